"""Initial solutions of the smallest A, whose two ways through the steps share
one launch: sparse and dense A, a few starts to many, at the edges of the groups
of four starts and 32 rows and of the shared memory that the launch may take."""
import pytest

from paper_2412_13576_gb300 import instances as I

from .test_gpu_init import M, test_init_per_step as per_step  # noqa: F401  (M: the fixture)

pytestmark = pytest.mark.gpu
per_step.__test__ = False


@pytest.mark.parametrize("n,m,density", [(2, 1, None), (6, 2, 0.1), (20, 5, 0.1), (20, 5, None), (33, 4, 0.05),
                                         (64, 4, 0.05), (64, 4, None), (40, 33, 0.05)])
@pytest.mark.parametrize("P", [2, 5, 133])
def test_small_per_step(M, n, m, density, P):  # noqa: F811
    per_step(M, lambda: I.make_instance("small", n, m, c_k=2, c_density=density, lo=-4, hi=6, q_k=1, q_density=0.01,
                                        lin_k=1, seed=n + m), P, 3)
