"""Initial solutions over the nonzero lists of A (a block of four warps per
start, moments in registers for n <= 512) and over the dense A, at the edges of
the lists' groups of 32, of the 128 threads and of the registers: the same
per-step comparison with the oracle as for the headline sizes."""
import pytest

from paper_2412_13576_gb300 import instances as I

from .test_gpu_init import M, test_init_per_step as per_step  # noqa: F401  (M: the fixture)

pytestmark = pytest.mark.gpu
per_step.__test__ = False


@pytest.mark.parametrize("n,m,density", [
    (33, 1, 0.1),      # one row; the last group of columns holds one
    (97, 64, 0.3),
    (128, 31, 0.05),   # exactly one coordinate a thread
    (129, 33, 0.2),    # ragged groups both ways
    (200, 90, 0.0),    # lists of one entry
    (512, 100, 0.02),  # the last n with the moments in registers
    (513, 129, 0.02),  # the first without
    (130, 40, None),   # rows more than half full: the dense A
    (513, 20, None),
])
def test_lists_and_dense_per_step(M, n, m, density):  # noqa: F811
    per_step(M, lambda: I.make_instance("lists", n, m, c_k=2, c_density=density, lo=-4, hi=6, q_k=1, q_density=0.01,
                                        lin_k=1, seed=n + m), 65, 3)
