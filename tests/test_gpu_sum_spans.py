"""The fused reductions of FP32 boxes add at most 256 nodes in plain FP32 before
a partial sum enters the warp's exact pair.

Rest populations of whole numbers between 61,000 and 65,535 make it visible:
any 256 of them add up below 2^24, so every FP32 sum is exact and the total
mass is the exact whole number; a sum over more nodes has to round.  The two
kernels of two nodes per thread: grouped rows, with several items per CTA, and
the direct kernel, with several groups per CTA."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(128, 64, 128), (96, 83, 128), (250, 61, 67)])
def test_mass_of_whole_numbers_is_exact(shape):
    from paper_2601_03806_gb300 import flbm
    nx, ny, nz = shape
    box = flbm.Lattice(nx, ny, nz, 0.8, 0.0, precision="fp32")
    g = np.zeros((27, nz, ny, nx), np.float32)
    g[0] = np.random.default_rng(7).integers(61000, 65536, size=(nz, ny, nx))
    box.set_state(g)
    box.step(1)
    assert box.stats()["mass"] == box.n + g[0].sum(dtype=np.int64)
    box.close()
