"""The direct kernel's shapes: flat nodes, one per thread in CTAs of a warp
(small boxes) and two per thread, 128 apart, with the next ones staged (from
65,536 nodes): ends of groups, rows shorter and longer than a group, one lane
without a partner.

One node per thread (FLBM_ROW_PAIRS=0) gives the same populations, bit for
bit, and both the oracle's to the FP32 step tolerance (2e-6 per step).
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def F():
    from paper_2601_03806_gb300 import flbm
    return flbm


def state(F, shape, steps, prec, scheme, seed=3):
    box = F.Lattice(*shape, 0.7, 1e-4, seed=seed, precision=prec, scheme=scheme)
    box.init_thermal(5)
    box.step(steps)
    return box.get_state(), box.stats()


# 65,537 nodes leave one lane without a partner; 65,536 + 128 exactly one
# half group; rows of 1, 3, 255, 257 and of the whole box
@pytest.mark.parametrize("prec", ["fp32", "fp16"])
@pytest.mark.parametrize("shape", [(65537, 1, 1), (1, 65664, 1), (3, 5, 4400), (255, 257, 1), (257, 1, 256),
                                   (37, 43, 61), (250, 31, 17)])
def test_two_nodes_per_thread_give_the_same_bits(F, monkeypatch, prec, shape):
    for scheme in ("gmf", "bgk", "reg"):
        a, sa = state(F, shape, 3, prec, scheme)
        monkeypatch.setenv("FLBM_ROW_PAIRS", "0")
        b, sb = state(F, shape, 3, prec, scheme)
        monkeypatch.delenv("FLBM_ROW_PAIRS")
        assert np.array_equal(a, b)
        assert np.allclose(sa["u2"], sb["u2"], rtol=1e-5) and np.allclose(sa["m_var"], sb["m_var"], rtol=1e-4)


# FP64: an SM's warps share 32 nodes up to 4,864
@pytest.mark.parametrize("shape", [(37, 43, 61), (31, 1, 1), (33, 1, 1), (5, 13, 31), (19, 16, 16), (4865, 1, 1)])
def test_against_the_oracle(F, oracle_mod, shape):
    nx, ny, nz = shape
    f0 = F.Lattice(nx, ny, nz, 0.8, 1e-4, seed=8)
    f0.init_thermal(4)
    f = f0.get_populations()
    for prec, tol in (("fp64", 1e-13), ("fp32", 2e-6)):
        box = F.Lattice(nx, ny, nz, 0.8, 1e-4, seed=8, precision=prec)
        box.set_populations(f)
        ref = oracle_mod.Box(nx, ny, nz, 0.8, 1e-4, seed=8)
        ref.set_f(f)
        for steps in (1, 2):
            box.step(steps)
            ref.step(steps)
            assert np.abs(box.get_populations() - ref.get_f()).max() <= tol * 3
