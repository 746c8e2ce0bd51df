"""Totals of the reduced steps (formed 16 steps at a time), the FP64 normals
from tables, and the training pairs, where their code branches."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def F():
    from paper_2601_03806_gb300 import flbm
    return flbm


@pytest.mark.parametrize("every", [1, 3])
@pytest.mark.parametrize("prec,shape", [("fp32", (64, 6, 5)), ("fp64", (5, 4, 3)), ("fp16", (256, 3, 2))])
def test_totals_do_not_depend_on_how_steps_are_called(F, every, prec, shape):
    """37 steps in one call, one by one, and 16 + 20 + 1: the same sums."""
    got = []
    for calls in ([37], [1] * 37, [16, 20, 1]):
        box = F.Lattice(*shape, 0.8, 1e-4, seed=2, precision=prec, stats_every=every)
        box.init_thermal(7)
        for n in calls:
            box.step(n)
        got.append(box.stats())
    assert got[0]["n_samples"] == (37 if every == 1 else 13)
    assert got[0]["step"] == 36
    assert got[0] == got[1] == got[2]


def test_moment_state_totals(F):
    """The first step's totals come from another kernel and grid."""
    a = F.Lattice(64, 20, 33, 0.8, 1e-4, seed=2, state_form="moments")
    b = F.Lattice(64, 20, 33, 0.8, 1e-4, seed=2)
    for box in (a, b):
        box.init_thermal(7)
        box.step(19)
    sa, sb = a.stats(), b.stats()
    assert sa["n_samples"] == sb["n_samples"] == 19
    assert np.allclose(sa["u2_avg"], sb["u2_avg"], rtol=1e-5)
    assert np.allclose(sa["m_var"], sb["m_var"], rtol=1e-4)


@pytest.mark.parametrize("shape", [(32, 31, 29), (37, 21, 19)])
def test_fp64_noise_matches_the_oracle(F, oracle_mod, shape):
    """One step from rest is the noise alone (27,000 nodes, 325,000 pairs of
    normals, row and direct kernels): a radius and an angle good to 2^-52 and
    2^-52, 23 terms of size sqrt(3 kT) at most, summed in three passes: 2^-46
    of that scale."""
    kT = 1e-2
    box = F.Lattice(*shape, 1.0, kT, seed=99, precision="fp64")
    ref = oracle_mod.Box(*shape, 1.0, kT, seed=99)
    box.step(1)
    ref.step(1)
    assert np.abs(box.get_populations() - ref.get_f()).max() <= 2.0 ** -46 * np.sqrt(3 * kT)


@pytest.mark.parametrize("prec", ["fp32", "fp16", "fp64"])
@pytest.mark.parametrize("shape,steps", [((1, 1, 1), 0), ((127, 1, 1), 1), ((43, 3, 1), 0), ((33, 5, 7), 1)])
def test_pairs_match_oracle_at_block_edges(F, oracle_mod, prec, shape, steps):
    """As the existing test of the pairs: FP64 results stored in FP32."""
    import torch
    from oracle import mlp as M
    tau, kT, rho0 = 0.7, 1e-5, 1.1
    box = F.Lattice(*shape, tau, kT, rho0=rho0, seed=4, scheme=F.FLBM_REG, precision=prec)
    box.init_thermal(9)
    box.step(steps)
    f = box.get_populations().reshape(27, -1).T
    n = f.shape[0]
    x, t = torch.full((n + 1, 28), 7.0, device="cuda"), torch.full((n + 1, 27), 7.0, device="cuda")
    box.mlp_pairs(x, t)
    x, t = x.cpu().numpy().astype(float), t.cpu().numpy().astype(float)
    assert (x[n] == 7).all() and (t[n] == 7).all()
    xo = M.features(f, rho0, kT, 1.0 / tau)
    to = np.array([M.target(v, tau, rho0, kT) for v in f])
    assert np.abs(x[:n] - xo).max() <= 1e-6 * (1 + np.abs(xo).max())
    assert np.abs(t[:n] - to).max() <= 2e-6 * np.abs(to).max() + 1e-7
