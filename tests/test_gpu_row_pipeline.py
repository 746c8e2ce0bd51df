"""The row pipelines (FLBM_ROWS=1; small boxes run the direct kernels by
default): populations against the oracle and, bit for bit, against the direct
kernels; the entry point without allocation; the padded layout; the reductions;
and that these boxes do run the kernels that the tests name.

Kernels: k_step_items (FP32 / FP16 rows of 32 to 256 nodes, several to an item
of up to 512 nodes), k_step_rows (FP64, and longer rows).  Tolerances are those
of the parity tests: 1e-12, 2e-6 and 2e-5 a step in FP64, FP32 and FP16.
"""
import ctypes as C

import numpy as np
import pytest

import reduction_sums as R
from synth import inputs

pytestmark = pytest.mark.gpu

TOL = {"fp64": 1e-12, "fp32": 2e-6, "fp16": 2e-5}


@pytest.fixture(autouse=True)
def rows(monkeypatch):
    monkeypatch.setenv("FLBM_ROWS", "1")


@pytest.fixture(scope="module")
def F():
    from paper_2601_03806_gb300 import flbm
    return flbm


def perturbed(O, shape, seed):
    nx, ny, nz = shape
    return O.tables()["w"][:, None, None, None] * (1.0 + 0.02 * inputs.population_perturbation(nx, ny, nz, seed))


# neighbours that coincide (one or two rows or planes), rows that fill an item
# of 512 nodes and rows that leave some of it empty (96, 160, 192, 224), items
# cut short by the plane's end, one node and two nodes per thread, 144 pairs
SHAPES = [(32, 3, 2), (64, 5, 4), (96, 2, 1), (32, 1, 1), (64, 1, 2), (256, 1, 1), (256, 2, 1), (512, 1, 2),
          (288, 3, 2), (32, 17, 2), (96, 7, 3), (128, 4, 1), (160, 4, 2), (192, 3, 3), (224, 5, 1), (224, 1, 3)]


@pytest.mark.parametrize("prec", ["fp64", "fp32", "fp16"])
@pytest.mark.parametrize("shape", SHAPES)
def test_populations_match_the_oracle(F, oracle_mod, shape, prec):
    f0 = perturbed(oracle_mod, shape, shape[1] * 7 + shape[2])
    for scheme in ("bgk", "gmf", "reg"):
        g = F.Lattice(*shape, 0.7, 1e-4, seed=13, scheme=scheme, precision=prec)
        o = oracle_mod.Box(*shape, 0.7, 1e-4, seed=13, scheme=F.SCHEMES[scheme])
        g.set_populations(f0)
        o.set_f(f0)
        for nsteps in (1, 2, 5):
            g.step(nsteps)
            o.step(nsteps)
            assert np.abs(g.get_populations() - o.get_f()).max() < TOL[prec] * nsteps
        g.close()


# more than five items per resident CTA (two per SM in FP32, three in FP16), so
# that the stages are reused, barriers wrap and sums are folded in the loop;
# planes whose last item is one row; an FP64 box of many rows per CTA
@pytest.mark.parametrize("prec,shape", [("fp32", (96, 41, 256)), ("fp16", (96, 41, 320)), ("fp32", (224, 33, 130)),
                                        ("fp16", (160, 31, 200)), ("fp32", (32, 49, 500)), ("fp32", (288, 40, 100)),
                                        ("fp16", (480, 40, 120)), ("fp64", (64, 40, 60)), ("fp64", (96, 10, 16))])
def test_many_items_per_cta_match_the_direct_kernel(F, monkeypatch, prec, shape):
    for scheme in ("bgk", "gmf", "reg"):
        a = F.Lattice(*shape, 0.7, 1e-4, seed=13, scheme=scheme, precision=prec)
        monkeypatch.setenv("FLBM_ROWS", "0")
        b = F.Lattice(*shape, 0.7, 1e-4, seed=13, scheme=scheme, precision=prec)
        monkeypatch.setenv("FLBM_ROWS", "1")
        for box in (a, b):
            box.init_thermal(8)
        for steps in (1, 3):
            for box in (a, b):
                box.step(steps)
            assert np.array_equal(a.get_state(), b.get_state())
        sa, sb = a.stats(), b.stats()
        rtol = 1e-12 if prec == "fp64" else 1e-5
        assert np.allclose(sa["u2_avg"], sb["u2_avg"], rtol=rtol) and np.allclose(sa["m_var"], sb["m_var"], rtol=rtol)
        a.close()
        b.close()


def kernels(run):
    """Names of the kernels that run() launches."""
    import torch
    from torch.profiler import ProfilerActivity, profile
    for _ in range(3):   # a process's first profile may miss everything
        with profile(activities=[ProfilerActivity.CUDA]) as p:
            run()
            torch.cuda.synchronize()
        names = {e.name for e in p.events()}
        if names:
            break
    return names


@pytest.mark.parametrize("prec,shape,name", [
    ("fp32", (32, 3, 2), "k_step_items"), ("fp32", (256, 2, 1), "k_step_items"), ("fp16", (96, 7, 3), "k_step_items"),
    ("fp32", (288, 3, 2), "k_step_rows"), ("fp16", (288, 3, 2), "k_step_rows"), ("fp32", (512, 1, 2), "k_step_rows"),
    ("fp16", (512, 1, 2), "k_step_rows"), ("fp64", (64, 5, 4), "k_step_rows"), ("fp64", (96, 10, 16), "k_step_rows"),
    # the direct kernels' boxes, as a check of the check
    ("fp32", (30, 4, 3), "k_step<"), ("fp64", (30, 4, 3), "k_step_few")])
def test_the_named_kernel_runs(F, prec, shape, name):
    box = F.Lattice(*shape, 0.7, 1e-4, seed=3, precision=prec)
    box.step(1)
    got = kernels(lambda: box.step(2))
    assert any(name in k for k in got), got
    assert not any("k_step" in k and name not in k for k in got), got
    box.close()


# boxes of 2^19 nodes and more: grouped rows from 224 nodes an item
@pytest.mark.parametrize("prec", ["fp32", "fp16"])
@pytest.mark.parametrize("shape,name", [((32, 1, 16384), "k_step<"), ((32, 6, 2731), "k_step<"),
                                        ((64, 3, 2731), "k_step<"), ((96, 2, 2731), "k_step<"),
                                        ((32, 7, 2341), "k_step_items"), ((64, 4, 2048), "k_step_items"),
                                        ((224, 1, 2341), "k_step_items"), ((256, 1, 2048), "k_step_items")])
def test_thin_boxes_take_the_direct_kernel(F, monkeypatch, prec, shape, name):
    """By default, and with the same populations as the pipeline's."""
    a = F.Lattice(*shape, 0.7, 1e-4, seed=3, precision=prec)
    monkeypatch.delenv("FLBM_ROWS")
    b = F.Lattice(*shape, 0.7, 1e-4, seed=3, precision=prec)
    for box in (a, b):
        box.init_thermal(6)
        box.step(1)
    got = kernels(lambda: b.step(2))
    assert any(name in k for k in got), got
    assert not any("k_step" in k and name not in k for k in got), got
    a.step(b.step_count - a.step_count)
    assert np.array_equal(a.get_state(), b.get_state())
    a.close()
    b.close()


@pytest.mark.parametrize("shape", [(64, 6, 5), (96, 5, 3), (256, 3, 2), (288, 3, 2), (512, 3, 2)])
def test_the_call_without_allocation_matches(F, oracle_mod, shape):
    import torch
    n = shape[0] * shape[1] * shape[2]
    for scheme in (0, 1, 2):
        box = F.Lattice(*shape, 0.7, 1e-4, seed=5, scheme=scheme, stats_every=1, torch_memory=True)
        f0 = perturbed(oracle_mod, shape, 11)
        box.set_populations(f0)
        o = oracle_mod.Box(*shape, 0.7, 1e-4, seed=5, scheme=scheme)
        o.set_f(f0)
        torch.cuda.synchronize()
        ns = int(F.flbm_state_bytes(C.byref(box.params))) // (27 * 4)
        slabs = box._buf.view(torch.float32).view(27, ns)[:, :n]
        state = slabs.clone(memory_format=torch.contiguous_format)
        sums = torch.zeros(13, dtype=torch.float64, device="cuda")
        for t in range(3):
            rc = F.flbm_step_noalloc(C.byref(box.params), C.c_void_p(state.data_ptr()), t, t % 2,
                                     C.c_void_p(sums.data_ptr()), C.c_void_p(box.stream.cuda_stream))
            assert rc == F.FLBM_OK, F.flbm_last_error(None)
            box.step(1)
            o.step(1)
            torch.cuda.synchronize()
            assert torch.equal(state, slabs)
            assert np.array_equal(box.stats()["mom"], sums.cpu().numpy()[1:4])
            assert np.abs(box.get_populations() - o.get_f()).max() < 2e-6 * (t + 1)
        box.close()


@pytest.mark.parametrize("prec", ["fp64", "fp32", "fp16"])
@pytest.mark.parametrize("shape", [(64, 5, 3), (96, 6, 2), (288, 3, 2), (512, 3, 2)])
def test_the_pad_is_invisible(F, monkeypatch, prec, shape):
    ref = None
    for pad in ("0", "2048", "1048576"):
        monkeypatch.setenv("FLBM_SLAB_PAD", pad)
        for torch_memory in (False, True):
            box = F.Lattice(*shape, 0.7, 1e-4, seed=9, precision=prec, torch_memory=torch_memory)
            box.init_thermal(4)
            box.step(5)
            got = box.get_state(), box.stats()
            box.close()
            ref = ref or got
            assert np.array_equal(got[0], ref[0]) and got[1] == ref[1]


# a thread adds at most 16 nodes to a lane in FP32 before its warp folds them
# (8 rows of two pairs in k_step_rows; 8 nodes in k_step_items)
@pytest.mark.parametrize("prec", ["fp32", "fp16"])
@pytest.mark.parametrize("shape", [(64, 12, 10), (96, 41, 30), (512, 16, 8), (288, 20, 40)])
def test_reductions_match_the_oracle(F, oracle_mod, prec, shape):
    n, rho0, kT = shape[0] * shape[1] * shape[2], 1.0, 1e-4
    box = F.Lattice(*shape, 0.7, kT, rho0=rho0, seed=21, precision=prec, stats_every=1)
    box.init_thermal(7)
    for _ in range(4):
        S, B = R.sums_and_bounds(oracle_mod, box.get_populations(), rho0, 16)
        ref, bound = R.stats_from_sums(S, n, rho0, kT), R.stats_bounds(S, B, n, rho0, kT)
        box.stats_reset()
        box.step(1)
        st = box.stats()
        for k in ref:
            assert np.all(np.abs(np.asarray(st[k], float) - np.asarray(ref[k], float)) <= np.asarray(bound[k], float)), k
    box.close()


@pytest.mark.parametrize("prec,shape", [("fp32", (64, 6, 5)), ("fp64", (32, 4, 3)), ("fp16", (256, 3, 2)),
                                        ("fp32", (512, 3, 2)), ("fp64", (64, 32, 8))])
def test_steps_of_one_call_are_those_of_many(F, prec, shape):
    """37 steps in one call (each launched while the one before still runs), one
    by one, and 16 + 20 + 1: the same populations and the same sums."""
    got = []
    for calls in ([37], [1] * 37, [16, 20, 1]):
        box = F.Lattice(*shape, 0.8, 1e-4, seed=2, precision=prec)
        box.init_thermal(7)
        for n in calls:
            box.step(n)
        got.append((box.get_state(), box.stats()))
        box.close()
    for g in got[1:]:
        assert np.array_equal(g[0], got[0][0]) and g[1] == got[0][1]


def test_fp64_noise_of_the_row_kernel_matches_the_oracle(F, oracle_mod):
    """One step from rest is the noise alone; the bound of the direct kernels'
    test: 2^-46 of sqrt(3 kT)."""
    shape, kT = (32, 31, 29), 1e-2
    box = F.Lattice(*shape, 1.0, kT, seed=99, precision="fp64")
    ref = oracle_mod.Box(*shape, 1.0, kT, seed=99)
    box.step(1)
    ref.step(1)
    assert np.abs(box.get_populations() - ref.get_f()).max() <= 2.0 ** -46 * np.sqrt(3 * kT)
