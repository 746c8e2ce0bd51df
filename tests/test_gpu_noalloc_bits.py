"""flbm_step_noalloc's sums are flbm_step's to the last bit: the interface says
that they equal those of flbm_step + flbm_stats, and both form them from the
same partials in the same order.  Densities over sixty binades, one per 256
nodes, so that FP64 rounds and the order shows; boxes of one CTA and of
hundreds, of the direct kernel and of the row pipeline."""
import ctypes as C

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows", ["0", "1"])
@pytest.mark.parametrize("shape", [(30, 4, 3), (64, 32, 31), (64, 64, 60), (160, 50, 40), (512, 20, 30)])
def test_sums_have_the_same_bits(monkeypatch, shape, rows):
    import torch

    from paper_2601_03806_gb300 import flbm

    monkeypatch.setenv("FLBM_ROWS", rows)
    n = shape[0] * shape[1] * shape[2]
    box = flbm.Lattice(*shape, 0.7, 0.0, seed=5, precision="fp32", stats_every=1, torch_memory=True)
    rng = np.random.default_rng(n)
    g = (rng.normal(size=(27, n)) * 2.0 ** -rng.uniform(8, 60, size=n // 256 + 1)[np.arange(n) // 256]).astype(np.float32)
    box.set_state(g.reshape(27, *shape[::-1]))
    torch.cuda.synchronize()
    ns = int(flbm.flbm_state_bytes(C.byref(box.params))) // (27 * 4)
    slabs = box._buf.view(torch.float32).view(27, ns)[:, :n]
    state = slabs.clone(memory_format=torch.contiguous_format)
    sums = torch.zeros(13, dtype=torch.float64, device="cuda")
    for t in range(3):
        rc = flbm.flbm_step_noalloc(C.byref(box.params), C.c_void_p(state.data_ptr()), t, t % 2,
                                    C.c_void_p(sums.data_ptr()), C.c_void_p(box.stream.cuda_stream))
        assert rc == flbm.FLBM_OK, flbm.flbm_last_error(None)
        box.stats_reset()
        box.step(1)
        torch.cuda.synchronize()
        assert torch.equal(state, slabs)
        s, st = sums.cpu().numpy(), box.stats()
        assert st["mass"] == n + s[0]
        assert np.array_equal(st["mom"], s[1:4])
        assert np.array_equal(st["u2"], s[4:7] / n)
        assert np.array_equal(st["m_mean"], np.array([s[0], (s[1] + s[2]) + s[3], s[7], s[8]]) / n)
    box.close()
