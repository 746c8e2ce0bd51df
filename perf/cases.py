"""The work that the library's performance is followed on: listed() and
draw() name cases, prepare() builds what a program holds before the call,
run() is one pass through the public entry points, work() the bytes and
operations a pass cannot do without, and exact() the same results in 64 bits
from plain torch / numpy.

A box keeps its populations in a torch buffer handed to flbm_create_ex (27
slabs of ns elements, slot i of node n at i ns + n) and starts from a sample
of the lattice invariant measure, as the equilibrium-fluctuation runs do.
Steps come in even numbers, after which the slabs are in natural order.

Results: the populations are the box's own buffer.  The fused statistics and
the training losses of FP32 arithmetic are returned as FP32 (their order of
addition is not part of the interface; it is fixed to 1e-5), those of FP64
boxes as FP64; spectra and moments as the library returns them.
"""
import ctypes
import math

import numpy as np
import torch

from paper_2601_03806_gb300 import flbm

Q = 27
OBSERVABLES = (flbm.FLBM_OBS_RHO, flbm.FLBM_OBS_JSUM, flbm.FLBM_OBS_PI_DIAG, flbm.FLBM_OBS_PI_OFFDIAG)
TORCH_TYPE = {"fp64": torch.float64, "fp32": torch.float32, "fp16": torch.float16}


def _box(name, nx, ny, nz, precision="fp32", scheme="gmf", tau=0.6, kT=1e-5, steps=2, spectra=0, moments=False):
    return {"name": name, "kind": "box", "nx": nx, "ny": ny, "nz": nz, "precision": precision, "scheme": scheme,
            "tau": tau, "kT": kT, "steps": steps, "spectra": spectra, "moments": moments}


def listed():
    return [
        # the parity box of the tests: FP64, launches and latency count
        _box("parity16_f64", 16, 16, 16, precision="fp64", tau=0.8, kT=1e-4, steps=20),
        # the flat-S(k) sampling loop: 25 steps, then the spectra and moments
        _box("sample64_f32", 64, 64, 64, tau=0.8, steps=24, spectra=4, moments=True),
        # the statistics box run for many tau: the everyday size
        _box("box128_f32", 128, 128, 128, steps=20),
        # row lengths that no tile divides
        _box("ragged_f32", 250, 243, 121, scheme="bgk", tau=1.0, steps=8),
        # the paper's lattice and kT, the regularized scheme it compares
        _box("box256_reg_f32", 256, 256, 256, scheme="reg", kT=1.0 / 3000, steps=8),
        # the headline box, in both storages it is run in
        _box("box512_f32", 512, 512, 512, steps=2),
        _box("box512_f16", 512, 512, 512, precision="fp16", steps=2),
        # double precision at the size of the statistics box
        _box("box128_f64", 128, 128, 128, precision="fp64", tau=0.8, kT=1e-4, steps=2),
        # a snapshot of the paper's lattice: the spectral ratios of its four
        # observables
        _box("spectra256_f32", 256, 256, 256, kT=1.0 / 3000, steps=0, spectra=4),
        # the mixed ensemble, sampled every 20 steps
        {"name": "ensemble", "kind": "ensemble", "n32": 256, "n64": 64, "n128": 8, "precision": "fp32",
         "scheme": "gmf", "kT": 1e-5, "steps": 20},
        # the learned collision on the paper's lattice
        _box("learned256", 256, 256, 256, scheme="learned", tau=0.8, steps=4),
        # training pairs of one 64^3 box and an epoch of training on them
        {"name": "train", "kind": "train", "nx": 64, "ny": 64, "nz": 64, "tau": 0.8, "kT": 1e-5,
         "batch": 1024, "epochs": 1},
    ]


def _size(rng, lo, hi):
    n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    return max(lo, min(hi, n))


def _row(rng, lo, hi):
    """A row length: half of them multiples of 32, the others any number."""
    n = _size(rng, lo, hi)
    return max(32, n // 32 * 32) if rng.random() < 0.5 else n


def draw(rng):
    kind = rng.choice(["box", "box", "box", "sample", "learned", "ensemble", "train"])
    tau = round(rng.choice([0.51, 0.55, 0.6, 0.8, 1.0, 2.0, 5.0]) + 0.001 * rng.randrange(10), 4)
    kT = rng.choice([1e-5, 1e-4, 1.0 / 3000])
    if kind == "ensemble":
        return {"kind": "ensemble", "n32": rng.randrange(1, 257), "n64": rng.randrange(0, 65),
                "n128": rng.randrange(0, 9), "precision": rng.choice(["fp32", "fp32", "fp16"]),
                "scheme": rng.choice(["gmf", "reg", "bgk"]), "kT": 1e-5, "steps": 2 * rng.randrange(1, 11)}
    if kind == "train":
        return {"kind": "train", "nx": _size(rng, 16, 64), "ny": _size(rng, 16, 64), "nz": _size(rng, 16, 64),
                "tau": tau, "kT": 1e-5, "batch": rng.choice([256, 500, 1024, 2048, 4096]), "epochs": 1}
    if kind == "learned":
        c = _box("", _row(rng, 16, 256), _size(rng, 16, 256), _size(rng, 16, 256), scheme="learned", tau=tau,
                 steps=2 * rng.randrange(1, 3))
    else:
        precision = rng.choice(["fp32", "fp32", "fp32", "fp16", "fp64"])
        hi = 128 if precision == "fp64" else 512
        c = _box("", _row(rng, 8, hi), _size(rng, 8, hi), _size(rng, 8, hi), precision=precision,
                 scheme=rng.choice(["gmf", "gmf", "bgk", "reg"]), tau=tau if tau > 0.52 else 0.6, kT=kT)
        n = c["nx"] * c["ny"] * c["nz"]
        c["steps"] = 2 * rng.randrange(1, 1 + max(1, min(10, (1 << 24) // n)))
        if kind == "sample" and n <= 1 << 24:
            c["spectra"], c["moments"] = 4, n <= 1 << 18
    del c["name"]
    return c


# ---------------------------------------------------------------------------
# what a program holds


class _Box:
    """One flbm_ctx on a torch buffer and torch's current stream."""

    def __init__(self, case, seed):
        self.params = flbm.make_params(case["nx"], case["ny"], case["nz"], case["tau"], case["kT"], seed=seed,
                                       scheme=case["scheme"], precision=case["precision"])
        n = case["nx"] * case["ny"] * case["nz"]
        nbytes = int(flbm.flbm_state_bytes(ctypes.byref(self.params)))
        self.buf = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
        self.g = self.buf.view(TORCH_TYPE[case["precision"]]).view(Q, -1)
        self.h = ctypes.c_void_p()
        self.check(flbm.flbm_create_ex(ctypes.byref(self.params), self.buf.data_ptr(), nbytes,
                                       torch.cuda.current_stream().cuda_stream, ctypes.byref(self.h)))
        _thermal_into(self.g, n, case["kT"], seed)
        torch.cuda.synchronize()

    def check(self, rc):
        if rc != flbm.FLBM_OK:
            raise flbm.FlbmError(rc, flbm.flbm_last_error(self.h).decode())

    def __del__(self):
        if getattr(self, "h", None):
            flbm.flbm_destroy(self.h)
            self.h = None


def _weights():
    """(c[27][3], w[27]) in the interface's velocity order."""
    c = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1)]
    for a, b in ((0, 1), (0, 2), (1, 2)):
        for s in ((1, 1), (-1, -1), (1, -1), (-1, 1)):
            v = [0, 0, 0]
            v[a], v[b] = s
            c.append(tuple(v))
    c += [(1, 1, 1), (-1, -1, -1), (1, 1, -1), (-1, -1, 1), (1, -1, 1), (-1, 1, -1), (-1, 1, 1), (1, -1, -1)]
    w = [{0: 8 / 27, 1: 2 / 27, 2: 1 / 54, 3: 1 / 216}[sum(x * x for x in v)] for v in c]
    return c, w


def _thermal_into(g, n, kT, seed):
    """Deviations of the invariant measure, N(0, kT w_i / c_s^2), rho0 = 1."""
    gen = torch.Generator(device=g.device)
    gen.manual_seed(seed)
    for i, w in enumerate(_weights()[1]):
        draw_type = torch.float64 if g.dtype == torch.float64 else torch.float32
        z = torch.randn(n, generator=gen, device=g.device, dtype=draw_type)
        g[i, :n] = z.mul_(math.sqrt(3.0 * kT * w)).to(g.dtype)


def _network(seed):
    """Initial parameters: normal weights of variance 1 / inputs, zero biases."""
    rng = np.random.default_rng(seed)
    parts = []
    for nin, nout in ((28, 64), (64, 64), (64, 27)):
        parts += [rng.normal(0, math.sqrt(1.0 / nin), nout * nin), np.zeros(nout)]
    return np.concatenate(parts).astype(np.float32)


def _replicas(case, seed):
    """(sizes, taus) of the ensemble's replicas; replica r has noise stream r."""
    sizes = [32] * case["n32"] + [64] * case["n64"] + [128] * case["n128"]
    return sizes, np.random.default_rng(seed).uniform(0.51, 3.0, size=len(sizes))


def _probes(sizes):
    """Replicas looked into (the first of each size) and the nodes there."""
    first = sorted({sizes.index(n) for n in sizes})
    return [(r, np.arange(0, sizes[r] ** 3, sizes[r] ** 3 // 2048 + 1, dtype=np.int64)) for r in first]


def prepare(case, seed):
    if case["kind"] == "ensemble":
        sizes, taus = _replicas(case, seed)
        ps = [flbm.make_params(n, n, n, float(tau), case["kT"], seed=seed, scheme=case["scheme"],
                               precision=case["precision"], noise_stream=r)
              for r, (n, tau) in enumerate(zip(sizes, taus))]
        ens = flbm.Ensemble(ps)
        ens.autotune(4)
        for r in range(len(sizes)):
            ens[r].init_thermal(seed + r)
        return {"case": case, "ens": ens, "probes": _probes(sizes)}
    if case["kind"] == "train":
        box = _Box(dict(case, scheme="reg", precision="fp32"), seed)
        n = case["nx"] * case["ny"] * case["nz"]
        return {"case": case, "box": box, "theta": _network(seed), "seed": seed,
                "x": torch.empty((n, 28), device="cuda"), "t": torch.empty((n, 27), device="cuda")}
    box = _Box(case, seed)
    if case["scheme"] == "learned":
        net = _network(seed)
        box.check(flbm.flbm_set_mlp(box.h, net.ctypes.data))
    return {"case": case, "box": box}


# ---------------------------------------------------------------------------
# one pass


def _read_stats(check, h, dtype):
    s = flbm.flbm_stats_t()
    check(flbm.flbm_stats(h, ctypes.byref(s)))
    return {"mass": np.array([s.mass], dtype), "mom": np.array(s.mom, dtype), "u2": np.array(s.u2, dtype),
            "u2_avg": np.array(s.u2_avg, dtype), "m_mean": np.array(s.m_mean, dtype),
            "m_var": np.array(s.m_var, dtype), "er": np.array(s.er, dtype)}


def _nshell(case):
    return min(case["nx"], case["ny"], case["nz"]) // 2 + 1


def run(state):
    case = state["case"]
    if case["kind"] == "ensemble":
        ens = state["ens"]
        ens.step(case["steps"])
        per = [_read_stats(r._check, r.handle, np.float32) for r in ens.replicas]
        out = {k: np.stack([p[k] for p in per]) for k in per[0]}
        out["f"] = [ens[r].probe(nodes) for r, nodes in state["probes"]]
        return out
    box = state["box"]
    if case["kind"] == "train":
        x, t = state["x"], state["t"]
        box.check(flbm.flbm_mlp_pairs(box.h, x.data_ptr(), t.data_ptr()))
        theta, losses = flbm.mlp_train(state["theta"], x, t, epochs=case["epochs"], batch=case["batch"], lr=1e-2,
                                       seed=state["seed"])
        return {"x": x, "t": t, "theta": theta, "losses": losses.astype(np.float32)}
    out = {}
    if case["steps"]:
        box.check(flbm.flbm_step(box.h, case["steps"]))
        out["g"] = box.g
        out["stats"] = _read_stats(box.check, box.h, np.float64 if case["precision"] == "fp64" else np.float32)
    if case["spectra"]:
        k = _nshell(case)
        out["er"] = np.zeros((case["spectra"], k))
        out["count"] = np.zeros((case["spectra"], k), np.int64)
        for o in range(case["spectra"]):
            box.check(flbm.flbm_spectral_er(box.h, OBSERVABLES[o], k, out["er"][o].ctypes.data,
                                            out["count"][o].ctypes.data))
    if case["moments"]:
        shape = (case["nz"], case["ny"], case["nx"])
        out["rho"], out["j"], out["pi"] = np.empty(shape), np.empty((3,) + shape), np.empty((6,) + shape)
        box.check(flbm.flbm_moments(box.h, out["rho"].ctypes.data, out["j"].ctypes.data, out["pi"].ctypes.data))
    return out


# A node's collision: two 27-point transforms in three 3-point passes of four
# operations, six relaxed moments, 13 statistics, 23 normals (a radius and an
# angle for two, the scaling and the addition).
STEP_FLOPS = 216 + 60 + 40 + 23 * 6
NET_FLOPS = 2 * (28 * 64 + 64 * 64 + 64 * 27)


def work(case):
    if case["kind"] == "ensemble":
        n = case["n32"] * 32 ** 3 + case["n64"] * 64 ** 3 + case["n128"] * 128 ** 3
        es = 2 if case["precision"] == "fp16" else 4
        return {"bytes": case["steps"] * n * 2 * Q * es, "flops": case["steps"] * n * STEP_FLOPS}
    n = case["nx"] * case["ny"] * case["nz"]
    if case["kind"] == "train":
        back = 2 * (64 * 64 + 64 * 27)
        return {"bytes": n * 4 * (Q + 55) + case["epochs"] * n * 4 * 55,
                "flops": case["epochs"] * n * (2 * NET_FLOPS + back)}
    es = {"fp64": 8, "fp32": 4, "fp16": 2}[case["precision"]]
    flops = STEP_FLOPS + (NET_FLOPS if case["scheme"] == "learned" else 0)
    b, f = case["steps"] * n * 2 * Q * es, case["steps"] * n * flops
    # a spectrum reads the populations its observable weighs, and a transform
    # is 2.5 N log2 N operations
    b += case["spectra"] * n * es * 18
    f += case["spectra"] * n * int(Q + 2.5 * math.log2(n))
    if case["moments"]:
        b += n * (es * Q + 80)
        f += n * 100
    return {"bytes": b, "flops": f}


# ---------------------------------------------------------------------------
# the same results in 64 bits

_DEG2 = [(2, 0, 0), (0, 2, 0), (0, 0, 2), (1, 1, 0), (1, 0, 1), (0, 1, 1)]
_DEGREES = [(0, 0, 0), (1, 0, 0), (0, 1, 0), (0, 0, 1)] + _DEG2 + [
    (2, 1, 0), (2, 0, 1), (1, 2, 0), (1, 0, 2), (0, 2, 1), (0, 1, 2), (1, 1, 1), (2, 2, 0), (2, 0, 2), (0, 2, 2),
    (1, 1, 2), (1, 2, 1), (2, 1, 1), (2, 1, 2), (2, 2, 1), (1, 2, 2), (2, 2, 2)]
_LOW = 0xFFFFFFFF


def _philox(c0, c1, c2, c3, key0, key1):
    """Philox4x32-10 on int64 tensors or numbers below 2^32."""
    x = [c0, torch.full_like(c0, c1), torch.full_like(c0, c2), torch.full_like(c0, c3)]
    for _ in range(10):
        p0, p1 = x[0] * 0xD2511F53, x[2] * 0xCD9E8D57   # bits modulo 2^64
        x = [((p1 >> 32) & _LOW) ^ x[1] ^ key0, p1 & _LOW, ((p0 >> 32) & _LOW) ^ x[3] ^ key1, p0 & _LOW]
        key0, key1 = (key0 + 0x9E3779B9) & _LOW, (key1 + 0xBB67AE85) & _LOW
    return x


def _normals(node, step, blocks, stream, key):
    """Four normals per Philox block (Box-Muller on word pairs)."""
    out = []
    for blk in blocks:
        w = _philox(node, step & _LOW, blk | (stream << 8), step >> 32, key & _LOW, key >> 32)
        for a, b in ((0, 1), (2, 3)):
            u1, u2 = (((w[k] >> 9).double() + 0.5) * 2.0 ** -23 for k in (a, b))
            rad = torch.sqrt(-2.0 * torch.log(u1))
            out += [rad * torch.cos(2.0 * math.pi * u2), rad * torch.sin(2.0 * math.pi * u2)]
    return out


class _Lattice64:
    """A batch of equal periodic boxes g[27][R][nz][ny][nx] in FP64."""

    def __init__(self, g, taus, streams, scheme, kT, seed, net=None):
        self.g, self.scheme, self.kT, self.seed, self.net, self.t = g, scheme, kT, seed, net, 0
        dev = g.device
        c, w = _weights()
        self.c = c
        self.w = torch.tensor(w, dtype=torch.float64, device=dev)
        poly = [lambda v: 1.0, lambda v: float(v), lambda v: v * v - 1.0 / 3.0]
        e = [[poly[a](v[0]) * poly[b](v[1]) * poly[d](v[2]) for v in c] for a, b, d in _DEGREES]
        self.e = torch.tensor(e, dtype=torch.float64, device=dev)
        self.b = [(1.0, 1.0 / 3.0, 2.0 / 9.0)[a] * (1.0, 1.0 / 3.0, 2.0 / 9.0)[b] * (1.0, 1.0 / 3.0, 2.0 / 9.0)[d]
                  for a, b, d in _DEGREES]
        self.back = (self.w[:, None] * self.e.t()) / torch.tensor(self.b, dtype=torch.float64, device=dev)[None]
        self.taus, self.streams = taus, streams
        self.sums = torch.zeros((len(taus), 13), dtype=torch.float64, device=dev)
        self.u2, self.m1, self.m2 = (torch.zeros((len(taus), k), dtype=torch.float64, device=dev) for k in (3, 4, 4))

    def collide(self, g, r, z0):
        """Post-collision deviations of planes z0.. of box r from g[27][n]; adds its sums."""
        om = 1.0 / self.taus[r]
        m = self.e @ g
        rho = 1.0 + m[0]
        u = m[1:4] / rho
        jsum, diag = m[1] + m[2] + m[3], m[4] + m[5] + m[6] + m[0]
        off = m[7] + m[8] + m[9]
        terms = [m[0], m[1], m[2], m[3], u[0] ** 2, u[1] ** 2, u[2] ** 2, diag, off, m[0] ** 2, jsum ** 2,
                 diag ** 2, off ** 2]
        self.sums[r] += torch.stack([t.sum() for t in terms])

        def eq(k):
            a = rho
            for ax in range(3):
                for _ in range(_DEGREES[k][ax]):
                    a = a * u[ax]
            return a

        node = torch.arange(g.shape[1], device=g.device) + z0 * self.g.shape[3] * self.g.shape[4]
        normals = _normals(node, self.t, range(6), self.streams[r], self.seed)
        amp_h = math.sqrt(3.0 * self.kT * om * (2.0 - om))
        amp_g = amp_h if self.scheme == "bgk" else math.sqrt(3.0 * self.kT)
        sr = torch.sqrt(rho)
        for k in range(4, Q):
            if k < 10:
                m[k] = om * eq(k) + (1.0 - om) * m[k]
            elif self.scheme == "bgk":
                m[k] *= 1.0 - om
            elif self.scheme == "reg":
                m[k] = eq(k)
            else:
                m[k] = 0.0
            m[k] += (amp_h if k < 10 else amp_g) * math.sqrt(self.b[k]) * sr * normals[k - 4]
        out = self.back @ m
        if self.net is not None:
            d = self.w[:, None] * self.kT ** 1.5 * _forward64(self.net, _features64(g, self.w, self.kT, om).t())[0].t()
            ci = torch.tensor(self.c, dtype=torch.float64, device=g.device)
            out += d - self.w[:, None] * (d.sum(0) + 3.0 * (ci @ (ci.t() @ d)))
        return out

    def step(self):
        new = torch.empty_like(self.g)
        _, boxes, nz, ny, nx = self.g.shape
        planes = max(1, (1 << 23) // (nx * ny))
        self.sums.zero_()
        for r in range(boxes):
            for z0 in range(0, nz, planes):
                z1 = min(nz, z0 + planes)
                out = self.collide(self.g[:, r, z0:z1].reshape(Q, -1), r, z0).view(Q, z1 - z0, ny, nx)
                for i, (cx, cy, cz) in enumerate(self.c):
                    v = torch.roll(out[i], (cy, cx), (1, 2))
                    to = torch.arange(z0 + cz, z1 + cz, device=v.device) % nz
                    new[i, r, to] = v
        self.g = new
        n = nx * ny * nz
        s = self.sums / n
        self.u2 += s[:, 4:7]
        self.m1 += torch.stack([s[:, 0], s[:, 1] + s[:, 2] + s[:, 3], s[:, 7], s[:, 8]], 1)
        self.m2 += s[:, 9:13]
        self.t += 1

    def stats(self):
        n = self.g[0, 0].numel()
        mean = self.m1 / self.t
        var = self.m2 / self.t - mean ** 2
        theory = torch.tensor([3.0, 3.0, 5.0, 1.0], dtype=torch.float64, device=mean.device) * self.kT
        return {"mass": n + self.sums[:, :1], "mom": self.sums[:, 1:4], "u2": self.sums[:, 4:7] / n,
                "u2_avg": self.u2 / self.t, "m_mean": mean, "m_var": var, "er": var / theory}


def _spectra64(field, nshell):
    nz, ny, nx = field.shape
    spec = torch.fft.rfftn(field - field.mean())
    n2 = torch.zeros(spec.shape, dtype=torch.int64, device=field.device)
    for ax, (n, k) in enumerate(((nz, nz), (ny, ny), (nx, nx // 2 + 1))):
        a = torch.arange(k, device=field.device)
        if ax < 2:
            a = torch.where(2 * a < n, a, a - n)
        n2 += (a * a).view([-1 if d == ax else 1 for d in range(3)])
    s = torch.round(torch.sqrt(n2.double())).long()
    weight = torch.full(spec.shape, 2.0, dtype=torch.float64, device=field.device)
    weight[..., 0] = 1.0
    if nx % 2 == 0:
        weight[..., nx // 2] = 1.0
    use = (n2 > 0) & (s < nshell)
    power = torch.zeros(nshell, dtype=torch.float64, device=field.device)
    count = torch.zeros_like(power)
    power.index_add_(0, s[use], (weight * spec.abs() ** 2)[use] / field.numel())
    count.index_add_(0, s[use], weight[use])
    return power / count.clamp(min=1.0), count.long()


def _moments64(g, c):
    c = torch.tensor(c, dtype=torch.float64, device=g.device)
    pairs = [(0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2)]
    rho = g.sum(0) + 1.0
    j = torch.stack([torch.einsum("i,izyx->zyx", c[:, a], g) for a in range(3)])
    pi = torch.stack([torch.einsum("i,izyx->zyx", c[:, a] * c[:, b], g) + (1.0 / 3.0 if a == b else 0.0)
                      for a, b in pairs])
    return rho, j, pi


def _features64(g, w, kT, omega):
    x = torch.empty((28, g.shape[1]), dtype=torch.float64, device=g.device)
    x[:27] = g / torch.sqrt(3.0 * kT * w)[:, None]
    x[27] = omega - 1.0
    return x


def _layers(theta):
    out, at = [], 0
    for nin, nout in ((28, 64), (64, 64), (64, 27)):
        out.append((theta[at:at + nin * nout].view(nout, nin), theta[at + nin * nout:at + nin * nout + nout]))
        at += nin * nout + nout
    return out


def _forward64(theta, x):
    layers, kept = _layers(theta), [x]
    for k, (w, b) in enumerate(layers):
        z = x @ w.t() + b
        x = z * torch.sigmoid(z) if k < 2 else z
        kept += [z, x]
    return x, kept


def _gradient64(theta, x, t):
    y, (h0, z1, h1, z2, h2, _, _) = _forward64(theta, x)
    (w1, _), (w2, _), (w3, _) = _layers(theta)

    def dsilu(z):
        s = torch.sigmoid(z)
        return s * (1.0 + z * (1.0 - s))

    d3 = 2.0 * (y - t) / y.numel()
    d2 = (d3 @ w3) * dsilu(z2)
    d1 = (d2 @ w2) * dsilu(z1)
    grads = []
    for d, h in ((d1, h0), (d2, h1), (d3, h2)):
        grads += [(d.t() @ h).reshape(-1), d.sum(0)]
    return torch.cat(grads), ((y - t) ** 2).sum()


class _Mt64:
    """The 64-bit Mersenne twister (Nishimura 2000): the epoch order's source."""

    def __init__(self, seed):
        mask = (1 << 64) - 1
        self.s = [seed & mask]
        for i in range(1, 312):
            self.s.append((6364136223846793005 * (self.s[-1] ^ (self.s[-1] >> 62)) + i) & mask)
        self.at = 312

    def __call__(self):
        if self.at == 312:
            for i in range(312):
                x = (self.s[i] & 0xFFFFFFFF80000000) | (self.s[(i + 1) % 312] & 0x7FFFFFFF)
                self.s[i] = self.s[(i + 156) % 312] ^ (x >> 1) ^ (0xB5026F5AA96619E9 if x & 1 else 0)
            self.at = 0
        x = self.s[self.at]
        self.at += 1
        x ^= (x >> 29) & 0x5555555555555555
        x ^= (x << 17) & 0x71D67FFFEDA60000
        x ^= (x << 37) & 0xFFF7EEE000000000
        return x ^ (x >> 43)


def _train64(theta, x, t, epochs, batch, lr, seed):
    n = x.shape[0]
    batch = min(batch, n)
    nb = -(-n // batch)
    rng, it, losses = _Mt64(seed), 0, []
    m1, m2 = torch.zeros_like(theta), torch.zeros_like(theta)
    for _ in range(epochs):
        mult = 1 + rng() % (n - 1)
        while math.gcd(mult, n) != 1:
            mult = 1 + rng() % (n - 1)
        off, total = rng() % n, 0.0
        order = (torch.arange(n, device=x.device) * mult + off) % n
        for b in range(nb):
            take = order[b * batch:(b + 1) * batch]
            grad, loss = _gradient64(theta, x[take], t[take])
            total = total + loss
            rate = lr * (0.05 + 0.475 * (1.0 + math.cos(math.pi * it / max(epochs * nb - 1, 1))))
            it += 1
            m1, m2 = 0.9 * m1 + 0.1 * grad, 0.999 * m2 + 0.001 * grad * grad
            theta = theta - rate * math.sqrt(1.0 - 0.999 ** it) / (1.0 - 0.9 ** it) * m1 / (torch.sqrt(m2) + 1e-8)
        losses.append(total / (n * 27))
    return theta, torch.stack(losses)


def _start64(case, seed):
    """The box's starting deviations as its storage holds them, in FP64, and its slab length."""
    n = case["nx"] * case["ny"] * case["nz"]
    p = flbm.make_params(case["nx"], case["ny"], case["nz"], case["tau"], case["kT"], precision=case["precision"],
                         scheme=case["scheme"])
    dtype = TORCH_TYPE[case["precision"]]
    ns = int(flbm.flbm_state_bytes(ctypes.byref(p))) // (Q * torch.empty(0, dtype=dtype).element_size())
    g = torch.empty((Q, n), dtype=dtype, device="cuda")
    _thermal_into(g, n, case["kT"], seed)
    return g.double(), n, ns


def _exact_ensemble(case, seed):
    sizes, taus = _replicas(case, seed)
    c, w = _weights()
    probes, stats, f = dict(_probes(sizes)), [], []
    es = {"fp32": torch.float32, "fp16": torch.float16}[case["precision"]]
    for size in sorted(set(sizes)):
        rs = [r for r, n in enumerate(sizes) if n == size]
        g = torch.empty((Q, len(rs), size ** 3), dtype=torch.float64, device="cuda")
        node = torch.arange(size ** 3, device="cuda")
        for k, r in enumerate(rs):
            xi = _normals(node, 0, range(6, 13), 0, seed + r)
            for i in range(Q):
                g[i, k] = (math.sqrt(3.0 * case["kT"] * w[i]) * xi[i]).to(es).double()
        lat = _Lattice64(g.view(Q, len(rs), size, size, size), [float(taus[r]) for r in rs], rs, case["scheme"],
                         case["kT"], seed)
        for _ in range(case["steps"]):
            lat.step()
        stats.append(lat.stats())
        weights = torch.tensor(w, dtype=torch.float64, device="cuda")
        f.append((lat.g[:, 0].reshape(Q, -1)[:, torch.from_numpy(probes[rs[0]]).cuda()] + weights[:, None]).t())
        del lat, g
    return dict({k: torch.cat([s[k] for s in stats]) for k in stats[0]}, f=f)


def exact(case, seed):
    if case["kind"] == "ensemble":
        # the time of one is that of its nodes and of its count of boxes
        return _exact_ensemble(case, seed)
    if case["kind"] == "train":
        g, n, _ = _start64(dict(case, scheme="reg", precision="fp32"), seed)
        lat = _Lattice64(g.view(Q, 1, case["nz"], case["ny"], case["nx"]), [case["tau"]], [0], "reg", case["kT"], seed)
        m = lat.e @ g
        rho, u = 1.0 + m[0], m[1:4] / (1.0 + m[0])
        for k in range(Q):
            m[k] = 0.0
            if k >= 10:
                m[k] = rho
                for ax in range(3):
                    for _ in range(_DEGREES[k][ax]):
                        m[k] *= u[ax]
        t = ((lat.back @ m) / (lat.w[:, None] * case["kT"] ** 1.5)).t()
        x = _features64(g, lat.w, case["kT"], 1.0 / case["tau"]).t()
        theta = torch.from_numpy(_network(seed)).double().cuda()
        theta, losses = _train64(theta, x.contiguous(), t.contiguous(), case["epochs"], case["batch"], 1e-2, seed)
        return {"x": x, "t": t, "theta": theta, "losses": losses}
    g, n, ns = _start64(case, seed)
    net = torch.from_numpy(_network(seed)).double().cuda() if case["scheme"] == "learned" else None
    scheme = "gmf" if case["scheme"] == "learned" else case["scheme"]
    lat = _Lattice64(g.view(Q, 1, case["nz"], case["ny"], case["nx"]), [case["tau"]], [0], scheme, case["kT"], seed,
                     net)
    del g
    out = {}
    for _ in range(case["steps"]):
        lat.step()
    if case["steps"]:
        out["g"] = torch.zeros((Q, ns), dtype=torch.float64, device="cuda")
        out["g"][:, :n] = lat.g.view(Q, n)
        out["stats"] = {k: v[0] for k, v in lat.stats().items()}
    now = lat.g[:, 0]
    if case["spectra"]:
        c = torch.tensor(lat.c, dtype=torch.float64, device="cuda")
        fields = [torch.ones(Q, dtype=torch.float64, device="cuda"), c.sum(1), (c * c).sum(1),
                  c[:, 0] * c[:, 1] + c[:, 0] * c[:, 2] + c[:, 1] * c[:, 2]]
        theory = [3.0, 3.0, 5.0, 1.0]
        got = [_spectra64(torch.einsum("i,izyx->zyx", fields[o], now), _nshell(case)) for o in range(case["spectra"])]
        out["er"] = torch.stack([s / (theory[o] * case["kT"]) for o, (s, _) in enumerate(got)])
        out["count"] = torch.stack([k for _, k in got])
    if case["moments"]:
        out["rho"], out["j"], out["pi"] = _moments64(now, lat.c)
    return out
