"""Cases for timing the Swendsen-Wang engine through its public calls.

Four kinds of work, each through the calls a program makes:
  sweep   one lattice: n measured sweeps (sw_sweep, sw_measure) or n update-only
          ones (sw_discard), and the state read back to a device buffer;
  batch   a ragged batch of 2D Ising / Potts lattices (sw_batch_sweep), every
          member's moments and state read back;
  stream  a state streamed in and out of the device per sweep with the
          asynchronous host I/O calls;
  label   canonical cluster labels of a bond mask on the device
          (sw_label_from_bonds_noalloc).
Every lattice is near its critical point, the regime the engine is run in, and
starts from sweeps that have built the clusters of that regime.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1403_7560_gb300 import sw

ISING, POTTS, XY, CLOCK = sw.SW_ISING, sw.SW_POTTS, sw.SW_XY, sw.SW_CLOCK
WARM = 30  # sweeps from the random start before the first pass
TORCH_SPIN = {ISING: torch.int8, POTTS: torch.uint8, XY: torch.float32, CLOCK: torch.int16}
SPIN_BYTES = {ISING: 1, POTTS: 1, XY: 4, CLOCK: 2}
# 3D Potts couplings 1/T_c (H = -sum delta): q = 2 is the Ising value, the others approximate
POTTS_3D_K = {2: 2 * 0.2216546, 3: 0.5505, 4: 0.6286, 8: 0.80}
SUMS = ("n_sweeps", "sum_M2", "sum_M4", "sum_E", "sum_E2", "sum_nclusters")


def critical(model, dim, q):
    if model == ISING:
        return 2.0 / math.log(1.0 + math.sqrt(2.0)) if dim == 2 else 1.0 / 0.2216546
    if model == POTTS:
        return 1.0 / math.log(1.0 + math.sqrt(q)) if dim == 2 else 1.0 / POTTS_3D_K[q]
    return 0.8929 if dim == 2 else 1.0 / 0.4541652


def _sweep(name, model, dim, L, q, sweeps, measured=True, tr=1.0):
    c = {"kind": "sweep", "model": model, "dim": dim, "L": L, "q": q, "tr": tr, "sweeps": sweeps,
         "measured": measured}
    return {"name": name, **c} if name else c


def listed():
    return [
        # a small lattice run for many sweeps: equilibration tests, teaching, finite-size scaling's small end
        _sweep("ising2d_L64", ISING, 2, 64, 2, 50),
        # a small XY lattice: launches and latency
        _sweep("xy3d_L16", XY, 3, 16, 2, 20),
        # an odd mid-size Potts lattice, rows not a multiple of a word
        _sweep("potts2d_q3_L515", POTTS, 2, 515, 3, 20),
        # a ragged mid-size 3D lattice of a finite-size-scaling series
        _sweep("ising3d_L100", ISING, 3, 100, 2, 20),
        # the large 2D lattice, thermalisation (update only)
        _sweep("ising2d_L4096_update", ISING, 2, 4096, 2, 6, measured=False),
        # the headline lattice, measured
        _sweep("ising3d_L256", ISING, 3, 256, 2, 6),
        # continuous XY at production size
        _sweep("xy3d_L256", XY, 3, 256, 2, 4),
        # the discretised XY model (q = 512) at a middle size of the paper's table
        _sweep("clock3d_q512_L128", CLOCK, 3, 128, 512, 10),
        # a ragged batch of independent 2D simulations
        {"name": "batch2d_ragged", "kind": "batch", "members": 48, "lo": 32, "hi": 1024, "step": 16, "pick": 1003,
         "sweeps": 30},
        # many small simulations at once
        {"name": "batch2d_small", "kind": "batch", "members": 128, "lo": 16, "hi": 90, "step": 1, "pick": 1005,
         "sweeps": 100},
        # states streamed in and out of the device, a sweep and a record each
        {"name": "stream3d_L256", "kind": "stream", "model": ISING, "dim": 3, "L": 256, "q": 2, "tr": 1.0, "steps": 4},
        # cluster labels of a device bond mask near the percolation threshold
        {"name": "label3d_L128", "kind": "label", "dim": 3, "L": 128, "density": 0.25},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choices(("sweep", "batch", "stream", "label"), (14, 3, 2, 2))[0]
    if kind == "batch":
        step = rng.choice((1, 16))
        hi = _log_int(rng, 64, 768)
        members = _log_int(rng, 8, 96)
        return {"kind": kind, "members": members, "lo": 16, "hi": hi, "step": step, "pick": rng.randrange(1 << 20),
                "sweeps": max(4, min(100, int(2e8 / (members * hi * hi))))}
    dim = rng.choice((2, 3))
    if kind == "label":
        return {"kind": kind, "dim": dim, "L": _log_int(rng, 32, 1448) if dim == 2 else _log_int(rng, 10, 128),
                "density": round(rng.uniform(0.4, 0.6) if dim == 2 else rng.uniform(0.2, 0.35), 4)}
    tr = round(rng.uniform(0.95, 1.05), 4)
    model = rng.choice((ISING, ISING, POTTS, POTTS, XY, CLOCK))
    q = 2
    if model == POTTS:
        q = rng.choice((2, 3, 4, 8))
    elif model == CLOCK:
        q = rng.choice((6, 37, 512))
    if kind == "stream":
        L = _log_int(rng, 64, 2048) if dim == 2 else _log_int(rng, 16, 160)
        return {"kind": kind, "model": model, "dim": dim, "L": L, "q": q, "tr": tr, "steps": rng.randint(2, 6)}
    L = _log_int(rng, 16, 4096) if dim == 2 else _log_int(rng, 8, 256)
    top = 6e7 if model in (XY, CLOCK) else 9e7
    n = max(1, min(_log_int(rng, 4, 100), int(top / L ** dim)))
    return _sweep(None, model, dim, L, q, n, measured=rng.random() < 0.75, tr=tr)


def _members(case, seed):
    """(model, L, q, T, seed) of a batch's lattices: model uniform over Ising and
    Potts q = 3, 4 and L uniform over the range, both by the case; T uniform in
    [0.8, 1.2] T_c and the random-number key by the seed."""
    pick, rng = np.random.default_rng(case["pick"]), np.random.default_rng([int(seed), 17])
    out = []
    n = (case["hi"] - case["lo"]) // case["step"]
    for _ in range(case["members"]):
        model, q = ((ISING, 2), (POTTS, 3), (POTTS, 4))[int(pick.integers(0, 3))]
        L = case["lo"] + case["step"] * int(pick.integers(0, n + 1))
        T = critical(model, 2, q) * float(rng.uniform(0.8, 1.2))
        out.append((model, L, q, T, int(rng.integers(1, 2 ** 62))))
    return out


class _State:
    """What a program keeps: the handles (freed with it) and its buffers."""

    def __init__(self):
        self.handles, self.batch = [], None

    def __del__(self):
        torch.cuda.synchronize()
        if self.batch is not None:
            sw.sw_batch_destroy(self.batch)
        for h in self.handles:
            sw.sw_destroy(h)


def _random_spins(model, n, q, rng):
    if model == ISING:
        return (rng.integers(0, 2, n, dtype=np.int8) * 2 - 1).astype(np.int8)
    if model == XY:
        return (rng.random(n, dtype=np.float32) * np.float32(6.2831)).astype(np.float32)
    return rng.integers(0, q, n).astype(np.uint8 if model == POTTS else np.uint16)


def _key(seed):
    return 0x9E3779B97F4A7C15 * (int(seed) + 1) & (2 ** 62 - 1)


def _mask(case, seed):
    """Random bond planes, each bond present with the case's density."""
    dim, L = case["dim"], case["L"]
    rng = np.random.default_rng([int(seed), 23])
    R, W = L ** (dim - 1), (L + 31) // 32
    bits = np.zeros((dim * R, W * 32), dtype=bool)
    bits[:, :L] = rng.random((dim * R, L), dtype=np.float32) < case["density"]
    return np.packbits(bits, axis=1, bitorder="little").view(np.uint32).reshape(-1)


def prepare(case, seed):
    s = _State()
    s.case = case
    kind = case["kind"]
    if kind == "label":
        s.mask = torch.from_numpy(_mask(case, seed).view(np.int32)).cuda()
        s.labels = torch.empty(case["L"] ** case["dim"], dtype=torch.int32, device="cuda")
        return s
    if kind == "batch":
        s.batch = sw.sw_batch_create(2)
        for model, L, q, T, key in _members(case, seed):
            h = sw.sw_create(model, 2, L, q, T, key)
            s.handles.append(h)
            sw.sw_batch_add(s.batch, h)
        sw.sw_batch_sweep(s.batch, WARM)
        for h in s.handles:
            sw.sw_measure(h)
        s.spins = torch.empty(sum(h.N for h in s.handles), dtype=torch.uint8, device="cuda")
        return s
    model, dim, L, q = case["model"], case["dim"], case["L"], case["q"]
    h = sw.sw_create(model, dim, L, q, case["tr"] * critical(model, dim, q), _key(seed))
    s.handles.append(h)
    if kind == "stream":
        # the states that arrive: configurations of the chain itself, in page-locked memory
        s.inputs, s.outputs = [], []
        for _ in range(case["steps"]):
            sw.sw_discard(h, 10)
            t = torch.empty(sw.sw_spin_bytes(h), dtype=torch.uint8, pin_memory=True)
            a = t.numpy().view(sw.spin_dtype(model))
            sw.sw_get_spins(h, a)
            s.inputs.append(a)
            s.outputs.append(torch.empty(sw.sw_spin_bytes(h), dtype=torch.uint8, pin_memory=True).numpy()
                             .view(sw.spin_dtype(model)))
        s.records = sw.record_buffer(case["steps"])
        sw.sw_set_sweep_counter(h, 0)
        return s
    sw.sw_discard(h, WARM)
    sw.sw_sync(h)
    s.spins = torch.empty(h.N, dtype=TORCH_SPIN[model], device="cuda")
    return s


def run(s):
    case = s.case
    kind = case["kind"]
    if kind == "label":
        sw.sw_label_from_bonds_noalloc(case["dim"], case["L"], s.mask.data_ptr(), s.labels.data_ptr(),
                                       torch.cuda.current_stream().cuda_stream)
        return s.labels
    if kind == "batch":
        sw.sw_batch_sweep(s.batch, case["sweeps"])
        at = s.spins.data_ptr()
        for h in s.handles:
            sw.sw_get_spins_device(h, at, h.N)
            at += h.N
        m = [sw.sw_measure(h) for h in s.handles]
        return {"spins": s.spins, "moments": np.array([[x[k] for k in SUMS] for x in m])}
    h = s.handles[0]
    if kind == "stream":
        k = sw.sw_sweep_counter(h)
        for j, (a, b) in enumerate(zip(s.inputs, s.outputs)):
            sw.sw_set_spins_async(h, a)
            sw.sw_sweep(h, 1)
            sw.sw_get_spins_async(h, b)
            sw.sw_get_record_async(h, k + j + 1, s.records[j])
        sw.sw_wait_io(h)
        return {"spins": s.outputs, "M2": [r.M2 for r in s.records], "E": [r.Ed for r in s.records],
                "nclusters": [int(r.nclusters) for r in s.records]}
    if not case["measured"]:
        sw.sw_discard(h, case["sweeps"])
        sw.sw_get_spins_device(h, s.spins.data_ptr(), sw.sw_spin_bytes(h))
        return {"spins": s.spins}
    sw.sw_sweep(h, case["sweeps"])
    sw.sw_get_spins_device(h, s.spins.data_ptr(), sw.sw_spin_bytes(h))
    return {"spins": s.spins, "moments": sw.sw_measure(h)}


def work(case):
    """The state read and written once per sweep (labels: the mask read, the
    labels written); the arithmetic is integer but for XY (about 40 floating
    operations a site and sweep: projection, bond probabilities, moments)."""
    if case["kind"] == "label":
        N = case["L"] ** case["dim"]
        return {"bytes": N * (case["dim"] / 8 + 4), "flops": 0}
    if case["kind"] == "batch":
        return {"bytes": 2 * sum(m[1] ** 2 for m in _members(case, 0)) * case["sweeps"], "flops": 0}
    n = case["steps"] if case["kind"] == "stream" else case["sweeps"]
    N = case["L"] ** case["dim"]
    return {"bytes": 2 * SPIN_BYTES[case["model"]] * N * n, "flops": 40 * N * n if case["model"] == XY else 0}


# ---------------------------------------------------------------- in 64 bits
# The definitions of the sweep (random numbers, bonds, labels, flip, moments)
# in plain torch, integers in int64 and reals in float64.
_M32 = 0xFFFFFFFF


def _philox(c0, c1, c2, c3, key):
    """Philox4x32-10; counter words as int64 tensors or numbers."""
    k0, k1 = key & _M32, key >> 32
    c0 = c0.clone()
    c1, c2, c3 = (x if torch.is_tensor(x) else torch.full_like(c0, x) for x in (c1, c2, c3))
    for _ in range(10):
        p0, p1 = c0 * 0xD2511F53, c2 * 0xCD9E8D57
        c0 = ((p1 >> 32) & _M32) ^ c1 ^ k0
        c1 = p1 & _M32
        c2 = ((p0 >> 32) & _M32) ^ c3 ^ k1
        c3 = p0 & _M32
        k0, k1 = (k0 + 0x9E3779B9) & _M32, (k1 + 0xBB67AE85) & _M32
    return c0, c1, c2, c3


def _roots(edges, N, dev):
    par = torch.arange(N, device=dev)
    while True:
        live = []
        for i, j in edges:
            a, b = par[i], par[j]
            keep = a != b
            if bool(keep.any()):
                live.append((a[keep], b[keep]))
        if not live:
            return par
        edges = live
        for a, b in edges:
            par.scatter_reduce_(0, torch.maximum(a, b), torch.minimum(a, b), "amin")
        while True:
            up = par[par]
            if torch.equal(up, par):
                break
            par = up


class _Exact:
    def __init__(self, model, dim, L, q, T, key, dev):
        self.model, self.dim, self.L, self.q, self.T, self.key, self.dev = model, dim, L, q, T, key, dev
        self.N, self.R, self.W = L ** dim, L ** (dim - 1), (L + 31) // 32
        self.i = torch.arange(self.N, device=dev)
        x, row = self.i % L, self.i // L
        self.g, self.bit = row * self.W + x // 32, x % 32
        at = self.i.view((L,) * dim)
        self.nb = [torch.roll(at, -1, dims=dim - 1 - d).reshape(-1) for d in range(dim)]
        w = _philox(self.i, 0, 0, 0, key)[0]
        if model == ISING:
            self.s = 1 - 2 * (w >> 31)
        elif model == XY:
            self.s = (w >> 8).double() * (float(np.float32(2 * math.pi)) / 2 ** 24)
        else:
            self.s = (w * q) >> 32
        if model == CLOCK:
            xk = [math.sin(math.pi * k / q) for k in range(2 * q)]
            self.x = torch.tensor(xk, dtype=torch.float64, device=dev)
            ang = [2 * math.pi * p / q for p in range(q)]
            self.c = torch.tensor([math.cos(a) for a in ang], dtype=torch.float64, device=dev)
            self.sn = torch.tensor([math.sin(a) for a in ang], dtype=torch.float64, device=dev)
        if model in (ISING, POTTS):
            self.t = min(int(math.floor(-math.expm1(-(2.0 if model == ISING else 1.0) / T) * 2 ** 32)), _M32)

    def _uniform(self, sweep, d):
        """The bit-sliced 32-bit uniforms of bond direction d."""
        words = torch.arange(self.R * self.W, device=self.dev)
        u = torch.zeros(self.N, dtype=torch.int64, device=self.dev)
        for c in range(8):
            for k, w in enumerate(_philox(words, sweep, 1, 8 * d + c, self.key)):
                u |= ((w[self.g] >> self.bit) & 1) << (31 - 4 * c - k)
        return u

    def sweep(self, sweep):
        q, s = self.q, self.s
        zero = torch.zeros(1, dtype=torch.int64, device=self.dev)
        edges = []
        if self.model in (ISING, POTTS):
            for d, j in enumerate(self.nb):
                on = (s == s[j]) & (self._uniform(sweep, d) < self.t)
                edges.append((self.i[on], j[on]))
        else:
            axis = int(_philox(zero, sweep, 3, 0, self.key)[0][0])
            w = _philox(self.i, sweep, 1, 0, self.key)
            if self.model == XY:
                phi = (axis >> 8) * float(np.float32(2 * math.pi)) / 2 ** 24
                x = torch.cos(s - phi)
            else:
                mirror = (axis * 2 * q) >> 32
                x = self.x[(2 * s - mirror) % (2 * q)]
            for d, j in enumerate(self.nb):
                a = x * x[j]
                p = -torch.expm1(-(2.0 / self.T) * a)
                u = (w[d] >> 8).double() / 2 ** 24 if self.model == XY else w[d].double()
                if self.model == CLOCK:
                    p = torch.floor(p * 2.0 ** 32)
                on = (a > 0) & (u < p)
                edges.append((self.i[on], j[on]))
        root = _roots(edges, self.N, self.dev)
        self.clusters = int((root == self.i).sum())
        if self.model == POTTS and q > 2:
            w = torch.stack(_philox(root >> 2, sweep, 2, 0, self.key))
            self.s = (w.gather(0, (root & 3)[None])[0] * q) >> 32
            return
        bit = (_philox(self.g, sweep, 2, 1, self.key)[0][root] >> self.bit[root]) & 1
        if self.model == ISING:
            self.s = 1 - 2 * bit
        elif self.model == POTTS:
            self.s = bit
        elif self.model == CLOCK:
            self.s = torch.where(bit == 1, (mirror - s) % q, s)
        else:
            self.s = torch.where(bit == 1, (2 * phi + math.pi - s) % (2 * math.pi), s)

    def moments(self):
        """(M2, E) of the state."""
        s, N = self.s, self.N
        if self.model == ISING:
            return float(int(s.sum()) ** 2), float(-sum(int((s * s[j]).sum()) for j in self.nb))
        if self.model == POTTS:
            n = torch.bincount(s, minlength=self.q).tolist()
            return ((self.q * sum(k * k for k in n) - N * N) / (self.q - 1),
                    float(sum(int((s != s[j]).sum()) for j in self.nb)))
        if self.model == CLOCK:
            m2 = float(self.c[s].sum()) ** 2 + float(self.sn[s].sum()) ** 2
            return m2, -sum(float(self.c[(s - s[j]) % self.q].sum()) for j in self.nb)
        m2 = float(torch.cos(s).sum()) ** 2 + float(torch.sin(s).sum()) ** 2
        return m2, -sum(float(torch.cos(s - s[j]).sum()) for j in self.nb)

    def run(self, first, n, measured=True):
        a = [0.0] * 6
        for k in range(first, first + n):
            self.sweep(k)
            if measured:
                m2, e = self.moments()
                for j, v in enumerate((1.0, m2, m2 * m2, e, e * e, float(self.clusters))):
                    a[j] += v
        return dict(zip(SUMS, a))


def exact(case, seed):
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    kind = case["kind"]
    if kind == "label":
        dim, L = case["dim"], case["L"]
        bits = np.unpackbits(_mask(case, seed).view(np.uint8), bitorder="little")
        on = torch.from_numpy(bits.reshape(dim, L ** (dim - 1), -1)[:, :, :L].reshape(dim, -1).astype(bool)).to(dev)
        i = torch.arange(L ** dim, device=dev)
        at = i.view((L,) * dim)
        nb = [torch.roll(at, -1, dims=dim - 1 - d).reshape(-1) for d in range(dim)]
        return _roots([(i[on[d]], nb[d][on[d]]) for d in range(dim)], L ** dim, dev)
    if kind == "batch":
        if case["members"] * (WARM + case["sweeps"]) > 1200:
            return None  # thousands of small lattice sweeps: minutes here
        out, spins = [], []
        for model, L, q, T, key in _members(case, seed):
            e = _Exact(model, 2, L, q, T, key, dev)
            e.run(1, WARM, measured=False)
            m = e.run(WARM + 1, case["sweeps"])
            out.append([m[k] for k in SUMS])
            spins.append(e.s)
        return {"spins": torch.cat(spins), "moments": np.array(out)}
    model, dim, L, q = case["model"], case["dim"], case["L"], case["q"]
    T = case["tr"] * critical(model, dim, q)
    if model == XY and L ** dim > 20000:
        return None  # a bond's float decision differs somewhere, and the trajectories part
    e = _Exact(model, dim, L, q, T, _key(seed), dev)
    if kind == "stream":
        states, out = [], {"spins": [], "M2": [], "E": [], "nclusters": []}
        for j in range(case["steps"]):
            e.run(10 * j + 1, 10, measured=False)
            states.append(e.s)
        for j, x in enumerate(states):
            e.s = x
            e.sweep(j + 1)
            m2, en = e.moments()
            for k, v in (("spins", e.s), ("M2", m2), ("E", en), ("nclusters", e.clusters)):
                out[k].append(v)
        return out
    e.run(1, WARM, measured=False)
    a = e.run(WARM + 1, case["sweeps"], case["measured"])
    if not case["measured"]:
        return {"spins": e.s}
    n, N = a["n_sweeps"], e.N
    m2, m4, e1, e2 = a["sum_M2"] / n, a["sum_M4"] / n, a["sum_E"] / n, a["sum_E2"] / n
    return {"spins": e.s, "moments": {**a, "U": m4 / (m2 * m2), "e_per_spin": e1 / N,
                                      "c_per_spin": (e2 - e1 * e1) / (N * T * T),
                                      "mean_cluster_size": N * n / a["sum_nclusters"]}}
