"""What this library is asked to do, as cases that can be timed and compared.

A case is one call (or one training step) through the public entry points on a named lattice
and filling: products y = H x, Lanczos solves (to convergence, or a fixed number of steps),
mixed-precision and batched solves, ground-state vectors with their double occupancy, and the
learned start vector's training and inference. Lattices and sizes are those of the
repository's benchmark and tests; draw() takes other sizes, fillings and types of the same
ranges.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1511_00863_gb300 as ed

DEV = "cuda"


# ------------------------------------------------------------------ cases
def listed() -> list[dict]:
    return [
        # the smallest call: one product on a 12-site ring (48,400 states), latency only
        dict(name="hv_ring12_f64", kind="hv", lattice="ring", L=12, up=3, dn=3, U=4.0, dtype="f64"),
        # an odd row length (3432 = C(14, 7)) in FP32, the product of a user's own iteration
        dict(name="hv_ring14_f32", kind="hv", lattice="ring", L=14, up=7, dn=7, U=4.0, dtype="f32"),
        # the 4x4 lattice of the benchmark, FP64 product
        dict(name="hv_torus16_f64", kind="hv", lattice="torus", L=16, Lx=4, up=5, dn=5, U=4.0, dtype="f64"),
        # a small solve to convergence: steps of a few microseconds, one check per step
        dict(name="solve_ring12_f64", kind="solve", lattice="ring", L=12, up=3, dn=3, U=4.0, dtype="f64",
             steps=200, tol=1e-12),
        # the benchmark's workload, default precision, to convergence
        dict(name="solve_torus16_f64", kind="solve", lattice="torus", L=16, Lx=4, up=5, dn=5, U=4.0,
             dtype="f64", steps=200, tol=1e-12),
        # the largest: the half-filled 16-site ring (166 M states), FP32 steps
        dict(name="solve_ring16_f32", kind="solve", lattice="ring", L=16, up=8, dn=8, U=4.0, dtype="f32",
             steps=20, tol=0.0),
        # complex hopping amplitudes, FP64: the checkerboard-type lattice, ten hops per site
        dict(name="solve_checker16_c64", kind="solve", lattice="checker", L=16, Lx=4, up=5, dn=5, U=4.0,
             dtype="c64", steps=6, tol=0.0),
        # E0 to FP64 accuracy with most steps in FP32
        dict(name="mixed_ring14", kind="mixed", lattice="ring", L=14, up=7, dn=7, U=4.0, steps=200, tol=1e-9),
        # a parameter scan: many small instances at once, to FP64 accuracy
        dict(name="batched_256", kind="batched", form="mixed", count=256, pick=4),
        # the ground-state vector and its double occupancy (the training data of the network)
        dict(name="ground_ring14", kind="ground", lattice="ring", L=14, up=7, dn=7, U=4.0, steps=200, tol=1e-12),
        # one training step of the start-vector network at the benchmark's batch
        dict(name="mlp_train_ring14", kind="mlp_train", lattice="ring", L=14, up=7, dn=7, U=4.0, batch=16384),
        # its prediction over the whole basis
        dict(name="mlp_infer_ring14", kind="mlp_infer", lattice="ring", L=14, up=7, dn=7, U=4.0, dtype="f32"),
    ]


def _draw_filling(rng, L, low, high):
    """A filling whose dimension lies in [low, high], spread over the logarithm."""
    fits = [(u, d) for u in range(1, L) for d in range(1, L)
            if low <= math.comb(L, u) * math.comb(L, d) <= high and 2 <= math.comb(L, d) <= 13000]
    if not fits:
        return None
    want = math.log(low) + rng.random() * (math.log(high) - math.log(low))
    fits.sort(key=lambda f: abs(math.log(math.comb(L, f[0]) * math.comb(L, f[1])) - want))
    return rng.choice(fits[:6])


def _draw_system(rng, low, high, kinds=("ring", "torus", "checker")):
    while True:
        lattice = rng.choice(kinds)
        if lattice == "ring":
            c = dict(lattice="ring", L=rng.randint(8, 16))
        elif lattice == "torus":
            Lx, Ly = rng.choice([(2, 4), (3, 3), (3, 4), (2, 7), (3, 5), (4, 4)])
            c = dict(lattice="torus", L=Lx * Ly, Lx=Lx)
        else:
            c = dict(lattice="checker", L=16, Lx=4)
        f = _draw_filling(rng, c["L"], low, high)
        if f:
            return dict(c, up=f[0], dn=f[1], U=round(8.0 * rng.random(), 3))


def draw(rng) -> dict:
    kind = rng.choice(["hv", "hv", "hv", "solve", "solve", "solve", "solve", "mixed", "batched", "ground",
                       "mlp_train", "mlp_infer"])
    if kind == "hv":
        dtype = rng.choice(["f64", "f32", "f64", "f32", "c64", "c32"])
        if dtype[0] == "c":
            return dict(kind=kind, dtype=dtype, **_draw_system(rng, 20_000, 20_000_000))
        return dict(kind=kind, dtype=dtype, **_draw_system(rng, 3_000, 60_000_000, ("ring", "torus")))
    if kind == "solve":
        dtype = rng.choice(["f64", "f64", "f64", "f32", "f32", "f64n", "c64", "c32"])
        if dtype == "f64":
            if rng.random() < 0.15:  # one species only (the paper's first workload)
                L = rng.randint(20, 24)
                return dict(kind=kind, dtype=dtype, lattice="ring", L=L, up=L // 2, dn=0, U=4.0,
                            steps=rng.randint(20, 60), tol=0.0)
            return dict(kind=kind, dtype=dtype, steps=300, tol=1e-12,
                        **_draw_system(rng, 20_000, 40_000_000, ("ring", "torus")))
        if dtype == "f32":
            if rng.random() < 0.15:  # rows too long for one block's shared memory
                return dict(kind=kind, dtype=dtype, lattice="ring", L=18, up=rng.randint(1, 2), dn=9, U=4.0,
                            steps=rng.randint(8, 16), tol=0.0)
            return dict(kind=kind, dtype=dtype, steps=rng.randint(10, 20), tol=0.0,
                        **_draw_system(rng, 20_000, 160_000_000, ("ring", "torus")))
        kinds = ("ring", "torus") if dtype == "f64n" else ("ring", "torus", "checker")
        return dict(kind=kind, dtype=dtype, steps=rng.randint(4, 10), tol=0.0,
                    **_draw_system(rng, 20_000, 20_000_000, kinds))
    if kind == "mixed":
        return dict(kind=kind, steps=200, tol=1e-9, **_draw_system(rng, 200_000, 20_000_000, ("ring", "torus")))
    if kind == "batched":
        return dict(kind=kind, form=rng.choice(["mixed", "f32", "f64n"]),
                    count=int(round(8 * 2 ** (5 * rng.random()))), pick=rng.randint(1, 10**6))
    if kind == "ground":
        return dict(kind=kind, steps=300, tol=1e-12, **_draw_system(rng, 20_000, 12_000_000, ("ring", "torus")))
    if kind == "mlp_train":
        return dict(kind=kind, batch=int(round(1024 * 2 ** (4 * rng.random()))),
                    **_draw_system(rng, 20_000, 12_000_000, ("ring", "torus")))
    return dict(kind=kind, dtype=rng.choice(["f32", "f64"]),
                **_draw_system(rng, 20_000, 20_000_000, ("ring", "torus")))


# ------------------------------------------------------------------ lattices
def _bonds(c):
    """(bonds, complex amplitudes or None): periodic ring, Lx x Ly square lattice, and the
    checkerboard-type lattice with complex nearest-neighbour amplitudes."""
    L = c["L"]
    if c["lattice"] == "ring":
        return [(i, (i + 1) % L) for i in range(L)], None
    Lx = c["Lx"]
    Ly = L // Lx
    at = lambda x, y: (x % Lx) + Lx * (y % Ly)  # noqa: E731
    out, amp = [], []
    for y in range(Ly):
        for x in range(Lx):
            if c["lattice"] == "torus":
                out += [(at(x, y), at(x + 1, y)), (at(x, y), at(x, y + 1))]
                continue
            s, a = at(x, y), 1.0 if (x + y) % 2 == 0 else -1.0
            out += [(s, at(x + 1, y)), (s, at(x, y + 1)), (s, at(x + 1, y + 1)), (s, at(x + 1, y - 1))]
            amp += [np.exp(0.25j * np.pi * a), np.exp(-0.25j * np.pi * a), 0.3 * a, -0.3 * a]
            if Lx != 4 or x < 2:
                out.append((s, at(x + 2, y)))
                amp.append(-0.2)
            if Ly != 4 or y < 2:
                out.append((s, at(x, y + 2)))
                amp.append(-0.2)
    return out, (np.array(amp, dtype=np.complex128) if amp else None)


def _instances(c, seed):
    """The systems of a batch: rings of 8 to 12 sites and 2x4, 3x4 rectangles at up to half
    filling (from the case), U uniform in [0, 8) (from the seed)."""
    r = np.random.RandomState(c["pick"] % 2**31)
    u = np.random.RandomState(seed % 2**31)
    got = []
    for _ in range(c["count"]):
        k = int(r.randint(7))
        d = dict(lattice="ring", L=8 + k) if k < 5 else dict(lattice="torus", L=8 if k == 5 else 12, Lx=2 if k == 5 else 3)
        d["up"], d["dn"] = int(r.randint(1, d["L"] // 2 + 1)), int(r.randint(1, d["L"] // 2 + 1))
        d["U"] = float(1.0 + 7.0 * u.rand())
        got.append(d)
    return got


class _Basis:
    """A basis handle, released with the state that holds it."""

    def __init__(self, c):
        bonds, amp = _bonds(c)
        self.h = ed.ed_build_basis(c["L"], bonds, c["up"], c["dn"], t_bond=amp)

    def __del__(self):
        ed.ed_basis_destroy(self.h)


class _Net:
    def __init__(self, L):
        self.h = ed.ed_mlp_create(L, 1)
        ptr, n = ed.ed_mlp_params(self.h)
        self.__cuda_array_interface__ = dict(shape=(n,), typestr="<f4", data=(ptr, False), version=3)
        self.params = torch.as_tensor(self, device=DEV)

    def __del__(self):
        torch.cuda.synchronize()
        ed.ed_mlp_destroy(self.h)


# ------------------------------------------------------------------ inputs
_TORCH = {"f64": torch.float64, "f32": torch.float32, "c64": torch.complex128, "c32": torch.complex64}


def _dim(c):
    return math.comb(c["L"], c["up"]) * math.comb(c["L"], c["dn"])


def _generator(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return g


def _x(c, seed):
    return torch.randn(_dim(c), dtype=_TORCH[c["dtype"]], device=DEV, generator=_generator(seed))


def _weights(c, seed):
    """Weights of the network: the spread that training leaves (Glorot-like layers, biases)."""
    nin = 2 * c["L"] + 1
    g = _generator(seed)
    shapes = [(nin, 64), (64,), (64, 64), (64,), (64, 2), (2,)]
    return [torch.randn(s, device=DEV, generator=g) * (0.3 if len(s) == 1 else math.sqrt(2.0 / sum(s)))
            for s in shapes]


def _amplitudes(c, seed):
    """A unit vector shaped like a ground state: random signs, amplitudes over some decades."""
    g = _generator(seed + 1)
    a = torch.randn(_dim(c), dtype=torch.float64, device=DEV, generator=g)
    s = torch.randn(_dim(c), dtype=torch.float64, device=DEV, generator=g)
    v = torch.exp(2.0 * a) * torch.sign(s)
    return v / v.norm()


def prepare(c, seed):
    kind = c["kind"]
    st = dict(case=c, seed=seed)
    if kind == "batched":
        inst = _instances(c, seed)
        st["bases"] = [_Basis(d) for d in inst]
        st["handles"] = [b.h for b in st["bases"]]
        st["ts"], st["Us"] = [1.0] * len(inst), [d["U"] for d in inst]
        f64 = c["form"] == "f64n"
        st["opts"] = ed.make_opts(max_steps=200, tol=1e-12 if f64 else 1e-9, seed=seed, schedule=6,
                                  dtype="f64n" if f64 else "f32")
        return st
    st["basis"] = _Basis(c)
    if kind == "hv":
        st["x"] = _x(c, seed)
        st["y"] = torch.empty_like(st["x"])
    elif kind == "solve":
        st["opts"] = ed.make_opts(max_steps=c["steps"], tol=c["tol"], seed=seed, dtype=c["dtype"])
    elif kind == "mixed":
        st["opts"] = ed.make_opts(max_steps=c["steps"], tol=c["tol"], seed=seed, dtype="f32")
    elif kind == "ground":
        st["opts"] = ed.make_opts(max_steps=c["steps"], tol=c["tol"], seed=seed, dtype="f64")
        st["psi"] = torch.empty(_dim(c), dtype=torch.float64, device=DEV)
    else:
        st["net"] = _Net(c["L"])
        st["net"].params.copy_(torch.cat([w.reshape(-1) for w in _weights(c, seed)]))
        if kind == "mlp_train":
            st["psi"] = _amplitudes(c, seed)
        else:
            st["out"] = torch.empty(_dim(c), dtype=_TORCH[c["dtype"]], device=DEV)
    return st


# ------------------------------------------------------------------ one pass
def run(st):
    c = st["case"]
    kind = c["kind"]
    if kind == "batched":
        if c["form"] == "mixed":
            # the steps at which FP32 rounding lets the first phase stop are left out
            r = ed.ed_lanczos_solve_batched_mixed(st["handles"], st["ts"], st["Us"], st["opts"], refine_steps=64,
                                                  refine_tol=1e-12, raise_not_converged=False)
            return {"E0": r["E0"]}
        r = ed.ed_lanczos_solve_batched(st["handles"], st["ts"], st["Us"], st["opts"], raise_not_converged=False)
        return {"E0": r["E0"].astype(np.float32) if c["form"] == "f32" else r["E0"]}
    h, U = st["basis"].h, c["U"]
    if kind == "hv":
        ed.ed_hv(h, 1.0, U, st["x"], st["y"])
        return st["y"]
    if kind == "solve":
        r = ed.ed_lanczos_solve(h, 1.0, U, st["opts"], raise_not_converged=False)
        if c["dtype"] in ("f32", "c32"):  # scalars of FP32 vectors: FP32 accuracy
            return {k: r[k].astype(np.float32) for k in ("alpha", "beta", "E0_hist")}
        if c["tol"] > 0.0:  # padded to the step limit: the number of steps depends on the start vector
            n = (0, c["steps"] - r["steps"])
            return {"E0": np.float64(r["E0"]), "steps": r["steps"],
                    **{k: np.pad(r[k], n) for k in ("alpha", "beta", "E0_hist")}}
        return {k: r[k] for k in ("alpha", "beta", "E0_hist")}
    if kind == "mixed":
        r = ed.ed_lanczos_solve_mixed(h, 1.0, U, st["opts"], refine_steps=64, refine_tol=1e-12,
                                      raise_not_converged=False)
        return {"E0": np.float64(r["E0"])}
    if kind == "ground":
        r = ed.ed_lanczos_ground_state(h, 1.0, U, st["opts"], st["psi"], raise_not_converged=False)
        D, site = ed.ed_double_occupancy(h, st["psi"])
        return {"E0": np.float64(r["E0"]), "steps": r["steps"], "psi": st["psi"], "D": np.float64(D), "site": site}
    if kind == "mlp_train":
        loss = ed.ed_mlp_train_step(st["net"].h, h, U, st["psi"], c["batch"], 3e-3, 1000 + st["seed"])
        return {"loss": torch.tensor(loss, dtype=torch.float32), "params": st["net"].params}
    ed.ed_mlp_infer(st["net"].h, h, U, st["out"])
    return st["out"]


# ------------------------------------------------------------------ what a pass cannot do without
def _hops(c):
    """Hops out of all states of each species, and their table bytes (target and sign)."""
    n = len(_bonds(c)[0])
    L = c["L"]
    of = lambda k: 2 * n * math.comb(L - 2, k - 1) if 1 <= k < L else 0  # noqa: E731
    return of(c["up"]), of(c["dn"])


def _step(c, width, cx):
    """Bytes (two vectors read, one written, the tables) and operations of a Lanczos step."""
    dim, (hu, hd) = _dim(c), _hops(c)
    terms = hu * math.comb(c["L"], c["dn"]) + hd * math.comb(c["L"], c["up"])
    return 3 * width * dim + 4 * (hu + hd), (8 if cx else 2) * terms + 10 * (2 if cx else 1) * dim


_WIDTH = {"f64": 8, "f32": 4, "f64n": 8, "c64": 16, "c32": 8}


def work(c):
    kind = c["kind"]
    if kind == "batched":
        b = f = 0
        for d in _instances(c, 0):
            s = _step(d, 8 if c["form"] == "f64n" else 4, False)
            n = min(_dim(d), 50)
            b, f = b + s[0] * n, f + s[1] * n
        return {"bytes": b, "flops": f}
    dim = _dim(c)
    if kind == "hv":
        b, f = _step(c, _WIDTH[c["dtype"]], c["dtype"][0] == "c")
        return {"bytes": b - dim * _WIDTH[c["dtype"]], "flops": f}
    if kind in ("solve", "mixed", "ground"):
        d = {"mixed": "f32", "ground": "f64"}.get(kind) or c["dtype"]
        # a run to convergence takes about 60 steps, a ground-state vector takes them twice
        n = c["steps"] if c["tol"] == 0.0 else 120 if kind == "ground" else 60
        b, f = _step(c, _WIDTH[d], d[0] == "c")
        return {"bytes": b * n, "flops": f * n}
    per = 2 * ((2 * c["L"] + 1) * 64 + 64 * 64 + 128)
    if kind == "mlp_train":
        return {"bytes": 8 * c["batch"] + 16 * 64 * (2 * c["L"] + 68), "flops": 3 * per * c["batch"]}
    return {"bytes": dim * (4 if c["dtype"] == "f32" else 8), "flops": per * dim}


# ------------------------------------------------------------------ the same in 64 bits
def _species(c, n):
    """(states, targets, amplitudes) of one species: for every bond and direction the state that
    hops into state r and its matrix element (hops that do not exist point at r with 0)."""
    L = c["L"]
    bonds, amp = _bonds(c)
    every = torch.arange(1 << L, dtype=torch.int64, device=DEV)
    ones = torch.zeros_like(every)
    for i in range(L):
        ones += (every >> i) & 1
    states = every[ones == n]
    del every, ones
    at = torch.arange(states.numel(), device=DEV)
    targets, elements = [], []
    for b, (i, j) in enumerate(bonds):
        a = complex(amp[b]) if amp is not None else 1.0
        lo, hi = min(i, j), max(i, j)
        between = (1 << hi) - (1 << (lo + 1))
        for src, dst, el in ((j, i, a), (i, j, np.conj(a))):  # element of c+_dst c_src
            # row r has dst occupied and src empty; its source has the particle at src
            ok = ((states >> dst) & 1 == 1) & ((states >> src) & 1 == 0)
            sign = torch.zeros_like(states)
            for k in range(lo + 1, hi):
                sign += ((states & between) >> k) & 1
            frm = torch.searchsorted(states, states ^ ((1 << dst) | (1 << src)))
            targets.append(torch.where(ok, frm.clamp(max=states.numel() - 1), at))
            e = torch.where(ok, 1.0 - 2.0 * (sign & 1).double(), torch.zeros((), dtype=torch.float64, device=DEV))
            elements.append(-e * el if amp is not None else -e)
    return states, targets, elements


class _Product:
    def __init__(self, c):
        self.U = c["U"]
        self.up, self.dn = _species(c, c["up"]), _species(c, c["dn"])
        occ = lambda s: torch.stack([((s >> i) & 1).double() for i in range(c["L"])], 1)  # noqa: E731
        nu, nd = occ(self.up[0]), occ(self.dn[0])
        self.shape = (nu.shape[0], nd.shape[0])
        self.D = nu @ nd.T
        self.cx = c["lattice"] == "checker"
        self.dense = []
        for s, t, e in (self.up, self.dn):
            n = s.numel()
            m = None
            if n <= 1000:
                m = torch.zeros(n, n, dtype=torch.complex128 if self.cx else torch.float64, device=DEV)
                for tk, ek in zip(t, e):
                    m[torch.arange(n, device=DEV), tk] += ek
            self.dense.append(m)

    def __call__(self, x):
        X = x.reshape(self.shape)
        Y = (self.U * self.D) * X
        if self.dense[0] is not None:
            Y += self.dense[0].to(X.dtype) @ X
        else:
            for t, e in zip(*self.up[1:]):
                Y += e[:, None] * X[t]
        if self.dense[1] is not None:
            Y += X @ self.dense[1].T.to(X.dtype)
        else:
            for t, e in zip(*self.dn[1:]):
                Y += e * X[:, t]
        return Y.reshape(-1)


def _splitmix(seed, n):
    """SplitMix64 outputs 1 .. n as int64 bit patterns."""
    wrap = lambda v: v - 2**64 if v >= 2**63 else v  # noqa: E731
    lsr = lambda z, k: (z >> k) & ((1 << (64 - k)) - 1)  # noqa: E731
    z = torch.arange(1, n + 1, dtype=torch.int64, device=DEV) * wrap(0x9E3779B97F4A7C15) + wrap(seed % 2**64)
    z = (z ^ lsr(z, 30)) * wrap(0xBF58476D1CE4E5B9)
    z = (z ^ lsr(z, 27)) * wrap(0x94D049BB133111EB)
    return z ^ lsr(z, 31)


def _start(seed, dim, cx):
    z = _splitmix(seed, 2 * dim if cx else dim)
    v = 2.0 * (((z >> 11) & ((1 << 53) - 1)).double() * 2.0**-53) - 1.0
    v /= v.norm()
    return torch.view_as_complex(v.reshape(-1, 2)) if cx else v


def _lowest(a, b):
    T = np.diag(a) + np.diag(b[:len(a) - 1], 1) + np.diag(b[:len(a) - 1], -1)
    return np.linalg.eigvalsh(T)[0]


def _lanczos(H, f, steps, tol=0.0, keep=None):
    """Plain Lanczos in FP64: (a, b, E0 after every step, or the last one with tol > 0)."""
    a, b, hist = [], [], []
    prev, beta = torch.zeros_like(f), 0.0
    for j in range(steps):
        if keep is not None:
            keep.append(f)
        q = H(f) - beta * prev
        al = torch.vdot(f, q).real.item()
        q -= al * f
        if keep is not None:
            for _ in range(2):
                for v in keep:
                    q -= torch.vdot(v, q) * v
        beta = q.norm().item()
        a.append(al)
        b.append(beta)
        if tol == 0.0 or j % 5 == 4:
            hist.append(_lowest(a, b))
            if tol > 0.0 and len(hist) > 1 and abs(hist[-1] - hist[-2]) <= tol * max(1.0, abs(hist[-1])):
                break
        if beta <= 1e-12:
            hist.append(_lowest(a, b))
            break
        prev, f = f, q / beta
    return np.array(a), np.array(b), np.array(hist or [_lowest(a, b)])


def _bf16(t):
    return t.to(torch.float32).to(torch.bfloat16).double()


def _net(ws, c, index):
    """Features, layers and outputs of the network for the states `index`, in 64 bits with the
    operand roundings of the model (bfloat16 weights, U and first-layer outputs)."""
    def states(n):
        s = torch.arange(1 << c["L"], device=DEV)
        ones = sum((s >> i) & 1 for i in range(c["L"]))
        return s[ones == n]
    up, dn = states(c["up"]), states(c["dn"])
    u, d = up[index // dn.numel()], dn[index % dn.numel()]
    X = torch.stack([((s >> i) & 1).double() for s in (u, d) for i in range(c["L"])]
                    + [_bf16(torch.full(index.shape, c["U"] / 8.0, device=DEV))], 1)
    h1 = torch.tanh(X @ ws[0] + ws[1])
    h1b = h1 + (_bf16(h1) - h1).detach()  # the rounding counts as the identity backwards
    h2 = torch.tanh(h1b @ ws[2] + ws[3])
    return h2 @ ws[4] + ws[5]


def exact(c, seed):
    kind = c["kind"]
    if kind == "batched":
        got = []
        for d in _instances(c, seed):
            a, b, hist = _lanczos(_Product(d), _start(seed, _dim(d), False), min(_dim(d), 140), tol=1e-14)
            got.append(hist[-1])
        return {"E0": np.array(got)}
    if kind == "hv":
        H = _Product(c)
        x = _x(c, seed)
        return H(x.to(torch.complex128 if x.is_complex() else torch.float64))
    if kind == "solve":
        a, b, hist = _lanczos(_Product(c), _start(seed, _dim(c), c["dtype"][0] == "c"), c["steps"], c["tol"] / 100)
        if c["tol"] > 0.0:
            return {"E0": np.float64(hist[-1]), "steps": None, "alpha": None, "beta": None, "E0_hist": None}
        return {"alpha": a, "beta": b, "E0_hist": hist}
    if kind == "mixed":
        return {"E0": np.float64(_lanczos(_Product(c), _start(seed, _dim(c), False), 300, 1e-14)[2][-1])}
    if kind == "ground":
        keep = []
        H = _Product(c)
        a, b, hist = _lanczos(H, _start(seed, _dim(c), False), 150, 1e-14, keep)
        T = np.diag(a) + np.diag(b[:-1], 1) + np.diag(b[:-1], -1)
        y = np.linalg.eigh(T)[1][:, 0]
        psi = sum(float(w) * v for w, v in zip(y, keep))
        psi /= psi.norm()
        if psi[psi.abs().argmax()] < 0:
            psi = -psi
        p2 = (psi * psi).reshape(H.shape)
        site = [float((((H.up[0] >> i) & 1).double()[:, None] * p2 * ((H.dn[0] >> i) & 1).double()).sum())
                for i in range(c["L"])]
        return {"E0": np.float64(hist[-1]), "steps": None, "psi": psi, "D": np.float64(sum(site)), "site": np.array(site)}
    ws = _weights(c, seed)
    if kind == "mlp_train":
        n, dim, psi = c["batch"], _dim(c), _amplitudes(c, seed)
        z = _splitmix(1000 + seed, n).cpu().numpy().astype(np.uint64)
        index = torch.tensor([(int(v) * dim) >> 64 for v in z], device=DEV)
        t = psi[index]
        leaf = [_bf16(w).requires_grad_(True) for w in ws]
        out = _net(leaf, c, index)
        w = dim * t * t
        loss = (w * ((out[:, 0] - t.abs().log()) ** 2 + torch.nn.functional.softplus(-t.sign() * out[:, 1]))).sum() / n
        loss.backward()
        g = torch.cat([v.grad.reshape(-1) for v in leaf])
        # one Adam step from zero moments
        m, v = 0.1 * g / (1 - 0.9), 0.001 * g * g / (1 - 0.999)
        params = torch.cat([w.double().reshape(-1) for w in ws]) - 3e-3 * m / (v.sqrt() + 1e-8)
        return {"loss": loss.detach(), "params": params}
    out = torch.empty(_dim(c), dtype=torch.float64, device=DEV)
    leaf = [_bf16(w) for w in ws]
    for at in range(0, out.numel(), 1 << 20):
        index = torch.arange(at, min(out.numel(), at + (1 << 20)), device=DEV)
        o = _net(leaf, c, index)
        out[index] = torch.exp(o[:, 0]) * torch.where(o[:, 1] >= 0, 1.0, -1.0)
    return out
