"""Performance cases of the ladder dual-fermion library.

Each case is work a user of the library has it do, through its public entry
points (the Python binding over include/df.h).  ``listed()`` holds the fixed
ones, ``draw(rng)`` gives further cases of the same ranges.  A case names its
kind:

* ``loop``     a whole short loop: Sigma~ set, ``passes`` passes of df_iterate,
               Sigma~ and the residual read back;
* ``ladders``  the ladder stage alone: df_bubble + df_bse, chi~ and the Eq. sd
               brackets read back (what a vertex or eigenvalue study reads);
* ``chi``      the charge and spin susceptibilities of a given Sigma~;
* ``batch``    one pass over a batch of uneven parameter points;
* ``train``    one training step of the warm-start network, with its gradients;
* ``predict``  a warm start: one network output expanded onto a handle.

``family`` selects the inputs: ``paper`` is the paper's Example I (Hubbard
atom, U around 20, beta around 1; the loop converges), ``tp`` the doped
t-t' square lattice with a perturbed vertex (ill-conditioned ladders),
``crit`` the half-filled cubic lattice near its magnetic instability,
``generic`` complex inputs without any symmetry.
"""
from __future__ import annotations

import ctypes
import math

import numpy as np
import torch

from paper_1507_00895_gb300 import df, inputs, warmstart

F64, MIXED = df.DF_FP64, df.DF_FP32_IR


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------

def listed():
    return [
        # one small point of the paper's Example I sweeps: launches and latency count
        dict(name="sweep_point_8sq_n16", kind="loop", family="paper", dim=2, nk=8, n_w=16, m_max=1,
             precision=F64, symmetry=0, passes=6),
        # the paper's Example I size, refined mixed precision (an order that is no power of two)
        dict(name="paper_16sq_n48_mixed", kind="loop", family="paper", dim=2, nk=16, n_w=48, m_max=1,
             precision=MIXED, symmetry=0, passes=2),
        # the benchmark's workload in plain FP64: the default precision of a handle
        dict(name="bench_32sq_n64_fp64", kind="loop", family="tp", dim=2, nk=32, n_w=64, m_max=7,
             precision=F64, symmetry=0, passes=1),
        # the benchmark's headline: every ladder solved, refined mixed precision
        dict(name="bench_32sq_n64_mixed", kind="loop", family="tp", dim=2, nk=32, n_w=64, m_max=7,
             precision=MIXED, symmetry=0, passes=1),
        # the same workload as a production run takes it, with both exact reductions
        dict(name="bench_32sq_n64_reduced", kind="loop", family="tp", dim=2, nk=32, n_w=64, m_max=7,
             precision=MIXED, symmetry=2, passes=1),
        # a pass of the 3D run towards criticality, both reductions
        dict(name="cubic16_n96_reduced", kind="loop", family="crit", dim=3, nk=16, n_w=96, m_max=10,
             precision=MIXED, symmetry=2, passes=1),
        # one training run's pass of the learned warm start at its stated grid
        dict(name="warm_64sq_n128_reduced", kind="loop", family="paper", dim=2, nk=64, n_w=128, m_max=15,
             precision=MIXED, symmetry=2, passes=1),
        # ladders of an uneven small order with generic complex vertices, 3D, no reductions
        dict(name="ladders_8cubed_n30", kind="ladders", family="generic", dim=3, nk=8, n_w=30, m_max=5,
             precision=MIXED, symmetry=0),
        # the observables at the end of a run
        dict(name="susceptibility_32sq_n64", kind="chi", family="tp", dim=2, nk=32, n_w=64, m_max=7,
             precision=MIXED, symmetry=0),
        # a parameter study: uneven points iterated together
        dict(name="batch_24_points", kind="batch", points=24, max_n_w=64, max_m=7, precision=MIXED, symmetry=2),
        # training the warm-start network at the stated grid's output size
        dict(name="train_512x71808", kind="train", n_in=260, width=512, n_out=71808, batch=256),
        # applying it to a new parameter point
        dict(name="predict_64sq_n128", kind="predict", nk=64, n_w=128, m_max=15, width=512),
    ]


_LATTICES = ((1, 64), (2, 8), (2, 16), (2, 32), (2, 64), (3, 8), (3, 16), (4, 4), (4, 8))


def _orbits(dim, nk):
    return math.comb(nk // 2 + dim, dim)


def _ladders(case):
    """(q, W, channel) systems a pass solves."""
    nb = 2 * case["m_max"] + 1
    if case["symmetry"] == 2:
        return 2 * (case["m_max"] + 1) * _orbits(case["dim"], case["nk"])
    return 2 * nb * case["nk"] ** case["dim"]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("loop",) * 5 + ("ladders",) * 2 + ("chi", "batch", "train", "predict"))
    if kind == "train":
        return dict(kind=kind, n_in=rng.randrange(8, 400), width=rng.choice((64, 128, 200, 256, 512)),
                    n_out=_logint(rng, 100, 71808), batch=_logint(rng, 16, 256))
    if kind == "predict":
        nk, n_w = rng.choice((8, 16, 32, 64)), 2 * _logint(rng, 6, 64)
        return dict(kind=kind, nk=nk, n_w=n_w, m_max=rng.randrange(0, 16), width=rng.choice((128, 256, 512)))
    if kind == "batch":
        return dict(kind=kind, points=rng.randrange(4, 25), max_n_w=8 * rng.randrange(3, 9), max_m=rng.randrange(1, 8),
                    precision=rng.choice((F64, MIXED)), symmetry=2)
    dim, nk = rng.choice(_LATTICES)
    n_w = 2 * _logint(rng, 4, 64)
    if kind == "chi":
        n_w = min(n_w, 64)                       # both precisions refine or factorise up to this order
    m_max = rng.randrange(0, 16)
    precision = rng.choice((F64, MIXED, MIXED))
    symmetry = rng.choice((0, 2)) if kind == "loop" else 0
    if symmetry:
        families = ("paper", "tp") if dim == 2 else ("crit",) if dim == 3 else ("paper",)
    else:
        families = ("paper", "tp", "generic") if dim == 2 else ("crit", "generic") if dim == 3 else ("paper", "generic")
    case = dict(kind=kind, family=rng.choice(families), dim=dim, nk=nk, n_w=n_w, m_max=m_max, precision=precision,
                symmetry=symmetry)
    # no more than the largest listed case (18k ladders of order 128 in mixed precision)
    cap = 0.8e11 if precision == F64 and kind != "chi" else 2.5e11
    while _ladders(case) * 8.0 * n_w ** 3 > cap and case["m_max"] > 0:
        case["m_max"] -= 1
    while _ladders(case) * 8.0 * n_w ** 3 > cap and case["nk"] > 4:
        case["nk"] //= 2
    if kind == "loop":
        case["passes"] = 1
    return case


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _workload(case, seed):
    rng = np.random.default_rng(seed)
    dim, nk, n_w, m_max = case["dim"], case["nk"], case["n_w"], case["m_max"]
    fam = case["family"]
    if fam == "paper":
        u, b = float(rng.uniform(16.0, 24.0)), float(rng.uniform(0.8, 1.2))
        return inputs.half_filled_atom("paper", dim, nk, U=u, beta=b, n_w=n_w, m_max=m_max)
    if fam == "tp":
        return inputs.workload("square32_tp", nk=nk, n_w=n_w, m_max=m_max, seed=seed)
    if fam == "crit":
        b = inputs.CUBIC16_BETA_LAMBDA098 * float(rng.uniform(0.97, 1.0))
        return inputs.half_filled_atom("crit", dim, nk, U=6.0, beta=b, n_w=n_w, m_max=m_max)
    if fam == "generic":
        return inputs.random_nonsymmetric(n_w, m_max, dim, nk, seed, scale=0.5)
    raise KeyError(fam)


def _batch_workloads(case, seed):
    """The uneven recipe's lattices and sizes (fixed by the case) at U and beta drawn from the seed."""
    sizes = inputs.uneven_batch(case["points"], seed=4, max_n_w=case["max_n_w"], max_m=case["max_m"],
                                grids=((2, 8), (2, 16), (2, 32), (4, 4)))
    rng = np.random.default_rng(seed)
    return [inputs.half_filled_atom(w.name, w.dim, w.nk, U=float(rng.uniform(1.0, 8.0)),
                                    beta=float(rng.uniform(2.0, 20.0)), n_w=w.n_w, m_max=w.m_max) for w in sizes]


def _weights(dims, seed):
    """Glorot-uniform weights and small biases, flat [W1 b1 ... W4 b4], on the GPU."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    parts = []
    for a, b in zip(dims[:-1], dims[1:]):
        lim = math.sqrt(6.0 / (a + b))
        parts.append((torch.rand(a * b, generator=gen, device="cuda") * 2 - 1) * lim)
        parts.append(torch.randn(b, generator=gen, device="cuda") * 0.01)
    return torch.cat(parts).contiguous()


def _train_data(case, seed):
    """Standardised features and targets."""
    gen = torch.Generator(device="cuda").manual_seed(seed + 1)
    x = torch.randn(case["batch"], case["n_in"], generator=gen, device="cuda")
    t = torch.randn(case["batch"], case["n_out"], generator=gen, device="cuda")
    return x, t


def _predict_sizes(case):
    _, rep = warmstart.wedge(case["nk"])
    half = case["n_w"] // 2
    return 4 + 4 * half, len(rep) * half * 2


def _predict_data(case, seed):
    n_in, n_out = _predict_sizes(case)
    w = inputs.warmstart_family(1, seed, nk=case["nk"], n_w=case["n_w"], m_max=case["m_max"])[0]
    gen = torch.Generator(device="cuda").manual_seed(seed + 1)
    x = torch.randn(1, n_in, generator=gen, device="cuda")
    mean = torch.randn(n_out, generator=gen, device="cuda") * 0.02
    sd = torch.rand(n_out, generator=gen, device="cuda") * 0.01 + 1e-4
    kmap = torch.from_numpy(warmstart.wedge(case["nk"])[0]).cuda()
    return w, x, mean, sd, kmap


def _mlp(dims, max_batch, seed):
    net = df.MLP(dims[0], dims[4], width=dims[1], max_batch=max_batch)
    p = _weights(dims, seed)
    s = net.lib.df_mlp_params(net.h, ctypes.c_void_p(p.data_ptr()), 1, 1)
    assert s == df.DF_OK
    return net


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("loop", "ladders", "chi"):
        w = _workload(case, seed)
        d = df.DualFermion.from_workload(w, precision=case["precision"], symmetry=case["symmetry"])
        st = dict(case=case, d=d)
        if kind == "loop":
            st["sigma0"] = torch.zeros(d.n_w, d.N, dtype=torch.complex128, device="cuda")
            st["sigma"] = torch.empty_like(st["sigma0"])
        elif kind == "ladders":
            st["chi"] = torch.empty(d.nb, d.n_w, d.N, dtype=torch.complex128, device="cuda")
            st["kernel"] = torch.empty(2, d.nb, d.n_w, d.N, dtype=torch.complex128, device="cuda")
        else:
            st["out"] = torch.empty(2, d.nb, d.N, dtype=torch.complex128, device="cuda")
        return st
    if kind == "batch":
        ws = _batch_workloads(case, seed)
        b = df.DualFermionBatch(ws, precision=case["precision"], symmetry=case["symmetry"])
        return dict(case=case, b=b,
                    out=[torch.empty(w.n_w, w.N, dtype=torch.complex128, device="cuda") for w in ws])
    if kind == "train":
        dims = (case["n_in"], case["width"], case["width"], case["width"], case["n_out"])
        net = _mlp(dims, case["batch"], seed)
        x, t = _train_data(case, seed)
        return dict(case=case, net=net, x=x, t=t, grads=torch.empty(net.nparam, device="cuda"))
    if kind == "predict":
        n_in, n_out = _predict_sizes(case)
        w, x, mean, sd, kmap = _predict_data(case, seed)
        net = _mlp((n_in, case["width"], case["width"], case["width"], n_out), 1, seed)
        d = df.DualFermion.from_workload(w, precision=MIXED, symmetry=2, eig_mode=0)
        return dict(case=case, net=net, d=d, x=x, y=torch.empty(1, n_out, device="cuda"), mean=mean, sd=sd, kmap=kmap,
                    sigma=torch.empty(d.n_w, d.N, dtype=torch.complex128, device="cuda"),
                    g=torch.empty(d.ne, d.N, dtype=torch.complex128, device="cuda"))
    raise KeyError(kind)


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "loop":
        d = state["d"]
        d.set_sigma(state["sigma0"])
        _, r, _ = d.iterate(case["passes"])
        d.get_sigma(state["sigma"])
        return {"sigma": state["sigma"], "residual": r}
    if kind == "ladders":
        d = state["d"]
        d.bubble()
        d.bse(3)
        d.get_chi(state["chi"])
        d.get_kernel(state["kernel"])
        return {"chi": state["chi"], "kernel": state["kernel"]}
    if kind == "chi":
        state["d"].susceptibility(state["out"])
        return {"chi": state["out"]}
    if kind == "batch":
        b = state["b"]
        b.reset()
        _, r, _, _ = b.iterate(1)
        for i, o in enumerate(state["out"]):
            b.get_sigma(i, o)
        return {"residual": r, "sigma": state["out"]}
    if kind == "train":
        net = state["net"]
        net.train_step(state["x"], state["t"], 1e-4)
        s = net.lib.df_mlp_grads(net.h, ctypes.c_void_p(state["grads"].data_ptr()), 1)
        assert s == df.DF_OK
        return {"grads": state["grads"]}
    if kind == "predict":
        d = state["d"]
        state["net"].forward(state["x"], state["y"])
        df.warmstart_sigma(d, state["y"], state["mean"], state["sd"], state["kmap"])
        d.get_sigma(state["sigma"])
        d.get_gtilde(state["g"])
        return {"y": state["y"], "sigma": state["sigma"], "g": state["g"]}
    raise KeyError(kind)


# ---------------------------------------------------------------------------
# work a pass cannot do without
# ---------------------------------------------------------------------------

def _fft(planes, n):
    return planes * 5.0 * n * max(1.0, math.log2(n))


def _pass_work(dim, nk, n_w, m_max, symmetry):
    """One loop pass: g, Delta, gamma and Sigma~ read, Sigma~ written; flops: the ladders
    (8 n^3 real each: diag Gamma by LU and truncated substitutions) and the lattice FFTs."""
    c = dict(dim=dim, nk=nk, n_w=n_w, m_max=m_max, symmetry=symmetry)
    n, nb, ne = nk ** dim, 2 * m_max + 1, n_w + 2 * m_max
    planes = (m_max + 1 if symmetry == 2 else nb) * n_w
    return {"bytes": 16.0 * (2 * ne + 2 * nb * n_w * n_w + 2 * n_w * n),
            "flops": _ladders(c) * 8.0 * n_w ** 3 + _fft(2 * planes + 2 * n_w, n)}


def work(case):
    kind = case["kind"]
    if kind == "train":
        dims = (case["n_in"], case["width"], case["width"], case["width"], case["n_out"])
        p = sum(a * b + b for a, b in zip(dims[:-1], dims[1:]))
        b = case["batch"]
        # parameters and both moments read and written, gradients written, the batch read
        return {"bytes": 4.0 * (7 * p + b * (case["n_in"] + case["n_out"])), "flops": 6.0 * b * p}
    if kind == "predict":
        n_in, n_out = _predict_sizes(case)
        dims = (n_in, case["width"], case["width"], case["width"], n_out)
        p = sum(a * b + b for a, b in zip(dims[:-1], dims[1:]))
        n, n_w, ne = case["nk"] ** 2, case["n_w"], case["n_w"] + 2 * case["m_max"]
        # weights, mean, sd and map read; output, Sigma~ and G~ written
        return {"bytes": 4.0 * (p + 3 * n_out + n) + 16.0 * (n_w * n + ne * n), "flops": 2.0 * p + _fft(n_w, n)}
    if kind == "batch":
        tot = {"bytes": 0.0, "flops": 0.0}
        for w in _batch_workloads(case, 0):
            one = _pass_work(w.dim, w.nk, w.n_w, w.m_max, case["symmetry"])
            tot = {k: tot[k] + one[k] for k in tot}
        return tot
    dim, nk, n_w, m_max = case["dim"], case["nk"], case["n_w"], case["m_max"]
    n, nb, ne = nk ** dim, 2 * m_max + 1, n_w + 2 * m_max
    if kind == "loop":
        one = _pass_work(dim, nk, n_w, m_max, case["symmetry"])
        return {"bytes": one["bytes"], "flops": case["passes"] * one["flops"]}
    gam = 16.0 * 2 * nb * n_w * n_w
    if kind == "ladders":
        return {"bytes": gam + 16.0 * (ne * n + 3 * nb * n_w * n),
                "flops": _ladders(case) * 8.0 * n_w ** 3 + _fft(nb * n_w, n)}
    # susceptibilities: one right-hand side per ladder
    return {"bytes": gam + 16.0 * (n_w * n + 2 * nb * n),
            "flops": _ladders(case) * (8.0 / 3.0 * n_w ** 3 + 24.0 * n_w ** 2) + _fft(3 * nb * n_w, n)}


# ---------------------------------------------------------------------------
# the same results in 64 bits by plain torch
# ---------------------------------------------------------------------------

def _t(a):
    return torch.as_tensor(np.ascontiguousarray(a)).cuda()


def _eps(w):
    k = 2.0 * math.pi * torch.arange(w.nk, dtype=torch.float64, device="cuda") / w.nk
    axes = torch.meshgrid(*([k] * w.dim), indexing="ij")
    e = sum(-2.0 * w.t * torch.cos(a) for a in axes)
    if w.dim == 2:
        e = e - 4.0 * w.tp * torch.cos(axes[0]) * torch.cos(axes[1])
    return e.reshape(-1)


class _Plain:
    """The loop's steps for one workload: complex128, torch.fft and batched LAPACK-style solves."""

    def __init__(self, w, reduce):
        self.w, self.reduce = w, reduce
        self.g, self.delta = _t(w.g)[:, None], _t(w.delta)[:, None]
        uu, ud = _t(w.gamma_uu), _t(w.gamma_ud)
        self.gamma = torch.stack([uu + ud, uu - ud])
        self.eps = _eps(w)[None, :]
        self.g0 = 1.0 / (1.0 / self.g + self.delta - self.eps) - self.g
        self.box = slice(w.m_max, w.m_max + w.n_w)

    def grid(self, x):
        return x.reshape(x.shape[:-1] + (self.w.nk,) * self.w.dim)

    def axes(self):
        return tuple(range(-self.w.dim, 0))

    def to_r(self, x):
        return torch.fft.ifftn(self.grid(x), dim=self.axes())

    def to_k(self, x):
        y = torch.fft.fftn(x, dim=self.axes())
        return y.reshape(y.shape[:-self.w.dim] + (-1,))

    def minus(self, x):
        return torch.roll(torch.flip(x, self.axes()), (1,) * self.w.dim, self.axes())

    def dyson(self, sigma):
        gt = self.g0.clone()
        gt[self.box] = 1.0 / (1.0 / self.g0[self.box] - sigma)
        return gt

    def bubble(self, planes):
        """-(T/N) sum_k A_w(k) A_{w+W}(k+q), [N_W][n_w][N]."""
        w = self.w
        r = self.to_r(planes)
        rm = self.minus(r)[self.box]
        out = torch.empty(w.n_bos, w.n_w, w.N, dtype=torch.complex128, device="cuda")
        for a in range(w.n_bos):
            out[a] = self.to_k(rm * r[a:a + w.n_w]) * (-1.0 / w.beta)
        return out

    def momenta(self):
        """(representatives, orbit of each momentum): one per class of axis permutations and sign
        flips for inputs that have that symmetry, else every momentum."""
        w = self.w
        if not self.reduce:
            i = torch.arange(w.N, device="cuda")
            return i, i
        i = np.indices((w.nk,) * w.dim).reshape(w.dim, -1)
        f = np.sort(np.minimum(i, w.nk - i), axis=0)
        key = np.ravel_multi_index(f, (w.nk,) * w.dim)
        _, first, inv = np.unique(key, return_index=True, return_inverse=True)
        return _t(first), _t(inv.reshape(-1))

    def solve(self, chi, a, c, q, rhs):
        """D^-1 rhs for the momenta q: D = 1 - gamma diag(chi~), [len(q)][n][.]."""
        n = self.w.n_w
        gam = self.gamma[c, a]
        d = torch.eye(n, dtype=torch.complex128, device="cuda") - gam[None] * chi[a][:, q].T[:, None, :]
        return torch.linalg.solve(d, rhs)

    def brackets(self, chi):
        """c (Gamma_ww - (gamma chi~ gamma)_ww / 2) per channel, [2][N_W][n_w][N]."""
        w = self.w
        rep, orb = self.momenta()
        out = torch.empty(2, w.n_bos, w.n_w, w.N, dtype=torch.complex128, device="cuda")
        step = max(1, (1 << 26) // (w.n_w * w.n_w))
        for c in range(2):
            for a in range(w.n_bos):
                if self.reduce and a < w.m_max:
                    continue
                gam = self.gamma[c, a]
                part = []
                for q0 in range(0, rep.numel(), step):
                    q = rep[q0:q0 + step]
                    s = self.solve(chi, a, c, q, gam[None].expand(q.numel(), -1, -1))
                    part.append(torch.diagonal(s, dim1=1, dim2=2).T)
                two = (gam * gam.T) @ chi[a][:, rep]
                k = (1.0 if c == 0 else 3.0) * (torch.cat(part, 1) - 0.5 * two)
                out[c, a] = k[:, orb]
                if self.reduce and a > w.m_max:        # -W: the frequency-reversed conjugate
                    out[c, 2 * w.m_max - a] = out[c, a].flip(0).conj()
        return out

    def one_pass(self, sigma):
        w = self.w
        gt = self.dyson(sigma)
        kern = self.brackets(self.bubble(gt)).sum(0)
        r = self.to_r(gt)
        acc = 0.0
        for a in range(w.n_bos):
            acc = acc + self.minus(self.to_r(kern[a])) * r[a:a + w.n_w]
        new = self.to_k(acc) * (0.5 / w.beta)
        return new, float((new - sigma).abs().max() / new.abs().max())

    def susceptibility(self, sigma):
        w = self.w
        gt = self.dyson(sigma)
        a_ = 1.0 / (self.delta - self.eps)
        g_lat = a_ + a_ / self.g * gt / self.g * a_
        frak = gt * (self.g0 + self.g) / self.g0
        chi, lv, bare = self.bubble(gt), self.bubble(frak), self.bubble(g_lat).sum(1)
        out = torch.empty(2, w.n_bos, w.N, dtype=torch.complex128, device="cuda")
        q = torch.arange(w.N, device="cuda")
        for c in range(2):
            for a in range(w.n_bos):
                rhs = (self.gamma[c, a] @ lv[a]).T[:, :, None]
                x = self.solve(chi, a, c, q, rhs)[:, :, 0]
                out[c, a] = bare[a] + (lv[a].T * x).sum(1)
        return out


def _zero_sigma(w):
    return torch.zeros(w.n_w, w.N, dtype=torch.complex128, device="cuda")


def _layers(flat, dims):
    """[(W, b)] in FP64 from the flat parameters."""
    out, o = [], 0
    for a, b in zip(dims[:-1], dims[1:]):
        out.append((flat[o:o + a * b].double().reshape(a, b), flat[o + a * b:o + a * b + b].double()))
        o += a * b + b
    return out


def exact(case, seed):
    kind = case["kind"]
    if kind in ("loop", "ladders", "chi"):
        w = _workload(case, seed)
        p = _Plain(w, case["symmetry"] == 2)
        if kind == "loop":
            s, r = _zero_sigma(w), 0.0
            for _ in range(case["passes"]):
                s, r = p.one_pass(s)
            return {"sigma": s, "residual": r}
        if kind == "ladders":
            chi = p.bubble(p.dyson(_zero_sigma(w)))
            return {"chi": chi, "kernel": p.brackets(chi)}
        return {"chi": p.susceptibility(_zero_sigma(w))}
    if kind == "batch":
        sig, res = [], []
        for w in _batch_workloads(case, seed):
            s, r = _Plain(w, case["symmetry"] == 2).one_pass(_zero_sigma(w))
            sig.append(s)
            res.append(r)
        return {"residual": np.array(res), "sigma": sig}
    if kind == "train":
        dims = (case["n_in"], case["width"], case["width"], case["width"], case["n_out"])
        layers = _layers(_weights(dims, seed), dims)
        x, t = _train_data(case, seed)
        acts = [x.double()]
        for l, (wt, b) in enumerate(layers):
            z = acts[-1] @ wt + b
            acts.append(torch.tanh(z) if l < 3 else z)
        dz = (acts[4] - t.double()) * (2.0 / t.numel())
        parts = []
        for l in (3, 2, 1, 0):
            parts[:0] = [(acts[l].T @ dz).reshape(-1), dz.sum(0)]
            if l:
                dz = (dz @ layers[l][0].T) * (1.0 - acts[l] ** 2)
        return {"grads": torch.cat(parts)}
    if kind == "predict":
        n_in, n_out = _predict_sizes(case)
        dims = (n_in, case["width"], case["width"], case["width"], n_out)
        w, x, mean, sd, kmap = _predict_data(case, seed)
        y = x.double()
        for l, (wt, b) in enumerate(_layers(_weights(dims, seed), dims)):
            y = y @ wt + b
            y = torch.tanh(y) if l < 3 else y
        half = w.n_w // 2
        s = (y[0] * sd.double() + mean.double()).reshape(-1, half, 2)
        s = torch.complex(s[..., 0], s[..., 1])[kmap.long()].T      # [half][N], w_n > 0
        s = torch.cat([s.flip(0).conj().resolve_conj(), s])
        p = _Plain(w, False)
        return {"y": y, "sigma": s, "g": p.dyson(s)}
    raise KeyError(kind)
