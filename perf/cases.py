"""Timed cases of the emulated ZGEMM and the KKR tau_00 solve.

A case is a dict of plain values; ``kind`` names the path:

* ``zgemm``    one product through ``ozaki_zgemm`` (S slices; S = 0: the selector chooses);
* ``combine``  two products into one matrix, C = a1 op(A1) op(B1), then C = a2 op(A2) op(B2) + b2 C;
* ``vbatch``   a batch of products of different sizes through ``ozaki_zgemm_vbatched``;
* ``single``   M = I - t G of one LIZ (``kkr_build_m``), then ``kkr_tau00``;
* ``step``     the M of every atom of one lattice at one energy (``kkr_build_m_shared_sizes``),
               then all their tau_00 (``kkr_tau00_batched`` with leaf panels).

Every pass starts from the inputs alone (a solve overwrites its M, so the pass builds M again)
and returns the whole product or every tau_00 block.  Inputs are drawn on the GPU from the seed:
matrix entries U(-1, 1) 2^round(N(0, 2)) for the products, and the KKR recipe of ``synth`` (bcc
LIZ, diagonal t of magnitude 0.05..0.15, G_ij = R_ij e^(-r/1.5) e^(ikr) scaled so that
||t G||_2 <= 0.9) for the solves.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

import paper_2603_29975_gb300 as ozk
import synth

C128 = torch.complex128
LIZ_LO, LIZ_HI = 27, 169                       # sites of the contour workload's LIZs


def listed():
    return [
        # the smallest product of a solve: one 64-wide pivot panel against a 64-wide block
        dict(name="zgemm_64", kind="zgemm", m=64, n=64, k=64, S=7, ta="N", tb="N"),
        # the accuracy study's square product at the 55-bit mode
        dict(name="zgemm_512", kind="zgemm", m=512, n=512, k=512, S=7, ta="N", tb="N"),
        # odd sizes, conjugate and plain transposes and general scalars at the 39-bit mode
        dict(name="combine_ragged", kind="combine", m=1001, n=777, k=389, k2=131, S=5, ta="C", tb="T"),
        # many bits: the selector's fallback slice count on a mid-sized product
        dict(name="zgemm_2048_s10", kind="zgemm", m=2048, n=2048, k=2048, S=10, ta="N", tb="N"),
        # the slice count chosen and the product checked by the library: a panel update
        dict(name="zgemm_auto", kind="zgemm", m=1536, n=1536, k=192, S=0, ta="N", tb="N"),
        # a large product: the order of the lmax = 4 matrix with spin
        dict(name="zgemm_5650", kind="zgemm", m=5650, n=5650, k=5650, S=7, ta="N", tb="N"),
        # products of different sizes in one call, as a user's own blocked algorithm issues them
        dict(name="vbatch_48", kind="vbatch", batch=48, mlo=200, mhi=1600, klo=16, khi=192, S=7, sizes=11),
        # one atom at one energy (65-site LIZ, lmax = 3)
        dict(name="single_1040", kind="single", L=65, b=16, S=7, nb=64, e_re=0.5, e_im=0.05),
        # a small system: 16 atoms of mixed LIZ at one energy, 39 bits
        dict(name="step_16_s5", kind="step", atoms=16, lo=LIZ_LO, hi=LIZ_HI, b=16, S=5, W=192, w=64, sizes=20260332,
             e_re=0.1, e_im=0.9),
        # one atom with lmax = 4 and spin (113 sites, n = 5650)
        dict(name="step_1_n5650", kind="step", atoms=1, lo=113, hi=113, b=50, S=7, W=200, w=50, sizes=1, e_re=0.5,
             e_im=0.05),
        # the contour workload's step: 256 atoms of mixed LIZ at one energy, 55 bits
        dict(name="step_256", kind="step", atoms=256, lo=LIZ_LO, hi=LIZ_HI, b=16, S=7, W=192, w=64, sizes=20260332,
             e_re=0.4, e_im=0.7),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["zgemm", "zgemm", "combine", "vbatch", "single", "step", "step"])
    # the precision modes of 31..63 bits, the two used most drawn more often
    S = rng.choice([4, 5, 5, 6, 7, 7, 7, 8])
    if kind in ("zgemm", "combine"):
        m, n, k = (_log_int(rng, 16, 6000) for _ in range(3))
        ta, tb = rng.choice("NNTC"), rng.choice("NNTC")
        if kind == "zgemm":
            return dict(kind=kind, m=m, n=n, k=k, S=rng.choice([S, S, S, 10]) if m * n * k < 2e10 else S, ta=ta, tb=tb)
        return dict(kind=kind, m=m, n=n, k=k, k2=_log_int(rng, 16, 2000), S=S, ta=ta, tb=tb)
    if kind == "vbatch":
        lo, klo = _log_int(rng, 16, 600), _log_int(rng, 8, 100)
        return dict(kind=kind, batch=rng.randint(2, 64), mlo=lo, mhi=min(1600, lo * rng.randint(1, 4)), klo=klo,
                    khi=klo * rng.randint(1, 4), S=S, sizes=rng.randrange(1 << 20))
    E = dict(e_re=round(rng.uniform(-1.2, 0.7), 3), e_im=round(math.exp(rng.uniform(math.log(0.005), 0.0)), 4))
    if kind == "single":
        b = rng.choice([16, 16, 9, 50])
        return dict(kind=kind, L=_log_int(rng, 3, 169 if b < 50 else 64), b=b, S=S, nb=b * rng.randint(1, 112 // b), **E)
    b, w = rng.choice([(16, 64), (16, 64), (16, 48), (16, 80), (50, 50), (9, 63)])
    lo = _log_int(rng, 9, 100 if b < 50 else 30)
    hi = rng.randint(lo, min(LIZ_HI, 3 * lo) if b < 50 else 2 * lo)
    return dict(kind=kind, atoms=_log_int(rng, 1, 200 if b < 50 else 48), lo=lo, hi=hi, b=b, S=S, W=w * rng.randint(1, 4),
                w=w, sizes=rng.randrange(1 << 20), **E)


# ----------------------------------------------------------------------------- inputs
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _scaled_uniform(g, rows, cols):
    """rows x cols complex128, column major: U(-1, 1) 2^round(N(0, 2)) per real and imaginary part."""
    x = torch.rand((cols, rows, 2), dtype=torch.float64, device="cuda", generator=g).mul_(2).sub_(1)
    e = torch.randn((cols, rows, 2), dtype=torch.float32, device="cuda", generator=g).mul_(2).round_()
    return torch.view_as_complex(torch.ldexp(x, e)).t()


def _empty(rows, cols):
    return torch.zeros((cols, rows), dtype=C128, device="cuda").t()


def _op_shape(rows, cols, op):
    return (rows, cols) if op == "N" else (cols, rows)


def _batch_sizes(case):
    r = random.Random(int(case["sizes"]))
    return [(r.randint(case["mlo"], case["mhi"]), r.randint(case["mlo"], case["mhi"]),
             r.randint(case["klo"], case["khi"])) for _ in range(case["batch"])]


def _site_counts(case):
    return [int(v) for v in synth.liz_sizes(case["atoms"], case["lo"], case["hi"], case["sizes"])]


def _t_blocks(g, L, b):
    """L diagonal b x b blocks, entries 0.1 (0.5 + U) e^(i phi)."""
    u = torch.rand((L, b), dtype=torch.float64, device="cuda", generator=g)
    phi = torch.rand((L, b), dtype=torch.float64, device="cuda", generator=g) * (2 * math.pi)
    return torch.diag_embed(torch.polar(0.1 * (0.5 + u), phi))


def _structure(g, L, b, E, t):
    """G (column major) of an L-site bcc LIZ at energy E for the single-site blocks t."""
    pos = synth.bcc_sites(L)
    d = np.sqrt(((pos[:, None, :] - pos[None, :, :]) ** 2).sum(-1))
    f = np.exp(-d / 1.5) * np.exp(1j * np.sqrt(complex(E)) * d)
    f[np.arange(L), np.arange(L)] = 0.0
    fd = torch.from_numpy(f).cuda()
    n = L * b
    R = torch.rand((n, n, 2), dtype=torch.float64, device="cuda", generator=g).mul_(2).sub_(1)
    G = (torch.view_as_complex(R).reshape(L, b, L, b) * fd[:, None, :, None]).reshape(n, n) / math.sqrt(b)
    tG = torch.diagonal(t, dim1=1, dim2=2).reshape(n, 1) * G
    v = torch.ones((n, 1), dtype=C128, device="cuda") / math.sqrt(n)
    s = torch.zeros((), dtype=torch.float64, device="cuda")
    for _ in range(20):
        v = tG.mH @ (tG @ v)
        s = torch.linalg.vector_norm(v)
        v = v / s.clamp_min(1e-300)
    norm = math.sqrt(float(s))
    if norm > 0.9:
        G = G * (0.9 / norm)
    return G.t().contiguous().t()


def _pointers(xs):
    return torch.tensor([x.data_ptr() for x in xs], dtype=torch.int64, device="cuda")


# ----------------------------------------------------------------------------- cases
def prepare(case, seed):
    g = _gen(seed)
    s = dict(case=case, h=ozk.Handle())
    kind = case["kind"]
    if kind in ("zgemm", "combine"):
        m, n = case["m"], case["n"]
        for i, k in enumerate([case["k"]] + ([case["k2"]] if kind == "combine" else [])):
            s["A%d" % i] = _scaled_uniform(g, *_op_shape(m, k, case["ta"]))
            s["B%d" % i] = _scaled_uniform(g, *_op_shape(k, n, case["tb"]))
        s["C"] = _empty(m, n)
        if case["S"] == 0:
            s["h"].selector_load()
    elif kind == "vbatch":
        sizes = _batch_sizes(case)
        s["A"] = [_scaled_uniform(g, m, k) for m, n, k in sizes]
        s["B"] = [_scaled_uniform(g, k, n) for m, n, k in sizes]
        s["C"] = [_empty(m, n) for m, n, k in sizes]
    elif kind == "single":
        L, b = case["L"], case["b"]
        s["t"] = _t_blocks(g, L, b)                       # diagonal blocks: either storage order
        s["G"] = _structure(g, L, b, complex(case["e_re"], case["e_im"]), s["t"])
        s["M"], s["tau"] = _empty(L * b, L * b), _empty(b, b)
    else:
        b, Ls = case["b"], _site_counts(case)
        ts = [_t_blocks(g, L, b) for L in Ls]
        big = max(range(len(Ls)), key=lambda a: Ls[a])
        s["Ls"], s["ns"], s["t"] = Ls, [L * b for L in Ls], ts
        s["G"] = _structure(g, Ls[big], b, complex(case["e_re"], case["e_im"]), ts[big])
        s["M"] = [torch.empty((n, n), dtype=C128, device="cuda") for n in s["ns"]]
        s["tau"] = torch.zeros((len(Ls), b, b), dtype=C128, device="cuda")   # column-major blocks
        s["pt"], s["pm"], s["ptau"] = _pointers(ts), _pointers(s["M"]), _pointers(list(s["tau"]))
    return s


ALPHA, ALPHA2, BETA2 = 0.75 - 0.5j, -1.25 + 0.25j, 0.5 + 1.0j   # the combine case's scalars


def run(s):
    case, h = s["case"], s["h"]
    kind, S = case["kind"], case["S"]
    if kind == "zgemm":
        return ozk.ozaki_zgemm(h, s["A0"], s["B0"], s["C"], S=S, transa=case["ta"], transb=case["tb"])
    if kind == "combine":
        ozk.ozaki_zgemm(h, s["A0"], s["B0"], s["C"], S=S, alpha=ALPHA, transa=case["ta"], transb=case["tb"])
        return ozk.ozaki_zgemm(h, s["A1"], s["B1"], s["C"], S=S, alpha=ALPHA2, beta=BETA2, transa=case["ta"],
                               transb=case["tb"])
    if kind == "vbatch":
        out, s["tables"] = ozk.ozaki_zgemm_vbatched(h, s["A"], s["B"], s["C"], S=S)
        return out
    if kind == "single":
        ozk.kkr_build_m(h, s["t"], s["G"], s["M"])
        return ozk.kkr_tau00(h, s["M"], s["t"][0], s["tau"], S=S, nb=case["nb"])
    ozk.kkr_build_m_shared_sizes_ptrs(h, s["Ls"], case["b"], s["pt"], s["G"], s["pm"], S=S)
    ozk.kkr_tau00_batched_ptrs(h, s["ns"], case["b"], s["pm"], s["pt"], s["ptau"], S=S, nb=case["W"], leaf=case["w"])
    return s["tau"]


def exact(case, seed):
    s = prepare(case, seed)
    kind = case["kind"]
    op = {"N": lambda x: x, "T": lambda x: x.t(), "C": lambda x: x.mH}
    if kind in ("zgemm", "combine"):
        Z = op[case["ta"]](s["A0"]) @ op[case["tb"]](s["B0"])
        if kind == "zgemm":
            return Z
        return ALPHA2 * (op[case["ta"]](s["A1"]) @ op[case["tb"]](s["B1"])) + BETA2 * (ALPHA * Z)
    if kind == "vbatch":
        return [a @ b for a, b in zip(s["A"], s["B"])]

    def tau(t, G):
        L, b = t.shape[0], t.shape[1]
        n = L * b
        M = torch.eye(n, dtype=C128, device="cuda") - torch.diagonal(t, dim1=1, dim2=2).reshape(n, 1) * G[:n, :n]
        rhs = torch.zeros((n, b), dtype=C128, device="cuda")
        rhs[:b] = torch.eye(b, dtype=C128, device="cuda")
        return torch.linalg.solve(M, rhs)[:b] @ t[0]

    if kind == "single":
        return tau(s["t"], s["G"])
    s["M"] = None
    return torch.stack([tau(t, s["G"]).t() for t in s["t"]])


def work(case):
    """Bytes: inputs once, outputs once (16 per complex element).  Flops: the integer products of
    the slice pairs, S (S + 1) / 2 times the 8 m n k (products) or (8/3) n^3 (solves) of the
    binary64 operation, plus 8 n^2 b per M built; S = 0 counts the smallest slice count, 3."""
    pairs = max(case["S"], 3) * (max(case["S"], 3) + 1) / 2
    kind = case["kind"]
    if kind in ("zgemm", "combine"):
        m, n = case["m"], case["n"]
        k = case["k"] + case.get("k2", 0)
        return {"bytes": 16.0 * (m * k + k * n + m * n), "flops": pairs * 8.0 * m * n * k}
    if kind == "vbatch":
        sz = _batch_sizes(case)
        return {"bytes": 16.0 * sum(m * k + k * n + m * n for m, n, k in sz),
                "flops": pairs * 8.0 * sum(float(m) * n * k for m, n, k in sz)}
    b = case["b"]
    Ls = [case["L"]] if kind == "single" else _site_counts(case)
    ns = [float(L * b) for L in Ls]
    nbytes = 16.0 * (sum(n * b for n in ns) + max(ns) ** 2 + len(ns) * b * b)
    build = sum(8.0 * n * n * b for n in ns) * (1.0 if kind == "single" else pairs)
    return {"bytes": nbytes, "flops": pairs * sum(8.0 / 3.0 * n ** 3 for n in ns) + build}
