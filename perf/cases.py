"""What a program asks of this library, as cases that can be timed.

Whole applications (chains, a tree, a lockstep group, a mixed serving set, the sketching
method) and the building blocks that the sweeps are made of (products, the truncation
eigensolver, the LQ), each through the entry point a program calls.  Inputs are random
networks of unit Frobenius norm per tensor, Gaussian, drawn on the GPU from the seed.

Gauge.  A compressed network is determined up to one phase per basis vector of every inner
bond (an eigenvector has no phase of its own), and an eigenvector up to one phase.  Results
are returned whole with those phases fixed: every basis vector is turned so that its
overlap with a fixed vector is positive (where that overlap is zero it is left alone).
"""
import ctypes
import math
import random

import numpy as np
import torch

from paper_2601_19650_gb300 import _cbc

DT = {"f32": (torch.float32, _cbc.CBC_F32), "f64": (torch.float64, _cbc.CBC_F64),
      "c64": (torch.complex64, _cbc.CBC_C64), "c128": (torch.complex128, _cbc.CBC_C128)}
WIDE = {"f32": "f64", "f64": "f64", "c64": "c128", "c128": "c128"}


def listed():
    return [
        # a first call, a unit test, an inner step of a small simulation: latency and launches
        dict(name="apply_tiny", kind="apply", topo="chain", L=8, d=2, chi=8, D=4, cap=8, tol=0.0,
             dtype="f64", prec="fp64"),
        # the default precision on a middle-sized chain, a cap and a tolerance together
        dict(name="apply_fp64", kind="apply", topo="chain", L=32, d=2, chi=64, D=8, cap=64,
             tol=1e-8, dtype="c128", prec="fp64"),
        # one application of the benchmark's MPO to its MPS in the mixed path
        dict(name="apply_mixed", kind="apply", topo="chain", L=64, d=2, chi=128, D=16, cap=128,
             tol=0.0, dtype="c64", prec="mixed"),
        # the benchmark's way of use: a lockstep group of equal shapes (a shorter chain)
        dict(name="apply_group", kind="group", topo="chain", L=24, d=2, chi=128, D=16, cap=128,
             tol=0.0, dtype="c64", prec="mixed", count=64),
        # a tree operator on a tree state, 64 leaves
        dict(name="apply_tree", kind="apply", topo="binary", L=6, d=2, chi=64, D=8, cap=64,
             tol=0.0, dtype="f32", prec="mixed"),
        # a serving set: chains of unlike shapes, one call
        dict(name="apply_serving", kind="serving", topo="chain", mix=10, count=6, top=256,
             dtype="f32", prec="mixed"),
        # the randomised method on the shape of the paper's benchmark
        dict(name="src_paper", kind="src", topo="chain", L=50, d=3, chi=40, D=40, cap=20,
             tol=0.0, dtype="c128", prec="mixed"),
        # the first contraction of a site of the large chain, a quarter of its rows
        dict(name="gemm_mixed", kind="gemm", M=8192, N=4096, K=1024, ta=0, ca=0, tb=0, cb=0,
             dtype="c128", prec="mixed", slices=5),
        # an FP64 product of ragged sizes with a conjugate transpose (a Gram-like shape)
        dict(name="gemm_fp64", kind="gemm", M=501, N=777, K=1030, ta=0, ca=0, tb=1, cb=1,
             dtype="c128", prec="fp64", slices=0),
        # the truncations of a lockstep group at one cut
        dict(name="heev_group", kind="heev", m=256, kmax=128, nb=64, dtype="c128", mixed=1),
        # one truncation of a large bond
        dict(name="heev_large", kind="heev", m=2048, kmax=512, nb=1, dtype="c128", mixed=0),
        # the LQ of a lockstep group at one site
        dict(name="cholqr_group", kind="cholqr", m=128, n=256, nb=64, dtype="c128"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["apply", "apply", "group", "tree", "serving", "src", "gemm", "gemm", "heev",
                       "heev", "cholqr"])
    if kind in ("apply", "group"):
        d = rng.choice([2, 2, 2, 3, 4])
        chi = _log(rng, 6, 128 if d == 2 else 64)
        c = dict(kind=kind, topo="chain", L=_log(rng, 4, 40), d=d, chi=chi, D=_log(rng, 2, 16),
                 cap=max(2, int(chi * rng.choice([1.0, 1.0, 0.5]))), tol=rng.choice([0.0, 0.0, 1e-8]),
                 dtype=rng.choice(["f32", "f64", "c64", "c128"]),
                 prec=rng.choice(["fp64", "mixed"]))
        if kind == "group":
            c.update(tol=0.0, prec="mixed", L=min(c["L"], 20), count=_log(rng, 3, 40))
        elif c["prec"] == "fp64" and chi > 48:
            c.update(chi=48, cap=min(c["cap"], 48))
        return c
    if kind == "tree":
        chi = _log(rng, 6, 48)
        return dict(kind="apply", topo="binary", L=rng.choice([3, 4, 5]), d=rng.choice([2, 3]),
                    chi=chi, D=_log(rng, 2, 8), cap=chi, tol=0.0,
                    dtype=rng.choice(["f32", "f64", "c64"]), prec=rng.choice(["fp64", "mixed"]))
    if kind == "serving":
        top = rng.choice([64, 128])
        return dict(kind="serving", topo="chain", mix=rng.randrange(1000),
                    count=2 if top > 64 else rng.choice([2, 3, 4]), top=top,
                    dtype=rng.choice(["f32", "c64"]), prec="mixed")
    if kind == "src":
        chi = _log(rng, 8, 64)
        return dict(kind="src", topo="chain", L=_log(rng, 6, 50), d=rng.choice([2, 3]), chi=chi,
                    D=_log(rng, 2, 40), cap=max(2, chi // 2), tol=0.0,
                    dtype=rng.choice(["f64", "c128"]), prec=rng.choice(["fp64", "mixed"]))
    if kind == "gemm":
        prec = rng.choice(["fp64", "mixed"])
        hi = 1500 if prec == "fp64" else 5000
        cplx = rng.random() < 0.6
        return dict(kind="gemm", M=_log(rng, 8, hi), N=_log(rng, 8, hi), K=_log(rng, 4, hi),
                    ta=rng.randrange(2), ca=int(cplx) * rng.randrange(2), tb=rng.randrange(2),
                    cb=int(cplx) * rng.randrange(2), dtype="c128" if cplx else "f64", prec=prec,
                    slices=0 if prec == "fp64" else rng.choice([0, 5]))
    if kind == "heev":
        if rng.random() < 0.5:
            m, nb = _log(rng, 200, 1800), 1
        else:
            m, nb = _log(rng, 8, 260), _log(rng, 2, 64)
        return dict(kind="heev", m=m, kmax=max(1, int(m * rng.choice([0.25, 0.5, 0.5, 1.0]))),
                    nb=nb, dtype=rng.choice(["f64", "c128"]), mixed=rng.randrange(2))
    m = _log(rng, 4, 300)
    return dict(kind="cholqr", m=m, n=int(m * rng.uniform(1.2, 4.0)) + 1,
                nb=1 if m > 160 else _log(rng, 1, 64), dtype=rng.choice(["f64", "c128"]))


# ---- shapes -------------------------------------------------------------------------

def _topology(c):
    """(parent, phys): a chain rooted at its first site, or a perfect binary tree of depth
    L whose leaves carry the physical legs."""
    if c["topo"] == "chain":
        return list(range(-1, c["L"] - 1)), [c["d"]] * c["L"]
    n = 2 ** (c["L"] + 1) - 1
    leaves = 2 ** c["L"]
    return [-1] + [(j - 1) // 2 for j in range(1, n)], [1] * (n - leaves) + [c["d"]] * leaves


def _children(parent):
    ch = [[] for _ in parent]
    for j, p in enumerate(parent):
        if p >= 0:
            ch[p].append(j)
    return ch


def _bonds(parent, phys, cap, power):
    """The bond of every node to its parent: the cap, or what the sites on either side span."""
    n, sub = len(parent), [p ** power for p in phys]
    for j in range(n - 1, 0, -1):
        sub[parent[j]] *= sub[j]
    return [1] + [min(cap, sub[j], sub[0] // sub[j]) for j in range(1, n)]


def _parts(c):
    """The chains of a serving set."""
    if c["kind"] != "serving":
        return [c]
    r = random.Random(c["mix"])
    out = []
    for _ in range(c["count"]):
        chi = r.choice([x for x in (32, 64, 128, 256) if x <= c["top"]])
        out.append(dict(c, kind="apply", L=r.randint(16, 64), d=2, chi=chi,
                        D=r.choice([4, 8, 16, 32]), cap=chi, tol=0.0))
    return out


# ---- inputs -------------------------------------------------------------------------

class _Handle:
    """A network of the library, freed with this object."""

    def __init__(self, parent, phys, bond, tensors, kind, stream):
        self.free = _cbc.ttn_destroy if kind == "state" else _cbc.ttno_destroy
        self.h = None
        self.h = _cbc.create_from_device(parent, phys, bond, tensors, kind, stream)

    def __del__(self):
        if self.h is not None:
            self.free(self.h)


def _tensors(c, gen, kind):
    parent, phys = _topology(c)
    ch = _children(parent)
    bond = _bonds(parent, phys, c["chi"] if kind == "state" else c["D"], 1 if kind == "state" else 2)
    out = []
    for j in range(len(parent)):
        site = (phys[j],) if kind == "state" else (phys[j], phys[j])
        shape = (bond[j], *site, *(bond[k] for k in ch[j]))
        x = torch.randn(shape, generator=gen, device="cuda", dtype=DT[c["dtype"]][0])
        out.append(x / torch.linalg.vector_norm(x))
    return parent, phys, bond, out


def _gen(seed, which=0):
    return torch.Generator(device="cuda").manual_seed(1_000_003 * (seed + 1) + which)


def _sketch(c, seed):
    """The random matrices of the sketching method, in host memory as a program draws them."""
    r = np.random.default_rng([seed, 3])
    _, phys = _topology(c)
    out = []
    for d in phys:
        x = r.standard_normal((d, c["cap"]))
        if c["dtype"] == "c128":
            x = (x + 1j * r.standard_normal((d, c["cap"]))) / math.sqrt(2.0)
        out.append(np.ascontiguousarray(x))
    return out


def _gemm_shapes(c):
    return (((c["K"], c["M"]) if c["ta"] else (c["M"], c["K"])),
            ((c["N"], c["K"]) if c["tb"] else (c["K"], c["N"])))


def _gram(c, seed):
    """Gram matrices as a cut of random networks has them: M M^H of an m x 8m matrix."""
    dt = DT[c["dtype"]][0]
    x = torch.randn((c["nb"], c["m"], 8 * c["m"]), generator=_gen(seed), device="cuda",
                    dtype=torch.complex64 if dt.is_complex else torch.float32)
    g = torch.matmul(x, x.mH).to(dt) / (8 * c["m"])
    return ((g + g.mH) / 2).contiguous()


def _rows(c, seed):
    """Blocks whose rows carry falling singular values, as the backward sweep has them."""
    x = torch.randn((c["nb"], c["m"], c["n"]), generator=_gen(seed), device="cuda",
                    dtype=DT[c["dtype"]][0])
    return x * torch.logspace(0, -3, c["m"], device="cuda", dtype=torch.float64)[None, :, None]


def prepare(case, seed):
    s = {"case": case}
    if case["kind"] == "gemm":
        g = _gen(seed)
        sa, sb = _gemm_shapes(case)
        dt = DT[case["dtype"]][0]
        s["A"] = torch.randn(sa, generator=g, device="cuda", dtype=dt)
        s["B"] = torch.randn(sb, generator=g, device="cuda", dtype=dt)
        return s
    if case["kind"] == "heev":
        return dict(s, A=_gram(case, seed))
    if case["kind"] == "cholqr":
        return dict(s, S=_rows(case, seed))
    parts = _parts(case) * (case["count"] if case["kind"] == "group" else 1)
    s["nets"] = []
    for j, c in enumerate(parts):
        g = _gen(seed, j)
        # chains of unlike shapes run side by side, each on a stream of its own
        st = torch.cuda.Stream() if case["kind"] == "serving" else torch.cuda.current_stream()
        state, op = _tensors(c, g, "state"), _tensors(c, g, "op")
        torch.cuda.synchronize()
        s["nets"].append((c, _Handle(*state, "state", st.cuda_stream),
                          _Handle(*op, "op", st.cuda_stream), st))
    prec = _cbc.CBC_PREC_MIXED if case["prec"] == "mixed" else _cbc.CBC_PREC_FP64
    s["opt"] = _cbc.make_options(prec, max_group=case["count"] if case["kind"] == "group" else 0)
    if case["kind"] == "src":
        s["omega"] = _sketch(case, seed)
    return s


# ---- one pass -----------------------------------------------------------------------

def _weights(n, like):
    """A fixed vector of n entries of mixed signs and sizes."""
    t = torch.arange(n, device=like.device, dtype=torch.float64)
    return (torch.cos(1.0 + 0.7 * t) + 0.3 * torch.cos(2.9 * t * t + 0.5)).to(like.dtype)


_W = {}


def _fixed(n, like):
    key = (like.dtype, like.device)
    w = _W.get(key)
    if w is None or w.numel() < n:
        w = _W[key] = _weights(max(n, 4096), like)
    return w[:n]


def _fix_network(flat, parent, phys, bond):
    """Networks of one shape, rows of `flat`, with the phases of their inner bonds fixed."""
    ch = _children(parent)
    b, off, nodes = flat.shape[0], 0, []
    for j in range(len(parent)):
        shape = (bond[j], phys[j], *(bond[k] for k in ch[j]))
        n = math.prod(shape)
        nodes.append(flat[:, off:off + n].view(b, *shape))
        off += n
    for j in range(len(parent) - 1, 0, -1):
        x, p = nodes[j], parent[j]
        k = bond[j]
        # the overlap with a vector on the first basis vector of every child's bond: a row's
        # phase then takes one phase of each child's along, and errors don't build up
        z = torch.matmul(x.reshape(b, k, phys[j], -1)[..., 0], _fixed(phys[j], flat))
        ph = torch.sgn(z) + (z == 0)
        x.mul_(ph.conj().view(b, k, *([1] * (x.dim() - 2))))
        slot = 2 + ch[p].index(j)
        view = [b] + [1] * (nodes[p].dim() - 1)
        view[slot + 1] = k
        nodes[p].mul_(ph.view(view))
    return flat


def _fetch(case, outs, parts):
    """Every result network, whole: one flat buffer for each (one for a whole group), its
    bonds and the logarithm of its norm."""
    dt = case["dtype"] if case["prec"] == "mixed" else WIDE[case["dtype"]]
    info = [_cbc.ttn_get_info(h) for h in outs]
    flats = []
    for (n, bonds, _), c in zip(info, parts):
        parent, phys = _topology(c)
        ch = _children(parent)
        flats.append(sum(int(bonds[j]) * phys[j] * math.prod(int(bonds[k]) for k in ch[j])
                         for j in range(n)))
    together = case["kind"] == "group" and all((b == info[0][1]).all() for _, b, _ in info)
    res = []
    sizes = [(len(outs), flats[0])] if together else [(1, n) for n in flats]
    bufs = [torch.empty(s, dtype=DT[dt][0], device="cuda") for s in sizes]
    if case["kind"] == "serving":  # the copies run on the networks' own streams
        torch.cuda.current_stream().synchronize()
    for j, h in enumerate(outs):
        dst = bufs[0][j] if together else bufs[j]
        rc = _cbc.lib().ttn_get_network(h, ctypes.c_void_p(dst.data_ptr()), 1, DT[dt][1])
        if rc:
            raise _cbc.CBCError(rc, _cbc.cbc_last_error())
        _cbc.ttn_destroy(h)
    for j, buf in enumerate(bufs):
        parent, phys = _topology(parts[j])
        res.append(_fix_network(buf, parent, phys, [int(x) for x in info[j][1]]))
    return {"nodes": res, "bonds": np.stack([b for _, b, _ in info]) if together else
            [b for _, b, _ in info], "log_norm": np.array([x for _, _, x in info])}


def _fetch_host(h, c):
    """A small network as host arrays, the phases fixed there."""
    parent, phys = _topology(c)
    tens, bonds, log_norm = _cbc.fetch_network(h, _cbc.output_shape_fn(parent, phys),
                                               c["dtype"] in ("c64", "c128"))
    _cbc.ttn_destroy(h)
    flat = torch.from_numpy(np.concatenate([t.reshape(-1) for t in tens]))[None]
    return {"nodes": [_fix_network(flat, parent, phys, [int(x) for x in bonds])],
            "bonds": [bonds], "log_norm": np.array([log_norm])}


def _fix_vectors(u):
    """Eigenvectors (columns) with their phases fixed."""
    ph = torch.sgn(torch.matmul(_fixed(u.shape[-2], u), u))
    return u.mul_(ph.conj()[..., None, :])


def run(state):
    c = state["case"]
    if c["kind"] == "gemm":
        A, B = state["A"], state["B"]
        C = torch.empty((c["M"], c["N"]), dtype=A.dtype, device="cuda")
        prec = _cbc.CBC_PREC_MIXED if c["prec"] == "mixed" else _cbc.CBC_PREC_FP64
        _cbc.cbc_gemm(prec, c["slices"], DT[c["dtype"]][1], c["M"], c["N"], c["K"], A.data_ptr(),
                      A.shape[1], c["ta"], c["ca"], B.data_ptr(), B.shape[1], c["tb"], c["cb"],
                      C.data_ptr(), c["N"], torch.cuda.current_stream().cuda_stream)
        return C
    if c["kind"] == "heev":
        A = state["A"].clone()  # the call overwrites it
        m, k, nb = c["m"], c["kmax"], c["nb"]
        lam = torch.empty((nb, m), dtype=torch.float64, device="cuda")
        U = torch.empty((nb, m, k), dtype=A.dtype, device="cuda")
        _cbc.cbc_heev(DT[c["dtype"]][1], m, k, nb, A.data_ptr(), lam.data_ptr(), U.data_ptr(),
                      bool(c["mixed"]), torch.cuda.current_stream().cuda_stream)
        # beyond the candidates the eigenvalues are single-precision estimates
        return {"lam": lam[:, :k], "lam_rest": lam[:, k:].float(), "U": _fix_vectors(U)}
    if c["kind"] == "cholqr":
        S = state["S"].clone()  # replaced by the result
        _cbc.cbc_cholqr2(DT[c["dtype"]][1], c["m"], c["n"], c["nb"], S.data_ptr(),
                         torch.cuda.current_stream().cuda_stream)
        return S
    nets, opt = state["nets"], state["opt"]
    if c["kind"] == "src":
        p, st, op, _ = nets[0]
        return _fetch(c, [_cbc.src_apply(st.h, op.h, c["cap"], state["omega"], opt)], [p])
    if c["kind"] == "apply":
        p, st, op, _ = nets[0]
        out = _cbc.cbc_apply(st.h, op.h, c["cap"], c["tol"], opt)
        if c["L"] * c["d"] * c["chi"] ** 2 <= 4096:
            return _fetch_host(out, c)
        return _fetch(c, [out], [p])
    outs = _cbc.cbc_apply_batched([st.h for _, st, _, _ in nets], [op.h for _, _, op, _ in nets],
                                  [p["cap"] for p, *_ in nets], [p["tol"] for p, *_ in nets], opt)
    return _fetch(c, outs, [p for p, *_ in nets])


# ---- what a pass cannot do without --------------------------------------------------

def _work_network(c):
    """Elements in and out, and multiply-adds of the contractions, Gram products (half of
    them: they are Hermitian) and LQs of the sweeps."""
    parent, phys = _topology(c)
    n, ch = len(parent), _children(parent)
    a, b = _bonds(parent, phys, c["chi"], 1), _bonds(parent, phys, c["D"], 2)
    # kept bonds: the cap, what the product holds, what the sites span
    k = [1] + [min(c["cap"], x, a[j] * b[j]) for j, x in
               enumerate(_bonds(parent, phys, 1 << 60, 1))][1:]
    elems = sum(a[j] * phys[j] * math.prod(a[i] for i in ch[j])
                + b[j] * phys[j] ** 2 * math.prod(b[i] for i in ch[j])
                + k[j] * phys[j] * math.prod(k[i] for i in ch[j]) for j in range(n))

    def chain(dims, j):
        """Multiply-adds of T with the first environment, then W, then the other ones."""
        legs = [(a[i], b[i], x) for i, x in dims]
        d, total = phys[j], 0
        left = math.prod(x for x, _, _ in legs) * a_free * d
        rest = b_free
        for q, (ai, bi, xi) in enumerate(legs):
            if q == 0:
                total += left * bi * xi
                left = left // ai * bi * xi
                total += left * d * rest * math.prod(y for _, y, _ in legs[1:])
                left = left // bi * rest * math.prod(y for _, y, _ in legs[1:])
            else:
                total += left * xi
                left = left // (ai * bi) * xi
        return total

    macs = 0
    for j in range(n):
        if j:  # the way up: Z, S and R of this node
            a_free, b_free = a[j], b[j]
            cols = phys[j] * math.prod(k[i] for i in ch[j])
            if ch[j]:
                macs += chain([(i, k[i]) for i in ch[j]], j)
            else:
                macs += a[j] * b[j] * phys[j] ** 2
            macs += 2 * k[j] * a[j] * b[j] * cols + 2 * k[j] * k[j] * cols
        for i in ch[j]:  # the cut below this node, seen from above
            a_free, b_free = a[i], b[i]
            around = [(j, k[j])] + [(q, k[q]) for q in ch[j] if q != i]
            macs += chain(around, j)
            m, nn = phys[j] * math.prod(x for _, x in around), a[i] * b[i]
            if c["kind"] != "src":
                macs += m * nn * min(m, nn) // 2 + k[i] * m * nn
        if j and len(ch[parent[j]]) > 1 and c["kind"] != "src":  # and from below, on a tree
            a_free, b_free = a[j], b[j]
            if ch[j]:
                macs += chain([(i, k[i]) for i in ch[j]], j)
            m, nn = phys[j] * math.prod(k[i] for i in ch[j]), a[j] * b[j]
            macs += m * nn * min(m, nn) // 2 + k[j] * m * nn
    return elems, macs


def work(case):
    c = case
    cplx = c["dtype"] in ("c64", "c128")
    fl = 8.0 if cplx else 2.0
    es = 16.0 if cplx else 8.0
    if c["kind"] == "gemm":
        M, N, K = c["M"], c["N"], c["K"]
        return {"bytes": es * (M * K + K * N + M * N), "flops": fl * M * N * K}
    if c["kind"] == "heev":
        m, k, nb = c["m"], c["kmax"], c["nb"]
        return {"bytes": nb * (es * (m * m + m * k) + 8.0 * m),
                "flops": nb * fl * (2.0 / 3.0 * m ** 3 + 1.0 * m * m * k)}
    if c["kind"] == "cholqr":
        m, n, nb = c["m"], c["n"], c["nb"]
        return {"bytes": nb * es * 2.0 * m * n, "flops": nb * fl * (2.0 * m * m * n + m ** 3 / 3.0)}
    total = {"bytes": 0.0, "flops": 0.0}
    size = {"f32": 4, "f64": 8, "c64": 8, "c128": 16}[c["dtype"]]
    for p in _parts(c) * (c["count"] if c["kind"] == "group" else 1):
        e, macs = _work_network(p)
        total["bytes"] += size * e
        total["flops"] += fl * macs
    return total


# ---- the same numbers in plain 64-bit torch -----------------------------------------

def _contract(x, lx, y, ly):
    """x and y over the legs they share; the result's legs are x's others, then y's."""
    sh = [q for q in lx if q in ly]
    z = torch.tensordot(x, y, ([lx.index(q) for q in sh], [ly.index(q) for q in sh]))
    return z, [q for q in lx if q not in sh] + [q for q in ly if q not in sh]


def _order(x, lx, want):
    return x.permute([lx.index(q) for q in want])


def _truncate(m, cap, tol):
    """U_k^H M for the dominant left singular vectors U_k of M, normalised."""
    if m.shape[0] <= m.shape[1]:
        w, v = torch.linalg.eigh(m @ m.mH)
        f = v.flip(1).mH @ m
    else:
        w, v = torch.linalg.eigh(m.mH @ m)
        w, v = w.flip(0).clamp(min=0), v.flip(1)
        f = w.sqrt()[:, None] * v.mH
    w = (f.abs() ** 2).sum(1)
    g = f.shape[0]
    k = min(cap, g)
    if tol > 0:
        tail = w.flip(0).cumsum(0).flip(0)
        k = min(k, max(1, int((tail > tol * tol * tail[0]).sum())))
    f = f[:k]
    return f / torch.linalg.vector_norm(f)


def _exact_network(c, seed, which, omega=None):
    g = _gen(seed, which)
    parent, phys, _, T = _tensors(c, g, "state")
    _, _, _, W = _tensors(c, g, "op")
    wide = DT[WIDE[c["dtype"]]][0]
    T, W = [t.to(wide) for t in T], [t.to(wide) for t in W]
    n, ch = len(parent), _children(parent)

    def around(j, skip, down, subs):
        """T, W and the environments of node j but that of its leg `skip`."""
        x, lx = T[j], [("a", j), "s", *(("a", i) for i in ch[j])]
        w, lw = W[j], [("b", j), "o", "s", *(("b", i) for i in ch[j])]
        envs = ([(down[j], [("x", j), ("b", j), ("a", j)])] if skip != j else []) + [
            (subs[i], [("x", i), ("b", i), ("a", i)]) for i in ch[j] if i != skip]
        if envs:
            x, lx = _contract(x, lx, *envs[0])
        x, lx = _contract(x, lx, w, lw)
        for e in envs[1:]:
            x, lx = _contract(x, lx, *e)
        rows = ["o"] + [e[1][0] for e in envs]
        x = _order(x, lx, rows + [("b", skip), ("a", skip)])
        return x.reshape(math.prod(x.shape[:-2]), -1), x.shape[:-2], x.shape[-2:]

    one = torch.ones((1, 1, 1), dtype=wide, device="cuda")
    subs, down = [None] * n, [None] * n
    down[0] = one
    if any(len(x) > 1 for x in ch):
        for j in range(n - 1, 0, -1):
            m, _, ba = around(j, j, down, subs)
            f = _truncate(m, c["cap"], c["tol"])
            subs[j] = f.reshape(-1, *ba)
    for j in range(n):
        for i in ch[j]:
            m, rs, ba = around(j, i, down, subs)
            if omega is not None:
                x = m.reshape(rs[0], rs[1], -1)  # (out, sketch row, (b a))
                om = torch.from_numpy(omega[j]).cuda().to(wide)
                if rs[1] == 1:
                    x = x.expand(rs[0], c["cap"], x.shape[2])
                f = torch.einsum("ojq,oj->jq", x, om)
                f = f / torch.linalg.vector_norm(f)
            else:
                f = _truncate(m, c["cap"], c["tol"])
            down[i] = f.reshape(-1, *ba)
    R, out, log, span = [None] * n, [None] * n, 0.0, 1
    for j in range(n - 1, -1, -1):
        z, rs, ba = around(j, j, down, R)
        S = down[j].reshape(down[j].shape[0], -1) @ z.T
        if j == 0:
            nrm = torch.linalg.vector_norm(S)
            out[0], log = S / nrm, log + float(torch.log(nrm))
            break
        if omega is not None:
            S = S[:max(1, min(S.shape[0], math.prod(phys[:j]), z.shape[1]))]
        if S.shape[0] < S.shape[1]:
            q, r = torch.linalg.qr((S / torch.linalg.vector_norm(S, dim=1)[:, None]).mH)
            q = (q * torch.sgn(torch.diagonal(r))).mH
        else:
            q = torch.eye(S.shape[1], dtype=wide, device="cuda")
        r = q.conj() @ z
        nrm = torch.linalg.vector_norm(r)
        log += float(torch.log(nrm))
        R[j] = (r / nrm).reshape(-1, *ba)
        out[j] = q.reshape(-1, *rs)
    bond = [1] + [x.shape[0] for x in out[1:]]
    # the legs of a node: its parent's, its site's, its children's in their order
    flat = torch.cat([x.reshape(-1) for x in out])[None].contiguous()
    return _fix_network(flat, parent, phys, bond), log


def exact(case, seed):
    c = case
    if c["kind"] == "gemm":
        s = prepare(case, seed)
        A, B = (x.mT if t else x for x, t in ((s["A"], c["ta"]), (s["B"], c["tb"])))
        return (A.conj() if c["ca"] else A) @ (B.conj() if c["cb"] else B)
    if c["kind"] == "heev":
        lam, U = [], []
        for g in _gram(c, seed):
            w, v = torch.linalg.eigh(g)
            lam.append(w.flip(0))
            U.append(v.flip(1)[:, :c["kmax"]])
        lam = torch.stack(lam)
        k = c["kmax"]
        return {"lam": lam[:, :k], "lam_rest": lam[:, k:],
                "U": _fix_vectors(torch.stack(U).contiguous())}
    if c["kind"] == "cholqr":
        S = _rows(c, seed)
        q, r = torch.linalg.qr(S.mH)
        return (q * torch.sgn(torch.diagonal(r, dim1=-2, dim2=-1))[:, None, :]).mH.resolve_conj().contiguous()
    if c["kind"] == "group" and c["count"] * c["L"] * c["cap"] > 250_000:
        return None  # too many eigenproblems for a few seconds
    parts = _parts(c) * (c["count"] if c["kind"] == "group" else 1)
    if sum(p["L"] * min(p["chi"], p["cap"]) ** 2 for p in parts) > 8_000_000:
        return None
    omega = _sketch(c, seed) if c["kind"] == "src" else None
    got = [_exact_network(p, seed, j, omega) for j, p in enumerate(parts)]
    nodes = [x for x, _ in got]
    if c["kind"] == "group":
        nodes = [torch.cat(nodes)]
    return {"nodes": nodes, "bonds": None, "log_norm": np.array([x for _, x in got])}
