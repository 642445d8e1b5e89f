"""Performance cases: what users of this package have it do, over the sizes it takes.

A case is a dict of plain values.  Its ``kind`` says which public entry points it goes through:

``step``     one time step of a circuit on a state of bond dimension ``chi``: a gate layer on the even bonds,
             then one on the odd bonds (each followed by ``g`` PtSU steps), through ``State.apply_layer``;
``circuit``  a whole brickwork circuit of ``depth`` layers from |0...0>, while the bond dimensions grow and the
             small Schmidt values have to be resolved, then one two-site observable in the middle of the chain;
``routed``   a 2D circuit (``lx`` x ``ly``) compiled onto the line: many sparse layers through ``apply_bonds``;
``batch``    several circuits of different lengths, depths and bond dimensions served together (``Batch``);
``svd``      ``svd_batched`` on matrices a caller holds;
``measure``  norm, overlap, one- and two-site expectation values of given states (the FP64 contractions);
``sample``   bit strings drawn from a given state.

Outputs are what the method fixes uniquely (Sec. II B of arXiv:2312.02667): the Schmidt values of every bond, bond
dimensions, discarded weights and nu factors, observables.  The Gamma tensors are fixed only up to a phase
per Schmidt vector; the Schmidt values after a further layer depend on them.  Values of a mixed-precision state
(complex64 tensors) are returned as float32, the type its arithmetic carries.
"""
import math

import numpy as np
import torch

from paper_2312_02667_gb300 import circuits2d, inputs, ptebd

CUTOFF = 1e-12


def listed():
    return [
        # the smallest calls: a few qubits, where launches and latency are all there is
        {"name": "step_n16_chi16", "kind": "step", "n": 16, "chi": 16, "prec": "mixed", "g": 1},
        # an ordinary circuit simulation step (the 128-qubit, chi 64 configuration)
        {"name": "step_n128_chi64", "kind": "step", "n": 128, "chi": 64, "prec": "mixed", "g": 1},
        # odd sizes: an odd number of sites, a bond dimension that fills no tile, no regauging
        {"name": "step_n75_chi100", "kind": "step", "n": 75, "chi": 100, "prec": "mixed", "g": 0},
        # the largest: the 1024-qubit, chi 256 configuration with regauging after every layer
        {"name": "step_n1024_chi256", "kind": "step", "n": 1024, "chi": 256, "prec": "mixed", "g": 1},
        # the complex128 path (the 128-qubit, chi 64 configuration in FP64)
        {"name": "step_n128_chi64_fp64", "kind": "step", "n": 128, "chi": 64, "prec": "fp64", "g": 1},
        # a circuit from the product state: growing bonds, resolved in FP64 where complex64 cannot decide
        {"name": "circuit_n50_chi64", "kind": "circuit", "n": 50, "chi": 64, "depth": 12, "prec": "mixed", "g": 0},
        # a routed 2D circuit: tens of sparse layers of a few bonds each
        {"name": "routed_8x8_chi32", "kind": "routed", "lx": 8, "ly": 8, "chi": 32, "depth": 4, "prec": "mixed"},
        # uneven circuits served together, one graph launch per layer
        {"name": "batch_6_circuits", "kind": "batch", "circuits": 6, "n_max": 100, "chi": 64, "depth_max": 10},
        # SVDs alone: the size of the largest layer, and small tall complex128 ones with their vectors
        {"name": "svd_c64_256x512x512", "kind": "svd", "batch": 256, "rows": 512, "cols": 512, "prec": "mixed",
         "spectrum": "graded", "vectors": False},
        {"name": "svd_c128_40x90x70", "kind": "svd", "batch": 40, "rows": 90, "cols": 70, "prec": "fp64",
         "spectrum": "ginibre", "vectors": True},
        # measurements on a finished state
        {"name": "measure_n128_chi64", "kind": "measure", "n": 128, "chi": 64, "prec": "mixed"},
        {"name": "sample_n64_chi32", "kind": "sample", "n": 64, "chi": 32, "samples": 500, "prec": "mixed"},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "step", "circuit", "routed", "batch", "svd", "svd", "measure", "sample"])
    prec = rng.choice(["mixed", "mixed", "mixed", "fp64"])
    if kind == "step":
        if prec == "fp64":
            n, chi = _log(rng, 8, 200), _log(rng, 8, 72)
        else:
            chi = _log(rng, 8, 256)
            n = _log(rng, 8, 1000 if chi <= 128 else 400)
        return {"kind": kind, "n": n, "chi": chi, "prec": prec, "g": rng.choice([0, 1, 1])}
    if kind == "circuit":
        return {"kind": kind, "n": rng.randint(20, 80), "chi": _log(rng, 12, 72), "depth": rng.randint(9, 13),
                "prec": prec, "g": rng.choice([0, 0, 1])}
    if kind == "routed":
        return {"kind": kind, "lx": rng.randint(4, 9), "ly": rng.randint(4, 9), "chi": _log(rng, 8, 32), "depth": 4,
                "prec": prec}
    if kind == "batch":
        return {"kind": kind, "circuits": rng.randint(2, 8), "n_max": rng.randint(40, 140), "chi": _log(rng, 16, 64),
                "depth_max": rng.randint(9, 11)}
    if kind == "svd":
        rows = 2 * _log(rng, 4, 256 if prec == "mixed" else 64)
        cols = rng.randint(max(1, rows // 4), rows)
        most = int(min(2000.0, 200 * (512.0 / rows) ** 3)) if prec == "mixed" else int(min(500.0, 100 * (128.0 / rows) ** 3))
        vectors = cols <= 0.8 * rows
        return {"kind": kind, "batch": rng.randint(max(1, most // 8), most), "rows": rows, "cols": cols, "prec": prec,
                "spectrum": "ginibre" if vectors else rng.choice(["ginibre", "graded"]), "vectors": vectors}
    if kind == "measure":
        return {"kind": kind, "n": rng.randint(8, 200), "chi": _log(rng, 8, 100), "prec": prec}
    return {"kind": kind, "n": rng.randint(16, 100), "chi": _log(rng, 8, 64), "samples": _log(rng, 10, 1500), "prec": prec}


# ------------------------------------------------------------------ inputs --

def _dims(n, chi):
    """Bond dimensions chi_{-1} .. chi_{n-1} of a state saturated at chi."""
    return [1] + [min(chi, 2 ** min(b + 1, n - b - 1, 30)) for b in range(n - 1)] + [1]


def _mps(n, chi, prec, seed, canonical=False):
    """A saturated random MPS: Gaussian Gamma of about unit norm per column, descending normalised Lambda.  With
    `canonical`, isometries from the left (norm 1) and flat Lambda, a state whose observables are of order 1."""
    gen = torch.Generator(device="cuda").manual_seed(1_000_003 * (seed + 1) + 7919 * n + chi)
    rng = np.random.default_rng([seed, n, chi, 0x51A7])
    dims = _dims(n, chi)
    lam = []
    for b in range(n - 1):
        k = dims[b + 1]
        x = np.ones(k) if canonical else np.sort(np.abs(rng.standard_normal(k)) + 0.1)[::-1]
        lam.append(np.ascontiguousarray(x / np.linalg.norm(x)))
    gam = []
    for s in range(n):
        shape = (2, dims[s], dims[s + 1])
        z = torch.view_as_complex(torch.randn(shape + (2,), generator=gen, device="cuda", dtype=torch.float64))
        if canonical:  # Gamma Lambda_s left-orthonormal: sum over (x, alpha) of conj(M) M = 1
            a = z.reshape(2 * dims[s], dims[s + 1]).cpu()
            if 2 * dims[s] >= dims[s + 1]:
                a = torch.linalg.qr(a)[0]
            else:
                a = a / torch.linalg.norm(a)
            z = a.reshape(shape)
            if s < n - 1:
                z = z / torch.from_numpy(lam[s].copy())
            else:
                z = z / torch.linalg.norm(z)
        else:
            z = z / math.sqrt(2 * dims[s + 1])
            # towards the ends of the chain, where a site's two square sides meet, a unitary (as in a real state)
            if 2 * dims[s] == dims[s + 1]:
                z = torch.linalg.qr(z.reshape(2 * dims[s], -1).cpu())[0].reshape(shape)
            elif dims[s] == 2 * dims[s + 1]:
                q = torch.linalg.qr(z.permute(1, 0, 2).reshape(dims[s], -1).cpu())[0]
                z = q.reshape(dims[s], 2, dims[s + 1]).permute(1, 0, 2).contiguous()
        if prec == "mixed":
            z = z.to(torch.complex64)
        gam.append(z.to(torch.complex128).cpu().numpy())
    return gam, lam


def _gates(n, layer, seed):
    return inputs.brickwork_layer(seed, n, layer, 17)[2]


def _op2(seed):
    return inputs.haar_u4(np.random.default_rng([seed, 0x0B2]))


def _routed(case, seed):
    layers = circuits2d.compile_layers(case["lx"], case["ly"],
                                       circuits2d.physical_layers(seed, case["lx"], case["ly"], case["depth"]))
    return [([int(b) for b in bonds], np.asarray(us, dtype=np.complex128)) for bonds, us in layers]


def _batch(case, seed):
    """(n, chi, depth) of each circuit: the sizes go with the case, the gates with the seed."""
    rng = np.random.default_rng([case["circuits"], case["n_max"], case["chi"], case["depth_max"]])
    return [(int(rng.integers(case["n_max"] // 2, case["n_max"] + 1)), case["chi"] if i % 2 else case["chi"] // 2,
             int(rng.integers(case["depth_max"] - 2, case["depth_max"] + 1))) for i in range(case["circuits"])]


def _matrices(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(31 * seed + case["rows"])
    b, m, k = case["batch"], case["rows"], case["cols"]
    real, cplx = (torch.float32, torch.complex64) if case["prec"] == "mixed" else (torch.float64, torch.complex128)
    z = torch.view_as_complex(torch.randn((b, m, k, 2), generator=gen, device="cuda", dtype=real)) / math.sqrt(2 * m)
    if case["spectrum"] == "graded":  # a spectrum falling over three decades, as Schmidt values do
        s = torch.logspace(0, -3, k, device="cuda", dtype=real)
        w = torch.view_as_complex(torch.randn((b, k, k, 2), generator=gen, device="cuda", dtype=real)) / math.sqrt(2 * k)
        z = torch.matmul(z * s.to(cplx), w)
    return z.contiguous()


# --------------------------------------------------------- prepare and run --

def prepare(case, seed):
    kind = case["kind"]
    prec = case.get("prec", "mixed")
    if kind == "step":
        n, chi = case["n"], case["chi"]
        st = ptebd.State(n, chi, prec, cutoff=CUTOFF, g=case["g"])
        gam, lam = _mps(n, chi, prec, seed)
        st.load(gam, lam)
        gates = [torch.from_numpy(_gates(n, p, seed)).cuda() for p in (0, 1)]
        return {"case": case, "st": st, "gates": gates}
    if kind == "circuit":
        st = ptebd.State(case["n"], case["chi"], prec, cutoff=CUTOFF, g=case["g"])
        layers = [inputs.brickwork_layer(seed, case["n"], l, 23) for l in range(case["depth"])]
        return {"case": case, "st": st, "layers": layers, "op2": _op2(seed)}
    if kind == "routed":
        st = ptebd.State(case["lx"] * case["ly"], case["chi"], prec, cutoff=CUTOFF)
        return {"case": case, "st": st, "layers": _routed(case, seed)}
    if kind == "batch":
        sizes = _batch(case, seed)
        sts = [ptebd.State(n, chi, "mixed", cutoff=CUTOFF) for n, chi, _ in sizes]
        gates = [[inputs.brickwork_layer(seed, n, l, 100 + i)[2] for l in range(d)] for i, (n, _, d) in enumerate(sizes)]
        return {"case": case, "sts": sts, "batch": ptebd.Batch(sts), "gates": gates}
    if kind == "svd":
        return {"case": case, "a": _matrices(case, seed)}
    st = ptebd.State(case["n"], case["chi"], prec, cutoff=CUTOFF)
    gam, lam = _mps(case["n"], case["chi"], prec, seed, canonical=True)
    st.load(gam, lam)
    if kind == "measure":
        other = ptebd.State(case["n"], case["chi"], prec, cutoff=CUTOFF)
        g2 = [g.copy() for g in gam]  # the same state after one-site rotations on three sites
        for j, s in enumerate((0, case["n"] // 2, case["n"] - 1)):
            u = np.linalg.qr(np.random.default_rng([seed, j]).standard_normal((2, 2)) + 1j)[0]
            g2[s] = np.einsum("xy,yab->xab", u, g2[s])
            if prec == "mixed":
                g2[s] = g2[s].astype(np.complex64).astype(np.complex128)
        other.load(g2, lam)
        return {"case": case, "st": st, "other": other, "op1": inputs.random_one_site_op(seed), "op2": _op2(seed)}
    return {"case": case, "st": st, "u": np.random.default_rng([seed, 5]).random((case["samples"], case["n"]))}


def _real(prec):
    return np.float32 if prec == "mixed" else np.float64


def _schmidt(st, prec):
    """Schmidt values of every bond (zero-padded), bond dimensions, discarded weights, nu."""
    lam = np.zeros((st.n_sites - 1, st.chi_max), dtype=_real(prec))
    chi = np.zeros(st.n_sites - 1, dtype=np.int32)
    for b in range(st.n_sites - 1):
        v = st.lam(b)
        lam[b, : len(v)] = v
        chi[b] = len(v)
    eps, nu, _ = st.bond_stats()
    return {"lam": lam, "chi": chi, "eps": eps.astype(_real(prec)), "nu": nu.astype(_real(prec))}


def _pair(z, prec):
    return np.array([z.real, z.imag], dtype=_real(prec))


def run(state):
    case = state["case"]
    kind = case["kind"]
    prec = case.get("prec", "mixed")
    if kind == "step":
        st = state["st"]
        for p in (0, 1):
            st.apply_layer(state["gates"][p], p)
        return _schmidt(st, prec)
    if kind == "circuit":
        st = state["st"]
        st.reset()
        for parity, _, gates in state["layers"]:
            st.apply_layer(gates, parity)
        out = _schmidt(st, prec)
        out["expect2"] = _pair(st.expect2(case["n"] // 2 - 1, state["op2"]), prec)
        return out
    if kind == "routed":
        st = state["st"]
        st.reset()
        for bonds, us in state["layers"]:
            st.apply_bonds(bonds, us)
        return _schmidt(st, prec)
    if kind == "batch":
        for st in state["sts"]:
            st.reset()
        depth = max(len(g) for g in state["gates"])
        none = np.zeros((0, 4, 4), complex)
        for l in range(depth):
            state["batch"].apply_layer([g[l] if l < len(g) else none for g in state["gates"]],
                                       [l % 2 if l < len(g) else -1 for g in state["gates"]])
        return [_schmidt(st, prec) for st in state["sts"]]
    if kind == "svd":
        a = state["a"]
        sigma, u = ptebd.svd_batched(a, want_u=case["vectors"])
        out = {"sigma": sigma.to(torch.float32 if prec == "mixed" else torch.float64)}
        if case["vectors"]:  # the isometry nearest to each matrix: U S^-1 (U^H A)
            out["isometry"] = torch.matmul(u / sigma.unsqueeze(1).to(u.real.dtype), torch.matmul(u.mH, a))
        return out
    if kind == "measure":
        st, n = state["st"], case["n"]
        return {"norm": np.array([st.norm()], dtype=_real(prec)),
                "overlap": _pair(st.overlap(state["other"]), prec),
                "expect": _pair(st.expect(n // 3, state["op1"]), prec),
                "expect2": _pair(st.expect2(n // 2, state["op2"]), prec)}
    return {"bits": state["st"].sample(state["u"])}


# ------------------------------------------------------------------- work --

def _svd_flops(m, n):
    """Real flops of an economy SVD of a complex m x n matrix, m >= n (Golub and Van Loan's 14 m n^2 + 8 n^3, times
    four for complex arithmetic)."""
    m, n = max(m, n), min(m, n)
    return 4.0 * (14.0 * m * n * n + 8.0 * n ** 3)


def _bond_work(cl, cm, cr, k, elem, gated):
    """A two-site update: theta, its SVD (of rank cm for an ungated bond: QR factors and a cm x cm core), both Gamma."""
    if gated:
        f = 32.0 * cl * cm * cr + _svd_flops(2 * cl, 2 * cr) + 8.0 * k * 4 * cl * cr
    else:
        f = 2 * 16.0 * (cl + cr) * cm * cm + _svd_flops(cm, cm) + 2 * 16.0 * (cl + cr) * cm * cm
    return {"flops": f, "bytes": float(elem) * 2 * (cl * cm + cm * cr + cl * k + k * cr)}


def _layer_work(dims, bonds, chi, elem, gated, total, rank=4):
    for b in bonds:
        cl, cm, cr = dims[b], dims[b + 1], dims[b + 2]
        k = min(chi, 2 * cl, 2 * cr, rank * cm) if gated else min(cm, 2 * cl, 2 * cr)
        w = _bond_work(cl, cm, cr, k, elem, gated)
        total["flops"] += w["flops"]
        total["bytes"] += w["bytes"]
        dims[b + 1] = k


def _circuit_work(n, chi, depth, g, elem, total, dims=None):
    dims = dims or [1] * (n + 1)
    for l in range(depth):
        _layer_work(dims, range(l % 2, n - 1, 2), chi, elem, True, total)
        for step in range(g):
            for p in (0, 1):
                if not (step == 0 and p == 0 and l % 2 == 0):  # just done by the gated layer itself
                    _layer_work(dims, range(p, n - 1, 2), chi, elem, False, total)
    return dims


def _contract_work(dims, elem, total):
    for s in range(len(dims) - 1):
        a, b = dims[s], dims[s + 1]
        total["flops"] += 2 * 8.0 * (a * a * b + a * b * b)
        total["bytes"] += elem * 2.0 * a * b


def work(case):
    total = {"bytes": 0.0, "flops": 0.0}
    kind = case["kind"]
    elem = 16 if case.get("prec") == "fp64" else 8
    if kind == "step":
        _circuit_work(case["n"], case["chi"], 2, case["g"], elem, total, _dims(case["n"], case["chi"]))
    elif kind == "circuit":
        dims = _circuit_work(case["n"], case["chi"], case["depth"], case["g"], elem, total)
        for _ in range(2):
            _contract_work(dims, elem, total)
    elif kind == "routed":
        dims = [1] * (case["lx"] * case["ly"] + 1)
        for bonds, us in _routed(case, 0):
            for b, u in zip(bonds, us):
                r = np.linalg.matrix_rank(u.reshape(2, 2, 2, 2).transpose(0, 2, 1, 3).reshape(4, 4), tol=1e-9)
                _layer_work(dims, [b], case["chi"], elem, True, total, rank=int(r))
    elif kind == "batch":
        for n, chi, depth in _batch(case, 0):
            _circuit_work(n, chi, depth, 0, 8, total)
    elif kind == "svd":
        b, m, n = case["batch"], case["rows"], case["cols"]
        total["flops"] = b * _svd_flops(m, n) * (1.0 if case["vectors"] else 0.4)
        total["bytes"] = float(b) * (elem * m * n * (2 if case["vectors"] else 1) + 8 * n)
    else:
        dims = _dims(case["n"], case["chi"])
        if kind == "measure":
            for _ in range(6):  # the norm, the overlap, and a numerator and a denominator of each expectation value
                _contract_work(dims, elem, total)
        else:
            _contract_work(dims, elem, total)
            for a, b in zip(dims[:-1], dims[1:]):
                total["flops"] += 8.0 * case["samples"] * (2 * a * b + 2 * a * a)
            total["bytes"] += case["samples"] * case["n"] * 12.0
    return total


# ------------------------------------------------------------------ exact --
# The method in complex128 numpy (Sec. II C, III B-D of arXiv:2312.02667), Schmidt reading of eps.

def _np_bond(gam, lam, b, gate, chi, stats):
    one = np.ones(1)
    n = len(gam)
    ll = lam[b - 1] if b > 0 else one
    lr = lam[b + 1] if b + 1 < n - 1 else one
    cl, cr = len(ll), len(lr)
    x = ll[None, :, None] * gam[b] * lam[b][None, None, :]
    y = gam[b + 1] * lr[None, None, :]
    th = np.einsum("sab,tbc->satc", x, y, optimize=True)
    if gate is not None:
        th = np.einsum("xyst,satc->xayc", gate.reshape(2, 2, 2, 2), th, optimize=True)
    u, s, vh = np.linalg.svd(th.reshape(2 * cl, 2 * cr), full_matrices=False)
    k = max(1, min(chi, int(np.sum(s > CUTOFF * s[0]))))
    scale = 1.0
    if gate is not None:
        tot = float(np.sum(s * s))
        eps = float(np.sum(s[k:] ** 2)) / tot
        nu = 1.0 / math.sqrt(1.0 - eps)
        scale = nu / math.sqrt(tot)
        stats[0][b], stats[1][b] = eps, nu
    gam[b] = u[:, :k].reshape(2, cl, k) / ll[None, :, None]
    gam[b + 1] = np.ascontiguousarray(vh[:k].reshape(k, 2, cr).transpose(1, 0, 2)) / lr[None, None, :]
    lam[b] = scale * s[:k]


def _np_layer(gam, lam, bonds, gates, chi, g, stats):
    for b, u in zip(bonds, gates):
        _np_bond(gam, lam, int(b), u, chi, stats)
    for _ in range(g):
        for p in (0, 1):
            for b in range(p, len(gam) - 1, 2):
                _np_bond(gam, lam, b, None, chi, stats)


def _np_zero(n):
    z = np.zeros((2, 1, 1), complex)
    z[0, 0, 0] = 1.0
    return [z.copy() for _ in range(n)], [np.ones(1) for _ in range(n - 1)]


def _np_out(lam, stats, chi_max):
    out = np.zeros((len(lam), chi_max))
    for b, v in enumerate(lam):
        out[b, : len(v)] = v
    return {"lam": out, "chi": np.array([len(v) for v in lam], dtype=np.int32), "eps": stats[0], "nu": stats[1]}


def _np_contract(ga, la, gb, lb, site=-1, op=None):
    """<a| op |b>, op on one site (2x2) or on (site, site + 1) (4x4)."""
    n = len(ga)
    ma = [g * (la[s] if s < n - 1 else np.ones(1))[None, None, :] for s, g in enumerate(ga)]
    mb = [g * (lb[s] if s < n - 1 else np.ones(1))[None, None, :] for s, g in enumerate(gb)]
    e = np.ones((1, 1), complex)
    s = 0
    while s < n:
        if s == site and op.shape == (4, 4):
            t = np.einsum("yab,zbc->yzac", mb[s], mb[s + 1], optimize=True)
            t = np.einsum("wxyz,yzac->wxac", op.reshape(2, 2, 2, 2), t, optimize=True)
            q = np.einsum("yab,zbc->yzac", ma[s], ma[s + 1], optimize=True)
            e = np.einsum("yzap,ab,yzbq->pq", q.conj(), e, t, optimize=True)
            s += 2
            continue
        t = np.einsum("xy,yab->xab", op, mb[s]) if s == site else mb[s]
        e = np.einsum("xap,ab,xbq->pq", ma[s].conj(), e, t, optimize=True)
        s += 1
    return complex(e[0, 0])


def _np_cost(case):
    """Seconds of exact(), roughly."""
    kind = case["kind"]
    if kind in ("step", "circuit"):
        per = 2 if kind == "step" else case["depth"]
        return 3e-8 * per * case["n"] * (0.5 + 1.0 * case["g"]) * (2 * case["chi"]) ** 3 / 3.0
    if kind == "routed":
        return 3e-8 * 60 * case["lx"] * case["ly"] * 0.3 * (2 * case["chi"]) ** 3 / 3.0
    if kind == "batch":
        return 3e-8 * case["circuits"] * case["n_max"] * 0.5 * case["depth_max"] * (2 * case["chi"]) ** 3 / 3.0
    if kind == "svd":
        return 3e-8 * case["batch"] * case["rows"] * case["cols"] ** 2
    return 3e-9 * 40 * case["n"] * case["chi"] ** 3


def exact(case, seed):
    if _np_cost(case) > 15.0:
        return None
    kind = case["kind"]
    prec = case.get("prec", "mixed")
    if kind == "step":
        n, chi = case["n"], case["chi"]
        gam, lam = _mps(n, chi, prec, seed)
        stats = (np.zeros(n - 1), np.ones(n - 1))
        for p in (0, 1):
            _np_layer(gam, lam, range(p, n - 1, 2), _gates(n, p, seed), chi, case["g"], stats)
        return _np_out(lam, stats, chi)
    if kind == "circuit":
        n, chi = case["n"], case["chi"]
        gam, lam = _np_zero(n)
        stats = (np.zeros(n - 1), np.ones(n - 1))
        for l in range(case["depth"]):
            _, bonds, gates = inputs.brickwork_layer(seed, n, l, 23)
            _np_layer(gam, lam, bonds, gates, chi, case["g"], stats)
        out = _np_out(lam, stats, chi)
        e = _np_contract(gam, lam, gam, lam, n // 2 - 1, _op2(seed)) / _np_contract(gam, lam, gam, lam).real
        out["expect2"] = np.array([e.real, e.imag])
        return out
    if kind == "routed":
        n = case["lx"] * case["ly"]
        gam, lam = _np_zero(n)
        stats = (np.zeros(n - 1), np.ones(n - 1))
        for bonds, us in _routed(case, seed):
            _np_layer(gam, lam, bonds, us, case["chi"], 0, stats)
        return _np_out(lam, stats, case["chi"])
    if kind == "batch":
        outs = []
        for i, (n, chi, depth) in enumerate(_batch(case, seed)):
            gam, lam = _np_zero(n)
            stats = (np.zeros(n - 1), np.ones(n - 1))
            for l in range(depth):
                _, bonds, gates = inputs.brickwork_layer(seed, n, l, 100 + i)
                _np_layer(gam, lam, bonds, gates, chi, 0, stats)
            outs.append(_np_out(lam, stats, chi))
        return outs
    if kind == "svd":
        a = _matrices(case, seed).to(torch.complex128).cpu().numpy()
        u, s, vh = np.linalg.svd(a, full_matrices=False)
        out = {"sigma": s}
        if case["vectors"]:
            out["isometry"] = np.matmul(u, vh)
        return out
    if kind == "sample":
        return None  # bits: whole numbers, compared as they are
    state_g, lam = _mps(case["n"], case["chi"], prec, seed, canonical=True)
    g2 = [g.copy() for g in state_g]
    for j, s in enumerate((0, case["n"] // 2, case["n"] - 1)):
        u = np.linalg.qr(np.random.default_rng([seed, j]).standard_normal((2, 2)) + 1j)[0]
        g2[s] = np.einsum("xy,yab->xab", u, g2[s])
        if prec == "mixed":
            g2[s] = g2[s].astype(np.complex64).astype(np.complex128)
    n2 = _np_contract(state_g, lam, state_g, lam).real
    ov = _np_contract(state_g, lam, g2, lam)
    e1 = _np_contract(state_g, lam, state_g, lam, case["n"] // 3, inputs.random_one_site_op(seed)) / n2
    e2 = _np_contract(state_g, lam, state_g, lam, case["n"] // 2, _op2(seed)) / n2
    return {"norm": np.array([math.sqrt(n2)]), "overlap": np.array([ov.real, ov.imag]),
            "expect": np.array([e1.real, e1.imag]), "expect2": np.array([e2.real, e2.imag])}
