"""What a user of this library has it do, as measurable cases.

A program that measures hadron correlators with stochastic LapH holds, on the GPU, the
orthonormal Laplacian eigenvectors V of one or more time slices, the coefficients phi of its
quark lines (one set per noise triple), a momentum list and a spin operator. It calls the
library once per time slice, or once for a batch of time slices and noise triples, and takes
the blocks B[p][d1][d2][d3]. ``listed`` holds those calls over the library's entry points,
arithmetic forms and sizes; ``draw`` gives further calls of the same ranges.

Sizes: the workloads of ``workloads.py`` (whole or with fewer time slices), the benchmark's
secondary measurements (the problem-size sweep, the mode triplet at L = 24) and the tests.
Values: V orthonormalised complex Gaussian, phi complex Gaussian, real spin coefficients.
"""
import math

import torch

import paper_2211_16278_gb300 as bb

# Momentum sets in units of 2 pi / L, |n|^2 <= 2, and spin operators (triples, coefficients).
_M9 = "0,0,0 1,0,0 -1,0,0 0,1,0 0,-1,0 0,0,1 0,0,-1 1,1,0 -1,-1,0"
_M7 = "0,0,0 1,0,0 -1,0,0 0,1,0 0,-1,0 0,0,1 0,0,-1"
_M5 = "0,0,0 1,0,0 0,1,0 0,0,1 1,1,0"
_M3 = "0,0,0 1,0,0 1,1,0"
_S1 = "0,0,0"
_S3 = "0,1,0 1,0,0 2,3,2"
_S4 = "0,1,0 1,0,0 2,3,2 3,2,2"


def _case(name, kind, form, L, n_ev, nd, n_t, momenta, spins, coeffs, **more):
    """nd: dilution sizes of the three lines of each noise triple, "a,b,c a,b,c ...". """
    return dict({"name": name, "kind": kind, "form": form, "products": 6, "L": L, "n_ev": n_ev,
                 "nd": nd, "n_t": n_t, "momenta": momenta, "spins": spins, "coeffs": coeffs}, **more)


def _cube(*sizes):
    return " ".join("%d,%d,%d" % (d, d, d) for d in sizes)


def listed():
    r2 = "0.7071067811865476 -0.7071067811865476 0.7071067811865476"
    h = "0.5 -0.5 0.5 -0.5"
    return [
        # the smallest call: one time slice of a 4^3 lattice, zero momentum, one spin triple
        _case("l4_fp64", "compute", "fp64", 4, 8, _cube(8), 1, "0,0,0", _S1, "1.0"),
        # the default form on an ordinary lattice: two time slices, three momenta
        _case("l24_fp64", "compute", "fp64", 24, 96, _cube(32), 2, _M3, _S3, r2),
        # the default form with a full momentum set, one time slice at a time (the size sweep)
        _case("l32_fp64", "compute", "fp64", 32, 96, _cube(32), 1, _M9, _S4, h),
        # a batch of uneven, odd dilution sizes (other sizes for each line and noise triple) in
        # double-float arithmetic, on a lattice that fills no tile
        _case("l19_ragged_df64", "batch", "df64", 19, 61, "33,17,29 21,40,13 27,27,31", 2, _M9, _S4, h),
        # the benchmark's workload, one time slice of it: six noise triples of N_dil 32, 48 and 64
        # sharing V, nine momenta, mixed precision; repeated on a stream of its own, as the
        # benchmark and a production loop call it (the library then replays a CUDA graph)
        _case("l32_batch_fp16x3", "batch", "fp16x3", 32, 128, _cube(64, 48, 32, 64, 48, 32), 1, _M9,
              _S4, h, stream=True),
        # the largest lattice, one time slice, mixed precision
        _case("l48_fp16x3", "compute", "fp16x3", 48, 264, _cube(64), 1, _M7, _S4, h),
        # eigenvectors and coefficients read from disk into pinned host memory, blocks written
        # back to it: eight time slices of the L = 24 workload
        _case("l24_host_fp16x3", "host", "fp16x3", 24, 96, _cube(32), 8, _M3, _S3, r2),
        # the BF16 split (six products) on the precision workload, one time slice
        _case("l32_bf16x6", "compute", "bf16", 32, 128, _cube(64), 1, _M5, _S4, h),
        # FP64-accurate blocks on the tensor cores, a batch of two noise triples
        _case("l32_batch_ozaki", "batch", "ozaki", 32, 128, _cube(48, 32), 1, _M9, _S4, h),
        # the mode triplet of one time slice, set up once for many noise and spin combinations ...
        _case("l24_mode_triplet", "triplet", "fp64", 24, 96, _cube(96), 1, _M3, _S1, "1.0"),
        # ... and the blocks of one noise triple taken from it
        _case("l24_from_triplet", "from_triplet", "fp64", 24, 96, _cube(32), 1, _M3, _S3, r2),
        # blocks from reconstructed fields, for a program whose memory manager owns the device
        _case("l16_noalloc", "noalloc", "fp64", 16, 1, _cube(32), 1, _M5, _S4, h),
    ]


# ---------------------------------------------------------------- reading a case

def _triples(text):
    return [tuple(int(v) for v in t.split(",")) for t in text.split()]


def _coeffs(case):
    return [float(v) for v in case["coeffs"].split()]


def _terms(case):
    """{gamma: {(alpha, beta): coefficient}} of the spin operator."""
    got = {}
    for (a, b, g), c in zip(_triples(case["spins"]), _coeffs(case)):
        got.setdefault(g, {})
        got[g][a, b] = got[g].get((a, b), 0.0) + c
    return got


def work(case):
    """Bytes: V of every time slice, phi of every noise triple and the blocks, once each.
    Flops (complex multiply-add = 8): the reconstruction of each line's spins (Eq. 2), the
    diquarks of the operator's (alpha, beta) pairs, one colour singlet per distinct gamma of the
    third quark, and the momentum sum with the phase factorised along one lattice axis."""
    L, n_ev, n_t, kind = case["L"], case["n_ev"], case["n_t"], case["kind"]
    X, mom, spins, by_gamma = L ** 3, _triples(case["momenta"]), _triples(case["spins"]), _terms(case)
    P, n0 = len(mom), len({n[0] % L for n in mom})
    al, be, ga = ({s[i] for s in spins} for i in range(3))
    pairs = {s[:2] for s in spins}
    nbytes = 0.0 if kind in ("from_triplet", "noalloc") else 16.0 * n_t * n_ev * 3 * X
    flops = 0.0
    for nd in _triples(case["nd"]):
        d1, d2, d3 = nd
        contract = 42.0 * len(pairs) * d1 * d2 * X
        contract += (24.0 * len(by_gamma) + 8.0 * (n0 + P / L)) * d1 * d2 * d3 * X
        if kind == "triplet":       # antisymmetric in its three indices
            flops += n_t * contract / 6
            nbytes += 16.0 * n_t * P * d1 * d2 * d3
            continue
        nbytes += 16.0 * n_t * P * d1 * d2 * d3
        if kind == "from_triplet":
            nbytes += 16.0 * n_t * (P * n_ev ** 3 + 4 * n_ev * sum(nd))
            flops += n_t * 8.0 * P * (len(ga) * n_ev * n_ev * n_ev * d3 +
                                      len({s[1:] for s in spins}) * n_ev * n_ev * d2 * d3 +
                                      len(al) * n_ev * d1 * d2 * d3)
        elif kind == "noalloc":
            nbytes += 16.0 * 3 * X * (len(al) * d1 + len(be) * d2 + len(ga) * d3)
            flops += contract
        else:
            nbytes += 16.0 * n_t * 4 * n_ev * sum(nd)
            flops += n_t * (8.0 * 3 * X * n_ev * (len(al) * d1 + len(be) * d2 + len(ga) * d3) + contract)
    return {"bytes": nbytes, "flops": flops}


# ---------------------------------------------------------------- drawn cases

# paper-ordering flop rates (TFLOP/s) that keep a drawn case below the largest listed one
_RATE = {"fp64": 0.7, "df64": 2.0, "ozaki": 3.0, "tf32x3": 10.0, "bf16": 15.0, "fp16x3": 40.0}
_MOMENTA = [(a, b, c) for a in (-1, 0, 1) for b in (-1, 0, 1) for c in (-1, 0, 1)
            if a * a + b * b + c * c <= 2]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _paper_flops(case):
    X, P, n_t = case["L"] ** 3, len(_triples(case["momenta"])), case["n_t"]
    pairs = len({s[:2] for s in _triples(case["spins"])})
    return n_t * sum((24.0 * pairs + 8.0 * P) * a * b * c * X + 50.0 * pairs * a * b * X +
                     24.0 * X * case["n_ev"] * 4 * (a + b + c) for a, b, c in _triples(case["nd"]))


def draw(rng):
    while True:
        kind = rng.choice(["compute"] * 5 + ["batch"] * 4 + ["host", "triplet", "from_triplet", "noalloc"])
        form = rng.choice(["fp64", "fp64", "fp16x3", "fp16x3", "ozaki", "df64", "bf16", "tf32x3"])
        if kind in ("from_triplet", "noalloc"):
            form = "fp64"
        if kind == "triplet":
            form = rng.choice(["fp64", "df64"])
        L = _log_int(rng, 4, 48 if kind in ("compute", "batch", "host") else 24)
        n_ev = _log_int(rng, 8, min(264, 3 * L ** 3))
        if kind in ("triplet", "from_triplet"):
            n_ev = _log_int(rng, 8, 96)
        n_noise = rng.randint(2, 4) if kind == "batch" else 1
        nd = []
        for _ in range(n_noise):
            d = _log_int(rng, 8, 64)
            nd.append((d, d, d) if rng.random() < 0.5 else
                      tuple(max(1, min(64, d + rng.randint(-d // 3, d // 3))) for _ in range(3)))
        if kind == "triplet":
            nd = [(n_ev,) * 3]
        n_mom = rng.choice([1, 2, 3, 5, 7, 8, 9])
        if kind == "noalloc":
            n_mom = min(n_mom, 8)
        mom = _triples(rng.choice([_M3, _M5, _M7])) if rng.random() < 0.4 else rng.sample(_MOMENTA, n_mom)
        if rng.random() < 0.5:
            spins = rng.choice([_S1, _S3, _S4])
        else:
            spins = " ".join("%d,%d,%d" % s for s in rng.sample(
                [(a, b, g) for a in range(4) for b in range(4) for g in range(4)], rng.randint(1, 4)))
        if kind == "triplet":
            spins = _S1
        n = len(spins.split())
        coeffs = " ".join(repr(rng.choice([1, -1]) / math.sqrt(n)) for _ in range(n))
        if kind == "triplet":
            coeffs = "1.0"
        case = _case("", kind, form, L, n_ev, " ".join("%d,%d,%d" % t for t in nd),
                     1 if kind in ("triplet", "noalloc") else rng.choice([1, 1, 2, 4, 8]),
                     " ".join("%d,%d,%d" % t for t in mom), spins, coeffs)
        del case["name"]
        if form == "bf16":
            case["products"] = rng.choice([3, 6, 9])
        if kind in ("compute", "batch") and rng.random() < 0.3:
            case["stream"] = True
        if kind == "noalloc" and len(mom) * nd[0][0] * nd[0][1] * nd[0][2] * 16 > 32 << 20:
            continue
        if _paper_flops(case) < 0.25 * _RATE[form] * 1e12 and 24.0 * 8 * L ** 3 * sum(
                t[0] * t[1] * t[2] for t in nd) * case["n_t"] < 2.4e13:
            return case


# ---------------------------------------------------------------- inputs

def _gauss(gen, *shape):
    s = math.sqrt(0.5)
    return torch.complex(torch.randn(*shape, generator=gen, dtype=torch.float64, device="cuda") * s,
                         torch.randn(*shape, generator=gen, dtype=torch.float64, device="cuda") * s)


def _eigenvectors(gen, L, n_ev):
    """n_ev orthonormal vectors of length 3 L^3 (Cholesky QR of a complex Gaussian), V[l][x][a]."""
    g = _gauss(gen, 3 * L ** 3, n_ev)
    if n_ev * 2 > g.shape[0]:
        q = torch.linalg.qr(g)[0]
    else:
        q = torch.linalg.solve_triangular(torch.linalg.cholesky(g.mH @ g).mH, g, upper=True, left=False)
    return q.T.reshape(n_ev, L ** 3, 3).contiguous()


def _inputs(case, seed):
    """Every tensor of a case on the GPU: V [n_t], phi [noise][line][n_t], or fields, or T."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    L, n_ev, n_t, kind = case["L"], case["n_ev"], case["n_t"], case["kind"]
    got = {}
    if kind == "noalloc":
        # fields of unit-normalised eigenvectors: entries of size sqrt(n_ev / 3 L^3), n_ev = 96
        got["q"] = [_gauss(gen, 4, L ** 3, 3, d) * math.sqrt(96 / (3 * L ** 3)) for d in _triples(case["nd"])[0]]
        return got
    if kind == "from_triplet":
        P = len(_triples(case["momenta"]))
        t = _gauss(gen, n_t, P, n_ev, n_ev, n_ev)
        t = t - t.transpose(-1, -2)
        t = t + t.movedim(-1, -3) + t.movedim(-3, -1)      # antisymmetric in l1, l2, l3
        got["T"] = (t / math.sqrt(6 * 3 * L ** 3)).contiguous()
    else:
        got["V"] = torch.stack([_eigenvectors(gen, L, n_ev) for _ in range(n_t)])
    if kind != "triplet":
        got["phi"] = [[_gauss(gen, n_t, 4 * n_ev, d) for d in nd] for nd in _triples(case["nd"])]
    return got


def prepare(case, seed):
    s = _inputs(case, seed)
    nds, mom = _triples(case["nd"]), _triples(case["momenta"])
    n_t, P, kind = case["n_t"], len(mom), case["kind"]
    s.update(kind=kind, L=case["L"], mom=mom, spins=_triples(case["spins"]), coeffs=_coeffs(case),
             stream=torch.cuda.Stream() if case.get("stream") else None)
    if kind != "noalloc":
        s["ctx"] = bb.bblock_create(case["L"], case["n_ev"], max(max(t) for t in nds), case["form"],
                                    bf16_products=case["products"])
    lead = () if kind == "noalloc" else (n_t,)
    s["B"] = [torch.empty(lead + (P,) + nd, dtype=torch.complex128, device="cuda") for nd in nds]
    if kind == "host":
        def pinned(t):
            h = torch.empty(t.shape, dtype=t.dtype, pin_memory=True)
            h.copy_(t)
            return h
        s["V"], s["phi"] = pinned(s["V"]), [[pinned(p) for p in line] for line in s["phi"]]
        s["B"] = [pinned(b.zero_()) for b in s["B"]]
    if kind == "batch":
        s["jobs"] = [(s["V"][t], *(p[t] for p in s["phi"][k]), s["B"][k][t])
                     for t in range(n_t) for k in range(len(nds))]
    return s


def run(s):
    if s["stream"] is not None:
        now = torch.cuda.current_stream()
        s["stream"].wait_stream(now)
        with torch.cuda.stream(s["stream"]):
            _call(s)
        now.wait_stream(s["stream"])
    else:
        _call(s)
    return s["B"]


def _call(s):
    op = (s["mom"], s["spins"], s["coeffs"])
    if s["kind"] == "compute":
        bb.bblock_compute(s["ctx"], s["V"], *s["phi"][0], *op, B_out=s["B"][0])
    elif s["kind"] == "batch":
        bb.bblock_compute_batch(s["ctx"], s["jobs"], *op)
    elif s["kind"] == "host":
        bb.bblock_compute_host(s["ctx"], s["V"], *s["phi"][0], *op, s["B"][0])
    elif s["kind"] == "triplet":
        bb.bblock_mode_triplet(s["ctx"], s["V"], s["mom"], T_out=s["B"][0])
    elif s["kind"] == "from_triplet":
        bb.bblock_from_triplet(s["ctx"], s["T"], *s["phi"][0], s["spins"], s["coeffs"], B_out=s["B"][0])
    else:
        bb.bblock_contract_noalloc(s["L"], *s["q"], *op, s["B"][0])


# ---------------------------------------------------------------- in 64 bits

def _exact_contract(L, q1, q2, q3, mom, by_gamma):
    """Eq. 1 of fields q[spin][x][c][d] (dicts by spin): B[p][d1][d2][d3], lattice rows at a time."""
    d1, d2, d3 = (next(iter(q.values())).shape[-1] for q in (q1, q2, q3))
    dev, X = next(iter(q1.values())).device, L ** 3
    n0s = sorted({n[0] % L for n in mom})
    w = torch.exp(-2j * math.pi * torch.arange(L, dtype=torch.float64, device=dev) / L)
    at = torch.arange(L, device=dev)
    B = torch.zeros(len(mom), d1 * d2, d3, dtype=torch.complex128, device=dev)
    for r in range(L * L):
        sl = slice(r * L, (r + 1) * L)
        a, b = [], []
        for g, pairs in by_gamma.items():
            A = 0
            for (al, be), c in pairs.items():
                u, v = q1[al][sl], q2[be][sl] * c
                A = A + torch.linalg.cross(u[:, :, :, None].expand(-1, -1, -1, d2),
                                           v[:, :, None, :].expand(-1, -1, d1, -1), dim=1)
            a.append(A.reshape(3 * L, d1 * d2))
            b.append(torch.stack([w[(n * at) % L][:, None, None] * q3[g][sl] for n in n0s], 2).reshape(3 * L, -1))
        T = (torch.cat(a).T @ torch.cat(b)).reshape(d1 * d2, len(n0s), d3)
        for p, n in enumerate(mom):
            B[p] += w[(n[1] * (r % L) + n[2] * (r // L)) % L] * T[:, n0s.index(n[0] % L)]
    return B.reshape(len(mom), d1, d2, d3)


def exact(case, seed):
    s = _inputs(case, seed)
    L, n_ev, n_t, mom = case["L"], case["n_ev"], case["n_t"], _triples(case["momenta"])
    spins, by_gamma, nds = _triples(case["spins"]), _terms(case), _triples(case["nd"])
    used = [sorted({t[i] for t in spins}) for i in range(3)]
    if case["kind"] == "noalloc":
        q = [{a: f[a] for a in u} for f, u in zip(s["q"], used)]
        return [_exact_contract(L, *q, mom, by_gamma)]
    if case["kind"] == "from_triplet":
        B = torch.zeros(n_t, len(mom), *nds[0], dtype=torch.complex128, device="cuda")
        phi = [p.reshape(n_t, 4, n_ev, -1) for p in s["phi"][0]]
        for g, pairs in by_gamma.items():
            U = s["T"] @ phi[2][:, g][:, None, None]
            for (al, be), c in pairs.items():
                B += c * torch.einsum("tad,tpaef->tpdef", phi[0][:, al],
                                      torch.einsum("tbe,tpabf->tpaef", phi[1][:, be], U))
        return [B]
    out = []
    for k, nd in enumerate(nds):
        B = torch.empty(n_t, len(mom), *nd, dtype=torch.complex128, device="cuda")
        for t in range(n_t):
            V = s["V"][t].reshape(n_ev, 3 * L ** 3)
            if case["kind"] == "triplet":
                q = [{0: V.T.reshape(L ** 3, 3, n_ev).contiguous()}] * 3
            else:
                q = [{a: (V.T @ s["phi"][k][i][t, a * n_ev:(a + 1) * n_ev]).reshape(L ** 3, 3, nd[i])
                      for a in used[i]} for i in range(3)]
            B[t] = _exact_contract(L, *q, mom, by_gamma)
        out.append(B)
    return out
