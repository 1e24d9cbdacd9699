"""Spin sums grouped by third-quark field and momenta summed along lattice rows.

The FP64-accurate forms sum Eq. 1 over groups of spin terms that share a third-quark field
(one group per (alpha, beta) pair, or one per gamma), and take the phase as
e^{-i p.x} = w^{n0 x0} w^{n1 x1 + n2 x2} along the axis with the fewest classes of +-n0. These
cases sit where the grouping, the axis, the classes (none, one to three per launch, more than
three, more than 32 momenta) and the tiles (one column to several ragged tiles) change.
"""
import numpy as np
import pytest

import oracle
import workloads

pytestmark = pytest.mark.gpu

TOL = 1e-12   # the FP64-accurate forms' parity target against the oracle

ALL27 = [(a, b, c) for a in (-1, 0, 1) for b in (-1, 0, 1) for c in (-1, 0, 1)]
CASES = {
    # pairs (a, b), (b, a) on one gamma: grouped by gamma; two terms a group
    "gamma": (5, 12, (6, 7, 17), [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (1, 1, 1)],
              [(0, 1, 0), (1, 0, 0), (2, 3, 2), (3, 2, 2)], [0.5, -0.5, 0.25j, 1.0]),
    # several betas folded into one line-2 field, a triple given twice
    "fold": (3, 9, (5, 4, 33), [(0, 0, 0), (0, 0, 1)],
             [(0, 0, 1), (0, 1, 1), (0, 2, 1), (0, 3, 1), (1, 3, 1), (0, 1, 1)],
             [1.0, 0.5j, -0.25, 2.0, 0.125, 0.5]),
    # more gammas than pairs: grouped by pair
    "pair": (4, 10, (3, 6, 16), [(1, 0, 2), (2, 0, 0), (-2, 1, 0)],
             [(0, 1, 0), (0, 1, 1), (0, 1, 2), (0, 1, 3)], [1.0, 0.5, -0.5j, 0.25]),
    # no class along the last axis
    "flat": (6, 8, (9, 4, 64), [(0, 0, 0), (1, 0, 0), (1, 1, 0), (5, 2, 0)],
             [(2, 1, 3), (1, 2, 3)], [1.0, -1.0]),
    # one site, one column
    "single": (1, 3, (1, 1, 1), [(0, 0, 0), (3, -1, 7)], [(0, 0, 0), (1, 1, 0)], [1.0, 1.0j]),
    # two and three classes, with L / 2 and momenta beyond L
    "two": (6, 8, (7, 5, 40), [(1, 1, 1), (2, 2, 2), (-1, 2, 1), (8, 1, 2)], [(0, 1, 2)], [1.0]),
    "three": (6, 8, (5, 7, 31), [(1, 2, 3), (2, 3, 1), (3, 1, 2), (-2, -1, -3), (0, 0, 0)],
              [(0, 1, 2), (1, 0, 2)], [1.0, 0.5]),
    # five classes on every axis: two launches
    "five": (11, 6, (4, 5, 18), [(k, (2 * k) % 11, (3 * k) % 11) for k in range(1, 11)],
             [(0, 1, 2), (1, 0, 2)], [1.0, 0.5]),
    # more momenta than one launch takes, two d3 tiles, a second one of one column
    "many": (4, 8, (3, 3, 65), ALL27 + [(2, 0, 0), (2, 1, 0), (0, 2, 1), (2, 2, 2), (1, 2, 0), (3, 0, 2),
                                        (0, 3, 2)], [(0, 0, 0), (0, 1, 0), (1, 0, 0)], [1.0, -1.0, 2.0]),
}


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2211_16278_gb300 as bb
    bb.load()
    return torch, bb


def rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


@pytest.mark.parametrize("slabs", [0, 1])
@pytest.mark.parametrize("name", CASES)
@pytest.mark.parametrize("form,options", [
    ("fp64", {}), ("df64", {}), ("ozaki", {"tc_rows": 2}), ("ozaki", {"tc_rows": 1}),
    ("ozaki", {"tc_rows": 1, "tc_cluster": 1, "tc_nc": 32}), ("ozaki", {"tc_rows": 1, "tc_cluster": 3}),
    ("ozaki", {"tc_rows": 1, "tc_cluster": 4, "tc_nc": 16})], ids=str)
def test_matches_oracle(env, form, options, name, slabs):
    torch, bb = env
    L, n_ev, nd, mom, spins, coeffs = CASES[name]
    inp = workloads.custom(L, n_ev, nd, 2, mom, spins, coeffs, seed=9000 + len(name))
    dev = torch.device("cuda:0")
    ctx = bb.bblock_create(L, n_ev, max(nd), form)
    bb.bblock_set_option(ctx, "slabs", slabs)
    for k, v in options.items():
        bb.bblock_set_option(ctx, k, v)
    B = bb.bblock_compute(ctx, torch.from_numpy(inp.V).to(dev),
                          *[torch.from_numpy(inp.phi[0][i]).to(dev) for i in range(3)],
                          inp.momenta, inp.spins, inp.coeffs)
    bb.bblock_status(ctx)
    for t in range(2):
        ref = oracle.bblock(L, inp.V[t], *[inp.phi[0][i][t] for i in range(3)], inp.momenta,
                            inp.spins, inp.coeffs)
        for p in range(len(mom)):
            assert rel(B[t, p].cpu().numpy(), ref[p]) <= TOL, (t, p)
    bb.bblock_destroy(ctx)


@pytest.mark.parametrize("name", [n for n in CASES if len(CASES[n][3]) <= 8])
def test_noalloc_matches_oracle(env, name):
    torch, bb = env
    L, n_ev, nd, mom, spins, coeffs = CASES[name]
    inp = workloads.custom(L, n_ev, nd, 1, mom, spins, coeffs, seed=9100 + len(name))
    dev = torch.device("cuda:0")
    phis = [inp.phi[0][i][0] for i in range(3)]
    used = [{s[i] for s in spins} for i in range(3)]
    # spins the operator does not name are not read
    qs = []
    for p, u in zip(phis, used):
        q = np.full((4, L ** 3, 3, p.shape[1]), np.nan, np.complex128)
        for a in u:
            q[a] = oracle.reconstruct(inp.V[0], p, a)
        qs.append(torch.from_numpy(q).to(dev))
    B = torch.full((len(mom), *nd), complex(np.nan, np.nan), dtype=torch.complex128, device=dev)
    bb.bblock_contract_noalloc(L, *qs, inp.momenta, inp.spins, inp.coeffs, B)
    torch.cuda.synchronize()
    ref = oracle.bblock(L, inp.V[0], *phis, inp.momenta, inp.spins, inp.coeffs)
    for p in range(len(mom)):
        assert rel(B[p].cpu().numpy(), ref[p]) <= TOL, p
