"""Momentum lists whose momenta hardly share a component along any axis.

A row-factored launch takes at most three classes of +-n0, and every launch repeats the colour
singlet and the diquarks: such lists run with a phase per momentum and site instead, up to ten
momenta a launch in FP64 (eight in double-float). Blocks against the oracle where the momentum
count crosses a launch's tiles (4, 5, 8, 9, 10, 11), at ragged sizes, with slabs that end inside
a staged chunk, and the number of launches. A call's blocks are compared as a whole: the momenta's
sums have the same terms, with phases of modulus one, so they share one error scale.
"""
import numpy as np
import pytest

import oracle
import workloads

pytestmark = pytest.mark.gpu

TOL = 1e-12   # the FP64-accurate forms' parity target against the oracle
SPINS = {"one": ([(0, 1, 2)], [1.0]), "three": ([(0, 1, 0), (1, 0, 0), (2, 3, 2)], [0.7, -0.7, 0.5j])}


def diagonal(n):
    """n momenta with n different components along every axis (L > 2 n)."""
    return [(k, 2 * k, -k) for k in range(n)]


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2211_16278_gb300 as bb
    bb.load()
    return torch, bb


@pytest.mark.parametrize("form,per_launch", [("fp64", 10), ("df64", 8)])
@pytest.mark.parametrize("op", SPINS)
@pytest.mark.parametrize("n_mom,nd,slabs", [(5, (3, 4, 5), 0), (8, (7, 5, 17), 0), (9, (4, 9, 33), 3), (10, (1, 1, 1), 1),
                                            (11, (5, 3, 64), 0), (17, (2, 3, 16), 0)])
def test_matches_oracle(env, form, per_launch, op, n_mom, nd, slabs):
    torch, bb = env
    L, n_ev, n_t = 23 if n_mom == 11 else 35 if n_mom == 17 else 21, 4, 1
    if n_mom <= 8:
        L, n_t = 17, 2
    spins, coeffs = SPINS[op]
    inp = workloads.custom(L, n_ev, nd, n_t, diagonal(n_mom), spins, coeffs, seed=9200 + n_mom)
    dev = torch.device("cuda:0")
    ctx = bb.bblock_create(L, n_ev, max(nd), form)
    bb.bblock_set_option(ctx, "slabs", slabs)
    bb.bblock_profile_enable(ctx)
    B = bb.bblock_compute(ctx, torch.from_numpy(inp.V).to(dev),
                          *[torch.from_numpy(inp.phi[0][i]).to(dev) for i in range(3)],
                          inp.momenta, inp.spins, inp.coeffs)
    bb.bblock_status(ctx)
    assert bb.bblock_profile_read(ctx)["contract"][0] == -(-n_mom // per_launch)
    for t in range(n_t):
        ref = oracle.bblock(L, inp.V[t], *[inp.phi[0][i][t] for i in range(3)], inp.momenta,
                            inp.spins, inp.coeffs)
        assert np.linalg.norm(B[t].cpu().numpy() - ref) <= TOL * np.linalg.norm(ref), t
    bb.bblock_destroy(ctx)


@pytest.mark.parametrize("form", ["fp64", "df64"])
@pytest.mark.parametrize("L,n_mom", [(2, 3), (3, 4), (4, 7), (5, 5)])
def test_small_lattices(env, form, L, n_mom):
    """Momenta beyond L, more of them than the lattice has distinct ones along an axis."""
    torch, bb = env
    n_ev, nd = 3, (9, 7, 37)
    mom = [(3 * k + 1, -k, 2 * k) for k in range(n_mom)]
    inp = workloads.custom(L, n_ev, nd, 2, mom, *SPINS["three"], seed=9300 + L)
    dev = torch.device("cuda:0")
    ctx = bb.bblock_create(L, n_ev, max(nd), form)
    B = bb.bblock_compute(ctx, torch.from_numpy(inp.V).to(dev),
                          *[torch.from_numpy(inp.phi[0][i]).to(dev) for i in range(3)],
                          inp.momenta, inp.spins, inp.coeffs)
    bb.bblock_status(ctx)
    for t in range(2):
        ref = oracle.bblock(L, inp.V[t], *[inp.phi[0][i][t] for i in range(3)], inp.momenta,
                            inp.spins, inp.coeffs)
        assert np.linalg.norm(B[t].cpu().numpy() - ref) <= TOL * np.linalg.norm(ref)
    bb.bblock_destroy(ctx)


@pytest.mark.parametrize("L,n_mom,nd", [(11, 5, (3, 4, 5)), (17, 8, (6, 7, 33)), (9, 4, (8, 8, 16)), (4, 8, (5, 6, 40))])
def test_noalloc_matches_oracle(env, L, n_mom, nd):
    torch, bb = env
    n_ev = 3
    spins, coeffs = SPINS["three"]
    inp = workloads.custom(L, n_ev, nd, 1, diagonal(n_mom), spins, coeffs, seed=9400 + n_mom)
    dev = torch.device("cuda:0")
    phis = [inp.phi[0][i][0] for i in range(3)]
    qs = [torch.from_numpy(np.stack([oracle.reconstruct(inp.V[0], p, a) for a in range(4)])).to(dev) for p in phis]
    B = torch.full((n_mom, *nd), complex(np.nan, np.nan), dtype=torch.complex128, device=dev)
    bb.bblock_contract_noalloc(L, *qs, inp.momenta, inp.spins, inp.coeffs, B)
    torch.cuda.synchronize()
    ref = oracle.bblock(L, inp.V[0], *phis, inp.momenta, inp.spins, inp.coeffs)
    assert np.linalg.norm(B.cpu().numpy() - ref) <= TOL * np.linalg.norm(ref)


@pytest.mark.parametrize("L", [16, 24])
def test_as_accurate_as_sums_by_row(env, L):
    """The double-float error of a list with a phase per site against that of as many momenta that are
    summed by rows (one component is 0 in all of them), each relative to its blocks. The FP64 form stands
    for the exact blocks: its error is a twentieth of either. Both errors are sums of the same roundings
    of the fields and of a like number of partial sums; they scatter by about 2 % over seeds."""
    torch, bb = env
    n_ev, n_mom, nd = 8, 8, (9, 8, 16)

    def error(momenta):
        inp = workloads.custom(L, n_ev, nd, 1, momenta, [(0, 1, 2)], [1.0], seed=9700 + L)
        args = [torch.from_numpy(x).to("cuda:0") for x in (inp.V, *inp.phi[0][:3])]
        blocks = {}
        for form in ("fp64", "df64"):
            ctx = bb.bblock_create(L, n_ev, max(nd), form)
            blocks[form] = bb.bblock_compute(ctx, *args, inp.momenta, inp.spins, inp.coeffs)
            bb.bblock_status(ctx)
            bb.bblock_destroy(ctx)
        return (torch.linalg.vector_norm(blocks["df64"] - blocks["fp64"]) / torch.linalg.vector_norm(blocks["fp64"])).item()

    assert error([(k, 2 * k, -k) for k in range(n_mom)]) <= 1.15 * error([(k, 2 * k, 0) for k in range(n_mom)])


@pytest.mark.parametrize("form", ["fp64", "df64"])
def test_mode_triplet(env, form):
    torch, bb = env
    L, n_ev = 13, 21
    mom = diagonal(6)
    inp = workloads.custom(L, n_ev, (1, 1, 1), 1, mom, [(0, 0, 0)], [1.0], seed=9500)
    ctx = bb.bblock_create(L, n_ev, n_ev, form)
    T = bb.bblock_mode_triplet(ctx, torch.from_numpy(inp.V).to("cuda:0"), mom).cpu().numpy()[0]
    bb.bblock_status(ctx)
    bb.bblock_destroy(ctx)
    ref = oracle.mode_triplet(L, inp.V[0], mom)
    assert np.linalg.norm(T - ref) <= TOL * np.linalg.norm(ref)


@pytest.mark.parametrize("form", ["fp64", "df64"])
@pytest.mark.parametrize("mom", [[(0, 0, 0), (1, 1, 1), (1, 0, 0)], [(2, 1, 1), (1, 1, 3), (-1, 1, 2)]])
@pytest.mark.parametrize("nd", [(3, 4, 16), (5, 6, 40)])
def test_a_coefficient_set_for_each_momentum(env, form, mom, nd):
    """A launch per momentum, all of one kind: some momenta alone would be row-factored, some not."""
    torch, bb = env
    L, n_ev = 9, 4
    spins, coeffs = SPINS["three"]
    per_mom = np.array([[c * (1 + p) for c in coeffs] for p in range(len(mom))], np.complex128)
    inp = workloads.custom(L, n_ev, nd, 2, mom, spins, coeffs, seed=9600)
    dev = torch.device("cuda:0")
    ctx = bb.bblock_create(L, n_ev, max(nd), form)
    B = bb.bblock_compute(ctx, torch.from_numpy(inp.V).to(dev),
                          *[torch.from_numpy(inp.phi[0][i]).to(dev) for i in range(3)],
                          inp.momenta, inp.spins, per_mom)
    bb.bblock_status(ctx)
    for t in range(2):
        for p in range(len(mom)):
            ref = oracle.bblock(L, inp.V[t], *[inp.phi[0][i][t] for i in range(3)], inp.momenta[p:p + 1],
                                inp.spins, per_mom[p])
            assert np.linalg.norm(B[t, p].cpu().numpy() - ref[0]) <= TOL * np.linalg.norm(ref), (t, p)
    bb.bblock_destroy(ctx)
