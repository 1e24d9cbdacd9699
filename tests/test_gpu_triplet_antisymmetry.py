"""The FP64 and double-float mode triplets are summed for l1 < l2 < l3 only and completed by
antisymmetry: every element against the oracle's Eq. (4) at eigenvector counts around the 16-
and 64-column tiles, several time slices and waves, and where a vector holds an infinity or a NaN.
"""
import numpy as np
import pytest

import oracle
import workloads

pytestmark = pytest.mark.gpu

TOL = 1e-12
MOM = [(0, 0, 0), (1, 0, 0), (-1, 2, 0), (1, 1, 1)]


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2211_16278_gb300 as bb
    bb.load()
    return torch, bb


@pytest.mark.parametrize("form", ["fp64", "df64"])
@pytest.mark.parametrize("L,n_ev", [(1, 1), (1, 2), (1, 3), (3, 16), (3, 17), (4, 33), (3, 65)])
def test_every_element(env, form, L, n_ev):
    torch, bb = env
    inp = workloads.custom(L, n_ev, (1, 1, 1), 3, MOM, [(0, 0, 0)], [1.0], seed=6400 + n_ev)
    V = torch.from_numpy(inp.V).to("cuda:0")
    ctx = bb.bblock_create(L, n_ev, n_ev, form)
    bb.bblock_set_option(ctx, "wave_mb", 1)
    T = bb.bblock_mode_triplet(ctx, V, MOM)
    bb.bblock_status(ctx)
    got = T.cpu().numpy()
    for t in range(3):
        ref = oracle.mode_triplet(L, inp.V[t], MOM)
        assert np.linalg.norm(got[t] - ref) <= TOL * max(np.linalg.norm(ref), np.linalg.norm(inp.V[t]) ** 3)
        for axes in ((0, 2, 1, 3), (0, 1, 3, 2), (0, 3, 2, 1)):
            assert np.array_equal(got[t], -got[t].transpose(axes))
    bb.bblock_destroy(ctx)


@pytest.mark.parametrize("form", ["fp64", "df64"])
def test_non_finite_vectors(env, form):
    """An element is finite exactly where none of its three vectors holds an infinity or a NaN
    (the general contraction, whose projection multiplies every vector by the identity
    coefficients, is not finite there either)."""
    torch, bb = env
    L, n_ev = 2, 7
    inp = workloads.custom(L, n_ev, (1, 1, 1), 1, MOM, [(0, 0, 0)], [1.0], seed=6500)
    clean = inp.V[0].copy()
    inp.V[0, 2, 3, 1] = np.nan
    inp.V[0, 5, 0, 0] = np.inf
    V = torch.from_numpy(inp.V).to("cuda:0")
    got = []
    for checks in (0, 1):
        ctx = bb.bblock_create(L, n_ev, n_ev, form)
        bb.bblock_set_option(ctx, "checks", checks)
        got.append(bb.bblock_mode_triplet(ctx, V, MOM).cpu().numpy()[0])
        bb.bblock_destroy(ctx)
    bad = np.zeros((n_ev,) * 3, bool)
    for ax in range(3):
        for l in (2, 5):
            bad.swapaxes(0, ax)[l] = True
    assert (np.isfinite(got[0]) == ~bad).all()
    assert not np.isfinite(got[1][:, bad]).any()
    ref = oracle.mode_triplet(L, clean, MOM)
    assert np.linalg.norm((got[0] - ref)[:, ~bad]) <= TOL * np.linalg.norm(ref)


def test_blocks_from_the_triplet_in_chunks_of_terms(env):
    """All 64 spin triples (16 terms in 4 groups) at a size whose intermediates exceed the
    chunk of terms taken at a time, and an operator grouped by gamma with several betas folded
    into one term; blocks of the direct contraction as the reference."""
    torch, bb = env
    L, n_ev, nd = 4, 128, (64, 60, 64)
    mom = [(a, b, c) for a in (0, 1, -1) for b in (0, 1, -1) for c in (0,)]
    rng = np.random.default_rng(6600)
    every = [(a, b, g) for a in range(4) for b in range(4) for g in range(4)]
    dev = torch.device("cuda:0")
    inp = workloads.custom(L, n_ev, nd, 1, mom, [(0, 0, 0)], [1.0], seed=6601)
    V = torch.from_numpy(inp.V).to(dev)
    phis = [torch.from_numpy(inp.phi[0][i]).to(dev) for i in range(3)]
    ctx = bb.bblock_create(L, n_ev, n_ev, "fp64")
    T = bb.bblock_mode_triplet(ctx, V, mom)
    for spins in (every, [(0, 0, 1), (0, 1, 1), (0, 2, 1), (1, 0, 1), (2, 3, 1)]):
        coeffs = rng.standard_normal(len(spins)) + 1j * rng.standard_normal(len(spins))
        via = bb.bblock_from_triplet(ctx, T, *phis, spins, coeffs)
        direct = bb.bblock_compute(ctx, V, *phis, mom, spins, coeffs)
        bb.bblock_status(ctx)
        err = (torch.linalg.norm(via - direct) / torch.linalg.norm(direct)).item()
        assert err <= TOL
    bb.bblock_destroy(ctx)
