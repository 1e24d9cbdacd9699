"""Blocks from the mode triplet: the intermediates of as many spin terms at a time as fit, and
shorter runs of terms where the device cannot hold them; the same blocks either way."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def case():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2211_16278_gb300 as bb
    rng = np.random.default_rng(9600)
    n_ev, nd, P = 64, (20, 24, 32), 4

    def gauss(*shape):
        return torch.from_numpy(rng.standard_normal(shape) + 1j * rng.standard_normal(shape)).cuda()

    T, phi = gauss(1, P, n_ev, n_ev, n_ev), [gauss(1, 4 * n_ev, d) for d in nd]
    spins = [(a, b, g) for a in range(4) for b in range(4) for g in range(4)]
    coeffs = rng.standard_normal(64)
    u1 = 16 * P * n_ev * n_ev * nd[2]        # T x3 phi3 of one group, the largest intermediate

    def run(ctx):
        return bb.bblock_from_triplet(ctx, T, *phi, spins, coeffs).cpu().numpy()

    def create():
        return bb.bblock_create(4, n_ev, n_ev, "fp64")

    ctx = create()
    ref = run(ctx)
    held = bb.bblock_workspace_bytes(ctx)
    bb.bblock_destroy(ctx)
    assert held > 4 * u1                     # 16 terms in 4 groups at once, and counted
    return bb, create, run, ref, u1, held


def test_a_failed_allocation_takes_shorter_runs(case):
    bb, create, run, ref, u1, held = case
    ctx = create()
    bb.bblock_set_option(ctx, "fail_next_alloc", 1)
    got = run(ctx)
    assert bb.bblock_get_option(ctx, "fail_next_alloc") == 0
    assert bb.bblock_last_error(ctx) == ""
    assert bb.bblock_workspace_bytes(ctx) < held
    bb.bblock_destroy(ctx)
    assert np.linalg.norm(got - ref) <= 1e-13 * np.linalg.norm(ref)


def test_the_workspace_limit_holds(case):
    bb, create, run, ref, u1, held = case
    limit = (2 * u1) >> 20                   # MiB: less than two groups take
    ctx = create()
    bb.bblock_set_option(ctx, "wave_mb", limit)
    got = run(ctx)
    assert bb.bblock_workspace_bytes(ctx) <= (limit << 20) + 4096
    bb.bblock_destroy(ctx)
    assert np.linalg.norm(got - ref) <= 1e-13 * np.linalg.norm(ref)
