"""Mode triplets repeated on a stream of their own: plain launches, capture, graph replays, with
several waves, vectors rewritten in place between the calls, and a NaN that comes and goes (the
per-vector flags are cleared by every replay)."""
import numpy as np
import pytest

import oracle
import workloads

pytestmark = pytest.mark.gpu

TOL = 1e-12   # the FP64-accurate forms' parity target
MOM = [(0, 0, 0), (1, 0, 0), (-1, 2, 0)]


@pytest.mark.parametrize("form", ["fp64", "df64"])
def test_replays_read_the_vectors_of_their_call(form):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2211_16278_gb300 as bb
    L, n_ev, n_t = 3, 19, 4
    sets = [workloads.custom(L, n_ev, (1, 1, 1), n_t, MOM, [(0, 0, 0)], [1.0], seed=9900 + k).V for k in range(3)]
    dirty = sets[1].copy()
    dirty[2, 5, 7, 1] = np.nan
    calls = [sets[0], sets[1], dirty, sets[1], sets[2], dirty, sets[0]]
    V = torch.from_numpy(sets[0].copy()).cuda()
    T = torch.empty((n_t, len(MOM), n_ev, n_ev, n_ev), dtype=torch.complex128, device="cuda")
    ctx = bb.bblock_create(L, n_ev, n_ev, form)
    bb.bblock_set_option(ctx, "wave_mb", 8)
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    for k, v in enumerate(calls):
        with torch.cuda.stream(stream):
            V.copy_(torch.from_numpy(v).pin_memory(), non_blocking=True)
            T.fill_(complex(1.0, 2.0))
            bb.bblock_mode_triplet(ctx, V, MOM, T_out=T)
        bb.bblock_status(ctx)
        assert bb.bblock_last_wave_count(ctx) > 1
        got = T.cpu().numpy()
        for t in range(n_t):
            bad = np.zeros((n_ev,) * 3, bool)
            if v is dirty and t == 2:
                bad[5], bad[:, 5], bad[:, :, 5] = True, True, True
            assert (np.isfinite(got[t]) == ~bad).all(), (k, t)
            ref = oracle.mode_triplet(L, np.nan_to_num(v[t]), MOM)
            assert np.linalg.norm((got[t] - ref)[:, ~bad]) <= TOL * np.linalg.norm(ref), (k, t)
    bb.bblock_destroy(ctx)
