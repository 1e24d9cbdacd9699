"""The Ozaki form's row-factored units keep row sums in a scratch of their own: it is part of the
workspace that "wave_mb" limits."""
import numpy as np
import pytest

import oracle
import workloads

pytestmark = pytest.mark.gpu


def test_the_row_scratch_counts_against_the_wave_budget():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2211_16278_gb300 as bb
    mom = [(0, 0, 0), (1, 0, 0), (0, 1, 0), (0, 0, 1), (1, 1, 0)]
    inp = workloads.custom(4, 8, (8, 8, 8), 1, mom, [(0, 1, 0), (1, 0, 0)], [1.0, -1.0], seed=9700)
    V = torch.from_numpy(inp.V).cuda()[0]
    phis = [torch.from_numpy(inp.phi[0][i]).cuda()[0] for i in range(3)]
    outs = [torch.empty((len(mom), 8, 8, 8), dtype=torch.complex128, device="cuda") for _ in range(60)]
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    scratch = sms * 48 * 128 * 16            # row sums of 48 columns by 128 rows a CTA
    limit = -(-scratch // (1 << 20)) + 6     # MiB: a few jobs beside it
    ctx = bb.bblock_create(4, 8, 8, "ozaki")
    bb.bblock_set_option(ctx, "tc_rows", 1)
    bb.bblock_set_option(ctx, "wave_mb", limit)
    bb.bblock_compute_batch(ctx, [(V, *phis, o) for o in outs], inp.momenta, inp.spins, inp.coeffs)
    bb.bblock_status(ctx)
    other = 1 << 18                          # phases, momenta and call tables
    assert scratch < bb.bblock_workspace_bytes(ctx) <= (limit << 20) + other
    assert bb.bblock_last_wave_count(ctx) > 1
    ref = oracle.bblock(4, inp.V[0], *[inp.phi[0][i][0] for i in range(3)], inp.momenta, inp.spins, inp.coeffs)
    for o in outs:
        assert np.linalg.norm(o.cpu().numpy() - ref) <= 1e-12 * np.linalg.norm(ref)
    bb.bblock_destroy(ctx)
