"""bblock_last_launch_count and the step times count every kernel of a call, the copy of each wave's
job table among them, and from one entry point as from another."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("on_stream", [False, True])
def test_every_kernel_is_counted(on_stream):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2211_16278_gb300 as bb
    inp = workloads.custom(4, 6, (8, 8, 8), 1, [(0, 0, 0), (1, 0, 0)], [(0, 1, 0)], [1.0], seed=9800)
    V = torch.from_numpy(inp.V).cuda()[0]
    phis = [torch.from_numpy(inp.phi[0][i]).cuda()[0] for i in range(3)]
    outs = [torch.empty((2, 8, 8, 8), dtype=torch.complex128, device="cuda") for _ in range(5)]
    jobs = [(V, *phis, o) for o in outs]
    ctx = bb.bblock_create(4, 6, 8, "fp64")
    bb.bblock_set_option(ctx, "wave_mb", 2)
    stream = torch.cuda.Stream() if on_stream else None   # plain launches, capture, replay
    bb.bblock_profile_enable(ctx)
    for call in range(4):
        bb.bblock_compute_batch(ctx, jobs, inp.momenta, inp.spins, inp.coeffs, stream=stream)
        bb.bblock_status(ctx)
        waves = bb.bblock_last_wave_count(ctx)
        steps = bb.bblock_profile_read(ctx)
        assert waves > 1 and steps["tables"][0] == waves
        # table copy, projection, contraction and slab sum of each wave, and w^k once
        assert bb.bblock_last_launch_count(ctx) == 4 * waves + (1 if call == 0 else 0)
        assert sum(n for n, _ in steps.values()) == bb.bblock_last_launch_count(ctx)
    bb.bblock_destroy(ctx)
