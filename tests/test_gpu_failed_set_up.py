"""A call that fails after its phase table was allocated leaves no unfilled table behind.

The failure is a host-side one: the call comes on a stream that is being captured (relaxed
mode, so the allocation goes through), where waiting for the table is refused. The next call on
the context must fill the table and match the oracle.
"""
import ctypes

import numpy as np
import pytest

import oracle
import workloads

pytestmark = pytest.mark.gpu

FEW = [(0, 0, 0), (1, 0, 0)]
MORE = [(0, 0, 0), (0, 1, 0), (1, 1, 0), (-1, 0, 0), (0, 0, 1)]


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2211_16278_gb300 as bb
    bb.load()
    return torch, bb


@pytest.mark.parametrize("after_a_call", [False, True])
@pytest.mark.parametrize("form,tol", [("fp64", 1e-12), ("df64", 1e-12), ("ozaki", 1e-12), ("fp16x3", 1e-6)])
def test_the_table_is_filled_again(env, form, tol, after_a_call):
    torch, bb = env
    dev = torch.device("cuda:0")
    inp = workloads.custom(7, 12, (9, 8, 10), 1, FEW, [(0, 1, 0), (1, 0, 2)], [1.0, 0.5], seed=8800)
    V = torch.from_numpy(inp.V).to(dev)
    phis = [torch.from_numpy(inp.phi[0][i]).to(dev) for i in range(3)]
    ctx = bb.bblock_create(7, 12, 10, form)
    out = {n: torch.empty((1, n, 9, 8, 10), dtype=torch.complex128, device=dev) for n in (len(FEW), len(MORE))}

    def call(mom):
        return bb.bblock_compute(ctx, V, *phis, mom, inp.spins, inp.coeffs, B_out=out[len(mom)])

    if after_a_call:
        call(FEW)
    torch.cuda.synchronize()
    rt = ctypes.CDLL("libcudart.so.13")
    stream = torch.cuda.Stream()
    handle = ctypes.c_void_p(stream.cuda_stream)
    with torch.cuda.stream(stream):
        assert rt.cudaStreamBeginCapture(handle, 2) == 0   # cudaStreamCaptureModeRelaxed
        try:
            if after_a_call and form in ("fp64", "df64"):
                refused = False   # one w^k table serves every momentum list: nothing to fill
            else:
                refused = True
                with pytest.raises(bb.BblockError):
                    call(MORE)
        finally:
            graph = ctypes.c_void_p()
            ended = rt.cudaStreamEndCapture(handle, ctypes.byref(graph))
            rt.cudaGetLastError()
    assert (ended != 0) == refused
    for mom in (FEW, MORE):
        got = call(mom)
        bb.bblock_status(ctx)
        ref = oracle.bblock(7, inp.V[0], *[inp.phi[0][i][0] for i in range(3)], np.array(mom, np.int32),
                            inp.spins, inp.coeffs)
        assert np.linalg.norm(got.cpu().numpy()[0] - ref) <= tol * np.linalg.norm(ref)
    bb.bblock_destroy(ctx)
