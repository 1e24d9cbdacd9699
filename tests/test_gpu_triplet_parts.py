"""Blocks from the mode triplet: the real and the imaginary part are each accurate to their own size.

T and the coefficients are positive and nearly real (imaginary parts 1e-8 of the real ones), so
no sum cancels and every product of a four-multiplication complex sum keeps 52 bits in both
parts: three products in a row of N_ev terms, the folds and the sum over spin terms round at most
8 N_ev + 64 times a part, each by 1.2e-16 of that part. Forms that share a product between the two
parts leave the imaginary one accurate to the modulus only, 1e-8 of what is asked here.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

OPERATORS = [([(0, 1, 0)], [1.0]),
             ([(0, 1, 0), (1, 0, 0), (2, 3, 2), (3, 2, 2)], [0.5, 0.25, 0.5, 1.0]),
             ([(0, 0, 1), (0, 1, 1), (0, 2, 1), (1, 0, 1)], [1.0, 0.5, 0.25, 2.0])]


@pytest.mark.parametrize("op", range(len(OPERATORS)))
@pytest.mark.parametrize("n_ev,nd", [(1, (1, 1, 1)), (17, (5, 33, 9)), (33, (9, 4, 31))])
def test_each_part_of_a_block(op, n_ev, nd):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2211_16278_gb300 as bb
    rng = np.random.default_rng(8900 + n_ev)
    spins, coeffs = OPERATORS[op]

    def positive(*shape):
        return rng.uniform(0.5, 1.5, shape) + 1e-8j * rng.uniform(0.5, 1.5, shape)

    T = positive(1, 2, n_ev, n_ev, n_ev)
    phi = [positive(1, 4 * n_ev, d) for d in nd]
    ctx = bb.bblock_create(4, n_ev, max(*nd, n_ev), "fp64")
    got = bb.bblock_from_triplet(ctx, torch.from_numpy(T).cuda(), *[torch.from_numpy(p).cuda() for p in phi],
                                 spins, coeffs).cpu().numpy()[0]
    bb.bblock_destroy(ctx)
    wide = [p[0].astype(np.clongdouble).reshape(4, n_ev, -1) for p in phi]
    Tw = T[0].astype(np.clongdouble)
    ref = 0
    for (a, b, g), c in zip(spins, coeffs):
        u = np.einsum("pabc,cf->pabf", Tw, wide[2][g])
        u = np.einsum("pabf,be->paef", u, wide[1][b])
        ref = ref + c * np.einsum("paef,ad->pdef", u, wide[0][a])
    tol = (8 * n_ev + 64) * 1.2e-16
    for part in ("real", "imag"):
        r = getattr(ref, part)
        assert (np.abs(getattr(got, part) - r) <= tol * np.abs(r)).all(), part
