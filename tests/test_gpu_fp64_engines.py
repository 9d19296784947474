"""The FP64 contraction kernels against sums in extended precision, at the
edges of their tiles.  Error bound of a chain of K FMAs: K 2^-53 sum |a b|,
with a factor two for the roundings of alpha and beta."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2401_11935_gb300 as P
    from synth import make_system
    eng = P.Engine.from_system(make_system((2, 40, 12), seed=3))
    yield eng
    eng.close()


def _exact(a, b):
    return np.asarray(a, dtype=np.longdouble) @ np.asarray(b, dtype=np.longdouble).T


def _bound(a, b, alpha, c0, beta):
    ab = np.abs(a) @ np.abs(b).T
    return 2 * 2.0 ** -53 * (abs(alpha) * (a.shape[1] + 1) * ab + abs(beta) * np.abs(c0))


def _run(eng, engine, a, b, alpha, beta, c0, spec="mk,nk->mn"):
    import torch
    from paper_2401_11935_gb300 import _lib as L
    A, B = torch.tensor(a).cuda(), torch.tensor(b).cuda()
    C = torch.tensor(c0).cuda()
    torch.cuda.synchronize()
    L.dcsd_einsum_device(eng.ctx, engine, spec, alpha, A, B, beta, C)
    torch.cuda.synchronize()
    return C.cpu().numpy()


# edges of the 8 x 8 and 16 x 16 tiles and of their k-chunks, few tiles (K split), many tiles
SHAPES = [(1, 1, 1), (3, 5, 2), (16, 16, 16), (17, 15, 33), (64, 64, 64), (65, 63, 65), (127, 16, 128), (128, 17, 63),
          (129, 255, 100), (130, 257, 31), (12, 12, 5000), (40, 300, 1024), (257, 33, 1025), (300, 530, 200),
          (9, 7, 20000), (513, 4, 513)]


@pytest.mark.parametrize("M,N,K", SHAPES)
@pytest.mark.parametrize("engine", [0, 1])
def test_contraction_error_bound(ctx, M, N, K, engine):
    rng = np.random.default_rng(M * 7 + N * 3 + K)
    a, b = rng.normal(size=(M, K)), rng.normal(size=(N, K))
    a *= np.exp(rng.normal(size=(M, 1)) * 10)  # rows of very different size
    b[rng.random(b.shape) < 0.5] = 0.0
    for alpha, beta in ((1.0, 0.0), (-0.5, 1.0)):
        c0 = rng.normal(size=(M, N)) if beta else np.full((M, N), np.nan)
        ref = np.longdouble(alpha) * _exact(a, b) + (np.longdouble(beta) * c0 if beta else 0)
        err = np.abs(_run(ctx, engine, a, b, alpha, beta, c0) - ref)
        assert (err <= _bound(a, b, alpha, c0 if beta else np.zeros((M, N)), beta)).all()


@pytest.mark.parametrize("engine", [0, 1])
@pytest.mark.parametrize("spec,sa,sb,sc", [
    ("Lac,Lbd->acbd", (9, 5, 7), (9, 6, 8), (5, 7, 6, 8)), ("ikac,kcjb->iajb", (4, 5, 9, 7), (5, 7, 3, 11), (4, 9, 3, 11)),
    ("klij,klab->ijab", (4, 5, 3, 2), (4, 5, 13, 17), (3, 2, 13, 17)), ("ijdc,kcbd->ijkb", (3, 3, 6, 6), (5, 6, 7, 6), (3, 3, 5, 7))])
@pytest.mark.parametrize("perm", [False, True])
def test_strided_views(ctx, engine, spec, sa, sb, sc, perm):
    """Several modes a side, transposed storage, an output view inside a
    larger array whose other elements stay as they are."""
    import torch
    from paper_2401_11935_gb300 import _lib as L
    rng = np.random.default_rng(5)
    a, b = rng.normal(size=sa), rng.normal(size=sb)
    A, B = torch.tensor(a).cuda(), torch.tensor(b).cuda()
    if perm:
        A = A.permute(*range(A.dim())[::-1]).contiguous().permute(*range(A.dim())[::-1])
        B = B.permute(*range(B.dim())[::-1]).contiguous().permute(*range(B.dim())[::-1])
    big = torch.full([n + 2 for n in sc], 7.0, dtype=torch.float64, device="cuda")
    C = big[tuple(slice(1, 1 + n) for n in sc)]
    torch.cuda.synchronize()
    L.dcsd_einsum_device(ctx.ctx, engine, spec, 2.0, A, B, 1.0, C)
    torch.cuda.synchronize()
    ref = 7.0 + 2.0 * np.einsum(spec, a, b)
    assert np.abs(C.cpu().numpy() - ref).max() < 1e-12
    C.fill_(7.0)
    assert (big == 7.0).all()
