"""The FP64 contraction engines (FP64 CUDA cores; modular GEMMs on the tensor
cores) against sums in extended precision, at the edges of their tiles.

Error bound of the modular engine: the rows of A and B are scaled to integers
of 2-norm in (2^57, 2^58] and (2^56, 2^57] and rounded (at most 1/2 per
element), the integer product is exact, and one rounding to FP64 follows:
|error| <= |a| |b| sqrt(K) / 2 (2^-57 + 2^-56) + 2^-53 |c| to first order.
The FMA chain of the CUDA cores: K 2^-53 sum |a b|.  Both bounds take a
factor two for the roundings of alpha and beta."""
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


def _bounds(a, b, alpha, c0, beta):
    K = a.shape[1]
    na, nb = np.linalg.norm(a, axis=1), np.linalg.norm(b, axis=1)
    ab = np.abs(a) @ np.abs(b).T
    tail = 2.0 ** -53 * (abs(alpha) * ab + abs(beta) * np.abs(c0))
    crt = abs(alpha) * np.outer(na, nb) * np.sqrt(K) * 0.5 * (2.0 ** -57 + 2.0 ** -56)
    return {1: 2 * (abs(alpha) * K * 2.0 ** -53 * ab + tail), 2: 2 * (crt + tail)}


def _run(eng, engine, a, b, alpha, beta, c0, spec="mk,nk->mn"):
    import torch
    from paper_2401_11935_gb300 import _lib as L
    A, B = torch.tensor(a).cuda(), torch.tensor(b).cuda()
    C = torch.tensor(c0).cuda()
    torch.cuda.synchronize()
    L.dcsd_einsum_device(eng.ctx, engine, spec, alpha, A, B, beta, C)
    torch.cuda.synchronize()
    return C.cpu().numpy()


# tile edges: 4, 16 and 64 (packing, CUDA cores), 128 and 256 (tensor-core tiles), k-blocks of
# 64, sums of 1024 k, norm blocks of 512 k, split k
SHAPES = [(1, 1, 1), (3, 5, 2), (16, 16, 16), (17, 15, 33), (64, 64, 64), (65, 63, 65), (127, 16, 128), (128, 17, 63),
          (129, 255, 100), (130, 257, 31), (12, 12, 5000), (40, 300, 1024), (257, 33, 1025), (300, 530, 200),
          (9, 7, 20000), (513, 4, 513)]


@pytest.mark.parametrize("M,N,K", SHAPES)
@pytest.mark.parametrize("engine", [0, 1, 2])
def test_contraction_error_bound(ctx, M, N, K, engine):
    rng = np.random.default_rng(M * 7 + N * 3 + K)
    a, b = rng.normal(size=(M, K)), rng.normal(size=(N, K))
    a *= np.exp(rng.normal(size=(M, 1)) * 10)  # rows of very different size
    b[rng.random(b.shape) < 0.5] = 0.0
    for alpha, beta in ((1.0, 0.0), (-0.5, 1.0)):
        c0 = rng.normal(size=(M, N)) if beta else np.full((M, N), np.nan)
        ref = np.longdouble(alpha) * _exact(a, b) + (np.longdouble(beta) * c0 if beta else 0)
        err = np.abs(_run(ctx, engine, a, b, alpha, beta, c0) - ref)
        bound = _bounds(a, b, alpha, c0 if beta else np.zeros((M, N)), beta)
        assert (err <= (np.maximum(bound[1], bound[2]) if engine == 0 else bound[engine])).all()


@pytest.mark.parametrize("K", [64, 1024, 4096, 9000])
def test_modular_sums_are_exact(ctx, K):
    """Integers: every residue sum has to be exact, also where all products
    have one sign (2^52 + 128 and 2^51 + 128 keep their unit bits at K = 1024
    and have residues 128 modulo 256, so that the FP32 sums reach 2^24)."""
    for va, vb in ((128, 128), (-128, 128), (127, 253), (2 ** 20 + 128, 3), (2 ** 52 + 128, 2 ** 51 + 128),
                   (-2 ** 52 - 128, 2 ** 51 + 128), (2 ** 52 + 127, 2 ** 51 + 125)):
        if K > 1024 and abs(va) > 2 ** 50:
            continue  # the rounding to integers then acts
        a, b = np.full((130, K), float(va)), np.full((24, K), float(vb))
        c = _run(ctx, 2, a, b, 1.0, 0.0, np.zeros((130, 24)))
        assert (c == float(va * vb * K)).all()
    rng = np.random.default_rng(K)
    a = rng.integers(-2 ** 18, 2 ** 18, (70, K)).astype(float)
    b = rng.integers(-2 ** 18, 2 ** 18, (50, K)).astype(float)
    ref = (a.astype(np.int64) @ b.astype(np.int64).T).astype(float)
    assert (_run(ctx, 2, a, b, 1.0, 0.0, np.zeros((70, 50))) == ref).all()


def test_modular_extreme_rows(ctx):
    """Zero rows, subnormals, the largest magnitudes; Inf and NaN stay in
    their rows and columns."""
    rng = np.random.default_rng(1)
    a, b = rng.normal(size=(20, 100)), rng.normal(size=(30, 100))
    a[0] = 0.0
    a[1] *= 1e-310
    a[2] *= 1e300
    a[3] *= 1e-200
    b[4] *= 1e-5
    a[5, 7] = np.inf
    b[6, 3] = np.nan
    c = _run(ctx, 2, a, b, 1.0, 0.0, np.zeros((20, 30)))
    good = np.ones((20, 30), bool)
    good[5] = good[:, 6] = False
    assert not np.isfinite(c[~good]).any() and np.isfinite(c[good]).all()
    a[5, 7] = b[6, 3] = 0.0
    ref = _exact(a, b)
    norm = np.outer(np.linalg.norm(a.astype(np.longdouble), axis=1), np.linalg.norm(b, axis=1))
    assert (np.abs(c - ref)[good] <= (1e-14 * norm + 1e-322)[good]).all()


@pytest.mark.parametrize("engine", [1, 2])
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


# What follows grades the elements along k: |a| |b| is then far above
# S = sum |a_k b_k|, and an error relative to the norms would be a loss of
# accuracy against the FMA chain.  Bound for every engine, in u = 2^-53: the
# chain's K u S.  The modular engine keeps a result only where S is at least
# 2^-7 in the units of its integers (2^-62 and 2^-61 of the norms' bounds, at
# least half of which the norms are): sqrt(K) / 2 (2^-62 + 2^-61) <= 0.375 sqrt(K) u S.


def _graded(rng, shape, decades):
    return rng.normal(size=shape) * 10.0 ** (-decades * np.arange(shape[1]) / max(1, shape[1] - 1))


@pytest.mark.parametrize("M,N,K", [(1, 1, 2), (17, 15, 33), (64, 64, 484), (130, 257, 31), (129, 33, 1025), (12, 12, 5000),
                                   (40, 300, 1024), (300, 530, 200)])
@pytest.mark.parametrize("decades", [4, 8, 30])
@pytest.mark.parametrize("engine", [0, 1, 2])
def test_rows_graded_along_k(ctx, M, N, K, decades, engine):
    rng = np.random.default_rng(M + 5 * N + 11 * K + decades)
    a, b = _graded(rng, (M, K), decades), _graded(rng, (N, K), decades)[:, ::-1].copy()
    for alpha, beta in ((1.0, 0.0), (-0.5, 1.0)):
        c0 = rng.normal(size=(M, N)) if beta else np.full((M, N), np.nan)
        ref = np.longdouble(alpha) * _exact(a, b) + (np.longdouble(beta) * c0 if beta else 0)
        err = np.abs(_run(ctx, engine, a, b, alpha, beta, c0) - ref)
        assert (err <= _bounds(a, b, alpha, c0 if beta else np.zeros((M, N)), beta)[1]).all()


@pytest.mark.parametrize("spec", ["mk,nk->mn", "km,nk->nm", "mk,kn->mn"])
def test_some_graded_rows_among_others(ctx, spec):
    """A few graded rows, rows and columns of zeros, products that are all zero:
    the elements computed again stand between others of their tiles."""
    rng = np.random.default_rng(17)
    M, N, K = 147, 290, 700
    a, b = rng.normal(size=(M, K)), rng.normal(size=(N, K))
    a[[0, 31, 100, 146]] = _graded(rng, (4, K), 12)
    b[[5, 256, 289]] = _graded(rng, (3, K), 12)[:, ::-1]
    a[7] = 0.0
    b[44] = 0.0
    a[20, ::2] = 0.0
    b[21, 1::2] = 0.0
    sa, rest = spec.split(",")
    sb, sc = rest.split("->")
    A, B = (a if sa == "mk" else a.T.copy()), (b if sb == "nk" else b.T.copy())
    c = _run(ctx, 2, A, B, 1.0, 0.0, np.full((M, N) if sc == "mn" else (N, M), np.nan), spec)
    c = c if sc == "mn" else c.T
    assert (np.abs(c - _exact(a, b)) <= _bounds(a, b, 1.0, np.zeros((M, N)), 0.0)[1]).all()
    assert (c[7] == 0).all() and (c[:, 44] == 0).all() and c[20, 21] == 0.0


def test_small_products_beside_large_elements(ctx):
    a, b = np.array([[1e9, 1e-9], [1.0, 1e-16]]), np.array([[0.0, 1.0], [1e-300, 1e-16]])
    for engine in (0, 1, 2):
        c = _run(ctx, engine, a, b, 1.0, 0.0, np.zeros((2, 2)))
        assert c[0, 0] == 1e-9 and c[1, 0] == 1e-16
        assert abs(c[0, 1] - 1e-25) <= 1e-40 and abs(c[1, 1] - 1e-32) <= 1e-47


def test_infinities_as_in_a_chain(ctx):
    rng = np.random.default_rng(2)
    a, b = np.abs(rng.normal(size=(40, 90))), np.abs(rng.normal(size=(50, 90)))
    a[3, 5], a[33, 8], b[17, 5], b[18, 0] = np.inf, -np.inf, 0.0, np.nan
    with np.errstate(invalid="ignore"):
        ref = a @ b.T
    for engine in (0, 1, 2):
        c = _run(ctx, engine, a, b, 1.0, 0.0, np.zeros((40, 50)))
        assert (np.isnan(c) == np.isnan(ref)).all() and (np.isposinf(c) == np.isposinf(ref)).all()
        assert (np.isneginf(c) == np.isneginf(ref)).all()
        ok = np.isfinite(ref)
        assert np.abs(c[ok] - ref[ok]).max() < 1e-11


@pytest.mark.parametrize("K", [64, 1024])
def test_modular_sums_at_the_integers_bounds(ctx, K):
    """Elements that are integers of the modular engine as they stand (the
    norms sqrt(K) 2^(61 - log2(K) / 2) and half of it are their bounds), with
    residues 128 modulo 256: FP32 sums of 2^24 and results of 2^122."""
    e = 61 - int(np.log2(K)) // 2
    for sa, sb in ((1, 1), (-1, 1), (-1, -1)):
        va, vb = sa * (2 ** e + 128), sb * (2 ** (e - 1) + 128)
        assert float(va) == va and float(vb) == vb
        c = _run(ctx, 2, np.full((130, K), float(va)), np.full((24, K), float(vb)), 1.0, 0.0, np.zeros((130, 24)))
        assert (c == float(va * vb * K)).all()


@pytest.mark.parametrize("warm", [False, True])
def test_contraction_under_capture(warm):
    """Captured by the caller: the workspace of the modular engine is not
    allocated there, so a context that does not have it yet records the CUDA
    cores' launches."""
    import torch
    import paper_2401_11935_gb300 as P
    from paper_2401_11935_gb300 import _lib as L
    from synth import make_system
    rng = np.random.default_rng(4)
    a, b = rng.normal(size=(500, 300)), rng.normal(size=(700, 300))
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        A, B = torch.tensor(a).cuda(), torch.tensor(b).cuda()
        C = torch.zeros(500, 700, dtype=torch.float64, device="cuda")
        eng = P.Engine.from_system(make_system((2, 40, 12), seed=3))
        # (loads the kernels of both engines)
        other = P.Engine.from_system(make_system((2, 40, 12), seed=3))
        for engine in (1, 2):
            L.dcsd_einsum_device(other.ctx, engine, "mk,nk->mn", 1.0, A, B, 0.0, C)
        if warm:
            L.dcsd_einsum_device(eng.ctx, 0, "mk,nk->mn", 1.0, A, B, 0.0, C)
        stream.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            L.dcsd_einsum_device(eng.ctx, 0, "mk,nk->mn", 1.0, A, B, 0.0, C)
        C.zero_()
        graph.replay()
        stream.synchronize()
    del graph
    c = C.cpu().numpy()
    eng.close()
    other.close()
    assert (np.abs(c - _exact(a, b)) <= _bounds(a, b, 1.0, np.zeros(c.shape), 0.0)[1]).all()
