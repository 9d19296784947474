"""The modular FP64 GEMM on pairs of SMs (the default) against its one-CTA
form (DCSD_TC_MULTICAST=0): the integer results are exact in both, so the
outputs are identical bit for bit, with one, even and odd numbers of 128-row
tiles, several column tiles and split sums over k.  The trace names the form
that ran."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SHAPES = [(100, 40, 70), (130, 300, 520), (300, 257, 1100), (513, 17, 64), (640, 530, 33), (200, 12, 6000)]


def _products(monkeypatch, capfd, pairs):
    import torch
    import paper_2401_11935_gb300 as P
    from paper_2401_11935_gb300 import _lib as L
    from synth import make_system
    monkeypatch.setenv("DCSD_TC_MULTICAST", "1" if pairs else "0")
    monkeypatch.setenv("DCSD_TRACE", "1")
    eng = P.Engine.from_system(make_system((2, 40, 12), seed=3))
    out = []
    for M, N, K in SHAPES:
        rng = np.random.default_rng(M + N + K)
        a, b = torch.tensor(rng.normal(size=(M, K))).cuda(), torch.tensor(rng.normal(size=(N, K))).cuda()
        a[M // 2] = 0.0
        a[M // 2, 0] = 1e3  # one row with small sums of magnitudes
        c = torch.full((N, M), np.nan, dtype=torch.float64, device="cuda")  # (m contiguous: the m side has the tiles)
        torch.cuda.synchronize()
        L.dcsd_einsum_device(eng.ctx, 2, "mk,nk->nm", 1.0, a, b, 0.0, c)
        torch.cuda.synchronize()
        out.append(c.cpu().numpy())
    eng.close()  # (prints the trace)
    return out, capfd.readouterr().err


def test_one_cta_and_paired_modular_gemms_are_identical(monkeypatch, capfd):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    c1, e1 = _products(monkeypatch, capfd, True)
    c0, e0 = _products(monkeypatch, capfd, False)
    for x, y in zip(c1, c0):
        assert np.isfinite(x).all() and np.array_equal(x, y)
    assert "crt-gemm-pairs" in e1 and "crt-gemm " in e1  # (one row of tiles: no pair)
    assert "crt-gemm-pairs" not in e0 and "crt-gemm " in e0
