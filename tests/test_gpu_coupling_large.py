"""Coupling terms with many virtual orbitals: a system embedded among virtuals
that have no amplitudes, no integrals and no Fock couplings keeps its residual.
At 802 union virtuals the group vectors of the separable FP64 form take 167 KB
of shared memory; beyond 1063 they do not fit and every element is evaluated
term by term, which takes seven times as long.  (BF16X6, whose coupling terms
are FP64 and whose ladder takes a second here.)"""
import dataclasses

import numpy as np
import pytest

from synth import make_system, random_amplitudes

pytestmark = pytest.mark.gpu


def _embedded(s, T, n_v):
    n0, n = s.n_c + 2 + s.n_v, s.n_c + 2 + n_v

    def pad(x, fill):
        y = np.zeros((n, n))
        y[:n0, :n0] = x
        y[np.arange(n0, n), np.arange(n0, n)] = fill
        return y

    B = np.zeros((s.naux, n, n))
    B[:, :n0, :n0] = s.B
    big = dataclasses.replace(s, n_v=n_v, eps=np.concatenate([s.eps, np.full(n - n0, 5.0)]),
                              parity=np.concatenate([s.parity, np.zeros(n - n0, s.parity.dtype)]), B=B,
                              fock_a=pad(s.fock_a, 5.0), fock_b=pad(s.fock_b, 5.0))
    add = n_v - s.n_v
    return big, [np.pad(t, [(0, 0)] * (t.ndim // 2) + [(0, add)] * (t.ndim // 2)) for t in T]


def test_embedded_system_keeps_its_residual(monkeypatch, capfd):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2401_11935_gb300 as P
    s = make_system((2, 30, 8), seed=4, ias=True)
    T = random_amplitudes(s, seed=5, scale1=0.05, scale2=0.05)
    eng = P.Engine.from_system(s)
    R0, W0, E0 = eng.residual(eng.to_device(T), method=0, precision=4)
    R0 = [x.cpu().numpy() for x in R0]
    eng.close()
    big, Tb = _embedded(s, T, 800)
    capfd.readouterr()
    monkeypatch.setenv("DCSD_TRACE", "1")
    eng = P.Engine.from_system(big)
    R, W, E = eng.residual(eng.to_device(Tb), method=0, precision=4)
    R = [x.cpu().numpy() for x in R]
    eng.close()
    assert "mterm_doubles_sep64" in capfd.readouterr().err
    v = s.n_v + 1
    rmax = max(np.abs(y).max() for y in R0)
    for x, y in zip(R, R0):
        sub = x[..., :v] if x.ndim == 2 else x[..., :v, :v]
        assert np.abs(sub - y).max() < 2e-5 * rmax  # (the split's precision, as elsewhere)
    assert abs(W - W0) < 2e-5 * rmax and abs(E - E0) < 1e-12 and abs(W) > 1e-3
