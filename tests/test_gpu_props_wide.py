"""The FP32 full properties pass on states with mass fractions of both signs and |X_k| >= 4, past the range of the FP16
terms of its tensor-core sums: such cells stay finite and match the FP64 pass on the same FP32-rounded state
within 1e-5 times the condition of each sum (sum of magnitudes over magnitude of the sum; FP32 rounding of N terms
times N and the tables' polynomials is below 1e-5), the cells beside them do not change by a bit, and states that are
themselves not finite stay so. The excess is a heavy species' and the deficit a light one's, whose Wilke weights are
small, so that no sum cancels (a bound by conditions is of first order)."""
import numpy as np
import pytest

from paper_2312_05800_gb300 import synth
from tests.gpu_util import to_dev
from tests.test_gpu_props_tc import _mech, _state

pytestmark = pytest.mark.gpu


def _conditions(m, T, Y):
    """Condition numbers of mu, lambda and D_k per cell, from the formulas in FP64."""
    X = Y / m.W[:, None]
    X = X / X.sum(0)
    x = np.log(T / 1000.0)
    mu = np.exp(sum(m.visc_fit[:, i, None] * x ** i for i in range(5)))
    a = np.where(T >= synth.T_MID, m.nasa_hi[:, :5, None], m.nasa_lo[:, :5, None])
    cp = sum(a[:, i] * T ** i for i in range(5))
    parts, conds, cD = np.zeros_like(Y), np.zeros_like(Y), np.zeros_like(Y)
    for k in range(m.N):
        phi = (1.0 + np.sqrt(mu[k] / mu) * (m.W / m.W[k])[:, None] ** 0.25) ** 2 / np.sqrt(8.0 * (1.0 + m.W[k] / m.W))[:, None]
        den = (X * phi).sum(0)
        parts[k], conds[k] = X[k] * mu[k] / den, (np.abs(X) * phi).sum(0) / np.abs(den)
        g = sum(m.diff_fit[k, :, i, None] * x ** i for i in range(5))
        g[k] = 0.0
        cD[k] = (np.abs(X) * np.abs(g)).sum(0) / np.abs((X * g).sum(0))
    lam = parts * (cp + 1.25) / m.W[:, None]
    return [(np.abs(q) * conds).sum(0) / np.abs(q.sum(0)) for q in (parts, lam)] + [cD]


@pytest.mark.parametrize("N", [14, 30, 53])
def test_wide_mole_fractions(N):
    import torch
    from paper_2312_05800_gb300 import binding
    m = _mech(N)
    dm = binding.Mech(m)
    n = 700
    ld = synth.padded_ld(n)
    T, p, Y = _state(m, n, ld, N)
    wide = np.arange(3, n, 7)
    order = np.argsort(m.W)
    Yw = Y.copy()
    for q, i in enumerate(wide):                     # mole fractions that sum to 1, one past 4 and one below -4
        X = Y[:, i] / m.W
        X *= 0.5 / X.sum()
        big = 4.7 + 0.1 * (q % 30)
        X[order[-1 - q % 2]] += big
        X[order[q % 2]] -= big - 0.5
        Yw[:, i] = X * m.W / (X * m.W).sum()
    Yw = np.asarray(Yw, np.float32).astype(np.float64)
    bad = [5, 12]
    Yw[0, bad[0]] = np.nan
    T[bad[1]] = np.inf

    def run(Ya, dtype, td):
        out = torch.full((4 + m.N, ld), -7.0, dtype=torch.float64 if td == torch.float64 and dtype == binding.CHEM_F64
                         else torch.float32, device="cuda")
        binding.props_eval(dm, n, ld, dtype, to_dev(T, td), to_dev(p, td), to_dev(Ya, td), out[0], out[1], out[2],
                           out[3], out[4:])
        torch.cuda.synchronize()
        return out.double().cpu().numpy()[:, :n]

    ref = run(Yw, binding.CHEM_F64, torch.float64)
    X = Yw[:, wide] / m.W[:, None]
    X = X / X.sum(0)
    assert np.all(np.abs(X).max(0) >= 4.0)
    cmu, clam, cD = _conditions(m, T[wide], Yw[:, wide])
    assert max(cmu.max(), clam.max()) < 1e3
    for dtype, td in ((binding.CHEM_F32, torch.float32), (binding.CHEM_F64_IN_F32, torch.float64)):
        got, plain = run(Yw, dtype, td), run(Y, dtype, td)
        rest = np.setdiff1d(np.arange(n), np.concatenate([wide, bad]))
        assert np.array_equal(got[:, rest], plain[:, rest])
        assert not np.isfinite(got[2, bad]).any()
        g, r = got[:, wide], ref[:, wide]
        assert np.isfinite(g).all()
        for row, cond in ((2, cmu), (3, clam)):
            assert np.all(np.abs(g[row] - r[row]) <= 1e-5 * cond * np.abs(r[row]))
        assert np.all(np.abs(g[4:] - r[4:]) <= 1e-5 * cD * np.abs(r[4:]))
