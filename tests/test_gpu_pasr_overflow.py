"""chem_pasr where one reaction's rate overflows FP64: only the species of that reaction lose their times; the
others' stay, so tau_c and kappa match the oracle. The overflowing reaction is the first and the last in the device's
order (the species' reaction lists are padded to one length)."""
import numpy as np
import pytest

from oracle import pasr as P
from paper_2312_05800_gb300 import synth
from tests.gpu_util import to_dev
from tests.test_gpu_pasr import _times

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,reaction", [(14, 0), (14, -1), (40, 0)])
def test_one_infinite_rate(oracle, N, reaction):
    import torch
    from paper_2312_05800_gb300 import binding
    m = synth.make_mech("o%d" % N, N, 2 * N, 0, 0, ["C", "H", "O", "N"], 5000 + N)   # elementary: file order
    m.A[reaction], m.beta[reaction] = 1e308, 12.0
    n = 96
    T, p, Y = synth.states_dirichlet(m, n, 77)
    T, p, Y = T[:n], p[:n], np.ascontiguousarray(Y[:, :n])
    T = np.maximum(T, 800.0)
    f = np.array([oracle.rhs(m, float(p[i]), np.concatenate([[T[i]], Y[:, i]])) for i in range(n)])[:, 1:]
    assert (~np.isfinite(f)).any(1).all() and np.isfinite(f).any(1).all()
    tt, tk = _times(n, 78)
    tc = torch.zeros(n, dtype=torch.float64, device="cuda")
    kp = torch.zeros(n, dtype=torch.float64, device="cuda")
    binding.chem_pasr(binding.Mech(m), n, n, 1e-6, to_dev(T), to_dev(p), to_dev(Y), to_dev(tt[:n]), to_dev(tk[:n]), None,
                      None, tc, kp)
    torch.cuda.synchronize()
    otc = P.chemical_time(m, T, p, Y, 1e-6)
    assert np.all(otc > 0.0) and np.all(np.isfinite(otc))
    assert np.allclose(tc.cpu().numpy(), otc, rtol=1e-9, atol=0)
    assert np.allclose(kp.cpu().numpy(), P.kappa(otc, tt[:n], tk[:n]), rtol=1e-9, atol=0)
