"""FP64 properties with several threads per cell (small calls): species counts around the thread counts per
cell (4, 8, 16, 32) and cell counts around the lines between them, up to the loop with one thread per cell,
against the FP64 oracle at 1e-12 relative (h: of sum_k Y_k |h_k|), as the other FP64 properties."""
import numpy as np
import pytest

from paper_2312_05800_gb300 import synth
from tests.gpu_util import h_scale, to_dev

pytestmark = pytest.mark.gpu


def _mech(N):
    if N < 12:
        return synth.make_mech("p%d" % N, N, 2 * N, 0, 2, ["H", "O", "N"], 7000 + N)
    return synth.make_mech("p%d" % N, N, 2 * N, 1, 2, ["C", "H", "O", "N"], 7000 + N)


@pytest.mark.parametrize("N,n", [(8, 1), (9, 4096), (9, 19455), (9, 19457), (15, 33), (16, 2500), (23, 1200), (24, 1000),
                                 (30, 2431), (33, 1217), (64, 131), (64, 4864)])
def test_threads_per_cell(oracle, N, n):
    import torch
    from paper_2312_05800_gb300 import binding
    m = _mech(N)
    dm = binding.Mech(m)
    ld = synth.padded_ld(n) + 4
    T, p, Y = synth.states_dirichlet(m, n, N, ld)
    Y[:, 0] = 0.0
    Y[N // 2, 0] = 1.0                                     # a pure species
    out = torch.full((4 + N, ld), float("nan"), dtype=torch.float64, device="cuda")
    binding.props_eval(dm, n, ld, binding.CHEM_F64, to_dev(T), to_dev(p), to_dev(Y), out[0], out[1], out[2], out[3], out[4:])
    thermo = torch.full((2, ld), float("nan"), dtype=torch.float64, device="cuda")
    binding.props_eval(dm, n, ld, binding.CHEM_F64, to_dev(T), to_dev(p), to_dev(Y), thermo[0], thermo[1])
    torch.cuda.synchronize()
    got = out.cpu().numpy()
    assert np.isnan(got[:, n:]).all() and torch.equal(thermo[:, :n], out[:2, :n])
    keep = np.unique(np.concatenate([np.arange(min(n, 300)), np.arange(max(0, n - 300), n)]))
    cp, h, mu, lam, Dk = oracle.props(m, T[keep], p[keep], np.ascontiguousarray(Y[:, keep]))
    hs = h_scale(oracle, m, T[keep], Y[:, keep], keep.size)
    for a, b, scale in ((got[0], cp, cp), (got[1], h, hs), (got[2], mu, mu), (got[3], lam, lam), (got[4:], Dk, Dk)):
        a = a[..., keep]
        assert np.all(np.abs(a - b) <= 1e-12 * np.abs(scale)), float((np.abs(a - b) / np.abs(scale)).max())
