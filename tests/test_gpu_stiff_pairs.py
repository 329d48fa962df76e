"""chem_step_stiff with two cells in a warp (many cells of up to 15 species): bitwise the results, status and
step counts of one warp per cell (the same cells in calls of at most 500), for even and odd cell counts,
at the edges of the species range, with cells that end early (a step limit, a NaN) beside others that
go on, in both modes."""
import numpy as np
import pytest

from paper_2312_05800_gb300 import synth
from tests.gpu_util import to_dev
from tests.test_gpu_stiff_sizes import DT, _mech

pytestmark = pytest.mark.gpu


def _run(dm, T, p, Y, **opts):
    import torch
    from paper_2312_05800_gb300 import binding
    n = T.size
    ld = (n + 3) // 4 * 4
    pad = lambda a: to_dev(np.concatenate([a, np.repeat(a[..., -1:], ld - n, axis=-1)], axis=-1))
    Td, Yd = pad(T), pad(Y)
    st = torch.zeros(ld, dtype=torch.int32, device="cuda")
    ns = torch.zeros(ld, dtype=torch.int32, device="cuda")
    binding.chem_step_stiff(dm, n, ld, DT, binding.make_opts(**opts), Td, pad(p), Yd, st, ns)
    torch.cuda.synchronize()
    return Td.cpu().numpy()[:n], Yd.cpu().numpy()[:, :n], st.cpu().numpy()[:n], ns.cpu().numpy()[:n]


@pytest.mark.parametrize("mode", ["fp64", "mixed"])
@pytest.mark.parametrize("kind,n", [(14, 4000), (15, 6001), ("forms", 4003)])
def test_pairs_bitwise(kind, n, mode):
    from paper_2312_05800_gb300 import binding
    m = _mech(kind)
    dm = binding.Mech(m)
    T, p, Y = synth.states_dirichlet(m, n, 5) if kind == "forms" else synth.states_profiles(m, n, 5)
    T, p, Y = T[:n].copy(), p[:n].copy(), Y[:, :n].copy()
    Y[0, 7::97] = np.nan
    opts = dict(rtol=1e-3, atol_Y=1e-10, atol_T=1e-3, h0=1e-9, max_steps=12)
    if mode == "mixed":
        opts["mode"] = binding.CHEM_ODE_MIXED
    whole = _run(dm, T, p, Y, **opts)
    parts = [_run(dm, T[i:i + 500], p[i:i + 500], Y[:, i:i + 500], **opts) for i in range(0, n, 500)]
    assert whole[2][7] != 0 and np.any(whole[2] == 0)
    for k, a in enumerate(whole):
        assert np.array_equal(a, np.concatenate([q[k] for q in parts], axis=-1), equal_nan=k < 2)
