"""chem_step_stiff where its kernel variants and index lists change: species counts at the edges of the
register factorisation (n = N + 1 = 16, 17, 32; 33 goes to the shared-memory one) and a mechanism whose
reactions use every form (three reactants, a species twice on a side, a species on both sides with and
without a net change, three-body and fall-off). Against the FP64 oracle at the parity tolerances (1e-8
relative, as the other stiff tests); the mixed mode within 20 rtol of the oracle's tight integration,
one warp per cell and a team per cell bitwise equal."""
import numpy as np
import pytest

from paper_2312_05800_gb300 import synth
from tests.gpu_util import to_dev
from tests.mechs import tiny_mech

pytestmark = pytest.mark.gpu
DT = 1.0e-6
PARITY = dict(rtol=1e-9, atol_Y=1e-15, atol_T=1e-9, h0=1e-9, max_steps=20000)


def _forms():
    sp = [(3.5, h, 20.0 + 0.3 * i) for i, h in enumerate((0.0, 2e4, -3e4, 1e4, -2e4, 0.0))]
    arr = dict(beta=0.3, Ea=2.0e4)
    fall = dict(A0=3.0e3, beta0=-0.5, Ea0=1.0e4, troe=[0.6, 100.0, 1500.0, 4000.0])
    eff = np.array([1.0, 2.0, 0.5, 1.0, 1.5, 1.0])
    return tiny_mech(sp, [
        dict(reac=[0, 1, 2], prod=[3, 4, 5], A=4.0e3, **arr),         # three reactants and products
        dict(reac=[0, 0, 1], prod=[2, 2, 3], A=2.0e3, **arr),         # twice on a side
        dict(reac=[3, 3, 3], prod=[0, 1, 4], A=3.0e3, **arr),         # three times
        dict(reac=[0, 3], prod=[0, 4], A=5.0e5, **arr),               # a catalyst: no net change of species 0
        dict(reac=[1, 2], prod=[1, 1], A=4.0e5, **arr),               # on both sides with a net change
        dict(reac=[4], prod=[2], A=2.0e6, **arr),
        dict(reac=[2, 3], prod=[4, 4], A=3.0e3, type=1, eff=eff, **arr),
        dict(reac=[1, 4], prod=[3, 5], A=2.0e5, type=2, eff=eff, **arr, **fall),
    ], W=[0.028] * 6, name="forms")


def _mech(kind):
    if kind == "forms":
        return _forms()
    return synth.make_mech("s%d" % kind, kind, 3 * kind, 2, 3, ["C", "H", "O", "N"], 6000 + kind)


def _run(dm, T, p, Y, n, **opts):
    import torch
    from paper_2312_05800_gb300 import binding
    Td, Yd = to_dev(T), to_dev(Y)
    st = torch.zeros(T.size, dtype=torch.int32, device="cuda")
    binding.chem_step_stiff(dm, n, T.size, DT, binding.make_opts(**opts), Td, to_dev(p), Yd, st)
    torch.cuda.synchronize()
    return Td.cpu().numpy()[:n], Yd.cpu().numpy()[:, :n], st.cpu().numpy()[:n]


@pytest.mark.parametrize("kind", [15, 16, 31, 32, "forms"])
def test_variant_edges(oracle, kind):
    from paper_2312_05800_gb300 import binding
    m = _mech(kind)
    dm = binding.Mech(m)
    n = 24
    T, p, Y = synth.states_dirichlet(m, n, 31) if kind == "forms" else synth.states_profiles(m, n, 31)
    To, Yo, so, _ = oracle.step_stiff(m, T, p, Y, DT, ncells=n, **PARITY)
    Tg, Yg, sg = _run(dm, T, p, Y, n, **PARITY)
    assert np.array_equal(sg, so[:n]) and np.all(sg == 0)
    assert np.all(np.abs(Tg - To[:n]) <= 1e-8 * To[:n])
    assert np.all(np.abs(Yg - Yo[:, :n]) <= 1e-8 * np.abs(Yo[:, :n]) + 1e-14)
    # mixed mode; 24 cells take a team each, 24 copies (576 cells) a warp each
    rtol = 1e-3
    mixed = dict(rtol=rtol, atol_Y=1e-10, atol_T=1e-3, h0=1e-9, max_steps=20000, mode=binding.CHEM_ODE_MIXED)
    Tm, Ym, sm = _run(dm, T, p, Y, n, **mixed)
    assert np.all(sm == 0)
    assert np.all(np.abs(Tm - To[:n]) <= 20 * rtol * To[:n])
    assert np.all(np.abs(Ym - Yo[:, :n]) <= 20 * rtol * np.abs(Yo[:, :n]) + 1e-8)
    Tw, Yw, sw = _run(dm, np.tile(T, 24), np.tile(p, 24), np.tile(Y, (1, 24)), 24 * n, **mixed)
    assert np.array_equal(Tw.reshape(24, n), np.tile(Tm, (24, 1)))
    assert np.array_equal(Yw.reshape(m.N, 24, n), np.repeat(Ym[:, None], 24, axis=1))
