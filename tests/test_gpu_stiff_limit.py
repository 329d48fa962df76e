"""chem_step_stiff at the largest mechanism the shared memory of the FP64 mode takes: 63 species and 271 third-body
reactions of six different species each (4 x (n^2 + 2 n + 9 N + 9 R) doubles and 4 n integers fill 227 KB, the layout
that set the limit). The species differ in their initial fractions only, so every reaction is balanced. One cell
per team of warps and one per warp, against the FP64 oracle at the parity tolerances."""
import numpy as np
import pytest

from paper_2312_05800_gb300 import synth
from tests.test_gpu_stiff_sizes import DT, PARITY, _run

pytestmark = pytest.mark.gpu


def _limit_mech():
    m = synth.make_mech("limit", 63, 126, 0, 0, ["C", "H", "O", "N"], 6063)
    R = 271
    rng = np.random.default_rng(9)
    six = np.array([rng.permutation(63)[:6] for _ in range(R)], np.int32)
    m.reac, m.prod, m.rtype = six[:, :3].copy(), six[:, 3:].copy(), np.ones(R, np.int32)
    m.W = np.full(63, 0.03)
    m.nasa_lo, m.nasa_hi = np.tile(m.nasa_lo[:1], (63, 1)), np.tile(m.nasa_hi[:1], (63, 1))
    m.A, m.beta, m.Ea = np.full(R, 1e4), np.zeros(R), np.zeros(R)
    m.A0 = m.beta0 = m.Ea0 = np.zeros(R)
    m.troe, m.eff = np.zeros((R, 4)), rng.uniform(0.5, 2.0, (R, 63))
    return m


@pytest.mark.parametrize("cells", [3, 160])
def test_largest_mechanism(oracle, cells):
    from paper_2312_05800_gb300 import binding
    m = _limit_mech()
    T, p, Y = synth.states_dirichlet(m, 4, 31)
    To, Yo, so, _ = oracle.step_stiff(m, T, p, Y, DT, ncells=4, **PARITY)
    rep = lambda a: np.ascontiguousarray(np.tile(a[..., :4], 40)[..., :max(4, cells)])
    Tg, Yg, sg = _run(binding.Mech(m), rep(T), rep(p), rep(Y), cells, **PARITY)
    i = np.arange(cells) % 4
    assert np.all(so[:4] == 0) and np.all(sg == 0)
    assert np.abs(Yo[:, :4] - Y[:, :4]).max() > 0.0
    assert np.all(np.abs(Tg - To[i]) <= 1e-8 * To[i])
    assert np.all(np.abs(Yg - Yo[:, i]) <= 1e-8 * np.abs(Yo[:, i]) + 1e-14)
