"""props_eval's bounded waits run out on purpose (failure detection without a GPU fault), with many tiles per CTA: with
no try at all every transport output (in the thermo pass: every output) is NaN, with one try every requested output
of every cell is either the value of an undisturbed call, bit for bit, or NaN. None keeps what the caller's arrays
held, none past ncells is written, and the next call with the default limit is undisturbed. The full FP32 pass at
its three sizes, and the thermo pass (cp and h alone)."""
import numpy as np
import pytest

from paper_2312_05800_gb300 import synth
from tests.gpu_util import to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mech,n,transport", [("c1", 500003, True), ("c2", 400003, True), ("c5", 150001, True),
                                              ("c2", 700001, False)])
def test_no_stale_outputs(mech, n, transport):
    import torch
    from paper_2312_05800_gb300 import binding
    m = synth.get_mech(mech)
    dm = binding.Mech(m)
    ld = synth.padded_ld(n)
    T, p, Y = synth.states_profiles(m, 4096, 11) if mech != "c1" else synth.states_dirichlet(m, 4096, 11)
    rep = lambda a: to_dev(np.tile(a[..., :4096], ld // 4096 + 1)[..., :ld], torch.float32)
    Td, pd, Yd = rep(T), rep(p), rep(Y)

    def call():
        out = torch.full((4 + m.N, ld), -7.0, dtype=torch.float32, device="cuda")
        more = (out[2], out[3], out[4:]) if transport else ()
        binding.props_eval(dm, n, ld, binding.CHEM_F32, Td, pd, Yd, out[0], out[1], *more)
        torch.cuda.synchronize()
        return out[:4 + m.N if transport else 2]

    good = call()
    assert torch.isfinite(good).all()
    for tries in (-1, 1, 1, 1):
        dm.set_wait_limit(tries)
        got = call()
        nan = torch.isnan(got[:, :n])
        assert torch.equal(torch.where(nan, good[:, :n], got[:, :n]), good[:, :n])
        assert torch.equal(got[:, n:], good[:, n:])
        if tries < 0:
            assert nan[2 if transport else 0:].all()
            # cp and h of the full pass need no wait: those of a CTA's first tile are there, later tiles have none
            assert not transport or (nan[:2].any() and not nan[:2].all())
    dm.set_wait_limit(0)
    assert torch.equal(call(), good)
