"""The FP32 full properties pass for tables that FP16 pairs cannot hold (diffusion fits scaled by 1e-30: every
coefficient lies below the range in which the tensor-core pass scales its rows), which the pair loop takes: its 16-,
32- and 64-species instances at the edges of their ranges, with FP32 and FP64 state. cp, h, mu and lambda do not know
the scale, and D is the unscaled mechanism's times 1e30: the two passes agree within 2e-5, the sum of the
1e-5 that each is held to against the oracle."""
import numpy as np
import pytest

from paper_2312_05800_gb300 import synth
from tests.gpu_util import to_dev
from tests.test_gpu_props_tc import _mech, _state

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,n", [(14, 1000), (16, 129), (17, 2001), (32, 300), (33, 130), (56, 257)])
def test_pair_loop_takes_what_does_not_split(N, n):
    import torch
    from paper_2312_05800_gb300 import binding
    m, tiny = _mech(N), _mech(N)
    tiny.diff_fit = m.diff_fit * 1e-30
    ld = synth.padded_ld(n)
    T, p, Y = _state(m, n, ld, N)
    for dtype, td in ((binding.CHEM_F32, torch.float32), (binding.CHEM_F64_IN_F32, torch.float64)):
        got = []
        for mech in (m, tiny):
            out = torch.full((4 + m.N, ld), float("nan"), dtype=torch.float32, device="cuda")
            binding.props_eval(binding.Mech(mech), n, ld, dtype, to_dev(T, td), to_dev(p, td), to_dev(Y, td), out[0],
                               out[1], out[2], out[3], out[4:])
            torch.cuda.synchronize()
            got.append(out.double().cpu().numpy()[:, :n])
        a, b = got
        b[4:] *= 1e-30
        assert np.isfinite(b).all()
        assert np.array_equal(a[:2], b[:2])
        assert np.all(np.abs(a[2:] - b[2:]) <= 2e-5 * np.abs(a[2:])), float((np.abs(a[2:] / b[2:] - 1)).max())
        assert not np.array_equal(a[2:], b[2:])          # the other route did run
