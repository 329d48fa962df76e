"""chem_step_stiff's mixed mode (FP32 rate exponentials and matrix, rtol 1e-2): bitwise the stored states and step
counts of a warp per cell with the LU in shared memory, the kernel that defined the mode, for 9, 30 and 53
species. The mode's exponentials cut their FP64 arguments to FP32, so one product fused or not in the stage sums moves
T by up to 2e-7 over an integration: no tolerance below the caller's own separates that from a wrong result, and
equality does. The cells are repeated to take the routes of one and of two cells per warp."""
import json
import os

import numpy as np
import pytest

from paper_2312_05800_gb300 import synth
from tests.gpu_util import to_dev

pytestmark = pytest.mark.gpu
GOLD = json.load(open(os.path.join(os.path.dirname(__file__), "golden", "stiff_mixed.json")))


def _floats(a):
    return np.array([[float.fromhex(v) for v in r] for r in a])


@pytest.mark.parametrize("cells", [200, 4000])
@pytest.mark.parametrize("case", GOLD["cases"], ids=lambda c: "%s-h%g" % (c["mech"], c["h0"]))
def test_mixed_mode_bits(case, cells):
    import torch
    from paper_2312_05800_gb300 import binding
    n = len(case["T"])
    rep = lambda a: to_dev(np.tile(a, cells // n + 1)[..., :cells])
    T, p, Y = rep(_floats([case["T"]])[0]), rep(_floats([case["p"]])[0]), rep(_floats(case["Y"]))
    st = torch.zeros(cells, dtype=torch.int32, device="cuda")
    ns = torch.zeros(cells, dtype=torch.int32, device="cuda")
    opts = binding.make_opts(h0=case["h0"], mode=binding.CHEM_ODE_MIXED, **GOLD["opts"])
    binding.chem_step_stiff(binding.Mech(synth.get_mech(case["mech"])), cells, cells, GOLD["dt"], opts, T, p, Y, st, ns)
    torch.cuda.synchronize()
    idx = np.arange(cells) % n
    assert not st.cpu().numpy().any()
    assert np.array_equal(ns.cpu().numpy(), np.array(case["steps"])[idx])
    assert np.array_equal(T.cpu().numpy(), _floats([case["T1"]])[0][idx])
    assert np.array_equal(Y.cpu().numpy(), _floats(case["Y1"])[:, idx])
