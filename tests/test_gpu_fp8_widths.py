"""E4M3 layer outputs stored in pairs of 16-column chunks: widths where a tile or the layer ends after the
first chunk of a pair. The same network with eight dead units (zero weights in and out, zero bias) added to a
layer has a width that is not a multiple of 16, which takes the element stores; dead units add exact
zeros, so both give the same bits."""
import numpy as np
import pytest

from paper_2312_05800_gb300 import synth
from tests.gpu_util import to_dev
from tests.test_gpu_fp8 import _mlp, _problem

pytestmark = pytest.mark.gpu


def _u(widths, layers, stats, scales, T, p, Y, n):
    import torch
    from paper_2312_05800_gb300 import binding
    net = _mlp(widths, layers, stats)
    binding.chem_mlp_set_fp8_scales(net, scales)
    u = torch.zeros((n, 32), dtype=torch.float32, device="cuda")
    binding.chem_mlp_forward_prec(net, binding.CHEM_PREC_FP8, n, T.shape[0], to_dev(T), to_dev(p), to_dev(Y), u, 32)
    torch.cuda.synchronize()
    assert net.error() == 0
    net.free()
    return u.cpu().numpy()


@pytest.mark.parametrize("n,hidden", [(1, (16, 48, 32)), (33, (208, 240, 16)), (300, (224, 416, 48)),
                                      (257, (464, 272, 96))])
def test_pair_stores_match_element_stores(n, hidden):
    mech, T, p, Y, widths, layers, stats, scales = _problem(300, hidden=hidden)
    want = layers
    wide = list(widths)
    for l in (0, 1):                                    # the layers whose outputs are E4M3
        W, b = want[l]
        W2, b2 = want[l + 1]
        want = list(want)
        want[l] = (np.vstack([W, np.zeros((8, W.shape[1]))]), np.concatenate([b, np.zeros(8)]))
        want[l + 1] = (np.hstack([W2, np.zeros((W2.shape[0], 8))]), b2)
        wide[l + 1] += 8
    a = _u(widths, layers, stats, scales, T, p, Y, n)
    b = _u(wide, want, stats, scales, T, p, Y, n)
    assert np.array_equal(a, b)
