"""Training gradients where the weight-gradient launch and the products with N-major weights change: batches
that end inside a 64-row k-block, widths below, at and past their 64- and 128-column tiles, multiples of 8
that take the element-store epilogue (not of 16). Against the oracle's FP64 backward, each element within
8 standard deviations of the device's BF16 rounding (tests/grad_bounds.py). The loss gradient is the one
the device stores, bf16(1 / B) with the residual's sign, so it carries no error of its own."""
import numpy as np
import pytest

from oracle import ann as A
from oracle import mlp as M
from paper_2312_05800_gb300 import synth
from tests.gpu_util import dev_mech, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,hidden", [(8, (8, 16, 24)), (72, (104, 56, 24)), (136, (256, 128, 64)), (264, (272, 136, 264))])
def test_gradients_at_tile_edges(B, hidden):
    import torch
    from paper_2312_05800_gb300 import binding
    from tests.grad_bounds import check, gradients_with_sigma, separated_targets
    mech = synth.get_mech("c2")
    n = 512
    T, p, Y = synth.states_profiles(mech, n, 11, synth.padded_ld(n))
    widths = [mech.N + 2, *hidden, mech.N - 1]
    layers = synth.mlp_layers(widths, 3011)
    x = M.features(T[:n], p[:n], Y[:, :n])
    mu_x, sd_x = M.zscore_stats(x)
    rng = np.random.default_rng(12)
    mu_u = rng.uniform(-1e-5, 1e-5, mech.N - 1)
    sd_u = 10.0 ** rng.uniform(-6, -3, mech.N - 1)
    z = ((x - mu_x) / sd_x)[:B]
    uq = A.network(layers, np.asarray(z, np.float32).astype(np.float64), round_bf16=True)
    target = separated_targets(uq, rng)
    Y1 = Y.copy()
    Y1[A.out_species(mech), :B] += (target * sd_u + mu_u).T
    net = binding.Mlp(dev_mech("c2"), hidden=list(hidden), max_batch=B)
    net.set_params(synth.flatten_layers(layers))
    net.set_norm(mu_x, sd_x, mu_u, sd_u)
    loss = torch.zeros(4, dtype=torch.float32, device="cuda")
    binding.mlp_train_step(net, B, None, T.shape[0], to_dev(T), to_dev(p), to_dev(Y), to_dev(Y1), 0.0, loss)
    torch.cuda.synchronize()
    assert net.error() == 0
    g = synth.unflatten(net.get_grads(), widths)
    step = float(torch.tensor(np.float32(1) / np.float32(B)).bfloat16())
    lo, go, sig, min_res = gradients_with_sigma(layers, z, target, uq, dout=np.sign(uq - target) * step)
    assert min_res >= 0.4 * np.sqrt(np.mean(uq ** 2))
    for l in range(4):
        for j, key in ((0, "W"), (1, "b")):
            check(g[l][j], go[l][j], sig[l][j], "layer %d d%s" % (l + 1, key))
    net.free()
