"""The FP32 full properties pass with its species-pair sums on the tensor cores, at the sizes where its
tiling can go wrong: species counts at the edges of the padded contraction length (16, 32, 48, 64) and of
the 8-species chunks, the largest it takes (56) and the first it does not (57, the pair loop); cell
counts at the edges of the 128-cell tile and past one tile per resident CTA; cells of one dominant species,
whose diffusivity sums run over traces. FP32 tolerance 1e-5 relative to the FP64 oracle on the same
FP32-rounded state, as for the other FP32 properties."""
import numpy as np
import pytest

from paper_2312_05800_gb300 import synth
from tests.gpu_util import h_scale, to_dev

pytestmark = pytest.mark.gpu


def _mech(N):
    return synth.make_mech("t%d" % N, N, 3 * N, 2, 3, ["C", "H", "O", "N"], 4000 + N)


def _state(m, n, ld, seed):
    rng = np.random.default_rng(seed)
    T, p, Y = np.zeros(ld), np.zeros(ld), np.zeros((m.N, ld))
    T[:n] = rng.uniform(300.0, 2500.0, n)
    p[:n] = synth.P_ATM * rng.uniform(0.5, 20.0, n)
    Y[:, :n] = rng.dirichlet(np.full(m.N, 0.5), size=n).T
    for q, eps in enumerate((1e-1, 1e-2, 1.5e-3, 1e-3, 1e-4, 1e-6)):    # nearly alone, both sides of the X = 0.999 line
        for i in range(q, n, 61):
            k = (i // 61) % m.N
            Y[:, i] *= eps
            Y[k, i] += 1.0 - eps
    return (np.asarray(a, np.float32).astype(np.float64) for a in (T, p, Y))


@pytest.mark.parametrize("N,n", [(16, 129), (17, 127), (30, 1), (32, 40000), (33, 128), (48, 257), (49, 20011),
                                 (56, 300), (57, 130)])
def test_species_and_tile_edges(oracle, N, n):
    import torch
    from paper_2312_05800_gb300 import binding
    m = _mech(N)
    dm = binding.Mech(m)
    ld = synth.padded_ld(n) + 4
    T, p, Y = _state(m, n, ld, N)
    keep = np.unique(np.concatenate([np.arange(min(n, 400)), np.arange(max(0, n - 400), n)]))
    cp, h, mu, lam, Dk = oracle.props(m, T[keep], p[keep], np.ascontiguousarray(Y[:, keep]))
    hs = h_scale(oracle, m, T[keep], Y[:, keep], keep.size)
    for dtype, td in ((binding.CHEM_F32, torch.float32), (binding.CHEM_F64_IN_F32, torch.float64)):
        out = torch.full((4 + m.N, ld), float("nan"), dtype=torch.float32, device="cuda")
        binding.props_eval(dm, n, ld, dtype, to_dev(T, td), to_dev(p, td), to_dev(Y, td), out[0], out[1], out[2],
                           out[3], out[4:])
        torch.cuda.synchronize()
        got = out.double().cpu().numpy()
        assert np.isnan(got[:, n:]).all()
        got = got[:, keep]
        for a, b, scale in ((got[0], cp, np.abs(cp)), (got[1], h, hs), (got[2], mu, mu), (got[3], lam, lam),
                            (got[4:], Dk, Dk)):
            assert np.all(np.abs(a - b) <= 1e-5 * scale), (dtype, float((np.abs(a - b) / scale).max()))
