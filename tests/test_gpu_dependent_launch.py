"""Products launched while the one before them still runs (at most two tiles per SM) and those that are not:
a chain of dense layers, each reading the one before, has the bits of the same chain with the device
synchronised after every layer, at row counts on both sides of the rule and for a ragged one."""
import pytest

pytestmark = pytest.mark.gpu


def _chain(x, ws, bs, sync):
    import torch
    from paper_2312_05800_gb300 import binding
    err = torch.zeros(4, dtype=torch.int32, device="cuda")
    ys = [torch.full((x.shape[0], w.shape[0]), float("nan"), dtype=torch.bfloat16, device="cuda") for w in ws]
    for w, b, y in zip(ws, bs, ys):                   # nothing launched between the products
        (M, K), N = x.shape, w.shape[0]
        rc = binding.lib().chem_dense_bf16(M, N, K, x.data_ptr(), K, w.data_ptr(), K, b.data_ptr(), 1, y.data_ptr(), N,
                                           0, err.data_ptr(), torch.cuda.current_stream().cuda_stream)
        assert rc == 0
        if sync:
            torch.cuda.synchronize()
        x = y
    torch.cuda.synchronize()
    assert int(err[0]) == 0
    return x


@pytest.mark.parametrize("M", [1, 1000, 4096, 128 * 304 // 4, 128 * 304 // 4 + 1, 128 * 400])
def test_chain_of_products(M):
    import torch
    g = torch.Generator(device="cuda")
    g.manual_seed(3)
    widths = [96, 800, 784, 800, 400, 32]
    x = torch.randn(M, widths[0], device="cuda", generator=g).bfloat16()
    ws = [(torch.randn(n, k, device="cuda", generator=g) / k ** 0.5).bfloat16() for k, n in zip(widths, widths[1:])]
    bs = [torch.randn(n, device="cuda", generator=g) for n in widths[1:]]
    want = _chain(x, ws, bs, True)
    assert bool(torch.isfinite(want.float()).all())
    for _ in range(3):
        assert torch.equal(_chain(x, ws, bs, False), want)
