"""The row-block GEMV (five sequences and more on the CUDA cores) against
float64, at the edges of its split: row blocks of 4, 512-byte chunks of a
row, K slices of 4096 inputs over a cluster, groups of 8 sequences, and
inputs that do not allow 16-byte loads, both sides of the rule that cuts long
fp32 rows in two."""
import pytest
import torch

from paper_2605_27255_gb300 import capi

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [0, 1])
@pytest.mark.parametrize("mode,N,K", [(0, 1, 8), (0, 3, 264), (0, 613, 4096), (1, 153, 4104), (0, 2560, 9728),
                                      (1, 5, 12296), (0, 40003, 4104), (0, 5003, 2056), (1, 2501, 2056),
                                      (0, 4863, 2056)])
@pytest.mark.parametrize("B,off", [(5, 0), (8, 1), (9, 0), (17, 3)])
def test_row_block_gemv_matches_float64(dtype, mode, N, K, B, off):
    g = torch.Generator(device="cuda").manual_seed(N + K + B)
    W = (torch.randn(N * (1 + mode), K, device="cuda", generator=g) * 0.05).to([torch.float32, torch.bfloat16][dtype])
    xbuf = torch.randn(B * K + off, device="cuda", generator=g)
    x = xbuf[off:].view(B, K)  # off elements past a 16-byte boundary
    y = torch.full((B, N), float("nan"), device="cuda")
    capi.pipo_op_gemv(dtype, mode, W.data_ptr(), N, K, x.data_ptr(), B, y.data_ptr())
    torch.cuda.synchronize()
    ref = x.double() @ W.double().t()
    mag = x.double().abs() @ W.double().abs().t()
    # a lane's running sum over K / 32 inputs, then a tree: well under 2^-24 (K / 32 + 64) of the sum of magnitudes
    bound = 2.0 ** -24 * (K / 32 + 64) * mag
    if mode:
        gate, up = ref[:, 0::2], ref[:, 1::2]
        sig = torch.sigmoid(gate)
        # |d(silu)| <= 1.1, and the rounding of the two factors
        bound = 1.1 * bound[:, 0::2] * up.abs() + (gate * sig).abs() * bound[:, 1::2] + 2.0 ** -20 * (gate * sig * up).abs()
        ref = gate * sig * up
    assert ((y.double() - ref).abs() <= bound + 1e-30).all()


@pytest.mark.parametrize("K", [2048, 2560, 4096, 5120])
def test_fp32_sums_of_whole_rows_are_chains_of_k_over_256(K):
    """Rows that one warp sums alone (many rows) in fp32: no less accurate than
    32 lanes that each add K / 256 sums of eight products (fused, in turn), then a
    tree.  2 %: the root mean square of 16000 rounding errors is known to
    1 / sqrt(2 x 16000) = 0.6 %."""
    g = torch.Generator(device="cuda").manual_seed(K)
    N, B = 40000, 8
    W = torch.randn(N, K, device="cuda", generator=g) * 0.02
    x = torch.randn(B, K, device="cuda", generator=g)
    y = torch.empty(B, N, device="cuda")
    capi.pipo_op_gemv(0, 0, W.data_ptr(), N, K, x.data_ptr(), B, y.data_ptr())
    torch.cuda.synchronize()
    ref = x.double() @ W.double().t()
    got = ((y.double() - ref).norm() / ref.norm()).item()
    n = 2000
    w8, x8 = W[:n].double().view(n, 1, K // 256, 32, 8), x.double().view(1, B, K // 256, 32, 8)
    s = torch.zeros(n, B, 32, device="cuda")
    for i in range(K // 256):
        p = torch.zeros_like(s)
        for j in range(8):
            p = (w8[:, :, i, :, j] * x8[:, :, i, :, j] + p.double()).float()
        s = s + p
    while s.shape[-1] > 1:
        s = s[..., ::2] + s[..., 1::2]
    r = ref.t()[:n]
    want = ((s[..., 0].double() - r).norm() / r.norm()).item()
    assert got <= 1.02 * want, (got, want)
