"""The network's convolutions at the largest edges that it accepts (128 and 256: several tiles and
x segments a row, offsets of 2^28 and more elements), against FP64 on the GPU: forward and data
gradient on planes at both ends and in the middle, the weight gradient whole.  Bounds as in
test_gpu_nn.py: one BF16 rounding (2^-8) and FP32 sums."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sur():
    import __graft_entry__ as g
    g.build()
    from paper_2112_10059_gb300 import surrogate as s
    return s


def _planes(x, w, z0, z1):
    """FP64 convolution of x [B, D, D, D, C] with w [N, 27, C] at planes z0 .. z1 - 1."""
    import torch
    d = x.shape[1]
    pad = torch.zeros((x.shape[0], z1 - z0 + 2, d + 2, d + 2, x.shape[4]), dtype=torch.float64, device="cuda")
    lo, hi = max(z0 - 1, 0), min(z1 + 1, d)
    pad[:, lo - z0 + 1:hi - z0 + 1, 1:-1, 1:-1] = x[:, lo:hi].double()
    out = 0.0
    for tap in range(27):
        k, j, i = tap // 9, tap // 3 % 3, tap % 3
        out = out + pad[:, k:k + z1 - z0, j:j + d, i:i + d] @ w[:, tap].double().T
    return out


def _tensors(C, N, edge, batch, seed):
    import torch
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    x = torch.randn((batch, edge, edge, edge, C), device="cuda", generator=g).to(torch.bfloat16)
    w = (0.2 * torch.randn((N, 27, C), device="cuda", generator=g)).to(torch.bfloat16)
    return x, w, g


CASES = [(16, 16, 128, 2), (32, 32, 128, 1), (16, 16, 256, 1), (32, 16, 256, 1)]


@pytest.mark.parametrize("C,N,edge,batch", CASES)
@pytest.mark.parametrize("mode", [0, 1])
def test_convolution(sur, C, N, edge, batch, mode):
    import torch
    # mode 1: x is the gradient [.., N], the weights flipped and transposed
    x, w, _ = _tensors(N if mode else C, N, edge, batch, 41 + edge + mode)
    if mode:
        w = (0.2 * torch.randn((N, 27, C), device="cuda")).to(torch.bfloat16)
    wr = w.flip(1).permute(2, 1, 0).contiguous() if mode else w
    out = sur.conv3d(mode, C, N, edge, batch, x.reshape(-1), w.float().reshape(-1), relu=False)
    out = out.reshape(batch, edge, edge, edge, C if mode else N)
    for z0, z1 in ((0, 2), (edge // 2 - 1, edge // 2 + 2), (edge - 2, edge)):
        ref = _planes(x, wr, z0, z1)
        got = out[:, z0:z1].double()
        bad = (got - ref).abs() > 2.0 ** -8 * ref.abs() + 2e-5 * ref.abs().max()
        assert not bool(bad.any()), (z0, int(bad.sum()))


@pytest.mark.parametrize("C,N,edge,batch", CASES)
def test_weight_gradient(sur, C, N, edge, batch):
    import torch
    x, _, g = _tensors(C, N, edge, batch, 61 + edge)
    dz = torch.randn((batch, edge, edge, edge, N), device="cuda", generator=g).to(torch.bfloat16)
    out = sur.conv3d_wgrad(C, N, edge, batch, x.reshape(-1), dz.reshape(-1)).double().cpu()
    ref = torch.zeros((N, 27, C), dtype=torch.float64, device="cuda")
    sl = lambda o, n: (slice(max(0, -o), n - max(0, o)), slice(max(0, o), n - max(0, -o)))   # of dz, of x
    for tap in range(27):
        oz, oy, ox = tap // 9 - 1, tap // 3 % 3 - 1, tap % 3 - 1
        (az, bz), (ay, by), (ax, bx) = sl(oz, edge), sl(oy, edge), sl(ox, edge)
        for b in range(batch):
            a = dz[b, az, ay, ax].reshape(-1, N).double()
            ref[:, tap] += a.T @ x[b, bz, by, bx].reshape(-1, C).double()
    ref = torch.cat([ref.reshape(-1), dz.reshape(-1, N).double().sum(dim=0)]).cpu()
    # the steps of a CTA's sums, each rounded towards zero (2^-23 of a partial sum of at most 5 sigma)
    voxels = batch * edge ** 3
    steps = -(-voxels // (64 * 152)) * 4
    assert float((out - ref).abs().max()) <= steps * 2.0 ** -23 * 5 * np.sqrt(voxels)
