"""The bias gradient of the convolutions on gradients that nearly cancel: smooth over the grid with a sum far
below the sum of magnitudes, as the gradient of the loss is.  Summed over runs of neighbouring rows such a
field loses digits that the sum over rows from everywhere keeps, so the order of the sum is part of the
result: block b of G adds 64-voxel row segments b, b + G, ... in 16 chains, the chains, then the blocks."""
import numpy as np
import pytest

from oracle import conv3d as C

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_1410_4054_gb300 import pk  # noqa: E402

DEV = "cuda:0"


def smooth(dims, seed):
    """[D, H, W, 16] BF16 values, one warm half and one cold half along each axis, sum near zero."""
    r = np.random.default_rng(seed)
    z, y, x = (np.linspace(0.0, 1.0, m) if m > 1 else np.zeros(1) for m in dims)
    a = r.uniform(0.5, 1.5, 16)
    f = a * (np.cos(np.pi * z)[:, None, None, None] + 0.5 * np.cos(np.pi * y)[None, :, None, None]
             + 0.1 * np.cos(2.0 * np.pi * x)[None, None, :, None]) + 1e-3 * r.standard_normal(dims + (16,))
    f -= f.mean(axis=(0, 1, 2))
    return C.bf16(1e-4 * f)


def in_order(g, blocks):
    """db in FP32, in the order above."""
    D, H, W, ch = g.shape
    nseg = (W + 63) // 64
    seg = np.zeros((D * H, nseg * 64, ch), np.float32)
    seg[:, :W] = g.reshape(D * H, W, ch)
    seg = seg.reshape(D * H * nseg, 4, 16, ch)
    block = np.zeros((blocks, ch), np.float32)
    for b in range(blocks):
        chain = np.zeros((16, ch), np.float32)
        for s in seg[b::blocks]:
            for k in range(4):
                chain += s[k]
        for i in range(16):
            block[b] += chain[i]
    out = np.zeros(ch, np.float32)
    for w in range(8):
        part = np.zeros(ch, np.float32)
        for b in range(w, blocks, 8):
            part += block[b]
        out += part
    return out


@pytest.mark.parametrize("dims", [(1, 1, 1), (1, 1, 65), (7, 9, 20), (18, 32, 39), (16, 41, 72), (33, 19, 28), (64, 64, 64)])
def test_bias_gradient_keeps_the_order_of_its_sum(dims):
    g = smooth(dims, sum(dims))
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    blocks = min(dims[0] * dims[1] * ((dims[2] + 63) // 64), sms, 256)
    G = torch.from_numpy(g.astype(np.float32)).to(DEV).to(torch.bfloat16).contiguous()
    X = torch.relu(torch.randn(dims + (16,), generator=torch.Generator(device=DEV).manual_seed(1), device=DEV)).to(torch.bfloat16)
    scratch = torch.zeros(pk.conv3d_wgrad_scratch_floats(dims), dtype=torch.float32, device=DEV)
    dW, db = torch.zeros(27, 16, 16, device=DEV), torch.zeros(16, device=DEV)
    pk.conv3d_wgrad(X, G, scratch, dW, db, dims)
    pk.conv3d_check()
    assert np.array_equal(db.cpu().numpy(), in_order(g.astype(np.float32), blocks))
