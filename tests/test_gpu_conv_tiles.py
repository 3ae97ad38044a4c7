"""The convolution kernels at the edges of their tiles and runs (8 x 16 columns and z runs forward,
64-voxel segments and 10-row runs in the weight gradient), the fused Adam step and the network's
input with and without its stash."""
import numpy as np
import pytest

from oracle import conv3d as C

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_1410_4054_gb300 import pk  # noqa: E402

DEV = "cuda:0"


def dev(a, dtype=torch.bfloat16):
    return torch.from_numpy(np.asarray(a, dtype=np.float32)).to(DEV).to(dtype).contiguous()


def host(t):
    return t.float().cpu().numpy().astype(np.float64)


# one voxel; one row past a segment; a run of one row per plane; more planes than accumulator slots in
# one column; more than one run of 10 rows per plane and block; several blocks of the grid with one unit
EDGES = [(1, 1, 1), (1, 1, 65), (3, 1, 64), (40, 3, 7), (1, 300, 2), (21, 23, 66), (70, 17, 9)]


@pytest.mark.parametrize("dims", EDGES)
def test_convolutions_at_tile_edges(dims):
    r = np.random.default_rng(sum(dims))
    x = C.bf16(np.maximum(r.standard_normal(dims + (16,)), 0.0))
    g = C.bf16(r.standard_normal(dims + (16,)))
    w = C.bf16(r.standard_normal((27, 16, 16)) * 0.1)
    b = r.standard_normal(16).astype(np.float32).astype(np.float64)
    X, G, Wt = dev(x), dev(g), dev(w)
    Yf = torch.zeros(dims, dtype=torch.float32, device=DEV)
    pk.conv3d_fwd(X, Wt, dev(b, torch.float32), Yf, dims, relu=False, out_f32=True)
    Y = torch.zeros(dims + (16,), dtype=torch.bfloat16, device=DEV)
    pk.conv3d_fwd(X, Wt, dev(b, torch.float32), Y, dims, relu=True)
    scratch = torch.zeros(pk.conv3d_wgrad_scratch_floats(dims), dtype=torch.float32, device=DEV)
    dW, db = torch.zeros(27, 16, 16, device=DEV), torch.zeros(16, device=DEV)
    pk.conv3d_wgrad(X, G, scratch, dW, db, dims)
    pk.conv3d_check()
    # sums of k FP32 terms, products exact: within k roundings (and truncations) of 2^-23 of the sum
    # of the magnitudes, whatever the order
    ref, mag = C.conv3d(x, w, b), C.conv3d(np.abs(x), np.abs(w), np.abs(b))
    assert np.all(np.abs(host(Yf) - ref[..., 0]) <= 440 * 2.0 ** -23 * mag[..., 0])
    y = np.maximum(ref, 0.0)
    assert np.all(np.abs(host(Y) - y) <= 2.0 ** -8 * y + 440 * 2.0 ** -22 * mag)
    n = int(np.prod(dims))
    dW_ref, dW_mag = C.conv3d_wgrad(x, g), C.conv3d_wgrad(np.abs(x), np.abs(g))
    db_ref, db_mag = g.sum(axis=(0, 1, 2)), np.abs(g).sum(axis=(0, 1, 2))
    assert np.all(np.abs(host(dW) - dW_ref) <= (n + 300) * 2.0 ** -23 * dW_mag)
    assert np.all(np.abs(host(db) - db_ref) <= (n + 300) * 2.0 ** -23 * db_mag)


def test_fused_adam_step_equals_the_single_steps():
    sizes = [27 * 256, 16, 27 * 256, 1, 257]

    def state():
        q = np.random.default_rng(4)
        return [[dev(q.standard_normal(k) ** (2 if j == 3 else 1), torch.float32) for k in sizes] for j in range(4)]

    one, many = state(), state()
    h1 = [torch.zeros(k, dtype=torch.bfloat16, device=DEV) for k in sizes]
    h2 = [torch.zeros(k, dtype=torch.bfloat16, device=DEV) for k in sizes]
    flipped = [torch.zeros(k, dtype=torch.bfloat16, device=DEV) if k == 27 * 256 else None for k in sizes]
    for k in range(len(sizes)):
        pk.adam_step(one[0][k], one[1][k], one[2][k], one[3][k], 1e-3, 5, p_bf16=h1[k])
    pk.adam_step_many(many[0], many[1], many[2], many[3], 1e-3, 5, p_bf16=h2, flipped=flipped)
    for a, b in zip(one[0] + one[2] + one[3] + h1, many[0] + many[2] + many[3] + h2):
        assert torch.equal(a, b)
    for k, f in enumerate(flipped):
        if f is not None:
            ref = torch.empty_like(f)
            pk.conv3d_flip(h1[k], ref)
            assert torch.equal(f, ref)
    too_many = [many[0][3]] * 17
    with pytest.raises(pk.PkError):
        pk.adam_step_many(too_many, too_many, too_many, too_many, 1e-3, 5)


@pytest.mark.parametrize("n", [1, 255, 4097])
def test_network_input_does_not_depend_on_the_alignment(n):
    r = np.random.default_rng(n)
    rp, ci, va = [0], [], []
    for i in range(n):
        cols = sorted(set(int(c) for c in r.integers(0, n, 5)) | ({i} if i % 7 else set()))
        ci += cols
        va += list(r.standard_normal(len(cols)))
        rp.append(len(ci))
    A = pk.CSRMatrix(torch.tensor(rp, dtype=torch.int32, device=DEV), torch.tensor(ci, dtype=torch.int32, device=DEV),
                     torch.tensor(va, dtype=torch.float64, device=DEV))
    x1, x2, b = (torch.from_numpy(r.standard_normal(n)).to(DEV) for _ in range(3))
    out = []
    for off in (0, 1):  # 16-byte aligned (the stash is used), then 2-byte aligned
        X = torch.zeros(16 * n + 8, dtype=torch.bfloat16, device=DEV)[off:off + 16 * n]
        scales = torch.zeros(3, dtype=torch.float64, device=DEV)
        scratch = torch.zeros(pk.warmstart_scratch_doubles(), dtype=torch.float64, device=DEV)
        pk.warmstart_input(A, x1, x2, b, X, scales, scratch)
        out.append((X.clone(), scales))
    torch.cuda.synchronize()
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
    assert bool((out[0][0].view(n, 16)[:, 3:] == 0).all())
