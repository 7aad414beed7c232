"""Convolution kernels of the warm-start network on integer-valued tensors:
every sum is an integer below 2^24, exact in FP32 in any order, so the
kernels must give the FP64 reference exactly (the forward result rounded
once to BF16).  Sizes: one plane, one voxel row, tiles with ragged edges,
z segments longer than the ring of accumulators (its window of three planes
wraps), every split of the channels, slices of one block, channel slices of
wider buffers.  Bias gradient and ReLU mask on both sides of their rules.
"""
import pytest

pytestmark = pytest.mark.gpu


def _ints(gen, shape, hi, dtype):
    import torch
    return torch.randint(-hi, hi + 1, shape, generator=gen, device="cuda").to(dtype)


def _shift(v, t, periodic):
    """v[n, z + dz, y + dy, x + dx] with zeros outside in x (and in y, z unless periodic)"""
    import torch
    for dim, d in ((3, t % 3 - 1), (2, t // 3 % 3 - 1), (1, t // 9 - 1)):
        if d == 0:
            continue
        v = torch.roll(v, -d, dim)
        if dim == 3 or not periodic:
            idx = [slice(None)] * 5
            idx[dim] = slice(-1, None) if d > 0 else slice(0, 1)
            v[tuple(idx)] = 0
    return v


FORWARD = [
    (16, 16, (1, 1, 1, 1), 1), (48, 16, (1, 2, 16, 8), 1), (16, 48, (2, 1, 17, 9), 1), (32, 64, (1, 3, 15, 7), 0),
    (32, 96, (1, 5, 33, 17), 1), (64, 16, (3, 4, 5, 23), 1), (64, 32, (1, 9, 18, 8), 0), (16, 112, (1, 6, 16, 16), 1),
    (16, 64, (1, 7, 256, 80), 1), (16, 48, (1, 13, 250, 77), 0), (48, 16, (1, 18, 256, 80), 1),
    # weights that stream: split and whole output channels, one to four channel chunks
    (64, 64, (1, 4, 12, 12), 1), (96, 32, (1, 4, 12, 12), 0), (128, 128, (1, 1, 1, 1), 1), (128, 128, (1, 2, 19, 9), 1),
    (192, 64, (2, 2, 7, 9), 0), (80, 48, (1, 3, 17, 8), 1), (96, 32, (1, 16, 40, 40), 1), (64, 256, (1, 2, 6, 6), 1),
    (32, 160, (1, 3, 33, 17), 0)]


@pytest.mark.parametrize("ci,co,shape,periodic", FORWARD)
def test_forward_exact(cuda_lib, ci, co, shape, periodic):
    import torch

    from paper_1410_1914_gb300 import warmstart as W
    gen = torch.Generator(device="cuda").manual_seed(ci * 1000 + co)
    N, D, H, X = shape
    xs, xo, ys, yo = ci + 16, 8, co + 24, 16  # channel slices of wider buffers
    xb = _ints(gen, (N, D, H, X, xs), 2, torch.bfloat16)
    w = _ints(gen, (27, co, ci), 2, torch.bfloat16)
    b = _ints(gen, (co,), 9, torch.float32)
    yb = torch.full((N, D, H, X, ys), 7.0, dtype=torch.bfloat16, device="cuda")
    W._call("cl_nn_conv3d", W._p(xb), W._p(w), W._p(b), W._p(yb), N, D, H, X, ci, co, xs, xo, ys, yo, 1, periodic, None)
    W._call("cl_nn_check", None)
    x = xb[..., xo:xo + ci].float()
    ref = b.expand(N, D, H, X, co).clone()
    for t in range(27):
        ref += _shift(x.clone(), t, periodic) @ w[t].float().T
    ref = ref.clamp(min=0).to(torch.bfloat16)
    assert torch.equal(yb[..., yo:yo + co], ref)
    assert bool((yb[..., :yo] == 7).all()) and bool((yb[..., yo + co:] == 7).all())


@pytest.mark.parametrize("ci,co,shape,periodic", [
    (16, 16, (1, 1, 1, 1), 1), (48, 16, (1, 2, 16, 8), 1), (64, 32, (2, 3, 17, 9), 0), (80, 16, (1, 4, 15, 7), 1),
    (128, 16, (1, 2, 5, 9), 1), (144, 48, (1, 3, 18, 10), 1), (256, 128, (1, 2, 4, 4), 1), (16, 112, (1, 3, 6, 6), 0),
    (48, 16, (1, 19, 40, 40), 1), (16, 16, (3, 21, 33, 25), 0)])
def test_weight_gradient_exact(cuda_lib, ci, co, shape, periodic):
    import torch

    from paper_1410_1914_gb300 import warmstart as W
    gen = torch.Generator(device="cuda").manual_seed(ci * 1000 + co + 1)
    N, D, H, X = shape
    xs, xo, ys, yo = ci + 8, 8, co + 24, 16
    xb = _ints(gen, (N, D, H, X, xs), 2, torch.bfloat16)
    gb = _ints(gen, (N, D, H, X, ys), 2, torch.bfloat16)
    ws = torch.empty(W._lib().cl_nn_wgrad_workspace(N, D, H, X, ci, co) // 4, dtype=torch.float32, device="cuda")
    dw = torch.empty(27, co, ci, dtype=torch.float32, device="cuda")
    W._call("cl_nn_conv3d_wgrad", W._p(xb), W._p(gb), W._p(ws), W._p(dw), N, D, H, X, ci, co, xs, xo, ys, yo, periodic,
            None)
    W._call("cl_nn_check", None)
    x, g = xb[..., xo:xo + ci].float(), gb[..., yo:yo + co].double().reshape(-1, co)
    for t in range(27):
        ref = g.T @ _shift(x.clone(), t, periodic).double().reshape(-1, ci)
        assert torch.equal(dw[t].double(), ref), t


# (voxels, channels, stride, offset, elements before the tensor's start): 16384 voxels is
# where the cluster takes over; odd strides, offsets, counts and bases keep the element kernels
@pytest.mark.parametrize("M,C,stride,off,skip", [
    (1, 8, 8, 0, 0), (16383, 16, 16, 0, 0), (16384, 16, 16, 0, 0), (50001, 24, 40, 8, 0), (20000, 12, 16, 0, 0),
    (20000, 16, 20, 0, 0), (20000, 16, 24, 4, 0), (20000, 16, 16, 0, 1), (20000, 8, 8, 0, 8)])
def test_bias_gradient_and_relu_mask(cuda_lib, M, C, stride, off, skip):
    import torch

    from paper_1410_1914_gb300 import warmstart as W
    gen = torch.Generator(device="cuda").manual_seed(M + C + skip)
    dy = _ints(gen, (M * stride + skip,), 3, torch.bfloat16)[skip:]
    y = _ints(gen, (M * stride + skip,), 1, torch.bfloat16)[skip:]
    y[:: 97] = float("nan")
    y[1:: 89] = -0.0
    db = torch.empty(C, dtype=torch.float32, device="cuda")
    W._call("cl_nn_bias_grad", W._p(dy), M, C, stride, off, W._p(db), None)
    cols = dy.view(M, stride)[:, off:off + C]
    assert torch.equal(db.double(), cols.double().sum(0))
    exp = dy.clone()
    part = exp.view(M, stride)[:, off:off + C]
    part[~(y.view(M, stride)[:, off:off + C] > 0)] = 0
    W._call("cl_nn_relu_bwd", W._p(y), W._p(dy), M, C, stride, off, None)
    torch.cuda.synchronize()
    assert torch.equal(dy, exp)


def test_calls_outside_the_kernels_range(cuda_lib):
    """Channel counts without a tensor-core weight gradient have a workspace
    size, and an empty box is refused."""
    import torch

    from paper_1410_1914_gb300 import _lib as L
    from paper_1410_1914_gb300 import warmstart as W
    assert W._lib().cl_nn_wgrad_workspace(1, 2, 3, 4, 16, 8) > 0
    assert W._lib().cl_nn_wgrad_workspace(1, 2, 3, 4, 16, 256) > 0
    t = torch.zeros(27 * 16 * 16, device="cuda")
    for call in ((0, 2, 3, 4, 16, 16), (1, 2, 3, 0, 16, 16), (1, 2, 3, 4, 16, 8)):
        with pytest.raises(L.ClError):
            W._call("cl_nn_conv3d_wgrad", W._p(t), W._p(t), W._p(t), W._p(t), *call, 16, 0, 16, 0, 1, None)
