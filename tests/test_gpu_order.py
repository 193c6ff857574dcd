"""GPU: calls on one stream take effect in order.  Every kernel is launched while its predecessor still runs, so an operand
that the call before produces may only be read behind the kernel's wait for it; the kernels of one forward read the
model's own parameters earlier, but not before work enqueued ahead of the forward has finished."""
import numpy as np
import pytest
import torch

from ivit_inputs import Scale
from ivit_inputs.gen import _Ids, dyadic, make_block, make_block_input, make_vit, make_image, scale_channels
from oracle import api as O

pytestmark = pytest.mark.gpu


def _g():
    import gpu_util
    return gpu_util


def rand_i8(rng, shape, std=32):
    return np.clip(np.rint(rng.standard_normal(shape) * std), -128, 127).astype(np.int8)


def gather(c, src, index, out):
    """ivit_gather_rows into a tensor of the caller's."""
    rc = c.lib.ivit_gather_rows(c.h, src.data_ptr(), src.stride(0), index.data_ptr(), index.numel(), src.shape[1],
                                out.data_ptr(), out.stride(0))
    assert rc == 0


# one small tile per SM / the persistent kernel
@pytest.mark.parametrize("Ma,Nb,K", [(128, 128, 4096), (200, 196, 48), (4096, 2048, 1024)])
def test_matmul_of_one_batch_waits_for_both_operands(Ma, Nb, K):
    """A and B are outputs of the two calls before, over buffers that held other values."""
    g = _g()
    c = g.ctx()
    rng = np.random.default_rng(Ma + Nb + K)
    X, Y = rand_i8(rng, (Ma, 512)), rand_i8(rng, (Nb, 512))
    W = rand_i8(rng, (K, 512))
    s1, s2 = Scale(*dyadic(30.0 / (np.sqrt(512) * 1024))), Scale(*dyadic(30.0 / (np.sqrt(K) * 900)))
    ds1, ds2 = g.binding.DevScale(s1, "cuda"), g.binding.DevScale(s2, "cuda")
    A, B = O.linear(X, W, None, s1), O.linear(Y, W, None, s1)
    want = O.matmul(A[None], B[None], True, s2)
    dX, dY, dW = g.dev(X), g.dev(Y), g.dev(W)
    for k in range(5):
        dA, dB = (g.dev(np.full((n, K), 7 + k, np.int8)) for n in (Ma, Nb))
        dC = g.dev(np.zeros((1, Ma, Nb), np.int8))
        torch.cuda.synchronize()
        c.linear(dX, dW, None, ds1, out=dA)
        c.linear(dY, dW, None, ds1, out=dB)
        c.matmul(dA[None], dB[None], True, ds2, out=dC)
        g.assert_equal(g.host(dC), want, f"matmul {k}")
    assert c.poll_status() == 0


@pytest.mark.parametrize("M,N,K", [(64, 256, 512), (9000, 512, 512)])
def test_linear_parameters_may_come_from_the_call_before(M, N, K):
    """W, then bias, then the per-channel scale written by the library call right in front of the Dense layer."""
    g = _g()
    c = g.ctx()
    rng = np.random.default_rng(M + N)
    A, W, W0 = rand_i8(rng, (M, K)), rand_i8(rng, (N, K)), rand_i8(rng, (N, 4096))
    one = np.zeros((1, 4096), np.int8)
    one[0, :64] = 1
    scale = scale_channels(rng.uniform(20, 60, N) / (np.sqrt(K) * 1024))
    flat = Scale(*dyadic(0.5))
    bias = O.linear(one, W0, None, flat, out_dtype=O.I32)[0]
    perm = rng.permutation(N).astype(np.int32)
    dA, dW, dW0, done, dperm = g.dev(A), g.dev(W), g.dev(W0), g.dev(one), torch.from_numpy(perm).cuda()
    ds, dflat = g.binding.DevScale(scale, "cuda"), g.binding.DevScale(flat, "cuda")
    # the multipliers as rows of bytes, brought to their place by a row gather
    mult = np.ascontiguousarray(scale.mult).astype(np.int32)
    src = torch.from_numpy(mult.view(np.int8).reshape(N // 4, 16)[::-1].copy()).cuda()
    back = torch.arange(N // 4 - 1, -1, -1, dtype=torch.int32, device="cuda")
    late = g.binding.DevScale(scale, "cuda")
    for k in range(5):
        w, b = g.dev(np.full((N, K), 5 + k, np.int8)), torch.full((1, N), 99 + k, dtype=torch.int32, device="cuda")
        late.mult_t.fill_(1 << 30)
        torch.cuda.synchronize()
        gather(c, dW, dperm, w)
        got = c.linear(dA, w, None, ds)
        g.assert_equal(g.host(got), O.linear(A, W[perm], None, scale), f"W {k}")
        c.linear(done, dW0, None, dflat, out=b, out_dtype=g.binding.I32)
        got = c.linear(dA, dW, b[0], ds)
        g.assert_equal(g.host(got), O.linear(A, W, bias, scale), f"bias {k}")
        gather(c, src, back, late.mult_t.view(torch.int8).view(N // 4, 16))
        got = c.linear(dA, dW, None, late)
        g.assert_equal(g.host(got), O.linear(A, W, None, scale), f"scale {k}")
    assert c.poll_status() == 0


@pytest.mark.parametrize("rows,C", [(197, 384), (5000, 384), (300, 1536), (200, 640)])
def test_layernorm_constants_may_come_from_the_call_before(rows, C):
    g = _g()
    c = g.ctx()
    rng = np.random.default_rng(rows + C)
    X, W0 = rand_i8(rng, (rows, C)), rand_i8(rng, (C, 4096))
    one = np.zeros((1, 4096), np.int8)
    one[0, 0] = 1
    flat = Scale(*dyadic(0.25))
    beta = O.linear(one, W0, None, flat, out_dtype=O.I32)[0]
    gamma = scale_channels(rng.uniform(0.8, 1.2, C) * 32.0 * np.sqrt(C) / 2.0 ** 20)
    dX, dW0, done = g.dev(X), g.dev(W0), g.dev(one)
    dgamma, dflat = g.binding.DevScale(gamma, "cuda"), g.binding.DevScale(flat, "cuda")
    want = O.layernorm(X, gamma, beta)
    for k in range(5):
        b = torch.full((1, C), 40 + k, dtype=torch.int32, device="cuda")
        torch.cuda.synchronize()
        c.linear(done, dW0, None, dflat, out=b, out_dtype=g.binding.I32)
        got = c.layernorm(dX, dgamma, b[0])
        g.assert_equal(g.host(got), want, f"layernorm {k}")
    assert c.poll_status() == 0


@pytest.mark.parametrize("B,T,D", [(1, 200, 48), (1, 196, 80), (2, 200, 48)])
def test_unfused_attention_of_one_head(B, T, D):
    """A head width that the fused kernels do not have: with one image and one head the keys are the second operand of a
    single product, and the block's QKV layer writes them right before it."""
    g = _g()
    c = g.ctx()
    blk = make_block(_Ids(400 + T + D), 1, B, T, D, 1, 4 * D)
    dblk = g.binding.DeviceBlock(blk, "cuda")
    for k in range(5):
        X = make_block_input(20 + k, B, T, D)
        dX, ws = torch.from_numpy(X).cuda(), dblk.workspace().fill_(k)
        torch.cuda.synchronize()
        Y = c.block_forward(dblk, dX, workspace=ws)
        g.assert_equal(g.host(Y), O.block_forward(blk, X), f"block {k}")
    assert c.poll_status() == 0


def test_forwards_see_parameters_written_by_the_call_before():
    """A weight of a block (of the first and of the only image) and of a model, brought to its place by the call right in
    front of the forward."""
    g = _g()
    c = g.ctx()
    blk = make_block(_Ids(77), 1, 1, 197, 192, 3, 768)
    X = make_block_input(3, 1, 197, 192)
    dblk, dX = g.binding.DeviceBlock(blk, "cuda"), torch.from_numpy(X).cuda()
    want = O.block_forward(blk, X)
    model, image = make_vit(5, 2, 64, 192, 3, 768, 2, patch=16, classes=16), make_image(5, 2, 64)
    dm, dimg = g.binding.DeviceVit(model, "cuda"), torch.from_numpy(image).cuda()
    want_m = O.vit_forward(model, image)

    def late(up, array):
        """The uploaded copy of `array` and what brings it back."""
        t = next(t for t in up.keep if torch.is_tensor(t) and t.dtype == torch.int8 and tuple(t.shape) == array.shape
                 and np.array_equal(t.cpu().numpy(), array))
        return t, t.clone(), torch.arange(t.shape[0], dtype=torch.int32, device="cuda")

    cases = [(dblk.up, blk.Wqkv), (dblk.up, blk.W2)]
    for k, (up, array) in enumerate(cases):
        t, good, idx = late(up, array)
        ws = dblk.workspace()
        t.fill_(1)
        torch.cuda.synchronize()
        gather(c, good, idx, t)
        Y = c.block_forward(dblk, dX, workspace=ws)
        g.assert_equal(g.host(Y), want, f"block {k}")
    for k, array in enumerate([model.Wpe, model.blocks[0].Wqkv, model.Whead]):
        t, good, idx = late(dm.up, array)
        ws = dm.workspace()
        t.fill_(1)
        torch.cuda.synchronize()
        gather(c, good, idx, t)
        logits = c.vit_forward(dm, dimg, workspace=ws)
        g.assert_equal(g.host(logits), want_m, f"model {k}")
    assert c.poll_status() == 0


def test_small_dense_layer_behind_a_long_kernel():
    """The limit of a kernel's own waits does not run while the kernel in front of it does: a CUDA-core product of some
    tenths of a second, then a layer of one wave that reads its output."""
    g = _g()
    c = g.ctx()
    n, K = 8192, 65536
    gen = torch.Generator(device="cuda").manual_seed(3)
    A, W = (torch.randint(-128, 128, (n, K), dtype=torch.int8, device="cuda", generator=gen) for _ in range(2))
    ds = g.binding.DevScale(Scale(*dyadic(30.0 / (np.sqrt(K) * 74.0 ** 2))), "cuda")
    rng = np.random.default_rng(4)
    W2 = rand_i8(rng, (128, n))
    s2 = Scale(*dyadic(30.0 / (np.sqrt(n) * 900)))
    dW2, ds2 = g.dev(W2), g.binding.DevScale(s2, "cuda")
    long_out = torch.zeros((n, n), dtype=torch.int8, device="cuda")
    torch.cuda.synchronize()
    c.set_gemm_engine(1)
    c.linear(A, W, None, ds, out=long_out)
    c.set_gemm_engine(0)
    got = g.host(c.linear(long_out[:64], dW2, None, ds2))
    assert c.poll_status() == 0
    x = g.host(long_out[:64])
    assert len(np.unique(x)) > 100
    g.assert_equal(got, O.linear(x, W2, None, s2), "layer behind a long kernel")
