"""Row operators inside the Dense kernels (I-LayerNorm after the projection / FC2, ShiftGELU after FC1):
the fused launch configuration, the one-kernel-per-operator configuration and the oracle give the same bytes, on
shapes that put one, several and many CTAs on a block of output rows, ragged last row blocks included."""
import numpy as np
import pytest
import torch

from ivit_inputs import make_config
from ivit_inputs.gen import _Ids, make_block, make_block_input
from oracle import api as O

pytestmark = pytest.mark.gpu


def _g():
    import gpu_util
    return gpu_util


@pytest.mark.parametrize("B,T,D,heads,H", [(1, 197, 192, 3, 768), (5, 197, 384, 6, 1536), (3, 50, 768, 12, 3072),
                                           (2, 130, 1024, 16, 4096), (40, 49, 96, 3, 384), (1, 9, 64, 1, 64),
                                           (17, 197, 384, 6, 1536)])
def test_block_fused_equals_unfused_equals_oracle(B, T, D, heads, H):
    g = _g()
    c = g.ctx()
    blk = make_block(_Ids(900 + B), 3, B, T, D, heads, H)
    X = make_block_input(900 + B, B, T, D)
    dblk = g.binding.DeviceBlock(blk, "cuda")
    dX = torch.from_numpy(X).cuda()
    want = O.block_forward(blk, X)
    c.block_forward(dblk, dX)          # builds the ShiftGELU table of this parameter set (a launch of its own)
    try:
        c.set_row_fusion(True)
        n0 = c.launch_count()
        fused = g.host(c.block_forward(dblk, dX))
        n_fused = c.launch_count() - n0
        c.set_row_fusion(False)
        n0 = c.launch_count()
        plain = g.host(c.block_forward(dblk, dX))
        n_plain = c.launch_count() - n0
        c.set_row_fusion(True)
        # repeated calls leave the arrival counters and ready flags at zero: same bytes again
        g.assert_equal(g.host(c.block_forward(dblk, dX)), want, "second fused call")
    finally:
        c.set_row_fusion(False)
    g.assert_equal(fused, want, "fused row operators vs oracle")
    g.assert_equal(plain, want, "separate row kernels vs oracle")
    # LayerNorm 2 and ShiftGELU ran inside the Dense kernels
    assert n_plain - n_fused == 2, (n_plain, n_fused)
    assert c.poll_status() == 0


def test_vit_forward_kernel_count_and_parity_with_fusion():
    """DeiT-S shapes, 3 blocks: LayerNorm 1 of blocks 1 and 2 comes out of the previous block's FC2 kernel."""
    g = _g()
    c = g.ctx()
    model, image = make_config(1, batch=5, depth=3)
    dm = g.binding.DeviceVit(model, "cuda")
    d_img = torch.from_numpy(image).cuda()
    tokens = torch.empty((5 * model.T, model.D), dtype=torch.int8, device="cuda")
    want_logits, want_tokens = O.vit_forward(model, image, return_tokens=True)
    c.vit_forward(dm, d_img)           # builds the ShiftGELU tables
    try:
        c.set_row_fusion(True)
        n0 = c.launch_count()
        logits = g.host(c.vit_forward(dm, d_img, tokens=tokens))
        n_fused = c.launch_count() - n0
        g.assert_equal(g.host(tokens), want_tokens, "tokens, fused")
        g.assert_equal(logits, want_logits, "logits, fused")
        c.set_row_fusion(False)
        n0 = c.launch_count()
        logits = g.host(c.vit_forward(dm, d_img, tokens=tokens))
        n_plain = c.launch_count() - n0
        g.assert_equal(g.host(tokens), want_tokens, "tokens, separate kernels")
        g.assert_equal(logits, want_logits, "logits, separate kernels")
    finally:
        c.set_row_fusion(False)
    # per block: LayerNorm 2 and ShiftGELU; between blocks: LayerNorm 1 of the next one
    assert n_plain - n_fused == 3 * 2 + 2, (n_plain, n_fused)
    assert c.poll_status() == 0


def test_linear_then_layernorm_tail_many_row_blocks_random_values():
    """The Dense + LayerNorm pair through the block entry point is covered above; here the arrival counters see
    a long run of row blocks (12 608 rows) at the benchmark's projection shape, twice in a row."""
    g = _g()
    c = g.ctx()
    blk = make_block(_Ids(77), 1, 64, 197, 384, 6, 1536)
    X = make_block_input(77, 64, 197, 384)
    dblk = g.binding.DeviceBlock(blk, "cuda")
    dX = torch.from_numpy(X).cuda()
    want = O.block_forward(blk, X)
    try:
        c.set_row_fusion(True)
        for k in range(2):
            g.assert_equal(g.host(c.block_forward(dblk, dX)), want, f"call {k}")
    finally:
        c.set_row_fusion(False)
    assert c.poll_status() == 0


@pytest.mark.parametrize("B,T,D,heads,H", [(1, 1, 16, 1, 16), (1, 33, 48, 1, 80), (1, 197, 192, 3, 768), (2, 257, 384, 6, 1536),
                                           (9, 197, 384, 6, 1552), (2, 65, 768, 12, 3072), (1, 130, 1024, 16, 4096),
                                           (24, 197, 384, 6, 1536), (60, 49, 768, 24, 3072), (1, 40, 1040, 5, 4112)])
def test_row_operators_in_front_of_the_dense_layers(B, T, D, heads, H):
    """Layers of few rows: LayerNorm (and, in model forwards, ShiftGELU) in front of the MMAs of the Dense layer that
    reads it.  Contraction tails of 16, ragged row blocks and channel groups, one to four channel tiles per CTA, sizes
    on both sides of what the kernel takes; the block as kernels of their own gives the same bytes."""
    import gpu_util as g
    c = g.binding.Context(0)
    blk = make_block(_Ids(5000 + B + D), 2, B, T, D, heads, H)
    X = make_block_input(B + D, B, T, D)
    dblk = g.binding.DeviceBlock(blk, "cuda")
    dX = torch.from_numpy(X).cuda()
    want = O.block_forward(blk, X)
    g.assert_equal(g.host(c.block_forward(dblk, dX)), want, "default")
    c.set_row_fusion(False)
    g.assert_equal(g.host(c.block_forward(dblk, dX)), want, "kernels of their own")
    assert c.poll_status() == 0


@pytest.mark.parametrize("batch,img,D,heads,H", [(1, 224, 192, 3, 768), (3, 160, 384, 6, 1536), (2, 64, 768, 12, 3072), (1, 32, 1024, 16, 4096)])
def test_small_model_forwards_with_prologues(batch, img, D, heads, H):
    """Two-block model forwards small enough for every Dense layer to take its row operator along."""
    import gpu_util as g
    from ivit_inputs.gen import make_image, make_vit
    c = g.binding.Context(0)
    model, image = make_vit(60 + batch, batch, img, D, heads, H, 2), make_image(61, batch, img)
    dm = g.binding.DeviceVit(model, "cuda")
    d_img = torch.from_numpy(image).cuda()
    c.vit_forward(dm, d_img)           # builds the ShiftGELU tables
    n0 = c.launch_count()
    got = g.host(c.vit_forward(dm, d_img))
    assert c.launch_count() - n0 == 3 + 5 * 2 + 1      # patches, embedding, class rows; five kernels per block; the head
    g.assert_equal(got, O.vit_forward(model, image), "logits")
    assert c.poll_status() == 0
