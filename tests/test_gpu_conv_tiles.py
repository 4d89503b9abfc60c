"""The tensor-core convolutions at the sizes where their tiles end: one tile of 8 or 16 columns (whose
MMAs read past the staged rows), fewer tiles than blocks, an odd number of tiles per block (two MMA
warps take alternate ones), two column blocks per row."""
import math

import numpy as np
import pytest

from oracle import cnn_oracle as C
from test_gpu_cnn import LAYERS, U32, assert_bf16_close, bf16_tensor, rand_bf16, tensor_bits

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SIZES = [(1, 16), (3, 112), (1, 256)]            # images, rows and columns


@pytest.mark.parametrize("B,H", SIZES)
@pytest.mark.parametrize("cin,cout,S", LAYERS)
@pytest.mark.parametrize("mode", [0, 1])
def test_tile_ends(built_lib, gpu_ctx, mode, cin, cout, S, B, H):
    """As the single-layer tests: the fp32 sum of K terms is within K u sum|terms| of the exact one
    (u = 2^-24; K = 9 cin + 1 forward, 9 cout for the input gradient), then one bf16 rounding."""
    if mode == 0 and (cin, S, H) == (64, 2, 256):
        pytest.skip("two stages of 130-column rows do not fit in shared memory")
    gfh = built_lib
    rng = np.random.default_rng(1000 * mode + cin + cout + S + H)
    wb = rand_bf16(rng, (cout, 3, 3, cin), scale=math.sqrt(2.0 / (9 * cin)))
    W, ho = C.bf16_value(wb).astype(np.float64), H // S
    if mode == 0:
        xb = rand_bf16(rng, (B, H, H, cin), relu=True)
        bias = (0.1 * rng.standard_normal(cout)).astype(np.float32)
        res = torch.empty((B, ho, ho, cout), dtype=torch.bfloat16, device="cuda")
        gfh.conv3x3(gpu_ctx, 0, cin, cout, S, B, H, inp=bf16_tensor(xb), w=bf16_tensor(wb),
                    bias=torch.from_numpy(bias).cuda(), res=res)
        x = C.bf16_value(xb).astype(np.float64)
        exact = np.maximum(C.conv3x3(x, W, S) + bias.astype(np.float64), 0.0)
        err = (9 * cin + 1) * U32 * (C.conv3x3(np.abs(x), np.abs(W), S) + np.abs(bias))
    else:
        ob, gb = rand_bf16(rng, (B, ho, ho, cout), relu=True), rand_bf16(rng, (B, ho, ho, cout))
        res = torch.empty((B, H, H, cin), dtype=torch.bfloat16, device="cuda")
        gfh.conv3x3(gpu_ctx, 1, cin, cout, S, B, H, w=bf16_tensor(wb), out=bf16_tensor(ob),
                    dout=bf16_tensor(gb), res=res)
        G = np.where(C.bf16_value(ob) > 0, C.bf16_value(gb), 0.0).astype(np.float64)
        exact = C.conv3x3_input_grad(G, W, S, H)
        err = 9 * cout * U32 * C.conv3x3_input_grad(np.abs(G), np.abs(W), S, H)
    torch.cuda.synchronize()
    assert gpu_ctx.check() == gfh.GFH_OK
    assert_bf16_close(C.bf16_value(tensor_bits(res)).astype(np.float64), exact, err)
