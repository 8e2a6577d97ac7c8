"""The projections at the edges of their tiling: row counts around the switches between one block per tile, pairs of 64 and
pairs of 128 rows, several row chunks, K that does not fill a pipeline stage, every tile width, and head-split activations
whose pair split falls inside a sequence.  Against the oracle."""
import pytest
import torch

import paper_2505_21467_b200 as dlm
from helpers import Dev
from test_gpu_projection import _close, _qkv_case, _rope_tables
from workloads import make_kv_rows, widen

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dev():
    return Dev()


@pytest.mark.parametrize("B,q_cap,dm,Hq,Hkv,D", [
    (1, 1, 64, 1, 1, 128),        # one row, one K panel
    (1, 64, 192, 2, 1, 128),      # the last row count of single blocks; K is 3 panels, less than a stage
    (1, 65, 320, 2, 1, 128),      # pairs of 64 rows, the second with one
    (2, 64, 320, 4, 2, 64),       # 128 rows exactly
    (1, 129, 64, 4, 4, 64),       # pairs of 128 rows
    (3, 171, 128, 3, 1, 128),     # 513 rows: three chunks
    (1, 20, 64, 32, 8, 64),       # 32-feature tiles, two per head of 64
    (1, 40, 192, 48, 16, 64),     # 64-feature tiles: a head of 64
    (1, 40, 128, 128, 16, 64),    # 128-feature tiles of single blocks: two heads of 64
    (1, 100, 192, 40, 4, 128),    # 128-feature pair tiles of 64 rows
    (1, 100, 128, 128, 16, 64),   # 256-feature pair tiles of 64 rows: four heads of 64
    (1, 250, 192, 88, 4, 64),     # 128-feature pair tiles of 128 rows: two heads of 64
    (1, 250, 64, 72, 4, 128),     # 192-feature pair tiles of 128 rows, units of heads of 128
    (1, 130, 64, 104, 4, 128),    # 256-feature pair tiles of 128 rows: two heads of 128
    (1, 300, 64, 104, 4, 64),     # the same, four heads of 64, two chunks of rows
    (1, 33, 128, 14, 1, 24),      # a head size without rotary embedding
    (1, 160, 64, 192, 10, 64),    # 192-feature tiles, units of 32 two to a group, the last tile ragged
    (1, 160, 128, 84, 8, 128),    # the same with heads of 128
    (4, 320, 128, 28, 4, 128),    # 1280 rows: tiles beyond 256 features, two MMAs each
    (1, 1801, 64, 28, 4, 128),    # the widest, 512
    (1, 1537, 64, 66, 2, 64),     # 448: MMAs of 256 and 192, heads of 64
    (2, 900, 64, 72, 4, 24),      # 320, the heads without rotary embedding
])
def test_qkv_projection_tiles(dev, oracle, B, q_cap, dm, Hq, Hkv, D):
    seed = 13 * B + q_cap
    # millions of sums: without the bias none is so large (8) that rounding it to bf16 alone exceeds the tolerance
    q, k, v = _qkv_case(dev, oracle, B, q_cap, dm, Hq, Hkv, D, B * q_cap < 1000, seed)
    if D == 24:
        return
    # the same sums turned in the epilogue and staged in a cache
    n_out = (Hq + 2 * Hkv) * D
    x = make_kv_rows((B, q_cap, dm), seed, "cuda")
    w = (torch.randn(n_out, dm, generator=torch.Generator("cuda").manual_seed(seed + 1), device="cuda") * dm ** -0.5).to(torch.bfloat16)
    bias = make_kv_rows((n_out,), seed + 2, "cuda") if B * q_cap < 1000 else None
    cs, sn = _rope_tables(B, q_cap, D, seed + 3)
    ck, cv = make_kv_rows((1, B, Hkv, q_cap + 9, D), 3, "cuda"), make_kv_rows((1, B, Hkv, q_cap + 9, D), 4, "cuda")
    cache = dlm.make_kv_cache(ck, cv, torch.arange(B, dtype=torch.int32, device="cuda"))
    q2, k2, v2 = torch.empty_like(q), torch.empty_like(k), torch.empty_like(v)
    ws = dev.workspace(dlm.dlm_window_proj_workspace_bytes(dev.ctx, B * q_cap, n_out, dm))
    dlm.dlm_window_qkv_project_stage(dev.ctx, x, w, bias, cs, sn, B, q_cap, dm, Hq, Hkv, D, None, q2, k2, v2, cache, 0, ws)
    assert dev.status() == 0
    rq, rk, rv = oracle.qkv_project_rope(widen(x), widen(w), None if bias is None else widen(bias), cs.cpu().numpy(), sn.cpu().numpy(), Hq, Hkv, D)
    _close(q2, rq, "q"); _close(k2, rk, "k")
    assert torch.equal(v2, v)
    for b in range(B):
        assert torch.equal(ck[0, b, :, b:b + q_cap], k2[b]) and torch.equal(cv[0, b, :, b:b + q_cap], v2[b])


@pytest.mark.parametrize("B,q_cap,dm,Hq,D", [
    (1, 1, 128, 1, 64),
    (5, 8, 256, 3, 64),           # single blocks, five sequences in one copy
    (3, 24, 128, 3, 128),         # 72 rows: two sequences and one
    (3, 40, 384, 2, 128),         # 120 rows: the pair's split falls inside the second sequence
    (1, 200, 256, 3, 64),
    (3, 80, 128, 5, 64),          # 240 rows: as above, with 128 rows a block
    (9, 24, 256, 2, 128),
    (3, 72, 128, 3, 64),          # 216 rows in pieces of 24
    (5, 48, 384, 2, 128),         # the same, five sequences
    (5, 24, 128, 3, 128),         # 120 rows whose half of the sequences exceeds the narrow pair's rows
    (3, 56, 256, 1, 192),         # heads of three panels
])
def test_out_projection_tiles(dev, oracle, B, q_cap, dm, Hq, D):
    seed = 17 * B + q_cap
    o = make_kv_rows((B, Hq, q_cap, D), seed, "cuda")
    wo = (torch.randn(dm, Hq * D, generator=torch.Generator("cuda").manual_seed(seed + 1), device="cuda") * (Hq * D) ** -0.5).to(torch.bfloat16)
    y = dev.guarded((B, q_cap, dm), torch.bfloat16, float("nan"))
    ws = dev.workspace(dlm.dlm_window_proj_workspace_bytes(dev.ctx, B * q_cap, dm, Hq * D))
    dlm.dlm_window_out_project(dev.ctx, o, wo, None, B, q_cap, dm, Hq, D, y, ws)
    assert dev.status() == 0
    _close(y, oracle.out_project(widen(o), widen(wo), None), "y")


# K of one stage, of two (a stage holds 256 elements of K, 128 with more than 64 rows, 64 where tiles are wide), of one more, and of more than the
# ring holds
@pytest.mark.parametrize("dm", [128, 256, 512, 576, 2304])
@pytest.mark.parametrize("q_cap", [17, 100, 200])
def test_qkv_projection_stages_of_k(dev, oracle, q_cap, dm):
    _qkv_case(dev, oracle, 1, q_cap, dm, 4, 1, 128, True, q_cap + dm)


# the same for stages of 64 elements: 256-feature pair tiles of 64 rows, 192 and 256 of 128 rows, 384
@pytest.mark.parametrize("dm", [64, 128, 192, 1024])
@pytest.mark.parametrize("B,q_cap,Hq,Hkv,D", [(1, 100, 128, 16, 64), (1, 250, 72, 4, 128), (1, 130, 104, 4, 128), (2, 640, 28, 4, 128)])
def test_qkv_projection_stages_of_one_panel(dev, oracle, B, q_cap, Hq, Hkv, D, dm):
    _qkv_case(dev, oracle, B, q_cap, dm, Hq, Hkv, D, B * q_cap < 1000, q_cap + dm)
