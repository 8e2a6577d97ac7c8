"""GPU parity of dlm_freecache_attn_step against the CPU oracle, through the C-ABI.
Tolerance (fp32 oracle, unit-scale bf16 inputs, bf16 output): max |err| <= 2e-2, mean |err| <= 2e-3."""
import numpy as np
import pytest
import torch

import paper_2505_21467_b200 as dlm
from workloads import get_config, make_attn_inputs, make_cache, seed_for
from helpers import Dev, assert_attn_close, gpu_attn_step, oracle_attn_layers

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dev():
    return Dev()


def _i32(a):
    return torch.tensor(np.asarray(a), dtype=torch.int32, device="cuda")


def _case(dev, oracle, NL, B, Hq, Hkv, D, Lcap, q_cap, cache_len, q_len=None, seed=1, layer_begin=0, nl=None,
          scale=0.0, layers=None, hint=0, device="cpu"):
    nl = NL - layer_begin if nl is None else nl
    ck, cv = make_cache(NL, B, Hkv, Lcap, D, seed, device=device)
    q, kn, vn = make_attn_inputs(nl, B, Hq, Hkv, q_cap, D, seed + 1, device=device)
    cl = _i32(cache_len)
    ql = None if q_len is None else _i32(q_len)
    out, lse = gpu_attn_step(dev, ck.cuda(), cv.cuda(), cl, q.cuda(), kn.cuda(), vn.cuda(), ql, scale, layer_begin,
                             layer_begin + nl, hint=hint)
    assert dev.status() == 0
    ref = oracle_attn_layers(oracle, ck, cv, cl, q, kn, vn, ql, scale if scale > 0 else None, layer_begin, layers)
    errs = [assert_attn_close(out, lse, ref[lc], lc) for lc in ref]
    return out, lse, errs


def _schedule(dev, NL, B, Hq, Hkv, D, Lcap, q_cap, nl, hint=0):
    ck = torch.empty(NL, B, Hkv, Lcap, D, dtype=torch.bfloat16, device="cuda")
    cache = dlm.make_kv_cache(ck, ck, _i32([0] * B))
    return dlm.dlm_selftest_attn_schedule(dev.ctx, cache, nl, Hq, q_cap, hint)


def _each_schedule(dev, names, NL, B, Hq, Hkv, D, Lcap, q_cap):
    """For every schedule of `names`, makes a call of this shape take it and yields the length hint to pass."""
    try:
        for name in names:
            hint = 1 if name == "whole" else 0
            dlm.dlm_selftest_set_attn_team_max(dev.ctx, 1 << 20 if name == "team" else 1)
            sch = _schedule(dev, NL, B, Hq, Hkv, D, Lcap, q_cap, NL, hint)
            assert name == ("team" if sch["team"] > 1 else "whole" if sch["whole_units"] else "split"), sch
            yield hint
    finally:
        dlm.dlm_selftest_set_attn_team_max(dev.ctx, 1 << 20)


def test_tiny_config_full(dev, oracle):
    cfg = get_config(0)
    _case(dev, oracle, cfg.n_layers, cfg.batch, cfg.n_q_heads, cfg.n_kv_heads, cfg.head_dim, cfg.capacity,
          cfg.block_len, [cfg.prompt_len], seed=seed_for(0))


@pytest.mark.parametrize("Hq,Hkv,D,Lcap,q_cap,cache_len,q_len", [
    (28, 4, 128, 700, 32, [517, 640], None),            # Dream group of 7: two M tiles, several K tiles, ragged tail
    (28, 4, 128, 700, 32, [517, 0], [32, 7]),           # ragged active rows, one empty cache
    (8, 8, 128, 400, 64, [333, 128], [64, 64]),         # MHA (LLaDA-like), block 64
    (4, 2, 64, 300, 32, [1, 299], [5, 32]),             # head_dim 64
    (2, 1, 64, 200, 128, [130, 77], [128, 100]),        # 256 query rows per KV head, fresh part spans a full tile
    (6, 2, 128, 260, 20, [256, 255], [20, 0]),          # q_cap not a multiple of 16; one element fully inactive
    (3, 3, 128, 129, 1, [129, 128], None),              # a single active row
])
def test_shapes_and_ragged_lengths(dev, oracle, Hq, Hkv, D, Lcap, q_cap, cache_len, q_len):
    out, lse, _ = _case(dev, oracle, 2, 2, Hq, Hkv, D, Lcap, q_cap, cache_len, q_len, seed=Hq * 100 + q_cap)
    if q_len is not None:
        for b, n in enumerate(q_len):
            assert torch.all(out[:, b, :, n:] == 0)


@pytest.mark.parametrize("name", ["whole", "split", "team"])
def test_each_schedule(dev, oracle, name):
    """How the units are dealt is the host's choice: whole, split across the SMs, or to teams; all three match the oracle."""
    for hint in _each_schedule(dev, [name], 2, 2, 28, 4, 128, 1400, 32):
        _case(dev, oracle, 2, 2, 28, 4, 128, 1400, 32, [1368, 900], [32, 17], seed=77, hint=hint)


@pytest.mark.parametrize("Hq,Hkv,D,Lcap,q_cap,cache_len,q_len", [
    (28, 4, 128, 600, 256, [300], None),                # the paper's window: 256 active rows, Dream heads (7 chunks of 256 rows)
    (4, 4, 128, 520, 512, [0, 0], [512, 333]),          # initial full pass: empty cache, 512 active rows, ragged
    (4, 2, 64, 400, 300, [77, 100], [300, 130]),        # rows per KV head not a multiple of 256, head_dim 64
    (16, 4, 64, 1100, 256, [1001, 844, 3], [256, 200, 256]),   # units of two M tiles when split
])
def test_large_windows_in_row_chunks(dev, oracle, Hq, Hkv, D, Lcap, q_cap, cache_len, q_len):
    B = len(cache_len)
    for hint in _each_schedule(dev, ["whole", "split", "team"], 1, B, Hq, Hkv, D, Lcap, q_cap):
        out, lse, _ = _case(dev, oracle, 1, B, Hq, Hkv, D, Lcap, q_cap, cache_len, q_len, seed=Hq * 1000 + q_cap, hint=hint)
        if q_len is not None:
            for b, n in enumerate(q_len):
                assert torch.all(out[:, b, :, n:] == 0)


@pytest.mark.parametrize("scale", [0.2, 1.0])
def test_scores_that_keep_outgrowing_the_running_maximum(dev, oracle, scale):
    """Keys grow along the cache and the softmax scale is large, so later tiles bring scores far above the
    maximum in use (by tens of powers of two): the deferred rescaling of O has to fire, repeatedly, and the result
    must still match.  Every schedule."""
    NL, B, Hq, Hkv, D, Lc, q_cap = 1, 2, 14, 2, 128, 1500, 32
    ck, cv = make_cache(NL, B, Hkv, Lc + 40, D, 91)
    q, kn, vn = make_attn_inputs(NL, B, Hq, Hkv, q_cap, D, 92)
    grow = (1.0 + 4.0 * torch.arange(Lc + 40, dtype=torch.float32) / Lc).view(1, 1, 1, -1, 1)
    ck = (ck.float() * grow).to(torch.bfloat16)
    cl = _i32([Lc, Lc - 333])
    for hint in _each_schedule(dev, ["whole", "split", "team"], NL, B, Hq, Hkv, D, Lc + 40, q_cap):
        out, lse = gpu_attn_step(dev, ck.cuda(), cv.cuda(), cl, q.cuda(), kn.cuda(), vn.cuda(), None, scale, hint=hint)
        assert dev.status() == 0
        ref = oracle_attn_layers(oracle, ck, cv, cl, q, kn, vn, None, scale)
        assert_attn_close(out, lse, ref[0], 0)


def test_many_batch_elements_with_random_lengths(dev, oracle):
    """600 sequences (the limit is 1024), each with its own cache length and window length, some empty."""
    rng = np.random.default_rng(3)
    B, Lcap, q_cap = 600, 70, 8
    cache_len = rng.integers(0, Lcap + 1, B).tolist()
    q_len = rng.integers(0, q_cap + 1, B).tolist()
    out, lse, _ = _case(dev, oracle, 1, B, 2, 1, 64, Lcap, q_cap, cache_len, q_len, seed=606)
    for b, n in enumerate(q_len):
        assert torch.all(out[:, b, :, n:] == 0)


def test_layer_range_and_explicit_scale(dev, oracle):
    _case(dev, oracle, 5, 1, 4, 2, 128, 300, 32, [290], seed=9, layer_begin=2, nl=2, scale=0.05)


@pytest.mark.parametrize("name,Lcap", [("whole", 520), ("team", 520), ("split", 1400)])
def test_poisoned_invisible_rows_do_not_leak(dev, oracle, name, Lcap):
    """Rows at or beyond cache_len / q_len may hold NaN: the result must not change (bit for bit)."""
    NL, B, Hq, Hkv, D, q_cap = 1, 2, 14, 2, 128, 32
    cl, ql = _i32([300, 5]), _i32([32, 9])
    for hint in _each_schedule(dev, [name], NL, B, Hq, Hkv, D, Lcap, q_cap):
        ck, cv = make_cache(NL, B, Hkv, Lcap, D, 31, device="cuda")
        q, kn, vn = make_attn_inputs(NL, B, Hq, Hkv, q_cap, D, 32, device="cuda")
        base, base_lse = gpu_attn_step(dev, ck, cv, cl, q, kn, vn, ql, hint=hint)
        nan = float("nan")
        ck[:, 0, :, 300:] = nan; cv[:, 0, :, 300:] = nan
        ck[:, 1, :, 5:] = nan; cv[:, 1, :, 5:] = nan
        kn[:, 1, :, 9:] = nan; vn[:, 1, :, 9:] = nan; q[:, 1, :, 9:] = nan
        out, lse = gpu_attn_step(dev, ck, cv, cl, q, kn, vn, ql, hint=hint)
        assert dev.status() == 0
        assert torch.equal(out, base) and torch.equal(lse, base_lse)
        assert torch.isfinite(out.float()).all()


@pytest.mark.parametrize("name", ["whole", "split", "team"])
def test_deterministic(dev, name):
    ck, cv = make_cache(2, 1, 4, 1100, 128, 41, device="cuda")
    q, kn, vn = make_attn_inputs(2, 1, 28, 4, 32, 128, 42, device="cuda")
    cl = _i32([1056])
    for hint in _each_schedule(dev, [name], 2, 1, 28, 4, 128, 1100, 32):
        a, al = gpu_attn_step(dev, ck, cv, cl, q, kn, vn, hint=hint)
        b, bl = gpu_attn_step(dev, ck, cv, cl, q, kn, vn, hint=hint)
        assert torch.equal(a, b) and torch.equal(al, bl)


def test_the_same_sizes_on_other_tensors(dev):
    """What a context keeps of a call (descriptors, plan) depends on sizes alone: calls of two shapes in turn, each time on
    other copies of the same tensors, one of them at an odd multiple of 16 bytes, give the same bits."""
    def shifted(t, n):      # a copy that starts n * 16 bytes into a buffer of its own
        buf = torch.empty(t.numel() + 8 * n, dtype=t.dtype, device="cuda")
        return buf[8 * n:].view_as(t).copy_(t)

    shapes = [(2, 1, 28, 4, 32, 128, 300, [280]), (1, 3, 4, 2, 40, 64, 500, [400, 0, 77])]
    first = {}
    for turn in range(3):
        for i, (NL, B, Hq, Hkv, q_cap, D, Lcap, lens) in enumerate(shapes):
            ck, cv = make_cache(NL, B, Hkv, Lcap, D, 60 + i, device="cuda")
            t = [ck, cv, *make_attn_inputs(NL, B, Hq, Hkv, q_cap, D, 70 + i, device="cuda")]
            ck, cv, q, kn, vn = [shifted(x, 2 * turn + 1) for x in t]
            out, lse = gpu_attn_step(dev, ck, cv, _i32(lens), q, kn, vn)
            assert dev.status() == 0
            a, b = first.setdefault(i, (out, lse))
            assert torch.equal(a, out) and torch.equal(b, lse)


def test_argument_errors(dev):
    ck, cv = make_cache(1, 1, 2, 64, 128, 1, device="cuda")
    cl = _i32([10])
    cache = dlm.make_kv_cache(ck, cv, cl)
    ws = dev.workspace(1 << 20)

    def call(Hq=4, q_cap=32, D=128, layer_end=1, ws_=ws):
        q = torch.zeros(1, 1, Hq, q_cap, D, dtype=torch.bfloat16, device="cuda")
        kn = torch.zeros(1, 1, 2, q_cap, D, dtype=torch.bfloat16, device="cuda")
        dlm.dlm_freecache_attn_step(dev.ctx, cache, 0, layer_end, q, kn, kn, Hq, q_cap, None, 0.0, 0,
                                    torch.empty_like(q), None, ws_)

    before = dlm.dlm_launch_count(dev.ctx)
    for kwargs, code in ((dict(Hq=3), dlm.DLM_ERR_UNSUPPORTED), (dict(Hq=4, q_cap=5000), dlm.DLM_ERR_UNSUPPORTED),
                         (dict(layer_end=2), dlm.DLM_ERR_SHAPE),
                         (dict(ws_=ws[8:]), dlm.DLM_ERR_WORKSPACE)):
        with pytest.raises(dlm.DlmError) as e:
            call(**kwargs)
        assert e.value.code == code, kwargs
    assert dlm.dlm_launch_count(dev.ctx) == before
    ck96, cv96 = make_cache(1, 1, 2, 64, 96, 1, device="cuda")
    cache96 = dlm.make_kv_cache(ck96, cv96, cl)
    q = torch.zeros(1, 1, 2, 8, 96, dtype=torch.bfloat16, device="cuda")
    with pytest.raises(dlm.DlmError) as e:
        dlm.dlm_freecache_attn_step(dev.ctx, cache96, 0, 1, q, q, q, 2, 8, None, 0.0, 0, torch.empty_like(q), None, ws)
    assert e.value.code == dlm.DLM_ERR_UNSUPPORTED


def test_out_of_range_lengths_are_clamped_and_reported(dev):
    ck, cv = make_cache(1, 2, 2, 64, 128, 1, device="cuda")
    q, kn, vn = make_attn_inputs(1, 2, 4, 2, 16, 128, 2, device="cuda")
    out, _ = gpu_attn_step(dev, ck, cv, _i32([65, 10]), q, kn, vn)
    assert dev.status() == dlm.DLM_ERR_CAPACITY
    ref, _ = gpu_attn_step(dev, ck, cv, _i32([64, 10]), q, kn, vn)
    assert dev.status() == 0 and torch.equal(out, ref)


def test_dream7b_full_size_layer_batched_first_and_last_step(dev, oracle):
    """The benchmark's launch: all 28 layers in one call at the Dream-7B shape, at the first step
    (cache 1024) and the last (cache 1248); oracle on layers {0, 14, 27}, all heads and rows."""
    cfg = get_config(1)
    for cache_len in (cfg.prompt_len, cfg.capacity - cfg.block_len):
        _case(dev, oracle, cfg.n_layers, cfg.batch, cfg.n_q_heads, cfg.n_kv_heads, cfg.head_dim, cfg.capacity,
              cfg.block_len, [cache_len], seed=seed_for(1, cache_len), layers=[0, 14, 27], hint=cache_len,
              device="cuda")


def test_guided_shape_ragged_batch8(dev, oracle):
    """Config 5's shape: batch 8 with ragged cache_len and q_len (accepted prefixes shrink the window)."""
    cfg = get_config(4)
    cache_len = [1024, 1031, 1056, 1100, 1247, 1279, 1088, 1150]
    q_len = [32, 25, 32, 20, 1, 1, 32, 2]
    _case(dev, oracle, 3, cfg.batch, cfg.n_q_heads, cfg.n_kv_heads, cfg.head_dim, cfg.capacity, cfg.block_len,
          cache_len, q_len, seed=seed_for(4), layers=[0, 2])


def test_guided_shape_more_units_than_sms_split_schedule(dev, oracle):
    """Config 5's launch form: more units (10 layers x 8 sequences x 4 KV heads = 320) than SMs and still split,
    so a block's share holds whole units and a partial unit at each end, with ragged lengths."""
    cfg = get_config(4)
    cache_len = [1024, 1031, 1056, 1100, 1247, 1279, 1088, 1150]
    q_len = [32, 25, 32, 20, 1, 1, 32, 2]
    sch = _schedule(dev, 10, cfg.batch, cfg.n_q_heads, cfg.n_kv_heads, cfg.head_dim, cfg.capacity, cfg.block_len, 10)
    assert sch["whole_units"] == 0 and sch["team"] == 1
    _case(dev, oracle, 10, cfg.batch, cfg.n_q_heads, cfg.n_kv_heads, cfg.head_dim, cfg.capacity, cfg.block_len,
          cache_len, q_len, seed=seed_for(4, 7), layers=[0, 9], device="cuda")


def test_longctx_shape_sampled_layers(dev, oracle):
    """Config 4: 16384 cached rows, Dream heads; 4 of the 28 layers resident, oracle on two of them."""
    cfg = get_config(3)
    _case(dev, oracle, 4, cfg.batch, cfg.n_q_heads, cfg.n_kv_heads, cfg.head_dim, cfg.prompt_len + cfg.block_len,
          cfg.block_len, [cfg.prompt_len], seed=seed_for(3), layers=[0, 3], device="cuda")


def test_llada_shape_sampled(dev, oracle):
    """Config 3's shape at full batch / heads / lengths, 2 layers resident; oracle on one layer."""
    cfg = get_config(2)
    _case(dev, oracle, 2, cfg.batch, cfg.n_q_heads, cfg.n_kv_heads, cfg.head_dim, cfg.capacity, cfg.block_len,
          [2048, 2112, 2496, 2300], seed=seed_for(2), layers=[1], device="cuda")


def test_a_wait_that_runs_out_reports_timeout_and_leaves_the_context_usable(dev, oracle):
    """The bounded device-side wait gives up after its limit (here 2 ms on a barrier nothing arrives at): the kernel
    ends normally, the status word says DLM_ERR_TIMEOUT, it is cleared by the read, and the next calls work."""
    dlm.dlm_selftest_wait_timeout(dev.ctx, 2_000_000)
    assert dev.status() == dlm.DLM_ERR_TIMEOUT
    assert dev.status() == 0
    _case(dev, oracle, 1, 1, 4, 2, 64, 200, 16, [150], seed=5)
    with pytest.raises(dlm.DlmError) as e:
        dlm.dlm_selftest_wait_timeout(dev.ctx, 5_000_000_000)
    assert e.value.code == dlm.DLM_ERR_SHAPE


@pytest.mark.parametrize("name", ["whole", "split"])
def test_the_attention_kernel_gives_up_cleanly_when_its_waits_may_not_wait(dev, oracle, name):
    """The kernel's own unwinding, units whole and split: with the wait limit set to 0 the first wait whose data is still
    on its way gives up; the producer lets its copies land, the MMA issuers drain, every role reaches the teardown,
    TMEM is released and the kernel ends normally with DLM_ERR_TIMEOUT.  With the limit restored the next call on the
    same context is correct again (nothing of the aborted launch is left behind, ticket words included)."""
    for hint in _each_schedule(dev, [name], 2, 2, 28, 4, 128, 700, 32):
        args = dict(NL=2, B=2, Hq=28, Hkv=4, D=128, Lcap=700, q_cap=32, cache_len=[517, 640], seed=4242, hint=hint)
        dlm.dlm_selftest_set_wait_limit(dev.ctx, 0)
        try:
            ck, cv = make_cache(2, 2, 4, 700, 128, 1, device="cuda")
            q, kn, vn = make_attn_inputs(2, 2, 28, 4, 32, 128, 2, device="cuda")
            gpu_attn_step(dev, ck, cv, _i32([517, 640]), q, kn, vn, hint=hint)
            torch.cuda.synchronize()
            assert dev.status() == dlm.DLM_ERR_TIMEOUT
        finally:
            dlm.dlm_selftest_set_wait_limit(dev.ctx, 2_000_000_000)
        assert dev.status() == 0
        _case(dev, oracle, **args)
    with pytest.raises(dlm.DlmError) as e:
        dlm.dlm_selftest_set_wait_limit(dev.ctx, 3_000_000_000)
    assert e.value.code == dlm.DLM_ERR_SHAPE


@pytest.mark.parametrize("D,cache_len,q_len", [
    (128, [100, 90], None),         # two key tiles: the producer has issued everything before it would have to wait
    (128, [100, 0], [16, 0]),       # a unit without key tiles, whose Q is copied all the same
    (64, [330, 200], [16, 9]),      # the deeper rings of heads of 64: up to four key tiles
])
def test_giving_up_lets_copies_land_that_nobody_waits_for(dev, oracle, D, cache_len, q_len):
    """A launch that gives up although its producer never had to wait ends only when its copies have landed: the blocks of the
    next launch, right behind it on the same SMs, take over that shared memory.  Units dealt whole (no counters to clear)."""
    ck, cv = make_cache(2, 2, 4, 400, D, 1)
    q, kn, vn = make_attn_inputs(2, 2, 28, 4, 16, D, 2)
    cl, ql = _i32(cache_len), None if q_len is None else _i32(q_len)
    args = [t.cuda() for t in (ck, cv)] + [cl] + [t.cuda() for t in (q, kn, vn)] + [ql]
    assert _schedule(dev, 2, 2, 28, 4, D, 400, 16, 2, 1)["whole_units"] == 1 == _schedule(dev, 2, 2, 28, 4, D, 400, 16, 2, 1)["team"]
    ref = oracle_attn_layers(oracle, ck, cv, cl, q, kn, vn, ql)
    gpu_attn_step(dev, *args, hint=1)
    for _ in range(4):
        dlm.dlm_selftest_set_wait_limit(dev.ctx, 0)
        try:
            gpu_attn_step(dev, *args, hint=1)
        finally:
            dlm.dlm_selftest_set_wait_limit(dev.ctx, 2_000_000_000)
        out, lse = gpu_attn_step(dev, *args, hint=1)
        assert dev.status() == dlm.DLM_ERR_TIMEOUT
        for lc in ref:
            assert_attn_close(out, lse, ref[lc], lc)


@pytest.mark.parametrize("NL,B,Hq,Hkv,D,Lcap,q_cap,cache_len,q_len", [
    (1, 1, 28, 4, 128, 2200, 32, [2048], None),          # one Dream layer at batch 1: 8 units of 128 rows, 17 key tiles each
    (1, 1, 28, 4, 128, 2200, 32, [2048], [19]),          # ragged active rows
    (1, 2, 28, 4, 128, 900, 32, [517, 0], [32, 7]),      # an empty cache: one key tile, most ranks get none
    (1, 2, 6, 2, 128, 700, 20, [256, 255], [20, 0]),     # one element fully inactive; 60 rows per unit
    (2, 1, 4, 2, 64, 1000, 32, [901], [5]),              # head_dim 64, 64 rows per unit
    (1, 1, 2, 1, 64, 700, 128, [650], [100]),            # 256 rows per unit (two M tiles), fresh part a whole tile
    (1, 1, 8, 8, 128, 1100, 64, [1000], None),           # MHA, 64 rows per unit
    (1, 1, 3, 3, 128, 300, 1, [129], None),              # a single row per unit
])
def test_team_schedule_against_the_oracle_at_every_team_size(dev, oracle, NL, B, Hq, Hkv, D, Lcap, q_cap, cache_len, q_len):
    """Calls with few units give each unit a team of blocks, which split its key tiles and then each reduce a share
    of its outputs over all the team's pieces.  Every team size, and the same call with the schedule switched off,
    matches the oracle."""
    outs = []
    try:
        for tmax in (1 << 20, 8, 3, 2, 1):
            dlm.dlm_selftest_set_attn_team_max(dev.ctx, tmax, force=True)
            sch = _schedule(dev, NL, B, Hq, Hkv, D, Lcap, q_cap, NL)
            assert (sch["team"] > 1) == (tmax > 1) and sch["team"] <= tmax and sch["grid"] % sch["team"] == 0
            out, lse, _ = _case(dev, oracle, NL, B, Hq, Hkv, D, Lcap, q_cap, cache_len, q_len, seed=Hq * 10 + q_cap)
            outs.append(out.float())
            if q_len is not None:
                for b, n in enumerate(q_len):
                    assert torch.all(out[:, b, :, n:] == 0)
    finally:
        dlm.dlm_selftest_set_attn_team_max(dev.ctx, 1 << 20)
    for o in outs[1:]:
        assert (o - outs[0]).abs().max().item() <= 2e-2
    with pytest.raises(dlm.DlmError) as e:
        dlm.dlm_selftest_set_attn_team_max(dev.ctx, 0)
    assert e.value.code == dlm.DLM_ERR_SHAPE
    with pytest.raises(dlm.DlmError) as e:
        dlm.dlm_selftest_set_attn_team_max(dev.ctx, 4, 2)
    assert e.value.code == dlm.DLM_ERR_SHAPE


def test_team_schedule_repeated_launches_leave_the_counters_clean(dev, oracle):
    """Teams meet on barriers of their own launch and count nothing in memory: many launches in a row on the same units (also of
    different team sizes) stay correct, and so does a split-schedule call, which does count, afterwards."""
    shape = dict(NL=1, B=1, Hq=28, Hkv=4, D=128, Lcap=2200, q_cap=32)
    try:
        for i, tmax in enumerate((1 << 20, 5, 1 << 20, 2, 9)):
            dlm.dlm_selftest_set_attn_team_max(dev.ctx, tmax, force=True)
            assert _schedule(dev, nl=1, **shape)["team"] > 1
            _case(dev, oracle, cache_len=[1500 + 100 * i], seed=300 + i, **shape)
    finally:
        dlm.dlm_selftest_set_attn_team_max(dev.ctx, 1 << 20)
    for hint in _each_schedule(dev, ["split"], 2, 2, 28, 4, 128, 1400, 32):
        _case(dev, oracle, 2, 2, 28, 4, 128, 1400, 32, [1368, 900], [32, 17], seed=77, hint=hint)


def test_team_members_without_key_tiles(dev, oracle):
    """Sequences much shorter than the hint: most blocks of a team have no key tile, send their rows' (m, l) only and are done while the Q and
    the key tile they asked for may still be on their way.  Many launches back to back, every one the same."""
    B, Lcap, q_cap = 2, 2200, 32
    assert _schedule(dev, 1, B, 28, 4, 128, Lcap, q_cap, 1)["team"] > 2
    out, lse, _ = _case(dev, oracle, 1, B, 28, 4, 128, Lcap, q_cap, [0, 60], [1, 32], seed=811)
    ck, cv = make_cache(1, B, 4, Lcap, 128, 811, device="cpu")
    q, kn, vn = make_attn_inputs(1, B, 28, 4, q_cap, 128, 812, device="cpu")
    args = [t.cuda() for t in (ck, cv)] + [_i32([0, 60])] + [t.cuda() for t in (q, kn, vn)] + [_i32([1, 32])]
    again = [gpu_attn_step(dev, *args) for _ in range(64)]
    assert dev.status() == 0
    for o, l in again:
        assert torch.equal(o, out) and torch.equal(l, lse)


def test_team_schedule_gives_up_cleanly_when_its_waits_may_not_wait(dev, oracle):
    """The give-up path under the team schedule: with the wait limit at 0 every wait, the one for the team's other
    blocks included, gives up at once.  The kernel ends normally with DLM_ERR_TIMEOUT and the next call is correct."""
    shape = dict(NL=1, B=1, Hq=28, Hkv=4, D=128, Lcap=2200, q_cap=32)
    assert _schedule(dev, nl=1, **shape)["team"] > 1
    dlm.dlm_selftest_set_wait_limit(dev.ctx, 0)
    try:
        ck, cv = make_cache(1, 1, 4, 2200, 128, 1, device="cuda")
        q, kn, vn = make_attn_inputs(1, 1, 28, 4, 32, 128, 2, device="cuda")
        gpu_attn_step(dev, ck, cv, _i32([2048]), q, kn, vn)
        torch.cuda.synchronize()
        assert dev.status() == dlm.DLM_ERR_TIMEOUT
    finally:
        dlm.dlm_selftest_set_wait_limit(dev.ctx, 2_000_000_000)
    assert dev.status() == 0
    _case(dev, oracle, cache_len=[2048], seed=99, **shape)


# as many units as SMs (a block of a single unit each) and a few more (some blocks have two), one M tile and two; with inactive elements
@pytest.mark.parametrize("B,Hkv,group,D,q_cap", [(37, 4, 2, 64, 40), (50, 3, 2, 128, 40), (37, 4, 7, 128, 20), (50, 3, 5, 64, 30)])
def test_whole_units_as_many_as_sms_and_more(dev, oracle, B, Hkv, group, D, q_cap):
    rng = np.random.default_rng(B + D)
    cl, ql = rng.integers(0, 201, B), rng.integers(0, q_cap + 1, B)
    ql[[0, B // 2]] = 0
    for hint in _each_schedule(dev, ["whole"], 1, B, Hkv * group, Hkv, D, 200, q_cap):
        out, lse, _ = _case(dev, oracle, 1, B, Hkv * group, Hkv, D, 200, q_cap, cl, ql, seed=B, hint=hint)
    for b in np.flatnonzero(ql == 0):
        assert not out[0, b].any() and bool((lse[0, b] == -float("inf")).all())


# teams on row chunks of 64: a ragged last chunk, inactive rows and an inactive element, blocks without a key tile, both head sizes
@pytest.mark.parametrize("B,Hq,Hkv,D,Lcap,q_cap,cache_len,q_len", [
    (1, 28, 4, 128, 1100, 32, [1024], None),
    (1, 28, 4, 128, 1100, 32, [500], [9]),
    (2, 9, 3, 64, 700, 24, [700, 3], [24, 0]),
    (1, 5, 1, 128, 1990, 13, [1500], None),
])
def test_teams_of_half_m_tiles(dev, oracle, B, Hq, Hkv, D, Lcap, q_cap, cache_len, q_len):
    sch = _schedule(dev, 2, B, Hq, Hkv, D, Lcap, q_cap, 1, max(cache_len))
    assert sch["team"] > 1 and sch["chunk_rows"] == 64, sch
    for _ in range(2):
        _case(dev, oracle, 2, B, Hq, Hkv, D, Lcap, q_cap, cache_len, q_len, seed=Hq, layer_begin=1, hint=max(cache_len))


# teams whose blocks split the keys: tiles that end in either half of the keys or at its edge, blocks whose second half has nothing, rows
# that end inside a warp or at its edge, chunks of 96, team sizes that do not divide the columns
@pytest.mark.parametrize("D,Hq,Hkv,q_cap", [(128, 1, 1, 31), (128, 3, 1, 32), (128, 1, 1, 128), (64, 2, 1, 65), (128, 7, 1, 32), (64, 5, 1, 33)])
@pytest.mark.parametrize("last", [1, 33, 63, 64, 65, 127])
def test_teams_that_split_the_keys_at_the_edges(dev, oracle, D, Hq, Hkv, q_cap, last):
    try:
        for team in (2, 3, 7):
            dlm.dlm_selftest_set_attn_team_max(dev.ctx, team, force=True)
            cache_len, q_len = [640 + last, last], [q_cap, max(1, q_cap - 3)]
            sch = _schedule(dev, 1, 2, Hq, Hkv, D, 1000, q_cap, 1, 640 + last)
            assert sch["team"] == team or team == 7 and sch["team"] > 3, sch
            _case(dev, oracle, 1, 2, Hq, Hkv, D, 1000, q_cap, cache_len, q_len, seed=last + team, hint=640 + last)
    finally:
        dlm.dlm_selftest_set_attn_team_max(dev.ctx, 1 << 20)


# blocks of a single unit ask for the key tile that the hint lets them expect before they read the lengths: hints below, at and beyond the lengths,
# sequences without cached rows or without active ones, whole units and teams
@pytest.mark.parametrize("D,Hq,Hkv,q_cap,nl", [(128, 4, 2, 24, 1), (64, 4, 2, 24, 1), (128, 28, 4, 32, 1), (64, 8, 8, 40, 3)])
@pytest.mark.parametrize("hint", [1, 130, 640, 1100, 0])
def test_lengths_other_than_the_hint(dev, oracle, D, Hq, Hkv, q_cap, nl, hint):
    for seed, (cache_len, q_len) in enumerate([([0, 640, 17], [q_cap, 1, q_cap]), ([1100, 128, 129], [q_cap, 0, 7]), ([641, 0, 700], None)]):
        _case(dev, oracle, nl, 3, Hq, Hkv, D, 1140, q_cap, cache_len, q_len, seed=seed + hint, hint=hint, layers=[nl - 1])


# teams of two M tiles: the chain that is through first lays its rows out over the K tiles, which the other one may still read.  Launches back to
# back with other lengths in between, every one the same
@pytest.mark.parametrize("B,Hq,Hkv,q_cap", [(6, 16, 8, 128), (8, 8, 8, 250), (6, 16, 8, 65)])
def test_teams_of_two_m_tiles(dev, oracle, B, Hq, Hkv, q_cap):
    cap = 1000
    try:
        dlm.dlm_selftest_set_attn_team_max(dev.ctx, 2, force=True)
        sch = _schedule(dev, 1, B, Hq, Hkv, 64, cap, q_cap, 1, 300)
        assert sch["team"] == 2 and sch["chunk_rows"] == 256, sch
        rng = np.random.default_rng(q_cap)
        ck, cv = make_cache(1, B, Hkv, cap, 64, 5, device="cuda")
        q, kn, vn = make_attn_inputs(1, B, Hq, Hkv, q_cap, 64, 6, device="cuda")
        calls = [(_i32(rng.integers(0, 700, B)), _i32(rng.integers(1, q_cap + 1, B))) for _ in range(3)]
        refs = [oracle_attn_layers(oracle, ck, cv, cl, q, kn, vn, ql)[0] for cl, ql in calls]
        got = [[gpu_attn_step(dev, ck, cv, cl, q, kn, vn, ql, hint=300) for cl, ql in calls] for _ in range(20)]
        assert dev.status() == 0
        for i, ref in enumerate(refs):
            assert_attn_close(got[0][i][0], got[0][i][1], ref, 0)
            for launch in got[1:]:
                assert torch.equal(launch[i][0], got[0][i][0]) and torch.equal(launch[i][1], got[0][i][1])
    finally:
        dlm.dlm_selftest_set_attn_team_max(dev.ctx, 1 << 20)


# a block reports a give-up of any of its roles, also one that comes after the rows of its other M tile are done: units whole (of one segment and
# of several), split, teams of one and of two M tiles; whichever waits happen to give up, a launch without an error status has every row right
@pytest.mark.parametrize("name,B,Hq,Hkv,D,q_cap", [("whole", 37, 8, 4, 64, 80), ("whole", 80, 16, 2, 128, 17), ("split", 2, 28, 4, 128, 32),
                                                   ("team", 1, 28, 4, 128, 32), ("team", 6, 16, 8, 64, 128)])
def test_no_launch_that_gave_up_passes_for_good(dev, oracle, name, B, Hq, Hkv, D, q_cap):
    cap = 300 if name == "whole" else 1400
    ck, cv = make_cache(1, B, Hkv, cap, D, 5, device="cuda")
    q, kn, vn = make_attn_inputs(1, B, Hq, Hkv, q_cap, D, 6, device="cuda")
    cl = _i32(np.random.default_rng(B).integers(0, cap - q_cap, B))
    try:
        for hint in _each_schedule(dev, [name], 1, B, Hq, Hkv, D, cap, q_cap):
            ref = oracle_attn_layers(oracle, ck, cv, cl, q, kn, vn)[0]
            for limit in (0, 0, 0, 2_000_000_000):
                dlm.dlm_selftest_set_wait_limit(dev.ctx, limit)
                out, lse = gpu_attn_step(dev, ck, cv, cl, q, kn, vn, hint=hint)
                status = dev.status()
                assert status == 0 or limit == 0 and status == dlm.DLM_ERR_TIMEOUT
                if status == 0:
                    assert_attn_close(out, lse, ref, 0)
    finally:
        dlm.dlm_selftest_set_wait_limit(dev.ctx, 2_000_000_000)


# a key of NaN or +-inf reaches every row that it makes undefined, whichever block or key half it falls to, and no other row
@pytest.mark.parametrize("name", ["whole", "split", "team"])
@pytest.mark.parametrize("D,Hq,Hkv", [(128, 28, 4), (64, 12, 2)])
@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
@pytest.mark.parametrize("at", [3, 70, 1111, 1300])
def test_a_key_that_is_not_finite(dev, name, D, Hq, Hkv, bad, at):
    B, cap, q_cap, cl = 2, 1400, 32, [1301, 1200]
    ck, cv = make_cache(1, B, Hkv, cap, D, 31, device="cuda")
    q, kn, vn = make_attn_inputs(1, B, Hq, Hkv, q_cap, D, 32, device="cuda")
    for hint in _each_schedule(dev, [name], 1, B, Hq, Hkv, D, cap, q_cap):
        good, good_lse = gpu_attn_step(dev, ck, cv, _i32(cl), q, kn, vn, hint=hint)
        ck[0, 0, 1, at, 5] = bad
        out, lse = gpu_attn_step(dev, ck, cv, _i32(cl), q, kn, vn, hint=hint)
        assert dev.status() == 0
    undefined = torch.zeros(lse.shape, dtype=torch.bool, device="cuda")
    group = Hq // Hkv
    rows = q[0, 0, group:2 * group, :, 5].float()
    undefined[0, 0, group:2 * group] = True if bad != bad else rows > 0     # a score of -inf only takes the key out
    untouched = torch.ones_like(undefined)
    untouched[0, 0, group:2 * group] = False
    assert torch.equal(out.isnan().all(-1), undefined) and torch.equal(out.isnan().any(-1), undefined) and torch.equal(lse.isnan(), undefined)
    assert torch.equal(out[untouched], good[untouched]) and torch.equal(lse[untouched], good_lse[untouched])


# teams that are no cluster: two M tiles of heads of 128, whose pieces have no room in shared memory, and more blocks a unit than clusters of that
# size fit the device; ragged rows, an inactive element, blocks without a key tile; many launches, which leave the counters clean, and one that gives up
@pytest.mark.parametrize("NL,B,Hq,Hkv,D,q_cap,lc", [(1, 2, 28, 4, 128, 200, 2000), (2, 3, 8, 2, 128, 32, 5000), (8, 1, 28, 4, 128, 32, 5000), (2, 2, 8, 2, 64, 32, 10000)])
def test_teams_that_exchange_through_l2(dev, oracle, NL, B, Hq, Hkv, D, q_cap, lc):
    cap = lc + q_cap
    sch = _schedule(dev, NL, B, Hq, Hkv, D, cap, q_cap, NL, lc)
    # (of clusters of 10 and more the device runs 7 at a time)
    assert sch["team"] > 1 and sch["chunk_rows"] == 256 and (Hq // Hkv * q_cap > 128 and D == 128 or sch["team"] > 9 and sch["grid"] > 7 * sch["team"]), sch
    cl, ql = [lc, lc // 2 + 3, 0][:B], [q_cap, q_cap // 2, 1][:B]
    out, lse, _ = _case(dev, oracle, NL, B, Hq, Hkv, D, cap, q_cap, cl, ql, seed=NL, hint=lc, layers=[NL - 1])
    _case(dev, oracle, NL, B, Hq, Hkv, D, cap, q_cap, [0, lc, 17][:B], [1, 0, q_cap][:B], seed=NL + 1, hint=lc, layers=[0])
    ck, cv = make_cache(NL, B, Hkv, cap, D, NL)
    q, kn, vn = make_attn_inputs(NL, B, Hq, Hkv, q_cap, D, NL + 1)
    args = [t.cuda() for t in (ck, cv)] + [_i32(cl)] + [t.cuda() for t in (q, kn, vn)] + [_i32(ql)]
    dlm.dlm_selftest_set_wait_limit(dev.ctx, 0)
    try:
        gpu_attn_step(dev, *args, hint=lc)
        assert dev.status() == dlm.DLM_ERR_TIMEOUT
    finally:
        dlm.dlm_selftest_set_wait_limit(dev.ctx, 2_000_000_000)
    again = [gpu_attn_step(dev, *args, hint=lc) for _ in range(20)]
    assert dev.status() == 0
    for o, l in again:
        assert torch.equal(o, out) and torch.equal(l, lse)
