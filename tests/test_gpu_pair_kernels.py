"""The kernels on CTA pairs (calls of more than 64 suffix tokens) against the oracle, at the edges of their tiles: token
counts around the 32-token steps of the tile width, one and several tiles per pair, every key-range split of the attention
kernel, prefixes with no full key tile, exactly one, and empty ranges; reproducible to the bit."""
import numpy as np
import pytest
import torch

from oracle import expert_oracle as O
from paper_2608_03682_b200 import binding, synth
from tests.helpers import BAR, rel_err, small_bf16_config

pytestmark = pytest.mark.gpu


def check(cfg, lens, n_steps, which, cfg_id=51, std=0.05, **options):
    batch = len(lens)
    W = synth.make_weights(cfg, cfg_id, std=std)
    kvs = [synth.make_prefix_kv(cfg, cfg_id, p, b) for b, p in enumerate(lens)]
    packed, cu = synth.pack_prefix_kv(kvs)
    states = torch.stack([synth.make_state(cfg, cfg_id, b) for b in range(batch)]) if cfg.has_state_token else None
    noise = torch.stack([synth.make_noise(cfg, cfg_id, b) for b in range(batch)])
    args = (packed.cuda(), torch.from_numpy(cu).cuda(), None if states is None else states.cuda(), noise.cuda(), n_steps)
    with binding.Expert(cfg, binding.weights_to_device(W)) as ex:
        for k, v in options.items():
            ex.set_option(k, v)
        out = ex.denoise_batched(*args).clone()
        again = ex.denoise_batched(*args)
        torch.cuda.synchronize()
        assert ex.poll_status() == 0 and torch.equal(out, again)
    Wf = O.Weights(W)
    for b in which:
        ref = O.denoise(cfg, Wf, kvs[b], lens[b], None if states is None else states[b], noise[b], n_steps)
        err = rel_err(out[b].double().cpu().numpy(), ref)
        assert err <= BAR["bf16"], (b, lens[b], err)


@pytest.mark.parametrize("cond,dtype,horizon,batch", [("pi0", "bf16", 12, 5), ("pi0", "bf16", 31, 3), ("pi05", "bf16", 33, 2),
                                                       ("pi05", "w8e4m3", 43, 3), ("pi0", "w4a16", 50, 11), ("pi0", "bf16", 63, 33)])
def test_pair_gemms_at_the_edges_of_their_token_tiles(cond, dtype, horizon, batch):
    cfg = small_bf16_config(cond, dtype=dtype, horizon=horizon, max_batch=batch, max_prefix_len=120, n_q_heads=4, mlp_dim=1024)
    check(cfg, [(37 * b) % 121 for b in range(batch)], 2, {0, batch // 2, batch - 1})


@pytest.mark.parametrize("cond,dtype,width,mlp,horizon,batch", [
    ("pi0", "bf16", 256, 512, 1, 1), ("pi05", "w8e4m3", 512, 1024, 16, 4), ("pi0", "w4a16", 384, 640, 15, 3),
    ("pi05", "bf16", 1024, 4096, 33, 1), ("pi0", "w8e4m3", 1024, 1152, 63, 1), ("pi0", "bf16", 1152, 1280, 20, 3)])
def test_single_tile_projections_on_pairs(cond, dtype, width, mlp, horizon, batch):
    """Fewest and most tokens of the tile, uneven k-ranges, all three weight codings, contractions up to and past one pair's
    (past it: both kernel families in one layer)."""
    cfg = small_bf16_config(cond, dtype=dtype, width=width, mlp_dim=mlp, horizon=horizon, max_batch=batch, max_prefix_len=200)
    for pair in (1, 0):
        check(cfg, [(200, 77, 0, 128)[b] for b in range(batch)], 2, range(batch), use_b1_pair=pair)


@pytest.mark.parametrize("cond,action_dim,width,horizon,batch", [("pi05", 33, 768, 60, 20), ("pi0", 7, 1280, 37, 32), ("pi05", 1, 256, 61, 2)])
def test_step_boundary_row_groups(cond, action_dim, width, horizon, batch):
    """Sixteen rows per block from 1185 action rows on, four below; ragged last groups; action widths around a warp's lanes."""
    cfg = small_bf16_config(cond, action_dim=action_dim, width=width, horizon=horizon, max_batch=batch, max_prefix_len=40, n_layers=2)
    check(cfg, [(13 * b) % 41 for b in range(batch)], 3, {0, batch - 1})


@pytest.mark.parametrize("head_dim,n_q,n_kv", [(256, 4, 1), (128, 8, 2)])
@pytest.mark.parametrize("ranges", [1, 2, 3, 4])
def test_pair_attention_key_ranges(head_dim, n_q, n_kv, ranges):
    cfg = small_bf16_config("pi0", head_dim=head_dim, n_q_heads=n_q, n_kv_heads=n_kv, max_batch=9, max_prefix_len=700, n_layers=2,
                            suffix_block_causal=ranges % 2 == 0)
    check(cfg, [700, 0, 1, 127, 128, 129, 512, 64, 386], 1, range(9), pair_attn_ranges=ranges)


@pytest.mark.parametrize("head_dim,n_q,n_kv,batch,horizon,top", [(256, 8, 1, 75, 12, 520), (128, 8, 2, 190, 50, 300), (256, 4, 1, 149, 63, 120)])
def test_attention_of_many_requests(head_dim, n_q, n_kv, batch, horizon, top):
    """More (request, head group) items than CTA pairs: two to six per pair, of one to five key tiles (no prefix, one key, whole and
    partial blocks of 64 keys, an odd and an even number of blocks), the last round of items incomplete."""
    cfg = small_bf16_config("pi0", head_dim=head_dim, n_q_heads=n_q, n_kv_heads=n_kv, max_batch=batch, max_prefix_len=top, n_layers=2,
                            horizon=horizon, suffix_block_causal=n_kv == 2)
    lens = [min(top, (0, 1, 63, 64, 65, top, 127, 128, 129)[b % 9]) if b < 18 else (53 * b) % (top + 1) for b in range(batch)]
    check(cfg, lens, 1, [*range(0, 18, 2), batch // 2, batch - 2, batch - 1])


@pytest.mark.parametrize("head_dim,n_q,n_kv,batch", [(256, 8, 1, 45), (128, 8, 2, 60), (256, 8, 1, 8), (128, 8, 2, 13)])
def test_rows_around_a_prefix_have_no_part_in_its_request(head_dim, n_q, n_kv, batch):
    """What lies around a prefix (every third request's cache is NaN or infinite, and so are the rows before the first one and behind the
    last) leaves the other requests' actions as they are, to the bit; a first block that would begin before the cache.  Rows that threads of
    both CTAs of a pair clear or store themselves, with one key range per request and with several."""
    cfg = small_bf16_config("pi0", head_dim=head_dim, n_q_heads=n_q, n_kv_heads=n_kv, max_batch=batch, max_prefix_len=300, n_layers=2, horizon=12)
    W = synth.make_weights(cfg, 53, std=0.05)
    lens = [(1, 63, 64, 65, 130, 300, 0, 191)[b % 8] for b in range(batch)]
    packed, cu = synth.pack_prefix_kv([synth.make_prefix_kv(cfg, 53, p, b) for b, p in enumerate(lens)])
    packed = torch.cat([torch.zeros_like(packed[:, :, :30]), packed, torch.zeros_like(packed[:, :, :70])], dim=2)
    cu = cu + np.int32(30)
    dirty = packed.clone()
    dirty[:, :, :30], dirty[:, :, int(cu[-1]):] = float("nan"), float("nan")
    for b in range(1, batch, 3):
        dirty[:, :, cu[b]:cu[b + 1]] = float("nan") if b % 2 else float("inf")
    states = torch.stack([synth.make_state(cfg, 53, b) for b in range(batch)]).cuda()
    noise = torch.stack([synth.make_noise(cfg, 53, b) for b in range(batch)]).cuda()
    with binding.Expert(cfg, binding.weights_to_device(W)) as ex:
        clean = ex.denoise_batched(packed.cuda(), torch.from_numpy(cu).cuda(), states, noise, 2).clone()
        out = ex.denoise_batched(dirty.cuda(), torch.from_numpy(cu).cuda(), states, noise, 2)
        torch.cuda.synchronize()
        assert ex.poll_status() == 0 and clean.isfinite().all()
    for b in range(batch):
        if b % 3 != 1 or lens[b] == 0:
            assert torch.equal(out[b], clean[b]), (b, lens[b])


@pytest.mark.parametrize("head_dim,n_kv", [(256, 1), (128, 2)])
def test_infinite_values_among_the_keys_of_a_partial_block(head_dim, n_kv):
    """The 64 rows that a partial last block is fetched from begin with keys of the block before: an infinite value there (and one among the
    block's own keys, and in a prefix of fewer than 64) gives its channel an infinite result and leaves the others as they are."""
    from tests.test_gpu_attention_op import make_case
    lens = [(130, 65, 191, 40, 127)[b % 5] for b in range(90)]
    qkv, kv, cu, _ = make_case(14, 4 * n_kv, n_kv, head_dim, 33, lens, theta=0.0)
    dirty = kv.clone()
    for b in range(0, 90, 2):
        dirty[1, 1, cu[b] + (100, 5, 180, 20, 64)[b % 5], :, 3] = float("inf")
        dirty[1, 1, cu[b + 1] - 1, :, 70] = float("-inf")
    desc = binding.attention_desc(4 * n_kv, n_kv, head_dim, 33, n_layers=2, layer=1)
    clean, out = (binding.suffix_attention(desc, qkv.cuda(), x.cuda(), torch.from_numpy(cu).cuda(), None)[0].view(90, 33, 4 * n_kv, head_dim) for x in (kv, dirty))
    torch.cuda.synchronize()
    want = clean.clone()
    want[::2, :, :, 3], want[::2, :, :, 70] = float("inf"), float("-inf")
    assert clean.isfinite().all() and torch.equal(out, want)


@pytest.mark.parametrize("horizon", [59, 60, 62, 63])
@pytest.mark.parametrize("ranges", [2, 3, 4])
def test_pair_attention_at_the_most_suffix_rows(ranges, horizon):
    """The fp32 partials of heads of 256 channels fit the shared memory for four ranges up to 60 rows, three up to 63 (one state
    token and the horizon): more ranges than that are reduced, and the fullest layouts are right to the last row."""
    cfg = small_bf16_config("pi0", head_dim=256, n_q_heads=4, max_batch=5, max_prefix_len=400, n_layers=2, horizon=horizon)
    check(cfg, [400, 0, 129, 256, 33], 1, range(5), pair_attn_ranges=ranges)


@pytest.mark.parametrize("head_dim,n_q,n_kv,lens", [(256, 4, 1, [960, 0, 1, 7, 8, 511, 959]), (128, 8, 2, [700, 129, 64]), (128, 4, 1, [256] * 7)])
def test_attention_of_a_few_requests(head_dim, n_q, n_kv, lens):
    """The library's own choice of key ranges for few requests (63 and 64 suffix rows: with 256 channels not four of them), empty and
    one-key ranges, a full last tile."""
    cfg = small_bf16_config("pi0", head_dim=head_dim, n_q_heads=n_q, n_kv_heads=n_kv, max_batch=len(lens), max_prefix_len=max(lens),
                            n_layers=2, horizon=63, suffix_block_causal=n_kv == 2)
    check(cfg, lens, 1, range(len(lens)))


@pytest.mark.parametrize("n_kv,head_dim,suffix,lens", [(1, 256, 51, [700, 0, 129]), (1, 256, 64, [1100]), (1, 256, 1, [0]), (1, 256, 64, [(53 * b) % 300 for b in range(40)]),
                                                      (2, 128, 17, [128] * 45)])
def test_attention_operator_on_the_pair_kernel(n_kv, head_dim, suffix, lens):
    """The library's own choice of kernel: one request (cluster kernel; two key tiles per range, no prefix), split key ranges, one range
    per request (row-major output), 128-channel heads."""
    from tests.test_gpu_attention_op import make_case, oracle_attention
    qkv, kv, cu, rope = make_case(9, 8, n_kv, head_dim, suffix, lens)
    desc = binding.attention_desc(8, n_kv, head_dim, suffix, n_layers=2, layer=1)
    out, status = binding.suffix_attention(desc, qkv.cuda(), kv.cuda(), torch.from_numpy(cu).cuda(), rope.cuda())
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    ref = oracle_attention(qkv, kv, cu, 8, n_kv, head_dim, suffix, 1, 10000.0)
    assert abs(out.double().cpu().numpy() - ref).max() <= 2e-2 * abs(ref).max()


@pytest.mark.parametrize("n_q,n_kv,head_dim,suffix,lens", [
    (8, 1, 256, 51, [816, 400, 130]), (8, 2, 128, 17, [700, 64, 1, 513, 250]), (8, 1, 256, 51, [(97 * b) % 900 for b in range(8)]),
    (8, 1, 256, 33, [600 + 13 * b for b in range(14)]),
    (4, 1, 256, 51, [(67 * b) % 500 for b in range(100)] + [(5 * b) % 65 for b in range(60)]), (8, 2, 128, 64, [(41 * b) % 420 for b in range(90)])])
def test_logits_that_grow_over_the_keys(n_q, n_kv, head_dim, suffix, lens):
    """Half of the rows see logits that grow by 11.5 (log2) with every 64 keys, up to the request's own: their accumulators are rescaled in
    every tile, beside rows that keep theirs.  Split key ranges, and several items per pair with prefixes of less than a tile last."""
    from tests.test_gpu_attention_op import oracle_attention
    rng = np.random.default_rng(12)
    B, T, scale = len(lens), sum(lens), head_dim ** -0.5
    u = rng.choice([-1.0, 1.0], head_dim)
    level = np.concatenate([8.0 * (np.arange(p) // 64) for p in lens])
    kv = rng.standard_normal((1, 2, T, n_kv, head_dim))
    kv[0, 0] += level[:, None, None] * u
    qkv = rng.standard_normal((B * suffix, n_q + 2 * n_kv, head_dim))
    qkv[:, :n_q] = rng.choice([-1.0, 1.0], (B * suffix, n_q, 1)) * u / (head_dim * scale)    # (scaled: exact in bf16; logit = +-level + noise)
    qkv[:, n_q:n_q + n_kv] += np.repeat([8.0 * ((p + 63) // 64) for p in lens], suffix)[:, None, None] * u
    kv = torch.from_numpy(kv).bfloat16()
    qkv = torch.from_numpy(qkv.reshape(B * suffix, -1)).float()
    qkv[:, n_q * head_dim:] = qkv[:, n_q * head_dim:].bfloat16().float()
    cu = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
    desc = binding.attention_desc(n_q, n_kv, head_dim, suffix, n_layers=1, layer=0)
    args = (desc, qkv.cuda(), kv.cuda(), torch.from_numpy(cu).cuda(), None)
    outs = [binding.suffix_attention(*args) for _ in range(8)]
    torch.cuda.synchronize()
    for out, status in outs:
        assert int(status.item()) == 0 and torch.equal(out, outs[0][0])
    ref = oracle_attention(qkv, kv, cu, n_q, n_kv, head_dim, suffix, 0, 0.0)
    qkv[:, (n_q + n_kv) * head_dim:].abs_(), kv[:, 1].abs_()
    mean_abs = oracle_attention(qkv, kv, cu, n_q, n_kv, head_dim, suffix, 0, 0.0)
    # P: one bf16 rounding (2^-9); logits of at most 2^7 in 16 truncated accumulations (2^-16 each, in product and sum: 2^-11); the result: one
    # bf16 rounding
    bound = mean_abs * 2.0 ** -8 + np.abs(ref) * 2.0 ** -8
    assert (np.abs(outs[0][0].double().cpu().numpy() - ref) <= bound).all(), (np.abs(outs[0][0].double().cpu().numpy() - ref) / bound).max()


@pytest.mark.parametrize("head_dim,n_kv,batch", [(256, 1, 150), (128, 1, 150), (256, 1, 301)])
def test_items_of_one_tile_at_the_end_of_a_pairs_list(head_dim, n_kv, batch):
    """The last two or three items of a pair are a long prefix and ones of a single tile: their outputs follow one another without a
    softmax in between.  Zero queries: every sum is the number of keys, 17 to 81 in the last items and 400 and more in those before."""
    from tests.test_gpu_attention_op import make_case, oracle_attention
    lens = [400 + b % 60 if b < batch // 2 else (b * 5) % 65 for b in range(batch)]
    qkv, kv, cu, _ = make_case(13, 4, n_kv, head_dim, 17, lens, theta=0.0)
    qkv[:, :4 * head_dim] = 0.0
    qkv[:, 4 * head_dim:] = qkv[:, 4 * head_dim:].bfloat16().float()
    desc = binding.attention_desc(4, n_kv, head_dim, 17, n_layers=2, layer=1)
    args = (desc, qkv.cuda(), kv.cuda(), torch.from_numpy(cu).cuda(), None)
    outs = [binding.suffix_attention(*args) for _ in range(8)]
    torch.cuda.synchronize()
    for out, status in outs:
        assert int(status.item()) == 0 and torch.equal(out, outs[0][0])
    ref = oracle_attention(qkv, kv, cu, 4, n_kv, head_dim, 17, 1, 0.0)
    # (P is exactly 1; at most 36 truncated additions of at most 2^9 x 4: 2^-12 each, over at least 17 keys; one bf16 rounding)
    assert (np.abs(outs[0][0].double().cpu().numpy() - ref) <= np.abs(ref) * 2.0 ** -8 + 36 * 2.0 ** -12 / 17).all()


@pytest.mark.parametrize("tokens,n_kv,dh,layers,shift", [(1, 1, 64, 3, 0), (65, 3, 64, 1, 4), (641, 1, 128, 5, 0), (200, 1, 192, 2, 4)])
def test_feature_projection_of_all_layers(tokens, n_kv, dh, layers, shift):
    """Row counts that leave the last 256 padded, warps whose 32 rows end a plane, planes at an 8-byte-aligned address."""
    from oracle import adapter_oracle as A
    F = synth.make_features(44, tokens, 192)
    g = torch.Generator().manual_seed(44)
    wk, wv = ([torch.randn(192, n_kv * dh, generator=g).mul(192 ** -0.5).bfloat16() for _ in range(layers)] for _ in range(2))
    n = layers * 2 * (tokens + 3) * n_kv * dh
    out = torch.full((n + 2 * shift,), 7.0, dtype=torch.bfloat16, device="cuda")
    planes = out[shift:shift + n].view(layers, 2, tokens + 3, n_kv, dh)
    with binding.KvProjector([w.cuda() for w in wk], [w.cuda() for w in wv], n_kv, dh, max_tokens=tokens) as proj:
        proj.run(F.cuda(), out=planes)
        torch.cuda.synchronize()
    ref = torch.from_numpy(A.project_features_kv(F.double().numpy(), [w.double().numpy() for w in wk], [w.double().numpy() for w in wv], n_kv, dh))
    got = planes.double().cpu()
    assert (got[:, :, tokens:] == 7).all() and (out[:shift] == 7).all() and (out[shift + n:] == 7).all()
    assert ((got[:, :, :tokens] - ref).abs() <= ref.abs() * 2.0 ** -8 + 1e-4).all()
