"""The few-row fp32 kernels against the oracle at the edges of their ranges: widths that leave ragged contraction ranges
and columns, one row, the switch from four to eight rows per block (64 rows), and the switch to the tiled kernel (512)."""
import pytest
import torch

from oracle import expert_oracle as O
from paper_2608_03682_b200 import binding, synth
from tests.helpers import BAR, rel_err

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("horizon,batch,width,mlp,head_dim,cond", [(1, 1, 36, 50, 12, "pi05"), (15, 1, 130, 66, 20, "pi0"),
                                                                  (15, 4, 64, 1028, 32, "pi0"), (12, 5, 64, 96, 16, "pi0"),
                                                                  (63, 8, 32, 40, 8, "pi05"), (64, 8, 32, 40, 8, "pi0")])
def test_few_row_fp32_kernels_match_oracle(horizon, batch, width, mlp, head_dim, cond):
    cfg = synth.ExpertConfig(n_layers=2, width=width, mlp_dim=mlp, n_q_heads=2, n_kv_heads=1, head_dim=head_dim, state_dim=3,
                             action_dim=5, horizon=horizon, has_state_token=cond == "pi0", max_prefix_len=70, max_batch=batch,
                             cond=cond, dtype="f32", suffix_block_causal=cond == "pi0")
    W = synth.make_weights(cfg, 61, std=0.08)
    lens = [(70 - 23 * b) % 71 for b in range(batch)]
    kvs = [synth.make_prefix_kv(cfg, 61, p, b) for b, p in enumerate(lens)]
    packed, cu = synth.pack_prefix_kv(kvs)
    states = torch.stack([synth.make_state(cfg, 61, b) for b in range(batch)]) if cfg.has_state_token else None
    noise = torch.stack([synth.make_noise(cfg, 61, b) for b in range(batch)])
    with binding.Expert(cfg, binding.weights_to_device(W)) as ex:
        out = ex.denoise_batched(packed.cuda(), torch.from_numpy(cu).cuda(), None if states is None else states.cuda(), noise.cuda(), 2)
        torch.cuda.synchronize()
        assert ex.poll_status() == 0
    Wf = O.Weights(W)
    for b in {0, batch - 1}:
        ref = O.denoise(cfg, Wf, kvs[b], lens[b], None if states is None else states[b], noise[b], 2)
        assert rel_err(out[b].double().cpu().numpy(), ref) <= BAR["f32"], b


def run_case(cfg_id, horizon, batch, width, mlp, n_q, head_dim, cond, action_dim, prefix, theta, n_steps):
    cfg = synth.ExpertConfig(n_layers=2, width=width, mlp_dim=mlp, n_q_heads=n_q, n_kv_heads=1, head_dim=head_dim, state_dim=3,
                             action_dim=action_dim, horizon=horizon, has_state_token=cond == "pi0", max_prefix_len=max(1, prefix),
                             rope_theta=theta, max_batch=batch, cond=cond, dtype="f32", suffix_block_causal=cond == "pi0")
    W = synth.make_weights(cfg, cfg_id, std=0.08)
    lens = [(prefix - 23 * b) % (prefix + 1) for b in range(batch)]
    kvs = [synth.make_prefix_kv(cfg, cfg_id, p, b) for b, p in enumerate(lens)]
    packed, cu = synth.pack_prefix_kv(kvs)
    states = torch.stack([synth.make_state(cfg, cfg_id, b) for b in range(batch)]) if cfg.has_state_token else None
    noise = torch.stack([synth.make_noise(cfg, cfg_id, b) for b in range(batch)])
    with binding.Expert(cfg, binding.weights_to_device(W)) as ex:
        out = ex.denoise_batched(packed.cuda(), torch.from_numpy(cu).cuda(), None if states is None else states.cuda(), noise.cuda(), n_steps)
        torch.cuda.synchronize()
        assert ex.poll_status() == 0
    Wf = O.Weights(W)
    for b in {0, batch - 1}:
        ref = O.denoise(cfg, Wf, kvs[b], lens[b], None if states is None else states[b], noise[b], n_steps)
        assert rel_err(out[b].double().cpu().numpy(), ref) <= BAR["f32"], b


@pytest.mark.parametrize("horizon,batch,width,mlp,n_q,head_dim,cond,theta,action_dim,prefix", [
    (47, 1, 36, 44, 2, 4, "pi0", 1e4, 5, 70), (48, 1, 100, 132, 1, 12, "pi0", 1e4, 5, 33), (1, 1, 4, 4, 3, 256, "pi05", 0.0, 1, 300),
    (16, 3, 676, 1028, 2, 64, "pi05", 1e4, 33, 129), (25, 10, 260, 520, 4, 64, "pi0", 1e4, 7, 64), (32, 8, 64, 64, 2, 128, "pi0", 0.0, 256, 0)])
def test_rolled_fp32_kernels_match_oracle(horizon, batch, width, mlp, n_q, head_dim, cond, theta, action_dim, prefix):
    """Four and eight rows to a block (48 and 49 rows), contractions that some warps have no part of, that end within a range and that
    do not fit the shared memory, ragged column blocks, heads of one and of many channel groups, no and many keys, an action per
    lane and more; 256 action rows (the most for a block per row) and 250 of them."""
    run_case(62, horizon, batch, width, mlp, n_q, head_dim, cond, action_dim, prefix, theta, 3)
