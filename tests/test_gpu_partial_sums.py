"""Attention with the keys of a request split over CTAs keeps its partial sums in 32 bits: value rows of +64 and -64 cancel
across the ranges, and what is left is smaller than the bf16 rounding of a range's partial sum (16 at 6528 = 102 rows of 64)
but 1e4 times its fp32 rounding."""
import numpy as np
import pytest
import torch

from oracle import expert_oracle as O
from paper_2608_03682_b200 import binding, synth
from tests.helpers import small_bf16_config
from tests.test_gpu_attention_op import oracle_attention

pytestmark = pytest.mark.gpu


def cancelling_kv(seed, L, P, Hkv, dh):
    """[L, 2, P, Hkv, dh]: any keys; values +64 in the first half, -64 + d_c in the second, d_c a multiple of 1/4 up to 2."""
    gen = torch.Generator().manual_seed(seed)
    kv = torch.randn(L, 2, P, Hkv, dh, generator=gen)
    kv[:, 1] = 64.0
    kv[:, 1, (P + 1) // 2:] = -64.0 + torch.randint(1, 9, (L, 1, Hkv, dh), generator=gen) / 4.0
    if P % 2:
        kv[:, 1, P // 2] = 0.0
    return kv.bfloat16()


@pytest.mark.parametrize("Hq,Hkv,dh,S,lens", [(8, 1, 256, 51, [816]), (4, 1, 128, 64, [899, 301, 640]), (8, 1, 256, 51, [816] * 4),
                                             (8, 2, 128, 17, [967, 600, 816, 300, 555, 960, 728, 968]), (4, 1, 256, 33, [513] * 9)])
def test_attention_operator_partial_sums(Hq, Hkv, dh, S, lens):
    L, B = 2, len(lens)
    kv = torch.cat([cancelling_kv(b, L, p, Hkv, dh) for b, p in enumerate(lens)], dim=2)
    qkv = torch.randn(B * S, (Hq + 2 * Hkv) * dh, generator=torch.Generator().manual_seed(5))
    qkv[:, :Hq * dh] = 0.0                       # uniform probabilities: every P is exactly 1
    qkv[:, Hq * dh:] = qkv[:, Hq * dh:].bfloat16().float()
    cu = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
    desc = binding.attention_desc(Hq, Hkv, dh, S, n_layers=L, layer=1)
    out, status = binding.suffix_attention(desc, qkv.cuda(), kv.cuda(), torch.from_numpy(cu).cuda(), None)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    ref = oracle_attention(qkv, kv, cu, Hq, Hkv, dh, S, 1, 0.0)
    # result: one bf16 rounding; sums: at most 128 truncated additions of at most 968 x 64 = 2^16 (ulp 2^-8), over >= 318 keys
    bound = np.abs(ref) * 2.0 ** -8 + 128 * 2.0 ** -8 / (np.repeat(lens, S)[:, None] + S)
    assert (np.abs(out.double().cpu().numpy() - ref) <= bound).all(), (np.abs(out.double().cpu().numpy() - ref) / bound).max()


@pytest.mark.parametrize("head_dim,n_q,batch", [(256, 8, 2), (256, 8, 3), (128, 4, 5), (256, 8, 8)])
def test_loop_partial_sums(head_dim, n_q, batch):
    """The denoising loop's kernels for few requests, one layer, one step: a wide output projection makes the attention's
    output the larger part of the residual stream."""
    P = 640
    cfg = small_bf16_config("pi0", head_dim=head_dim, n_q_heads=n_q, n_kv_heads=1, max_batch=batch, max_prefix_len=P, n_layers=1, horizon=50)
    W = synth.make_weights(cfg, 71, std=0.05)
    W["wq.0"] = torch.zeros_like(W["wq.0"])
    W["wo.0"] = (W["wo.0"].float() * 8).bfloat16()
    kvs = [cancelling_kv(b, 1, P - 40 * b, 1, head_dim) for b in range(batch)]
    packed, cu = synth.pack_prefix_kv(kvs)
    states = torch.stack([synth.make_state(cfg, 71, b) for b in range(batch)])
    noise = torch.stack([synth.make_noise(cfg, 71, b) for b in range(batch)])
    with binding.Expert(cfg, binding.weights_to_device(W)) as ex:
        out = ex.denoise_batched(packed.cuda(), torch.from_numpy(cu).cuda(), states.cuda(), noise.cuda(), 1)
        torch.cuda.synchronize()
        assert ex.poll_status() == 0
    errs = []
    for b in range(batch):
        ref = O.denoise(cfg, O.Weights(W), kvs[b], P - 40 * b, states[b], noise[b], 1)
        errs.append(O.max_rel_err(out[b].double().cpu().numpy(), ref))
    assert max(errs) <= 2e-2, errs
