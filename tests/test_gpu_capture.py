"""Operator calls inside a captured CUDA graph: every call carries its own clearing of the status word, so that graphs may be
replayed in any order, and an error of one replay does not stick to the next."""
import subprocess
import sys

import pytest
import torch

from oracle import adapter_oracle as A
from paper_2608_03682_b200 import binding
from tests.test_gpu_attention_op import make_case, oracle_attention

pytestmark = pytest.mark.gpu


def attention_call(seed, Hq, Hkv, dh, S, lens):
    """(the call, its lengths on the device, a check of its output)"""
    qkv, kv, cu, rope = make_case(seed, Hq, Hkv, dh, S, lens)
    desc = binding.attention_desc(Hq, Hkv, dh, S, n_layers=2, layer=1)
    args = (desc, qkv.cuda(), kv.cuda(), torch.from_numpy(cu).cuda(), rope.cuda())
    ref = torch.from_numpy(oracle_attention(qkv, kv, cu, Hq, Hkv, dh, S, 1, 10000.0))

    def check(result):
        assert (result[0].double().cpu() - ref).abs().max() <= 2e-2 * ref.abs().max()
    return lambda: binding.suffix_attention(*args), args[3], check


def pack_call(seed, lens):
    gen = torch.Generator().manual_seed(seed)
    k, v = (torch.randn(2, len(lens), 40, 1, 64, generator=gen).bfloat16() for _ in range(2))
    args = (k.cuda(), v.cuda(), torch.tensor(lens, dtype=torch.int32, device="cuda"))
    ref, cu_ref = A.pack_prefix_kv(k.float().numpy(), v.float().numpy(), lens)

    def check(result):
        n = sum(lens)
        assert result[1].tolist() == list(cu_ref)
        assert torch.equal(result[0][:, :, :n].float().cpu(), torch.from_numpy(ref)) and (result[0][:, :, n:] == 0).all()
    return lambda: binding.pack_prefix_kv(*args), args[2], check


CALLS = {"tcgen05": (attention_call, (8, 1, 256, 17, [100]), (8, 1, 256, 17, [70, 40])),
         "mma.sync": (attention_call, (2, 1, 64, 17, [100]), (2, 1, 64, 17, [70, 40])),
         "kv-writer": (pack_call, ([40, 0, 7],), ([1, 39],))}


@pytest.mark.parametrize("kind", list(CALLS))
def test_captured_operator_calls_clear_their_own_status_word(kind):
    make, first, second = CALLS[kind]
    calls = [make(3, *first), make(4, *second)]
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        for call, _, check in calls:              # (kernels loaded, as by a program's warm-up)
            check(call())
    stream.synchronize()
    graphs, results = [], []
    for call, _, _ in calls:
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=stream):
            results.append(call())
        graphs.append(g)
    for i in (1, 0):                              # the graph captured second is replayed first
        _, lens, check = calls[i]
        good = lens.clone()
        for attempt in range(3):
            for t in results[i]:
                t.fill_(-3)
            lens.copy_(torch.full_like(lens, -1) if attempt == 1 else good)
            graphs[i].replay()
            torch.cuda.synchronize()
            status = int(results[i][-1].item())
            assert status == (binding.ERR_INVALID_ARG if attempt == 1 else 0), (i, attempt)
            if attempt != 1:
                check(results[i])


def test_first_operator_call_of_a_process_may_be_a_captured_one():
    code = """
import torch
from tests.test_gpu_capture import attention_call
call, _, check = attention_call(3, 8, 1, 256, 17, [100])
stream, g = torch.cuda.Stream(), torch.cuda.CUDAGraph()
with torch.cuda.graph(g, stream=stream):
    result = call()
g.replay()
torch.cuda.synchronize()
assert int(result[1].item()) == 0
check(result)
"""
    r = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
