"""Device memory of a handle: the weight images its default kernels read, and no others."""
import pytest
import torch

from paper_2608_03682_b200 import binding, synth
from tests.helpers import gpu_single

pytestmark = pytest.mark.gpu


def free_bytes():
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return torch.cuda.mem_get_info()[0]


@pytest.mark.parametrize("dtype", ["bf16", "w8e4m3", "w4a16"])
@pytest.mark.parametrize("batch", [1, 8])
def test_handle_keeps_the_images_its_kernels_read(dtype, batch):
    cfg = synth.ExpertConfig(n_layers=6, width=1024, mlp_dim=4096, n_q_heads=8, n_kv_heads=1, head_dim=256, state_dim=32, action_dim=32,
                             horizon=50, has_state_token=True, max_prefix_len=300, max_batch=batch, cond="pi0", dtype=dtype)
    W = binding.weights_to_device(synth.make_weights(cfg, 61))
    binding.Expert(cfg, W).close()                        # (the library's kernels are loaded)
    before = free_bytes()
    with binding.Expert(cfg, W) as ex:
        used = before - free_bytes()
        qkv, o, gate_up, down = 1024 * 2560, 2048 * 1024, 2 * 1024 * 4096, 4096 * 1024
        # calls of more than 64 tokens read q|k|v and gate|up in another row order; the rest: workspaces and tables (70 MB at 8)
        images = 6 * 2 * (qkv + o + gate_up + down + (qkv + gate_up if batch > 1 else 0))
        assert images <= used <= images + (96 << 20), (used, images)
        kv, state, noise = synth.make_prefix_kv(cfg, 61, 300), synth.make_state(cfg, 61), synth.make_noise(cfg, 61)
        call = lambda: torch.from_numpy(gpu_single(cfg, W, kv, 300, state, noise, 2, expert=ex))
        out = call()
        for key, value, default in (("use_w8_inkernel", 1, 0), ("use_pair_gemm", 0, 1)):     # images made when an option asks for them
            ex.set_option(key, value)
            got = call()
            assert (got - out).abs().max() <= 2e-2 * out.abs().max()
            assert key != "use_w8_inkernel" or torch.equal(got, out)
            ex.set_option(key, default)
