"""Backward pass (sh_backward, fp32 configuration) on the GPU against the backward oracle: dx and the gradients of
all six weight tensors, on the tiny workload and on shapes with a padded d_head, one and three selections,
without the causal mask; argument checks."""
import numpy as np
import pytest
import torch

from oracle.switchhead_backward import switchhead_backward
from paper_2312_07987_b200 import binding, inputs

pytestmark = pytest.mark.gpu
TOL = 2e-4          # max-abs error / RMS of the gradient: fp32 products, sums and atomics against fp64


def check(cfg, causal=True, batch=None, causal_after=None):
    inp = inputs.make_inputs(cfg, batch=batch)
    layer = binding.layer_from_inputs(inp)
    if not causal:
        layer.sh_set_causal(False)
    x = binding.to_device(inp.x, cfg.dtype)
    rg = np.random.default_rng(cfg.seed + 1)
    G = rg.standard_normal(inp.x.shape).astype(np.float32)
    layer.sh_forward(x)
    if causal_after is not None:
        layer.sh_set_causal(causal_after)
    got = layer.sh_backward(x, torch.from_numpy(G).cuda())
    torch.cuda.synchronize()
    assert layer.sh_last_status() == 0
    ref = switchhead_backward(inp.x, inp.Wq, inp.Wk, inp.Wv, inp.Wo, inp.Ws, inp.Wd, cfg.k, G, inp.bias_s, inp.bias_d, causal=causal)
    for name in ("dx", "dWq", "dWk", "dWv", "dWo", "dWs", "dWd"):
        a, r = got[name].cpu().numpy().astype(np.float64), ref[name]
        err = np.abs(a - r).max() / np.sqrt((r ** 2).mean())
        assert err < TOL, (name, err)
    layer.sh_check_guards()
    layer.close()


def test_backward_tiny_f32():
    check(inputs.CONFIGS["tiny_f32"])


@pytest.mark.parametrize("T,B,M,H,D,E,k,causal", [(70, 2, 128, 2, 40, 5, 3, True), (33, 3, 64, 3, 64, 4, 1, False), (150, 1, 192, 1, 132, 6, 2, True)])
def test_backward_shapes(T, B, M, H, D, E, k, causal):
    check(inputs.LayerConfig("bw", inputs.DTYPE_F32, B, T, M, H, D, E, k, seed=900 + T, zipf_bias=1.2 if E == 5 else 0.0), causal=causal)


@pytest.mark.parametrize("T,E,k", [(27, 32, 1), (5, 16, 3), (2, 16, 3)])
def test_backward_with_fewer_selections_than_experts(T, E, k):
    # (most experts' lists are empty: their gradients are zeros, which nothing but the kernel writes)
    cfg = inputs.LayerConfig("bw", inputs.DTYPE_F32, 1, T, 128, 3, 40, E, k, seed=930 + T)
    torch.full((1 << 24,), float("nan"), device="cuda")     # what the gradients' memory holds before
    check(cfg)


@pytest.mark.parametrize("causal", [True, False])
def test_backward_takes_the_mask_of_the_forward_pass(causal):
    # (sh_set_causal takes effect with the next forward pass)
    check(inputs.CONFIGS["tiny_f32"], causal=causal, causal_after=not causal)


def test_weights_loaded_again_keep_the_intermediates():
    # d_head 40 is stored as 64 columns
    inp = inputs.make_inputs(inputs.LayerConfig("bw", inputs.DTYPE_F32, 2, 70, 128, 2, 40, 5, 3, seed=970))
    layer = binding.layer_from_inputs(inp)
    x = binding.to_device(inp.x, inp.cfg.dtype)
    G = torch.ones(inp.x.shape, dtype=torch.float32, device="cuda")
    layer.sh_forward(x)
    want = layer.sh_backward(x, G)
    layer.sh_set_weights(*[binding.to_device(a, inp.cfg.dtype) for a in (inp.Wq, inp.Wk, inp.Wv, inp.Wo, inp.Ws, inp.Wd)])
    got = layer.sh_backward(x, G)
    for name, w in want.items():
        assert float((got[name] - w).abs().max() / w.abs().max()) < 1e-5, name      # (sums in another order)
    layer.close()


def test_backward_wants_the_intermediates_of_a_plain_pass_on_this_input():
    inp = inputs.make_inputs(inputs.CONFIGS["tiny_f32"])
    cfg = inp.cfg
    layer = binding.layer_from_inputs(inp)
    x = binding.to_device(inp.x, cfg.dtype)
    G = torch.ones(inp.x.shape, dtype=torch.float32, device="cuda")

    def refused():
        with pytest.raises(binding.SwitchHeadError, match="NOT_CONFIGURED"):
            layer.sh_backward(x, G)

    layer.sh_forward(x)
    layer.sh_gate_topk(x)                                  # the same selections once more
    layer.sh_set_rope(10000.0)                             # (for the next forward pass)
    layer.sh_set_rope(0.0)
    layer.sh_backward(x, G)
    other = x + 1
    layer.sh_gate_topk(other)                              # another input's selections
    refused()
    for positional in (True, False):
        layer.sh_set_rope(10000.0 if positional else 0.0)
        layer.sh_forward(x)
        layer.sh_set_rope(0.0)
        if positional:
            refused()
    layer.sh_backward(x, G)
    layer.sh_set_xl_positions(torch.zeros(cfg.n_heads, cfg.d_model, cfg.d_head, device="cuda"))
    layer.sh_forward(x)
    layer.sh_set_xl_positions(None)
    refused()
    layer.sh_forward(x)
    layer.sh_configure(cfg.dtype, *inp.x.shape[:2])        # a workspace without any pass's intermediates
    layer.sh_set_weights(*[binding.to_device(a, cfg.dtype) for a in (inp.Wq, inp.Wk, inp.Wv, inp.Wo, inp.Ws, inp.Wd)])
    refused()
    layer.close()


def test_backward_argument_checks():
    inp = inputs.make_inputs(inputs.CONFIGS["tiny_f32"])
    layer = binding.layer_from_inputs(inp)
    x = binding.to_device(inp.x, inp.cfg.dtype)
    G = torch.zeros(inp.x.shape, dtype=torch.float32, device="cuda")
    with pytest.raises(binding.SwitchHeadError):          # no forward pass on this x yet
        layer.sh_backward(x, G)
    layer.sh_forward(x)
    layer.sh_backward(x, G)
    layer.close()
    bf = binding.layer_from_inputs(inputs.make_inputs(inputs.CONFIGS["small_bf16"], batch=1))
    xb = binding.to_device(inputs.make_inputs(inputs.CONFIGS["small_bf16"], batch=1).x, inputs.DTYPE_BF16)
    bf.sh_forward(xb)
    with pytest.raises(binding.SwitchHeadError):          # tensor-core path: forward only
        bf.sh_backward(xb, torch.zeros((1, 256, 512), dtype=torch.float32, device="cuda"))
    bf.close()
