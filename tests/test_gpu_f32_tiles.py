"""The fp32 configuration's tensor-core GEMMs (split bf16), attention tiles and one-launch selection at the edges of
their tiles: d_head off the 16-column grid and across 64 / 128 columns, token counts around 32 / 64 / 128, more than one
selection sweep (1024 tokens), empty experts, split contractions, operands that are only 4-byte aligned."""
import numpy as np
import pytest
import torch

from oracle.switchhead_backward import switchhead_backward
from oracle.switchhead_oracle import switchhead_forward
from paper_2312_07987_b200 import binding, inputs

pytestmark = pytest.mark.gpu
# max-abs error / largest value (an expert nobody selects makes most of a gradient zero, and an RMS over it means
# nothing).  An fp32 sum of K products differs from the fp64 one by about sqrt(K) 2^-24 of its own size, times 5 for the
# largest of ~1e5 values: K <= 2100 tokens, 1.4e-5.
TOL = 1.4e-5


def run(B, T, M, H, D, E, k, causal=True, offset=0, zipf=0.0, change=None):
    cfg = inputs.LayerConfig("tiles", inputs.DTYPE_F32, B, T, M, H, D, E, k, seed=77 + T + D, zipf_bias=zipf)
    inp = inputs.make_inputs(cfg)
    G = np.random.default_rng(3).standard_normal(inp.x.shape).astype(np.float32)
    if change:
        change(inp, G)
    layer = binding.layer_from_inputs(inp)
    layer.sh_set_causal(causal)
    x = binding.to_device(inp.x, cfg.dtype)
    g = torch.empty(G.size + offset, dtype=torch.float32, device="cuda")[offset:].view(G.shape)
    g.copy_(torch.from_numpy(G))
    y = layer.sh_forward(x)
    got = layer.sh_backward(x, g)
    torch.cuda.synchronize()
    assert layer.sh_last_status() == 0
    layer.sh_check_guards()
    args = (inp.x, inp.Wq, inp.Wk, inp.Wv, inp.Wo, inp.Ws, inp.Wd, cfg.k)
    want = dict(switchhead_backward(*args, G, inp.bias_s, inp.bias_d, causal=causal))
    want["y"] = switchhead_forward(*args, inp.bias_s, inp.bias_d, causal=causal, return_stages=False)["y"]
    got["y"] = y
    for name in ("y", "dx", "dWq", "dWk", "dWv", "dWo", "dWs", "dWd"):
        a, r = got[name].cpu().numpy().astype(np.float64).reshape(want[name].shape), want[name]
        # (one token attends to itself alone: dQ and dK are exactly zero, and what is left of them is the rounding of
        #  two sums of order one)
        err = np.abs(a - r).max() / (np.abs(r).max() or 1.0)
        assert err < TOL, (name, err)
    layer.close()


@pytest.mark.parametrize("B,T,M,H,D,E,k", [
    (1, 1, 64, 1, 1, 1, 1),          # one of everything
    (1, 31, 64, 3, 17, 2, 1),        # d_head off the 16-column grid; fewer tokens than a tile
    (2, 33, 128, 1, 64, 3, 3),       # every expert selected; one token into the second query tile
    (1, 129, 192, 2, 65, 4, 2),      # one column into the second 64-column tile, one row into the second row tile
    (1, 127, 64, 1, 128, 2, 2),
    (1, 65, 448, 2, 129, 5, 2),      # 129: two 128-column tiles, the 256-wide attention kernels
    (3, 50, 128, 1, 256, 3, 1),
    (1, 2100, 64, 1, 40, 1, 1),      # three selection sweeps; contractions over tokens in parts
    (2, 600, 128, 2, 76, 32, 4),     # 32 experts, hardly a full tile among them
    (64, 64, 64, 1, 16, 3, 2),       # the most tokens of the one-block sort
    (41, 100, 64, 2, 16, 5, 2),      # ... and just past it: a block per 128 tokens
])
def test_f32_tile_edges(B, T, M, H, D, E, k):
    run(B, T, M, H, D, E, k)


def test_f32_empty_experts_and_no_mask():
    run(1, 200, 128, 2, 48, 8, 1, causal=False, zipf=4.0)


def test_f32_gradient_input_off_its_alignment():
    run(1, 90, 128, 2, 76, 4, 2, offset=1)


def large_weight(inp, G):
    inp.Wo[0, 0, 0, 0] = 3.4e38
    G *= 1e-3


def large_gradient(inp, G):
    G[0, 0, 0] = -3.4e38
    inp.Wo *= 1e-3                   # (no partial sum overflows)


@pytest.mark.parametrize("change", [large_weight, large_gradient])
def test_f32_values_past_the_largest_bf16(change):
    # (half a bf16 step past 3.3895e38; results and gradients stay finite)
    run(1, 90, 128, 2, 76, 4, 2, causal=False, change=change)


def test_f32_selection_of_an_input_off_its_alignment():
    cfg = inputs.LayerConfig("tiles", inputs.DTYPE_F32, 1, 70, 128, 2, 32, 4, 2, seed=5)
    inp = inputs.make_inputs(cfg)
    layer = binding.layer_from_inputs(inp)
    x = binding.to_device(inp.x, cfg.dtype)
    shifted = torch.empty(x.numel() + 1, dtype=torch.float32, device="cuda")[1:].view(x.shape)
    shifted.copy_(x)
    for a, b in zip(layer.sh_gate_topk(x), layer.sh_gate_topk(shifted)):
        assert torch.equal(a, b)
    layer.close()


@pytest.mark.parametrize("cache,shared,positions", [(0, False, False), (0, True, False), (64, False, True)])
def test_f32_output_in_place_of_the_input(cache, shared, positions):
    # the first rows of a larger x hold the output (with a cache there are fewer of them than tokens)
    cfg = inputs.LayerConfig("tiles", inputs.DTYPE_F32, 2, 300 + cache, 448, 2, 76, 5, 3, seed=17)
    inp = inputs.make_inputs(cfg)
    layer = binding.layer_from_inputs(inp, shared_selection=shared, cache_len=cache)
    if positions:
        g = torch.Generator(device="cuda").manual_seed(1)
        layer.sh_set_xl_positions(torch.randn(2, 448, 76, generator=g, device="cuda") / 21, None, None)
    x = binding.to_device(inp.x, cfg.dtype)
    want = layer.sh_forward(x)
    out = x.view(-1)[:want.numel()].view(want.shape)
    layer.sh_forward(x, out=out)
    assert float((out - want).abs().max() / want.abs().max()) < TOL
    layer.close()


@pytest.mark.parametrize("blocks", ["8 tokens", "16 tokens"])
@pytest.mark.parametrize("M,H,E,k", [
    (64, 1, 2, 1),                   # fewer gate columns than warps
    (512, 3, 16, 4),                 # 96: three rounds of 32
    (576, 2, 9, 3),                  # rows staged in 1024 columns, 36 gate columns
    (1088, 2, 4, 2),                 # one piece of 64 behind the first 1024
    (2112, 1, 17, 2),                # three pieces, two rounds
])
def test_f32_gate_kernel_sums_as_the_allocation_free_one(M, H, E, k, blocks):
    # blocks of 16 tokens from 32 tokens per SM on; every output bit for bit: both sum a logit in the same order
    N = 69 if blocks == "8 tokens" else 32 * torch.cuda.get_device_properties(0).multi_processor_count + 5
    g = torch.Generator(device="cuda").manual_seed(M + N)
    normal = lambda *shape: torch.randn(*shape, generator=g, device="cuda")
    W = [normal(H, M, E) / M ** 0.5 for _ in range(2)]
    bias = [normal(H, E) for _ in range(2)]
    layer = binding.Layer(M, H, 16, E, k)
    layer.sh_configure(binding.SH_F32, 1, N)
    layer.sh_set_weights(normal(H, M, 16), normal(H, M, 16), normal(H, E, M, 16), normal(H, E, 16, M), *W, *bias)
    x = normal(1, N, M)
    got = layer.sh_gate_topk(x)
    want = binding.sh_noalloc_gate_topk(binding.SH_F32, x[0], torch.cat([w.transpose(1, 2).reshape(H * E, M) for w in W]).contiguous(),
                                        torch.cat([b.reshape(-1) for b in bias]), H, E, k)
    for a, b in zip(got, want):
        assert torch.equal(a, b)
    layer.close()


@pytest.mark.parametrize("D", [32, 64, 128, 200])
def test_f32_overflow_of_one_token_stays_behind_the_mask(D):
    # finite inputs, but token 40's value row overflows (first column of x times that row of W_V): earlier rows of the
    # output never see it; then token 40's dAhat overflows: later rows of dx never see that
    B, T, M, H, E, k, t0 = 1, 100, 128, 2, 4, 2, 40
    inp = inputs.make_inputs(inputs.LayerConfig("tiles", inputs.DTYPE_F32, B, T, M, H, D, E, k, seed=31 + D))
    for W in (inp.Wq, inp.Wk, inp.Ws, inp.Wd):
        W[:, 0] = 0.0
    inp.Wv[:, :, 0] = 10.0
    inp.Wo[:, :, :, 0] = 10.0
    layer = binding.layer_from_inputs(inp)
    x = binding.to_device(inp.x, inp.cfg.dtype)
    G = torch.ones(B, T, M, device="cuda")
    close = lambda a, b: float((a - b).abs().max() / b.abs().max()) < TOL
    want_y, want_dx = layer.sh_forward(x), layer.sh_backward(x, G)["dx"]
    G[0, t0, 0] = 1e38
    dx = layer.sh_backward(x, G)["dx"]
    assert close(dx[:, t0 + 1:], want_dx[:, t0 + 1:]) and not bool(torch.isfinite(dx[:, :t0 + 1]).all())
    x[0, t0, 0] = 1e38
    y = layer.sh_forward(x)
    assert close(y[:, :t0], want_y[:, :t0]) and not bool(torch.isfinite(y[:, t0:]).all())
    layer.close()


def test_f32_forward_and_backward_in_a_captured_graph():
    cfg = inputs.LayerConfig("tiles", inputs.DTYPE_F32, 2, 150, 128, 2, 76, 4, 2, seed=23)
    inp = inputs.make_inputs(cfg)
    layer = binding.layer_from_inputs(inp)
    x = binding.to_device(inp.x, cfg.dtype)
    other = x.flip(1).contiguous()
    G = torch.ones_like(x)
    layer.sh_forward(other)
    want = dict(layer.sh_backward(other, G), y=layer.sh_forward(other))
    layer.sh_forward(x)
    layer.sh_backward(x, G)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        y = layer.sh_forward(x)
        got = dict(layer.sh_backward(x, G), y=y)
    x.copy_(other)
    for _ in range(3):
        graph.replay()
    torch.cuda.synchronize()
    for name, w in want.items():
        assert float((got[name] - w).abs().max() / w.abs().max()) < TOL, name
    assert layer.sh_last_status() == 0
    layer.close()
