"""fp32 attention of long sequences, forward on the tensor cores: the shortest sequence that takes it and its neighbours,
query tiles of 128 and key tiles of 64 with one row more or less, keys in parts (one query tile's up to as many as there are
SMs) and in one, stored widths of 32, 64 and 128 columns, no mask, a cache; scores and values that are not finite."""
import numpy as np
import pytest
import torch

from oracle.switchhead_backward import switchhead_backward
from oracle.switchhead_oracle import switchhead_forward, switchhead_xl_forward
from paper_2312_07987_b200 import binding, inputs

pytestmark = pytest.mark.gpu
# max-abs error / largest value: fp32 sums of up to K terms, sqrt(K) 2^-24 of their size, times 5 for the largest of
# ~1e5 values: K <= 1100, 1e-5
TOL = 1e-5


@pytest.mark.parametrize("B,T,H,D,causal", [
    (1, 320, 1, 32, True),           # the first length; three query tiles of six parts in all
    (1, 321, 2, 64, False),          # one key into the sixth key tile, no mask
    (2, 385, 1, 112, True),          # one row into the fourth query tile
    (1, 383, 3, 76, True),           # one row less than three
    (1, 1025, 1, 20, True),          # nine query tiles; five parts for the last one (the scratch holds no more)
    (40, 130, 2, 128, True),         # many heads: parts of the whole row, nothing to join
])
def test_f32_attention_parts(B, T, H, D, causal):
    M, E, k = 64, 2, 1
    cfg = inputs.LayerConfig("parts", inputs.DTYPE_F32, B, T, M, H, D, E, k, seed=T + D)
    inp = inputs.make_inputs(cfg)
    layer = binding.layer_from_inputs(inp)
    layer.sh_set_causal(causal)
    x = binding.to_device(inp.x, cfg.dtype)
    ones = np.ones(inp.x.shape, dtype=np.float32)
    y = [layer.sh_forward(x).cpu().numpy() for _ in range(3)]
    dx = layer.sh_backward(x, torch.from_numpy(ones).cuda())["dx"].cpu().numpy()      # (with the pass's maxima and normalisers)
    assert layer.sh_last_status() == 0
    layer.sh_check_guards()
    args = (inp.x, inp.Wq, inp.Wk, inp.Wv, inp.Wo, inp.Ws, inp.Wd, k)
    want = switchhead_forward(*args, inp.bias_s, inp.bias_d, causal=causal, return_stages=False)["y"]
    for got in y:
        assert np.abs(got - want).max() / np.abs(want).max() < TOL
    want = switchhead_backward(*args, ones, inp.bias_s, inp.bias_d, causal=causal)["dx"]
    assert np.abs(dx - want.reshape(dx.shape)).max() / np.abs(want).max() < TOL
    layer.close()


@pytest.mark.parametrize("D", [32, 64, 128])
@pytest.mark.parametrize("t0", [40, 300])
def test_f32_overflow_of_one_value_row_stays_behind_the_mask(D, t0):
    # finite inputs, but token t0's value row overflows (first column of x times that row of W_V): earlier rows never see it
    B, T, M, H, E, k = 1, 400, 128, 2, 4, 2
    inp = inputs.make_inputs(inputs.LayerConfig("parts", inputs.DTYPE_F32, B, T, M, H, D, E, k, seed=31 + D))
    for W in (inp.Wq, inp.Wk, inp.Ws, inp.Wd):
        W[:, 0] = 0.0
    inp.Wv[:, :, 0] = 10.0
    layer = binding.layer_from_inputs(inp)
    x = binding.to_device(inp.x, inp.cfg.dtype)
    want = layer.sh_forward(x)
    x[0, t0, 0] = 1e38
    y = layer.sh_forward(x)
    close = lambda a, b: float((a - b).abs().max() / b.abs().max()) < TOL
    assert close(y[:, :t0], want[:, :t0]) and not bool(torch.isfinite(y[:, t0:]).all())
    x.copy_(binding.to_device(inp.x, inp.cfg.dtype))
    assert close(layer.sh_forward(x), want)                 # and nothing of it is left behind
    layer.close()


@pytest.mark.parametrize("wk,wq", [(10.0, -5.0),                        # the key is infinite
                                   (1.0046875, -1.3e6)])                # it is finite, its products with the queries are not
@pytest.mark.parametrize("D", [32, 64, 128])
@pytest.mark.parametrize("T", [100, 400, 700])
def test_f32_score_of_minus_infinity_weighs_nothing(T, D, wk, wq):
    # one key's score overflows to minus infinity for every query that sees it: its weight is zero and the row stays finite
    M, H, E, k, t0 = 128, 2, 4, 2, 40
    inp = inputs.make_inputs(inputs.LayerConfig("parts", inputs.DTYPE_F32, 1, T, M, H, D, E, k, seed=57 + D + T))
    inp.x[0, :, 0] = 0.0
    inp.x[0, t0, 0] = 2.0 ** 126
    inp.x[0, :, 1] = 1.0
    for W in (inp.Wq, inp.Wk, inp.Ws, inp.Wd, inp.Wv):
        W[..., :2, :] = 0.0
    inp.Wq[:, :, 0] = inp.Wk[:, :, 0] = 0.0                 # the first position of q and k is made of x's first two columns alone
    inp.Wq[:, 1, 0] = wq
    inp.Wk[:, 0, 0] = wk
    layer = binding.layer_from_inputs(inp)
    y = layer.sh_forward(binding.to_device(inp.x, inp.cfg.dtype)).cpu().numpy()
    assert layer.sh_last_status() == 0
    layer.close()
    want = switchhead_forward(inp.x, inp.Wq, inp.Wk, inp.Wv, inp.Wo, inp.Ws, inp.Wd, k, inp.bias_s, inp.bias_d, return_stages=False)["y"]
    assert np.isfinite(want).all()
    assert np.abs(y - want).max() / np.abs(want).max() < TOL


def parts_of(B, T, Tc, H, D):
    """Parts of the last query tile's keys: two key tiles of 64 each or as many as keep the units at or below the number of SMs and their
    partial results (128 rows of the stored width and two values) in the backward pass's scratch, four rows of it a token and head."""
    Dp = 32 if D <= 32 else 64 if D <= 64 else 128
    tiles = [-(-min(T, Tc + 128 * (i + 1)) // 64) for i in range(-(-(T - Tc) // 128))]
    cap = min(torch.cuda.get_device_properties(0).multi_processor_count, 4 * B * T * H * Dp // (128 * (Dp + 2)))
    for per in range(2, -(-T // 64)):
        if sum(-(-n // per) for n in tiles) * B * H <= cap:
            return -(-tiles[-1] // per)
    return 1


@pytest.mark.parametrize("T,Tc,B,H,D,parts", [
    (330, 70, 1, 2, 76, 4),          # the cache ends inside a key tile, the chunk inside a query tile
    (129, 200, 2, 1, 32, 3),         # one row into the second query tile
    (1, 400, 1, 1, 112, 4),          # one query
    (33, 399, 10, 8, 64, 1),         # whole rows: nothing to join
    (100, 9000, 1, 1, 32, 72),       # the weights of many parts
    (100, 18840, 1, 1, 20, 148),     # as many as there are SMs
    (1, 400, 10, 8, 112, 0),         # one query for each of many heads: on the CUDA cores
    (32, 400, 19, 8, 32, 0),         # ... and 32 for more of them than there are SMs
])
def test_f32_attention_behind_a_cache(T, Tc, B, H, D, parts):
    M, E, k = 64, 2, 1
    if parts:
        assert parts_of(B, T + Tc, Tc, H, D) == parts
    cfg = inputs.LayerConfig("parts", inputs.DTYPE_F32, B, Tc + T, M, H, D, E, k, seed=T + Tc)
    inp = inputs.make_inputs(cfg)
    layer = binding.layer_from_inputs(inp, cache_len=Tc)
    x = binding.to_device(inp.x, cfg.dtype)
    y = [layer.sh_forward(x).cpu().numpy() for _ in range(2)]
    assert layer.sh_last_status() == 0
    layer.sh_check_guards()
    A = layer.sh_debug_buffer("AHAT").cpu().numpy().reshape(B, Tc + T, H, D)[:, Tc:]
    layer.close()
    # (the longest chain of additions is a thread's keys of a part, then the parts: shorter than the K of the bound)
    want = switchhead_xl_forward(inp.x[:, Tc:], inp.x[:, :Tc], inp.Wq, inp.Wk, inp.Wv, inp.Wo, inp.Ws, inp.Wd, k, inp.bias_s, inp.bias_d)
    assert np.abs(A - want["Ahat"]).max() / np.abs(want["Ahat"]).max() < TOL
    for got in y:
        assert np.abs(got - want["y"]).max() / np.abs(want["y"]).max() < TOL


@pytest.mark.parametrize("cache", [0, 70])
def test_f32_long_output_in_place_of_the_input(cache):
    cfg = inputs.LayerConfig("parts", inputs.DTYPE_F32, 2, 400 + cache, 128, 2, 76, 4, 2, seed=19)
    inp = inputs.make_inputs(cfg)
    layer = binding.layer_from_inputs(inp, cache_len=cache)
    x = binding.to_device(inp.x, cfg.dtype)
    want = layer.sh_forward(x)
    out = x.view(-1)[:want.numel()].view(want.shape)
    layer.sh_forward(x, out=out)
    assert float((out - want).abs().max() / want.abs().max()) < TOL
    layer.close()


def test_f32_long_sequence_with_rotary_positions_in_a_captured_graph():
    cfg = inputs.LayerConfig("parts", inputs.DTYPE_F32, 2, 400, 128, 2, 64, 4, 2, seed=23)
    inp = inputs.make_inputs(cfg)
    layer = binding.layer_from_inputs(inp)
    layer.sh_set_rope(10000.0)
    x = torch.zeros(inp.x.shape, device="cuda")
    layer.sh_forward(x)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        y = layer.sh_forward(x)
    x.copy_(binding.to_device(inp.x, cfg.dtype))
    want = switchhead_forward(inp.x, inp.Wq, inp.Wk, inp.Wv, inp.Wo, inp.Ws, inp.Wd, cfg.k, inp.bias_s, inp.bias_d, rope_base=10000.0,
                              return_stages=False)["y"]
    for _ in range(3):                                      # (the counters of a tile's parts go back to zero by themselves)
        y.fill_(7.0)
        graph.replay()
        assert np.abs(y.cpu().numpy() - want).max() / np.abs(want).max() < TOL
    del graph
    layer.close()
