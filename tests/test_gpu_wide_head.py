"""bf16 storage with d_head above 128 (256 stored columns): the attention kernel's 64-key steps and 128-query tiles, the
16-column slices and 64-column blocks that d_head reaches, with rotary positions, without the mask, with more selections
than the output projection's shared memory holds, and with more gate columns than the tensor-core gate kernel takes."""
import numpy as np
import pytest
import torch

from paper_2312_07987_b200 import binding, inputs
from tests import parity_util as pu
from tests.test_gpu_parity import full_check

pytestmark = pytest.mark.gpu


def config(B, T, M, H, D, E, k, seed=0):
    return inputs.LayerConfig("wide", inputs.DTYPE_BF16, B, T, M, H, D, E, k, seed=500 + D + T + seed)


@pytest.mark.parametrize("D", [129, 144, 145, 160, 161, 176, 192, 193, 224, 256])
def test_widths(D):
    full_check(inputs.make_inputs(config(2, 130, 128, 2, D, 4, 2)))


@pytest.mark.parametrize("T", [1, 63, 64, 65, 127, 128, 129, 257])
def test_lengths(T):
    full_check(inputs.make_inputs(config(2, T, 256, 1, 132, 3, 2)))


@pytest.mark.parametrize("H,E,k", [(1, 1, 1), (3, 16, 4), (12, 4, 3), (8, 17, 2)])
def test_heads_experts_and_selections(H, E, k):
    # (12 x 3 selections a token: read from global memory; 2 x 8 x 17 gate columns: the CUDA-core gate kernel)
    full_check(inputs.make_inputs(config(1, 150, 128, H, 168, E, k)))


@pytest.mark.parametrize("causal,rope", [(False, None), (True, 10000.0), (False, 10000.0)])
def test_mask_and_rotary_positions(causal, rope):
    inp = inputs.make_inputs(config(2, 200, 256, 2, 132, 4, 2))
    layer = binding.layer_from_inputs(inp)
    layer.sh_set_causal(causal)
    if rope:
        layer.sh_set_rope(rope)
    y = layer.sh_forward(binding.to_device(inp.x, inp.cfg.dtype)).cpu().numpy()
    assert layer.sh_last_status() == 0
    ref = pu.oracle_for(inp, rope_base=rope, causal=causal)["y"]
    assert pu.rel_rms_err(y, ref) < pu.TOL_Y[inputs.DTYPE_BF16]
    layer.sh_check_guards()
    layer.close()


def test_half_precision_output_stays_refused():
    inp = inputs.make_inputs(config(1, 64, 128, 1, 132, 2, 1))
    layer = binding.layer_from_inputs(inp)
    layer.sh_set_output_f16(True)
    with pytest.raises(binding.SwitchHeadError):
        layer.sh_forward(binding.to_device(inp.x, inp.cfg.dtype))
    layer.close()


def test_selection_of_an_input_off_its_alignment():
    inp = inputs.make_inputs(config(1, 70, 128, 2, 132, 4, 2))
    layer = binding.layer_from_inputs(inp)
    x = binding.to_device(inp.x, inp.cfg.dtype)
    shifted = torch.empty(x.numel() + 1, dtype=x.dtype, device="cuda")[1:].view(x.shape)
    shifted.copy_(x)
    idx, gate, off, lists = (t.cpu().numpy() for t in layer.sh_gate_topk(shifted))
    ref = pu.oracle_selection(inp)
    pu.check_selection(idx, gate, ref, 70, 2e-5)
    pu.check_lists(off, lists, ref)
    layer.close()


def test_small_probabilities_keep_their_bits():
    # token 0 takes all but 2^-24 of the attention and has no value; what a row reads is the sum over the others.  Two fp16
    # parts of 2^7 p leave each of them an error of 2^-25 against 2^-17, 2^-8, which averages out over 100 keys and more;
    # fp16 queries, keys and values add 2^-11 each
    T, M, D = 256, 128, 132
    g = torch.Generator(device="cuda").manual_seed(4)
    x = torch.zeros(T, M, device="cuda")
    x[1:, 0] = 1.0
    x[0, 1] = 1.0
    x[1:, 2:] = torch.randn(T - 1, M - 2, generator=g, device="cuda")
    Wq, Wk = torch.zeros(1, M, D, device="cuda"), torch.zeros(1, M, D, device="cuda")
    Wq[0, 0, 0] = 13.8
    Wk[0, 1, 0] = 13.8
    Wk[0, 2:, 0] = 0.05 * torch.randn(M - 2, generator=g, device="cuda")
    Wv = torch.zeros(1, 1, M, D, device="cuda")
    Wv[0, 0, 2:] = 4096 * torch.randn(M - 2, D, generator=g, device="cuda") / M ** 0.5     # (the sums are normal fp16 numbers)
    Wo, Ws = torch.zeros(1, 1, D, M, device="cuda"), torch.zeros(1, M, 1, device="cuda")
    x, Wq, Wk, Wv, Wo, Ws = (a.bfloat16() for a in (x, Wq, Wk, Wv, Wo, Ws))
    layer = binding.Layer(M, 1, D, 1, 1)
    layer.sh_configure(binding.SH_BF16, 1, T)
    layer.sh_set_weights(Wq, Wk, Wv, Wo, Ws, Ws)
    layer.sh_forward(x.view(1, T, M))
    got = layer.sh_debug_buffer("AHAT")[100:, 0].double()
    x, Wq, Wk, Wv = x.double(), Wq[0].double(), Wk[0].double(), Wv[0, 0].double()
    s = (x @ Wq) @ (x @ Wk).T / D ** 0.5
    p = torch.softmax(s.masked_fill(torch.ones(T, T, device="cuda").triu(1).bool(), -torch.inf), dim=1)
    want = (p @ (0.5 * x @ Wv))[100:]
    assert float((got - want).norm() / want.norm()) < 4e-3
    layer.close()


def test_overflow_of_one_token_stays_behind_the_mask():
    # finite inputs, but token 70's value row passes fp16's range (first column of x times that row of W_V)
    cfg = config(1, 200, 128, 2, 132, 4, 2)
    inp = inputs.make_inputs(cfg)
    for W in (inp.Wq, inp.Wk, inp.Ws, inp.Wd):
        W[:, 0] = 0.0
    inp.Wv[:, :, 0] = 128.0
    inp.x[0, :, 0] = 0.0
    layer = binding.layer_from_inputs(inp)
    x = binding.to_device(inp.x, cfg.dtype)
    want = layer.sh_forward(x)
    x[0, 70, 0] = 8192.0
    y = layer.sh_forward(x)
    # (the rows of that token's tile are summed once more in another order: an fp16 unit, 2^-10, in what they read)
    assert pu.rel_rms_err(y[:, :70].cpu().numpy(), want[:, :70].cpu().numpy()) < 1e-2 and not bool(torch.isfinite(y[:, 70:]).all())
    assert layer.sh_last_status() == 0
    layer.close()


def test_overflowing_weight_reaches_the_tokens_that_selected_its_expert():
    # 1e5 is a finite bf16 weight, but past fp16's range: feature 3 of head 1's output expert 2
    cfg = config(1, 150, 256, 2, 168, 4, 2)
    inp = inputs.make_inputs(cfg)
    layer = binding.layer_from_inputs(inp)
    x = binding.to_device(inp.x, cfg.dtype)
    want = layer.sh_forward(x)
    hit = (layer.sh_gate_topk(x)[0][1, :, 1] == 2).any(dim=1)
    assert 0 < int(hit.sum()) < 150
    inp.Wo[1, 2, 0, 3] = 1e5
    layer.sh_set_weights(*[binding.to_device(a, cfg.dtype) for a in (inp.Wq, inp.Wk, inp.Wv, inp.Wo, inp.Ws, inp.Wd)])
    y = layer.sh_forward(x)
    assert pu.rel_rms_err(y[:, ~hit].cpu().numpy(), want[:, ~hit].cpu().numpy()) < 1e-5      # (two fp32 orders)
    assert not bool(torch.isfinite(y[0, hit, 3]).any())
    keep = torch.arange(256, device="cuda") != 3
    assert torch.equal(y[..., keep], want[..., keep])
    layer.close()


@pytest.mark.parametrize("T,M,H,E,k", [(70, 128, 1, 2, 1), (300, 1152, 2, 9, 3), (5000, 1024, 2, 8, 4), (130, 1536, 4, 16, 4)])
def test_gates_are_the_allocation_free_entry_points_bit_for_bit(T, M, H, E, k):
    # fp32 FMA chains in both: one and several passes a block, rows in one and two pieces, up to 128 gate columns
    inp = inputs.make_inputs(config(1, T, M, H, 132, E, k))
    layer = binding.layer_from_inputs(inp)
    x = binding.to_device(inp.x, inp.cfg.dtype)
    wg = torch.from_numpy(np.concatenate([np.transpose(w, (0, 2, 1)).reshape(-1, M) for w in (inp.Ws, inp.Wd)])).to(x).contiguous()
    layer.sh_forward(x)
    for a, b in zip(layer.sh_gate_topk(x), binding.sh_noalloc_gate_topk(inp.cfg.dtype, x[0], wg, None, H, E, k)):
        assert torch.equal(a, b)
    assert layer.sh_last_status() == 0
    layer.close()


def test_shared_selection():
    full_check(inputs.make_inputs(config(2, 150, 128, 2, 132, 5, 2)), shared_selection=True)
