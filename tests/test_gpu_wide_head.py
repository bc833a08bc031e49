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
