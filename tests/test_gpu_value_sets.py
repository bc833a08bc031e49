"""The value projection by sets of selected experts (bf16 storage, up to 256 columns of k experts): two, three and four
experts of 64 stored columns, one set and as many as are taken (35), tiles of 256 entries with one token more or less,
sets nobody selects, d_head below its stored width, a model dimension of one ring turn and more."""
import numpy as np
import pytest
import torch

from paper_2312_07987_b200 import inputs
from tests import parity_util as pu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,T,M,H,D,E,k,zipf", [
    (1, 255, 128, 1, 64, 3, 3, 0.0),     # one set: a tile less one row
    (1, 257, 256, 2, 64, 4, 4, 0.0),     # ... and one row into the second tile; 256 columns
    (2, 300, 384, 2, 48, 5, 3, 1.2),     # 10 sets, uneven; zero columns behind d_head
    (3, 1000, 512, 2, 64, 7, 3, 0.0),    # 35 sets
    (2, 700, 640, 3, 40, 6, 4, 3.0),     # 15 sets, most of them empty
    (8, 401, 128, 1, 64, 8, 2, 0.0),     # pairs of 64 columns
])
def test_sets_of_experts(B, T, M, H, D, E, k, zipf):
    cfg = inputs.LayerConfig("sets", inputs.DTYPE_BF16, B, T, M, H, D, E, k, seed=7 * T + E, zipf_bias=zipf)
    inp = inputs.make_inputs(cfg)
    layer, x, y = pu.run_layer(inp)
    ref = pu.oracle_for(inp)
    # a value row: fp16 stored once, of an fp32 sum (no reductions in fp16)
    got = layer.sh_debug_buffer("V").float().cpu().numpy().astype(np.float64).transpose(0, 2, 1, 3)
    want = ref["V"]
    tol = 2.0 ** -11 * np.abs(want) + 3e-4 * np.sqrt((want ** 2).mean())      # half a unit of fp16; bf16 products in fp32
    assert not (np.abs(got - want) > tol).any(), float(np.abs(got - want).max())
    assert pu.rel_rms_err(y.cpu().numpy(), ref["y"]) < pu.TOL_Y[cfg.dtype]
    for _ in range(3):                                      # nothing depends on the order of arrival
        assert torch.equal(layer.sh_forward(x), y)
    layer.sh_check_guards()
    layer.close()
