"""Work units of 64 and 128 output features in the CTA-pair output projections (calls with too few tokens for units of 256):
one unit's worth of tokens and its neighbours, d_model off the 256 grid, both kernels (2:4 sparse, masked), fp16 output."""
import numpy as np
import pytest
import torch

from paper_2312_07987_b200 import binding, inputs
from tests import parity_util as pu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D,E,k", [(128, 4, 2), (128, 8, 1), (128, 5, 3), (64, 4, 2), (128, 16, 4)])
@pytest.mark.parametrize("T,M", [(255, 384), (257, 1024), (3000, 512)])      # 64, 64 and 128 features a unit
def test_narrow_units(T, M, D, E, k):
    cfg = inputs.LayerConfig("units", inputs.DTYPE_BF16, 1, T, M, 2, D, E, k, seed=T + E)
    inp = inputs.make_inputs(cfg)
    layer, x, y = pu.run_layer(inp)
    ref = pu.oracle_for(inp)["y"]
    assert pu.rel_rms_err(y.cpu().numpy(), ref) < pu.TOL_Y[inputs.DTYPE_BF16]
    if k <= 2:                                              # (the value rows of k >= 3 are summed in no fixed order)
        layer.sh_set_output_f16(True)
        assert torch.equal(layer.sh_forward(x), y.half())
    layer.sh_check_guards()
    layer.close()
