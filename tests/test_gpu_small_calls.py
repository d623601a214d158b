"""Calls of at most 256 tokens of one routing group, whose dispatch plan and gather are one launch: checked like every other
layer, on both sides of the limit."""
import pytest

from paper_2101_03961_b200 import inputs as si
from paper_2101_03961_b200 import switch_moe as sm
from tests.gpu_helpers import TOL_BF16, TOL_F32
from tests.test_gpu_parity import _check_layer


@pytest.mark.gpu
@pytest.mark.parametrize("T,d,E,cf,kw", [
    (1, 64, 1, 1.0, {}), (31, 64, 3, 1.0, dict(residual=True)), (33, 192, 5, 2.0, {}), (96, 256, 8, 2.0, dict(residual=True)),
    (129, 128, 64, 2.0, {}), (255, 64, 65, 1.25, dict(jitter_eps=0.2)), (256, 320, 128, 2.0, dict(noise_eps=0.3)),
    (256, 128, 129, 2.0, {}), (256, 64, 256, 1.0, dict(residual=True)), (200, 64, 126, 4.0, dict(geglu=True)),
    (256, 64, 2, 0.5, dict(residual=True)), (250, 64, 3, 4.0, {}), (257, 128, 128, 2.0, {}), (256, 64, 8, 1.0, dict(reroute=True)),
])
@pytest.mark.parametrize("dtype", [si.DTYPE_BF16, si.DTYPE_F32])
def test_small_calls_match_oracle(T, d, E, cf, kw, dtype):
    cfg = si.SwitchConfig("small", T, d, 128, E, cf, bias_std=0.3, dtype=dtype)
    _check_layer(cfg, sm.GEMM_DEFAULT, TOL_F32 if dtype == si.DTYPE_F32 else TOL_BF16, **kw)


@pytest.mark.gpu
def test_small_float32_call_with_tensor_core_products_matches_oracle():
    cfg = si.SwitchConfig("small_tc", 250, 320, 576, 3, 1.25, bias_std=0.3, dtype=si.DTYPE_F32)
    _check_layer(cfg, sm.GEMM_DEFAULT, TOL_F32, residual=True)


def test_small_calls_have_fewer_launches():
    small, large = (sm.switch_moe_stage_launches(sm.make_config(T, 256, 512, 64, 2.0)) for T in (256, 257))
    assert (small["dispatch_plan"], small["gather_x"]) == (0, 1) and (large["dispatch_plan"], large["gather_x"]) == (2, 1)
    rerouted = sm.switch_moe_stage_launches(sm.make_config(256, 256, 512, 64, 2.0, reroute=True))
    assert rerouted["dispatch_plan"] == 2 + 4
