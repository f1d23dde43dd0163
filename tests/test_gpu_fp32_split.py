"""fp32 forward on either side of the pair and block counts at which its scan and softmax kernels cut their work finer,
against the oracle."""
import pytest

from paper_2602_03681_b200 import inputs
from test_gpu_parity import TOL, check_fwd, run_fwd, run_oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,H,L", [(1, 73, 64), (2, 37, 64), (1, 49, 192), (1, 50, 192), (3, 25, 320)])
def test_fp32_forward(B, H, L):
    wl = inputs.WORKLOADS["cfg0_f32_tiny_fwd"]
    x = inputs.make_layer_inputs(wl, B=B, H=H, L=L)
    check_fwd(wl, run_fwd(wl, x), run_oracle(wl, x), TOL["f32"])
