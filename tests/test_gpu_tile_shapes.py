"""GEMM tiles whose width is no power of two and whose channels lie between the multiples of 128 (needs a B200): whole rows of 13, 14, 19
and 42 columns (117, 126, 114 and 126 rows of the MMA used), sector-aligned splits of a row, parity classes of 14 columns, one
accumulator of 160 to 256 channels, narrow channel tiles where SMs are idle, block pairs on short tiles.  fp32 outputs against
the CPU oracle within the bound of the other GEMM tests."""
import pytest

from paper_2609_28358_b200 import inputs, mq
from parity_util import OracleLayer, check_convs, check_quantize

pytestmark = pytest.mark.gpu

# N, C_in, H, W, C_out, kernel, stride, padding; knobs forced beside the rules
CASES = [
    ("w13", (19, 64, 3, 13, 96, 3, 1, 1), {}),
    ("w14", (10, 128, 5, 14, 224, 3, 1, 1), {}),                    # narrow channel tiles: few row tiles
    ("w19", (7, 96, 4, 19, 160, 3, 1, 1), {}),
    ("w42", (5, 64, 3, 42, 64, 3, 1, 1), {}),
    ("w60_split", (3, 64, 3, 60, 64, 5, 1, 2), {}),                 # more taps than the whole-tile kernel takes
    ("s2_28", (11, 64, 6, 28, 128, 3, 2, 1), {}),                   # 14 output columns; input gradient: classes of 14, pairs of columns
    ("s2_38", (6, 64, 5, 38, 128, 3, 2, 1), {}),                    # 19 columns
    ("bn160", (9, 128, 4, 14, 160, 3, 1, 1), {"MQ_TC_BN": "160"}),  # one accumulator copied into registers, 80 columns a half
    ("bn192", (9, 128, 4, 14, 192, 3, 1, 1), {"MQ_TC_BN": "192"}),
    ("bn224_tail", (9, 128, 4, 14, 250, 3, 1, 1), {"MQ_TC_BN": "224"}),
    ("k1_bn160", (9, 512, 4, 16, 250, 1, 1, 0), {"MQ_TC_BN": "160"}),   # 1x1: staged stores where the halves are whole boxes, else direct ones
    ("k1_bn192", (9, 512, 4, 16, 250, 1, 1, 0), {"MQ_TC_BN": "192"}),
    ("k1_bn224", (9, 512, 4, 16, 250, 1, 1, 0), {"MQ_TC_BN": "224"}),
    ("k1_bn256", (9, 512, 4, 16, 600, 1, 1, 0), {"MQ_TC_BN": "256"}),
    ("pairs_14", (9, 256, 4, 14, 256, 3, 1, 1), {"MQ_TC_BN": "256"}),   # four tiles of 126 rows: block pairs, E4M3 and E2M1
]


@pytest.mark.parametrize("fmts", [(mq.E4M3, mq.E4M3, mq.E5M2), (mq.E2M1,) * 3], ids=["fp8", "fp4"])
@pytest.mark.parametrize("name,shape,env", CASES, ids=[c[0] for c in CASES])
def test_gemms(name, shape, env, fmts, knobs):
    d = inputs.conv_desc(*shape)
    ol = OracleLayer(inputs.Layer(name, d, *fmts, "relu", "kaiming", "gauss", 47))
    qs = check_quantize(ol)
    knobs(**env)
    check_convs(ol, qs, layouts=(mq.NCHW, mq.HWNC))
    assert mq.last_device_status() == 0


@pytest.mark.parametrize("cout", [64, 96])
def test_outputs_beyond_l2(cout):
    """More than 110 MB of output in NCHW rows that 8 columns cut inside a sector: the whole-tile kernel up to 64 output channels,
    per-tap tiles of whole rows above.  Sampled outputs, the borders among them."""
    d = inputs.conv_desc(340 * 64 // cout, 32, 36, 36, cout, 3, 1, 1)
    ol = OracleLayer(inputs.Layer("beyond l2", d, mq.E4M3, mq.E4M3, mq.E5M2, "relu", "kaiming", "gauss", 48))
    check_convs(ol, check_quantize(ol), samples=3000, ops=("fwd",))
    assert mq.last_device_status() == 0
