"""Contractions too small for tiles of 256 columns on every SM take tiles of 128 or 64 columns, one CTA each."""
import numpy as np
import pytest

from oracle import eqat_oracle as O
from test_gpu_parity import check_block_ap, check_e2e, eqat, f32, run_block_ap, run_e2e, small_cfg  # noqa: F401
from workloads import weight_for

pytestmark = pytest.mark.gpu


# tiles of 64 columns while a tile of 128 rows each fits the chip (148 SMs) and a group lies in a tile, then 128, then 256
@pytest.mark.parametrize("out,in_f,tokens,bits,group", [
    (64, 128, 1, 2, 64),            # one tile of 64 columns, half of a tile's rows
    (576, 1152, 129, 4, 32),        # ragged rows, an odd number of K blocks
    (320, 896, 300, 3, 128),        # groups of 128: 64 columns for Y and dX, 128 for the weight gradient
    (1088, 1152, 600, 2, 64),       # the weight gradient has 9 x 18 tiles of 64 columns, more than SMs: 128
    (1408, 1408, 1100, 4, 128),     # Y and dX have 9 x 22 tiles of 64 columns: 128
    (2112, 2304, 1300, 2, 256),     # groups of 256, and more tiles of 128 columns than SMs: pairs of CTAs
])
@pytest.mark.parametrize("kind", ["block_ap", "e2e"])
def test_narrow_tiles(eqat, kind, out, in_f, tokens, bits, group):  # noqa: F811
    cfg = small_cfg(f"narrow_{out}_{in_f}_{tokens}", out, in_f, bits, group, tokens, "student_t4", 0.02, 0.01)
    lin = cfg.linears[0]
    if kind == "e2e":
        return check_e2e(run_e2e(eqat, cfg, lin, tokens, real_z=bits == 4), group)
    s, z = O.minmax_init(f32(weight_for(cfg, lin)), bits, group)
    s = (s * np.float32(0.8)).astype(np.float32)
    check_block_ap(run_block_ap(eqat, cfg, lin, tokens, s, z), s, z, bits, group)


@pytest.mark.parametrize("out,in_f,tokens,bits,group,columns", [
    (64, 128, 1, 2, 64, (64, 64)),
    (576, 1152, 129, 4, 32, (64, 64)),
    (320, 896, 300, 3, 128, (64, 128)),
    (1088, 1152, 600, 2, 64, (64, 128)),
    (1408, 1408, 1100, 4, 128, (128, 128)),
    (2112, 2304, 1300, 2, 256, (256, 256)),
])
def test_columns_of_the_problems_above(eqat, out, in_f, tokens, bits, group, columns):  # noqa: F811
    """The comments above by the host query, on this device: columns of Y and dX, and of the weight and step-size gradients."""
    d = eqat.make_desc(bits, group, out, in_f, tokens)
    Y, dX, dW, packed_dX, ds = (eqat.eqat_gemm_tile(d, c)[1] for c in (eqat.EQAT_GEMM_Y, eqat.EQAT_GEMM_DX, eqat.EQAT_GEMM_DW,
                                                                      eqat.EQAT_GEMM_PACKED_DX, eqat.EQAT_GEMM_PACKED_DS))
    assert ((Y, dW), (dX, ds)) == (columns, columns) and packed_dX == max(128, columns[0])
