"""Every shape of output tile of the GEMM kernels, with rows that do not fill the last one.

Which tiles a contraction takes follows its sizes and the number of SMs; the host tells (eqat_gemm_tile).  The problems below
reach every kernel that the library has for a B200 of 148 SMs, which is checked without a GPU, and on a GPU each problem has
to take the same tiles there.
"""
import numpy as np
import pytest

from oracle import eqat_oracle as O
from helpers import f32
from test_gpu_parity import check_block_ap, check_e2e, eqat as gpu_eqat, run_block_ap, run_e2e, small_cfg  # noqa: F401
from workloads import weight_for

SMS = 148

# (out, in, tokens, bits, group); group 0: one per row.  Tiles of Y, dX and the weight gradient:
BLOCK_AP = [
    (320, 384, 165, 3, 384),        # 128 x 64 each; the weight gradient goes through memory
    (64, 128, 132, 3, 32),          # 128 x 64 each, Eqs. 3-5 in the epilogue
    (64, 128, 162, 3, 128),         # 128 x 128 for the weight gradient: a group lies in a tile
    (64, 256, 133, 2, 256),         # one CTA with 256 columns
    (192, 256, 141, 4, 256),        # a pair of CTAs, the second with 64 rows
    (11264, 384, 99, 2, 384),       # 128 x 128 for Y, pairs for the weight gradient
    (320, 9984, 66, 3, 128),        # 128 x 128 for dX, pairs for the weight gradient
    (19008, 384, 71, 4, 64),        # one CTA with 256 columns for Y
    (320, 21504, 70, 4, 256),       # and for dX
    (64, 13568, 174, 4, 13568),     # 128 x 128 for the weight gradient through memory
    (64, 23552, 138, 3, 23552),     # one CTA with 256 columns for it
    (320, 6656, 257, 3, 6656),      # pairs of 128 rows for dX and the weight gradient through memory
    (10816, 384, 210, 2, 384),      # pairs of 128 rows for Y, of 256 for the weight gradient through memory
    (9536, 384, 274, 4, 384),       # pairs of 256 rows for Y and the weight gradient through memory
    (320, 9856, 287, 2, 64),        # pairs of 256 rows for dX
]
LATENT = [
    (320, 384, 70, 2, 64),          # W_hat not stored: 256 rows on one CTA
    (320, 384, 259, 4, 64),         # a pair of them, the second with three rows
]
# the same and the zero points: trained (fp16) or bytes.  Tiles of the tiled forward, dX and the step-size gradient:
E2E_QP = [
    (64, 128, 135, 2, 64, False), (64, 128, 142, 3, 64, True), (64, 128, 142, 4, 32, False),     # ds on 128 x 64
    (64, 128, 130, 2, 128, True), (64, 128, 137, 3, 128, False), (64, 384, 622, 4, 128, True),   # on 128 x 128
    (64, 384, 589, 2, 384, False), (64, 384, 482, 3, 384, True), (64, 256, 158, 4, 256, True),   # on one CTA with 256 columns
    (10816, 384, 261, 2, 384, False),     # ds on pairs of 256 rows, Y on pairs
    (9664, 384, 325, 4, 32, True),
    (20032, 640, 136, 3, 640, True),      # Y on one CTA with 256 rows
    (20736, 384, 68, 2, 128, False),
    (23168, 512, 66, 4, 128, False),
    (320, 20608, 66, 2, 128, True),       # dX on one CTA with 256 rows
    (384, 20480, 65, 3, 128, False),
    (320, 22400, 67, 4, 32, False),
] + [
    # Y on pairs; dX on pairs and ds on pairs of 128 rows: every width of codes with groups shorter than a unit of 64 codes,
    # longer than one, and one per row, and both kinds of zero points
    case for bits in (2, 3, 4) for g, (group, real_z) in enumerate(((32, bits != 3), (256, bits == 3), (0, bits == 4)))
    for case in ((576, 512, 4098 + g, bits, group, real_z), (320, 7168, 300, bits, group, not real_z))
]


@pytest.fixture(scope="module")
def lib():
    from paper_2407_11062_b200.build import build_library
    build_library()
    from paper_2407_11062_b200 import binding
    return binding


def kernels(eqat, kind, out, in_f, tokens, bits, group, real_z=False, sms=SMS):
    """{(what selects the kernel): (tile, rows of the result)} of the GEMM kernels that a call of this kind launches."""
    d = eqat.make_desc(bits, group or in_f, out, in_f, tokens, 0, int(real_z))

    def tile(contraction):
        return eqat.eqat_gemm_tile(d, contraction, sms)

    if kind == "block_ap":
        grad = "dW" if d.group > 256 else "STE"
        return {("Y",): (tile(eqat.EQAT_GEMM_Y), tokens), ("dX",): (tile(eqat.EQAT_GEMM_DX), tokens),
                (grad,): (tile(eqat.EQAT_GEMM_DW), out)}
    if kind == "latent":
        return {("latent Y",): (tile(eqat.EQAT_GEMM_LATENT_Y), tokens), ("latent dX",): (tile(eqat.EQAT_GEMM_LATENT_DX), tokens)}
    found = {("packed dX", bits): (tile(eqat.EQAT_GEMM_PACKED_DX), tokens), ("ds", bits): (tile(eqat.EQAT_GEMM_PACKED_DS), out)}
    if eqat.eqat_packed_fwd_route(d, sms)[0] == eqat.EQAT_ROUTE_TILED:
        found["packed Y", bits] = tile(eqat.EQAT_GEMM_PACKED_Y), tokens
    return found


def problems():
    return ([("block_ap",) + p for p in BLOCK_AP] + [("latent",) + p for p in LATENT] + [("e2e",) + p for p in E2E_QP])


def test_every_kernel_is_reached_with_a_ragged_last_tile(lib):
    dense = {(128, 64, 1), (128, 128, 1), (128, 256, 1), (128, 256, 2), (256, 256, 2)}
    packed = {(128, 128, 1), (256, 256, 1), (256, 256, 2)}
    want = {(name, t) for name in ("Y", "dX", "dW") for t in dense} | {("STE", t) for t in dense - {(256, 256, 2)}}
    want |= {(name, t) for name in ("latent Y", "latent dX") for t in packed - {(128, 128, 1)}}
    want |= {(name, bits, t) for name, tiles in (("packed Y", packed), ("packed dX", packed), ("ds", dense))
             for bits in (2, 3, 4) for t in tiles}
    got = set()
    for p in problems():
        for key, (tile, rows) in kernels(lib, *p).items():
            if rows % (tile[0] * tile[2]):
                got.add(key + (tile,))
    assert got == want


def test_pairs_take_codes_of_every_width_group_and_zero_point(lib):
    got = {"packed Y": set(), "packed dX": set(), "ds": set()}
    for p in problems():
        for key, (tile, _) in kernels(lib, *p).items():
            if key[0] in got and tile[2] == 2:
                got[key[0]] |= {(p[4], "row" if p[5] in (0, p[2]) else p[5]), (p[4], p[6])}
    want = {(bits, group) for bits in (2, 3, 4) for group in (32, 256, "row")} | {(bits, z) for bits in (2, 3, 4) for z in (False, True)}
    for name, reached in got.items():
        assert reached >= want, name


def test_tiles_of_a_contraction(lib):
    """A group that the epilogue sums up lies in a tile; narrow tiles only while all of them fit the SMs; bad arguments."""
    for out in (64, 512, 1408, 2112, 11008):
        for in_f in (128, 512, 1408, 4096):
            for group in (32, 64, 128, 256):
                if in_f % group:
                    continue
                for tokens in (1, 300, 2048):
                    d = lib.make_desc(2, group, out, in_f, tokens)
                    for contraction in range(lib.EQAT_GEMM_Y, lib.EQAT_GEMM_PACKED_DS + 1):
                        rows, cols, ctas = lib.eqat_gemm_tile(d, contraction, SMS)
                        if contraction in (lib.EQAT_GEMM_DW, lib.EQAT_GEMM_PACKED_DS):
                            assert cols >= group
                        if cols < 256:
                            M, N = {lib.EQAT_GEMM_Y: (tokens, out), lib.EQAT_GEMM_PACKED_Y: (tokens, out), lib.EQAT_GEMM_DX: (tokens, in_f),
                                    lib.EQAT_GEMM_PACKED_DX: (tokens, in_f)}.get(contraction, (out, in_f))
                            assert (rows, ctas) == (128, 1) and -(-M // rows) * -(-N // cols) <= SMS
    # the 70B k/v projections in training, and what the GPU tests of small problems name
    assert lib.eqat_gemm_tile(lib.make_desc(4, 128, 1024, 8192, 2048), lib.EQAT_GEMM_Y, SMS) == (128, 128, 1)
    assert lib.eqat_gemm_tile(lib.make_desc(2, 64, 512, 512, 256), lib.EQAT_GEMM_Y, SMS) == (128, 64, 1)
    assert lib.eqat_gemm_tile(lib.make_desc(4, 128, 4096, 4096, 4096), lib.EQAT_GEMM_DW, SMS) == (128, 256, 2)
    with pytest.raises(lib.EqatError):
        lib.eqat_gemm_tile(lib.make_desc(2, 64, 512, 512, 4), 8, SMS)
    with pytest.raises(lib.EqatError):
        lib.eqat_gemm_tile(lib.make_desc(2, 64, 512, 512, 4), lib.EQAT_GEMM_Y, -1)
    with pytest.raises(lib.EqatError):
        lib.eqat_gemm_tile(lib.make_desc(2, 512, 512, 1024, 4), lib.EQAT_GEMM_PACKED_DX, SMS)


@pytest.mark.gpu
@pytest.mark.parametrize("problem", problems(), ids=lambda p: "-".join(str(v) for v in p))
def test_ragged_tiles(gpu_eqat, problem):  # noqa: F811
    kind, out, in_f, tokens, bits, group = problem[:6]
    group = group or in_f
    assert kernels(gpu_eqat, *problem, sms=0) == kernels(gpu_eqat, *problem)
    cfg = small_cfg(f"tiles_{out}_{in_f}_{tokens}_{group}", out, in_f, bits, group, tokens, "student_t4", 0.02, 0.01)
    lin = cfg.linears[0]
    if kind == "e2e":
        return check_e2e(run_e2e(gpu_eqat, cfg, lin, tokens, real_z=problem[6]), group)
    s, z = O.minmax_init(f32(weight_for(cfg, lin)), bits, group)
    s = (s * np.float32(0.8)).astype(np.float32)
    check_block_ap(run_block_ap(gpu_eqat, cfg, lin, tokens, s, z, store_what=kind == "block_ap"), s, z, bits, group)
