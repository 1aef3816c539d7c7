"""2-bit codes are decided by comparing a weight with its group's three thresholds, the smallest bf16 numbers of codes 1 to 3."""
import numpy as np
import pytest
import torch

from helpers import bits_to_torch, f32, torch_to_f64
from test_gpu_parity import dev, eqat  # noqa: F401
from workloads import to_bf16_bits

ZERO_POINTS = (0.0, 1.0, 2.0, 3.0, -2.0, 5.0, 16.0)


def steps():
    for base in (1.0, 0.75, 1.0 / 3.0, 0.0234375, 6.1e-5, 1.5e-30, 1.0e36):
        for ulps in (-2, -1, 0, 1, 2):
            s = np.float32(base)
            for _ in range(abs(ulps)):
                s = np.nextafter(s, np.float32(np.inf if ulps > 0 else 0.0), dtype=np.float32)
            yield s


def codes_of(w, s, z):
    """Eq. 1 in binary32: the definition."""
    with np.errstate(all="ignore"):
        p = np.rint(w / s) + z
    return np.clip(np.nan_to_num(p, nan=0.0, posinf=3.0, neginf=0.0), 0, 3).astype(np.uint8)


def test_three_comparisons_give_every_code():
    """The construction of the thresholds, over all 65536 bf16 numbers: the one nearest the rounding boundary, or the next."""
    w = f32(np.arange(65536, dtype=np.uint16))
    for s in steps():
        for z in ZERO_POINTS:
            got = np.zeros(65536, np.uint8)
            for k in (1, 2, 3):
                m = np.float32(k - z)
                v = int(to_bf16_bits(np.array([(m - np.float32(0.5)) * s]))[0])
                if not codes_of(f32(np.array([v], np.uint16)), s, z)[0] >= k:
                    v = (1 if v == 0x8000 else v - 1) if v & 0x8000 else v + 1
                with np.errstate(invalid="ignore"):
                    got += w >= f32(np.array([v], np.uint16))[0]
            assert np.array_equal(got, codes_of(w, s, z)), (s, z)


@pytest.mark.gpu
@pytest.mark.parametrize("group", [32, 256, 512])
def test_codes_on_and_beside_the_thresholds(eqat, group):  # noqa: F811
    """The bf16 numbers around the rounding boundaries of a group, for step sizes whose boundaries are bf16 numbers or a few
    fp32 ulps beside one, and for zero points inside and outside the grid; infinities and both zeros among the weights."""
    rng = np.random.default_rng(group)
    rows, s_rows, z_rows = [], [], []
    for s in steps():
        for z in ZERO_POINTS:
            marks = np.float32([k - z - 0.5 for k in (1, 2, 3)]) * s
            near = (marks.view(np.uint32) >> 16).astype(np.int64)[:, None] + np.arange(-2, 4)[None, :]
            w = np.resize((near.reshape(-1).astype(np.uint32) << 16).view(np.float32), group).copy()
            w[18:22] = np.float32([0.0, -0.0, np.inf, -np.inf])
            w[22:] = rng.standard_normal(group - 22).astype(np.float32) * s * np.float32(2.0)
            rows.append(w); s_rows.append(s); z_rows.append(np.float32(z))
    while len(rows) % 4:
        rows.append(rows[0]); s_rows.append(s_rows[0]); z_rows.append(z_rows[0])
    per_row = max(1, 128 // group)
    out, in_f = len(rows) // per_row, group * per_row
    bits16 = to_bf16_bits(np.stack(rows).reshape(out, in_f))
    W = f32(bits16)
    s, z = np.asarray(s_rows, np.float32).reshape(out, per_row), np.asarray(z_rows, np.float32).reshape(out, per_row)
    d = eqat.make_desc(2, group, out, in_f)
    P = torch.empty(out, in_f // 4, dtype=torch.uint8, device="cuda")
    z8, s16 = torch.empty(out, per_row, dtype=torch.uint8, device="cuda"), torch.empty(out, per_row, dtype=torch.float16, device="cuda")
    codes, What = torch.empty(out, in_f, dtype=torch.uint8, device="cuda"), torch.empty(out, in_f, dtype=torch.bfloat16, device="cuda")
    eqat.eqat_quantize_pack(d, bits_to_torch(bits16), dev(s), dev(z), P, z8, s16)
    eqat.eqat_unpack(d, P, codes)
    eqat.eqat_fakequant_weight(d, bits_to_torch(bits16), dev(s), dev(z), What)
    s_all, z_all = np.repeat(s, group, 1), np.repeat(z, group, 1)
    want = codes_of(W, s_all, z_all)
    assert np.array_equal(codes.cpu().numpy(), want)
    value = (want.astype(np.float32) - z_all) * s_all                     # binary32, then rounded to bf16
    assert np.array_equal(torch_to_f64(What), f32(to_bf16_bits(value)).astype(np.float64))


def end_steps():
    """The ends of what the comparisons stand for, below which 1 / s overflows and above which it is subnormal; there
    thresholds are subnormal, and boundaries overflow."""
    for base in (1.0e-38, 2.94e-39, 8.4e37, 8.5e37):
        s = np.float32(base)
        down, up = (np.nextafter(s, np.float32(to), dtype=np.float32) for to in (0.0, np.inf))
        yield from (np.nextafter(down, np.float32(0.0), dtype=np.float32), down, s, up,
                    np.nextafter(up, np.float32(np.inf), dtype=np.float32))


@pytest.mark.gpu
@pytest.mark.filterwarnings("ignore:overflow:RuntimeWarning")
@pytest.mark.parametrize("group", [32, 64, 256, 512])
def test_all_bf16_numbers(eqat, group):  # noqa: F811
    """Every bf16 number, NaN and subnormal ones among them, through quantise + pack and the fake quantiser.  W_hat bit for bit
    what Eq. 2 gives in binary32, rounded to bf16: its zeros are +0, as the difference of equal integers is."""
    bits16 = np.arange(65536, dtype=np.uint16).reshape(-1, 512)
    W, Wd = f32(bits16), bits_to_torch(bits16)
    out, in_f = bits16.shape
    d = eqat.make_desc(2, group, out, in_f)
    P = torch.empty(out, in_f // 4, dtype=torch.uint8, device="cuda")
    z8, s16 = (torch.empty(out, in_f // group, dtype=t, device="cuda") for t in (torch.uint8, torch.float16))
    codes, What = torch.empty(out, in_f, dtype=torch.uint8, device="cuda"), torch.empty(out, in_f, dtype=torch.bfloat16, device="cuda")
    for s in (*steps(), *end_steps()):
        for z in ZERO_POINTS:
            sd, zd = dev(np.full((out, in_f // group), s, np.float32)), dev(np.full((out, in_f // group), z, np.float32))
            eqat.eqat_quantize_pack(d, Wd, sd, zd, P, z8, s16)
            eqat.eqat_unpack(d, P, codes)
            eqat.eqat_fakequant_weight(d, Wd, sd, zd, What)
            want = codes_of(W, s, np.float32(z))
            assert np.array_equal(codes.cpu().numpy(), want), (s, z)
            value = to_bf16_bits((want.astype(np.float32) - np.float32(z)) * s)
            assert np.array_equal(What.view(torch.int16).cpu().numpy().view(np.uint16), value), (s, z)
