"""Packed forward for prompts: whole rounds of clusters, and a rest that is split finer over K in a launch of its own."""
import pytest

import test_gpu_parity as parity
from test_gpu_parity import eqat  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("out,in_f,tokens,bits,group,real_z", [
    (19200, 1024, 100, 2, 64, False),     # 75 pairs of row tiles: 74 at once, the last one over a cluster of eight CTAs
    (19008, 1024, 100, 4, 32, True),      # 64 live rows in the rest
    (19840, 1152, 97, 3, 128, False),     # nine runs over a split of K, ragged tokens
])
def test_rest_of_the_rounds(eqat, out, in_f, tokens, bits, group, real_z):  # noqa: F811
    assert eqat.eqat_packed_fwd_route(eqat.make_desc(bits, group, out, in_f, tokens, 0, int(real_z)))[0] == eqat.EQAT_ROUTE_WEIGHT_ROW_PAIRS
    parity.test_packed_forward_for_prompts(eqat, out, in_f, tokens, bits, group, real_z)


# (problem, token tiles, split of K of the rest); the first three are those above
REST = [
    ((19200, 1024, 100, 2, 64, False), 1, 4),
    ((19008, 1024, 100, 4, 32, True), 1, 4),      # 64 live rows in the rest
    ((19840, 1152, 97, 3, 128, False), 1, 4),
    ((9600, 2048, 257, 2, 2048, False), 2, 4),    # two ragged token tiles, half of the last pair's rows; one group per row
    ((9536, 2048, 257, 4, 64, False), 2, 4),
    ((4736, 2048, 777, 2, 256, True), 5, 2),      # five token tiles, the rest over clusters of four CTAs
    ((13952, 2048, 520, 3, 128, False), 3, 2),
]


@pytest.mark.parametrize("problem,tiles,rest_split", REST)
def test_rest_with_several_token_tiles(eqat, problem, tiles, rest_split):  # noqa: F811
    """The plan, second launch included, on this device; and the results where the test above has no such problem."""
    out, in_f, tokens, bits, group, real_z = problem
    d = eqat.make_desc(bits, group, out, in_f, tokens, 0, int(real_z))
    kernel, (token_tiles, _, split) = eqat.eqat_packed_fwd_route(d)
    assert (kernel, token_tiles, split) == (eqat.EQAT_ROUTE_WEIGHT_ROW_PAIRS, tiles, 1)
    rows, second = eqat.eqat_packed_fwd_rest(d)
    assert 0 < rows < out and second == rest_split
    if tiles > 1:
        parity.test_packed_forward_for_prompts(eqat, out, in_f, tokens, bits, group, real_z)
