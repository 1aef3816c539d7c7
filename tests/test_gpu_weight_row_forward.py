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
