"""Which kernel a packed forward goes to (decided on the host; here for a device of 148 SMs)."""
import random

import pytest

SMS = 148


@pytest.fixture(scope="module")
def eqat():
    from paper_2407_11062_b200.build import build_library
    build_library()
    from paper_2407_11062_b200 import binding
    return binding


def route(eqat, out, in_f, tokens, bits, group, fp16_z=False):
    zfmt = eqat.EQAT_ZP_FP16 if fp16_z else eqat.EQAT_ZP_U8
    return eqat.eqat_packed_fwd_route(eqat.make_desc(bits, group, out, in_f, tokens, 0, zfmt), SMS)


def test_few_tokens_keep_exact_codes_on_long_rows(eqat):
    """Up to 64 tokens neither kernel that takes them rounds (q - z) * s to bf16.  A token tile that does not fit shared
    memory is no reason to leave them: narrower tiles do (here 49152 and 53248 columns, among a grid of shapes)."""
    few = (eqat.EQAT_ROUTE_MATRIX_VECTOR, eqat.EQAT_ROUTE_WEIGHT_ROWS)
    assert route(eqat, 2048, 49152, 40, 3, 64) == (eqat.EQAT_ROUTE_WEIGHT_ROWS, (2, 32, 4))
    for in_f in (128, 384, 1024, 4096, 8192, 11008, 28672, 49152, 53248, 57344):
        for out in (64, 1024, 2048, 28672):
            for bits in (2, 3, 4):
                for group in {32, 64, 128, min(in_f, 32768)} | ({256} if in_f % 256 == 0 else set()):
                    if in_f % group or (group > 256 and group != in_f):
                        continue
                    for tokens in (1, 3, 8, 9, 13, 16, 17, 31, 33, 40, 48, 49, 64):
                        for fp16_z in (False, True):
                            assert route(eqat, out, in_f, tokens, bits, group, fp16_z)[0] in few, (out, in_f, bits, group, tokens)


def test_small_weights_take_one_kernel_up_to_sixteen_tokens(eqat):
    """The range over which a token's bits do not depend on its batch, and both sides of its boundary."""
    def kernels(out, in_f, bits, group, tokens):
        return {route(eqat, out, in_f, t, bits, group)[0] for t in tokens}

    inside = {eqat.EQAT_ROUTE_MATRIX_VECTOR}
    for in_f in (1024, 1152, 1408, 2048, 2944, 3072, 4096):
        for bits in (2, 3, 4):
            for group in {64, 128, in_f}:
                largest = (8 * 3000000 - 1) // (in_f * bits) // 64 * 64
                for out in {64, 192, 512, largest} if in_f % group == 0 else ():
                    assert kernels(out, in_f, bits, group, range(1, 17)) == inside, (out, in_f, bits, group)
                    assert kernels(out, in_f, bits, group, range(17, 65)) == {eqat.EQAT_ROUTE_WEIGHT_ROWS}
    # outside: larger weights, longer and shorter rows and groups of 32 go by time
    assert kernels(512, 384, 2, 64, range(9, 17)) == {eqat.EQAT_ROUTE_WEIGHT_ROWS}
    assert kernels(2944, 4096, 2, 64, (1, 2)) == inside                     # 3,014,656 bytes
    assert kernels(2944, 4096, 2, 64, range(9, 17)) == {eqat.EQAT_ROUTE_WEIGHT_ROWS}
    assert kernels(1024, 5120, 2, 64, range(9, 17)) == {eqat.EQAT_ROUTE_WEIGHT_ROWS}
    assert kernels(1024, 8192, 2, 64, (8, 16)) == {eqat.EQAT_ROUTE_WEIGHT_ROWS}
    assert kernels(1024, 2048, 2, 32, range(1, 17)) == {eqat.EQAT_ROUTE_WEIGHT_ROWS}


def test_an_odd_number_of_ctas_per_sm_is_not_taken_for_free(eqat):
    """Three CTAs on nearly every SM, of which two run at a time: 13824 x 5120 at seven and eight tokens was estimated at 15.5
    us, took 21.5, and the matrix-vector kernel 18.9 to 20.8 us."""
    for bits in (3, 4):
        for tokens in (7, 8):
            assert route(eqat, 13824, 5120, tokens, bits, 128)[0] == eqat.EQAT_ROUTE_MATRIX_VECTOR
    assert route(eqat, 13824, 5120, 16, 4, 128) == (eqat.EQAT_ROUTE_WEIGHT_ROWS, (1, 16, 2))
    assert route(eqat, 12288, 6144, 8, 4, 128) == (eqat.EQAT_ROUTE_WEIGHT_ROWS, (1, 16, 4))   # on 88 of the 148 SMs only


def test_large_batches_of_4_bit_codes_keep_the_tiled_kernel(eqat):
    assert route(eqat, 8192, 28672, 2048, 4, 128)[0] == eqat.EQAT_ROUTE_TILED            # 705 to 850 against 825 to 920 us
    assert route(eqat, 8192, 28672, 2300, 4, 128)[0] == eqat.EQAT_ROUTE_WEIGHT_ROW_PAIRS   # 1161 against 798 us
    assert route(eqat, 4096, 4096, 333, 4, 128)[0] == eqat.EQAT_ROUTE_WEIGHT_ROW_PAIRS


def test_the_tiled_kernel_is_priced_by_the_tiles_it_takes(eqat):
    """128 x 128 where all of them fit the chip at once: with few columns those are ahead of the weight-row pairs."""
    for out, in_f, tokens, bits in ((64, 128, 1022, 3),           # 3.8 against 5.8 us
                                    (640, 256, 1816, 2),          # 5.4 against 7.5
                                    (1536, 512, 1536, 2),         # 8.0 against 9.0
                                    (128, 384, 3938, 3)):         # 7.0 against 9.7
        assert route(eqat, out, in_f, tokens, bits, 64)[0] == eqat.EQAT_ROUTE_TILED, (out, in_f, tokens)
    for out, in_f, tokens, bits in ((1536, 1024, 1536, 2),        # 11.1 against 12.0
                                    (256, 512, 256, 4),           # 4.9 against 7.5
                                    (3392, 1024, 417, 4)):        # 10.2 against 12.4
        assert route(eqat, out, in_f, tokens, bits, 64)[0] == eqat.EQAT_ROUTE_WEIGHT_ROW_PAIRS, (out, in_f, tokens)


def test_plans_cover_all_tokens(eqat):
    rng = random.Random(3)
    for _ in range(3000):
        in_f, out = 128 * rng.randint(1, 224), 64 * rng.randint(1, 448)
        tokens, bits = int(4096 ** rng.random()) or 1, rng.choice([2, 3, 4])
        kernel, (parts, each, split) = route(eqat, out, in_f, tokens, bits, rng.choice([32, 64, 128, in_f]))
        if kernel == eqat.EQAT_ROUTE_TILED:
            assert (parts, each, split) == (0, 0, 1)
        else:
            assert (parts - 1) * each < tokens <= parts * each and split in (1, 2, 4, 8)


def test_the_rest_of_a_prompt_is_told(eqat):
    """Where a prompt goes out as two launches, the second one's rows and its split of K."""
    def rest(out, in_f, tokens, bits, group, fp16_z=False):
        zfmt = eqat.EQAT_ZP_FP16 if fp16_z else eqat.EQAT_ZP_U8
        return eqat.eqat_packed_fwd_rest(eqat.make_desc(bits, group, out, in_f, tokens, 0, zfmt), SMS)

    assert route(eqat, 11008, 4096, 333, 2, 64) == (eqat.EQAT_ROUTE_WEIGHT_ROW_PAIRS, (2, 192, 1))
    assert rest(11008, 4096, 333, 2, 64) == (1536, 4)           # 86 clusters, 74 resident: the last six pairs of row tiles
    assert rest(4096, 11008, 1531, 4, 64, True) == (1024, 2)
    assert rest(4096, 4096, 333, 2, 64) == (0, 0)               # one round
    assert rest(512, 512, 4, 2, 64) == (0, 0)                   # another kernel
    # one launch: a second one would come with more and narrower token tiles, and more expansions of the weight
    assert (route(eqat, 22976, 25216, 949, 4, 64)[1], rest(22976, 25216, 949, 4, 64)) == ((4, 256, 1), (0, 0))     # 969 against 1082 us
    assert (route(eqat, 4352, 25728, 1653, 2, 64)[1], rest(4352, 25728, 1653, 2, 64)) == ((8, 224, 1), (0, 0))     # 272 against 283
    import test_gpu_weight_row_forward as gpu
    for problem, tiles, split in gpu.REST:
        kernel, (token_tiles, _, first) = route(eqat, *problem)
        assert (kernel, token_tiles, first) == (eqat.EQAT_ROUTE_WEIGHT_ROW_PAIRS, tiles, 1), problem
        rows, second = rest(*problem)
        assert 0 < rows < problem[0] and second == split, problem
    with pytest.raises(eqat.EqatError):
        eqat.eqat_packed_fwd_rest(eqat.make_desc(2, 64, 512, 512, 4), -1)


def test_the_query_checks_its_descriptor(eqat):
    with pytest.raises(eqat.EqatError):
        eqat.eqat_packed_fwd_route(eqat.make_desc(2, 64, 96, 512, 4), SMS)
    with pytest.raises(eqat.EqatError):
        eqat.eqat_packed_fwd_route(eqat.make_desc(2, 64, 512, 512, 4), -1)


def test_the_gpu_tests_reach_the_kernels_they_name(eqat):
    """The sizes of the GPU tests, by the kernel that each test is about."""
    import test_gpu_parity as gpu

    def sizes(test):
        return next(m.args[1] for m in test.pytestmark if m.name == "parametrize")

    for out, in_f, tokens, bits, group, real_z in sizes(gpu.test_packed_forward_on_weight_row_tiles):
        assert route(eqat, out, in_f, tokens, bits, group, real_z)[0] == eqat.EQAT_ROUTE_WEIGHT_ROWS, (out, in_f, tokens)
    for out, in_f, tokens, bits, group, real_z in sizes(gpu.test_packed_forward_for_prompts):
        kernel = eqat.EQAT_ROUTE_TILED if out == 11008 else eqat.EQAT_ROUTE_WEIGHT_ROW_PAIRS
        assert route(eqat, out, in_f, tokens, bits, group, real_z)[0] == kernel, (out, in_f, tokens)
    for out, in_f, tokens, bits, group, real_z in sizes(gpu.test_packed_forward_of_large_batches):
        assert route(eqat, out, in_f, tokens, bits, group, real_z)[0] == eqat.EQAT_ROUTE_TILED, (out, in_f, tokens)
    for bits, group, in_f in next(m.args[1] for m in gpu.test_few_token_forward_takes_any_zero_point_byte.pytestmark
                                  if m.args[0].startswith("bits")):
        for tokens in (1, 2, 8):
            assert route(eqat, 320, in_f, tokens, bits, group)[0] == eqat.EQAT_ROUTE_MATRIX_VECTOR
    for bits, group, in_f, tokens in sizes(gpu.test_e2e_few_tokens_with_trained_zero_points):
        assert route(eqat, 320, in_f, tokens, bits, group, True)[0] == eqat.EQAT_ROUTE_MATRIX_VECTOR
    for bits, group in sizes(gpu.test_few_token_forward_does_not_depend_on_the_slicing):
        assert route(eqat, 1280, 4096, 13, bits, group) == (eqat.EQAT_ROUTE_MATRIX_VECTOR, (2, 7, 1))
    for out, in_f, bits, group in sizes(gpu.test_small_weights_give_a_token_the_same_bits_in_any_batch_of_up_to_sixteen):
        assert route(eqat, out, in_f, 16, bits, group) == (eqat.EQAT_ROUTE_MATRIX_VECTOR, (2, 8, 1))
