"""Launches overlap: a kernel starts while the ones before it in the stream still run and waits for them before it touches
global memory.  What an earlier launch writes must therefore not be read through the read-only path, which is for data
that nobody writes while the kernel lives."""
import glob
import os
import re

import numpy as np
import pytest
import torch

from conftest import ROOT


def sources():
    for path in sorted(glob.glob(os.path.join(ROOT, "paper_2407_11062_b200", "csrc", "*.cu*"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        yield os.path.basename(path), text


def test_no_operand_is_read_through_the_read_only_path():
    found = []
    for name, text in sources():
        found += [(name, m) for m in re.findall(r"__ldg\s*\(|ld\.global\.nc\S*|const\s+\w+\s*\*\s*(?:const\s+)?__restrict__", text)]
    assert not found


def test_tensor_memory_of_overlapped_and_paired_launches():
    """Read in the sources: a kernel takes its tensor memory before it lets the next launch start (a CTA of that launch that
    took the columns first would wait for this grid, and this grid for the columns); a pair takes its columns when both CTAs
    are known to run and no CTA leaves before both have given theirs back."""
    checked = 0
    for name, text in sources():
        for kernel in re.split(r"__global__", text)[1:]:
            alloc = [m.start() for m in re.finditer(r"tmem_alloc(?:_pair)?\(", kernel)]
            if not alloc:
                continue
            checked += 1
            starts = [m.start() for m in re.finditer(r"grid_dependents_launch\(", kernel)]
            assert len(starts) == 1 and starts[0] > max(alloc), name
            if "tmem_alloc_pair(" in kernel:
                waits = [m.start() for m in re.finditer(r"cluster_wait\(", kernel)]
                assert min(waits) < kernel.index("tmem_alloc_pair("), name
                assert max(waits) > kernel.index("tmem_dealloc_pair("), name
    assert checked == 3


def test_warps_give_up_a_wait_together():
    """Read in the sources: only waits of a single lane (producers, teardown) are decided lane by lane.  What a whole warp
    waits for goes through the form that votes, or its result is voted on before the warp goes on, since elect.sync,
    shuffles and tensor-core instructions follow."""
    one_lane, waits, alone = {"WAIT_PRODUCER_EMPTY", "WAIT_STREAM_EMPTY", "WAIT_TEARDOWN"}, 0, []
    for name, text in sources():
        for m in re.finditer(r"([^;{}]*?)(\w+)(?:<\w+>)?\(\s*ptx::smem_addr\(&ctl->[^;{]*?abort_flag,\s*(WAIT_\w+)", text):
            waits += 1
            before, function, site = m.groups()
            result = re.search(r"(\w+) = [^;]*$", before)
            rest = text[m.end():m.end() + 6000]
            into = result and re.search(r"(\w+) = %s &&" % result.group(1), rest)          # or with the wait that follows
            voted = result and any(re.search(r"(?:warp_agrees\(|__all_sync\(0xFFFFFFFFu, )%s\)" % v.group(1), rest) for v in (result, into) if v)
            if site not in one_lane and function != "bounded_wait_warp" and not voted:
                alone.append((name, function, site))
    assert waits >= 20 and not alone


@pytest.mark.gpu
@pytest.mark.parametrize("bits,group", [(2, 64), (3, 128), (4, 512), (4, 32)])
def test_operands_rewritten_between_overlapped_launches(bits, group):
    """One layer of 512 x 512 whose step sizes, zero points and codes are rewritten in place from another weight each time,
    between kernels that read them, without a pause and again with a synchronise after every call."""
    from paper_2407_11062_b200 import binding as eqat
    n, ng, rounds, tokens = 512, 512 // group, 12, (1, 8, 12, 40, 100, 300)
    gen = torch.Generator(device="cuda").manual_seed(bits)

    def empty(*shape, dtype=torch.bfloat16):
        return torch.zeros(shape, dtype=dtype, device="cuda")

    def normal(*shape):
        return torch.randn(shape, device="cuda", generator=gen).to(torch.bfloat16)

    Ws = [normal(n, n) * (0.01 * (1 + i % 3)) for i in range(rounds)]
    Xs, dYs = {t: normal(t, n) for t in tokens}, normal(300, n)

    def run(pause):
        s, z = empty(n, ng, dtype=torch.float32), empty(n, ng, dtype=torch.float32)
        P, z8, s16 = empty(n, n * bits // 8, dtype=torch.uint8), empty(n, ng, dtype=torch.uint8), empty(n, ng, dtype=torch.float16)
        d0 = eqat.make_desc(bits, group, n, n, 300)
        scratch = [torch.empty(max(256, eqat.workspace_bytes(d0, op)), dtype=torch.uint8, device="cuda")
                   for op in (eqat.EQAT_OP_FAKEQUANT_BWD, eqat.EQAT_OP_PACKED_BWD_DS)]
        outs = []
        for _ in Ws:
            outs.append({"codes": empty(n, n, dtype=torch.uint8), "W_hat": empty(n, n), "Y": {t: empty(t, n) for t in tokens},
                         "Y0": {t: empty(t, n) for t in tokens}, "dX": empty(300, n), "ds": empty(n, ng, dtype=torch.float32),
                         "dz": empty(n, ng, dtype=torch.float32), "Yap": empty(300, n), "dXap": empty(300, n), "dW": empty(n, n),
                         "dsap": empty(n, ng, dtype=torch.float32), "dzap": empty(n, ng, dtype=torch.float32)})
        torch.cuda.synchronize()

        def call(fn, *args):
            fn(*args)
            if pause:
                torch.cuda.synchronize()

        for W, o in zip(Ws, outs):
            d = eqat.make_desc(bits, group, n, n)
            call(eqat.eqat_minmax_init, d, W, s, z)
            call(eqat.eqat_quantize_pack, d, W, s, z, P, z8, s16)
            call(eqat.eqat_unpack, d, P, o["codes"])
            for t in tokens:
                call(eqat.qlinear_packed_fwd, eqat.make_desc(bits, group, n, n, t), Xs[t], P, s16, z8, o["Y"][t])
            call(eqat.qlinear_packed_bwd_dx, d0, dYs, P, s16, z8, o["dX"])
            call(eqat.qlinear_packed_bwd_ds, d0, Xs[300], dYs, P, z8, s16, o["ds"], o["dz"], scratch[1])
            call(eqat.qlinear_fakequant_fwd, d0, Xs[300], W, s, z, o["Yap"], o["W_hat"])
            call(eqat.qlinear_fakequant_bwd, d0, Xs[300], dYs, W, s, z, o["W_hat"], o["dXap"], o["dW"], o["dsap"], o["dzap"],
                 scratch[0])
            call(eqat.eqat_pack, d, o["codes"], P)                          # the same codes again, and read at once
            for t in tokens:
                call(eqat.qlinear_packed_fwd, eqat.make_desc(bits, group, n, n, t), Xs[t], P, s16, z8, o["Y0"][t])
        torch.cuda.synchronize()
        return [t for o in outs for v in o.values() for t in (v.values() if isinstance(v, dict) else [v])]

    ref = run(True)
    assert all(np.isfinite(float(t.float().abs().max())) for t in ref)
    for _ in range(5):
        for got, want in zip(run(False), ref):
            assert torch.equal(got.view(torch.uint8), want.view(torch.uint8))
    assert eqat.device_status() == (0, 0)
