"""Forms of the resident decode that depend on a code's mixture of degrees,
compared bit for bit with the pass kernels (a profiled decode runs those)."""
import subprocess
import sys
from pathlib import Path

import numpy as np
import pytest

from paper_1609_01567_gb300 import inputs as I
from tests.test_resident import decodes, ldpc, random_code  # noqa: F401  (ldpc is a fixture)

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ROOT = Path(__file__).resolve().parent.parent


# Checks on both sides of degree 16, whose sign rule for an input of exactly +0
# differs: (m, n, degrees that the checks cycle through). The pass kernels serve
# degrees 17-32 by the register kernel in batches of up to 32 frames (largest
# degree 18), always (above 18), or never (2048 such checks or more).
MIXED_DEGREES = {
    "up_to_18": (97, 402, [5, 9, 10, 11, 13, 15, 17, 18]),
    "up_to_32": (97, 603, [9, 10, 12, 14, 15, 20, 27, 32]),
    "many_wide": (3200, 3003, [18, 17, 10]),
}


@pytest.mark.parametrize("frames", [3, 40, 70])
@pytest.mark.parametrize("name", list(MIXED_DEGREES))
def test_erased_inputs_of_checks_on_both_sides_of_degree_16(ldpc, name, frames):  # noqa: F811
    m, n, degrees = MIXED_DEGREES[name]
    rows, cols = random_code(m, n, degrees, seed=m)
    if name == "many_wide":
        assert int((np.bincount(rows) > 16).sum()) >= 2048
    h = ldpc.ldpc_code_create(m, n, rows, cols)
    gen = torch.Generator(device="cuda").manual_seed(frames)
    llr = torch.randn((frames, n), generator=gen, device="cuda") * 4.0 - 3.0
    for c in range(7):  # about a seventh of the bits, other ones in each frame
        llr[c::7, c::7] = 0.0
    llr[-1] = 0.0
    for msg in ("f32", "bf16"):
        for max_iter in (1, 8):
            got, ref = decodes(ldpc, h, llr, max_iter, early_exit=False, msg_dtype=msg)
            for k in ref:
                assert torch.equal(got[k], ref[k]), (msg, max_iter, k)


def test_kernels_are_counted_as_launched(ldpc):  # noqa: F811
    """A batch above 8192 frames whose last chunk of passes would hold 1 to 32
    frames runs as two kernels, other sum-product batches and min-sum as one."""
    code = I.small_code_n1008()
    h = ldpc.code_from_inputs(code)
    llr = torch.full((8200, code.n), -3.0, device="cuda")
    for frames, rule, kernels in ((8200, "sum_product", 2), (8192, "sum_product", 1), (20, "sum_product", 1),
                                  (8200, "min_sum", 1)):
        ldpc.ldpc_prof_read(h, reset=True)
        ldpc.ldpc_decode(h, llr[:frames], 3, rule=rule, want_post=False)
        torch.cuda.synchronize()
        assert ldpc.ldpc_prof_read(h, reset=True)["kernels"] == kernels, (frames, rule)


def test_batch_info_tells_which_decode_an_item_runs(ldpc):  # noqa: F811
    """A short code's item runs one kernel (streams 0); with a layout option, or
    a code too long for one SM, it runs the pass kernels."""
    short, long_ = I.small_code_n1008(), I.mixed_code(6)
    hs = [ldpc.code_from_inputs(short), ldpc.code_from_inputs(long_)]
    assert long_.n == 32400
    b = ldpc.ldpc_batch_create(hs, [64, 3], 4)
    assert [ldpc.ldpc_batch_info(b, i)["streams"] for i in range(2)] == [0, 1]
    llrs = [torch.full((f, h.n), -3.0, device="cuda") for f, h in zip((64, 3), hs)]
    ldpc.ldpc_prof_read(hs[0], reset=True)
    ldpc.ldpc_batch_run(b, llrs)
    torch.cuda.synchronize()
    assert ldpc.ldpc_prof_read(hs[0], reset=True)["kernels"] == 1
    b = ldpc.ldpc_batch_create(hs, [64, 3], 4, frames_per_lane=2)
    assert [ldpc.ldpc_batch_info(b, i)["streams"] for i in range(2)] == [1, 1]


def test_batch_tuning_tries_the_resident_decode_every_time(ldpc):  # noqa: F811
    """Frames that use all their iterations tune this item to the pass kernels
    (or nearly); frames that stop early, tuned afterwards, take it back to the
    resident decode, as in a batch tuned with those alone."""
    code, entries = I.qc_stand_in_code(16000)
    h = ldpc.ldpc_code_create_qc(4, 8, 2000, entries)
    gen = torch.Generator(device="cuda").manual_seed(1)
    noise = torch.randn((64, code.n), generator=gen, device="cuda")
    clean = noise - 6.0
    kw = dict(msg_dtype="bf16")
    fresh = ldpc.ldpc_batch_create([h], [64], 50, **kw)
    ldpc.ldpc_batch_tune(fresh, [clean])
    assert ldpc.ldpc_batch_info(fresh, 0)["streams"] == 0
    again = ldpc.ldpc_batch_create([h], [64], 50, **kw)
    ldpc.ldpc_batch_tune(again, [noise])
    first = ldpc.ldpc_batch_info(again, 0)["streams"]
    ldpc.ldpc_batch_tune(again, [clean])
    assert ldpc.ldpc_batch_info(again, 0)["streams"] == 0, first
    out = ldpc.ldpc_batch_run(again, [clean])[0]
    ref = ldpc.ldpc_decode(h, clean, 50, profile=True, **kw)
    for k in ("bits", "iters", "ok"):
        assert torch.equal(out[k], ref[k]), k


def test_choice_between_one_sm_and_the_passes(ldpc):  # noqa: F811
    """Few frames of long codes of wide checks, and fixed iterations of many int8
    frames, run the pass kernels (more than one launch); short codes, and frames
    that may stop early, run one kernel. Both give the same results."""
    wide = I.ira_code(16000, 12000, {4: 1.0}, seed=16000)
    half = I.ira_code(8000, 4000, {6: 1.0}, seed=8000)
    short = I.small_code_n1008()
    for code, frames, max_iter, early, msg, one in (
            (wide, 8, 10, False, "bf16", False), (wide, 8, 50, True, "bf16", False), (half, 1600, 3, False, "i8", False),
            (half, 1600, 50, True, "i8", True), (half, 100, 10, False, "f16", True), (short, 1, 50, True, "f32", True),
            (short, 3000, 10, False, "i8", True)):
        h = ldpc.code_from_inputs(code)
        gen = torch.Generator(device="cuda").manual_seed(frames)
        llr = torch.randn((frames, code.n), generator=gen, device="cuda") * 2.0 - 4.0
        ldpc.ldpc_prof_read(h, reset=True)
        got = ldpc.ldpc_decode(h, llr, max_iter, early_exit=early, msg_dtype=msg)
        torch.cuda.synchronize()
        assert (ldpc.ldpc_prof_read(h, reset=True)["kernels"] == 1) == one, (code.n, frames, max_iter, msg)
        ref = ldpc.ldpc_decode(h, llr, max_iter, early_exit=early, msg_dtype=msg, streams=1)
        for k in ref:
            assert torch.equal(got[k], ref[k]), (code.n, frames, k)


@pytest.mark.parametrize("rule", ["sum_product", "min_sum"])
def test_channel_values_outside_shared_memory(ldpc, rule):  # noqa: F811
    """n = 16200 with FP32 messages: the channel LLRs do not fit beside them."""
    code = I.mixed_code(5)
    assert code.n == 16200
    h = ldpc.code_from_inputs(code)
    gen = torch.Generator(device="cuda").manual_seed(5)
    llr = torch.randn((304, code.n), generator=gen, device="cuda") * 1.6 - 1.3
    for early in (True, False):
        kw = dict(rule=rule, rule_beta=0.15 if rule == "min_sum" else 0.0, early_exit=early)
        ldpc.ldpc_prof_read(h, reset=True)
        got = ldpc.ldpc_decode(h, llr, 30 if early else 6, **kw)
        torch.cuda.synchronize()
        assert ldpc.ldpc_prof_read(h, reset=True)["kernels"] == 1
        ref = ldpc.ldpc_decode(h, llr, 30 if early else 6, streams=1, **kw)
        for k in ref:
            assert torch.equal(got[k], ref[k]), (early, k)


def test_last_chunk_of_few_frames_with_erased_inputs(ldpc):  # noqa: F811
    """The zero rule changes within a batch above 8192 frames whose last chunk of
    passes holds 1 to 32."""
    code = I.small_code_n1008()
    h = ldpc.code_from_inputs(code)
    gen = torch.Generator(device="cuda").manual_seed(8)
    for frames in (8193, 8224, 8225):
        llr = torch.randn((frames, code.n), generator=gen, device="cuda") * 4.0 - 5.0
        llr[:, 7::11] = 0.0
        llr[::5, 3::4] = 0.0
        got = ldpc.ldpc_decode(h, llr, 6)
        ref = ldpc.ldpc_decode(h, llr, 6, streams=1)
        for k in ref:
            assert torch.equal(got[k], ref[k]), (frames, k)


@pytest.mark.parametrize("frames", [3, 33, 70])
@pytest.mark.parametrize("degrees", [[3, 4, 6], [7, 12], [5, 17, 18], [8, 25]])
def test_nan_inputs(ldpc, degrees, frames):  # noqa: F811
    """A channel value that is no number enters every check as it does in the
    pass kernels, and spoils the same decisions."""
    m, n = 97, 410
    rows, cols = random_code(m, n, degrees, seed=sum(degrees))
    h = ldpc.ldpc_code_create(m, n, rows, cols)
    gen = torch.Generator(device="cuda").manual_seed(frames)
    llr = torch.randn((frames, n), generator=gen, device="cuda") * 4.0 - 3.0
    llr[::2, 5::37] = float("nan")
    for msg in ("f32", "f16", "bf16", "i8"):
        for rule in ("sum_product", "min_sum"):
            for max_iter in (0, 1, 7):
                got, ref = decodes(ldpc, h, llr, max_iter, early_exit=False, msg_dtype=msg, rule=rule)
                for k in ref:
                    assert torch.equal(torch.nan_to_num(got[k].float(), 123.0), torch.nan_to_num(ref[k].float(), 123.0)), (
                        msg, rule, max_iter, k)
                assert torch.equal(got["post"].isnan(), ref["post"].isnan())


@pytest.mark.parametrize("msg", ["f32", "f16", "bf16", "i8"])
def test_variables_without_a_check(ldpc, msg):  # noqa: F811
    """Their posteriors are their channel values, -0 included, in every format."""
    m, n = 40, 600
    rows, cols = random_code(m, n, [3, 6], seed=1)
    free = np.setdiff1d(np.arange(n), cols)
    assert free.size > 300
    h = ldpc.ldpc_code_create(m, n, rows, cols)
    gen = torch.Generator(device="cuda").manual_seed(2)
    llr = torch.randn((40, n), generator=gen, device="cuda") * 4.0
    llr[:, ::3] = -0.0
    got, ref = decodes(ldpc, h, llr, 5, early_exit=False, msg_dtype=msg)
    for k in ref:
        a, b = (x.view(torch.int32) if x.dtype == torch.float32 else x for x in (got[k], ref[k]))  # -0 is not +0
        assert torch.equal(a, b), k
    at = torch.from_numpy(free).cuda()
    assert torch.equal(got["post"][:, at].view(torch.int32), llr[:, at].view(torch.int32))


REFUSED_IN_A_CAPTURE = """
import torch
from paper_1609_01567_gb300 import inputs, ldpc
code = inputs.small_code_n1008()
h = ldpc.code_from_inputs(code)
llr = torch.full((8, code.n), -3.0, device="cuda")
out = ldpc.ldpc_decode(h, llr, 5)
torch.cuda.synchronize()
refused = False
try:
    with torch.cuda.graph(torch.cuda.CUDAGraph()):
        ldpc.ldpc_decode(h, llr, 5, out=out)  # waits for the decode before it, which the capture does not hold
except Exception:
    refused = True
again = ldpc.ldpc_decode(h, llr, 5)
torch.cuda.synchronize()
assert refused and not again["bits"].any() and again["ok"].all()
"""


def test_decode_after_one_that_a_capture_refused(ldpc):  # noqa: F811
    r = subprocess.run([sys.executable, "-c", REFUSED_IN_A_CAPTURE], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
