"""The pass kernels on short codes, with the options that keep a decode on them
(streams, frames_per_lane, check_schedule): graph capture and replay, workspace
growth, chunks, and the kernel forms that a code short enough for one SM does
not reach by default. Every decode here launches more than one kernel, and its
results equal the default decode's bit for bit."""
import numpy as np
import pytest

from paper_1609_01567_gb300 import inputs as I
from tests.test_graph_replay import ldpc, llrs  # noqa: F401  (ldpc is a fixture)
from tests.test_resident import random_code

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

KEYS = ("bits", "iters", "ok", "post")


def passes(ldpc, h, llr, max_iter, **kw):  # noqa: F811
    """A decode that has to run the pass kernels; direct, captured and replayed
    calls count their kernels alike."""
    ldpc.ldpc_prof_read(h, reset=True)
    out = ldpc.ldpc_decode(h, llr, max_iter, **kw)
    torch.cuda.synchronize()
    assert ldpc.ldpc_prof_read(h, reset=True)["kernels"] > 1, kw
    return out


def same(got, ref, what=None):
    for k in KEYS:
        if k in ref:
            assert torch.equal(got[k], ref[k]), (k, what)


@pytest.mark.parametrize("kw", [dict(streams=1), dict(streams=2, msg_dtype="bf16", early_exit=False),
                                dict(streams=1, rule="min_sum", rule_alpha=0.8), dict(streams=1, msg_dtype="i8")])
def test_replays_follow_buffer_contents(ldpc, kw):  # noqa: F811
    code = I.small_code_n1008()
    h = ldpc.code_from_inputs(code)
    buf = llrs(code, 300, 1.5, seed=1)
    plain = {k: v for k, v in kw.items() if k != "streams"}
    out, counts = None, []
    for rnd in range(4):  # direct, captured, replayed, replayed
        buf.copy_(llrs(code, 300, 1.5, seed=10 + rnd))
        ldpc.ldpc_prof_read(h, reset=True)
        out = ldpc.ldpc_decode(h, buf, 25, out=out, **kw)
        torch.cuda.synchronize()
        counts.append(ldpc.ldpc_prof_read(h, reset=True)["kernels"])
        same(out, ldpc.ldpc_decode(h, buf, 25, **plain), rnd)
    assert counts[0] > 1 and len(set(counts)) == 1, counts


def test_alternating_buffers_workspace_growth_and_chunks(ldpc):  # noqa: F811
    code = I.small_code_n1008()
    h = ldpc.code_from_inputs(code)
    a, b = llrs(code, 64, 2.0, seed=3), llrs(code, 64, 2.0, seed=4)
    big = llrs(code, 8192 + 300, 2.0, seed=5)  # two chunks; grows the workspace, which drops the captured graphs
    oa = ob = obig = None
    for llr_set in ((a, b), (a, b), (a, b), (big,), (big,), (big,), (a,), (a,), (a,)):
        for x in llr_set:
            if x is a:
                oa = passes(ldpc, h, a, 20, out=oa, streams=1)
            elif x is b:
                ob = passes(ldpc, h, b, 20, out=ob, streams=1)
            else:
                obig = passes(ldpc, h, big, 6, out=obig, streams=1)
    same(oa, ldpc.ldpc_decode(h, a, 20))
    same(ob, ldpc.ldpc_decode(h, b, 20))
    same(obig, ldpc.ldpc_decode(h, big, 6))


def test_host_entry_replays_and_counts_kernels(ldpc):  # noqa: F811
    code = I.small_code_n1008()
    h = ldpc.code_from_inputs(code)
    host = llrs(code, 100, 1.75, seed=6).cpu().pin_memory()
    ref = ldpc.ldpc_decode(h, host.cuda(), 15)
    torch.cuda.synchronize()
    ldpc.ldpc_prof_read(h, reset=True)
    for _ in range(3):
        got = ldpc.ldpc_decode_host(h, host, 15, streams=1)
        for k in ("bits", "iters", "ok"):
            np.testing.assert_array_equal(np.asarray(got[k]), ref[k].cpu().numpy(), err_msg=k)
    k3 = ldpc.ldpc_prof_read(h, reset=True)["kernels"]
    ldpc.ldpc_decode_host(h, host, 15, streams=1)
    k1 = ldpc.ldpc_prof_read(h, reset=True)["kernels"]
    assert k1 > 1 and k3 == 3 * k1


def test_replays_read_the_current_rule_table(ldpc):  # noqa: F811
    code = I.small_code_n1008()
    h = ldpc.code_from_inputs(code)
    buf = llrs(code, 300, 1.5, seed=21)
    out = None
    for a5, a6 in ((0.7, 0.9), (0.7, 0.9), (0.7, 0.9), (0.95, 0.6), (0.6, 0.8)):
        ldpc.ldpc_code_set_rule_table(h, [1.0] * 5 + [a5, a6], [0.0] * 5 + [0.1, 0.2])
        out = passes(ldpc, h, buf, 25, out=out, rule="min_sum_adaptive", streams=1)
        same(out, ldpc.ldpc_decode(h, buf, 25, rule="min_sum_adaptive"), (a5, a6))


def test_halves_that_stop_far_apart(ldpc):  # noqa: F811
    code = I.small_code_n1008()
    h = ldpc.code_from_inputs(code)
    buf = torch.cat([llrs(code, 256, 4.0, seed=31), llrs(code, 256, 1.2, seed=32)])
    for max_iter in (50, 23):
        out = None
        for _ in range(4):  # direct, captured, replayed, replayed
            out = passes(ldpc, h, buf, max_iter, out=out, streams=2)
        same(out, ldpc.ldpc_decode(h, buf, max_iter), max_iter)
        assert int(out["iters"][:256].max()) < 16 and int(out["iters"][256:].max()) >= 20


def test_unaligned_caller_buffers(ldpc):  # noqa: F811
    code = I.small_code_n1008()
    h = ldpc.code_from_inputs(code)
    f, n = 70, code.n
    llr = llrs(code, f, 2.0, seed=8)
    lbuf = torch.zeros(f * n + 1, device="cuda")
    lbuf[1:] = llr.flatten()
    out = {"bits": torch.zeros(f * n + 1, dtype=torch.uint8, device="cuda")[1:].view(f, n),
           "post": torch.zeros(f * n + 1, device="cuda")[1:].view(f, n)}
    same(passes(ldpc, h, lbuf[1:].view(f, n), 12, out=out, streams=1), ldpc.ldpc_decode(h, llr, 12))


# The check kernels' slot counts: 10 (largest degree 9 or 10), 12, 16 and 18, in
# batches of whole 64-frame groups; check_schedule 1 runs the direct-load forms.
@pytest.mark.parametrize("msg", ["f32", "f16", "bf16", "i8"])
@pytest.mark.parametrize("degrees", [[9], [10, 9], [12, 11], [13, 16], [18, 17]])
def test_slot_counts_of_the_pipelined_check_kernel(ldpc, degrees, msg):  # noqa: F811
    m, n = 97, 520
    rows, cols = random_code(m, n, degrees, seed=m + degrees[0])
    h = ldpc.ldpc_code_create(m, n, rows, cols)
    gen = torch.Generator(device="cuda").manual_seed(degrees[0])
    for frames, rule in ((70, "sum_product"), (300, "sum_product"), (70, "min_sum")):
        llr = torch.randn((frames, n), generator=gen, device="cuda") * 4.0 - 3.0
        kw = dict(msg_dtype=msg, rule=rule, early_exit=False)
        ring = passes(ldpc, h, llr, 7, streams=1, **kw)
        same(passes(ldpc, h, llr, 7, streams=1, check_schedule=1, **kw), ring, (frames, rule, "direct loads"))
        same(ldpc.ldpc_decode(h, llr, 7, **kw), ring, (frames, rule, "default"))


@pytest.mark.parametrize("idx,ebn0", [(0, 4.0), (1, 3.6), (2, 3.0), (4, 2.8)])
def test_named_short_codes(ldpc, idx, ebn0):  # noqa: F811
    """The 18-, 12- and 10-slot rings and the degree-96 check of the mixed codes."""
    code = I.mixed_code(idx)
    h = ldpc.code_from_inputs(code)
    llr = llrs(code, 256, ebn0, seed=77 + idx)
    for msg in ("f32", "bf16", "i8"):
        base = passes(ldpc, h, llr, 15, msg_dtype=msg, streams=1)
        same(passes(ldpc, h, llr, 15, msg_dtype=msg, frames_per_lane=1, check_schedule=1, streams=1), base, msg)
        same(ldpc.ldpc_decode(h, llr, 15, msg_dtype=msg), base, msg)
    part = passes(ldpc, h, llr[:20], 15, streams=1)
    full = ldpc.ldpc_decode(h, llr, 15)
    same(part, {k: v[:20] for k, v in full.items()}, "20 frames")
