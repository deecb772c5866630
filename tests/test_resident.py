"""The resident decode (a frame's iterations inside one CTA) gives the results
of the pass kernels bit for bit. A profiled decode runs the pass kernels."""
import numpy as np
import pytest

from paper_1609_01567_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ldpc():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1609_01567_gb300 import build
    build.build()
    from paper_1609_01567_gb300 import ldpc as mod
    return mod


def random_code(m, n, degrees, seed, wide_vars=0):
    """m checks whose degrees cycle through ``degrees``; ``wide_vars`` variables
    enter every third check."""
    rng = np.random.default_rng(seed)
    rows, cols = [], []
    for i in range(m):
        c = set(rng.choice(n, size=min(n, degrees[i % len(degrees)]), replace=False).tolist())
        if i % 3 == 0:
            c |= set(range(wide_vars))
        rows += [i] * len(c)
        cols += sorted(c)
    order = rng.permutation(len(rows))
    return np.asarray(rows, np.int32)[order], np.asarray(cols, np.int32)[order]


# one group of 32 checks and its edges, pairs of groups, every row width, the
# border between checks of at most four inputs and larger ones, nodes worked on
# by a whole warp, lengths that are no multiple of four
CODES = {
    "one_check": (1, 5, [3], 0),
    "32_checks": (32, 61, [4], 0),
    "33_checks": (33, 64, [6], 0),
    "65_checks": (65, 130, [8], 0),
    "small_degrees": (96, 203, [1, 2, 3, 4], 0),
    "border": (97, 256, [3, 4, 5, 6], 0),
    "mixed": (130, 411, [2, 6, 7, 9, 12, 13], 0),
    "degree_18": (70, 302, [5, 17, 18], 0),
    "degree_32": (40, 500, [4, 20, 32], 0),
    "wide": (80, 349, [3, 6, 11, 40], 2),
}


def decodes(ldpc, h, llr, max_iter, **kw):
    got = ldpc.ldpc_decode(h, llr, max_iter, **kw)
    ref = ldpc.ldpc_decode(h, llr, max_iter, profile=True, **kw)
    torch.cuda.synchronize()
    ldpc.ldpc_prof_read(h, reset=True)
    return got, ref


@pytest.mark.parametrize("msg", ["f32", "f16", "bf16", "i8"])
@pytest.mark.parametrize("name", list(CODES))
def test_equals_the_pass_kernels(ldpc, name, msg):
    m, n, degrees, wide_vars = CODES[name]
    rows, cols = random_code(m, n, degrees, seed=m + n, wide_vars=wide_vars)
    h = ldpc.ldpc_code_create(m, n, rows, cols)
    gen = torch.Generator(device="cuda").manual_seed(n)
    ldpc.ldpc_code_set_rule_table(h, [0.9 - 0.02 * (d % 7) for d in range(50)], [0.05 * (d % 3) for d in range(50)])
    for frames, max_iter, early, rule in ((1, 20, True, "sum_product"), (40, 9, False, "sum_product"),
                                          (70, 20, True, "sum_product"), (5, 0, True, "sum_product"),
                                          (70, 20, True, "min_sum"), (70, 6, False, "min_sum_adaptive")):
        llr = torch.randn((frames, n), generator=gen, device="cuda") * 4.0 - 3.0
        got, ref = decodes(ldpc, h, llr, max_iter, early_exit=early, msg_dtype=msg, rule=rule,
                           rule_beta=0.15 if rule == "min_sum" else 0.0)
        for k in ref:
            assert torch.equal(got[k], ref[k]), (name, msg, frames, rule, k)


@pytest.mark.parametrize("frames", [3, 40])
@pytest.mark.parametrize("rule", ["sum_product", "min_sum"])
def test_erased_saturated_and_infinite_inputs(ldpc, frames, rule):
    code = I.small_code_n1008()
    h = ldpc.code_from_inputs(code)
    gen = torch.Generator(device="cuda").manual_seed(frames)
    llr = torch.randn((frames, code.n), generator=gen, device="cuda") * 4.0 - 6.0
    llr[:, 7::11] = 0.0
    llr[:, 3::97] = -0.0
    llr[:, 5::89] = -300.0
    llr[:, 2::83] = float("-inf")
    llr[-1] = 0.0  # a frame of erasures only
    got, ref = decodes(ldpc, h, llr, 12, rule=rule)
    for k in ref:
        assert torch.equal(got[k], ref[k]), k


def test_odd_buffers_and_other_stream(ldpc):
    """Outputs that are not word-aligned, no posteriors, a side stream."""
    code = I.small_code_n1008()
    h = ldpc.code_from_inputs(code)
    gen = torch.Generator(device="cuda").manual_seed(3)
    llr = torch.randn((37, code.n), generator=gen, device="cuda") * 4.0 - 5.0
    raw = torch.zeros(37 * code.n + 1, dtype=torch.uint8, device="cuda")
    out = {"bits": raw[1:].view(37, code.n)}
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        got = ldpc.ldpc_decode(h, llr, 15, want_post=False, out=out, stream=side)
    side.synchronize()
    ref = ldpc.ldpc_decode(h, llr, 15, want_post=False, profile=True)
    for k in ("bits", "iters", "ok"):
        assert torch.equal(got[k], ref[k]), k
    assert int(raw[0]) == 0
