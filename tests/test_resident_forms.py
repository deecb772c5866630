"""Forms of the resident decode that depend on a code's mixture of degrees,
compared bit for bit with the pass kernels (a profiled decode runs those)."""
import numpy as np
import pytest

from tests.test_resident import decodes, ldpc, random_code  # noqa: F401  (ldpc is a fixture)

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


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
