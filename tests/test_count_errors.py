"""The error counter over its forms: a warp or a CTA a frame, loads of 16, 4 and
1 bytes, more frames than the grid holds at once."""
import pytest

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


@pytest.mark.parametrize("frames,n", [(1, 1), (9, 15), (33, 16), (6000, 36), (7, 4096), (3, 4097), (700, 4100), (5, 64800)])
@pytest.mark.parametrize("with_ref", [False, True])
def test_counts(ldpc, frames, n, with_ref):
    gen = torch.Generator(device="cuda").manual_seed(frames + n)

    def draw(hi, shape):
        return torch.randint(0, hi, shape, generator=gen, device="cuda", dtype=torch.int32)

    bits, ref = draw(2, (frames, n)).to(torch.uint8), draw(2, (frames, n)).to(torch.uint8)
    bits[::3] = ref[::3] if with_ref else 0  # frames without an error
    iters, ok = draw(50, (frames,)), draw(2, (frames,)).to(torch.uint8)
    wrong = (bits != (ref if with_ref else 0)).sum(1)
    want = torch.stack([wrong.sum(), (wrong > 0).sum(), iters.sum(), (ok == 0).sum()])
    counts = torch.full((4,), 5, dtype=torch.int64, device="cuda")  # added to what is there
    ldpc.ldpc_count_errors(bits, ref if with_ref else None, iters, ok, counts=counts)
    assert torch.equal(counts - 5, want)
    odd = torch.empty(frames * n + 1, dtype=torch.uint8, device="cuda")[1:].view(frames, n)
    odd.copy_(bits)
    assert torch.equal(ldpc.ldpc_count_errors(odd, ref if with_ref else None)[:2], want[:2])
