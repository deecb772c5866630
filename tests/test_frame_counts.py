"""Calls whose frame count is close to 2^31: every frame is reached, and no
frame index wraps. Single frames are compared with short calls."""
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


def test_channel_noise(ldpc):
    """Rows of one sample (8.6 GB): the frame loop steps by up to 65,535 frames."""
    frames = 2 ** 31 - 1
    llr = torch.full((frames, 1), 7.0e30, device="cuda")
    ldpc.ldpc_gen_awgn(11, 0, frames, 1, 0.5, out=llr)
    for at, count in ((0, 4096), (65535 * 17 - 100, 200), (2 ** 30 - 50, 100), (frames - 70000, 70000)):
        want = ldpc.ldpc_gen_awgn(11, at, count, 1, 0.5)
        assert torch.equal(llr[at:at + count], want), at
    assert float(llr.max()) < 1.0e30  # every sample was written


def test_dense_encoder(ldpc):
    """One information bit a word (2.1 GB in, 4.3 GB out), encoded in rounds of
    65,536 frames: the word repeats its bit."""
    frames = 2 ** 31 - 64
    h = ldpc.ldpc_code_create(1, 2, [0, 0], [0, 1])
    info = torch.empty((frames, 1), dtype=torch.uint8, device="cuda").random_(0, 2)
    words = torch.full((frames, 2), 2, dtype=torch.uint8, device="cuda")
    ldpc.ldpc_encode(h, info, out=words)
    for part, bits in zip(words.split(2 ** 28), info.split(2 ** 28)):
        assert torch.equal(part, bits.expand(-1, 2))


@pytest.mark.parametrize("n", [1, 4, 7, 33, 128, 129, 516, 1023, 1028, 2052])
def test_channel_noise_of_short_and_odd_rows(ldpc, n):
    """Frames beside each other in a CTA: every frame's noise is that of the frame
    alone, and its codeword enters it."""
    for frames in (1, 2, 700):
        cw = torch.randint(0, 2, (frames, n), dtype=torch.uint8, device="cuda")
        for words in (None, cw):
            llr = ldpc.ldpc_gen_awgn(5, 100, frames, n, 0.8, words)
            for f in sorted({0, frames // 2, frames - 1}):
                one = ldpc.ldpc_gen_awgn(5, 100 + f, 1, n, 0.8, None if words is None else words[f:f + 1].clone())
                assert torch.equal(llr[f:f + 1], one), (frames, f)


@pytest.mark.parametrize("n", [2047, 2049, 2052, 4092, 4095, 4098])
def test_error_counts_of_unaligned_words(ldpc, n):
    """Loads of one and four bytes on both sides of the lengths where a CTA takes
    over from a warp, and more frames than CTAs in flight."""
    for frames in (3, 2500):
        bits = torch.randint(0, 2, (frames, n), dtype=torch.uint8, device="cuda")
        ref = torch.randint(0, 2, (frames, n), dtype=torch.uint8, device="cuda")
        ref[::2] = bits[::2]
        for r in (None, ref):
            wrong = (bits != (0 if r is None else r)).sum(1)
            got = ldpc.ldpc_count_errors(bits, r)
            assert got.tolist() == [int(wrong.sum()), int((wrong > 0).sum()), 0, 0]
