"""The one-kernel IRA encoder around the amounts of shared memory where its
launch changes: 48 KB, from where a launch needs an opt-in, and the longest word
that it serves. The opt-in lasts for a process and a kernel form, so the words
around 48 KB are encoded in a process of their own, in rising order."""
import subprocess
import sys
from pathlib import Path

import numpy as np
import pytest

from tests.test_encode_shapes import parity

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ROOT = Path(__file__).resolve().parent.parent


def long_staircase(m, k, seed):
    """H = [H1 | dual diagonal] with up to three columns of H1 a check."""
    rng = np.random.default_rng(seed)
    at = np.unique(np.repeat(np.arange(m, dtype=np.int64), 3) * k + rng.integers(0, k, 3 * m))
    i = np.arange(m, dtype=np.int64)
    rows = np.concatenate([at // k, i, i[1:]])
    cols = np.concatenate([at % k, k + i, k + i[:-1]])
    return rows.astype(np.int32), cols.astype(np.int32)


def encode(n, k, frames=9):
    from paper_1609_01567_gb300 import ldpc
    m = n - k
    rows, cols = long_staircase(m, k, seed=n)
    h = ldpc.ldpc_code_create(m, n, rows, cols)
    info = np.random.default_rng(k).integers(0, 2, size=(frames, k), dtype=np.uint8)
    got = ldpc.ldpc_encode_ira(h, torch.from_numpy(info).cuda()).cpu().numpy()
    np.testing.assert_array_equal(got, np.concatenate([info, parity(rows, cols, m, k, info)], axis=1), err_msg=str(n))


# accesses of 16, four and one bytes: n and k are multiples of 16, of four, odd
@pytest.mark.parametrize("k,step", [(24512, 16), (24508, 4), (24001, 2)])
def test_words_around_48_kilobytes(k, step):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    run = (f"from tests.test_encode_limits import encode\n"
           f"for n in [*range(48960 + {k % 2}, 49200, {step * 4}), 49160]:\n"
           f"    encode(n, {k})\n")
    r = subprocess.run([sys.executable, "-c", run], cwd=ROOT, capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stderr[-2000:]


# the longest words of one kernel (229,376 - 48 bits), and the first without it
@pytest.mark.parametrize("n", [229312, 229328, 229329])
def test_longest_words(n):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    for frames in (9, 40):  # few words this long take the general path
        encode(n, 114656, frames)


# information rows of one to nine bits at every byte offset: the words around the
# first and the last byte belong to the buffers' neighbours and hold other values
@pytest.mark.parametrize("k", [1, 2, 3, 4, 5, 9])
def test_dense_encoder_ends_of_the_information(k):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1609_01567_gb300 import ldpc
    rows, cols = [0] * (k + 1), list(range(k + 1))  # one check over all bits: the last one is the parity
    h = ldpc.ldpc_code_create(1, k + 1, rows, cols)
    assert ldpc.ldpc_code_build_encoder(h) == k
    for frames in (1, 2, 3, 31, 33):
        for off in range(4):
            raw = torch.full((off + frames * k + 8,), 255, dtype=torch.uint8, device="cuda")
            info = raw[off:off + frames * k].view(frames, k)
            info.random_(0, 2)
            want = torch.cat([info, info.sum(1, keepdim=True).remainder(2).to(torch.uint8)], 1)
            assert torch.equal(ldpc.ldpc_encode(h, info), want), (frames, off)


# few words of 200,001 bits take the general path, many the one-kernel form
@pytest.mark.parametrize("frames", [1, 8, 200])
def test_long_odd_words(frames):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    encode(200001, 100000, frames)
