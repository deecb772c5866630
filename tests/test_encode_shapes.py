"""The encoders over the shapes where their kernels change: word lengths and
buffers of every alignment, frame counts around eight and 32, checks around the
groups and warps, and the codes that the one-kernel form leaves to the general
path."""
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


def staircase(m, k, seed, heavy=0):
    """H = [H1 | dual diagonal]; the first check holds ``heavy`` more columns."""
    rng = np.random.default_rng(seed)
    rows, cols = [], []
    for i in range(m):
        d = min(k, int(rng.integers(0, 6)) + (heavy if i == 0 else 0))
        c = rng.choice(k, size=d, replace=False) if k else np.empty(0, int)
        rows += [i] * len(c)
        cols += c.tolist()
        rows.append(i)
        cols.append(k + i)
        if i:
            rows.append(i)
            cols.append(k + i - 1)
    return np.asarray(rows, np.int32), np.asarray(cols, np.int32)


def parity(rows, cols, m, k, info):
    s = np.zeros((m, info.shape[0]), np.uint8)
    sel = cols < k
    np.bitwise_xor.at(s, rows[sel], info.T[cols[sel]])
    return (np.cumsum(s, axis=0) & 1).T.astype(np.uint8)


@pytest.mark.parametrize("m,k,heavy", [(1, 1, 0), (7, 0, 0), (31, 17, 0), (32, 32, 0), (33, 35, 0), (128, 64, 0),
                                       (129, 127, 0), (1000, 1032, 0), (2048, 2064, 0), (5001, 3000, 0),
                                       (16400, 400, 0), (300, 4000, 3500), (230000, 40, 0)])
def test_ira_encoder(ldpc, m, k, heavy):
    rows, cols = staircase(m, k, seed=m + k, heavy=heavy)
    h = ldpc.ldpc_code_create(m, m + k, rows, cols)
    rng = np.random.default_rng(k)
    for frames in (1, 8, 9, 33):
        info = rng.integers(0, 2, size=(frames, k), dtype=np.uint8)
        want = np.concatenate([info, parity(rows, cols, m, k, info)], axis=1)
        got = ldpc.ldpc_encode_ira(h, torch.from_numpy(info).cuda())
        np.testing.assert_array_equal(got.cpu().numpy(), want, err_msg=f"{frames} frames")
        raw = torch.zeros(frames * (m + k) + 1, dtype=torch.uint8, device="cuda")  # rows at odd addresses
        src = torch.zeros(frames * k + 1, dtype=torch.uint8, device="cuda")
        src[1:] = torch.from_numpy(info).cuda().flatten()
        ldpc.ldpc_encode_ira(h, src[1:].view(frames, k), out=raw[1:].view(frames, m + k))
        np.testing.assert_array_equal(raw[1:].view(frames, m + k).cpu().numpy(), want)
        assert int(raw[0]) == 0


@pytest.mark.parametrize("n", [264, 520, 1032])
def test_dense_encoder(ldpc, n):
    code, entries = I.qc_stand_in_code(n)
    h = ldpc.ldpc_code_create_qc(4, 8, n // 8, entries)
    k = ldpc.ldpc_code_build_encoder(h)
    gen = torch.Generator(device="cuda").manual_seed(n)
    # the code words of the unit vectors give every other word
    unit = ldpc.ldpc_encode(h, torch.eye(k, dtype=torch.uint8, device="cuda")).float()
    for frames in (1, 31, 33, 1024, 1030):
        info = torch.randint(0, 2, (frames, k), generator=gen, device="cuda", dtype=torch.uint8)
        want = (info.double() @ unit.double()).remainder(2).to(torch.uint8)
        assert torch.equal(ldpc.ldpc_encode(h, info), want), frames
        raw = torch.zeros(frames * n + 1, dtype=torch.uint8, device="cuda")
        ldpc.ldpc_encode(h, info, out=raw[1:].view(frames, n))
        assert torch.equal(raw[1:].view(frames, n), want), frames
    s = torch.zeros((code.m, k), device="cuda", dtype=torch.float64)
    s.index_add_(0, torch.from_numpy(code.rows.astype(np.int64)).cuda(),
                 unit.double().t()[torch.from_numpy(code.cols.astype(np.int64)).cuda()])
    assert not s.remainder(2).any()
