"""Encoder and channel rows on and off the alignment their wide accesses need: buffers that start one
element late and codes of every length modulo 4 give the bytes that aligned rows give."""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1204_0334_gb300 as p

    p.lib()
    return p


@pytest.mark.parametrize("p", [20, 21, 22, 23])  # N = 9 p: 0, 1, 2, 3 mod 4
@pytest.mark.parametrize("gamma", [1, 32, 37])
def test_rows_on_and_off_alignment(pkg, p, gamma):
    shifts = synth.qc_shifts(3, 9, p, seed=4)
    code = pkg.QCCode(shifts, p)
    H = np.asarray(oracle.qc_parity_check(shifts, p), dtype=np.int64)
    k, pos = code.info_set()
    rng = np.random.default_rng(p * 100 + gamma)
    info = torch.from_numpy(rng.integers(0, 2, (gamma, k)).astype(np.uint8)).cuda()

    def late(shape, dtype):  # a contiguous tensor one element past an aligned start
        n = int(np.prod(shape))
        return torch.empty(n + 1, dtype=dtype, device="cuda")[1:].view(shape)

    cw = code.encode(info)
    got = cw.cpu().numpy()
    assert np.array_equal(got[:, pos], info.cpu().numpy()) and not ((got.astype(np.int64) @ H.T) % 2).any()
    cw2, info2 = late((gamma, code.N), torch.uint8), late((gamma, k), torch.uint8)
    info2.copy_(info)
    pkg.ldpc_encode(code.handle, info2, cw2)
    assert torch.equal(cw, cw2)
    llr = code.channel_codewords(2.0, 9, 5, cw)
    llr2 = late((gamma, code.N), torch.float32)
    pkg.ldpc_channel_codewords(code.handle, 2.0, 9, 5, cw2, llr2)
    assert torch.equal(llr, llr2)
    zero = torch.zeros_like(cw)
    out = late((gamma, code.N), torch.float32)
    pkg.ldpc_channel(code.handle, 2.0, 9, 5, out)
    assert torch.equal(out, code.channel(2.0, 9, 5, gamma))
    assert torch.equal(out, code.channel_codewords(2.0, 9, 5, zero))
    sigma = oracle.sigma_from_ebn0(2.0, code.K / code.N)
    assert np.array_equal(out.cpu().numpy(), oracle.channel_awgn(9, 5, gamma, code.N, sigma))
