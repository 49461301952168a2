"""ldpc_decode of few frames of a short code (a package per thread-block cluster, everything on chip)
against the same frames in a batch too large for it, bit for bit; and the flow decoder at the edges of
its tiles on codes too long for a cluster, against the oracle."""
import numpy as np
import pytest

import oracle
import synth
from test_gpu_flow import pkg, setup  # noqa: F401  (the module's fixture)

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


# J, L, p, zero blocks: fewer variables than blocks of a cluster, ragged shares of them, rows of 6, 8, 12
# and 24 edges with and without zero blocks, more than four block rows
@pytest.mark.parametrize("J,L,p,zero", [(1, 2, 1, 0), (2, 5, 3, 1), (3, 6, 16, 0), (3, 6, 37, 2), (4, 8, 25, 0),
                                        (4, 12, 13, 0), (4, 16, 11, 3), (4, 24, 17, 0), (5, 10, 9, 4), (8, 32, 3, 20)])
@pytest.mark.parametrize("algo,msg", [(0, 0), (0, 1), (1, 2), (2, 0), (2, 1)])
def test_parts_equal_large_batch(pkg, J, L, p, zero, algo, msg):
    code, rp, col = setup(pkg, J, L, p, zero, 9)
    W = 32 << msg
    mu = torch.from_numpy(synth.gaussian_llrs(153 * W + 1, code.N, seed=L, ebn0_db=2.0, rate=0.5)).cuda()
    mu[0, : code.N // 2] = 0.0  # erased inputs: infinite transforms
    mu[1] *= 1e6
    prm = torch.from_numpy(np.random.default_rng(1).uniform(0.05, 0.9, (11, J * L, 2)).astype(np.float32)).cuda()

    def decode(x, early):
        o = pkg.default_opts(max_iter=11, early_stop=early, algo=algo, msg=msg)
        o.noms_params = prm.data_ptr() if algo == 2 else None
        n = x.shape[0]
        out = (torch.empty((n, code.N), device="cuda"), torch.empty((n, code.N), dtype=torch.uint8, device="cuda"),
               torch.empty(n, dtype=torch.int32, device="cuda"), torch.empty(n, dtype=torch.int32, device="cuda"))
        pkg.ldpc_decode(code.handle, x, o, *out)
        return out

    for early in (0, 1):
        whole = decode(mu, early)
        for at, n in ((0, 1), (0, W - 1), (3 * W, W + 1), (W, 10 * W), (0, 40 * W), (2 * W, 130 * W)):
            for a, b in zip(whole, decode(mu[at:at + n], early)):
                assert torch.equal(a[at:at + n], b), (early, at, n)


# codes of more lines than a cluster takes: ragged last rows and variables, 6 to 32 edges a row
@pytest.mark.parametrize("J,L,p,zero,gamma", [(3, 6, 715, 0, 33), (4, 12, 271, 0, 65), (4, 24, 137, 0, 40),
                                              (4, 20, 169, 3, 31), (3, 32, 149, 4, 36), (5, 12, 233, 4, 34),
                                              (8, 32, 61, 20, 66)])
def test_flow_long_codes_against_oracle(pkg, J, L, p, zero, gamma):
    """Min-sum bit for bit; sum-product posteriors after five iterations within the suite's 1e-4 (FP32) and
    1.2e-2 (FP16 storage, twice the 6e-3 that test_gpu_qc measures)."""
    code, rp, col = setup(pkg, J, L, p, zero, 5)
    mu = synth.integer_llrs(gamma, code.N, seed=J + L + p, lo=-30, hi=60, scale=0.25)
    out = code.decode(torch.from_numpy(mu).cuda(), max_iter=9, early_stop=True, algo=pkg.ALGO_MS)
    po, ho, io, oo = oracle.ms_decode(rp, col, code.N, mu, 9, early_stop=True)
    post, hard, iters, ok = [x.cpu().numpy() for x in out]
    assert np.array_equal(post, po.astype(np.float32) * 0.25)
    assert np.array_equal(hard, ho) and np.array_equal(iters, io) and np.array_equal(ok, oo)
    mu = synth.gaussian_llrs(gamma, code.N, seed=p, ebn0_db=1.0, rate=0.5)  # no frame stops early
    po, _, io, _ = oracle.sp_decode(rp, col, code.N, mu, 5, early_stop=True, nthreads=8)
    for msg, tol in ((pkg.MSG_F32, 1e-4), (pkg.MSG_F16, 1.2e-2)):
        post, _, it, _ = code.decode(torch.from_numpy(mu).cuda(), max_iter=5, early_stop=True, msg=msg)
        same = it.cpu().numpy() == io
        assert same.any()
        err = np.abs(post.cpu().numpy() - po) / np.maximum(1.0, np.abs(po))
        assert np.max(err[same]) <= tol, msg
