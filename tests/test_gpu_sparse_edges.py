"""General codes whose columns have every degree from 1 to 8 and rows every kernel width up to 32, with
ragged variable and frame counts; and convolutional codes with an odd number of variables a frame."""
import numpy as np
import pytest

import oracle
import synth
from test_gpu_ldpccc import compare, pkg, run_gpu  # noqa: F401  (the module's fixture)

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


# rows of about 7, 14, 21 and 28 edges
@pytest.mark.parametrize("N,M,gamma", [(203, 130, 130), (202, 65, 33), (201, 43, 64), (203, 33, 1)])
@pytest.mark.parametrize("early", [0, 1])
def test_every_degree(pkg, N, M, gamma, early):
    """Min-sum bit for bit; sum-product posteriors after five iterations within the suite's 1e-4 (FP32) and
    1.2e-2 (FP16 storage, twice the 6e-3 that test_gpu_qc measures)."""
    rp, col = synth.random_ldpc(N, M, seed=N, var_degrees=(1, 2, 3, 4, 5, 6, 7, 8))
    code = pkg.SparseCode(rp, col, N)
    mu = synth.integer_llrs(gamma, N, seed=M, lo=-60, hi=90, scale=0.25)
    out = code.decode(torch.from_numpy(mu).cuda(), max_iter=8, early_stop=bool(early), algo=pkg.ALGO_MS)
    po, ho, io, oo = oracle.ms_decode(rp, col, N, mu, 8, early_stop=bool(early))
    post, hard, iters, ok = [x.cpu().numpy() for x in out]
    assert np.array_equal(post, po.astype(np.float32) * 0.25)
    assert np.array_equal(hard, ho) and np.array_equal(iters, io) and np.array_equal(ok, oo)
    mu = synth.gaussian_llrs(gamma, N, seed=M, ebn0_db=0.0, rate=0.5)  # no frame stops
    mu[0, ::7] = 0.0  # erased inputs: infinite transforms
    po = oracle.sp_decode(rp, col, N, mu, 5, nthreads=8)[0]
    for msg, tol in ((pkg.MSG_F32, 1e-4), (pkg.MSG_F16, 1.2e-2)):
        post, _, it, _ = code.decode(torch.from_numpy(mu).cuda(), max_iter=5, early_stop=bool(early), msg=msg)
        run = it.cpu().numpy() == 5
        assert run.any()
        err = np.abs(post.cpu().numpy() - po) / np.maximum(1.0, np.abs(po))
        assert np.max(err[run]) <= tol, msg


@pytest.mark.parametrize("J,L,p", [(3, 9, 7), (1, 5, 11)])
def test_ldpccc_odd_frames(pkg, J, L, p):
    shifts = synth.qc_shifts(J, L, p, seed=3)
    c = pkg.LDPCCC(shifts, p, 3, 40).c
    assert c % 2 == 1
    mu = synth.gaussian_llrs(40, 14 * c, seed=2, ebn0_db=2.0, rate=0.5).reshape(40, 14, c)
    hard, post, decided = run_gpu(pkg, shifts, p, 3, mu, [5, 9])
    compare(shifts, p, 3, mu, hard, post, decided, f"odd frames {J}x{L}")
