"""The flow decoder (ldpc_decode on QC codes) at the edges of its tiles: codes and batches whose rows,
columns, packages and circulant wraps do not fill them, every message rule, with and without early
stop, against the oracle; and more packages than it keeps in work at once."""
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


def setup(pkg, J, L, p, zero, seed):
    shifts = synth.qc_shifts(J, L, p, seed=seed, zero_blocks=zero)
    rp, col = oracle.csr_rows(oracle.qc_parity_check(shifts, p))
    return pkg.QCCode(shifts, p), rp, col


# J, L, p, zero blocks, frames: one-row circulants, a tile's rows and variables +-1, 16/24/32-edge
# rows, more than four block rows, packages with one frame, the regular 4 x 24 shape
SHAPES = [(1, 2, 1, 0, 3), (2, 3, 25, 1, 65), (3, 6, 48, 0, 129), (3, 6, 97, 2, 31), (4, 12, 24, 5, 260),
          (4, 24, 23, 0, 70), (4, 24, 49, 0, 33), (4, 20, 95, 7, 40), (3, 32, 17, 3, 36), (5, 12, 51, 4, 34),
          (8, 32, 13, 20, 66)]


@pytest.mark.parametrize("J,L,p,zero,gamma", SHAPES)
@pytest.mark.parametrize("early", [0, 1])
def test_min_sum_bit_exact(pkg, J, L, p, zero, gamma, early):
    code, rp, col = setup(pkg, J, L, p, zero, 5)
    mu = synth.integer_llrs(gamma, code.N, seed=J + L + p, lo=-30, hi=60, scale=0.25)
    out = code.decode(torch.from_numpy(mu).cuda(), max_iter=9, early_stop=bool(early), algo=pkg.ALGO_MS)
    po, ho, io, oo = oracle.ms_decode(rp, col, code.N, mu, 9, early_stop=bool(early))
    post, hard, iters, ok = [x.cpu().numpy() for x in out]
    assert np.array_equal(post, po.astype(np.float32) * 0.25)
    assert np.array_equal(hard, ho) and np.array_equal(iters, io) and np.array_equal(ok, oo)


@pytest.mark.parametrize("J,L,p,zero,gamma", SHAPES)
def test_sum_product_against_oracle(pkg, J, L, p, zero, gamma):
    """Five iterations: FP32 posteriors within the suite's 1e-4; FP16 storage within 1.2e-2, twice what
    its storage rounding gives per iteration (test_gpu_qc measures 6e-3 after five)."""
    code, rp, col = setup(pkg, J, L, p, zero, 6)
    mu = synth.gaussian_llrs(gamma, code.N, seed=p, ebn0_db=3.0, rate=max(0.5, 1 - J / L))
    mu[0, : code.N // 2] = 0.0  # erased inputs: infinite transforms
    po = oracle.sp_decode(rp, col, code.N, mu, 5, nthreads=8)[0]
    for msg, tol in ((pkg.MSG_F32, 1e-4), (pkg.MSG_F16, 1.2e-2)):
        post = code.decode(torch.from_numpy(mu).cuda(), max_iter=5, msg=msg)[0].cpu().numpy()
        assert np.max(np.abs(post - po) / np.maximum(1.0, np.abs(po))) <= tol, msg


def test_more_packages_than_slots(pkg):
    """9000 frames of a small code (282 packages, 256 in work): every frame's result is that of the same
    frame decoded in a batch of its own package."""
    code, rp, col = setup(pkg, 2, 6, 20, 0, 7)
    mu = torch.from_numpy(synth.gaussian_llrs(9000, code.N, seed=3, ebn0_db=2.0, rate=2 / 3)).cuda()
    whole = code.decode(mu, max_iter=12, early_stop=True)
    for f in (0, 4096, 8992):
        part = code.decode(mu[f:f + 32], max_iter=12, early_stop=True)
        for a, b in zip(whole, part):
            assert torch.equal(a[f:f + 32], b)


@pytest.mark.parametrize("J,L,p,slots,frames", [(3, 6, 17, 32, 1), (3, 6, 64, 128, 700), (4, 12, 31, 4096, 5000),
                                                (5, 10, 33, 64, 333)])
@pytest.mark.parametrize("algo,msg", [(0, 0), (1, 2)])
def test_refill_equals_batch_decode(pkg, J, L, p, slots, frames, algo, msg):
    """The simulation with a target that cannot be met (one launch, lanes refilled) counts what a batch
    decode of the same frames counts; fewer frames than lanes, ragged variable counts, several packages."""
    code = pkg.QCCode(synth.qc_shifts(J, L, p, seed=8), p)
    r = code.ber_sim(2.0, seed=11, first_frame=5, max_frames=frames, target_frame_errors=1 << 40, gamma=slots,
                     max_iter=14, early_stop=1, algo=algo, msg=msg)
    llr = code.channel(2.0, 11, 5, frames)
    _, hard, it, ok = code.decode(llr, max_iter=14, early_stop=True, algo=algo, msg=msg, want_post=False)
    e = hard.sum(dim=1).long()
    assert r["frames"] == frames and r["iters_sum"] == int(it.sum())
    assert r["bit_errors"] == int(e.sum()) and r["frame_errors"] == int((e > 0).sum())
    assert r["bit_errors_sq"] == int((e * e).sum()) and r["undetected"] == int(((e > 0) & (ok == 1)).sum())
