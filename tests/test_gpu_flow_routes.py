"""The flow decoder on calls that are seen to reach it (two launches, whatever the iterations): more packages
than there are slots, every message rule and kernel width, with a fixed count and with early stop, and the
streaming decode, against the same frames decoded by themselves or by a launch per pass."""
import numpy as np
import pytest

import synth
from test_gpu_flow import pkg, setup  # noqa: F401  (the module's fixture)

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def launches(pkg, call):
    pkg.ldpc_profile_enable(False)  # clears the count
    out = call()
    return out, pkg.ldpc_profile_read()["launches"]


@pytest.mark.parametrize("algo,msg,slots", [(0, 1, 16384), (1, 2, 32768)])
def test_simulation_on_256_packages(pkg, algo, msg, slots):
    """A short code's simulation on the most slots there are counts what the simulation by a launch a step
    counts on the same frames (a target that can be met, and is not), and with integer messages what a batch
    decode of them counts (binary16 messages start from rounded channel values there, from FP32 in a batch)."""
    code = pkg.QCCode(synth.qc_shifts(3, 6, 64, seed=8), 64)
    frames = 2 * slots + 77
    kw = dict(max_iter=14, early_stop=1, algo=algo, msg=msg)

    def sim(target):
        r, n = launches(pkg, lambda: code.ber_sim(2.0, seed=11, first_frame=5, max_frames=frames,
                                                  target_frame_errors=target, gamma=slots, **kw))
        r.pop("seconds")
        return r, n

    r, n = sim(1 << 40)
    assert n == 2
    other, n = sim(frames)
    assert n > 2 and r == other
    if msg == 2:
        _, hard, it, ok = code.decode(code.channel(2.0, 11, 5, frames), want_post=False, **kw)
        e = hard.sum(dim=1).long()
        assert r["frames"] == frames and r["iters_sum"] == int(it.sum())
        assert r["bit_errors"] == int(e.sum()) and r["frame_errors"] == int((e > 0).sum())
        assert r["bit_errors_sq"] == int((e * e).sum()) and r["undetected"] == int(((e > 0) & (ok == 1)).sum())


def test_decode_of_more_packages_than_slots(pkg):
    """282 packages of a small code, 256 in work at once."""
    code, _, _ = setup(pkg, 2, 4, 20, 0, 7)
    mu = torch.from_numpy(synth.gaussian_llrs(9000, code.N, seed=3, ebn0_db=2.0, rate=0.5)).cuda()
    whole, n = launches(pkg, lambda: code.decode(mu, max_iter=12, early_stop=True))
    assert n == 2
    for f in range(0, 9000, 3000):
        part, n = launches(pkg, lambda: code.decode(mu[f:f + 3000], max_iter=12, early_stop=True))
        assert n == 1  # on chip
        for a, b in zip(whole, part):
            assert torch.equal(a[f:f + 3000], b)


def test_captured_decodes(pkg):
    """A decode captured after a larger batch that ran in another form, and one replayed after decodes of the
    same frames with other messages and outputs have run on the object."""
    shifts = synth.qc_shifts(4, 24, 765, seed=2)
    code, other = pkg.QCCode(shifts, 765), pkg.QCCode(shifts, 765)
    mu = code.channel(3.0, 5, 0, 600)
    opts = pkg.default_opts(max_iter=6)

    def outputs(n):
        return (torch.empty((n, code.N), device="cuda"), torch.empty((n, code.N), dtype=torch.uint8, device="cuda"),
                torch.empty(n, dtype=torch.int32, device="cuda"), torch.empty(n, dtype=torch.int32, device="cuda"))

    code.decode(mu, max_iter=6, early_stop=True)
    small, whole = outputs(32), outputs(600)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        pkg.ldpc_decode(code.handle, mu[:32], opts, *small)
        pkg.ldpc_decode(code.handle, mu, opts, None, *whole[1:])
    for msg, algo in ((pkg.MSG_F16, pkg.ALGO_SP), (pkg.MSG_I8, pkg.ALGO_MS)):
        code.decode(mu, max_iter=6, msg=msg, algo=algo)
    graph.replay()
    torch.cuda.synchronize()
    for a, b in zip(small, other.decode(mu[:32], max_iter=6)):
        assert torch.equal(a, b)
    for a, b in zip(whole[1:], other.decode(mu, max_iter=6)[1:]):
        assert torch.equal(a, b)


@pytest.mark.parametrize("post,frames,gamma", [(True, 8000, None), (False, 9001, None), (False, 9001, 512)])
def test_several_launches_for_one_call(pkg, post, frames, gamma):
    """A decode (in a batch, and streamed) and a simulation whose iteration limit allows more work than one
    launch may hold the chip for give what the same frames give with a lower limit, which none of them reaches."""
    code = pkg.QCCode(synth.qc_shifts(4, 24, 765, seed=2), 765)
    if gamma is None:
        mu = code.channel(3.5, 7, 0, frames)
        one, n1 = launches(pkg, lambda: code.decode(mu, max_iter=60, early_stop=True, want_post=post))
        many, n = launches(pkg, lambda: code.decode(mu, max_iter=2000, early_stop=True, want_post=post))
        part = 2 ** 39 // (73440 * 2000)  # frames of a launch; whole packages in a batch
        assert int(one[2].max()) < 60 and n1 == 2 and n == 2 * -(-frames // (part // 32 * 32 if post else part))
        for a, b in zip(one, many):
            assert a is b is None or torch.equal(a, b)
    else:
        def sim(max_iter):
            r, n = launches(pkg, lambda: code.ber_sim(3.5, seed=7, max_frames=frames, target_frame_errors=1 << 40,
                                                      gamma=gamma, max_iter=max_iter, early_stop=1))
            r.pop("seconds")
            return r, n

        one, many = sim(60), sim(2000)
        assert one[1] == 2 and many[1] == 6 and one[0] == many[0] and one[0]["frame_errors"] == 0


# J, L, p, zero blocks: the kernels of 8, 16, 24 (full and with empty slots) and 32 edges a row, more than
# four block rows; ragged last rows and variables; none fits a cluster
WIDTHS = [(3, 8, 619, 1), (4, 13, 271, 0), (4, 24, 137, 0), (4, 20, 179, 3), (3, 32, 149, 4), (5, 12, 233, 4),
          (8, 32, 61, 20)]


@pytest.mark.parametrize("J,L,p,zero", WIDTHS)
@pytest.mark.parametrize("algo,msg", [(0, 0), (0, 1), (1, 2), (2, 0), (2, 1)])
def test_more_packages_than_slots(pkg, J, L, p, zero, algo, msg):
    """Slots that take package after package: outputs of a large batch, bit for bit those of its parts, which
    go by launches with a fixed count (posteriors of the last iteration) and with early stop through the flow
    with a slot for every package."""
    code, _, _ = setup(pkg, J, L, p, zero, 9)
    W = 32 << msg
    slot = 128 * code.E + 128 * code.N * (1 if algo == 1 else W // 32) + 4 * code.N * (W + W // 32)
    packages = 96 * 2 ** 20 // slot + 9
    frames = packages * W - 5
    mu = torch.from_numpy(synth.gaussian_llrs(6 * W, code.N, seed=L, ebn0_db=2.0, rate=0.5)).cuda()
    mu = mu.repeat(-(-frames // (6 * W)), 1)[:frames].contiguous()
    mu[::5] *= 1.25
    mu[0, : code.N // 2] = 0.0  # erased inputs: infinite transforms
    prm = torch.from_numpy(np.random.default_rng(1).uniform(0.05, 0.9, (7, J * L, 2)).astype(np.float32)).cuda()

    def decode(x, early):
        o = pkg.default_opts(max_iter=7, early_stop=early, algo=algo, msg=msg)
        o.noms_params = prm.data_ptr() if algo == 2 else None
        n = x.shape[0]
        out = (torch.empty((n, code.N), device="cuda"), torch.empty((n, code.N), dtype=torch.uint8, device="cuda"),
               torch.empty(n, dtype=torch.int32, device="cuda"), torch.empty(n, dtype=torch.int32, device="cuda"))
        return launches(pkg, lambda: pkg.ldpc_decode(code.handle, x, o, *out) or out)

    for early in (0, 1):
        whole, n = decode(mu, early)
        assert n == 2
        for at in (0, (packages // 2) * W, (packages - 4) * W):
            part, n = decode(mu[at:at + 4 * W], early)
            assert n == 2 if early else n > 2
            for a, b in zip(whole, part):
                assert torch.equal(a[at:at + 4 * W], b), (early, at)


@pytest.mark.parametrize("J,L,p", [(4, 13, 251), (4, 14, 247), (4, 16, 203)])  # N: 3, 2 and 0 mod 4
@pytest.mark.parametrize("algo,msg", [(0, 0), (1, 2)])
def test_streaming(pkg, J, L, p, algo, msg):
    """A batch that streams through refilled lanes: decisions, iterations and flags of the batch decode, with
    rows on and off the alignment of wide accesses, from device and pinned host memory, and without decisions."""
    code = pkg.QCCode(synth.qc_shifts(J, L, p, seed=8), p)
    frames = 8209
    o = pkg.default_opts(max_iter=25, early_stop=1, algo=algo, msg=msg)
    mu = code.channel(4.0, 3, 0, frames)
    _, *want = code.decode(mu, max_iter=25, early_stop=True, algo=algo, msg=msg)
    assert 0 < int(want[2].sum()) and int(want[1].min()) < int(want[1].max())
    for device, late in (("cuda", 0), ("cuda", 1), ("cpu", 1)):
        def buffer(shape, dtype):
            n = int(np.prod(shape)) + late
            return torch.empty(n, dtype=dtype, device=device, pin_memory=device == "cpu")[late:].view(shape)

        llr = buffer(mu.shape, torch.float32).copy_(mu)
        hard, iters, ok = buffer(mu.shape, torch.uint8), buffer(frames, torch.int32), buffer(frames, torch.int32)
        for h in (hard, None):
            iters.zero_(), ok.zero_()
            _, n = launches(pkg, lambda: pkg.ldpc_decode(code.handle, llr, o, None, h, iters, ok))
            assert n == 2
            torch.cuda.synchronize()
            assert torch.equal(iters.cuda(), want[1]) and torch.equal(ok.cuda(), want[2])
        assert torch.equal(hard.cuda(), want[0])
