"""The flow decoder's host part on a machine without a GPU (fake_device.py): what its launches are given,
what it allocates and when, and what a caller is told when a device-side wait gives up."""
import pytest

from fake_device import FakeDevice


@pytest.fixture(scope="module")
def built(tmp_path_factory):
    return FakeDevice(tmp_path_factory.mktemp("fake"))


@pytest.fixture
def dev(built):
    built.reset()
    return built


def phases_while_one_block_waits(slots, blocks, cycle):
    """Phases that can be open or done from the one on whose tile a block is held up, all other blocks being
    done with theirs at once: tile t of all belongs to block t mod blocks, a slot goes through the phases
    of `cycle` (tiles each), and stops at the first that has a tile of the held-up block."""
    opened = tiles = 0
    at = [0] * slots
    running = list(range(slots))
    while running:
        still = []
        for s in running:
            n = cycle[at[s] % len(cycle)]
            first = -tiles % blocks  # the phase's first tile of block 0
            tiles += n
            opened += 1
            at[s] += 1
            if first >= n:
                still.append(s)
        running = still
    return opened


# J, L, p: the shortest codes (a tile or a few a phase), short ones on many slots, longer ones on few
@pytest.mark.parametrize("J,L,p", [(1, 2, 1), (2, 6, 20), (3, 6, 64), (4, 12, 31), (4, 12, 211), (4, 24, 100),
                                   (4, 24, 765), (8, 32, 61)])
@pytest.mark.parametrize("algo,msg", [(0, 0), (0, 1), (1, 2)])
def test_phase_log_holds_what_a_late_block_has_not_read(dev, J, L, p, algo, msg):
    """A log entry is not overwritten while a block may still have to read it, whatever the number of slots
    and however long one block is held up."""
    code = dev.code(J, L, p)
    N = L * p
    opts = dict(algo=algo, msg=msg, max_iter=20, early_stop=1)
    seen = 0
    for frames in (33, 300, 10000, 70000):
        if frames * N <= 1 << 24:
            assert dev.decode(code, N, frames, post=True, **opts) == 0
    for slots in (64, 1024, 16384, 32768):
        assert dev.sim(code, 5 * slots, slots, **opts) == 0
    for f in dev.flows():
        fewest = min(f["nsyn"], f["cn_tiles"], f["vn_tiles"], -(-N // 256))
        for cycle in ([f["nsyn"], f["cn_tiles"], f["vn_tiles"]], [1], [fewest]):
            assert phases_while_one_block_waits(f["W"], f["blocks"], cycle) < f["log_len"], f
        seen = max(seen, f["W"])
    if msg and N < 1000:
        assert seen == 256  # the most slots there are
    dev.c.ldpc_code_destroy(code)


def test_phase_log_of_the_allocation_free_decode(dev):
    code = dev.code(2, 4, 20)
    assert dev.decode(code, 80, 256 * 32, noalloc=True, max_iter=9, early_stop=1) == 0
    (f,) = dev.flows()
    assert f["W"] == 256 and f["log_len"] > phases_while_one_block_waits(f["W"], f["blocks"], [1])
    dev.c.ldpc_code_destroy(code)


@pytest.mark.parametrize("length", [64, 2048, 65536])
def test_log_entry_read_in_two_parts(dev, length):
    """A block that finds one word of an entry and the other of the entry before it in that place looks again,
    whichever came first; words past the wrap of the sequence number too."""
    here, past, ahead = 0, 1, 2
    for n in (0, 5, length - 1, length, 12345, (1 << 22) - 1, 1 << 22, (1 << 22) + 77, (1 << 24) + 1, (1 << 32) - 3):
        before, after = (n - length) % (1 << 32), (n + length) % (1 << 32)
        assert dev.c.fake_entry_is(n, n, n) == here
        assert dev.c.fake_entry_is(before, before, n) == ahead
        assert dev.c.fake_entry_is(before, n, n) == ahead and dev.c.fake_entry_is(n, before, n) == ahead
        assert dev.c.fake_entry_is(after, after, n) == past and dev.c.fake_entry_is(n, after, n) == past
        assert dev.c.fake_entry_is(after, n, n) == ahead  # read again: n has been overwritten


@pytest.mark.parametrize("J,L,p", [(4, 24, 211), (4, 24, 765), (8, 32, 200)])
def test_buffers_are_kept_while_batches_do_not_grow(dev, J, L, p):
    """Once a batch has been decoded, no decode of as many frames or fewer and no simulation on as many slots
    frees a buffer (one that a captured graph of the first call holds) or needs memory that the first did not."""
    code = dev.code(J, L, p)
    N, frames = L * p, 700
    assert dev.decode(code, N, frames, max_iter=30) == 0
    assert len(dev.flows()) == 1
    had = dev.calls("cudaMalloc")
    for algo, msg in ((0, 0), (0, 1), (1, 2), (2, 0), (2, 1)):
        for post in (False, True):
            for early in (0, 1):
                for n in (frames, 701 - 128, 33):
                    assert dev.decode(code, N, n, post=post, algo=algo, msg=msg, early_stop=early, max_iter=30) == 0
    flows = dev.flows()
    assert len(flows) > 40 and dev.calls("cudaFree") == 0
    # (the calls that go by launches have a workspace of their own: eight buffers)
    assert dev.calls("cudaMalloc") <= had + 8
    assert dev.sim(code, 2000, 700, early_stop=1) == 0  # and the simulation its state: one
    assert dev.calls("cudaMalloc") <= had + 9 and dev.calls("cudaFree") == 0
    dev.c.ldpc_code_destroy(code)


def form(dev):
    """how the last decode ran"""
    last = dev.names()[-1]
    return "chip" if "chip_kernel" in last else "flow" if "tile_kernel" in last else "launches"


# a batch decoded first, then one of no more frames that by itself takes another form
OTHERS = [((4, 24, 765), dict(gamma=2048, early_stop=1), dict(gamma=32), "flow", "launches"),
          ((4, 24, 211), dict(gamma=96), dict(gamma=33, early_stop=1), "launches", "flow"),
          ((4, 12, 200), dict(gamma=512, algo=1, msg=2), dict(gamma=128, algo=1, msg=2), "chip", "launches")]


@pytest.mark.parametrize("shape,first,then,before,alone", OTHERS)
def test_smaller_batch_without_new_memory(dev, shape, first, then, before, alone):
    """Under capture, and where no memory is left, a batch of no more frames than an earlier one is decoded
    by the form whose workspace is there."""
    N = shape[1] * shape[2]
    for how in ("alone", "capture", "no memory"):
        code = dev.code(*shape)
        if how != "alone":
            assert dev.decode(code, N, max_iter=20, **first) == 0 and form(dev) == before
        dev.c.fake_capturing(how == "capture")
        if how == "no memory":
            dev.c.fake_budget(0)
        st = dev.decode(code, N, max_iter=20, **then)
        dev.c.fake_capturing(0)
        dev.c.fake_budget(-1)
        assert st == 0 and form(dev) == (alone if how == "alone" else before), how
        dev.c.ldpc_code_destroy(code)


OK, ETIMEOUT = 0, 4


def test_a_wait_given_up_is_told_by_the_next_call(dev):
    """A device-side wait that gave up is told by the next call on the object, whichever way that runs, and
    by no other and no later one."""
    code, other = dev.code(4, 24, 211), dev.code(4, 24, 211)
    N = 24 * 211
    big, few = dict(gamma=4096, max_iter=30), dict(gamma=32, max_iter=30)
    for then in (lambda: dev.decode(code, N, **big), lambda: dev.decode(code, N, **few),
                 lambda: dev.sim(code, 500, 64, early_stop=1), lambda: dev.sim(code, 500, 64, target=100),
                 lambda: dev.decode(code, N, gamma=8192, early_stop=1, max_iter=30)):
        assert then() == OK  # each of them runs by itself
        dev.c.fake_give_up(1)
        assert dev.decode(code, N, **big) == OK and form(dev) == "flow"
        n = len(dev.names())
        assert dev.decode(other, N, **big) == OK
        assert then() == ETIMEOUT
        assert then() == OK and len(dev.names()) > n
    dev.c.fake_give_up(2)  # a call that waits tells of its own
    assert dev.sim(code, 500, 64, early_stop=1) == ETIMEOUT
    assert dev.decode(code, N, **big) == OK
    dev.c.ldpc_code_destroy(code)
    dev.c.ldpc_code_destroy(other)


def test_a_wait_given_up_with_pageable_outputs(dev):
    """Outputs in pageable host memory are there when the call returns: it tells of its own time-out."""
    code = dev.code(4, 24, 211)
    big = dict(gamma=4096, max_iter=30)
    dev.c.fake_give_up(3)
    assert dev.decode(code, 24 * 211, host_out=True, **big) == ETIMEOUT
    assert dev.decode(code, 24 * 211, host_out=True, **big) == OK
    assert dev.decode(code, 24 * 211, **big) == OK
    dev.c.ldpc_code_destroy(code)


def test_a_wait_given_up_in_the_fixed_scratch(dev):
    """The allocation-free decode's time-out is told by the next such call on the same code, not on another."""
    codes = [dev.code(4, 24, 150) for _ in range(2)]
    N = 24 * 150
    call = dict(gamma=32, max_iter=30, early_stop=1, noalloc=True)
    for code in codes:
        assert dev.decode(code, N, **call) == OK and form(dev) == "flow"
        dev.c.fake_give_up(1)
        assert dev.decode(code, N, **call) == OK
    assert dev.decode(codes[0], N, gamma=32, max_iter=30) == OK  # ldpc_decode has its own
    for code in codes:
        assert dev.decode(code, N, **call) == ETIMEOUT
        assert dev.decode(code, N, **call) == OK
    for code in codes:
        dev.c.ldpc_code_destroy(code)


def test_a_second_device(dev):
    """What a kernel may have and how many of its blocks fit are asked for on each device: the first call of
    every form on a second device, after the same calls on the first."""
    for d in (0, 1):
        dev.c.fake_device(d)
        code, long = dev.code(3, 6, 64), dev.code(4, 24, 211)
        assert dev.decode(code, 384, 32, max_iter=30) == 0 and form(dev) == "chip"
        assert dev.decode(code, 384, 8192, max_iter=30) == 0 and form(dev) == "launches"
        assert dev.decode(long, 24 * 211, 4096, max_iter=30) == 0 and form(dev) == "flow"
        assert dev.c.fake_refused() == 0
        dev.c.ldpc_code_destroy(code)
        dev.c.ldpc_code_destroy(long)


@pytest.mark.parametrize("algo,msg", [(0, 0), (0, 1), (1, 2)])
def test_tuner_times_the_form_that_the_slots_decide(dev, algo, msg):
    """The slot count's candidates are timed as the runs that it decides are run: by launches on that many
    slots, where the flow decoder keeps the same few packages in work at every candidate."""
    import ctypes

    code = dev.code(4, 24, 40)
    o = dev.opts(max_iter=5, early_stop=1, algo=algo, msg=msg)
    picked = ctypes.c_int32()
    assert dev.c.ldpc_tune_slots(code, 2.0, 1, ctypes.byref(o), ctypes.byref(picked), None, None) == 0
    assert not dev.flows() and sum("sim_check_kernel" in n for n in dev.names()) >= 10
    assert dev.sim(code, 500, 64, algo=algo, msg=msg, early_stop=1) == 0 and len(dev.flows()) == 1
    dev.c.ldpc_code_destroy(code)


@pytest.mark.parametrize("J,L,p,max_iter,frames", [(4, 24, 765, 30, 1 << 20), (4, 24, 4200, 100, 1 << 20),
                                                   (3, 6, 64, 30, 3 << 20), (4, 24, 765, 30, 131072),
                                                   (4, 8, 300000, 50, 4000)])
def test_simulation_launches_are_bounded_in_work(dev, J, L, p, max_iter, frames):
    """A launch holds every SM until it ends: edges x frames x iterations of one stay below 2^39, about a
    second, whatever the code and the iterations, unless that would leave lanes without a frame."""
    code = dev.code(J, L, p)
    assert dev.sim(code, frames, 1024, max_iter=max_iter, early_stop=1) == 0
    flows = dev.flows()
    assert sum(f["frames"] for f in flows) == frames
    for f in flows:
        assert f["frames"] * J * L * p * max_iter <= 1 << 39 or f["frames"] <= 32 * f["W"]
    if frames == 131072:
        assert len(flows) == 1
    dev.c.ldpc_code_destroy(code)


def test_decode_launches_are_bounded_in_work(dev):
    code = dev.code(4, 24, 765)
    for kw, n in ((dict(gamma=4001, max_iter=100000), 16), (dict(gamma=2048, max_iter=30), 1)):
        at = len(dev.flows())
        assert dev.decode(code, 18360, post=True, **kw) == 0
        flows = dev.flows()[at:]
        assert len(flows) > 15 if n > 1 else len(flows) == 1
        assert sum(f["frames"] for f in flows) == kw["gamma"]
        for f in flows:
            assert f["frames"] * 73440 * kw["max_iter"] <= 1 << 39 or f["frames"] <= 32 * f["W"]
    dev.c.ldpc_code_destroy(code)
