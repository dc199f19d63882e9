"""A pool's work follows the pool's work before it whatever stream that ran on,
also where equal stream handles name different streams (cudaStreamPerThread in
two threads, a destroyed stream's handle) and for what is not a tick: a
camera's admission and release, state reads, the host's wait. The stream of the
earlier work is held back by other work, so that later work that did not wait
would overtake it; the results equal a pool that keeps to one stream."""
import ctypes
import itertools
import queue
import threading

import numpy as np
import pytest

import paper_2110_14934_gb300 as G
from parity import scene_frames, to_dev

pytestmark = pytest.mark.gpu

H, W, M, N = 240, 320, 3, 6
PER_THREAD = 2  # cudaStreamPerThread


class Handle:
    """A stream known by its handle alone."""

    def __init__(self, handle):
        self.cuda_stream = handle


@pytest.fixture(scope="module")
def setup():
    """Frames, and what holds a stream back: some 4 ms of full-HD ticks, on a
    model of their own at each call (four in turn; a test waits for the GPU
    before it makes a fifth)."""
    import torch
    rgb, depth, _ = scene_frames(81, H, W, 1, 44, N)
    frames = [to_dev(r, d) for r, d in zip(rgb, depth)]
    models = [G.GMM(1080, 1920, 3) for _ in range(4)]
    masks = [g.new_mask() for g in models]
    turn = itertools.cycle(zip(models, masks))
    br, bd = (torch.zeros(s, dtype=t, device="cuda") for s, t in (((1080, 1920, 3), torch.uint8), ((1080, 1920), torch.int16)))

    def hold(stream):
        g, m = next(turn)
        for _ in range(100):
            g.apply(br, bd, m, stream=stream)

    torch.cuda.synchronize()
    yield frames, hold
    torch.cuda.synchronize()
    for g in models:
        g.set_stream(torch.cuda.default_stream())
        g.close()


def _run(frames, tick):
    """Masks of every tick and the final state of a pool of one camera."""
    import torch
    p = G.Pool()
    cam = p.admit(H, W, M)
    masks = [torch.zeros((H, G.mask_words_per_row(W)), dtype=torch.int32, device="cuda") for _ in frames]
    torch.cuda.synchronize()
    for t, (r, d) in enumerate(frames):
        p.submit(cam, r, d, masks[t])
        tick(p, t)
    planes = p.planes(cam)  # (follows the ticks by itself)
    torch.cuda.synchronize()
    p.close()
    return [m.cpu().numpy() for m in masks], planes


def _same(a, b):
    assert all(np.array_equal(x, y) for x, y in zip(a[0], b[0]))
    assert np.array_equal(a[1], b[1])


def test_per_thread_streams_of_two_threads(setup):
    """Two threads, which live until the work is done, tick in turn."""
    frames, hold = setup
    jobs, done = [queue.Queue(), queue.Queue()], queue.Queue()

    def worker(i):
        for p in iter(jobs[i].get, None):
            try:
                if i == 0:
                    hold(Handle(PER_THREAD))
                p.tick(stream=Handle(PER_THREAD))
                done.put(None)
            except Exception as e:  # noqa: BLE001 (raised below)
                done.put(e)

    def in_turn(p, t):
        jobs[t % 2].put(p)
        e = done.get(timeout=20)
        if e is not None:
            raise e

    threads = [threading.Thread(target=worker, args=(i,), daemon=True) for i in range(2)]
    for th in threads:
        th.start()
    moved = _run(frames, in_turn)
    for q in jobs:
        q.put(None)
    for th in threads:
        th.join(20)
    _same(moved, _run(frames, lambda p, t: p.tick()))


def test_stream_destroyed_with_a_tick_queued(setup):
    import torch
    frames, hold = setup
    cu = ctypes.CDLL("libcuda.so.1")
    torch.cuda.current_stream()

    def create():
        s = ctypes.c_void_p()
        assert cu.cuStreamCreate(ctypes.byref(s), 1) == 0  # 1: does not wait for the default stream
        return s

    def destroy(s):
        assert cu.cuStreamDestroy_v2(s) == 0

    live = []

    def on_new_streams(p, t):
        s = create()
        if t % 2 == 0:
            hold(Handle(s.value))
        p.tick(stream=Handle(s.value))
        if t < N - 1:
            destroy(s)
        else:
            live.append(s)

    _same(_run(frames, on_new_streams), _run(frames, lambda p, t: p.tick()))
    for s in live:
        destroy(s)


def test_admission_release_reads_and_waits_follow_the_work_before(setup):
    import torch
    frames, hold = setup
    alone = _run(frames, lambda p, t: p.tick())
    side = torch.cuda.Stream()
    p = G.Pool(max_cams=2)
    masks = [torch.zeros((H, G.mask_words_per_row(W)), dtype=torch.int32, device="cuda") for _ in frames]
    torch.cuda.synchronize()
    hold(torch.cuda.default_stream())
    cam = p.admit(H, W, M)  # its clearing of the state waits on the default stream
    for t, (r, d) in enumerate(frames):
        p.submit(cam, r, d, masks[t])
        if t == 3:
            hold(side)
        p.tick(stream=side)
    p.set_stream(torch.cuda.default_stream())
    assert np.array_equal(p.planes(cam), alone[1])
    # a camera in the memory of one whose last tick is still queued elsewhere
    hold(side)
    p.submit(cam, *frames[0], masks[0])
    p.tick(stream=side)
    p.set_stream(torch.cuda.default_stream())
    p.release(cam)
    cam = p.admit(H, W, M)
    for t, (r, d) in enumerate(frames):
        p.submit(cam, r, d, masks[t])
        p.tick()
    assert np.array_equal(p.planes(cam), alone[1])
    assert all(np.array_equal(m.cpu().numpy(), a) for m, a in zip(masks, alone[0]))
    # the host's wait for the pool covers a tick on an earlier stream
    masks[0].fill_(-1)
    torch.cuda.synchronize()
    hold(side)
    p.submit(cam, *frames[0], masks[0])
    p.tick(stream=side)
    p.set_stream(torch.cuda.default_stream())
    p.sync()
    assert side.query()
    p.close()
