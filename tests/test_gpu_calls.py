"""Sequences of calls on one handle, and the kernels that single options take: each call's result equals that of a
handle of its own or of the CPU oracle."""

from __future__ import annotations

import numpy as np
import pytest

import oracle
import synth
from gpu_util import dev, gpu_clean, host, params_of

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1008_2192_gb300 import Cleaner, Server, poisson_into  # noqa: E402


# calls of one pixel count, tile count, number of words, cells and zeroed bytes: single frames that differ in their
# strips, and pairs of frames whose maps end 1 KiB apart after rounding
SAME_SUMS = [([(4096, 2560)], [(2560, 4096)]), ([(1536, 6144)], [(6144, 1536)]), ([(2304, 4608)], [(4608, 2304)]),
             ([(124, 73), (117, 96)], [(116, 91), (128, 76)]), ([(120, 86), (110, 71)], [(121, 70), (115, 84)])]


@pytest.mark.parametrize("a,b", SAME_SUMS, ids=[f"{a}-{b}".replace(" ", "") for a, b in SAME_SUMS])
def test_graphs_of_calls_with_equal_sums(a, b):
    """A replayed graph is the one captured for the call's own sizes: calls whose totals agree, one after the
    other and back on one handle, equal the launched ones."""
    plain = Cleaner(niter=4, pipeline="queue")
    graphs = Cleaner(niter=4, pipeline="queue", use_graphs=True)
    scenes = [[dev(synth.frame(w, h, seed=81 + j, index=i)) for i, (w, h) in enumerate(s)] for j, s in enumerate((a, b))]
    want = [plain.clean_batch(s) for s in scenes]
    plain.sync()
    big = torch.zeros((4096 if a[0][0] > 1000 else 300, 4096 if a[0][0] > 1000 else 300), device="cuda")
    graphs.clean(big)  # the workspace then serves all the others, at one address
    for j in (0, 1, 0, 1):
        outs, masks = graphs.clean_batch(scenes[j])
        graphs.sync()
        for o, m, wo, wm in zip(outs, masks, *want[j]):
            assert torch.equal(m, wm) and torch.equal(o, wo), j
    assert all(int(m.sum()) > 0 for _, ms in want for m in ms)


def test_server_of_transposed_frames():
    """Single-frame waves replay graphs: a frame and its transpose, which have the same totals, alternate."""
    imgs = [dev(synth.frame(w, h, seed=83)) for w, h in [(4096, 2560), (2560, 4096)]]
    plain = Cleaner(gain=7.0, readnoise=5.0, niter=4, pipeline="queue")
    want = [plain.clean(x) for x in imgs]
    plain.sync()
    srv = Server(niter=4, max_inflight=1)  # one context for all waves
    try:
        for i in (0, 1, 0, 1):
            o, m = torch.empty_like(imgs[i]), torch.empty(imgs[i].shape, dtype=torch.uint8, device="cuda")
            srv.submit(imgs[i], o, m, i, 7.0, 5.0)
            done = []
            for _ in range(200):
                done += srv.poll(block_ms=100)
                if done:
                    break
            assert [d[0] for d in done] == [i]
            assert torch.equal(m, want[i][1]) and torch.equal(o, want[i][0]), i
    finally:
        srv.close()


@pytest.mark.parametrize("w,h", [(800, 800), (768, 616), (1216, 670), (1217, 700)])
def test_separate_launches_by_rounds_of_tiles(w, h):
    """Without fusion, tile_shape 0 takes 64x32 tiles or, where only those of 64x28 fit one round of resident blocks
    (the first and third), these: sizes either side of both lines equal the FP32 oracle."""
    img = synth.frame(w, h, seed=85)
    out, mask = gpu_clean(Cleaner(niter=3, pipeline="tile", fusion=False), img)
    r32 = oracle.clean(img, params_of({}), 3, precision="f32")
    assert np.array_equal(mask, r32.mask) and np.array_equal(out, r32.clean)


@pytest.mark.parametrize("autotune", [False, True], ids=["shapes", "pipelines-too"])
def test_autotuned_shape_is_the_fastest(autotune):
    """tile_shape -1 tries the row kernels beside the detection shapes, none of which is within a factor of two of
    them here, and the trial of the tile pipeline against the queue pipeline runs what the call then takes. The work
    counters tell the kernels apart: the row kernels decide the objlim tests by counting, the others by a 7x7 median each."""
    for w, h in ((800, 800), (2048, 1100)):
        img = synth.frame(w, h, seed=87)
        want = Cleaner(niter=4, pipeline="tile")
        o, m = gpu_clean(want, img)
        c = Cleaner(niter=4, tile_shape=-1, pipeline="auto" if autotune else "tile", autotune=autotune)
        for _ in range(2):
            out, mask = gpu_clean(c, img)
            assert np.array_equal(mask, m) and np.array_equal(out, o)
            assert c.last_work() == want.last_work() and c.tuned_config()[2] == "tile"
            assert c.last_launches() == want.last_launches()


@pytest.mark.parametrize("kw", [dict(fusion=False), dict(fuse2=True), dict(tile_shape=1), dict(tile_shape=99), dict(tile_shape=-1)],
                         ids=["two-launch", "two-iterations", "shape-1", "past-the-last", "tuned-shape"])
def test_autotune_with_tile_options(kw):
    """The tile pipeline that the autotuner tries is the one the options ask for: results of the first (tuning) and
    later calls equal the FP32 oracle."""
    img = synth.frame(500, 331, seed=88)
    r32 = oracle.clean(img, params_of({}), 4, precision="f32")
    c = Cleaner(niter=4, autotune=True, **kw)
    for _ in range(2):
        out, mask = gpu_clean(c, img)
        assert np.array_equal(mask, r32.mask) and np.array_equal(out, r32.clean)


@pytest.mark.parametrize("given", [False, True])
def test_given_mask_does_not_take_the_tuned_row_kernels(given):
    """A handle tuned to the row kernels by a call without a previous mask keeps to the detection kernels where one is
    given, and the other way round."""
    img = synth.frame(300, 200, seed=89)
    M = np.zeros(img.shape, np.uint8)
    M[::7, ::5] = 1
    c = Cleaner(niter=1, tile_shape=-1, pipeline="tile")
    for k in (0, 1, 0, 1):
        mp = M if bool(k) != given else None
        r = oracle.iterate(img, M if mp is not None else np.zeros_like(M), params_of({}), precision="f32")
        gJ, gM, _ = c.iterate(dev(img), dev(mp) if mp is not None else None)
        c.sync()
        assert np.array_equal(host(gM), r.Mk) and np.array_equal(host(gJ), r.Ik), k


@pytest.mark.parametrize("niter", [2, 4])
def test_fused_64x32_tiles_and_graphs_of_shapes(niter):
    """The fused 64x32 detection kernel (an index past the last) and the capture of detection kernels in a graph,
    both launched and replayed, on a frame of several tiles with remainders and on a batch."""
    img = synth.frame(333, 251, seed=90)
    r32 = oracle.clean(img, params_of({}), niter, precision="f32")
    for shape in (99, 1, 5):
        for graphs in (False, True):
            c = Cleaner(niter=niter, tile_shape=shape, use_graphs=graphs, pipeline="tile")
            for _ in range(2):
                out, mask = gpu_clean(c, img)
                assert np.array_equal(mask, r32.mask) and np.array_equal(out, r32.clean), (shape, graphs)
            outs, masks = c.clean_batch([dev(img), dev(img[:97].copy())])
            c.sync()
            r2 = oracle.clean(img[:97].copy(), params_of({}), niter, precision="f32")
            assert np.array_equal(host(masks[0]), r32.mask) and np.array_equal(host(outs[0]), r32.clean)
            assert np.array_equal(host(masks[1]), r2.mask) and np.array_equal(host(outs[1]), r2.clean)


@pytest.mark.parametrize("graphs", [False, True])
def test_autotune_finds_the_tile_pipeline_above_10_mpix(graphs):
    """On a frame of noise with flags everywhere the tile pipeline takes little more than half the queue pipeline's
    time; the tuner tries it up to 2^25 pixels, and the result is the same."""
    rng = np.random.default_rng(91)
    x = dev((rng.standard_normal((3300, 3300)) * 50 + 200).astype(np.float32))
    q = Cleaner(niter=2, sigclip=2.5, pipeline="queue")
    wo, wm = q.clean(x)
    q.sync()
    c = Cleaner(niter=2, sigclip=2.5, autotune=True, use_graphs=graphs)
    for _ in range(2):
        o, m = c.clean(x)
        c.sync()
        assert torch.equal(m, wm) and torch.equal(o, wo)
    assert c.tuned_config()[2] == "tile"


CHAIN_SIZES = [(137, 137), (400, 300), (401, 299), (800, 800), (801, 799), (1200, 1000), (1201, 999)]


@pytest.mark.parametrize("niter", [1, 2, 4])
def test_chained_calls_without_a_wait(niter):
    """One stream and one handle, nothing waited for in between: a clean of the output of the one before, POISSON
    into the input of the next clean, and an input that a kernel overwrites between two calls, with the frame size, gain
    and buffers changing from call to call. Each result equals that of calls waited for one by one."""
    rng = np.random.default_rng(93)
    calls = []
    for w, h in CHAIN_SIZES:
        a, b = (synth.frame(w, h, seed=94, index=i) for i in range(2))
        mean = np.full((h, w), 24.3, np.float32)
        calls.append(dict(a=dev(a), b=dev(b), mean=dev(mean), g=[float(np.float32(rng.uniform(2, 7))) for _ in range(3)]))

    def go(c, wait):
        outs = []
        step = c.sync if wait else (lambda: None)
        for rep in range(3):
            for k in calls:
                x = k.setdefault("x", torch.empty_like(k["a"]))
                bufs = [torch.empty_like(x) for _ in range(5)]
                masks = [torch.empty(x.shape, dtype=torch.uint8, device="cuda") for _ in range(5)]

                def clean(src, i, g):
                    c.clean_batch_into([src], [bufs[i]], [masks[i]], [g], [5.0])
                    step()

                x.copy_(k["a"])
                clean(x, 0, k["g"][0])
                x.copy_(k["b"])
                clean(x, 1, k["g"][1])
                clean(bufs[1], 2, k["g"][2])
                poisson_into(k["mean"], x, 95 + rep)
                step()
                clean(x, 3, k["g"][0])
                x.add_(k["a"])
                clean(x, 4, k["g"][1])
                outs += bufs + masks
        c.sync()
        return outs

    want = go(Cleaner(niter=niter), True)
    for _ in range(3):
        got = go(Cleaner(niter=niter), False)
        assert len(got) == len(want) and all(torch.equal(p, q) for p, q in zip(got, want))


def test_chained_batches_without_a_wait():
    """Batches of changing sizes and numbers of frames, the input of each being the output of the one before."""
    sizes = [[(137, 137), (200, 100)], [(801, 799)], [(401, 299), (64, 64), (400, 300)], [(1201, 999), (97, 61)]]
    frames = [[dev(synth.frame(w, h, seed=96, index=i)) for i, (w, h) in enumerate(s)] for s in sizes]

    def go(c, wait):
        outs = []
        for f in frames * 3:
            for _ in range(2):
                f, masks = c.clean_batch(f, [6.5 - len(f)] * len(f), [4.0 + len(f)] * len(f))
                if wait:
                    c.sync()
                outs += f + masks
        c.sync()
        return outs

    want = go(Cleaner(niter=4), True)
    for _ in range(3):
        got = go(Cleaner(niter=4), False)
        assert all(torch.equal(p, q) for p, q in zip(got, want))


@pytest.mark.parametrize("w,h", [(137, 90), (150, 331), (1153, 781)])
@pytest.mark.parametrize("kw", [dict(objlim=1e-29), dict(objlim=1e-35), dict(objlim=450.0), dict(objlim=450.0, objlim_form=1),
                                dict(sigclip=1e-3, objlim=1e-38), dict(amp=1e33), dict(amp=1e36), dict(amp=1e38)],
                         ids=lambda k: "-".join(f"{a}{b:g}" for a, b in k.items()))
def test_objlim_beyond_counting(w, h, kw):
    """The row kernels' objlim test where a count of the window decides at scales near float's range, and where it
    cannot decide and the steps are taken value by value (S'/objlim near 0.01; scales out of range): masks, images and
    counters equal the FP32 oracle's, on tiles of 14 and 30 rows, in one round and in more."""
    kw = dict(kw)
    img = synth.frame(w, h, seed=97, ncr=max(1, int(3 * w * h * synth.CR_DENSITY)))
    amp = kw.pop("amp", None)
    if amp:
        rng = np.random.default_rng(98)
        hit = rng.random(img.shape) < 0.01
        img[hit] = (rng.uniform(-1.0, 1.0, int(hit.sum())) * amp).astype(np.float32)
    c = Cleaner(niter=3, pipeline="tile", **kw)
    out, mask = gpu_clean(c, img)
    r32 = oracle.clean(img, params_of(kw), 3, precision="f32")
    assert np.array_equal(mask, r32.mask) and np.array_equal(out, r32.clean)
    assert c.last_counts() == list(zip(r32.n_new, r32.n_none_left))


def test_tuning_leaves_fixed_grids():
    """Kernels whose grid follows no occupancy are reported with that grid's blocks per SM, tuned or not: the row forms
    below 2^26 pixels, and the growth of iteration 1."""
    img = synth.frame(900, 700, seed=99)
    plain, tuned = (Cleaner(niter=4, pipeline="queue", autotune=t) for t in (False, True))
    (o, m), (o2, m2) = gpu_clean(plain, img), gpu_clean(tuned, img)
    assert np.array_equal(m, m2) and np.array_equal(o, o2)
    a, b = plain.tuned_config()[0], tuned.tuned_config()[0]
    names = list(a)
    rows = [names[i] for i in (1, 4, 11, 18, 19, 20)]  # need, tests (three forms), d2, grow_first
    segs = [names[i] for i in (16, 17)]
    assert all(a[k] == b[k] == 64 for k in rows) and all(a[k] == b[k] == 8 for k in segs), (a, b)


def test_chained_calls_on_two_streams():
    """One handle, calls alternating between two streams with no wait on the host: each call's upload and kernels, launched
    ahead of time, start after the call before on the other stream, whose workspace and descriptors they take over."""
    sizes = [(137, 137), (801, 799), (401, 299), (1201, 999)]
    imgs = [dev(synth.frame(w, h, seed=100, index=i)) for i, (w, h) in enumerate(sizes)]
    c = Cleaner(niter=4)
    want = []
    for x in imgs:
        want.append(c.clean(x))
        c.sync()
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    torch.cuda.synchronize()
    outs = [(torch.empty_like(imgs[i % 4]), torch.empty(imgs[i % 4].shape, dtype=torch.uint8, device="cuda")) for i in range(60)]
    torch.cuda.synchronize()
    for i, (o, m) in enumerate(outs):
        c.clean_into(imgs[i % 4], o, m, stream=streams[(i // 3 + i) % 2])
    torch.cuda.synchronize()
    for i, (o, m) in enumerate(outs):
        assert torch.equal(m, want[i % 4][1]) and torch.equal(o, want[i % 4][0]), i
