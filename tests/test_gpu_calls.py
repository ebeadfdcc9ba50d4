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

from paper_1008_2192_gb300 import Cleaner, Server  # noqa: E402


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
