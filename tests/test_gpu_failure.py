"""Failure detection without a GPU fault: every device-side spin wait of the
work queues (the reconstruction's, and the growth's under Canny and red blood
cells) is bounded by the pipe's cycle budget.  With a budget of a few hundred
cycles the idle workers give up, the kernel returns, the status word reports
PIPE_ETIMEOUT, and the context stays usable: a pipe with the normal budget
then matches the oracle on the same input.  The status word keeps the first
error until it is read."""
import numpy as np
import pytest

import synth
from tests.gpu_util import assert_planes_equal, oracle_all, run_gpu

pytestmark = pytest.mark.gpu


def test_wait_budget_exhaustion_is_reported_and_recoverable():
    import paper_1209_3332_gb300 as P
    from paper_1209_3332_gb300 import build
    build.build()
    rgb = synth.tile(1024, 1024, 61, n_nuclei=200, frac_cluster=0.2)
    tight = P.Pipe(0, wait_budget_cycles=300)
    run_gpu(tight, rgb, want_planes=False)
    assert tight.status() == P.PIPE_ETIMEOUT
    assert tight.status() == P.PIPE_OK  # reading the status clears it
    tight.close()
    normal = P.Pipe(0)
    g = run_gpu(normal, rgb)
    assert_planes_equal(g, oracle_all(rgb))
    assert normal.status() == P.PIPE_OK
    normal.close()


def spiral(n, pitch=12.0):
    """A plane whose edges form two spiral arms, strong near the centre only, so
    that the hysteresis follows them through the work tiles one after the other."""
    yy, xx = np.mgrid[0:n, 0:n].astype(np.float64)
    dx, dy = xx - n / 2 + 0.3, yy - n / 2 + 0.2
    r, turn = np.hypot(dx, dy), np.arctan2(dy, dx) / (2 * np.pi)
    amp = np.where(r < 3 * pitch, 60, 20)
    return np.where((r / pitch - turn) % 1.0 < 0.5, 100 + amp, 100).astype(np.uint8)


def snake_rgb(n):
    """Red rows joined at alternate ends, one strong pixel at the start."""
    rgb = np.full((n, n, 3), 200, np.uint8)
    red = np.zeros((n, n), bool)
    red[::4] = True
    for i, y in enumerate(range(0, n - 4, 4)):
        red[y:y + 4, n - 1 if i % 2 == 0 else 0] = True
    rgb[red] = (200, 140, 140)
    rgb[0, 0] = (250, 100, 100)
    return rgb


# Wait budgets in cycles that the idle workers of a large call exceed many times
# and a call of one work tile does not: the growth of a long path takes milliseconds,
# and its idle warps wait for one tile in the small call; the reconstruction of
# one tile has one worker, which waits for nobody.
WAIT = dict(canny=400000, rbc=400000, plain=300, batch=300, overflow=1 << 32)


class Calls:
    """The calls under test on one pipe; each returns the planes it wrote."""

    def __init__(self, pipe):
        import torch
        self.pipe, self.dev = pipe, torch.device("cuda", 0)
        self.keep = []  # nothing waits between the calls

    def put(self, a):
        import torch
        t = torch.from_numpy(np.ascontiguousarray(a)).to(self.dev)
        self.keep.append(t)
        return t

    def canny(self, img):
        import torch
        I = self.put(img)
        E = torch.full_like(I, 7)
        self.pipe.canny(I, E)
        return E

    def rbc(self, rgb):
        import torch
        src = self.put(rgb)
        out = torch.full(rgb.shape[:2], 7, dtype=torch.uint8, device=self.dev)
        self.pipe.rbc(src, out)
        return out

    def batch(self, rgbs, cap):
        import torch
        tiles = []
        for a in rgbs:
            H, W = a.shape[:2]
            tiles.append(dict(rgb=self.put(a), hem8=torch.empty((H, W), dtype=torch.uint8, device=self.dev),
                              labels=torch.full((H, W), -1, dtype=torch.int32, device=self.dev),
                              edt=torch.empty((H, W), dtype=torch.int32, device=self.dev),
                              n_objects=torch.zeros(1, dtype=torch.int32, device=self.dev),
                              feats=torch.zeros((cap, 15), dtype=torch.float32, device=self.dev)))
        self.keep.append(tiles)
        self.pipe.seg_features_batch(tiles)
        return tiles

    def plain(self, rgb):
        import torch
        H, W = rgb.shape[:2]
        out = (torch.empty((H, W), dtype=torch.uint8, device=self.dev), torch.full((H, W), -1, dtype=torch.int32, device=self.dev),
               torch.empty((H, W), dtype=torch.int32, device=self.dev), torch.zeros(1, dtype=torch.int32, device=self.dev))
        self.keep.append(out)
        self.pipe.seg_tile(self.put(rgb), *out)
        return out


BLANK = np.full((64, 64, 3), 200, np.uint8)
NUCLEI = dict(n_nuclei=200, frac_cluster=0.2)


@pytest.mark.parametrize("late,then", [("canny", "rbc"), ("rbc", "canny"), ("canny", "canny"), ("plain", "plain"),
                                       ("batch", "batch"), ("overflow", "batch")])
def test_status_outlives_the_calls_behind(late, then):
    """The status word holds the first error since it was last read, whatever
    runs between the call that failed and the read."""
    import paper_1209_3332_gb300 as P
    pipe = P.Pipe(0, autotune=0, wait_budget_cycles=WAIT[late])
    c = Calls(pipe)
    tile = synth.tile(1024, 1024, 61, **NUCLEI)
    small = dict(canny=lambda: c.canny(BLANK[..., 0]), rbc=lambda: c.rbc(BLANK), plain=lambda: c.plain(BLANK),
                 batch=lambda: c.batch([BLANK], 8))[then]
    small()
    assert pipe.status() == P.PIPE_OK
    dict(canny=lambda: c.canny(spiral(1024)), rbc=lambda: c.rbc(snake_rgb(1024)), plain=lambda: c.plain(tile),
         batch=lambda: c.batch([tile], 400), overflow=lambda: c.batch([tile], 3))[late]()
    small()
    assert pipe.status() == (P.PIPE_EOVERFLOW if late == "overflow" else P.PIPE_ETIMEOUT)
    assert pipe.status() == P.PIPE_OK
    small()
    assert pipe.status() == P.PIPE_OK
    pipe.close()


@pytest.mark.parametrize("form", ["teams", "warps", "canny", "rbc"])
def test_wait_budget_exhaustion_of_every_queue(form):
    """Both kernels of the reconstruction -- teams of warps take a launch of
    less than two work tiles per resident warp, single warps the larger ones --
    and the growth under Canny and red blood cells."""
    import oracle
    import paper_1209_3332_gb300 as P
    tight, normal = P.Pipe(0, autotune=0, wait_budget_cycles=300), P.Pipe(0, autotune=0)
    tile = synth.tile(512, 512, 62, n_nuclei=60, frac_cluster=0.2)  # 64 work tiles
    if form in ("teams", "warps"):
        Calls(normal).batch([tile], 200)
        warps = normal.autotune_info()["recon_workers"]
        n = -(-2 * warps // 64) - (form == "teams")  # 2 * warps work tiles, or just fewer
        Calls(tight).batch([tile] * n, 200)
    elif form == "canny":
        Calls(tight).canny(spiral(768))
    else:
        Calls(tight).rbc(snake_rgb(768))
    assert tight.status() == P.PIPE_ETIMEOUT
    assert tight.status() == P.PIPE_OK
    tight.close()
    if form == "canny":
        assert np.array_equal(Calls(normal).canny(spiral(768)).cpu().numpy(), oracle.canny(spiral(768)))
    elif form == "rbc":
        assert np.array_equal(Calls(normal).rbc(snake_rgb(768)).cpu().numpy(), oracle.rbc(snake_rgb(768)))
    else:
        want = oracle_all(tile)
        for t in Calls(normal).batch([tile] * n, 200):
            assert np.array_equal(t["labels"].cpu().numpy(), want["labels"])
    assert normal.status() == P.PIPE_OK
    normal.close()
