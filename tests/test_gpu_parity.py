"""Parity of the CUDA path (through the C ABI) with the CPU oracle: every
integer plane and the object count bit for bit, every feature within 1e-4
relative or 1e-6 absolute of the FP64 oracle."""
import numpy as np
import pytest

import oracle
import synth
from tests.gpu_util import assert_feats_close, assert_planes_equal, oracle_all, run_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pipe():
    import torch
    import paper_1209_3332_gb300 as P
    from paper_1209_3332_gb300 import build
    build.build()
    torch.cuda.init()
    p = P.Pipe(0)
    yield p
    assert p.status() == P.PIPE_OK
    p.close()


def check(pipe, rgb, **kw):
    g = run_gpu(pipe, rgb)
    r = oracle_all(rgb, **kw)
    assert_planes_equal(g, r)
    assert_feats_close(g["feats"], r["feats"])
    return g, r


def test_cfg0_512(pipe):
    g, r = check(pipe, synth.cfg0())
    assert r["K"] > 20


@pytest.mark.parametrize("W,H,n", [(77, 133, 6), (33, 65, 3), (1, 1, 0), (1, 300, 0), (300, 1, 0),
                                   (1000, 999, 120), (2049, 1025, 300), (31, 32, 1), (64, 64, 2)])
def test_ragged_sizes(pipe, W, H, n):
    rgb = synth.tile(W, H, 7 + W + H, n_nuclei=n, frac_overlap=0.1, frac_cluster=0.2, n_stroma=n // 20)
    check(pipe, rgb)


def test_empty_tile(pipe):
    rgb = synth.tile(700, 500, 3, n_nuclei=0)
    g, r = check(pipe, rgb)
    assert g["K"] == 0


def test_all_foreground_small_tile_has_no_background(pipe):
    rgb = np.zeros((30, 30, 3), np.uint8)  # hem8 = 255 everywhere -> one object, no background
    g, r = check(pipe, rgb)
    assert g["K"] == 1 and (g["edt"] == 2 ** 31 - 1).all()


def test_uniform_random_rgb(pipe):
    rng = np.random.default_rng(0)
    rgb = rng.integers(0, 256, (257, 300, 3)).astype(np.uint8)
    check(pipe, rgb)


def test_dense_chains_and_corridor(pipe):
    rgb = synth.tile(1536, 1280, 99, n_nuclei=1500, frac_chain=0.5, corridor=True)
    check(pipe, rgb)


def test_cfg1_full_4096(pipe):
    g, r = check(pipe, synth.cfg1())
    assert r["K"] > 1000


def test_repeat_is_deterministic(pipe):
    rgb = synth.tile(900, 700, 5, n_nuclei=200, frac_cluster=0.3)
    a = run_gpu(pipe, rgb)
    b = run_gpu(pipe, rgb)
    for k in ("hem8", "R", "labels", "edt"):
        assert np.array_equal(a[k], b[k])
    assert np.array_equal(a["feats"], b["feats"])


def test_all_rgb_triples_through_the_whole_path(pipe):
    # every 24-bit colour once: hem8 must match the oracle exactly everywhere,
    # and the rest of the path must agree on this far-from-natural image too
    v = np.arange(1 << 24, dtype=np.uint32)
    rgb = np.stack([(v >> 16) & 255, (v >> 8) & 255, v & 255], -1).astype(np.uint8).reshape(4096, 4096, 3)
    check(pipe, rgb)


def ring_tile(W=620, H=530):
    """White tile with black annuli: each annulus is a flat dome of the
    hematoxylin plane, so it is foreground and its inside a hole -- holes of
    2 to 230 pixels across, inside one 32x32 labelling block or spanning
    many, nested rings, and rings cut by the tile border (their inside
    touches the border and is no hole)."""
    yy, xx = np.mgrid[:H, :W]
    rgb = np.full((H, W, 3), 255, np.uint8)
    rings = [(40, 40, 2, 4), (31, 95, 5, 3), (100, 63, 9, 4), (160, 160, 14, 5), (300, 120, 30, 4),
             (300, 120, 12, 3), (420, 330, 115, 6), (420, 330, 60, 5), (420, 330, 20, 3), (5, 300, 25, 4),
             (600, 500, 40, 5), (250, 480, 33, 4), (96, 400, 31, 2)]
    for cx, cy, r, t in rings:
        d2 = (xx - cx) ** 2 + (yy - cy) ** 2
        rgb[(d2 >= r * r) & (d2 < (r + t) ** 2)] = 0
    return rgb


def test_holes_of_every_size(pipe):
    rgb = ring_tile()
    g, r = check(pipe, rgb)
    holes = int(r["filled"].sum()) - int(r["fg"].sum())
    assert holes > 20000  # the rings' insides were filled


@pytest.mark.parametrize("W,H,off,pad", [(16, 1, 1, 0), (17, 2, 2, 1), (35, 3, 3, 5), (64, 65, 1, 0), (79, 33, 2, 7),
                                         (130, 67, 3, 0), (193, 129, 1, 2)])
def test_unaligned_buffers(pipe, W, H, off, pad):
    """RGB rows and a hem8 plane that start on no 4-byte boundary, at widths
    around the 16-pixel loads and the 64-pixel work tiles."""
    import torch
    import synth
    rgb = synth.tile(W, H, 31 + W, n_nuclei=max(1, W * H // 400), frac_cluster=0.3)
    dev = torch.device("cuda", 0)
    pitch = 3 * W + pad
    src = torch.zeros(off + H * pitch, dtype=torch.uint8, device=dev)
    view = src[off:].view(H, pitch)[:, :3 * W]
    view.copy_(torch.from_numpy(rgb.reshape(H, 3 * W)).to(dev))
    hem = torch.full((off + H * W,), 7, dtype=torch.uint8, device=dev)[off:].view(H, W)
    lab = torch.empty((H, W), dtype=torch.int32, device=dev)
    edt = torch.empty_like(lab)
    nobj = torch.zeros(1, dtype=torch.int32, device=dev)
    pipe.seg_tile(view.view(H, W, 3) if pad == 0 else view.as_strided((H, W, 3), (pitch, 3, 1)), hem, lab, edt, nobj)
    R = torch.empty((H, W), dtype=torch.uint8, device=dev)
    pipe.debug_plane(0, R)
    torch.cuda.synchronize()
    ref = oracle_all(rgb)
    assert_planes_equal(dict(hem8=hem.cpu().numpy(), R=R.cpu().numpy(), labels=lab.cpu().numpy(), edt=edt.cpu().numpy(),
                             K=int(nobj.item())), ref)


@pytest.mark.parametrize("W", [720, 721, 722, 8, 4])
def test_distances_of_large_objects(W):
    """Objects wider and taller than several 32-row chunks, whose pixels look
    for background far beyond their own group of four columns, up to and past
    the widest search (128), at the image's sides too; widths that are and are
    not a multiple of four."""
    import paper_1209_3332_gb300 as P
    rgb = ring_tile(720, 530)
    yy, xx = np.mgrid[:530, :720]
    for cx, cy, rad in ((150, 330, 140), (700, 120, 90), (0, 0, 50)):
        rgb[(xx - cx) ** 2 + (yy - cy) ** 2 <= rad * rad] = 0
    rgb = np.concatenate([rgb, np.full((530, 2, 3), 255, np.uint8)], 1)[:, :W] if W > 720 else rgb[:, :W]
    p = P.Pipe(0, area_max=10 ** 6)
    g, r = check(p, np.ascontiguousarray(rgb), amax=10 ** 6)
    if W >= 720:
        assert int(r["edt"].max()) > 128 * 128
    p.close()


@pytest.mark.parametrize("bw,bh", [(62, 42), (63, 42), (54, 51), (78, 62), (79, 62), (936, 1), (937, 2), (1, 1200), (1, 1), (300, 15)])
def test_features_at_the_stage_sizes(pipe, bw, bh):
    """Objects whose box plus margin just fits the features' stage (2816
    pixels), is staged in bands of rows (up to 5120), or is not staged: full
    and ragged ones, inside the image and in its corners, under noise."""
    import torch
    rng = np.random.default_rng(bw * 1000 + bh)
    W, H = 2 * bw + 12, 2 * bh + 12
    hem8 = rng.integers(0, 256, (H, W)).astype(np.uint8)
    labels = np.zeros((H, W), np.int32)
    for k, (x, y) in enumerate(((0, 0), (W - bw, 0), (3, H - bh - 3), (W - bw, H - bh))):
        m = rng.random((bh, bw)) < (1.0 if k % 2 else 0.6)
        m[0, 0] = m[-1, -1] = True
        labels[y:y + bh, x:x + bw][m] = k + 1
    ref = oracle.features(hem8, labels, 4)
    dev = torch.device("cuda", 0)
    out = torch.zeros((4, 15), dtype=torch.float32, device=dev)
    pipe.features_tile(torch.from_numpy(hem8).to(dev), torch.from_numpy(labels).to(dev), 4, out)
    torch.cuda.synchronize()
    assert_feats_close(out.cpu().numpy(), ref)


@pytest.mark.parametrize("bw,bh", [(79, 64), (80, 64), (100, 100), (300, 200), (936, 6), (937, 6), (1200, 5), (4, 1500), (1, 4000)])
def test_features_of_objects_beyond_the_stage(pipe, bw, bh):
    """Regions of more than 5120 pixels, whose sums are taken in 64 bits: staged
    in bands of many rows down to one, whose first two rows are the last two of
    the band before, and read from global memory where not even three rows fit;
    at the image's sides, and touching other objects."""
    import torch
    rng = np.random.default_rng(bw * 1000 + bh)
    W, H = 2 * bw + 5, 2 * bh + 1
    hem8 = rng.integers(0, 256, (H, W)).astype(np.uint8)
    labels = np.zeros((H, W), np.int32)
    for k, (x, y) in enumerate(((0, 0), (W - bw, 0), (2, H - bh), (W - bw, H - bh))):
        m = rng.random((bh, bw)) < (1.0 if k % 2 else 0.6)
        m[0, 0] = m[-1, -1] = True
        labels[y:y + bh, x:x + bw][m] = k + 1
    ref = oracle.features(hem8, labels, 4)
    dev = torch.device("cuda", 0)
    out = torch.zeros((4, 15), dtype=torch.float32, device=dev)
    pipe.features_tile(torch.from_numpy(hem8).to(dev), torch.from_numpy(labels).to(dev), 4, out)
    torch.cuda.synchronize()
    assert_feats_close(out.cpu().numpy(), ref)
