"""The renderer's alternative paths against each other and against the oracles:
depth ranking (crowded and equal depths, windows of any size), binning by
difference arrays and by noted places, the compositor's CTA form, warp form and
teams, LiDAR boxes, the no-allocation entry.  Orders, lists and counts are
exact; images of two paths are equal bit for bit, since every path blends the
same splats in the same order with the same arithmetic."""
import dataclasses

import numpy as np
import pytest

from gpu_helpers import ensure_built, gpu_render
from oracle import oracle
from paper_2604_25459_gb300 import gsbatch, synth
from test_gpu_lidar import _oracle_scan, _sensors

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _build():
    ensure_built()


def _check_lists(w, tile, W, H):
    """Counts and depth-ordered lists of env 0, from the GPU's own records."""
    out = gpu_render(w, tile=tile, debug=True, keep_scene=True)
    rec = out["scene"].debug_records(0, w.background.n + w.links.n)
    vis = np.nonzero(rec["visible"])[0]
    counts, lists = out["scene"].debug_tiles(0, (-(-W // tile[0])) * (-(-H // tile[1])))
    out["scene"].close()
    oc, ol = oracle.bin_records(rec["u"][vis], rec["v"][vis], rec["hx"][vis], rec["hy"][vis],
                                rec["z"][vis].view(np.uint32), vis.astype(np.uint32), W, H, *tile)
    np.testing.assert_array_equal(counts.astype(np.int64), oc)
    np.testing.assert_array_equal(lists, ol)
    return len(vis)


@pytest.mark.parametrize("depths", ["equal", "half_equal", "steps"])
@pytest.mark.parametrize("n", [1, 33, 767, 2049, 9_000, 70_000])
def test_ranking_of_crowded_depths(n, depths):
    """Keys with one depth, a crowd among spread ones, and few distinct depths:
    ranges that a counting sort cannot split, windows above one block's."""
    w = synth.make_c0(n=n)
    mean = w.background.mean.copy()
    if depths == "equal":
        mean[:, 2] = 0.0
    elif depths == "half_equal":
        mean[::2, 2] = 0.25
    else:
        mean[:, 2] = np.round(mean[:, 2] * 2.0) / 2.0
    w = dataclasses.replace(w, background=dataclasses.replace(w.background, mean=mean))
    vis = _check_lists(w, (16, 16), 128, 96)
    assert vis > 0 or n == 1


@pytest.mark.parametrize("n", [0, 32, 1024, 1025, 2048, 2049])
def test_ranking_of_small_scenes(n):
    """Scenes ranked whole by one block, up to 2048 slots, and the first above."""
    w = synth.make_c0(n=max(n, 1))
    if n == 0:  # nothing visible
        w = dataclasses.replace(w, background=dataclasses.replace(w.background, mean=w.background.mean - [0, 0, 9]))
    assert (_check_lists(w, (16, 16), 128, 96) > 0) == (n > 0)


@pytest.mark.parametrize("width,height,tile", [(255, 240, (16, 16)), (257, 241, (16, 16)), (641, 479, (16, 16)),
                                               (129, 121, (8, 8)), (333, 251, (32, 8)), (520, 33, (16, 8))])
def test_binning_of_long_spans(width, height, tile):
    """Grids around 256 tiles, some splats spanning the whole image."""
    w = synth.make_c1(n_envs=1, width=width, height=height, f=0.8 * width, n_bg=12_000, per_link=100)
    ls = w.background.log_scale.copy()
    ls[::97] += 3.0
    w = dataclasses.replace(w, background=dataclasses.replace(w.background, log_scale=ls))
    assert _check_lists(w, tile, width, height) > 1000


@pytest.mark.parametrize("width,height", [(7, 5), (17, 33), (130, 94), (373, 375), (374, 375)])
def test_images_do_not_depend_on_the_compositor_form(width, height):
    """Square tiles take the warp form up to 140,000 pixels (few items: teams),
    other tiles the CTA form."""
    w = synth.make_c1(n_envs=2, width=width, height=height, f=0.8 * width, n_bg=150_000, per_link=1000)
    scene = gsbatch.scene_from_workload(w)
    ref = gpu_render(w, tile=(32, 16), scene=scene)
    for tile in ((16, 16), (8, 8), (16, 8), (32, 8)):
        out = gpu_render(w, tile=tile, scene=scene)
        for k in ("rgb", "depth", "alpha"):
            np.testing.assert_array_equal(out[k], ref[k], err_msg=f"{tile} {k}")
    scene.close()


def test_images_do_not_depend_on_the_batch():
    """Alone a view's items go to teams of four warps; among 480 views its long
    buckets go to single warps."""
    w = synth.make_c1(n_envs=480, width=128, height=96, f=100.0, n_bg=30_000, per_link=200)
    scene = gsbatch.scene_from_workload(w)
    out = gpu_render(w, scene=scene)
    for e in (0, 479):
        alone = gpu_render(w, scene=scene, envs=[e])
        for k in ("rgb", "depth", "alpha"):
            np.testing.assert_array_equal(out[k][e], alone[k][0], err_msg=f"env {e} {k}")
    scene.close()


def test_mixed_resolutions_take_the_form_of_their_size():
    """render_v, largest image first: each env as alone."""
    import torch

    sizes = [(640, 240), (64, 48), (374, 375), (33, 21), (200, 120)]
    ws = [synth.make_c1(n_envs=1, width=a, height=b, f=0.8 * a, n_bg=20_000, per_link=200) for a, b in sizes]
    envs = gsbatch.make_envs(np.concatenate([w.cams for w in ws]),
                             link_ranges=np.tile([0, ws[0].n_links], (len(ws), 1)),
                             pose_offsets=np.zeros(len(ws)))
    scene = gsbatch.scene_from_workload(ws[0])
    poses = torch.from_numpy(ws[0].link_poses).cuda()
    npx = sum(a * b for a, b in sizes)
    rgb, depth, alpha = (torch.full((npx * k,), -1.0, device="cuda") for k in (3, 1, 1))
    scene.render_v(envs, poses, rgb, depth, alpha)
    torch.cuda.synchronize()
    for e, (a, b) in enumerate(sizes):
        cams = ws[e].cams
        r = [t.cpu().numpy() for t in scene.render(poses, cams)]
        o = int(envs["pixel_offset"][e])
        np.testing.assert_array_equal(rgb[3 * o:3 * (o + a * b)].cpu().numpy().reshape(b, a, 3), r[0][0])
        np.testing.assert_array_equal(depth[o:o + a * b].cpu().numpy().reshape(b, a), r[1][0])
        np.testing.assert_array_equal(alpha[o:o + a * b].cpu().numpy().reshape(b, a), r[2][0])
    scene.close()


@pytest.mark.parametrize("rows,cols", [(5, 40), (16, 64), (33, 47)])
def test_lidar_boxes_hold_near_and_steep_gaussians(rows, cols):
    """Gaussians around a sensor, up to half a metre wide, at elevations up to
    1.45: a ray that a box misses would lose a whole Gaussian.  Tolerances as
    for the other scans (threshold flips only)."""
    import torch

    w = synth.make_c1(n_envs=1, width=64, height=48, f=50.0, n_bg=600, per_link=20)
    rng = np.random.default_rng(rows)
    g = w.background
    d = rng.normal(size=(g.n, 3))
    d /= np.linalg.norm(d, axis=1, keepdims=True)
    sens = _sensors(1, rows=rows, cols=cols)
    sens["elev_min"], sens["elev_max"] = -1.45, 1.45
    mean = -sens["t_ws"][0] + d * rng.uniform(1.0, 6.0, (g.n, 1))
    ls = np.log(rng.uniform(0.02, 0.5, (g.n, 3)))
    w = dataclasses.replace(w, background=dataclasses.replace(g, mean=mean.astype(np.float32),
                                                              log_scale=ls.astype(np.float32)))
    scene = gsbatch.scene_from_workload(w)
    rng_m, hit = (t.cpu().numpy()[0] for t in scene.render_lidar(torch.from_numpy(w.link_poses).cuda(), sens))
    scene.close()
    ref = _oracle_scan(w, 0, sens[0])
    dh = np.abs(hit - ref["hit"])
    both = (ref["hit"] >= 0.5) & (hit >= 0.5)
    rel = np.abs(rng_m - ref["range"])[both] / ref["range"][both]
    assert both.sum() > 50
    assert np.quantile(dh, 0.99) <= 2e-3 and dh.max() <= 0.05
    assert np.quantile(rel, 0.99) <= 1e-4 and rel.max() <= 1e-2


@pytest.mark.parametrize("n,width,height,E", [(300, 40, 24, 1), (16_384, 128, 96, 3), (17_001, 129, 97, 2),
                                              (1500, 64, 48, 24), (700, 40, 24, 130),
                                              (30_000, 400, 360, 1)])
def test_noalloc_is_the_batched_render(n, width, height, E):
    import torch

    w = synth.make_c1(n_envs=E, width=width, height=height, f=0.8 * width, n_bg=n, per_link=40)
    scene = gsbatch.scene_from_workload(w)
    poses = torch.from_numpy(w.link_poses).cuda()
    ref = scene.render(poses, w.cams)
    out = [torch.empty_like(t) for t in ref]
    scene.render_noalloc(poses, w.cams, *out)
    torch.cuda.synchronize()
    for a, b in zip(out, ref):
        assert torch.equal(a, b)
    scene.close()
