"""Edges of the renderer's binning, ranking and host paths that ordinary scenes
do not reach."""
import ctypes
import dataclasses
import os
import subprocess

import numpy as np
import pytest

from gpu_helpers import ensure_built, gpu_render
from oracle import oracle
from paper_2604_25459_gb300 import build as cuda_build
from paper_2604_25459_gb300 import gsbatch, synth
from test_gpu_lidar import _check_scan, _oracle_rays, _ray_sensors, _sensors

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _build():
    ensure_built()


def _check_lists(scene, w, e, tile, W, H):
    """Counts and depth-ordered lists of env e of the last debug render, from the GPU's own records."""
    rec = scene.debug_records(e, w.background.n + w.links.n)
    vis = np.nonzero(rec["visible"])[0]
    counts, lists = scene.debug_tiles(e, (-(-W // tile[0])) * (-(-H // tile[1])))
    oc, ol = oracle.bin_records(rec["u"][vis], rec["v"][vis], rec["hx"][vis], rec["hy"][vis],
                                rec["z"][vis].view(np.uint32), vis.astype(np.uint32), W, H, *tile)
    np.testing.assert_array_equal(counts.astype(np.int64), oc)
    np.testing.assert_array_equal(lists, ol)
    return rec, vis


@pytest.mark.parametrize("tile,n_envs,words", [((16, 16), 192, 64), ((32, 8), 192, 64), ((16, 16), 1, 16)])
def test_blocks_full_of_long_spans(tile, n_envs, words):
    """A robot whose Gaussians cover a third of the image and more, in blocks of the
    scatter of `words` visibility words (2048 slots in large batches, 512 for one
    view): a block lists more spans of over 64 tiles than its list holds, so it
    drains the list several times before its last round.  Keys with subtile
    masks (square tiles) and without."""
    W = H = 256
    w = synth.make_c1(n_envs=n_envs, width=W, height=H, f=200.0, n_bg=100_000, per_link=300)
    links = dataclasses.replace(w.links, log_scale=(w.links.log_scale + np.float32(2.0)).astype(np.float32))
    w = dataclasses.replace(w, links=links)
    out = gpu_render(w, tile=tile, debug=True, keep_scene=True)
    most = 0
    for e in {0, n_envs // 2, n_envs - 1}:
        rec, vis = _check_lists(out["scene"], w, e, tile, W, H)
        r = rec["range"][vis].astype(np.int64)
        tiles = (r[:, 1] // tile[0] - r[:, 0] // tile[0] + 1) * (r[:, 3] // tile[1] - r[:, 2] // tile[1] + 1)
        far = vis[(tiles > 64) & (vis >= w.background.n)]  # links keep their storage order
        block = (far - w.background.n + (w.background.n + 31) // 32 * 32) // (32 * words)
        most = max(most, int(np.bincount(block).max()))
    out["scene"].close()
    assert most > (1024 if words == 64 else 384)


def _native(name, folder):
    """tests/<name>.cu, linked with the library; its function <name>."""
    so = str(folder / f"{name}.so")
    here = os.path.dirname(os.path.abspath(__file__))
    libdir = os.path.dirname(cuda_build.LIB)
    subprocess.run([cuda_build.nvcc(), *cuda_build.ARCH, "-O1", "-std=c++17", "-Xcompiler", "-fPIC",
                    "--expt-relaxed-constexpr", "-I", cuda_build.INCLUDE, "-I", cuda_build.CSRC, "-shared", "-cudart",
                    "static", "-o", so, os.path.join(here, f"{name}.cu"), "-L", libdir, "-l:libgsbatch.so",
                    "-Xlinker", "-rpath", "-Xlinker", libdir], check=True)
    f = getattr(ctypes.CDLL(so), name)
    f.restype = ctypes.c_int
    return f


@pytest.fixture(scope="module")
def corrupt_bucket(tmp_path_factory):
    native = _native("corrupt_bucket", tmp_path_factory.mktemp("native"))

    def run(form, n, bad):
        alpha, status = np.full((16, 16), -1.0, np.float32), ctypes.c_uint32(0)
        assert native(form, n, bad, alpha.ctypes.data_as(ctypes.c_void_p), ctypes.byref(status)) == 0
        return alpha, status.value

    return run


@pytest.mark.parametrize("form", [0, 1, 2])
@pytest.mark.parametrize("n", [40, 600, 1490])
def test_rank_beyond_the_ranked_records_is_left_out(corrupt_bucket, form, n):
    """A key that names no ranked record (a corrupted bucket): its place in the
    order is not read and the other splats are blended; the CTA form, which
    accounts for every key of a bucket, also sets the status word."""
    alpha, status = corrupt_bucket(form, n, 0)
    assert status == 0 and np.all(np.abs(alpha - (1.0 - (1.0 - 0.0045) ** n)) < 5e-3)
    again, status = corrupt_bucket(form, n, 1)
    assert status == (4 if form == 0 else 0)
    np.testing.assert_array_equal(again, alpha)


@pytest.mark.parametrize("wave", [0, 2])
def test_tile_counts_of_mixed_resolutions_are_the_named_envs(wave):
    """render_v orders a batch by resolution; the counts it leaves are looked up by
    the caller's index, and an env outside the last wave is refused."""
    import torch

    sizes = [(320, 240), (64, 48), (130, 94), (96, 200), (33, 21)]
    ws = [synth.make_c1(n_envs=1, width=a, height=b, f=0.8 * a, n_bg=20_000, per_link=200) for a, b in sizes]
    envs = gsbatch.make_envs(np.concatenate([w.cams for w in ws]),
                             link_ranges=np.tile([0, ws[0].n_links], (len(ws), 1)),
                             pose_offsets=np.zeros(len(ws)))
    scene = gsbatch.scene_from_workload(ws[0])
    poses = torch.from_numpy(ws[0].link_poses).cuda()
    tiles = [(-(-a // 16)) * (-(-b // 16)) for a, b in sizes]
    alone = []
    for w, t in zip(ws, tiles):
        scene.render(poses, w.cams)
        alone.append(scene.debug_tiles(0, t, with_lists=False)[0])
    scene.set_wave(wave)
    npx = sum(a * b for a, b in sizes)
    scene.render_v(envs, poses, torch.empty(npx * 3, device="cuda"), torch.empty(npx, device="cuda"))
    last = range(len(sizes)) if wave == 0 else range(0, 1)  # the largest image is the last wave of two
    for e in range(len(sizes)):
        if e in last:
            np.testing.assert_array_equal(scene.debug_tiles(e, tiles[e], with_lists=False)[0], alone[e])
        else:
            with pytest.raises(gsbatch.GsError):
                scene.debug_tiles(e, tiles[e], with_lists=False)
    scene.close()


def test_tile_counts_outlive_a_plan():
    """A plan measures its batch with eager passes in its own scratch; the
    scene's counts of its last render stay readable, also when the plan is gone."""
    import torch

    w = synth.make_c1(n_envs=1, width=130, height=94, f=100.0, n_bg=20_000, per_link=200)
    other = synth.make_c1(n_envs=3, width=200, height=120, f=160.0, n_bg=20_000, per_link=200)
    scene = gsbatch.scene_from_workload(w)
    scene.render(torch.from_numpy(w.link_poses).cuda(), w.cams)
    before = scene.debug_tiles(0, 54, with_lists=False)[0]
    envs = gsbatch.make_envs(other.cams, link_ranges=np.tile([0, w.n_links], (3, 1)),
                             pose_offsets=np.arange(3) * w.n_links)
    npx = 3 * 200 * 120
    plan = scene.plan(envs)
    plan.launch(torch.from_numpy(other.link_poses).cuda(), torch.empty(npx * 3, device="cuda"),
                torch.empty(npx, device="cuda"))
    torch.cuda.synchronize()
    np.testing.assert_array_equal(scene.debug_tiles(0, 54, with_lists=False)[0], before)
    plan.close()
    np.testing.assert_array_equal(scene.debug_tiles(0, 54, with_lists=False)[0], before)
    scene.close()


@pytest.mark.parametrize("width,height,tile,quad", [(200, 120, (16, 16), 1), (640, 480, (16, 16), 0),
                                                    (200, 120, (32, 8), 0)])
def test_plan_info_names_the_form_that_runs(width, height, tile, quad):
    """An untuned plan takes the warp form by resolution, on square tiles."""
    import torch

    w = synth.make_c1(n_envs=2, width=width, height=height, f=0.8 * width, n_bg=20_000, per_link=200)
    scene = gsbatch.scene_from_workload(w)
    scene.set_tile(*tile)
    envs = gsbatch.make_envs(w.cams, link_ranges=np.tile([0, w.n_links], (2, 1)), pose_offsets=np.arange(2) * w.n_links)
    plan = scene.plan(envs, autotune=False)
    npx = 2 * width * height
    plan.launch(torch.from_numpy(w.link_poses).cuda(), torch.empty(npx * 3, device="cuda"),
                torch.empty(npx, device="cuda"))
    torch.cuda.synchronize()
    assert plan.info()["quad"] == quad
    plan.close()
    scene.close()


@pytest.mark.parametrize("kind,width,height,mib", [("render", 64, 48, 24), ("render", 320, 240, 40), ("lidar", 128, 32, 24),
                                                   ("rays", 64, 64, 24)])
def test_scratch_stays_within_the_budget(kind, width, height, mib):
    """Several waves of 24 envs of 22,000 slots under a small budget: the scratch
    that the scene then holds, every table of it, is within the budget."""
    import torch

    n = 24
    w = synth.make_c1(n_envs=n, width=width, height=height, f=0.8 * width, n_bg=20_000, per_link=100)
    scene = gsbatch.scene_from_workload(w)
    scene.set_budget(mib << 20)
    poses = torch.from_numpy(w.link_poses).cuda()
    if kind == "render":
        scene.render(poses, w.cams)
    else:
        sens = _sensors(n, rows=height, cols=width)
        if kind == "lidar":
            scene.render_lidar(poses, sens)
        else:
            scene.render_rays(poses, sens, torch.from_numpy(synth.rosette_rays(n, 500)).cuda())
    torch.cuda.synchronize()
    st = scene.stats()
    assert st["waves"] > 1
    assert st["scratch_bytes"] <= mib << 20
    scene.close()


@pytest.mark.parametrize("n,width,height", [(20_000, 64, 48), (15_000, 1000, 30), (70_000, 33, 21)])
def test_one_environment_fits_the_budget_it_always_fitted(n, width, height):
    """64 bytes a slot and 12 a tile within 60 % of the budget: what one env
    needed before records were ranked is still enough for it."""
    import torch

    w = synth.make_c0(n=n, width=width, height=height, f=0.8 * width)
    slots, tiles = (n + 31) // 32 * 32, (-(-width // 16)) * (-(-height // 16))
    scene = gsbatch.scene_from_workload(w)
    scene.set_budget(int((slots * 64 + slots // 32 * 4 + tiles * 12 + 600) / 0.6))
    scene.render(None, w.cams)
    torch.cuda.synchronize()
    scene.close()


def test_server_scratch_stays_within_its_budget():
    """Requests of low resolution, whose scratch is records and ranking and few
    keys: the device memory that a slot takes is within what admission allowed it,
    up to the rounding of 17 buffers to 2 MiB."""
    import torch

    E, budget = 96, 2 << 30
    w = synth.make_c1(n_envs=E, width=64, height=48, f=50.0, n_bg=600_000, per_link=200)
    scene = gsbatch.scene_from_workload(w)
    for rounds, limit in ((1, 256 << 20), (3, budget)):  # the first server loads the kernels
        sv = gsbatch.Server(budget_bytes=limit, max_inflight=1, max_batch_envs=E)
        sid = sv.add_scene(scene)
        ids = [sv.add_env(sid, w.cams[e:e + 1], 0, w.n_links) for e in range(E)]
        sv.start()
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        for _ in range(rounds):
            for e in ids:
                sv.submit(e, w.link_poses[e])
            sv.drain(300.0)
        used = free - torch.cuda.mem_get_info()[0]
        most = sv.stats()["max_batch"]
        sv.close()
    scene.close()
    assert 8 <= most < E
    assert used <= budget + (17 * 2 << 20)


def test_threads_may_render_grids_of_different_sizes():
    """Scenes of their own on threads and streams of their own, on grids whose
    histograms need shared memory beyond the default, of three sizes: no launch
    may depend on what another thread's last one needed."""
    import threading

    import torch

    errors = []

    def work(width, height, tile, seed):
        try:
            w = synth.make_c0(seed=seed, n=300, width=width, height=height, f=0.8 * width)
            scene = gsbatch.scene_from_workload(w)
            scene.set_tile(*tile)
            stream = torch.cuda.Stream()
            out = [torch.empty((1, height, width) + s, device="cuda") for s in ((3,), (), ())]
            torch.cuda.synchronize()
            for _ in range(400):
                scene.render(None, w.cams, *out, stream=stream)
            stream.synchronize()
            scene.close()
        except Exception as e:
            errors.append(e)

    jobs = [(1920, 1080, (16, 16), 0), (2560, 1440, (16, 16), 1), (1024, 1024, (8, 8), 2)]
    threads = [threading.Thread(target=work, args=j) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors[0]


@pytest.mark.parametrize("width,height,tile", [(16384, 64, (8, 8)), (64, 16384, (8, 8)), (2048, 2048, (16, 16))])
def test_largest_grids(width, height, tile):
    """16384 tiles, the most an image may have, square and in the longest rows."""
    w = synth.make_c0(n=3000, width=width, height=height, f=60.0)
    out = gpu_render(w, tile=tile, debug=True, keep_scene=True)
    _, vis = _check_lists(out["scene"], w, 0, tile, width, height)
    out["scene"].close()
    assert len(vis) > 1000


@pytest.mark.parametrize("depths", ["spread", "equal", "half_equal"])
def test_ranking_of_a_window_that_the_sample_missed(depths):
    """Of 20,000 slots the ranking samples every third; with all of those culled
    (too faint) it has no splitters, so 13,333 records share one depth range: a
    window far above what one block sorts, cut by radix selection."""
    w = synth.make_c0(n=20_000)
    g = w.background
    mean = g.mean.copy()
    if depths == "equal":
        mean[:, 2] = 0.0
    elif depths == "half_equal":
        mean[::2, 2] = 0.25
    g = dataclasses.replace(g, mean=mean)
    scene = gsbatch.scene_from_workload(dataclasses.replace(w, background=g))
    order = scene.storage_order()  # by the means alone
    scene.close()
    opacity = np.maximum(g.opacity, np.float32(0.1))
    opacity[order[::3]] = 0.001
    w = dataclasses.replace(w, background=dataclasses.replace(g, opacity=opacity))
    out = gpu_render(w, debug=True, keep_scene=True)
    assert np.array_equal(out["scene"].storage_order(), order)
    _, vis = _check_lists(out["scene"], w, 0, (16, 16), 128, 96)
    out["scene"].close()
    assert len(vis) > 10_000 and not np.isin(vis, order[::3]).any()


def _shell(n, half_az, half_el, seed):
    """n faint Gaussians of 2 cm, 2 to 6 m around the origin, within +-half_az and +-half_el."""
    rng = np.random.default_rng([seed, 91])
    w = synth.make_c0(seed=seed, n=n)
    az, el, r = rng.uniform(-half_az, half_az, n), rng.uniform(-half_el, half_el, n), rng.uniform(2.0, 6.0, n)
    mean = np.stack([r * np.cos(el) * np.cos(az), r * np.cos(el) * np.sin(az), r * np.sin(el)], 1)
    return dataclasses.replace(w, background=dataclasses.replace(
        w.background, mean=mean.astype(np.float32), log_scale=np.full((n, 3), np.log(0.02), np.float32),
        opacity=rng.uniform(0.02, 0.2, n).astype(np.float32)))


def _at(sens, n, pos_seed=7):
    s = np.repeat(sens[:1], n)
    s["t_ws"] = -np.random.default_rng(pos_seed).uniform(-0.05, 0.05, (n, 3))
    return s


def test_scans_of_many_gaussians_in_short_buckets():
    """300,000 ranked Gaussians and buckets of some 2,000 keys: with 24 sensors a
    warp orders a bucket by runs of a histogram over the ranks; alone, a scan's
    buckets go to teams and their bitmaps.  The same bits either way."""
    import torch

    w = _shell(300_000, np.pi, 0.5, 1)
    scene = gsbatch.scene_from_workload(w)
    sens = _at(_sensors(1, rows=64, cols=1024), 24)
    rng, hit = scene.render_lidar(None, sens)
    torch.cuda.synchronize()
    scene.sync_status()
    assert 0.2 < float(hit.mean()) < 0.95
    for e in (0, 23):
        r1, h1 = scene.render_lidar(None, sens[e:e + 1])
        assert torch.equal(hit[e], h1[0]) and torch.equal(rng[e], r1[0])
    scene.close()


def test_rays_through_many_gaussians_in_short_buckets():
    """The same for rays, 72 sensors and one, and a part of them against the oracle."""
    import torch

    n_env, n_rays = 72, 16_000
    w = _shell(150_000, 0.65, 0.65, 2)
    w = dataclasses.replace(w, link_poses=np.zeros((n_env, 0, 7), np.float32))
    scene = gsbatch.scene_from_workload(w)
    sens = _at(_ray_sensors(1, rows=256, cols=256), n_env)
    dirs = synth.rosette_rays(n_env, n_rays, seed=5)
    rng, hit = scene.render_rays(None, sens, torch.from_numpy(dirs).cuda())
    torch.cuda.synchronize()
    scene.sync_status()
    for e in (0, n_env - 1):
        r1, h1 = scene.render_rays(None, sens[e:e + 1], torch.from_numpy(dirs[e:e + 1].copy()).cuda())
        assert torch.equal(hit[e], h1[0]) and torch.equal(rng[e], r1[0])
    scene.close()
    some = np.arange(0, n_rays, 160)
    _check_scan(rng[0, some].cpu().numpy(), hit[0, some].cpu().numpy(),
                _oracle_rays(w, 0, sens[0], dirs[0][some].copy()), "rays of the shell")


@pytest.fixture(scope="module")
def rank_ranges(tmp_path_factory):
    return _native("rank_ranges", tmp_path_factory.mktemp("native"))


@pytest.mark.parametrize("n", [5000, 8192, 20_000, 120_000, 300_000])
@pytest.mark.parametrize("seen", [1.0, 0.5])
def test_depth_ranges_are_balanced(rank_ranges, n, seen):
    """The sample is kept from all over the storage order, whatever share of it is
    seen: no range of an env whose depths follow the order holds more than three
    times the average (a range spans two to thirty samples, evenly spaced but for what is not seen)."""
    rng = np.random.default_rng([n, int(10 * seen)])
    bits = rng.random(n) < seen if seen < 1.0 else np.ones(n, bool)
    mask = np.packbits(np.pad(bits, (0, -n % 32)), bitorder="little").view(np.uint32)
    per = np.zeros(4096, np.uint32)
    bins = rank_ranges(n, mask.ctypes.data_as(ctypes.c_void_p), per.ctypes.data_as(ctypes.c_void_p), len(per))
    assert bins > 0 and per[:bins].sum() == bits.sum()
    assert per[:bins].max() <= 3.0 * bits.sum() / bins


@pytest.mark.parametrize("scene,n,width,height,envs", [("cube", 30_000, 300, 250, 8), ("cube", 30_000, 64, 48, 3),
                                                       ("cube", 120_000, 40, 30, 2), ("room", 5_000, 200, 150, 4),
                                                       ("room", 60_000, 200, 150, 4), ("cube", 60_000, 64, 48, 110)])
def test_images_do_not_depend_on_the_buckets_form(scene, n, width, height, envs):
    """Even and uneven scenes with short and long buckets, few and many tiles: the
    buckets decide between the compositor's forms, and the images are those of
    32x16 tiles, which know one form only."""
    import torch

    if scene == "cube":
        w = synth.make_c0(n=n)
        cams, poses = np.repeat(synth.make_c0(n=1, width=width, height=height, f=0.86 * width).cams, envs), None
    else:
        w = synth.make_c1(n_envs=envs, width=width, height=height, f=0.8 * width, n_bg=n, per_link=n // 100)
        cams, poses = w.cams, torch.from_numpy(w.link_poses).cuda()
    s = gsbatch.scene_from_workload(w)
    out = [t.clone() for t in s.render(poses, cams)]
    s.set_tile(32, 16)
    for a, b in zip(out, s.render(poses, cams)):
        assert torch.equal(a, b)
    s.close()


@pytest.mark.parametrize("n", [31, 1000, 1024, 1025, 2000, 2048, 2049, 3000, 4096, 4097])
@pytest.mark.parametrize("depths", ["equal", "crowd", "far"])
def test_ranking_of_small_scenes_of_crowded_depths(n, depths):
    """Scenes ranked by one block (up to 4096 slots, and the first above) whose depths
    fill one counting range or a few: all equal, a crowd among spread ones, and one
    splat far behind the others."""
    w = synth.make_c0(n=n)
    mean = w.background.mean.copy()
    if depths == "equal":
        mean[:, 2] = 0.0
    elif depths == "crowd":
        mean[: n // 20 + 33, 2] = 0.25
    else:
        mean[0] = [0.0, 0.0, 4000.0]
    w = dataclasses.replace(w, background=dataclasses.replace(w.background, mean=mean))
    out = gpu_render(w, debug=True, keep_scene=True)
    _, vis = _check_lists(out["scene"], w, 0, (16, 16), 128, 96)
    out["scene"].close()
    assert len(vis) > n // 2
