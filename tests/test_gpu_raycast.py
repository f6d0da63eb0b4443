"""GPU parity of shm_raycast against the FP64 oracle ray caster (§3.1).

Several results can be correct where a march sample of F lies within rounding of 0: a float32
and a float64 evaluation may then bracket different roots.  The oracle reports, per pixel, the
smallest |F| over its march samples; pixels with margin < 1e-4 R_max are excluded from the exact
comparison of hit object, and must stay a small fraction.  Elsewhere: identical object ids, depth
within 2e-5 relative (bisection + Newton in float32), normals and shading within 2e-3.
"""
import math

import numpy as np
import pytest
import torch

import oracle as O
import shm_inputs as I
from gpu_common import shm, upload_pool

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def S():
    return shm()


def camera_frame(eye, target=(0.0, 0.0, 0.0), up=(0.0, 1.0, 0.0)):
    eye = np.asarray(eye, dtype=np.float64)
    fwd = np.asarray(target) - eye
    fwd /= np.linalg.norm(fwd)
    right = np.cross(fwd, up)
    right /= np.linalg.norm(right)
    upv = np.cross(right, fwd)
    return eye, fwd, right, upv


def _scene(n_obj, seed, choices=(16, 32)):
    counts, offs, mu, amp, width = I.bump_params(n_obj, seed)
    Ns = I.uneven_N(n_obj, seed + 1, choices=choices)
    luts = []
    for o in range(n_obj):
        s = slice(offs[o], offs[o + 1])
        luts.append(O.bake_fd(int(Ns[o]), O.sample_grid_bumps(int(Ns[o]), mu[s], amp[s], width[s]), r0=1.0))
    return luts, Ns


def _run(S, luts, centres, scale, W, H, eye, fov=45.0, prm_kw=None):
    n = len(luts)
    r0 = np.ones(n, np.float32)
    L, stored = upload_pool(S, luts, r0=r0)
    rmax_dev = S.lut_bounds(L).cpu().numpy() * np.asarray(scale, np.float32)
    objs = S.objects_tensor(centres, scale, rmax_dev, np.arange(n))
    eye, fwd, right, up = camera_frame(eye)
    cam = S.make_camera(eye, fwd, right, up, fov, W, H)
    prm = S.make_raycast_params(**(prm_kw or {}))
    out = S.raycast(L, objs, n, cam, prm)
    torch.cuda.synchronize()
    pool = stored.reshape(-1, 4)
    off, Ns = O.make_pool(luts)[1:]
    rmax_o = np.array([O.lut_bound(pool[off[g]:off[g] + 6 * (Ns[g] + 2) ** 2].reshape(6, Ns[g] + 2, Ns[g] + 2, 4),
                                   int(Ns[g]), 1.0) for g in range(n)]) * np.asarray(scale)
    ocam = O.make_camera(eye, fwd, right, up, fov, W, H)
    oprm = O.make_raycast_params(**(prm_kw or {}))
    ref = O.raycast(pool, off, Ns, centres, scale, rmax_o, np.arange(n), ocam, oprm, r0=r0.astype(np.float64))
    return out, ref, rmax_o


def _seam_pixels(ref, centres, eye, fwd, right, up, fov, W, H, eps=1e-4):
    """Pixels whose oracle hit direction lies within eps of a cube-face tie: the two sides may take
    the hit on different faces there, whose interpolants differ by the seam jump."""
    th = math.tan(math.radians(fov) / 2.0)
    yy, xx = np.meshgrid(np.arange(H), np.arange(W), indexing="ij")
    xn = (2 * (xx.ravel() + 0.5) / W - 1) * th * W / H
    yn = (1 - 2 * (yy.ravel() + 0.5) / H) * th
    d = fwd[None, :] + xn[:, None] * right[None, :] + yn[:, None] * up[None, :]
    d /= np.linalg.norm(d, axis=1, keepdims=True)
    ids = ref["obj_id"]
    seam = np.zeros(W * H, bool)
    hit = ids >= 0
    x = eye[None, :] + ref["depth"][hit, None] * d[hit] - np.asarray(centres)[ids[hit]]
    a = np.sort(np.abs(x), axis=1)
    seam[hit] = (a[:, 2] - a[:, 1]) <= eps * a[:, 2]
    return seam


def _compare(out, ref, rmax, W, H, depth_abs=None, seam=None):
    ids = out["obj_id"].cpu().numpy().reshape(-1)
    depth = out["depth"].double().cpu().numpy().reshape(-1)
    nrm = out["normal"].double().cpu().numpy().reshape(-1, 3)
    rgba = out["rgba"].double().cpu().numpy().reshape(-1, 4)
    amb = ref["margin"] < 1e-4 * rmax.max()
    same = ids == ref["obj_id"]
    assert np.all(same[~amb]), np.nonzero(~same & ~amb)[0][:10]
    assert amb.mean() < 0.01
    hit = same & (ids >= 0) & ~amb
    assert hit.sum() > 0.05 * W * H
    rel = np.abs(depth[hit] - ref["depth"][hit]) / ref["depth"][hit]
    if depth_abs is None:
        assert rel.max() <= 2e-5, rel.max()
    else:
        # allowed: 2e-5 relative, or the final bisection bracket of the hit object where a Newton
        # step is rejected (grazing rays) and the two sides stop one halving apart
        allow = np.maximum(2e-5 * ref["depth"][hit], depth_abs[ref["obj_id"][hit]])
        assert np.all(np.abs(depth[hit] - ref["depth"][hit]) <= allow)
    # a hit point moved by dt along the ray turns the normal by at most ~ (a / w^2) dt for bumps of
    # amplitude a <= 0.2 and width w >= 0.05: 100 dt (only where the depth allowance above was used)
    dt = np.abs(depth[hit] - ref["depth"][hit])
    tol = 2e-3 + (100.0 * dt if depth_abs is not None else 0.0)
    smooth = np.ones(hit.sum(), bool) if seam is None else ~seam[hit]
    assert np.all((np.abs(nrm[hit] - ref["normal"][hit]).max(1) <= tol)[smooth])
    assert np.all((np.abs(rgba[hit] - ref["rgba"][hit]).max(1) <= 2 * tol)[smooth])
    miss = same & (ids < 0)
    assert np.all(np.isinf(depth[miss]))
    return hit.sum()


def test_sphere_closed_form(S):
    N = 8
    lut = np.zeros((6, N + 2, N + 2, 4))
    lut[..., 0] = 0.0
    L, _ = upload_pool(S, [lut], r0=np.array([1.0], np.float32))
    objs = S.objects_tensor([[0.3, -0.2, 0.0]], [1.2], [1.5], [0])
    eye, fwd, right, up = camera_frame((0.0, 0.0, 6.0))
    W, H = 64, 48
    cam = S.make_camera(eye, fwd, right, up, 40.0, W, H)
    out = S.raycast(L, objs, 1, cam, S.make_raycast_params())
    depth = out["depth"].double().cpu().numpy()
    th = math.tan(math.radians(20.0))
    c = np.array([0.3, -0.2, 0.0])
    n_hit = 0
    for py in range(H):
        for px in range(W):
            xn = (2 * (px + 0.5) / W - 1) * th * W / H
            yn = (1 - 2 * (py + 0.5) / H) * th
            d = fwd + xn * right + yn * up
            d /= np.linalg.norm(d)
            oc = eye - c
            b = oc @ d
            disc = b * b - (oc @ oc - 1.44)
            if disc < 1e-4:
                continue
            t = -b - math.sqrt(disc)
            assert abs(depth[py, px] - t) <= 2e-5 * t
            n_hit += 1
    assert n_hit > 100


def test_bump_scene_parity(S):
    luts, Ns = _scene(8, 300)
    centres = np.array([[x, y, z] for x in (-1.6, 1.6) for y in (-1.6, 1.6) for z in (-1.6, 1.6)])
    out, ref, rmax = _run(S, luts, centres, np.ones(8), 96, 64, eye=(2.5, 3.0, 9.0))
    _compare(out, ref, rmax, 96, 64)


def test_sampled_pixels_full_size_grid(S):
    """8x8x8 grid of 512 objects at 1920x1080 (the impostor workload): sampled pixels vs the oracle."""
    n = 512
    luts, Ns = _scene(n, 20063 + 2, choices=(16, 32, 64, 128))
    g = (np.arange(8) - 3.5) * 3.0
    centres = np.array([[x, y, z] for x in g for y in g for z in g])
    r0 = np.ones(n, np.float32)
    L, stored = upload_pool(S, luts, r0=r0)
    rmax = S.lut_bounds(L).cpu().numpy()
    objs = S.objects_tensor(centres, np.ones(n), rmax, np.arange(n))
    R_scene = math.sqrt(3) * 10.5 + float(rmax.max())
    dist = R_scene / math.sin(math.radians(22.5))
    eye, fwd, right, up = camera_frame((0.0, 0.0, dist))
    W, H = 1920, 1080
    cam = S.make_camera(eye, fwd, right, up, 45.0, W, H)
    out = S.raycast(L, objs, n, cam, S.make_raycast_params())
    torch.cuda.synchronize()
    rng = np.random.default_rng(5)
    px = rng.integers(0, W, 400).astype(np.int32)
    py = rng.integers(0, H, 400).astype(np.int32)
    pool = stored.reshape(-1, 4)
    off, Nn = O.make_pool(luts)[1:]
    rmax_o = np.array([O.lut_bound(pool[off[k]:off[k] + 6 * (Nn[k] + 2) ** 2].reshape(6, Nn[k] + 2, Nn[k] + 2, 4),
                                   int(Nn[k]), 1.0) for k in range(n)])
    ref = O.raycast(pool, off, Nn, centres, np.ones(n), rmax_o, np.arange(n),
                    O.make_camera(eye, fwd, right, up, 45.0, W, H), O.make_raycast_params(), px=px, py=py,
                    r0=r0.astype(np.float64))
    ids = out["obj_id"].cpu().numpy()[py, px]
    depth = out["depth"].double().cpu().numpy()[py, px]
    amb = ref["margin"] < 1e-4 * rmax_o.max()
    assert np.all((ids == ref["obj_id"])[~amb])
    hit = (ids >= 0) & ~amb
    assert hit.sum() > 50
    assert (np.abs(depth[hit] - ref["depth"][hit]) / ref["depth"][hit]).max() <= 2e-5
    assert S.raycast_query_count(out["_ws"]) > 0


def test_workspace_too_small(S):
    lut = np.zeros((6, 6, 6, 4))
    L, _ = upload_pool(S, [lut], r0=np.array([1.0], np.float32))
    objs = S.objects_tensor([[0, 0, 0]], [1.0], [1.0], [0])
    eye, fwd, right, up = camera_frame((0.0, 0.0, 5.0))
    cam = S.make_camera(eye, fwd, right, up, 40.0, 32, 32)
    with pytest.raises(S.ShmError):
        S.raycast(L, objs, 1, cam, S.make_raycast_params(), ws=torch.empty(16, dtype=torch.uint8, device="cuda"))


def test_lod_refinement_parity(S):
    """Projected-size refinement (§3.1) with the paper's ranges (bisection 8-16, Newton 2-4):
    objects at several depths get different counts; device and oracle take the same per-object
    decision (float32 projected radius) and agree to the usual bar."""
    luts, Ns = _scene(8, 310)
    centres = np.array([[-3.0, -1.0, -30.0], [3.0, 1.5, -18.0], [-1.5, 2.0, -8.0], [1.0, -2.0, -4.0],
                        [0.0, 0.0, 2.0], [4.0, 3.0, -50.0], [-1.2, -0.9, 6.4], [0.9, 0.6, 7.3]])
    kw = dict(lod=1, bisect=16, newton=4, bisect_min=8, newton_min=2)
    W, H = 256, 192
    out, ref, rmax = _run(S, luts, centres, np.ones(8), W, H, eye=(0.0, 0.0, 9.0), prm_kw=kw)
    ocam = O.make_camera(*camera_frame((0.0, 0.0, 9.0)), 45.0, W, H)
    alloc = [O.lod_steps(ocam, O.make_raycast_params(**kw), centres[k], rmax[k]) for k in range(8)]
    bracket = np.array([2 * rmax[k] / (32 * 2.0 ** alloc[k][0]) for k in range(8)])
    eye, fwd, right, up = camera_frame((0.0, 0.0, 9.0))
    seam = _seam_pixels(ref, centres, eye, fwd, right, up, 45.0, W, H)
    assert seam.mean() < 0.01
    _compare(out, ref, rmax, W, H, depth_abs=bracket, seam=seam)
    steps = {a[:2] for a in alloc}
    assert len(steps) >= 3   # the scene exercises several allocations, Newton counts included


@pytest.mark.parametrize("method", [1, 2])  # SHM_RECON_BILINEAR (FD normals), SHM_RECON_BICUBIC (Catmull-Rom)
def test_value_only_raycast_parity(S, method):
    """The value-only baselines ray cast (the equal-storage renders of §4.5): one L = 8 SH glyph as a
    value table at 2N = 32 (the storage of a Hermite table at N = 16), device vs the oracle's value-only
    ray caster on identical stored values, with the same bars as the Hermite renders (face seams
    excluded: each face's gutter is evaluated in its own chart)."""
    c = I.sh_coeffs(1, 8, 20063 + 41)[0]
    N2 = 32
    grid = O.value_grid_sh(N2, 8, c).astype(np.float32)
    L = S.alloc_lut(1, N2, S.SHM_F32, S.SHM_LAYOUT_VALUE)
    L.data.copy_(torch.from_numpy(grid.ravel()))
    stored = grid.astype(np.float64)
    rmax = np.array([1.3 * float(np.abs(stored).max())])
    centres = np.zeros((1, 3))
    objs = S.objects_tensor(centres, [1.0], rmax.astype(np.float32), [0])
    W, H, fov = 96, 72, 40.0
    eye, fwd, right, up = camera_frame((0.4, 0.5, 3.6))
    out = S.raycast(L, objs, 1, S.make_camera(eye, fwd, right, up, fov, W, H), S.make_raycast_params(recon=method))
    torch.cuda.synchronize()
    pool, off, Ns = O.make_value_pool([stored.reshape(6, N2 + 4, N2 + 4)])
    ref = O.raycast(pool, off, Ns, centres, [1.0], rmax, [0], O.make_camera(eye, fwd, right, up, fov, W, H),
                    O.make_raycast_params(recon=method))
    seam = _seam_pixels(ref, centres, eye, fwd, right, up, fov, W, H)
    assert _compare(out, ref, rmax, W, H, seam=seam) > 500


def test_value_only_raycast_rejects_unknown_method(S):
    L = S.alloc_lut(1, 8, S.SHM_F32, S.SHM_LAYOUT_VALUE, zero=True)
    objs = S.objects_tensor(np.zeros((1, 3)), [1.0], [1.0], [0])
    eye, fwd, right, up = camera_frame((0.0, 0.0, 4.0))
    with pytest.raises(S.ShmError, match="invalid"):
        S.raycast(L, objs, 1, S.make_camera(eye, fwd, right, up, 40.0, 16, 16), S.make_raycast_params(recon=7))


def _frame(S, centres, W, H, eye=(0.0, 0.0, 40.0), fov=40.0):
    lut = S.alloc_lut(1, 8, r0=[1.0], zero=True)
    n = len(centres)
    e, fwd, right, up = camera_frame(eye)
    return S.raycast(lut, S.objects_tensor(centres, np.ones(n), np.ones(n), np.zeros(n, int)), n,
                     S.make_camera(e, fwd, right, up, fov, W, H), S.make_raycast_params())


@pytest.mark.parametrize("n", [4096, 4097, 9001])
def test_many_objects_in_depth_order(S, n):
    """Up to 4,096 objects each warp forms the keys it ranks against, beyond they are formed once: overlapping
    spheres at many depths (equal ones among them: the lower index is in front) between objects behind the
    camera give the frame of the visible ones alone."""
    rng = np.random.default_rng(n)
    seen = np.sort(rng.choice(n, 300, replace=False))
    near = np.stack([rng.uniform(-9, 9, 300), rng.uniform(-6, 6, 300), np.round(rng.uniform(-9, 9, 300), 0)], 1)
    near[7] = near[3]  # the same sphere twice
    centres = np.tile([0.0, 0.0, 900.0], (n, 1)) + rng.uniform(-50, 50, (n, 3))
    centres[seen] = near
    full, part = _frame(S, centres, 320, 200), _frame(S, near, 320, 200)
    ids = part["obj_id"].long()
    assert (ids >= 0).float().mean() > 0.2
    mapped = torch.where(ids >= 0, torch.from_numpy(seen).cuda()[ids.clamp(min=0)], ids)
    assert torch.equal(full["obj_id"].long(), mapped)
    for k in ("rgba", "depth", "normal"):
        assert torch.equal(full[k].view(torch.int32), part[k].view(torch.int32)), k


def test_image_wider_than_packed_tiles(S):
    """Above 4,096 pixels a side the tiles work out the objects' rectangles themselves: bump objects across an
    image of 4,300 x 32, sampled pixels against the oracle, bars of the full-size grid."""
    n, W, H, fov = 8, 4300, 32, 0.5
    luts, Ns = _scene(n, 320)
    centres = np.stack([np.linspace(-4.2, 4.2, n), 0.3 * np.sin(np.arange(n)), np.linspace(-0.5, 0.5, n)], 1)
    r0 = np.ones(n, np.float32)
    L, stored = upload_pool(S, luts, r0=r0)
    rmax = S.lut_bounds(L).cpu().numpy()
    eye, fwd, right, up = camera_frame((0.0, 0.0, 8.0))
    out = S.raycast(L, S.objects_tensor(centres, 0.5 * np.ones(n), 0.5 * rmax, np.arange(n)), n,
                    S.make_camera(eye, fwd, right, up, fov, W, H), S.make_raycast_params())
    rng = np.random.default_rng(5)
    px, py = rng.integers(0, W, 400).astype(np.int32), rng.integers(0, H, 400).astype(np.int32)
    pool = stored.reshape(-1, 4)
    off, Nn = O.make_pool(luts)[1:]
    rmax_o = np.array([O.lut_bound(pool[off[k]:off[k] + 6 * (Nn[k] + 2) ** 2].reshape(6, Nn[k] + 2, Nn[k] + 2, 4),
                                   int(Nn[k]), 1.0) for k in range(n)]) * 0.5
    ref = O.raycast(pool, off, Nn, centres, 0.5 * np.ones(n), rmax_o, np.arange(n),
                    O.make_camera(eye, fwd, right, up, fov, W, H), O.make_raycast_params(), px=px, py=py,
                    r0=r0.astype(np.float64))
    ids = out["obj_id"].cpu().numpy()[py, px]
    depth = out["depth"].double().cpu().numpy()[py, px]
    amb = ref["margin"] < 1e-4 * rmax_o.max()
    assert np.all((ids == ref["obj_id"])[~amb])
    hit = (ids >= 0) & ~amb
    assert hit.sum() > 50 and (ids < 0).sum() > 20 and len(set(ids[hit])) == n
    assert (np.abs(depth[hit] - ref["depth"][hit]) / ref["depth"][hit]).max() <= 2e-5
