"""The bootstrap passes decide in FP32 (pairs) where FP32 is sure and in FP64
elsewhere; their results are those of FP64 throughout.

The depth of bootstrap(T_1) is compared bit for bit with the same FP64 expressions
in NumPy, operation by operation, over images that are not a multiple of a warp or
a block, motions forwards, sideways, without translation (a.b = 0 everywhere) and
turned by half a turn, flows that are zero, ordinary and far outside the image, and
clamps that cut both ends.

The cheirality counts of the epipolar bootstrap equal FP64's, but for pixels whose
FP64 value is below 1e-12 of its terms (there a fused and an unfused product differ
in sign); these are counted in the test."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def vd():
    from paper_2104_06789_gb300 import build, voldor
    build.build()
    return voldor


def _pose(axis, angle, t):
    a = np.asarray(axis, float) / np.linalg.norm(axis)
    X = np.array([[0, -a[2], a[1]], [a[2], 0, -a[0]], [-a[1], a[0], 0]])
    T = np.eye(4)
    T[:3, :3] = np.eye(3) + np.sin(angle) * X + (1 - np.cos(angle)) * X @ X
    T[:3, 3] = t
    return T


MOTIONS = {"forward": ((1, 2, 0.5), 0.01, (0.02, -0.01, -1.0)), "sideways": ((0, 1, 0), 0.03, (0.7, 0.05, 0.1)),
           "still": ((0, 0, 1), 0.02, (0.0, 0.0, 0.0)), "turned": ((0, 1, 0.1), 3.1, (0.3, 0.2, 0.9))}


def _flows(W, H, T, K, rng):
    x, y = np.meshgrid(np.arange(W, dtype=np.float64), np.arange(H, dtype=np.float64))
    fx, fy, cx, cy = K
    z = rng.uniform(1.0, 30.0, (H, W))
    Y = np.stack([(x - cx) / fx * z, (y - cy) / fy * z, z], -1) @ T[:3, :3].T + T[:3, 3]
    f = np.stack([fx * Y[..., 0] / Y[..., 2] + cx - x, fy * Y[..., 1] / Y[..., 2] + cy - y], -1)
    f = np.clip(f + rng.normal(0, 0.3, f.shape), -5e3, 5e3)
    f[rng.random((H, W)) < 0.05] = 0.0
    f[rng.random((H, W)) < 0.02] = 5.0e3
    return f.astype(np.float32)


def _depth64(f, K, T, imin, imax):
    H, W = f.shape[:2]
    x, y = np.meshgrid(np.arange(W, dtype=np.float64), np.arange(H, dtype=np.float64))
    fx, fy, cx, cy = K
    ifx, ify = 1.0 / fx, 1.0 / fy
    u, v = f[..., 0].astype(np.float64), f[..., 1].astype(np.float64)
    dx, dy, mx, my = (x - cx) * ifx, (y - cy) * ify, (x + u - cx) * ifx, (y + v - cy) * ify
    R, t = T[:3, :3], T[:3, 3]
    Rx, Ry, Rz = ((R[i, 0] * dx + R[i, 1] * dy) + R[i, 2] for i in range(3))
    ax, ay, bx, by = Rx - mx * Rz, Ry - my * Rz, mx * t[2] - t[0], my * t[2] - t[1]
    num, den = ax * ax + ay * ay, ax * bx + ay * by
    with np.errstate(all="ignore"):
        r = num / den
        ok = (den > 0) & np.isfinite(r)
        lo, hi = np.float64(np.float32(imin)), np.float64(np.float32(imax))
        inv = np.where(ok, np.minimum(np.maximum(r, lo), hi), lo)
        return (1.0 / inv).astype(np.float32)


@pytest.mark.parametrize("motion", sorted(MOTIONS))
@pytest.mark.parametrize("W,H,dtype,clamp", [(33, 9, np.float32, (0.05, 1.0)), (160, 121, np.float16, (0.05, 0.3)),
                                             (257, 65, np.float32, (1e-4, 1e3))])
def test_depth_equals_fp64_bit_for_bit(vd, motion, W, H, dtype, clamp):
    rng = np.random.default_rng(W + H)
    K = (0.8 * W, 0.83 * W, 0.47 * W, 0.52 * H)
    T = _pose(*MOTIONS[motion])
    f = _flows(W, H, T, K, rng).astype(dtype)
    p = vd.default_params(inv_depth_min=clamp[0], inv_depth_max=clamp[1], hyps_per_frame=64)
    g = vd.Window(np.repeat(f[None], 2, 0), K, p)
    g.bootstrap(T)
    _, D, Wm = g.get_pose_depth_rigidness(poses=False)
    ref = _depth64(f, K, T, *clamp)
    assert np.array_equal(D.view(np.uint32), ref.view(np.uint32))
    assert np.all(Wm == 1.0)
    g.destroy()


@pytest.mark.parametrize("W,H,M", [(33, 20, 64), (160, 121, 64)])
def test_cheirality_counts_equal_fp64(vd, W, H, M):
    rng = np.random.default_rng(7 * W + H)
    K = (0.8 * W, 0.83 * W, 0.47 * W, 0.52 * H)
    f = _flows(W, H, _pose(*MOTIONS["sideways"]), K, rng)
    g = vd.Window(np.repeat(f[None], 2, 0), K, vd.default_params(inv_depth_min=0.01, inv_depth_max=2.0, hyps_per_frame=64))
    T1 = g.bootstrap_epipolar(M, 1.0)
    r = g.epipolar_results()
    x, y = np.meshgrid(np.arange(W, dtype=np.float64), np.arange(H, dtype=np.float64))
    fx, fy, cx, cy = K
    u, v = x + f[..., 0].astype(np.float64), y + f[..., 1].astype(np.float64)
    valid = (u >= 0) & (u <= W - 1) & (v >= 0) & (v <= H - 1)
    assert r["n_valid"] == valid.sum()
    m0x, m0y, m1x, m1y = (x - cx) / fx, (y - cy) / fy, (u - cx) / fx, (v - cy) / fy
    Wm = np.array([[0, -1, 0], [1, 0, 0], [0, 0, 1.0]])
    best = None
    for a, Wa in enumerate((Wm, Wm.T)):
        R = r["U"] @ Wa @ r["V"].T
        for sg in range(2):
            t = (1.0, -1.0)[sg] * r["U"][:, 2]
            Rx, Ry, Rz = (R[i, 0] * m0x + R[i, 1] * m0y + R[i, 2] for i in range(3))
            ax, bx, ay, by = Rx - m1x * Rz, m1x * t[2] - t[0], Ry - m1y * Rz, m1y * t[2] - t[1]
            aa, ab = ax * ax + ay * ay, ax * bx + ay * by
            with np.errstate(all="ignore"):
                z = ab / aa * Rz + t[2]
            edge = valid & ((np.abs(ab) < 1e-12 * (np.abs(ax * bx) + np.abs(ay * by)) + 1e-16)
                            | (np.abs(z) < 1e-12 * (np.abs(ab / aa * Rz) + 1)))
            n = (valid & (aa > 0) & (ab > 0) & (z > 0)).sum()
            got = r["counts"][2 * a + sg]
            assert abs(int(got) - int(n)) <= edge.sum(), (a, sg)
            if best is None or got > best[0]:
                best = (got, R, t)
    assert np.abs(T1[:3, :3] - best[1]).max() < 1e-12 and np.abs(T1[:3, 3] - best[2]).max() < 1e-12
    g.destroy()
