"""Composition culls (ray, primitive) pairs by the ball around the primitive's
box before it forms the exact local ray.  No pair that meets the box may be
lost: small primitives far from the world's origin, seen from nearby, where the
FP32 spacing of world coordinates is a sizeable part of the ball; and short
ray directions, whose squared length nears the end of the FP32 range.

Reference: the FP64 oracle on the same FP32 inputs, at the bar of 1e-4 that
tests/test_gpu_compose.py holds every pixel to whose early stop is not
ambiguous.  The tree is filled to its corners, so a lost corner shows."""
import numpy as np
import pytest

import oracle
from paper_2202_06088_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B(cuda_lib):
    from paper_2202_06088_gb300 import binding
    return binding


@pytest.fixture(scope="module")
def cube():
    cells = np.stack(np.meshgrid(*[np.arange(8)] * 3, indexing="ij"), -1).reshape(-1, 3)
    st = I.build_tree(3, np.full(512, 3), cells)
    return I.make_coefficients(np.random.default_rng(2), st, K=8, T=5, hh_degree=2, mean_sigma=30.0)


def _rotation(seed):
    q, _ = np.linalg.qr(np.random.default_rng(seed).standard_normal((3, 3)))
    return q * np.sign(np.linalg.det(q))


@pytest.mark.parametrize("where,scale,length", [
    ((0.0, 0.0, 0.0), 0.3, 1.0),            # at the origin
    ((1.0e5, -7.0e4, 4.0e4), 0.3, 1.0),     # spacing of coordinates 2^-7, radius 0.26
    ((-3.0e5, 2.0e5, 1.0e5), 1.0, 1.0),
    ((1.0e3, 5.0e2, -8.0e2), 0.01, 1.0),
    ((0.0, 0.0, 0.0), 1e-3, 1e-18),         # squared direction lengths of 1e-36
])
def test_no_ray_that_meets_the_box_is_culled(B, cube, where, scale, length):
    xf, rays = [], None
    tree_d = B.Tree(cube, "f32")
    for seed in range(4):
        M = np.concatenate([scale * _rotation(seed), np.asarray(where)[:, None]], 1).astype(np.float32)
        centre = M.astype(np.float64) @ np.array([0.5, 0.5, 0.5, 1.0])
        v = np.random.default_rng(10 + seed).standard_normal(3)
        cam = I.look_at(centre + 1.5 * scale * v / np.linalg.norm(v), centre, 64, 64, fov_y_deg=75.0)
        rays, _ = I.camera_rays(cam, 0.4)
        rays.dirs = (rays.dirs * np.float32(length)).astype(np.float32)
        xf = [M.astype(np.float64)]
        ref = oracle.compose([cube], xf, [0.0], [np.ones(3)], rays)
        got = B.neuvv_compose([tree_d], xf, [0.0], [np.ones(3)], B.DeviceRays.from_host(rays))
        ok = ref["stop_margin"] > 1e-3
        assert ok.mean() > 0.95 and (ref["alpha"] > 0.01).mean() > 0.1
        for k in ("rgb", "alpha"):
            err = np.abs(got[k].cpu().numpy() - ref[k])[ok]
            assert err.max() <= 1e-4, (seed, k, err.max())
