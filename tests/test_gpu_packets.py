"""The packet forward's routes -- parts of packets, the triage of packets and of
rays, ray orders -- against the plain kernel (one thread per ray): the same
walk and the same arithmetic per ray, so every segment count and every hit is
equal and the images differ by the compiler's contraction alone (1e-5, the bar
of the ray-order check in smoke()).  Sizes: one ray, a ragged packet, one warp
of parts, about a packet per resident warp, and above four of them, where the
triage lists packets.  With a log the adjoint replays what the forward formed:
its gradient equals the walking adjoint's within 1e-5 of the largest entry
(FP32 summation order)."""
import numpy as np
import pytest
import torch

from paper_2202_06088_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B(cuda_lib):
    from paper_2202_06088_gb300 import binding
    return binding


@pytest.fixture(scope="module")
def scenes():
    rng = np.random.default_rng(5)
    mixed = I.make_coefficients(rng, I.random_mixed_tree(6, 7, p_leaf=0.2, p_empty=0.3), K=16, T=9, hh_degree=3,
                                mean_sigma=8.0)
    return {"solid": I.config1_tree(), "mixed": mixed}


def _rays(W, H, shuffle=False):
    rays, _ = I.camera_rays(I.sphere_cameras(43, 1, 2.5, W, H)[0], 0.37)
    return rays.subset(np.random.default_rng(1).permutation(rays.n)) if shuffle else rays


def _same(got, ref):
    assert torch.equal(got["nseg"], ref["nseg"])
    assert torch.equal(torch.isfinite(got["depth"]), torch.isfinite(ref["depth"]))
    for k in ("rgb", "alpha"):
        assert (got[k] - ref[k]).abs().max().item() <= 1e-5, k
    assert (got["tau"] - ref["tau"]).abs().max().item() <= 1e-5 * max(1.0, ref["tau"].max().item())


@pytest.mark.parametrize("W,H", [(1, 1), (33, 1), (130, 121), (421, 307), (901, 703)])
@pytest.mark.parametrize("scene,dtype", [("solid", "f32"), ("mixed", "bf16"), ("mixed", "f32")])
def test_packet_routes_equal_the_plain_kernel(B, scenes, scene, dtype, W, H):
    tree_d = B.Tree(scenes[scene], dtype)
    dr = B.DeviceRays.from_host(_rays(W, H))
    ref = B.neuvv_render(tree_d, dr, kernel="plain")
    _same(B.neuvv_render(tree_d, dr, kernel="packet"), ref)
    _same(B.neuvv_render(tree_d, dr, kernel="packet", out=B.alloc_out(dr.n, log_bytes_per_ray=512)), ref)
    assert tree_d.status() == 0


@pytest.mark.parametrize("order", ["given", "region", "rays"])
@pytest.mark.parametrize("reserve", [0, 1 << 22])
def test_logged_routes_give_the_walks_gradient(B, scenes, order, reserve):
    tree = scenes["solid"]
    tree_d = B.Tree(tree, "f32")
    dr = B.DeviceRays.from_host(_rays(401, 307, shuffle=True))   # more packets than resident warps, uneven rays
    g = torch.from_numpy(np.random.default_rng(3).standard_normal((dr.n, 3)).astype(np.float32)).cuda()
    plain = B.neuvv_render(tree_d, dr, kernel="plain")
    walk = B.neuvv_render_backward(tree_d, dr, plain, g, kernel="packet")
    tree_d.set_packet_order({"given": B.ORDER_AS_GIVEN, "region": B.ORDER_BY_REGION, "rays": B.ORDER_BY_RAY}[order])
    out = B.neuvv_render(tree_d, dr, kernel="packet", out=B.alloc_out(dr.n, log_bytes_per_ray=512))
    _same(out, plain)
    log = B.neuvv_log_read(out, dr.n, 8)
    assert torch.equal(log["count"], out["nseg"])
    tree_d.reserve_adjoint(reserve)
    got = B.neuvv_render_backward(tree_d, dr, out, g, kernel="packet")
    assert (got - walk).abs().max().item() <= 1e-5 * walk.abs().max().item()
    assert tree_d.status() == 0
