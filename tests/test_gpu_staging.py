"""Records of a shading batch are staged in shared memory or read in place, by
record shape and block size.  Every form against the plain kernel: the same walk
and the same arithmetic per ray, so segment counts and hits are equal and the
images differ by the compiler's contraction alone (1e-5, the bar of
tests/test_gpu_packets.py).  Shapes on both sides of the rule, with blocks that
leave room for the staging and blocks that do not, and a ragged last packet."""
import numpy as np
import pytest
import torch

from paper_2202_06088_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B(cuda_lib):
    from paper_2202_06088_gb300 import binding
    return binding


@pytest.mark.parametrize("block", [32, 64, 256])
@pytest.mark.parametrize("K,degree,dtype,bricks", [
    (8, 3, "f32", True), (16, 3, "f32", True), (16, 3, "bf16", True), (16, 3, "f32", False),   # staged where they fit
    (8, 3, "bf16", True), (16, 2, "f32", True), (32, 2, "f32", True), (32, 3, "bf16", True),   # in place
])
def test_staged_and_in_place_records_give_the_plain_image(B, K, degree, dtype, bricks, block):
    tree = I.make_coefficients(np.random.default_rng(6), I.random_mixed_tree(6, 8, p_leaf=0.2, p_empty=0.3), K=K, T=5,
                               hh_degree=degree, mean_sigma=8.0)
    rays, _ = I.camera_rays(I.sphere_cameras(11, 1, 2.5, 131, 97)[0], 0.4)
    tree_d, dr = B.Tree(tree, dtype, bricks=bricks), B.DeviceRays.from_host(rays)
    tree_d.set_launch(block, 8, 32)
    ref = B.neuvv_render(tree_d, dr, kernel="plain")
    got = [B.neuvv_render(tree_d, dr, kernel="packet"),
           B.neuvv_render(tree_d, dr, kernel="packet", out=B.alloc_out(dr.n, log_bytes_per_ray=512))]
    if (K, degree) == (16, 3):   # the edited render, with no edit active
        got.append(B.neuvv_render_edit(tree_d, dr, B.new_edits(tree_d), beta=0.5))
    assert ref["nseg"].max().item() > 8
    for g in got:
        assert torch.equal(g["nseg"], ref["nseg"])
        assert torch.equal(torch.isfinite(g["depth"]), torch.isfinite(ref["depth"]))
        for k in ("rgb", "alpha"):
            assert (g[k] - ref[k]).abs().max().item() <= 1e-5, k
    assert tree_d.status() == 0
