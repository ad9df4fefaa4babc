"""How many segments a log of a given size holds: 8 bytes a slot (leaf and lane
in one word, chord), 256 slots a chunk, one link per chunk.  A log with exactly
one chunk per packet holds every packet of up to 256 segments; one chunk less
leaves one packet out."""
import numpy as np
import pytest
import torch

from paper_2202_06088_gb300 import inputs as I

pytestmark = pytest.mark.gpu

PACKETS = 200
FIXED = 64 + 3 * 4 * PACKETS + 4 * 32 * PACKETS + 4 * 4096 + 16    # header, per packet, per ray, sort bins, alignment
CHUNK = 4 + 256 * 8


@pytest.fixture(scope="module")
def B(cuda_lib):
    from paper_2202_06088_gb300 import binding
    return binding


@pytest.mark.parametrize("missing", [0, 1])
def test_one_chunk_per_packet_is_room_for_every_packet(B, missing):
    rng = np.random.default_rng(4)
    cells = np.stack(np.meshgrid(*[np.arange(4)] * 3, indexing="ij"), -1).reshape(-1, 3)
    tree = I.make_coefficients(rng, I.build_tree(2, np.full(64, 2), cells), K=4, T=3, hh_degree=2, mean_sigma=0.5)
    n = 32 * PACKETS
    d = rng.standard_normal((3, n))
    d /= np.linalg.norm(d, axis=0)
    o = 0.5 + rng.uniform(-0.3, 0.3, (3, n)) - 3.0 * d     # aimed at the inside of a filled cube
    rays = I.Rays(o.astype(np.float32), d.astype(np.float32), np.full(n, 0.5, np.float32))
    tree_d, dr = B.Tree(tree, "f32"), B.DeviceRays.from_host(rays)
    out = B.alloc_out(n, dr.o.device)
    out["log"] = torch.empty((FIXED + (PACKETS - missing) * CHUNK + 3) // 4, device=dr.o.device, dtype=torch.int32)
    B.neuvv_render(tree_d, dr, kernel="packet", out=out)
    segments = out["nseg"].view(PACKETS, 32).sum(1)
    assert segments.min().item() > 0 and segments.max().item() <= 256
    count = B.neuvv_log_read(out, n, 16)["count"].view(PACKETS, 32)
    held = (count >= 0).all(1)
    assert held.sum().item() == PACKETS - missing
    assert torch.equal(count[held], out["nseg"].view(PACKETS, 32)[held])
    # the adjoint takes the packet that is left out by walking
    g = torch.from_numpy(rng.standard_normal((n, 3)).astype(np.float32)).to(dr.o.device)
    ref = B.neuvv_render_backward(tree_d, dr, B.neuvv_render(tree_d, dr, kernel="plain"), g, kernel="plain")
    got = B.neuvv_render_backward(tree_d, dr, out, g, kernel="packet")
    assert (got - ref).abs().max().item() <= 1e-5 * ref.abs().max().item()
    assert tree_d.status() == 0
