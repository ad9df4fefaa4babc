"""The triage of packets: a forward call without a log, of more than two packets
per resident warp, on a sparse tree of depth 8 or more lists its packets by an
estimate of their work and runs the long ones first, in two or four parts.

Each ray is computed by the same walk and arithmetic whatever packet, part or
order it comes in, so every output of a call that lists its packets equals, bit
for bit, that of the same rays in calls too small to list (no triage up to two
packets per resident warp); the plain kernel differs by the compiler's contraction
alone (1e-5 in images; 2e-5 of the depth, a quotient of two sums of up to 64
terms with two roundings of 2^-24 each).  Whether a call lists its packets is read
from its captured graph: the counter's reset, the triage and the render."""
import ctypes

import numpy as np
import pytest
import torch

from paper_2202_06088_gb300 import inputs as I

pytestmark = pytest.mark.gpu

DEPTH = 8
LONG = 0.4          # bricks per ray, per packet of a resident warp's share, of a long packet


@pytest.fixture(scope="module")
def B(cuda_lib):
    from paper_2202_06088_gb300 import binding
    return binding


def _cells(kind):
    """Finest cells of a ball's surface (an eighth of its bricks' cells) or of a ball."""
    n = 1 << DEPTH
    x = (np.arange(n) + 0.5) / n - 0.5
    r = np.sqrt(x[:, None, None] ** 2 + x[None, :, None] ** 2 + x[None, None, :] ** 2)
    return np.argwhere((np.abs(r - 0.35) < 0.8 / n) if kind == "shell" else (r < 0.2))


def _merged(cells):
    """The same cells with every full node a leaf of its own."""
    level, out = DEPTH, []
    while level > 1 and len(cells):
        key = I.morton3(cells)
        parents, first, count = np.unique(key >> 3, return_index=True, return_counts=True)
        full = np.isin(key >> 3, parents[count == 8])
        out.append((np.full((~full).sum(), level), cells[~full]))
        order = np.argsort(key)
        cells = np.unique(cells[order][full[order]] >> 1, axis=0)
        level -= 1
    out.append((np.full(len(cells), level), cells))
    return np.concatenate([a for a, _ in out]), np.concatenate([c for _, c in out])


@pytest.fixture(scope="module")
def shell_cells():
    return _cells("shell")


@pytest.fixture(scope="module")
def trees(B, shell_cells):
    st = I.build_tree(DEPTH, np.full(len(shell_cells), DEPTH), shell_cells)

    def make(K, degree, dtype):
        host = I.make_coefficients(np.random.default_rng(3), st, K=K, T=5, hh_degree=degree, mean_sigma=40.0)
        return B.Tree(host, dtype)
    return {"f32": make(8, 2, "f32"), "bf16": make(16, 3, "bf16")}


def _rays(W, H, shuffle):
    rays, _ = I.camera_rays(I.sphere_cameras(5, 1, 1.6, W, H)[0], 0.6)
    return rays.subset(np.random.default_rng(1).permutation(rays.n)) if shuffle else rays


def _graph_nodes(call):
    call()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(g):
        call()
    n = ctypes.c_size_t()
    assert ctypes.CDLL("libcuda.so.1").cuGraphGetNodes(ctypes.c_void_p(g.raw_cuda_graph()), None, ctypes.byref(n)) == 0
    return n.value


def _resident_warps(tree_d):
    # blocks of 64 threads at 128 registers: 16 warps per multiprocessor
    return 16 * torch.cuda.get_device_properties(tree_d.info.device).multi_processor_count


def _parts_of_packets(rays, cells, n_resident):
    """Whole, halved and quartered packets by the estimate: of each ray one point of
    its chord of the box, at a fraction of its own within the packet."""
    o, d = rays.origins.astype(np.float64), rays.dirs.astype(np.float64)
    with np.errstate(divide="ignore"):
        a, b = (0.0 - o) / d, (1.0 - o) / d
    s0, s1 = np.maximum(np.minimum(a, b).max(0), 0.0), np.maximum(a, b).min(0)
    hit = s0 < s1
    lane = np.arange(rays.n) & 31
    rev = np.array([int(f"{k:05b}"[::-1], 2) for k in range(32)])[lane]
    p = o + (s0 + (rev + 0.5) / 32.0 * (s1 - s0)) * d
    N = 1 << (DEPTH - 3)
    grid = np.zeros((N, N, N), bool)
    grid[tuple((cells >> 3).T)] = True
    at = np.clip((p * N).astype(int), 0, N - 1)
    bricks = np.where(hit & grid[tuple(at)], (s1 - s0) * N / 32.0, 0.0)
    per = np.add.reduceat(bricks, np.arange(0, rays.n, 32))
    half = LONG * len(per) / n_resident
    any_hit = np.add.reduceat(hit.astype(int), np.arange(0, rays.n, 32)) > 0
    return (any_hit & (per < 0.9 * half)).sum(), ((per > 1.1 * half) & (per < 1.8 * half)).sum(), (per > 2.2 * half).sum()


def _in_small_calls(B, call, rays, n_resident):
    step = 32 * n_resident          # one packet per resident warp: no list
    parts = [call(B.DeviceRays.from_host(rays.subset(np.arange(k, min(k + step, rays.n))))) for k in range(0, rays.n, step)]
    return {k: torch.cat([p[k] for p in parts]) for k in parts[0]}


@pytest.mark.parametrize("shuffle", [False, True])
@pytest.mark.parametrize("W,H", [(521, 401), (701, 503)])     # 2.7 and 4.5 packets per resident warp, ragged
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_listed_packets_compute_the_same_rays(B, trees, shell_cells, dtype, W, H, shuffle):
    tree_d, rays = trees[dtype], _rays(W, H, shuffle)
    n_resident, dr = _resident_warps(tree_d), B.DeviceRays.from_host(rays)
    assert rays.n % 32 and 2 * n_resident < rays.n // 32
    if not shuffle:
        assert min(_parts_of_packets(rays, shell_cells, n_resident)) > 20      # all three kinds are listed
    sl = B.neuvv_slice(tree_d, 0.6)
    edits = B.new_edits(tree_d)
    pick = torch.from_numpy(np.random.default_rng(7).random(edits.shape[0]) < 0.3).to(edits.device)
    edits[pick, :3], edits[pick, 3], edits[pick, 4] = 0.8, 25.0, 0.2
    calls = {"render": lambda r: B.neuvv_render(tree_d, r, kernel="packet"),
             "slice": lambda r: B.neuvv_render_slice(tree_d, sl, r),
             "edit": lambda r: B.neuvv_render_edit(tree_d, r, edits, beta=0.6)}
    got = {}
    for name, call in calls.items():
        out = B.alloc_out(rays.n, dr.o.device)
        inside = {"render": lambda: B.neuvv_render(tree_d, dr, kernel="packet", out=out),
                  "slice": lambda: B.neuvv_render_slice(tree_d, sl, dr, out=out),
                  "edit": lambda: B.neuvv_render_edit(tree_d, dr, edits, beta=0.6, out=out)}[name]
        assert _graph_nodes(inside) == 3, name
        got[name] = call(dr)
        ref = _in_small_calls(B, call, rays, n_resident)
        for k in ("rgb", "alpha", "depth", "tau", "nseg"):
            assert torch.equal(got[name][k], ref[k]), (name, k)
    plain, r = B.neuvv_render(tree_d, dr, kernel="plain"), got["render"]
    assert torch.equal(r["nseg"], plain["nseg"]) and plain["nseg"].max().item() > 4
    fin = torch.isfinite(plain["depth"])
    assert torch.equal(fin, torch.isfinite(r["depth"]))
    assert ((r["depth"] - plain["depth"]).abs()[fin] <= 2e-5 * plain["depth"][fin]).all()
    for k in ("rgb", "alpha"):
        assert (r[k] - plain[k]).abs().max().item() <= 1e-5, k
    assert not torch.equal(got["edit"]["rgb"], r["rgb"]) and tree_d.status() == 0


@pytest.mark.parametrize("leaves", ["finest", "merged"])
def test_solids_are_not_listed(B, leaves):
    """Whether a solid's leaves are finest cells or its full nodes."""
    cells = _cells("ball")
    level, cells = (np.full(len(cells), DEPTH), cells) if leaves == "finest" else _merged(cells)
    host = I.make_coefficients(np.random.default_rng(3), I.build_tree(DEPTH, level, cells), K=8, T=5, hh_degree=2,
                               mean_sigma=40.0)
    tree_d, dr = B.Tree(host, "f32"), B.DeviceRays.from_host(_rays(521, 401, False))
    out = B.alloc_out(dr.n, dr.o.device)
    assert _graph_nodes(lambda: B.neuvv_render(tree_d, dr, kernel="packet", out=out)) == 2     # reset, render
