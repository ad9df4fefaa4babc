"""The sparse Adam step over record lengths: records that half a warp covers, that a
warp covers partly and fully, and longer ones, each with its own grouping of
rows.  Leaf counts with a ragged last word of the touched bitmap, and words with
none, one, an odd number and all of their leaves touched.  Against the FP64 oracle
at the bars of test_sparse_adam_matches_oracle (tests/test_gpu_backward.py)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2202_06088_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B(cuda_lib):
    from paper_2202_06088_gb300 import binding
    return binding


@pytest.mark.parametrize("K,degree,entries", [(8, 2, 58), (16, 2, 74), (8, 3, 106), (16, 3, 122), (32, 3, 154)])
@pytest.mark.parametrize("n_cells", [1, 33, 203])
def test_adam_step_over_record_lengths(B, K, degree, entries, n_cells):
    rng = np.random.default_rng(17)
    cells = np.stack(np.unravel_index(rng.choice(512, n_cells, replace=False), (8, 8, 8)), -1)
    tree = I.make_coefficients(rng, I.build_tree(3, np.full(n_cells, 3), cells), K=K, T=4, hh_degree=degree)
    tree_d = B.Tree(tree, "bf16", with_optimizer=True)
    info = tree_d.info
    assert info.rec_len == entries
    w = tree_d.master().cpu().numpy().astype(np.float64)
    m, v = np.zeros_like(w), np.zeros_like(w)
    for step in (1, 2):
        touched = rng.random(n_cells) < 0.5
        touched[:32] = True                       # a full word, then one empty and one with a single leaf
        touched[32:64] = False
        touched[70:96] = False
        gnp = np.zeros((n_cells, info.rec_stride_f32), np.float32)
        gnp[touched, :info.rec_len] = rng.standard_normal((touched.sum(), info.rec_len)).astype(np.float32)
        bits = np.zeros((n_cells + 31) // 32, np.uint32)
        for leaf in np.nonzero(touched)[0]:
            bits[leaf >> 5] |= np.uint32(1 << (leaf & 31))
        grad, tb = torch.from_numpy(gnp).cuda(), torch.from_numpy(bits.view(np.int32)).cuda()
        B.neuvv_adam_step(tree_d, grad, tb, lr=0.01, beta1=0.9, beta2=0.99, eps=1e-8, step=step)
        oracle.adam(w, m, v, gnp.astype(np.float64), touched.astype(np.uint8), 0.01, 0.9, 0.99, 1e-8, step)
        assert torch.count_nonzero(grad).item() == 0 and torch.count_nonzero(tb).item() == 0
    got = tree_d.master()
    assert np.abs(got.cpu().numpy() - w).max() <= 1e-5
    for a, b in zip(tree_d.adam_state(), (m, v)):
        assert np.abs(a.cpu().numpy() - b).max() <= 1e-6
    assert torch.equal(tree_d.storage()[:, :info.rec_len].float(), got[:, :info.rec_len].bfloat16().float())
