"""Edges of the kernels that multiply on tensor cores, against the fp64 oracle."""
import numpy as np
import pytest
import torch

import oracle
from gpu_util import check_y, dev, pack_on_gpu, packed_to_host
from paper_2511_04477_b200 import binding, inputs

pytestmark = pytest.mark.gpu

FORMATS = [(4, 128), (4, 64), (3, 128), (3, 64)]


def growing_activations(n, seed):
    """Magnitudes from about 1e-1 to 1e3 in ascending order: the running scale of the fp16 operands changes along the
    list.  (With weights of order 1: results below the fp16 normal range would round to more than the tolerance.)"""
    x = inputs.activations(n, seed).astype(np.float32)
    return (x * np.logspace(-1, 3, n).astype(np.float32)).clip(-6e4, 6e4).astype(np.float16)


@pytest.mark.parametrize("bits,group", FORMATS)
@pytest.mark.parametrize("m_blocks,n,batch", [(1, 1, 2), (1, 8, 5), (2, 31, 4), (3, 33, 8), (2, 257, 3), (37, 264, 6), (101, 300, 4),
                                              (5, 2049, 8), (20, 2056, 2)])
def test_small_batch_at_chunk_part_and_split_edges(bits, group, m_blocks, n, batch):
    m = m_blocks * group
    W = inputs.weights(m, n, seed=m + n, std=0.5)
    X = np.stack([growing_activations(n, seed=70 + b)[:: 1 if b % 2 else -1] for b in range(batch)])
    p = pack_on_gpu(np.ascontiguousarray(W), bits, group)
    codes, s, z = packed_to_host(p)
    ws = binding.new_gemm_small_workspace(p)
    Xd = dev(np.ascontiguousarray(X))
    Y = binding.spqt_dense_gemm_small(p, Xd, ws)
    t = inputs.threshold_for_sparsity(X[0], 0.3)
    Ys, idx, cnt = binding.spqt_sparse_gemm_small(p, Xd, t, ws)
    torch.cuda.synchronize()
    ref_idx, ref_cnt = oracle.union_sparsify(X, t)
    assert int(cnt.item()) == ref_cnt and np.array_equal(idx.cpu().numpy()[:ref_cnt], ref_idx)
    Ys_ref, bound = oracle.sparse_gemm_small(codes, s, z, m, n, X, ref_idx, bits, group)
    for b in range(batch):
        y_ref, dbound = oracle.dense_gemv(codes, s, z, m, n, X[b], bits, group)
        check_y(Y.cpu().numpy()[b], y_ref, dbound, "dense row %d" % b)
        check_y(Ys.cpu().numpy()[b], Ys_ref[b], bound[b], "row %d" % b)
