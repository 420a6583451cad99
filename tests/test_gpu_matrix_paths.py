"""Edges of the kernels that multiply on tensor cores, against the fp64 oracle, and of the conversion that feeds them."""
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


@pytest.mark.parametrize("bits,group,m_blocks,n,batch", [(4, 128, 16, 3072, 8), (3, 64, 19, 3080, 3), (4, 64, 25, 2055, 6), (3, 128, 33, 2048, 2)])
def test_small_batch_in_clusters_with_an_sm_for_each_cta(bits, group, m_blocks, n, batch):
    test_small_batch_at_chunk_part_and_split_edges(bits, group, m_blocks, n, batch)


def share_not_nearest(y, exact):
    """Share of the outputs that are not the fp16 nearest to the exact value.  A value lands on the other side of a rounding
    boundary with a probability of its error before the rounding over the spacing of fp16: the mean error in those units."""
    return float(np.mean(y.view(np.uint16) != exact.astype(np.float16).view(np.uint16)))


# fp32 FMAs in sequence leave 0.2 to 0.5 % on such inputs, multipliers cut by the alignment of the tensor core's products 1 to
# 5 %, sums cut when the scale changes 0.8 % (the last case).  The bound is twice the mean of the first; a share of 0.3 % of
# 8192 values has a deviation of 0.06 %.
NOT_NEAREST = 0.006


@pytest.mark.parametrize("bits,group,n", [(4, 128, 602), (4, 64, 1490), (3, 128, 543), (3, 64, 293), (4, 128, 4100), (3, 128, 9000)])
def test_sums_are_as_exact_as_fp32(bits, group, n):
    m, batch = 8192, 8
    W = inputs.weights(m, n, seed=n)
    X = np.stack([inputs.activations(n, seed=40 + b) for b in range(batch)])
    for b in range(1, batch, 2):   # outliers: the scale of the multipliers changes along the list
        X[b, np.random.Generator(np.random.PCG64(b)).random(n) < 0.01] *= 20
    p = pack_on_gpu(W, bits, group)
    codes, s, z = packed_to_host(p)
    Xd = dev(X)
    small = binding.new_gemm_small_workspace(p)
    rows = [oracle.dense_gemv(codes, s, z, m, n, X[b], bits, group)[0] for b in range(batch)]
    for b in (0, 1):
        y = binding.spqt_dense_gemv(p, Xd[b].contiguous(), binding.new_workspace(m, n, bits, group)).cpu().numpy()
        assert share_not_nearest(y, rows[b]) < NOT_NEAREST, "one row, %d" % b
    for rows_at_once in (4, 8):
        Y = binding.spqt_dense_gemm_small(p, Xd[:rows_at_once], small).cpu().numpy()
        assert share_not_nearest(Y, np.stack(rows[:rows_at_once])) < NOT_NEAREST, "%d rows" % rows_at_once


# (0.17 to 0.27 % with fp32 FMAs in sequence: multipliers cut by the alignment leave 0.5 to 0.7 %)
@pytest.mark.parametrize("bits,n", [(2, 700), (4, 300)])
def test_two_level_sums_are_as_exact_as_fp32(bits, n):
    m = 8192
    W = inputs.weights(m, n, seed=n)
    x = inputs.activations(n, seed=50)
    y_ref, _ = oracle.kq_gemv(*oracle.kq_quantize(W, bits=bits), x)
    p = binding.spqt_kqw_pack(dev(W), bits)
    y = binding.spqt_kqw_dense_gemv(p, dev(x), binding.new_kq_workspace(p)).cpu().numpy()
    assert share_not_nearest(y, y_ref) < 0.004


@pytest.mark.parametrize("bits,group", FORMATS)
@pytest.mark.parametrize("m_blocks,n,ctas", [(1, 1, 0), (2, 31, 0), (3, 33, 2), (7, 257, 4), (40, 300, 7), (19, 2049, 8), (5, 8193, 0), (9, 300, 72),
                                             (101, 33, 0), (149, 260, 0), (299, 40, 0), (149, 8191, 0), (200, 8192, 0), (149, 8200, 0), (3, 8200, 0)])
def test_single_row_at_chunk_part_slice_and_piece_edges(bits, group, m_blocks, n, ctas):
    """Clusters, one CTA per block-row with 16 and with 8 warps, equal pieces of all block-rows; the list given, collected in
    the call (the same bits) and absent."""
    m = m_blocks * group
    W = inputs.weights(m, n, seed=m + n, std=0.1)
    x = growing_activations(n, seed=90)
    p = pack_on_gpu(W, bits, group)
    codes, s, z = packed_to_host(p)
    ws = binding.new_workspace(m, n, bits, group)
    t = inputs.threshold_for_sparsity(x, 0.4) if n != 8192 else -1.0   # (the longest list of one CTA)
    try:
        binding.spqt_set_tuning(ctas)
        y, idx, cnt = binding.spqt_sparsify_gemv(p, dev(x), t, ws)
        y_list = binding.spqt_sparse_gemv(p, dev(x), idx, cnt, ws)
        y_dense = binding.spqt_dense_gemv(p, dev(x), ws)
        torch.cuda.synchronize()
    finally:
        binding.spqt_set_tuning(0)
    ref_idx, ref_cnt = oracle.sparsify(x, t)
    assert int(cnt.item()) == ref_cnt and np.array_equal(idx.cpu().numpy()[:ref_cnt], ref_idx)
    y_ref, bound = oracle.sparse_gemv(codes, s, z, m, n, x, ref_idx, bits, group)
    check_y(y.cpu().numpy(), y_ref, bound, "list collected")
    assert torch.equal(y, y_list)
    y_ref, bound = oracle.sparse_gemv(codes, s, z, m, n, x, np.arange(n, dtype=np.int32), bits, group)
    check_y(y_dense.cpu().numpy(), y_ref, bound, "dense")
    assert binding.spqt_workspace_status(ws, m, group) == 0 and int(ws.count_nonzero()) == 0


@pytest.mark.parametrize("bits,group", FORMATS)
@pytest.mark.parametrize("m_blocks,n,pad,shift", [(1, 1, 0, 0), (2, 16, 2, 0), (1, 66, 0, 0), (3, 130, 2, 2), (2, 258, 2, 1), (2, 257, 0, 0), (1, 31, 3, 0)])
def test_conversion_at_the_edges_of_tiles_and_alignments(bits, group, m_blocks, n, pad, shift):
    """Pairs of columns as words, single columns, bytes equal to the oracle's: quotients in the middle between two codes, groups
    over many orders of magnitude, constant ones, scales that are subnormal or round to zero."""
    m = m_blocks * group
    rng = np.random.Generator(np.random.PCG64(m * 1000 + n + bits))
    W = (rng.standard_normal((m, n)) * 10.0 ** rng.uniform(-6, 3, n)).astype(np.float16)
    qmax = (1 << bits) - 1
    ties = rng.integers(0, 2 * qmax + 1, (m, n)) * 0.5   # multiples of half the scale
    ties[::group // 2] = 0.0
    ties[1::group // 2] = qmax
    pick = rng.integers(0, 4, n)
    W = np.where(pick == 1, (ties * 2.0 ** rng.integers(-12, 5, n)).astype(np.float16), W)
    W = np.where(pick == 2, (W * np.logspace(-3, 0, m)[:, None]).astype(np.float16), W)
    W[:, n // 2] = W[0, n // 2]
    buf = torch.zeros(shift + m * (n + pad), dtype=torch.float16, device="cuda")
    Wd = buf[shift:].view(m, n + pad)[:, :n]
    Wd.copy_(dev(np.ascontiguousarray(W)))
    p = binding.spqt_pack(Wd, bits, group)
    codes, s, z = packed_to_host(p)
    ref_codes, ref_s, ref_z = oracle.pack(W, bits, group)
    assert np.array_equal(np.asarray(codes).reshape(-1), np.asarray(ref_codes).reshape(-1))
    assert np.array_equal(s.view(np.uint16).reshape(-1), ref_s.view(np.uint16).reshape(-1))
    assert np.array_equal(z.view(np.uint16).reshape(-1), ref_z.view(np.uint16).reshape(-1))


@pytest.mark.parametrize("bits,group", FORMATS)
@pytest.mark.parametrize("m_blocks,n,pad,shift", [(1, 1, 7, 0), (1, 8, 0, 0), (2, 31, 1, 8), (3, 33, 7, 0), (1, 64, 0, 8), (2, 65, 7, 0), (99, 997, 3, 0)])
def test_conversion_in_tiles(bits, group, m_blocks, n, pad, shift):
    """Rows of 16-byte pieces: ragged and odd widths, and more tiles than the persistent warps take at once."""
    test_conversion_at_the_edges_of_tiles_and_alignments(bits, group, m_blocks, n, pad, shift)


@pytest.mark.parametrize("bits", [2, 4, 5, 6, 8])
@pytest.mark.parametrize("m_blocks,n,pad,shift", [(1, 1, 0, 0), (2, 64, 2, 0), (1, 66, 0, 0), (2, 130, 2, 1), (2, 129, 0, 0), (1, 31, 3, 0)])
def test_two_level_conversion_at_the_edges_of_tiles_and_alignments(bits, m_blocks, n, pad, shift):
    """As above; blocks of one sign, of zeros, and of very different sizes in one superblock."""
    m = 256 * m_blocks
    rng = np.random.Generator(np.random.PCG64(m * 1000 + n + bits))
    W = rng.standard_normal((m, n)) * 10.0 ** rng.uniform(-4, 2, n) * np.repeat(10.0 ** rng.uniform(-2, 0, (m // 32, n)), 32, axis=0)
    pick = rng.integers(0, 5, n)
    W = np.where(pick == 1, np.abs(W), np.where(pick == 2, -np.abs(W), np.where(pick == 3, np.round(W * 8) / 8, W))).astype(np.float16)
    W[32:64, n // 2] = 0.0
    buf = torch.zeros(shift + m * (n + pad), dtype=torch.float16, device="cuda")
    Wd = buf[shift:].view(m, n + pad)[:, :n]
    Wd.copy_(dev(np.ascontiguousarray(W)))
    got = binding.spqt_kqw_pack(Wd, bits).records.cpu().numpy()
    want = oracle.kq_pack(*oracle.kq_quantize(W, bits=bits), bits=bits)
    assert np.array_equal(got, np.asarray(want).reshape(-1))


@pytest.mark.parametrize("bits", [2, 4, 5, 6, 8])
@pytest.mark.parametrize("m_blocks,n", [(1, 1), (2, 17), (1, 2049), (20, 300), (37, 1030), (60, 264), (101, 129), (149, 40), (3, 16421)])
def test_two_level_products_at_chunk_part_and_cluster_edges(bits, m_blocks, n):
    m = 256 * m_blocks
    W = inputs.weights(m, n, seed=m + n, std=0.1)
    x = growing_activations(n, seed=91)
    parts = oracle.kq_quantize(W, bits=bits)
    p = binding.spqt_kqw_pack(dev(W), bits)
    ws = binding.new_kq_workspace(p)
    t = inputs.threshold_for_sparsity(x, 0.4)
    xd = dev(x)
    idx, cnt = binding.spqt_sparsify(xd, t)
    y = binding.spqt_kqw_sparse_gemv(p, xd, idx, cnt, ws)
    again = binding.spqt_kqw_sparse_gemv(p, xd, idx, cnt, ws)
    y_dense = binding.spqt_kqw_dense_gemv(p, xd, ws)
    torch.cuda.synchronize()
    ref_idx, _ = oracle.sparsify(x, t)
    y_ref, bound = oracle.kq_gemv(*parts, x, ref_idx)
    check_y(y.cpu().numpy(), y_ref, bound, "sparse")
    assert torch.equal(y, again)
    y_ref, bound = oracle.kq_gemv(*parts, x)
    check_y(y_dense.cpu().numpy(), y_ref, bound, "dense")


def test_two_level_sparse_product_refuses_a_missing_list():
    p = binding.spqt_kqw_pack(dev(inputs.weights(256, 64, seed=3)), 4)
    x, ws = dev(inputs.activations(64, seed=4)), binding.new_kq_workspace(p)
    idx, cnt = binding.spqt_sparsify(x, 0.5)
    before = binding.spqt_launch_count()
    for product in (binding.spqt_kqw_sparse_gemv, binding.spqt_kq_sparse_gemv):
        for i, c in ((None, None), (idx, None), (None, cnt)):
            with pytest.raises(TypeError):
                product(p, x, i, c, ws)
    assert binding.spqt_launch_count() == before


@pytest.mark.parametrize("bits,m_blocks,n", [(8, 1, 16384), (4, 1, 60001), (4, 3, 16421), (2, 4, 28672)])
def test_two_level_products_leave_the_workspace_zero(bits, m_blocks, n):
    """Several clusters of a block-row: their sums lie where a shape with more block-rows has its counters."""
    p = binding.spqt_kqw_pack(dev(inputs.weights(256 * m_blocks, n, seed=n)), bits)
    x, ws = dev(inputs.activations(n, seed=5)), binding.new_kq_workspace(p)
    idx, cnt = binding.spqt_sparsify(x, 0.5)
    for _ in range(2):
        y, y_dense = binding.spqt_kqw_sparse_gemv(p, x, idx, cnt, ws), binding.spqt_kqw_dense_gemv(p, x, ws)
        assert int(ws.count_nonzero()) == 0
    assert torch.equal(y, binding.spqt_kqw_sparse_gemv(p, x, idx, cnt, ws)) and torch.equal(y_dense, binding.spqt_kqw_dense_gemv(p, x, ws))


def random_matrix(bits, group, m_blocks, n):
    """Any bytes are a packed matrix: quick for large ones."""
    rng = np.random.Generator(np.random.PCG64(m_blocks * group + n))
    codes = rng.integers(0, 256, binding.spqt_packed_sizes(m_blocks * group, n, bits, group).codes_bytes, dtype=np.uint8)
    pairs = np.stack([rng.uniform(0.001, 0.01, m_blocks * n), rng.uniform(-0.1, 0.0, m_blocks * n)], axis=1).astype(np.float16)
    p = binding.Packed(dev(codes), dev(pairs.reshape(-1)), m_blocks * group, n, bits, group)
    return (p, codes) + tuple(np.ascontiguousarray(pairs[:, i]).reshape(m_blocks, n) for i in (0, 1))


@pytest.mark.parametrize("bits,group,m_blocks,n,batch", [(4, 64, 101, 8192, 3), (3, 128, 100, 8193, 8), (4, 128, 36, 4097, 5), (3, 64, 99, 1536, 4)])
def test_small_batch_at_the_lines_between_cluster_sizes(bits, group, m_blocks, n, batch):
    p, codes, s, z = random_matrix(bits, group, m_blocks, n)
    X = np.stack([growing_activations(n, seed=93 + b) for b in range(batch)])
    ws = binding.new_gemm_small_workspace(p)
    t = inputs.threshold_for_sparsity(X[0], 0.4)
    Y, idx, cnt = binding.spqt_sparse_gemm_small(p, dev(X), t, ws)
    Yd = binding.spqt_dense_gemm_small(p, dev(X), ws)
    ref_idx, ref_cnt = oracle.union_sparsify(X, t)
    assert int(cnt.item()) == ref_cnt and np.array_equal(idx.cpu().numpy()[:ref_cnt], ref_idx)
    Y_ref, bound = oracle.sparse_gemm_small(codes, s, z, p.m, n, X, ref_idx, bits, group)
    for b in range(batch):
        check_y(Y.cpu().numpy()[b], Y_ref[b], bound[b], "row %d" % b)
        check_y(Yd.cpu().numpy()[b], *oracle.dense_gemv(codes, s, z, p.m, n, X[b], bits, group), "dense row %d" % b)


@pytest.mark.parametrize("bits,group,m_blocks,n", [(4, 128, 92, 9505), (4, 64, 95, 20049), (3, 128, 90, 5665), (3, 64, 92, 11720), (4, 128, 301, 2048),
                                                   (3, 64, 150, 4501), (3, 128, 298, 3072), (3, 64, 32, 28672), (3, 64, 33, 22001), (4, 64, 36, 20485)])
def test_pieces_where_the_last_round_of_block_rows_leaves_sms_idle(bits, group, m_blocks, n):
    """Equal pieces with fewer block-rows than SMs (a block-row's sums come from up to three CTAs) and with little more than one
    or two rounds of them; each just above its line.  The last three: clusters of 24-byte blocks up to the least that a long
    x needs, pieces one block-row further on, and an odd cluster that nearly fills the device."""
    p, codes, s, z = random_matrix(bits, group, m_blocks, n)
    m = p.m
    x = growing_activations(n, seed=92)
    ws = binding.new_workspace(m, n, bits, group)
    t = inputs.threshold_for_sparsity(x, 0.4)
    y, idx, cnt = binding.spqt_sparsify_gemv(p, dev(x), t, ws)
    y_list = binding.spqt_sparse_gemv(p, dev(x), idx, cnt, ws)
    y_dense = binding.spqt_dense_gemv(p, dev(x), ws)
    again = binding.spqt_dense_gemv(p, dev(x), ws)
    ref_idx, ref_cnt = oracle.sparsify(x, t)
    assert int(cnt.item()) == ref_cnt and np.array_equal(idx.cpu().numpy()[:ref_cnt], ref_idx)
    check_y(y.cpu().numpy(), *oracle.sparse_gemv(codes, s, z, m, n, x, ref_idx, bits, group), "list collected")
    assert torch.equal(y, y_list) and torch.equal(y_dense, again)
    check_y(y_dense.cpu().numpy(), *oracle.dense_gemv(codes, s, z, m, n, x, bits, group), "dense")
    assert int(ws.count_nonzero()) == 0


@pytest.mark.parametrize("word", [1, 2])
def test_status_words_of_other_shapes_are_not_taken_for_sums(word):
    """A word that is no sum, where CTAs' sums meet, does not get into y; nor does what the built-in scratch still holds."""
    bits, group, m_blocks, n = 3, 64, 33, 22001   # pieces
    p, _, _, _ = random_matrix(bits, group, m_blocks, n)
    x = dev(growing_activations(n, seed=94))
    idx, cnt = binding.spqt_sparsify(x, 0.5)
    want = binding.spqt_sparse_gemv(p, x, idx, cnt, binding.new_workspace(p.m, n, bits, group))
    ws = binding.new_workspace(p.m, n, bits, group)
    ws.view(torch.int32)[64::7] = word
    assert torch.equal(binding.spqt_sparse_gemv(p, x, idx, cnt, ws), want)
    assert torch.equal(binding.spqt_sparse_gemv_static(p, x, idx, cnt, torch.empty_like(want)), want)


def test_status_word_survives_calls_of_other_shapes():
    """One workspace for a shape with more block-rows, whose list checked mode refuses, and one with fewer that CTAs share in pieces:
    the status stays until the workspace is zeroed, and the sums have other places."""
    bits, group = 3, 64
    many, few = random_matrix(bits, group, 150, 512)[0], random_matrix(bits, group, 33, 22001)[0]
    ws = torch.zeros(max(w.numel() for w in (binding.new_workspace(p.m, p.n, bits, group) for p in (many, few))), dtype=torch.uint8, device="cuda")
    x = dev(growing_activations(few.n, seed=95))
    idx, cnt = binding.spqt_sparsify(x, 0.5)
    want = binding.spqt_sparse_gemv(few, x, idx, cnt, ws)
    assert int(ws.count_nonzero()) == 0
    binding.spqt_set_debug(True)
    try:
        binding.spqt_sparse_gemv(many, x[:512].clone(), torch.full((512,), 3, dtype=torch.int32, device="cuda"), torch.full((1,), 2, dtype=torch.int32, device="cuda"), ws)
    finally:
        binding.spqt_set_debug(False)
    for _ in range(2):
        assert binding.spqt_workspace_status(ws, many.m, group) == 2 and binding.spqt_workspace_status(ws, few.m, group) == 2
        assert torch.equal(binding.spqt_sparse_gemv(few, x, idx, cnt, ws), want)


@pytest.mark.parametrize("length", [-1, -9, -2 ** 31])
def test_list_without_a_length_gives_not_a_number(length):
    """What the index collection leaves if it finds no places: block-rows in clusters, whole, in pieces, and of the two-level format
    in one cluster and in several; the next call is as if nothing had been."""
    cnt = torch.full((1,), length, dtype=torch.int32, device="cuda")
    for bits, group, m_blocks, n in [(4, 128, 8, 4096), (4, 64, 300, 512), (3, 64, 33, 22001)]:
        p = random_matrix(bits, group, m_blocks, n)[0]
        ws, x, idx = binding.new_workspace(p.m, n, bits, group), dev(inputs.activations(n, seed=96)), torch.zeros(n, dtype=torch.int32, device="cuda")
        assert bool(binding.spqt_sparse_gemv(p, x, idx, cnt, ws).isnan().all())
        assert binding.spqt_workspace_status(ws, p.m, group) == 1
        assert bool((binding.spqt_sparse_gemv(p, x, idx, cnt * 0, ws) == 0).all())
    for bits, m_blocks, n in [(4, 8, 512), (8, 4, 28672), (5, 300, 64)]:
        p = binding.spqt_kqw_pack(dev(inputs.weights(256 * m_blocks, n, seed=6)), bits)
        ws, x, idx = binding.new_kq_workspace(p), dev(inputs.activations(n, seed=97)), torch.zeros(n, dtype=torch.int32, device="cuda")
        assert bool(binding.spqt_kqw_sparse_gemv(p, x, idx, cnt, ws).isnan().all()) and int(ws.count_nonzero()) == 0
        assert bool((binding.spqt_kqw_sparse_gemv(p, x, idx, cnt * 0, ws) == 0).all())


@pytest.mark.parametrize("n", [1, 63, 64, 65, 2047, 2048, 2049, 4096, 4097, 8192, 16385, 32768, 32769, 49152, 49153, 65535, 65536, 65537])
def test_index_collection_at_word_and_cluster_edges(n):
    """One CTA, a cluster with 1 to 16 words per lane, and beyond; x on an odd boundary too; entries and thresholds that are
    extreme, infinite or no numbers."""
    x = inputs.activations(n, seed=n)
    rng = np.random.Generator(np.random.PCG64(n))
    for value in (np.nan, np.inf, -np.inf, -0.0, 6e-8, 65504.0, -0.5):
        x[rng.integers(0, n, max(1, n // 50))] = value
    for shift in (0, 1):
        buf = torch.full((n + shift + 8,), float("inf"), dtype=torch.float16, device="cuda")   # (active, if it were read)
        xd = buf[shift:shift + n]
        xd.copy_(dev(x))
        for t in (0.5, 0.0, -0.0, -1.0, 3e-8, 0.4999, 65504.0, 1e6, float("inf"), float("nan")):
            idx, cnt = binding.spqt_sparsify(xd, t)
            ref_idx, ref_cnt = oracle.sparsify(x, t)
            assert int(cnt.item()) == ref_cnt and np.array_equal(idx.cpu().numpy()[:ref_cnt], ref_idx), (shift, t)


@pytest.mark.parametrize("shared", [False, True])
def test_recorded_step_in_branches(shared):
    """More linears than a step has branches, of all formats, one with a list of its own launch; also where linears write their
    lists to the same place."""
    sizes = [(4, 128, 8, 512), (3, 64, 33, 1030), (4, 64, 149, 260), (3, 128, 5, 2049), (4, 128, 2, 33000), (4, 128, 40, 300), (3, 64, 150, 4501)]
    linears = []
    for i, (bits, group, m_blocks, n) in enumerate(sizes):
        p = random_matrix(bits, group, m_blocks, n)[0]
        h = binding.HostLinear(p)
        if shared and i > 0 and h.idx.numel() <= linears[0].idx.numel():
            h.idx, h.count = linears[0].idx, linears[0].count
        linears.append(h)
    if shared:
        linears[1].count = linears[0].count
    ts = [0.4 + 0.05 * i for i in range(len(linears))]
    step = binding.HostStep(linears, ts)
    for replay in range(3):
        for i, h in enumerate(linears):
            h.x_host.copy_(torch.from_numpy(inputs.activations(h.p.n, seed=100 * replay + i)))
            h.y_host.zero_()
        step.launch()
        torch.cuda.synchronize()
        for h, t in zip(linears, ts):
            y, _, _ = binding.spqt_sparsify_gemv(h.p, h.x_host.cuda(), t, binding.new_workspace(h.p.m, h.p.n, h.p.bits, h.p.group))
            assert torch.equal(y.cpu(), h.y_host)
            assert int(h.workspace.count_nonzero()) == 0


def test_calls_behind_one_another_see_what_the_previous_one_wrote():
    """Every call starts while the previous one of the stream drains: a list, its length and x that the previous call has just
    written, other ones each time, give what the same calls give one at a time."""
    m = n = 2048
    W = inputs.weights(m, n, seed=5, std=n ** -0.5)   # (y is about as large as x)
    p, pr, pk = pack_on_gpu(W, 4, 128), binding.spqt_rowwise_pack(dev(W), 4, 128), binding.spqt_kqw_pack(dev(W), 6)
    ws, wk, wsm = binding.new_workspace(m, n), binding.new_kq_workspace(pk), binding.new_gemm_small_workspace(p)
    idx, cnt = torch.empty(n, dtype=torch.int32, device="cuda"), torch.empty(1, dtype=torch.int32, device="cuda")
    Y = torch.empty((5, 2, m), dtype=torch.float16, device="cuda")
    starts = dev(np.stack([inputs.activations(n, seed=80 + i) for i in range(12)]))

    def chain(wait):
        """Products whose x is the y of the call before; lists that are collected over and over into the same places."""
        outs = []

        def call(f, *a, **k):
            r = f(*a, **k)
            if wait:
                torch.cuda.synchronize()
            return r

        for i, x in enumerate(starts):
            t = 0.1 + 0.05 * (i % 5)
            call(binding.spqt_sparsify, x, t, idx, cnt)
            a = call(binding.spqt_sparse_gemv, p, x, idx, cnt, ws)
            call(binding.spqt_sparsify, a, 2 * t, idx, cnt)
            b = call(binding.spqt_kqw_sparse_gemv, pk, a, idx, cnt, wk)
            c = call(binding.spqt_dense_gemv, p, b, ws)
            d = call(binding.spqt_kqw_dense_gemv, pk, c, wk)
            e = call(binding.spqt_rowwise_dense_gemv, pr, d)
            f = call(binding.spqt_sparsify_gemv, p, e, t, ws, idx=idx, count=cnt)[0]
            Z = Y[i % 5]
            call(binding.spqt_dense_gemv, p, f, ws, y=Z[0])
            call(binding.spqt_dense_gemv, p, a, ws, y=Z[1])
            g = call(binding.spqt_sparse_gemm_small, p, Z, t, wsm, idx=idx, count=cnt)[0]
            h = call(binding.spqt_dense_gemm_small, p, g, wsm)
            outs += [a, b, c, d, e, f, g, h]
        torch.cuda.synchronize()
        return outs

    want = chain(True)
    assert all(bool(v.isfinite().all()) and float(v.float().std()) > 1e-2 for v in want)
    for got in (chain(False), chain(False)):
        assert all(torch.equal(a, b) for a, b in zip(want, got))


@pytest.mark.parametrize("shared", ["idx", "count", "workspace", "y_host"])
def test_recorded_step_keeps_the_order_of_linears_with_a_buffer_in_common(shared):
    """Linear 5, whose predecessors in a branch of its own would be quick, has a buffer in common with linear 4, which a large one
    would hold up: what the buffer holds in the end, and what the linears read from it meanwhile, is as in the order given."""
    sizes = [(4, 128, 400, 8192)] + 3 * [(4, 128, 2, 256)] + 2 * [(3, 64, 33, 33001)] + [(4, 64, 3, 300)]
    linears = [binding.HostLinear(random_matrix(*size)[0]) for size in sizes]
    setattr(linears[5], shared, getattr(linears[4], shared))
    ts = [0.6] * 4 + [1.5, 0.3, 0.6]
    xs = [inputs.activations(h.p.n, seed=110 + i) for i, h in enumerate(linears)]
    for h, x in zip(linears, xs):
        h.x_host.copy_(torch.from_numpy(x))
    step = binding.HostStep(linears, ts)
    for _ in range(5):
        for h in linears:
            h.y_host.zero_()
        step.launch()
        torch.cuda.synchronize()
        for i, (h, x, t) in enumerate(zip(linears, xs, ts)):
            y, idx, cnt = binding.spqt_sparsify_gemv(h.p, dev(x), t, binding.new_workspace(h.p.m, h.p.n, h.p.bits, h.p.group))
            if i != 4 or shared != "y_host":
                assert torch.equal(y.cpu(), h.y_host), i
            if i != 4 or shared != "count":
                assert int(h.count) == int(cnt), i
            if i != 4 or shared != "idx":
                assert torch.equal(h.idx[:int(cnt)], idx[:int(cnt)]), i
            assert int(h.workspace.count_nonzero()) == 0


@pytest.mark.parametrize("bits,group,m_blocks,n", [(4, 128, 88, 8200), (3, 128, 53, 14337), (4, 64, 36, 14336), (3, 64, 25, 4099), (4, 128, 24, 4096)])
def test_clusters_that_leave_together(bits, group, m_blocks, n):
    """Clusters that nearly fill the device, calls behind one another."""
    p, codes, s, z = random_matrix(bits, group, m_blocks, n)
    m, ws = p.m, binding.new_workspace(p.m, n, bits, group)
    x = growing_activations(n, seed=98)
    t = inputs.threshold_for_sparsity(x, 0.5)
    y, idx, cnt = binding.spqt_sparsify_gemv(p, dev(x), t, ws)
    ref_idx, ref_cnt = oracle.sparsify(x, t)
    assert int(cnt.item()) == ref_cnt and np.array_equal(idx.cpu().numpy()[:ref_cnt], ref_idx)
    y_dense = binding.spqt_dense_gemv(p, dev(x), ws)
    check_y(y.cpu().numpy(), *oracle.sparse_gemv(codes, s, z, m, n, x, ref_idx, bits, group), "list collected")
    check_y(y_dense.cpu().numpy(), *oracle.dense_gemv(codes, s, z, m, n, x, bits, group), "dense")
    for _ in range(20):
        assert torch.equal(binding.spqt_sparse_gemv(p, dev(x), idx, cnt, ws), y) and torch.equal(binding.spqt_dense_gemv(p, dev(x), ws), y_dense)
    assert binding.spqt_workspace_status(ws, m, group) == 0 and int(ws.count_nonzero()) == 0


@pytest.mark.parametrize("bits,m_blocks,n", [(4, 53, 8192), (8, 36, 4100), (6, 90, 4097), (2, 88, 1537), (5, 52, 2560)])
def test_two_level_clusters_that_leave_together(bits, m_blocks, n):
    m = 256 * m_blocks
    W = inputs.weights(m, n, seed=m + n)
    p, parts = binding.spqt_kqw_pack(dev(W), bits), oracle.kq_quantize(W, bits=bits)
    x, ws = growing_activations(n, seed=99), binding.new_kq_workspace(p)
    idx, cnt = binding.spqt_sparsify(dev(x), 0.5)
    ref_idx, _ = oracle.sparsify(x, 0.5)
    rows = np.unique(np.concatenate([np.arange(0, m, 97), np.arange(256), np.arange(m - 256, m)]))
    y, y_dense = binding.spqt_kqw_sparse_gemv(p, dev(x), idx, cnt, ws), binding.spqt_kqw_dense_gemv(p, dev(x), ws)
    check_y(y.cpu().numpy()[rows], *oracle.kq_gemv(*parts, x, ref_idx, rows=rows), "list")
    check_y(y_dense.cpu().numpy()[rows], *oracle.kq_gemv(*parts, x, rows=rows), "dense")
    for _ in range(20):
        assert torch.equal(binding.spqt_kqw_sparse_gemv(p, dev(x), idx, cnt, ws), y) and torch.equal(binding.spqt_kqw_dense_gemv(p, dev(x), ws), y_dense)
