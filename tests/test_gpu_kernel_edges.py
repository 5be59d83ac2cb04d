"""The kernels that a dispatch chooses among, at the sizes where each can go wrong: edges of tiles and of row groups, remainders,
the smallest and largest of its range.  Attention in float32 I/O against the float64 oracle (the tolerance of one kernel's
arithmetic, see parity_utils); encoders against the codes of the same tokens encoded in other pieces, because every decision is
exact whatever kernel takes it."""
import numpy as np
import pytest
import torch

import paper_2502_02617_b200 as pq
from paper_2502_02617_b200 import synthetic
from oracle import polarquant_oracle as orc
from parity_utils import (TOL_ATTENTION_F32_IO, assert_codes_match, assert_radii_match, code_mismatch_report, oracle_codebooks,
                          radii_ulp_report, rel_l2, to_f64)
from test_gpu_parity import _encode_and_compare, _oracle_cache

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _filled(lens, Hq, Hkv, d, seed, dtype=torch.bfloat16, paged=False, codebooks=None):
    if paged:
        pages = -(-max(lens) // 128)
        table = torch.randperm(len(lens) * pages, generator=torch.Generator().manual_seed(seed)).view(len(lens), pages)
        cache = pq.PagedPolarQuantCache(len(lens), Hq, Hkv, d, 128, len(lens) * pages, table, seed=seed, device=DEV, codebooks=codebooks)
    else:
        cache = pq.PolarQuantCache(len(lens), Hq, Hkv, d, capacity=max(lens), seed=seed, device=DEV, codebooks=codebooks)
    K, V = synthetic.kv_like(seed + 1, sum(lens), Hkv, d, dtype, DEV, n_outliers=4 if d >= 64 else 0)
    cache.encode(K, V, torch.tensor(np.concatenate(([0], np.cumsum(lens))), dtype=torch.int32, device=DEV))
    return cache, _oracle_cache(cache, K, V, lens)


CLUSTER, PERSISTENT, ROWS, TCGEN05 = 6, 7, 8, 9    # pq_debug_fail_next_wait: the next attention call runs this kernel


def _check_multi(cache, ref, q, lens, kernel):
    pq.pq_debug_fail_next_wait(kernel)
    out = to_f64(cache.attend_multi(q))
    n_q = q.shape[1]
    want = orc.multi_query_attention(to_f64(q), ref.k_codes, ref.k_radii, ref.v_codes, ref.v_radii, ref.lens, ref.cb, ref.S, 128 ** -0.5)
    for b in range(len(lens)):
        for j in range(n_q):
            if lens[b] - (n_q - 1 - j) <= 0:
                assert np.all(out[b, j] == 0)
            else:
                assert rel_l2(out[b, j], want[b, j]) < TOL_ATTENTION_F32_IO, (kernel, b, j)


# Rows of a kv head (queries x heads of the group) on both sides of every group of four that the rows kernel is built for
# (8, 12, 16, 20, 24, 32) and beyond one row block, odd groups whose rows do not end with a query; lengths around its 16-token
# tiles and 128-token stages; contiguous and behind a block table.
@pytest.mark.parametrize("paged", [False, True])
@pytest.mark.parametrize("g,n_q", [(1, 1), (1, 5), (1, 8), (1, 9), (4, 3), (1, 13), (8, 2), (1, 17), (5, 4), (7, 3), (6, 4), (1, 25), (7, 4),
                                   (4, 8), (8, 4), (1, 32), (8, 5), (3, 23)])
def test_rows_kernel(g, n_q, paged):
    lens, Hkv = [16, 129, 397, 2, 128], 2
    cache, ref = _filled(lens, g * Hkv, Hkv, 128, 60 + g, paged=paged)
    q = torch.randn((len(lens), n_q, g * Hkv, 128), generator=torch.Generator(device=DEV).manual_seed(n_q), device=DEV)
    _check_multi(cache, ref, q, lens, ROWS)


def test_a_named_kernel_that_does_not_take_the_call_is_refused():
    cache = pq.PolarQuantCache(2049, 2, 1, 128, capacity=64, device=DEV)   # more units than the persistent schedules handle
    q = synthetic.queries(1, 2049, 2, 128, torch.bfloat16, DEV)
    for kernel in (PERSISTENT, ROWS):
        pq.pq_debug_fail_next_wait(kernel)
        with pytest.raises(pq.PolarQuantError) as e:
            cache.attend(q)
        assert e.value.status == pq.ERR_UNSUPPORTED


# The persistent kernel with five to eight heads per kv head, a unit per query, both cache layouts.
@pytest.mark.parametrize("paged", [False, True])
@pytest.mark.parametrize("g,n_q", [(5, 3), (8, 5), (7, 12)])
def test_persistent_kernel_with_two_groups_of_heads(g, n_q, paged):
    lens, Hkv = [16, 129, 1397, 12, 128], 2
    cache, ref = _filled(lens, g * Hkv, Hkv, 128, 40 + g, paged=paged)
    q = torch.randn((len(lens), n_q, g * Hkv, 128), generator=torch.Generator(device=DEV).manual_seed(n_q), device=DEV)
    _check_multi(cache, ref, q, lens, PERSISTENT)


# The tcgen05 kernel: an odd count of 64-token blocks (half of a tile pair), fewer blocks than ranges (empty parts), more rows than
# one pair of CTAs holds, a group size that leaves rows of the 128 unused, and 64-row tiles in the rotation kernels.
@pytest.mark.parametrize("g,Hkv,n_q,lens", [(8, 1, 16, [1, 64, 65, 700]), (7, 2, 19, [1473, 40]), (4, 1, 70, [1000, 71, 64]),
                                            (8, 8, 75, [90, 75, 300, 65, 76, 80, 91, 99]), (4, 2, 8, [130] * 64), (1, 1, 32, [64, 3])])
def test_tcgen05_multi_query_kernel_parts(g, Hkv, n_q, lens):
    cache, ref = _filled(lens, g * Hkv, Hkv, 128, 70 + g)
    q = torch.randn((len(lens), n_q, g * Hkv, 128), generator=torch.Generator(device=DEV).manual_seed(n_q), device=DEV)
    _check_multi(cache, ref, q, lens, TCGEN05)


# The cluster kernel: lengths around its 16-token tiles, a warp without tokens, one head and every padding of the heads of a group;
# at head_dim 128 the persistent kernel (both instantiations) and the rows kernel on the same.
@pytest.mark.parametrize("d,g", [(128, 1), (128, 3), (128, 5), (128, 8), (64, 2), (64, 7), (32, 4), (16, 1), (16, 8)])
def test_single_query_kernels(d, g):
    lens, Hkv = [1, 15, 16, 17, 63, 64, 65, 255, 257, 1025], 2
    cache, ref = _filled(lens, g * Hkv, Hkv, d, 80 + g, torch.float32)
    q = synthetic.queries(5, len(lens), g * Hkv, d, torch.float32, DEV)
    want = ref.attend(to_f64(q), d ** -0.5)
    for kernel in (0,) if d < 128 else (CLUSTER, PERSISTENT, ROWS):
        pq.pq_debug_fail_next_wait(kernel)
        out = to_f64(cache.attend(q))
        for b in range(len(lens)):
            assert rel_l2(out[b], want[b]) < TOL_ATTENTION_F32_IO, (kernel, lens[b])


# The tensor-core encoder where a group's queue of uncertified decisions fills up again and again (zero rows, rows on the boundaries of an
# unrotated codebook), at every number of tiles that its three groups of warps can be left with, against the float32 encoder: the same
# codes and status counts, radii that are neighbours at most.  One to six tiles per CTA: the last of one or four is shared by two groups.
@pytest.mark.parametrize("n", [128, 129, 640, 1700, 2500, 4700, 6000])
@pytest.mark.parametrize("analytic", [True, False])
def test_tensor_core_encoder_with_many_uncertified_decisions(n, analytic):
    Hkv = 8
    K, V = synthetic.kv_like(n, n, Hkv, 128, torch.bfloat16, DEV)
    K[::3] = 0
    V[5:90] = 1.0
    cen, bnd = (t.clone() for t in pq.pq_fit_codebooks())
    if not analytic:
        cen[:16] += 0.01 * torch.cos(torch.arange(16, dtype=torch.float64))
        bnd[:15] = 0.5 * (cen[:15] + cen[1:16])
    cu = torch.tensor([0, n], dtype=torch.int32, device=DEV)
    got = []
    for dtype in (torch.bfloat16, torch.float32):
        c = pq.PolarQuantCache(1, Hkv, Hkv, 128, capacity=n, S=torch.eye(128), device=DEV, codebooks=(cen, bnd))
        c.encode(K.to(dtype), V.to(dtype), cu)
        got.append((*c.unpack(n), c.status[:3].tolist()))
    assert torch.equal(got[0][0], got[1][0]) and got[0][2] == got[1][2]
    assert torch.all((got[0][1].float() - got[1][1].float()).abs() <= 2.0 ** -10 * got[1][1].float())


# Codebooks without the symmetries of the analytic one: every level moved, or the top level alone, in the three kernels that read the decode
# tables.
@pytest.mark.parametrize("moved", [slice(0, 28), slice(24, 28)])
@pytest.mark.parametrize("g,paged", [(4, False), (4, True), (7, False)])
def test_attention_with_codebooks_that_are_not_analytic(g, paged, moved):
    cen, bnd = (t.clone() for t in pq.pq_fit_codebooks())
    cen[moved] += 0.01 * torch.cos(torch.arange(28, dtype=torch.float64))[moved]
    for c0, b0, n in ((0, 0, 16), (16, 15, 4), (20, 18, 4), (24, 21, 4)):
        bnd[b0:b0 + n - 1] = 0.5 * (cen[c0:c0 + n - 1] + cen[c0 + 1:c0 + n])
    lens, Hkv = [1, 15, 16, 17, 127, 129, 1025], 2
    cache, ref = _filled(lens, g * Hkv, Hkv, 128, 30 + g, paged=paged, codebooks=(cen, bnd))
    for n_q, kernels in ((1, (PERSISTENT, ROWS)), (16, (TCGEN05,))):
        q = torch.randn((len(lens), n_q, g * Hkv, 128), generator=torch.Generator(device=DEV).manual_seed(g), device=DEV)
        for kernel in kernels:
            _check_multi(cache, ref, q, lens, kernel)


# The rotations around several queries take 8, 16, 32 or 64 rows per block: one sequence of 64 rows on both sides of where each begins,
# and a number of rows that leaves a remainder of every tile.
@pytest.mark.parametrize("per_sm,more", [(8, 0), (8, 1), (16, 1), (32, 0), (32, 1)])
@pytest.mark.parametrize("kernel,n_q", [(ROWS, 16), (TCGEN05, 16), (ROWS, 15)])
def test_rotations_of_many_rows(kernel, n_q, per_sm, more):
    B = per_sm * torch.cuda.get_device_properties(0).multi_processor_count // 64 + more
    lens = [1 + 7 * b % 40 for b in range(B)]
    cache, ref = _filled(lens, 4, 1, 128, 80)
    q = torch.randn((B, n_q, 4, 128), generator=torch.Generator(device=DEV).manual_seed(n_q), device=DEV)
    _check_multi(cache, ref, q, lens, kernel)


# Scores of a few hundred: an error of the keys' factors that a softmax over small scores hides moves the log-sum-exp by its share of them.
# Keys and queries are fp16 values with fp16 residuals, 22 bits of each coordinate: 2^-22 of sum |q_i||k_i| <= |q||k| for each of the
# two, and the float32 sums of the score take as much again.
@pytest.mark.parametrize("g", [4, 8])
@pytest.mark.parametrize("fitted", [False, True])
def test_large_scores_keep_the_precision_of_keys_and_queries(g, fitted):
    cen, bnd = (t.clone() for t in pq.pq_fit_codebooks())
    if fitted:
        cen[:16] += 0.01 * torch.cos(torch.arange(16, dtype=torch.float64))
        bnd[:15] = 0.5 * (cen[:15] + cen[1:16])
    lens, Hkv = [600, 33], 2
    cache, ref = _filled(lens, g * Hkv, Hkv, 128, 70 + g, codebooks=(cen, bnd))
    q = 16 * synthetic.queries(5, len(lens), g * Hkv, 128, torch.float32, DEV)
    for kernel in (PERSISTENT, ROWS):
        pq.pq_debug_fail_next_wait(kernel)
        _, lse = cache.attend_lse(q)
        for b in range(len(lens)):
            for h in range(g * Hkv):
                K, qh = orc.dequant(ref.k_codes[b, h // g, :lens[b]], ref.k_radii[b, h // g, :lens[b]], ref.cb, ref.S), to_f64(q[b, h])
                bound = 2.0 ** -20 * np.linalg.norm(qh) * np.linalg.norm(K, axis=1).max() * 128 ** -0.5
                assert abs(float(lse[b, h]) - orc.log_sum_exp_scores(qh, K, 128 ** -0.5)) < bound, (kernel, b, h)


# One or two units of a longer sequence: clusters of sixteen blocks (the limit), also where a block un-rotates one coordinate.
@pytest.mark.parametrize("d,g,Hkv", [(128, 1, 1), (128, 8, 2), (64, 4, 1), (32, 2, 2), (16, 1, 1), (16, 8, 1)])
def test_cluster_kernel_with_sixteen_blocks(d, g, Hkv):
    lens = [4101]
    cache, ref = _filled(lens, g * Hkv, Hkv, d, 90 + g, torch.float32)
    q = synthetic.queries(5, 1, g * Hkv, d, torch.float32, DEV)
    if d == 128:
        pq.pq_debug_fail_next_wait(CLUSTER)
    assert rel_l2(to_f64(cache.attend(q)), ref.attend(to_f64(q), d ** -0.5)) < TOL_ATTENTION_F32_IO


# Calls below 32 tokens have a kernel of their own (one block per sequence), larger ones tiles of 64 rows (float32 or d < 128)
# or of 128 (bf16, d = 128): the same codes whatever pieces the tokens come in, and the first piece against the oracle.  The radii
# are float32 sums in another order before they are rounded to fp16: neighbours at most, 2^-10 apart.
@pytest.mark.parametrize("d,dtype", [(128, torch.bfloat16), (128, torch.float32), (64, torch.bfloat16), (32, torch.float32), (16, torch.bfloat16)])
def test_encoders_give_the_same_codes_in_any_pieces(d, dtype):
    Hkv, pieces = 3, [31, 1, 32, 2, 17, 63, 65, 16, 15, 129, 3]
    n = sum(pieces)
    K, V = synthetic.kv_like(90 + d, n, Hkv, d, dtype, DEV, n_outliers=4 if d >= 64 else 0)
    V[7] = 0                                                    # a zero vector
    whole, cut = (pq.PolarQuantCache(1, Hkv, Hkv, d, capacity=n, seed=6, device=DEV) for _ in range(2))
    whole.encode(K, V, torch.tensor([0, n], dtype=torch.int32, device=DEV))
    at = 0
    for m in pieces:
        cut.encode(K[at:at + m], V[at:at + m], torch.tensor([0, m], dtype=torch.int32, device=DEV))
        at += m
    (codes, radii), (codes_cut, radii_cut) = whole.unpack(n), cut.unpack(n)
    assert torch.equal(codes, codes_cut) and cut.lens.tolist() == [n]
    assert torch.all((radii.float() - radii_cut.float()).abs() <= 2.0 ** -10 * radii.float())
    few = pq.PolarQuantCache(2, Hkv, Hkv, d, capacity=32, seed=6, device=DEV)
    _encode_and_compare(few, K[:31], V[:31], [17, 14])          # one launch, odd counts


# head_dim 128 on both sides of four vectors per SM, where bf16 goes on with the tensor cores, of sixteen, where a second pass of the few-rows
# kernel begins, and of 128, where float32 goes on with tiles of 128 rows; the pieces are all few rows.
@pytest.mark.parametrize("dtype,per_sm,Hkv", [(torch.bfloat16, 4, 2), (torch.float32, 16, 4), (torch.float32, 128, 4)])
def test_encoders_on_both_sides_of_the_few_rows_kernel(dtype, per_sm, Hkv):
    edge = per_sm * torch.cuda.get_device_properties(0).multi_processor_count // (2 * Hkv)
    K, V = synthetic.kv_like(17, edge + 1, Hkv, 128, dtype, DEV, n_outliers=4)
    cut = pq.PolarQuantCache(1, Hkv, Hkv, 128, capacity=edge + 1, seed=6, device=DEV)
    for at in range(0, edge + 1, 31):
        m = min(31, edge + 1 - at)
        cut.encode(K[at:at + m], V[at:at + m], torch.tensor([0, m], dtype=torch.int32, device=DEV))
    codes_cut, radii_cut = cut.unpack(edge + 1)
    for n in (edge, edge + 1):
        whole = pq.PolarQuantCache(1, Hkv, Hkv, 128, capacity=n, seed=6, device=DEV)
        whole.encode(K[:n], V[:n], torch.tensor([0, n], dtype=torch.int32, device=DEV))
        codes, radii = whole.unpack(n)
        assert torch.equal(codes, codes_cut[:, :, :, :n]) and whole.lens.tolist() == [n]
        assert torch.all((radii.float() - radii_cut[:, :, :, :n].float()).abs() <= 2.0 ** -10 * radii.float())


# The tensor-core encoder's radii are float32 sums rounded to fp16.  An error of e row norms, sqrt(8) radii, brings e sqrt(8) 2^11 of them
# across a boundary: with the smallest term of S multiplied first e is 0.2 * 2^-24 on average, 0.013 % of the radii are neighbours of
# the exact norm's rounding; with the largest first 0.089 %.
def test_radii_of_the_tensor_core_encoder():
    n, Hkv = 4096, 8
    K, V = synthetic.kv_like(5, n, Hkv, 128, torch.bfloat16, DEV)
    c = pq.PolarQuantCache(1, Hkv, Hkv, 128, capacity=n, seed=0, device=DEV)
    c.encode(K, V, torch.tensor([0, n], dtype=torch.int32, device=DEV))
    radii = c.unpack(n)[1][0]                                   # [head, K | V, token, block]
    want = torch.stack([(X.double() @ c.S_host.double().to(DEV)).view(n, Hkv, 8, 16).norm(dim=-1).half() for X in (K, V)], dim=2).permute(1, 2, 0, 3)
    assert (radii != want).double().mean() < 3e-4
    assert torch.all((radii.float() - want.float()).abs() <= 2.0 ** -10 * want.float())


# What is stored for a row with a non-finite input does not depend on which kernel takes the call: bf16 calls of 128 tokens and more are the
# tensor-core encoder's or, up to four vectors per SM, the few-rows kernel's, and store the zero vector; tiles of 128 rows (float32, or
# bf16 rows that are not aligned, above 128 vectors per SM) store what the arithmetic gives, as fewer tokens do.  The other rows are the
# ones of a clean call, the elements are counted.
@pytest.mark.parametrize("dtype,per_sm,Hkv,pad", [(torch.bfloat16, 4, 2, 0), (torch.float32, 128, 8, 0), (torch.bfloat16, 128, 8, 1)])
def test_rows_that_are_not_finite_on_both_sides_of_the_few_rows_kernel(dtype, per_sm, Hkv, pad):
    edge = per_sm * torch.cuda.get_device_properties(0).multi_processor_count // (2 * Hkv)
    for n in (edge, edge + 1):
        K, V = synthetic.kv_like(19, n, Hkv, 128, dtype, DEV)
        got = []
        for spoilt in (False, True):
            if spoilt:
                K[3, 0, 5], V[n - 4, 1, 6], V[n - 4, 1, 7] = float("nan"), float("inf"), float("-inf")
            k, v = (torch.nn.functional.pad(t, (0, pad))[..., :128] for t in (K, V))
            c = pq.PolarQuantCache(1, Hkv, Hkv, 128, capacity=n, seed=6, device=DEV)
            c.encode(k, v, torch.tensor([0, n], dtype=torch.int32, device=DEV))
            got.append((*(t.movedim(3, 0) for t in c.unpack(n)), c.status.tolist()))
        (codes, radii, status), (codes_bad, radii_bad, status_bad) = got
        assert status[:2] == [0, 0] and status_bad[:2] == [pq.ERR_NONFINITE, 3]
        if dtype == torch.bfloat16 and pad == 0:
            assert status_bad[2] == 0
            for bad in ((3, 0, 0, 0), (n - 4, 0, 1, 1)):
                assert not codes_bad[bad].any() and not radii_bad[bad].any()
        keep = torch.ones(codes.shape[:4], dtype=torch.bool, device=DEV)
        keep[3, 0, 0, 0] = keep[n - 4, 0, 1, 1] = False
        assert torch.equal(codes[keep], codes_bad[keep]) and torch.equal(radii[keep], radii_bad[keep])


# bf16 rows that do not begin on 16-byte boundaries, in more passes than the few-rows kernel takes: tiles of 128 rows, whose float64
# decisions read the rows again.  The same codes as from the same rows in one piece, radii that are neighbours at most.
@pytest.mark.parametrize("pad,shift", [(1, 0), (4, 0), (0, 1), (0, 4)])
def test_encode_of_many_rows_that_are_not_aligned(pad, shift):
    Hkv, n = 8, 1300
    K, V = synthetic.kv_like(23, n, Hkv, 128, torch.bfloat16, DEV, n_outliers=4)
    K[::5], V[3::7] = 1.0, 0.0
    moved = []
    for t in (K, V):
        t = torch.nn.functional.pad(t, (0, pad))
        whole = torch.empty(t.numel() + shift, dtype=t.dtype, device=DEV)
        moved.append(whole[shift:].view(t.shape).copy_(t)[..., :128])
    got = []
    for k, v in ((K, V), moved):
        c = pq.PolarQuantCache(1, Hkv, Hkv, 128, capacity=n, seed=6, device=DEV)
        c.encode(k, v, torch.tensor([0, n], dtype=torch.int32, device=DEV))
        got.append((*c.unpack(n), c.status[:3].tolist()))
    assert n * 2 * Hkv > 128 * torch.cuda.get_device_properties(0).multi_processor_count
    assert torch.equal(got[0][0], got[1][0]) and got[0][2] == got[1][2]
    assert torch.all((got[0][1].float() - got[1][1].float()).abs() <= 2.0 ** -10 * got[1][1].float())


@pytest.mark.parametrize("d,bits", [(128, (3,) * 7), (64, (4, 2)), (16, (2,) * 4)])
def test_general_encoder_writes_the_same_bytes_in_any_pieces(d, bits):
    # up to 3072 or 4096 vectors a block each, in float64; above them tiles of 16 to 256 vectors
    Hkv, pieces = 3, [1, 20, 21, 22, 43, 64, 2, 700, 701]
    n = sum(pieces)
    K, V = synthetic.kv_like(95 + d, n, Hkv, d, torch.float32, DEV, n_outliers=4 if d >= 64 else 0)
    whole, cut = (pq.GeneralPolarQuantCache(1, Hkv, Hkv, d, bits, n, seed=6, device=DEV) for _ in range(2))
    whole.encode(K, V, torch.tensor([0, n], dtype=torch.int32, device=DEV))
    at = 0
    for m in pieces:
        cut.encode(K[at:at + m], V[at:at + m], torch.tensor([0, m], dtype=torch.int32, device=DEV))
        at += m
    assert torch.equal(whole.cache, cut.cache)


# Rows in bf16 are rotated on tensor cores where there are enough of them, the same values in float32 by multiply-adds: every decision
# and every radius is exact, so the bytes are the same.  Head dims of every warp layout of the product, a remainder of its tiles, rows
# that cannot be read 16 bytes at a time, outlier channels, a zero vector and rows near the ends of the float32 range.
@pytest.mark.parametrize("strided", [False, True])
@pytest.mark.parametrize("d,bits,n", [(16, None, 2500), (32, None, 1301), (64, None, 645), (128, (3,) * 7, 333), (256, (4, 2, 2, 2, 2), 167)])
def test_the_encoder_on_tensor_cores_writes_the_bytes_of_the_float32_one(d, bits, n, strided):
    Hkv = 8
    K, V = synthetic.kv_like(d + n, n, Hkv, d, torch.bfloat16, DEV, n_outliers=4 if d >= 64 else 0)
    V[7] = 0
    K[3::17] *= 1e-18
    K[5::19] *= 1e15
    if strided:
        K, V = (torch.nn.functional.pad(t, (0, 1))[..., :d] for t in (K, V))
    cu = torch.tensor([0, n], dtype=torch.int32, device=DEV)
    caches = []
    for dtype in (torch.bfloat16, torch.float32):
        c = (pq.PolarQuantCache(1, Hkv, Hkv, d, capacity=n, seed=6, device=DEV) if bits is None else
             pq.GeneralPolarQuantCache(1, Hkv, Hkv, d, bits, n, seed=6, device=DEV))
        c.cache.zero_()
        c.encode(*((K, V) if dtype == torch.bfloat16 else (K.float(), V.float())), cu)
        caches.append(c)
    assert torch.equal(caches[0].cache, caches[1].cache) and caches[0].status[:3].tolist() == caches[1].status[:3].tolist()


# The product's sums are truncated, so rows whose products all have one sign are its largest errors: columns of S, scaled, with a little of
# another row.  The bytes are those of the float32 path all the same.
@pytest.mark.parametrize("d,bits", [(16, None), (32, None), (64, None), (64, (4, 3, 2)), (128, (3,) * 7), (128, (4, 2, 2, 2)), (256, (4, 2, 2, 2, 2))])
def test_the_encoder_on_tensor_cores_where_its_sums_have_one_sign(d, bits):
    Hkv, n = 8, 40960 // d
    make = lambda: (pq.PolarQuantCache(1, Hkv, Hkv, d, capacity=n, seed=6, device=DEV) if bits is None else
                    pq.GeneralPolarQuantCache(1, Hkv, Hkv, d, bits, n, seed=6, device=DEV))
    c = make()
    K, V = synthetic.kv_like(d + n, n, Hkv, d, torch.bfloat16, DEV, n_outliers=0)
    columns = c.S.t()[torch.arange(n * Hkv, device=DEV) % d].view(n, Hkv, d)
    K, V = ((columns * 3 + amount * t.float()).bfloat16() for t, amount in ((K, 2.0 ** -8), (V, 2.0 ** -4)))
    cu = torch.tensor([0, n], dtype=torch.int32, device=DEV)
    caches = []
    for k, v in ((K, V), (K.float(), V.float())):
        c = make()
        c.cache.zero_()
        c.encode(k, v, cu)
        caches.append(c)
    assert torch.equal(caches[0].cache, caches[1].cache) and caches[0].status[:3].tolist() == caches[1].status[:3].tolist()


# Four coordinates per thread where the pointers allow it, else one.  A weighted mean of three float32 values: 1e-6 is eight
# roundings of 2^-23.
@pytest.mark.parametrize("d,shift", [(16, 0), (16, 1), (128, 0), (128, 3)])
def test_merge_of_parts(d, shift):
    gen = torch.Generator(device=DEV).manual_seed(d + shift)
    parts = torch.randn(3 * 5 * 7 * d + shift, generator=gen, device=DEV)[shift:].view(3, 5, 7, d)
    lse = torch.randn((3, 5, 7), generator=gen, device=DEV)
    lse[1, 2, 3] = -float("inf")                                # a part without tokens
    out, status = torch.empty((5, 7, d), device=DEV), torch.zeros(4, dtype=torch.int32, device=DEV)
    pq.pq_merge_attention(parts, lse, out, status)
    w = torch.softmax(lse.double(), 0)[..., None]
    assert rel_l2(to_f64(out), (w * parts.double()).sum(0).cpu().numpy()) < 1e-6


# Fewer stages of work than SMs: two units of 32 stages (and 7 empty positions each) over 148 blocks leave more than half of the
# blocks without a segment.  They have started the copy of S all the same; the calls in between put other kernels' shared
# memory where it lands.
def test_rows_kernel_with_blocks_that_own_nothing():
    lens, g, Hkv = [4096], 8, 2
    cache, ref = _filled(lens, g * Hkv, Hkv, 128, 31)
    other, _ = _filled([4096], 4, 2, 128, 32)
    q, q4 = synthetic.queries(6, 1, g * Hkv, 128, torch.float32, DEV), synthetic.queries(7, 1, 4, 128, torch.float32, DEV)
    pq.pq_debug_fail_next_wait(PERSISTENT)
    first4 = other.attend(q4)
    outs, outs4 = [], []
    for _ in range(20):
        pq.pq_debug_fail_next_wait(ROWS)
        outs.append(cache.attend(q))
        pq.pq_debug_fail_next_wait(PERSISTENT)
        outs4.append(other.attend(q4))
    assert rel_l2(to_f64(outs[0]), ref.attend(to_f64(q), 128 ** -0.5)) < TOL_ATTENTION_F32_IO
    assert all(torch.equal(o, outs[0]) for o in outs) and all(torch.equal(o, first4) for o in outs4)
    cache.check_status()


# The persistent kernel's ring holds the scratch of the work split and the merge of the segment before when a segment's first copies
# go into it: more units than blocks (several segments per block), some of one stage, repeated on changing neighbours.
def test_persistent_kernel_reuses_its_ring_between_segments():
    rng = np.random.default_rng(5)
    lens, Hkv = [int(x) for x in rng.integers(1, 400, size=60)] + [2000], 8
    cache, ref = _filled(lens, 4 * Hkv, Hkv, 128, 33)
    q = synthetic.queries(8, len(lens), 4 * Hkv, 128, torch.float32, DEV)
    outs = []
    for _ in range(10):
        pq.pq_debug_fail_next_wait(PERSISTENT)
        outs.append(cache.attend(q))
    assert all(torch.equal(o, outs[0]) for o in outs)
    out, want = to_f64(outs[0]), ref.attend(to_f64(q), 128 ** -0.5)
    for b in range(len(lens)):
        assert rel_l2(out[b], want[b]) < TOL_ATTENTION_F32_IO, lens[b]


# Fewer than 32 tokens, spread unevenly over the sequences: all in one of them, most of them without any, more vectors than a
# cluster's single pass.
@pytest.mark.parametrize("d,Hkv", [(128, 3), (128, 32), (64, 8), (32, 5), (16, 8)])
@pytest.mark.parametrize("lens", [[0] * 7 + [31] + [0] * 8, [3, 0, 0, 11, 1, 0, 14], [31], [0] * 299 + [2]])
def test_few_tokens_spread_unevenly(d, Hkv, lens):
    n = sum(lens)
    cache = pq.PolarQuantCache(len(lens), Hkv, Hkv, d, capacity=64, seed=7, device=DEV)
    K, V = synthetic.kv_like(50 + d, n, Hkv, d, torch.bfloat16, DEV, n_outliers=4 if d >= 64 else 0)
    cache.encode(K, V, torch.tensor(np.concatenate(([0], np.cumsum(lens))), dtype=torch.int32, device=DEV))
    assert cache.lens.tolist() == lens
    cache.check_status()
    codes, radii = (x.cpu().numpy() for x in cache.unpack(max(lens)))
    cb, S, row, off = oracle_codebooks(cache), cache.S_host.double().numpy(), 0, [0, 0]
    for b, m in enumerate(lens):
        for kv, X in ((0, to_f64(K)), (1, to_f64(V))):
            for h in range(Hkv if m else 0):
                rep = code_mismatch_report(codes[b, h, kv, :m], X[row:row + m, h], S, cb)
                assert_codes_match(rep)
                off = [x + y for x, y in zip(off, radii_ulp_report(radii[b, h, kv, :m], rep["radii16"]))]
        row += m
    assert_radii_match(counts=off)


# cu_seqlens that names more rows than K and V have: the missing rows are neither read (the inputs are the front of a larger
# tensor here) nor written.
@pytest.mark.parametrize("lens", [[5], [3, 4]])
def test_rows_past_the_inputs_are_not_touched(lens):
    n, Hkv, d = 3, 2, 64
    cache = pq.PolarQuantCache(len(lens), Hkv, Hkv, d, capacity=64, seed=7, device=DEV)
    cache.cache.fill_(0xA5)
    K, V = synthetic.kv_like(51, 40, Hkv, d, torch.bfloat16, DEV)
    K[n:], V[n:] = float("nan"), float("nan")
    cache.encode(K[:n], V[:n], torch.tensor([0] + list(np.cumsum(lens)), dtype=torch.int32, device=DEV))
    assert cache.status.tolist()[:2] == [pq.OK, 0]              # no non-finite input was seen
    codes, radii = cache.unpack(max(lens))
    untouched = torch.full((), 0xA5A5 - 0x10000, dtype=torch.int16).view(torch.float16).to(DEV)
    assert torch.all(radii[0, :, :, n:] == untouched) and not torch.any(radii[0, :, :, :n] == untouched)


def _codes_and_radii(cache, K, V, pieces):
    """Encodes the pieces one after the other; (codes, radii) of the cache and of the oracle, [vectors, ...]."""
    at = 0
    for m in pieces:
        cache.encode(K[at:at + m], V[at:at + m], torch.tensor([0, m], dtype=torch.int32, device=DEV))
        at += m
    bits = (4, 2, 2, 2) if not hasattr(cache, "bits") else tuple(cache.bits)
    cb = orc.codebooks_from_arrays(bits, cache.centroids.numpy(), cache.boundaries.numpy())
    codes, radii = (x.cpu().numpy()[0].transpose(1, 2, 0, 3).reshape(2 * at * cache.n_kv_heads, -1) for x in cache.unpack(at))
    X = np.stack([to_f64(K[:at]), to_f64(V[:at])]).reshape(2 * at * cache.n_kv_heads, -1)
    rep = code_mismatch_report(codes, X, cache.S_host.double().numpy(), cb)
    return rep, radii, rep["radii16"]


def _cache_of(d, bits, Hkv, n):
    if bits is None:
        return pq.PolarQuantCache(1, Hkv, Hkv, d, capacity=n, seed=6, device=DEV)
    cache = pq.GeneralPolarQuantCache(1, Hkv, Hkv, d, bits, n, seed=6, device=DEV)
    cache.bits = bits
    return cache


# Vectors whose norm lies in one rotated block: the float32 rotation's error follows the norm of the vector, not that of a block, and
# the radii of the small blocks are the one rounding of the exact norm all the same.
@pytest.mark.parametrize("d,bits", [(64, None), (32, None), (128, (4, 2, 2, 2)), (64, (4, 3, 2)), (256, (3,) * 5)])
def test_radii_of_vectors_concentrated_in_a_block(d, bits):
    Hkv, pieces = 2, [20, 1400]                                 # few vectors and tiles have kernels of their own
    n = sum(pieces)
    cache = _cache_of(d, bits, Hkv, n)
    gen = torch.Generator(device=DEV).manual_seed(d)
    Y = torch.randn((2, n, Hkv, d // 16, 16), generator=gen, device=DEV, dtype=torch.float64)
    small = 10.0 ** (-1.5 - 2.5 * torch.rand((2, n, Hkv, d // 16, 1), generator=gen, device=DEV, dtype=torch.float64))
    big = torch.randint(0, d // 16, (2, n, Hkv, 1, 1), generator=gen, device=DEV)
    Y *= small.scatter(3, big, 1.0)
    K, V = (Y.view(2, n, Hkv, d) @ cache.S_host.double().to(DEV).T).float()
    rep, radii, want = _codes_and_radii(cache, K, V, pieces)
    assert_codes_match(rep)
    assert np.array_equal(radii.view(np.uint16), want.astype(np.float16).view(np.uint16))


# Rows so small that squares, or the squares of squares that the sign tests compare, leave the float32 range.
@pytest.mark.parametrize("scale", [3e-21, 2e-10, 1.0])
@pytest.mark.parametrize("d,bits", [(128, None), (64, None), (16, None), (128, (3,) * 7), (64, (4, 3, 2)), (32, (5,)), (128, (6, 5, 4, 3, 2, 1, 1))])
def test_codes_of_tiny_rows(d, bits, scale):
    Hkv, pieces = 2, [20, 1400]
    cache = _cache_of(d, bits, Hkv, sum(pieces))
    K, V = (x * scale for x in synthetic.kv_like(52, sum(pieces), Hkv, d, torch.float32, DEV, n_outliers=0))
    rep, radii, want = _codes_and_radii(cache, K, V, pieces)
    assert_codes_match(rep)
    if d < 128 or bits is not None:
        assert np.array_equal(radii, want)
    else:
        assert_radii_match(radii, want)


# A query that is not finite gives a row that is not finite -- not zeros, and not an empty sequence -- and leaves the others alone.
@pytest.mark.parametrize("kernel", [CLUSTER, PERSISTENT, ROWS, TCGEN05])
def test_a_nan_query_gives_a_nan_row(kernel):
    lens, n_q, Hq = [700, 40], 8, 8
    cache, ref = _filled(lens, Hq, 2, 128, 77)
    q = torch.randn((2, n_q, Hq, 128), generator=torch.Generator(device=DEV).manual_seed(3), device=DEV)
    bad = q.clone()
    bad[0, 3, 5, 17] = float("nan")
    bad[1, 7, 0, 0] = float("inf")
    outs = []
    for x in (q, bad):
        pq.pq_debug_fail_next_wait(kernel)
        outs.append(cache.attend_multi(x))
    cache.check_status()
    for b, j, h in ((0, 3, 5), (1, 7, 0)):
        assert bool(torch.isnan(outs[1][b, j, h]).all())
        outs[1][b, j, h] = outs[0][b, j, h]
    assert torch.equal(outs[0], outs[1])


# Where the tcgen05 kernel does not fit, a long chunk runs on the others.
def test_long_chunk_without_the_tcgen05_kernel():
    lens, n_q = [700, 300], 64
    cache, ref = _filled(lens, 8, 2, 128, 78)
    q = torch.randn((2, n_q, 8, 128), generator=torch.Generator(device=DEV).manual_seed(4), device=DEV)
    _check_multi(cache, ref, q, lens, 10)
    pq.pq_debug_fail_next_wait(TCGEN05)
    other = cache.attend_multi(q)
    pq.pq_debug_fail_next_wait(10)
    assert not torch.equal(cache.attend_multi(q), other)


# The window on tensor cores (bf16 rows of 128, up to four heads per kv head) against the float32 kernel on the same rows: windows that end
# around its 16-token tiles and its warps' shares, empty ones, more splits than tokens.  Exact products, float32 sums in another order:
# 1e-5 is 2^-24 times the 128 terms of a score in the exponent.  Infinite and NaN rows give what the float32 kernel gives.
@pytest.mark.parametrize("io", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("g,n_splits", [(1, 1), (2, 3), (3, 1), (4, 7)])
def test_window_on_tensor_cores(g, n_splits, io):
    lens, T, Hkv = [0, 1, 15, 16, 17, 63, 64, 65, 129, 300, 300, 300], 300, 2
    B = len(lens)
    K, V = (t.view(B, T, Hkv, 128) for t in synthetic.kv_like(g, B * T, Hkv, 128, torch.bfloat16, DEV))
    K[10, 7, 0, 3], V[10, 200, 1, 5], V[11, 3, 0, 9], K[11, 250, 1, 0] = -float("inf"), float("inf"), float("nan"), float("nan")
    q = synthetic.queries(3, B, g * Hkv, 128, io, DEV)
    n = torch.tensor(lens, dtype=torch.int32, device=DEV)
    got = []
    for kv in ((K, V), (K.float(), V.float())):
        out, lse = torch.empty((n_splits, *q.shape), dtype=io, device=DEV), torch.empty((n_splits, *q.shape[:2]), device=DEV)
        pq.pq_tail_attention(q, *kv, n, 128 ** -0.5, out, lse, torch.zeros(4, dtype=torch.int32, device=DEV), n_splits)
        got.append((out.float(), lse))
    tol = 1e-5 if io == torch.float32 else 2.0 ** -8
    for a, b in zip(*got):
        assert torch.equal(a.isnan(), b.isnan()) and torch.equal(a.isinf(), b.isinf())
        ok = a.isfinite() & b.isfinite()
        assert torch.all((a - b)[ok].abs() <= tol * b[ok].abs().clamp(min=1.0))
