"""Sizes at which a tile, a remainder or a choice between kernels can go wrong, one small case per edge, against the
oracles."""
import numpy as np
import pytest
import torch

from paper_2609_35465_b200 import synth
from helpers import assert_gemv_close, make_matrix, oracle_product

pytestmark = pytest.mark.gpu
GAIN = synth.DEFAULT_GAIN


@pytest.fixture(scope="module")
def tt():
    from paper_2609_35465_b200 import tetra
    return tetra


@pytest.fixture(scope="module")
def table(tt):
    return tt.tetra_build_table(GAIN)


def device_matrix(tt, table, m, x):
    codes = tt.tetra_pack_codes(torch.from_numpy(m["codes"]).cuda(), table, m["N"], m["B"])
    return dict(codes=codes, row_scales=torch.from_numpy(m["sigma"]).cuda(), x=x, N=m["N"], K=m["K"],
                tail=torch.from_numpy(m["tail"]).cuda() if m["tail"] is not None else None,
                y=torch.full((m["N"],), float("nan"), dtype=torch.float32, device="cuda"))


def check(orc, m, y, what, vector=0):
    assert np.isfinite(y).all(), what
    ref = oracle_product(orc, m, GAIN, batch_index=vector)
    assert_gemv_close(y, ref, what)
    assert np.max(np.abs(y - ref["y"]) / ref["abssum"]) < 1e-5


# Row groups of eight and of four rows, one and several chunks of rows per CTA, fewer columns than lanes, K too large
# for the activations' image in shared memory.
@pytest.mark.parametrize("N,K,tail_mode", [
    (1, 24, True), (4, 25, True), (5, 47, False), (8, 24 * 31, True), (9, 24 * 32, True), (1183, 24 * 33 + 1, True),
    (1185, 24 * 5, True), (148 * 8 * 3 + 4, 24 * 40, True), (148 * 16 + 12, 24 * 64 + 23, True), (20001, 96, True),
    (64, 24 * 1400, True), (24, 49152, True),
])
def test_single_matrix(tt, table, orc, N, K, tail_mode):
    m = make_matrix(71, N + K, N, K, tail_mode, batch=1)
    d = device_matrix(tt, table, m, torch.from_numpy(m["x"][0]).cuda())
    if tail_mode:
        tt.tetra_gemv_tail(d["codes"], d["row_scales"], table, d["x"], d["y"], N, K, 1, d["tail"])
    else:
        tt.tetra_gemv(d["codes"], d["row_scales"], table, d["x"], d["y"], N, K)
    torch.cuda.synchronize()
    check(orc, m, d["y"].cpu().numpy(), "%d x %d" % (N, K))


# The activations' image by sections or by columns: on both sides of a section per thread and of a column per thread.
@pytest.mark.parametrize("N,K,tail_mode", [(9, 24 * 170 + 7, True), (9, 24 * 170 + 7, False), (9, 24 * 171, True), (33, 24 * 512 + 3, True),
                                           (33, 24 * 512 + 3, False), (8, 24 * 1024 + 1, True)])
def test_image_by_columns(tt, table, orc, N, K, tail_mode):
    test_single_matrix(tt, table, orc, N, K, tail_mode)


# A CTA works on one matrix: lists of very unequal matrices, of more and of fewer row groups than CTAs; long rows that leave
# the other matrix's rows room for half a CTA's share.
@pytest.mark.parametrize("rows,K", [((1, 1, 1, 1, 1, 1, 1, 1), 24), ((4000, 8), 24 * 40), ((8, 9000, 16, 1), 24 * 12 + 7),
                                    ((700, 700, 700), 24 * 70 + 2), ((60001, 64), (24, 24 * 1250))])
def test_list_split(tt, table, orc, rows, K):
    Ks = K if isinstance(K, tuple) else (K,) * len(rows)
    ms = [make_matrix(72, 10 * i + k, n, k, True, batch=1) for i, (n, k) in enumerate(zip(rows, Ks))]
    items = [device_matrix(tt, table, m, torch.from_numpy(m["x"][0]).cuda()) for m in ms]
    tt.tetra_gemv_list(tt.make_problems(items), table)
    torch.cuda.synchronize()
    for m, it in zip(ms, items):
        check(orc, m, it["y"].cpu().numpy(), "list %s" % (rows,))


# Block-diagonal up to four vectors, dense from five on; one to four row tiles per step and several steps of rows; column
# quads that are not full; clusters (few rows, many columns); rows of x that are not 16-byte aligned.
@pytest.mark.parametrize("N,K,tail_mode,batch", [
    (1, 24, True, 2), (15, 24 * 3, True, 3), (16, 24 * 4, True, 4), (17, 24 * 5, True, 5), (33, 24 * 65 + 1, True, 2),
    (33, 24 * 65 + 3, False, 7), (64, 24 * 600, True, 2), (64, 24 * 600 + 8, True, 11), (148 * 16, 24 * 9, True, 4),
    (148 * 16 + 1, 24 * 9, True, 9), (148 * 48, 24 * 7, True, 3), (148 * 64 + 5, 24 * 6, True, 6), (148 * 80, 24 * 2, True, 16),
    (148 * 96 + 3, 24 * 5 + 2, True, 2),
])
def test_batched_shapes(tt, table, orc, N, K, tail_mode, batch):
    m = make_matrix(73, N + K + batch, N, K, tail_mode, batch=batch)
    d = device_matrix(tt, table, m, torch.from_numpy(m["x"]).cuda())
    y = torch.full((batch, N), float("nan"), dtype=torch.float32, device="cuda")
    tt.tetra_gemv_batched(d["codes"], d["row_scales"], table, d["x"], y, N, K, batch, d["tail"])
    torch.cuda.synchronize()
    for v in sorted({0, batch // 2, batch - 1}):
        check(orc, m, y[v].cpu().numpy(), "%d x %d, vector %d of %d" % (N, K, v, batch), v)


# Rows of x at every 2-byte place of 16 bytes: copied as they lie and shifted on the chip.  What lies around x is NaN and may
# not reach a result.  (What the copies bring along ahead of a vector is the end of the one before: see the non-finite
# activations below.)
@pytest.mark.parametrize("batch", [2, 3, 8, 16])
@pytest.mark.parametrize("K,tail_mode,offset", [(24 * 9, True, 0), (24 * 9, True, 1), (24 * 70 + 4, True, 2), (24 * 70 + 5, True, 3),
                                                (24 * 70 + 2, False, 6), (24 * 71 + 7, False, 7), (24 * 4, True, 5)])
def test_batched_unaligned_activations(tt, table, orc, K, tail_mode, offset, batch):
    N = 41
    m = make_matrix(77, K + batch, N, K, tail_mode, batch=batch)
    buf = torch.full((batch * K + 32,), float("nan"), dtype=torch.float16, device="cuda")
    x = buf[8 + offset:8 + offset + batch * K].view(batch, K)
    x.copy_(torch.from_numpy(m["x"]))
    d = device_matrix(tt, table, m, x)
    y = torch.full((batch, N), float("nan"), dtype=torch.float32, device="cuda")
    tt.tetra_gemv_batched(d["codes"], d["row_scales"], table, x, y, N, K, batch, d["tail"])
    torch.cuda.synchronize()
    for v in range(batch):
        check(orc, m, y[v].cpu().numpy(), "K %d, offset %d, vector %d of %d" % (K, offset, v, batch), v)


# Rows shorter than 16 bytes: several begin in the 16 bytes that x begins in.
@pytest.mark.parametrize("batch", [2, 4, 7, 16])
@pytest.mark.parametrize("K,offset", [(1, 3), (3, 5), (6, 7)])
def test_batched_rows_shorter_than_a_unit(tt, table, orc, K, offset, batch):
    N = 17
    m = make_matrix(78, K + batch, N, K, False, batch=batch)
    buf = torch.full((batch * K + 32,), float("nan"), dtype=torch.float16, device="cuda")
    x = buf[8 + offset:8 + offset + batch * K].view(batch, K)
    x.copy_(torch.from_numpy(m["x"]))
    d = device_matrix(tt, table, m, x)
    y = torch.full((batch, N), float("nan"), dtype=torch.float32, device="cuda")
    tt.tetra_gemv_batched(d["codes"], d["row_scales"], table, x, y, N, K, batch)
    torch.cuda.synchronize()
    for v in range(batch):
        ref = oracle_product(orc, m, GAIN, batch_index=v)
        # a row's few coordinates may all be zero: the bound is then zero, and so is the result
        assert (np.abs(y[v].cpu().numpy() - ref["y"]) <= 1e-5 * ref["abssum"]).all(), "K %d, vector %d of %d" % (K, v, batch)


@pytest.mark.parametrize("bad", [float("nan"), float("inf"), float("-inf")])
@pytest.mark.parametrize("batch", [3, 6])
def test_batched_non_finite_activation(tt, table, bad, batch):
    m = make_matrix(74, batch, 70, 24 * 20, True, batch=batch)
    x = torch.from_numpy(m["x"]).cuda()
    x[1, 24 * 7 + 5] = bad
    d = device_matrix(tt, table, m, x)
    y = torch.zeros((batch, 70), dtype=torch.float32, device="cuda")
    tt.tetra_gemv_batched(d["codes"], d["row_scales"], table, x, y, 70, 24 * 20, batch)
    torch.cuda.synchronize()
    assert torch.isnan(y[1]).all() and torch.isfinite(y[0]).all() and torch.isfinite(y[2:]).all()


# The same in rows that are not 16-byte aligned, where a copy brings the end of a vector along ahead of the next: first and
# last activation of a vector in the middle, and one that two quads of columns share a copy of.
@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
@pytest.mark.parametrize("place", [0, 96, 24 * 20 + 4])
@pytest.mark.parametrize("batch", [3, 4, 6, 16])
def test_batched_non_finite_activation_in_unaligned_rows(tt, table, bad, place, batch):
    N, K = 70, 24 * 20 + 5
    m = make_matrix(79, batch, N, K, False, batch=batch)
    for offset in (0, 3):
        buf = torch.zeros(batch * K + 16, dtype=torch.float16, device="cuda")
        x = buf[offset:offset + batch * K].view(batch, K)
        x.copy_(torch.from_numpy(m["x"]))
        x[1, place] = bad
        d = device_matrix(tt, table, m, x)
        y = torch.zeros((batch, N), dtype=torch.float32, device="cuda")
        tt.tetra_gemv_batched(d["codes"], d["row_scales"], table, x, y, N, K, batch)
        torch.cuda.synchronize()
        assert torch.isnan(y[1]).all() and torch.isfinite(y[0]).all() and torch.isfinite(y[2:]).all()


# Rows of x that are not 16-byte aligned have kernels of their own: two, three and four row tiles a step for each class of
# vectors, three steps to a warp, and a second round of rows (six tiles to a CTA are two rounds of three).  The tiles follow
# from the rows; with 41 quads of columns a CTA has them to itself.  x at a 2-byte and at a 4-byte place: dense fragments are
# shifted or read as words.  Then a cluster of two CTAs (few rows, many columns).  Sampled rows, every vector.
_MATRICES = {}


def sampled_batched(tt, table, orc, N, K, offset, batch):
    if (N, K) not in _MATRICES:
        m = make_matrix(80, N + K, N, K, True, batch=16)
        _MATRICES[N, K] = m, device_matrix(tt, table, m, None)
    m, d = _MATRICES[N, K]
    buf = torch.full((batch * K + 16,), float("nan"), dtype=torch.float16, device="cuda")
    x = buf[offset:offset + batch * K].view(batch, K)
    x.copy_(torch.from_numpy(m["x"][:batch]))
    y = torch.full((batch, N), float("nan"), dtype=torch.float32, device="cuda")
    tt.tetra_gemv_batched(d["codes"], d["row_scales"], table, x, y, N, K, batch, d["tail"])
    torch.cuda.synchronize()
    yh = y.cpu().numpy()
    assert np.isfinite(yh).all()
    rows = np.unique([r for r in (0, 15, 16, 31, 32, 47, 48, 63, N // 2, N - 17, N - 16, N - 1) if 0 <= r < N])
    for v in range(batch):
        ref = oracle_product(orc, m, GAIN, rows=rows, batch_index=v, threads=4)
        assert_gemv_close(yh[v][rows], ref, "%d x %d, offset %d, vector %d of %d" % (N, K, offset, v, batch))
        assert np.max(np.abs(yh[v][rows] - ref["y"]) / ref["abssum"]) < 1e-5


@pytest.mark.parametrize("K,offset", [(24 * 162 + 5, 3), (24 * 162 + 4, 2)])
@pytest.mark.parametrize("tiles", [2, 3, 4, 6])
@pytest.mark.parametrize("batch", [2, 4, 7, 16])
def test_batched_unaligned_tiles(tt, table, orc, tiles, K, offset, batch):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    sampled_batched(tt, table, orc, 16 * sms * (tiles - 1) + 17, K, offset, batch)


@pytest.mark.parametrize("K,offset", [(24 * 600 + 1, 0), (24 * 600 + 4, 0), (24 * 600, 5)])
@pytest.mark.parametrize("batch", [2, 4, 7, 16])
def test_batched_unaligned_cluster(tt, table, orc, K, offset, batch):
    sampled_batched(tt, table, orc, 64, K, offset, batch)


# Copies out of 16, 8 and 4 bytes (odd block counts, outputs that are not aligned), part-filled row groups and columns.
@pytest.mark.parametrize("N,B", [(1, 1), (7, 31), (8, 32), (9, 33), (17, 64), (16, 65)])
def test_decode_packed_shapes(tt, table, orc, N, B):
    words = synth.words_to_bytes(synth.words(75, N * 100 + B, N * B))
    # word addresses that are 2, but not 4 bytes aligned as well
    buf = torch.zeros(6 * N * B + 2, dtype=torch.uint8, device="cuda")
    buf[2:] = torch.from_numpy(words.reshape(-1)).cuda()
    Y, M, G = orc.decode_blocks(words)
    for codes in (torch.from_numpy(words).cuda().reshape(N, B, 6), buf[2:].reshape(N, B, 6)):
        packed = tt.tetra_pack_codes(codes, table, N, B)
        y, mg = tt.tetra_decode_packed(packed, table, N, B)
        out = torch.zeros(24 * N * B + 4, dtype=torch.int8, device="cuda")
        lib, p = tt.lib(), tt._ptr
        assert lib.tetra_decode_packed(p(packed), p(table), p(out[4:]), None, N, B, tt._stream()) == 0
        torch.cuda.synchronize()
        assert np.array_equal(y.cpu().numpy().reshape(-1, 24), Y)
        assert np.array_equal(mg.cpu().numpy().reshape(-1, 2), np.stack([M, G], 1))
        assert np.array_equal(out[4:].cpu().numpy().reshape(-1, 24), Y)


# Strips of 32 rows shared by two and more warps, CTAs with fewer chunks than warps, both group sizes.
@pytest.mark.parametrize("N,K,G,batch", [(1, 64, 64, 1), (31, 128, 128, 8), (33, 192, 64, 1), (64, 15 * 64, 64, 3),
                                         (32 * 148, 128 * 7, 128, 1), (32 * 148 * 2 + 1, 64 * 3, 64, 2), (96, 64 * 257, 64, 1)])
def test_q4_shapes(tt, N, K, G, batch):
    from oracle import q4 as oq
    q = synth.q4_nibbles(76, N, N, K)
    sc, of = synth.q4_scales_offsets(76, N, N, K // G)
    packed = tt.tetra_q4_pack(torch.from_numpy(q).cuda(), torch.from_numpy(sc).cuda(), torch.from_numpy(of).cuda(), N, K, G)
    x = synth.activations(76, K, K, batch)
    y = torch.full((batch, N), float("nan"), dtype=torch.float32, device="cuda")
    tt.tetra_q4_gemv(packed, torch.from_numpy(x).cuda(), y, N, K, G, batch)
    ids = synth.token_ids(76, 1, 9, N)
    buf = torch.zeros(9 * K + 4, dtype=torch.float16, device="cuda")
    rows, rows8 = torch.zeros((9, K), dtype=torch.float16, device="cuda"), buf[4:].reshape(9, K)  # 16 and 8 byte stores
    for out in (rows, rows8):
        tt.tetra_q4_rows(packed, torch.from_numpy(ids).cuda(), out, N, K, G)
    torch.cuda.synchronize()
    want, tn = oq.gemv(q, sc, of, x, N, K, G, batch)
    assert_gemv_close(y.cpu().numpy(), {"y": want, "termnorm": tn}, "q4 %d x %d" % (N, K))
    want_rows = oq.rows(q, sc, of, ids, N, K, G).view(np.uint16)
    for out in (rows, rows8):
        assert np.array_equal(out.cpu().numpy().view(np.uint16), want_rows)


# Lists with fewer chunks than warps, strips that many warps share, many small matrices, more groups per CTA than are held.
@pytest.mark.parametrize("shapes,G", [([(1, 64)], 64), ([(40, 128), (1, 256), (33, 128)], 128), ([(32, 64 * 900)], 64),
                                      ([(64, 64)] * 300, 64), ([(32, 65536)] * 40, 64),
                                      ([(64, 1280)] * 200, 128), ([(32, 64 * 320)] * 20, 64)])
def test_q4_list_shapes(tt, shapes, G):
    from oracle import q4 as oq
    items, hosts = [], []
    for i, (N, K) in enumerate(shapes):
        q = synth.q4_nibbles(77, i % 3, N, K)
        sc, of = synth.q4_scales_offsets(77, i % 3, N, K // G)
        x = synth.activations(77, i, K, 1)
        hosts.append((q, sc, of, x, N, K))
        items.append(dict(packed=tt.tetra_q4_pack(torch.from_numpy(q).cuda(), torch.from_numpy(sc).cuda(),
                                                  torch.from_numpy(of).cuda(), N, K, G),
                          x=torch.from_numpy(x[0]).cuda(), y=torch.zeros(N, dtype=torch.float32, device="cuda"), N=N, K=K))
    ws = tt.tetra_q4_list_plan(tt.make_q4_problems(items), G)
    first = None
    for _ in range(2):  # the counters of shared strips start over
        for it in items:
            it["y"].fill_(float("nan"))
        tt.tetra_q4_list_run(ws, G)
        torch.cuda.synchronize()
        got = [it["y"].cpu().numpy() for it in items]
        assert first is None or all(np.array_equal(a, b) for a, b in zip(got, first))
        first = got
    for k in sorted({0, len(items) // 2, len(items) - 1}):
        q, sc, of, x, N, K = hosts[k]
        want, tn = oq.gemv(q, sc, of, x, N, K, G, 1)
        assert_gemv_close(got[k][None], {"y": want, "termnorm": tn}, "list matrix %d, %d x %d" % (k, N, K))


def test_encode_points_at_the_limits_of_the_lists(tt, table, orc):
    """The last rows of every list and the rows just inside its last shell, both parities, come back as the same point:
    these rows decide where the search's tables end."""
    fields = []
    for i1, i2, i3 in ((2047, 1239, 2047), (2046, 1238, 1256), (1256, 1240 + 807, 1255), (1255, 1240, 2047), (2047, 1240 + 806, 1816),
                       (1816, 499, 1815), (1815, 498, 2047)):
        for path in (0, 777, 4095):
            for p in (0, 1):
                for r in (0, 1):
                    fields.append(i1 | (i2 << 11) | (i3 << 22) | (path << 33) | (p << 45) | (r << 46))
    words = np.array(fields, dtype=np.uint64)
    Y, _, _ = orc.decode_blocks(synth.words_to_bytes(words))
    w = Y.astype(np.float32)
    codes, cos = tt.tetra_encode_blocks(torch.from_numpy(w).cuda(), table)
    torch.cuda.synchronize()
    got, _, _ = orc.decode_blocks(codes.cpu().numpy())
    got = got.astype(np.float64)
    c = (got * w).sum(1) / (np.linalg.norm(got, axis=1) * np.linalg.norm(w.astype(np.float64), axis=1))
    assert np.all(c >= 1 - 1e-12) and np.max(np.abs(cos.cpu().numpy() - 1)) <= 1e-6


@pytest.mark.parametrize("n", [1, 2, 147, 148, 149, 296, 297, 444, 445])
def test_encode_block_counts(tt, table, n):
    """Blocks are dealt to three groups of threads per CTA: every count gives what the blocks give on their own."""
    w = torch.from_numpy(synth.normal(78, 0, 20, 445 * 24).reshape(445, 24).astype(np.float32)).cuda()
    w[5] = 0
    all_codes, all_cos = tt.tetra_encode_blocks(w, table)
    codes, cos = tt.tetra_encode_blocks(w[445 - n:].contiguous(), table)
    torch.cuda.synchronize()
    assert torch.equal(codes, all_codes[445 - n:]) and torch.equal(cos, all_cos[445 - n:])


# Planned lists are cut into the warps' ranges by passes (32 columns of a row group): one unit shared by many ranges, fewer
# passes than CTAs and than warps, joint passes over three row groups' last columns on either side of a cut, a last unit with
# fewer row groups, units of one pass, several matrices in a range, the plan's order against the caller's.
@pytest.mark.parametrize("mats", [
    [(8, 24 * 32 * 63, True)], [(8, 24 * 32 * 40, True), (1, 24, True)], [(24, 24 * 42, True)], [(200, 24 * (32 * 5 + 10), True)],
    [(17, 24 * 37, True), (1, 24 * 33, False), (8 * 148, 24 * 32, True)], [(8 * 2368 + 9, 24 * 5, True)],
    [(3000, 24 * 42, True), (40, 24 * 700 + 7, True), (3001, 24 * 32, True)], [(1, 24 * 3, True)] * 40,
    [(8 * 300, 24 * 32 * 9, True), (16 * 75 + 3, 24 * (32 * 9 + 11) + 5, True)],
])
def test_planned_list_ranges(tt, table, orc, mats):
    ms = [make_matrix(83, 1000 * i + N, N, K, tail, batch=1) for i, (N, K, tail) in enumerate(mats)]
    items = [device_matrix(tt, table, m, torch.from_numpy(m["x"][0]).cuda()) for m in ms]
    problems = tt.make_problems(items)
    ws = torch.full((tt.tetra_grouped_workspace_bytes(problems),), 0xA5, dtype=torch.uint8, device="cuda")
    tt.tetra_gemv_grouped(problems, table, ws)
    first = [it["y"].clone() for it in items]
    for it in items:
        it["y"].fill_(float("nan"))
    tt.tetra_gemv_grouped_run(ws, table)
    torch.cuda.synchronize()
    for m, it, y in zip(ms, items, first):
        assert torch.equal(it["y"], y)
        check(orc, m, y.cpu().numpy(), "%d x %d of %d" % (m["N"], m["K"], len(ms)))


# No more pairs of eight rows and 32 columns than warps: units of one row group, and a pass for each range; one pair more; far fewer;
# ranges that begin in a joint pass.
@pytest.mark.parametrize("mats", [
    [(8 * 1184, 24 * 42, True)], [(8 * 1184 + 1, 24 * 42, True)], [(64, 768, True)], [(1024, 2560, True), (8, 24 * 3, True)],
    [(8 * 147, 24 * 45 + 11, True)], [(512, 24 * 170 + 16, True), (24, 24 * 170 + 16, True), (9, 24 * 700, True)],
])
def test_planned_list_of_few_passes(tt, table, orc, mats):
    test_planned_list_ranges(tt, table, orc, mats)


# A plan in place of another one between runs, copied by an ordinary kernel (test_gpu_order.py has one that lets the run start early).
def test_plan_written_by_the_kernel_before(tt, table, orc):
    sizes = [[(2048, 24 * 85, True), (17, 24 * 33 + 5, True)], [(40, 24 * 700 + 7, True), (3001, 24 * 32, True), (9, 24 * 5, True)]]
    plans, items, mats = [], [], []
    for i, shapes in enumerate(sizes):
        ms = [make_matrix(84, 1000 * i + N, N, K, tail, batch=1) for N, K, tail in shapes]
        its = [device_matrix(tt, table, m, torch.from_numpy(m["x"][0]).cuda()) for m in ms]
        problems = tt.make_problems(its)
        ws = torch.zeros(tt.tetra_grouped_workspace_bytes(problems), dtype=torch.uint8, device="cuda")
        tt.tetra_gemv_grouped_plan(problems, ws)
        plans.append(ws)
        items.append(its)
        mats.append(ms)
    shared = torch.zeros(max(p.numel() for p in plans), dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    for turn in range(40):
        torch.bitwise_or(plans[turn % 2], 0, out=shared[:plans[turn % 2].numel()])
        tt.tetra_gemv_grouped_run(shared, table)
    torch.cuda.synchronize()
    for ms, its in zip(mats, items):
        for m, it in zip(ms, its):
            check(orc, m, it["y"].cpu().numpy(), "%d x %d" % (m["N"], m["K"]))


# The largest K of the call that brings its own scratch, both rules; one weight more is refused.
@pytest.mark.parametrize("K,tail_mode", [(24576, True), (24575, False), (24575, True)])
def test_noalloc_largest_rows(tt, table, orc, K, tail_mode):
    m = make_matrix(87, K, 41, K, tail_mode, batch=1)
    d = device_matrix(tt, table, m, torch.from_numpy(m["x"][0]).cuda())
    tt.tetra_gemv_noalloc(d["codes"], d["row_scales"], table, d["x"], d["y"], 41, K, d["tail"])
    torch.cuda.synchronize()
    check(orc, m, d["y"].cpu().numpy(), "noalloc 41 x %d" % K)
    p = tt._ptr
    assert tt.lib().tetra_gemv_noalloc(p(d["codes"]), p(d["row_scales"]), p(table), p(d["x"]), p(d["y"]), 41, tt.NOALLOC_MAX_K + 1,
                                       None, tt._stream()) == -6


# A plan made for a grid of another size deals its units round-robin: here because the number of warps in the plan is overwritten.
def test_planned_list_dealt_round_robin(tt, table, orc):
    ms = [make_matrix(88, 1000 * i + N, N, K, tail, batch=1)
          for i, (N, K, tail) in enumerate([(8 * 2600 + 1, 24 * 32, True), (3001, 24 * 42 + 3, True), (40, 24 * 700 + 7, True), (33, 749, False)])]
    items = [device_matrix(tt, table, m, torch.from_numpy(m["x"][0]).cuda()) for m in ms]
    problems = tt.make_problems(items)
    ws = torch.zeros(-(-tt.tetra_grouped_workspace_bytes(problems) // 4), dtype=torch.int32, device="cuda")
    tt.tetra_gemv_grouped_plan(problems, ws)
    warps = torch.cuda.get_device_properties(0).multi_processor_count * 16
    assert int(ws[5]) == warps and int(ws[1]) > warps  # its warps; its units
    ws[5] = 0
    tt.tetra_gemv_grouped_run(ws, table)
    torch.cuda.synchronize()
    for m, it in zip(ms, items):
        check(orc, m, it["y"].cpu().numpy(), "%d x %d" % (m["N"], m["K"]))


# One matrix of more than 64 GB: places of records beyond 2^32 sixteen-byte units.  All rows are the origin but the first row
# group's and the last two's, which lie where a place in 32 bits would wrap around to rows of the beginning.
@pytest.mark.parametrize("entry,B", [("grouped", 2048), ("noalloc", 1024), ("list", 2048)])
def test_matrix_beyond_64_gigabytes(tt, table, orc, entry, B):
    G = (1 << 32) // (3 * B) + 3
    N, K = 8 * G, 24 * B
    torch.cuda.empty_cache()
    if torch.cuda.mem_get_info()[0] < (72 << 30):
        pytest.skip("less than 72 GB free")
    m = make_matrix(85, B, 24, K, True, batch=1)
    codes = torch.zeros(G * 3 * B * 16, dtype=torch.uint8, device="cuda")
    packed = tt.tetra_pack_codes(torch.from_numpy(m["codes"]).cuda(), table, 24, B)
    part = 3 * B * 16
    codes[:part] = packed[:part]
    codes[-2 * part:] = packed[part:]
    rows = torch.cat([torch.arange(8), torch.arange(N - 16, N)]).cuda()
    scales = torch.ones(N, device="cuda")
    scales[rows] = torch.from_numpy(m["sigma"]).cuda()
    x, y = torch.from_numpy(m["x"][0]).cuda(), torch.full((N,), float("nan"), device="cuda")
    problems = tt.make_problems([dict(codes=codes, row_scales=scales, x=x, tail=None, y=y, N=N, K=K)])
    if entry == "grouped":
        ws = torch.empty(tt.tetra_grouped_workspace_bytes(problems), dtype=torch.uint8, device="cuda")
        tt.tetra_gemv_grouped(problems, table, ws)
    elif entry == "noalloc":
        tt.tetra_gemv_noalloc(codes, scales, table, x, y, N, K)
    else:
        tt.tetra_gemv_list(problems, table)
    torch.cuda.synchronize()
    check(orc, m, y[rows].cpu().numpy(), "%s, %d x %d" % (entry, N, K))
    y[rows] = 0
    assert torch.count_nonzero(y) == 0
    del codes
    torch.cuda.empty_cache()


def least_workspace(mats):
    """What a plan has always been given at least: 80 bytes a column, room for the plan, and for a list of at most 65,536 pairs of
    eight rows and 32 columns what their sums take."""
    cols = groups = pairs = 0
    for N, K, tail in mats:
        B = K // 24 if tail or K % 24 == 0 else -(-K // 24)
        cols += B
        groups += -(-N // 8)
        pairs += -(-N // 8) * -(-B // 32)
    up = lambda v: -(-v // 256) * 256  # noqa: E731
    size = up(56 + 72 * len(mats) + 8 + 4 * 8193) + 80 * cols
    return size if pairs > 65536 else up(size) + 4 * groups + 256 + 32 * pairs


# A workspace of that size and not a byte more: ranges cut inside units, between units where the list is too long for the
# pieces' sums, more matrices than there is room to align.
@pytest.mark.parametrize("mats", [
    [(1024, 4096, True)], [(8, 24, True)], [(1, 24 * 3, True)] * 40, [(8, 24 * 5, True)] * 700,
    [(40, 24 * 700 + 7, True), (3001, 24 * 32, True), (33, 749, False)], [(3000, 24 * 42, True)], [(8 * 32769, 24 * 33, True)],
    [(8 * 22000 + 3, 24 * 75 + 1, True), (16, 24 * 2047, True)],
])
def test_planned_list_in_the_smallest_workspace(tt, table, orc, mats):
    ms = [make_matrix(86, 1000 * i + N, N, K, tail, batch=1) for i, (N, K, tail) in enumerate(mats)]
    items = [device_matrix(tt, table, m, torch.from_numpy(m["x"][0]).cuda()) for m in ms]
    problems = tt.make_problems(items)
    n = least_workspace(mats)
    assert n <= tt.tetra_grouped_workspace_bytes(problems)
    buf = torch.full((n + 4096,), 0xA5, dtype=torch.uint8, device="cuda")
    with pytest.raises(tt.TetraError, match="-6"):
        tt.tetra_gemv_grouped_plan(problems, buf[:n - 1])
    tt.tetra_gemv_grouped_plan(problems, buf[:n])
    for _ in range(2):
        for it in items:
            it["y"].fill_(float("nan"))
        tt.tetra_gemv_grouped_run(buf[:n], table)
    torch.cuda.synchronize()
    assert bool((buf[n:] == 0xA5).all())
    for m, it in list(zip(ms, items))[:12] + list(zip(ms, items))[-1:]:
        rows = np.unique(np.concatenate([np.arange(0, m["N"], max(1, m["N"] // 4000)), np.arange(max(0, m["N"] - 50), m["N"])]))
        y = it["y"].cpu().numpy()
        assert np.isfinite(y).all()
        assert_gemv_close(y[rows], oracle_product(orc, m, GAIN, rows=rows), "%d x %d" % (m["N"], m["K"]))
