"""The branches that a call's sizes select, at the sizes where they change over: the plan's mask products
(integer matrix units or walk over the set bits, one CTA or a cluster, Stage 2 by counting or by a sort),
the list conversions, the pairing of 64-row blocks across blocks of positions, the longest-first tail of
the tickets, tasks of zero to a few tiles back to back, and a captured call."""
import ctypes
import threading

import numpy as np
import pytest
import torch

from oracle import waveal_oracle as wo
from paper_2609_34814_b200 import binding as wb

pytestmark = pytest.mark.gpu


def _pack(mask):
    """[heads, rows, columns] of bool on the GPU -> bitmap words."""
    H, m, n = mask.shape
    bits = torch.zeros((H, m, (n + 63) // 64 * 64), dtype=torch.int64, device="cuda")
    bits[..., :n] = mask
    return (bits.view(H, m, -1, 64) << torch.arange(64, device="cuda")).sum(3).contiguous()


def _mask(H, m, n, density, seed):
    g = torch.Generator("cuda")
    g.manual_seed(seed)
    x = torch.rand((H, m, n), generator=g, device="cuda") < density
    x |= (torch.arange(m, device="cuda")[:, None] * n // m - torch.arange(n, device="cuda")[None]).abs() < 2
    return x


def _plan(mask, wave=148, mode=wb.FORCE_REORDER):
    H, m, n = mask.shape
    d = wb.plan_desc_default(heads=H, n_q_blocks=m, n_kv_blocks=n, wave_size=wave, mode=mode, seed=5)
    return wb.plan_bitmap(d, _pack(mask), debug=True)


# 256 / 257 rows: one CTA or a cluster; 255 / 256 / 257 columns: one 256-column chunk or two; wave 220 / 221: Stage 2 by
# counting or by the sort; one row or one column; 14,336 / 14,337 rows: digits in shared memory and the state in the workspace, or
# the walk by a cluster over that state; 16,384 rows: the most the plan takes, and the longest strip of the transpose
@pytest.mark.parametrize("H,m,n,wave", [(2, 1, 1, 148), (2, 1, 300, 7), (2, 33, 1, 7), (3, 31, 255, 16), (2, 256, 256, 220),
                                        (2, 257, 257, 221), (1, 600, 511, 148),
                                        (2, 14336, 200, 148), (2, 14337, 200, 148), (1, 16384, 200, 148)])
def test_plan_products_match_the_oracle(H, m, n, wave):
    mask = _mask(H, m, n, 0.2, m + n)
    r = _plan(mask, wave)
    for h in range(H):
        mk = mask[h].cpu().numpy()
        u = wo.mfcsi(mk, 5, wo.start_block(5, h, m))
        e = r.embedding[h].cpu().numpy()
        # fp64 on both sides, entries below 1; ~n roundings of 1e-16 per sum and 12 sums in a row
        assert np.abs(e - u).max() <= 12 * (m + n) * 2.3e-16 + 1e-15
        order1 = r.order1[h].cpu().numpy().astype(np.int64)
        assert np.array_equal(order1, wo.stage1_order(wo.polar_angles(e)))
        assert np.array_equal(r.row_order[h].cpu().numpy(), wo.stage2_order(order1, mk.sum(1), wave))
        st = wo.guard_stats(mk, wave)
        assert r.stats[h].tolist()[:3] == [st["nnz"], st["ov_nat"], st["pair2"]]
        assert np.array_equal(r.row_nnz[h].cpu().numpy(), mk.sum(1)) and np.array_equal(r.col_count[h].cpu().numpy(), mk.sum(0))


# a wave of the head's length or more is one wave, up to the largest value the descriptor holds
@pytest.mark.parametrize("m", [2, 100, 300, 9700])
def test_waves_longer_than_the_head(m):
    mask = _mask(2, m, 70, 0.2, m)
    ref = _plan(mask, wave=m)
    for wave in (m + 1, 2 ** 31 - m, 2 ** 31 - 1):
        r = _plan(mask, wave=wave)
        assert torch.equal(r.row_order, ref.row_order) and torch.equal(r.order1, ref.order1) and torch.equal(r.stats, ref.stats)
    nnz = ref.row_nnz.long().gather(1, ref.row_order.long())
    assert (nnz[:, :-1] >= nnz[:, 1:]).all()
    st = wo.guard_stats(mask[0].cpu().numpy(), m)
    assert ref.stats[0].tolist()[:3] == [st["nnz"], st["ov_nat"], st["pair2"]]


# columns that select nothing change no product: the same mask with 10,000 of them goes through the walk over the
# set bits, widened to 4,700 x 4,700 or 5,000 x 5,000 through the shared Y / Z buffer or the workspace
# (4,768: the last square whose digits fit beside the state; then the walk; columns beyond 14,336: the walk over the workspace)
@pytest.mark.parametrize("m,n,wide", [(100, 300, 10000), (4700, 300, 4700), (4768, 300, 4768), (4769, 300, 4769),
                                      (5000, 300, 5000), (2000, 300, 14336), (2000, 300, 14400)])
def test_plan_products_agree_between_their_forms(m, n, wide):
    mask = _mask(2, m, n, 0.1, 9)
    padded = torch.zeros((2, m, wide), dtype=torch.bool, device="cuda")
    padded[..., :n] = mask
    a, b = _plan(mask), _plan(padded)
    assert (a.embedding - b.embedding).abs().max().item() <= 12 * (m + n) * 2.3e-16 + 1e-15
    assert torch.equal(a.order1, b.order1) and torch.equal(a.row_order, b.row_order)


# 512 / 513 rows: angles by merging or by bins; equal rows that fill a bin, or are too many for it (64 up to 1,024 rows, an
# eighth of the rows up to 192 above); 1,024 / 1,025 rows:
# Stage 2 by counting or a warp per bucket, buckets of 63 / 64 / 219 / 220 rows and of what is left
@pytest.mark.parametrize("m,wave,equal", [(512, 148, 0), (513, 148, 0), (700, 148, 150), (700, 148, 250), (1024, 64, 0), (1025, 63, 0),
                                          (1025, 64, 20), (1300, 219, 0), (1500, 220, 700), (2841, 148, 0), (7168, 148, 300),
                                          (700, 148, 64), (700, 148, 65), (1024, 64, 64), (1024, 64, 65), (1025, 64, 127), (1025, 64, 129),
                                          (1536, 148, 192), (1536, 148, 193), (2841, 148, 193)])
def test_sorts_of_the_plan(m, wave, equal):
    mask = _mask(2, m, 300, 0.1, m + wave)
    mask[0, torch.randperm(m, generator=torch.Generator().manual_seed(m))[:equal].cuda()] = True
    r = _plan(mask, wave)
    nnz = mask.sum(2).cpu().numpy()
    for h in range(2):
        first, order = r.order1[h].cpu().numpy(), r.row_order[h].cpu().numpy()
        u = r.embedding[h].cpu().numpy()[first]
        a = np.arctan2(u[:, 1], u[:, 0])
        assert np.array_equal(np.sort(first), np.arange(m))
        assert (np.diff(a) > -1e-14).all()                 # (NumPy's and the device's arctangents are an ulp or two apart)
        same = (np.diff(u, axis=0) == 0).all(1)
        assert (np.diff(first)[same] > 0).all()
        for lo in range(0, m, wave):
            bucket = first[lo:lo + wave]
            assert np.array_equal(order[lo:lo + wave], bucket[np.argsort(-nnz[h][bucket], kind="stable")])


# a head with many rows of one angle is planned as fast as by the merge sort alone (walked as one bin of 190: 4.5 to 7 % slower)
@pytest.mark.parametrize("m", [520, 700])
def test_equal_rows_do_not_slow_a_plan(m):
    def best(equal):
        mask = _mask(5, m, m, 0.1, m)
        mask[:, torch.randperm(m, generator=torch.Generator().manual_seed(m))[:equal].cuda()] = True
        bits = _pack(mask)
        d = wb.plan_desc_default(heads=5, n_q_blocks=m, n_kv_blocks=m, wave_size=148, mode=wb.FORCE_REORDER, seed=5)
        ws = torch.empty((wb.plan_workspace_bytes(d) + 256,), dtype=torch.uint8, device="cuda")
        out = []
        for _ in range(10):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            torch.cuda._sleep(4_000_000)             # the calls are queued before the first one starts
            a.record()
            for _ in range(20):
                wb.plan_bitmap(d, bits, workspace=ws)
            b.record()
            torch.cuda.synchronize()
            out.append(a.elapsed_time(b))
        return min(out)

    assert best(190) <= 1.02 * best(m // 2)          # (half of the rows go through the merge sort)


def _first_sweep(rows, cols, m, n, real):
    """Q factor after one sweep of Algorithm 1 over the sorted (row, column) pairs, in NumPy at the precision `real`."""
    def product(out, src, size, x):               # sums of x[src] over equal, ascending `out`
        at = np.flatnonzero(np.r_[True, out[1:] != out[:-1]])
        y = np.zeros((size, 2), real)
        y[out[at]] = np.add.reduceat(x[src], at, axis=0)
        return y

    def qr(z):
        q1 = z[:, 0] / np.sqrt((z[:, 0] ** 2).sum())
        y = z[:, 1] - (q1 * z[:, 1]).sum() * q1
        y = y - (q1 * y).sum() * q1
        return np.stack([q1, y / np.sqrt((y * y).sum())], 1)

    c = np.bincount(cols, minlength=n).astype(real)[:, None]
    by_col = np.argsort(cols, kind="stable")
    x = qr(wo.start_block(5, 0, m).astype(real))
    y = product(cols[by_col], rows[by_col], n, x) - c * (x.sum(0) / m)
    return qr(product(rows, cols, m, y) - (c * y).sum(0) / m)


# rows of one or two blocks: the entries of a sweep are far below what a mask of that size can reach
@pytest.mark.parametrize("m,blocks", [(14336, 1), (14336, 2), (2841, 1), (300, 2)])
def test_products_of_sparse_masks_are_as_close_as_fp64_sums(m, blocks):
    rng = np.random.default_rng(3)
    mask = torch.zeros((1, m, m), dtype=torch.bool, device="cuda")
    mask[0, torch.arange(m, device="cuda").repeat_interleave(blocks), torch.from_numpy(rng.integers(0, m, m * blocks)).cuda()] = True
    rows, cols = (x.cpu().numpy() for x in mask[0].nonzero(as_tuple=True))
    d = wb.plan_desc_default(heads=1, n_q_blocks=m, n_kv_blocks=m, wave_size=148, mode=wb.FORCE_REORDER, seed=5, svd_iters=1)
    e = wb.plan_bitmap(d, _pack(mask), debug=True).embedding[0].cpu().numpy()
    exact = _first_sweep(rows, cols, m, m, np.longdouble)

    def off(u):                                   # part of u outside the exact plane (rotation, sign and scale drop out)
        u = u.astype(np.longdouble)
        r = u - exact @ (exact.T @ u)
        return float(np.sqrt((r * r).sum() / (u * u).sum()))

    # (the last QR step's own rounding is in both; 1.5: the kernel's sums are not NumPy's)
    assert off(e) <= 1.5 * off(_first_sweep(rows, cols, m, m, np.float64))


@pytest.mark.parametrize("m", [9600, 9601])       # the second sort buffer fits shared memory, or not
def test_sorts_of_many_rows(m):
    mask = _mask(1, m, 64, 0.3, m)
    mask[0, 1::3] = mask[0, 0]                    # equal rows, equal angles: ties by row
    r = _plan(mask, wave=500)
    order1 = r.order1[0].cpu().numpy().astype(np.int64)
    assert np.array_equal(order1, wo.stage1_order(wo.polar_angles(r.embedding[0].cpu().numpy())))
    assert np.array_equal(r.row_order[0].cpu().numpy(), wo.stage2_order(order1, mask[0].sum(1).cpu().numpy(), 500))


# 16,384 words: the last size without a counting launch; blocks of one step, then of more; a row of several blocks
@pytest.mark.parametrize("H,m,n", [(1, 1, 1), (1, 16384, 64), (1, 16385, 64), (2, 8192, 64 * 32 + 1), (1, 3, 70001)])
def test_list_conversions(H, m, n):
    mask = _mask(H, m, n, 0.05, 3)
    mask[:, 0] = True
    mask[:, m // 2] = m == 1
    bm = _pack(mask)
    ptr, idx = wb.bitmap_to_csr(bm, n)
    flat = mask.reshape(H * m, n)
    assert torch.equal(ptr[1:].long(), flat.sum(1).cumsum(0)) and ptr[0].item() == 0
    assert torch.equal(idx, flat.nonzero()[:, 1].int())
    # either can be kept without the other
    assert ptr.untyped_storage().nbytes() <= 8 * ptr.numel() and idx.untyped_storage().nbytes() == 4 * max(1, idx.numel())
    half, first = wb.bitmap_to_csr(bm, n, capacity=idx.numel() // 2)       # lists that end early: the rest is left out
    assert torch.equal(half, ptr) and torch.equal(first, idx[:idx.numel() // 2])
    if m <= 8192:                                                          # and back (8,192 columns at a time)
        d = wb.plan_desc_default(heads=H, n_q_blocks=m, n_kv_blocks=n, wave_size=148, mode=wb.FORCE_NATURAL)
        a, b = wb.plan_csr(d, ptr, idx, debug=True), wb.plan_bitmap(d, bm, debug=True)
        assert torch.equal(a.col_count, b.col_count) and torch.equal(a.row_nnz, b.row_nnz) and a.dev_status.tolist() == [0] * 4


# one piece of 8,192 columns, and rows of two and three: runs of eight entries inside a piece, across its end, repeated, descending
# and with entries out of range in them
@pytest.mark.parametrize("n", [8191, 8192, 8193, 16384, 20000])
def test_lists_of_any_order_with_entries_out_of_range(n):
    rng = np.random.default_rng(n)
    bad = np.array([-1, n, n + 5, -2 ** 31, 2 ** 31 - 1])
    lists = [rng.permutation(n)[:1000], np.arange(n), np.arange(n)[::-1], np.repeat(rng.integers(0, n, 50), 3), [], [n - 1],
             np.arange(max(0, 8192 - 21), min(n, 8192 + 20)), np.concatenate([rng.integers(0, n, 101), bad, rng.integers(0, n, 7)]),
             np.insert(np.sort(rng.permutation(n)[:300]), [0, 13, 100, 299, 300], bad)]
    lists = [np.asarray(l, dtype=np.int64) for l in lists]
    mask = np.zeros((len(lists), n), dtype=bool)
    for i, l in enumerate(lists):
        mask[i, l[(l >= 0) & (l < n)]] = True
    d = wb.plan_desc_default(heads=1, n_q_blocks=len(lists), n_kv_blocks=n, wave_size=148, mode=wb.FORCE_NATURAL)
    for keep in (lists[:7] + [np.zeros(0, np.int64)] * 2, lists):
        ptr = torch.tensor([0] + [len(l) for l in keep]).cumsum(0).int().cuda()
        r = wb.plan_csr(d, ptr, torch.from_numpy(np.concatenate(keep)).int().cuda(), debug=True)
        rows = 7 if keep is not lists else 9
        assert r.row_nnz[0, :rows].tolist() == mask[:rows].sum(1).tolist()
        assert np.array_equal(r.col_count[0].cpu().numpy(), mask[:rows].sum(0))
        st = r.dev_status.tolist()
        assert st == [0] * 4 if rows == 7 else (st[:3] == [wb.ERR_BAD_MASK, 1, 0] and st[3] in bad)


def test_host_threads_plan_different_sizes():
    """A small plan must not take from a large one, between that one's set-up and its launches, the shared
    memory they need."""
    lib, jobs, failed = wb.load(), [], []
    for m, n in ((64, 64), (16384, 64), (128, 64), (4700, 300)):
        mask = _mask(1, m, n, 0.1, m)
        d = wb.plan_desc_default(heads=1, n_q_blocks=m, n_kv_blocks=n, wave_size=148, mode=wb.FORCE_NATURAL, seed=5)
        ws = torch.empty((wb.plan_workspace_bytes(d) + 256,), dtype=torch.uint8, device="cuda")
        jobs.append((d, _pack(mask), ws, wb.plan_bitmap(d, _pack(mask), workspace=ws), mask.sum(2), torch.cuda.Stream()))
    torch.cuda.synchronize()

    def work(d, bits, ws, res, nnz, stream):
        out = wb.PlanOut(row_order=res.row_order.data_ptr(), row_nnz=res.row_nnz.data_ptr())
        args = (ctypes.byref(d), bits.data_ptr(), ws.data_ptr(), ws.numel(), ctypes.byref(out), stream.cuda_stream)
        for _ in range(4000):                     # (the library call alone: the threads run it side by side)
            status = lib.waveal_plan_bitmap(*args)
            if status != wb.OK:
                failed.append((d.n_q_blocks, status, wb.last_error()))
                return

    threads = [threading.Thread(target=work, args=j) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not failed, failed
    for _, _, _, res, nnz, _ in jobs:
        assert torch.equal(res.row_nnz.long(), nnz)


def _attend(q, k, v, block, ptr, idx, T, order=None, flags=0, interleaved=False):
    o = torch.full_like(q, float("nan"))
    lse = torch.full(q.shape[:2], float("nan"), device="cuda")
    d = wb.attn_desc(q, k, v, o, T, T, block, interleaved, flags=flags)
    ws = torch.empty((wb.bsattn_workspace_bytes(d),), dtype=torch.uint8, device="cuda")
    st = torch.zeros((4,), dtype=torch.int32, device="cuda")
    wb.bsattn_fwd(d, q, k, v, o, ptr, idx, row_order=order, lse=lse, workspace=ws, dev_status=st)
    torch.cuda.synchronize()
    assert st.tolist() == [0] * 4
    return o, lse, ws.view(torch.int32)[:8].tolist()


def _inputs(H, T, D, seed):
    g = torch.Generator("cuda")
    g.manual_seed(seed)
    return [torch.randn((H, T, D), generator=g, device="cuda").to(torch.bfloat16) for _ in range(3)]


# tasks of 0 to 5 blocks one behind the other (1,023 to 1,025 of them: the tail takes the last 1,024), in natural and
# reversed order, with a ragged last block
@pytest.mark.parametrize("block,D", [(128, 128), (128, 64), (64, 128), (64, 64)])
@pytest.mark.parametrize("tasks", [1, 150, 1023, 1025])
def test_short_tasks_back_to_back(block, D, tasks):
    T = tasks * block - 37 if tasks > 1 else 90 - block // 2
    nb = (T + block - 1) // block
    counts = torch.tensor([(1, 0, 2, 1, 1, 3, 0, 0, 5, 1, 2, 4)[i % 12] for i in range(nb)]).clamp(max=nb)
    g = torch.Generator().manual_seed(tasks)
    lists = [torch.randperm(nb, generator=g)[:c].sort().values for c in counts.tolist()]
    ptr = torch.cat([torch.zeros(1, dtype=torch.long), counts.cumsum(0)]).int().cuda()
    idx = torch.cat(lists).int().cuda()
    q, k, v = _inputs(1, T, D, 1)
    o, lse, _ = _attend(q, k, v, block, ptr, idx, T)
    back, lse_back, _ = _attend(q, k, v, block, ptr, idx, T, order=torch.arange(nb - 1, -1, -1, device="cuda", dtype=torch.int32))
    assert torch.equal(o, back) and torch.equal(lse, lse_back)
    pad = torch.nn.functional.pad
    qf, kf, vf, of = (pad(x[0].double(), (0, 0, 0, nb * block - T)).view(nb, block, D) for x in (q, k, v, o))
    lf = pad(lse[0].double(), (0, nb * block - T)).view(nb, block)
    exists = torch.arange(nb * block, device="cuda").view(nb, block) < T
    for c in counts.unique().tolist():
        rows = (counts == c).nonzero()[:, 0].cuda()
        live, got, got_lse = exists[rows], of[rows], lf[rows]
        if c == 0:
            assert (got[live] == 0).all() and (got_lse[live] == -float("inf")).all()
            continue
        sel = torch.stack([lists[i] for i in rows.tolist()]).cuda()
        K, V = kf[sel].flatten(1, 2), vf[sel].flatten(1, 2)
        s = (qf[rows] @ K.transpose(1, 2) / D ** 0.5).masked_fill(~exists[sel].flatten(1)[:, None, :], -float("inf"))
        p = s.softmax(-1)
        ref = p @ V
        # P is cut to bf16 (each weight within 2^-8 of itself) and O rounded to bf16
        bound = 2.0 ** -8 * (p @ V.abs()) + 2.0 ** -8 * ref.abs() + 1e-6
        assert ((got - ref).abs() <= bound)[live].all()
        # the polynomial share of the exponentials is within 7.5e-5 of itself, fp32 scores and logarithm add a few 1e-6
        assert ((got_lse - s.logsumexp(-1)).abs() <= 1.5e-4)[live].all()


# O leaves in boxes of 32 rows and half of head_dim: the last box whole, cut and left out; rows of O with other tensors'
# rows between them, at 16-byte boundaries, and nothing written behind seq_q
@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("cut", [0, 1, 31, 32, 33, 64, 95, 96, 127])
def test_stores_end_with_the_sequence(D, cut):
    H, nb, block = 2, 3, 128
    T = nb * block - cut
    q, k, v = _inputs(H, nb * block, D, cut)
    ptr = torch.arange(0, 2 * H * nb + 1, 2, device="cuda", dtype=torch.int32)
    idx = torch.tensor([0, 2, 0, 1, 1, 2], device="cuda", dtype=torch.int32).repeat(H)
    buf = torch.full((nb * block, H, D + 8), float("nan"), dtype=torch.bfloat16, device="cuda")
    o = buf[:, :, 8:].permute(1, 0, 2)
    st = torch.zeros((4,), dtype=torch.int32, device="cuda")
    wb.bsattn_fwd(wb.attn_desc(q, k, v, o, T, T, block), q, k, v, o, ptr, idx, dev_status=st)
    torch.cuda.synchronize()
    assert st.tolist() == [0] * 4
    assert torch.isnan(buf[:, :, :8]).all() and torch.isnan(buf[T:]).all()
    for i, pair in enumerate(((0, 2), (0, 1), (1, 2))):
        sel = torch.cat([torch.arange(j * block, min((j + 1) * block, T)) for j in pair]).cuda()
        rows = slice(i * block, min((i + 1) * block, T))
        p = (q[:, rows].double() @ k[:, sel].double().transpose(1, 2) / D ** 0.5).softmax(-1)
        ref = p @ v[:, sel].double()
        bound = 2.0 ** -8 * (p @ v[:, sel].double().abs()) + 2.0 ** -8 * ref.abs() + 1e-6      # as in the test above
        assert ((o[:, rows].double() - ref).abs() <= bound).all()


# heads of unequal row lengths, more tickets than the sorted tail: no order of heads or rows shows in the results
@pytest.mark.parametrize("block,nb", [(128, 420), (64, 420), (128, 300)])
def test_tail_over_several_heads(block, nb):
    H = 3
    mask = torch.cat([_mask(1, nb, nb, dens, nb + i) for i, dens in enumerate((0.01, 0.08, 0.03))])
    mask[1, 5] = True
    mask[2, 9] = False
    ptr, idx = wb.bitmap_to_csr(_pack(mask), nb)
    T = nb * block - 11
    q, k, v = _inputs(H, T, 64, 6)
    order = torch.stack([torch.randperm(nb, generator=torch.Generator().manual_seed(h)) for h in range(H)]).int().cuda()
    o, lse, w = _attend(q, k, v, block, ptr, idx, T)
    for order_i in (None, order):
        for interleaved in (False, True):
            o2, lse2, w2 = _attend(q, k, v, block, ptr, idx, T, order=order_i, interleaved=interleaved)
            assert torch.equal(o, o2) and torch.equal(lse, lse2)
            assert w2[0] >= H * nb
    assert (o[2, 9 * block:10 * block] == 0).all() and not torch.isnan(o).any()
    for h, i in ((0, 0), (1, 5), (2, nb - 1)):
        blocks = mask[h, i].nonzero()[:, 0]
        sel = (blocks[:, None] * block + torch.arange(block, device="cuda")).flatten()
        sel = sel[sel < T]
        s = q[h, i * block:(i + 1) * block].double() @ k[h, sel].double().T / 8.0
        p = s.softmax(-1)
        ref = p @ v[h, sel].double()
        bound = 2.0 ** -8 * (p @ v[h, sel].double().abs()) + 2.0 ** -8 * ref.abs() + 1e-6      # as in the test above
        assert ((o[h, i * block:(i + 1) * block].double() - ref).abs() <= bound).all()


# rows that select everything stand in several blocks of 64 positions, an odd number of them, besides equal neighbours
@pytest.mark.parametrize("nb,full", [(65, [0, 63, 64]), (150, [5, 63, 64, 66, 128, 130, 149]), (130, [70])])
def test_pairs_across_blocks_of_positions(nb, full):
    mask = _mask(2, nb, nb, 0.15, nb)
    mask[:, full] = True
    mask[0, 21] = mask[0, 20]
    mask[1, 23] = mask[1, 22]
    mask[1, 25] = mask[1, 24]
    ptr, idx = wb.bitmap_to_csr(_pack(mask), nb)
    q, k, v = _inputs(2, nb * 64, 64, 2)
    order = torch.stack([torch.randperm(nb, generator=torch.Generator().manual_seed(h)) for h in range(2)]).int().cuda()
    o, lse, w = _attend(q, k, v, 64, ptr, idx, nb * 64)
    alone, lse_alone, w_alone = _attend(q, k, v, 64, ptr, idx, nb * 64, flags=wb.ATTN_NO_ROW_PAIRING)
    mixed, lse_mixed, w_mixed = _attend(q, k, v, 64, ptr, idx, nb * 64, order=order)
    assert torch.equal(o, alone) and torch.equal(lse, lse_alone) and torch.equal(o, mixed) and torch.equal(lse, lse_mixed)
    tiles = int(((mask.sum(2) + 1) // 2).sum())
    assert w_alone[6] == 0 and w_alone[7] == tiles
    assert w[6] == 2 * (len(full) // 2) + 3 and w_mixed[6] >= 2 * (len(full) // 2)
    shared = 2 * (len(full) // 2) * ((nb + 1) // 2) + sum(int((mask[h, i].sum() + 1) // 2) for h, i in ((0, 20), (1, 22), (1, 24)))
    assert w[7] == tiles - shared


@pytest.mark.parametrize("block", [64, 128])
def test_a_captured_step_replays(block):
    nb, D = 200, 64
    mask = _mask(2, nb, nb, 0.1, 4)
    bm, pairs = _pack(mask), int(mask.sum())
    q, k, v = _inputs(2, nb * block, D, 3)
    o = torch.zeros_like(q)
    pd = wb.plan_desc_default(heads=2, n_q_blocks=nb, n_kv_blocks=nb, wave_size=148, mode=wb.FORCE_REORDER, seed=1)
    pws = torch.empty((wb.plan_workspace_bytes(pd) + 256,), dtype=torch.uint8, device="cuda")
    ad = wb.attn_desc(q, k, v, o, nb * block, nb * block, block)
    aws = torch.empty((wb.bsattn_workspace_bytes(ad),), dtype=torch.uint8, device="cuda")

    def step():
        ptr, idx = wb.bitmap_to_csr(bm, nb, capacity=pairs)
        plan = wb.plan_bitmap(pd, bm, workspace=pws)
        wb.bsattn_fwd(ad, q, k, v, o, ptr, idx, row_order=plan.row_order, workspace=aws)
        return plan.row_order

    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        order = step().clone()
    torch.cuda.synchronize()
    ref = o.clone()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        replayed = step()
    o.zero_()
    graph.replay()
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(o, ref) and torch.equal(replayed, order)
    del graph
