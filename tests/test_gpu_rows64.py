"""64-row blocks: the first launch of large calls runs them in products of 64 rows, an item (one block, 128 keys) at a time, four
softmax groups and three P buffers in turn, or in products of 128 rows, whichever is quicker for the call's lists; small calls in
products of 128.  Lengths at every remainder, blocks that share their tiles with a second one, half tiles and ragged ends, tasks
that are computed again, malformed lists, strides, captured calls, and a tile that never comes, with the choice looked at."""
import time

import pytest
import torch

from paper_2609_34814_b200 import binding as wb

pytestmark = pytest.mark.gpu


def _call(q, k, v, ptr, idx, T, order=None, flags=0, ws=None, seq_kv=None):
    o, lse = torch.full_like(q, float("nan")), torch.full(q.shape[:2], float("nan"), device="cuda")[:, :T].contiguous()
    d = wb.attn_desc(q, k, v, o, T, seq_kv or T, 64, flags=flags)
    # (as an earlier call may have left it)
    ws = torch.full((wb.bsattn_workspace_bytes(d),), 127, dtype=torch.uint8, device="cuda") if ws is None else ws
    st = torch.zeros((4,), dtype=torch.int32, device="cuda")
    wb.bsattn_fwd(d, q, k, v, o, ptr, idx, row_order=order, lse=lse, workspace=ws, dev_status=st)
    torch.cuda.synchronize()
    return o, lse, ws.view(torch.int32), st.tolist()


def _rows128(w, tasks):
    """The choice that the call made on the device: products of 128 rows (1) or of 64 (0)."""
    return w[(32 + 8 * tasks + 31) // 32 * 8 + 7].item()


def _case(D, nb, cut, seed, full=True):
    """Rows of 0 to 45 blocks; every fifth row has its neighbour's list, every eleventh selects everything (`full`)."""
    g = torch.Generator().manual_seed(seed)
    lists = []
    for i in range(nb):
        n = min(int(torch.randint(0, 46, (1,), generator=g)), nb)
        l = torch.randperm(nb, generator=g)[:n].sort().values
        lists.append(lists[-1] if i % 5 == 1 else torch.arange(nb) if full and i % 11 == 3 else l)
    ptr = torch.tensor([0] + [len(l) for l in lists]).cumsum(0).int().cuda()
    gg = torch.Generator("cuda")
    gg.manual_seed(seed)
    q, k, v = (torch.randn((1, nb * 64, D), generator=gg, device="cuda").to(torch.bfloat16) for _ in range(3))
    return q, k, v, ptr, torch.cat(lists).int().cuda(), lists, nb * 64 - cut


@pytest.mark.parametrize("D", [128, 64])
@pytest.mark.parametrize("nb,cut,full", [(3, 1, True), (90, 63, True), (310, 1, True), (700, 0, True), (701, 40, True),
                                         (700, 0, False), (701, 40, False), (760, 63, False)])
def test_items_of_single_and_shared_blocks(D, nb, cut, full):
    q, k, v, ptr, idx, lists, T = _case(D, nb, cut, nb + D, full)
    o, lse, w, st = _call(q, k, v, ptr, idx, T)
    assert st == [0] * 4 and w[2] == 0
    alone, lse_alone, w_alone, _ = _call(q, k, v, ptr, idx, T, flags=wb.ATTN_NO_ROW_PAIRING)
    if nb >= 310:                                 # pairs of full rows outlast the call in products of 64 rows; short ones run there
        assert _rows128(w, nb) == full and _rows128(w_alone, nb) == 0
    assert w_alone[6] == 0 and w_alone[7] == sum((len(l) + 1) // 2 for l in lists) and (nb < 90 or w[6] > nb // 30)
    back, lse_back, _, _ = _call(q, k, v, ptr, idx, T, order=torch.arange(nb - 1, -1, -1, device="cuda", dtype=torch.int32))
    for other, lse_other in ((alone, lse_alone), (back, lse_back)):
        assert torch.equal(o[:, :T], other[:, :T]) and torch.equal(lse, lse_other)
    assert torch.isnan(o[:, T:].float()).all()
    for i in sorted({0, 1, 2, nb - 1, *range(3, nb, 13)}):
        rows = slice(i * 64, min((i + 1) * 64, T))
        if len(lists[i]) == 0:
            assert (o[0, rows] == 0).all() and (lse[0, rows] == -float("inf")).all()
            continue
        sel = (lists[i][:, None] * 64 + torch.arange(64)).flatten().cuda()
        sel = sel[sel < T]
        s = q[0, rows].double() @ k[0, sel].double().T / D ** 0.5
        p = s.softmax(-1)
        ref = p @ v[0, sel].double()
        # each weight is cut to bf16 (within 2^-8 of itself) and O rounded to bf16; 1e-6 for the fp32 sums
        bound = 2.0 ** -8 * (p @ v[0, sel].double().abs()) + 2.0 ** -8 * ref.abs() + 1e-6
        assert ((o[0, rows].double() - ref).abs() <= bound).all(), i
        # the polynomial share of the exponentials is within 7.5e-5 of itself, fp32 scores and logarithm add a few 1e-6
        assert ((lse[0, rows].double() - s.logsumexp(-1)).abs() <= 1.5e-4).all(), i


# full rows in pairs have all of the tiles, half or a few of them (products of 128 rows); the blocks on their own run in products of 64
# from 310 rows on, with the same bits
@pytest.mark.parametrize("D", [128, 64])
@pytest.mark.parametrize("nb,full", [(320, 320), (320, 120), (320, 12), (200, 80)])
def test_either_kernel_gives_the_same_bits(D, nb, full):
    g = torch.Generator().manual_seed(full)                   # (320 rows: up to 346 tiles an SM, 200: 135)
    lists = [torch.arange(nb) if i < full else torch.randperm(nb, generator=g)[:40 + i % 7].sort().values for i in range(nb)]
    ptr = torch.tensor([0] + [len(l) for l in lists]).cumsum(0).int().cuda()
    gg = torch.Generator("cuda")
    gg.manual_seed(full)
    T = nb * 64 - 21
    q, k, v = (torch.randn((1, nb * 64, D), generator=gg, device="cuda").to(torch.bfloat16) for _ in range(3))
    idx = torch.cat(lists).int().cuda()
    o, lse, w, st = _call(q, k, v, ptr, idx, T)
    alone, lse_alone, w_alone, _ = _call(q, k, v, ptr, idx, T, flags=wb.ATTN_NO_ROW_PAIRING)
    assert st == [0] * 4 and w[6] == full // 2 and w_alone[6] == 0 and w[7] == w_alone[7] - full // 2 * nb // 2
    assert nb == 200 or (_rows128(w, nb) == 1 and _rows128(w_alone, nb) == 0)
    assert torch.equal(o[:, :T], alone[:, :T]) and torch.equal(lse, lse_alone)
    for i in (0, 1, full - 1, min(full, nb - 1), nb - 1):
        rows = slice(i * 64, min((i + 1) * 64, T))
        sel = (lists[i][:, None] * 64 + torch.arange(64)).flatten().cuda()
        sel = sel[sel < T]
        p = (q[0, rows].double() @ k[0, sel].double().T / D ** 0.5).softmax(-1)
        ref = p @ v[0, sel].double()
        bound = 2.0 ** -8 * (p @ v[0, sel].double().abs()) + 2.0 ** -8 * ref.abs() + 1e-6      # as in the test above
        assert ((o[0, rows].double() - ref).abs() <= bound).all(), i


# one pair of 350 tiles among blocks of 10 to 15: it outlasts the call in products of 64 rows, in front of the last 1,024 tickets too
@pytest.mark.parametrize("D", [128, 64])
@pytest.mark.parametrize("at", [0, 1376])
def test_a_long_pair_decides_wherever_it_stands(D, at):
    heads, nb = 2, 700
    g = torch.Generator().manual_seed(at)
    lists = [torch.arange(nb) if t in (at, at + 1) else torch.randperm(nb, generator=g)[:20 + t % 11].sort().values for t in range(heads * nb)]
    ptr = torch.tensor([0] + [len(l) for l in lists]).cumsum(0).int().cuda()
    gg = torch.Generator("cuda")
    gg.manual_seed(at)
    q, k, v = (torch.randn((heads, nb * 64, D), generator=gg, device="cuda").to(torch.bfloat16) for _ in range(3))
    idx = torch.cat(lists).int().cuda()
    o, lse, w, st = _call(q, k, v, ptr, idx, nb * 64)
    alone, lse_alone, w_alone, st_alone = _call(q, k, v, ptr, idx, nb * 64, flags=wb.ATTN_NO_ROW_PAIRING)
    assert st == [0] * 4 and st_alone == [0] * 4 and w[6] == 1 and w_alone[6] == 0
    assert _rows128(w, heads * nb) == 1 and _rows128(w_alone, heads * nb) == 0
    assert torch.equal(o, alone) and torch.equal(lse, lse_alone)


# the single-launch variant has one kernel: nothing is chosen, and long pairs are not put in front of longer blocks
@pytest.mark.parametrize("D", [128, 64])
def test_the_single_launch_variant_chooses_nothing(D):
    nb, heads = 320, 2
    lists = [torch.arange(nb) if t % 8 < 2 else torch.arange(0, nb, 2) if t % 8 < 4 else torch.arange(t % 7, 250 + t % 7) for t in range(heads * nb)]
    ptr = torch.tensor([0] + [len(l) for l in lists]).cumsum(0).int().cuda()
    q, k, v = (torch.randn((heads, nb * 64, D), generator=torch.Generator("cuda").manual_seed(D), device="cuda").to(torch.bfloat16) for _ in range(3))
    o, _, w, st = _call(q, k, v, ptr, torch.cat(lists).int().cuda(), nb * 64, flags=wb.ATTN_ONLINE_MAX_ONLY)
    tasks = heads * nb
    table = w[(32 + 8 * tasks + 31) // 32 * 8:][:8 * tasks].view(tasks, 8)
    n = table[:, 3].tolist()                       # tiles of a ticket, longest first (absorbed ones last); 160 and 80 of the pairs
    assert st == [0] * 4 and wb.last_launch_count() == 3 and w[6] == tasks // 4 and not table[:, 7].any()
    assert n == sorted(n, reverse=True) and max(n) == 160


# calls on either side of the number of tiles from which the choice of kernel is made on the device, and of as many blocks as SMs
@pytest.mark.parametrize("D", [128, 64])
@pytest.mark.parametrize("nb,heads", [(100, 9), (200, 4)])
def test_a_head_has_the_same_bits_in_every_call(D, nb, heads):
    _, _, _, ptr, idx, lists, T = _case(D, nb, 13, nb + D)
    g = torch.Generator("cuda")
    g.manual_seed(nb)
    q, k, v = (torch.randn((heads, nb * 64, D), generator=g, device="cuda").to(torch.bfloat16) for _ in range(3))
    n = ptr[-1]
    all_ptr = torch.cat([ptr[:1]] + [ptr[1:] + h * n for h in range(heads)])
    o, lse, w, st = _call(q, k, v, all_ptr, idx.repeat(heads), T)
    assert st == [0] * 4 and w[2] == 0
    for h in range(heads):
        one, lse_one, w, st = _call(q[h:h + 1], k[h:h + 1], v[h:h + 1], ptr, idx, T)
        assert st == [0] * 4 and w[2] == 0
        assert torch.equal(one[0, :T], o[h, :T]) and torch.equal(lse_one[0], lse[h]), h


M, N = 500, 200                                  # query and key blocks: 337 tiles an SM that lists could have


def _lists(pairs, seed, first=()):
    """[M] lists of 4 to 19 of blocks 4 to N - 1, behind those of `first`; of the rows 2i + 1 none, a sixth or all have their neighbour's."""
    g = torch.Generator().manual_seed(seed)
    lists = []
    for i in range(M):
        l = torch.cat([torch.tensor(list(first), dtype=torch.long), 4 + torch.randperm(N - 4, generator=g)[:4 + i % 16].sort().values])
        lists.append(lists[-1] if i % 2 and (pairs == "all" or pairs == "some" and i % 6 == 1) else l)
    ptr = torch.tensor([0] + [len(l) for l in lists]).cumsum(0).int().cuda()
    return lists, ptr, torch.cat(lists).int().cuda()


def _tensors(D, seed):
    g = torch.Generator("cuda")
    g.manual_seed(seed)
    return [torch.randn((1, n * 64, D), generator=g, device="cuda").to(torch.bfloat16) for n in (M, N, N)]


def _assert_rows(q, k, v, o, lists, rows, T, S):
    for i in rows:
        at = slice(i * 64, min((i + 1) * 64, T))
        sel = (lists[i][:, None] * 64 + torch.arange(64)).flatten().cuda()
        sel = sel[sel < S]
        s = q[0, at].double() @ k[0, sel].double().T / q.shape[2] ** 0.5
        p = s.masked_fill(s < -1e30, -float("inf")).softmax(-1)
        V = v[0, sel].double()
        # as above; and fp32 scores of up to 200 nats: 200 * 2^-23 of every weight
        bound = (2.0 ** -8 + 2.5e-5) * (p @ V.abs()) + 2.0 ** -8 * (p @ V).abs() + 1e-6 * V.abs().max()
        assert ((o[0, at].double() - p @ V).abs() <= bound).all(), i


# What sends a task to the second launch: a key 60 or 200 nats above the rest behind a row's first 128 keys; V of 2^90 under sums of
# 2^46; a first tile without a finite score.  Query blocks whose first component is 0 do not see the key, but a pair is listed as two.
@pytest.mark.parametrize("D", [128, 64])
@pytest.mark.parametrize("pairs", ["none", "some", "all"])
@pytest.mark.parametrize("what", ["60 nats", "200 nats", "large values", "no reference", "nothing"])
def test_tasks_that_are_computed_again(D, pairs, what):
    hot, col, T, S = 150, 41, M * 64 - 9, N * 64 - 30
    q, k, v = _tensors(D, D)
    lists, ptr, idx = _lists(pairs, 3, first=(0, 1) if what == "no reference" else ())
    blind = torch.arange(M) % 4 == 1              # (second blocks of pairs, and single ones)
    if what == "no reference":
        q.abs_()
        k[0, :128] = -3e38
        k[0, 64 * 50:64 * 51] = -3e38             # (behind a reference: weights of 0)
        expected = list(range(M))
    else:
        q[0, :, 0] = torch.where(blind, 0.0, 8.0).repeat_interleave(64).cuda()
        k[..., 0] = 0.0
        k[0, hot * 64 + col] = 0.0
        k[0, hot * 64 + col, 0] = {"60 nats": 60.0, "200 nats": 200.0, "large values": 36.0, "nothing": 20.0}[what] * D ** 0.5 / 8
        if what == "large values":
            v.mul_(2.0 ** 90)
        late = [hot in l.tolist() and l.tolist().index(hot) >= 2 for l in lists]
        partner = [i ^ 1 if lists[i] is lists[i ^ 1] else i for i in range(M)]
        expected = [i for i in range(M) if what != "nothing" and late[i] and not (blind[i] and blind[partner[i]])]
        alone = [i for i in expected if not blind[i]]
    for flags in (0, wb.ATTN_NO_ROW_PAIRING):
        o, lse, w, st = _call(q, k, v, ptr, idx, T, flags=flags, seq_kv=S)
        assert st == [0] * 4 and (w[6] > 0) == (pairs != "none" and not flags)
        assert _rows128(w, M) == (pairs == "all" and not flags)
        listed = sorted(w[8:8 + 2 * int(w[2])].view(-1, 2)[:, 1].tolist())
        assert listed == (alone if flags and what != "no reference" else expected) and (what == "nothing" or len(listed) > 15)
        assert torch.isfinite(o[:, :T].float()).all() and torch.isfinite(lse).all() and torch.isnan(o[:, T:].float()).all()
        _assert_rows(q, k, v, o, lists, sorted({0, 1, 2, M - 1, *listed[:12], *range(5, M, 41)}), T, S)


# an index out of range inside a list (the last one is looked at before): reported once, block 0 in its place, the other rows as ever
@pytest.mark.parametrize("D", [128, 64])
@pytest.mark.parametrize("pairs", ["none", "all"])
def test_an_index_out_of_range_inside_a_list(D, pairs):
    q, k, v = _tensors(D, 1)
    lists, ptr, idx = _lists(pairs, 1)
    for row, at, bad in ((0, 0, -4), (77, 3, N), (M - 2, 8, 2 ** 31 - 1)):
        broken, zero = idx.clone(), idx.clone()
        for r in [row, row + 1] if pairs == "all" and row % 2 == 0 else [row]:       # (a pair's lists stay equal)
            e = int(ptr[r]) + min(at, len(lists[r]) - 2)
            broken[e], zero[e] = bad, 0
        o, lse, w, st = _call(q, k, v, ptr, broken, M * 64, seq_kv=N * 64)
        assert st == [wb.ERR_BAD_MASK, 30, 0, bad] and _rows128(w, M) == (pairs == "all")
        ref, lse_ref, _, st = _call(q, k, v, ptr, zero, M * 64, seq_kv=N * 64)
        assert st == [0] * 4 and torch.equal(o, ref) and torch.equal(lse, lse_ref)


# Q, K and V in one tensor, O between other tensors' columns at 32- and at 16-byte boundaries: the bits of the contiguous call
@pytest.mark.parametrize("D", [128, 64])
@pytest.mark.parametrize("pad", [8, 16])
@pytest.mark.parametrize("full", [False, True])
def test_strided_tensors(D, pad, full):
    _, _, _, ptr, idx, lists, T = _case(D, 310, 21, 8, full)
    H, nb = 2, 310
    ptr, idx = torch.cat([ptr, ptr[1:] + ptr[-1]]), idx.repeat(H)
    g = torch.Generator("cuda")
    g.manual_seed(D)
    fused = torch.randn((nb * 64, 3, H, D), generator=g, device="cuda").to(torch.bfloat16)
    views = [fused[:, i].permute(1, 0, 2) for i in range(3)]
    ref, lse_ref, w, st = _call(*(x.contiguous() for x in views), ptr, idx, T)
    assert st == [0] * 4 and _rows128(w, H * nb) == full
    buf = torch.full((nb * 64, H, D + pad), float("nan"), dtype=torch.bfloat16, device="cuda")
    o, lse = buf[:, :, pad:].permute(1, 0, 2), torch.full_like(lse_ref, float("nan"))
    st = torch.zeros((4,), dtype=torch.int32, device="cuda")
    wb.bsattn_fwd(wb.attn_desc(*views, o, T, T, 64), *views, o, ptr, idx, lse=lse, dev_status=st)
    torch.cuda.synchronize()
    assert st.tolist() == [0] * 4 and torch.equal(o[:, :T], ref[:, :T]) and torch.equal(lse, lse_ref)
    assert torch.isnan(buf[:, :, :pad]).all() and torch.isnan(buf[T:]).all()


# one captured call, replayed on lists that want the one kernel, the other, and the first again
@pytest.mark.parametrize("D", [128, 64])
def test_a_captured_call_chooses_at_every_replay(D):
    q, k, v = _tensors(D, 2)
    cases = []
    for pairs in ("none", "all"):
        _, ptr, idx = _lists(pairs, 4)
        o, _, w, st = _call(q, k, v, ptr, idx, M * 64, seq_kv=N * 64)
        assert st == [0] * 4 and _rows128(w, M) == (pairs == "all")
        cases.append((ptr, idx, o, _rows128(w, M)))
    ptr, idx = (torch.zeros((max(c[i].numel() for c in cases),), dtype=torch.int32, device="cuda") for i in (0, 1))
    o = torch.zeros_like(q)
    d = wb.attn_desc(q, k, v, o, M * 64, N * 64, 64)
    ws = torch.full((wb.bsattn_workspace_bytes(d),), 127, dtype=torch.uint8, device="cuda")
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        wb.bsattn_fwd(d, q, k, v, o, ptr, idx, workspace=ws)
    assert wb.last_launch_count() == 5
    for i in (0, 1, 0):
        ptr.copy_(cases[i][0])
        idx[:cases[i][1].numel()] = cases[i][1]
        o.zero_()
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(o, cases[i][2]) and _rows128(ws.view(torch.int32), M) == cases[i][3]
    del graph


@pytest.mark.parametrize("D", [128, 64])
@pytest.mark.parametrize("flags,rows128", [(0, 1), (wb.ATTN_NO_ROW_PAIRING, 0)])
def test_a_tile_that_never_comes(D, flags, rows128):
    q, k, v, ptr, idx, lists, T = _case(D, 400, 17, 5)
    good, _, w, st = _call(q, k, v, ptr, idx, T, flags=flags)
    assert st == [0] * 4 and _rows128(w, 400) == rows128
    t0 = time.perf_counter()
    _, _, w, st = _call(q, k, v, ptr, idx, T, flags=flags | wb.ATTN_SELFTEST_LOST_TILE)
    assert time.perf_counter() - t0 < 1.0
    assert st[0] == wb.ERR_TIMEOUT and w[1] == 1 and _rows128(w, 400) == rows128, st
    for _ in range(8):                            # tensor memory was given back, the workspace is as good as new
        o, _, w, st = _call(q, k, v, ptr, idx, T, flags=flags, ws=w.view(torch.uint8))
        assert st == [0] * 4 and torch.equal(o[:, :T], good[:, :T])
