"""64-row blocks: the first launch runs them in products of 64 rows, an item (one block, 128 keys) at a time, four softmax
groups and three P buffers in turn.  Lengths at every remainder of those, blocks that share their tiles with a second one,
half tiles and ragged ends, and what the kernel does when a tile never comes."""
import time

import pytest
import torch

from paper_2609_34814_b200 import binding as wb

pytestmark = pytest.mark.gpu


def _call(q, k, v, ptr, idx, T, order=None, flags=0, ws=None):
    o, lse = torch.full_like(q, float("nan")), torch.full(q.shape[:2], float("nan"), device="cuda")[:, :T].contiguous()
    d = wb.attn_desc(q, k, v, o, T, T, 64, flags=flags)
    ws = torch.zeros((wb.bsattn_workspace_bytes(d),), dtype=torch.uint8, device="cuda") if ws is None else ws
    st = torch.zeros((4,), dtype=torch.int32, device="cuda")
    wb.bsattn_fwd(d, q, k, v, o, ptr, idx, row_order=order, lse=lse, workspace=ws, dev_status=st)
    torch.cuda.synchronize()
    return o, lse, ws.view(torch.int32), st.tolist()


def _rows128(w, tasks):
    """The choice that the call made on the device: products of 128 rows (1) or of 64 (0)."""
    return w[(32 + 8 * tasks + 31) // 32 * 8 + 7].item()


def _case(D, nb, cut, seed):
    """Rows of 0 to 45 blocks; every fifth row has its neighbour's list, every eleventh selects everything."""
    g = torch.Generator().manual_seed(seed)
    lists = []
    for i in range(nb):
        n = min(int(torch.randint(0, 46, (1,), generator=g)), nb)
        l = torch.randperm(nb, generator=g)[:n].sort().values
        lists.append(lists[-1] if i % 5 == 1 else torch.arange(nb) if i % 11 == 3 else l)
    ptr = torch.tensor([0] + [len(l) for l in lists]).cumsum(0).int().cuda()
    gg = torch.Generator("cuda")
    gg.manual_seed(seed)
    q, k, v = (torch.randn((1, nb * 64, D), generator=gg, device="cuda").to(torch.bfloat16) for _ in range(3))
    return q, k, v, ptr, torch.cat(lists).int().cuda(), lists, nb * 64 - cut


@pytest.mark.parametrize("D", [128, 64])
@pytest.mark.parametrize("nb,cut", [(3, 1), (90, 63), (310, 1), (700, 0), (701, 40)])
def test_items_of_single_and_shared_blocks(D, nb, cut):
    q, k, v, ptr, idx, lists, T = _case(D, nb, cut, nb + D)
    o, lse, w, st = _call(q, k, v, ptr, idx, T)
    assert st == [0] * 4 and w[2] == 0
    alone, lse_alone, w_alone, _ = _call(q, k, v, ptr, idx, T, flags=wb.ATTN_NO_ROW_PAIRING)
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


# pairs have all of the tiles, half or a few of them: products of 128 rows or of 64, with the same bits as the blocks on their own
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


@pytest.mark.parametrize("D", [128, 64])
def test_a_tile_that_never_comes(D):
    q, k, v, ptr, idx, lists, T = _case(D, 400, 17, 5)        # (541 tiles an SM: products of 64 rows)
    good, _, _, st = _call(q, k, v, ptr, idx, T)
    assert st == [0] * 4
    t0 = time.perf_counter()
    _, _, w, st = _call(q, k, v, ptr, idx, T, flags=wb.ATTN_SELFTEST_LOST_TILE)
    assert time.perf_counter() - t0 < 1.0
    assert st[0] == wb.ERR_TIMEOUT and w[1] == 1, st
    for _ in range(8):                            # tensor memory was given back, the workspace is as good as new
        o, _, w, st = _call(q, k, v, ptr, idx, T, ws=w.view(torch.uint8))
        assert st == [0] * 4 and torch.equal(o[:, :T], good[:, :T])
