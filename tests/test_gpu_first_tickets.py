"""128-row blocks and two tasks an SM or more: every thread block takes the ticket of its own number before the kernel in
front of the call has made the task table and cleared the counters.  What a first task can meet besides its plain
path: it ends before that kernel and has to be computed again, its lists are malformed, a wait of it runs out."""
import time

import pytest
import torch

from paper_2609_34814_b200 import binding as wb

pytestmark = pytest.mark.gpu
H, NB, BLOCK, FIRST = 2, 160, 128, 148            # 320 tasks; tickets of the first tasks on a GPU of 148 SMs
T = NB * BLOCK


def _case(D, lists, seed=3):
    assert wb.default_wave_size() <= FIRST and 2 * wb.default_wave_size() <= H * NB
    g = torch.Generator("cuda")
    g.manual_seed(seed)
    q, k, v = (torch.randn((H, T, D), generator=g, device="cuda").to(torch.bfloat16) for _ in range(3))
    ptr = torch.tensor([0] + [len(x) for x in lists]).cumsum(0).int().cuda()
    return q, k, v, ptr, torch.tensor(sum(lists, []), dtype=torch.int32, device="cuda")


def _run(q, k, v, ptr, idx, order=None, ws=None, flags=0):
    o = torch.full_like(q, float("nan"))
    d = wb.attn_desc(q, k, v, o, T, T, BLOCK, flags=flags)
    if ws is None:
        # (as an earlier call may have left it: the counters are cleared by the call)
        ws = torch.full((wb.bsattn_workspace_bytes(d),), 127, dtype=torch.uint8, device="cuda")
    st = torch.zeros((4,), dtype=torch.int32, device="cuda")
    wb.bsattn_fwd(d, q, k, v, o, ptr, idx, row_order=order, workspace=ws, dev_status=st)
    torch.cuda.synchronize()
    return o, ws.view(torch.int32), st.tolist()


def _assert_close(q, k, v, o, lists, tasks):
    for t in tasks:
        h, i = divmod(t, NB)
        rows = slice(i * BLOCK, (i + 1) * BLOCK)
        sel = (torch.tensor(lists[t], device="cuda")[:, None] * BLOCK + torch.arange(BLOCK, device="cuda")).flatten()
        p = (q[h, rows].double() @ k[h, sel].double().T / q.shape[2] ** 0.5).softmax(-1)
        V = v[h, sel].double()
        # P and O are rounded to bf16 (2^-9 of each, twice that for P, which is cut); 1e-6 for the fp32 sums
        bound = 2.0 ** -8 * (p @ V.abs()) + 2.0 ** -8 * (p @ V).abs() + 1e-6
        assert ((o[h, rows].double() - p @ V).abs() <= bound).all(), t


def _plain_lists():
    """Two tiles a first task (it ends before the table is there), one to five the others."""
    return [[i % 7, 20 + i % 100] if t < FIRST else [0, 9, 30 + i % 50, 100, 140][:1 + i % 5]
            for t in range(H * NB) for i in (t % NB,)]


@pytest.mark.parametrize("D", [128, 64])
def test_first_tasks_that_are_computed_again(D):
    hot = 150
    lists = _plain_lists()
    for t in range(H * NB):
        if t % 3 == 1:
            lists[t] = lists[t][:1] + [hot]       # 200 nats above the reference, in the second tile
        elif t % 12 == 2:
            lists[t] = [hot] + lists[t][1:2]      # in the first one: it is the reference
    q, k, v, ptr, idx = _case(D, lists)
    q[..., 0] = 8.0
    k[..., 0] = 0.0
    k[:, hot * BLOCK + 57] = 0.0
    k[:, hot * BLOCK + 57, 0] = 200.0 * D ** 0.5 / 8.0
    o, w, st = _run(q, k, v, ptr, idx)
    assert st == [0] * 4
    listed = sorted(NB * h + i for h, i in w[8:8 + 2 * int(w[2])].view(-1, 2).tolist())
    assert listed == [t for t in range(H * NB) if t % 3 == 1]
    assert not torch.isnan(o).any()
    _assert_close(q, k, v, o, lists, range(H * NB))


@pytest.mark.parametrize("D", [128, 64])
def test_malformed_lists_of_first_tasks_are_reported_not_followed(D):
    lists = _plain_lists()
    q, k, v, ptr, idx = _case(D, lists)
    good, _, st = _run(q, k, v, ptr, idx)
    assert st == [0] * 4
    _assert_close(q, k, v, good, lists, list(range(0, H * NB, 9)))
    blocks = lambda x: x.view(H, NB, BLOCK, D)

    def check(result, status, empty=(), other=()):
        o, _, st = result
        assert st == status
        same = torch.ones((H, NB), dtype=torch.bool, device="cuda")
        for i in (*empty, *other):
            same[0, i] = False
        for i in empty:
            assert (blocks(o)[0, i] == 0).all()
        assert torch.equal(blocks(o)[same], blocks(good)[same])

    order = torch.arange(NB, dtype=torch.int32, device="cuda").repeat(H, 1)
    order[0, 5] = NB + 3
    check(_run(q, k, v, ptr, idx, order=order), [wb.ERR_BAD_MASK, 31, 0, NB + 3], empty=(5,))
    bad = ptr.clone()
    bad[41] = bad[40] - 1                         # row 40's list ends before it starts, row 41's starts there
    check(_run(q, k, v, bad, idx), [wb.ERR_BAD_MASK, 32, 0, int(bad[41])], empty=(40,), other=(41,))
    bad = idx.clone()
    bad[int(ptr[78]) - 1] = NB + 7                # the last entry of row 77
    check(_run(q, k, v, ptr, bad), [wb.ERR_BAD_MASK, 33, 0, NB + 7], empty=(77,))
    bad = idx.clone()
    bad[int(ptr[FIRST - 1])] = -4                 # an entry inside a list: block 0 in its place
    check(_run(q, k, v, ptr, bad), [wb.ERR_BAD_MASK, 30, 0, -4], other=(FIRST - 1,))
    check(_run(q, k, v, ptr, idx), [0] * 4)


@pytest.mark.parametrize("D", [128, 64])
def test_a_first_task_whose_wait_runs_out(D):
    """The loader never requests the first K tile of ticket 0, which a thread block has without asking."""
    lists = _plain_lists()
    q, k, v, ptr, idx = _case(D, lists)
    t0 = time.perf_counter()
    _, w, st = _run(q, k, v, ptr, idx, flags=wb.ATTN_SELFTEST_LOST_TILE)
    assert time.perf_counter() - t0 < 1.0
    assert st[0] == wb.ERR_TIMEOUT and st[1] in (3, 4, 12, 14, 21) and st[2] == 0, st
    assert int(w[1]) == 1                         # the flag that the other thread blocks see
    for _ in range(3):                            # ordinary calls on the same workspace
        o, w, st = _run(q, k, v, ptr, idx, ws=w.view(torch.uint8))
        assert st == [0] * 4 and w[1:4].tolist()[:2] == [0, 0]
    _assert_close(q, k, v, o, lists, list(range(0, H * NB, 5)))
