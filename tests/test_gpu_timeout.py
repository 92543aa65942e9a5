"""The path a kernel takes when one of its bounded waits runs out.

Every wait inside the tensor-core kernels gives up after a clock budget, sets the device status word and lets the CTA
wind down: in-flight copies and products are awaited, tensor memory is released, nothing further is written, and the
CTAs that start afterwards return at once.  cosa_options.wait_cycles sets that budget per call; a budget of one cycle
makes every wait that is not satisfied on the spot run out, so the path is reached without any kernel ever waiting
for something that does not come.  After such a call cosa_device_status() reports COSA_ERR_DEVICE_TIMEOUT once, and
the same call with the default budget then gives the regular result.
"""
import numpy as np
import pytest
import torch

import paper_2607_25291_b200 as cosa
from synth.configs import WORKLOADS
from tests.helpers import alloc_lists, alloc_outputs, to_dev

pytestmark = pytest.mark.gpu

TIMEOUT = -5


@pytest.fixture(scope="module")
def cfg1():
    w = WORKLOADS["gqa4_4k"]
    qb, kb, vb, _ = w.make()
    return dict(w=w, dev=tuple(to_dev(x) for x in (qb, kb, vb)))


def test_kap_wait_budget_of_one_cycle_reports_a_timeout_and_the_next_call_is_clean(cfg1):
    w, (q, k, _) = cfg1["w"], cfg1["dev"]
    nqb = w.n // 128
    ref_order, ref_count = alloc_lists(w.hq, nqb)
    cosa.cosa_kap_select(q, k, w.kap_budget, ref_order, ref_count, opt=cosa.default_options(stride=w.stride))
    assert cosa.cosa_device_status() == 0
    order, count = alloc_lists(w.hq, nqb)
    cosa.cosa_kap_select(q, k, w.kap_budget, order, count, opt=cosa.default_options(stride=w.stride, wait_cycles=1))
    assert cosa.cosa_device_status() == TIMEOUT        # reported once ...
    assert cosa.cosa_device_status() == 0              # ... then cleared
    assert int((count == -7).sum()) == count.numel()   # the later kernels of the call wrote nothing
    cosa.cosa_kap_select(q, k, w.kap_budget, order, count, opt=cosa.default_options(stride=w.stride))
    assert cosa.cosa_device_status() == 0
    assert torch.equal(order, ref_order) and torch.equal(count, ref_count)


@pytest.mark.parametrize("impl", [0, 4, 5])     # one work item at a time, two side by side, the two row tiles of a 256-row block per CTA
def test_osk_wait_budget_of_one_cycle_reports_a_timeout_and_the_next_call_is_clean(cfg1, impl):
    w, (q, k, v) = cfg1["w"], cfg1["dev"]
    nqb = w.n // 128
    order, count = alloc_lists(w.hq, nqb)
    cosa.cosa_kap_select(q, k, w.kap_budget, order, count, opt=cosa.default_options(stride=w.stride),
                         block_q=256 if impl == 5 else 128)
    ref = alloc_outputs(q, nqb)
    cosa.cosa_osk_attention(q, k, v, order, count, w.osk_budget, ref["out"], ref["lse"], ref["visited"],
                            opt=cosa.default_options(skip_scale=w.skip_scale, impl=impl))
    assert cosa.cosa_device_status() == 0
    for _ in range(2):                                  # twice: a timed-out call leaves nothing behind that trips the next
        bufs = alloc_outputs(q, nqb)
        bufs["visited"].fill_(-7)
        cosa.cosa_osk_attention(q, k, v, order, count, w.osk_budget, bufs["out"], bufs["lse"], bufs["visited"],
                                opt=cosa.default_options(skip_scale=w.skip_scale, wait_cycles=1, impl=impl))
        assert cosa.cosa_device_status() == TIMEOUT
        assert cosa.cosa_device_status() == 0
        assert int((bufs["visited"] == -7).sum()) > 0   # the CTAs that started after the first timeout returned at once
    bufs = alloc_outputs(q, nqb)
    cosa.cosa_osk_attention(q, k, v, order, count, w.osk_budget, bufs["out"], bufs["lse"], bufs["visited"],
                            opt=cosa.default_options(skip_scale=w.skip_scale, impl=impl))
    assert cosa.cosa_device_status() == 0
    assert torch.equal(bufs["out"], ref["out"]) and torch.equal(bufs["visited"], ref["visited"])
    assert torch.equal(bufs["lse"], ref["lse"])


def test_status_word_set_by_hand_makes_both_stages_return_at_once(cfg1):
    """The same early return, reached without any wait: with the status word already set when the kernels start, they
    leave their outputs untouched; reading the status clears it."""
    w, (q, k, v) = cfg1["w"], cfg1["dev"]
    nqb = w.n // 128
    good_order, good_count = alloc_lists(w.hq, nqb)
    cosa.cosa_kap_select(q, k, w.kap_budget, good_order, good_count, opt=cosa.default_options(stride=w.stride))
    assert cosa.cosa_device_status() == 0
    cosa.cosa_debug_set_device_status(TIMEOUT)
    order, count = alloc_lists(w.hq, nqb)
    cosa.cosa_kap_select(q, k, w.kap_budget, order, count, opt=cosa.default_options(stride=w.stride))
    bufs = alloc_outputs(q, nqb)
    bufs["visited"].fill_(-7)
    bufs["out"].fill_(3.0)
    cosa.cosa_osk_attention(q, k, v, good_order, good_count, w.osk_budget, bufs["out"], bufs["lse"], bufs["visited"],
                            opt=cosa.default_options(skip_scale=w.skip_scale))
    assert cosa.cosa_device_status() == TIMEOUT
    assert cosa.cosa_device_status() == 0
    assert int((count == -7).sum()) == count.numel() and int((order == -7).sum()) == order.numel()
    assert int((bufs["visited"] == -7).sum()) == bufs["visited"].numel()
    assert bool((bufs["out"] == 3.0).all())


def test_osk_writes_no_decisions_of_a_walk_that_was_given_up(cfg1):
    """Budgets at which waits run out at every stage of a walk: the decisions of a work item (its 32 positions are one word,
    written when the walk reaches its end) are those of an undisturbed call or not written at all."""
    w, (q, k, v) = cfg1["w"], cfg1["dev"]
    nqb = w.n // 128
    order = torch.arange(nqb, dtype=torch.int32, device="cuda").expand(1, w.hq, nqb, nqb).contiguous()
    count = torch.full((1, w.hq, nqb), nqb, dtype=torch.int32, device="cuda")

    def words_and_visited(**kw):
        bufs = alloc_outputs(q, nqb)
        bufs["visited"].fill_(-7)
        cosa.cosa_osk_attention(q, k, v, order, count, 0.999, bufs["out"], bufs["lse"], bufs["visited"], causal=False,
                                opt=cosa.default_options(skip_scale=w.skip_scale, out_decisions=bufs["decisions"], **kw))
        assert cosa.cosa_device_status() in (0, TIMEOUT)
        return bufs["decisions"][0, :, :, 0], bufs["visited"][0]

    want, want_visited = words_and_visited()
    assert int((want == -1).sum()) < want.numel() // 2     # (most walks skip something)
    given_up = 0
    for cycles in range(200, 6200, 100):
        words, visited = words_and_visited(wait_cycles=cycles)
        done = visited != -7
        assert torch.equal(words[done], want[done]) and torch.equal(visited[done], want_visited[done]), cycles
        assert bool(((words == 0) | (words == want)).all()), cycles
        given_up += int((~done).sum())
    assert given_up > 0


@pytest.mark.parametrize("blocks,hq,hkv,lens", [
    (31, 32, 8, None), (61, 32, 8, None), (97, 32, 8, None), (257, 8, 2, None),      # a call of each form of the screen
    (32, 16, 4, (5, 32)), (64, 16, 4, (7, 50)), (100, 16, 4, (100, 9)), (260, 4, 1, (30, 260))])
def test_kap_call_that_gave_up_leaves_the_lists_as_they_were(blocks, hq, hkv, lens):
    """Budgets at which the waits of some CTAs run out and those of others do not: a call that reports a timeout has written no
    list and no count, those of query blocks that are padding included."""
    batch = 1 if lens is None else len(lens)
    g = torch.Generator(device="cuda").manual_seed(blocks)
    q, k = (torch.randn(batch, heads, blocks * 128, 128, device="cuda", generator=g).to(torch.bfloat16) for heads in (hq, hkv))
    extra = {} if lens is None else dict(seq_lens=torch.tensor([x * 128 for x in lens], dtype=torch.int32, device="cuda"))

    def lists(**kw):
        order = torch.full((batch, hq, blocks, blocks + 1), -7, dtype=torch.int32, device="cuda")
        count = torch.full((batch, hq, blocks), -7, dtype=torch.int32, device="cuda")
        cosa.cosa_kap_select(q, k, 0.3, order, count, opt=cosa.default_options(**extra, **kw))
        return order, count, cosa.cosa_device_status()

    want_order, want_count, status = lists()
    assert status == 0 and int(want_count.min()) >= (0 if lens else 1)
    given_up = 0
    for cycles in [1, 50, *range(200, 8200, 160), 20000, 50000]:
        order, count, status = lists(wait_cycles=cycles)
        if status == 0:
            assert torch.equal(order, want_order) and torch.equal(count, want_count), cycles
        else:
            assert status == TIMEOUT and bool((order == -7).all()) and bool((count == -7).all()), cycles
            given_up += 1
    assert given_up > 0
    for _ in range(20):          # a wait that is not satisfied on the spot is not slept through, either
        assert lists(wait_cycles=1)[2] == TIMEOUT
    cosa.cosa_debug_set_device_status(TIMEOUT)
    order, count, status = lists()
    assert status == TIMEOUT and bool((order == -7).all()) and bool((count == -7).all())


@pytest.mark.parametrize("tb", [1.0, 0.999])
def test_osk_writes_a_work_item_whole_or_not_at_all(tb):
    """Budgets at which waits run out at every stage of a walk, and, as one CTA does many short walks, in the load and issue warps
    while the rows write: out, lse, visited and scored of a work item are those of an undisturbed call, or all as they were."""
    hq, hkv, nqb = 32, 8, 31
    g = torch.Generator(device="cuda").manual_seed(3)
    q, k, v = (torch.randn(1, heads, nqb * 128, 128, device="cuda", generator=g).to(torch.bfloat16) for heads in (hq, hkv, hkv))
    order = torch.arange(nqb, dtype=torch.int32, device="cuda").expand(1, hq, nqb, nqb).contiguous()
    count = (torch.arange(nqb, dtype=torch.int32, device="cuda") % 6).expand(1, hq, nqb).contiguous()     # (and some empty ones)

    def call(**kw):
        bufs = alloc_outputs(q, nqb)
        bufs["out"].fill_(77.0)
        bufs["lse"].fill_(77.0)
        bufs["visited"].fill_(-7)
        bufs["scored"].fill_(-7)
        cosa.cosa_osk_attention(q, k, v, order, count, tb, bufs["out"], bufs["lse"], bufs["visited"], causal=False,
                                opt=cosa.default_options(skip_scale=500.0, out_scored=bufs["scored"], **kw))
        status = cosa.cosa_device_status()
        return [bufs["out"].view(-1, 128 * 128), bufs["lse"].view(-1, 128), bufs["visited"].view(-1, 1), bufs["scored"].view(-1, 1)], status

    want, status = call()
    assert status == 0
    in_part = 0
    for cycles in [*range(1000, 6000, 10)]:
        got, status = call(wait_cycles=cycles)
        assert status in (0, TIMEOUT)
        done = got[2][:, 0] != -7
        for a, b, blank in zip(got, want, (77.0, 77.0, -7, -7)):
            assert bool(torch.where(done[:, None], a == b, a == blank).all()), cycles
        in_part += int(bool(done.any()) and not bool(done.all()))
    assert in_part > 0


# the forms of the OSK kernel that the lists above (pitch 31 and 32) do not reach: (list pitch, Stage-2 cap, page size in place or 0)
SHORT_FORMS = [(8, 0.999, 0), (8, 0.999, 16), (31, 0.999, 16), (4, 1.0, 16), (31, 1.0, 16), (8, 1.0, 0)]


def _short_call(pitch, tb, page_size):
    """hq 32, hkv 8, 31 query blocks, lists of 0 to min(pitch, 5) blocks; returns call(**options) -> ([out, lse, visited, scored] by work
    item, status)."""
    hq, hkv, nqb = 32, 8, 31
    n = nqb * 128
    g = torch.Generator(device="cuda").manual_seed(3)
    q, k, v = (torch.randn(1, heads, n, 128, device="cuda", generator=g).to(torch.bfloat16) for heads in (hq, hkv, hkv))
    order = torch.arange(pitch, dtype=torch.int32, device="cuda").expand(1, hq, nqb, pitch).contiguous()
    count = (torch.arange(nqb, dtype=torch.int32, device="cuda") % (min(pitch, 5) + 1)).expand(1, hq, nqb).contiguous()
    paging = {}
    if page_size:
        table = torch.randperm(n // page_size, device="cuda", generator=g).to(torch.int32).view(1, -1).contiguous()
        pools = []
        for x in (k, v):
            pool = torch.empty(n // page_size, hkv, page_size, 128, dtype=torch.bfloat16, device="cuda")
            pool[table.view(-1).long()] = x.view(hkv, n // page_size, page_size, 128).transpose(0, 1)
            pools.append(pool)
        k, v = pools
        paging = dict(kv_page_table=table, kv_page_size=page_size, kv_num_pages=n // page_size, kv_pages_in_place=1)

    def call(**kw):
        bufs = alloc_outputs(q, nqb)
        bufs["out"].fill_(77.0)
        bufs["lse"].fill_(77.0)
        bufs["visited"].fill_(-7)
        bufs["scored"].fill_(-7)
        cosa.cosa_osk_attention(q, k, v, order, count, tb, bufs["out"], bufs["lse"], bufs["visited"], causal=False,
                                opt=cosa.default_options(skip_scale=500.0 if tb < 1 else -1.0, out_scored=bufs["scored"], order_stride=pitch, **paging, **kw))
        status = cosa.cosa_device_status()
        return [bufs["out"].view(-1, 128 * 128), bufs["lse"].view(-1, 128), bufs["visited"].view(-1, 1), bufs["scored"].view(-1, 1)], status

    return call


@pytest.mark.parametrize("pitch,tb,page_size", SHORT_FORMS)
def test_osk_writes_a_work_item_whole_or_not_at_all_on_every_form(pitch, tb, page_size):
    """The same budgets, and some at which the load warp leaves before it has read a work item (its first tile is then on its way all
    the same where the item warp asks for it)."""
    call = _short_call(pitch, tb, page_size)
    want, status = call()
    assert status == 0
    in_part = 0
    for cycles in [1, 20, 100, *range(200, 1000, 50), *range(1000, 9000, 25)]:
        got, status = call(wait_cycles=cycles)
        assert status in (0, TIMEOUT)
        done = got[2][:, 0] != -7
        for a, b, blank in zip(got, want, (77.0, 77.0, -7, -7)):
            assert bool(torch.where(done[:, None], a == b, a == blank).all()), cycles
        in_part += int(bool(done.any()) and not bool(done.all()))
    assert in_part > 0
    got, status = call()
    assert status == 0 and all(torch.equal(a, b) for a, b in zip(got, want))


@pytest.mark.parametrize("pitch,tb,page_size", SHORT_FORMS)
def test_osk_wait_budget_of_one_cycle_on_every_form(pitch, tb, page_size):
    call = _short_call(pitch, tb, page_size)
    want, status = call()
    assert status == 0
    for _ in range(20):
        got, status = call(wait_cycles=1)
        assert status == TIMEOUT and cosa.cosa_device_status() == 0
        assert int((got[2] == -7).sum()) > 0
    got, status = call()
    assert status == 0 and all(torch.equal(a, b) for a, b in zip(got, want))
