"""Device route planner vs the oracle: lists, lengths and pair counts must match bit for bit."""
import numpy as np
import pytest
import torch

import bf1_inputs as I
import paper_2608_20427_b200 as bf1
from oracle import bf1_oracle as O

pytestmark = pytest.mark.gpu

CASES = [
    [1], [63], [64], [65], [128], [257], [512], [1000], [2048], [4096], [8192], [16384], [32768],
    [3001, 8192, 12345, 16384], [130, 0, 257, 64, 1], [0, 0, 5], [70000],
]
CFGS = [dict(), dict(local_blocks=0), dict(local_blocks=5, global_first=0, dyadic=0),
        dict(global_first=0), dict(local_blocks=1, dyadic=0)]


def oracle_route(seqlens, kw, max_deg):
    c = O.cfg(**kw)
    seq, blk, cnt, idx, pairs = [], [], [], [], []
    for s, n in enumerate(seqlens):
        if n == 0:
            continue
        i, c_, p, _ = O.route(c, n, max_deg)
        B = len(c_)
        seq += [s] * B
        blk += list(range(B))
        cnt.append(c_)
        idx.append(i)
        pairs.append(p)
    if not cnt:
        return (np.zeros(0, np.int32),) * 3 + (np.zeros((0, max_deg), np.int32), np.zeros(0, np.int64))
    return (np.array(seq, np.int32), np.array(blk, np.int32), np.concatenate(cnt), np.concatenate(idx),
            np.concatenate(pairs))


@pytest.mark.parametrize("seqlens", CASES, ids=lambda s: "-".join(map(str, s)))
@pytest.mark.parametrize("kw", CFGS, ids=lambda k: ",".join("%s=%s" % i for i in k.items()) or "paper")
def test_planner_matches_oracle_bit_exact(seqlens, kw):
    dev = torch.device("cuda:0")
    cu = bf1.cu_seqlens_tensor(seqlens, dev)
    route = bf1.plan_route(cu, max(seqlens), bf1.RouteCfg(**kw))
    torch.cuda.synchronize()
    route.check_status()
    nqb = int(route.num_qblocks.item())
    seq, blk, cnt, idx, pairs = oracle_route(seqlens, kw, route.max_degree)
    assert nqb == len(seq)
    assert np.array_equal(route.qb_seq[:nqb].cpu().numpy(), seq)
    assert np.array_equal(route.qb_block[:nqb].cpu().numpy(), blk)
    assert np.array_equal(route.kv_count[:nqb].cpu().numpy(), cnt)
    assert np.array_equal(route.kv_idx[:nqb].cpu().numpy(), idx)
    assert np.array_equal(route.pair_count[:nqb].cpu().numpy().astype(np.int64), pairs)
    assert int(route.total_pairs.item()) == int(pairs.sum())
    # hand-out order: a permutation of the slots with non-increasing list length
    order = route.order[:nqb].cpu().numpy()
    assert np.array_equal(np.sort(order), np.arange(nqb))
    assert (np.diff(cnt[order]) <= 0).all()


def test_planner_flags_bad_sequence_lengths_without_faulting():
    dev = torch.device("cuda:0")
    cu = torch.tensor([0, 100, 90, 300], dtype=torch.int32, device=dev)   # decreasing
    cap, deg = bf1.route_capacity(3, 300, 300)
    route = bf1.Route.empty(cap, deg, dev)
    cu._bf1_total = 300
    bf1.plan_route(cu, 300, route=route)
    torch.cuda.synchronize()
    assert int(route.status.item()) & 1 and int(route.num_qblocks.item()) == 0
    # a sequence longer than max_seqlen
    cu = bf1.cu_seqlens_tensor([100, 200], dev)
    route = bf1.Route.empty(cap, deg, dev)
    bf1.plan_route(cu, 150, route=route)
    torch.cuda.synchronize()
    assert int(route.status.item()) & 1
    # too few slots
    cu = bf1.cu_seqlens_tensor([1000], dev)
    route = bf1.Route.empty(4, 6, dev)
    bf1.plan_route(cu, 1000, route=route)
    torch.cuda.synchronize()
    assert int(route.status.item()) & 2 and int(route.num_qblocks.item()) == 0
    # list pitch too small is caught on the host
    route = bf1.Route.empty(16, 3, dev)
    with pytest.raises(bf1.Bf1Error):
        bf1.plan_route(cu, 1000, route=route)
    # and a good plan afterwards clears the status word
    route = bf1.plan_route(cu, 1000)
    torch.cuda.synchronize()
    assert int(route.status.item()) == 0 and int(route.num_qblocks.item()) == 16


@pytest.mark.parametrize("seqlens,kw", [([1] * 9000, dict()),                                   # more slots than one sweep of the list CTAs
                                        ([64 * 1100, 65], dict(local_blocks=2000)),             # lists longer than a CTA has threads
                                        ([64 * 257 + 1, 64 * 127], dict(local_blocks=4))],      # window and dyadic predecessors overlap
                         ids=["many-slots", "long-lists", "overlap"])
def test_planner_at_the_edges_of_its_work_split(seqlens, kw):
    test_planner_matches_oracle_bit_exact(seqlens, kw)


@pytest.mark.parametrize("batch", [1, 7, 8, 9, 40])
def test_decode_planner_at_the_edges_of_its_work_split(batch):
    """A warp per sequence, eight to a CTA; one bad length anywhere flags the batch and empties that sequence only."""
    dev = torch.device("cuda:0")
    rng = np.random.default_rng(batch)
    lens = [int(x) for x in rng.integers(0, 64 * 70, size=batch)]
    lens[-1] = 64 * 70
    table = torch.from_numpy(rng.permutation(batch * 70).astype(np.int32).reshape(batch, 70)).to(dev)
    for bad in (False, True):
        if bad:
            lens[-1] += 1
        plan = bf1.plan_decode(torch.tensor(lens, dtype=torch.int32, device=dev), table)
        torch.cuda.synchronize()
        assert int(plan.status.item()) == (1 if bad else 0)
        for s, n in enumerate(lens):
            want = []
            if n > 0 and not (bad and s == batch - 1):
                idx, cnt, _, _ = O.route(O.cfg(), n, plan.max_degree)
                want = table[s].cpu().numpy()[idx[-1, :cnt[-1]]].tolist()
            assert plan.count[s].item() == len(want) and plan.page[s].tolist() == want + [-1] * (plan.max_degree - len(want))


@pytest.mark.parametrize("batch", [31, 32, 33])
def test_planner_where_the_scan_of_the_lengths_changes(batch):
    """Up to 32 sequences every warp scans the lengths, beyond that the CTA does; one bad length flags the batch in both."""
    lens = [int(x) for x in np.random.default_rng(batch).integers(0, 400, size=batch)]
    lens[0], lens[-1] = 0, 401
    test_planner_matches_oracle_bit_exact(lens, dict())
    cu = bf1.cu_seqlens_tensor(lens, torch.device("cuda:0"))
    cap, deg = bf1.route_capacity(batch, sum(lens), 401)
    for bad, slots, longest in ((1, cap, 400), (2, cap // 2, 401)):
        route = bf1.plan_route(cu, longest, route=bf1.Route.empty(slots, deg, cu.device))
        torch.cuda.synchronize()
        assert int(route.status.item()) == bad and int(route.num_qblocks.item()) == 0


@pytest.mark.parametrize("batch", [11200, 11800, 12270, 12300, 50000])
def test_planner_where_its_shared_memory_passes_what_needs_no_leave(batch):
    """One word for a sequence: 48 KB are passed, together with what the kernel declares itself, at about 12,200 of them."""
    test_planner_matches_oracle_bit_exact([1] * batch, dict())
