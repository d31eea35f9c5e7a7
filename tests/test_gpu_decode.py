"""Cached one-token decode over selected pages (Section 3.2, Section 5.4) vs the CPU oracle.

The oracle for a decode step is the last row of the routed attention over the same (logical) keys
and values: the newest token reads P(block of n-1), the self block up to itself.  The gates are the
paper's: agreement with that reference, tail handling, page-permutation invariance, zero decoy-page
leakage, and one plan serving a whole 64-token route epoch."""
import numpy as np
import pytest
import torch

import bf1_inputs as I
import paper_2608_20427_b200 as bf1
from oracle import bf1_oracle as O

from gpu_util import LSE_ABS, O_MAX_ABS, O_REL_RMS

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def paged_cache(w, k, v, seed, decoys=7, decoy_scale=50.0):
    """Scatter the logical K/V of a packed batch into randomly permuted physical pages, with decoy
    pages (large finite garbage) in between.  Returns k_pages, v_pages, page_table (CPU tensors)."""
    g = torch.Generator().manual_seed(seed)
    blocks = [(n + 63) // 64 for n in w.seqlens]
    total = sum(blocks) + decoys
    perm = torch.randperm(total, generator=g)
    k_pages = (torch.randn((total, 64, w.hkv, w.d), generator=g) * decoy_scale).to(torch.bfloat16)
    v_pages = (torch.randn((total, 64, w.hkv, w.d), generator=g) * decoy_scale).to(torch.bfloat16)
    table = torch.full((len(blocks), max(max(blocks), 1)), -1, dtype=torch.int32)
    cu = w.cu_seqlens()
    nxt = 0
    for s, nb in enumerate(blocks):
        for b in range(nb):
            pg = int(perm[nxt]); nxt += 1
            table[s, b] = pg
            lo, hi = cu[s] + 64 * b, min(cu[s] + 64 * b + 64, cu[s + 1])
            k_pages[pg, :hi - lo] = k[lo:hi]
            v_pages[pg, :hi - lo] = v[lo:hi]
    return k_pages, v_pages, table


def run_decode(w, q, k_pages, v_pages, table, seqlens=None, plan=None):
    dev = torch.device(DEV)
    sl = torch.tensor(list(w.seqlens if seqlens is None else seqlens), dtype=torch.int32, device=dev)
    cu = w.cu_seqlens()
    last = [cu[s] + (n - 1) for s, n in enumerate(sl.tolist())]
    qd = torch.stack([q[i] if n > 0 else torch.zeros_like(q[0]) for i, n in zip(last, sl.tolist())]).to(dev)
    tb = table.to(dev)
    if plan is None:
        plan = bf1.plan_decode(sl, tb)
    ws = bf1.decode_workspace(len(w.seqlens), w.hq, w.hkv, plan.max_degree, w.d, dev)
    out = torch.full((len(w.seqlens), w.hq, w.d), float("nan"), dtype=torch.bfloat16, device=dev)
    lse = torch.full((w.hq, len(w.seqlens)), float("nan"), dtype=torch.float32, device=dev)
    for _ in range(2):   # twice: a call leaves nothing behind (the scratch is looked at below)
        bf1.decode_fwd(qd, k_pages.to(dev), v_pages.to(dev), sl, plan, ws, out=out, lse=lse)
    torch.cuda.synchronize()
    pairs = (w.hq // w.hkv + 1) // 2
    assert int(ws.view(torch.int32)[-len(w.seqlens) * w.hkv * pairs:].abs().sum().item()) == 0
    return out.float().cpu().numpy(), lse.cpu().numpy(), plan, last


def check(w, q, k, v, out, lse, last):
    rows = [r for r, n in zip(last, w.seqlens) if n > 0]
    o_ref, lse_ref = O.attn_route(O.cfg(), q, k, v, w.cu_seqlens(), rows=rows)
    live = [s for s, n in enumerate(w.seqlens) if n > 0]
    diff = out[live].astype(np.float64) - o_ref[rows]
    assert not np.isnan(out[live]).any() and not np.isnan(lse[:, live]).any()
    assert np.abs(diff).max() <= O_MAX_ABS
    assert np.sqrt((diff ** 2).mean() / (o_ref[rows].astype(np.float64) ** 2).mean()) <= O_REL_RMS
    assert np.abs(lse[:, live] - lse_ref[:, rows]).max() <= LSE_ABS


@pytest.mark.parametrize("d", [64, 128])
def test_decode_matches_oracle_with_tails_and_empty_sequences(d):
    lens = [1, 64, 65, 257, 1000, 0, 4097, 12345]
    w = I.custom(lens, hq=4, hkv=2, d=d, seed=3000 + d)
    q, k, v = I.draw_qkv(w)
    k_pages, v_pages, table = paged_cache(w, k, v, seed=1)
    out, lse, plan, last = run_decode(w, q, k_pages, v_pages, table)
    assert int(plan.status.item()) == 0
    check(w, q, k, v, out, lse, last)
    # the plan: physical pages of Eq. 1's list for the newest token's block, self page last
    cnt, pages = plan.count.cpu().numpy(), plan.page.cpu().numpy()
    for s, n in enumerate(lens):
        if n == 0:
            assert cnt[s] == 0 and np.isnan(out[s]).all()
            continue
        j = (n - 1) // 64
        idx, c, _, _ = O.route(O.cfg(), n, plan.max_degree)
        want = [int(table[s, b]) for b in idx[j, :c[j]]]
        assert cnt[s] == c[j] and list(pages[s, :cnt[s]]) == want and (pages[s, cnt[s]:] == -1).all()


def test_long_context_decode_32k_and_64k():
    w = I.custom([32768, 65536], hq=16, hkv=8, d=128, seed=3100)
    q, k, v = I.draw_qkv(w)
    k_pages, v_pages, table = paged_cache(w, k, v, seed=2)
    out, lse, plan, last = run_decode(w, q, k_pages, v_pages, table)
    assert plan.count.tolist() == [11, 12]      # 3 + floor(log2 511), 3 + floor(log2 1023)
    check(w, q, k, v, out, lse, last)


@pytest.mark.parametrize("d", [64, 128])
def test_large_batch_takes_the_one_cta_per_list_path(d):
    """batch x KV heads >= number of SMs: one CTA walks a whole page list with an online softmax."""
    rng = np.random.default_rng(7)
    lens = [int(x) for x in rng.integers(1, 3000, size=40)] + [1, 64, 65, 0, 4097]
    w = I.custom(lens, hq=8, hkv=4, d=d, seed=3500 + d)    # 45 x 4 = 180 pairs
    q, k, v = I.draw_qkv(w)
    k_pages, v_pages, table = paged_cache(w, k, v, seed=5)
    out, lse, plan, last = run_decode(w, q, k_pages, v_pages, table)
    assert int(plan.status.item()) == 0
    check(w, q, k, v, out, lse, last)
    # NaN behind the newest token and in unselected pages must not leak on this path either
    used = set(int(x) for x in table.flatten().tolist() if x >= 0)
    for pg in range(k_pages.shape[0]):
        if pg not in used:
            k_pages[pg] = float("nan")
            v_pages[pg] = float("nan")
    for s_, n_ in enumerate(w.seqlens):
        if n_ % 64:
            pg = int(table[s_, (n_ - 1) // 64])
            k_pages[pg, n_ % 64:] = float("nan")
            v_pages[pg, n_ % 64:] = float("nan")
    out1, lse1, _, _ = run_decode(w, q, k_pages, v_pages, table)
    live = [i for i, n_ in enumerate(lens) if n_ > 0]
    assert np.array_equal(out[live], out1[live]) and np.array_equal(lse[:, live], lse1[:, live])


def test_page_permutation_invariance_and_zero_decoy_leakage():
    w = I.custom([700, 3001], hq=4, hkv=2, d=128, seed=3200)
    q, k, v = I.draw_qkv(w)
    ref = None
    for seed, scale in ((10, 50.0), (11, 50.0), (10, 1000.0)):   # another permutation; other decoy contents
        k_pages, v_pages, table = paged_cache(w, k, v, seed=seed, decoy_scale=scale)
        out, lse, _, _ = run_decode(w, q, k_pages, v_pages, table)
        if ref is None:
            ref = (out, lse)
        assert np.array_equal(out, ref[0]) and np.array_equal(lse, ref[1])


def test_unwritten_page_tails_may_hold_anything():
    """The part of the newest page behind the newest token is unwritten cache memory: NaN there
    (and in pages the route does not select) must not reach the output."""
    w = I.custom([1000, 65], hq=4, hkv=2, d=128, seed=3400)
    q, k, v = I.draw_qkv(w)
    k_pages, v_pages, table = paged_cache(w, k, v, seed=4)
    out0, lse0, _, _ = run_decode(w, q, k_pages, v_pages, table)
    used = set(int(x) for x in table.flatten().tolist() if x >= 0)
    for pg in range(k_pages.shape[0]):
        if pg not in used:
            k_pages[pg] = float("nan")
            v_pages[pg] = float("nan")
    for s, n in enumerate(w.seqlens):
        tail = n % 64
        if tail:
            pg = int(table[s, (n - 1) // 64])
            k_pages[pg, tail:] = float("nan")
            v_pages[pg, tail:] = float("nan")
    out1, lse1, _, _ = run_decode(w, q, k_pages, v_pages, table)
    assert np.array_equal(out0, out1) and np.array_equal(lse0, lse1)


def test_one_plan_serves_a_route_epoch_and_refuses_the_next():
    n0 = 64 * 9 + 1                                       # first token of block 9
    w = I.custom([n0 + 63], hq=4, hkv=2, d=128, seed=3300)
    q, k, v = I.draw_qkv(w)
    k_pages, v_pages, table = paged_cache(w, k, v, seed=3)
    dev = torch.device(DEV)
    plan = bf1.plan_decode(torch.tensor([n0], dtype=torch.int32, device=dev), table.to(dev))
    for n in (n0, n0 + 1, n0 + 31, n0 + 63):              # same plan, growing tail
        wn = I.custom([n], hq=4, hkv=2, d=128, seed=0)
        out, lse, _, last = run_decode(wn, q[:n], k_pages, v_pages, table, plan=plan)
        assert int(plan.status.item()) == 0
        check(wn, q[:n], k[:n], v[:n], out, lse, last)
    # one token further the newest token lives in block 10: the stale plan is flagged, nothing is read
    dev_sl = torch.tensor([n0 + 64], dtype=torch.int32, device=dev)
    ws = bf1.decode_workspace(1, 4, 2, plan.max_degree, 128, dev)
    bf1.decode_fwd(q[:1].to(dev), k_pages.to(dev), v_pages.to(dev), dev_sl, plan, ws)
    torch.cuda.synchronize()
    assert int(plan.status.item()) & 8


def test_decode_plan_flags_a_sequence_longer_than_its_page_table():
    dev = torch.device(DEV)
    table = torch.zeros((1, 4), dtype=torch.int32, device=dev)
    plan = bf1.plan_decode(torch.tensor([4 * 64 + 1], dtype=torch.int32, device=dev), table)
    torch.cuda.synchronize()
    assert int(plan.status.item()) & 1 and int(plan.count.item()) == 0


@pytest.mark.parametrize("hq,hkv", [(8, 2), (3, 3)], ids=["G4", "G1"])
@pytest.mark.parametrize("batch_kind", ["few", "many"])
def test_decode_with_four_and_with_one_query_head_per_kv_head(hq, hkv, batch_kind):
    """G = 4 runs two CTAs (pairs of query heads) per KV head, G = 1 half a pair; both forms of the kernel
    are exercised: lists cut into runs with a combine (few sequences) and one CTA per list (many)."""
    lens = [1, 64, 65, 257, 1000, 0, 4097] if batch_kind == "few" else [1 + (37 * i) % 700 for i in range(90)]
    w = I.custom(lens, hq=hq, hkv=hkv, d=128, seed=7100 + hq + len(lens))
    q, k, v = I.draw_qkv(w)
    k_pages, v_pages, table = paged_cache(w, k, v, seed=7200 + hq)
    out, lse, plan, last = run_decode(w, q, k_pages, v_pages, table)
    assert int(plan.status.item()) == 0
    check(w, q, k, v, out, lse, last)


@pytest.mark.parametrize("hq,hkv,d", [(16, 8, 128), (8, 2, 64), (3, 3, 128)], ids=["G2-d128", "G4-d64", "G1-d128"])
@pytest.mark.parametrize("batch", [1, 5, 19, 40])
@pytest.mark.parametrize("local_blocks", [2, 40], ids=["short-lists", "long-lists"])
def test_decode_however_a_list_is_cut_into_runs(hq, hkv, d, batch, local_blocks):
    """Few lists: clusters of up to eight CTAs, with runs of one page up to more pages than a CTA's ring holds, and CTAs
    without a run (short sequences beside long ones, an empty sequence); many lists: a CTA for a list."""
    rng = np.random.default_rng(batch + d)
    lens = [int(x) for x in rng.integers(1, 64 * 60, size=batch)]
    lens[0] = 64 * 59 + 1
    if batch > 1:
        lens[1:5] = [0, 1, 64, 65]
    w = I.custom(lens, hq=hq, hkv=hkv, d=d, seed=3900 + batch + d, local_blocks=local_blocks)
    q, k, v = I.draw_qkv(w)
    k_pages, v_pages, table = paged_cache(w, k, v, seed=9)
    dev = torch.device(DEV)
    plan = bf1.plan_decode(torch.tensor(lens, dtype=torch.int32, device=dev), table.to(dev), bf1.RouteCfg(64, local_blocks, 1, 1))
    out, lse, plan, last = run_decode(w, q, k_pages, v_pages, table, plan=plan)
    assert int(plan.status.item()) == 0
    rows = [r for r, n in zip(last, lens) if n > 0]
    live = [s for s, n in enumerate(lens) if n > 0]
    o_ref, lse_ref = O.attn_route(O.cfg(local_blocks=local_blocks), q, k, v, w.cu_seqlens(), rows=rows)
    assert np.abs(out[live] - o_ref[rows]).max() <= O_MAX_ABS
    assert np.abs(lse[:, live] - lse_ref[:, rows]).max() <= LSE_ABS
    assert np.isnan(out[[s for s in range(batch) if lens[s] == 0]]).all()


@pytest.mark.parametrize("hq,hkv,d", [(16, 8, 128), (2, 1, 64), (4, 1, 128)], ids=["G2-d128", "G2-d64", "G4-d128"])
def test_few_lists_are_rounded_page_by_page(hq, hkv, d):
    """Nothing but the result is rounded where a list is cut (P is multiplied with V unrounded), and nothing but it where a part is
    a page and P is rounded against the maximum of its 16 keys.  Here one key of every 16 has a score of O(1) and the others at
    most -300, whose weight is 0 in fp32.
    The fp32 sums behind a score (d products, sum of magnitudes about 25) are off by d * 2^-23 * 25 at most, a weight
    relatively by that times the scale, 3.4e-5: a result comes to lie on the other side of a rounding boundary in about 2 *
    3.4e-5 / 2^-8 = 2 % of the elements at worst.  Rounded weights in parts of two pages round every other weight by up to 2^-9."""
    lens = [64 * 500 + 17, 64 * 130]
    w = I.custom(lens, hq=hq, hkv=hkv, d=d, seed=4100 + d)
    q, k, v = I.draw_qkv(w)
    k = (k.float() * 0.3).to(torch.bfloat16)
    k[..., 0] = -448.0
    q[..., 0] = 8.0
    cu = w.cu_seqlens()
    for s, n in enumerate(lens):
        g = torch.arange(n // 16)
        k[cu[s] + 16 * g + (7 * g) % 16, :, 0] = 0.0
    k_pages, v_pages, table = paged_cache(w, k, v, seed=12)
    out, lse, plan, last = run_decode(w, q, k_pages, v_pages, table)
    assert int(plan.status.item()) == 0 and plan.count.tolist() == [11, 10]
    for s, n in enumerate(lens):
        j = (n - 1) // 64
        idx, c, _, _ = O.route(O.cfg(), n, plan.max_degree)
        rows = torch.cat([torch.arange(64 * b, min(64 * b + 64, n)) for b in idx[j, :c[j]]]) + cu[s]
        kk, vv = (t[rows].double().repeat_interleave(hq // hkv, 1) for t in (k, v))
        p = torch.softmax(torch.einsum("hd,nhd->hn", q[last[s]].double(), kk) * d ** -0.5, 1)
        want = torch.einsum("hn,nhd->hd", p, vv).to(torch.bfloat16).float().numpy()
        assert (out[s] != want).mean() <= 0.03, (out[s] != want).mean()


def test_a_plan_that_changes_between_the_ctas_of_a_list_stays_in_bounds():
    """Sequences without a plan, and of another route epoch, among others: all CTAs of their clusters go through the whole
    kernel, nothing of theirs is written, and the others' rows are those of a batch without them."""
    lens = [64 * 70, 130, 64 * 300 + 9, 5000]
    w = I.custom(lens, hq=4, hkv=2, d=128, seed=4200)
    q, k, v = I.draw_qkv(w)
    k_pages, v_pages, table = paged_cache(w, k, v, seed=13)
    dev = torch.device(DEV)
    ref, ref_lse, _, _ = run_decode(w, q, k_pages, v_pages, table)
    plan = bf1.plan_decode(torch.tensor(lens, dtype=torch.int32, device=dev), table.to(dev))
    plan.count[1] = -3
    plan.block[2] += 1
    plan.count[3] = 1 << 20                       # (kept to the row pitch)
    plan.page[3, int((plan.page[3] >= 0).sum()):] = plan.page[3, 0]
    out, lse, plan, _ = run_decode(w, q, k_pages, v_pages, table, plan=plan)
    assert int(plan.status.item()) == 8
    assert np.isnan(out[[1, 2]]).all() and np.isnan(lse[:, [1, 2]]).all()
    assert np.array_equal(out[0], ref[0]) and np.array_equal(lse[:, 0], ref_lse[:, 0])
    assert np.isfinite(out[3]).all()


def distances_from_64_bits(w, q, k, v, out, last):
    """Relative distance from 64 bits, over the sequences of more than ten blocks (in a short one the first keys' V fills the norm, and the
    rounding of P does not show), of `out` and of a result whose weights are rounded to bf16 where that costs least: every weight
    against the maximum of its own 16 keys."""
    off = planted = norm = 0.0
    cu, bf16 = w.cu_seqlens(), lambda x: x.to(torch.bfloat16).double()
    for s, n in enumerate(w.seqlens):
        if n <= 64 * 10:
            continue
        j = (n - 1) // 64
        idx, c, _, _ = O.route(O.cfg(), n)
        blocks = [torch.arange(64 * b, min(64 * b + 64, n)) + cu[s] for b in idx[j, :c[j]]]
        rows = torch.cat(blocks)
        kk, vv = (t[rows].double().repeat_interleave(w.hq // w.hkv, 1) for t in (k, v))
        score = torch.einsum("hd,nhd->hn", q[last[s]].double(), kk) * w.d ** -0.5
        p = torch.exp(score - score.max(1, keepdim=True).values)
        piece = torch.cat([(torch.arange(len(b)) // 16) + 4 * i for i, b in enumerate(blocks)]).expand_as(p)
        top = torch.zeros(w.hq, 4 * len(blocks), dtype=torch.float64).scatter_reduce(1, piece, p, "amax").gather(1, piece)
        want, rounded = (torch.einsum("hn,nhd->hd", x, vv) / p.sum(1, keepdim=True) for x in (p, bf16(p / top) * top))
        off += float(((torch.from_numpy(out[s]).double() - want) ** 2).sum())
        planted += float(((bf16(rounded) - want) ** 2).sum())
        norm += float((want ** 2).sum())
    return (off / norm) ** 0.5, (planted / norm) ** 0.5


# The rounding of a result to bf16 is 1.64e-3 to 1.69e-3 of its norm in the cases below, computed in 64 bits, and with rounded
# weights, page by page, 1.9e-3 and more.
UNROUNDED = 1.78e-3


@pytest.mark.parametrize("hq,hkv,d,batch", [(16, 4, 128, 18), (16, 4, 128, 19), (8, 2, 64, 70), (8, 8, 64, 3), (4, 2, 128, 37)],
                         ids=["G4-parts", "G4-whole", "G4-d64", "G1", "G2"])
def test_parts_of_a_list_lose_nothing_but_the_rounding_of_the_result(hq, hkv, d, batch):
    """Where a list is cut (all of these but "G4-whole") P is multiplied with V unrounded."""
    rng = np.random.default_rng(batch)
    lens = [int(x) for x in rng.integers(64 * 20, 64 * 130, size=batch)]
    lens[:3] = [64 * 129 + 5, 1, 65]
    w = I.custom(lens, hq=hq, hkv=hkv, d=d, seed=4300 + batch)
    q, k, v = I.draw_qkv(w)
    k_pages, v_pages, table = paged_cache(w, k, v, seed=14)
    out, lse, plan, last = run_decode(w, q, k_pages, v_pages, table)
    assert int(plan.status.item()) == 0
    check(w, q, k, v, out, lse, last)
    off, planted = distances_from_64_bits(w, q, k, v, out, last)
    assert planted > UNROUNDED
    if (hq, hkv, d, batch) != (16, 4, 128, 19):
        assert off <= UNROUNDED, off


@pytest.mark.parametrize("hq,hkv,d,blocks", [(1, 1, 128, 520), (4, 2, 64, 520), (4, 2, 128, 520), (8, 2, 64, 520), (8, 2, 64, 32), (8, 2, 128, 520)],
                         ids=["G1", "G2-d64", "G2", "G4-d64", "G4-d64-brief", "G4"])
def test_what_is_not_finite_in_v_comes_out_the_same_however_the_lists_are_walked(hq, hkv, d, blocks):
    """One sequence alone, whose list is cut (into parts of a page, and longer ones), and batches of it that fill the GPU, whose
    lists are walked whole.  Every column but the last 8 has an infinity at one selected key, with a weight that is not zero:
    the result is that infinity.  Of the others some have both infinities or a NaN at a key: NaN."""
    n = 64 * blocks
    w = I.custom([n], hq=hq, hkv=hkv, d=d, seed=4400 + d + hq)
    q, k, v = I.draw_qkv(w)
    idx, c, _, _ = O.route(O.cfg(), n, 16)
    listed = [int(b) for b in idx[n // 64 - 1, :c[n // 64 - 1]]]
    want = torch.zeros(d)
    for col in range(d - 8):
        key = 64 * listed[col % len(listed)] + (col * 29) % 64
        want[col] = float("inf") if col % 2 else float("-inf")
        v[key, :, col] = want[col]
    for col in (d - 8, d - 7):
        v[64 * listed[0] + col % 64, :, col] = float("inf")
        v[64 * listed[-1], :, col] = float("-inf")
        v[64 * listed[-1] + 1, :, col + 2] = float("nan")
        want[col] = want[col + 2] = float("nan")
    k_pages, v_pages, table = (t.to(DEV) for t in paged_cache(w, k, v, seed=15))
    last = None
    for batch in (1, 30 // hkv, 60 // hkv, 100 // hkv, 160 // hkv):
        sl = torch.full((batch,), n, dtype=torch.int32, device=DEV)
        plan = bf1.plan_decode(sl, table.repeat(batch, 1))
        ws = bf1.decode_workspace(batch, hq, hkv, plan.max_degree, d, torch.device(DEV))
        out, _ = bf1.decode_fwd(q[-1].to(DEV).repeat(batch, 1, 1), k_pages, v_pages, sl, plan, ws)
        out = out.float().cpu()
        assert torch.equal(out.isnan(), want.isnan().expand_as(out)), batch
        assert torch.equal(torch.where(out.isinf(), out, 0.0), torch.where(want.isinf(), want, 0.0).expand_as(out)), batch
        if last is not None:
            assert (out - last)[..., d - 4:].abs().max() <= O_MAX_ABS
        last = out[:1]


@pytest.mark.parametrize("hq,hkv,d", [(4, 2, 64), (4, 2, 128), (8, 2, 128)], ids=["G2-d64", "G2", "G4"])
def test_an_infinity_under_a_weight_of_zero_is_nan_however_the_lists_are_walked(hq, hkv, d):
    """The keys of one listed page have scores some 300 below the others', a weight of 0 in fp32, and an infinity in the first
    column: 0 times infinity.  Where the page is a part by itself the part is fine and its weight among the parts is 0."""
    n = 64 * 520
    w = I.custom([n], hq=hq, hkv=hkv, d=d, seed=4500 + d + hq)
    q, k, v = I.draw_qkv(w)
    idx, c, _, _ = O.route(O.cfg(), n, 16)
    low = int(idx[n // 64 - 1, 4])
    q[..., 0] = 8.0
    k[..., 0] = 0.0
    k[64 * low:64 * low + 64, :, 0] = -448.0
    v[64 * low + 5, :, 0] = float("inf")
    k_pages, v_pages, table = (t.to(DEV) for t in paged_cache(w, k, v, seed=16))
    for batch in (1, 30 // hkv, 60 // hkv, 160 // hkv):
        sl = torch.full((batch,), n, dtype=torch.int32, device=DEV)
        plan = bf1.plan_decode(sl, table.repeat(batch, 1))
        ws = bf1.decode_workspace(batch, hq, hkv, plan.max_degree, d, torch.device(DEV))
        out, _ = bf1.decode_fwd(q[-1].to(DEV).repeat(batch, 1, 1), k_pages, v_pages, sl, plan, ws)
        assert bool(out[..., 0].isnan().all()) and bool(out[..., 1:].isfinite().all()), batch


@pytest.mark.parametrize("d,blocks,batch", [(64, 32, 86), (64, 32, 87), (64, 32, 147), (64, 32, 148), (64, 3, 3), (64, 4, 3), (128, 3, 3),
                                            (128, 4, 3), (128, 3, 73), (128, 3, 74), (128, 1, 5)])
def test_brief_lists_of_four_heads_are_walked_whole_and_unrounded(d, blocks, batch):
    """One KV head, 148 SMs.  Seven pages (32 blocks): cut up to 86 lists, whole and unrounded from 87, whole and rounded from 148.  Up to
    three pages: whole and unrounded however many lists there are, with d = 128 rounded from 74.  Four pages: cut."""
    rng = np.random.default_rng(blocks + batch)
    lens = [int(x) for x in rng.integers(64 * 12 if blocks == 32 else 1, 64 * blocks, size=batch)]
    lens[:3] = [64 * blocks, 1, 64 * (blocks // 2) + 1]
    w = I.custom(lens, hq=4, hkv=1, d=d, seed=4600 + batch)
    q, k, v = I.draw_qkv(w)
    k_pages, v_pages, table = paged_cache(w, k, v, seed=17)
    out, lse, plan, last = run_decode(w, q, k_pages, v_pages, table)
    assert int(plan.status.item()) == 0 and plan.max_degree == {32: 7, 4: 4, 3: 3, 1: 1}[blocks]
    check(w, q, k, v, out, lse, last)
    if blocks == 32:
        off, planted = distances_from_64_bits(w, q, k, v, out, last)
        assert planted > UNROUNDED and (batch == 148 or off <= UNROUNDED), (off, planted)
