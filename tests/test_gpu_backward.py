"""Gradients of the routed attention on the GPU vs the fp64 CPU oracle (Section 4.2's gradient gate).  The
kernels round P and dS to bf16 before their MMAs and their outputs to bf16, so the comparison is by relative RMS
and by the largest error relative to the gradient's scale.  Nothing is added with atomics: the three gradients
must come out bit-identical on every run."""
import numpy as np
import pytest
import torch

import bf1_inputs as I
import paper_2608_20427_b200 as bf1
from oracle import bf1_oracle as O

from gpu_util import oracle_cfg, lib_cfg

pytestmark = pytest.mark.gpu
REL_RMS = 1e-2          # P, dS and the outputs are bf16 (2^-9 relative each); observed 2e-3 .. 5e-3
REL_MAX = 2e-2          # of the gradient's largest magnitude; observed <= 6e-3
ZERO_ABS = 1e-4         # where the exact gradient is zero: fp32 rounding of O(10) dot products, times P <= 1


def run_case(w, seed):
    dev = torch.device("cuda:0")
    q, k, v = I.draw_qkv(w)
    g = torch.Generator().manual_seed(seed)
    d_o = torch.randn(q.shape, generator=g).to(torch.bfloat16)
    cu = bf1.cu_seqlens_tensor(w.seqlens, dev)
    route = bf1.plan_route(cu, w.max_seqlen, lib_cfg(w))
    qd, kd, vd, gd = q.to(dev), k.to(dev), v.to(dev), d_o.to(dev)
    o, lse = bf1.attn_fwd(qd, kd, vd, cu, w.max_seqlen, route)
    dq, dk, dv = bf1.attn_bwd(qd, kd, vd, o, lse, gd, cu, w.max_seqlen, route)
    torch.cuda.synchronize()
    route.check_status()
    rq, rk, rv = O.attn_route_bwd(oracle_cfg(w), q, k, v, d_o.float().numpy().astype(np.float64), w.cu_seqlens())
    out = {}
    for name, got, ref in (("dq", dq, rq), ("dk", dk, rk), ("dv", dv, rv)):
        got = got.float().cpu().numpy().astype(np.float64)
        assert np.isfinite(got).all(), name
        diff = got - ref
        scale = float(np.abs(ref).max())
        if scale < 1e-9:
            # a gradient that is zero by definition (a token whose only key is itself has dq = dk = 0):
            # the kernel's D = <dO, O> and dP = <dO, V> differ by fp32 rounding only, so what is left
            # must be tiny in absolute terms -- no relative floor to hide behind
            assert float(np.abs(got).max()) <= ZERO_ABS, (name, float(np.abs(got).max()))
            out[name] = (0.0, 0.0)
            continue
        rms_ref = float(np.sqrt((ref ** 2).mean()))
        out[name] = (float(np.sqrt((diff ** 2).mean())) / rms_ref, float(np.abs(diff).max()) / scale)
    return out


@pytest.mark.parametrize("lens", [[64], [1], [65], [257], [1000], [130, 0, 257, 64, 1, 700]],
                         ids=lambda x: "-".join(map(str, x)))
def test_gradients_match_the_oracle(lens):
    w = I.custom(lens, hq=4, hkv=2, d=128, seed=6000 + sum(lens))
    res = run_case(w, seed=1)
    print(lens, res)
    for name, (rms, mx) in res.items():
        assert rms <= REL_RMS and mx <= REL_MAX, (name, rms, mx)


def test_gradients_4k_qwen_geometry():
    w = I.custom([4096], hq=16, hkv=8, d=128, seed=6100, sink_scale=4.0)
    res = run_case(w, seed=2)
    print("4k", res)
    for name, (rms, mx) in res.items():
        assert rms <= REL_RMS and mx <= REL_MAX, (name, rms, mx)


@pytest.mark.parametrize("n", [8192, 32768])
def test_gradients_at_the_benchmarked_lengths(n):
    """The sizes bench.py's `backward` block times: several waves of units, lists of 9 to 11 entries,
    up to eleven query blocks adding into one KV block.  All of dQ, dK, dV against the fp64 oracle."""
    w = I.custom([n], hq=16, hkv=8, d=128, seed=6200 + n)
    res = run_case(w, seed=3)
    print(n, res)
    for name, (rms, mx) in res.items():
        assert rms <= REL_RMS and mx <= REL_MAX, (name, rms, mx)


@pytest.mark.parametrize("hq,hkv,d", [(4, 2, 64), (8, 2, 128), (8, 2, 64), (3, 3, 128), (2, 2, 64)],
                         ids=["G2-d64", "G4-d128", "G4-d64", "G1-d128", "G1-d64"])
def test_gradients_in_every_geometry_the_forward_takes(hq, hkv, d):
    """Section 4.2's gradient gate per geometry: head dimension 64, four query heads per KV head (two CTAs per unit
    whose dK / dV contributions add up), one query head per KV head (half of the tile idle)."""
    for lens in ([1, 65, 257, 1000], [2500]):
        w = I.custom(lens, hq=hq, hkv=hkv, d=d, seed=6300 + hq + d + len(lens))
        res = run_case(w, seed=4)
        print(hq, hkv, d, lens, res)
        for name, (rms, mx) in res.items():
            assert rms <= REL_RMS and mx <= REL_MAX, (name, rms, mx)


@pytest.mark.parametrize("route", [dict(local_blocks=9, global_first=0, dyadic=0),      # sliding window: ten readers per block
                                   dict(local_blocks=40, global_first=1, dyadic=1),     # 41+ readers per block: cut into runs
                                   dict(local_blocks=0, global_first=0, dyadic=1)],     # dyadic predecessors only
                         ids=["sliding", "wide", "dyadic-only"])
def test_gradients_over_other_routes(route):
    """dK / dV walk the INVERSE of whatever lists the route holds; these routes give it other shapes than BF1's."""
    w = I.custom([4096, 700], hq=4, hkv=2, d=128, seed=6400, **route)
    res = run_case(w, seed=5)
    print(route, res)
    for name, (rms, mx) in res.items():
        assert rms <= REL_RMS and mx <= REL_MAX, (name, rms, mx)


def test_gradients_of_many_short_sequences():
    """Hundreds of sequences of one to three blocks: more units than the persistent kernels have CTAs, nearly all of
    one or two list entries, so every ring, buffer pair and barrier phase changes hands at every step; units of
    sequences with a single token have nothing but the self block."""
    rng = np.random.default_rng(77)
    lens = [int(x) for x in rng.integers(1, 190, size=700)]
    lens[5] = 0
    lens[100:108] = [1, 64, 65, 128, 129, 1, 63, 2]
    w = I.custom(lens, hq=4, hkv=2, d=64, seed=6600)
    res = run_case(w, seed=7)
    print(len(lens), sum(lens), res)
    for name, (rms, mx) in res.items():
        assert rms <= REL_RMS and mx <= REL_MAX, (name, rms, mx)


def test_gradients_over_a_dense_route():
    """Every predecessor selected (lists of up to 32 entries, every block with many readers): long units in the dQ
    kernel, every KV block of the first half cut into runs in the dK/dV kernel."""
    w = I.custom([2048], hq=4, hkv=2, d=128, seed=6700, local_blocks=64, global_first=1, dyadic=1)
    res = run_case(w, seed=8)
    print(res)
    for name, (rms, mx) in res.items():
        assert rms <= REL_RMS and mx <= REL_MAX, (name, rms, mx)


def test_backward_over_a_damaged_route_is_the_backward_of_the_repaired_route():
    """Entries outside [0, j], a list that does not end in its query block, counts past the pitch: every kernel of the
    library reads a list the same repaired way (the forward flags it), so the gradients over the damaged route are,
    bit for bit, those over the route with the repairs written in -- and nothing faults."""
    dev = torch.device("cuda:0")
    w = I.custom([1500, 300], hq=4, hkv=2, d=128, seed=6800)
    q, k, v = (t.to(dev) for t in I.draw_qkv(w))
    d_o = torch.randn(q.shape, generator=torch.Generator().manual_seed(9)).to(torch.bfloat16).to(dev)
    cu = bf1.cu_seqlens_tensor(w.seqlens, dev)

    def grads(damage):
        route = bf1.plan_route(cu, w.max_seqlen)
        deg = route.max_degree
        cnt = route.kv_count.cpu()
        blk = route.qb_block.cpu()
        idx = route.kv_idx.cpu().clone()
        kc = cnt.clone()
        g1, g2, g3 = 7, 12, 20            # slots of the first sequence (24 blocks)
        if damage:
            idx[g1, 0] = 1000             # out of range            -> read as block 0
            idx[g2, 1] = -5               # negative                -> read as block 0
            idx[g3, int(cnt[g3]) - 1] = 3 # last entry not the self block -> read as the self block
            kc[g2] = deg + 50             # count past the pitch    -> cut to the pitch
        else:
            idx[g1, 0] = 0
            idx[g2, 1] = 0
            idx[g3, int(cnt[g3]) - 1] = int(blk[g3])
            # kc[g2] cut to the pitch: the entries past the old count are the -1 padding, read as block 0, and the
            # last one as the self block
            kc[g2] = deg
            idx[g2, int(cnt[g2]) - 1] = 0
            idx[g2, int(cnt[g2]):deg - 1] = 0
            idx[g2, deg - 1] = int(blk[g2])
        route.kv_idx.copy_(idx.to(dev))
        route.kv_count.copy_(kc.to(dev))
        o, lse = bf1.attn_fwd(q, k, v, cu, w.max_seqlen, route)
        out = bf1.attn_bwd(q, k, v, o, lse, d_o, cu, w.max_seqlen, route)
        torch.cuda.synchronize()
        return out, int(route.status.item())

    bad, status_bad = grads(True)
    good, status_good = grads(False)
    assert status_bad & 8 and not status_good & 8
    for x, y in zip(bad, good):
        assert torch.isfinite(x.float()).all()
        assert torch.equal(x, y)


def test_backward_is_bitwise_reproducible():
    """No floating-point atomics: two runs give the same bits, whatever the workspace held before (block 0 of the
    long sequence has 64 readers and goes through the partial-sum path)."""
    dev = torch.device("cuda:0")
    w = I.custom([4096, 1000, 65], hq=8, hkv=2, d=128, seed=6500)
    q, k, v = (t.to(dev) for t in I.draw_qkv(w))
    d_o = torch.randn(q.shape, generator=torch.Generator().manual_seed(6)).to(torch.bfloat16).to(dev)
    cu = bf1.cu_seqlens_tensor(w.seqlens, dev)
    route = bf1.plan_route(cu, w.max_seqlen)
    o, lse = bf1.attn_fwd(q, k, v, cu, w.max_seqlen, route)
    ws = bf1.bwd_workspace(route, w.total_tokens, w.hq, w.hkv, w.d, dev)
    runs = []
    for fill in (0x00, 0xFF, 0x7F):          # 0xFF bytes are NaNs as fp32, 0x7F.. huge ints as counters
        ws.fill_(fill)
        runs.append(bf1.attn_bwd(q, k, v, o, lse, d_o, cu, w.max_seqlen, route, workspace=ws))
        torch.cuda.synchronize()
        route.check_status()
    for other in runs[1:]:
        for x, y in zip(runs[0], other):
            assert torch.equal(x, y)
    assert all(torch.isfinite(t.float()).all() for t in runs[0])


def test_backward_rejects_what_it_does_not_support():
    dev = torch.device("cuda:0")
    w = I.custom([128], hq=2, hkv=1, d=64, seed=1)
    q, k, v = (t.to(dev) for t in I.draw_qkv(w))
    cu = bf1.cu_seqlens_tensor(w.seqlens, dev)
    route = bf1.plan_route(cu, 128)
    o, lse = bf1.attn_fwd(q, k, v, cu, 128, route)
    lib = bf1.load()
    rc = lib.bf1_attn_bwd(q.data_ptr(), k.data_ptr(), v.data_ptr(), o.data_ptr(), lse.data_ptr(), q.data_ptr(),
                          cu.data_ptr(), 1, 128, 128, 6, 1, 64, 0.0, route.c, q.data_ptr(), q.data_ptr(), q.data_ptr(),
                          q.data_ptr(), None)
    assert rc == -2 and b"group" in lib.bf1_last_error()      # G = 6
    rc = lib.bf1_attn_bwd(q.data_ptr(), k.data_ptr(), v.data_ptr(), o.data_ptr(), lse.data_ptr(), q.data_ptr(),
                          cu.data_ptr(), 1, 128, 128, 2, 1, 96, 0.0, route.c, q.data_ptr(), q.data_ptr(), q.data_ptr(),
                          q.data_ptr(), None)
    assert rc == -2 and b"dimension" in lib.bf1_last_error()  # d = 96


@pytest.mark.parametrize("hq,hkv,d", [(4, 2, 128), (8, 2, 64), (2, 2, 128)], ids=["G2-d128", "G4-d64", "G1-d128"])
@pytest.mark.parametrize("tiles_bytes", [300 << 20, 700 << 20, 9 << 30], ids=["several-launches", "head-by-head", "recompute"])
def test_backward_does_not_depend_on_the_row_pitch_of_the_lists(hq, hkv, d, tiles_bytes):
    """The pitch of the lists sizes the workspace, and its size chooses how dS is kept (all heads, head by head, not at
    all) and how the inverse route is made (one CTA or several launches).  A pitch far wider than the lists takes a
    small problem through each choice; the gradients are those of the ordinary pitch.  Recomputed dS has the same bits
    (same MMAs, same D), only its sum runs through other instructions: fp32 sums of at most 448 products of O(1) in
    another order differ by 448 * 2^-24 relative to the sum of magnitudes, far below a bf16 step (2^-8), so an element
    moves by one step at most."""
    dev = torch.device("cuda:0")
    w = I.custom([897, 130], hq=hq, hkv=hkv, d=d, seed=6900 + d + hq)
    q, k, v = (t.to(dev) for t in I.draw_qkv(w))
    d_o = torch.randn(q.shape, generator=torch.Generator().manual_seed(10)).to(torch.bfloat16).to(dev)
    cu = bf1.cu_seqlens_tensor(w.seqlens, dev)

    def grads(pitch):
        cap, deg = bf1.route_capacity(len(w.seqlens), w.total_tokens, w.max_seqlen)
        route = bf1.plan_route(cu, w.max_seqlen, route=bf1.Route.empty(cap, pitch or deg, dev))
        o, lse = bf1.attn_fwd(q, k, v, cu, w.max_seqlen, route)
        out = bf1.attn_bwd(q, k, v, o, lse, d_o, cu, w.max_seqlen, route)
        torch.cuda.synchronize()
        route.check_status()
        return out

    cap, _ = bf1.route_capacity(len(w.seqlens), w.total_tokens, w.max_seqlen)
    pairs = 2 if hq == 4 * hkv else 1
    base, wide = grads(None), grads(tiles_bytes // (cap * pairs * 16384))
    for name, x, y in zip(("dq", "dk", "dv"), base, wide):
        if tiles_bytes > 8 << 30 and name == "dq":
            diff = (x.float() - y.float()).abs()
            assert bool((diff <= 2.0 ** -7 * x.float().abs() + 1e-6).all()), float(diff.max())
        else:
            assert torch.equal(x, y), name


@pytest.mark.parametrize("lens,spare,route", [([1] * 1100 + [700], 0, dict()),                    # more slots than threads
                                              ([8192], 0, dict(local_blocks=9)),                 # runs of more than 16 readers, and a rest
                                              ([64 * 16], 0, dict(local_blocks=16)),             # 16 readers: one full run, no rest
                                              ([1000, 65], 1500, dict())],                       # nothing behind the last slot is read as a slot
                         ids=["slots", "runs", "full-run", "spare-capacity"])
def test_gradients_at_the_edges_of_the_inverse_route(lens, spare, route):
    dev = torch.device("cuda:0")
    w = I.custom(lens, hq=2, hkv=1, d=64, seed=7000 + len(lens), **route)
    q, k, v = I.draw_qkv(w)
    d_o = torch.randn(q.shape, generator=torch.Generator().manual_seed(11)).to(torch.bfloat16)
    cu = bf1.cu_seqlens_tensor(w.seqlens, dev)
    cap, deg = bf1.route_capacity(len(w.seqlens), w.total_tokens, w.max_seqlen, lib_cfg(w))
    r = bf1.Route.empty(cap + spare, deg, dev, lib_cfg(w))
    for t in (r.qb_seq, r.qb_block, r.kv_count, r.kv_idx, r.order):
        t.fill_(0x7f7f7f7f)
    bf1.plan_route(cu, w.max_seqlen, lib_cfg(w), route=r)
    qd, kd, vd, gd = q.to(dev), k.to(dev), v.to(dev), d_o.to(dev)
    o, lse = bf1.attn_fwd(qd, kd, vd, cu, w.max_seqlen, r)
    grads = bf1.attn_bwd(qd, kd, vd, o, lse, gd, cu, w.max_seqlen, r)
    torch.cuda.synchronize()
    r.check_status()
    ref = O.attn_route_bwd(oracle_cfg(w), q, k, v, d_o.float().numpy().astype(np.float64), w.cu_seqlens())
    for name, got, want in zip(("dq", "dk", "dv"), grads, ref):
        diff = got.float().cpu().numpy().astype(np.float64) - want
        assert np.isfinite(diff).all(), name
        rms = float(np.sqrt((diff ** 2).mean() / (want ** 2).mean()))
        assert rms <= REL_RMS and float(np.abs(diff).max()) <= REL_MAX * float(np.abs(want).max()), (name, rms)


def _hand_written(route, slots, pitch, dev):
    """The planned route with its slots in another order (or some of them only), uploaded as a caller's."""
    t = {n: getattr(route, n).cpu()[slots] for n in ("qb_seq", "qb_block", "kv_count", "kv_idx", "pair_count")}
    if pitch:
        t["kv_idx"] = torch.nn.functional.pad(t["kv_idx"], (0, pitch - t["kv_idx"].shape[1]), value=-1)
    return bf1.Route.from_host(order=torch.arange(len(slots)), total_pairs=0, device=dev, **t)


def _raw_backward(q, k, v, d_o, cu, max_len, route):
    """Forward, then the C entry point with gradients that hold NaN beforehand; they, and the status words after each."""
    o, lse = bf1.attn_fwd(q, k, v, cu, max_len, route, out=torch.zeros_like(q), lse=torch.zeros((q.shape[1], q.shape[0]), device=q.device))
    after_forward = int(route.status.item())
    ws = bf1.bwd_workspace(route, q.shape[0], q.shape[1], k.shape[1], q.shape[2], q.device)
    grads = [torch.full_like(t, float("nan")) for t in (q, k, v)]
    rc = bf1.load().bf1_attn_bwd(q.data_ptr(), k.data_ptr(), v.data_ptr(), o.data_ptr(), lse.data_ptr(), d_o.data_ptr(), cu.data_ptr(),
                                 cu.numel() - 1, q.shape[0], max_len, q.shape[1], k.shape[1], q.shape[2], 0.0, route.c, ws.data_ptr(),
                                 *(t.data_ptr() for t in grads), torch.cuda.current_stream().cuda_stream)
    assert rc == 0
    torch.cuda.synchronize()
    return grads, after_forward, int(route.status.item())


@pytest.mark.parametrize("pitch", [0, 500, 19000], ids=["one-cta", "several-launches", "recompute"])
def test_routes_whose_blocks_are_not_found_where_the_planner_puts_them(pitch):
    """The backward looks for block p of an entry as many slots in front of its query slot as p lies in front of the query
    block.  Routes for which another slot, or none, is there run forward; their backward flags them and writes nothing."""
    dev = torch.device("cuda:0")
    w = I.custom([64 * 9 + 5, 64 * 6], hq=4, hkv=2, d=64, seed=7300)
    q, k, v = (t.to(dev) for t in I.draw_qkv(w))
    d_o = torch.randn(q.shape, generator=torch.Generator().manual_seed(12)).to(torch.bfloat16).to(dev)
    cu = bf1.cu_seqlens_tensor(w.seqlens, dev)
    planned = bf1.plan_route(cu, w.max_seqlen)
    want, _, st = _raw_backward(q, k, v, d_o, cu, w.max_seqlen, planned)
    assert st == 0
    first, second = list(range(10)), list(range(10, 16))
    # the sequences in the other order: every sequence's slots still follow each other
    got, st_fwd, st = _raw_backward(q, k, v, d_o, cu, w.max_seqlen, _hand_written(planned, second + first, pitch, dev))
    assert st_fwd == 0 and st == 0
    for x, y in zip(got, want):
        assert pitch > 1000 or torch.equal(x, y)      # (recomputed dS: see the test of the row pitch)
        assert bool((x.float() - y.float()).abs().max() <= 2.0 ** -7 * y.float().abs().max())
    for name, slots in (("reversed", first[::-1] + second), ("two swapped", [0, 2, 1] + first[3:] + second), ("no first block", first[1:] + second),
                        ("a block missing", first[:4] + first[5:] + second), ("interleaved", [x for p in zip(first, second) for x in p])):
        got, st_fwd, st = _raw_backward(q, k, v, d_o, cu, w.max_seqlen, _hand_written(planned, slots, pitch, dev))
        assert st_fwd == 0 and st == 8, (name, st_fwd, st)
        assert all(bool(t.isnan().all()) for t in got), name


def test_a_shard_route_has_no_backward_and_a_window_in_mid_sequence_has():
    dev = torch.device("cuda:0")
    n = 64 * 20
    w = I.custom([n], hq=2, hkv=1, d=128, seed=7400)
    q, k, v = (t.to(dev) for t in I.draw_qkv(w))
    d_o = torch.randn(q.shape, generator=torch.Generator().manual_seed(13)).to(torch.bfloat16).to(dev)
    # blocks 12 .. 19 as a shard
    needed = bf1.shard_needed_blocks(n, 12, 20)
    route, cu = bf1.plan_route_shard(n, 12, 20, torch.tensor(needed, dtype=torch.int32, device=dev))
    rows = torch.cat([torch.arange(64 * b, 64 * b + 64) for b in needed + list(range(12, 20))]).to(dev)
    got, st_fwd, st = _raw_backward(q[rows], k[rows], v[rows], d_o[rows], cu, rows.numel(), route)
    assert st_fwd == 0 and st == 8 and all(bool(t.isnan().all()) for t in got)
    # blocks 12 .. 19 with a window of two, those lists cut off at block 12: every block that is named has its slot
    cfg = bf1.RouteCfg(64, 2, 0, 0)
    cu = bf1.cu_seqlens_tensor([n], dev)
    planned = bf1.plan_route(cu, n, cfg)
    idx = planned.kv_idx.cpu()[12:].clone()
    count = planned.kv_count.cpu()[12:].clone()
    idx[0], count[0] = torch.tensor([12, -1, -1]), 1
    idx[1], count[1] = torch.tensor([12, 13, -1]), 2
    part = bf1.Route.from_host(torch.zeros(8), torch.arange(12, 20), count, idx, torch.zeros(8), torch.arange(8), 0, dev, cfg)
    got, st_fwd, st = _raw_backward(q, k, v, d_o, cu, n, part)
    alone = bf1.cu_seqlens_tensor([64 * 8], dev)
    want, _, _ = _raw_backward(q[64 * 12:], k[64 * 12:], v[64 * 12:], d_o[64 * 12:], alone, 64 * 8, bf1.plan_route(alone, 64 * 8, cfg))
    assert st_fwd == 0 and st == 0
    for x, y in zip(got, want):
        assert torch.equal(x[64 * 12:], y) and bool(x[:64 * 12].isnan().all())


@pytest.mark.parametrize("lens,kw", [([64 * 257], dict()), ([64 * 700 - 9], dict(local_blocks=0, dyadic=0)),
                                     ([64 * 300, 64 * 280, 70], dict(local_blocks=1, dyadic=0)), ([64 * 256, 64 * 40], dict())],
                         ids=["257", "700", "two-of-them", "256"])
def test_blocks_with_many_readers_are_the_same_however_the_inverse_route_is_made(lens, kw):
    """Block 0 of a sequence is read by all of its blocks.  In one CTA more than 256 readers are put in order by going
    through all entries; a pitch too wide for one CTA sorts them in a launch of its own.  The sums run in that order."""
    dev = torch.device("cuda:0")
    w = I.custom(lens, hq=2, hkv=1, d=64, seed=7500 + len(lens), **kw)
    q, k, v = (t.to(dev) for t in I.draw_qkv(w))
    d_o = torch.randn(q.shape, generator=torch.Generator().manual_seed(14)).to(torch.bfloat16).to(dev)
    cu = bf1.cu_seqlens_tensor(w.seqlens, dev)
    cap, deg = bf1.route_capacity(len(lens), w.total_tokens, w.max_seqlen, lib_cfg(w))
    assert 2 * cap + 1 + 2 * cap * deg <= 24576 < 2 * cap + 1 + 2 * cap * 60
    grads = []
    for pitch in (deg, 60):
        route = bf1.plan_route(cu, w.max_seqlen, lib_cfg(w), route=bf1.Route.empty(cap, pitch, dev, lib_cfg(w)))
        o, lse = bf1.attn_fwd(q, k, v, cu, w.max_seqlen, route)
        grads.append(bf1.attn_bwd(q, k, v, o, lse, d_o, cu, w.max_seqlen, route))
        torch.cuda.synchronize()
        route.check_status()
    assert all(torch.equal(x, y) for x, y in zip(*grads))
    assert all(bool(x.isfinite().all()) for x in grads[0])


def runs_of_readers(w):
    """(units, readers, run length, partial sums, blocks cut) that a backward leaves in its workspace: the last words of its
    integers, which lie behind one float per row and head."""
    dev = torch.device("cuda:0")
    q, k, v = (t.to(dev) for t in I.draw_qkv(w))
    cu = bf1.cu_seqlens_tensor(w.seqlens, dev)
    route = bf1.plan_route(cu, w.max_seqlen, lib_cfg(w))
    o, lse = bf1.attn_fwd(q, k, v, cu, w.max_seqlen, route)
    ws = bf1.bwd_workspace(route, w.total_tokens, w.hq, w.hkv, w.d, dev)
    bf1.attn_bwd(q, k, v, o, lse, torch.ones_like(q), cu, w.max_seqlen, route, workspace=ws)
    cap, deg = route.capacity_qblocks, route.max_degree
    parts = max(cap, min(cap * deg, 2 * 148 // w.hkv + 1))
    ints = 3 * (cap + 1) + 3 * cap + cap * deg + 8 * (cap + parts) + 8 * cap + w.hkv + 8
    at = (w.total_tokens * w.hq * 4 + 255) // 256 * 256 + 4 * (ints - 8)
    return ws[at:at + 20].view(torch.int32).tolist()


@pytest.mark.parametrize("lens,hq,hkv,d,kw,chunk", [
    ([64 * 2 + 1], 1, 1, 64, dict(), 2),
    ([64 * 31 + 7], 2, 1, 128, dict(local_blocks=0, dyadic=0), 2),        # 16 runs of block 0, the last block short
    ([1000], 8, 4, 128, dict(), 4),
    ([700, 33, 64 * 9], 16, 4, 64, dict(), 4),                            # two pairs of heads, short and empty tails
    ([64 * 33], 16, 8, 64, dict(), 12),
    ([64 * 64], 8, 8, 64, dict(), 16)],                                   # the longest; block 0 in four
    ids=["2", "2-window", "4", "G4", "12", "16"])
def test_few_units_are_cut_into_short_runs(lens, hq, hkv, d, kw, chunk):
    w = I.custom(lens, hq=hq, hkv=hkv, d=d, seed=7700 + sum(lens), **kw)
    readers = []
    for n in lens:
        idx, count, _, _ = O.route(oracle_cfg(w), n)
        readers += list(np.bincount(np.concatenate([row[:c] for row, c in zip(idx, count)]), minlength=len(count)))
    cut = [-(-int(r) // chunk) for r in readers]
    assert chunk == min(sum(readers) * hkv // 148 + 2, 16)
    assert runs_of_readers(w) == [sum(cut), sum(readers), chunk, sum(c for c in cut if c > 1), sum(c > 1 for c in cut)]
    for name, (rms, mx) in run_case(w, seed=15).items():
        assert rms <= REL_RMS and mx <= REL_MAX, (name, rms, mx)
