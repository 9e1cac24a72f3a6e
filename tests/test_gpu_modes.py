"""Element-by-element parity (GPU against the float64 oracle) of the attention kernel variants and
unpack paths that the five workloads do not reach, each case pinned to the variant it selects.

The attention kernel is compiled four times, attention_kernel<D, kIndep> for D in {64, 128} and
kIndep in {false, true}; the host scheduler picks kIndep from the packing (mean key tiles per query
tile) and, in the shared-stream mode (kIndep = false), pairs either two query heads of one KV head
(even GQA group) or two consecutive row tiles of one head (odd group). Each case below states the
variant and pairing it must select; the test recomputes that choice from the rule and also asks the
library (pp_prefill_schedule_info), so a case cannot silently drift to another variant.

case                         D    group  variant                    pairing       what it adds
[3000,1500,700]    2/2       64   1      <64,false>                 row tiles     D=64 shared-stream (4-stage rings, N=64 P.V)
[3000,1500,700]    4/1       64   4      <64,false>                 head pairs    the same with two heads per item
[2500,1300,129]    2/2       128  1      <128,false>                row tiles     slot 1 joins the key stream late (jb1 > 0)
[2432,640]         2/2       128  1      <128,false>                row tiles     odd tile counts: unpaired last row tile
[2500,1300,129]    3/1       64   3      <64,false>                 row tiles     odd group > 1, late join, D=64
[2432,640]         3/1       64   3      <64,false>                 row tiles     odd group > 1, unpaired tile, D=64
Padded mode declares every prompt as long as the longest, so these cases stay in the shared-stream
mode there as well (asserted)."""
import numpy as np
import pytest
import torch

import paper_2404_09529_b200 as pp
from parity_utils import compare_with_refs, expected_schedule, oracle_refs, run_cuda, table_ints
from paper_2404_09529_b200.runner import DecodeBatch, PrefillBatch
from workloads import split_by_prompt

pytestmark = pytest.mark.gpu


def _case(lengths, hq, hkv, d, seed):
    g = torch.Generator().manual_seed(seed)
    t = int(np.sum(lengths))
    mk = lambda h: torch.randn((t, h, d), generator=g).to(torch.bfloat16)
    return mk(hq), mk(hkv), mk(hkv)


def _assert_schedule(batch, hq, hkv, want_mode, want_pairing, unpaired=None, late=None):
    pk = batch.pack
    seg_bins = [[int(x) for x in pk.seg_len[pk.bin_seg_ptr[b]:pk.bin_seg_ptr[b + 1]]] for b in range(pk.n_bins)]
    assert expected_schedule(seg_bins, hq, hkv) == (want_mode, want_pairing)
    info = pp.pp_prefill_schedule_info(batch.params, pk)
    assert (info["mode"], info["pairing"]) == (want_mode, want_pairing), info
    if unpaired is not None:
        assert (info["unpaired_entries"] > 0) == unpaired, info
    if late is not None:
        assert (info["late_joining_entries"] > 0) == late, info


# lengths, Hq, Hkv, D, pairing (0 = head pairs, 1 = row tiles), unpaired last tile?, late-joining slot?
SHARED_CASES = [
    ([3000, 1500, 700], 2, 2, 64, 1, False, False),
    ([3000, 1500, 700], 4, 1, 64, 0, False, False),
    ([2500, 1300, 129], 2, 2, 128, 1, False, True),
    ([2432, 640], 2, 2, 128, 1, True, False),
    ([2500, 1300, 129], 3, 1, 64, 1, False, True),
    ([2432, 640], 3, 1, 64, 1, True, False),
]


@pytest.mark.parametrize("lengths,hq,hkv,d,pairing,unpaired,late", SHARED_CASES)
def test_shared_stream_variants_full_parity(lengths, hq, hkv, d, pairing, unpaired, late):
    lengths = np.asarray(lengths, np.int32)
    base = 500000.0
    q, k, v = _case(lengths, hq, hkv, d, seed=int(lengths.sum()) + d + hq)
    refs = oracle_refs(lengths, q, k, v, base)
    for mode in ("packed", "padded"):
        for fused in (False, True):
            b = run_cuda(lengths, q, k, v, hq, hkv, d, base, mode, fused=fused, guard=True)
            if mode == "packed":
                _assert_schedule(b, hq, hkv, 0, pairing, unpaired, late)
            else:
                _assert_schedule(b, hq, hkv, 0, pairing)
            compare_with_refs(b, lengths, refs)


# lengths, Hq, Hkv, D, query heads folded into a query tile (independent mode: the largest of 8, 4, 2
# that divides the GQA group; 1 = MHA or an odd group)
FOLD_CASES = [
    ([129, 1, 1, 127, 40, 3], 2, 1, 64, 2),
    ([300, 5, 129, 64, 1, 250, 33, 8, 8, 8, 90, 2], 8, 2, 128, 4),
    ([515, 130, 129, 128, 64, 33, 17, 9, 3, 2, 1], 8, 1, 64, 8),
    ([8] * 40 + [31, 33, 65], 16, 1, 128, 8),                  # group 16: two folds of 8 per KV head
    ([200, 77, 130, 31, 12], 6, 2, 64, 1),                     # group 3: no fold
    ([200, 77, 130, 31, 12], 12, 2, 128, 2),                   # group 6: folds of 2
]


@pytest.mark.parametrize("lengths,hq,hkv,d,fold", FOLD_CASES)
def test_head_folding_variants_full_parity(lengths, hq, hkv, d, fold):
    """Independent mode with GQA: the query tile is 128 / fold bin rows x fold heads. Every fold the
    scheduler can choose, both batch modes, both routes, guard regions around every output."""
    lengths = np.asarray(lengths, np.int32)
    base = 10000.0
    q, k, v = _case(lengths, hq, hkv, d, seed=hq * 100 + d)
    refs = oracle_refs(lengths, q, k, v, base)
    for mode in ("packed", "padded"):
        for fused in (False, True):
            b = run_cuda(lengths, q, k, v, hq, hkv, d, base, mode, fused=fused, guard=True)
            info = pp.pp_prefill_schedule_info(b.params, b.pack)
            assert info["mode"] == 1 and info["heads_folded"] == fold, info
            compare_with_refs(b, lengths, refs)


# KV heads that are drawn one after another and those drawn together at the end of the work list: all of them together (one
# head, several), two of four, two of three with three query heads each that are not folded, two of three in the shared-stream mode
@pytest.mark.parametrize("lengths,hq,hkv,d,mode,entries_per_head", [
    ([50, 20, 300], 1, 1, 64, 1, 4), ([50, 20, 300], 5, 5, 128, 1, 4), ([130] * 300, 4, 4, 64, 1, 600),
    ([130] * 100, 9, 3, 64, 1, 600), ([4000, 3000, 2600], 12, 3, 64, 0, 154)])
def test_every_head_is_drawn_once(lengths, hq, hkv, d, mode, entries_per_head):
    lengths = np.asarray(lengths, np.int32)
    q, k, v = _case(lengths, hq, hkv, d, seed=len(lengths) + hq)
    b = run_cuda(lengths, q, k, v, hq, hkv, d, 10000.0, "packed", fused=True, guard=True)
    info = pp.pp_prefill_schedule_info(b.params, b.pack)
    assert info["mode"] == mode
    heads_per_entry = info["heads_folded"] if mode == 1 else 2
    assert info["entries"] * (hq // hkv) // heads_per_entry == entries_per_head
    compare_with_refs(b, lengths, oracle_refs(lengths, q, k, v, 10000.0))


@pytest.mark.parametrize("room", [1, 7, 64])
@pytest.mark.parametrize("lengths,hq,hkv,d", [
    ([112, 87, 73, 46, 50, 20, 24, 17], 4, 4, 64),          # several prompts per bin, independent mode
    ([300, 5, 129, 64, 1, 250, 33, 8, 8, 8, 90, 2], 8, 2, 128),
])
def test_caches_with_spare_rows_and_guards(lengths, hq, hkv, d, room):
    """cache_cap = length + room: UNPACK writes rows [0, length) of every cache block and nothing
    else. The pools are pre-filled with a sentinel and every output buffer sits between sentinel
    guard regions; spare rows and guards must come back bit-unchanged from pp_unpack_kv, from
    pp_prefill_fused and from pp_unpack_kv_static, and the filled rows must match the oracle."""
    lengths = np.asarray(lengths, np.int32)
    base = 10000.0
    q, k, v = _case(lengths, hq, hkv, d, seed=room)
    refs = oracle_refs(lengths, q, k, v, base)
    rooms = room if room != 7 else (np.arange(len(lengths)) % 3 * 7 + 1).astype(np.int32)   # mixed spare rows
    for mode in ("packed", "padded"):
        three = run_cuda(lengths, q, k, v, hq, hkv, d, base, mode, fused=False, room=rooms, guard=True)
        compare_with_refs(three, lengths, refs)
        fused = run_cuda(lengths, q, k, v, hq, hkv, d, base, mode, fused=True, room=rooms, guard=True)
        compare_with_refs(fused, lengths, refs)
        assert torch.equal(three.k_cache, fused.k_cache) and torch.equal(three.v_cache, fused.v_cache)
        # the entry point without a workspace, on the same packed tensors, into fresh sentinel pools
        st = PrefillBatch(lengths, hq, hkv, d, base, mode=mode, room=rooms, guard=True)
        pp.pp_unpack_kv_static(three.params, three.bin_of, three.off_of, three.lengths, three.kk, three.v,
                               st.k_cache, st.v_cache, st.cache_off, st.cache_cap,
                               torch.cuda.current_stream().cuda_stream)
        torch.cuda.synchronize()
        st.assert_untouched()
        assert torch.equal(st.k_cache, three.k_cache) and torch.equal(st.v_cache, three.v_cache)


def test_prefill_with_room_then_decode_on_the_same_caches():
    """The hand-over of Section 7: UNPACK fills cache blocks that have room to grow, and the decode
    step appends to and reads those very blocks (no copy in between)."""
    from oracle import prepack_oracle as orc
    from parity_utils import MAX_ABS_TOL, MEAN_ABS_TOL, to64
    lengths = np.array([300, 17, 255, 256, 257, 64], np.int32)
    hq, hkv, d, base, n_steps = 8, 2, 128, 500000.0, 3
    q, k, v = _case(lengths, hq, hkv, d, seed=31)
    refs = oracle_refs(lengths, q, k, v, base)
    pre = run_cuda(lengths, q, k, v, hq, hkv, d, base, fused=True, room=n_steps + 2, guard=True)
    compare_with_refs(pre, lengths, refs)
    dec = DecodeBatch.from_prefill(pre)
    kc, vc = [r[1] for r in refs], [r[2] for r in refs]
    g = torch.Generator().manual_seed(77)
    for step in range(n_steps):
        qn, kn, vn = (torch.randn(len(lengths), h, d, generator=g).to(torch.bfloat16) for h in (hq, hkv, hkv))
        got = to64(dec.step(qn.cuda(), kn.cuda(), vn.cuda()))
        torch.cuda.synchronize()
        errs = []
        for i in range(len(lengths)):
            o_ref, kc[i], vc[i] = orc.decode_step(to64(qn[i]), to64(kn[i]), to64(vn[i]), kc[i], vc[i], base)
            errs.append(np.abs(got[i] - o_ref).ravel())
            l = int(lengths[i]) + step + 1
            ck, cv = dec.caches(i)
            assert np.max(np.abs(to64(ck[:, :l]) - kc[i])) <= MAX_ABS_TOL
            assert np.array_equal(to64(cv[:, :l]), vc[i])
            assert bool((ck[:, l:] == PrefillBatch.SENTINEL).all()) and bool((cv[:, l:] == PrefillBatch.SENTINEL).all())
        e = np.concatenate(errs)
        assert e.max() <= MAX_ABS_TOL and e.mean() <= MEAN_ABS_TOL, (step, e.max(), e.mean())


def test_unknown_flag_bits_are_rejected():
    lengths = np.array([40, 9], np.int32)
    b = PrefillBatch(lengths, 2, 2, 64, 10000.0)
    for bad in (0x100, 0x200, 0x8, 1 << 20):
        with pytest.raises(pp.PrepackError) as err:
            b.run(flags=bad)
        assert err.value.status == -1
        with pytest.raises(pp.PrepackError):
            b.run_fused(flags=bad)
    torch.cuda.synchronize()


def test_keep_rope_table_flag_gives_identical_results():
    lengths = np.array([700, 300, 250, 150, 90, 5, 5], np.int32)
    q, k, v = _case(lengths, 8, 2, 128, seed=3)
    b = PrefillBatch(lengths, 8, 2, 128, 500000.0)
    b.load(q, k, v)
    b.run_fused()
    torch.cuda.synchronize()
    ref = (b.o_tokens().clone(), b.k_cache.clone(), b.v_cache.clone())
    b.load(q, k, v)
    b.k_cache.zero_(); b.v_cache.zero_(); b.o.zero_()
    b.run_fused(flags=pp.PP_FLAG_KEEP_ROPE_TABLE)
    torch.cuda.synchronize()
    assert b.device_status() == 0
    for a, c in zip(ref, (b.o_tokens(), b.k_cache, b.v_cache)):
        assert torch.equal(a, c)


# whether the fused and the three-call table travel as kernel parameters: the sizes next to the line, without and with heads
# folded into the query tiles
@pytest.mark.parametrize("hq,hkv,d,k,fused_as_parameter,three_as_parameter", [
    (4, 4, 64, 1, True, True), (4, 4, 64, 37, True, True), (4, 4, 64, 38, False, True), (4, 4, 64, 45, False, True),
    (4, 4, 64, 46, False, False),
    (4, 2, 128, 1, True, True), (4, 2, 128, 22, True, True), (4, 2, 128, 23, False, True), (4, 2, 128, 24, False, True),
    (4, 2, 128, 25, False, False)])
def test_table_as_parameter_or_uploaded(hq, hkv, d, k, fused_as_parameter, three_as_parameter):
    """Both forms of the prefill table give the oracle's results, on the first and on a repeated call on the
    same workspace (the work counter starts anew), and whole or split by flags."""
    lengths = np.asarray([100 - 3 * (i % 7) for i in range(k)], np.int32)
    base = 10000.0
    q, kk, v = _case(lengths, hq, hkv, d, seed=k + d)
    refs = oracle_refs(lengths, q, kk, v, base)
    fused = PrefillBatch(lengths, hq, hkv, d, base, guard=True)
    three = PrefillBatch(lengths, hq, hkv, d, base, guard=True)
    three_ints, fused_ints, may = table_ints(fused.params, fused.pack)
    line = pp.binding.PARAMETER_TABLE_INTS
    assert (may and fused_ints <= line, may and three_ints <= line) == (fused_as_parameter, three_as_parameter)
    for _ in range(2):
        for b, call in ((fused, fused.run_fused), (three, three.run)):
            b.load(q, kk, v)
            call()
            torch.cuda.synchronize()
            assert b.device_status() == 0
            b.assert_untouched()
            compare_with_refs(b, lengths, refs)
    o = fused.o.clone()
    fused.load(q, kk, v)
    fused.o.zero_()
    fused.run_fused(flags=pp.PP_FLAG_ROPE_ONLY)
    fused.run_fused(flags=pp.PP_FLAG_SKIP_ROPE)
    torch.cuda.synchronize()
    assert fused.device_status() == 0 and torch.equal(fused.o_tokens(), o.view(-1, hq, d)[fused.token_rows])


# prompts: only the unpack table is uploaded (31, 45), the fused table too (70), all three (120, 333)
@pytest.mark.parametrize("k,uploaded", [(31, (False, False)), (45, (False, False)), (70, (False, True)), (120, (True, True)), (333, (True, True))])
@pytest.mark.parametrize("staging", ["pinned", "pinned + 16", "pinned + 8", "pageable"])
def test_tables_from_any_staging_memory(k, uploaded, staging):
    """Tables are read by a kernel from aligned pinned memory and copied from any other, several calls in a row
    through the ring of staging buffers."""
    lengths = np.asarray([60 - 7 * (i % 9) for i in range(k)], np.int32)
    q, kk, v = _case(lengths, 2, 1, 64, seed=k)
    refs = oracle_refs(lengths, q, kk, v, 10000.0)
    at = int(staging.split("+")[1]) if "+" in staging else 0
    fused = PrefillBatch(lengths, 2, 1, 64, 10000.0, guard=True)
    three = PrefillBatch(lengths, 2, 1, 64, 10000.0, guard=True)
    assert tuple(n > pp.binding.PARAMETER_TABLE_INTS for n in table_ints(three.params, three.pack)[:2]) == uploaded

    def buffer(like):
        t = torch.empty(like.numel() + at, dtype=torch.uint8)
        return (t if staging == "pageable" else t.pin_memory())[at:]

    for b, call in ((fused, fused.run_fused), (three, three.run)):
        b.ws._fused_host = [buffer(t) for t in b.ws._fused_host]
        b.ws._ring = [(buffer(a), buffer(u), fence) for a, u, fence in b.ws._ring]
        for _ in range(6):
            b.load(q, kk, v)
            call()
        torch.cuda.synchronize()
        assert b.device_status() == 0
        b.assert_untouched()
        compare_with_refs(b, lengths, refs)


# Multi-head, D = 128, independent mode: the attention kernel fills the V caches from 32 rows per prompt on, the rotation
# kernel below that. Prompts at the edges of the 64-key and the 128-row tiles, many in a tile, and streams of many items.
@pytest.mark.parametrize("lengths,room", [
    ([1], 0), ([32], 0), ([63, 1, 64, 65, 127], 3), ([128, 129, 1, 1, 1, 191, 193], 0), ([700, 3, 640, 257], 5),
    ([31] * 9, 0), ([32] * 9, 2), ([97 + i % 64 for i in range(70)], 0)])
@pytest.mark.parametrize("h", [1, 3])
def test_v_caches_filled_by_either_kernel(lengths, room, h):
    lengths = np.asarray(lengths, np.int32)
    base = 10000.0
    q, k, v = _case(lengths, h, h, 128, seed=int(lengths.sum()) + h)
    b = PrefillBatch(lengths, h, h, 128, base, room=room, guard=True)
    _assert_schedule(b, h, h, 1, 2)
    refs = oracle_refs(lengths, q, k, v, base)
    for _ in range(2):
        b.load(q, k, v)
        b.run_fused()
        torch.cuda.synchronize()
        assert b.device_status() == 0
        b.assert_untouched()
        compare_with_refs(b, lengths, refs)


def _scaled_inputs(kind, lengths, hq, hkv, d):
    q, k, v = _case(lengths, hq, hkv, d, seed=d + hq)
    t = q.shape[0]
    pos = torch.cat([torch.arange(int(l)) / int(l) for l in lengths]).view(-1, 1, 1)
    if kind == "unbounded":
        q, k = q * 4, k * 4
    elif kind == "rising":                       # later key tiles exceed the first one by far more than 2^90
        q, k = q * 6, k * (0.1 + 16 * pos)
    elif kind == "mixed":                        # rows within and beyond the bound side by side
        q = q * (0.5 + 8 * (torch.arange(t) % 3 == 0)).view(-1, 1, 1)
    elif kind == "nan":                          # one key is not a number: rows that do not see it stay right
        q, k = q * 4, k * 4
        k[int(lengths[0]) - 1] = float("nan")
    return q.to(torch.bfloat16), k.to(torch.bfloat16), v


@pytest.mark.parametrize("kind", ["bounded", "unbounded", "rising", "mixed", "nan"])
@pytest.mark.parametrize("lengths,hq,hkv,d", [([2432, 640], 2, 2, 128), ([3000, 1500, 700], 4, 1, 64)])
def test_rows_with_and_without_a_running_maximum(lengths, hq, hkv, d, kind):
    """Shared-stream mode: rows whose scores the norms bound drop the running maximum, others rescale. Reference: float64
    attention on the rotated q and k that the library returns (their own parity is tested above), so that the
    scores agree to fp32 and the rest is rounding: P to bf16 (2^-9 of each term, of which the sum of weights is 1),
    the sum of weights with or without it (as much again) and O to bf16, together below 2^-7 of the largest |v|."""
    lengths = np.asarray(lengths, np.int32)
    q, k, v = _scaled_inputs(kind, lengths, hq, hkv, d)
    fused = PrefillBatch(lengths, hq, hkv, d, 10000.0, guard=True)
    three = PrefillBatch(lengths, hq, hkv, d, 10000.0, guard=True)
    for b, call in ((fused, fused.run_fused), (three, three.run)):
        _assert_schedule(b, hq, hkv, 0, 0 if (hq // hkv) % 2 == 0 else 1)
        b.load(q, k, v)
        call()
        torch.cuda.synchronize()
        assert b.device_status() == 0
        b.assert_untouched()
    rows = three.token_rows.long()
    qr = three.q.reshape(-1, hq, d)[rows].double()
    kr = three.kk.reshape(-1, hkv, d)[rows].double().repeat_interleave(hq // hkv, 1)
    vr = v.cuda().double().repeat_interleave(hq // hkv, 1)
    tol = 2.0 ** -7 * float(v.abs().max())
    start = 0
    for i, l in enumerate(int(x) for x in lengths):
        part = slice(start, start + l)
        seen = l - 1 if kind == "nan" and i == 0 else l
        s = torch.einsum("qhd,khd->hqk", qr[part], kr[part]) / d ** 0.5
        s = s.masked_fill(torch.ones(l, l, dtype=torch.bool, device=s.device).triu(1), float("-inf"))
        ref = torch.einsum("hqk,khd->qhd", torch.softmax(s, -1), vr[part])
        for b in (fused, three):
            err = (b.o_tokens()[part].double() - ref).abs()[:seen].max().item()
            assert err <= tol, (i, err, tol)
        start += l


def _climbing_scores(climb, lengths, hq, hkv, d):
    """q and k along one slowly turning direction, so that a row's scores climb from -climb to climb (log2 units) with
    the key's place in its prompt; a little noise on top."""
    q, k, v = _case(lengths, hq, hkv, d, seed=d + hq)
    pos = torch.cat([torch.arange(int(l)) / int(l) for l in lengths]).view(-1, 1)
    amp = (climb * d ** 0.5 / 1.4426950408889634) ** 0.5
    q, k = q * 0.02, k * 0.02
    q[:, :, d // 2 - 1] += amp
    k[:, :, d // 2 - 1] += amp * (2 * pos - 1)
    return q.to(torch.bfloat16), k.to(torch.bfloat16), v


def _float64_attention(rotated, values, lengths, scale):
    """O of every prompt in float64 from the rotated q and k that the library handed back."""
    qr, kr = (x.double() for x in rotated)
    group = qr.shape[1] // kr.shape[1]
    kr, vr = kr.repeat_interleave(group, 1), values.cuda().double().repeat_interleave(group, 1)
    out, start = [], 0
    for l in (int(x) for x in lengths):
        part = slice(start, start + l)
        s = torch.einsum("qhd,khd->hqk", qr[part], kr[part]) * scale
        s = s.masked_fill(torch.ones(l, l, dtype=torch.bool, device=s.device).triu(1), float("-inf"))
        out.append(torch.einsum("hqk,khd->qhd", torch.softmax(s, -1), vr[part]))
        start += l
    return torch.cat(out)


@pytest.mark.parametrize("v_scale", [1.0, 2.0 ** 60, 2.0 ** 100])
@pytest.mark.parametrize("climb", [38, 300])           # within the bound on the scores, beyond it
@pytest.mark.parametrize("lengths,hq,hkv,d", [([2432, 640], 2, 2, 128), ([3000, 1500, 700], 4, 1, 64)])
def test_large_values_where_scores_climb(lengths, hq, hkv, d, climb, v_scale):
    """Shared-stream mode: however far a row's scores climb above those of its first key tile, O stays finite for values up
    to 2^100, and all routes give the same bits. Tolerance as in test_rows_with_and_without_a_running_maximum."""
    lengths = np.asarray(lengths, np.int32)
    q, k, v = _climbing_scores(climb, lengths, hq, hkv, d)
    v = (v * v_scale).to(torch.bfloat16)
    routes = {"three calls": lambda b: b.run(), "fused": lambda b: b.run_fused(),
              "three calls, split": lambda b: (b.run(flags=pp.PP_FLAG_ROPE_ONLY, unpack=False), b.run(flags=pp.PP_FLAG_SKIP_ROPE)),
              "fused, split": lambda b: (b.run_fused(flags=pp.PP_FLAG_ROPE_ONLY), b.run_fused(flags=pp.PP_FLAG_SKIP_ROPE))}
    first = None
    for name, call in routes.items():
        b = PrefillBatch(lengths, hq, hkv, d, 10000.0)
        _assert_schedule(b, hq, hkv, 0, 0 if (hq // hkv) % 2 == 0 else 1)
        b.load(q, k, v)
        call(b)
        torch.cuda.synchronize()
        assert b.device_status() == 0
        got = (b.o_tokens(), b.k_cache, b.v_cache)
        if first is None:
            first = got
            err = (got[0].double() - _float64_attention(b.rotated_tokens(), v, lengths, d ** -0.5)).abs().max().item()
            assert err <= 2.0 ** -7 * float(v.abs().max()), err
        for x, y in zip(first, got):
            assert torch.equal(x, y), name


@pytest.mark.parametrize("end", ["no bound", "infinite"])
@pytest.mark.parametrize("lengths,hq,hkv,d", [([2432, 640], 2, 2, 128), ([3000, 1500, 700], 4, 1, 64)])
def test_bound_on_the_scores_at_its_ends(lengths, hq, hkv, d, end):
    """Shared-stream mode, scores that climb by thousands, where the limit on |q|^2 is at an end of its range. "no bound":
    squares of the keys overflow and those of the queries come to 0; "infinite": the scale is so small that the
    limit itself overflows. Tolerance as in test_rows_with_and_without_a_running_maximum."""
    lengths = np.asarray(lengths, np.int32)
    scale, q_size, k_size = {"no bound": (0.0, 1e-23, 4e27), "infinite": (1e-20, 1e12, 3.5e11)}[end]
    q, k, v = _case(lengths, hq, hkv, d, seed=d + hq)
    pos = torch.cat([torch.arange(int(l)) / int(l) for l in lengths]).view(-1, 1)
    q, k = q.float() * 0.01, k.float() * 0.01
    q[:, :, d // 2 - 1] += 1
    k[:, :, d // 2 - 1] += 0.05 + pos
    q, k = (q * q_size).to(torch.bfloat16), (k * k_size).to(torch.bfloat16)
    three, fused = (PrefillBatch(lengths, hq, hkv, d, 10000.0, softmax_scale=scale) for _ in range(2))
    for b, call in ((three, three.run), (fused, fused.run_fused)):
        _assert_schedule(b, hq, hkv, 0, 0 if (hq // hkv) % 2 == 0 else 1)
        b.load(q, k, v)
        call()
        torch.cuda.synchronize()
        assert b.device_status() == 0
    ref = _float64_attention(three.rotated_tokens(), v, lengths, scale or d ** -0.5)
    for b in (three, fused):
        err = (b.o_tokens().double() - ref).abs().max().item()
        assert err <= 2.0 ** -7 * float(v.abs().max()), err
