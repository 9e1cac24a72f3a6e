"""Generation step over the per-prompt caches (pp_decode_step) against the float64 oracle."""
import numpy as np
import pytest
import torch

from oracle import prepack_oracle as orc
from parity_utils import MAX_ABS_TOL, MEAN_ABS_TOL, decode_bytes, to64
from workloads import split_by_prompt

pytestmark = pytest.mark.gpu


def _case(lengths, hq, hkv, d, seed):
    g = torch.Generator().manual_seed(seed)
    t = int(np.sum(lengths))
    mk = lambda h: torch.randn(t, h, d, generator=g).to(torch.bfloat16)
    return mk(hq), mk(hkv), mk(hkv)


@pytest.mark.parametrize("lengths,hq,hkv,d,base", [
    (np.array([1, 1, 1, 1000, 1, 1, 1, 1, 1, 1], np.int32), 8, 8, 128, 10000.0),   # the paper's toy mix
    (np.array([300, 17, 255, 256, 257, 64], np.int32), 8, 2, 128, 500000.0),
    (np.array([40, 9, 513], np.int32), 4, 4, 64, 10000.0),
    # many prompts at the edges of chunks of 256 keys (the batches above run chunks of 64)
    (np.array([255, 256, 257, 511, 512, 513, 767, 768, 300, 64, 1000, 129] * 4, np.int32), 16, 16, 64, 10000.0),
])
def test_decode_steps_match_oracle(lengths, hq, hkv, d, base):
    from paper_2404_09529_b200.runner import DecodeBatch, PrefillBatch
    n_steps = 3
    q, k, v = _case(lengths, hq, hkv, d, seed=21)
    pre = PrefillBatch(lengths, hq, hkv, d, base)
    pre.load(q, k, v)
    pre.run_fused()
    torch.cuda.synchronize()
    assert pre.device_status() == 0
    dec = DecodeBatch(lengths, hq, hkv, d, base, room=n_steps + 1)
    dec.adopt(pre)
    # oracle state: caches of every prompt alone
    qs, ks, vs = (split_by_prompt(x, lengths) for x in (q, k, v))
    ref = [orc.prefill_prompt(to64(a), to64(b), to64(c), base) for a, b, c in zip(qs, ks, vs)]
    kc = [r[1] for r in ref]
    vc = [r[2] for r in ref]
    g = torch.Generator().manual_seed(99)
    for step in range(n_steps):
        qn = torch.randn(len(lengths), hq, d, generator=g).to(torch.bfloat16)
        kn = torch.randn(len(lengths), hkv, d, generator=g).to(torch.bfloat16)
        vn = torch.randn(len(lengths), hkv, d, generator=g).to(torch.bfloat16)
        o = dec.step(qn.cuda(), kn.cuda(), vn.cuda())
        torch.cuda.synchronize()
        got = to64(o)
        errs = []
        for i in range(len(lengths)):
            o_ref, kc[i], vc[i] = orc.decode_step(to64(qn[i]), to64(kn[i]), to64(vn[i]), kc[i], vc[i], base)
            errs.append(np.abs(got[i] - o_ref))
            l = int(lengths[i]) + step + 1
            ck, cv = dec.caches(i)
            assert np.max(np.abs(to64(ck[:, :l]) - kc[i])) <= MAX_ABS_TOL       # rotated keys, bf16-rounded
            assert np.array_equal(to64(cv[:, :l]), vc[i])                       # values are copied bit for bit
        e = np.concatenate([x.ravel() for x in errs])
        assert e.max() <= MAX_ABS_TOL and e.mean() <= MEAN_ABS_TOL, (step, e.max(), e.mean())


def test_decode_argument_checks():
    import paper_2404_09529_b200 as pp
    params = pp.AttnParams(4, 4, 64, 10000.0, 0.0, 1, 1, 0)
    lengths = np.array([5, 3], np.int32)
    nb = pp.pp_decode_workspace_bytes(params, lengths)
    assert nb > 0
    ws = torch.empty(nb, dtype=torch.uint8, device="cuda")
    host = torch.empty(nb, dtype=torch.uint8).pin_memory()
    x = torch.zeros(2, 4, 64, dtype=torch.bfloat16, device="cuda")
    cache = torch.zeros(2 * 4 * 8 * 64, dtype=torch.bfloat16, device="cuda")
    off = np.array([0, 4 * 8 * 64], np.int64)
    with pytest.raises(pp.PrepackError):       # no room for the new token of prompt 0
        pp.pp_decode_step(params, lengths, x, x, x, x.clone(), cache, cache.clone(), off, np.array([5, 8], np.int32),
                          ws, host, nb)
    with pytest.raises(pp.PrepackError):       # workspace too small
        pp.pp_decode_step(params, lengths, x, x, x, x.clone(), cache, cache.clone(), off, np.array([8, 8], np.int32),
                          ws, host, 16)


@pytest.mark.parametrize("lengths,hq,hkv,d,chunk_keys", [
    # every remainder of a 16-key step and of a 64-key chunk, in one chunk and in several; group 8
    (np.array([1, 2, 15, 16, 17, 31, 32, 33, 47, 48, 49, 63, 64, 65, 127, 128, 129, 191, 192, 193], np.int32), 16, 2, 128, 64),
    (np.array([1, 15, 16, 17, 63, 64, 65, 129, 255, 257], np.int32), 6, 2, 64, 64),      # group 3: absent head columns
    (np.array([4096, 3], np.int32), 2, 1, 128, 64),                                      # 64 chunks, the most of a prompt
    (np.array([4097, 3], np.int32), 2, 1, 128, 128),                                     # one key more: larger chunks
    (np.arange(600, dtype=np.int32) % 37 + 1, 2, 2, 64, 64),                             # table uploaded, not in the parameters
    (np.array([70] * 40 + [200], np.int32), 4, 1, 128, 64),                              # the larger parameter block
    (np.array([3000] * 3 + [512, 513], np.int32), 128, 32, 64, 192),                     # between the smallest and the largest
    (np.array([9000] * 3 + [1536, 512, 513], np.int32), 64, 32, 64, 512),                # the largest
    (np.array([18943] * 3 + [1], np.int32), 32, 32, 64, 512),                            # the last before the line
    (np.array([18944] * 3 + [1], np.int32), 32, 32, 64, 1024),                           # and past it
])
def test_decode_chunks_and_tables(lengths, hq, hkv, d, chunk_keys):
    """The generation step on caches of random contents at the edges of its steps, chunks and table forms,
    spare rows untouched. The chunks are those that the step takes: it runs in the workspace that they need and in no less."""
    import paper_2404_09529_b200 as pp
    from paper_2404_09529_b200.runner import DecodeBatch
    dec = DecodeBatch(lengths, hq, hkv, d, 10000.0, room=2)
    need = decode_bytes(dec.params, lengths, chunk_keys)
    assert pp.pp_decode_workspace_bytes(dec.params, lengths) == decode_bytes(dec.params, lengths, min(chunk_keys, 512))
    g = torch.Generator().manual_seed(int(lengths.sum()))
    for pool in (dec.k_cache, dec.v_cache):
        pool.copy_(torch.randn(pool.shape, generator=g).to(torch.bfloat16))
    before = [tuple(c.clone() for c in dec.caches(i)) for i in range(dec.k)]
    qn, kn, vn = (torch.randn(dec.k, h, d, generator=g).to(torch.bfloat16) for h in (hq, hkv, hkv))
    ws, host = torch.empty(need, dtype=torch.uint8, device="cuda"), torch.empty(need, dtype=torch.uint8).pin_memory()
    step = lambda nbytes: pp.pp_decode_step(dec.params, lengths, qn.cuda(), kn.cuda(), vn.cuda(), dec.o, dec.k_cache, dec.v_cache,
                                            dec.cache_off, dec.cache_cap, ws, host, nbytes)
    with pytest.raises(pp.PrepackError):
        step(need - 1)
    step(need)
    got = to64(dec.o)
    errs = []
    for i in range(dec.k):
        l = int(lengths[i])
        kc, vc = (to64(c[:, :l]) for c in before[i])
        o_ref, k_ref, v_ref = orc.decode_step(to64(qn[i]), to64(kn[i]), to64(vn[i]), kc, vc, 10000.0)
        errs.append(np.abs(got[i] - o_ref).ravel())
        ck, cv = dec.caches(i)
        assert np.max(np.abs(to64(ck[:, l]) - k_ref[:, l])) <= MAX_ABS_TOL
        assert torch.equal(cv[:, l].cpu(), vn[i])
        for now, was in zip((ck, cv), before[i]):
            assert torch.equal(now[:, :l], was[:, :l]) and torch.equal(now[:, l + 1:], was[:, l + 1:])
    e = np.concatenate(errs)
    assert e.max() <= MAX_ABS_TOL and e.mean() <= MEAN_ABS_TOL, (e.max(), e.mean())


@pytest.mark.parametrize("sized,used,keys", [
    ([18955] * 3, [18900] * 3, 512),         # sized where a step takes chunks of 1024, used where it takes 512
    ([18900] * 3, [18955] * 3, 1024),        # the other way round
])
def test_decode_workspace_on_the_other_side_of_the_line(sized, used, keys):
    """A workspace that was sized on one side of the line between chunks of 512 and of 1024 keys holds a step on the other side;
    the step gives what it gives in a workspace of its own."""
    import paper_2404_09529_b200 as pp
    from paper_2404_09529_b200.runner import DecodeBatch
    sized, used = np.array(sized, np.int32), np.array(used, np.int32)
    h, d = 32, 64
    dec = DecodeBatch(used, h, h, d, 10000.0, room=2)
    nbytes = pp.pp_decode_workspace_bytes(dec.params, sized)
    assert decode_bytes(dec.params, used, keys) <= nbytes
    g = torch.Generator(device="cuda").manual_seed(7)
    for pool in (dec.k_cache, dec.v_cache):
        pool.copy_(torch.randn(pool.shape, generator=g, device="cuda"))
    new = [torch.randn(dec.k, h, d, generator=g, device="cuda").to(torch.bfloat16) for _ in range(3)]
    ws, host = torch.empty(nbytes, dtype=torch.uint8, device="cuda"), torch.empty(nbytes, dtype=torch.uint8).pin_memory()
    o = torch.zeros_like(dec.o)
    pp.pp_decode_step(dec.params, used, *new, o, dec.k_cache, dec.v_cache, dec.cache_off, dec.cache_cap, ws, host, nbytes)
    assert torch.equal(o, dec.step(*new))


@pytest.mark.parametrize("hq,hkv,d", [(2, 2, 128), (8, 1, 128), (6, 2, 64)])
def test_decode_with_infinite_values(hq, hkv, d):
    """An infinity among the cached values, or in the new token's, makes that element of O infinite (with both signs, or a
    NaN, not a number) and no other: the first, a middle and the last key of a step, in one chunk and in several."""
    from paper_2404_09529_b200.runner import DecodeBatch
    lengths = np.array([1, 16, 17, 50, 64, 65, 200, 700], np.int32)
    dec = DecodeBatch(lengths, hq, hkv, d, 10000.0, room=2)
    g = torch.Generator().manual_seed(hq + d)
    for pool in (dec.k_cache, dec.v_cache):
        pool.copy_(torch.randn(pool.shape, generator=g).to(torch.bfloat16))
    qn, kn, vn = (torch.randn(dec.k, h, d, generator=g).to(torch.bfloat16) for h in (hq, hkv, hkv))
    inf = float("inf")
    for i, l in enumerate(int(x) for x in lengths):
        cv = dec.caches(i)[1]
        cv[0, 0, 1] = inf
        cv[hkv - 1, l - 1, d - 1] = -inf
        cv[0, l // 2, d // 2 + 3] = inf
        cv[0, l - 1, 8] = float("nan")
        vn[i, 0, 5] = -inf if i % 2 else inf
        cv[0, l // 3, 6] = inf
        vn[i, 0, 6] = -inf
        cv[0, l:] = inf                        # spare rows are not read
        dec.caches(i)[0][0, l:] = float("nan")
    before = [tuple(to64(c[:, :int(l)]) for c in dec.caches(i)) for i, l in enumerate(lengths)]
    got = to64(dec.step(qn.cuda(), kn.cuda(), vn.cuda()))
    for i in range(dec.k):
        with np.errstate(invalid="ignore"):
            ref = orc.decode_step(to64(qn[i]), to64(kn[i]), to64(vn[i]), *before[i], 10000.0)[0]
        assert np.isinf(ref).any() and np.isnan(ref).any()
        finite = np.isfinite(ref)
        assert np.array_equal(np.isnan(got[i]), np.isnan(ref)), i
        assert np.array_equal(got[i][np.isinf(ref)], ref[np.isinf(ref)]), i
        assert np.isfinite(got[i][finite]).all() and np.abs(got[i] - ref)[finite].max() <= MAX_ABS_TOL, i


@pytest.mark.parametrize("lengths", [[40], [64, 65, 200], [700]])
def test_decode_with_scores_of_minus_infinity(lengths):
    """Keys with an infinite element whose score is -inf weigh nothing, whether they are some of a 16-key step, all of it or
    a whole chunk."""
    from paper_2404_09529_b200.runner import DecodeBatch
    lengths = np.asarray(lengths, np.int32)
    h, d, base = 2, 128, 10000.0
    dec = DecodeBatch(lengths, h, h, d, base, room=2)
    g = torch.Generator().manual_seed(5)
    for pool in (dec.k_cache, dec.v_cache):
        pool.copy_(torch.randn(pool.shape, generator=g).to(torch.bfloat16))
    qn, kn, vn = (torch.randn(dec.k, h, d, generator=g).to(torch.bfloat16) for _ in range(3))
    for i, l in enumerate(int(x) for x in lengths):
        q_rot = orc.rope_rotate(to64(qn[i])[None], np.array([l]), base)[0]
        for key in list(range(18)) + [l // 2] + list(range(64, min(l, 128))) + list(range(320, min(l, 640))):
            for head in range(h):
                dec.caches(i)[0][head, key, 7] = -float("inf") * float(np.sign(q_rot[head, 7]))
    before = [tuple(to64(c[:, :int(l)]) for c in dec.caches(i)) for i, l in enumerate(lengths)]
    got = to64(dec.step(qn.cuda(), kn.cuda(), vn.cuda()))
    for i in range(dec.k):
        ref = orc.decode_step(to64(qn[i]), to64(kn[i]), to64(vn[i]), *before[i], base)[0]
        assert np.isfinite(ref).all() and np.isfinite(got[i]).all(), i
        assert np.abs(got[i] - ref).max() <= MAX_ABS_TOL, i


@pytest.mark.parametrize("hq,hkv,d", [(2, 2, 128), (6, 2, 64)])
def test_decode_with_huge_values_of_no_weight(hq, hkv, d):
    """The largest finite bf16 among the values of keys whose weight underflows to 0 adds nothing: in the middle of a chunk and
    in the last row, of which the rows past the end are copies."""
    from paper_2404_09529_b200.runner import DecodeBatch
    lengths = np.array([1, 16, 17, 50, 64, 65, 200, 700], np.int32)
    dec = DecodeBatch(lengths, hq, hkv, d, 10000.0, room=2)
    g = torch.Generator().manual_seed(hq + d)
    for pool in (dec.k_cache, dec.v_cache):
        pool.copy_(torch.randn(pool.shape, generator=g).to(torch.bfloat16))
    qn, kn, vn = (torch.randn(dec.k, h, d, generator=g).to(torch.bfloat16) for h in (hq, hkv, hkv))
    qn[:, :, d // 2 - 1] = 20                     # slowly turning: hardly rotated, positive at every position here
    qn[:, :, d - 1] = 0
    for i, l in enumerate(int(x) for x in lengths):
        ck, cv = dec.caches(i)
        for key in {l // 3, l // 2, l - 1}:
            ck[:, key, d // 2 - 1] = -100         # weight exp(-170) or less
            cv[:, key] = 3.3e38
    before = [tuple(to64(c[:, :int(l)]) for c in dec.caches(i)) for i, l in enumerate(lengths)]
    got = to64(dec.step(qn.cuda(), kn.cuda(), vn.cuda()))
    for i in range(dec.k):
        kc, vc = before[i]
        vc = np.where(vc > 1e38, 0.0, vc)         # (their part of O is below 1e-30, but not of an fp64 sum of 1e38 exp(-170))
        ref = orc.decode_step(to64(qn[i]), to64(kn[i]), to64(vn[i]), kc, vc, 10000.0)[0]
        assert np.abs(got[i] - ref).max() <= MAX_ABS_TOL, (i, np.abs(got[i] - ref).max())
