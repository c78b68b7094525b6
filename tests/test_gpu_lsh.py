"""GPU parity of the SimHash-indexed key check (Eq. 1; Algorithm 1's cache search) against the oracle.

Signatures are sign decisions of fp32 tensor-core dot products; the oracle takes them in fp64. Bits whose
projection is within 1e-4 of zero may legitimately differ: they are counted, and the queries whose outcome such
a bit could change are excluded from the exact comparison (reported, at most a few)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2608_01718_gb300 import build
from paper_2608_01718_gb300 import lacache as L
from paper_2608_01718_gb300 import workloads as wl

from parity import compare, fill, gpu_lookup, log_report, new_cache, oracle_queries, oracle_store, params

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def library():
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    build.build()
    L.load()


def _unpack(words, bits):
    w = words.astype(np.uint64)
    out = np.zeros((w.shape[0], bits), dtype=bool)
    for i in range(bits):
        out[:, i] = (w[:, i // 32] >> np.uint64(i % 32)) & np.uint64(1)
    return out


@pytest.mark.parametrize("bits", [128, 256, 512])
def test_signatures_match_the_oracle(bits):
    w = wl.WORKLOADS["mid-1m"].scaled(n=20_000)
    R = wl.hyperplanes(bits, w.d, device="cuda")
    st = oracle_store(w)
    with new_cache(w, L.LACACHE_STAGE1_LSH) as cache:
        fill(cache, w)
        L.lacache_enable_lsh(cache.h, bits, 40, R)
        sig = torch.empty((w.n, bits // 32), dtype=torch.int32, device="cuda")
        L.lacache_read_signatures(cache.h, 0, w.n, sig)
        torch.cuda.synchronize()
    got = _unpack(sig.cpu().numpy().view(np.uint32), bits)
    want, amb = oracle.signatures(st.key, wl.bf16_bits(R))
    diff = got != want
    assert not np.any(diff & ~amb), "a signature bit differs away from a zero projection"
    assert amb.mean() < 1e-3


def _expected_lsh_kernel(batch, bits):
    # the tensor-core scan from 48 queries at 256 bits and from 40 at 128 and 512 bits (on stores of fewer than 131,072
    # entries; the callers' larger ones see at most 32 queries, which the popcount scan has below 2,097,152 entries)
    return L.LACACHE_STAGE1_LSH_TENSOR if batch >= (48 if bits == 256 else 40) else L.LACACHE_STAGE1_LSH


# popcount-1 / -2: a pass of fewer queries than one group of 8 (only their distances are computed);
# tensor-40: the tensor-core scan at 128 and 512 bits, two passes of the popcount scan at 256 bits (its switch is at
# 48);
# popcount-36: two passes of 32 queries; tensor-200: two passes of 128 queries, the last one ragged
@pytest.mark.parametrize("batch", [1, 2, 5, 32, 36, 40, 64, 200],
                         ids=["popcount-1", "popcount-2", "popcount-5", "popcount-32", "popcount-36", "tensor-40",
                              "tensor-64", "tensor-200"])
@pytest.mark.parametrize("bits", [128, 256, 512])
def test_lsh_lookup_matches_the_oracle(bits, batch):
    _check_lsh_lookup(wl.WORKLOADS["mid-1m"].scaled(n=70_000, batch=batch), bits)


@pytest.mark.parametrize("batch", [1, 5])
@pytest.mark.parametrize("bits", [128, 256, 512])
def test_lsh_lookup_at_a_low_threshold_matches_the_oracle(bits, batch):
    # tau_c = 0.8 gives radii of 45, 79 and 142 bits, too wide for the scan's prefix test to reject unrelated
    # pairs: it tests whole signatures (at 512 bits through its shared-memory ring)
    _check_lsh_lookup(wl.WORKLOADS["mid-1m"].scaled(n=70_000, batch=batch, tau_c=0.8), bits)


@pytest.mark.parametrize("bits", [128, 256])
def test_single_query_lookups_on_a_large_store_match_the_oracle(bits):
    # 2.6M entries of d = 64: 304 splits of about 8,553 entries (17 tiles, the last one ragged). One-query lookups
    # on splits of at least 16 tiles stream the signatures through the scan's shared-memory ring (at 512 bits every
    # lookup does, and the cases above cover it); eight such lookups, compared as one batch
    _check_lsh_lookup(wl.WORKLOADS["mid-1m"].scaled(n=2_600_000, d=64, batch=8), bits, one_at_a_time=True)


@pytest.mark.slow
@pytest.mark.parametrize("bits", [128, 256, 512])
def test_lsh_lookup_at_full_size_matches_the_oracle(bits):
    # mid-1m at full size (1,048,576 entries, B = 32), as the benchmark's SimHash line times it: the popcount scan
    # with its prefix test, in its register form at 128 and 256 bits and its shared-memory ring form at 512
    _check_lsh_lookup(wl.WORKLOADS["mid-1m"], bits)


@pytest.mark.parametrize("top_c", [1, 32])
@pytest.mark.parametrize("batch", [16, 64], ids=["popcount", "tensor"])
def test_lsh_top_c_extremes_match_the_oracle(batch, top_c):
    # one candidate per query (every list insertion replaces the head) and the longest lists the kernels hold
    _check_lsh_lookup(wl.WORKLOADS["mid-1m"].scaled(n=40_000, batch=batch, top_c=top_c), 256)


def _check_lsh_lookup(w, bits, one_at_a_time=False):
    batch = w.batch
    radius = wl.lsh_radius(w.tau_c, bits)
    R = wl.hyperplanes(bits, w.d, device="cuda")
    st = oracle_store(w)
    with new_cache(w, L.LACACHE_STAGE1_LSH) as cache:
        fill(cache, w)
        L.lacache_enable_lsh(cache.h, bits, radius, R)
        q = wl.batch(w, 0, device="cuda")
        if one_at_a_time:
            parts = []
            for i in range(batch):
                parts.append(gpu_lookup(cache, {k: q[k][i:i + 1] for k in ("emb", "prefix", "ids")}))
                assert cache.last_launch()[1] == L.LACACHE_STAGE1_LSH
            g = {k: np.concatenate([r[k] for r in parts]) for k in parts[0]}
        else:
            g = gpu_lookup(cache, q)
            assert cache.last_launch()[1] == _expected_lsh_kernel(batch, bits)
    oq = oracle_queries(q)
    p = params(w)
    res, amb = oracle.lookup_lsh(st, oq, p, wl.bf16_bits(R), radius)
    keep = np.nonzero(~amb)[0]
    sub = oracle.Result(**{f: getattr(res, f)[keep] for f in res.__dataclass_fields__})
    rep = compare(g, sub, p, rows=keep)
    amb_n = w.batch - len(keep)
    log_report(f"lsh bits={bits} B={batch} c={w.top_c} radius={radius} ({amb_n} queries with ambiguous bits)", rep)
    # queries with a signature bit within the fp32/fp64 ambiguity of zero are set aside: at most 1 in 50
    assert rep.exact + rep.band == len(keep) and len(keep) >= w.batch - max(2, w.batch // 50)
    if batch >= 16:
        assert rep.hits > 0 and rep.rejects > 0 and rep.misses > 0
    # at this radius the index keeps every near-duplicate's target: the decisions equal the exact lookup's
    exact = oracle.lookup(st, oq, p)
    assert np.array_equal(res.status, exact.status) and np.array_equal(res.entry_id, exact.entry_id)


@pytest.mark.parametrize("bits", [256, 512])
@pytest.mark.parametrize("batch", [16, 64], ids=["popcount", "tensor"])
def test_full_radius_equals_the_exact_scan_and_appends_are_signed(batch, bits):
    # radius = bits admits every pair: the queue overflows on every tile (at 512 bits the popcount scan's ring form,
    # whose queue is a quarter of the register form's), and appended entries must be signed before the next lookup
    w = wl.WORKLOADS["serve-2m"].scaled(n=30_000, batch=batch, clusters=300)
    R = wl.hyperplanes(bits, w.d, device="cuda")
    with new_cache(w, L.LACACHE_STAGE1_TENSOR, capacity=w.n + 4 * w.batch) as exact_cache, \
            new_cache(w, L.LACACHE_STAGE1_LSH, capacity=w.n + 4 * w.batch) as lsh_cache:
        fill(exact_cache, w)
        fill(lsh_cache, w)
        L.lacache_enable_lsh(lsh_cache.h, bits, bits, R)      # radius = bits: nothing is pruned
        for step in range(3):
            q = wl.batch(w, step, device="cuda")
            a = exact_cache.lookup(q["emb"], q["prefix"], q["ids"])
            b = lsh_cache.lookup(q["emb"], q["prefix"], q["ids"])
            assert lsh_cache.last_launch()[1] == _expected_lsh_kernel(batch, bits)
            assert torch.equal(a["status"], b["status"]) and torch.equal(a["entry_id"], b["entry_id"])
            assert torch.equal(a["cand_id"], b["cand_id"])
            assert torch.allclose(a["cand_score"], b["cand_score"], atol=2e-3, equal_nan=True)
            exact_cache.append_misses(q["emb"], q["prefix"], q["ids"], a["status"])
            first, m = lsh_cache.append_misses(q["emb"], q["prefix"], q["ids"], b["status"])
        sig = torch.empty((m, bits // 32), dtype=torch.int32, device="cuda")
        L.lacache_read_signatures(lsh_cache.h, first, m, sig)
        torch.cuda.synchronize()
        # the appended entries are the last batch's non-HIT queries, in query order
        miss = torch.nonzero(b["status"] != L.LACACHE_HIT).flatten()
        assert len(miss) == m
        rows = wl.bf16_bits(q["emb"][miss])
    want, amb = oracle.signatures(rows, wl.bf16_bits(R))
    assert not np.any((_unpack(sig.cpu().numpy().view(np.uint32), bits) != want) & ~amb)


@pytest.mark.parametrize("n", [1, 127, 129, 255, 2_200, 38_913])
@pytest.mark.parametrize("bits,batch", [(128, 65), (128, 129), (256, 48), (256, 300), (512, 97)])
def test_tensor_scan_block_and_pass_edges_equal_the_exact_scan(bits, batch, n):
    # the tensor-core scan at the edges of its 128-entry blocks and 8 KB stages (a ragged last block, one block per
    # split, 38,913 entries = 2 blocks on all splits and 3 on some), of its 128-query passes and of its 32-query
    # column chunks; radius = bits admits every pair, so the lookup is the exact scan's and the queue runs over
    w = wl.WORKLOADS["mid-1m"].scaled(n=n, d=64, batch=batch, clusters=8)
    R = wl.hyperplanes(bits, w.d, device="cuda")
    with new_cache(w, L.LACACHE_STAGE1_TENSOR) as exact_cache, new_cache(w, L.LACACHE_STAGE1_LSH) as cache:
        fill(exact_cache, w)
        fill(cache, w)
        L.lacache_enable_lsh(cache.h, bits, bits, R)
        q = wl.batch(w, 0, device="cuda")
        a = exact_cache.lookup(q["emb"], q["prefix"], q["ids"])
        b = cache.lookup(q["emb"], q["prefix"], q["ids"])
        cache.sync()
        assert cache.last_launch()[1] == L.LACACHE_STAGE1_LSH_TENSOR
        # fp32 sums of 64 products of bf16 unit rows in two orders: |difference| <= 64 * 2^-24 * sum |x y| < 4e-6
        assert torch.equal(a["n_cand"], b["n_cand"])
        assert torch.allclose(a["key_score"], b["key_score"], rtol=0, atol=4e-6)
        assert torch.allclose(a["cand_score"], b["cand_score"], rtol=0, atol=4e-6, equal_nan=True)


@pytest.mark.parametrize("batch", [8, 64], ids=["popcount", "tensor"])
def test_host_buffer_lookups_through_the_index_match_device_lookups(batch):
    # inputs from mapped pinned host memory: the gather kernel writes them, the query-signature kernel waits for
    # it before reading, and three lookups are in flight on one stream (each gather runs under the stage 2 before)
    w = wl.WORKLOADS["mid-1m"].scaled(n=40_000, batch=batch)
    bits = 256
    R = wl.hyperplanes(bits, w.d, device="cuda")
    with new_cache(w, L.LACACHE_STAGE1_LSH) as cache:
        fill(cache, w)
        L.lacache_enable_lsh(cache.h, bits, wl.lsh_radius(w.tau_c, bits), R)
        qs = [wl.batch(w, i, device="cuda") for i in range(3)]
        want = [gpu_lookup(cache, q) for q in qs]
        hq = [{k: q[k].cpu().pin_memory() for k in ("emb", "prefix", "ids")} for q in qs]
        outs = [L.alloc_result(w.batch, w.top_c, "cpu", pinned=True) for _ in qs]
        stream = torch.cuda.current_stream()
        for q, o in zip(hq, outs):
            L.lacache_lookup_host_async(cache.h, q["emb"], q["prefix"], q["ids"], o, stream)
        stream.synchronize()
        cache.sync()
        assert cache.last_launch()[1] == _expected_lsh_kernel(batch, bits)
        for o, g in zip(outs, want):
            for k, v in o.items():
                assert np.array_equal(v.numpy(), g[k], equal_nan=True), k


def test_lookup_before_the_index_is_enabled_is_refused():
    w = wl.WORKLOADS["mid-1m"].scaled(n=5_000, batch=8)
    q = wl.batch(w, 0, device="cuda")
    with new_cache(w, L.LACACHE_STAGE1_LSH) as cache:
        fill(cache, w)
        with pytest.raises(L.LacacheError) as e:
            cache.lookup(q["emb"], q["prefix"], q["ids"])
        assert e.value.status == L.LACACHE_ERR_INVALID_ARG
        L.lacache_enable_lsh(cache.h, 256, 256, wl.hyperplanes(256, w.d, device="cuda"))
        out = cache.lookup(q["emb"], q["prefix"], q["ids"])
        torch.cuda.synchronize()
        assert out["status"].shape == (w.batch,)


@pytest.mark.parametrize("n,bits,batch", [(131_071, 128, 33), (131_072, 128, 33), (131_072, 512, 39),
                                          (2_097_151, 256, 24), (2_097_152, 128, 32), (2_097_152, 256, 23),
                                          (2_097_152, 256, 24), (2_097_152, 512, 18)])
def test_large_stores_take_the_tensor_scan_earlier_and_equal_the_exact_scan(n, bits, batch):
    # both sides of the store sizes and batches at which lookups change from the popcount to the tensor-core scan. An
    # entry at the key threshold differs in about acos(0.9) / pi = 0.14 of the bits, with a standard deviation of 0.031
    # of 128 bits, so the radius of 0.375 (seven of them) keeps every candidate, and the lookup is the exact scan's
    w = wl.WORKLOADS["mid-1m"].scaled(n=n, d=64, batch=batch)
    first = (18 if bits == 512 else 24 if bits == 256 else 32) if n >= 1 << 21 else \
        33 if n >= 1 << 17 else 48 if bits == 256 else 40
    with new_cache(w, L.LACACHE_STAGE1_TENSOR) as exact_cache, new_cache(w, L.LACACHE_STAGE1_LSH) as cache:
        for c in (exact_cache, cache):
            fill(c, w)
        L.lacache_enable_lsh(cache.h, bits, bits // 2 - bits // 8, wl.hyperplanes(bits, w.d, device="cuda"))
        q = wl.batch(w, 0, device="cuda")
        a, b = gpu_lookup(exact_cache, q), gpu_lookup(cache, q)
        assert cache.last_launch()[1] == (L.LACACHE_STAGE1_LSH_TENSOR if batch >= first else L.LACACHE_STAGE1_LSH)
    hit = a["status"] == L.LACACHE_HIT
    assert hit.any()
    assert np.array_equal(a["status"], b["status"]) and np.array_equal(a["n_cand"], b["n_cand"])
    assert np.array_equal(a["entry_id"][hit], b["entry_id"][hit])


def test_tensor_scan_goes_on_after_the_queue_filled_up():
    # 72 blocks per CTA in rounds of 32, a pass of 128 queries and one of 3, every pair admitted: each round fills the queue
    # over and over, and the scan goes on after it, with whole and ragged rounds and an idle column chunk
    w = wl.WORKLOADS["mid-1m"].scaled(n=1_400_001, d=64, batch=131, clusters=5_000)
    with new_cache(w, L.LACACHE_STAGE1_TENSOR) as exact_cache, new_cache(w, L.LACACHE_STAGE1_LSH) as cache:
        for c in (exact_cache, cache):
            fill(c, w)
        L.lacache_enable_lsh(cache.h, 128, 128, wl.hyperplanes(128, w.d, device="cuda"))
        q = wl.batch(w, 0, device="cuda")
        a, b = gpu_lookup(exact_cache, q), gpu_lookup(cache, q)
        assert cache.last_launch()[1] == L.LACACHE_STAGE1_LSH_TENSOR
    # fp32 sums of 64 products of bf16 unit rows in two orders: |difference| <= 64 * 2^-24 * sum |x y| < 4e-6
    assert np.array_equal(a["n_cand"], b["n_cand"]) and np.array_equal(a["status"], b["status"])
    assert np.allclose(a["key_score"], b["key_score"], rtol=0, atol=4e-6)
    assert np.allclose(a["cand_score"], b["cand_score"], rtol=0, atol=4e-6, equal_nan=True)


@pytest.mark.slow
def test_a_long_drain_of_the_queue_is_not_a_timeout():
    # radius = bits on 48 blocks of 128 rows per CTA: a round of 32 blocks leaves 524,288 pairs to a queue of 4,096. Rows
    # of 8,192 elements whose scores rise along each CTA's range, so that every pair enters a list of 32, make their
    # checks take a quarter of a second (0.8 s when the checker warps did them alone), and for that long the loader, the
    # expanders and the MMA issuer stand still. The budget of their waits, a second, has to count the drain's progress.
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    per, d, batch, bits, top_c, chunk = 48 * 128, 8192, 128, 256, 32, 1 << 15
    n = per * sms
    g = torch.Generator(device="cuda").manual_seed(d)
    u, v = torch.linalg.qr(torch.randn((d, 2), generator=g, device="cuda", dtype=torch.float64))[0].float().T
    q = dict(emb=u.bfloat16().expand(batch, d).contiguous(),
             prefix=torch.zeros((batch, 8), dtype=torch.bfloat16, device="cuda"),
             ids=torch.zeros((batch, 1), dtype=torch.int32, device="cuda"))
    with L.LaCache(d, 1, n, 0.3, 0.5, top_c, max_batch=batch, stage1=L.LACACHE_STAGE1_LSH, prefix_dims=[8],
                   tau_a_models=[0.5]) as cache:
        for r in range(0, n, chunk):
            m = min(chunk, n - r)
            a = (0.5 + 0.49 * ((r + torch.arange(m, device="cuda")) % per) / per).unsqueeze(1)
            key = (a * u + (1 - a * a).sqrt() * v).bfloat16()
            cache.insert(key, torch.zeros((m, 8), dtype=torch.bfloat16, device="cuda"),
                         torch.zeros((m, 1), dtype=torch.int32, device="cuda"))
        L.lacache_enable_lsh(cache.h, bits, bits, wl.hyperplanes(bits, d, device="cuda"))
        got = gpu_lookup(cache, q)   # raises on a timeout
        assert cache.last_launch()[1] == L.LACACHE_STAGE1_LSH_TENSOR
    # the last row of every CTA's range is the same row, and the largest: a tie that goes to the lowest ids
    want = per * np.arange(top_c, dtype=np.int32) + per - 1
    assert np.all(got["cand_id"] == want) and np.all(got["cand_score"] == got["key_score"][:, None])
    # an fp32 sum of 8,192 products of unit rows: within 8192 * 2^-24 * sum |x y| < 5e-4 of the exact one
    best = float(key[-1].double() @ u.bfloat16().double())
    assert np.allclose(got["key_score"], best, rtol=0, atol=5e-4)


@pytest.mark.parametrize("bits,batch,radius,tensor", [(128, 33, 48, True), (128, 33, 49, False), (128, 39, 64, False),
                                                      (128, 40, 64, True), (256, 47, 112, False), (512, 33, 512, False)])
def test_wide_radii_keep_the_switch_of_small_stores(bits, batch, radius, tensor):
    # both sides of the radius and of the batch at which lookups on 131,072 entries go to the tensor-core scan: 33 queries
    # admit 0.098 unrelated pairs per entry at radius 48 of 128 bits and 0.17 at 49. Every radius here keeps all candidates
    # (test_large_stores_take_the_tensor_scan_earlier_and_equal_the_exact_scan), so the lookup is the exact scan's
    w = wl.WORKLOADS["mid-1m"].scaled(n=131_072, d=64, batch=batch)
    with new_cache(w, L.LACACHE_STAGE1_TENSOR) as exact_cache, new_cache(w, L.LACACHE_STAGE1_LSH) as cache:
        for c in (exact_cache, cache):
            fill(c, w)
        L.lacache_enable_lsh(cache.h, bits, radius, wl.hyperplanes(bits, w.d, device="cuda"))
        q = wl.batch(w, 0, device="cuda")
        a, b = gpu_lookup(exact_cache, q), gpu_lookup(cache, q)
        assert cache.last_launch()[1] == (L.LACACHE_STAGE1_LSH_TENSOR if tensor else L.LACACHE_STAGE1_LSH)
    hit = a["status"] == L.LACACHE_HIT
    assert hit.any()
    assert np.array_equal(a["status"], b["status"]) and np.array_equal(a["n_cand"], b["n_cand"])
    assert np.array_equal(a["entry_id"][hit], b["entry_id"][hit])
