"""Sizes at which a kernel or a rule of a dispatch can go wrong (edges of tiles, remainders, the smallest and largest of a
range), against the CPU oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_2412_14468_b200 import binding as ha
from paper_2412_14468_b200 import workloads as wl
from tests._fake import BATCH_CASES, NEXT_TO_BATCH_CASES, PER_HEAD_BATCH_CASES, budgets, ragged
from tests._util import OUT_TOL, assert_out_close, max_abs_diff_bf16, u16
from tests.test_gpu_parity import _attn_inputs, _check_gather, _run_step, _check_score_topk, _check_score_topk_wide, _page_codes, _wide_codes, _wide_mapping, \
    test_whole_step_with_keys_values_and_signatures_all_paged as _whole_paged_step

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("n_bits", [64, 128, 256, 512])
@pytest.mark.parametrize("B,G", [(1, 1), (3, 8), (40, 8)])
def test_encode_wide_of_single_vectors_at_every_item_width(n_bits, B, G):
    """One token per head takes the vector kernel: few vectors (one per CTA), more than CTA slots (items of several
    vectors, several items per CTA), signatures shared by n_bits / 128 CTAs; strided inputs, no biases for the first."""
    Hkv, W = 2, n_bits // 64
    m = _wide_mapping(Hkv, n_bits, 60 + n_bits)
    if B == 1:
        m = {k: v for k, v in m.items() if k.startswith("w")}
    mn = wl.mapping_numpy(m)
    bias = lambda name, g: mn[name][g] if name in mn else None  # noqa: E731
    x = torch.randn(B, Hkv * G, 3, 128, device=DEV, generator=torch.Generator(DEV).manual_seed(B)).to(torch.bfloat16)[:, :, 1]
    codes = torch.full((B, Hkv * G, 2, W), -1, dtype=torch.int64, device=DEV)
    ha.ha_encode_wide(ha.MappingWide(m), G, x, codes)
    got = codes.cpu().numpy().view(np.uint64)
    xu = u16(x.contiguous()).reshape(B, Hkv, G, 128)
    for g in range(Hkv):
        ref = oracle.encode_wide(np.ascontiguousarray(xu[:, g].reshape(B * G, 128)), mn["w1"][g], mn["w2"][g], mn["w3"][g],
                                 bias("b1", g), bias("b2", g), bias("b3", g))
        assert np.array_equal(got[:, g * G:(g + 1) * G, 0].reshape(B * G, W), ref)
    assert (codes[:, :, 1] == -1).all()


@pytest.mark.parametrize("n_bits", [64, 512])
@pytest.mark.parametrize("lens", [(2047, 2048, 2049), (16383, 16385), (131071, 131072), (131073,), tuple(range(1, 1601, 23))])
def test_score_topk_wide_at_row_and_cluster_edges(n_bits, lens):
    """Rows of 2048 tokens, the longest sequence of the one-kernel path and the first beyond it, and a batch that takes
    smaller clusters."""
    rng = np.random.default_rng(len(lens))
    W, Hkv, G = n_bits // 64, 2, 2
    n_cap = max(lens)
    kc = _wide_codes(rng, len(lens) * Hkv * n_cap, W).reshape(len(lens), Hkv, n_cap, W)
    qc = _wide_codes(rng, len(lens) * Hkv * G, W).reshape(len(lens), Hkv * G, W)
    _check_score_topk_wide(n_bits, qc, kc, list(lens), [max(1, n // 5) for n in lens], Hkv * G, Hkv, 3, 5)


@pytest.mark.parametrize("page_size", [2, 4, 8, 32])
@pytest.mark.parametrize("lens", [(255, 256, 257), (2049, 16383, 16385), (131072, 131071), (131073,), tuple(range(1, 2200, 29))])
def test_score_topk_paged_at_row_page_and_cluster_edges(page_size, lens):
    """Pages below and above a lane's eight tokens; rows of 256 tokens, slices of 2048, the longest sequence of the cluster
    kernel and the first beyond it, and a batch that takes smaller clusters."""
    rng = np.random.default_rng(page_size + len(lens))
    B, Hq, Hkv, G = len(lens), 8, 2, 4
    n_cap, ks = max(lens), [max(1, n // 7) for n in lens]
    n_sink, n_local = 2, 9
    codes = rng.integers(0, 2**32, size=(B, Hkv, n_cap), dtype=np.uint64).astype(np.uint32)
    qc = rng.integers(0, 2**32, size=(B, Hq), dtype=np.uint64).astype(np.uint32)
    pool, table = _page_codes(codes, lens, page_size, rng)
    k_max = max(ks) + n_sink + n_local
    shape = ha.make_shape(B, Hq, Hkv, 1.0, n_sink=n_sink, n_local=n_local)
    ws = ha.alloc_workspace(shape, n_cap, k_max)
    idx = torch.full((B, Hkv, k_max), 5, dtype=torch.int32, device=DEV)
    cnt = torch.full((B, Hkv), 5, dtype=torch.int32, device=DEV)
    to = lambda a: torch.from_numpy(a.view(np.int32)).to(DEV)  # noqa: E731
    ha.ha_score_topk_paged(shape, to(qc), to(pool), to(table), torch.tensor(lens, dtype=torch.int32, device=DEV),
                           torch.tensor(ks, dtype=torch.int32, device=DEV), 0, n_cap, k_max, idx, cnt, ws)
    got, n_got = idx.cpu().numpy(), cnt.cpu().numpy()
    for b, n in enumerate(lens):
        for g in range(Hkv):
            ref = oracle.topk_windows(oracle.score(qc[b, g * G:(g + 1) * G], codes[b, g, :n]), ks[b], n_sink, n_local)
            assert n_got[b, g] == len(ref) and np.array_equal(got[b, g, :len(ref)], ref) and (got[b, g, len(ref):] == -1).all()


@pytest.mark.parametrize("page_size,B", [(4, 2), (16, 45), (2, 45)])
def test_whole_paged_step_in_one_launch_and_in_three(page_size, B):
    """Few units take the one-kernel step over the pools, 90 units ENCODE, SCORE + TOPK and GATHER-ATT one by one."""
    _whole_paged_step(page_size, B)


@pytest.mark.parametrize("G", [1, 8])
@pytest.mark.parametrize("lens", [(65537,) + (4095, 4096, 4097) + (0, 1) * 4, (262144,) + (70001,) * 11, (262145,) + (33000,) * 11,
                                  (131072,) * 3 + tuple(range(60000, 60015))])
@pytest.mark.parametrize("page_size", [0, 16])
def test_score_topk_on_clusters_of_large_ctas(G, lens, page_size):
    """24 to 36 units with sequences of 65537 to 262144 tokens: slices of 4096 tokens, one row and eight, sequences shorter than
    a slice beside long ones, and the first length beyond the range."""
    rng = np.random.default_rng(G + len(lens))
    B, Hkv = len(lens), 2
    Hq, n_cap, ks = Hkv * G, max(lens) // 64 * 64 + 64, [max(1, n // 9) for n in lens]
    n_sink, n_local = 130, 7
    k_max = max(ks) + n_sink + n_local
    codes = rng.integers(0, 2**32, size=(B, Hkv, n_cap), dtype=np.uint64).astype(np.uint32)
    codes[0, 0, :200] = codes[0, 0, 5]                              # ties decided by token index
    qc = rng.integers(0, 2**32, size=(B, Hq), dtype=np.uint64).astype(np.uint32)
    shape = ha.make_shape(B, Hq, Hkv, 1.0, n_sink=n_sink, n_local=n_local)
    ws = ha.alloc_workspace(shape, n_cap, k_max)
    idx = torch.full((B, Hkv, k_max), 5, dtype=torch.int32, device=DEV)
    cnt = torch.full((B, Hkv), 5, dtype=torch.int32, device=DEV)
    to = lambda a: torch.from_numpy(a.view(np.int32)).to(DEV)  # noqa: E731
    lt, kt = torch.tensor(lens, dtype=torch.int32, device=DEV), torch.tensor(ks, dtype=torch.int32, device=DEV)
    if page_size:
        pool, table = _page_codes(codes, lens, page_size, rng)
        ha.ha_score_topk_paged(shape, to(qc), to(pool), to(table), lt, kt, 0, max(lens), k_max, idx, cnt, ws)
    else:
        ha.ha_score_topk(shape, to(qc), to(codes), lt, kt, 0, max(lens), k_max, idx, cnt, ws)
    got, n_got = idx.cpu().numpy(), cnt.cpu().numpy()
    for b, n in enumerate(lens):
        for g in range(Hkv):
            s = oracle.score(qc[b, g * G:(g + 1) * G], codes[b, g, :n]) if n else np.zeros(0, np.int32)
            ref = oracle.topk_windows(s, ks[b], n_sink, n_local)
            assert n_got[b, g] == len(ref) and np.array_equal(got[b, g, :len(ref)], ref) and (got[b, g, len(ref):] == -1).all()


@pytest.mark.parametrize("G,Hkv,lens,page_size", [(c[0], c[1], c[2], page) for c in BATCH_CASES + NEXT_TO_BATCH_CASES for page in c[3]],
                         ids=lambda v: f"{len(v)}x{max(v)}" if isinstance(v, list) else None)
def test_score_topk_with_several_units_per_cluster(G, Hkv, lens, page_size):
    """Every cluster size of the batch kernel at the edges of its rule, and the other kernels beside them: lengths dealt out,
    several batches per cluster, windows, ties at the threshold, budgets of nothing and of everything, contiguous and in pages.
    (test_dispatch.py holds the cases to their kernels, batches and staged tables.)"""
    rng = np.random.default_rng(len(lens) + page_size)
    B, Hq, n_cap = len(lens), Hkv * G, max(lens) // 128 * 128 + 128
    ks = budgets(lens)
    n_sink, n_local = (130, 7) if page_size == 16 else (0, 0)
    k_max = max(max(ks) + n_sink + n_local, 1)
    codes = rng.integers(0, 2**32, size=(B, Hkv, n_cap), dtype=np.uint64).astype(np.uint32)
    codes[:, :, 100:400] = codes[:, :, 100:101]                     # ties decided by token index
    qc = rng.integers(0, 2**32, size=(B, Hq), dtype=np.uint64).astype(np.uint32)
    qc[:, 0] = codes[:, 0, 100]                                     # ... at the highest score for the first unit
    shape = ha.make_shape(B, Hq, Hkv, 1.0, n_sink=n_sink, n_local=n_local)
    ws = ha.alloc_workspace(shape, n_cap, k_max)
    idx = torch.full((B, Hkv, k_max), 5, dtype=torch.int32, device=DEV)
    cnt = torch.full((B, Hkv), 5, dtype=torch.int32, device=DEV)
    hist = torch.full((B, Hkv, 33), 5, dtype=torch.int32, device=DEV)
    to = lambda a: torch.from_numpy(a.view(np.int32)).to(DEV)  # noqa: E731
    lt, kt = torch.tensor(lens, dtype=torch.int32, device=DEV), torch.tensor(ks, dtype=torch.int32, device=DEV)
    if page_size:
        pool, table = _page_codes(codes, lens, page_size, rng)
        ha.ha_score_topk_paged(shape, to(qc), to(pool), to(table), lt, kt, 0, max(lens), k_max, idx, cnt, ws, hist_out=hist)
    else:
        ha.ha_score_topk(shape, to(qc), to(codes), lt, kt, 0, max(lens), k_max, idx, cnt, ws, hist_out=hist)
    got, n_got, h_got = idx.cpu().numpy(), cnt.cpu().numpy(), hist.cpu().numpy()
    for b, n in enumerate(lens):
        free = np.ones(n, bool)
        free[:n_sink] = False
        free[max(n - n_local, 0):] = False
        for g in range(Hkv):
            s = oracle.score(qc[b, g * G:(g + 1) * G], codes[b, g, :n]) if n else np.zeros(0, np.int32)
            ref = oracle.topk_windows(s, ks[b], n_sink, n_local)
            assert n_got[b, g] == len(ref) and np.array_equal(got[b, g, :len(ref)], ref) and (got[b, g, len(ref):] == -1).all()
            assert np.array_equal(h_got[b, g], np.bincount(s[free], minlength=33))


@pytest.mark.parametrize("B,Hkv,G,longest,_cs", PER_HEAD_BATCH_CASES)
@pytest.mark.parametrize("page_size", [16, 64])
def test_score_topk_per_head_with_several_units_per_cluster(B, Hkv, G, longest, _cs, page_size):
    """Lists per query head over pages: G units share the signatures of a KV head."""
    rng = np.random.default_rng(B + page_size)
    lens = ragged(B, longest)
    ks = budgets(lens)
    k_max, Hq = max(ks), Hkv * G
    codes = rng.integers(0, 2**32, size=(B, Hkv, longest), dtype=np.uint64).astype(np.uint32)
    codes[:, :, 100:400] = codes[:, :, 100:101]                     # ties decided by token index
    qc = rng.integers(0, 2**32, size=(B, Hq), dtype=np.uint64).astype(np.uint32)
    pool, table = _page_codes(codes, lens, page_size, rng)
    shape = ha.make_shape(B, Hq, Hkv, 1.0)
    ws = ha.alloc_workspace(ha.make_shape(B, Hq, Hq, 1.0), longest, k_max)
    idx = torch.full((B, Hq, k_max), 5, dtype=torch.int32, device=DEV)
    cnt = torch.full((B, Hq), 5, dtype=torch.int32, device=DEV)
    to = lambda a: torch.from_numpy(a.view(np.int32)).to(DEV)  # noqa: E731
    ha.ha_score_topk_per_head_paged(shape, to(qc), to(pool), to(table), torch.tensor(lens, dtype=torch.int32, device=DEV),
                                    torch.tensor(ks, dtype=torch.int32, device=DEV), 0, longest, k_max, idx, cnt, ws)
    got, n_got = idx.cpu().numpy(), cnt.cpu().numpy()
    for b, n in enumerate(lens):
        for h in range(Hq):
            ref = oracle.topk(oracle.score(qc[b, h:h + 1], codes[b, h // G, :n]) if n else np.zeros(0, np.int32), ks[b])
            assert n_got[b, h] == len(ref) and np.array_equal(got[b, h, :len(ref)], ref) and (got[b, h, len(ref):] == -1).all()


def test_score_topk_of_many_short_sequences_of_one_length():
    """464 units of at most 10240 tokens, one budget: one CTA a cluster."""
    rng = np.random.default_rng(9)
    B, Hkv, G, n = 58, 8, 4, 1111
    codes = rng.integers(0, 2**32, size=(B, Hkv, 1112), dtype=np.uint64).astype(np.uint32)
    qc = rng.integers(0, 2**32, size=(B, Hkv * G), dtype=np.uint64).astype(np.uint32)
    _check_score_topk(qc, codes, [n] * B, [40] * B, Hkv * G, Hkv, k_uniform=40)


@pytest.mark.parametrize("G", [1, 4, 8])
@pytest.mark.parametrize("lens,sparsity", [((32769, 1), 32), ((65536, 33000), 64), ((65535,), 16), ((65537, 4), 64), ((131072, 70001), 100)])
def test_one_launch_step_of_long_sequences(G, lens, sparsity):
    """Sequences beyond 32768 tokens in one launch (one row stage up to 65536 tokens and 2560 entries, two up to 131072): lists
    and signatures equal to those of the entry points one by one, outputs to fp32 reordering; the same over pages, and from
    host buffers."""
    n_sink, n_local = 70, 40
    cfg = wl.Config("long-fused", 71, len(lens), list(lens), None, 0.01, n_q_heads=2 * G, n_kv_heads=2, sparsity=sparsity)
    w = wl.make_workload(cfg, DEV)
    B, Hq, Hkv, n_cap = cfg.batch, 2 * G, 2, (w["n_cap"] + 63) // 64 * 64
    k_max = w["k_max"] + n_sink + n_local
    shape = ha.make_shape(B, Hq, Hkv, w["sm_scale"], n_sink=n_sink, n_local=n_local)
    ws = ha.alloc_workspace(shape, n_cap, k_max)
    mq, mk = ha.Mapping(w["map_q"]), ha.Mapping(w["map_k"])
    clean = torch.zeros(B, Hkv, n_cap, dtype=torch.int32, device=DEV)
    ha.ha_encode(mk, 1, w["K"], clean)
    for b, n in enumerate(lens):                                   # slots past a sequence stay untouched by a step
        clean[b, :, n:] = 0x11111111
    last = w["seq_lens"].long() - 1
    stale = clean.clone()
    stale[torch.arange(B, device=DEV), :, last] = 0x0BADF00D
    new = lambda *s, t=torch.int32: torch.zeros(*s, dtype=t, device=DEV)  # noqa: E731

    qr, ir, cr, outr = new(B, Hq), new(B, Hkv, k_max), new(B, Hkv), new(B, Hq, 128, t=torch.bfloat16)
    ha.ha_encode(mq, G, w["q"], qr.unsqueeze(2))
    ha.ha_score_topk(shape, qr, clean, w["seq_lens"], w["k_per_seq"], 0, w["n_cap"], k_max, ir, cr, ws)
    ha.ha_gather_attn(shape, w["q"], w["K"], w["V"], w["seq_lens"], ir, cr, k_max, outr, ws)

    def check(idx, cnt, out, qc=None):
        assert torch.equal(idx, ir) and torch.equal(cnt, cr) and (qc is None or torch.equal(qc, qr))
        assert max_abs_diff_bf16(u16(out), u16(outr)) <= OUT_TOL
        assert ha.ha_read_device_status(ws) == 0

    def step(fn, *args):
        qc, idx, cnt, out = new(B, Hq), new(B, Hkv, k_max), new(B, Hkv), new(B, Hq, 128, t=torch.bfloat16)
        before = ha.ha_kernel_launches()
        fn(shape, mq, mk, w["q"], w["k_new"], *args, w["seq_lens"], w["k_per_seq"], 0, w["n_cap"], k_max, qc, idx, cnt, out, ws)
        assert ha.ha_kernel_launches() - before == 1
        check(idx, cnt, out, qc)

    codes = stale.clone()
    step(ha.ha_sparse_decode, w["K"], w["V"], codes)
    assert torch.equal(codes, clean)
    page = 16
    pps = n_cap // page
    table = torch.randperm(B * pps, device=DEV, generator=torch.Generator(DEV).manual_seed(3)).view(B, pps)

    def pool(x):
        x = torch.nn.functional.pad(x, (0, 0) * (x.dim() - 3) + (0, n_cap - x.shape[2]))
        p = torch.empty((B * pps, Hkv, page) + tuple(x.shape[3:]), dtype=x.dtype, device=DEV)
        for b in range(B):
            p[table[b]] = x[b].reshape((Hkv, pps, page) + tuple(x.shape[3:])).transpose(0, 1)
        return p

    pc = pool(stale)
    step(ha.ha_sparse_decode_paged_codes, pool(w["K"]), pool(w["V"]), pc, table.to(torch.int32))
    assert torch.equal(pc, pool(clean))
    pin = lambda t: t.cpu().pin_memory()  # noqa: E731
    codes, idx, cnt, out = stale.clone(), new(B, Hkv, k_max), new(B, Hkv), torch.zeros(B, Hq, 128, dtype=torch.bfloat16).pin_memory()
    ha.ha_sparse_decode_host(shape, mq, mk, pin(w["q"]), pin(w["k_new"]), pin(w["v_new"]), w["K"].clone(), w["V"].clone(), codes,
                             w["seq_lens"], w["k_per_seq"], 0, w["n_cap"], k_max, idx, cnt, out, ws)
    check(idx, cnt, out)
    assert torch.equal(codes, clean)


@pytest.mark.parametrize("B", [10, 30])
@pytest.mark.parametrize("k,launches", [(2560, 1), (2561, 3)])
def test_step_at_the_longest_list_of_one_launch(B, k, launches):
    """20 and 60 units (clusters of 8 and of 4): the longest list that one launch takes and the first beyond it give the lists and
    outputs of the entry points one by one; GATHER-ATT at these lengths against the oracle."""
    cfg = wl.Config("longest-list", 72, B, [2 * k] * B, None, 0.02, n_q_heads=8, n_kv_heads=2, sparsity=2)
    w = wl.make_workload(cfg, DEV)
    _run_step(w)
    before = ha.ha_kernel_launches()
    r = _run_step(w)
    assert ha.ha_kernel_launches() - before == launches + 1        # and the signature cache
    shape = ha.make_shape(B, 8, 2, w["sm_scale"])
    ws = ha.alloc_workspace(shape, 2 * k, k)
    idx, cnt, out = torch.zeros_like(r["idx"]), torch.zeros_like(r["cnt"]), torch.zeros_like(r["out"])
    ha.ha_score_topk(shape, r["qc"], r["kc"], w["seq_lens"], w["k_per_seq"], 0, 2 * k, k, idx, cnt, ws)
    ha.ha_gather_attn(shape, w["q"], w["K"], w["V"], w["seq_lens"], idx, cnt, k, out, ws)
    assert torch.equal(idx, r["idx"]) and torch.equal(cnt, r["cnt"]) and max_abs_diff_bf16(u16(out), u16(r["out"])) <= OUT_TOL
    n = 3000
    lists = np.random.default_rng(k).integers(0, n, size=(1, 2, k)).astype(np.int32)
    _check_gather(*_attn_inputs(1, 8, 2, n, 5), [n], lists, np.full((1, 2), k, np.int32), 0.09)


@pytest.mark.parametrize("k", [4095, 4096, 4097])
def test_gather_attn_at_the_longest_list_of_clusters_of_four(k):
    """44 units: up to 4096 entries on clusters of 4, more on the split-K kernel; full and ragged lists."""
    B, Hkv, G, n = 22, 2, 2, 5000
    rng = np.random.default_rng(k)
    lists = rng.integers(0, n, size=(B, Hkv, k)).astype(np.int32)
    cnt = np.where(np.arange(B * Hkv).reshape(B, Hkv) % 3 == 0, k, rng.integers(0, k, size=(B, Hkv))).astype(np.int32)
    _check_gather(*_attn_inputs(B, Hkv * G, Hkv, n, 6), [n] * B, lists, cnt, 0.09)


@pytest.mark.parametrize("B,G", [(1, 8), (17, 4), (18, 4), (17, 8), (18, 8), (17, 1), (300, 1), (592, 2)])
def test_gather_attn_split_k_merges_of_many_and_of_few_parts(B, G):
    """One unit cut over every CTA, 17 CTAs per unit (the first grid whose merge takes the wide pass) and 16, units that are cut
    in two, and whole units per CTA; lists in any order."""
    n, k = 300, 4200
    lists = np.random.default_rng(B).integers(0, n, size=(B, 1, k)).astype(np.int32)
    cnt = np.full((B, 1), k, np.int32)
    cnt[::3] -= 1001
    _check_gather(*_attn_inputs(B, G, 1, n, 6), [n] * B, lists, cnt, 0.09)


@pytest.mark.parametrize("n_bits,B,n", [(64, 37, 2049), (64, 38, 2100), (128, 112, 300), (256, 18, 9000), (256, 19, 9000),
                                        (512, 27, 4097), (512, 28, 4097), (512, 60, 300), (64, 30, 66000), (512, 2, 131072)])
def test_score_topk_wide_where_the_cluster_size_changes(n_bits, B, n):
    """Two units a sequence: as many clusters of 8 or 4 as are resident at once and one more, at few and at eight rows per CTA."""
    rng = np.random.default_rng(B)
    W, Hkv = n_bits // 64, 2
    lens = [n - 7 * (b % 5) for b in range(B)]
    kc = _wide_codes(rng, B * Hkv * n, W).reshape(B, Hkv, n, W)
    qc = _wide_codes(rng, B * Hkv, W).reshape(B, Hkv, W)
    _check_score_topk_wide(n_bits, qc, kc, lens, [max(1, m // 9) for m in lens], Hkv, Hkv, 2, 3)


@pytest.mark.parametrize("uniform,k", [(True, 2048), (True, 2049), (True, 4100), (False, 2048), (False, 2049), (False, 4100)])
def test_step_on_the_split_k_kernel_with_two_and_with_three_row_stages(uniform, k):
    """160 units: one budget for all sequences takes two row stages at any length, a budget per sequence up to 2048 entries.  All
    signatures, lists and outputs against the oracle."""
    B, Hq, Hkv = 80, 4, 2
    n = 4200 if k > 3000 else 2100
    cfg = wl.Config("row-stages", 73, B, [n] * B, k, 0.02, n_q_heads=Hq, n_kv_heads=Hkv)
    w = wl.make_workload(cfg, DEV)
    lens = [n - (0 if uniform else 3 * (b % 7)) for b in range(B)]
    ks = [k - (0 if uniform else 5 * (b % 11)) for b in range(B)]
    shape = ha.make_shape(B, Hq, Hkv, w["sm_scale"])
    ws = ha.alloc_workspace(shape, n, k)
    mq, mk = ha.Mapping(w["map_q"]), ha.Mapping(w["map_k"])
    kc = torch.zeros(B, Hkv, -(-n // 4) * 4, dtype=torch.int32, device=DEV)
    ha.ha_encode(mk, 1, w["K"], kc)
    new = lambda *s, t=torch.int32: torch.zeros(*s, dtype=t, device=DEV)  # noqa: E731
    qc, idx, cnt, out = new(B, Hq), new(B, Hkv, k), new(B, Hkv), new(B, Hq, 128, t=torch.bfloat16)
    i32 = lambda v: torch.tensor(v, dtype=torch.int32, device=DEV)  # noqa: E731
    Kc = kc.cpu().numpy().view(np.uint32)[:, :, :n].copy()
    ha.ha_sparse_decode(shape, mq, None, w["q"], None, w["K"], w["V"], kc, i32(lens), None if uniform else i32(ks), k if uniform else 0, n, k,
                        qc, idx, cnt, out, ws)
    ref = oracle.decode_step(u16(w["q"]), None, u16(w["K"]), u16(w["V"]), Kc, wl.mapping_numpy(w["map_q"]), wl.mapping_numpy(w["map_k"]),
                             lens, ks, sm_scale=w["sm_scale"], n_threads=4)
    got, n_got = idx.cpu().numpy(), cnt.cpu().numpy()
    assert np.array_equal(n_got, ref["count"])
    for b in range(B):
        assert np.array_equal(got[b, :, :ks[b]], ref["idx"][b, :, :ks[b]]) and (got[b, :, ks[b]:] == -1).all()
    assert_out_close(u16(out), ref["out"])
    assert ha.ha_read_device_status(ws) == 0
