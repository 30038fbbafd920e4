"""What the library is timed at: the calls that a user of it makes, over the range of sizes that they meet.

Six kinds of case, each one pass through the public entry points of `binding`:

  step      `ha_sparse_decode`, the layer-step of a decoder (signatures of q and of the appended key, scores, top-k,
            gather-attention) on contiguous caches
  paged     `ha_sparse_decode_paged_codes`, the same step with K, V and signatures in pages behind one block table
  host      `SparseDecodeHostStep`, the same step from pinned host buffers, its result back on the host
  prefill   `ha_encode_prefill`, the signature cache of a prompt
  per_head  `ha_encode` (queries; appended keys), `ha_score_topk_per_head`, `ha_gather_attn_per_head`: one list per query head
  wide      `ha_encode_wide` (queries; appended keys), `ha_score_topk_wide`, `ha_gather_attn`: signatures of 64 to 512 bits

Inputs come from `workloads.make_workload` (unit normals in bf16, a share of the keys planted along the queries, random
mapping networks); the signature cache is filled by the library's own exact ENCODE, as a program that follows the cache
token by token would have it.  K and V hold the appended row already, except for `host`, which appends it itself.
"""
from __future__ import annotations

import math
import random

import torch

from paper_2412_14468_b200 import binding as ha
from paper_2412_14468_b200 import workloads as wl

MAX_TOKENS = 64 * 32768          # cached tokens of one case over all sequences: 8.6 GB of K and V at 8 KV heads
SIDE_BYTES = 2 * (128 * 128 * 2 + 128 * 32) + 4 * (128 + 128 + 32)   # one KV head's mapping network, 32 bits


def _case(kind, batch, n, n_lo=0, lens_seed=0, sparsity=32, q_heads=32, kv_heads=8, window=0, planted=0.01, lse=False,
          page=0, bits=32):
    """n_lo > 0: ragged lengths in [n_lo, n] from lens_seed; window: tokens always kept at each end of a sequence."""
    return {"kind": kind, "batch": batch, "n": n, "n_lo": n_lo, "lens_seed": lens_seed, "sparsity": sparsity,
            "q_heads": q_heads, "kv_heads": kv_heads, "window": window, "planted": planted, "lse": lse, "page": page,
            "bits": bits}


def listed():
    return [
        # one short conversation: launches and host work are all there is
        dict(_case("step", 1, 4096, sparsity=16, planted=0.0), name="step_b1_4k"),
        # the headline: one sequence at 32K, 32x
        dict(_case("step", 1, 32768), name="step_b1_32k"),
        # a handful of sequences of odd lengths with the first and last 128 tokens always kept, as in the paper's
        # experiments, and the log-sum-exp asked for
        dict(_case("step", 5, 23457, n_lo=1001, lens_seed=3, window=128, lse=True), name="step_b5_ragged_windows"),
        # batched decode at 16x
        dict(_case("step", 16, 32768, sparsity=16), name="step_b16_32k"),
        # a full serving batch at 32K, 32x
        dict(_case("step", 64, 32768), name="step_b64_32k"),
        # one very long document
        dict(_case("step", 1, 524288, planted=0.001), name="step_b1_512k"),
        # a serving batch of very different lengths
        dict(_case("step", 32, 131072, n_lo=8192, lens_seed=5), name="step_b32_ragged_128k"),
        # a paged server in mid-flight: pages of 16 tokens, lengths of every kind
        dict(_case("paged", 24, 65536, n_lo=2000, lens_seed=7, page=16), name="paged_b24_ragged_64k"),
        # a decoder that keeps its activations on the host
        dict(_case("host", 1, 32768), name="host_b1_32k"),
        # the signature cache of a 32K prompt
        dict(_case("prefill", 1, 32768, planted=0.0), name="prefill_32k"),
        # the paper's own selection, one list per query head
        dict(_case("per_head", 2, 32768), name="per_head_b2_32k"),
        # more bits per signature
        dict(_case("wide", 4, 32768, bits=128), name="wide128_b4_32k"),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng: random.Random):
    kind = rng.choice(["step"] * 6 + ["paged"] * 2 + ["host", "prefill", "per_head", "wide"])
    tokens = {"step": MAX_TOKENS, "paged": MAX_TOKENS // 2, "host": 8 * 32768, "prefill": 4 * 32768,
              "per_head": 8 * 32768, "wide": 8 * 32768}[kind]
    n_hi = {"step": 524288, "paged": 131072, "host": 131072, "prefill": 131072, "per_head": 65536, "wide": 65536}[kind]
    sparsity = rng.choice([8, 16, 32, 32, 32]) if kind not in ("prefill", "per_head") else 32
    heads = rng.choice([4, 4, 4, 2, 8]) if kind in ("step", "paged") else 4      # query heads of a KV head
    tokens = tokens * sparsity * 4 // (32 * max(4, heads))   # no dearer than the dearest listed case
    n = _log_int(rng, 1000, min(n_hi, tokens))
    batch = _log_int(rng, 1, max(1, min(64 if kind in ("step", "paged") else 8, tokens // n)))
    ragged = batch > 1 and kind != "prefill" and rng.random() < 0.5
    return _case(kind, batch, n, n_lo=max(1, n // rng.choice([2, 8, 16])) if ragged else 0, lens_seed=rng.randrange(1 << 20),
                 sparsity=sparsity, q_heads=8 * heads, window=rng.choice([0, 0, 128]) if kind in ("step", "paged") else 0,
                 planted=0.0 if kind == "prefill" else rng.choice([0.001, 0.01]),
                 lse=kind in ("step", "paged") and rng.random() < 0.25, page=rng.choice([16, 16, 64]) if kind == "paged" else 0,
                 bits=rng.choice([64, 128, 256, 512]) if kind == "wide" else 32)


def _lens(case):
    if not case["n_lo"]:
        return [case["n"]] * case["batch"]
    r = random.Random(case["lens_seed"])
    return [r.randint(case["n_lo"], case["n"]) for _ in range(case["batch"])]


def _budgets(case):
    return [max(1, n // case["sparsity"]) for n in _lens(case)]


class _State:
    pass


def _in_pages(t, page, order):
    """[B, H, n, ...] with n a multiple of `page` -> pool [n_pages, H, page, ...] in which page p of the batch lies at
    order[p]."""
    B, H, n = t.shape[:3]
    pages = t.view(B, H, n // page, page, *t.shape[3:]).transpose(1, 2)
    pool = torch.empty((B * (n // page), H, page) + tuple(t.shape[3:]), dtype=t.dtype, device=t.device)
    where = order.view(B, n // page)
    for b in range(B):
        pool[where[b]] = pages[b]
    return pool


def prepare(case, seed):
    dev = torch.device("cuda", torch.cuda.current_device())
    s = _State()
    s.kind, s.bits, s.page = case["kind"], case["bits"], case["page"]
    B, Hq, Hkv = case["batch"], case["q_heads"], case["kv_heads"]
    G = Hq // Hkv
    base = wl.BASE_SEED + 7919 * int(seed)

    if s.kind == "prefill":
        g = torch.Generator(dev).manual_seed(base)
        s.x = torch.randn(B, Hkv, case["n"], 128, device=dev, generator=g, dtype=torch.float32).to(torch.bfloat16)
        s.map = ha.Mapping(wl.make_mapping(Hkv, g, dev))
        s.codes = torch.zeros(B, Hkv, case["n"], dtype=torch.int32, device=dev)
        s.ws = ha.alloc_workspace(ha.make_shape(B, Hq, Hkv, 1.0), case["n"], 1, device=dev)
        return s

    lens, ks = _lens(case), _budgets(case)
    page = s.page or 1
    s.n_max, s.k_max = max(lens), max(ks) + 2 * case["window"]
    room = -(-s.n_max // 64) * 64     # whole pages; rows of the signature cache stay 16-byte aligned
    cfg = wl.Config("case", 0, B, tuple(lens), None, case["planted"], Hq, Hkv, case["sparsity"])
    w = wl.make_workload(cfg, device=dev, seed=base)
    s.q, s.k_new, s.v_new = w["q"], w["k_new"], w["v_new"]
    s.K, s.V = w["K"], w["V"]
    s.seq_lens = w["seq_lens"]
    s.ragged = len(set(lens)) > 1
    s.k_per_seq = torch.tensor(ks, dtype=torch.int32, device=dev) if s.ragged else None
    s.k_uniform = 0 if s.ragged else ks[0]
    s.shape = ha.make_shape(B, Hq, Hkv, w["sm_scale"], n_sink=case["window"], n_local=case["window"])
    units = Hq if s.kind == "per_head" else Hkv
    s.idx = torch.zeros(B, units, s.k_max, dtype=torch.int32, device=dev)
    s.count = torch.zeros(B, units, dtype=torch.int32, device=dev)
    s.out = torch.zeros(B, Hq, 128, dtype=torch.bfloat16, device=dev)
    s.lse = torch.zeros(B, Hq, dtype=torch.float32, device=dev) if case["lse"] else None

    if s.kind == "wide":
        W = s.bits // 64
        g = torch.Generator(dev).manual_seed(base + 3001)
        maps = []
        for _ in range(2):
            m = wl.make_mapping(Hkv, g, dev)
            bound = 1.0 / math.sqrt(128)
            m["w3"] = ((torch.rand(Hkv, 128, s.bits, device=dev, generator=g) * 2 - 1) * bound).to(torch.bfloat16)
            m["b3"] = (torch.rand(Hkv, s.bits, device=dev, generator=g) * 2 - 1) * bound
            maps.append(ha.MappingWide(m))
        s.map_q, s.map_k = maps
        s.G, s.slot = G, s.seq_lens - 1
        s.q_codes = torch.zeros(B, Hq, 1, W, dtype=torch.int64, device=dev)
        s.codes = torch.zeros(B, Hkv, room, W, dtype=torch.int64, device=dev)
        ha.ha_encode_wide(s.map_k, 1, s.K, s.codes)
        s.ws_score = ha.alloc_workspace_wide(s.shape, s.n_max, device=dev)
        s.ws = ha.alloc_workspace(s.shape, s.n_max, s.k_max, device=dev)
        return s

    s.map_q, s.map_k = ha.Mapping(w["map_q"]), ha.Mapping(w["map_k"])
    s.codes = torch.zeros(B, Hkv, room, dtype=torch.int32, device=dev)
    ha.ha_encode(s.map_k, 1, s.K, s.codes)
    s.q_codes = torch.zeros(B, Hq, dtype=torch.int32, device=dev)

    if s.kind == "per_head":
        s.G, s.slot = G, s.seq_lens - 1
        s.q_codes = s.q_codes.unsqueeze(2)
        s.ws = ha.alloc_workspace(ha.make_shape(B, Hq, Hq, w["sm_scale"]), s.n_max, s.k_max, device=dev)
        return s

    s.ws = ha.alloc_workspace(s.shape, s.n_max, s.k_max, device=dev)
    if s.kind == "paged":
        g = torch.Generator(dev).manual_seed(base + 6001)
        pages = room // page
        order = torch.randperm(B * pages, device=dev, generator=g)
        short = room - s.K.shape[2]
        for name in ("K", "V"):
            t = getattr(s, name)
            t = torch.nn.functional.pad(t, (0, 0, 0, short)) if short else t
            setattr(s, name, _in_pages(t, page, order))
            del t
        s.codes = _in_pages(s.codes, page, order)
        s.table = order.view(B, pages).to(torch.int32)
    if s.kind == "host":
        pin = lambda t: t.cpu().pin_memory()  # noqa: E731
        s.host = [pin(s.q), pin(s.k_new), pin(s.v_new)]
        s.out_host = torch.zeros(B, Hq, 128, dtype=torch.bfloat16).pin_memory()
        last = [n - 1 for n in lens]
        for b, t in enumerate(last):
            s.K[b, :, t] = 0
            s.V[b, :, t] = 0
        s.step = ha.SparseDecodeHostStep(s.shape, s.map_q, s.map_k, *s.host, s.K, s.V, s.codes, s.seq_lens, s.k_per_seq,
                                         s.k_uniform, s.n_max, s.k_max, s.idx, s.count, s.out_host, s.ws)
    return s


def run(s):
    if s.kind == "step":
        ha.ha_sparse_decode(s.shape, s.map_q, s.map_k, s.q, s.k_new, s.K, s.V, s.codes, s.seq_lens, s.k_per_seq, s.k_uniform,
                            s.n_max, s.k_max, s.q_codes, s.idx, s.count, s.out, s.ws, lse=s.lse)
    elif s.kind == "paged":
        ha.ha_sparse_decode_paged_codes(s.shape, s.map_q, s.map_k, s.q, s.k_new, s.K, s.V, s.codes, s.table, s.seq_lens,
                                        s.k_per_seq, s.k_uniform, s.n_max, s.k_max, s.q_codes, s.idx, s.count, s.out, s.ws,
                                        lse=s.lse)
    elif s.kind == "host":
        s.step()
        return {"out": s.out_host, "idx": s.idx, "count": s.count, "codes": s.codes, "K": s.K, "V": s.V}
    elif s.kind == "prefill":
        ha.ha_encode_prefill(s.map, 1, s.x, s.codes, workspace=s.ws)
        return s.codes
    elif s.kind == "per_head":
        ha.ha_encode(s.map_k, 1, s.k_new, s.codes, slot=s.slot)
        ha.ha_encode(s.map_q, s.G, s.q, s.q_codes)
        ha.ha_score_topk_per_head(s.shape, s.q_codes, s.codes, s.seq_lens, s.k_per_seq, s.k_uniform, s.k_max, s.idx, s.count)
        ha.ha_gather_attn_per_head(s.shape, s.q, s.K, s.V, s.seq_lens, s.idx, s.count, s.k_max, s.out, s.ws)
    elif s.kind == "wide":
        ha.ha_encode_wide(s.map_k, 1, s.k_new, s.codes, slot=s.slot)
        ha.ha_encode_wide(s.map_q, s.G, s.q, s.q_codes)
        ha.ha_score_topk_wide(s.shape, s.bits, s.q_codes, s.codes, s.seq_lens, s.k_per_seq, s.k_uniform, s.n_max, s.k_max,
                              s.idx, s.count, s.ws_score)
        ha.ha_gather_attn(s.shape, s.q, s.K, s.V, s.seq_lens, s.idx, s.count, s.k_max, s.out, s.ws)
    return {"out": s.out, "lse": s.lse, "idx": s.idx, "count": s.count, "q_codes": s.q_codes, "codes": s.codes}


def work(case):
    """Bytes: signatures scanned, selected K and V rows, mapping networks, q, k_new, index lists and out.  Operations: the
    mapping networks and the attention over the selected rows (the bit counts are not floating-point operations)."""
    B, Hq, Hkv, bits = case["batch"], case["q_heads"], case["kv_heads"], case["bits"]
    G = Hq // Hkv
    net = 2 * (128 * 128 * 2 + 128 * bits)                      # operations of one vector
    side = SIDE_BYTES + (2 * 128 + 4) * (bits - 32)
    if case["kind"] == "prefill":
        keys = B * Hkv * case["n"]
        return {"bytes": keys * (256 + 4) + Hkv * side, "flops": keys * net}
    lists = G if case["kind"] == "per_head" else 1
    nbytes, flops = 2 * Hkv * side, B * (Hq + Hkv) * net
    for n, k in zip(_lens(case), _budgets(case)):
        k = min(n, k + 2 * case["window"])
        nbytes += Hkv * (bits // 8 * n + 512 * min(n, k * lists) + 4 * k * lists + 256) + Hq * (2 * 256)
        flops += 4 * 128 * k * Hq
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    if case["kind"] == "prefill":
        # tensor-core sums: a bit whose output lies within about 1e-5 of zero may fall either way
        return {"rel": 0.0, "differ": 1e-3}
    # out is bf16 from fp32 sums: one unit in the last place; lists, counts and signatures are whole numbers
    return {"rel": 5e-3, "max": 2e-2}
