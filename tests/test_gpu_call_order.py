"""Library kernels start while the kernel in front of them is finishing.  A call that writes one signature at any slot directly
in front of a call that scans the cache: the scan has to see it.  Key networks equal query networks and the key is the query, so
the written signature scores 32 of 32 (or n_bits of n_bits) and is on the list exactly if the scan has read it; what lies there
before is its complement, which is on no list."""
import numpy as np
import pytest
import torch

import oracle
from paper_2412_14468_b200 import binding as ha
from paper_2412_14468_b200 import workloads as wl
from tests._fake import SEVERAL_UNITS_PER_CLUSTER
from tests._util import u16
from tests.test_gpu_parity import _wide_mapping

pytestmark = pytest.mark.gpu
DEV = "cuda"
K, REPEATS, PAGE = 16, 12, 16


class _Calls:
    """One cache with heads of one query each, and the calls that append to it and scan it."""

    def __init__(self, B, H, n, paged=False, bits=32, budgets=False):
        g = torch.Generator(DEV).manual_seed(B + n)
        rng = np.random.default_rng(n)
        self.B, self.H, self.n, self.W, self.bits, self.paged = B, H, n, bits // 64, bits, paged
        room = -(-n // 64) * 64
        self.q = torch.randn(B, H, 128, device=DEV, generator=g).to(torch.bfloat16)
        self.K = torch.randn(B, H, room, 128, device=DEV, generator=g).to(torch.bfloat16)
        self.lens = torch.full((B,), n, dtype=torch.int32, device=DEV)
        self.budget = (torch.full((B,), K, dtype=torch.int32, device=DEV), 0) if budgets else (None, K)   # one per sequence, or one for all
        self.shape = ha.make_shape(B, H, H, 0.09)
        self.ws, self.ws_wide = ha.alloc_workspace(self.shape, n, K), ha.alloc_workspace_wide(self.shape, n)
        new = lambda *s, t=torch.int32: torch.zeros(*s, dtype=t, device=DEV)  # noqa: E731
        self.idx, self.cnt, self.out = new(B, H, K), new(B, H), new(B, H, 128, t=torch.bfloat16)
        m = _wide_mapping(H, bits, 3) if bits > 32 else wl.make_mapping(H, g, torch.device(DEV))
        mn, qu = wl.mapping_numpy(m), u16(self.q)
        self.map = ha.MappingWide(m) if bits > 32 else ha.Mapping(m)
        enc = oracle.encode_wide if bits > 32 else oracle.encode
        self.code = np.stack([enc(qu[:, h], mn["w1"][h], mn["w2"][h], mn["w3"][h], mn["b1"][h], mn["b2"][h], mn["b3"][h])
                              for h in range(H)], 1)                               # [B, H] or [B, H, W]
        words = (self.W,) if bits > 32 else ()
        self.base = rng.integers(0, 2**(64 if bits > 32 else 32), size=(B, H, room) + words, dtype=np.uint64).astype(self.code.dtype)
        view = lambda a: torch.from_numpy(np.ascontiguousarray(a).view(np.int64 if bits > 32 else np.int32)).to(DEV)  # noqa: E731
        self.clean, self.complement = view(self.base), view(~self.code)
        self.q_codes = view(self.code)
        if paged:
            self.table = torch.randperm(B * room // PAGE, device=DEV, generator=g).view(B, -1).to(torch.int32)
            pool = self.clean.new_empty(B * room // PAGE, H, PAGE)
            kv = torch.empty(B * room // PAGE, H, PAGE, 128, dtype=torch.bfloat16, device=DEV)
            for b in range(B):
                pool[self.table[b].long()] = self.clean[b].view(H, -1, PAGE).transpose(0, 1)
                kv[self.table[b].long()] = self.K[b].view(H, -1, PAGE, 128).transpose(0, 1)
            self.clean, self.K = pool, kv
        self.codes = self.clean.clone()
        # the best of the other tokens, best first, of which a slot may be one
        self.best = []
        for b in range(B):
            for h in range(H):
                s = oracle.score_wide(self.code[b, h], self.base[b, h, :n]) if bits > 32 else oracle.score(self.code[b, h:h + 1], self.base[b, h, :n])
                self.best.append(np.argsort(-s.astype(np.int64), kind="stable")[:K + 1])

    def reset(self, slot):
        self.codes.copy_(self.clean)
        ar = torch.arange(self.B, device=DEV)
        if self.paged:
            self.codes[self.table[ar, slot.long() // PAGE].long(), :, slot.long() % PAGE] = self.complement
        else:
            self.codes[ar, :, slot.long()] = self.complement

    def append(self, how, slot):
        if how == "encode" and self.bits > 32:
            ha.ha_encode_wide(self.map, 1, self.q.unsqueeze(2), self.codes, slot=slot)
        elif how == "encode" and self.paged:
            ha.ha_encode_append_paged(self.map, self.q, self.codes, self.table, slot + 1)
        elif how == "encode":
            ha.ha_encode(self.map, 1, self.q.unsqueeze(2), self.codes, slot=slot)
        else:
            self.step(slot + 1, self.q)

    def step(self, lens, k_new):
        common = (lens, *self.budget, self.n, K, torch.zeros_like(self.q_codes), self.idx, self.cnt, self.out, self.ws)
        if self.paged:
            ha.ha_sparse_decode_paged_codes(self.shape, self.map, self.map, self.q, k_new, self.K, self.K, self.codes, self.table, *common)
        else:
            ha.ha_sparse_decode(self.shape, self.map, self.map, self.q, k_new, self.K, self.K, self.codes, *common)

    def scan(self, how):
        args = (self.lens, *self.budget)
        if how == "step":
            self.step(self.lens, None)
        elif how == "wide":
            ha.ha_score_topk_wide(self.shape, self.bits, self.q_codes, self.codes, *args, self.n, K, self.idx, self.cnt, self.ws_wide)
        elif how == "topk" and self.paged:
            ha.ha_score_topk_paged(self.shape, self.q_codes, self.codes, self.table, *args, self.n, K, self.idx, self.cnt, self.ws)
        elif how == "topk":
            ha.ha_score_topk(self.shape, self.q_codes, self.codes, *args, self.n, K, self.idx, self.cnt, self.ws)
        else:
            (ha.ha_score_topk_sum if how == "sum" else ha.ha_score_topk_per_head)(self.shape, self.q_codes, self.codes, *args, K, self.idx, self.cnt)

    def check(self, slot):
        got, slots = self.idx.cpu().numpy().reshape(-1, K), slot.cpu().numpy().repeat(self.H)
        for u, best in enumerate(self.best):
            ref = np.sort(np.concatenate([[slots[u]], best[best != slots[u]][:K - 1]]))
            assert np.array_equal(got[u], ref), (u, slots[u])


def _run(c, append, scan):
    for r in range(REPEATS):
        # any slot, then the last three tokens of the sequence
        slot = (torch.arange(c.B, device=DEV) * 331 + 977 * r) % c.n if r < REPEATS - 3 else torch.full((c.B,), c.n - 1 - (REPEATS - 1 - r), device=DEV)
        slot = slot.to(torch.int32)
        c.reset(slot)
        torch.cuda.synchronize()
        c.append(append, slot)
        c.scan(scan)
        c.check(slot)
    assert ha.ha_read_device_status(c.ws) == 0


# few units (one-launch step, large clusters), many units (three launches), a sequence beyond the cluster kernels
@pytest.mark.parametrize("B,n", [(2, 20000), (20, 3001), (1, 262147)])
@pytest.mark.parametrize("scan", ["topk", "sum", "per_head", "step"])
@pytest.mark.parametrize("append", ["encode", "step"])
def test_a_signature_written_directly_in_front_of_a_scan(B, n, scan, append):
    _run(_Calls(B, 4, n), append, scan)


@pytest.mark.parametrize("B,n", [(2, 20000), (20, 3001), (1, 262147)])
@pytest.mark.parametrize("scan", ["topk", "step"])
@pytest.mark.parametrize("append", ["encode", "step"])
def test_a_signature_written_into_a_page_directly_in_front_of_a_scan(B, n, scan, append):
    _run(_Calls(B, 4, n, paged=True), append, scan)


@pytest.mark.parametrize("B,H,n,_cs", SEVERAL_UNITS_PER_CLUSTER)
@pytest.mark.parametrize("paged,scan,append", [(False, "topk", "encode"), (False, "step", "step"), (False, "topk", "step"),
                                               (True, "topk", "encode"), (True, "step", "step")])
def test_a_signature_written_directly_in_front_of_clusters_of_several_units(B, H, n, _cs, paged, scan, append):
    _run(_Calls(B, H, n, paged=paged, budgets=True), append, scan)


@pytest.mark.parametrize("B,n", [(2, 20000), (20, 3001), (1, 140001)])
@pytest.mark.parametrize("bits", [64, 256])
def test_a_wide_signature_written_directly_in_front_of_its_selection(B, n, bits):
    _run(_Calls(B, 4, n, bits=bits), "encode", "wide")


# the kernel in front: lets the kernels behind it start at once and writes its buffer some 20 us later
LATE_COPY = """
extern "C" __global__ void late_copy(const int *src, int *dst, int n) {
    asm volatile("griddepcontrol.launch_dependents;");
    for (int i = 0; i < 20; ++i) __nanosleep(1000);
    for (int i = threadIdx.x; i < n; i += blockDim.x) dst[i] = src[i];
}"""


@pytest.mark.parametrize("B,H,n,budgets", [(2, 4, 20000, False), (20, 4, 3001, False), (1, 4, 100003, False), (1, 4, 262147, False)] +
                         [(B, H, n, True) for B, H, n, _ in SEVERAL_UNITS_PER_CLUSTER])
@pytest.mark.parametrize("scan", ["topk", "step"])
def test_a_block_table_is_read_behind_whatever_writes_it(B, H, n, budgets, scan):
    """The table names other pages of the same pool until the kernel in front has written it."""
    c = _Calls(B, H, n, paged=True, budgets=budgets)
    late_copy = torch.cuda._compile_kernel(LATE_COPY, "late_copy")
    table = c.table
    slot = torch.full((B,), n // 2, dtype=torch.int32, device=DEV)
    c.reset(slot)
    c.append("encode", slot)
    c.table = torch.empty_like(table)
    for _ in range(3):
        c.table.copy_(table.roll(1, 1))
        torch.cuda.synchronize()
        late_copy(grid=(1, 1, 1), block=(1024, 1, 1), args=[table, c.table, table.numel()])
        c.scan(scan)
        c.check(slot)
    assert ha.ha_read_device_status(c.ws) == 0


@pytest.mark.parametrize("n", [20000, 262147])
def test_a_call_of_empty_sequences_between_the_two(n):
    """A grid in which no CTA has work still waits for the kernels in front of it."""
    c = _Calls(2, 4, n)
    empty = torch.zeros_like(c.lens)
    idx, cnt = torch.zeros_like(c.idx), torch.zeros_like(c.cnt)
    for r in range(REPEATS):
        slot = torch.full((2,), 977 * r, dtype=torch.int32, device=DEV)
        c.reset(slot)
        torch.cuda.synchronize()
        c.append("step", slot)
        ha.ha_score_topk(c.shape, c.q_codes, c.codes, empty, None, K, n, K, idx, cnt, c.ws)
        c.scan("topk")
        c.check(slot)
    assert (cnt == 0).all()


@pytest.mark.parametrize("B,n", [(2, 20000), (20, 3001), (1, 262147)])
def test_a_prompt_is_encoded_over_signatures_that_the_call_in_front_still_scans(B, n):
    """ha_encode_prefill starts while the selection in front of it runs, and overwrites the cache that it reads."""
    c = _Calls(B, 4, n)
    for r in range(REPEATS):
        slot = torch.full((B,), 977 * r % n, dtype=torch.int32, device=DEV)
        c.reset(slot)
        c.append("encode", slot)
        torch.cuda.synchronize()
        c.scan("topk")
        ha.ha_encode_prefill(c.map, 1, c.K, c.codes, workspace=c.ws)
        c.check(slot)
    assert ha.ha_read_device_status(c.ws) == 0


@pytest.mark.parametrize("B,n", [(2, 20000), (1, 130), (3, 8192)])
def test_a_prompt_is_encoded_behind_whatever_writes_its_tokens(B, n):
    """The tokens are other ones until the kernel in front, which lets its dependents start at once, has written them."""
    c = _Calls(B, 4, n)
    late_copy = torch.cuda._compile_kernel(LATE_COPY, "late_copy")
    want, x = torch.zeros_like(c.codes), torch.empty_like(c.K)
    ha.ha_encode_prefill(c.map, 1, c.K, want, workspace=c.ws)
    words, to = c.K.view(torch.int32), x.view(torch.int32)
    for _ in range(3):
        x.copy_(c.K.roll(1, 2))
        c.codes.zero_()
        torch.cuda.synchronize()
        late_copy(grid=(1, 1, 1), block=(1024, 1, 1), args=[words, to, words.numel()])
        ha.ha_encode_prefill(c.map, 1, x, c.codes, workspace=c.ws)
        assert torch.equal(c.codes, want)
    assert ha.ha_read_device_status(c.ws) == 0
