"""The library linked against a CUDA runtime that launches nothing (fake_cudart.cpp), and its entry points with made-up device
addresses: what the host side decides for a call, without a GPU."""
import ctypes as C
import glob
import os
import re
import subprocess

from paper_2412_14468_b200 import binding as ha
from paper_2412_14468_b200 import build as ha_build

CUDA = os.environ.get("CUDA_HOME", "/usr/local/cuda")
SRC = os.path.join(os.path.dirname(os.path.abspath(__file__)), "fake_cudart.cpp")
RESIDENT = {1: 296, 2: 148, 4: 71, 8: 33}          # clusters of 512-thread CTAs, two per SM, at once on 148 SMs in two dies
PTR = 1 << 20                                       # an address that nothing looks behind
BATCH = "score_select_batch_kernel"

# (sequences, KV heads of one query head, tokens, CTAs per cluster): with one budget per sequence these take clusters of several units
SEVERAL_UNITS_PER_CLUSTER = [(120, 4, 3001, 1), (62, 4, 33000, 2), (12, 4, 140001, 4), (6, 4, 270001, 8)]


def ragged(n_seqs, longest):
    """Unequal lengths with the edges of a row of 128 tokens and of a group of 32 among them, not in order."""
    edges = [0, 1, 31, 32, 33, 127, 128, 129, 255, 257]
    step = max(1, longest // n_seqs)
    lens = [max(1, longest - 3 - i * step) for i in range(n_seqs - len(edges) - 1)]
    return edges[::2] + lens[::2] + [longest] + edges[1::2] + lens[1::2]


# Calls of SCORE + TOPK with one budget per sequence that take clusters of several units:
# (group size, KV heads, lengths, page sizes, CTAs per cluster, batches of the busiest cluster, block table staged)
BATCH_CASES = [
    (4, 8, ragged(58, 5120), (0, 16, 128, 4096), 1, 1, True),        # the fewest units of one CTA, the longest for their share
    (4, 8, ragged(64, 10240), (0, 16), 1, 1, True),                  # the longest, CTAs filled evenly
    (8, 8, ragged(64, 5120), (0, 16), 1, 1, True),
    (1, 2, ragged(240, 900), (0, 16, 128, 4096), 1, 1, True),        # lengths sorted by the whole CTA
    (1, 8, ragged(65, 300), (0, 16, 128), 1, 1, True),               # one sequence more than one warp sorts
    (1, 1, ragged(512, 300), (0, 16, 128), 1, 1, True),              # as many as are sorted
    (1, 1, [0] * 511 + [1], (0, 16, 128), 1, 1, True),               # ... and hardly any step between their lengths
    (2, 1, ragged(700, 700), (0, 16, 128, 4096), 1, 1, True),        # more than are sorted
    (1, 8, ragged(300, 300), (0, 16, 4096), 1, 2, True),             # nine units a cluster: eight at a time, two warps each
    (8, 8, ragged(32, 32769), (0, 16, 128, 4096), 2, 1, True),       # beyond the clusters of 2 of one unit
    (4, 8, ragged(23, 40000), (16, 4096), 2, 1, True),               # fewer units in pages
    (4, 8, ragged(24, 65537), (0, 16), 2, 1, True),                  # ... and contiguous from here on
    (1, 4, ragged(31, 65537), (16,), 2, 1, True),                    # 124 units in pages: one a cluster
    (2, 8, [100000] * 38 + [1, 131072], (0, 16), 2, 3, True),         # more than two long units a cluster: one at a time
    (2, 4, ragged(17, 98305), (0, 16, 4096), 4, 1, True),
    (4, 4, ragged(12, 131073), (0, 16, 128, 4096), 4, 1, True),      # beyond the one-unit clusters
    (2, 8, [150000] * 23 + [140], (0, 16), 2, 2, True),              # two units a cluster that do not fit together
    (1, 8, [170000] * 12 + [33], (16, 64), 2, 1, None),              # staged in pages of 64, no room for the entries of pages of 16
    (1, 8, [190000] * 13, (0, 16), 4, 2, True),                      # two units a cluster of 4 that do not fit together
    (1, 8, [300000] * 9, (0,), 8, 2, True),                          # three units a cluster of 8: two and one
    (1, 8, [300000] * 9, (16,), 8, 3, True),                         # ... with the entries of pages of 16 one at a time
    (1, 2, ragged(12, 262145), (0, 16, 128, 4096), 8, 1, True),      # beyond the large CTAs
    (1, 2, ragged(12, 393000), (0, 16, 128, 4096), 8, 1, True),
    (1, 4, [330000] * 11 + [330001], (16,), 4, 1, False),            # no room for the entries
]
# ... and calls beside the lines of the rule, which the other kernels take
NEXT_TO_BATCH_CASES = [
    (4, 4, ragged(58, 8193), (0, 16, 128)),          # 232 units
    (4, 8, ragged(57, 5120), (0, 16)),               # 456 units
    (4, 8, ragged(58, 5121), (0,)),                  # CTAs filled unevenly
    (8, 8, ragged(64, 5121), (0,)),
    (4, 8, ragged(64, 10241), (0, 16)),
    (8, 8, ragged(24, 16385), (0, 16, 128)),
    (4, 8, ragged(48, 8193), (0, 16, 128)),
    (4, 8, ragged(32, 32768), (0, 16)),
    (4, 8, ragged(24, 65536), (0,)),
    (4, 8, ragged(22, 65536), (16,)),
    (4, 8, ragged(13, 49153), (0, 16, 128)),
    (2, 2, ragged(20, 98305), (0, 16, 128)),         # 40 units
    (2, 4, ragged(15, 131072), (0, 16)),             # 60 units
    (4, 4, ragged(17, 98304), (0,)),
    (1, 3, ragged(12, 262145), (0, 16)),             # 36 units beyond 131072 tokens: two rounds of few clusters
    (8, 4, [140000] * 9 + [1], (0,)),                # 40 units in groups of 8
    (1, 8, [200, 4095, 4096, 4097, 0] * 5 + [8193, 200000], (0, 16)),   # 216 short units in a capacity that takes clusters of 4
]

# lists per query head over pages: (sequences, KV heads, group size, longest, CTAs per cluster)
PER_HEAD_BATCH_CASES = [(58, 2, 4, 900, 1), (15, 8, 4, 12000, 1), (37, 8, 2, 32768, 1), (23, 2, 4, 40000, 2), (13, 4, 2, 140000, 2)]


def budgets(lens):
    """A budget per sequence: among short ones nothing and everything."""
    return [(0, n, max(1, n // 11), max(1, n // 40))[i % 4] if n < 600 else n // 40 for i, n in enumerate(lens)]


def batches(Hkv, lens, cs, clusters, page=0, staged=False, most=8, pool=96 * 1024):
    """Batches of the busiest cluster: units by falling length, dealt out forth and back, as many at a time as fit the pool."""
    order = sorted(range(len(lens)), key=lambda b: -lens[b]) if len(lens) <= 512 else range(len(lens))
    need = []
    for b in order:
        rows = -(-(-(-lens[b] // 128)) // cs)
        need += [33 * 128 + rows * 128 + ((rows * 128 // page + 5) // 4 * 16 if staged else 0)] * Hkv
    worst = 0
    for c in range(clusters):
        mine = [u for j in range(0, len(need), clusters) for u in [j + (clusters - 1 - c if j // clusters & 1 else c)] if u < len(need)]
        n, used, held = 0, 0, 0
        for u in mine:
            if n == 0 or held == most or used + need[u] > pool:
                n, used, held = n + 1, 0, 0
            used, held = used + need[u], held + 1
        worst = max(worst, n)
    return worst


class Fake:
    def __init__(self, directory, name="fake"):
        ha_build.build()
        path = os.path.join(str(directory), f"lib{name}.so")
        subprocess.run(["g++", "-std=c++17", "-O1", "-fPIC", "-shared", "-I", os.path.join(CUDA, "include"), SRC,
                        *sorted(glob.glob(os.path.join(ha_build.OBJ, "*.o"))), "-o", path, "-Wl,-Bsymbolic"], check=True)
        self.lib, real = C.CDLL(path), ha.lib()
        for fn in ha.EXPORTS:
            getattr(self.lib, fn).argtypes, getattr(self.lib, fn).restype = getattr(real, fn).argtypes, getattr(real, fn).restype
        self.lib.fake_launch.restype = C.c_char_p
        self.lib.fake_answers(*(RESIDENT[c] for c in (1, 2, 4, 8)))
        self.lib.fake_clear()

    def launches(self):
        """[(kernel, its template arguments, CTAs, CTAs per cluster, dynamic shared memory, last argument)] since the last look."""
        out, v = [], [C.c_int() for _ in range(4)]
        for i in range(self.lib.fake_launches()):
            name = self.lib.fake_launch(i, *(C.byref(x) for x in v)).decode()
            m = re.match(r"_ZN2ha\d+(\w+?_kernel)(I[\w]*?EE)?", name)
            args = [int(a) for a in re.findall(r"L[ib](\d+)E", m.group(2) or "")]
            out.append((m.group(1), args, v[0].value, v[1].value, v[2].value, v[3].value))
        self.lib.fake_clear()
        return out

    def score_topk(self, B, G, Hkv, max_len, array=True, page=0, per_head=False, k_max=64):
        """Status of SCORE + TOPK over `B` sequences of at most `max_len` tokens; array: one budget per sequence."""
        L, shape = self.lib, ha.make_shape(B, G * Hkv, Hkv, 1.0)
        units = ha.make_shape(B, G * Hkv, G * Hkv if per_head else Hkv, 1.0)
        ws = L.ha_workspace_bytes(C.byref(units), max_len, k_max)
        room = -(-max_len // 64) * 64
        tail = (PTR, PTR if array else None, 0 if array else 7, max_len, k_max, PTR, units.n_kv_heads * k_max, k_max, PTR, None, PTR, ws, None)
        if not page:
            return L.ha_score_topk(C.byref(shape), PTR, PTR, Hkv * room, room, *tail)
        fn = L.ha_score_topk_per_head_paged if per_head else L.ha_score_topk_paged
        return fn(C.byref(shape), PTR, PTR, Hkv * page, page, PTR, -(-max_len // page), page, *tail)

    def step(self, B, G, Hkv, max_len, k_max):
        """Status of the whole layer-step on contiguous caches."""
        L, shape = self.lib, ha.make_shape(B, G * Hkv, Hkv, 1.0)
        m = ha.ha_mapping(Hkv, 128, 128, 32, *([PTR] * 6))
        kv = ha.ha_tensor(PTR, Hkv * max_len * 128, max_len * 128, 128)
        ws, row = L.ha_workspace_bytes(C.byref(shape), max_len, k_max), -(-max_len // 4) * 4
        return L.ha_sparse_decode(C.byref(shape), C.byref(m), C.byref(m), PTR, PTR, C.byref(kv), C.byref(kv), PTR, Hkv * row, row, PTR,
                                  None, k_max, max_len, k_max, PTR, PTR, Hkv * k_max, k_max, PTR, PTR, None, PTR, ws, None)
