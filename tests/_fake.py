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
        """[(kernel with its template arguments, CTAs, CTAs per cluster, last argument)] since the last look."""
        out, v = [], [C.c_int() for _ in range(4)]
        for i in range(self.lib.fake_launches()):
            name = self.lib.fake_launch(i, *(C.byref(x) for x in v)).decode()
            m = re.match(r"_ZN2ha\d+(\w+?_kernel)(I[\w]*?EE)?", name)
            args = [int(a) for a in re.findall(r"L[ib](\d+)E", m.group(2) or "")]
            out.append((m.group(1), args, v[0].value, v[2].value, v[3].value))
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
