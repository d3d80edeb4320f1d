"""The rules by which the kernels choose the way of a step's attention (csrc/att_plan.h), compiled for the host."""
import ctypes as C
import functools
import os
import subprocess
import tempfile

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2604_07609_b200", "csrc")

WRAPPER = r"""
#include "att_plan.h"
extern "C" int pair_rows() { return blink::ATT_PAIR_ROWS; }
extern "C" int on_pairs(int keys) { return blink::att_on_pairs(keys); }
extern "C" int one_round(int p, int s, int n, int longest) { return blink::att_one_round_on_ctas(p, s, n, longest); }
extern "C" void decode_way(long long TT, int units, int maxkb, int cta_C, int cta_items, int n_ctas, int prompt_rows, long long* out) {
  const blink::AttDecodeWay w = blink::att_decode_way({TT, units, maxkb, cta_C, cta_items, n_ctas, 8, prompt_rows != 0, 1ll << 40});
  out[0] = w.S; out[1] = w.C; out[2] = w.half;
}
"""


@functools.lru_cache(None)
def lib():
    with tempfile.TemporaryDirectory() as d:
        src, so = os.path.join(d, "plan.cpp"), os.path.join(d, "plan.so")
        with open(src, "w") as f:
            f.write(WRAPPER)
        subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", CSRC, src, "-o", so], check=True)
        return C.CDLL(so)


def prompts_on_pairs(requests, n_kv_heads, n_ctas, n_rep=4):
    """requests: (first position, rows) of the requests of several rows in a step.  The number of them that go to CTA pairs."""
    L, pairs, ctas, longest, n = lib(), 0, 0, 0, 0
    for start, rows in requests:
        ctas += -(-rows * n_rep // 128)
        if L.on_pairs(start + rows):
            n += 1
            pairs += -(-rows // L.pair_rows())
            longest = max(longest, start + rows)
    return 0 if L.one_round(pairs * n_kv_heads, ctas * n_kv_heads, n_ctas, longest) else n


def decode_way(keys, n_kv_heads, n_ctas):
    """'half', 'cta', 'units' or 'stream' for a step of single rows that see `keys` keys each."""
    kb = [-(-k // 16) for k in keys]
    U = len(kb) * n_kv_heads
    cta_C = items = 0
    if U <= 2 * n_ctas:   # the smallest of 32 part sizes whose parts fit the CTAs at once, else whole units
        share = max(24, -(-sum(kb) * n_kv_heads // n_ctas))
        cta_C, items = max(kb), U
        for i in range(32):
            c = share + i * -(-share // 8)
            parts = sum(-(-k // c) for k in kb) * n_kv_heads
            if parts <= n_ctas:
                cta_C, items = c, parts
                break
    out = (C.c_longlong * 3)()
    lib().decode_way(C.c_longlong(sum(kb) * n_kv_heads), U, max(kb), cta_C, items, n_ctas, 0, out)
    return ("half" if out[2] else "cta") if out[1] else "stream" if out[0] else "units"
