"""The buffer plan on devices that are not here: a host program calls the library's
make_plan (csrc/plan.h) with other SM counts.  No GPU."""
import os
import shutil
import subprocess

import pytest

from paper_2608_24204_gb300 import build

CSRC = build.CSRC


def test_the_decode_grid_and_its_row_shares_fit_every_device(tmp_path):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("needs g++")
    lib = build.build()
    src, exe = tmp_path / "t.cc", tmp_path / "t"
    src.write_text(r"""
#include "plan.h"
#include <cstdio>
#include <cstring>
using namespace wici;
int main() {
    wici_config c;
    std::memset(&c, 0, sizeof c);
    c.n_layers = 2; c.hidden = 3072; c.n_q_heads = 24; c.n_kv_heads = 8; c.head_dim = 128; c.ffn_dim = 8192;
    c.vocab = 1024; c.max_tokens = 64; c.max_chunk = 64; c.page_tokens = 16; c.rms_eps = 1e-5f; c.rope_theta = 1e4;
    const int sms[] = {0, 1, 132, 152, 256, 257, 400};
    for (int n : sms)
        for (int share : {0, 38, 300}) {
            c.max_sms = share;
            Plan p;
            if (make_plan(&c, n, &p)) return 1;
            // one row share per thread of the eight consumer warps, and a table entry for each
            int want = n < 1 ? 1 : n < 256 ? n : 256;
            if (share && share < want) want = share;
            const bool room = p.ws_mega_time - p.ws_mega_bound >= (size_t)(p.num_sms + 1) * 4;
            if (p.num_sms != want || !room) {
                std::printf("%d SMs, share %d: %d CTAs, wanted %d\n", n, share, p.num_sms, want);
                return 1;
            }
        }
    return 0;
}
""")
    libdir = os.path.dirname(lib)
    subprocess.run([cxx, "-std=c++17", "-I", CSRC, str(src), "-L" + libdir, "-l:libwici.so", "-Wl,-rpath," + libdir,
                    "-Wl,--allow-shlib-undefined", "-o", str(exe)], check=True)
    env = dict(os.environ)
    env["LD_LIBRARY_PATH"] = "/usr/local/cuda/lib64:" + env.get("LD_LIBRARY_PATH", "")
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120, env=env)
    assert r.returncode == 0, r.stdout + r.stderr
