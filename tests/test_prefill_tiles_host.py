"""The rule that picks a prefill GEMM's tile (pick_tile, csrc/prefill_gemm.cuh) on devices and
SM shares without resident pairs or clusters of four: a host program built with nvcc, no GPU."""
import os
import subprocess

from paper_2608_24204_gb300 import build


def test_tiles_without_resident_clusters(tmp_path):
    lib = build.build()
    src, exe = tmp_path / "t.cu", tmp_path / "t"
    src.write_text(r"""
#include "prefill_gemm.cuh"
#include <cstdio>
using namespace wici;
int main() {
    const int counts[][3] = {{152, 76, 36}, {38, 19, 9}, {3, 1, 0}, {1, 0, 0}, {152, 0, 0}};
    for (auto &n : counts)
        for (int T : {1, 32, 64, 65, 128, 129, 300, 2048, 9000})
            for (int N : {256, 2000, 6144, 28672})
                for (int K : {64, 264, 4096, 16384})
                    for (int at : {2, 3})
                        for (int wu : {1, at}) {
                            PrefillMaps mp;
                            mp.sms = n[0];
                            mp.pairs = n[1];
                            mp.quads = n[2];
                            const TileChoice c = pick_tile(T, N, K, at, wu, mp);
                            const int tiles = (T + 127) / 128 * ((N + c.bn - 1) / c.bn);
                            bool ok = c.pair ? c.bn == 192 || c.bn == 224 || c.bn == 256
                                             : c.bn == 128 || c.bn == 192 || (c.bn == 224 && at == 2 && c.split == 1);
                            ok = ok && (c.split == 1 || c.split == 2 || c.split == 4);
                            ok = ok && !(c.pair && (mp.pairs < 1 || c.split != 1 || c.stack));
                            // split tiles run as one wave
                            if (c.split > 1) ok = ok && c.split * tiles <= (c.split == 2 ? 2 * mp.pairs : 4 * mp.quads);
                            if (c.stack) ok = ok && T <= 64 && at == 2 && c.split * tiles <= mp.sms &&
                                              (c.bn == 128 || c.split == 1);
                            if (!ok) {
                                std::printf("sms %d T %d N %d K %d at %d wu %d: bn %d split %d pair %d stack %d\n",
                                            n[0], T, N, K, at, wu, c.bn, c.split, c.pair, c.stack);
                                return 1;
                            }
                        }
    return 0;
}
""")
    libdir = os.path.dirname(lib)
    subprocess.run([build._nvcc(), "-std=c++17", *build.ARCH, "--expt-relaxed-constexpr", "-I", build.CSRC, str(src),
                    "-L" + libdir, "-l:libwici.so", "-Xlinker", "-rpath", "-Xlinker", libdir, "-Xlinker",
                    "--allow-shlib-undefined", "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout + r.stderr
