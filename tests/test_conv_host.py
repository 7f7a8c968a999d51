"""The convolution layer's host-side bookkeeping (csrc/conv_plan.h, csrc/device_table.h), compiled
by itself with the host compiler: no GPU and no CUDA."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2608_24204_gb300", "csrc")


def run_host(tmp_path, body):
    """Compiles and runs a main() with `body`; it returns 0 when every check holds."""
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("needs g++")
    src, exe = tmp_path / "t.cc", tmp_path / "t"
    src.write_text('#include "conv_plan.h"\n#include "device_table.h"\n#include <cstdio>\n#include <thread>\n#include <vector>\nusing namespace wici;\n'
                   '#define CHECK(x) do { if (!(x)) { std::printf("failed: %s\\n", #x); return 1; } } while (0)\n'
                   "int main() {\n" + body + "\nreturn 0;\n}\n")
    subprocess.run([cxx, "-std=c++17", "-O1", "-pthread", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, f"exit {r.returncode}: {r.stdout}{r.stderr}"


def test_each_device_keeps_its_own_counts(tmp_path):
    # two threads on two devices with different counts: each call gets its own device's, and a
    # device is asked once; a failed query is returned and asked again
    run_host(tmp_path, r"""
    DeviceTable<ConvDevice> devs;
    int asked[2] = {0, 0};
    auto query = [&](int dev) {
        return [&asked, dev](ConvDevice *d) {
            ++asked[dev];
            d->sms = 100 + dev;
            for (int i = 0; i < 4; ++i) d->clusters[i] = 10 * (dev + 1) + i;
            return 0;
        };
    };
    ConvDevice none;
    CHECK(devs.get(0, &none, [](ConvDevice *d) { d->sms = 7; return 3; }) == 3);
    CHECK(none.sms == 0);
    CHECK(devs.get(1000, &none, [](ConvDevice *d) { d->sms = 9; return 0; }) == 0 && none.sms == 9);
    int wrong[2] = {0, 0};
    std::vector<std::thread> threads;
    for (int dev = 0; dev < 2; ++dev)
        threads.emplace_back([&, dev] {
            for (int i = 0; i < 20000; ++i) {
                ConvDevice d;
                if (devs.get(dev, &d, query(dev)) != 0 || d.sms != 100 + dev || d.clusters[3] != 10 * (dev + 1) + 3)
                    ++wrong[dev];
            }
        });
    for (auto &t : threads) t.join();
    CHECK(wrong[0] == 0 && wrong[1] == 0);
    CHECK(asked[0] == 1 && asked[1] == 1);
    // counts of zero are an answer like any other
    int n = 0;
    for (int i = 0; i < 2; ++i) CHECK(devs.get(2, &none, [&](ConvDevice *) { ++n; return 0; }) == 0 && none.sms == 0);
    CHECK(n == 1);
    """)


def test_ctas_per_tile_on_devices_without_some_cluster_sizes(tmp_path):
    # no resident pair (a small or partitioned device): one CTA per tile is always there; where
    # pairs and clusters exist, large layers take pairs and small ones clusters
    run_host(tmp_path, r"""
    ConvDevice none, solo, all;
    none.sms = solo.sms = all.sms = 152;
    solo.clusters[0] = 1;
    const int n[4] = {152, 76, 36, 16};
    for (int i = 0; i < 4; ++i) all.clusters[i] = n[i];
    for (int tiles : {1, 2, 3, 9, 64, 1000, 50000})
        for (int nkb : {1, 4, 36, 144, 800}) {
            CHECK(pick_ctas(none, tiles, (tiles + 1) / 2, nkb) == 1);
            CHECK(pick_ctas(solo, tiles, (tiles + 1) / 2, nkb) == 1);
            const int c = pick_ctas(all, tiles, (tiles + 1) / 2, nkb);
            CHECK(c == 0 || c == 1 || c == 2 || c == 4 || c == 8);
        }
    CHECK(pick_ctas(all, 1568, 784, 144) == 0);
    CHECK(pick_ctas(all, 2, 1, 144) == 8);
    """)
