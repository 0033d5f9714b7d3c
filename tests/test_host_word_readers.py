"""Which workers look at the host's abort word: enough of them in every grid, and few in a large one."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_readers_for_every_grid_size(tmp_path):
    src = tmp_path / "readers.cpp"
    src.write_text("""
#include <algorithm>
#include <cstdio>
#include "gtap_internal.h"
int main() {
    for (unsigned n = 1; n <= 8192; ++n) {
        unsigned readers = 0;
        for (unsigned w = 0; w < n; ++w) readers += gtap::reads_host_word(w, n) ? 1 : 0;
        if (readers < std::min(n, 64u) || readers > 128) { std::printf("%u workers: %u readers\\n", n, readers); return 1; }
    }
    return 0;
}
""")
    exe = tmp_path / "readers"
    subprocess.run(["g++", "-std=c++17", "-I" + os.path.join(ROOT, "paper_2604_05982_gb300", "csrc"),
                    str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
