"""Sizes of the step's scratch that other passes reuse (no GPU needed): the
photon stage keeps a record of every pair in the emission records (two words
each) and in the staging records (eight Reals each), and all photons of a full
species may convert in one step, so both hold max_particles pairs -- for every
max_particles, the edges of the two minimum sizes (16384 pairs, 131072 pairs)
among them."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_pair_records_hold_every_photon(tmp_path):
    src = tmp_path / "scratch.cpp"
    src.write_text("""
        #include <cstdio>
        #include "qed_scratch.h"
        using namespace qed;
        static bool ok(int64_t m) {
          return rec_entries(m) * SUB_REC >= 2 * m && stage_records(m) * 16 >= 8 * m;
        }
        int main() {
          for (int64_t m = 1; m <= (1 << 21); ++m)
            if (!ok(m)) { printf("%lld\\n", (long long)m); return 1; }
          for (int k = 20; k <= 30; ++k)
            for (int64_t m = ((int64_t)1 << k) - 5000; m <= ((int64_t)1 << k) + 5; ++m)
              if (!ok(m)) { printf("%lld\\n", (long long)m); return 1; }
          return 0;
        }""")
    exe = tmp_path / "scratch"
    inc = os.path.join(ROOT, "paper_1608_06356_gb300", "csrc")
    subprocess.check_call(["g++", "-std=c++17", "-I" + inc, str(src), "-o", str(exe)])
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, f"max_particles {r.stdout.strip()}"
