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


def test_field_slabs_number_their_threads_in_32_bits(tmp_path):
    """Every thread number of a field pass fits 32 bits, the slabs cover all rows,
    and grids below 4.2e9 cells take one launch (a Yee grid and its nodes are 68
    bytes a cell: 4.3e9 cells still fit the device)."""
    src = tmp_path / "slabs.cpp"
    src.write_text("""
        #include <initializer_list>
        #include "qed_scratch.h"
        using namespace qed;
        int main() {
          for (int64_t per_row : {1, 2, 3, 127, 128, 129, 1000, 1639, 16384, 65535, 65536}) {
            const int64_t s = slab_rows(per_row, 128);
            const int64_t threads = (s * per_row + 127) / 128 * 128;
            if (s < 1 || threads > ((int64_t)1 << 32) || s * per_row < 4200000000ll) return 1;
          }
          return 0;
        }""")
    exe = tmp_path / "slabs"
    inc = os.path.join(ROOT, "paper_1608_06356_gb300", "csrc")
    subprocess.check_call(["g++", "-std=c++17", "-I" + inc, str(src), "-o", str(exe)])
    assert subprocess.run([str(exe)]).returncode == 0
