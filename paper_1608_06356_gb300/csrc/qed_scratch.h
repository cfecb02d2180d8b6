// qed_scratch.h -- sizes of the step's scratch and of launches (plain C++).
#ifndef QED_SCRATCH_H
#define QED_SCRATCH_H

#include <cstdint>

namespace qed {

constexpr int SUB_REC = 8;  // emission records kept per particle by the sub-step counting pass

// Emission records of the multi-pass step (SUB_REC per entry, for the first
// rec_entries entries) and staging records (16 Reals each).  The photon stage
// keeps a record per pair in the same memory -- two words of rec_k and eight
// Reals of the stage -- and every photon may convert in one step, so both must
// hold max_particles pairs, whatever the rounding of the divisions.  (The ordered
// single pass keeps the photon count of every lepton to replay, 2 max_particles
// words at most, in rec_k too: the same size.)
constexpr int64_t rec_entries(int64_t max_particles) {
  const int64_t r = max_particles / 4 + 1;
  return r > 4096 ? r : 4096;
}
constexpr int64_t stage_records(int64_t max_particles) {
  const int64_t r = max_particles / 2 + 1;
  return r > 65536 ? r : 65536;
}
constexpr bool holds_pairs(int64_t max_particles) {
  return rec_entries(max_particles) * SUB_REC / 2 >= max_particles && 2 * stage_records(max_particles) >= max_particles;
}
static_assert(holds_pairs(1) && holds_pairs(16384) && holds_pairs(16385) && holds_pairs(16387) && holds_pairs(16388) &&
                  holds_pairs(131072) && holds_pairs(131073) && holds_pairs(((int64_t)1 << 30) - 4096),
              "a record for every pair");

// Rows of a launch with `per_row` threads a row, CTAs of `block`: thread numbers
// up to the last CTA's fit 32 bits.
constexpr int64_t slab_rows(int64_t per_row, int64_t block) {
  return (((int64_t)1 << 32) - block) / per_row;
}

}  // namespace qed

#endif
