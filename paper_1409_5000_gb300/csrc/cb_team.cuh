// Launch interface of the team kernel (cb_team.cu).
#pragma once

#include "cb_step.cuh"

namespace cb {

constexpr uint32_t kMaxTeams = 160;     // realisations of one cooperative launch
constexpr uint32_t kMaxTeamCtas = 160;  // its CTAs (one per SM)
constexpr uint32_t kCtrStride = 32;     // counters a cache line apart

struct TeamArgs {
  double *parts;  // [2][kMaxTeamCtas] partials of the CTAs
  uint32_t *ctr;  // barrier counter of team q at q kCtrStride, 0 before the launch
  double *xd;             // [pass][CTA][ms] dot products of the Gram-Schmidt passes
  uint64_t whole_x;  // bit q: team q keeps all of W_j in shared memory
  uint32_t nteams;   // 0: one CTA per realisation, any number of them
  uint32_t smem;     // dynamic shared memory of a CTA
  uint32_t rowdiv;   // a row weighs as much as mean degree / rowdiv entries
  uint32_t reorth;
  uint64_t wait_ns;  // limit of a barrier's wait
  uint32_t stall;    // test hook: the last CTA of each team never arrives
  uint16_t first[kMaxTeams + 1];  // first CTA of each team
};

// Whether the recurrence over realisations [r0, r1) with elements of esz bytes
// runs as one launch; its grid and arguments (the buffers left to the caller).
bool team_plan(const cb_graph *h, uint32_t r0, uint32_t r1, size_t esz, bool reorth, TeamArgs *out,
               uint32_t *grid, bool *cooperative);
// Whether one CTA per realisation (lanczos_small_kernel) is the better route for FP32
// realisations that are small enough for it and that no team takes.
bool small_launch_pays(const cb_graph *h, uint32_t r0, uint32_t r1);
template <typename T>
int team_launch(const LArgs &a, TeamArgs t, uint32_t r0, uint32_t m, uint32_t grid, bool cooperative,
                cudaStream_t s);

}  // namespace cb
