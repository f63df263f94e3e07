// gm_em.cu -- the EM kernel's launch: instantiation and launch shape.
#include "em_launch.cuh"

namespace gmcr {

// The launch shape: one CTA per SM, T teams of `team` threads, a cell each.
// Results do not depend on it (the sums' order is the groups', see Team).
//   * A cell of more than 128 pairs takes 4 warps, up to 5 teams per SM: the
//     serial M-steps of one cell overlap the passes of the others, and 640
//     threads leave 96 registers, which the passes need without spilling.
//     4096 1V cells of 2000 particles, 16384 3V cells of 572 on average (ms, one
//     run of the variants on the same inputs):
//     5 x 128 threads 102, 126; 4 x 128 119, 138; 8 x 64 -, 144; 8 x 128 at
//     64 registers 109, -; one CTA of 256 threads per cell (two or four per
//     SM, the same work) 113, 284.
//   * Smaller cells have only 1 to 4 groups of pairs: 2 warps, up to 10 teams.
//     So do cells with the FP32 M-step, a tenth of the FP64 one, where at least 8
//     tiles fit and more than 5 cells wait: the passes' latency is what is left
//     to hide (4096 cells of 785, 24 sweeps: 1V 3.75 -> 3.15 ms, 3V 8.2 -> 8.1; 300
//     particles 2.80 -> 2.13, 5.2 -> 4.3; 1216 cells of 785 1.31 -> 0.98, 2.88 -> 2.21;
//     with 4 cells per SM two warps take 1.12 times as long).
//   * No more teams than tiles of the mean size fit the pool (but two: a
//     team without a tile works in L2, at once if the tile is larger than its
//     share; 888 3V cells of 4500 particles 11.5 -> 8.8 ms against waiting for
//     the other's tile, 500 1V cells of 8000 4.9 -> 4.2, 1216 3V cells of 600 and 6000
//     13.9 -> 8.1), and no more than the SM's share of
//     the cells; with one or two cells per SM a cell gets 8 warps, one group
//     each (32 cells of 156 particles: 3.9 ms with 256 threads, 4.8 with 64).
cudaError_t launch_em(int D, int fp64_mstep, EmParams p, int sms, cudaStream_t s) {
  constexpr int64_t kSmem = 227 * 1024;  // a CTA's dynamic shared memory, at most
  const int64_t ctl = (int64_t)(D == 1 ? (fp64_mstep ? em_ctl_size<1, double>() : em_ctl_size<1, float>())
                                       : (fp64_mstep ? em_ctl_size<3, double>() : em_ctl_size<3, float>()));
  const int64_t mean = (p.n + p.C - 1) / p.C;
  const int64_t per_sm = (p.C + sms - 1) / sms;
  EmShape sh;
  const int64_t each2 = ctl + 2 * em_buf_bytes(D) + em_tile_bytes(D, mean, true);  // with 2 warps
  sh.team = mean > 256 && (fp64_mstep || per_sm <= 5 || kSmem / each2 < 8) ? 128 : 64;
  const int64_t each = each2 + (sh.team / 32 - 2) * em_buf_bytes(D);
  int64_t T = kSmem / each;
  if (T < 2) T = 2;
  if (T > kEmThreads / sh.team) T = kEmThreads / sh.team;
  if (T > per_sm) T = per_sm;
  if (T <= 2) sh.team = 256;
  sh.teams = (int)T;
  const int64_t need = (p.C + T - 1) / T;
  sh.grid = (int)(need < sms ? need : sms);
  p.team = sh.team;
  p.patience = 1 << 15;  // 2 us each: a cell's fit takes a few ms
  p.granules = (int)((kSmem - 64 - T * ctl - T * sh.team / 32 * em_buf_bytes(D)) / kPoolGranule);
  if (p.granules > 32 * kPoolWords) p.granules = 32 * kPoolWords;
  // a team's share; where the others' tiles, at twice the mean, leave room for
  // more, up to half of the pool (16384 log-normal 3V cells of 572: a cell of
  // three times the mean waits for a hole rather than work in L2)
  const int64_t mean_gn = (em_tile_bytes(D, mean, true) + kPoolGranule - 1) / kPoolGranule;
  int64_t share = p.granules - 2 * (T - 1) * mean_gn;
  if (share > p.granules / 2) share = p.granules / 2;
  if (share < p.granules / T) share = p.granules / T;
  p.share = (int)share;
  if (D == 1)
    return fp64_mstep ? em_go<1, double>(p, sh, kSmem, s) : em_go<1, float>(p, sh, kSmem, s);
  return fp64_mstep ? em_go<3, double>(p, sh, kSmem, s) : em_go<3, float>(p, sh, kSmem, s);
}

}  // namespace gmcr
