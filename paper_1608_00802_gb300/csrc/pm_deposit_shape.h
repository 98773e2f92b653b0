// The deposit's launch: tile shape, blocks, helper blocks for crowded rows and shared memory.  Host code without CUDA
// types, so that the rules can be tested by themselves.
#pragma once
#include <stddef.h>
#include <stdint.h>

#include <algorithm>

#ifdef __CUDACC__
#define PM_DEP_HD __host__ __device__
#else
#define PM_DEP_HD
#endif

namespace pm {

// Mesh rows with more records than this are "crowded": the deposit computes the rows they add to by whole
// blocks instead of one warp each.  A tile's warp takes 0.4 us per batch of 32 records when few warps are busy, so
// nine rows of 256 records are ~30 us, the length of the whole kernel at 2 10^6 particles.  The blocks take ten times
// as long for a record as all the warps together, so a tile is theirs only if its chain would outlast the rest of the
// kernel: the rest takes 1.4e-5 us a particle, the chain 9/32 * 0.4 us for each record of a row, equal near N_p / 6000
// records.  And where every row is long, none is crowded (twice the mean: a uniform state's rows differ by a few
// sqrt(mean)).
// Uniform, a particle per cell: 256^3 by blocks (256 records, whatever the state) 2320 us, by tiles 228; 2 10^6
// particles on 32^3 2377 and 221.  Clustered (a power law of 300 cores), N_p / 6000 against 256 records or
// twice the mean: 256^3 550 and 830, 2 10^6 particles on 256^3 104 and 137; a core of 10^6 on 128^3 keeps 256.
// The word after the row starts, row_start[N^2 + 1], says whether any row is (CROWD_WORDS entries follow
// the N^2 row starts: the closing one and the flag).
inline uint32_t deposit_crowd(int64_t n_part, int n_mesh) {
  int64_t c = 256;
  const int64_t mean = n_part / (int64_t(n_mesh) * n_mesh);
  if (2 * mean > c) c = 2 * mean;
  if (n_part / 6000 > c) c = n_part / 6000;
  return uint32_t(c);
}
constexpr size_t CROWD_WORDS = 2;

constexpr int DEP_WARPS = 8;  // most warps of a block
// what fits an SM: blocks of 40 warps together with the kernel's 48 registers; its shared memory, of which a block takes
// 1040 bytes of its own and 1 KB of the system's besides the dynamic
constexpr unsigned DEP_SMS = 152, DEP_SM_WARPS = 40;
constexpr size_t DEP_SM_SMEM = 228 * 1024, DEP_BLOCK_SMEM = 2064;

// slots of a deposit row: N + 1 rounded up to 16 bytes
template <typename R>
PM_DEP_HD inline int deposit_stride_of(int n) {
  const int q = 16 / int(sizeof(R));
  return (n + 1 + q - 1) / q * q;
}

// deposit tile of TY x TZ rows per warp: by size the largest of 2 x 4, 2 x 2, 1 x 2, 1 x 1 whose rows fit
// PM_DEPOSIT_WARP_BYTES of shared memory per 4-byte accumulator (4.25 KB: 2 x 2 rows of a 256^3
// fp32 mesh; measured there: 43 us against 53 us for 2 x 4 rows, whose 8.3 KB per warp leave
// too few resident warps)
#ifndef PM_DEP_HELPERS
#define PM_DEP_HELPERS 608
#endif
#ifndef PM_DEPOSIT_WARP_BYTES
#define PM_DEPOSIT_WARP_BYTES 4352
#endif
// Small meshes take fewer planes per tile while the launch's tiles (of all nm members of a packed group) are fewer
// than PM_DEPOSIT_MIN_TILES warps (16 per SM): a warp's time is its chain of batches, one or two per plane, so 64^3
// goes from 512 tiles of five source planes (6.9 us) to 2048 of two (4.2 us; 4096 particles on 32^3 7.2 -> 3.9 us).  A
// packed group that has the warps anyway keeps the thick tiles, which read each record less often (16 members: 64^3
// 124 -> 119 us a step, 128^3 645 -> 637).  Not in fp64, whose pipe pays
// for every record read again (14.1 -> 14.7 us).  The planes of a tile do not enter its result: a row's batches
// are cut by its chain, which only the rows in y decide, and added plane by plane.
#ifndef PM_DEPOSIT_MIN_TILES
#define PM_DEPOSIT_MIN_TILES 2432
#endif
template <typename R>
inline int deposit_shape(int n, int nm, int& ty, int& tz) {
  static const int shapes[5][2] = {{2, 4}, {2, 2}, {2, 1}, {1, 2}, {1, 1}};
  const size_t row = size_t(deposit_stride_of<R>(n)) * sizeof(R);
  const size_t most = size_t(PM_DEPOSIT_WARP_BYTES) * sizeof(R) / 4;
  int s = 0;
  while (s < 4 && (size_t(shapes[s][0] * shapes[s][1]) * row > most || s == 2)) ++s;
  while (sizeof(R) == 4 && s < 2 && nm * ((n + 1) / 2) * ((n + shapes[s][1] - 1) / shapes[s][1]) < PM_DEPOSIT_MIN_TILES) ++s;
  ty = shapes[s][0], tz = shapes[s][1];
  return s;
}

// most records per window of a helper block (the batch sums of a window are kept in shared memory)
template <typename R>
constexpr int DEP_WINDOW = sizeof(R) == 4 ? 2048 : 1024;
// shared memory of a helper block with a window of w records: the window's sums, the row, each cell's first and last
// record of the window
template <typename R>
inline size_t deposit_crowd_smem(int n, int w) {
  return size_t(2 * w + deposit_stride_of<R>(n)) * sizeof(R) + size_t(2 * n) * sizeof(uint16_t);
}
// Shared memory of a deposit block of `warps` warps whose tiles take `tiles` bytes, and its helpers' window.  The
// window does not enter the result (it is whole batches), so a block of few warps takes a small one, a full window with
// 8 warps: with a full one for any block, blocks of 1 and 2 warps on 256^3 took 88 and 55 us for 43 and 41, and a batch
// of mixed sizes with 4 warps 2796 us a step for 2552.
#ifndef PM_DEP_CROWD_WARP
#define PM_DEP_CROWD_WARP 2304
#endif
template <typename R>
inline size_t deposit_smem(int n, int warps, size_t tiles, int* window) {
  size_t smem = std::max(tiles, std::min(deposit_crowd_smem<R>(n, DEP_WINDOW<R>), size_t(warps) * PM_DEP_CROWD_WARP));
  smem = std::max(smem, deposit_crowd_smem<R>(n, 64));
  const int w = int((smem - deposit_crowd_smem<R>(n, 0)) / (2 * sizeof(R))) & ~31;
  *window = std::min(w, DEP_WINDOW<R>);
  return smem;
}

struct DepositLaunch {
  int shape, ty, tz;         // tile shape (index of deposit_shape, rows x planes)
  int warps;                 // per block
  unsigned blocks, helpers;  // of the tiles, and after them for the crowded rows
  uint32_t crowd;            // deposit_crowd
  int window;                // records of a helper's window
  size_t smem;               // dynamic shared memory of a block
};

// the launch for n_part particles (in each of nm members of a packed group) in blocks of `warps` warps
template <typename R>
inline DepositLaunch deposit_launch(int64_t n_part, int n_mesh, int warps, int nm) {
  DepositLaunch d = {};
  // A packed group fills the chip with any block size, and beside other groups small blocks get in the way of kernels
  // that need much of an SM (8 members each of 64^3, 128^3 and 256^3: 2761 us a step with 2 warps, 2552 with 4)
  if (nm > 1 && warps < 4) warps = 4;
  d.shape = deposit_shape<R>(n_mesh, nm, d.ty, d.tz);
  d.warps = warps;
  const unsigned N = unsigned(n_mesh), n2 = N * N;
  d.blocks = unsigned((n_mesh + warps * d.ty - 1) / (warps * d.ty)) * unsigned((n_mesh + d.tz - 1) / d.tz);
  d.smem = size_t(warps) * d.ty * d.tz * deposit_stride_of<R>(n_mesh) * sizeof(R);
  d.crowd = deposit_crowd(n_part, n_mesh);
  // helper blocks for crowded tiles (none with so few particles): at most PM_DEP_HELPERS of 8 warps in all,
  // and no fewer than 16 rows each.  A helper takes every helpers-th row, and rows crowd together, so their
  // number is q N + 0.382 N: a block's rows then lie far apart in y from plane to plane (a core of 10^6
  // particles on 128^3: the longest share is one row's, 1.0 .. 1.1 of it over meshes of 64 .. 160; with
  // 2 N + 1 blocks it is 7 of them, 800 us instead of 87)
  if (n_part <= int64_t(d.crowd)) return d;
  const unsigned most = std::max(8u, std::min(unsigned(PM_DEP_HELPERS * DEP_WARPS / (warps * nm)), n2 / 16 + 1));
  const unsigned part = unsigned(0.382 * n_mesh);
  d.helpers = most >= N + part ? (most - part) / N * N + part : most;
  d.smem = deposit_smem<R>(n_mesh, warps, d.smem, &d.window);
  // The helpers come at the end of the tiles' grid.  Where the tiles alone leave room on the SMs, the longer grid is
  // no longer spread evenly over them and some SMs get more than their share of the tiles (128^3 with a particle
  // per cell: fp64 359 -> 527 us, fp32 43 -> 51; 64^3 particles in fp64 57 -> 78), so shared memory keeps an SM
  // to its even share: 357, 43 and 57 us again.  In fp32 only when not all blocks are resident at once and from 2^21
  // particles: the other kernels' share of the SM changes with the deposit's, which costs ~4 us a call, as
  // much as the even spread saves there (10^6 particles in a core: 3147 -> 3180 us a run).  Not in packed groups: they
  // run beside others, which lose more by the shared memory (8 members each of 64^3, 128^3, 256^3: 2552 -> 2728 us).
  if (nm == 1 && (sizeof(R) == 8 || n_part >= int64_t(1) << 21)) {
    const unsigned share = (d.blocks + DEP_SMS - 1) / DEP_SMS;
    const unsigned per_sm = std::min(DEP_SM_WARPS / unsigned(warps), unsigned(DEP_SM_SMEM / (d.smem + DEP_BLOCK_SMEM)));
    if (share < per_sm && d.blocks + d.helpers > DEP_SMS * (sizeof(R) == 8 ? share : per_sm))
      d.smem = std::max(d.smem, (DEP_SM_SMEM / (share + 1) - DEP_BLOCK_SMEM) / 256 * 256 + 256);
  }
  return d;
}

}  // namespace pm
