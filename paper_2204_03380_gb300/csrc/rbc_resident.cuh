// rbc_resident.cuh -- tables of the resident 2-D time loops (rbc_resident.cu),
// shared by the single-shot contexts (rbc_abi.cu) and the batches (rbc_batch.cu).
#pragma once

#include <vector>

#include "rbc_internal.cuh"

namespace rbc {

enum { kResFwd = 0, kResRev = 1, kResStore = 2 };  // the loops: forward, reverse (imaging, FWI), storage-RTM reverse

// One block's tile: 128 columns x `rows` rows of one shot's padded grid.
struct ResTile {
  int shot;
  int x0, z0;
  int rows;       // rows of the grid in this tile (the last tile of a column may have fewer than H)
  int up, dn, lf, rt;  // neighbouring tiles (index into the tile table), or -1
};

// One shot: its fields in the pitched layout and the per-call tables.
struct ResShot {
  Lay L;
  const float *a;
  float *p[2];              // level m in p[m & 1]: written by the forward loop, read by the reverse loop
  float *q[2];              // pbar's level m in q[m & 1], sums in cnum / cden (pitched): what a reverse loop of several
  float *cnum, *cden;       // parts leaves for the next part (unused with one part)
  const ShotInfo *info;
  float *seis_t;            // [levels][nrec] time-major record
  const int *cell_ptr;      // receivers of each (tile, warp) of this shot's tile range (CSR)
  const int2 *cell_rec;     // {node's place in the tile (row * 128 + column), receiver index}
  float *num, *den;         // outputs of the reverse loop (see ResArgs)
  int tile0;                // this shot's first tile
  int ix0, ix1, iz0, iz1;   // interior box in padded nodes
};

struct ResArgs {
  const ResTile *tiles;
  const ResShot *shots;
  unsigned long long *ll;   // halo exchange words, zeroed before the launch
  const float *wav;         // f[0..nt-1]
  int nt;
  int t0, t1;               // this part's steps (res_launch)
  int sample;               // forward: record every level at the receivers
  int grad;                 // reverse: 1 = FWI gradient (num += mu p_tt), 0 = imaging integrals
  int overwrite;            // reverse: outputs are set, not added to
  int dense;                // reverse: num / den are dense interior arrays (else pitched)
  float *store;             // storage RTM: the kept levels, every `stride` steps (0: none kept)
  int stride;
  int *err;
  int *gave_up;             // this loop's own mark of a wait that gave up (behind its exchange words), for its later parts
};

// Tiling of a resident loop over one or several grids: `warps` warps of `rz`
// rows per block (H = warps * rz rows per tile), `blocks` blocks, all resident.
struct ResPlan {
  int variant = -1;         // index into the kernel variants, -1: does not fit
  int rz = 0, warps = 0, H = 0;
  int blocks = 0;
  int steps = 1;            // most steps of one launch (a longer loop runs in parts)
  size_t smem = 0;
  std::vector<ResTile> tiles;
  std::vector<int> tile0;   // first tile of each shot, then the tile count
};

// Plan for one loop (dir) of the given layouts (variant -1 when
// they do not fit on this device at once); share: the device is shared by that
// many such loops.
bool res_plan(const Lay *L, int nshots, int dir, int share, ResPlan *out);
// Plan for one of `loops` such loops that run at a time: chosen for the time of all of them; false where it does not
// fit or (steps) one launch per step is through sooner.
bool res_plan_shared(const Lay *L, int nshots, int dir, int loops, bool steps, ResPlan *out);
// A context or batch whose loops may run beside others', and the number of them in flight with a call of it.
struct LoopUser {
  int dev = 0;
  unsigned long long called = 0, on_stream = 0;  // its last counted call (0: none yet) and that call's stream
  unsigned long long born = 0;                   // calls counted before it was added
};
void flight_add(LoopUser *u);
void flight_remove(LoopUser *u);
int flight_count(LoopUser *u, cudaStream_t s);
// Shots of a batch sorted into groups whose loops run at once: groups of shot
// indices, or none when a shot does not fit.
std::vector<std::vector<int>> res_groups(const Lay *L, int nshots);
size_t res_ll_bytes(const ResPlan &P, int dir);
// At least res_ll_bytes of any plan of these grids on half of the device or less, for loops of nf fields.
size_t res_ll_bound(const Lay *L, int nshots, int nf);
// cudaMalloc for the loops' own tables, without which a context or batch takes the step path; res_fail_alloc(true)
// makes the next one fail (rbc_inject_fault).
cudaError_t res_malloc(void **p, size_t bytes);
void res_fail_alloc(bool on);
// The (tile, warp) cell that owns a node, within its shot's tiles, and the
// node's place in the tile.
void res_cell(const ResPlan &P, const Lay &L, int x, int z, int *cell, int *loc);
// Receiver cells of one shot (its tiles * warps cells): CSR pointers and
// {place in the tile, receiver}, positions offset by `base`.
void res_cells(const ResPlan &P, const Lay &L, int cells, int nrec, const int *rec, int base, int *ptr, int2 *out);
// Whether a forward loop that records nrec receivers is through sooner by launches.
bool res_many_receivers(const ResPlan &P, int nrec);
// Parts of a loop of n steps (forward: nt; reverse: nt + 1).
inline int res_parts(const ResPlan &P, int n) { return (n + P.steps - 1) / P.steps; }
// withhold: the first of several parts is not launched (rbc_inject_fault), so that the second waits in vain.
cudaError_t res_launch(const ResPlan &P, int dir, const ResArgs &A, cudaStream_t s, long long *launches,
                       bool withhold = false);

} // namespace rbc
