// rbc_resident.cu -- 2-D time loops that stay on the chip.
//
// A launch per time step moves every field through L2 at every step (forward
// 16 bytes per node, fused reverse 60) and pays a launch's latency.  A grid of
// up to about 2.1 M padded nodes (the 2421 x 871 survey grid, at 7 fields) has
// room on the chip: 152 SMs hold 34 MB of shared memory and 39 MB of tensor
// memory.  Here one cooperative launch runs a whole loop, or a part of it of
// some two milliseconds (res_plan).  Each block keeps a
// tile of 128 columns x H rows for all the launch's steps: the two levels of each field
// in shared memory; a and the imaging sums in registers and shared memory
// (tiles of one or two rows per warp) or in tensor memory, which serves as a
// thread-private store (32 lanes of a quarter x 512 columns; no MMA runs) and
// leaves shared memory to the fields.  Only the tile's four edge rows and
// columns leave the SM: they go to the neighbouring tiles as 8-byte words of
// {value, level} through L2, so that a reader that finds the level it waits
// for has the value with it -- no fence, no flag, one L2 round trip.  A word's
// place alternates between even and odd levels: a writer is at most one level
// ahead of its reader, because it needs the reader's own words to get there.
// All blocks are resident (the launch is cooperative) and every wait is bounded.
//
// What bounds it: one block by itself takes 0.9 us per level and field plus
// 0.69 us for every ten-row warp on a scheduler (143 clocks per row; 59 packed
// operations take 118), so a survey tile (11 warps) 2.9 us, and the exchange
// adds 0.5 us; on small grids the fixed part and the exchange are all there
// is.  Measured (us per step; before, one launch per step): survey forward 3.5
// (6.1), forward + reverse 10.5 (18.8); 300 x 300 forward 1.5 (2.7), forward +
// reverse 4.4 (6.7).  Tensor memory for a and the sums: 8 us per reverse step
// against 12.4 with the sums in registers (spilled) and a read from L2 twice.
// Reverse kernels of 16 warps have 128 registers a thread and still spill some:
// 156 bytes stored (7 rows per warp, imaging), 134 (7, gradient), 64 (2,
// imaging), 28 and 4 (4); ten rows of 11 warps, with 162 registers, none.
// Tried and not kept: a warp-to-warp order (mbarriers) instead of the block
// barrier at each step -- the warps drift apart and their unrolled rows no
// longer fit the instruction cache (18 us per reverse step); the same with the
// rows rolled up into a loop of two (9.8 us); the tile's outer columns updated
// last, so that nothing else waits for the words beside it (forward 3.8 us
// against 3.4: the wait is not what bounds a step); 16 warps of 7 rows instead
// of 11 of 10 (the same).
#include <algorithm>
#include <atomic>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <mutex>
#include <type_traits>

#include "rbc_resident.cuh"
#include "rbc_tile2d.cuh"

namespace rbc {

namespace {

typedef unsigned long long u64;
constexpr int kSpins = 2000000;               // polls of a wait before it gives up (each an L2 round trip: about a second)
constexpr int kEdge = 4 * kTileX;             // words of a top or bottom halo (4 rows)

__device__ __forceinline__ void ll_ld(const u64 *p, u64 &a, u64 &b) {
  asm volatile("ld.relaxed.gpu.global.v2.b64 {%0, %1}, [%2];" : "=l"(a), "=l"(b) : "l"(p) : "memory");
}
__device__ __forceinline__ void ll_st(u64 *p, float x, float y, uint32_t tag) {
  u64 a, b;
  asm volatile("mov.b64 %0, {%1, %2};" : "=l"(a) : "r"(__float_as_uint(x)), "r"(tag));
  asm volatile("mov.b64 %0, {%1, %2};" : "=l"(b) : "r"(__float_as_uint(y)), "r"(tag));
  asm volatile("st.relaxed.gpu.global.v2.b64 [%0], {%1, %2};" ::"l"(p), "l"(a), "l"(b) : "memory");
}
__device__ __forceinline__ float ll_val(u64 v) { return __uint_as_float((uint32_t)v); }
__device__ __forceinline__ bool ll_ok(u64 v, uint32_t tag) { return (uint32_t)(v >> 32) == tag; }

// Four consecutive halo values of one lane: two 16-byte loads.
struct Ll4 {
  u64 v[4];
  __device__ __forceinline__ void load(const u64 *p0, const u64 *p1) {
    ll_ld(p0, v[0], v[1]);
    ll_ld(p1, v[2], v[3]);
  }
  __device__ __forceinline__ bool ok(uint32_t tag) const {
    return ll_ok(v[0], tag) && ll_ok(v[1], tag) && ll_ok(v[2], tag) && ll_ok(v[3], tag);
  }
  __device__ __forceinline__ float4 value() const {
    return make_float4(ll_val(v[0]), ll_val(v[1]), ll_val(v[2]), ll_val(v[3]));
  }
  // Poll, from a first load, until the values are those of `tag`; false if it gave up.
  __device__ __forceinline__ bool wait(const u64 *p0, const u64 *p1, uint32_t tag) {
#pragma unroll 1
    for (int i = 0; !ok(tag); ++i) {
      if (i == kSpins) return false;
      load(p0, p1);
    }
    return true;
  }
};

// Halo words of one tile, field and parity: rows above [4][2][32][2], rows
// below [4][2][32][2], columns to the left [H][4], columns to the right [H][4].
__host__ __device__ __forceinline__ int ll_words(int H) { return 2 * kEdge + 8 * H; }

__device__ __forceinline__ float4 lds4(const float *p) { return *reinterpret_cast<const float4 *>(p); }

// A warp's place in its tile (rows r0 .. r0 + RZ - 1) and this lane's ends of
// the halo words (offsets from the exchange buffer, field 0, even levels).
struct Place {
  int lane, r0, rows, H;
  bool up, dn, lr;            // rows above / below come from another tile; this lane moves a column halo
  bool right;                 // ... of the right-hand side
  u64 *in_lr, *in_tb;         // own tile: column halo of this lane's row; rows above (below: + kEdge)
  u64 *out_lr, *out_up, *out_dn;
};

template <int RZ>
__device__ __forceinline__ Place place_of(const ResArgs &A, const ResTile &T, int w, int lane, int H, int nf) {
  Place W;
  W.lane = lane;
  W.r0 = w * RZ;
  W.rows = T.rows;
  W.H = H;
  W.up = T.up >= 0;
  W.dn = T.dn >= 0;
  const size_t tw = (size_t)ll_words(H) * 2 * nf;
  const int j = lane & 15;   // lane j: the left of row j, lane 16 + j: the right
  W.right = lane >= 16;
  const int side = W.right ? T.rt : T.lf;
  W.lr = j < RZ && W.r0 + j < T.rows && side >= 0;
  const int col = 4 * (W.r0 + (j < RZ ? j : 0));
  W.in_lr = A.ll + blockIdx.x * tw + 2 * kEdge + (W.right ? 4 * H : 0) + col;
  W.out_lr = A.ll + max(side, 0) * tw + 2 * kEdge + (W.right ? 0 : 4 * H) + col;
  W.in_tb = A.ll + blockIdx.x * tw + 2 * lane;
  W.out_up = A.ll + max(T.up, 0) * tw + kEdge + 2 * lane;
  W.out_dn = A.ll + max(T.dn, 0) * tw + 2 * lane;
  return W;
}

// Offset of a field's words of level `tag`, opaque so that the addresses
// formed from it are not all kept in registers across the time loop.
__device__ __forceinline__ int ll_off(int f, uint32_t tag, int H) {
  int o = (2 * f + (int)(tag & 1)) * ll_words(H);
  asm volatile("" : "+r"(o));
  return o;
}

// Halo of level `tag` for this warp: the columns beside its rows into s_lr
// ([H][2][4]); where its stencil reaches over the tile's edge, the rows above
// into s_up[4][128] (or, for TIGHT, into the row queue's first four entries)
// and the rows below into s_dn[4][128].
template <int RZ, bool TIGHT>
__device__ __forceinline__ bool halo_in(const Place &W, int f, uint32_t tag, float *s_lr, float *s_up, float *s_dn,
                                        float4 *qa) {
  const int o = ll_off(f, tag, W.H);
  Ll4 c;
  if (W.lr) c.load(W.in_lr + o, W.in_lr + o + 2);
  bool ok = true;
  // Rows k0 .. k1 of the four of a side, polled together.  With fewer than
  // four rows per warp, a warp reads only the halo rows its own rows reach
  // (the others' next level may already be on its way): the rest of its four
  // loads repeat the nearest of those.  (One short loop per side: with a wait
  // of its own behind every load the code a warp jumps over costs more
  // instruction fetches than it saves polls.)
  auto rows_in = [&](const u64 *b, int k0, int k1, auto put) {
    Ll4 t[4];
    bool all;
    int i = 0;
#pragma unroll 1
    do {
      all = true;
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const u64 *p = b + (RZ < 4 ? min(max(k, k0), k1) : k) * kTileX;
        t[k].load(p, p + 64);
      }
#pragma unroll
      for (int k = 0; k < 4; ++k) all = all && t[k].ok(tag);
    } while (!all && ++i < kSpins);
    ok = ok && all;
#pragma unroll
    for (int k = 0; k < 4; ++k) put(RZ < 4 ? min(max(k, k0), k1) : k, k, t[k].value());
  };
  if (W.up && W.r0 < 4)  // rows r0 .. 3 of the four above
    rows_in(W.in_tb + o, W.r0, 3, [&](int kk, int k, float4 v) {
      if (TIGHT) qa[k] = v;
      else st4(s_up + kk * kTileX + 4 * W.lane, v);
    });
  if (W.dn && W.r0 + RZ + 3 >= W.H)  // rows 0 .. r0 + RZ + 3 - H of the four below
    rows_in(W.in_tb + o + kEdge, 0, W.r0 + RZ + 3 - W.H,
            [&](int kk, int, float4 v) { st4(s_dn + kk * kTileX + 4 * W.lane, v); });
  if (W.lr) {
    ok = c.wait(W.in_lr + o, W.in_lr + o + 2, tag) && ok;
    *reinterpret_cast<float4 *>(s_lr + ((W.r0 + (W.lane & 15)) * 2 + (W.right ? 1 : 0)) * 4) = c.value();
  }
  __syncwarp();
  return ok;
}

// This warp's edge rows and columns of a finished level, from shared memory,
// to the neighbours' halo words.
template <int RZ>
__device__ __forceinline__ void halo_out(const Place &W, int f, uint32_t tag, const float *s) {
  const int o = ll_off(f, tag, W.H);
  if (W.lr) {
    const float4 v = lds4(s + (W.r0 + (W.lane & 15)) * kTileX + (W.right ? kTileX - 4 : 0));
    ll_st(W.out_lr + o, v.x, v.y, tag);
    ll_st(W.out_lr + o + 2, v.z, v.w, tag);
  }
  if (W.up && W.r0 < 4) {
#pragma unroll
    for (int i = 0; i < (RZ < 4 ? RZ : 4); ++i) {
      const int r = W.r0 + i;
      if (RZ >= 4 || r < 4) {  // rows past a short last tile are zero in its buffer, and are sent
        const float4 v = lds4(s + r * kTileX + 4 * W.lane);
        u64 *b = W.out_up + o + r * kTileX;
        ll_st(b, v.x, v.y, tag);
        ll_st(b + 64, v.z, v.w, tag);
      }
    }
  }
  if (W.dn && W.r0 + RZ > W.H - 4) {
#pragma unroll
    for (int i = 0; i < (RZ < 4 ? RZ : 4); ++i) {
      const int r = W.r0 + (RZ < 4 ? i : RZ - 4 + i), k = r - (W.H - 4);
      if (RZ >= 4 || k >= 0) {
        const float4 v = lds4(s + r * kTileX + 4 * W.lane);
        u64 *b = W.out_dn + o + k * kTileX;
        ll_st(b, v.x, v.y, tag);
        ll_st(b + 64, v.z, v.w, tag);
      }
    }
  }
}

// One level of one field over this warp's rows: pre(j) starts the loads of
// what is kept elsewhere (a, the imaging sums), body(j, c, old, lap) finishes
// row j and stores it.  The z differences D_k (rbc_stencil.cuh) march down the
// rows in registers.  c0 / n0: the level's / the overwritten level's tile rows
// in shared memory; up / dn: the four rows above / below the warp's rows.
template <int RZ, bool TIGHT, typename Pre, typename Body>
__device__ __forceinline__ void sweep(const Place &W, const float *smem, int c0, int n0, const float *up,
                                      const float *dn, bool have_up, const float4 *qa, int lofs, int lstep, int rofs,
                                      int rstep, Pre pre, Body body) {
  const int lane = W.lane;
  const float *own = smem + c0 + W.r0 * kTileX + 4 * lane;
  const float *lp = smem + lofs + (lane == 0 ? 0 : c0), *rp = smem + rofs + (lane == 31 ? 0 : c0);
  const float *np = smem + n0 + W.r0 * kTileX + 4 * lane;
  auto row = [&](int i) {  // row i - 4 of the warp
    return i < 4 ? (TIGHT && have_up ? qa[i < 4 ? i : 0] : lds4(up + i * kTileX + 4 * lane))
                 : i < RZ + 4 ? lds4(own + (i - 4) * kTileX) : lds4(dn + (i - RZ - 4) * kTileX + 4 * lane);
  };
  float4 q[RZ + 8], D[4][RZ + 4];  // D[k - 1][i] = D_k at row i - 4 (of each k, the last k rows are live)
#pragma unroll
  for (int i = 0; i < 8; ++i) q[i] = row(i);
#pragma unroll
  for (int k = 1; k <= 4; ++k)
#pragma unroll
    for (int i = 4 - k; i < 4; ++i) D[k - 1][i] = sub4(q[i + k], q[i]);
#pragma unroll
  for (int j = 0; j < RZ; ++j) {
    if (W.r0 + j >= W.rows) break;
    pre(j);
    const float4 lf = lds4(lp + j * lstep), rt = lds4(rp + j * rstep), po = lds4(np + j * kTileX);
    q[j + 8] = row(j + 8);
    float4 z[4];
#pragma unroll
    for (int k = 1; k <= 4; ++k) {
      D[k - 1][j + 4] = sub4(q[j + 4 + k], q[j + 4]);
      z[k - 1] = sub4(D[k - 1][j + 4], D[k - 1][j + 4 - k]);
    }
    body(j, q[j + 4], po, lap_shared(lf, q[j + 4], rt, z));
  }
}

// This warp's receivers: the first K * 32 in registers (node's place in the
// tile, receiver), the rest read from the table at every step.
constexpr int rec_regs(int rz) { return rz < 4 ? 4 : 1; }  // K of the forward loop
template <int K>
struct Recs {
  int beg, end, loc[K], id[K];
  __device__ __forceinline__ void load(const int *ptr, const int2 *rec, int cell, int lane, bool any) {
    beg = any ? ptr[cell] : 0;
    end = any ? ptr[cell + 1] : 0;
#pragma unroll
    for (int i = 0; i < K; ++i) {
      const int k = beg + lane + 32 * i;
      const int2 c = k < end ? __ldg(rec + k) : make_int2(0, -1);
      loc[i] = c.x;
      id[i] = c.y;
    }
  }
};

// Shared memory of one field's buffer: H rows, and unless TIGHT four rows
// above and below that the halo is received into.
template <bool TIGHT>
__host__ __device__ __forceinline__ int buf_floats(int H) { return (H + (TIGHT ? 0 : 8)) * kTileX; }

// The interior nodes of this warp's rows of level n to its slot of the store
// (lane l writes columns l, l + 32, ...: whole sectors).
template <int RZ>
__device__ __forceinline__ void keep_level(const ResArgs &A, const ResShot &S, const ResTile &T, const Place &W, int n,
                                           const float *cur) {
  const int nx = S.ix1 - S.ix0;
  float *slot = A.store + (long long)(n / A.stride) * nx * (S.iz1 - S.iz0);
#pragma unroll 1
  for (int j = 0; j < RZ; ++j) {
    const int r = W.r0 + j, z = T.z0 + r;
    if (r >= W.rows || z < S.iz0 || z >= S.iz1) continue;
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int c = W.lane + 32 * e, x = T.x0 + c;
      if (x >= S.ix0 && x < S.ix1) slot[(long long)(z - S.iz0) * nx + x - S.ix0] = cur[r * kTileX + c];
    }
  }
}

// Whether an earlier part gave up waiting (its words never came: no use waiting for them in this one).  A block barrier.
__device__ __forceinline__ bool given_up(const ResArgs &A, int tid) {
  return __syncthreads_or(A.t0 > 0 && tid == 0 && *(volatile const int *)A.gave_up != 0);
}

__device__ __forceinline__ void give_up(const ResArgs &A) {
  *(volatile int *)A.gave_up = 1;
  atomicOr_system(A.err, 1);  // reported by the next call, which clears it: later parts go by the mark above
}

// ------------------------------------------------------------- forward ----
template <int RZ, int MAXW>
__global__ void __launch_bounds__(32 * MAXW, 1) k_res_fwd(const ResArgs A, const int H) {
  extern __shared__ __align__(16) float smem[];
  const int fl = buf_floats<false>(H), h4 = 4 * kTileX;
  float *s_a = smem + 2 * fl;
  float *s_lr = s_a + H * kTileX;       // [H][2][4]
  const ResTile T = A.tiles[blockIdx.x];
  const ResShot &S = A.shots[T.shot];
  const int lane = threadIdx.x, w = threadIdx.y, nthr = 32 * blockDim.y, tid = 32 * w + lane;
  const int origin = S.L.origin, pitch = S.L.pitch, NX4 = S.L.NX4;
  const Place W = place_of<RZ>(A, T, w, lane, H, 1);
  for (int i = tid; i < (2 * fl + H * kTileX + 8 * H) / 4; i += nthr) *reinterpret_cast<float4 *>(smem + 4 * i) = zero4();
  if (given_up(A, tid)) return;
  for (int i = tid; i < T.rows * 32; i += nthr) {
    const int r = i >> 5, x = T.x0 + 4 * (i & 31), o = origin + (T.z0 + r) * pitch + x;
    if (x < NX4) {
      *reinterpret_cast<float4 *>(s_a + 4 * i) = ldg4(S.a + o);
      if (A.t0 > 0) {  // the part before left its last two levels
        st4(smem + h4 + 4 * i, ld4(S.p[0] + o));
        st4(smem + fl + h4 + 4 * i, ld4(S.p[1] + o));
      }
    }
  }
  const int x0 = T.x0 + 4 * lane;
  const bool xok = x0 < NX4;
  const int nrec = S.info->nrec;
  const int src = S.info->src_off;
  const float fsc = S.info->src_fwd;
  const int2 *cell_rec = S.cell_rec;
  float *seis_t = S.seis_t;
  const int cell = (blockIdx.x - S.tile0) * blockDim.y + w;
  constexpr int K = rec_regs(RZ);
  Recs<K> rec;
  rec.load(S.cell_ptr, cell_rec, cell, lane, A.sample != 0);
  auto record = [&](int n, const float *p) {  // p^n at this warp's receivers
    float *row = seis_t + (long long)n * nrec;
#pragma unroll
    for (int i = 0; i < K; ++i)
      if (rec.id[i] >= 0) row[rec.id[i]] = p[rec.loc[i]];
    for (int k = rec.beg + 32 * K + lane; k < rec.end; k += 32) {
      const int2 c = __ldg(cell_rec + k);
      row[c.y] = p[c.x];
    }
  };
  const int row0 = origin + (T.z0 + W.r0) * pitch;  // this warp's first row
  const bool has_src = src >= row0 + T.x0 && src < row0 + T.x0 + RZ * pitch;
  // left / right neighbours of the lane's four columns: the tile's own row, or the halo columns
  const int lstep = lane == 0 ? 8 : kTileX, rstep = lane == 31 ? 8 : kTileX;
  const int lofs = lane == 0 ? (int)(s_lr - smem) + W.r0 * 8 : W.r0 * kTileX + 4 * lane - 4;
  const int rofs = lane == 31 ? (int)(s_lr - smem) + W.r0 * 8 + 4 : W.r0 * kTileX + 4 * lane + 4;
  const float *pa = s_a + W.r0 * kTileX + 4 * lane;
  __syncthreads();
  const int nt = A.nt;
  bool ok = true;
  float f = has_src ? A.wav[A.t0] * fsc : 0.f, f_next = 0.f;
  int keep = A.stride > 0 ? (A.t0 + A.stride - 1) / A.stride * A.stride : -1;  // the next level kept
  for (int n = A.t0; n < A.t1; ++n) {
    if (has_src && n + 1 < nt) f_next = A.wav[n + 1];  // in flight during this step
    const int c0 = (n & 1 ? fl : 0) + h4, n0 = (n & 1 ? 0 : fl) + h4;
    float *cur = smem + c0, *np = smem + n0 + W.r0 * kTileX + 4 * lane;
    if (n > 0) ok = halo_in<RZ, false>(W, 0, (uint32_t)n, s_lr, cur - h4, cur + H * kTileX, nullptr);
    sweep<RZ, false>(W, smem, c0, n0, cur + W.r0 * kTileX - h4, cur + (W.r0 + RZ) * kTileX, false, nullptr, lofs, lstep,
                     rofs, rstep, [](int) {},
                     [&](int j, const float4 c, const float4 po, const float4 lap) {
                       const float4 av = lds4(pa + j * kTileX);
                       float4 v = leap_fin<false>(c, po, av, lap, nullptr);
                       if (has_src) {
                         const int d = src - (row0 + j * pitch + x0);
                         if ((unsigned)d < 4u) point_sub(v, d, cmp(av, d) * f);
                       }
                       if (xok) st4(np + j * kTileX, v);
                     });
    __syncwarp();
    if (n + 1 < nt) halo_out<RZ>(W, 0, (uint32_t)n + 1, smem + n0);
    if (n == keep) {
      keep_level<RZ>(A, S, T, W, n, cur);
      keep += A.stride;
    }
    if (rec.end > rec.beg) record(n, cur);
    f = f_next * fsc;
    if (__syncthreads_or(!ok)) {
      if (tid == 0) give_up(A);
      return;
    }
  }
  if (A.t1 == nt) {
    record(nt, smem + (nt & 1 ? fl : 0) + h4);
    if (nt == keep) keep_level<RZ>(A, S, T, W, nt, smem + (nt & 1 ? fl : 0) + h4);
  }
  // the last two levels, for the next part, or the reverse loop and rbc_get_panels
  for (int j = 0; j < RZ; ++j) {
    const int r = W.r0 + j;
    if (r < W.rows && xok) {
      const int o = row0 + j * pitch + x0;
      st4(S.p[0] + o, lds4(smem + h4 + r * kTileX + 4 * lane));
      st4(S.p[1] + o, lds4(smem + fl + h4 + r * kTileX + 4 * lane));
    }
  }
}

// ------------------------------------------------------------- reverse ----
// acc + a b, rounded as the one-launch-per-step kernels round it: product and
// sum (their products are masked), or once (k_store_image)
template <int MODE>
__device__ __forceinline__ float4 add_prod(const float4 a, const float4 b, const float4 c) {
  float2 l, h;
  if (MODE == 2) {
    l = __ffma2_rn(lo2(a), lo2(b), lo2(c));
    h = __ffma2_rn(hi2(a), hi2(b), hi2(c));
  } else {
    l = __fadd2_rn(__fmul2_rn(lo2(a), lo2(b)), lo2(c));
    h = __fadd2_rn(__fmul2_rn(hi2(a), hi2(b)), hi2(c));
  }
  return make_float4(l.x, l.y, h.x, h.y);
}

// What a thread keeps of its own nodes besides the fields: a and the imaging
// sums (FWI: the gradient sum in num).  Small tiles: a in shared memory, the
// sums in registers.
template <int RZ, int MODE>
struct KeepReg {
  static constexpr bool kGrad = MODE == 1;
  const float *pa;
  float4 num[RZ], den[kGrad ? 1 : RZ];
  __device__ __forceinline__ void init(float *s_a, const Place &W) {
    pa = s_a + W.r0 * kTileX + 4 * W.lane;
#pragma unroll
    for (int j = 0; j < RZ; ++j) {
      num[j] = zero4();
      if (!kGrad) den[j] = zero4();
    }
  }
  __device__ __forceinline__ void pre_a(int) {}
  __device__ __forceinline__ void pre_all(int) {}
  __device__ __forceinline__ float4 a(int j) { return lds4(pa + j * kTileX); }
  __device__ __forceinline__ void add(int j, const float4 c, const float4 b) {
    num[j] = add_prod<MODE>(c, b, num[j]);
    if (!kGrad) den[j] = add_prod<MODE>(c, c, den[j]);
  }
  __device__ __forceinline__ void flush() {}
  __device__ __forceinline__ void sums(int j, float4 &n, float4 &d) {
    n = num[j];
    if (!kGrad) d = den[j];
  }
};

__device__ __forceinline__ void tm_ld4(uint32_t ta, float4 &v) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
               : "r"(ta));
}
__device__ __forceinline__ void tm_st4(uint32_t ta, const float4 v) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1, %2, %3, %4};" ::"r"(ta), "f"(v.x), "f"(v.y), "f"(v.z),
               "f"(v.w)
               : "memory");
}
// st4 to shared memory where `on`, as one predicated store: the lanes of a warp do not part at it, so that the
// whole-warp (.sync.aligned) accesses of the next row need no __syncwarp (one per row cost the survey's reverse
// loop 3 %).  Not ordered against other shared-memory accesses by itself: every reader of the row is behind a
// __syncwarp or __syncthreads, and the thread's own earlier load of the place feeds the stored value.
__device__ __forceinline__ void st4_if(bool on, float *p, const float4 v) {
  asm volatile("{\n.reg .pred q;\nsetp.ne.u32 q, %0, 0;\n@q st.shared.v4.f32 [%1], {%2, %3, %4, %5};\n}" ::"r"((uint32_t)on),
               "r"((uint32_t)__cvta_generic_to_shared(p)), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w));
}
// Wait for this thread's tensor-memory loads; the loaded values are used after it only.
__device__ __forceinline__ void tm_wait(float4 &a) {
  asm volatile("tcgen05.wait::ld.sync.aligned;" : "+f"(a.x), "+f"(a.y), "+f"(a.z), "+f"(a.w)::"memory");
}
__device__ __forceinline__ void tm_tie(float4 &a) { asm volatile("" : "+f"(a.x), "+f"(a.y), "+f"(a.z), "+f"(a.w)); }

// Large tiles: a and the sums in tensor memory, used as a thread-private store
// (a warp reaches the 32 lanes of its quarter; 12 columns per row: a, num, den).
// Its accesses are the whole warp's: the lanes are together before a sweep and do not part in its rows.
template <int RZ, int MODE>
struct KeepTm {
  static constexpr bool kGrad = MODE == 1;
  uint32_t ta;
  float4 av, nv, dv;
  __device__ __forceinline__ void pre_a(int j) { tm_ld4(ta + 12 * j, av); }
  __device__ __forceinline__ void pre_all(int j) {
    tm_ld4(ta + 12 * j, av);
    tm_ld4(ta + 12 * j + 4, nv);
    if (!kGrad) tm_ld4(ta + 12 * j + 8, dv);
  }
  __device__ __forceinline__ float4 a(int) {
    tm_wait(av);
    return av;
  }
  __device__ __forceinline__ void add(int j, const float4 c, const float4 b) {
    tm_tie(nv);
    nv = add_prod<MODE>(c, b, nv);
    if (!kGrad) {
      tm_tie(dv);
      dv = add_prod<MODE>(c, c, dv);
    }
    __syncwarp();
    tm_st4(ta + 12 * j + 4, nv);
    if (!kGrad) tm_st4(ta + 12 * j + 8, dv);
  }
  __device__ __forceinline__ void flush() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
  __device__ __forceinline__ void sums(int j, float4 &n, float4 &d) {
    tm_ld4(ta + 12 * j + 4, nv);
    if (!kGrad) tm_ld4(ta + 12 * j + 8, dv);
    tm_wait(nv);
    n = nv;
    if (!kGrad) {
      tm_tie(dv);
      d = dv;
    }
  }
};
constexpr int tm_cols(int rz, int warps) {
  const int c = (warps + 3) / 4 * rz * 12;
  return c <= 128 ? 128 : c <= 256 ? 256 : 512;
}

// MODE 0: imaging integrals (Eq. 3); 1: FWI gradient; 2: RTM with wavefield storage (Algorithm 2: only pbar is
// stepped, and the integrals are formed at the kept levels, with p^n read from the store)
template <int RZ, int MAXW, bool TIGHT, bool TM, int MODE>
__global__ void __launch_bounds__(32 * MAXW, 1) k_res_rev(const ResArgs A, const int H) {
  constexpr bool kGrad = MODE == 1, kStore = MODE == 2;
  constexpr int NB = kStore ? 2 : 4, B0 = kStore ? 0 : 2, FB = kStore ? 0 : 1;  // buffers; pbar's first, its exchange field
  extern __shared__ __align__(16) float smem[];
  const int fl = buf_floats<TIGHT>(H), h4 = TIGHT ? 0 : 4 * kTileX;
  float *s_lr = smem + NB * fl;        // [H][2][4], the warp's own rows: both fields in turn
  // TIGHT: [4][128] rows below, read by the last warp, both fields in turn; without TM: a [H][128]
  float *s_x = s_lr + 8 * H;
  const int xfl = ((TIGHT ? 4 : 0) + (TM ? 0 : H)) * kTileX;
  uint32_t *s_tm = reinterpret_cast<uint32_t *>(s_x + xfl);  // TM: the tensor memory's address
  static_assert(TM || !TIGHT, "the tight layout leaves no shared memory for a");
  const ResTile T = A.tiles[blockIdx.x];
  const ResShot &S = A.shots[T.shot];
  const int lane = threadIdx.x, w = threadIdx.y, nthr = 32 * blockDim.y, tid = 32 * w + lane;
  const int origin = S.L.origin, pitch = S.L.pitch, NX4 = S.L.NX4;
  const Place W = place_of<RZ>(A, T, w, lane, H, kStore ? 1 : 2);
  const int nt = A.nt;
  constexpr int TC = tm_cols(RZ, MAXW);
  if (given_up(A, tid)) return;
  if (TM && w == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
        (uint32_t)__cvta_generic_to_shared(s_tm)), "r"(TC));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  for (int i = tid; i < (NB * fl + 8 * H + xfl) / 4; i += nthr)
    *reinterpret_cast<float4 *>(smem + 4 * i) = zero4();
  if (TM) asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (TM) asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  for (int i = tid; i < T.rows * 32; i += nthr) {
    const int r = i >> 5, x = T.x0 + 4 * (i & 31), o = origin + (T.z0 + r) * pitch + x;
    if (x < NX4) {
      if (!kStore) {
        st4(smem + h4 + 4 * i, ld4(S.p[0] + o));
        st4(smem + fl + h4 + 4 * i, ld4(S.p[1] + o));
      }
      if (A.t0 > 0) {  // left by the part before
        st4(smem + B0 * fl + h4 + 4 * i, ld4(S.q[0] + o));
        st4(smem + (B0 + 1) * fl + h4 + 4 * i, ld4(S.q[1] + o));
      }
      if (!TM) st4(s_x + 4 * i, ldg4(S.a + o));
    }
  }
  const int x0 = T.x0 + 4 * lane;
  const bool xok = x0 < NX4;
  const int nrec = S.info->nrec;
  const int src = S.info->src_off;
  const float fsc = S.info->src_rev, rsc = S.info->rec_scale;
  const int2 *cell_rec = S.cell_rec;
  const float *seis_t = S.seis_t, *sa = S.a + origin + T.z0 * pitch + T.x0;
  const int cell = (blockIdx.x - S.tile0) * blockDim.y + w;
  constexpr int K = TIGHT ? 1 : 4;
  Recs<K> rec;
  rec.load(S.cell_ptr, cell_rec, cell, lane, true);
  float rec_a[K], rec_s[K];  // scale * a at the receivers; the record's values, loaded a step ahead
  auto load_s = [&](int row) {
#pragma unroll
    for (int i = 0; i < K; ++i)
      if (rec.id[i] >= 0) rec_s[i] = seis_t[(long long)row * nrec + rec.id[i]];
  };
#pragma unroll
  for (int i = 0; i < K; ++i)
    rec_a[i] = rec.id[i] >= 0 ? rsc * __ldg(sa + (rec.loc[i] / kTileX) * pitch + rec.loc[i] % kTileX) : 0.f;
  load_s((kGrad ? nt + 1 : nt) - A.t0);
  const int row0 = origin + (T.z0 + W.r0) * pitch;
  const bool has_src = src >= row0 + T.x0 && src < row0 + T.x0 + RZ * pitch;
  const int lstep = lane == 0 ? 8 : kTileX, rstep = lane == 31 ? 8 : kTileX;
  const int lofs = lane == 0 ? (int)(s_lr - smem) + W.r0 * 8 : W.r0 * kTileX + 4 * lane - 4;
  const int rofs = lane == 31 ? (int)(s_lr - smem) + W.r0 * 8 + 4 : W.r0 * kTileX + 4 * lane + 4;
  const int own = W.r0 * kTileX + 4 * lane;
  const bool top = W.r0 == 0, last = W.r0 + RZ == H;  // TIGHT: the warps at the tile's edges
  uint32_t tmem = 0;
  std::conditional_t<TM, KeepTm<RZ, MODE>, KeepReg<RZ, MODE>> keep;
  if constexpr (TM) {
    tmem = *s_tm;
    keep.ta = tmem + ((uint32_t)(32 * (w & 3)) << 16) + (uint32_t)((w >> 2) * RZ * 12);
#pragma unroll 1
    for (int j = 0; j < RZ; ++j) {
      const bool in = W.r0 + j < T.rows && xok, sums = in && A.t0 > 0;
      const int o = row0 + j * pitch + x0;
      const float4 av = in ? ldg4(S.a + o) : zero4();
      const float4 n4 = sums ? ld4(S.cnum + o) : zero4(), d4 = sums && !kGrad ? ld4(S.cden + o) : zero4();
      __syncwarp();
      tm_st4(keep.ta + 12 * j, av);
      tm_st4(keep.ta + 12 * j + 4, n4);
      tm_st4(keep.ta + 12 * j + 8, d4);
    }
    keep.flush();
  } else {
    keep.init(s_x, W);
    if (A.t0 > 0) {
#pragma unroll
      for (int j = 0; j < RZ; ++j)
        if (W.r0 + j < T.rows && xok) {
          keep.num[j] = ld4(S.cnum + row0 + j * pitch + x0);
          if constexpr (!kGrad) keep.den[j] = ld4(S.cden + row0 + j * pitch + x0);
        }
    }
  }
  __syncthreads();
  bool ok = true;
  float f_next = has_src && A.t0 > 0 ? A.wav[nt - A.t0] : 0.f;
#pragma unroll 1
  for (int t = A.t0; t != A.t1; ++t) {
    const float f = f_next * fsc;
    if (has_src && t < nt) f_next = A.wav[nt - 1 - t];  // in flight during this step
    // p^R level n; pbar level n (FWI: adjoint level n + 1)
    const int n = nt - t, pr = n & 1, pb = kGrad ? pr ^ 1 : pr;
    const int rc0 = pr * fl + h4, rn0 = (pr ^ 1) * fl + h4, bc0 = (B0 + pb) * fl + h4, bn0 = (B0 + (pb ^ 1)) * fl + h4;
    const bool do_r = !kStore && t > 0 && (kGrad || n > 0), do_b = kGrad || n > 0;
    float4 qa[4];
    if (TIGHT) qa[0] = qa[1] = qa[2] = qa[3] = zero4();
    if (do_r) {
      float *rc = smem + rc0;
      ok = halo_in<RZ, TIGHT>(W, 0, (uint32_t)t, s_lr, rc - h4, TIGHT ? s_x : rc + H * kTileX, qa) && ok;
      sweep<RZ, TIGHT>(W, smem, rc0, rn0, rc + W.r0 * kTileX - 4 * kTileX,
                       TIGHT && last ? s_x : rc + (W.r0 + RZ) * kTileX, top, qa, lofs, lstep, rofs, rstep,
                       [&](int j) { keep.pre_all(j); },
                       [&](int j, const float4 c, const float4 po, const float4 lap) {
                         const float4 cb = lds4(smem + bc0 + own + j * kTileX), av = keep.a(j);
                         float4 inc, v = leap_fin<kGrad>(c, po, av, lap, &inc);
                         if (has_src) {
                           const int d = src - (row0 + j * pitch + x0);
                           if ((unsigned)d < 4u) {
                             point_sub(v, d, cmp(av, d) * f);
                             if (kGrad) point_sub(inc, d, cmp(av, d) * f);
                           }
                         }
                         keep.add(j, kGrad ? inc : c, cb);
                         st4_if(xok, smem + rn0 + own + j * kTileX, v);
                       });
      keep.flush();
    } else if (kStore) {
      if (n % A.stride == 0) {  // Eq. 3 at a kept level
        const int nx = S.ix1 - S.ix0;
        const float *slot = A.store + (long long)(n / A.stride) * nx * (S.iz1 - S.iz0);
#pragma unroll
        for (int j = 0; j < RZ; ++j) {
          if (W.r0 + j >= W.rows) break;
          const int z = T.z0 + W.r0 + j;
          float v[4];
#pragma unroll
          for (int e = 0; e < 4; ++e)
            v[e] = z >= S.iz0 && z < S.iz1 && x0 + e >= S.ix0 && x0 + e < S.ix1
                       ? slot[(long long)(z - S.iz0) * nx + x0 + e - S.ix0] : 0.f;
          __syncwarp();
          keep.pre_all(j);
          keep.a(j);
          keep.add(j, make_float4(v[0], v[1], v[2], v[3]), lds4(smem + bc0 + own + j * kTileX));
        }
        keep.flush();
      }
    } else if (!kGrad) {
#pragma unroll
      for (int j = 0; j < RZ; ++j) {
        if (W.r0 + j >= W.rows) break;
        keep.pre_all(j);
        keep.a(j);
        keep.add(j, lds4(smem + rc0 + own + j * kTileX), lds4(smem + bc0 + own + j * kTileX));
      }
      keep.flush();
    }
    __syncwarp();
    if (!kStore && t < nt) halo_out<RZ>(W, 0, (uint32_t)t + 1, smem + rn0);
    if (do_b) {
      float *bc = smem + bc0, *bn = smem + bn0;
      // (level nt is zero everywhere, as the words are before the first)
      ok = halo_in<RZ, TIGHT>(W, FB, (uint32_t)t, s_lr, bc - h4, TIGHT ? s_x : bc + H * kTileX, qa) && ok;
      sweep<RZ, TIGHT>(W, smem, bc0, bn0, bc + W.r0 * kTileX - 4 * kTileX,
                       TIGHT && last ? s_x : bc + (W.r0 + RZ) * kTileX, top, qa, lofs, lstep, rofs, rstep,
                       [&](int j) { keep.pre_a(j); },
                       [&](int j, const float4 c, const float4 po, const float4 lap) {
                         const float4 v = leap_fin<false>(c, po, keep.a(j), lap, nullptr);
                         st4_if(xok, bn + own + j * kTileX, v);
                       });
      __syncwarp();
      if (rec.end > rec.beg) {
#pragma unroll
        for (int i = 0; i < K; ++i)
          if (rec.id[i] >= 0) atomicAdd(bn + rec.loc[i], rec_a[i] * rec_s[i]);
        const int r = kGrad ? n + 1 : n;  // row of the record
        for (int k = rec.beg + 32 * K + lane; k < rec.end; k += 32) {
          const int2 c = __ldg(cell_rec + k);
          const float av = __ldg(sa + (c.x / kTileX) * pitch + c.x % kTileX);
          atomicAdd(bn + c.x, rsc * av * __ldg(seis_t + (long long)r * nrec + c.y));
        }
        load_s(r - 1);
        __syncwarp();
      }
      if (t < nt) halo_out<RZ>(W, FB, (uint32_t)t + 1, bn);
    }
    if (__syncthreads_or(!ok)) {
      if (tid == 0) give_up(A);
      break;
    }
  }
  // outputs (not after a wait that gave up)
#pragma unroll
  for (int j = 0; j < RZ; ++j) {
    const int z = T.z0 + W.r0 + j;
    float4 n4, d4;
    __syncwarp();  // (the row before ended with lanes that had nothing to write)
    keep.sums(j, n4, d4);
    if (!ok || W.r0 + j >= W.rows) continue;
    if (A.t1 <= nt) {  // another part follows
      if (xok) {
        const int o = row0 + j * pitch + x0;
        const float *b = smem + h4 + own + j * kTileX;
        if (!kStore) {
          st4(S.p[0] + o, lds4(b));
          st4(S.p[1] + o, lds4(b + fl));
        }
        st4(S.q[0] + o, lds4(b + B0 * fl));
        st4(S.q[1] + o, lds4(b + (B0 + 1) * fl));
        st4(S.cnum + o, n4);
        if (!kGrad) st4(S.cden + o, d4);
      }
      continue;
    }
    if (z < S.iz0 || z >= S.iz1) continue;
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int x = x0 + e;
      if (x < S.ix0 || x >= S.ix1) continue;
      const long long o = A.dense ? (long long)(z - S.iz0) * (S.ix1 - S.ix0) + x - S.ix0
                                  : (long long)(row0 + j * pitch + x);
      S.num[o] = A.overwrite ? cmp(n4, e) : S.num[o] + cmp(n4, e);
      if (!kGrad) S.den[o] = A.overwrite ? cmp(d4, e) : S.den[o] + cmp(d4, e);
    }
  }
  if (TM) {
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (w == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TC));
  }
}

// ----------------------------------------------------------- host side ----
inline int cdiv(int a, int b) { return (a + b - 1) / b; }

struct Variant {
  int rz, maxw;
  bool tight, tm;
  const void *fn[4];  // forward, imaging, FWI gradient, storage
};
#define RBC_RES_VARIANT(RZ, MAXW, TIGHT, TM)                                                                 \
  {RZ, MAXW, TIGHT, TM,                                                                                      \
   {(const void *)k_res_fwd<RZ, MAXW>, (const void *)k_res_rev<RZ, MAXW, TIGHT, TM, 0>,                \
    (const void *)k_res_rev<RZ, MAXW, TIGHT, TM, 1>, (const void *)k_res_rev<RZ, MAXW, TIGHT, TM, 2>}}
// Rows per warp, most warps per block, layout; one block per SM.  res_plan takes
// the first that holds the grid: with few rows per warp a step is short (300 x
// 300 forward: 1.6 / 1.9 / 2.5 / 2.8 / 3.1 us with 1 / 2 / 4 / 7 / 10 rows),
// and as few warps as fit, which spreads the grid over the SMs (1500 x 800 forward +
// reverse: 9.3 us with 10 warps of 7 rows, 11.2 with 15), but eight at least with
// one or two rows (300 x 300: 1.52 us with 8, 1.72 with 6).  Blocks of 8 warps, two to
// an SM, left some SMs two and some one: forward / RTM step of 400 x 400 1.79 / 5.40 us against
// 1.58 / 4.71 now, 700 x 500 2.05 / 5.74 against 1.90 / 5.54.  The last is the
// tallest tile whose four buffers fit 227 KB: TIGHT keeps no halo rows in them.
const Variant kVariants[] = {
    RBC_RES_VARIANT(1, 16, false, false), RBC_RES_VARIANT(2, 16, false, false),
    RBC_RES_VARIANT(4, 16, false, true), RBC_RES_VARIANT(7, 16, true, true),
    RBC_RES_VARIANT(10, 11, true, true),
};

size_t res_smem(int dir, int H, const Variant &V) {
  const int nb = dir == kResRev ? 4 : 2;  // field buffers
  size_t rows;
  if (dir == kResFwd) rows = 2 * (H + 8) + H;
  else rows = V.tight ? nb * H + 4 : nb * (H + 8) + (V.tm ? 0 : H);
  const size_t need = sizeof(float) * (rows * kTileX + 8 * (size_t)H) + (dir != kResFwd && V.tm ? 16 : 0);
  // More than half an SM's shared memory keeps a second loop's block off it.  Loops in flight together otherwise land
  // on the same SMs while others idle (four shots of 300 x 300 at once: 3.6 -> 2.4 us a step;
  // one shot of 2301 x 751: 3.64 -> 3.42), and two loops whose blocks share SMs could each hold tensor memory that
  // the other waits for.
  return std::max(need, (size_t)116 * 1024);
}

} // namespace

bool res_plan(const Lay *L, int nshots, int dir, int share, ResPlan *out) {
  out->variant = -1;
  const char *env = getenv("RBC_RESIDENT");  // 0: one launch per step
  if (env && env[0] == '0') return false;
  int dev = 0, sms = 0, maxsm = 0, coop = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&maxsm, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) != cudaSuccess || !coop) {
    cudaGetLastError();
    return false;
  }
  int force_v = -1, force_w = -1;
  if (const char *e = getenv("RBC_RES_TILE")) sscanf(e, "%d,%d", &force_v, &force_w);
  int best_v = -1, best_w = 0;
  for (int v = 0; best_v < 0 && v < (int)(sizeof kVariants / sizeof kVariants[0]); ++v) {
    const Variant &V = kVariants[v];
    int nzmax = 1;
    for (int s = 0; s < nshots; ++s) nzmax = std::max(nzmax, L[s].NZ);
    // the lowest tiles that fit; with one or two rows per warp at least eight warps
    const int top = std::min(V.maxw, std::max(cdiv(nzmax, V.rz), cdiv(4, V.rz)));
    for (int nw = V.rz < 4 && force_w <= 0 ? std::min(8, top) : 1; best_v < 0 && nw <= top; ++nw) {
      if (force_v >= 0 && (v != force_v || (force_w > 0 && nw != force_w))) continue;
      const int H = nw * V.rz;
      if (H < 4) continue;
      const size_t sm = res_smem(dir, H, V);
      if (sm > (size_t)maxsm) continue;
      long long blocks = 0;
      for (int s = 0; s < nshots; ++s) blocks += (long long)cdiv(L[s].NX, kTileX) * cdiv(L[s].NZ, H);
      if (blocks * share > sms) continue;  // (one block per SM: no need to ask the runtime)
      int per = 1 << 20;
      for (int f = dir == kResStore ? 3 : dir; f <= (dir == kResRev ? 2 : dir == kResStore ? 3 : 0); ++f) {
        const void *fn = V.fn[f];
        int k = 0;
        // the limit is raised to the device's for every plan alike: contexts on other threads share it
        if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, maxsm) != cudaSuccess ||
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&k, fn, 32 * nw, sm) != cudaSuccess)
          k = 0;
        per = std::min(per, k);
      }
      if (blocks * share <= (long long)per * sms) best_v = v, best_w = nw;
    }
  }
  cudaGetLastError();
  if (best_v < 0) return false;
  const Variant &V = kVariants[best_v];
  out->variant = best_v;
  out->rz = V.rz;
  out->warps = best_w;
  out->H = best_w * V.rz;
  out->smem = res_smem(dir, out->H, V);
  // A loop holds its SMs: a kernel on another stream that needs them starts where a part ends, so a part takes some
  // two milliseconds, by the estimates of res_plan_shared.  (A denoiser call beside a survey shot waited 15 ms, a
  // whole loop; 1.8 ms with such parts.)  A part costs 5 us on 300 x 300 (reverse 7) and 11 on 2421 x 871, for the
  // fields to global memory and back; the survey's reverse loop gains 3 % by them.
  const int r = V.rz * cdiv(best_w, 4);
  const char *est = getenv("RBC_RES_STEPS");
  out->steps = est && atoi(est) > 0 ? atoi(est) : (int)(2000 / (dir == kResRev ? 2.6 + 0.15 * r : 1.5 + 0.075 * r));
  out->tiles.clear();
  out->tile0.assign(1, 0);
  for (int s = 0; s < nshots; ++s) {
    const int gx = cdiv(L[s].NX, kTileX), gz = cdiv(L[s].NZ, out->H), t0 = (int)out->tiles.size();
    for (int bz = 0; bz < gz; ++bz)
      for (int bx = 0; bx < gx; ++bx) {
        const int i = t0 + bz * gx + bx;
        ResTile T;
        T.shot = s;
        T.x0 = bx * kTileX;
        T.z0 = bz * out->H;
        T.rows = std::min(out->H, L[s].NZ - T.z0);
        T.up = bz > 0 ? i - gx : -1;
        T.dn = bz + 1 < gz ? i + gx : -1;
        T.lf = bx > 0 ? i - 1 : -1;
        T.rt = bx + 1 < gx ? i + 1 : -1;
        out->tiles.push_back(T);
      }
    out->tile0.push_back((int)out->tiles.size());
  }
  out->blocks = (int)out->tiles.size();
  return true;
}

// Several loops of a grid at a time, each on its own stream.  Side by side each has fewer blocks, taller tiles and a
// longer step; loops that do not fit together follow one another; and with one launch per step the loops fill each
// other's gaps.  The way that is through first is taken, by these estimates of a step of all k loops (us; measured
// forward and forward + reverse for 1 to 6 loops of 200 x 200 to 2421 x 871): resident 1.5 + 0.075 r, reverse 2.6 +
// 0.15 r, with r the rows on the fullest of an SM's four schedulers; by launches 2.3 + 0.2 k + 1.3 M or 2.3 k M,
// reverse 3.9 + 0.3 k + 3.3 M or 5.5 k M (6.7 where the fields leave L2), for M million nodes.  Steps are taken where
// they are a fifth quicker: a context's first call by steps makes its graphs (5 us per step).
// Four loops of 400 x 400 take 2.42 / 6.52 us so (forward / both), 6.09 / 17.77 with the whole device each and
// 3.45 / 9.47 by launches; three of 1100 x 700 6.6 / 18.5 in turn, 7.3 / 22.6 as two and one, 5.4 / 17.4 by launches; two of
// 2421 x 871 7.05 / 21.3 in turn, 8.8 / 36.4 by launches.
bool res_plan_shared(const Lay *L, int nshots, int dir, int loops, bool steps, ResPlan *out) {
  if (loops == 1) return res_plan(L, nshots, dir, 1, out);
  int dev = 0, sms = 1;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  out->variant = -1;
  const bool rev = dir == kResRev;
  double best = 1e30;
  if (steps) {
    const double m = 1e-6 * L->NX * L->NZ, km = loops * m;
    best = 1.25 * (rev ? std::max(3.9 + 0.3 * loops + 3.3 * m, (km > 3.3 ? 6.7 : 5.5) * km)
                       : std::max(2.3 + 0.2 * loops + 1.3 * m, 2.3 * km));
  }
  for (int j = 1; j <= std::min(loops, 16); ++j) {  // (plans for a sixteenth of the device leave room for more)
    ResPlan P;
    if (!res_plan(L, nshots, dir, j, &P)) break;
    const int r = P.rz * cdiv(P.warps, 4);
    const double t = cdiv(loops, sms / P.blocks) * (rev ? 2.6 + 0.15 * r : 1.5 + 0.075 * r);
    if (t < 0.98 * best) best = t, *out = P;  // (with nothing in it, the shorter steps)
  }
  return out->variant >= 0;
}

// A warp records what its registers do not hold in turns of 32, each a table read from L2 behind its sweep: a step of
// 1100 x 700 takes 2.4 us with 1100 receivers, 6.0 with 86 k (22 more per warp), 10.3 with 193 k (90 more) and 35 with
// every node; by launches, whose blocks hide the reads behind one another, 3.7, 6.4, 10.0 and 30.  (2421 x 871: 9.4
// against 10.3 with 132 k receivers, 26.9 against 24.1 with 528 k.)
bool res_many_receivers(const ResPlan &P, int nrec) {
  return nrec > (64 + 32LL * rec_regs(P.rz)) * P.blocks * P.warps;
}

size_t res_ll_bytes(const ResPlan &P, int dir) {
  return sizeof(u64) * ((size_t)P.blocks * (dir == kResRev ? 2 : 1) * 2 * ll_words(P.H) + 2);  // (words, then the mark)
}

size_t res_ll_bound(const Lay *L, int nshots, int nf) {
  int dev = 0, sms = 0, hmax = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  for (const Variant &V : kVariants) hmax = std::max(hmax, V.maxw * V.rz);
  // ll_words(H) per block; a shot's blocks * H <= gx * (NZ + H - 1)
  long long blocks = 0, rows = 0;
  for (int s = 0; s < nshots; ++s) {
    const long long gx = cdiv(L[s].NX, kTileX);
    blocks += gx * cdiv(L[s].NZ, 4);
    rows += gx * (L[s].NZ + hmax - 1);
  }
  return sizeof(u64) * (nf * 2 * (size_t)(std::min((long long)sms / 2, blocks) * 2 * kEdge + 8 * rows) + 2);
}

namespace {
// The contexts and batches with resident loops that are alive, and the number of their calls so far.
struct Flight {
  std::mutex m;
  std::vector<LoopUser *> live;
  unsigned long long calls = 0;
};
Flight &flight() {
  static Flight *f = new Flight();  // (outlives what is destroyed at exit)
  return *f;
}
}

void flight_add(LoopUser *u) {
  Flight &f = flight();
  std::lock_guard<std::mutex> lock(f.m);
  cudaGetDevice(&u->dev);
  u->born = f.calls;
  f.live.push_back(u);
}

void flight_remove(LoopUser *u) {
  Flight &f = flight();
  std::lock_guard<std::mutex> lock(f.m);
  f.live.erase(std::remove(f.live.begin(), f.live.end(), u), f.live.end());
}

// Users whose loops may run beside this call's, itself included: those called on other streams since its own last
// call.  A program that runs k contexts on k streams calls the others in between; one that uses its contexts in turn
// on one stream, or one context at a time, is counted as one.  At its first call (on a stream of the caller's making)
// users that have not been called yet count too, so that a first round of calls runs side by side as well.
// Nothing but the plan depends on the count.
int flight_count(LoopUser *u, cudaStream_t s) {
  unsigned long long id = 0;
  if (cudaStreamGetId(s, &id) != cudaSuccess) {
    cudaGetLastError();
    return 1;
  }
  Flight &f = flight();
  std::lock_guard<std::mutex> lock(f.m);
  std::vector<unsigned long long> seen(1, id);
  int n = 1;
  for (const LoopUser *x : f.live) {
    if (x == u || x->dev != u->dev) continue;
    if (!x->called) {
      n += !u->called && s != nullptr && s != cudaStreamLegacy;
    } else if (x->called > std::max(u->called, u->born) &&
               std::find(seen.begin(), seen.end(), x->on_stream) == seen.end()) {
      seen.push_back(x->on_stream);
      ++n;
    }
  }
  u->called = ++f.calls;
  u->on_stream = id;
  return n;
}

namespace {
std::atomic<bool> g_fail_alloc{false};
}

cudaError_t res_malloc(void **p, size_t bytes) {
  return g_fail_alloc.exchange(false) ? cudaErrorMemoryAllocation : cudaMalloc(p, bytes);
}

void res_fail_alloc(bool on) { g_fail_alloc = on; }

void res_cell(const ResPlan &P, const Lay &L, int x, int z, int *cell, int *loc) {
  const int t = (z / P.H) * cdiv(L.NX, kTileX) + x / kTileX, r = z % P.H;
  *cell = t * P.warps + r / P.rz;
  *loc = r * kTileX + x % kTileX;
}

void res_cells(const ResPlan &P, const Lay &L, int cells, int nrec, const int *rec, int base, int *ptr, int2 *out) {
  std::vector<int> cell(nrec), loc(nrec), fill(cells + 1, 0);
  for (int r = 0; r < nrec; ++r) {
    res_cell(P, L, rec[3 * r], rec[3 * r + 2], &cell[r], &loc[r]);
    ++fill[cell[r] + 1];
  }
  for (int k = 0; k < cells; ++k) fill[k + 1] += fill[k];
  for (int k = 0; k <= cells; ++k) ptr[k] = base + fill[k];
  for (int r = 0; r < nrec; ++r) out[fill[cell[r]]++] = make_int2(loc[r], r);
}

// Every variant's tiles, first-fit by falling tile count; the variant whose
// groups take the least time in all is kept.  Time of a forward and a reverse
// step by rows per warp, measured on grids that fill the device (us).
std::vector<std::vector<int>> res_groups(const Lay *L, int nshots) {
  const double step_us[] = {4.4, 5.5, 7.3, 9.4, 11.0};
  int dev = 0, sms = 0, maxsm = 0;
  std::vector<std::vector<int>> best;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&maxsm, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return best;
  std::vector<int> order(nshots);
  for (int i = 0; i < nshots; ++i) {
    ResPlan f, r;
    if (!res_plan(L + i, 1, kResFwd, 1, &f) || !res_plan(L + i, 1, kResRev, 1, &r)) return best;
    order[i] = i;
  }
  double best_us = 1e30;
  for (int v = 0; v < (int)(sizeof kVariants / sizeof kVariants[0]); ++v) {
    const Variant &V = kVariants[v];
    const int cap = sms;
    int hmax = V.maxw * V.rz;
    while (hmax > V.rz && res_smem(kResRev, hmax, V) > (size_t)maxsm) hmax -= V.rz;
    std::vector<int> tiles(nshots);
    bool fits = true;
    for (int i = 0; i < nshots; ++i) {
      tiles[i] = cdiv(L[i].NX, kTileX) * cdiv(L[i].NZ, hmax);
      fits = fits && tiles[i] <= cap;
    }
    if (!fits) continue;
    std::sort(order.begin(), order.end(), [&](int a, int b) { return tiles[a] != tiles[b] ? tiles[a] > tiles[b] : a < b; });
    std::vector<std::vector<int>> g;
    std::vector<int> room;
    for (int i : order) {
      size_t k = 0;
      while (k < g.size() && room[k] < tiles[i]) ++k;
      if (k == g.size()) {
        g.push_back({});
        room.push_back(cap);
      }
      g[k].push_back(i);
      room[k] -= tiles[i];
    }
    if (g.size() * step_us[v] < best_us) best_us = g.size() * step_us[v], best = g;
  }
  return best;
}

cudaError_t res_launch(const ResPlan &P, int dir, const ResArgs &A, cudaStream_t s, long long *launches,
                       bool withhold) {
  const Variant &V = kVariants[P.variant];
  const void *fn = V.fn[dir == kResStore ? 3 : dir == kResRev && A.grad ? 2 : dir];
  cudaError_t e = cudaMemsetAsync(A.ll, 0, res_ll_bytes(P, dir), s);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(P.blocks);
  cfg.blockDim = dim3(32, P.warps);
  cfg.dynamicSmemBytes = P.smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  ResArgs a = A;
  a.gave_up = reinterpret_cast<int *>(A.ll + res_ll_bytes(P, dir) / sizeof(u64) - 2);
  int H = P.H;
  void *args[2] = {&a, &H};
  const int n = dir == kResFwd ? A.nt : A.nt + 1, parts = res_parts(P, n);
  for (int k = withhold && parts > 1 ? 1 : 0; k < parts && e == cudaSuccess; ++k) {
    a.t0 = (int)((long long)n * k / parts);
    a.t1 = (int)((long long)n * (k + 1) / parts);
    e = cudaLaunchKernelExC(&cfg, fn, args);
    if (e == cudaSuccess) ++*launches;
  }
  return e;
}

} // namespace rbc
