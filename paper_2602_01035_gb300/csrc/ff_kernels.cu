// ff_kernels.cu - sm_103a kernels of the FUSE-Flow per-frame fusion path.
//
// Launch sequence of one frame (all on the caller's stream; from the level step on,
// optionally as programmatic dependent launches, see pdl_release / pdl_wait):
//   screen   (only with a depth screen set) D^r of Eq. 8 into the context's buffers
//   count    (a) decode + gate (Eq. 9) of units of 32x8 pixels, a warp each; the gated pixels are
//            listed, back-projected (Eq. 8) and counted per coarse cell (Sec. II.5(1)c); per-block
//            pixel counts and extent (Sec. II.5(1)b)
//   levels   level of each coarse cell (Sec. II.5(1)d) and its range of 8^level dense
//            cell slots
//   weigh    per listed pixel: (b) consistency V (Eq. 4-7) on the rig's grid, omega = C V (Eq. 10)
//            as mantissa/exponent; (c) cell key (Sec. II.5(1)e) and dense slot; per cell its
//            representative (Sec. II.5(2)a) and smallest weight exponent
//   sum      (d) exact fixed-point sums of omega, omega P, omega RGB per cell (Eq. 11) at the scale
//            of its smallest exponent; the representatives are marked, the coarse entries cleared
//            (top-k variant: k_assign_topk keeps each tile's most confident members of a cell
//            instead of weigh, and k_reduce_topk weighs and fuses each cell's k instead of sum)
//   emit     ranks of the representatives (output order), Eq. 11 from each cell's sums, output and
//            frame statistics; the used slots, the bitmap and the counters are cleared for the next
//            frame
// Outside the frame sequence: k_copyout (served frames: cloud into pinned host memory),
// k_mc (the multi-camera depth consistency error of Eq. 12 on a point set), k_confidence
// (Eq. 3 confidence from depth) and the stand-alone depth screen.
//
// Every reduction of the frame is order-independent (integer counts, max, min and
// fixed-point sums), so its output is bitwise reproducible.
#include <algorithm>
#include <atomic>
#include <climits>
#include <cmath>
#include <cstring>
#include <cstdint>

#include "ff_internal.h"

namespace ffl {

namespace {

constexpr int kThreads = 256;
constexpr int kTileW = 32;                        // tiles: 32 columns by TH rows
constexpr int kMaxProbe = 1 << 14;
constexpr float kLn2H = 0.693147182464599609375f;         // float(ln 2)
constexpr float kLn2L = -1.904654299957768e-09f;          // ln 2 - kLn2H
constexpr float kInvLn2 = 1.44269504088896340736f;

// ------------------------------------------------------------------ global hash tables
__device__ __forceinline__ unsigned coarse_slot(unsigned long long key, unsigned cmask) {
  return coarse_hash((int)((key >> 40) & 0xfffff), (int)((key >> 20) & 0xfffff), (int)(key & 0xfffff)) & cmask;
}
// n points of coarse cell (x, y, z) (Sec. II.5(1)c) into the table; its position there.  Called by whole
// warps, lanes without a cell (`act` false) too: the warp's new cells take their places in the list of used
// positions with one atomic, as one each on the same counter takes about 1 ns a cell.
__device__ __forceinline__ unsigned count_cell(const Tables& t, bool act, int x, int y, int z, unsigned n) {
  const int lane = threadIdx.x & 31;
  unsigned slot = kSlotNone;
  bool fresh = false;
  if (act) {
    const unsigned long long key = pack_key(0, x, y, z);
    unsigned h = coarse_slot(key, t.cmask);
    for (int probe = 0; probe < kMaxProbe; ++probe) {
      // most keys are there already: a look first keeps their lines free of serialised swaps
      unsigned long long cur = __ldcg(&t.coarse[h].key);
      if (cur == kKeyEmpty) {
        cur = atomicCAS(&t.coarse[h].key, kKeyEmpty, key);
        fresh = cur == kKeyEmpty;
      }
      if (cur == key || fresh) {
        slot = h;
        break;
      }
      h = (h + 1) & t.cmask;
    }
    if (slot != kSlotNone)
      atomicAdd(&t.coarse[slot].count, n);
    else
      atomicOr(&t.cnt->error, kErrCoarseFull);
  }
  const unsigned m = __ballot_sync(0xffffffffu, fresh);
  if (m != 0u) {
    unsigned first = 0;
    if (lane == 0) first = atomicAdd(&t.cnt->n_coarse, (unsigned)__popc(m));
    first = __shfl_sync(0xffffffffu, first, 0) + (unsigned)__popc(m & ((1u << lane) - 1u));
    if (fresh && first <= t.cmask) t.cused[first] = slot;
  }
  return slot;
}

// One point each of K cells a lane (key kKeyEmpty: none), for whole warps: the K places are tried together,
// each at once with a swap.
template <int K>
__device__ __forceinline__ void count_points(const Tables& t, const unsigned long long (&key)[K]) {
  unsigned h[K], pending = 0, fresh = 0;
#pragma unroll
  for (int k = 0; k < K; ++k) {
    h[k] = coarse_slot(key[k], t.cmask);
    pending |= key[k] != kKeyEmpty ? 1u << k : 0u;
  }
#pragma unroll 1
  for (int probe = 0; probe < kMaxProbe && pending; ++probe) {
    unsigned long long old[K];
#pragma unroll
    for (int k = 0; k < K; ++k)
      if ((pending >> k) & 1u) old[k] = atomicCAS(&t.coarse[h[k]].key, kKeyEmpty, key[k]);
#pragma unroll
    for (int k = 0; k < K; ++k)
      if ((pending >> k) & 1u) {
        if (old[k] == kKeyEmpty) fresh |= 1u << k;
        if (old[k] == kKeyEmpty || old[k] == key[k]) {
          pending &= ~(1u << k);
          atomicAdd(&t.coarse[h[k]].count, 1u);
        } else {
          h[k] = (h[k] + 1) & t.cmask;
        }
      }
  }
  if (pending) atomicOr(&t.cnt->error, kErrCoarseFull);
  __syncwarp();
  const int lane = threadIdx.x & 31;
  const unsigned mine = (unsigned)__popc(fresh);
  unsigned sum = mine;                                               // of the lanes up to this one
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned v = __shfl_up_sync(0xffffffffu, sum, o);
    if (lane >= o) sum += v;
  }
  const unsigned total = __shfl_sync(0xffffffffu, sum, 31);
  if (total == 0u) return;
  unsigned at = 0;
  if (lane == 0) at = atomicAdd(&t.cnt->n_coarse, total);
  at = __shfl_sync(0xffffffffu, at, 0) + sum - mine;
#pragma unroll
  for (int k = 0; k < K; ++k)
    if ((fresh >> k) & 1u) {
      if (at <= t.cmask) t.cused[at] = h[k];
      ++at;
    }
}

// Level and slot base (packed level << 27 | base) of an existing coarse key.
__device__ __forceinline__ unsigned coarse_lvbase(const Tables& t, unsigned long long key) {
  unsigned h = coarse_slot(key, t.cmask);
  for (int probe = 0; probe < kMaxProbe; ++probe) {
    const ulonglong2 e = __ldcg(reinterpret_cast<const ulonglong2*>(&t.coarse[h]));
    if (e.x == key) return (unsigned)(e.y >> 32);
    if (e.x == kKeyEmpty) break;
    h = (h + 1) & t.cmask;
  }
  atomicOr(&t.cnt->error, kErrCoarseMiss);
  return kBaseNone;
}

// Programmatic dependent launch between the kernels of one frame: each kernel lets the next
// one start launching as soon as all of its own blocks are running (pdl_release), and a
// kernel waits for the previous one to complete, its memory visible, before it touches
// anything that one (or any earlier kernel of the frame) wrote (pdl_wait).  Outside such a
// launch both are no-ops.
__device__ __forceinline__ void pdl_release() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Frame of a block of a one-dimensional grid that concatenates the frames' blocks
// (first[f] = the frame's first block), and the block's index within its frame.
template <int NB>
__device__ __forceinline__ int batch_frame(const int (&first)[NB + 1], int n, int b, int& local) {
  int f = 0;
#pragma unroll
  for (int k = 1; k < NB; ++k)
    if (k < n && b >= first[k]) f = k;
  local = b - first[f];
  return f;
}
// Frame of a block of a grid whose y dimension runs over the frames.
template <int NB>
__device__ __forceinline__ int batch_frame_y() { return NB == 1 ? 0 : (int)blockIdx.y; }

// Sec. II.5(1)d for every coarse cell once all counts are in: its level l and a range of
// 8^l dense cell slots.  Ranges are claimed with one atomic per warp (an inclusive scan of
// the sizes inside the warp), so their placement depends on scheduling; no result does.
template <int NB>
__global__ void __launch_bounds__(kThreads) k_levels(const __grid_constant__ BatchArgs<NB> args) {
  const Tables& t = args.f[batch_frame_y<NB>()].t;
  pdl_release();
  pdl_wait();
  const unsigned n_coarse = min(t.cnt->n_coarse, t.cmask + 1u);
  const int lane = threadIdx.x & 31;
  const unsigned long long cap = t.max_slots;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < t.n_wblocks; i += gridDim.x * blockDim.x) t.bsum[i] = 0u;
  if (blockIdx.x == 0 && threadIdx.x == 0) t.cnt->n_cells = 0u;      // the last frame's
  for (unsigned base = blockIdx.x * blockDim.x; base < n_coarse; base += gridDim.x * blockDim.x) {
    const unsigned i = base + threadIdx.x;
    unsigned cs = 0, l = 0;
    unsigned long long size = 0;
    if (i < n_coarse) {
      cs = t.cused[i];
      l = (unsigned)level_for(t.coarse[cs].count, t.n_min, t.max_level);
      size = min(1ull << (3 * l), cap + 1ull);           // 8^l, clamped: never fits then
    }
    unsigned long long x = size;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned long long y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    unsigned long long wbase = 0;
    if (lane == 31 && x) wbase = atomicAdd(&t.cnt->n_slots, x);
    wbase = __shfl_sync(0xffffffffu, wbase, 31);
    if (i < n_coarse) {
      const unsigned long long b = wbase + x - size;
      const bool fits = b + size <= cap;
      t.coarse[cs].lvbase = (l << 27) | (fits ? (unsigned)b : kBaseNone);
      if (!fits) atomicOr(&t.cnt->error, kErrSlots);
    }
  }
}

// Block-local open addressing of dense cell slots (shared memory, Fibonacci hash); returns the table
// position or -1, and sets `fresh` when this call inserted the slot.
template <int TS>
__device__ __forceinline__ int local_pos(unsigned* tab, unsigned key, bool& fresh) {
  constexpr int kBits = TS == 512 ? 9 : TS == 1024 ? 10 : TS == 2048 ? 11 : 0;
  static_assert(kBits > 0, "block table size");
  unsigned h = (key * 0x9E3779B1u) >> (32 - kBits);
  fresh = false;
  for (int probe = 0; probe < TS; ++probe) {
    const unsigned cur = *static_cast<volatile unsigned*>(&tab[h]);
    if (cur == key) return (int)h;
    if (cur == kSlotNone) {
      const unsigned prev = atomicCAS(&tab[h], kSlotNone, key);
      fresh = prev == kSlotNone;
      if (fresh || prev == key) return (int)h;
    }
    h = (h + 1) & (TS - 1);
  }
  return -1;
}

// ------------------------------------------------------------------ Eq. 4-7 per point
// Exact floor(u + 1/2) for u = fx a_x / a_z + cx near a tie at integer r (a_z > 0):
// u + 1/2 >= r  <=>  fx a_x + (cx + 1/2 - r) a_z >= 0, evaluated in double-float.
__device__ __forceinline__ int exact_round(float fh, float fl, float ch, float cl, float axh,
                                           float axl, float azh, float azl, float r) {
  float p1, e1, c0, ce, p2, e2, s, q;
  two_prod(fh, axh, p1, e1);
  e1 = __fmaf_rn(fh, axl, __fmaf_rn(fl, axh, e1));
  two_sum(ch, __fsub_rn(0.5f, r), c0, ce);
  ce = __fadd_rn(ce, cl);
  two_prod(c0, azh, p2, e2);
  e2 = __fmaf_rn(c0, azl, __fmaf_rn(ce, azh, e2));
  two_sum(p1, p2, s, q);
  const float f = __fadd_rn(s, __fadd_rn(__fadd_rn(e1, e2), q));
  return (f >= 0.0f) ? (int)r : (int)r - 1;
}

// Pair rays of a tile of TH rows staged in shared memory (pixel (lx, ly) of the tile): the
// tile's column group, then its row groups (layout: kPrayColGroup, kPrayRowGroup).
template <int TH>
struct TilePairRays {
  const float4* a4;
  const float2* a2;
  const float4* b4;
  const float2* b2;
  __device__ __forceinline__ TilePairRays(const float4* s_cols, const float4* s_rows, int k1, int lx, int ly)
      : a4(s_cols + lx), a2(reinterpret_cast<const float2*>(s_cols + 32) + lx) {
    const float4* rows = s_rows + (ly >> 3) * k1 * kPrayRowGroup;
    b4 = rows + (ly & 7);
    b2 = reinterpret_cast<const float2*>(rows + 8) + (ly & 7);
  }
  __device__ __forceinline__ void operator()(int q, float4& a, float2& al, float4& b, float2& bl) const {
    a = a4[q * kPrayColGroup];
    al = a2[q * 2 * kPrayColGroup];
    b = b4[q * kPrayRowGroup];
    bl = b2[q * 2 * kPrayRowGroup];
  }
};

// Pair rays read from the global tables: pixel (x, y) of a camera of width W whose rays start
// at pray.
struct GlobalPairRays {
  const float4* cols;
  const float4* rows;
  int ix, iy;
  __device__ __forceinline__ GlobalPairRays(const float4* pray, int W, int k1, int x, int y)
      : cols(pray + (long long)(x >> 5) * k1 * kPrayColGroup),
        rows(pray + ((long long)((W + 31) >> 5) * kPrayColGroup + (long long)(y >> 3) * kPrayRowGroup) * k1),
        ix(x & 31), iy(y & 7) {}
  __device__ __forceinline__ void operator()(int q, float4& a, float2& al, float4& b, float2& bl) const {
    const float4* c = cols + q * kPrayColGroup;
    const float4* r = rows + q * kPrayRowGroup;
    a = __ldg(c + ix);
    al = __ldg(reinterpret_cast<const float2*>(c + 32) + ix);
    b = __ldg(r + iy);
    bl = __ldg(reinterpret_cast<const float2*>(r + 8) + iy);
  }
};

__device__ __forceinline__ float rcp_approx(float v) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v));
  return r;
}

// Nearest pixel floor(u + 1/2) along one axis from the float32 estimate u5 of u + 1/2 (out-of-range
// and non-finite estimates give an index outside every image).  The estimate's error is below
// (W + |c|) 2^-21 (six float32 roundings of u - c and the rounding of c + 1/2), half of the view's
// band; inside the band the pixel is decided exactly.
template <bool Y>
__device__ __forceinline__ int nearest_pixel(float u5, float band, const CamDev* J, float ah, float al,
                                             float azh, float azl) {
  const float t = __fadd_rn(u5, kGridM);
  const float r = __fsub_rn(t, kGridM), d = __fsub_rn(u5, r);
  int p = __float_as_int(t) - kGridBits - (d < 0.0f ? 1 : 0);
  if (fabsf(d) < band) {
    fast_two_sum(ah, al, ah, al);
    fast_two_sum(azh, azl, azh, azl);
    p = Y ? exact_round(J->fyh, J->fyl, J->cyh, J->cyl, ah, al, azh, azl, r)
          : exact_round(J->fxh, J->fxl, J->cxh, J->cxl, ah, al, azh, azl, r);
  }
  return p;
}

// Sum over the K-1 neighbour views of d_ij^2 (Eq. 6) in grid units^2, as ff (sh, sl): the general
// evaluation in double-float for depths of any size.  A pixel at z-depth z; the transform into view
// j (Eq. 4) uses the pixel's separable pair rays, a = z (A(x) + B(y)) + t_ji.
template <typename DT>
__device__ __noinline__ void residual_general(const BlockConst* bc, int k1, const RigDev* rig,
                                              GlobalPairRays prays, const float2* __restrict__ rays,
                                              const FramePtrs* fp, float z, float* res, int* views) {
  float sh = 0.0f, sl = 0.0f;
  int nview = 0;
  const float ginv = rig->hot.ginv;
  for (int q = 0; q < k1; ++q) {
    const ViewHot& V = bc->view[q];
    const PairDev& P = rig->pair[bc->cam.pair0 + q];
    const CamDev* J = &rig->cam[V.j];
    float4 a4, b4;
    float2 a2, b2;
    float ah[3], al[3];
    prays(q, a4, a2, b4, b2);
    ff_ray_affine(a4.x, a4.w, b4.x, b4.w, z, P.th[0], P.tl[0], ah[0], al[0]);
    ff_ray_affine(a4.y, a2.x, b4.y, b2.x, z, P.th[1], P.tl[1], ah[1], al[1]);
    ff_ray_affine(a4.z, a2.y, b4.z, b2.y, z, P.th[2], P.tl[2], ah[2], al[2]);
    fast_two_sum(ah[2], al[2], ah[2], al[2]);             // sign of a_z is that of ah
    if (!(ah[2] > 0.0f)) continue;                        // behind camera j
    const float fu = __fmaf_rn(V.fx, __fdividef(ah[0], ah[2]), V.cx5);
    const float fv = __fmaf_rn(V.fy, __fdividef(ah[1], ah[2]), V.cy5);
    const int px = nearest_pixel<false>(fu, V.band, J, ah[0], al[0], ah[2], al[2]);
    const int py = nearest_pixel<true>(fv, V.band, J, ah[1], al[1], ah[2], al[2]);
    if ((unsigned)px >= (unsigned)V.W || (unsigned)py >= (unsigned)V.H) continue;
    const DT D = __ldg(static_cast<const DT*>(fp->depth[V.j]) + (unsigned)(py * V.W + px));
    if (!Depth<DT>::valid(D)) continue;
    // Q = D_j(u_j) (rx_j, ry_j, 1) in camera-j coordinates (rigid motion keeps d)
    const float zj = __fmul_rn(Depth<DT>::z(D), ginv);
    const float2 qx = __ldg(rays + V.ray_x + px), qy = __ldg(rays + V.ray_y + py);
    float qh[3], ql[3];
    two_prod(zj, qx.x, qh[0], ql[0]);
    ql[0] = __fmaf_rn(zj, qx.y, ql[0]);
    two_prod(zj, qy.x, qh[1], ql[1]);
    ql[1] = __fmaf_rn(zj, qy.y, ql[1]);
    qh[2] = zj;
    ql[2] = 0.0f;
#pragma unroll
    for (int k = 0; k < 3; ++k) {                         // d^2 = |a - Q|^2 in ff
      float s, e, p, pe, tt;
      two_sum(ah[k], -qh[k], s, e);
      e = __fadd_rn(e, __fsub_rn(al[k], ql[k]));
      // (s + e)^2 = s^2 + 2 s e + e^2; e^2 is below the ff rounding of the sum
      two_prod(s, s, p, pe);
      pe = __fmaf_rn(__fmul_rn(2.0f, s), e, pe);
      two_sum(sh, p, sh, tt);
      sl = __fadd_rn(sl, __fadd_rn(tt, pe));
    }
    ++nview;
  }
  res[0] = sh;
  res[1] = sl;
  *views = nview;
}

// The same sum for depths up to the rig's zmax, on the rig's grid (all coordinates below 2^22 grid
// units): every coordinate is kept as an integral float plus a remainder below one unit.  Adding
// kGridM in the FMA that forms a product rounds it to an integer, a second FMA gives the exact rest,
// and integral parts add exactly; the difference D of two integral parts is the difference of their
// bits, so that sum D^2 is exact in 64-bit integers, and float32 carries the remainders alone:
// d^2 = D^2 + l (2 D + l).  A remainder is off by a few 2^-26 grid units, 2^-47 of the rig's extent.
// 16 operations a coordinate where the double-float evaluation takes 41; with it the consistency step of
// the 8x1280x720 rig (3.7 M points, 3 views) went from 269 to 216 us in the kernel it then was part of.
// Measured slower: two points a thread side by side (+16 us, spills), three views at once (+15 us).
// Views whose sample is beyond zmax return false (the point then takes the general evaluation).
template <typename DT, typename PR>
__device__ __forceinline__ bool residual_grid(const ViewHot* views, int k1, const PR& prays,
                                              const RigDev* __restrict__ rig, const RigHot& hot,
                                              const float2* __restrict__ rays, const FramePtrs& fp,
                                              float z, float& sh, float& sl, int& nview) {
  long long S = 0;
  float c = 0.0f;
  bool fits = sizeof(DT) == 2 || z <= hot.zmax;
#pragma unroll 1
  for (int q = 0; q < k1; ++q) {
    const float4* vw = reinterpret_cast<const float4*>(views + q);
    const float4 w0 = vw[0], w1 = vw[1], w2 = vw[2], w3 = vw[3];
    const float mt[3] = {w0.x, w0.y, w0.z}, tl[3] = {w0.w, w1.x, w1.y};
    const int W = __float_as_int(w2.z), H = __float_as_int(w2.w), j = __float_as_int(w3.w);
    float4 a4, b4;
    float2 a2, b2;
    prays(q, a4, a2, b4, b2);
    const float gh[3] = {__fadd_rn(a4.x, b4.x), __fadd_rn(a4.y, b4.y), __fadd_rn(a4.z, b4.z)};
    const float gl[3] = {__fadd_rn(a4.w, b4.w), __fadd_rn(a2.x, b2.x), __fadd_rn(a2.y, b2.y)};
    float s[3], l[3], ah[3], f[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {                         // Eq. 4: a = z (A + B) + t
      s[k] = __fmaf_rn(z, gh[k], mt[k]);
      l[k] = __fmaf_rn(z, gh[k], -__fsub_rn(s[k], mt[k]));
      l[k] = __fadd_rn(__fmaf_rn(z, gl[k], l[k]), tl[k]);
      ah[k] = __fsub_rn(s[k], kGridM);
      f[k] = __fadd_rn(ah[k], l[k]);
    }
    if (!(f[2] > 0.0f)) continue;                          // behind camera j
    const float inv = rcp_approx(f[2]);
    const float fu = __fmaf_rn(w1.z, __fmul_rn(f[0], inv), w2.x);
    const float fv = __fmaf_rn(w1.w, __fmul_rn(f[1], inv), w2.y);
    const int px = nearest_pixel<false>(fu, w3.z, &rig->cam[j], ah[0], l[0], ah[2], l[2]);
    const int py = nearest_pixel<true>(fv, w3.z, &rig->cam[j], ah[1], l[1], ah[2], l[2]);
    if ((unsigned)px >= (unsigned)W || (unsigned)py >= (unsigned)H) continue;
    const DT Dj = __ldg(static_cast<const DT*>(fp.depth[j]) + (unsigned)(py * W + px));
    const float2 qx = __ldg(rays + __float_as_int(w3.x) + px), qy = __ldg(rays + __float_as_int(w3.y) + py);
    if (!Depth<DT>::valid(Dj)) continue;
    if (sizeof(DT) == 4) fits = fits && Depth<DT>::z(Dj) <= hot.zmax;
    // Q = D_j(u_j) (rx_j, ry_j, 1) in camera-j coordinates (rigid motion keeps d)
    const float zj = __fmul_rn(Depth<DT>::z(Dj), hot.ginv);
    const float r[3] = {qx.x, qy.x, 1.0f}, rl[3] = {qx.y, qy.y, 0.0f};
#pragma unroll
    for (int k = 0; k < 3; ++k) {                         // Eq. 5, 6
      const float t = __fmaf_rn(zj, r[k], kGridM);
      float e = __fmaf_rn(zj, r[k], -__fsub_rn(t, kGridM));
      if (k < 2) e = __fmaf_rn(zj, rl[k], e);
      const int D = __float_as_int(s[k]) - __float_as_int(t);
      const float dl = __fsub_rn(l[k], e);
      S += (long long)D * D;
      c = __fmaf_rn(dl, __fmaf_rn(2.0f, __fsub_rn(s[k], t), dl), c);
    }
    ++nview;
  }
  // S = hi 2^25 + lo, -2^24 <= lo < 2^24, and the remainders' sum c as one ff.  Both parts are exact:
  // a point and the sample at its pixel lie along one ray of the view, so that |D| < 2^22 and
  // S < 3 kMaxK1 2^44 < 2^49
  static_assert(3 * kMaxK1 <= 32, "the high part of a residual sum fits 24 bits");
  const int hn = (int)((S + (1 << 24)) >> 25);
  const float hi = __fmul_rn((float)hn, 33554432.0f), lo = (float)(int)((unsigned)S - ((unsigned)hn << 25));
  float s1, e1, e2;
  two_sum(lo, c, s1, e1);
  fast_two_sum(hi, s1, sh, e2);
  sl = __fadd_rn(e1, e2);
  return fits;
}

// Residual sum of a point over its camera's views (block constants bc in shared or global
// memory): the grid evaluation, or the general one where a depth is beyond the rig's zmax.
template <typename DT, typename PR>
__device__ __forceinline__ void residual_sum(const BlockConst* bc, const Tables& t, int cam, int k1, const PR& prays,
                                             const RigDev* __restrict__ rig, const RigHot& hot,
                                             const float2* __restrict__ rays, const FramePtrs& fp, float z,
                                             int x, int y, float& sh, float& sl, int& nview) {
  nview = 0;
  const bool fits = residual_grid<DT>(bc->view, k1, prays, rig, hot, rays, fp, z, sh, sl, nview);
  if constexpr (sizeof(DT) == 4) {
    if (!fits) {
      const BlockConst* g = t.bconst + cam;
      float res[2];
      residual_general<DT>(g, k1, rig, GlobalPairRays(t.pray + g->cam.pray, rig->cam[cam].W, k1, x, y), rays, &fp,
                           z, res, &nview);
      sh = res[0];
      sl = res[1];
    }
  }
}

// Eq. 7 and 10 from the residual sum (sh, sl): omega = C' exp(-e) = mu 2^-m with
// e = m ln 2 + f, f in [0, ln 2), so that mu never underflows (C' = C, or 1 without the
// confidence term).  A residual beyond float32 (a view's sample near the format's largest value)
// leaves e infinite or not a number; its weight is 0 at an exponent above every other, so that it
// adds nothing to a sum and does not set the sum's scale.  Confidences above 1 move into the
// exponent (exactly), which keeps mu below 2 for the fixed-point terms.  Returns e (high part) for
// traces.
constexpr int kFarExponent = 1500000000;   // other exponents are at most 1e9 / ln 2
__device__ __forceinline__ float joint_weight(const RigHot& rig, int k1, float sh, float sl,
                                              float c, float& mu, int& m) {
  float eh = 0.0f, el = 0.0f;
  if (rig.use_cons && k1 > 0) {
    fast_two_sum(sh, sl, sh, sl);
    two_prod(sh, rig.einv_h, eh, el);                                  // Eq. 7 exponent
    el = __fmaf_rn(sh, rig.einv_l, __fmaf_rn(sl, rig.einv_h, el));
    fast_two_sum(eh, el, eh, el);
  }
  m = 0;
  float fh = eh, fl = el;
  if (eh > 0.0f) {
    m = (int)floorf(__fmul_rn(fminf(eh, 1.0e9f), kInvLn2));
    const float mf = (float)m;
    float p, pe;
    two_prod(mf, kLn2H, p, pe);
    fh = __fsub_rn(eh, p);
    fl = __fsub_rn(__fsub_rn(el, pe), __fmul_rn(mf, kLn2L));
  }
  const float base = rig.use_conf ? c : 1.0f;                          // Eq. 10
  mu = __fmul_rn(__fmul_rn(base, expf(-fh)), __fsub_rn(1.0f, fl));
  if (!(mu < 2.0f)) {                       // confidences above 1, or no number
    if (mu != mu) {
      mu = 0.0f;
      m = kFarExponent;
      eh = __int_as_float(0x7f800000);
    } else if (mu < __int_as_float(0x7f800000)) {
      const int bits = __float_as_int(mu);
      m -= (bits >> 23) - 127;
      mu = __int_as_float((bits & 0x7fffff) | 0x3f800000);
    }
  }
  return eh;
}

// ------------------------------------------------------------------ count step
// Position of a cell key in a warp's table of kUnitCells, inserted if new; -1 after 4 probes.
__device__ __forceinline__ int unit_cell(unsigned* tab, unsigned key) {
  unsigned h = (key * 0x9E3779B1u) >> 26;
#pragma unroll 1
  for (int probe = 0; probe < 4; ++probe) {
    const unsigned cur = *static_cast<volatile unsigned*>(&tab[h]);
    if (cur == key) return (int)h;
    if (cur == 0xffffffffu) {
      const unsigned prev = atomicCAS(&tab[h], 0xffffffffu, key);
      if (prev == 0xffffffffu || prev == key) return (int)h;
    }
    h = (h + 1) & (kUnitCells - 1);
  }
  return -1;
}

// Camera and first pixel of unit u.
__device__ __forceinline__ void unit_of(const TileIndex& ti, int u, int& cam, int& x0, int& y0) {
  int lu = u, ux;
  if (ti.units_per_cam) {
    cam = fast_div(u, ti.units_per_cam, ti.div_units, lu);
  } else {
    cam = 0;
    for (int lo = 0, hi = ti.n_cams - 1; lo <= hi;) {
      const int mid = (lo + hi) >> 1;
      if (ti.unit[mid] <= u) { cam = mid; lo = mid + 1; } else { hi = mid - 1; }
    }
    lu = u - ti.unit[cam];
  }
  y0 = fast_div(lu, (ti.W[cam] + kTileW - 1) / kTileW, ti.div_x[cam], ux) * kUnitH;
  x0 = ux * kTileW;
}
constexpr unsigned kUnnumbered = 0x80000000u;   // on a unit's count while points of it are left

// A warp takes units of 32 columns by 8 rows with no block-wide step in between: gate (Eq. 9) and
// compaction of the gated pixels, a column a lane; then a gated pixel a lane, full warps: back-projection
// (Eq. 8), extent (Sec. II.5(1)b), and the coarse cell (Sec. II.5(1)c), counted in a small table of the
// warp.  Each cell goes to the global table once per unit, with its number of points, and its position
// in the warp's table is its number in the unit; the gated pixels are listed (pixel and cell number,
// depth, confidence) for the next steps, which then neither gate again nor probe the global table.
// 8x1280x720 (7.4 Mpx, 28,800 units): 49 us, bound by instruction issue (69 % of the slots used);
// blocks with a table of 2048 cells and runs of equal cells merged across the warp took 59 us.  Finding a
// unit's cells one after another as the smallest key left took 49 us there, but 236 instead of 154 us
// where units hold many cells (16x1024^2).
constexpr int kCountFew = 2 * 4 * (kThreads / 32);   // units a multiprocessor: two rounds of 4 blocks

// FEW: launches of no more units than the chip takes at once or twice (whatever the units per block), where the step is as long as a crowded
// unit's chain of probes.  There a unit whose first 32 points have more than 14 cells puts no more into its
// table, and 8 of its points instead of 4 are under way together: frames of 5x326x319 in a room 94 -> 85 us,
// 8x248x228 95 -> 87 us (limits of 10 and 20 cells: 87 and 87).  With the test in it the loop takes 3 to 5 %
// longer in large frames (51.4 us instead of 49.6 at 8x1280x720, 169 instead of 161 at 16x1024x1024), which
// go without.
template <typename DT, int NB, bool FEW>
__global__ void __launch_bounds__(kThreads, 4) k_count(const __grid_constant__ BatchArgs<NB> args) {
  int local;
  const FrameArgs& fa = args.f[batch_frame<NB>(args.count_first, args.n, (int)blockIdx.x, local)];
  const float2* __restrict__ rays = fa.rays;
  const FramePtrs& fp = fa.fp;
  const Tables& t = fa.t;
  const TileIndex& ti = fa.ti;
  pdl_release();
  constexpr int kUnitPx = kTileW * kUnitH;
  __shared__ DT s_d[kThreads / 32][kUnitPx];
  __shared__ float s_c[kThreads / 32][kUnitPx];
  __shared__ unsigned char s_p[kThreads / 32][kUnitPx];
  __shared__ CamHot s_cam[kThreads / 32];
  __shared__ unsigned char s_occ[kThreads / 32][kUnitCells];
  __shared__ unsigned s_key[kThreads / 32][kUnitCells], s_cnt[kThreads / 32][kUnitCells];
  static_assert(kUnitCells == 64, "two positions a lane, 6-bit hash");
  constexpr int kMissed = FEW ? 8 : 4;                                         // points without a number tried together by a lane
  __shared__ unsigned s_red[kThreads / 32][9];
  const float tau = fa.hot.tau, inv_s0u = fa.hot.inv_s0u;
  const bool use_conf = fa.hot.use_conf != 0;
  const int lim = kKeyBias >> fa.hot.max_level;                      // a power of two
  const unsigned window = (unsigned)min(1024, 2 * lim);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const float qnan = __int_as_float(0x7fffffff), inf = __int_as_float(0x7f800000);
  unsigned nv = 0, ng = 0, noor = 0;
  bool any_rest = false;
  float fmn[3] = {inf, inf, inf}, fmx[3] = {-inf, -inf, -inf};
  const int u0 = local * fa.count_chunks * (kThreads / 32);
  const int u1 = min(u0 + fa.count_chunks * (kThreads / 32), t.n_units);
#pragma unroll 1
  for (int u = u0 + warp; u < u1; u += kThreads / 32) {
    int cam, x0, y0;
    unit_of(ti, u, cam, x0, y0);
    const int W = ti.W[cam], H = ti.H[cam];
    int n = 0;
    {
      const DT* __restrict__ dep = static_cast<const DT*>(fp.depth[cam]);
      const float* __restrict__ cf = fp.conf[cam];
      const int rows = x0 + lane < W ? min(kUnitH, H - y0) : 0;
      DT D[kUnitH];
      float C[kUnitH];
      unsigned li = (unsigned)(y0 * W + x0 + lane);                  // W H <= 2^30
#pragma unroll
      for (int k = 0; k < kUnitH; ++k, li += W) {
        D[k] = (DT)0;
        C[k] = 0.0f;
        if (k < rows) {
          D[k] = dep[li];
          C[k] = cf[li];
        }
      }
#pragma unroll
      for (int k = 0; k < kUnitH; ++k) {
        const bool valid = Depth<DT>::valid(D[k]);
        const bool gated = valid && (!use_conf || C[k] > tau);       // Eq. 9
        nv += valid ? 1u : 0u;
        const unsigned m = __ballot_sync(0xffffffffu, gated);
        if (gated) {
          const int pos = n + __popc(m & ((1u << lane) - 1u));
          s_d[warp][pos] = D[k];
          s_c[warp][pos] = C[k];
          s_p[warp][pos] = (unsigned char)(k * kTileW + lane);
        }
        n += __popc(m);
      }
    }
    if (n == 0) {                                                    // uniform over the warp
      if (lane == 0) t.lcount[u] = 0u;
      continue;
    }
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      s_key[warp][lane + 32 * q] = 0xffffffffu;
      s_cnt[warp][lane + 32 * q] = 0u;
    }
    if (lane < 4) reinterpret_cast<float4*>(&s_cam[warp])[lane] = __ldg(reinterpret_cast<const float4*>(t.bconst + cam) + lane);
    __syncwarp();
    const CamHot cam_c = s_cam[warp];
    // the rays of the unit's columns (a lane one) and rows (the first lanes)
    const float ray_x = __ldg(&rays[cam_c.ray_x + min(x0 + lane, W - 1)].x);
    const float ray_y = __ldg(&rays[cam_c.ray_y + min(y0 + (lane & (kUnitH - 1)), H - 1)].x);
    auto point = [&](int i, float z, float P[3]) {                   // Eq. 8 of list entry i at depth z
      const int p = s_p[warp][i];
      world_point(cam_c, z, __shfl_sync(0xffffffffu, ray_x, p & (kTileW - 1)),
                  __shfl_sync(0xffffffffu, ray_y, p / kTileW), P);
    };
    // Coarse cells as keys of 10 bits an axis, relative to the first point's cell - 512, or to the first
    // cell in range where there are no more than 1024 (a cell index is read off the bits of kGridM +
    // v rounded down: grid_coords); `ok`: the window holds only cells in range.  Other points go to the
    // global table by themselves.
    int ref[3] = {kGridBits - lim, kGridBits - lim, kGridBits - lim};
    bool ok = true;
    if (lim > 512) {
      float P[3];
      point(0, Depth<DT>::z(s_d[warp][0]), P);
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        ref[a] = __float_as_int(__fadd_rd(__fmul_rn(P[a], inv_s0u), kGridM)) - 512;
        ok = ok && (unsigned)(ref[a] - kGridBits + lim) < (unsigned)(2 * lim - 1024);
      }
    }
    const long long at = unit_list(ti.off[cam], W, H, x0, y0);
    DT* __restrict__ ld = static_cast<DT*>(t.ldepth) + at;
    float* __restrict__ lc = t.lconf + at;
    unsigned short* __restrict__ lp = t.lpix + at;
    bool sparse = false;                                             // hardly two points in a cell
    bool missed = false;                                             // a point without a number
#pragma unroll 1
    for (int i0 = 0; i0 < n; i0 += 32) {
      const int i = i0 + lane;
      const bool act = i < n;
      const DT d = s_d[warp][i];
      float P[3];
      point(i, act ? Depth<DT>::z(d) : qnan, P);                     // NaN: no minimum or maximum takes it
      unsigned q[3];
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        fmn[a] = fminf(fmn[a], P[a]);
        fmx[a] = fmaxf(fmx[a], P[a]);
        q[a] = (unsigned)(__float_as_int(__fadd_rd(__fmul_rn(P[a], inv_s0u), kGridM)) - ref[a]);
      }
      const bool in = ok && (q[0] | q[1] | q[2]) < window;
      const unsigned key = act && in ? (q[0] << 20) + (q[1] << 10) + q[2] : 0xffffffffu;
      const unsigned key0 = __shfl_sync(0xffffffffu, key, 0);
      int number = -1;
      if (__all_sync(0xffffffffu, key == key0 || !act) && key0 != 0xffffffffu) {   // one cell: one insertion
        if (lane == 0) {
          number = unit_cell(s_key[warp], key0);
          if (number >= 0) s_cnt[warp][number] += (unsigned)min(32, n - i0);
        }
        number = __shfl_sync(0xffffffffu, number, 0);
      } else {
        if (key != 0xffffffffu && !(FEW && sparse)) {
          number = unit_cell(s_key[warp], key);
          if (number >= 0) atomicAdd(&s_cnt[warp][number], 1u);
        }
        if (FEW && i0 == 0) {
          __syncwarp();
          sparse = __popc(__ballot_sync(0xffffffffu, s_key[warp][lane] != 0xffffffffu)) +
                       __popc(__ballot_sync(0xffffffffu, s_key[warp][lane + 32] != 0xffffffffu)) > 14;
        }
      }
      if (act) {
        missed = missed || number < 0;
        ld[i] = d;
        lc[i] = s_c[warp][i];
        lp[i] = (unsigned short)(s_p[warp][i] | ((unsigned)(number & 0xff) << 8));
      }
      __syncwarp();
    }
    ng += lane == 0 ? (unsigned)n : 0u;
    // the unit's cells into the global table, one a lane
    const unsigned o0 = __ballot_sync(0xffffffffu, s_key[warp][lane] != 0xffffffffu);
    const unsigned o1 = __ballot_sync(0xffffffffu, s_key[warp][lane + 32] != 0xffffffffu);
    const unsigned below = (1u << lane) - 1u;
    if ((o0 >> lane) & 1u) s_occ[warp][__popc(o0 & below)] = (unsigned char)lane;
    if ((o1 >> lane) & 1u) s_occ[warp][__popc(o0) + __popc(o1 & below)] = (unsigned char)(lane + 32);
    __syncwarp();
    const int cells = __popc(o0) + __popc(o1);
    for (int q = lane; q - lane < cells; q += 32) {
      const bool act = q < cells;
      const int h = act ? s_occ[warp][q] : 0;
      const unsigned key = s_key[warp][h];
      const unsigned slot =
          count_cell(t, act, ref[0] - kGridBits + (int)(key >> 20), ref[1] - kGridBits + (int)((key >> 10) & 1023u),
                     ref[2] - kGridBits + (int)(key & 1023u), s_cnt[warp][h]);
      if (act) t.lcell[(long long)u * kUnitCells + h] = slot;
    }
    const bool rest = __any_sync(0xffffffffu, missed);
    if (lane == 0) t.lcount[u] = (unsigned)n | (rest ? kUnnumbered : 0u);
    any_rest = any_rest || rest;
    __syncwarp();                                                    // the staged pixels are free again
  }
  // The points without a number (far-flung ones, and of units with more cells than the table takes) go to the
  // global table by themselves, from the lists.  After the other units: inside their loop this costs its
  // registers, 3 to 9 % of the step.
  if (any_rest) {                                                    // uniform over the warp
    __syncwarp();
#pragma unroll 1
    for (int u = u0 + warp; u < u1; u += kThreads / 32) {
      const unsigned marked = __ldcg(t.lcount + u);
      if (!(marked & kUnnumbered)) continue;
      const int n = (int)(marked & ~kUnnumbered);
      int cam, x0, y0;
      unit_of(ti, u, cam, x0, y0);
      const int W = ti.W[cam], H = ti.H[cam];
      const long long at = unit_list(ti.off[cam], W, H, x0, y0);
      const DT* ld = static_cast<const DT*>(t.ldepth) + at;
      const unsigned short* lp = t.lpix + at;
      if (lane < 4) reinterpret_cast<float4*>(&s_cam[warp])[lane] = __ldg(reinterpret_cast<const float4*>(t.bconst + cam) + lane);
      __syncwarp();
      const CamHot& cam_c = s_cam[warp];
#pragma unroll 1
      for (int i0 = 0; i0 < n; i0 += 32 * kMissed) {
        unsigned long long key[kMissed];
        unsigned e[kMissed];
        DT d[kMissed];
#pragma unroll
        for (int k = 0; k < kMissed; ++k) {                          // the lane's own stores above
          const int i = i0 + 32 * k + lane;
          e[k] = i < n ? __ldcg(lp + i) : 0u;
          d[k] = i < n ? __ldcg(ld + i) : (DT)0;
        }
#pragma unroll
        for (int k = 0; k < kMissed; ++k) {
          key[k] = kKeyEmpty;
          if ((e[k] >> 8) == kNoCellNumber) {
            float P[3], r[3];
            int c[3];
            world_point(cam_c, Depth<DT>::z(d[k]), __ldg(&rays[cam_c.ray_x + x0 + (int)(e[k] & (kTileW - 1))].x),
                        __ldg(&rays[cam_c.ray_y + y0 + (int)((e[k] & 0xffu) / kTileW)].x), P);
            if (grid_coords(fa.hot, P, r, c))
              key[k] = pack_key(0, c[0], c[1], c[2]);
            else
              ++noor;
          }
        }
        count_points<kMissed>(t, key);
      }
      __syncwarp();
      if (lane == 0) t.lcount[u] = (unsigned)n;
    }
  }
  // per-block pixel counts and extent
  unsigned vals[9] = {nv, ng, noor};
#pragma unroll
  for (int a = 0; a < 3; ++a) { vals[3 + a] = ordered(fmn[a]); vals[6 + a] = ordered(fmx[a]); }
  vals[0] = __reduce_add_sync(0xffffffffu, vals[0]);
  vals[1] = __reduce_add_sync(0xffffffffu, vals[1]);
  vals[2] = __reduce_add_sync(0xffffffffu, vals[2]);
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    vals[3 + a] = __reduce_min_sync(0xffffffffu, vals[3 + a]);
    vals[6 + a] = __reduce_max_sync(0xffffffffu, vals[6 + a]);
  }
  if (lane == 0) {
#pragma unroll
    for (int a = 0; a < 9; ++a) s_red[warp][a] = vals[a];
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    BlockStats b = {};
    for (int k = 0; k < 3; ++k) { b.bmin[k] = 0xffffffffu; b.bmax[k] = 0u; }
    for (int w = 0; w < kThreads / 32; ++w) {
      b.n_valid += s_red[w][0];
      b.n_gated += s_red[w][1];
      b.n_oor += s_red[w][2];
      if (s_red[w][1] == 0u) continue;                               // no point: no extent
      for (int k = 0; k < 3; ++k) {
        b.bmin[k] = min(b.bmin[k], s_red[w][3 + k]);
        b.bmax[k] = max(b.bmax[k], s_red[w][6 + k]);
      }
    }
    t.bstats[local] = b;
  }
}

__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src));
}
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// Camera and first pixel of tile T (tiles of TH rows): divisions by known divisors when every camera
// has the same size, else a binary search of the per-camera tile ranges (constant bank).
template <int TH>
__device__ __forceinline__ void tile_of(const TileIndex& ti, int T, int& cam, int& x0, int& y0) {
  int local = T;
  if (ti.per_cam) {
    cam = fast_div(T, ti.per_cam, ti.div_cam, local);
  } else {
    cam = 0;
    for (int lo = 0, hi = ti.n_cams - 1; lo <= hi;) {
      const int mid = (lo + hi) >> 1;
      if (ti.first[mid] <= T) { cam = mid; lo = mid + 1; } else { hi = mid - 1; }
    }
    local = T - ti.first[cam];
  }
  int tx;
  y0 = fast_div(local, (ti.W[cam] + kTileW - 1) / kTileW, ti.div_x[cam], tx) * TH;
  x0 = tx * kTileW;
}

// ------------------------------------------------------------------ ranks and statistics
// A slot without representative, number or weight exponent.
#define kSlotClear make_uint4(0u, 0u, kSlotNone, (unsigned)INT_MAX)

// Marks cell `id` as having its representative at pixel g: a bit of the pixel and the cell's number there
// (over the list's confidences, which no step reads any more).  The caller counts the bits of each emit
// block's share of the bitmap.
__device__ __forceinline__ void mark_cell(const Tables& t, unsigned g, unsigned id) {
  atomicOr(&t.bitmap[g >> 5], 1u << (g & 31));
  t.cell_at[g] = id;
}

// The frame's statistics from the count step's blocks and the counters, by one block, which clears the
// counters for the next frame (but the number of cells, which other blocks of its kernel read).
template <bool TOPK>
__device__ __forceinline__ void frame_stats(const Tables& t, const OutDev& out) {
  __shared__ unsigned long long s_l[3][kThreads / 32];
  __shared__ unsigned s_b[6][kThreads / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  unsigned long long n[3] = {0ull, 0ull, 0ull};
  unsigned mn[3] = {0xffffffffu, 0xffffffffu, 0xffffffffu}, mx[3] = {0u, 0u, 0u};
  for (int i = threadIdx.x; i < t.n_bstats; i += kThreads) {
    const BlockStats b = t.bstats[i];
    n[0] += b.n_valid;
    n[1] += b.n_gated;
    n[2] += b.n_oor;
    for (int k = 0; k < 3; ++k) { mn[k] = min(mn[k], b.bmin[k]); mx[k] = max(mx[k], b.bmax[k]); }
  }
  const unsigned nc = __ldcg(&t.cnt->n_cells);
  // cells without a record, as these ran out (reported), are not in the list of cells that the reduce
  // step clears, but their keys are in their slots
  if (TOPK && __ldcg(&t.cnt->n_partials) > t.max_partials) {
    const unsigned n_slots = (unsigned)min(__ldcg(&t.cnt->n_slots), (unsigned long long)t.max_slots);
    for (unsigned i = threadIdx.x; i < n_slots; i += kThreads) *reinterpret_cast<uint4*>(t.frec + i) = kSlotClear;
  }
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    for (int o = 16; o > 0; o >>= 1) n[k] += __shfl_xor_sync(0xffffffffu, n[k], o);
    mn[k] = __reduce_min_sync(0xffffffffu, mn[k]);
    mx[k] = __reduce_max_sync(0xffffffffu, mx[k]);
    if (lane == 0) { s_l[k][warp] = n[k]; s_b[k][warp] = mn[k]; s_b[3 + k][warp] = mx[k]; }
  }
  __syncthreads();
  if (threadIdx.x != 0) return;
  for (int q = 1; q < kThreads / 32; ++q)
    for (int k = 0; k < 3; ++k) {
      n[k] += s_l[k][q];
      mn[k] = min(mn[k], s_b[k][q]);
      mx[k] = max(mx[k], s_b[3 + k][q]);
    }
  fuseflow_stats st = {};
  st.n_valid = (int64_t)n[0];
  st.n_gated = (int64_t)n[1];
  st.n_out_of_range = (int64_t)n[2];
  unsigned err = __ldcg(&t.cnt->error);
  if ((long long)nc > out.max_cells) err |= kErrCells;
  if (TOPK && __ldcg(&t.cnt->n_partials) > t.max_partials) err |= kErrPartials;
  st.n_cells = (int64_t)(nc < out.max_cells ? nc : out.max_cells);
  for (int k = 0; k < 3; ++k) {
    st.bbox[k] = n[1] ? (float)((double)from_ordered(mn[k]) * out.unit_m) : __int_as_float(0x7f800000);
    st.bbox[3 + k] = n[1] ? (float)((double)from_ordered(mx[k]) * out.unit_m) : __int_as_float(0xff800000);
  }
  st.error = (int32_t)err;
  st.n_coarse = (int32_t)__ldcg(&t.cnt->n_coarse);
  *out.stats = st;
  t.cnt->n_coarse = 0u;                         // n_cells: by the level step
  t.cnt->error = 0u;
  t.cnt->n_partials = 0u;
  t.cnt->n_slots = 0ull;
}

// u64 -> float32 through two 32-bit conversions (at most two roundings)
__device__ __forceinline__ float u64_to_f32(unsigned long long x) {
  return __fmaf_rn(__uint2float_rn((unsigned)(x >> 32)), 4294967296.0f, __uint2float_rn((unsigned)x));
}

// ------------------------------------------------------------------ weigh step
// A block takes one tile of 32 columns by TH rows (TH = 8, 16 or 32: a launch-geometry choice), a
// thread up to four of its gated pixels, one after another, with no step of the whole block between
// the staging of the tile's constants and the claims at the end.  Frames of few tiles take more
// threads a block, down to a pixel a thread (weigh_threads).
template <int TH>
struct WeighTile {
  static_assert(TH == 8 || TH == 16 || TH == 32, "tile heights");
  static constexpr int Px = kTileW * TH, Threads = 8 * TH, Units = TH / kUnitH;
  // claimed cells (slot, key), level and first slot of the units' numbered coarse cells, camera and view
  // constants, the tile's pair rays
  static constexpr size_t Key = 0;                                 // u64[Px]
  static constexpr size_t Slot = Key + 8 * Px;                     // u32[Px]
  static constexpr size_t LB = Slot + 4 * Px;                      // u32[Units][kUnitCells]
  static constexpr size_t BC = LB + 4 * Units * kUnitCells;
  // 16-byte words of the constants of k1 views, and of the pair rays of the tile's columns and rows
  static __host__ __device__ constexpr int const_words(int k1) { return 4 * (1 + k1); }
  static __host__ __device__ constexpr int col_words(int k1) { return k1 * kPrayColGroup; }
  static __host__ __device__ constexpr int row_words(int k1) { return k1 * Units * kPrayRowGroup; }
  static constexpr size_t smem(int k1) { return BC + 16 * (size_t)(const_words(k1) + col_words(k1) + row_words(k1)); }
};

// The tile's gated pixels are its units' lists, one after the other: entry i of the tile is entry
// i + shift of the frame's lists, for the unit it falls into.
template <int kUnits>
struct TileList {
  int n, end[kUnits];            // pixels of the tile; of the units up to each one
  unsigned shift[kUnits];
  __device__ __forceinline__ TileList(const Tables& t, const TileIndex& ti, int cam, unsigned off, int W, int H, int x0,
                                      int y0) {
    const int tiles_x = (W + kTileW - 1) / kTileW, u0 = ti.unit[cam] + (y0 >> 3) * tiles_x + (x0 >> 5);
    unsigned listed[kUnits];
#pragma unroll
    for (int k = 0; k < kUnits; ++k) listed[k] = y0 + k * kUnitH < H ? __ldcg(t.lcount + u0 + k * tiles_x) : 0u;
    n = 0;
#pragma unroll
    for (int k = 0; k < kUnits; ++k) {
      shift[k] = (unsigned)unit_list(off, W, H, x0, y0 + k * kUnitH) - (unsigned)n;
      n += (int)listed[k];
      end[k] = n;
    }
  }
  // unit of entry i, and its entry in the frame's lists
  __device__ __forceinline__ unsigned at(int i, int& unit) const {
    unit = 0;
    unsigned s = shift[0];
#pragma unroll
    for (int q = 1; q < kUnits; ++q)
      if (i >= end[q - 1]) { unit = q; s = shift[q]; }
    return s + (unsigned)i;
  }
};

// Levels and first slots of the units' numbered coarse cells (Sec. II.5(1)d).  (A number that the unit
// does not use still names some position of the coarse table, an earlier frame's.)
template <int kUnits>
__device__ __forceinline__ void load_cell_levels(const Tables& t, const TileIndex& ti, const TileList<kUnits>& list, int cam,
                                                 int W, int x0, int y0, unsigned* s_lb) {
  const int tiles_x = (W + kTileW - 1) / kTileW, u0 = ti.unit[cam] + (y0 >> 3) * tiles_x + (x0 >> 5);
  for (int i = threadIdx.x; i < kUnits * kUnitCells; i += (int)blockDim.x) {
    const int k = i / kUnitCells;
    bool listed = false;                          // the unit has a list, and so its numbers
#pragma unroll
    for (int q = 0; q < kUnits; ++q)
      if (k == q) listed = list.end[q] > (q ? list.end[q > 0 ? q - 1 : 0] : 0);
    if (listed) {
      const unsigned slot = __ldcg(t.lcell + (long long)(u0 + k * tiles_x) * kUnitCells + (i & (kUnitCells - 1)));
      s_lb[i] = slot == kSlotNone ? kBaseNone : __ldcg(&t.coarse[slot].lvbase);
    }
  }
}

// Dense slot of a point: level << 27 | slot, from its coarse cell's level << 27 | first slot; its cell
// key's parts in kk and its place in the cell in frac.  kBaseNone in the slot field: none.
__device__ __forceinline__ unsigned point_slot(unsigned lb, const float r[3], int kk[3], float frac[3]) {
  const int l = (int)(lb >> 27);
  const float sl = pow2f(l);
#pragma unroll
  for (int a = 0; a < 3; ++a) {                   // floor of r 2^l (below 2^19 in size) and the rest
    const float t = __fmaf_rd(r[a], sl, kGridM);
    kk[a] = __float_as_int(t) - kGridBits;
    frac[a] = __fmaf_rn(r[a], sl, -__fsub_rn(t, kGridM));
  }
  // sub-cell of the coarse cell: k - (coarse << l) = k & (2^l - 1)
  const unsigned mask = (1u << l) - 1u;
  const unsigned local = ((((unsigned)kk[0] & mask) << l | ((unsigned)kk[1] & mask)) << l) | ((unsigned)kk[2] & mask);
  return (lb & kBaseNone) == kBaseNone ? lb : lb + local;
}

// Per gated pixel: Eq. 8, its cell (Sec. II.5(1)d-e), its joint weight (Eq. 4-7, 10) as mantissa and
// exponent; per cell, kept in its slot: the representative (Sec. II.5(2)a) as the largest
// (ordered(C) << 32) | ~g, the smallest weight exponent, and the cell's number, claimed by the first
// point that finds none.  All are order-independent but the numbering, which no result depends on.
// A point looks at its slot first and sends an atomic only where that would change it: most do not.
// Bound by latency and issue (gathers of the views' depths): 48 registers for uint16 depth, as 40 warps
// an SM hide more than 32 do (weigh + sum of 8x1280x720 when they were split: 185 us against 193 at 64); float32 depth, with
// its checks, is faster at 64 (50 against 53 us on five ragged cameras).
template <typename DT, bool TRACE, int NB, int TH>
__global__ void __maxnreg__(sizeof(DT) == 2 ? 48 : 64) k_weigh(const __grid_constant__ BatchArgs<NB> args) {
  using WT = WeighTile<TH>;
  int T;
  const FrameArgs& fa = args.f[batch_frame<NB>(args.tile_first, args.n, (int)blockIdx.x, T)];
  const float2* __restrict__ rays = fa.rays;
  const FramePtrs& fp = fa.fp;
  const Tables& t = fa.t;
  const TraceDev& tr = fa.tr;
  const TileIndex& ti = fa.ti;
  const RigHot& hot = fa.hot;
  pdl_release();
  extern __shared__ __align__(16) unsigned char smem[];
  unsigned long long* s_key = reinterpret_cast<unsigned long long*>(smem + WT::Key);
  unsigned* s_slot = reinterpret_cast<unsigned*>(smem + WT::Slot);
  unsigned* s_lb = reinterpret_cast<unsigned*>(smem + WT::LB);
  const BlockConst& bc = *reinterpret_cast<const BlockConst*>(smem + WT::BC);
  __shared__ unsigned s_claims, s_first;

  int cam, x0, y0;
  tile_of<TH>(ti, T, cam, x0, y0);
  const int W = ti.W[cam], H = ti.H[cam], k1 = ti.k1;
  const unsigned off = (unsigned)ti.off[cam];
  // the camera's and its views' constants and the tile's pair rays (Eq. 4), asynchronously
  const int n_views = hot.use_cons ? k1 : 0;
  const int n_const = WT::const_words(n_views), n_cols = WT::col_words(n_views);
  const float4* const s_cols = reinterpret_cast<const float4*>(smem + WT::BC) + n_const;
  const float4* const s_rows = s_cols + n_cols;
  {
    const float4* gc = reinterpret_cast<const float4*>(t.bconst + cam);
    const float4* ga = t.pray + ti.pray[cam] + (x0 >> 5) * k1 * kPrayColGroup;
    const float4* gb = t.pray + ti.pray[cam] + (((W + 31) >> 5) * kPrayColGroup + (y0 >> 3) * kPrayRowGroup) * k1;
    const int n = n_const + n_cols + WT::row_words(n_views);
    for (int i = threadIdx.x; i < n; i += (int)blockDim.x) {
      const float4* src = i < n_const ? gc + i : i < n_const + n_cols ? ga + (i - n_const) : gb + (i - n_const - n_cols);
      cp_async16(smem + WT::BC + 16 * i, src);
    }
  }
  // warm L2 with the colours of a tile further on: the sum step reads them
  if (threadIdx.x < 2 * TH && T + ti.ahead < t.n_tiles) {
    int pc, px0, py0;
    tile_of<TH>(ti, T + ti.ahead, pc, px0, py0);
    const int row = py0 + (int)(threadIdx.x >> 1);
    if (row < ti.H[pc]) {                     // every address lies inside its image
      const long long li = (long long)row * ti.W[pc] + ((threadIdx.x & 1) ? min(px0 + kTileW, ti.W[pc]) - 1 : px0);
      asm volatile("prefetch.global.L2 [%0];" ::"l"(fp.rgb[pc] + 3 * li));
    }
  }
  if (threadIdx.x == 0) s_claims = 0u;
  if (TRACE) {                              // every pixel as not gated; the gated ones follow
    const float qnan = __int_as_float(0x7fc00000);
    for (int i = threadIdx.x; i < WT::Px; i += (int)blockDim.x) {
      const int x = x0 + (i & (kTileW - 1)), y = y0 + i / kTileW;
      if (x >= W || y >= H) continue;
      const long long g = (long long)off + (long long)y * W + x;
      if (tr.pw) { tr.pw[3 * g] = qnan; tr.pw[3 * g + 1] = qnan; tr.pw[3 * g + 2] = qnan; }
      if (tr.e) tr.e[g] = qnan;
      if (tr.omega) tr.omega[g] = qnan;
      if (tr.nview) tr.nview[g] = -1;
      if (tr.key) tr.key[g] = kKeyEmpty;
    }
  }
  // everything above used only the context's constants; the lists (count step), the coarse table
  // (level step) and every table written below need the earlier kernels
  pdl_wait();
  const TileList<WT::Units> list(t, ti, cam, off, W, H, x0, y0);
  if (list.n == 0) return;                  // uniform over the block
  load_cell_levels<WT::Units>(t, ti, list, cam, W, x0, y0, s_lb);
  cp_async_wait();
  __syncthreads();
#pragma unroll 1
  for (int i = threadIdx.x; i < list.n; i += (int)blockDim.x) {
    int unit;
    const unsigned at = list.at(i, unit);
    const unsigned e = __ldcg(t.lpix + at);
    const float z = Depth<DT>::z(__ldcg(static_cast<const DT*>(t.ldepth) + at)), c = __ldcg(t.lconf + at);
    const int lx = (int)(e & (kTileW - 1)), ly = (int)((e & 0xffu) / kTileW) + unit * kUnitH, x = x0 + lx, y = y0 + ly;
    const unsigned g = off + (unsigned)(y * W + x);                   // W H <= 2^30
    const float rx = __ldg(&rays[bc.cam.ray_x + x].x), ry = __ldg(&rays[bc.cam.ray_y + y].x);
    float P[3], r[3], frac[3];
    int cc[3], kk[3];
    world_point(bc.cam, z, rx, ry, P);                                // Eq. 8
    unsigned lb = kBaseNone;
    if (grid_coords(hot, P, r, cc))
      lb = (e >> 8) != kNoCellNumber ? s_lb[(e >> 8) + (unsigned)(unit * kUnitCells)]
                                     : coarse_lvbase(t, pack_key(0, cc[0], cc[1], cc[2]));
    const unsigned ls = point_slot(lb, r, kk, frac), slot = ls & kBaseNone;
    // representative; number and exponent.  In two words of 64 bits: other blocks raise the key meanwhile,
    // and only a word is read whole
    ulonglong2 rec = make_ulonglong2(0ull, 0ull);
    if (slot != kBaseNone) rec = __ldcg(reinterpret_cast<const ulonglong2*>(t.frec + slot));
    float sh = 0.0f, sl = 0.0f, mu = 0.0f;
    int nview = 0, m = 0;
    if (n_views > 0)
      residual_sum<DT>(&bc, t, cam, k1, TilePairRays<TH>(s_cols, s_rows, k1, lx, ly), fa.rig, hot, rays, fp, z, x, y,
                       sh, sl, nview);
    const float eh = joint_weight(hot, k1, sh, sl, c, mu, m);
    t.wslot[at] = ls;
    t.wmant[at] = mu;
    t.wexp[at] = m;
    if (slot != kBaseNone) {                    // else out of range, or no slot left (reported)
      SlotRec* s = t.frec + slot;
      const unsigned long long key = ((unsigned long long)ordered(c) << 32) | (unsigned)(~g);
      if (rec.x < key) atomicMax(&s->key, key);
      if ((int)(rec.y >> 32) > m) atomicMin(&s->mmin, m);
      if ((unsigned)rec.y == kSlotNone && atomicCAS(&s->head, kSlotNone, kSlotPending) == kSlotNone) {
        const unsigned q = atomicAdd(&s_claims, 1u);
        s_slot[q] = slot;
        s_key[q] = pack_key((int)(ls >> 27), kk[0], kk[1], kk[2]);
      }
    }
    if (TRACE) {
      const float unit_m = fa.unit_m;
      if (tr.pw) {
        tr.pw[3ll * g + 0] = P[0] * unit_m;
        tr.pw[3ll * g + 1] = P[1] * unit_m;
        tr.pw[3ll * g + 2] = P[2] * unit_m;
      }
      if (tr.e) tr.e[g] = eh;
      if (tr.omega) tr.omega[g] = ldexpf(mu, -m);
      if (tr.nview) tr.nview[g] = nview;
      if (tr.key) tr.key[g] = slot != kBaseNone ? pack_key((int)(ls >> 27), kk[0], kk[1], kk[2]) : kKeyEmpty;
    }
  }
  __syncthreads();
  // the cells claimed by the tile: numbers from one counter update, their keys, sums cleared
  const unsigned n = s_claims;
  if (n == 0u) return;                      // uniform over the block
  if (threadIdx.x == 0) s_first = atomicAdd(&t.cnt->n_cells, n);
  __syncthreads();
  for (unsigned q = threadIdx.x; q < n; q += blockDim.x) {
    const unsigned id = s_first + q, slot = s_slot[q];
    t.frec[slot].head = id;
    if ((long long)id < fa.out.max_cells) {
      uint4* a = reinterpret_cast<uint4*>(t.rows + id);
#pragma unroll
      for (int k = 0; k < 4; ++k) a[k] = make_uint4(0u, 0u, 0u, 0u);
      a[4] = make_uint4((unsigned)s_key[q], (unsigned)(s_key[q] >> 32), slot, 0u);
    } else {
      t.fused[id] = slot;                   // past the capacity; a number for each slot at most
    }
  }
}

// ------------------------------------------------------------------ sum step
// rint(v) for 0 <= v < 2^45 as an integer, without 64-bit conversions (terms are below 2^37, as
// weights are below 2: joint_weight): floor(v 2^-22) and rint of the rest (exact: both are
// multiples of ulp(v)) are read off sums with 2^23, and adding the even integer hi 2^22 does not
// change a round-half-even decision.
__device__ __forceinline__ unsigned long long fixed_term(float v) {
  constexpr unsigned kBits = 0x4B000000u;                  // 2^23
  const float h = __fmaf_rd(v, 1.0f / 4194304.0f, 8388608.0f);
  const float lo = __fadd_rn(__fmaf_rn(-__fsub_rn(h, 8388608.0f), 4194304.0f, v), 8388608.0f);
  return (unsigned long long)(__float_as_uint(h) - kBits) * 4194304ull + (__float_as_uint(lo) - kBits);
}

// Shared memory of a warp of the sum step, in 16-byte words: 36 rows of 64 bytes, 32 cell numbers.
constexpr int kSumWarpWords = 36 * 4 + 32 / 4;
constexpr int kTileShares = 16;              // emit blocks that a tile counts representatives for

// Eq. 11: the sums of w, w P and w RGB of each cell as exact integers at the scale 2^-(36 + m_min) of
// its smallest weight exponent, one 64-byte row a cell {w, w frac xyz, w rgb / 256, members}, added
// with 64-bit reductions.  A warp lays the terms of its 32 points out in shared memory; eight lanes
// then take a row each of eight successive points, a lane a term, and send one reduction of 64
// contiguous bytes per run of points of one cell (eight lanes on a row measured 3 times faster than
// a lane a row: the reductions of a row travel together).  8x1280x720: 74 us for 3.73 M points, which
// send 2.87 M rows (2.15 M more than there are cells in the tiles, as only successive points of a
// cell are merged); a probe that did nothing but add rows of 64 bytes sent 75 G a second, 38 us for these,
// so that about half of the time is L2's reductions and the rest the points' own instructions and loads.
// Weigh and sum took 185 us together before the marks of representatives were added here (10 us), where
// one kernel that gathered each tile's cells in shared-memory tables and wrote a record per tile and cell
// for a later walk of the cells' record lists took 211 (tables, records and their barriers: 120).
template <typename DT, int NB, int TH>
__global__ void k_sum(const __grid_constant__ BatchArgs<NB> args) {
  using WT = WeighTile<TH>;
  int T;
  const FrameArgs& fa = args.f[batch_frame<NB>(args.tile_first, args.n, (int)blockIdx.x, T)];
  const float2* __restrict__ rays = fa.rays;
  const Tables& t = fa.t;
  const TileIndex& ti = fa.ti;
  pdl_release();
  // rows of 64 bytes, a spare one after each eight; a row's four 16-byte chunks are permuted by its
  // number so that neither the writes nor the reads conflict
  extern __shared__ __align__(16) unsigned char smem[];
  int cam, x0, y0;
  tile_of<TH>(ti, T, cam, x0, y0);
  const int W = ti.W[cam], H = ti.H[cam];
  const unsigned off = (unsigned)ti.off[cam];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  __shared__ unsigned s_share[kTileShares];
  uint4* const s_row = reinterpret_cast<uint4*>(smem) + warp * kSumWarpWords;
  unsigned* const s_id = reinterpret_cast<unsigned*>(s_row + 36 * 4);
  const CamHot& cc = t.bconst[cam].cam;
  const uint8_t* __restrict__ col = fa.fp.rgb[cam];
  pdl_wait();
  const TileList<WT::Units> list(t, ti, cam, off, W, H, x0, y0);
  const unsigned max_cells = (unsigned)fa.out.max_cells;
  // representatives of the tile by emit block, from the first pixel's on; counted here before they go to
  // the frame's counters (an update a cell took 10 us more on 8x1280x720, 170 us on 16x1024^2)
  const unsigned share0 = (off + (unsigned)(y0 * W + x0)) / (32u * kRankWords);
  if (threadIdx.x < kTileShares) s_share[threadIdx.x] = 0u;
  __syncthreads();
  // beside the tile's points, a part of the coarse entries to clear (no later step reads them)
  {
    const unsigned n_coarse = min(__ldcg(&t.cnt->n_coarse), t.cmask + 1u), step = (unsigned)t.n_tiles * blockDim.x;
    for (unsigned i = (unsigned)T * blockDim.x + threadIdx.x; i < n_coarse; i += step) {
      const unsigned cs = __ldcg(t.cused + i);
      t.coarse[cs].key = kKeyEmpty;
      t.coarse[cs].count = 0u;
    }
  }
  const int term = lane & 7, group = lane >> 3;
#pragma unroll 1
  for (int i0 = warp * 32; i0 < list.n; i0 += (int)blockDim.x) {
    const int i = i0 + lane;
    unsigned id = kSlotNone;
    if (i < list.n) {
      int unit;
      const unsigned at = list.at(i, unit);
      const unsigned ls = __ldcg(t.wslot + at), slot = ls & kBaseNone;
      if (slot != kBaseNone) {
        const uint4 rec = __ldcg(reinterpret_cast<const uint4*>(t.frec + slot));   // representative, number, exponent
        const unsigned e = __ldcg(t.lpix + at);
        const float z = Depth<DT>::z(__ldcg(static_cast<const DT*>(t.ldepth) + at)), mu = __ldcg(t.wmant + at);
        const int sh = __ldcg(t.wexp + at) - (int)rec.w;
        const int x = x0 + (int)(e & (kTileW - 1)), y = y0 + (int)((e & 0xffu) / kTileW) + unit * kUnitH;
        const uint8_t* p3 = col + 3u * (unsigned)(y * W + x);
        const unsigned rgb[3] = {__ldg(p3), __ldg(p3 + 1), __ldg(p3 + 2)};
        float P[3], r[3], frac[3];
        int c[3], kk[3];
        world_point(cc, z, __ldg(&rays[cc.ray_x + x].x), __ldg(&rays[cc.ray_y + y].x), P);
        grid_coords(fa.hot, P, r, c);
        point_slot(ls, r, kk, frac);
        const float w = sh > 62 ? 0.0f : __fmul_rn(mu, pow2f(kFixShift - sh));
        unsigned long long v[8];
        v[0] = fixed_term(w);
#pragma unroll
        for (int a = 0; a < 3; ++a) {
          v[1 + a] = fixed_term(__fmul_rn(w, frac[a]));
          // byte / 256: the byte in the last bits of 2^15
          v[4 + a] = fixed_term(__fmul_rn(w, __fsub_rn(__uint_as_float(0x47000000u | rgb[a]), 32768.0f)));
        }
        v[7] = 1ull;
        if (rec.z < max_cells) {
          id = rec.z;
          const unsigned g = off + (unsigned)(y * W + x);
          if (rec.x == ~g) {                    // the cell's representative
            t.rows[id].mmin = (int)rec.w;       // the emit step would read slots in another order, 4 times slower
            mark_cell(t, g, id);
            const unsigned q = g / (32u * kRankWords) - share0;
            if (q < kTileShares) atomicAdd(&s_share[q], 1u);
            else atomicAdd(&t.bsum[share0 + q], 1u);
          }
        }
        uint4* row = s_row + (lane + (lane >> 3)) * 4;
#pragma unroll
        for (int k = 0; k < 4; ++k)
          row[k ^ ((lane >> 1) & 3)] = make_uint4((unsigned)v[2 * k], (unsigned)(v[2 * k] >> 32), (unsigned)v[2 * k + 1],
                                                  (unsigned)(v[2 * k + 1] >> 32));
      }
    }
    s_id[lane] = id;
    __syncwarp();
    unsigned cur = kSlotNone;
    unsigned long long sum = 0ull;
#pragma unroll
    for (int s = 0; s < 8; ++s) {
      const int p = group * 8 + s;
      const unsigned next = s_id[p];
      const uint2 q = reinterpret_cast<const uint2*>(s_row + (p + group) * 4 + ((term >> 1) ^ ((p >> 1) & 3)))[term & 1];
      if (next != cur) {
        if (cur != kSlotNone) atomicAdd(&t.rows[cur].sum[term], sum);
        cur = next;
        sum = 0ull;
      }
      sum += ((unsigned long long)q.y << 32) | q.x;
    }
    if (cur != kSlotNone) atomicAdd(&t.rows[cur].sum[term], sum);
    __syncwarp();
  }
  __syncthreads();
  if (threadIdx.x < kTileShares && s_share[threadIdx.x]) atomicAdd(&t.bsum[share0 + threadIdx.x], s_share[threadIdx.x]);
}

// ------------------------------------------------------------------ assign step
constexpr size_t align16(size_t v) { return (v + 15) / 16 * 16; }
// The top-k assign step's tile: 32 columns by TH rows, one warp per two rows, two pixels a thread,
// and its shared-memory layout.
// Distinct cells of a tile with shared-memory lists: NL.  In a tile with more distinct cells (sparse,
// noisy tiles only) the cells with two or more members in the tile take the lists and every other
// member files a single-member partial, which is the record the list would have produced for it; if
// even the multi-member cells are too many, every member files alone.
template <int TH>
struct AssignTile {
  static_assert(TH == 8 || TH == 16 || TH == 32, "tile heights");
  static constexpr int Px = kTileW * TH;
  static constexpr int Threads = 16 * TH;
  static constexpr int Units = TH / kUnitH;
  static constexpr int TS = 2 * Px;                         // shared hash positions
  static constexpr int NL = Px / 2;                         // lists
  static constexpr size_t FK = 0;                           // u32 cell slot of a position
  static constexpr size_t CntP = FK + 4 * TS;               // u32 members of a position
  static constexpr size_t FI = CntP + 4 * TS;               // u16 list of a position
  static constexpr size_t EP = align16(FI + 2 * TS);        // u16 hash position of a list
  static constexpr size_t Top = align16(EP + 2 * NL);       // u64[NL][kMaxTopK]
  static constexpr size_t LB = Top + 8 * kMaxTopK * NL;     // u32[Units][kUnitCells]
  static constexpr size_t Bytes = LB + 4 * Units * kUnitCells;
};

// Writes partial p as record pi and pushes it onto its cell's list; true when it is the
// cell's first partial of the frame (the caller then lists the cell).
__device__ __forceinline__ bool file_partial(const Tables& t, Partial& p, unsigned slot, unsigned pi) {
  p.next = atomicExch(&t.frec[slot].head, pi);  // list push
  t.part[pi] = p;
  return p.next == kSlotNone;
}

// Sec. II.5(2)a variant: members are keyed and counted, and a tile keeps each cell's top-k members by C
// (packed (ordered(C) << 32) | ~g keys); the consistency and weights of those members are computed per
// cell by k_reduce_topk.
template <typename DT, bool TRACE, int NB, int TH>
__global__ void __launch_bounds__(AssignTile<TH>::Threads) k_assign_topk(const __grid_constant__ BatchArgs<NB> args) {
  using AT = AssignTile<TH>;
  constexpr int kAssignThreads = AT::Threads, kAssignTS = AT::TS, kAssignNL = AT::NL, kUnits = AT::Units;
  int T;
  const FrameArgs& fa = args.f[batch_frame<NB>(args.tile_first, args.n, (int)blockIdx.x, T)];
  const float2* __restrict__ rays = fa.rays;
  const Tables& t = fa.t;
  const TraceDev& tr = fa.tr;
  const TileIndex& ti = fa.ti;
  const RigHot& hot = fa.hot;
  pdl_release();
  extern __shared__ __align__(16) unsigned char smem[];
  unsigned* s_fk = reinterpret_cast<unsigned*>(smem + AT::FK);
  unsigned* s_cntp = reinterpret_cast<unsigned*>(smem + AT::CntP);
  unsigned short* s_fi = reinterpret_cast<unsigned short*>(smem + AT::FI);
  unsigned short* s_ep = reinterpret_cast<unsigned short*>(smem + AT::EP);
  unsigned long long* s_top = reinterpret_cast<unsigned long long*>(smem + AT::Top);
  unsigned* s_lb = reinterpret_cast<unsigned*>(smem + AT::LB);
  __shared__ unsigned s_n, s_base, s_nm;

  int cam, x0, y0;
  tile_of<TH>(ti, T, cam, x0, y0);
  const int W = ti.W[cam], H = ti.H[cam];
  const unsigned off = (unsigned)ti.off[cam];
  const int lane = threadIdx.x & 31;
  const CamHot& camc = t.bconst[cam].cam;
  // clear the per-position arrays: slot none, count 0
  for (int i = threadIdx.x; i < kAssignTS / 2; i += kAssignThreads) {
    const unsigned v = i < kAssignTS / 4 ? kSlotNone : 0u;
    reinterpret_cast<uint4*>(smem + AT::FK)[i] = make_uint4(v, v, v, v);
  }
  if (threadIdx.x == 0) s_n = 0u;
  // everything above used only the context's constants; the lists (count step), the coarse table
  // (level step) and every table written below need the earlier kernels
  pdl_wait();
  const TileList<kUnits> list(t, ti, cam, off, W, H, x0, y0);
  if (TRACE) {                              // the pixels that are not listed
    __shared__ unsigned s_listed[TH];
    if (threadIdx.x < TH) s_listed[threadIdx.x] = 0u;
    __syncthreads();
    for (int i = threadIdx.x; i < list.n; i += kAssignThreads) {
      int unit;
      const unsigned e = __ldcg(t.lpix + list.at(i, unit)) & 0xffu;
      atomicOr(&s_listed[unit * kUnitH + e / kTileW], 1u << (e & (kTileW - 1)));
    }
    __syncthreads();
    const float qnan = __int_as_float(0x7fc00000);
    for (int i = threadIdx.x; i < AT::Px; i += kAssignThreads) {
      const int lx = i & (kTileW - 1), ly = i / kTileW, x = x0 + lx, y = y0 + ly;
      if (x >= W || y >= H || (s_listed[ly] >> lx) & 1u) continue;
      const long long g = (long long)off + (long long)y * W + x;
      if (tr.pw) { tr.pw[3 * g] = qnan; tr.pw[3 * g + 1] = qnan; tr.pw[3 * g + 2] = qnan; }
      if (tr.e) tr.e[g] = qnan;
      if (tr.omega) tr.omega[g] = qnan;
      if (tr.nview) tr.nview[g] = -1;
      if (tr.key) tr.key[g] = kKeyEmpty;
    }
  }
  if (list.n == 0) return;                  // uniform over the block
  load_cell_levels<kUnits>(t, ti, list, cam, W, x0, y0, s_lb);
  __syncthreads();

  // Eq. 8 and Sec. II.5(1)d-e for each gated point
  bool has[2] = {false, false};
  int hpos[2] = {0, 0};
  unsigned long long pkey[2] = {0ull, 0ull};
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    const int i = threadIdx.x + j * kAssignThreads;
    if (i >= list.n) continue;
    int unit;
    const unsigned at = list.at(i, unit);
    const unsigned e = __ldcg(t.lpix + at);
    const float z = Depth<DT>::z(__ldcg(static_cast<const DT*>(t.ldepth) + at)), c = __ldcg(t.lconf + at);
    const int x = x0 + (int)(e & (kTileW - 1)), y = y0 + (int)((e & 0xffu) / kTileW) + unit * kUnitH;
    const unsigned g = off + (unsigned)(y * W + x);
    float P[3], r[3], frac[3];
    int cc[3], kk[3];
    world_point(camc, z, __ldg(&rays[camc.ray_x + x].x), __ldg(&rays[camc.ray_y + y].x), P);
    unsigned lb = kBaseNone;
    if (grid_coords(hot, P, r, cc))
      lb = (e >> 8) != kNoCellNumber ? s_lb[(e >> 8) + (unsigned)(unit * kUnitCells)]
                                     : coarse_lvbase(t, pack_key(0, cc[0], cc[1], cc[2]));
    const unsigned ls = point_slot(lb, r, kk, frac), slot = ls & kBaseNone;
    unsigned long long fkey = kKeyEmpty;
    if (slot != kBaseNone) {                  // else out of range, or no slot left (reported)
      fkey = pack_key((int)(ls >> 27), kk[0], kk[1], kk[2]);
      pkey[j] = ((unsigned long long)ordered(c) << 32) | (unsigned)(~g);
      bool fresh;
      const int h = local_pos<kAssignTS>(s_fk, slot, fresh);
      hpos[j] = h;
      has[j] = h >= 0;
      if (h < 0) {
        atomicOr(&t.cnt->error, kErrSlots);
      } else {
        if (fresh) {                          // the cell's list
          t.frec[slot].key = fkey;            // the same from every tile
          const int q = (int)atomicAdd(&s_n, 1u);
          s_fi[h] = (unsigned short)q;
          if (q < kAssignNL) {
            s_ep[q] = (unsigned short)h;
#pragma unroll
            for (int a = 0; a < kMaxTopK; ++a) s_top[q * kMaxTopK + a] = 0ull;
          }
        }
        atomicAdd(&s_cntp[h], 1u);
      }
    }
    if (TRACE) {
      const float unit_m = fa.unit_m;
      if (tr.pw) {
        tr.pw[3ll * g + 0] = P[0] * unit_m;
        tr.pw[3ll * g + 1] = P[1] * unit_m;
        tr.pw[3ll * g + 2] = P[2] * unit_m;
      }
      if (tr.nview) tr.nview[g] = -2;         // weighed per cell: gated, weight not evaluated here
      if (tr.key) tr.key[g] = fkey;
    }
  }
  __syncthreads();
  // more cells than lists: the multi-member cells take them (see AssignTile)
  const bool renumber = s_n > (unsigned)kAssignNL;         // the same in every thread
  bool all_alone = false;
  unsigned n_local = s_n;
  if (renumber) {
    if (threadIdx.x == 0) s_nm = 0u;
    __syncthreads();
    for (int h = threadIdx.x; h < kAssignTS; h += kAssignThreads) {
      if (s_fk[h] == kSlotNone) continue;
      int e = kAssignNL;
      if (s_cntp[h] >= 2u) {
        e = min((int)atomicAdd(&s_nm, 1u), kAssignNL);
        if (e < kAssignNL) {
          s_ep[e] = (unsigned short)h;
#pragma unroll
          for (int a = 0; a < kMaxTopK; ++a) s_top[e * kMaxTopK + a] = 0ull;
        }
      }
      s_fi[h] = (unsigned short)e;
    }
    __syncthreads();
    all_alone = s_nm > (unsigned)kAssignNL;
    n_local = all_alone ? 0u : s_nm;
  }
  // reserve the tile's partial records now; the index is needed only at the end
  unsigned base_pi = 0u;
  if (threadIdx.x == 0) base_pi = atomicAdd(&t.cnt->n_partials, n_local);
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    if (!has[j]) continue;
    const int h = hpos[j], e = s_fi[h];
    if (!(all_alone || e >= kAssignNL)) {
      // insert the member into its cell's sorted top-k list; each slot keeps the largest key that
      // reaches it and passes the smaller one down, so the list ends as the k largest keys whatever
      // the order of the atomics
      unsigned long long key = pkey[j];
      for (int q = 0; q < fa.top_k && key; ++q) {
        const unsigned long long old = atomicMax(&s_top[e * kMaxTopK + q], key);
        key = old < key ? old : key;
      }
    } else {                                  // a single-member partial of its own
      Partial p;
      const unsigned slot = s_fk[h];
      p.count = 1u;
      p.top[0] = pkey[j];
#pragma unroll
      for (int a = 1; a < kMaxTopK; ++a) p.top[a] = 0ull;
      const unsigned pi = atomicAdd(&t.cnt->n_partials, 1u);
      if (pi >= t.max_partials) {
        atomicOr(&t.cnt->error, kErrPartials);
      } else if (file_partial(t, p, slot, pi)) {
        const unsigned n = atomicAdd(&t.cnt->n_cells, 1u);
        if (n < t.max_slots) t.fused[n] = slot;
      }
    }
  }
  if (threadIdx.x == 0) s_base = base_pi;
  __syncthreads();
  // one partial record per (tile, cell), pushed onto its cell's list
  for (int e0 = 0; e0 < (int)n_local; e0 += kAssignThreads) {
    const int e = e0 + threadIdx.x;
    bool first = false;
    unsigned slot = 0u;
    if (e < (int)n_local) {
      const unsigned pi = s_base + (unsigned)e;
      if (pi >= t.max_partials) {
        atomicOr(&t.cnt->error, kErrPartials);
      } else {
        const unsigned h = s_ep[e];
        Partial p;
        slot = s_fk[h];
        p.count = s_cntp[h];
#pragma unroll
        for (int a = 0; a < kMaxTopK; ++a) p.top[a] = s_top[e * kMaxTopK + a];
        first = file_partial(t, p, slot, pi);
      }
    }
    // one counter update per warp for the cells claimed in it
    const unsigned claim = __ballot_sync(0xffffffffu, first);
    unsigned nb = 0u;
    if (lane == 0 && claim) nb = atomicAdd(&t.cnt->n_cells, (unsigned)__popc(claim));
    nb = __shfl_sync(0xffffffffu, nb, 0);
    if (first) {
      const unsigned n = nb + __popc(claim & ((1u << lane) - 1u));
      if (n < t.max_slots) t.fused[n] = slot;
    }
  }
}

// ------------------------------------------------------------------ top-k reduce
// Sec. II.5(2) variant, per cell: merge the tiles' top-k lists (the k largest packed
// (ordered(C) << 32) | ~g keys of the union: order-independent), then for each of the
// cell's k representatives recompute the world point (Eq. 8, the same float32 sequence as
// the other steps), its consistency over its camera's K-1 views (Eq. 4-7, global pair rays)
// and omega = C V (Eq. 10), and fuse them (Eq. 11, normalised, weights scaled by the
// largest).  Members are counted over the whole cell; the representative is the cell's top
// member.
// A block merges the lists of 128 / k cells, a thread a cell, then weighs their representatives, a thread
// each, and fuses them, a thread a cell again.  Bound by the latency of the lists, of the scattered samples
// and between the block's steps (33 % of the issue slots).  k = 3, 187,000 cells of 8x1280x720: 73 us; a
// thread a cell throughout, its k representatives one after another, 84 us unrolled and 78 us rolled; k = 6
// on 4x187x146: 12 us instead of 29.  10 blocks an SM (48 registers, spills) 79 us, 6 blocks 89 us; blocks of
// 64 or 32 threads 76 us.
constexpr int kTopThreads = 128;
template <typename DT, int NB>
__global__ void __launch_bounds__(kTopThreads, 8) k_reduce_topk(const __grid_constant__ BatchArgs<NB> args) {
  const FrameArgs& fa = args.f[batch_frame_y<NB>()];
  const RigDev* __restrict__ rigp = fa.rig;
  const float2* __restrict__ rays = fa.rays;
  const FramePtrs& fp = fa.fp;
  const Tables& t = fa.t;
  const OutDev& out = fa.out;
  __shared__ unsigned long long s_key[kTopThreads];                  // a cell's k keys side by side, 0: none
  __shared__ float s_mu[kTopThreads], s_val[6][kTopThreads];         // mantissa; world point and colour
  __shared__ int s_mx[kTopThreads];                                  // exponent of the weight
  pdl_release();
  pdl_wait();
  const RigDev& rig = *rigp;
  const unsigned n_cells = min(t.cnt->n_cells, t.max_slots);
  const unsigned n_coarse = min(t.cnt->n_coarse, t.cmask + 1u);
  const unsigned n_part = min(t.cnt->n_partials, t.max_partials);
  const int K = fa.top_k;
  const unsigned per = (unsigned)(kTopThreads / K);
  for (unsigned i = blockIdx.x * kTopThreads + threadIdx.x; i < n_coarse; i += gridDim.x * kTopThreads) {
    const unsigned cs = t.cused[i];
    t.coarse[cs].key = kKeyEmpty;
    t.coarse[cs].count = 0u;
  }
#pragma unroll 1
  for (unsigned c0 = blockIdx.x * per; c0 < n_cells; c0 += gridDim.x * per) {
    const unsigned i = c0 + threadIdx.x;
    const bool mine = threadIdx.x < per && i < n_cells;
    CellOut cell;
    s_key[threadIdx.x] = 0ull;
    __syncthreads();
    if (mine) {
      const unsigned slot = t.fused[i];
      const SlotRec rec = t.frec[slot];
      unsigned long long top[kMaxTopK];
#pragma unroll
      for (int q = 0; q < kMaxTopK; ++q) top[q] = 0ull;
      unsigned count = 0u, steps = 0u;
      for (unsigned p = rec.head; p != kSlotNone && steps <= n_part; ++steps) {
        const Partial P = t.part[p];
        count += P.count;
        for (int a = 0; a < K; ++a) {           // insert the tile's key a into the sorted list
          unsigned long long key = P.top[a];
#pragma unroll
          for (int q = 0; q < kMaxTopK; ++q) {
            if (q < K && key > top[q]) {
              const unsigned long long tmp = top[q];
              top[q] = key;
              key = tmp;
            }
          }
        }
        p = P.next;
      }
      if (steps > n_part) atomicOr(&t.cnt->error, kErrList);
#pragma unroll
      for (int q = 0; q < kMaxTopK; ++q)
        if (q < K) s_key[threadIdx.x * K + q] = top[q];
      cell.count = count;
      cell.key = rec.key;
      *reinterpret_cast<uint4*>(t.frec + slot) = kSlotClear;         // ready for the next frame
    }
    __syncthreads();
    if (s_key[threadIdx.x]) {                   // weight and world point of a representative
      const unsigned g = ~(unsigned)(s_key[threadIdx.x] & 0xffffffffull);
      if ((long long)g >= rig.n_px) {           // not a pixel: a corrupted list (reported)
        atomicOr(&t.cnt->error, kErrList);
        s_key[threadIdx.x] = 0ull;
      } else {
        int cam = 0;
        for (int lo = 0, hi = fa.ti.n_cams - 1; lo <= hi;) {
          const int mid = (lo + hi) >> 1;
          if (fa.ti.off[mid] <= (long long)g) { cam = mid; lo = mid + 1; } else { hi = mid - 1; }
        }
        const int W = fa.ti.W[cam];
        const unsigned li = g - (unsigned)fa.ti.off[cam];
        const int y = (int)(li / (unsigned)W), x = (int)(li - (unsigned)y * (unsigned)W);
        const float z = Depth<DT>::z(static_cast<const DT*>(fp.depth[cam])[li]);
        const float c = fp.conf[cam][li];
        const uint8_t* px = fp.rgb[cam] + 3 * (long long)li;
        const BlockConst* bc = t.bconst + cam;
        float P[3], mu, sh = 0.0f, sl = 0.0f;
        int mx, nview = 0;
        s_val[3][threadIdx.x] = (float)px[0];
        s_val[4][threadIdx.x] = (float)px[1];
        s_val[5][threadIdx.x] = (float)px[2];
        world_point(bc->cam, z, __ldg(&rays[bc->cam.ray_x + x].x), __ldg(&rays[bc->cam.ray_y + y].x), P);
        if (fa.hot.use_cons && rig.k1 > 0)
          residual_sum<DT>(bc, t, cam, rig.k1, GlobalPairRays(t.pray + fa.ti.pray[cam], W, rig.k1, x, y),
                           rigp, fa.hot, rays, fp, z, x, y, sh, sl, nview);
        joint_weight(fa.hot, rig.k1, sh, sl, c, mu, mx);
        s_mu[threadIdx.x] = mu;
        s_mx[threadIdx.x] = mx;
#pragma unroll
        for (int a = 0; a < 3; ++a) s_val[a][threadIdx.x] = P[a];
      }
    }
    __syncthreads();
    if (mine) {
      const int e0 = (int)threadIdx.x * K;
      int mmin = INT_MAX;
      bool any = false;
      for (int q = 0; q < K; ++q)
        if (s_key[e0 + q]) {
          mmin = min(mmin, s_mx[e0 + q]);
          any = true;
        }
      float sw = 0.0f, sp[3] = {0.0f, 0.0f, 0.0f}, sc[3] = {0.0f, 0.0f, 0.0f};
      for (int q = 0; q < K; ++q) {             // Eq. 11, weights relative to the largest
        if (!s_key[e0 + q]) continue;
        const int sh = s_mx[e0 + q] - mmin;
        const float w = sh > 126 ? 0.0f : __fmul_rn(s_mu[e0 + q], pow2f(-sh));
        sw = __fadd_rn(sw, w);
#pragma unroll
        for (int a = 0; a < 3; ++a) {
          sp[a] = __fmaf_rn(w, s_val[a][e0 + q], sp[a]);
          sc[a] = __fmaf_rn(w, s_val[3 + a][e0 + q], sc[a]);
        }
      }
      const float inv = any ? __frcp_rn(sw) : __int_as_float(0x7fc00000);
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        cell.pos[a] = __fmul_rn(__fmul_rn(sp[a], inv), out.unit_f);
        cell.rgb[a] = __fmul_rn(sc[a], inv);
      }
      cell.weight = any ? ldexpf(sw, -min(mmin, 1 << 30)) : 0.0f;
      const bool have = s_key[e0] != 0ull;
      const unsigned g = have ? ~(unsigned)(s_key[e0] & 0xffffffffull) : 0xffffffffu;
      cell.rep = g;
      cell.pad = 0u;
      if ((long long)i < out.max_cells) {
        t.staged[i] = cell;
        if (have) {                             // g < n_px (checked above)
          mark_cell(t, g, i);
          // one update for the lanes whose pixels fall into one share
          const unsigned share = g / (32u * kRankWords), peers = __match_any_sync(__activemask(), share);
          if ((threadIdx.x & 31) == __ffs(peers) - 1) atomicAdd(&t.bsum[share], (unsigned)__popc(peers));
        }
      }
    }
    __syncthreads();                            // the keys are free again
  }
}

// ------------------------------------------------------------------ point-wise (No SA)
// Table II's "No SA" ablation: fusion without the spatial hash, every gated pixel an output
// point with its own joint weight.  Per pixel: Eq. 8-9 (gate, back-projection), Eq. 4-7 over
// the camera's K-1 views (the same evaluation and global pair rays as the top-k reduce step)
// and Eq. 10; outputs are indexed by the global pixel index (position in
// metres and weight; NaN position and weight 0 for pixels that are not gated, 8-bit colour
// copied), so the cloud is in pixel order without a compaction pass.
// A block takes a tile of 32 columns by 16 rows, as the weigh step does: the gated pixels compacted in
// shared memory and weighed with full warps, the view constants and pair rays staged, and the results
// laid out by pixel for stores in order.  The tile's samples and colours are asked for first, from sizes
// and offsets in the constant bank, and few tiles take more threads a block, down to a pixel a thread
// (weigh_threads).  8x1280x720 (7.4 Mpx): 117 us with half of the pixels gated, 49 us with 2 %; without
// these two points 129 and 66 us, and a thread a pixel with rays and view constants from global memory
// 189 and 57 us.  2x160x120: 8.2, 10.4 and 7.8 us.  Bound by the residual's instructions.
struct PointsTile {
  static constexpr int H = 16, Px = kTileW * H;
  static constexpr size_t Out = 0;                                 // f32[4][Px]: pos xyz, weight, by pixel
  static constexpr size_t P = Out + 16 * Px;                       // u16[Px]: the gated pixels
  static constexpr size_t BC = P + 2 * Px;                         // constants, column and row pair rays
  static constexpr size_t smem(int k1) { return BC + 16 * (size_t)(4 * (1 + k1) + k1 * (kPrayColGroup + H / 8 * kPrayRowGroup)); }
};

template <typename DT, int Threads>
__global__ void __maxnreg__(sizeof(DT) == 2 ? 48 : 64)
k_points(const RigDev* __restrict__ rigp, const __grid_constant__ RigHot hot, const float2* __restrict__ rays,
         const __grid_constant__ FramePtrs fp, const __grid_constant__ Tables t, const __grid_constant__ TileIndex ti,
         PointsDev out) {
  using PT = PointsTile;
  constexpr int kWarps = Threads / 32, kRows = PT::H / kWarps;      // rows a warp
  static_assert(kRows * kWarps == PT::H, "whole rows a warp");
  extern __shared__ __align__(16) unsigned char smem[];
  float* const s_out = reinterpret_cast<float*>(smem + PT::Out);
  unsigned short* const s_p = reinterpret_cast<unsigned short*>(smem + PT::P);
  const BlockConst& bc = *reinterpret_cast<const BlockConst*>(smem + PT::BC);
  __shared__ unsigned s_n, s_valid;
  const int cam = blockIdx.y, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int W = ti.W[cam], H = ti.H[cam], k1 = ti.k1, tiles_x = (W + kTileW - 1) / kTileW;
  int tx;
  const int y0 = fast_div((int)blockIdx.x, tiles_x, ti.div_x[cam], tx) * PT::H, x0 = tx * kTileW;
  if (y0 >= H) return;                                              // uniform over the block
  const int w = min(kTileW, W - x0);
  const long long p0 = (long long)y0 * W + x0;                      // the tile's first pixel
  const DT* __restrict__ dep = static_cast<const DT*>(fp.depth[cam]) + p0;
  const float* __restrict__ cf = fp.conf[cam] + p0;
  const uint8_t* __restrict__ col = fp.rgb[cam] + 3 * p0;
  const float qnan = __int_as_float(0x7fc00000);
  DT D[kRows];
  float c[kRows];
  uint8_t rgb[kRows][3];
#pragma unroll
  for (int k = 0; k < kRows; ++k) {
    const int y = warp + kWarps * k;
    const unsigned li = (unsigned)(y * W + lane);                   // W H <= 2^30
    D[k] = (DT)0;
    c[k] = 0.0f;
    if (lane < w && y0 + y < H) {
      D[k] = dep[li];
      c[k] = cf[li];
    }
#pragma unroll
    for (int a = 0; a < 3; ++a)                                     // a row's colours, a byte a lane
      rgb[k][a] = lane + 32 * a < 3 * w && y0 + y < H ? __ldg(col + 3u * (unsigned)(y * W) + lane + 32 * a) : (uint8_t)0;
  }
  const int n_views = hot.use_cons ? k1 : 0, n_const = 4 * (1 + n_views), n_cols = n_views * kPrayColGroup;
  const float4* const s_cols = reinterpret_cast<const float4*>(smem + PT::BC) + n_const;
  {
    const float4* gc = reinterpret_cast<const float4*>(t.bconst + cam);
    const float4* ga = t.pray + ti.pray[cam] + (x0 >> 5) * k1 * kPrayColGroup;
    const float4* gb = t.pray + ti.pray[cam] + (tiles_x * kPrayColGroup + (y0 >> 3) * kPrayRowGroup) * k1;
    const int n = n_const + n_cols + n_views * (PT::H / 8) * kPrayRowGroup;
    for (int i = threadIdx.x; i < n; i += Threads) {
      const float4* src = i < n_const ? gc + i : i < n_const + n_cols ? ga + (i - n_const) : gb + (i - n_const - n_cols);
      cp_async16(smem + PT::BC + 16 * i, src);
    }
  }
  if (threadIdx.x == 0) { s_n = 0u; s_valid = 0u; }
  __syncthreads();
  const long long g0 = ti.off[cam] + p0;
  unsigned nv = 0u;
#pragma unroll
  for (int k = 0; k < kRows; ++k) {
    const int r = warp + kWarps * k, i = r * kTileW + lane;
    const bool valid = Depth<DT>::valid(D[k]);
    const bool gated = valid && (!hot.use_conf || c[k] > hot.tau);  // Eq. 9
    nv += __popc(__ballot_sync(0xffffffffu, valid));
    const unsigned m = __ballot_sync(0xffffffffu, gated);
    unsigned base = 0u;
    if (lane == 0 && m) base = atomicAdd(&s_n, (unsigned)__popc(m));
    base = __shfl_sync(0xffffffffu, base, 0);
    if (gated) {
      s_p[base + __popc(m & ((1u << lane) - 1u))] = (unsigned short)i;
      s_out[3 * i] = Depth<DT>::z(D[k]);                            // until the pixel is weighed
      s_out[3 * i + 1] = c[k];
    } else {
      s_out[3 * i] = qnan;
      s_out[3 * i + 1] = qnan;
      s_out[3 * i + 2] = qnan;
      s_out[3 * PT::Px + i] = 0.0f;
    }
#pragma unroll
    for (int a = 0; a < 3; ++a)
      if (lane + 32 * a < 3 * w && y0 + r < H) out.rgb[3 * (g0 + (long long)r * W) + lane + 32 * a] = rgb[k][a];
  }
  if (lane == 0 && nv) atomicAdd(&s_valid, nv);
  cp_async_wait();
  __syncthreads();
  const int n = (int)s_n;
#pragma unroll 1
  for (int i = threadIdx.x; i < n; i += Threads) {
    const int q = s_p[i], lx = q & (kTileW - 1), ly = q / kTileW, x = x0 + lx, y = y0 + ly;
    const float z = s_out[3 * q], cq = s_out[3 * q + 1];
    float P[3];
    world_point(bc.cam, z, __ldg(&rays[bc.cam.ray_x + x].x), __ldg(&rays[bc.cam.ray_y + y].x), P);   // Eq. 8
    float sh = 0.0f, sl = 0.0f, mu;
    int nview = 0, m;
    if (n_views > 0)
      residual_sum<DT>(&bc, t, cam, k1, TilePairRays<PT::H>(s_cols, s_cols + n_cols, k1, lx, ly), rigp, hot, rays, fp, z, x,
                       y, sh, sl, nview);
    joint_weight(hot, k1, sh, sl, cq, mu, m);                         // Eq. 7, 10
#pragma unroll
    for (int a = 0; a < 3; ++a) s_out[3 * q + a] = __fmul_rn(P[a], out.unit_f);
    s_out[3 * PT::Px + q] = ldexpf(mu, -min(m, 1 << 30));
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < kRows; ++k) {                                   // a warp a row
    const int r = warp + kWarps * k;
    if (y0 + r >= H) break;
    const long long g = g0 + (long long)r * W;
#pragma unroll
    for (int a = 0; a < 3; ++a)
      if (lane + 32 * a < 3 * w) out.pos[3 * g + lane + 32 * a] = s_out[3 * r * kTileW + lane + 32 * a];
    if (lane < w) out.weight[g + lane] = s_out[3 * PT::Px + r * kTileW + lane];
  }
  if (threadIdx.x == 0) {
    if (s_valid) atomicAdd(&out.counts[0], (unsigned long long)s_valid);
    if (n) atomicAdd(&out.counts[1], (unsigned long long)n);
  }
}

// ------------------------------------------------------------------ emit
// Block b of a frame takes pixels [8192 b, 8192 (b + 1)): the ranks of their representatives follow from
// the earlier blocks' counts and the bits of the block's own 256 words, which it leaves clear for the next frame; then a thread a cell, in rank order, so that
// the output is written in order: Eq. 11 from the cell's sums, or the cell that the top-k reduce step
// staged.  One block more writes the frame's statistics and clears the counters.  Bound by the latency of
// the scattered row reads: 19 us for 187,000 cells, 116 us for 1.7 M; a reduce, a scan and an emit kernel
// and a clear before the frame took 22 + 12 + 17 + 6 us and 255 + 25 + 134 + 6 us.  All blocks together read
// the square of their number / 2 counts, from L2: 64x3840x2160 (64,800 blocks, 61 M cells) takes 4.24 ms, and
// 4.15 with a kernel before it that adds the counts up by 256, so that even the largest frames accepted (8
// times as many pixels) spend a few percent of the frame on it.
template <bool TOPK, int NB>
__global__ void __launch_bounds__(kThreads) k_emit(const __grid_constant__ BatchArgs<NB> args) {
  static_assert(kRankWords == kThreads, "a bitmap word a thread");
  __shared__ unsigned s_w[kThreads / 32][2];
  __shared__ unsigned short s_px[32 * kRankWords];
  const Tables& t = args.f[batch_frame_y<NB>()].t;
  const OutDev& out = args.f[batch_frame_y<NB>()].out;
  pdl_release();
  pdl_wait();
  const int b = (int)blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (b >= t.n_wblocks) {
    if (b == t.n_wblocks) frame_stats<TOPK>(t, out);
    return;
  }
  const unsigned n_cells = TOPK ? 0u : __ldcg(&t.cnt->n_cells);      // for the end: all in flight together
  unsigned before = 0u;
  for (int i = threadIdx.x; i < b; i += kThreads) before += __ldcg(t.bsum + i);
  const long long w = (long long)b * kRankWords + threadIdx.x;
  unsigned v = w < t.n_words ? __ldcg(t.bitmap + w) : 0u;
  if (v) t.bitmap[w] = 0u;
  const unsigned mine = __popc(v);
  unsigned x = mine;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  before = __reduce_add_sync(0xffffffffu, before);
  if (lane == 31) {
    s_w[warp][0] = x;
    s_w[warp][1] = before;
  }
  __syncthreads();
  unsigned base = 0u, at = x - mine, total = 0u;
#pragma unroll
  for (int k = 0; k < kThreads / 32; ++k) {
    base += s_w[k][1];
    if (k < warp) at += s_w[k][0];
    total += s_w[k][0];
  }
  for (; v; v &= v - 1u) s_px[at++] = (unsigned short)(threadIdx.x * 32 + __ffs(v) - 1);
  __syncthreads();
  for (unsigned r = threadIdx.x; r < total; r += kThreads) {
    const unsigned g = (unsigned)b * (32u * kRankWords) + s_px[r];
    const unsigned id = __ldcg(t.cell_at + g);
    const unsigned long long rank = (unsigned long long)base + r;
    if (rank >= (unsigned long long)out.max_cells) continue;         // marked cells never exceed it
    CellOut c;
    if constexpr (TOPK) {
      c = t.staged[id];
    } else {
      const CellRow* row = t.rows + id;
      unsigned long long S[8];
#pragma unroll
      for (int a = 0; a < 4; ++a) {
        const ulonglong2 p = __ldcg(reinterpret_cast<const ulonglong2*>(row->sum) + a);
        S[2 * a] = p.x;
        S[2 * a + 1] = p.y;
      }
      const ulonglong2 p = __ldcg(reinterpret_cast<const ulonglong2*>(&row->key));
      const unsigned slot = (unsigned)p.y;
      const int mmin = (int)(p.y >> 32);
      *reinterpret_cast<uint4*>(t.frec + slot) = kSlotClear;         // ready for the next frame
      // Eq. 11 in float32: position = edge (k + S_k / S_0), colour = 256 S_c / S_0,
      // weight = S_0 2^-(36 + mmin); each result is within a few float32 roundings
      const int l = (int)(p.x >> 60);
      const float edge = __fmul_rn(out.s0_m, pow2f(-l));
      const float Wf = u64_to_f32(S[0]);
      const float inv = S[0] ? __frcp_rn(Wf) : __int_as_float(0x7fc00000);
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        const int ka = (int)((p.x >> (40 - 20 * a)) & 0xfffff) - kKeyBias;
        c.pos[a] = __fmaf_rn(edge, (float)ka, __fmul_rn(edge, __fmul_rn(u64_to_f32(S[1 + a]), inv)));
        c.rgb[a] = __fmul_rn(256.0f, __fmul_rn(u64_to_f32(S[4 + a]), inv));
      }
      c.weight = ldexpf(Wf, -kFixShift - min(mmin, 1 << 30));
      c.count = (unsigned)S[7];
      c.key = p.x;
    }
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      out.pos[3 * rank + a] = c.pos[a];
      out.rgb[3 * rank + a] = c.rgb[a];
    }
    out.weight[rank] = c.weight;
    out.count[rank] = c.count;
    out.rep[rank] = g;
    out.key[rank] = c.key;
  }
  // slots of cells past the output's capacity (reported)
  for (unsigned i = (unsigned)out.max_cells + (unsigned)b * kThreads + threadIdx.x; i < min(n_cells, t.max_slots);
       i += (unsigned)t.n_wblocks * kThreads)
    *reinterpret_cast<uint4*>(t.frec + t.fused[i]) = kSlotClear;
}

// Served frames: the cloud's first n cells (n = min(n_cells, capacity)) and the
// statistics, written into pinned host memory through its mapped addresses.
__global__ void __launch_bounds__(kThreads) k_copyout(fuseflow_cloud src, HostOutDev dst) {
  const long long nc = src.stats->n_cells;
  const long long n = nc < dst.capacity ? nc : dst.capacity;
  if (blockIdx.x == 0 && threadIdx.x == 0) *dst.stats = *src.stats;
  // word ranges of the six arrays, back to back: pos 3n, rgb 3n, weight n, count n,
  // rep n, key 2n
  const long long total = 11 * n;
  for (long long w = blockIdx.x * (long long)blockDim.x + threadIdx.x; w < total;
       w += (long long)gridDim.x * blockDim.x) {
    long long o = w;
    const uint32_t* from;
    uint32_t* to;
    if (o < 3 * n) { from = reinterpret_cast<const uint32_t*>(src.pos); to = reinterpret_cast<uint32_t*>(dst.pos); }
    else if ((o -= 3 * n) < 3 * n) { from = reinterpret_cast<const uint32_t*>(src.rgb); to = reinterpret_cast<uint32_t*>(dst.rgb); }
    else if ((o -= 3 * n) < n) { from = reinterpret_cast<const uint32_t*>(src.weight); to = reinterpret_cast<uint32_t*>(dst.weight); }
    else if ((o -= n) < n) { from = src.count; to = dst.count; }
    else if ((o -= n) < n) { from = src.rep; to = dst.rep; }
    else { o -= n; from = reinterpret_cast<const uint32_t*>(src.key); to = reinterpret_cast<uint32_t*>(dst.key); }
    if (to) to[o] = from[o];
  }
}

// ------------------------------------------------------------------ Eq. 12 (MC error)
// Per point P_k (world, metres): the cameras that see it (in front, nearest pixel inside
// the image, valid D_i there) and the mean of |z(T_i P_k) - D_i(pi(T_i P_k))| over them.
// Each block leaves the sum (depth units) and the number of points with a visible camera
// in bsum/bcnt; the host adds the blocks in order, so the mean does not depend on timing.
constexpr int kMcBlocks = 1024;

template <typename DT>
__global__ void __launch_bounds__(kThreads) k_mc(const RigDev* __restrict__ rigp, FramePtrs fp,
                                                 const float* __restrict__ pos, long long n,
                                                 float inv_unit, float unit_m, float occl_u,
                                                 float* err, int* nvis, double* bsum,
                                                 long long* bcnt) {
  __shared__ double s_sum[kThreads / 32];
  __shared__ long long s_cnt[kThreads / 32];
  const RigDev& rig = *rigp;
  double tsum = 0.0;
  long long tcnt = 0;
  for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < n;
       k += (long long)gridDim.x * blockDim.x) {
    const float P[3] = {__fmul_rn(pos[3 * k], inv_unit), __fmul_rn(pos[3 * k + 1], inv_unit),
                        __fmul_rn(pos[3 * k + 2], inv_unit)};
    float sum = 0.0f;
    int vis = 0;
    for (int i = 0; i < rig.n_cams; ++i) {
      const CamDev& C = rig.cam[i];
      const float d[3] = {__fsub_rn(P[0], C.cwc[0]), __fsub_rn(P[1], C.cwc[1]), __fsub_rn(P[2], C.cwc[2])};
      float a[3];
#pragma unroll
      for (int q = 0; q < 3; ++q)                     // T_i P = R (P - c), R = Rwc^T
        a[q] = __fmaf_rn(C.Rwc[q], d[0], __fmaf_rn(C.Rwc[3 + q], d[1], __fmul_rn(C.Rwc[6 + q], d[2])));
      if (!(a[2] > 0.0f)) continue;
      const float fu = __fadd_rn(__fmaf_rn(C.fx, __fdiv_rn(a[0], a[2]), C.cx), 0.5f);
      const float fv = __fadd_rn(__fmaf_rn(C.fy, __fdiv_rn(a[1], a[2]), C.cy), 0.5f);
      if (!(fu >= 0.0f && fu < (float)C.W && fv >= 0.0f && fv < (float)C.H)) continue;
      const int px = (int)fu, py = (int)fv;            // floor, both non-negative
      const DT D = __ldg(static_cast<const DT*>(fp.depth[i]) + (long long)py * C.W + px);
      if (!Depth<DT>::valid(D)) continue;
      const float zD = Depth<DT>::z(D);
      if (a[2] > __fadd_rn(zD, occl_u)) continue;       // hidden behind the observed surface
      sum = __fadd_rn(sum, fabsf(__fsub_rn(a[2], zD)));
      ++vis;
    }
    const float e = vis ? __fdiv_rn(sum, (float)vis) : __int_as_float(0x7fc00000);
    if (err) err[k] = vis ? __fmul_rn(e, unit_m) : e;
    if (nvis) nvis[k] = vis;
    if (vis) {
      tsum += (double)e;
      ++tcnt;
    }
  }
  // fixed-order block reduction
  for (int o = 16; o > 0; o >>= 1) {
    tsum += __shfl_down_sync(0xffffffffu, tsum, o);
    tcnt += __shfl_down_sync(0xffffffffu, tcnt, o);
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (lane == 0) { s_sum[warp] = tsum; s_cnt[warp] = tcnt; }
  __syncthreads();
  if (threadIdx.x == 0) {
    double bs = 0.0;
    long long bc = 0;
    for (int w = 0; w < kThreads / 32; ++w) { bs += s_sum[w]; bc += s_cnt[w]; }
    bsum[blockIdx.x] = bs;
    bcnt[blockIdx.x] = bc;
  }
}

// ------------------------------------------------------------------ Eq. 3 confidence
// One 128x32 pixel tile per block, staged with its one-pixel halo in shared memory (raw
// depth samples; vector loads for the interior columns).  Each thread computes four
// consecutive pixels in each of four rows, 8 apart, and stores each quadruple as one float4;
// the four windows share one load of their 3x6 samples, and each window's variance is taken
// relative to its centre depth.  Depth
// gradient G: central difference where both neighbours are valid, one-sided with one, 0
// with none; sigma_local: population variance of the window's valid depths (m^2); C is
// normalised by alpha + gamma and is 0 where the depth is invalid.
// 7.4 Mpx of uint16: 28.7 us, bound by instruction issue (about 110 instructions a pixel; 150, and 37 us,
// with each window's count and sum taken over its nine samples and each sample converted and tested apart).
constexpr int kConfW = 128, kConfH = 32;

// Six samples of a row from p on (p + 1 on an 8-byte boundary) as depths, 0 where invalid, and validity
// 1 or 0.
__device__ __forceinline__ void load_six(const uint16_t* p, float z[6], float v[6]) {
  const uint2 u = *reinterpret_cast<const uint2*>(p + 1);
  const unsigned d[6] = {p[0], u.x & 0xffffu, u.x >> 16, u.y & 0xffffu, u.y >> 16, p[5]};
#pragma unroll
  for (int c = 0; c < 6; ++c) {                           // the integer in the last bits of 2^23
    z[c] = __fsub_rn(__uint_as_float(0x4B000000u | d[c]), 8388608.0f);
    v[c] = fminf(z[c], 1.0f);
  }
}
__device__ __forceinline__ void load_six(const float* p, float z[6], float v[6]) {
  const float4 u = *reinterpret_cast<const float4*>(p + 1);
  const float d[6] = {p[0], u.x, u.y, u.z, u.w, p[5]};
#pragma unroll
  for (int c = 0; c < 6; ++c) {
    const bool ok = Depth<float>::valid(d[c]);
    z[c] = ok ? d[c] : 0.0f;
    v[c] = ok ? 1.0f : 0.0f;
  }
}

template <typename DT>
__global__ void __launch_bounds__(kThreads) k_confidence(ConfArgs a) {
  constexpr int kVec = 16 / sizeof(DT);                  // samples per 16-byte load
  constexpr int kRowVecs = kConfW / kVec;
  constexpr int kOff = kVec;                             // tile column c at c + kOff: the
  constexpr int kRow = kConfW + 2 * kVec;                // interior starts 16-byte aligned
  __shared__ __align__(16) DT t[kConfH + 2][kRow];
  const int cam = blockIdx.z;
  const int W = a.W[cam], H = a.H[cam];
  const int x0 = blockIdx.x * kConfW, y0 = blockIdx.y * kConfH;
  if (x0 >= W || y0 >= H) return;                       // uniform over the block
  const DT* __restrict__ dep = static_cast<const DT*>(a.depth[cam]);
  const bool vec_ok = (W % kVec) == 0 && ((reinterpret_cast<uintptr_t>(dep) & 15) == 0);
  // interior columns: rows y0-1 .. y0+8, 16-byte loads where the whole vector is inside
  for (int i = threadIdx.x; i < (kConfH + 2) * kRowVecs; i += kThreads) {
    const int r = i / kRowVecs, v = i - r * kRowVecs;
    const int y = y0 - 1 + r, x = x0 + v * kVec;
    DT* dst = &t[r][kOff + v * kVec];
    if (y >= 0 && y < H && vec_ok && x + kVec <= W) {
      *reinterpret_cast<uint4*>(dst) = __ldcs(reinterpret_cast<const uint4*>(dep + (long long)y * W + x));
    } else {
#pragma unroll
      for (int k = 0; k < kVec; ++k)
        dst[k] = (y >= 0 && y < H && x + k < W) ? dep[(long long)y * W + x + k] : (DT)0;
    }
  }
  // halo columns x0-1 and x0+128 (invalid outside the image)
  if (threadIdx.x < 2 * (kConfH + 2)) {
    const int r = threadIdx.x >> 1, side = threadIdx.x & 1;
    const int y = y0 - 1 + r, x = side ? x0 + kConfW : x0 - 1;
    t[r][side ? kOff + kConfW : kOff - 1] = (y >= 0 && y < H && x >= 0 && x < W) ? dep[(long long)y * W + x] : (DT)0;
  }
  __syncthreads();
  const int tx = threadIdx.x & 31, xb = x0 + 4 * tx;
  if (xb >= W) return;
  const int c0 = kOff + 4 * tx - 1;                       // smem column of pixel xb - 1
  for (int ty = threadIdx.x / 32; ty < kConfH; ty += kThreads / 32) {
    const int y = y0 + ty;
    if (y >= H) break;
    // the 3x6 samples of the thread's four windows, once, as depth z (0 where invalid) and validity v
    // (1 or 0); per column of three, the sums of both
    float zz[3][6], vv[3][6], nc[6], sc[6];
#pragma unroll
    for (int r = 0; r < 3; ++r) load_six(&t[ty + r][c0], zz[r], vv[r]);
#pragma unroll
    for (int c = 0; c < 6; ++c) {
      nc[c] = __fadd_rn(__fadd_rn(vv[0][c], vv[1][c]), vv[2][c]);
      sc[c] = __fadd_rn(__fadd_rn(zz[0][c], zz[1][c]), zz[2][c]);
    }
    float res[4];
#pragma unroll
    for (int p = 0; p < 4; ++p) {
      const float z0 = zz[1][p + 1];
      // window variance relative to the centre sample (one pass: the centre is one of the
      // samples, so the cancellation costs at most a factor 9 in relative precision); a sample's
      // distance e is z - v z0, 0 where it is invalid
      float e[3][3], sq = 0.0f, sm = 0.0f;
#pragma unroll
      for (int r = 0; r < 3; ++r)
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          if (r == 1 && c == 1) continue;
          e[r][c] = __fmaf_rn(vv[r][p + c], -z0, zz[r][p + c]);
          sq = __fmaf_rn(e[r][c], e[r][c], sq);
          if (sizeof(DT) == 4) sm = __fadd_rn(sm, e[r][c]);
        }
      const float n = __fadd_rn(__fadd_rn(nc[p], nc[p + 1]), nc[p + 2]);
      // sums of up to nine 16-bit samples, and n z0, are exact in float32
      if (sizeof(DT) == 2) sm = __fmaf_rn(n, -z0, __fadd_rn(__fadd_rn(sc[p], sc[p + 1]), sc[p + 2]));
      // gradient: half the difference of two valid neighbours, else the one-sided difference
      float g[2];
#pragma unroll
      for (int axis = 0; axis < 2; ++axis) {
        const float vm = axis == 0 ? vv[1][p] : vv[0][p + 1], vp = axis == 0 ? vv[1][p + 2] : vv[2][p + 1];
        float diff;
        if (sizeof(DT) == 2) {                            // differences of 16-bit samples are exact
          diff = __fsub_rn(axis == 0 ? e[1][2] : e[2][1], axis == 0 ? e[1][0] : e[0][1]);
        } else {
          const float zm = axis == 0 ? zz[1][p] : zz[0][p + 1], zp = axis == 0 ? zz[1][p + 2] : zz[2][p + 1];
          diff = __fsub_rn(vp != 0.0f ? zp : z0, vm != 0.0f ? zm : z0);
        }
        g[axis] = __fmul_rn(__fmul_rn(diff, __fmaf_rn(-0.5f * vm, vp, 1.0f)), a.scale);
      }
      const float G2 = __fmaf_rn(g[0], g[0], __fmul_rn(g[1], g[1]));
      const float G = G2 > 0.0f ? __fmul_rn(G2, rsqrtf(G2)) : 0.0f;   // |g|, a few ulp
      const float rn = __fdividef(1.0f, n);
      const float var = __fmul_rn(fmaxf(__fmul_rn(__fsub_rn(sq, __fmul_rn(__fmul_rn(sm, sm), rn)), rn), 0.0f),
                                  __fmul_rn(a.scale, a.scale));
      const float ta = __fdividef(a.alpha, __fmaf_rn(a.beta, G, 1.0f));
      const float tb = __fdividef(a.gamma, __fmaf_rn(a.delta, var, 1.0f));
      res[p] = vv[1][p + 1] != 0.0f ? __fmul_rn(__fadd_rn(ta, tb), a.inv_ag) : 0.0f;
    }
    float* __restrict__ out = a.out[cam] + (long long)y * W + xb;
    if (xb + 4 <= W && (W & 3) == 0 && ((reinterpret_cast<uintptr_t>(a.out[cam]) & 15) == 0)) {
      __stcs(reinterpret_cast<float4*>(out), make_float4(res[0], res[1], res[2], res[3]));
    } else {
#pragma unroll
      for (int p = 0; p < 4; ++p)
        if (xb + p < W) out[p] = res[p];
    }
  }
}

__global__ void k_init_tables(Tables t, unsigned fcap, unsigned ccap) {
  const unsigned n = max(fcap, ccap);
  for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    if (i < fcap) {
      t.frec[i].key = 0ull;
      t.frec[i].head = kSlotNone;
      t.frec[i].mmin = INT_MAX;
    }
    if (i < ccap) {
      t.coarse[i].key = kKeyEmpty;
      t.coarse[i].count = 0u;
      t.coarse[i].lvbase = 0u;
    }
  }
}

// ------------------------------------------------------------------ depth screen
// D^r of Eq. 8 (stated rule: include/fuseflow.h, fuseflow_params): a valid sample within
// the depth-unit bounds is kept unless a valid in-bounds 4-neighbour differs from it by more
// than edge_rel times its value; every decision in float32, screened samples become 0.
template <typename DT>
__device__ __forceinline__ bool screen_keep(DT d, float min_u, float max_u) {
  if (!Depth<DT>::valid(d)) return false;
  const float z = Depth<DT>::z(d);
  return (min_u <= 0.0f || z >= min_u) && (max_u <= 0.0f || z <= max_u);
}

template <typename DT>
__global__ void __launch_bounds__(kThreads) k_screen(ScreenArgs a) {
  const int cam = blockIdx.y;
  const unsigned W = (unsigned)a.W[cam], H = (unsigned)a.H[cam], n = W * H;   // W H <= 2^30
  const DT* __restrict__ in = static_cast<const DT*>(a.in[cam]);
  DT* __restrict__ out = static_cast<DT*>(a.out[cam]);
  for (unsigned p = blockIdx.x * blockDim.x + threadIdx.x; p < n; p += gridDim.x * blockDim.x) {
    const DT d = __ldg(in + p);
    bool keep = screen_keep<DT>(d, a.min_u, a.max_u);
    if (keep && a.edge_rel > 0.0f) {
      const unsigned y = p / W, x = p - y * W;
      const float z = Depth<DT>::z(d), thr = __fmul_rn(a.edge_rel, z);
      auto jump = [&](unsigned q) {
        const DT e = __ldg(in + q);
        return screen_keep<DT>(e, a.min_u, a.max_u) && fabsf(__fsub_rn(z, Depth<DT>::z(e))) > thr;
      };
      if ((x > 0 && jump(p - 1)) || (x + 1 < W && jump(p + 1)) || (y > 0 && jump(p - W)) ||
          (y + 1 < H && jump(p + W)))
        keep = false;
    }
    out[p] = keep ? d : (DT)0;
  }
}

// The same screen for images whose rows start on 16-byte boundaries (every width a
// multiple of 8, 16-byte aligned buffers): a block covers 8 rows x 256 columns of one
// camera, a thread 8 consecutive pixels of one row, read and written as 16-byte vectors
// (two for float32).  The rows above and below come from the neighbouring warps' loads
// through L1/L2; left and right neighbours from the adjacent lanes, the warp's two outer
// ones by scalar loads.
template <typename DT>
__device__ __forceinline__ void load_row8(const DT* __restrict__ p, DT v[8]) {
  if constexpr (sizeof(DT) == 2) {
    const uint4 u = __ldg(reinterpret_cast<const uint4*>(p));
    const unsigned w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
    for (int k = 0; k < 4; ++k) { v[2 * k] = (DT)(w[k] & 0xffffu); v[2 * k + 1] = (DT)(w[k] >> 16); }
  } else {
    const float4 f0 = __ldg(reinterpret_cast<const float4*>(p));
    const float4 f1 = __ldg(reinterpret_cast<const float4*>(p) + 1);
    v[0] = f0.x; v[1] = f0.y; v[2] = f0.z; v[3] = f0.w;
    v[4] = f1.x; v[5] = f1.y; v[6] = f1.z; v[7] = f1.w;
  }
}

template <typename DT>
__device__ __forceinline__ void store_row8(DT* __restrict__ p, const DT v[8]) {
  if constexpr (sizeof(DT) == 2) {
    uint4 u;
    u.x = (unsigned)v[0] | ((unsigned)v[1] << 16);
    u.y = (unsigned)v[2] | ((unsigned)v[3] << 16);
    u.z = (unsigned)v[4] | ((unsigned)v[5] << 16);
    u.w = (unsigned)v[6] | ((unsigned)v[7] << 16);
    *reinterpret_cast<uint4*>(p) = u;
  } else {
    reinterpret_cast<float4*>(p)[0] = make_float4(v[0], v[1], v[2], v[3]);
    reinterpret_cast<float4*>(p)[1] = make_float4(v[4], v[5], v[6], v[7]);
  }
}

template <typename DT>
__device__ __forceinline__ DT shfl_depth(DT v, int delta, bool up) {
  if constexpr (sizeof(DT) == 2) {
    const unsigned u = up ? __shfl_up_sync(0xffffffffu, (unsigned)v, delta)
                          : __shfl_down_sync(0xffffffffu, (unsigned)v, delta);
    return (DT)u;
  } else {
    return up ? __shfl_up_sync(0xffffffffu, v, delta) : __shfl_down_sync(0xffffffffu, v, delta);
  }
}

template <typename DT>
__global__ void __launch_bounds__(kThreads) k_screen_rows(ScreenArgs a) {
  const int cam = blockIdx.z;
  const int W = a.W[cam], H = a.H[cam];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int y = blockIdx.y * 8 + warp;
  const int x0 = blockIdx.x * 256 + lane * 8;
  const bool active = y < H && x0 < W;              // W % 8 == 0: all 8 pixels inside
  const DT* __restrict__ in = static_cast<const DT*>(a.in[cam]);
  DT v[8], up[8], dn[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) { v[k] = (DT)0; up[k] = (DT)0; dn[k] = (DT)0; }
  if (active) {
    const size_t row = (size_t)y * (size_t)W + (size_t)x0;
    load_row8<DT>(in + row, v);
    if (y > 0) load_row8<DT>(in + row - W, up);
    if (y + 1 < H) load_row8<DT>(in + row + W, dn);
  }
  // neighbours across the thread's 8-pixel group: adjacent lanes, or a scalar load at the
  // warp's edges (a sample outside the image counts as invalid: it never screens)
  DT left = shfl_depth<DT>(v[7], 1, true), right = shfl_depth<DT>(v[0], 1, false);
  if (lane == 0) left = (active && x0 > 0) ? __ldg(in + (size_t)y * W + x0 - 1) : (DT)0;
  if (lane == 31) right = (active && x0 + 8 < W) ? __ldg(in + (size_t)y * W + x0 + 8) : (DT)0;
  if (x0 + 8 >= W) right = (DT)0;
  if (!active) return;
  // valid and within the bounds as two compares: z >= lo and z <= hi, with lo the lower
  // bound or the smallest positive float (so that 0, negatives and NaN fail) and hi the
  // upper bound or the largest finite float (so that +inf fails); the same decision as
  // screen_keep (no flush of subnormals in this build)
  const float lo = a.min_u > 0.0f ? a.min_u : __int_as_float(1);
  const float hi = a.max_u > 0.0f ? a.max_u : __int_as_float(0x7f7fffff);
  float zc[8], zu[8], zd[8];
  bool oc[8], ou[8], od[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    zc[k] = Depth<DT>::z(v[k]);
    zu[k] = Depth<DT>::z(up[k]);
    zd[k] = Depth<DT>::z(dn[k]);
    oc[k] = zc[k] >= lo && zc[k] <= hi;
    ou[k] = zu[k] >= lo && zu[k] <= hi;
    od[k] = zd[k] >= lo && zd[k] <= hi;
  }
  const float zl = Depth<DT>::z(left), zr = Depth<DT>::z(right);
  const bool ol = zl >= lo && zl <= hi, orr = zr >= lo && zr <= hi;
  const float rel = a.edge_rel;
  DT o[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    bool keep = oc[k];
    if (rel > 0.0f) {
      const float z = zc[k], thr = __fmul_rn(rel, z);
      const float zw = k > 0 ? zc[k - 1] : zl, ze = k < 7 ? zc[k + 1] : zr;
      const bool ow = k > 0 ? oc[k - 1] : ol, oe = k < 7 ? oc[k + 1] : orr;
      const bool jump = (ow && fabsf(__fsub_rn(z, zw)) > thr) || (oe && fabsf(__fsub_rn(z, ze)) > thr) ||
                        (ou[k] && fabsf(__fsub_rn(z, zu[k])) > thr) ||
                        (od[k] && fabsf(__fsub_rn(z, zd[k])) > thr);
      keep = keep && !jump;
    }
    o[k] = keep ? v[k] : (DT)0;
  }
  store_row8<DT>(static_cast<DT*>(a.out[cam]) + (size_t)y * W + x0, o);
}

template <typename DT, int TH>
cudaError_t set_tile_attributes_th() {
  const int sm = (int)WeighTile<TH>::smem(kMaxK1);
  const cudaFuncAttribute at = cudaFuncAttributeMaxDynamicSharedMemorySize;
  cudaError_t e = cudaFuncSetAttribute(k_weigh<DT, false, 1, TH>, at, sm);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_weigh<DT, true, 1, TH>, at, sm);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_weigh<DT, false, kMaxBatch, TH>, at, sm);
  const int tk = (int)AssignTile<TH>::Bytes;
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_assign_topk<DT, false, 1, TH>, at, tk);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_assign_topk<DT, true, 1, TH>, at, tk);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_assign_topk<DT, false, kMaxBatch, TH>, at, tk);
  return e;
}

// Dynamic shared memory limits of the tile kernels for one depth type, set once per device
// (the first call comes from context creation, outside any stream capture).  The attribute
// call is idempotent, so two host threads that race here only repeat it.
template <typename DT>
cudaError_t set_tile_attributes() {
  static std::atomic<unsigned long long> done{0ull};       // one bit per device (< 64)
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return cudaErrorInvalidDevice;
  const unsigned long long bit = dev < 64 ? 1ull << dev : 0ull;
  if (bit && (done.load(std::memory_order_acquire) & bit)) return cudaSuccess;
  cudaError_t e = set_tile_attributes_th<DT, 8>();
  if (e == cudaSuccess) e = set_tile_attributes_th<DT, 16>();
  if (e == cudaSuccess) e = set_tile_attributes_th<DT, 32>();
  if (e == cudaSuccess) done.fetch_or(bit, std::memory_order_release);
  return e;
}

// Launch of one of the frame's kernels; pdl: programmatic stream serialization with the
// kernel before it on the stream (the kernel must call pdl_wait before using its results).
template <typename... P, typename... A>
cudaError_t launch_k(bool pdl, void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                     A... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pdl ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}

// Threads of a weigh or sum block: a thread for four pixels, or fewer while all of a launch's blocks
// fit on the chip at once (a frame of 80 tiles then takes a pixel a thread instead of four in turn).
int weigh_threads(int tiles, int th, int sms) {
  int n = 8 * th;
  while (n < 32 * th && n < 512 && 2ll * n * tiles <= 1024ll * sms) n *= 2;
  return n;
}

// The assign step over the batch's tiles (TH rows a tile; the traced instantiations exist for
// single frames only): the weigh kernel, or the top-k variant's.
template <typename DT, int NB, int TH>
cudaError_t launch_assign(const BatchArgs<NB>& a, int n, bool top_k, bool traced, int max_k1, int sms, bool pdl,
                          cudaStream_t s) {
  const dim3 tiles(a.tile_first[n]), at(AssignTile<TH>::Threads), wt(weigh_threads(a.tile_first[n], TH, sms));
  const size_t tk = AssignTile<TH>::Bytes, sm = WeighTile<TH>::smem(max_k1);
  if constexpr (NB == 1)
    if (traced)
      return top_k ? launch_k(pdl, k_assign_topk<DT, true, NB, TH>, tiles, at, tk, s, a)
                   : launch_k(pdl, k_weigh<DT, true, NB, TH>, tiles, wt, sm, s, a);
  return top_k ? launch_k(pdl, k_assign_topk<DT, false, NB, TH>, tiles, at, tk, s, a)
               : launch_k(pdl, k_weigh<DT, false, NB, TH>, tiles, wt, sm, s, a);
}

template <typename DT, int NB, int TH>
cudaError_t launch_sum(const BatchArgs<NB>& a, int n, int sms, bool pdl, cudaStream_t s) {
  const int threads = weigh_threads(a.tile_first[n], TH, sms);
  return launch_k(pdl, k_sum<DT, NB, TH>, dim3(a.tile_first[n]), dim3(threads), 16 * kSumWarpWords * (threads / 32), s, a);
}

// The frame kernels over n frames (NB = 1: one frame; NB = kMaxBatch: a batch of up to
// that many frames of any rigs, every kernel launched once for all of them).
template <typename DT, int NB>
cudaError_t launch_frames(const FrameLaunch* fr, int n, cudaStream_t s, cudaEvent_t* ev) {
  const cudaError_t ae = set_tile_attributes<DT>();
  if (ae != cudaSuccess) return ae;
  if (n < 1 || n > NB) return cudaErrorInvalidValue;
  auto mark = [&](int i) { if (ev) cudaEventRecord(ev[i], s); };
  mark(0);
  static thread_local BatchArgs<NB> a;
  std::memset(&a, 0, sizeof(a));
  a.n = n;
  int emit = 1, pdl_level = 2, max_wblocks = 1, max_k1 = 0;
  long long units = 0;
  const Geometry& g0 = *fr[0].geo;
  cudaError_t err = cudaSuccess;
  for (int f = 0; f < n; ++f) {
    const Geometry& geo = *fr[f].geo;
    const Tables& t = fr[f].t;
    FrameArgs& fa = a.f[f];
    fa.rig = fr[f].rig;
    fa.rays = fr[f].rays;
    fa.fp = fr[f].fp;
    fa.t = t;
    fa.tr = fr[f].tr;
    fa.out = fr[f].out;
    fa.ti = geo.tiles;
    fa.hot = geo.hot;
    fa.top_k = geo.top_k;
    fa.count_chunks = geo.count_chunks;
    fa.unit_m = (float)fr[f].out.unit_m;
    if (geo.screen) {                      // D^r of Eq. 8 into the context's buffers
      ScreenArgs sa = geo.scr;
      for (int i = 0; i < geo.n_cams; ++i) {
        sa.in[i] = fr[f].fp.depth[i];
        fa.fp.depth[i] = sa.out[i];
      }
      if ((err = launch_screen(sa, sizeof(DT) == 4, geo.max_px, s)) != cudaSuccess) return err;
    }
    a.count_first[f + 1] = a.count_first[f] + geo.count_blocks;
    a.tile_first[f + 1] = a.tile_first[f] + t.n_tiles;
    units += t.n_units;
    emit = std::max(emit, geo.emit_blocks);
    pdl_level = std::min(pdl_level, geo.pdl);
    max_wblocks = std::max(max_wblocks, t.n_wblocks);
    max_k1 = std::max(max_k1, geo.tiles.k1);
  }
  mark(1);
  // programmatic launches between the kernels when the geometry asks for them (level 2
  // also between the assign and reduce steps), never while stage events are recorded
  const bool pdl = pdl_level >= 1 && ev == nullptr;
  const bool pdl_reduce = pdl_level >= 2 && ev == nullptr;
  const dim3 eb(emit, n), th3(kThreads);
  const bool few = units <= (long long)kCountFew * g0.sms;
  if ((err = few ? launch_k(false, k_count<DT, NB, true>, dim3(a.count_first[n]), th3, 0, s, a)
                 : launch_k(false, k_count<DT, NB, false>, dim3(a.count_first[n]), th3, 0, s, a)) != cudaSuccess ||
      (err = launch_k(pdl, k_levels<NB>, eb, th3, 0, s, a)) != cudaSuccess)
    return err;
  mark(2);
  bool traced = false;
  for (int f = 0; f < n; ++f) {
    const TraceDev& tr = fr[f].tr;
    traced = traced || tr.pw || tr.omega || tr.e || tr.nview || tr.key;
  }
  const int th = g0.tiles.th;
  const bool topk = g0.top_k != 0;
  if (th == 8) err = launch_assign<DT, NB, 8>(a, n, topk, traced, max_k1, g0.sms, pdl, s);
  else if (th == 32) err = launch_assign<DT, NB, 32>(a, n, topk, traced, max_k1, g0.sms, pdl, s);
  else err = launch_assign<DT, NB, 16>(a, n, topk, traced, max_k1, g0.sms, pdl, s);
  if (err != cudaSuccess) return err;
  mark(3);
  if (topk) err = launch_k(pdl_reduce, k_reduce_topk<DT, NB>, dim3(2 * emit, n), dim3(kTopThreads), 0, s, a);
  else if (th == 8) err = launch_sum<DT, NB, 8>(a, n, g0.sms, pdl_reduce, s);
  else if (th == 32) err = launch_sum<DT, NB, 32>(a, n, g0.sms, pdl_reduce, s);
  else err = launch_sum<DT, NB, 16>(a, n, g0.sms, pdl_reduce, s);
  if (err != cudaSuccess) return err;
  mark(4);
  mark(5);
  const dim3 rb(max_wblocks + 1, n);
  if ((err = topk ? launch_k(pdl, k_emit<true, NB>, rb, th3, 0, s, a) : launch_k(pdl, k_emit<false, NB>, rb, th3, 0, s, a)) !=
      cudaSuccess)
    return err;
  mark(6);
  return cudaGetLastError();
}

}  // namespace

namespace {
template <int TH>
int resident_th(int k1) {
  static std::atomic<int> cache[kMaxK1 + 1];             // 0: not yet asked
  k1 = std::max(0, std::min(k1, kMaxK1));
  const int known = cache[k1].load(std::memory_order_relaxed);
  if (known > 0) return known;
  int n = 0;
  const int sm = (int)WeighTile<TH>::smem(k1);
  if (set_tile_attributes<uint16_t>() != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_weigh<uint16_t, false, 1, TH>, WeighTile<TH>::Threads, sm) !=
          cudaSuccess) {
    cudaGetLastError();
    return 1024 / WeighTile<TH>::Threads;
  }
  n = std::max(1, n);
  cache[k1].store(n, std::memory_order_relaxed);
  return n;
}
}  // namespace

int assign_resident_blocks(int th, int k1) {
  return th == 8 ? resident_th<8>(k1) : th == 32 ? resident_th<32>(k1) : resident_th<16>(k1);
}

int retile(TileIndex* ti, int th) {
  ti->th = th;
  int n = 0, u = 0;
  bool same = true;
  for (int i = 0; i < ti->n_cams; ++i) {
    const int tx = (ti->W[i] + kTileW - 1) / kTileW;
    ti->first[i] = n;
    ti->unit[i] = u;
    ti->div_x[i] = fast_div_factor((unsigned)tx);
    n += tx * ((ti->H[i] + th - 1) / th);
    u += tx * ((ti->H[i] + kUnitH - 1) / kUnitH);
    same = same && ti->W[i] == ti->W[0] && ti->H[i] == ti->H[0];
  }
  ti->first[ti->n_cams] = n;
  ti->unit[ti->n_cams] = u;
  ti->per_cam = same && ti->n_cams > 0 ? ti->first[1] : 0;
  ti->units_per_cam = same && ti->n_cams > 0 ? ti->unit[1] : 0;
  ti->div_cam = ti->per_cam ? fast_div_factor((unsigned)ti->per_cam) : 0u;
  ti->div_units = ti->units_per_cam ? fast_div_factor((unsigned)ti->units_per_cam) : 0u;
  return n;
}

int fill_tile_index(const RigDev& rig, TileIndex* out, int th) {
  memset(out, 0, sizeof(*out));
  out->n_cams = rig.n_cams;
  out->k1 = rig.k1;
  long long pray = 0;
  for (int i = 0; i < rig.n_cams; ++i) {
    out->W[i] = rig.cam[i].W;
    out->H[i] = rig.cam[i].H;
    out->off[i] = rig.cam[i].off;
    out->pray[i] = (int)pray;
    pray += pray_cam_size(rig.cam[i].W, rig.cam[i].H, rig.k1);
  }
  out->ahead = kNoPrefetch;                      // no prefetch unless the caller sets it
  return retile(out, th);
}

void fill_block_consts(const RigDev& rig, BlockConst* out) {
  long long pray = 0;
  for (int i = 0; i < rig.n_cams; ++i) {
    BlockConst& b = out[i];
    memset(&b, 0, sizeof(b));
    const CamDev& c = rig.cam[i];
    memcpy(b.cam.Rwc, c.Rwc, sizeof(c.Rwc));
    memcpy(b.cam.cwc, c.cwc, sizeof(c.cwc));
    b.cam.ray_x = c.ray_x;
    b.cam.ray_y = c.ray_y;
    b.cam.pray = (int)pray;
    b.cam.pair0 = c.pair0;
    pray += pray_cam_size(c.W, c.H, rig.k1);
    for (int q = 0; q < rig.k1; ++q) {
      const PairDev& p = rig.pair[c.pair0 + q];
      const CamDev& n = rig.cam[p.j];
      ViewHot& v = b.view[q];
      for (int a = 0; a < 3; ++a) {
        v.mt[a] = kGridM + p.th[a];
        v.tl[a] = p.tl[a];
      }
      v.fx = n.fx;
      v.fy = n.fy;
      v.cx5 = (float)((double)n.cxh + (double)n.cxl + 0.5);
      v.cy5 = (float)((double)n.cyh + (double)n.cyl + 0.5);
      v.W = n.W;
      v.H = n.H;
      v.ray_x = n.ray_x;
      v.ray_y = n.ray_y;
      // twice the error bound of the float32 projection (nearest_pixel)
      v.band = (float)std::max(n.W + std::fabs((double)n.cx), n.H + std::fabs((double)n.cy)) / 1048576.0f;
      v.j = p.j;
    }
  }
}

cudaError_t launch_init_tables(const Tables& t, unsigned fcap, unsigned ccap, cudaStream_t s) {
  k_init_tables<<<1024, 256, 0, s>>>(t, fcap, ccap);
  return cudaGetLastError();
}

cudaError_t launch_copyout(const fuseflow_cloud& src, const HostOutDev& dst, cudaStream_t s) {
  k_copyout<<<4 * 152, kThreads, 0, s>>>(src, dst);
  return cudaGetLastError();
}

cudaError_t launch_confidence(const ConfArgs& a, bool depth_f32, int max_w, int max_h,
                              cudaStream_t s) {
  const dim3 g((max_w + kConfW - 1) / kConfW, (max_h + kConfH - 1) / kConfH, a.n_cams);
  if (depth_f32) k_confidence<float><<<g, kThreads, 0, s>>>(a);
  else k_confidence<uint16_t><<<g, kThreads, 0, s>>>(a);
  return cudaGetLastError();
}

int mc_blocks(long long n) { return (int)std::max(1ll, std::min<long long>(kMcBlocks, (n + kThreads - 1) / kThreads)); }

cudaError_t launch_mc(const RigDev* rig, const FramePtrs& fp, bool depth_f32, const float* pos,
                      long long n, double unit_m, double occlusion_m, float* err, int* nvis,
                      double* bsum, long long* bcnt, cudaStream_t s) {
  const int g = mc_blocks(n);
  const float inv = (float)(1.0 / unit_m), um = (float)unit_m;
  const float occl = (float)(occlusion_m / unit_m);      // +inf stays +inf
  if (depth_f32) k_mc<float><<<g, kThreads, 0, s>>>(rig, fp, pos, n, inv, um, occl, err, nvis, bsum, bcnt);
  else k_mc<uint16_t><<<g, kThreads, 0, s>>>(rig, fp, pos, n, inv, um, occl, err, nvis, bsum, bcnt);
  return cudaGetLastError();
}

// Tiles of the point-wise path over all cameras, and the largest camera's.
static int points_tiles(const TileIndex& ti, int* most = nullptr) {
  int sum = 0, top = 1;
  for (int i = 0; i < ti.n_cams; ++i) {
    const int n = (ti.W[i] + kTileW - 1) / kTileW * ((ti.H[i] + PointsTile::H - 1) / PointsTile::H);
    sum += n;
    top = std::max(top, n);
  }
  if (most) *most = top;
  return sum;
}

template <int Threads>
static cudaError_t launch_points_n(const RigDev* rig, const RigHot& hot, const float2* rays, const FramePtrs& fp,
                                   const Tables& t, const PointsDev& out, bool depth_f32, const TileIndex& ti,
                                   cudaStream_t s) {
  int most;
  points_tiles(ti, &most);
  const dim3 g((unsigned)most, ti.n_cams);
  const size_t sm = PointsTile::smem(ti.k1);                  // at most 23 KB
  if (depth_f32) k_points<float, Threads><<<g, Threads, sm, s>>>(rig, hot, rays, fp, t, ti, out);
  else k_points<uint16_t, Threads><<<g, Threads, sm, s>>>(rig, hot, rays, fp, t, ti, out);
  return cudaGetLastError();
}

cudaError_t launch_points(const RigDev* rig, const RigHot& hot, const float2* rays, const FramePtrs& fp, const Tables& t,
                          const PointsDev& out, bool depth_f32, const TileIndex& ti, int sms, cudaStream_t s) {
  cudaError_t e = cudaMemsetAsync(out.counts, 0, 2 * sizeof(unsigned long long), s);
  if (e != cudaSuccess) return e;
  const int th = weigh_threads(points_tiles(ti), PointsTile::H, sms);
  return th == 128   ? launch_points_n<128>(rig, hot, rays, fp, t, out, depth_f32, ti, s)
         : th == 256 ? launch_points_n<256>(rig, hot, rays, fp, t, out, depth_f32, ti, s)
                     : launch_points_n<512>(rig, hot, rays, fp, t, out, depth_f32, ti, s);
}

cudaError_t launch_screen(const ScreenArgs& a, bool depth_f32, long long max_px, cudaStream_t s) {
  bool rows = true;                                   // 16-byte rows: the vector kernel
  int max_w = 1, max_h = 1;
  for (int i = 0; i < a.n_cams; ++i) {
    rows = rows && a.W[i] % 8 == 0 && (reinterpret_cast<uintptr_t>(a.in[i]) & 15) == 0 &&
           (reinterpret_cast<uintptr_t>(a.out[i]) & 15) == 0;
    max_w = std::max(max_w, a.W[i]);
    max_h = std::max(max_h, a.H[i]);
  }
  if (rows) {
    const dim3 grid((unsigned)((max_w + 255) / 256), (unsigned)((max_h + 7) / 8), (unsigned)a.n_cams);
    if (depth_f32) k_screen_rows<float><<<grid, kThreads, 0, s>>>(a);
    else k_screen_rows<uint16_t><<<grid, kThreads, 0, s>>>(a);
  } else {
    const unsigned bx = (unsigned)std::min<long long>((max_px + kThreads - 1) / kThreads, 4096);
    const dim3 grid(std::max(1u, bx), a.n_cams);
    if (depth_f32) k_screen<float><<<grid, kThreads, 0, s>>>(a);
    else k_screen<uint16_t><<<grid, kThreads, 0, s>>>(a);
  }
  return cudaGetLastError();
}

cudaError_t prepare_launch(bool depth_f32) {
  return depth_f32 ? set_tile_attributes<float>() : set_tile_attributes<uint16_t>();
}

cudaError_t launch_frame(const RigDev* rig, const float2* rays, const FramePtrs& fp, const Tables& t,
                         const TraceDev& tr, const OutDev& out, const Geometry& geo, cudaStream_t s,
                         cudaEvent_t* ev) {
  const FrameLaunch fl{rig, rays, fp, t, tr, out, &geo};
  if (geo.depth_f32) return launch_frames<float, 1>(&fl, 1, s, ev);
  return launch_frames<uint16_t, 1>(&fl, 1, s, ev);
}

cudaError_t launch_batch(const FrameLaunch* frames, int n, cudaStream_t s) {
  if (n < 1 || n > kMaxBatch) return cudaErrorInvalidValue;
  for (int f = 1; f < n; ++f)                       // one depth type and one fusion variant
    if (frames[f].geo->depth_f32 != frames[0].geo->depth_f32 || frames[f].geo->top_k != frames[0].geo->top_k ||
        frames[f].geo->tiles.th != frames[0].geo->tiles.th)
      return cudaErrorInvalidValue;
  if (frames[0].geo->depth_f32) return launch_frames<float, kMaxBatch>(frames, n, s, nullptr);
  return launch_frames<uint16_t, kMaxBatch>(frames, n, s, nullptr);
}

}  // namespace ffl
