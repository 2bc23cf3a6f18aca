// ff_device.cuh - device data layout and per-pixel arithmetic of the sm_103a fusion path.
//
// Geometry is carried in "depth units" (metres per unit = depth_scale), so that the depth
// sample z of a pixel is exact in float32 (uint16 codes and float32 samples both are).
// World points, cell keys and the projection that selects a pixel are float32; the 3D
// residual of Eq. 6 is evaluated in double-float ("ff", an unevaluated hi + lo pair of
// float32) so that the joint weight of Eq. 10 keeps ~1e-7 relative accuracy although the
// residual is a difference of two metre-scale vectors.  The error-free transformations are
// Knuth's TwoSum, Dekker's Fast2Sum and the FMA TwoProduct, combined as in the compensated
// dot product of Ogita, Rump and Oishi (SIAM J. Sci. Comput. 26(6), 2005).
#pragma once

#include <cstdint>
#include <cstring>
#include <cuda_runtime.h>

namespace ffl {

constexpr int kMaxCams = 64;
constexpr int kMaxK1 = 8;
constexpr int kMaxTopK = 7;              // top-k keys travel in a partial record
constexpr unsigned long long kKeyEmpty = ~0ull;
constexpr uint32_t kSlotNone = 0xffffffffu;
constexpr uint32_t kSlotPending = 0xfffffffeu;
constexpr int kFixShift = 36;            // per-cell fixed point: largest member weight ~ 2^36
constexpr int kKeyBias = 1 << 19;        // cell index range [-2^19, 2^19) per axis
constexpr float kGridM = 12582912.0f;    // 1.5 2^23: adding it rounds |v| < 2^22 to an integer
constexpr int kGridBits = 0x4B400000;    // its bits: an integer n is bits(kGridM + n) - kGridBits

// error bits of FrameCounters::error
constexpr unsigned kErrSlots = 1u;       // the cells' dense slot ranges exceed the slot capacity
constexpr unsigned kErrCoarseFull = 2u;  // coarse hash table could not take a key
constexpr unsigned kErrCells = 4u;       // more cells than the output capacity
constexpr unsigned kErrCoarseMiss = 8u;  // a point's coarse cell was not found (internal)
constexpr unsigned kErrPartials = 16u;   // more (tile, cell) partials than the buffer holds
constexpr unsigned kErrList = 32u;       // a cell list was longer than the partials written

struct CamDev {
  int W, H;
  long long off;                 // global index of pixel (0, 0)
  float fx, fy, cx, cy;          // float32 intrinsics (projection into this camera)
  float fxh, fxl, fyh, fyl;      // ff intrinsics for exact half-pixel decisions
  float cxh, cxl, cyh, cyl;
  float Rwc[9];                  // world-from-camera rotation R^T, row-major
  float cwc[3];                  // camera centre (depth units)
  int ray_x, ray_y;              // offsets of this camera's ray tables
  int pair0;                     // first neighbour pair of this camera
  int pad;
};

struct PairDev {                 // camera i -> neighbour j: a = R_ji p_c + t_ji
  float th[3], tl[3];            // t_ji = t_j - R_ji t_i in grid units: th integral, tl the rest
  int j;
};

// Scalars of a rig that the frame kernels use per pixel; passed by value (constant bank).
// The consistency step works in "grid units" (kGridM below): ginv grid units per depth unit, a
// power of two chosen so that every camera-frame coordinate of the rig (depths up to zmax) is
// below 2^22 of them.
struct RigHot {
  float tau;                     // Eq. 9 gate
  int use_conf, use_cons;
  int max_level;
  float inv_s0u;                 // 1 / s0 in 1 / depth units
  float einv_h, einv_l;          // 1 / (sigma^2 (K-1)) in 1 / grid units^2, as ff
  float ginv;                    // grid units per depth unit
  float zmax;                    // largest depth (depth units) the grid evaluation covers
};

struct RigDev {
  int n_cams, k1;                // k1 = K - 1 neighbours per camera
  RigHot hot;
  int n_min;
  int depth_f32;
  long long n_px;
  CamDev cam[kMaxCams];
  PairDev pair[kMaxCams * kMaxK1];
};

// What the consistency step reads of one camera's tiles, packed so that a tile copies it in a
// few 16-byte words: the camera's pose and, per neighbour view, its projection.  Everything in
// grid units; rare exact decisions read RigDev instead.
struct __align__(16) CamHot {
  float Rwc[9], cwc[3];          // world-from-camera pose (depth units)
  int ray_x, ray_y;              // offsets of the camera's ray tables
  int pray;                      // float4 index of its pair rays
  int pair0;                     // its first PairDev
};
struct __align__(16) ViewHot {
  float mt[3];                   // kGridM + integral part of t_ji
  float tl[3];                   // rest of t_ji
  float fx, fy, cx5, cy5;        // projection into view j; principal point + 1/2
  int W, H;
  int ray_x, ray_y;              // offsets of view j's ray tables
  float band;                    // |u - integer| below this is decided exactly (pixels)
  int j;
};
struct BlockConst {
  CamHot cam;
  ViewHot view[kMaxK1];
};
static_assert(sizeof(CamHot) == 64 && sizeof(ViewHot) == 64, "16-byte words of a tile's constants");

// Separable pair rays (Eq. 4): with p_c = z (rx(x), ry(y), 1), R_ji p_c = z (A(x) + B(y)),
// A_k(x) = R_ji[k][0] rx(x) + R_ji[k][2] and B_k(y) = R_ji[k][1] ry(y), in grid units per depth
// unit, each an ff whose high parts are multiples of one power of two, so that the sum of two
// high parts is exact.  Per camera, columns go in groups of 32 and rows in groups of 8; a group
// holds, view after view, a plane of (0h, 1h, 2h, 0l) and a plane of (1l, 2l), so that a tile's
// share is contiguous and its planes are read without bank conflicts.  Padded to 32 columns / rows.
constexpr int kPrayColGroup = 48;          // float4 per view and 32 columns
constexpr int kPrayRowGroup = 12;          // float4 per view and 8 rows
__host__ __device__ inline long long pray_cam_size(int W, int H, int k1) {   // float4 of one camera
  return (long long)k1 * ((W + 31) / 32 * kPrayColGroup + (H + 31) / 32 * 4 * kPrayRowGroup);
}

// Where the assign step's tiles are: camera i owns tiles [first[i], first[i+1]), row-major over its
// ceil(W/32) x ceil(H/th) grid; and its units of 32 x 8 pixels, the count step's share of a warp and
// the grain of the lists of gated pixels: units [unit[i], unit[i+1]), row-major over ceil(W/32) x
// ceil(H/8).  A unit's list starts where its pixels would if the image were stored unit by unit
// (unit_list).  Passed by value (constant bank) to the kernels.
struct TileIndex {
  int n_cams, k1;
  int th;                        // tile height (8, 16 or 32 rows of 32 columns)
  int first[kMaxCams + 1];
  int unit[kMaxCams + 1];
  int W[kMaxCams], H[kMaxCams];
  unsigned div_x[kMaxCams];      // fast_div factor of the camera's tile columns
  long long off[kMaxCams];       // global index of each camera's pixel (0, 0)
  int pray[kMaxCams];            // float4 index of the camera's pair rays: column groups, then rows
  int per_cam, units_per_cam;    // tiles and units per camera when all cameras share W and H, else 0
  unsigned div_cam, div_units;   // their fast_div factors
  int ahead;                     // tiles resident at once: block b prefetches tile b + ahead
};
constexpr int kUnitH = 8;
constexpr int kUnitCells = 64;   // numbers that a unit's coarse cells can have
constexpr unsigned kNoCellNumber = 0xffu;

// First list entry of the unit at (x0, y0) of a camera of W x H pixels whose first pixel is off.
__host__ __device__ inline long long unit_list(long long off, int W, int H, int x0, int y0) {
  return off + (long long)y0 * W + (long long)x0 * (H - y0 < kUnitH ? H - y0 : kUnitH);
}

// n / d and the remainder, for a divisor whose factor floor((2^32 - 1) / d) is known: the product's
// upper half is the quotient or one or two below it.
__host__ __device__ inline unsigned fast_div_factor(unsigned d) { return 0xffffffffu / d; }
__device__ __forceinline__ int fast_div(int n, int d, unsigned factor, int& rem) {
  int q = (int)__umulhi((unsigned)n, factor);
  rem = n - q * d;
  if (rem >= d) { ++q; rem -= d; }
  if (rem >= d) { ++q; rem -= d; }
  return q;
}

// Top-k variant: per (tile, cell) partial result of the assign step, pushed onto its cell's list when
// it is written; two aligned 32-byte sectors.
struct __align__(64) Partial {
  unsigned next;                 // next partial of the same cell, kSlotNone at the end
  unsigned count;                // members in the tile
  unsigned long long top[kMaxTopK];       // the tile's k largest ordered(C) << 32 | ~g, then 0
};
static_assert(sizeof(Partial) == 64, "partial record layout");

// Per dense cell slot, in one 16-byte record so that a point reads a single sector.
struct __align__(16) SlotRec {
  unsigned long long key;        // representative: largest ordered(C) << 32 | ~g (top-k: the cell's key)
  unsigned head;                 // the cell's number, kSlotPending while its claim is under way (top-k:
                                 // last partial pushed); kSlotNone if none
  int mmin;                      // smallest weight exponent of the cell's members
};

// Coarse hash-table record: key, density count (Sec. II.5(1)c) and, once every count is
// in, the level and first dense cell slot packed as level << 27 | base.
struct __align__(16) CoarseEntry {
  unsigned long long key;
  unsigned count;
  unsigned lvbase;
};
constexpr unsigned kBaseNone = (1u << 27) - 1u;    // base field of a coarse cell without slots

// By cell number: exact sums of Eq. 11 {w, w frac xyz, w rgb / 256, members} in units of
// 2^-(kFixShift + mmin), the cell's key and slot.
struct __align__(32) CellRow {
  unsigned long long sum[8];
  unsigned long long key;
  unsigned slot;
  int mmin;                      // smallest exponent, once the weigh step is over
  unsigned pad[4];
};
static_assert(sizeof(CellRow) == 96, "three sectors a cell");

// Bitmap words of an emit block's share.
constexpr int kRankWords = 256;

// Fused cell staged by the top-k reduce step (by cell number) for the emit step.
struct __align__(16) CellOut {
  float pos[3];
  float rgb[3];
  float weight;
  unsigned count;
  unsigned rep;
  unsigned pad;
  unsigned long long key;
};
static_assert(sizeof(CellOut) == 48, "staged cell layout");

struct FrameCounters {           // zero between frames, but n_cells, which the level step clears
  unsigned n_cells, n_coarse;
  unsigned error;
  unsigned n_partials;
  unsigned long long n_slots;    // dense cell slots claimed (sum over coarse cells of 8^l)
};

struct BlockStats {              // per block of the coarse-count step
  unsigned n_valid, n_gated, n_oor, pad;
  unsigned bmin[3], bmax[3];     // ordered-integer encodings
  unsigned pad2[2];
};

// ----------------------------------------------------------------------------- helpers
__device__ __forceinline__ unsigned ordered(float f) {
  unsigned u = __float_as_uint(f);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__host__ __device__ inline float from_ordered(unsigned u) {
#ifdef __CUDA_ARCH__
  return __uint_as_float((u & 0x80000000u) ? (u & 0x7fffffffu) : ~u);
#else
  unsigned v = (u & 0x80000000u) ? (u & 0x7fffffffu) : ~u;
  float f;
  memcpy(&f, &v, 4);
  return f;
#endif
}

// First table position of coarse cell (x, y, z).  The two last lines scatter the cells of a wall: without
// them its rows lie side by side, overlap, and linear probing needs 8 to 15 probes a cell instead of 1.4 to
// 2.1 at loads of 0.46 and 0.69 (the longest chain 250 to 550 instead of 18 to 70).
__device__ __forceinline__ unsigned coarse_hash(int x, int y, int z) {
  unsigned h = (unsigned)x * 0xC2B2AE3Du + (unsigned)y * 0x9E3779B1u + (unsigned)z * 0x85EBCA77u;
  h = (h ^ (h >> 15)) * 0x2C1B3C6Du;
  return h ^ (h >> 16);
}

__device__ __forceinline__ unsigned long long pack_key(int l, int kx, int ky, int kz) {
  return ((unsigned long long)l << 60) | ((unsigned long long)(kx + kKeyBias) << 40) |
         ((unsigned long long)(ky + kKeyBias) << 20) | (unsigned long long)(kz + kKeyBias);
}

// --------------------------------------------------------------------------- double-float
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
  s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}
__device__ __forceinline__ void fast_two_sum(float a, float b, float& s, float& e) {
  s = __fadd_rn(a, b);
  e = __fsub_rn(b, __fsub_rn(s, a));
}
__device__ __forceinline__ void two_prod(float a, float b, float& p, float& e) {
  p = __fmul_rn(a, b);
  e = __fmaf_rn(a, b, -p);
}

// One component of a = z (A + B) + t in ff (A, B, t as ff, z exact); the result (oh, ol)
// is not renormalised (|ol| stays within a few ulp of oh, unless z(A + B) and t cancel).
__device__ __forceinline__ void ff_ray_affine(float Ah, float Al, float Bh, float Bl, float z,
                                              float th, float tl, float& oh, float& ol) {
  float gh, ge, p, pe, e;
  two_sum(Ah, Bh, gh, ge);
  ge = __fadd_rn(ge, __fadd_rn(Al, Bl));
  two_prod(z, gh, p, pe);
  pe = __fmaf_rn(z, ge, pe);
  two_sum(p, th, oh, e);
  ol = __fadd_rn(e, __fadd_rn(pe, tl));
}

// --------------------------------------------------------------------------- depth decode
template <typename DT> struct Depth;
template <> struct Depth<uint16_t> {
  static __device__ __forceinline__ bool valid(uint16_t d) { return d != 0; }
  static __device__ __forceinline__ float z(uint16_t d) { return (float)d; }
};
template <> struct Depth<float> {
  static __device__ __forceinline__ bool valid(float d) { return d > 0.0f && d < __int_as_float(0x7f800000); }
  static __device__ __forceinline__ float z(float d) { return d; }
};

// Eq. 8 in float32: world point (depth units) of pixel ray (rx, ry, 1) at z-depth z.
// Every step uses the same rounding-explicit sequence so all kernels agree bit for bit.
template <typename Cam>                  // CamDev or CamHot
__device__ __forceinline__ void world_point(const Cam& c, float z, float rx, float ry,
                                            float P[3]) {
  const float px = __fmul_rn(z, rx), py = __fmul_rn(z, ry);
#pragma unroll
  for (int k = 0; k < 3; ++k)
    P[k] = __fmaf_rn(c.Rwc[3 * k + 0], px,
                     __fmaf_rn(c.Rwc[3 * k + 1], py, __fmaf_rn(c.Rwc[3 * k + 2], z, c.cwc[k])));
}

// 2^e as a float for -126 <= e <= 127, built from its bits (exact scaling by a product).
__device__ __forceinline__ float pow2f(int e) { return __int_as_float((127 + e) << 23); }

// Sec. II.5(1): coarse-grid coordinate r = P / s0 and the range test at the finest level:
// floor(r 2^Lmax) in [-2^19, 2^19)  <=>  r 2^Lmax in [-2^19, 2^19).
// The range test is on floor(r): in [-2^(19-Lmax), 2^(19-Lmax)).  floor(v) of |v| < 2^22 is read
// off the bits of kGridM + v rounded down; outside, and for NaN, the bits give an integer that
// fails the range test (they are monotonic in v, and at least 2^22 away once wrapped).
__device__ __forceinline__ bool grid_coords(const RigHot& rig, const float P[3], float r[3], int c[3]) {
  const unsigned lim = (unsigned)kKeyBias >> rig.max_level;
  bool ok = true;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    r[k] = __fmul_rn(P[k], rig.inv_s0u);
    c[k] = __float_as_int(__fadd_rd(r[k], kGridM)) - kGridBits;
    ok = ok && (unsigned)c[k] + lim < 2u * lim;
  }
  return ok;
}

// Sec. II.5(1)d: level of a coarse cell holding n_c points: largest l <= Lmax with
// n_c >= n_min 4^l, else 0.
__device__ __forceinline__ int level_for(unsigned n_c, int n_min, int max_level) {
  int l = 0;
  for (int c = 1; c <= max_level; ++c)
    if ((unsigned long long)n_c >= ((unsigned long long)n_min << (2 * c))) l = c;
  return l;
}

}  // namespace ffl
