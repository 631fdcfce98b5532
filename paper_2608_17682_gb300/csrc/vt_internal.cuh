// vt_internal.cuh -- internal layout of a scene and helpers shared by the
// translation units of libvt.so (never installed, never seen by callers).
//
// Device layout of a scene (cells in Morton order of the sites):
//   rec  [units]  the cells' walk records, 32-byte units. Cell i's record
//               starts at unit unit[i]: a header unit {x, y, z, sigma, cell id,
//               pairs, user id, nmax} and then its neighbours in CSR order, four
//               to a quad of two units: {x0..x3}, {y0..y3}, {z0..z3},
//               {u0..u3}, where (x, y, z) = s_j - s_i (each component rounded
//               to FP32) and u is the unit of neighbour j's own record. pairs =
//               ceil(degree / 2); the places past the degree hold NaN offsets
//               (never a crossing) and kNoUnit. nmax (float bits) = max over
//               the neighbours of |s_j - s_i|.
//   unit [N]    first unit of each cell's record
//   site [N]    {x, y, z, bits of the user id}: the nearest-site scan's copy
//   body [N]    {x, y, z, sigma}: all that a backward along a record needs
//   tex  [N*R*R] RGBA texel: float4 (FP32) or 4 x 16-bit (FP16 / BF16)
//   perm [N]    Morton index -> user id,  inv [N] user id -> Morton index
// A walk knows a cell by its unit, so one address leads to everything that a
// step reads. Offsets come as operand pairs of the two-wide FP32 arithmetic,
// and the units, of which a step needs one, are not loaded with them.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>
#include <mutex>

#include "vt.h"

#define VT_MAX_ANCHORS 64

// error bits recorded on the device (scene->d_err[0])
#define VT_EBIT_MAX_STEPS 1u
#define VT_EBIT_CAPACITY 2u
#define VT_EBIT_BAD_RAY 4u

constexpr unsigned kNoUnit = 0xffffffffu;

// Start cells of the anchors, written by the start-cell search and read by the
// walks: the origin and (as bits) the record unit of its nearest cell, per
// anchor and for the n_uniq different ones among them (anchor a's is uniq[
// slot[a]]), of which a ray of a 1-D batch may match the first n_search.
struct vt_anchors {
  float4 at[VT_MAX_ANCHORS];
  float4 uniq[VT_MAX_ANCHORS];
  int slot[VT_MAX_ANCHORS];
  int n_uniq, n_search;
};
// blocks of the nearest-site scan
constexpr int kAnchorSitesPerBlock = 1024, kAnchorMaxBlocks = 304;
static inline int vt_anchor_blocks(int64_t n) {
  const int64_t g = (n + kAnchorSitesPerBlock - 1) / kAnchorSitesPerBlock;
  return (int)(g < kAnchorMaxBlocks ? g : kAnchorMaxBlocks);
}

// Lanes of a team walk, and units that they may read past the last record (the
// first quads are loaded with the header).
#ifndef VT_TEAM
#define VT_TEAM 8
#endif
constexpr int kTeam = VT_TEAM;
constexpr int64_t kRecPad = 2 * kTeam + 1;

struct vt_scene {
  int64_t n = 0;
  int64_t E = 0;
  int32_t R = 0;
  int32_t dtype = VT_F32;
  int64_t units = 0;
  float4* rec = nullptr;  // two float4 per unit
  uint32_t* unit = nullptr;
  float4* site = nullptr;
  float4* body = nullptr;
  // optional FP16 offsets (VT_SCENE_HALF_OFFSETS), 16 bytes per unit of rec: a
  // quad's {x0..x3, y0..y3}, {z0..z3, 0}
  uint4* rec_h = nullptr;
  void* tex = nullptr;
  void* tex_vd = nullptr;  // view-dependent texture (appearance 1), same layout as tex
  int32_t* perm = nullptr;
  int32_t* inv = nullptr;
  // kernel-detected errors [0], FP64 recheck counter [1]
  unsigned long long* d_err = nullptr;
  // start-cell search: its result and the scan's per-block minima
  vt_anchors* anchors = nullptr;
  unsigned long long* anchor_part = nullptr;
  // validation of an update: the device word that its kernels look at, its copy
  // for the host, the events behind the copy and behind the last of the kernels
  // (made by the first update); one update at a time
  std::mutex update_mu;
  unsigned* bad = nullptr;
  unsigned* host_bad = nullptr;
  cudaEvent_t bad_copied = nullptr;
  cudaEvent_t bad_read = nullptr;
  // backward scratch: per-cell {dL/ds_x, dL/ds_y, dL/ds_z, dL/dsigma} (twice: even
  // and odd warps' sums), per-texel RGBA
  float4* g_cell = nullptr;
  float4* g_tex = nullptr;
  float4* g_tex_vd = nullptr;
  // cells whose texel scratch holds sums (set by the backward walk, cleared
  // by the gradient permute, which also re-zeroes those cells' scratch);
  // g_tex_clean: the texel scratch is zero outside the flagged cells
  uint8_t* g_touched = nullptr;
  bool g_tex_clean = false;
  // g_held: the flagged cells' blocks hold the sums of a scene-order backward
  // (vt_render_bwd_scene_order) that the caller may still read
  bool g_held = false;
};

// Kernels this library has launched since the process started (all devices
// and threads), read with vt_kernel_launches(); every launch site adds one.
extern std::atomic<unsigned long long> g_vt_launches;
static inline void vt_note_launch() { g_vt_launches.fetch_add(1, std::memory_order_relaxed); }

static inline size_t vt_texel_bytes(int32_t dtype) { return dtype == VT_F32 ? 16 : 8; }

#define VT_CUDA_TRY(expr)                     \
  do {                                        \
    cudaError_t e_ = (expr);                  \
    if (e_ != cudaSuccess) {                  \
      if (e_ == cudaErrorMemoryAllocation) {  \
        cudaGetLastError();                   \
        return VT_ERR_OOM;                    \
      }                                       \
      return VT_ERR_CUDA;                     \
    }                                         \
  } while (0)

// W consecutive floats, a 16-byte access for W = 4
template <int W>
struct Chan {
  float x[W];
};
template <int W>
__device__ __forceinline__ Chan<W> load_chan(const float* p) {
  Chan<W> c;
  if constexpr (W == 4) {
    const float4 q = *reinterpret_cast<const float4*>(p);
    c.x[0] = q.x, c.x[1] = q.y, c.x[2] = q.z, c.x[3] = q.w;
  } else {
#pragma unroll
    for (int i = 0; i < W; ++i) c.x[i] = p[i];
  }
  return c;
}
template <int W>
__device__ __forceinline__ void store_chan(float* p, const Chan<W>& c) {
  if constexpr (W == 4)
    *reinterpret_cast<float4*>(p) = make_float4(c.x[0], c.x[1], c.x[2], c.x[3]);
  else
#pragma unroll
    for (int i = 0; i < W; ++i) p[i] = c.x[i];
}

// a + b = s + e exactly (TwoSum, Knuth)
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
  s = __fadd_rn(a, b);
  float bb = __fsub_rn(s, a);
  e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}

// A thread's share of a loss sum: FP32 pairs with error-free sums and products,
// 48 bits to FP64's 53, as an FP64 operation takes as long as 64 FP32 ones and one
// per channel costs more than the memory. (Against exact sums of squares, worst of
// uniform, normal and log-normal terms: 1.2e-13 of 128, 1e-12 of 4,096; the losses
// are then rounded to FP32, 6e-8.) What FP32 does not hold goes
// to an FP64 sum: terms beyond 2^100, infinities and NaN; chunks whose largest
// number is beyond 2^50 or below 2^-51 (the errors of smaller squares are not FP32
// numbers; beside a larger square of the chunk they do not count).
struct LossSum {
  float hi = 0.f, lo = 0.f;
  double far = 0.0;
  __device__ __forceinline__ void add_pair(float x, float xe) {
    float s, e;
    two_sum(hi, x, s, e);
    hi = s;
    lo = __fadd_rn(lo, __fadd_rn(e, xe));
  }
  __device__ __forceinline__ void add(float x) {
    if (fabsf(x) <= 0x1p100f)
      add_pair(x, 0.f);
    else
      far += (double)x;
  }
  // Where a chunk's squares are at most the sum so far, hi - s below is exact
  // (s <= 2 hi): one rounding each of a square's sum and of that sum's error.
  template <int W>
  __device__ __forceinline__ void add_squares(const Chan<W>& r) {
    float m = 0.f;
#pragma unroll
    for (int i = 0; i < W; ++i) m = fmaxf(m, fabsf(r.x[i]));
    if (__fmul_rn(m, m) <= hi && hi >= 0x1p-100f && hi <= 0x1p110f) {  // (a NaN in r makes hi one)
#pragma unroll
      for (int i = 0; i < W; ++i) {
        const float s = __fmaf_rn(r.x[i], r.x[i], hi);
        lo = __fadd_rn(lo, __fmaf_rn(r.x[i], r.x[i], __fsub_rn(hi, s)));
        hi = s;
      }
      return;
    }
    bool near = m >= 0x1p-51f || m == 0.f;
#pragma unroll
    for (int i = 0; i < W; ++i) near = near && fabsf(r.x[i]) <= 0x1p50f;  // (false for NaN)
    if (near) {
#pragma unroll
      for (int i = 0; i < W; ++i) {
        const float p = __fmul_rn(r.x[i], r.x[i]);
        add_pair(p, __fmaf_rn(r.x[i], r.x[i], -p));
      }
    } else {
#pragma unroll
      for (int i = 0; i < W; ++i) far += (double)r.x[i] * (double)r.x[i];
    }
  }
  __device__ __forceinline__ double total() const { return far + ((double)hi + (double)lo); }
};

static inline int vt_grid(int64_t n, int block, int64_t cap = 1 << 30) {
  int64_t g = (n + block - 1) / block;
  if (g < 1) g = 1;
  if (g > cap) g = cap;
  return (int)g;
}
