// FFT passes of the PM step, with the k-space operations of the method fused
// into the passes that already hold the data in shared memory.
//
// A 3-D real transform is three passes over HBM: rows along x (contiguous,
// real <-> half spectrum by the two-for-one packing z = x[2j] + i x[2j+1]),
// then columns along y and along z (tiles of TW >= 4 adjacent kx columns, so
// every row segment of a tile is at least one whole 32-byte sector).
//
// Every pass is a persistent kernel (grid = SMs x resident CTAs) that walks
// its tiles in a software pipeline: the next tile is staged with cp.async into
// a second shared-memory buffer while the current tile is transformed.  The
// half spectra use the plane-interleaved layout of cola_internal.h.
//
// Most k-space operations and output stores run inside the tile transforms,
// through their load hook (first step) and store hook (last step), so a tile
// makes one round trip through shared memory per transform step and outputs
// leave for HBM from registers.
//
// Fusions:
//   * the z pass of a forward transform also applies the Green's function
//     (and G_eff, screening coupling, gradient) and runs the inverse z pass of
//     each output before writing it back (Poisson solve, App. B);
//   * the y inverse pass can emit the y derivative as a second output;
//   * the x inverse pass can apply the x derivative on load, and transforms up
//     to six independent arrays in one launch;
//   * the screening source S = delta * eps is formed between an inverse and a
//     forward x pass in one kernel (Sec. 6.1, Sec. 6.2);
//   * the LPT reweight by the per-k growth tables (Sec. 4.1, App. A) happens
//     on load of the z inverse pass.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <algorithm>
#include <mutex>
#include <type_traits>
#include <vector>

#include "cola_internal.h"
#include "fft.cuh"

namespace cola {
namespace {

constexpr int NT = 256;

// Column tile width: about 4096 complex values per buffer, between 4 and 16
// columns; 8 columns (64-byte row segments) for single-array 1024-point columns.
constexpr int col_tw(int N, int NBUF) {
  return (N == 1024 && NBUF == 1) ? 8
         : (4096 / (N * NBUF)) < 4 ? 4 : ((4096 / (N * NBUF)) > 16 ? 16 : 4096 / (N * NBUF));
}
// Tile and CTA of an x pass over rows of N reals: rows per tile, threads, resident
// CTAs per SM it is compiled for.  RowBig: about 8192 staged values (~64 KB in flight
// per CTA pair), 8..64 rows, 256 threads.  RowSmall: 128 threads that are all busy in
// both steps (at 1024 points 8 rows give 128 items of the radix-32 step).
struct RowShape {
  int rows, threads, ctas;
};
constexpr RowShape row_big(int N) {
  return N >= 1024 ? RowShape{8, 256, 2} : N == 512 ? RowShape{16, 256, 3} : N == 256 ? RowShape{32, 256, 2} : RowShape{64, 256, 3};
}
constexpr RowShape row_small(int N) {
  return N >= 1024 ? RowShape{8, 128, 2} : N == 512 ? RowShape{8, 128, 5} : N == 256 ? RowShape{16, 128, 5} : N == 128 ? RowShape{16, 128, 6} : RowShape{32, 128, 6};
}
// Measured on GB300 (us per launch, big / small, with CTA barriers between the steps): x r2c
// 512: 179 / 188, 256: 28.0 / 27.3; force c2r (pair and F_z) 1024: 4332 / 4032, 512: 538 / 540,
// 256: 82 / 78; LPT c2r (six fields) 512: 1006 / 1091, 256: 139 / 146; screening 1024: 3237 /
// 3386 (big with its radix-32 step on lane pairs), 512: 351 / 329, 256: 54 / 50.  With whole rows
// per warp and warp barriers only (fft_rowtile) and the tile staged by the CTA in memory order:
// force c2r 1024: 3876, 512: 522; LPT c2r 256: 130; r2c 512: 179, 1024: 1318 (small).  The
// screening pass, the one far from the DRAM rate, also stages per warp and has no CTA barrier:
// 1024: 2409, 512: 298, 256: 45; the others lose 3-10 % to the shorter pieces that way.
constexpr RowShape r2c_shape(int N) { return N == 256 || N >= 1024 ? row_small(N) : row_big(N); }
constexpr RowShape c2r_shape(int N) { return N >= 1024 ? row_small(N) : row_big(N); }
constexpr RowShape pair_shape(int N) { return N >= 1024 || N == 256 ? row_small(N) : row_big(N); }
constexpr RowShape screen_shape(int N) { return N >= 1024 ? row_big(N) : row_small(N); }

// Resident CTAs per SM that the shared memory of a kernel allows (1..3); used
// as the register bound of __launch_bounds__ so registers never limit occupancy
// below it.  Transforms of 512 points and more, and the force-side z passes
// (two transforms per tile), would spill at 3 and take at most 2.
constexpr int blocks_for_smem(size_t bytes, int N) {
  return bytes > 112 * 1024 ? 1 : (bytes > 72 * 1024 || N >= 512 ? 2 : 3);
}
// Stage buffer of a column tile: fft_rows rows (the transform's padding rows
// follow the N data rows) of NBUF arrays x TW columns.
constexpr int col_rows(int N) { return N + (1 << (ilog2(N) - ilog2(N) / 2)); }
constexpr size_t col_smem_c(int N, int NBUF) {
  return (N + 2 * (size_t)col_rows(N) * NBUF * col_tw(N, NBUF)) * 8;
}
// the same for an explicit tile width
constexpr size_t col_smem_tw(int N, int TW) { return (N + 2 * (size_t)col_rows(N) * TW) * 8; }
// Tiles and threads of the fused force-side z passes (screening field, force).  What
// bounds them is latency: two or three transforms per tile, each a chain of shared
// memory, arithmetic and barriers, at about 40 % of the issue and half of the DRAM
// rate.  Small CTAs that keep every thread busy in every step and drift apart hide it:
// 128 threads on 8 columns (16 up to 128 points) with all the registers the items of a
// radix-32 step take.  Per launch, against one or two CTAs of 256 threads (half of them
// idle in the longer step below 1024 points), us, screening field / force: 512^3 mesh
// 326 / 565 -> 271 / 498, 256^3 47 / 80 -> 42 / 59, 256 meshes of 128^3 642 / 1148 ->
// 533 / 964.  At 1024 points two tiles of 8 columns fill shared memory (one CTA of 256
// threads); 4-column tiles in CTAs of 128 threads lose more to their 32-byte rows
// (2.35 / 4.17 -> 2.84 / 4.94 ms).
constexpr int ztw(int N) { return N == 256 ? 8 : col_tw(N, 1); }
constexpr int zt(int N) { return N <= 512 ? 128 : NT; }
// Resident CTAs per SM they are compiled for (shared memory; 3 at 512 points: 295 us).
constexpr int zblocks(int N) { return N <= 256 ? 4 : N <= 512 ? 2 : 1; }

// Tiles, threads and resident CTAs per SM of the y passes (and the plain z pass): as the
// fused z passes, small CTAs without idle threads; the y inverse with its derivative reads
// each input once and starts both transforms from it (fft_tile_inv_deriv).  Per launch,
// us: y forward 512^3 216 -> 190, 256^3 31.2 -> 27.5; force y inverse (three arrays in two
// launches and the screening field's) 512^3 238 -> 222 mean, 1024^3 1810 -> 1713.
__host__ __device__ constexpr int ytw(int N) { return N >= 256 ? 8 : 16; }
__host__ __device__ constexpr int yt(int N) { return N >= 1024 ? 256 : 128; }
constexpr int ycol_blocks(int N) { return N >= 1024 ? 1 : N == 512 ? 3 : 5; }
// The plain forward passes of 128 points (P(k), initial conditions: the step transforms such a
// mesh plane by plane) keep CTAs of 256 threads, three per SM: P(k) of 128 meshes in one
// launch sequence 3.44 -> 3.31 ms.  The inverse ones do not: initial conditions of eight lattices
// of 128^3 2.79 ms, 2.84 with the larger CTAs.
__host__ __device__ constexpr int ct(int N, bool INV) { return N == 128 && !INV ? 256 : yt(N); }
constexpr int ct_blocks(int N, bool INV) { return N == 128 && !INV ? 3 : ycol_blocks(N); }
constexpr int yinv_blocks(int N) { return N >= 1024 ? 1 : N == 512 ? 2 : 4; }

int sm_count() {
  static int n = 0;
  if (n == 0) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    if (n <= 0) n = 1;
  }
  return n;
}

thread_local int g_grid_cap = 0;  // 0: no cap (see set_grid_cap)

struct KernelInfo {
  const void* fn;
  size_t smem;
  int per_sm;
};
std::mutex g_kinfo_mu;
std::vector<KernelInfo> g_kinfo;

// Largest dynamic shared memory a CTA may be given on this device.
size_t smem_most() {
  static const size_t most = [] {
    int dev = 0, n = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    return n > 0 ? (size_t)n : (size_t)48 * 1024;
  }();
  return most;
}

// Raises the shared-memory limit of a kernel where a launch needs more than those before, and
// caches its resident CTAs per SM for each size.  The limit is never lowered: launches of
// every size seen so far rely on it.
template <class K>
cudaError_t resident_ctas(K kernel, size_t smem, int& per_sm, int threads) {
  std::lock_guard<std::mutex> lk(g_kinfo_mu);
  size_t limit = 48 * 1024;
  for (const KernelInfo& k : g_kinfo)
    if (k.fn == (const void*)kernel) {
      if (k.smem == smem) {
        per_sm = k.per_sm;
        return cudaSuccess;
      }
      limit = std::max(limit, k.smem);
    }
  if (smem > limit) {
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
  }
  cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, smem);
  if (e != cudaSuccess) return e;
  g_kinfo.push_back({(const void*)kernel, smem, per_sm});
  return cudaSuccess;
}

// Persistent grid: resident CTAs x SMs, at most one CTA per tile, at most the
// calling thread's grid cap (used when many small simulations run concurrently).
template <class K>
cudaError_t prep(K kernel, size_t smem, int64_t ntiles, unsigned& grid, int threads = NT) {
  if (ntiles >= ((int64_t)1 << 31)) return cudaErrorInvalidValue;  // tile indices are 32-bit
  int per_sm = 0;
  cudaError_t e = resident_ctas(kernel, smem, per_sm, threads);
  if (e != cudaSuccess) return e;
  if (per_sm < 1) return cudaErrorInvalidConfiguration;
  int64_t g = std::min<int64_t>(ntiles, (int64_t)per_sm * sm_count());
  if (g_grid_cap > 0) g = std::min<int64_t>(g, g_grid_cap);
  grid = (unsigned)std::max<int64_t>(g, 1);
  return cudaSuccess;
}

template <int T = NT>
__device__ __forceinline__ void load_tw(float2* tw, const float2* __restrict__ twg, int n) {
  for (int i = threadIdx.x; i < n; i += T) tw[i] = twg[i];
}

// Twiddles of an x pass over rows of N reals (M = N/2 complex): entries 0..M the
// table exp(-2 pi i k / N) of the real <-> half-spectrum split, entry M + k1 R2 + n2
// (k1 >= 1) the row transform's first-step twiddle (fft_rowtile), which therefore
// takes w1 = tw + M.  Together they fill the N entries of the plain table.
template <int N, int T>
__device__ __forceinline__ void load_row_tw(float2* tw, const float2* __restrict__ twg) {
  constexpr int M = N / 2;
  for (int i = threadIdx.x; i < N; i += T) {
    const int j = i - M;
    if (i <= M || j >= Split<M>::R2) tw[i] = twg[i <= M ? i : 2 * row_twiddle<M>(j)];
  }
}

// Start of a kernel launched with launch_pdl: the twiddle table to the start of shared
// memory, then the wait for the kernels before.
template <int T>
__device__ __forceinline__ void pdl_begin(const float2* __restrict__ twg, int n) {
  extern __shared__ __align__(128) float2 sm[];
  load_tw<T>(sm, twg, n);
  pdl_wait();
}

// ---------------------------------------------------------------- cp.async helpers
__device__ __forceinline__ void cp_async16(void* smem, const void* gmem, bool valid) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
  const int sz = valid ? 16 : 0;  // 0: zero-fill, nothing read
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(s), "l"(gmem), "r"(sz)
               : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int n>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;\n" ::"n"(n) : "memory");
}

// ---------------------------------------------------------------- column tiles
// Tile element (n, c) of sub-block `sub` lives at buf[n * TP + sub * TW + c];
// global element at g[base + row(n) + hcol(c)] with row(n) = (n / HQ) ra +
// (n mod HQ) rb (the half-spectrum layout of cola_internal.h); only columns
// c0 + c < N/2 + 1 exist.  Each thread keeps one 16-byte piece (or one column)
// and walks rows n0, n0 + step, ... (HQ | step, so n mod HQ stays fixed).
template <int N, int TW, int TP, int T = NT>
__device__ __forceinline__ void col_issue(float2* buf, int sub, const float2* __restrict__ g,
                                          int64_t base, int64_t ra, int64_t rb, int c0) {
  constexpr int CH = TW / 2;  // 16-byte pieces per row segment
  constexpr int STEP = T / CH;
  static_assert(STEP % HQ == 0, "row step: whole plane groups");
  const int j = threadIdx.x % CH, n0 = threadIdx.x / CH;
  const bool v = c0 + 2 * j < N / 2 + 1;
  const float2* src = g + base + (n0 / HQ) * ra + (n0 % HQ) * rb + hcol(2 * j);
  float2* dst = buf + n0 * TP + sub * TW + 2 * j;
#pragma unroll 4
  for (int n = n0; n < N; n += STEP) {
    cp_async16(dst, v ? (const void*)src : (const void*)g, v);
    src += (STEP / HQ) * ra;
    dst += STEP * TP;
  }
}

// 16-bit seeds: 4 complex values (uint32 each) per 16-byte chunk.  Field f of
// row n is staged raw in the sub-block 2/3 area of that row:
// raw(f, n, c) = ((uint32*)buf)[8 n TW + 4 TW + f TW + c]  (TP = 4 TW).
template <int N, int TW>
__device__ __forceinline__ void col_issue_raw(uint32_t* rb_, int f, const uint32_t* __restrict__ g,
                                              int64_t base, int64_t ra, int64_t rb, int c0) {
  constexpr int CH = TW / 4;
  constexpr int STEP = NT / CH;
  static_assert(STEP % HQ == 0, "row step: whole plane groups");
  const int j = threadIdx.x % CH, n0 = threadIdx.x / CH;
  const bool v = c0 + 4 * j < N / 2 + 1;
  const uint32_t* src = g + base + (n0 / HQ) * ra + (n0 % HQ) * rb + hcol(4 * j);
  uint32_t* dst = rb_ + 8 * n0 * TW + 4 * TW + f * TW + 4 * j;
#pragma unroll 4
  for (int n = n0; n < N; n += STEP) {
    cp_async16(dst, v ? (const void*)src : (const void*)g, v);
    src += (STEP / HQ) * ra;
    dst += 8 * STEP * TW;
  }
}

template <int N, int TW, int TP>
__device__ __forceinline__ void col_store(const float2* buf, int sub, float2* __restrict__ g,
                                          int64_t base, int64_t ra, int64_t rb, int c0) {
  constexpr int STEP = NT / TW;
  static_assert(STEP % HQ == 0, "row step: whole plane groups");
  const int c = threadIdx.x % TW, n0 = threadIdx.x / TW;
  if (c0 + c >= N / 2 + 1) return;
  float2* dst = g + base + (n0 / HQ) * ra + (n0 % HQ) * rb + hcol(c);
  const float2* src = buf + n0 * TP + sub * TW + c;
#pragma unroll 4
  for (int n = n0; n < N; n += STEP) {
    *dst = *src;
    dst += (STEP / HQ) * ra;
    src += STEP * TP;
  }
}

// The elements of an N x TW column tile that a thread owns: column c = tid mod
// TW and rows n = n0 + i STEP, i < E (STEP = NT / TW, n0 = tid / TW).  |n|^2
// of element (kx, ky, n) is sxy + fz(n)^2 with sxy = kx^2 + ky^2 kept per
// thread; the integer sum is exact, so k^2 = kf^2 |n|^2 rounds once.
template <int N, int TW>
struct TileLane {
  static constexpr int STEP = NT / TW, E = N * TW / NT;
  int c, n0, sxy;
  __device__ __forceinline__ TileLane(int c0, int iy) {
    c = threadIdx.x % TW;
    n0 = threadIdx.x / TW;
    const int fx = c0 + c, fy = freq_index(iy, N);
    sxy = fx * fx + fy * fy;
  }
  __device__ __forceinline__ int row(int i) const { return n0 + i * STEP; }
  __device__ __forceinline__ float k2(int n, float kf2) const {
    const int fz = freq_index(n, N);
    return kf2 * (float)(sxy + fz * fz);
  }
};

// Store hook of a column transform that writes element (n, c) straight to
// g[(n / HQ) ra + (n mod HQ) rb + hcol(c)] (g = the tile's base, columns c < live
// exist) instead of through the tile and col_store: a warp's stores cover whole
// 64-byte chunks.
struct ColOut {
  static constexpr bool kSmem = false;
  float2* g;
  int64_t ra, rb;
  int live;
  __device__ __forceinline__ float2 operator()(float2 v, int n, int c, int) const {
    if (c < live) g[(n / HQ) * ra + (n % HQ) * rb + hcol(c)] = v;
    return v;
  }
};

// Column geometry: tile t -> (simulation b, outer index o, column block c0);
// base = the element offset of (o, row 0, c0) and `by` = the byte shift of
// simulation b's buffers.  Outer index o sits at (o / HQ) oa + (o mod HQ) ob and
// tile row n at (n / HQ) ra + (n mod HQ) rb.  Along y, consecutive tiles take the
// HQ planes o of one group at the same column block (the parts of each chunk
// group are read by neighbouring CTAs together).
template <int N, int TW>
struct ColGeo {
  static constexpr int ntx = (N / 2) / TW + 1;
  static constexpr int64_t tps = (int64_t)N * ntx;  // tiles per simulation
  int64_t oa, ob, ra, rb;
  int zaxis;  // 1: tiles run along z (o = y), 0: along y (o = z)
  Multi m;
  // t < 2^31 (prep checks the tile count); divisions by compile-time constants
  __device__ __forceinline__ void tile(int64_t t64, int& o, int& c0, int64_t& base, int64_t& by) const {
    uint32_t t = (uint32_t)t64;
    const uint32_t b = t / (uint32_t)tps;
    t -= b * (uint32_t)tps;
    by = shift_of(m, (int)b);
    if (!zaxis) {
      const uint32_t q = t / (HQ * ntx), r = t - q * (HQ * ntx);
      o = (int)(q * HQ + r % HQ);
      c0 = (int)(r / HQ) * TW;
    } else {
      const uint32_t q = t / ntx;
      o = (int)q;
      c0 = (int)(t - q * ntx) * TW;
    }
    base = (o / HQ) * oa + (o % HQ) * ob + hcol(c0);
  }
};

// Software pipeline over the tiles of one launch.  Op supplies
//   issue(buf, t): cp.async the inputs of tile t into buf (no commit)
//   process(buf, tw, t): transform + store (leaves buf free after a final barrier)
// and, with kSide (a second input, landing in op.extra),
//   issue_side(t): cp.async of tile t's second input (no commit)
//   process(buf, tw, t, next): next() once op.extra has been read; it issues the
//     next tile's second input and commits it, so that it lands while this tile's
//     outputs are formed.  process() waits for its own with cp_async_wait<1>(),
//     which leaves the prefetch of tile t + grid in flight.
template <int N, int BUFELEMS, int T = NT, class Op>
__device__ __forceinline__ void col_pipeline(Op op, const float2* __restrict__ twg,
                                             int64_t ntiles) {
  extern __shared__ __align__(128) float2 sm[];
  float2* tw = sm;
  float2* b0 = sm + N;
  float2* b1 = b0 + BUFELEMS;
  op.extra = b1 + BUFELEMS;  // optional per-op scratch after the two stage buffers
  if (!Op::kTwReady) load_tw<T>(tw, twg, N);
  int64_t t = blockIdx.x;
  if (t < ntiles) op.issue(b0, t);
  cp_async_commit();
  if constexpr (Op::kSide) {
    if (t < ntiles) op.issue_side(t);
    cp_async_commit();
  }
  int cur = 0;
  for (; t < ntiles; t += gridDim.x) {
    const int64_t tn = t + gridDim.x;
    if (tn < ntiles) op.issue(cur ? b0 : b1, tn);
    cp_async_commit();
    cp_async_wait<Op::kSide ? 2 : 1>();  // tile t's main input has landed
    __syncthreads();
    if (Op::kTwReady && tn >= ntiles) pdl_go();  // the CTA's last tile
    if constexpr (Op::kSide) {
      op.process(cur ? b1 : b0, tw, t, [&] {
        if (tn < ntiles) op.issue_side(tn);
        cp_async_commit();
      });
    } else {
      op.process(cur ? b1 : b0, tw, t);
    }
    __syncthreads();
    cur ^= 1;
  }
  cp_async_wait<0>();
}

// ---------------------------------------------------------------- TMA tile loads
// Single-simulation launches of the long column passes stage their tiles with
// the tensor-memory accelerator: thread 0 issues a few cp.async.bulk.tensor
// copies per tile, completion is tracked by an mbarrier per stage buffer, and
// the transform warps issue no load instructions.  The half spectrum is seen
// as a 5-D array of 8-byte elements (column within a 64-byte chunk, plane
// within its group, chunk, y, plane group), byte strides 8, 64, 64 HQ, 8 HQ P,
// 8 HQ N P: the interleaved layout of cola_internal.h.  A z tile (TW <= 8 columns
// of one y) is boxes of {TW, HQ, 1, 1, <= 256 groups}, landing as rows n = HQ j +
// plane of TW values; a y tile (one z) boxes of {TW, 1, 1, <= 256 rows, 1}.
__device__ unsigned int g_tile_load_failures;  // waits that ran out (host: tile_load_failures)

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void bar_init(uint64_t* b) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(smem_u32(b)) : "memory");
}
__device__ __forceinline__ void bar_expect(uint64_t* b, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(smem_u32(b)), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ bool bar_try(uint64_t* b, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(smem_u32(b)), "r"(parity)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ uint64_t global_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
// Wait for phase `parity` of b to complete, for limit_ns (one second) at most.
__device__ __forceinline__ bool bar_wait(uint64_t* b, uint32_t parity,
                                         uint64_t limit_ns = 1000000000ull) {
  if (bar_try(b, parity)) return true;
  const uint64_t t0 = global_ns();
  while (!bar_try(b, parity))
    if (global_ns() - t0 > limit_ns) return false;
  return true;
}
// orders this CTA's earlier generic-proxy accesses to shared memory before
// later async-proxy (TMA) writes
__device__ __forceinline__ void fence_async_smem() {
  asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
}
__device__ __forceinline__ void fence_bar_init() {
  asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
}
__device__ __forceinline__ void tma_load5(void* dst, const CUtensorMap* map, int c0, int c1, int c2, int c3,
                                          int c4, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.5d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, "
      "%4, %5, %6}], [%7];\n" ::"r"(smem_u32(dst)),
      "l"(map), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(c4), "r"(smem_u32(bar))
      : "memory");
}

// 1-D bulk copy of `bytes` (a multiple of 16; both addresses 16-byte aligned)
// from global memory into shared memory, completing on bar.
__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(
          smem_u32(dst)),
      "l"(src), "r"(bytes), "r"(smem_u32(bar))
      : "memory");
}

// Zero fill by bulk stores from a zeroed shared-memory region (thread 0): `bytes`
// (a multiple of 16) at dst, in pieces of at most ZB bytes, one bulk group; at
// most eight groups stay outstanding (the region is never written again, so
// only the count is bounded).
__device__ __forceinline__ void bulk_zero(char* dst, int64_t bytes, const void* zeros, uint32_t ZB) {
  for (int64_t o = 0; o < bytes; o += ZB) {
    const uint32_t len = (uint32_t)(bytes - o < (int64_t)ZB ? bytes - o : (int64_t)ZB);
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;\n" ::"l"(dst + o),
                 "r"(smem_u32(zeros)), "r"(len)
                 : "memory");
  }
  asm volatile("cp.async.bulk.commit_group;\n" ::: "memory");
  asm volatile("cp.async.bulk.wait_group.read 8;\n" ::: "memory");
}
__device__ __forceinline__ void bulk_store_drain() { asm volatile("cp.async.bulk.wait_group 0;\n" ::: "memory"); }

// Issue the loads of column tile t of `geo` into buf (thread 0; buf 128-byte aligned).
template <int N, int TW>
__device__ __forceinline__ void tma_tile(const ColGeo<N, TW>& geo, const CUtensorMap* map, float2* buf,
                                         int64_t t, uint64_t* bar) {
  static_assert(TW <= 8 && TW % 2 == 0, "TMA tiles: at most one 64-byte chunk");
  int o, c0;
  int64_t base, by;
  geo.tile(t, o, c0, base, by);
  bar_expect(bar, (uint32_t)(N * TW * sizeof(float2)));
  if (geo.zaxis) {
    constexpr int B = N / HQ < 256 ? N / HQ : 256;
#pragma unroll
    for (int k = 0; k < N / HQ; k += B) tma_load5(buf + HQ * k * TW, map, c0 & 7, 0, c0 >> 3, o, k, bar);
  } else {
    constexpr int B = N < 256 ? N : 256;
#pragma unroll
    for (int k = 0; k < N; k += B) tma_load5(buf + k * TW, map, c0 & 7, o % HQ, c0 >> 3, k, o / HQ, bar);
  }
}

// col_pipeline with TMA staging (one simulation).  Op supplies geo, process()
// and, for a side input (kSide), the members sbar / spar that its process()
// waits on through tma_side_wait; map1 is the side input's tensor map.
// Barriers: bars[0], bars[1] for the two stage buffers, bars[2] for the side
// input (landing in op.extra, N x TW).  A wait that runs out stops the CTA
// (counted in g_tile_load_failures) after a bounded wait for its copies.
struct TmaSide {
  uint64_t* bar = nullptr;
  uint32_t parity = 0;
  int* fail = nullptr;
  // thread 0 waits; the caller's next barrier publishes the data
  __device__ __forceinline__ void wait() const {
    if (bar && threadIdx.x == 0 && !bar_wait(bar, parity)) *fail = 1;
  }
};

// Shared memory: twiddles (N), two stage buffers, EXTRA float2 of op.extra,
// then the three barriers and the failure flag.
template <int N, int BUFELEMS, int EXTRA>
constexpr size_t tma_smem() {
  return ((size_t)N + 2 * (size_t)BUFELEMS + EXTRA) * sizeof(float2) + 4 * sizeof(uint64_t);
}

template <int N, int BUFELEMS, bool SIDE, int EXTRA, int T, class Op>
__device__ __forceinline__ void col_pipeline_tma(Op op, const float2* __restrict__ twg, int64_t ntiles,
                                                 const CUtensorMap* map0, const CUtensorMap* map1) {
  static_assert((N * sizeof(float2)) % 128 == 0 && (BUFELEMS * sizeof(float2)) % 128 == 0,
                "TMA destinations 128-byte aligned");
  extern __shared__ __align__(128) float2 sm[];
  float2* tw = sm;
  float2* b0 = sm + N;
  float2* b1 = b0 + BUFELEMS;
  op.extra = b1 + BUFELEMS;
  uint64_t* bars = reinterpret_cast<uint64_t*>(op.extra + EXTRA);
  int& fail = *reinterpret_cast<int*>(bars + 3);
  const bool lead = threadIdx.x == 0;
  if (lead) {
    bar_init(&bars[0]);
    bar_init(&bars[1]);
    bar_init(&bars[2]);
    fence_bar_init();
    fail = (smem_u32(sm) & 127) ? 1 : 0;  // no copy goes into a misaligned buffer
  }
  if (!Op::kTwReady) load_tw<T>(tw, twg, N);
  __syncthreads();
  if (fail) {
    if (lead) atomicAdd(&g_tile_load_failures, 1u);
    return;
  }
  // thread 0: parity of each barrier's next phase (bit i) and copies issued but
  // not yet waited for (bit i)
  uint32_t par = 0, pend = 0;
  int64_t t = blockIdx.x;
  if (lead && t < ntiles) {
    tma_tile(op.geo, map0, b0, t, &bars[0]);
    pend |= 1u;
    if (SIDE) {
      tma_tile(op.geo, map1, op.extra, t, &bars[2]);
      pend |= 4u;
    }
  }
  int cur = 0;
  for (; t < ntiles; t += gridDim.x) {
    const int64_t tn = t + gridDim.x;
    if (lead) {
      fence_async_smem();  // the previous tile's accesses to the buffers are done
      if (tn < ntiles) {
        tma_tile(op.geo, map0, cur ? b0 : b1, tn, &bars[cur ^ 1]);
        pend |= 1u << (cur ^ 1);
      }
      if (bar_wait(&bars[cur], (par >> cur) & 1u)) {
        par ^= 1u << cur;
        pend &= ~(1u << cur);
      } else {
        fail = 1;
      }
    }
    __syncthreads();
    if (fail) break;
    if (Op::kTwReady && tn >= ntiles) pdl_go();  // the CTA's last tile
    if constexpr (SIDE) {
      op.side = TmaSide{&bars[2], (par >> 2) & 1u, &fail};
      // after the tile's second input has been read: the next tile's (unless this one's
      // wait ran out, in which case its copy is still pending)
      op.process(cur ? b1 : b0, tw, t, [&] {
        if (!lead || fail) return;
        par ^= 4u;
        pend &= ~4u;
        if (tn < ntiles) {
          fence_async_smem();
          tma_tile(op.geo, map1, op.extra, tn, &bars[2]);
          pend |= 4u;
        }
      });
    } else if constexpr (Op::kSide) {
      op.process(cur ? b1 : b0, tw, t, [] {});
    } else {
      op.process(cur ? b1 : b0, tw, t);
    }
    __syncthreads();
    if (fail) break;
    cur ^= 1;
  }
  if (lead && fail) {
    atomicAdd(&g_tile_load_failures, 1u);
    for (int i = 0; i < 3; ++i)
      if ((pend >> i) & 1u) bar_wait(&bars[i], (par >> i) & 1u);  // bounded: copies in flight land before exit
  }
}

// Self-test of the bounded wait: one thread arms a barrier phase for 16 bytes
// that no copy will deliver and waits on it with bar_wait; g_wait_probe = 1 when
// the wait gave up after limit_ns, 0 if the phase completed.
__device__ int g_wait_probe;
__global__ void k_wait_probe(uint64_t limit_ns) {
  __shared__ __align__(8) uint64_t bar;
  if (threadIdx.x != 0) return;
  bar_init(&bar);
  fence_bar_init();
  bar_expect(&bar, 16);
  g_wait_probe = bar_wait(&bar, 0, limit_ns) ? 0 : 1;
}

// ---------------------------------------------------------------- plain column pass
// Dense half spectra [z][y][kx] of the public API (rows of N/2 + 1 values, no padding) as
// the far side of a y pass: stores of a column transform, and the staging of its tiles
// (8-byte pieces: an odd row length leaves no 16-byte alignment).
template <int N>
struct DenseOut {
  static constexpr bool kSmem = false;
  float2* g;  // element (row 0, column 0) of the tile
  int live;
  __device__ __forceinline__ float2 operator()(float2 v, int n, int c, int) const {
    if (c < live) g[n * (N / 2 + 1) + c] = v;
    return v;
  }
};
template <int N, int TW, int T>
__device__ __forceinline__ void col_issue_dense(float2* buf, const float2* __restrict__ g, int live) {
  const int c = threadIdx.x % TW;
  const int sz = c < live ? 8 : 0;  // 0: zero-fill, nothing read
#pragma unroll 4
  for (int n = threadIdx.x / TW; n < N; n += T / TW)
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;\n" ::"r"(smem_u32(buf + n * TW + c)),
                 "l"(g + (c < live ? n * (N / 2 + 1) + c : 0)), "r"(sz)
                 : "memory");
}

// out = transform of in along the tile axis; out may alias in.  DENSE (along y): 1 the
// output, 2 the input is a dense half spectrum.
template <int N, int TW, bool INV, int DENSE>
struct OpCol {
  static constexpr bool kTwReady = false;
  static constexpr int T = ct(N, INV);
  ColGeo<N, TW> geo;
  const float2* in;
  float2* out;
  float2* extra = nullptr;  // scratch after the stage buffers (set by col_pipeline)
  static constexpr bool kSide = false;
  __device__ __forceinline__ void issue(float2* buf, int64_t t) const {
    int o, c0;
    int64_t base, by;
    geo.tile(t, o, c0, base, by);
    if constexpr (DENSE == 2)
      col_issue_dense<N, TW, T>(buf, in + (int64_t)o * N * (N / 2 + 1) + c0, N / 2 + 1 - c0);
    else col_issue<N, TW, TW, T>(buf, 0, moved(in, by), base, geo.ra, geo.rb, c0);
  }
  // outputs go to HBM from the last step's registers
  __device__ __forceinline__ void process(float2* buf, const float2* tw, int64_t t) const {
    int o, c0;
    int64_t base, by;
    geo.tile(t, o, c0, base, by);
    if constexpr (DENSE == 1)
      fft_tile<N, TW, TW, T, INV, 1, TileLoad, DenseOut<N>>(
          buf, tw, TileLoad{}, DenseOut<N>{out + (int64_t)o * N * (N / 2 + 1) + c0, N / 2 + 1 - c0});
    else
      fft_tile<N, TW, TW, T, INV, 1, TileLoad, ColOut>(
          buf, tw, TileLoad{}, ColOut{moved(out, by) + base, geo.ra, geo.rb, N / 2 + 1 - c0});
  }
};

template <int N, int TW, bool INV, bool TMA, int DENSE>
__global__ void __launch_bounds__(ct(N, INV), ct_blocks(N, INV)) k_col(OpCol<N, TW, INV, DENSE> op, const float2* __restrict__ twg,
                                            int64_t ntiles, const __grid_constant__ CUtensorMap map) {
  constexpr int T = ct(N, INV);
  if constexpr (TMA) col_pipeline_tma<N, fft_rows<N>() * TW, false, 0, T>(op, twg, ntiles, &map, nullptr);
  else col_pipeline<N, fft_rows<N>() * TW, T>(op, twg, ntiles);
}

// ---------------------------------------------------------------- y inverse, two outputs
// y inverse with the y derivative as a second output: three tile buffers rotate
// between the input (its intermediate written in place for the plain output), the
// derivative's intermediate and the prefetch of the next input, so the input is read
// from HBM once, and from shared memory once (fft_tile_inv_deriv).  Given input
// buffer I, the derivative goes to (I + 1) mod 3 and the prefetch to (I + 2) mod 3,
// which holds the next tile's input.
template <int N, int TW>
constexpr size_t yinv2r_smem() {
  return (N + 3 * (size_t)fft_rows<N>() * TW) * sizeof(float2);
}

// Both transforms of tile t from input buffer bi (the derivative's intermediate in bd).
template <int N, int TW>
__device__ __forceinline__ void yinv2r_tile(const ColGeo<N, TW>& geo, float2* bi, float2* bd,
                                            const float2* tw, float2* __restrict__ outp,
                                            float2* __restrict__ outd, float kfs, int64_t t) {
  int o, c0;
  int64_t base, by;
  geo.tile(t, o, c0, base, by);
  const ColOut op{moved(outp, by) + base, geo.ra, geo.rb, N / 2 + 1 - c0};
  const ColOut od{moved(outd, by) + base, geo.ra, geo.rb, N / 2 + 1 - c0};
  fft_tile_inv_deriv<N, TW, TW, yt(N)>(bi, bd, tw, kfs, op, od);
}

// TMA: buffer i's copies complete on barrier i (after the three buffers; the
// failure flag follows), as in col_pipeline_tma.
template <int N, int TW, bool TMA>
__global__ void __launch_bounds__(yt(N), yinv_blocks(N)) k_yinv2r(
    ColGeo<N, TW> geo, const float2* __restrict__ in, float2* __restrict__ outp,
    float2* __restrict__ outd, float kfs, const float2* __restrict__ twg, int64_t ntiles,
    const __grid_constant__ CUtensorMap map) {
  constexpr int B = fft_rows<N>() * TW;
  extern __shared__ __align__(128) float2 sm[];
  float2* tw = sm;
  auto buf = [&](int i) { return sm + N + i * B; };
  if constexpr (TMA) {
    static_assert((N * sizeof(float2)) % 128 == 0 && (B * sizeof(float2)) % 128 == 0,
                  "TMA destinations 128-byte aligned");
    uint64_t* bars = reinterpret_cast<uint64_t*>(buf(3));
    int& fail = *reinterpret_cast<int*>(bars + 3);
    const bool lead = threadIdx.x == 0;
    if (lead) {
      bar_init(&bars[0]);
      bar_init(&bars[1]);
      bar_init(&bars[2]);
      fence_bar_init();
      fail = (smem_u32(sm) & 127) ? 1 : 0;
    }
    load_tw<yt(N)>(tw, twg, N);
    __syncthreads();
    if (fail) {
      if (lead) atomicAdd(&g_tile_load_failures, 1u);
      return;
    }
    uint32_t par = 0, pend = 0;  // thread 0: next phase parity and pending copies, bit i = barrier i
    int64_t t = blockIdx.x;
    if (lead && t < ntiles) {
      tma_tile(geo, &map, buf(0), t, &bars[0]);
      pend |= 1u;
    }
    int I = 0;
    for (; t < ntiles; t += gridDim.x) {
      const int D = I == 2 ? 0 : I + 1, F = I == 0 ? 2 : I - 1;
      if (lead) {
        fence_async_smem();
        const int64_t tn = t + gridDim.x;
        if (tn < ntiles) {
          tma_tile(geo, &map, buf(F), tn, &bars[F]);
          pend |= 1u << F;
        }
        if (bar_wait(&bars[I], (par >> I) & 1u)) {
          par ^= 1u << I;
          pend &= ~(1u << I);
        } else {
          fail = 1;
        }
      }
      __syncthreads();
      if (fail) break;
      yinv2r_tile<N, TW>(geo, buf(I), buf(D), tw, outp, outd, kfs, t);
      __syncthreads();  // both buffers are free for later prefetches
      I = F;
    }
    if (lead && fail) {
      atomicAdd(&g_tile_load_failures, 1u);
      for (int i = 0; i < 3; ++i)
        if ((pend >> i) & 1u) bar_wait(&bars[i], (par >> i) & 1u);
    }
  } else {
    load_tw<yt(N)>(tw, twg, N);
    int64_t t = blockIdx.x;
    if (t < ntiles) {
      int o, c0;
      int64_t base, by;
      geo.tile(t, o, c0, base, by);
      col_issue<N, TW, TW, yt(N)>(buf(0), 0, moved(in, by), base, geo.ra, geo.rb, c0);
    }
    cp_async_commit();
    int I = 0;
    for (; t < ntiles; t += gridDim.x) {
      const int D = I == 2 ? 0 : I + 1, F = I == 0 ? 2 : I - 1;
      const int64_t tn = t + gridDim.x;
      if (tn < ntiles) {
        int o, c0;
        int64_t base, by;
        geo.tile(tn, o, c0, base, by);
        col_issue<N, TW, TW, yt(N)>(buf(F), 0, moved(in, by), base, geo.ra, geo.rb, c0);
      }
      cp_async_commit();
      cp_async_wait<1>();  // tile t's input has landed
      __syncthreads();
      yinv2r_tile<N, TW>(geo, buf(I), buf(D), tw, outp, outd, kfs, t);
      __syncthreads();  // both buffers are free for later prefetches
      I = F;
    }
    cp_async_wait<0>();
  }
}

// ---------------------------------------------------------------- screening field (z pass)
// Smoothing window of the Vainshtein density (App. B) at h = k^2 R^2 / 2:
// 0 Gaussian exp(-h); 1 top-hat 3 (sin x - x cos x) / x^3 with x^2 = 2h, by its
// Taylor series below x = 1/2 where the closed form cancels; 2 sharp-k, 1 for
// kR <= 1 (h <= 1/2) and 0 beyond.
__device__ __forceinline__ float smoothing_window(float h, int filter) {
  if (filter == 0) return __expf(-h);
  if (filter == 2) return h <= 0.5f ? 1.f : 0.f;
  const float x2 = 2.f * h;
  if (x2 < 0.25f)
    return fmaf(x2, fmaf(x2, fmaf(x2, fmaf(x2, 1.f / 1330560.f, -1.f / 15120.f), 1.f / 280.f), -0.1f), 1.f);
  const float x = sqrtf(x2);
  float s, c;
  sincospif(x * 0.318309886f, &s, &c);  // argument reduction exact in units of pi
  return 3.f * (s - x * c) / (x * x2);
}

// MODEL: 1 the Newtonian potential (chameleon-type screening); 2 the density
// smoothed by the Gaussian window; 3 the density smoothed by the top-hat or
// sharp-k window (fp.filter).  The Gaussian keeps a kernel of its own: a
// per-element switch over the windows slows the pass by a third.
template <int N, int TW, int MODEL, int T>
struct OpZScreenField {
  static constexpr bool kTwReady = true;
  // Between the forward and the inverse transform: delta(k) out to HBM (chameleon-type
  // models: the force pass needs it; the Vainshtein source carries its delta), the
  // field's multiplier (-kappa/k^2, or the smoothing window) applied.
  struct Field {
    float2* dk;  // delta(k) of the tile: element (n, c) at dk[(n / HQ) ra + (n mod HQ) rb + hcol(c)]
    int64_t ra, rb;
    int c0, fy2;
    float kf2, kappa_norm, R2half, norm;
    int filter;
    __device__ __forceinline__ float2 operator()(float2 v, int n, int c, int) const {
      if (MODEL == 1 && c0 + c < N / 2 + 1) dk[(n / HQ) * ra + (n % HQ) * rb + hcol(c)] = v;
      const int fx = c0 + c, fz = freq_index(n, N);
      const float k2 = kf2 * (float)(fx * fx + fy2 + fz * fz);
      float m = 0.f;
      if (k2 > 0.f) {
        if (MODEL == 1) m = __fdividef(-kappa_norm, k2);
        else if (MODEL == 2) m = __expf(-k2 * R2half) * norm;
        else m = smoothing_window(k2 * R2half, filter) * norm;
      }
      return cscale(v, m);
    }
  };
  ColGeo<N, TW> geo;
  const float2* in;
  float2 *dk_out, *w_out;
  ForceParams fp;
  float2* extra = nullptr;  // scratch after the stage buffers (set by col_pipeline)
  static constexpr bool kSide = false;
  __device__ __forceinline__ void issue(float2* buf, int64_t t) const {
    int o, c0;
    int64_t base, by;
    geo.tile(t, o, c0, base, by);
    col_issue<N, TW, TW, T>(buf, 0, moved(in, by), base, geo.ra, geo.rb, c0);
  }
  __device__ __forceinline__ void process(float2* buf, const float2* tw, int64_t t) const {
    int iy, c0;
    int64_t base, by;
    geo.tile(t, iy, c0, base, by);
    ForceParams fp = this->fp;
    resolve(fp, by);
    const int fy = freq_index(iy, N);
    const Field f{moved(dk_out, by) + base, geo.ra, geo.rb, c0, fy * fy, fp.kf * fp.kf, fp.kappa_norm,
                  fp.R2half, fp.norm, fp.filter};
    fft_tile_fwd_inv<N, TW, TW, T>(buf, tw, f, ColOut{moved(w_out, by) + base, geo.ra, geo.rb, N / 2 + 1 - c0});
  }
};

template <int N, int TW, int MODEL, bool TMA, int T>
__global__ void __launch_bounds__(T, zblocks(N)) k_z_screen_field(OpZScreenField<N, TW, MODEL, T> op,
                                                       const float2* __restrict__ twg,
                                                       int64_t ntiles, const __grid_constant__ CUtensorMap map) {
  pdl_begin<T>(twg, N);
  if (!op.geo.m.shift) resolve(op.fp, 0);  // one simulation: once per launch
  if constexpr (TMA) col_pipeline_tma<N, fft_rows<N>() * TW, false, 0, T>(op, twg, ntiles, &map, nullptr);
  else col_pipeline<N, fft_rows<N>() * TW, T>(op, twg, ntiles);
}

// ---------------------------------------------------------------- force (z pass)
// Per tile: the source (S, or delta when unscreened) is staged and transformed
// forward while delta(k) lands in a second shared-memory tile (screened runs);
// Phi_tot(k) is formed from both in registers, and the inverse transforms of Phi
// and of -i kz Phi start from there.  The next tile's delta(k) is on its way while
// they run.
template <int N, int TW>
constexpr size_t zforce_smem() {  // twiddles, two stage buffers, delta(k)
  return col_smem_tw(N, TW) + (size_t)N * TW * sizeof(float2);
}
template <int N, int TW, bool SCREENED, int T>
struct OpZForce {
  static constexpr bool kTwReady = true;
  // Phi_tot(k) (App. B) from the transform of S and delta(k) in `dk`; ready() waits for
  // this tile's delta(k) between the forward transform's steps.
  struct Combine {
    const float2* dk;
    int c0, fy2;
    float kf2, a2m2, kappa_norm, C;
    __device__ __forceinline__ float2 operator()(float2 src, int n, int c, int at) const {
      const int fx = c0 + c, fz = freq_index(n, N);
      const float k2 = kf2 * (float)(fx * fx + fy2 + fz * fz);
      float2 phi = make_float2(0.f, 0.f);
      if (k2 > 0.f) {
        const float yuk = __fdividef(k2, k2 + a2m2);
        const float g = __fdividef(-kappa_norm, k2);
        if (SCREENED) phi = cscale(cadd(dk[at], cscale(src, C * yuk)), g);
        else phi = cscale(src, g * (1.f + C * yuk));
      }
      return phi;
    }
    TmaSide side;  // TMA staging: the barrier of delta(k)'s copy
    __device__ __forceinline__ void ready() const {
      if (!SCREENED) return;
      if (side.bar) side.wait();  // thread 0; the transform's next barrier publishes the tile
      else cp_async_wait<1>();    // delta(k); the next tile's prefetch may stay in flight
    }
  };
  // -i kz Phi_tot(k), zero on the Nyquist row.
  struct GradZ {
    float mkf;
    __device__ __forceinline__ float2 operator()(float2 phi, int n) const {
      const float kzs = (n == N / 2) ? 0.f : mkf * (float)freq_index(n, N);
      return cscale(cmul_i(phi), kzs);
    }
  };
  ColGeo<N, TW> geo;
  const float2 *in, *dk;
  float2 *phi_out, *phiz_out;
  ForceParams fp;
  float2* extra = nullptr;  // scratch after the stage buffers (set by col_pipeline)
  TmaSide side;             // set per tile by col_pipeline_tma
  __device__ __forceinline__ void issue(float2* buf, int64_t t) const {
    int o, c0;
    int64_t base, by;
    geo.tile(t, o, c0, base, by);
    col_issue<N, TW, TW, T>(buf, 0, moved(in, by), base, geo.ra, geo.rb, c0);
  }
  static constexpr bool kSide = true;
  // delta(k) of the tile into extra; lands while S is transformed
  __device__ __forceinline__ void issue_side(int64_t t) const {
    if (SCREENED) {
      int o, c0;
      int64_t base, by;
      geo.tile(t, o, c0, base, by);
      col_issue<N, TW, TW, T>(extra, 0, moved(dk, by), base, geo.ra, geo.rb, c0);
    }
  }
  template <class Next>
  __device__ __forceinline__ void process(float2* buf, const float2* tw, int64_t t, Next next) const {
    int iy, c0;
    int64_t base, by;
    geo.tile(t, iy, c0, base, by);
    ForceParams fp = this->fp;
    resolve(fp, by);
    const int fy = freq_index(iy, N);
    // a Vainshtein source already holds its fifth force (screen_source)
    const float C = !SCREENED && fp.screened ? 0.f : fp.C;
    const Combine cmb{extra, c0, fy * fy, fp.kf * fp.kf, fp.a2m2, fp.kappa_norm, C, side};
    const ColOut op{moved(phi_out, by) + base, geo.ra, geo.rb, N / 2 + 1 - c0};
    const ColOut oz{moved(phiz_out, by) + base, geo.ra, geo.rb, N / 2 + 1 - c0};
    fft_tile_fwd_inv2<N, TW, TW, T>(buf, tw, cmb, GradZ{-fp.kf}, next, op, oz);
  }
};

template <int N, int TW, bool SCREENED, bool TMA, int T>
__global__ void __launch_bounds__(T, zblocks(N)) k_z_force(
    OpZForce<N, TW, SCREENED, T> op, const float2* __restrict__ twg, int64_t ntiles,
    const __grid_constant__ CUtensorMap map, const __grid_constant__ CUtensorMap dmap) {
  pdl_begin<T>(twg, N);
  if (!op.geo.m.shift) resolve(op.fp, 0);  // one simulation: once per launch
  if constexpr (TMA) col_pipeline_tma<N, fft_rows<N>() * TW, SCREENED, N * TW, T>(op, twg, ntiles, &map, &dmap);
  else col_pipeline<N, fft_rows<N>() * TW, T>(op, twg, ntiles);
}

// ---------------------------------------------------------------- LPT reweight (z pass)
template <int PREC>
__device__ __forceinline__ float2 dequant(uint32_t w, float scale) {
  float re, im;
  if constexpr (PREC == 1) {
    re = __uint_as_float(w << 16);
    im = __uint_as_float(w & 0xFFFF0000u);
  } else {
    re = __half2float(__ushort_as_half((unsigned short)(w & 0xFFFFu)));
    im = __half2float(__ushort_as_half((unsigned short)(w >> 16)));
  }
  return make_float2(re * scale, im * scale);
}

template <int N, int TW, int PREC>
struct OpLptZ {
  static constexpr bool kTwReady = true;
  ColGeo<N, TW> geo;
  const void *phi1, *phi2;
  float2 *o0, *o1, *o2, *o3;
  LptParams lp;
  int tab_smem;             // 1: the (single) table row is staged in extra once per CTA
  // zero fill riding on this issue-bound pass: each tile clears its share (zchunk bytes)
  // of zdst (zbytes per simulation, moved by the simulation's shift), by bulk stores
  // from a zeroed 16 KB region after the table row; nullptr: none
  char* zdst = nullptr;
  int64_t zbytes = 0, zchunk = 0;
  float2* extra = nullptr;  // scratch after the stage buffers (set by col_pipeline)
  static constexpr uint32_t kZero = 16384;
  static constexpr bool kSide = false;
  __device__ __forceinline__ void issue(float2* buf, int64_t t) const {
    int o, c0;
    int64_t base, by;
    geo.tile(t, o, c0, base, by);
    if constexpr (PREC == 0) {
      col_issue<N, TW, 4 * TW>(buf, 0, moved(static_cast<const float2*>(phi1), by), base, geo.ra, geo.rb, c0);
      col_issue<N, TW, 4 * TW>(buf, 1, moved(static_cast<const float2*>(phi2), by), base, geo.ra, geo.rb, c0);
    } else {
      // raw 16-bit pairs staged in the (still unused) output sub-blocks 2 and 3
      uint32_t* rb = reinterpret_cast<uint32_t*>(buf);
      col_issue_raw<N, TW>(rb, 0, moved(static_cast<const uint32_t*>(phi1), by), base, geo.ra, geo.rb, c0);
      col_issue_raw<N, TW>(rb, 1, moved(static_cast<const uint32_t*>(phi2), by), base, geo.ra, geo.rb, c0);
    }
  }
  __device__ __forceinline__ void process(float2* buf, const float2* tw, int64_t t) const {
    constexpr int TP = 4 * TW;
    int iy, c0;
    int64_t base, by;
    geo.tile(t, iy, c0, base, by);
    LptParams lp = this->lp;
    resolve(lp, by);  // no-op when resolved once for the launch
    const float4* tab = lp.row;
    if (tab_smem) {
      float4* st = reinterpret_cast<float4*>(extra);
      if (t == blockIdx.x) {  // this CTA's first tile: stage the row
        for (int i = threadIdx.x; i < lp.nk; i += NT) st[i] = tab[i];
        __syncthreads();
      }
      tab = st;
    }
    if (zdst) {
      float4* zr = reinterpret_cast<float4*>(extra) + (tab_smem ? lp.nk : 0);
      if (t == blockIdx.x) {  // first tile: zero the region for the async proxy
        for (int i = threadIdx.x; i < (int)(kZero / 16); i += NT) zr[i] = make_float4(0.f, 0.f, 0.f, 0.f);
        fence_async_smem();
        __syncthreads();
      }
      if (threadIdx.x == 0) {
        const int64_t tps = ColGeo<N, TW>::tps, tl = t % tps;
        const int64_t a = tl * zchunk, b = a + zchunk < zbytes ? a + zchunk : zbytes;
        if (a < b) bulk_zero(moved(zdst, by) + a, b - a, zr, kZero);
      }
    }
    if constexpr (PREC != 0) {
      const uint32_t* rb = reinterpret_cast<const uint32_t*>(buf);
      const float sc1 = lp.scale[0], sc2 = lp.scale[1];
      for (int e = threadIdx.x; e < N * TW; e += NT) {
        const int c = e % TW, n = e / TW;
        const float2 a = dequant<PREC>(rb[8 * n * TW + 4 * TW + c], sc1);
        const float2 b = dequant<PREC>(rb[8 * n * TW + 5 * TW + c], sc2);
        buf[n * TP + c] = a;
        buf[n * TP + TW + c] = b;
      }
      __syncthreads();  // the raw staging (sub-blocks 2, 3) is consumed
    }
    const TileLane<N, TW> ln(c0, iy);
    const float kf2 = lp.kf * lp.kf;
    const int c = ln.c;
#pragma unroll 2
    for (int i = 0; i < ln.E; ++i) {
      const int n = ln.row(i);
      const float k2 = ln.k2(n, kf2);
      float2 d = make_float2(0.f, 0.f), A = make_float2(0.f, 0.f);
      if (k2 > 0.f) {
        const float u = (0.5f * __logf(k2) - lp.lnk0) * lp.inv_dlnk;
        int i0 = (int)floorf(u);
        i0 = min(max(i0, 0), lp.nk - 2);
        const float f = u - (float)i0;
        const float4 t0 = tab[i0], t1 = tab[i0 + 1];
        const float c1 = t0.x * (1.f - f) + t1.x * f;
        const float c2 = t0.y * (1.f - f) + t1.y * f;
        const float e1 = t0.z * (1.f - f) + t1.z * f;
        const float e2 = t0.w * (1.f - f) + t1.w * f;
        const float2 p1 = buf[n * TP + c], p2 = buf[n * TP + TW + c];
        d = cscale(cadd(cscale(p1, c1), cscale(p2, c2)), lp.norm);
        A = cscale(cadd(cscale(p1, e1), cscale(p2, e2)), lp.norm);
      }
      const float kz = (n == N / 2) ? 0.f : lp.kf * (float)freq_index(n, N);
      buf[n * TP + c] = d;
      buf[n * TP + TW + c] = cscale(cmul_i(d), kz);
      buf[n * TP + 2 * TW + c] = A;
      buf[n * TP + 3 * TW + c] = cscale(cmul_i(A), kz);
    }
    __syncthreads();
    fft_tile<N, TP, TP, NT, true>(buf, tw);
    col_store<N, TW, TP>(buf, 0, moved(o0, by), base, geo.ra, geo.rb, c0);
    col_store<N, TW, TP>(buf, 1, moved(o1, by), base, geo.ra, geo.rb, c0);
    col_store<N, TW, TP>(buf, 2, moved(o2, by), base, geo.ra, geo.rb, c0);
    col_store<N, TW, TP>(buf, 3, moved(o3, by), base, geo.ra, geo.rb, c0);
  }
};

template <int N, int TW, int PREC>
__global__ void __launch_bounds__(NT, blocks_for_smem(col_smem_c(N, 4), N)) k_lpt_z(OpLptZ<N, TW, PREC> op,
                                              const float2* __restrict__ twg, int64_t ntiles) {
  pdl_begin<NT>(twg, N);
  if (!op.geo.m.shift) resolve(op.lp, 0);  // one simulation: once per launch
  col_pipeline<N, fft_rows<N>() * 4 * TW>(op, twg, ntiles);
  if (op.zdst && threadIdx.x == 0) bulk_store_drain();  // the zero fill completes with the kernel
}

// The LPT z pass for 16-bit seeds with 8-column tiles (N = 256, 512), where four 4-column
// output arrays would otherwise fill shared memory: an 8-column tile reads and
// writes whole chunks of the interleaved layout (4-column tiles move halves of
// them).  Shared memory: two input buffers of raw seeds (phi1 words 0..7, phi2 words
// 8..15 of each 32-word row; double-buffered) and one work buffer that first holds
// (d, i kz d) and then (A, i kz A), formed from the dequantised seeds, each pair inverse
// transformed as one 16-column tile whose outputs leave for HBM from the last
// step's registers.  The table row is read through L1.
template <int N>
struct LptZ8 {
  static constexpr int TW = 8, TP = 16, ROWS = fft_rows<N>(), BUF = ROWS * TP;
  static constexpr size_t smem = (N + 3 * (size_t)BUF) * sizeof(float2);
};

// Store hook: columns c < 8 to ga, 8..15 to gb (columns c0 + c < N/2 + 1 exist).
struct PairColOut {
  static constexpr bool kSmem = false;
  float2 *ga, *gb;
  int64_t ra, rb;
  int live;
  __device__ __forceinline__ float2 operator()(float2 v, int n, int c, int) const {
    const bool b = c >= 8;
    const int cc = b ? c - 8 : c;
    if (cc < live) (b ? gb : ga)[(n / HQ) * ra + (n % HQ) * rb + hcol(cc)] = v;
    return v;
  }
};

// 16-bit seeds of one field, raw, into words f*8 .. f*8+7 of each 32-word staged row.
template <int N>
__device__ __forceinline__ void col_issue_raw8(uint32_t* sb, int f, const uint32_t* __restrict__ g, int64_t base,
                                               int64_t ra, int64_t rb, int c0) {
  constexpr int STEP = NT / 2;  // two 16-byte pieces (8 words) per row and field
  const int j = threadIdx.x & 1, n0 = threadIdx.x >> 1;
  const bool v = c0 + 4 * j < N / 2 + 1;
  const uint32_t* src = g + base + (n0 / HQ) * ra + (n0 % HQ) * rb + hcol(4 * j);
  uint32_t* dst = sb + n0 * 32 + f * 8 + 4 * j;
#pragma unroll 4
  for (int n = n0; n < N; n += STEP) {
    cp_async16(dst, v ? (const void*)src : (const void*)g, v);
    src += (STEP / HQ) * ra;
    dst += STEP * 32;
  }
}

template <int N, int PREC>
__global__ void __launch_bounds__(NT, 1) k_lpt_z8(ColGeo<N, 8> geo, const uint32_t* __restrict__ phi1,
                                                   const uint32_t* __restrict__ phi2, float2* __restrict__ o0,
                                                   float2* __restrict__ o1, float2* __restrict__ o2,
                                                   float2* __restrict__ o3, LptParams lp0,
                                                   const float2* __restrict__ twg, int64_t ntiles) {
  static_assert(PREC == 1 || PREC == 2, "16-bit seeds");
  using C = LptZ8<N>;
  extern __shared__ __align__(128) float2 sm[];
  float2* tw = sm;
  float2* const S0 = sm + N;
  float2* const S1 = sm + N + C::BUF;
  float2* const W = sm + N + 2 * C::BUF;
  load_tw(tw, twg, N);
  auto issue = [&](float2* buf, int64_t t) {
    int o, c0;
    int64_t base, by;
    geo.tile(t, o, c0, base, by);
    uint32_t* sb = reinterpret_cast<uint32_t*>(buf);
    col_issue_raw8<N>(sb, 0, moved(phi1, by), base, geo.ra, geo.rb, c0);
    col_issue_raw8<N>(sb, 1, moved(phi2, by), base, geo.ra, geo.rb, c0);
  };
  if (!geo.m.shift) resolve(lp0, 0);  // one simulation: once per launch
  int64_t t = blockIdx.x;
  if (t < ntiles) issue(S0, t);
  cp_async_commit();
  int cur = 0;
  for (; t < ntiles; t += gridDim.x) {
    const int64_t tn = t + gridDim.x;
    if (tn < ntiles) issue(cur ? S0 : S1, tn);
    cp_async_commit();
    cp_async_wait<1>();  // tile t's seeds have landed
    __syncthreads();
    int iy, c0;
    int64_t base, by;
    geo.tile(t, iy, c0, base, by);
    LptParams lp = lp0;
    resolve(lp, by);
    const float4* __restrict__ tab = lp.row;
    const uint32_t* sb = reinterpret_cast<const uint32_t*>(cur ? S1 : S0);
    const TileLane<N, 8> ln(c0, iy);
    const float kf2 = lp.kf * lp.kf;
    const int c = ln.c;
    // pass 0: (d, i kz d) with (c1, c2); pass 1: (A, i kz A) with (e1, e2)
#pragma unroll 1
    for (int pass = 0; pass < 2; ++pass) {
#pragma unroll 2
      for (int i = 0; i < ln.E; ++i) {
        const int n = ln.row(i);
        const float k2 = ln.k2(n, kf2);
        float2 v = make_float2(0.f, 0.f);
        if (k2 > 0.f) {
          const float u = (0.5f * __logf(k2) - lp.lnk0) * lp.inv_dlnk;
          int i0 = (int)floorf(u);
          i0 = min(max(i0, 0), lp.nk - 2);
          const float f = u - (float)i0;
          const float4 t0 = __ldg(tab + i0), t1 = __ldg(tab + i0 + 1);
          const float a = pass == 0 ? t0.x * (1.f - f) + t1.x * f : t0.z * (1.f - f) + t1.z * f;
          const float b = pass == 0 ? t0.y * (1.f - f) + t1.y * f : t0.w * (1.f - f) + t1.w * f;
          const float2 p1 = dequant<PREC>(sb[n * 32 + c], lp.scale[0]);
          const float2 p2 = dequant<PREC>(sb[n * 32 + 8 + c], lp.scale[1]);
          v = cscale(cadd(cscale(p1, a), cscale(p2, b)), lp.norm);
        }
        const float kz = (n == N / 2) ? 0.f : lp.kf * (float)freq_index(n, N);
        W[n * 16 + c] = v;
        W[n * 16 + 8 + c] = cscale(cmul_i(v), kz);
      }
      __syncthreads();
      const PairColOut out{moved(pass == 0 ? o0 : o2, by) + base, moved(pass == 0 ? o1 : o3, by) + base, geo.ra,
                           geo.rb, N / 2 + 1 - c0};
      fft_tile_call<N, 16, 16, NT, true, 1, TileLoad, PairColOut>(W, tw, TileLoad{}, out);
    }
    cur ^= 1;
  }
  cp_async_wait<0>();
}

// The LPT z pass for FP32 seeds up to 256 points: small CTAs as in the other z passes.  A
// thread reads the seeds of its first-step items, forms d = c1 phi1 + c2 phi2 and A = e1
// phi1 + e2 phi2 (one table lookup per mode for all four coefficients) and keeps them in
// registers; the four outputs d, i kz d, A, i kz A are then transformed one after the other
// through one tile buffer.  Three buffers rotate: the two seed tiles, whose room is free once
// they are in registers, and one more, so that the next tile's seeds land meanwhile.
// Against two- and four-array tiles of 256 threads: 142 -> 104 us at
// 256^3, 718 -> 488 us over 256 lattices of 64^3.  A launch of few tiles (one lattice of 64^3
// or 128^3) is bound by the length of one tile's chain instead and keeps k_lpt_z (10.5 and
// 24.8 us against 11.1 and 26.8).  Both forms give the same bits, so a lattice's fields
// do not depend on how many others share its launch: a product that k_lpt_z leaves in shared
// memory is rounded on its own here too (cmul_if).
template <int N>
struct LptZr {
  static constexpr int TW = ztw(N), T = 128, BUF = fft_rows<N>() * TW;
  static constexpr size_t smem = (N + 3 * (size_t)BUF) * sizeof(float2);
};

template <int N>
__global__ void __launch_bounds__(128, 4) k_lpt_zr(ColGeo<N, LptZr<N>::TW> geo, const float2* __restrict__ phi1,
                                                   const float2* __restrict__ phi2, float2* __restrict__ o0,
                                                   float2* __restrict__ o1, float2* __restrict__ o2,
                                                   float2* __restrict__ o3, LptParams lp0,
                                                   const float2* __restrict__ twg, int64_t ntiles) {
  using C = LptZr<N>;
  constexpr int TW = C::TW, T = C::T, R1 = Split<N>::R1, R2 = Split<N>::R2;
  constexpr int U = TW * R2, P = (U + T - 1) / T;
  extern __shared__ __align__(128) float2 sm[];
  float2* tw = sm;
  float2 *X = sm + N, *Y = X + C::BUF, *Z = Y + C::BUF;
  pdl_begin<T>(twg, N);
  auto issue = [&](float2* a, float2* b, int64_t t) {
    int o, c0;
    int64_t base, by;
    geo.tile(t, o, c0, base, by);
    col_issue<N, TW, TW, T>(a, 0, moved(phi1, by), base, geo.ra, geo.rb, c0);
    col_issue<N, TW, TW, T>(b, 0, moved(phi2, by), base, geo.ra, geo.rb, c0);
  };
  if (!geo.m.shift) resolve(lp0, 0);  // one simulation: once per launch
  int64_t t = blockIdx.x;
  if (t < ntiles) issue(X, Y, t);
  cp_async_commit();
  for (; t < ntiles; t += gridDim.x) {
    cp_async_wait<0>();
    __syncthreads();  // tile t's seeds have landed
    int iy, c0;
    int64_t base, by;
    geo.tile(t, iy, c0, base, by);
    LptParams lp = lp0;
    resolve(lp, by);
    const float4* __restrict__ tab = lp.row;
    const float kf2 = lp.kf * lp.kf;
    const int fy = freq_index(iy, N);
    float2 d[P][R1], A[P][R1];
#pragma unroll
    for (int i = 0; i < P; ++i) {
      const int u = threadIdx.x + i * T;
      if ((U % T) == 0 || u < U) {
        const int c = u % TW, n2 = u / TW, fx = c0 + c;
#pragma unroll
        for (int n1 = 0; n1 < R1; ++n1) {
          const int n = R2 * n1 + n2, fz = freq_index(n, N);
          const float k2 = kf2 * (float)(fx * fx + fy * fy + fz * fz);
          d[i][n1] = A[i][n1] = make_float2(0.f, 0.f);
          if (k2 > 0.f) {
            const float uu = (0.5f * __logf(k2) - lp.lnk0) * lp.inv_dlnk;
            const int i0 = min(max((int)floorf(uu), 0), lp.nk - 2);
            const float f = uu - (float)i0;
            const float4 t0 = __ldg(tab + i0), t1 = __ldg(tab + i0 + 1);
            const float2 p1 = X[n * TW + c], p2 = Y[n * TW + c];
            d[i][n1] = cscale(cadd(cscale(p1, t0.x * (1.f - f) + t1.x * f), cscale(p2, t0.y * (1.f - f) + t1.y * f)),
                              lp.norm);
            A[i][n1] = cscale(cadd(cscale(p1, t0.z * (1.f - f) + t1.z * f), cscale(p2, t0.w * (1.f - f) + t1.w * f)),
                              lp.norm);
          }
        }
      }
    }
    __syncthreads();  // every thread has its seeds
    if (t + gridDim.x < ntiles) issue(Y, Z, t + gridDim.x);
    else pdl_go();  // the CTA's last tile
    cp_async_commit();
    auto emit = [&](const float2 (&src)[P][R1], bool deriv, float2* out) {
#pragma unroll
      for (int i = 0; i < P; ++i) {
        const int u = threadIdx.x + i * T;
        if ((U % T) == 0 || u < U) {
          const int c = u % TW, n2 = u / TW;
          float2 v[R1];
#pragma unroll
          for (int n1 = 0; n1 < R1; ++n1) {
            const int n = R2 * n1 + n2;
            const float kz = (n == N / 2) ? 0.f : lp.kf * (float)freq_index(n, N);
            v[pos_of<R1>(n1)] = deriv ? cmul_if(src[i][n1], kz) : src[i][n1];
          }
          dftR<R1, true>(v);
          float2* y = X + n2 * (R1 + 1) * TW + c;
          y[0] = v[0];
#pragma unroll
          for (int k1 = 1; k1 < R1; ++k1) y[k1 * TW] = n2 > 0 ? cmul_conj(v[k1], tw[n2 * k1]) : v[k1];
        }
      }
      __syncthreads();
      col_inv2<R1, R2, TW, TW, T>(X, ColOut{moved(out, by) + base, geo.ra, geo.rb, N / 2 + 1 - c0});
    };
    emit(d, false, o0);
    __syncthreads();
    emit(d, true, o1);
    __syncthreads();
    emit(A, false, o2);
    __syncthreads();
    emit(A, true, o3);
    float2* x = X;
    X = Y;
    Y = Z;
    Z = x;
  }
  cp_async_wait<0>();
}

// ---------------------------------------------------------------- x passes (rows)
// A row tile holds TWX rows of the half-length complex transform (M = N/2)
// row-major in shared memory, row r at st[r * CW + k] (CW = rowtile_pitch<M>),
// exactly as cp.async staged them; the transform runs in place
// (fft_rowtile).  Tiles are double-buffered: the next tile is staged into the
// other buffer while the current one is transformed.
template <int N, int TWX>
struct RowCfg {
  static constexpr int M = N / 2;
  static constexpr int CW = rowtile_pitch<M>();    // complex values per staged row (>= M + 2)
  static constexpr size_t stage = (size_t)TWX * CW;  // float2 per buffer
  static constexpr size_t smem = (N + 2 * stage) * sizeof(float2);
};

// The rows of a row tile (first group-major row q0, HQ | TWX) are the rows (z, y) ..
// (z + HQ - 1, y) of TWX/HQ consecutive y: in the half spectrum one contiguous block
// of TWX/HQ interleaved row groups (HQ P complex values each), in real space HQ
// blocks of TWX/HQ consecutive rows, one per plane, N rows apart (the first from
// real row real_row_q(q0)).  Tile row r (plane r mod HQ, y r / HQ) is staged at
// st[r * CW ...].
//
// Walk over the NG row groups of a tile in memory order, LEN positions per
// group: warps take whole groups, or split each group into NW / NG segments
// when there are fewer groups than warps; f(group, p0, p1) visits p = p0, p0 +
// 32, ... < p1 with p0 = segment start + lane (segment starts are multiples of
// 32, so each warp reads or writes whole lines).
template <int T, int NG, int LEN, class F>
__device__ __forceinline__ void for_groups(F f) {
  constexpr int NW = T / 32;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if constexpr (NG >= NW) {
    for (int g = warp; g < NG; g += NW) f(g, lane, LEN);
  } else {
    constexpr int S = NW / NG;
    constexpr int SEG = (LEN + 32 * S - 1) / (32 * S) * 32;
    const int s = warp % S;
    f(warp / S, s * SEG + lane, (s + 1) * SEG < LEN ? (s + 1) * SEG : LEN);
  }
}

// 16-byte piece p of a row group holds values 2 (p mod 4), + 1 of chunk p / (4 HQ) of
// row (p / 4) mod HQ; piece p + 32 is the same row, columns + KSTEP.
constexpr int KSTEP = 64 / HQ;
static_assert(32 % (4 * HQ) == 0 && KSTEP * HQ == 64, "32 pieces are whole chunk groups");
__device__ __forceinline__ int piece_col(int p) { return p / (4 * HQ) * 8 + 2 * (p & 3); }
__device__ __forceinline__ int piece_row(int p) { return (p >> 2) % HQ; }

// Complex half rows (M + 1 values, staged as M + 2 to keep 16-byte pieces).
template <int N, int TWX, int T>
__device__ __forceinline__ void stage_complex_rows(float2* st, const float2* __restrict__ in,
                                                   int64_t q0) {
  using C = RowCfg<N, TWX>;
  constexpr int P = (int)half_pitch(N), LEN = HQ * P / 2;  // 16-byte pieces per row group
  const float2* src = in + hrow_q(q0, P);
  for_groups<T, TWX / HQ, LEN>([&](int gr, int p0, int p1) {
    int k = piece_col(p0);
    float2* d = st + (HQ * gr + piece_row(p0)) * C::CW + k;
    const float2* g = src + (int64_t)gr * HQ * P + 2 * p0;
    for (int p = p0; p < p1; p += 32, k += KSTEP, d += KSTEP, g += 64)
      if (k < C::M + 2) cp_async16(d, g, true);
  });
}

// A pair tile: TWX/2 rows of a and the same rows of b (first group-major row q0), row
// group i of a at tile rows 2 HQ i + 2 j (plane j), of b at 2 HQ i + 2 j + 1, so that
// tile rows 2w and 2w + 1 are the same real row of a and of b.
template <int N, int TWX, int T>
__device__ __forceinline__ void stage_complex_rows_pair(float2* st, const float2* __restrict__ a,
                                                        const float2* __restrict__ b, int64_t q0) {
  using C = RowCfg<N, TWX>;
  static_assert(TWX % (2 * HQ) == 0, "whole row groups of a and b");
  constexpr int P = (int)half_pitch(N), LEN = HQ * P / 2;
  const float2* srca = a + hrow_q(q0, P);
  const float2* srcb = b + hrow_q(q0, P);
  for_groups<T, TWX / HQ, LEN>([&](int gr, int p0, int p1) {
    const int job = gr & 1, i = gr >> 1;
    int k = piece_col(p0);
    float2* d = st + (2 * HQ * i + 2 * piece_row(p0) + job) * C::CW + k;
    const float2* g = (job ? srcb : srca) + (int64_t)i * HQ * P + 2 * p0;
    for (int p = p0; p < p1; p += 32, k += KSTEP, d += KSTEP, g += 64)
      if (k < C::M + 2) cp_async16(d, g, true);
  });
}

// real rows of N floats: row r at floats [pitch r, pitch r + N), i.e. the M
// complex values z[j] = x[2j] + i x[2j+1] at st[r * CW + j] when pitch = 2 CW
template <int N, int TWX, int T>
__device__ __forceinline__ void stage_real_rows(float* st, const float* __restrict__ in, int64_t q0,
                                                int pitch_floats) {
  constexpr int CH = N / 4;             // 16-byte pieces per row
  constexpr int BLK = TWX / HQ * CH;    // pieces per plane
  const float* src = in + real_row_q(q0, N) * N;
  if constexpr (BLK % T == 0) {
#pragma unroll
    for (int i = 0; i < HQ * BLK / T; ++i) {
      const int h = i * T / BLK;  // plane, constant per iteration
      const int e = threadIdx.x + i * T - h * BLK;
      cp_async16(st + (HQ * (e / CH) + h) * pitch_floats + 4 * (e % CH), src + (int64_t)h * N * N + 4 * e, true);
    }
  } else {
    for (int i = threadIdx.x; i < HQ * BLK; i += T) {
      const int h = i / BLK, e = i - h * BLK;
      cp_async16(st + (HQ * (e / CH) + h) * pitch_floats + 4 * (e % CH), src + (int64_t)h * N * N + 4 * e, true);
    }
  }
}

// A warp stages its own RW = TWX 32 / T rows (RowMap), so a row pass needs no barrier
// of the CTA: 16-byte pieces of R rows of one group, 64 R / HQ-th parts of it,
// R = min(RW, HQ); lane l takes piece l of each run of 32, which covers 8 / R chunks.
template <int N, int CW, int R, int RSTEP>
__device__ __forceinline__ void stage_group_rows(float2* st, const float2* __restrict__ g) {
  // rows j = 0 .. R - 1 of the group part at g, row j at st + j RSTEP CW
  static_assert(8 % R == 0, "whole chunks per 32 pieces");
  const int lane = threadIdx.x & 31, j = (lane >> 2) % R;
  int k = lane / (4 * R) * 8 + 2 * (lane & 3);
  const float2* src = g + lane / (4 * R) * (8 * HQ) + j * 8 + 2 * (lane & 3);
  float2* d = st + j * RSTEP * CW + k;
#pragma unroll 4
  for (; k < N / 2 + 2; k += 64 / R, d += 64 / R, src += 8 / R * (8 * HQ)) cp_async16(d, src, true);
}

template <int N, int TWX, int T>
__device__ __forceinline__ void stage_complex_rows_warp(float2* st, const float2* __restrict__ in,
                                                   int64_t q0) {
  using C = RowCfg<N, TWX>;
  constexpr int P = (int)half_pitch(N), RW = TWX * 32 / T, R = RW < HQ ? RW : HQ;
  const int c0 = (threadIdx.x >> 5) * RW;
#pragma unroll
  for (int b = 0; b < RW; b += R)
    stage_group_rows<N, C::CW, R, 1>(st + (c0 + b) * C::CW, in + hrow_q(q0 + c0 + b, P));
}

// Real row of tile row r relative to the tile's first: plane r mod HQ, y r / HQ.
template <int N>
__device__ __forceinline__ int tile_real_row(int r) {
  return (r % HQ) * N + r / HQ;
}

// Store hook of the forward row transforms (fft_rowtile_r2c): X[k] of tile row r into
// the interleaved half spectrum, g = the tile's first row group.  A warp holds 16 (or
// fewer) consecutive k of adjacent tile rows: whole 64-byte chunks of adjacent planes.
template <int P>
struct HalfRowOut {
  static constexpr bool kSmem = false;
  float2* g;
  __device__ __forceinline__ float2 operator()(float2 v, int r, int k) const {
    g[(r / HQ) * HQ * P + (r % HQ) * 8 + (k >> 3) * (8 * HQ) + (k & 7)] = v;
    return v;
  }
};

// The c2r input convention on a staged spectrum value X[k] (k = 0..M): the
// optional derivative i kfs k (zero at the Nyquist k = M), and the imaginary
// parts of X[0], X[M] dropped.
template <int M>
__device__ __forceinline__ float2 c2r_in(float2 x, int k, float kfs) {
  if (kfs != 0.f) x = (k == M) ? make_float2(0.f, 0.f) : cscale(cmul_i(x), kfs * (float)k);
  if (k == 0 || k == M) x.y = 0.f;
  return x;
}

// c2r pre-processing (unnormalised inverse, 2x folded in) as the first step of
// the inverse row transform loads element n of tile row r: with E = X[n] +
// conj X[M-n] and O = w^-n (X[n] - conj X[M-n]), Z[n] = E + i O.  The partner
// M - n is read from the staged row itself, which no thread overwrites before
// every load of that step is done (no separate pass over the tile).  Pitch CW.
template <int N, int CW>
struct C2rCombine {
  const float2* buf;
  const float2* tw;
  float kfs;
  __device__ __forceinline__ float2 operator()(float2 zn, int r, int n) const {
    constexpr int M = N / 2;
    const float2 a = c2r_in<M>(zn, n, kfs);
    const float2 b = cconj(c2r_in<M>(buf[r * CW + M - n], M - n, kfs));
    const float2 E = cadd(a, b);
    const float2 O = cmul(cconj(tw[n]), csub(a, b));
    return cadd(E, cmul_i(O));
  }
};

struct ScaleOffset {
  float scale, offset;
  __device__ __forceinline__ float2 operator()(float2 v, int, int) const {
    return make_float2(fmaf(v.x, scale, offset), fmaf(v.y, scale, offset));
  }
};

// Row tile t of a multi-simulation launch: simulation t / tps, first row (t mod tps) TWX
// in the group-major row order q of the half-spectrum layout (HQ | TWX).
struct RowTile {
  int64_t row0, by;
};
template <int N, int TWX>
__device__ __forceinline__ RowTile row_tile(int64_t t64, const Multi& m) {
  constexpr uint32_t TPS = (uint32_t)N * N / TWX;  // tiles per simulation
  const uint32_t t = (uint32_t)t64, b = t / TPS;     // t < 2^31 (checked by prep)
  return RowTile{(int64_t)(t - b * TPS) * TWX, shift_of(m, (int)b)};
}

// The real rows of row tile q0 into st by 1-D bulk copies (thread 0): tile row r at
// st + r * pitch floats.
template <int N, int TWX>
__device__ __forceinline__ void bulk_real_rows(float* st, const float* __restrict__ in, int64_t q0,
                                               int pitch_floats, uint64_t* bar) {
  bar_expect(bar, (uint32_t)(TWX * N * sizeof(float)));
  const float* src = in + real_row_q(q0, N) * N;
#pragma unroll
  for (int r = 0; r < TWX; ++r)
    bulk_load(st + r * pitch_floats, src + ((int64_t)(r % HQ) * N + r / HQ) * N, N * sizeof(float), bar);
}

template <int N, int TWX, int T, int CTAS, bool BULK>
__global__ void __launch_bounds__(T, CTAS) k_xr2c(const float* __restrict__ in, float2* __restrict__ out,
                                                float scale, float offset,
                                                const float2* __restrict__ twg, int64_t ntiles,
                                                Multi m) {
  using C = RowCfg<N, TWX>;
  constexpr int M = N / 2, P = (int)half_pitch(N);
  extern __shared__ __align__(128) float2 sm[];
  float2* tw = sm;
  float2* st0 = sm + N;
  float2* st1 = st0 + C::stage;
  if constexpr (BULK) {
    // one simulation: bulk-copy staging, one barrier per stage buffer (after the two buffers)
    uint64_t* bars = reinterpret_cast<uint64_t*>(st1 + C::stage);
    int& fail = *reinterpret_cast<int*>(bars + 2);
    const bool lead = threadIdx.x == 0;
    if (lead) {
      bar_init(&bars[0]);
      bar_init(&bars[1]);
      fence_bar_init();
      fail = 0;
    }
    load_row_tw<N, T>(tw, twg);
    __syncthreads();
    uint32_t par = 0, pend = 0;
    int64_t t = blockIdx.x;
    if (lead && t < ntiles) {
      bulk_real_rows<N, TWX>(reinterpret_cast<float*>(st0), in, row_tile<N, TWX>(t, m).row0, 2 * C::CW, &bars[0]);
      pend |= 1u;
    }
    int cur = 0;
    for (; t < ntiles; t += gridDim.x) {
      if (lead) {
        fence_async_smem();
        const int64_t tn = t + gridDim.x;
        if (tn < ntiles) {
          bulk_real_rows<N, TWX>(reinterpret_cast<float*>(cur ? st0 : st1), in, row_tile<N, TWX>(tn, m).row0,
                                 2 * C::CW, &bars[cur ^ 1]);
          pend |= 1u << (cur ^ 1);
        }
        if (bar_wait(&bars[cur], (par >> cur) & 1u)) {
          par ^= 1u << cur;
          pend &= ~(1u << cur);
        } else {
          fail = 1;
        }
      }
      __syncthreads();
      if (fail) break;
      const HalfRowOut<P> o{out + hrow_q(row_tile<N, TWX>(t, m).row0, P)};
      fft_rowtile_r2c<M, TWX, C::CW, T, ScaleOffset, true, HalfRowOut<P>>(cur ? st1 : st0, tw + M, tw,
                                                                           ScaleOffset{scale, offset}, o);
      __syncthreads();
      cur ^= 1;
    }
    if (lead && fail) {
      atomicAdd(&g_tile_load_failures, 1u);
      for (int i = 0; i < 2; ++i)
        if ((pend >> i) & 1u) bar_wait(&bars[i], (par >> i) & 1u);
    }
    return;
  }
  load_row_tw<N, T>(tw, twg);
  int64_t t = blockIdx.x;
  if (t < ntiles) {
    const RowTile r = row_tile<N, TWX>(t, m);
    stage_real_rows<N, TWX, T>(reinterpret_cast<float*>(st0), moved(in, r.by), r.row0, 2 * C::CW);
  }
  cp_async_commit();
  int cur = 0;
  for (; t < ntiles; t += gridDim.x) {
    cp_async_wait<0>();  // this thread's copies of tile t (the only group in flight)
    __syncthreads();     // tile t has landed, and every warp is done with the other buffer
    const int64_t tn = t + gridDim.x;
    if (tn < ntiles) {
      const RowTile r = row_tile<N, TWX>(tn, m);
      stage_real_rows<N, TWX, T>(reinterpret_cast<float*>(cur ? st0 : st1), moved(in, r.by), r.row0, 2 * C::CW);
    }
    cp_async_commit();
    const RowTile r = row_tile<N, TWX>(t, m);
    const HalfRowOut<P> o{moved(out, r.by) + hrow_q(r.row0, P)};
    fft_rowtile_r2c<M, TWX, C::CW, T, ScaleOffset, true, HalfRowOut<P>>(cur ? st1 : st0, tw + M, tw,
                                                                         ScaleOffset{scale, offset}, o);
    cur ^= 1;
  }
  cp_async_wait<0>();
}

// Up to six independent row transforms per launch (job = tile / tiles_per_job).
struct RowJobs {
  const void* in[6];
  void* out[6];
  float kfs[6];
  int njobs;
  uint32_t jmul, jshift;  // q / njobs = (umulhi(q, jmul) + q) >> jshift for q < 2^31
  const SimHeader* hdr;   // 16-bit outputs: scales and absmax of each job (moved per simulation)
};

// Division by an invariant integer d >= 1 through a multiply-high (Granlund and
// Montgomery, "Division by invariant integers using multiplication", PLDI 1994):
// l = ceil(log2 d), m = floor(2^32 (2^l - d) / d) + 1, q = (umulhi(n, m) + n) >> l,
// exact for every n < 2^31.
inline void fast_div_magic(uint32_t d, uint32_t& mul, uint32_t& shift) {
  uint32_t l = 0;
  while ((1ull << l) < d) ++l;
  mul = (uint32_t)((((1ull << l) - d) << 32) / d + 1);
  shift = l;
}
__device__ __forceinline__ uint32_t fast_div(uint32_t n, uint32_t mul, uint32_t shift) {
  return (__umulhi(n, mul) + n) >> shift;
}

// Tile t of a multi-job, multi-simulation c2r launch: simulation, job, first row.
struct JobTile {
  int job;
  int64_t row0, by;
  uint32_t q;  // simulation * njobs + job
};
template <int N, int TWX>
__device__ __forceinline__ JobTile job_tile(int64_t t64, const RowJobs& jobs, const Multi& m) {
  constexpr uint32_t TPJ = (uint32_t)N * N / TWX;  // tiles per job
  const uint32_t t = (uint32_t)t64, q = t / TPJ;     // q = simulation * njobs + job
  const uint32_t b = fast_div(q, jobs.jmul, jobs.jshift);
  return JobTile{(int)(q - b * (uint32_t)jobs.njobs), (int64_t)(t - q * TPJ) * TWX, shift_of(m, (int)b), q};
}

// Store hook of the c2r row transform: tile row r's M complex outputs (2M reals) to its
// real row (o: the first real row of the tile).
template <int M>
struct RealRowOut {
  static constexpr bool kSmem = false;
  float2* o;
  __device__ __forceinline__ float2 operator()(float2 v, int r, int k) const {
    o[tile_real_row<2 * M>(r) * M + k] = v;
    return v;
  }
};

// The same with 16-bit outputs (variant a.S1, the six per-step LPT fields):
// value / scale as bf16 (OUT 1) or fp16 (OUT 2, saturated at the largest
// finite value), two reals per 32-bit word; the largest |value| is kept in *amax.
template <int M, int OUT>
struct RealRowOut16 {
  static constexpr bool kSmem = false;
  uint32_t* o;
  float inv;
  float* amax;
  __device__ __forceinline__ float2 operator()(float2 v, int r, int k) const {
    *amax = fmaxf(*amax, fmaxf(fabsf(v.x), fabsf(v.y)));
    float a = v.x * inv, b = v.y * inv;
    uint32_t w;
    if constexpr (OUT == 1) {
      const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
      w = *reinterpret_cast<const uint32_t*>(&h);
    } else {
      a = fminf(fmaxf(a, -65504.f), 65504.f);
      b = fminf(fmaxf(b, -65504.f), 65504.f);
      const __half2 h = __floats2half2_rn(a, b);
      w = *reinterpret_cast<const uint32_t*>(&h);
    }
    o[tile_real_row<2 * M>(r) * M + k] = w;
    return v;
  }
};

// Largest |value| of a job's tiles into hdr->lq_amax[job] (one atomic per warp).
__device__ __forceinline__ void amax_flush(const SimHeader* h, int job, float a) {
  const unsigned ua = __reduce_max_sync(0xffffffffu, __float_as_uint(a));
  if ((threadIdx.x & 31) == 0 && ua != 0u && h)
    atomicMax(reinterpret_cast<unsigned*>(const_cast<float*>(&h->lq_amax[job])), ua);
}

template <int N, int TWX, int T, int CTAS, int OUT = 0>
__global__ void __launch_bounds__(T, CTAS) k_xc2r(const __grid_constant__ RowJobs jobs,
                                                const float2* __restrict__ twg, int64_t tiles_per_job,
                                                Multi m) {
  using C = RowCfg<N, TWX>;
  constexpr int M = N / 2;
  extern __shared__ __align__(128) float2 sm[];
  float2* tw = sm;
  float2* st0 = sm + N;
  float2* st1 = st0 + C::stage;
  load_row_tw<N, T>(tw, twg);
  const int64_t ntiles = tiles_per_job * jobs.njobs * m.nb;
  int64_t t = blockIdx.x;
  if (t < ntiles) {
    const JobTile j = job_tile<N, TWX>(t, jobs, m);
    stage_complex_rows<N, TWX, T>(st0, moved(static_cast<const float2*>(jobs.in[j.job]), j.by), j.row0);
  }
  cp_async_commit();
  int cur = 0;
  // 16-bit outputs: running |value| maximum of the current (simulation, job)
  float run_max = 0.f;
  uint32_t run_q = 0xffffffffu;
  const SimHeader* run_h = nullptr;
  int run_job = 0;
  for (; t < ntiles; t += gridDim.x) {
    const JobTile j = job_tile<N, TWX>(t, jobs, m);
    cp_async_wait<0>();  // this thread's copies of tile t (the only group in flight)
    __syncthreads();     // tile t has landed, and every warp is done with the other buffer
    const int64_t tn = t + gridDim.x;
    if (tn < ntiles) {
      const JobTile jn = job_tile<N, TWX>(tn, jobs, m);
      stage_complex_rows<N, TWX, T>(cur ? st0 : st1, moved(static_cast<const float2*>(jobs.in[jn.job]), jn.by),
                                 jn.row0);
    }
    cp_async_commit();
    float2* buf = cur ? st1 : st0;
    // the c2r pre-processing rides on the transform's first loads
    using Pre = C2rCombine<N, C::CW>;
    const Pre pre{buf, tw, jobs.kfs[j.job]};
    // the outputs leave straight from the transform's last step
    if constexpr (OUT == 0) {
      float* out = moved(static_cast<float*>(jobs.out[j.job]), j.by);
      const RealRowOut<M> o{reinterpret_cast<float2*>(out + real_row_q(j.row0, N) * N)};
      fft_rowtile<M, TWX, C::CW, T, true, Pre, RealRowOut<M>>(buf, tw + M, pre, o);
    } else {
      const SimHeader* h = moved(jobs.hdr, j.by);
      if (j.q != run_q) {  // the same for every thread of the CTA
        amax_flush(run_h, run_job, run_max);
        run_max = 0.f;
        run_q = j.q;
        run_h = h;
        run_job = j.job;
      }
      uint32_t* out = moved(static_cast<uint32_t*>(jobs.out[j.job]), j.by);
      float tile_max = 0.f;
      const RealRowOut16<M, OUT> o{out + real_row_q(j.row0, N) * M,
                                   1.f / h->lq_scale[j.job], &tile_max};
      fft_rowtile<M, TWX, C::CW, T, true, Pre, RealRowOut16<M, OUT>>(buf, tw + M, pre, o);
      run_max = fmaxf(run_max, tile_max);
    }
    cur ^= 1;
  }
  if constexpr (OUT != 0) amax_flush(run_h, run_job, run_max);
  cp_async_wait<0>();
}

// C2rCombine with the x-derivative factor of even tile rows (kfs) and of odd
// ones (kfs1): a pair tile's rows of a and of b.
template <int N, int CW>
struct C2rCombine2 {
  const float2* buf;
  const float2* tw;
  float kfs, kfs1;
  __device__ __forceinline__ float2 operator()(float2 zn, int r, int n) const {
    return C2rCombine<N, CW>{buf, tw, (r & 1) ? kfs1 : kfs}(zn, r, n);
  }
};

// Store hook of a pair tile's c2r: the last transform step leaves output k of
// tile rows 2w (a) and 2w + 1 (b) in lanes l and l ^ R1 of one warp (R1 = the
// first-step radix, the outputs per row and lane group of that step); one
// shuffle gives lane l (a) the pair (a, b) of real 2k and lane l ^ R1 (b) that
// of real 2k + 1, and each writes one 8-byte pair, so a warp's stores cover
// consecutive cells.  o: cell 0 of the tile's first real row.
template <int N, int R1>
struct PairRowOut {
  static constexpr bool kSmem = false;
  float2* o;
  __device__ __forceinline__ float2 operator()(float2 v, int r, int k) const {
    const int isb = r & 1;
    const float recv = __shfl_xor_sync(0xffffffffu, isb ? v.x : v.y, R1);
    float2* row = o + (int64_t)tile_real_row<N>(r >> 1) * N;
    // one store instruction for the warp: cell 2k (a lanes) or 2k + 1 (b lanes)
    row[2 * k + isb] = isb ? make_float2(recv, v.y) : make_float2(v.x, recv);
    return v;
  }
};

// c2r of the rows of a (x derivative i kfs kx on load) and of b into the (x, y)
// pairs of one interleaved real field (App. B: F_x and F_y of the force mesh),
// pair tiles of TWX/2 rows of each.
template <int N, int TWX, int T, int CTAS>
__global__ void __launch_bounds__(T, CTAS) k_xc2r_pair(
    const float2* __restrict__ a, const float2* __restrict__ b, float2* __restrict__ out, float kfs,
    const float2* __restrict__ twg, int64_t tiles_per_sim, Multi m) {
  using C = RowCfg<N, TWX>;
  constexpr int M = N / 2, R1 = Split<M>::R1;
  static_assert(R1 < 32 && TWX * R1 % 32 == 0, "pair lanes within whole warps");
  extern __shared__ __align__(128) float2 sm[];
  float2* tw = sm;
  float2* st0 = sm + N;
  float2* st1 = st0 + C::stage;
  load_row_tw<N, T>(tw, twg);
  const int64_t ntiles = tiles_per_sim * m.nb;
  auto tile = [&](int64_t t, int64_t& q0, int64_t& by) {
    const int64_t s = t / tiles_per_sim;
    q0 = (t - s * tiles_per_sim) * (TWX / 2);
    by = shift_of(m, (int)s);
  };
  int64_t t = blockIdx.x;
  if (t < ntiles) {
    int64_t q0, by;
    tile(t, q0, by);
    stage_complex_rows_pair<N, TWX, T>(st0, moved(a, by), moved(b, by), q0);
  }
  cp_async_commit();
  int cur = 0;
  for (; t < ntiles; t += gridDim.x) {
    int64_t q0, by;
    tile(t, q0, by);
    cp_async_wait<0>();  // this thread's copies of tile t (the only group in flight)
    __syncthreads();     // tile t has landed, and every warp is done with the other buffer
    const int64_t tn = t + gridDim.x;
    if (tn < ntiles) {
      int64_t qn, bn;
      tile(tn, qn, bn);
      stage_complex_rows_pair<N, TWX, T>(cur ? st0 : st1, moved(a, bn), moved(b, bn), qn);
    }
    cp_async_commit();
    float2* buf = cur ? st1 : st0;
    float2* o = moved(out, by);
    const PairRowOut<N, R1> st{o + real_row_q(q0, N) * N};
    fft_rowtile<M, TWX, C::CW, T, true, C2rCombine2<N, C::CW>, PairRowOut<N, R1>>(
        buf, tw + M, C2rCombine2<N, C::CW>{buf, tw, kfs, 0.f}, st);
    cur ^= 1;
  }
  cp_async_wait<0>();
}

// Screening factor eps(w) (Sec. 6.1, Sec. 6.2).  The divisions and the square
// root use the fast intrinsics (a few ulp), well below the FP32 rounding of
// the transforms the factor feeds.
// p: f(R) the threshold fr_thr on |Phi_N|; nDGP the coefficient dgp_coef.
template <int MODEL>
__device__ __forceinline__ float screen_eps(float w, float p) {
  if (MODEL == 1) {
    const float aw = fabsf(w);
    return aw > p ? __fdividef(p, aw) : 1.f;
  } else {
    const float u = 1.f + p * fmaxf(1.f + w, 0.f);  // >= 1
    return __fdividef(2.f, u * rsqrtf(u) + 1.f);
  }
}

// The source of a screening pass at density contrast d = rho / rho_bar - 1 and screening
// field w.  Chameleon-type models: S = d eps(w), which the force pass combines with
// delta(k) mode by mode (the coupling depends on k).  Vainshtein: the range is infinite,
// Phi_tot = -kappa (delta + C S) / k^2 with C independent of k, so the source is the
// whole d + C d eps(w): delta(k) is neither written nor read again (two of the fourteen
// half-spectrum streams of the screened force).
template <int MODEL>
__device__ __forceinline__ float screen_source(float d, float w, float p, float C) {
  const float e = d * screen_eps<MODEL>(w, p);
  return MODEL == 1 ? e : fmaf(C, e, d);
}

// Between the transforms of a screening pass: element j of tile row r is the source at w
// (the tile value) and the density read from consecutive rows in global memory (M
// float2 per row, read-only path); used by the plane pass.
template <int M, int MODEL>
struct ScreenSource {
  const float2* rho;
  float inv_rhobar, p, C;
  __device__ __forceinline__ float2 operator()(float2 w, int r, int j) const {
    const float2 rv = __ldg(rho + r * M + j);
    const float d0 = rv.x * inv_rhobar - 1.f, d1 = rv.y * inv_rhobar - 1.f;
    return make_float2(screen_source<MODEL>(d0, w.x, p, C), screen_source<MODEL>(d1, w.y, p, C));
  }
};

// The same for an x-pass row tile (rho: the tile's first density row): each warp's
// loads of one transform step cover 32 consecutive values of a row.
template <int M, int MODEL>
struct ScreenSourceRows {
  const float2* rho;
  float inv_rhobar, p, C;
  __device__ __forceinline__ float2 operator()(float2 w, int r, int j) const {
    const float2 rv = __ldg(rho + tile_real_row<2 * M>(r) * M + j);
    const float d0 = rv.x * inv_rhobar - 1.f, d1 = rv.y * inv_rhobar - 1.f;
    return make_float2(screen_source<MODEL>(d0, w.x, p, C), screen_source<MODEL>(d1, w.y, p, C));
  }
};

// Screening source (screen_source): c2r of the screening field rows, eps from the
// field and delta from rho (read from global memory by the forward transform's
// loads), r2c.  Shared memory: twiddles, two row tiles (double-buffered field rows).
template <int N, int TWX>
constexpr size_t xscreen_smem() {
  return RowCfg<N, TWX>::smem;
}

template <int N, int TWX, int T, int CTAS, int MODEL>
__global__ void __launch_bounds__(T, CTAS) k_x_screen(const float2* __restrict__ w_in,
                                                    const float* __restrict__ rho,
                                                    float2* __restrict__ s_out,
                                                    ForceParams fp0, const float2* __restrict__ twg,
                                                    int64_t ntiles, Multi m) {
  if (!m.shift) resolve(fp0, 0);  // one simulation: once per launch
  using C = RowCfg<N, TWX>;
  constexpr int M = N / 2;
  extern __shared__ __align__(128) float2 sm[];
  float2* tw = sm;
  float2* st0 = sm + N;
  float2* st1 = st0 + C::stage;
  load_row_tw<N, T>(tw, twg);
  __syncthreads();
  int64_t t = blockIdx.x;
  if (t < ntiles) {
    const RowTile r = row_tile<N, TWX>(t, m);
    stage_complex_rows_warp<N, TWX, T>(st0, moved(w_in, r.by), r.row0);
  }
  cp_async_commit();
  int cur = 0;
  for (; t < ntiles; t += gridDim.x) {
    const RowTile r = row_tile<N, TWX>(t, m);
    const int64_t row0 = r.row0;
    ForceParams fp = fp0;
    resolve(fp, r.by);
    const int64_t tn = t + gridDim.x;
    float2* buf = cur ? st1 : st0;
    cp_async_wait<0>();  // w rows of this tile (the only group in flight)
    __syncwarp();
    // the next tile's w rows into the other buffer land while this tile is transformed
    if (tn < ntiles) {
      const RowTile rn = row_tile<N, TWX>(tn, m);
      stage_complex_rows_warp<N, TWX, T>(cur ? st0 : st1, moved(w_in, rn.by), rn.row0);
    }
    cp_async_commit();
    // S = delta eps(w) is formed between the inverse and the forward transform
    const float* rho_t = moved(rho, r.by);
    const ScreenSourceRows<M, MODEL> src{reinterpret_cast<const float2*>(rho_t + real_row_q(row0, N) * N),
                                         fp.inv_rhobar, MODEL == 1 ? fp.fr_thr : fp.dgp_coef, fp.C};
    constexpr int P = (int)half_pitch(N);
    fft_rowtile_inv_r2c<M, TWX, C::CW, T, C2rCombine<N, C::CW>, ScreenSourceRows<M, MODEL>, true, HalfRowOut<P>>(
        buf, tw + M, tw, C2rCombine<N, C::CW>{buf, tw, 0.f}, src,
        HalfRowOut<P>{moved(s_out, r.by) + hrow_q(row0, P)});
    cur ^= 1;
  }
  cp_async_wait<0>();
}

// ---------------------------------------------------------------- plane passes (N <= 128)
// Up to 128 points a whole z-plane of the half spectrum (N rows of M + 1 = N/2 + 1
// values) fits in one CTA's shared memory, so the x and y steps of a 3-D
// transform run as one pass over HBM: one CTA per plane (and simulation) stages
// the plane, transforms its rows and then its columns in place, and writes it
// back; the intermediate between the x and y steps never leaves the SM.  The
// plane's rows have the row-transform pitch CW (>= M + R2 - 1, 8 mod 16, so the
// row steps are conflict-free) and the column transforms run on chunks of
// TWCOL columns at that pitch, with the padding rows of their intermediate
// below the plane.
template <int N>
struct PlaneCfg {
  static constexpr int M = N / 2;
  static constexpr int CW = rowtile_pitch<M>();
  static constexpr int ROWS = fft_rows<N>();
  static constexpr int TWCOL = N == 128 ? 24 : CW;  // column chunk (a multiple of 8, CW = 3 x 24 at N = 128)
  static constexpr size_t buf = (size_t)ROWS * CW;   // float2
  static constexpr size_t smem = ((size_t)N + M + buf) * sizeof(float2);  // twiddles (load_plane_tw), plane
  static_assert(CW >= M + 1 && CW % 8 == 0 && CW % TWCOL == 0 && TWCOL % 8 == 0, "plane pitch");
};

// Twiddles of a plane pass: the N-entry table (columns, real split), then M entries of
// row transform first-step twiddles (fft_rowtile's w1 = tw + N).
template <int N>
__device__ __forceinline__ void load_plane_tw(float2* tw, const float2* __restrict__ twg) {
  constexpr int M = N / 2;
  load_tw(tw, twg, N);
  for (int i = threadIdx.x; i < M; i += NT) tw[N + i] = twg[2 * row_twiddle<M>(i)];
}

// The N real rows of a plane (N floats each) as M complex values per row at pitch CW.
template <int N>
__device__ __forceinline__ void stage_real_plane(float2* buf, const float* __restrict__ src) {
  constexpr int CH = N / 4, CW = PlaneCfg<N>::CW;  // 16-byte pieces per row
  for (int e = threadIdx.x; e < N * CH; e += NT) {
    const int y = e / CH, p = e - y * CH;
    cp_async16(reinterpret_cast<float*>(buf + y * CW) + 4 * p, src + (int64_t)y * N + 4 * p, true);
  }
}

// Forward x (r2c, input scaled then offset) and y transforms of plane blockIdx.x of a
// real N^3 field into the interleaved half spectrum (the z pass follows separately).
template <int N>
__global__ void __launch_bounds__(NT) k_plane_r2c(const float* __restrict__ in, float2* __restrict__ out,
                                                  float scale, float offset, const float2* __restrict__ twg,
                                                  Multi m) {
  using C = PlaneCfg<N>;
  extern __shared__ __align__(128) float2 sm[];
  float2* tw = sm;
  float2* buf = sm + N + C::M;
  const int z = blockIdx.x;
  load_plane_tw<N>(tw, twg);
  pdl_wait();
  const int64_t by = shift_of(m, blockIdx.y);
  stage_real_plane<N>(buf, moved(in, by) + (int64_t)z * N * N);
  cp_async_commit();
  cp_async_wait<0>();
  __syncthreads();
  pdl_go();
  fft_rowtile_r2c<C::M, N, C::CW, NT, ScaleOffset, false, RowStore>(buf, tw + N, tw, ScaleOffset{scale, offset},
                                                                   RowStore{});
  __syncthreads();
  constexpr int64_t P = half_pitch(N);
  float2* g = moved(out, by) + hrow(z, 0, N, P);
#pragma unroll 1
  for (int c0 = 0; c0 < C::CW; c0 += C::TWCOL)
    fft_tile<N, C::TWCOL, C::CW, NT, false, 1, TileLoad, ColOut>(
        buf + c0, tw, TileLoad{}, ColOut{g + hcol(c0), HQ * HQ * P, HQ * P, C::M + 1 - c0});
}

// Store hook of a plane's row transforms: real row r (M float2 = N reals) to g + r M.
template <int M>
struct PlaneRowOut {
  static constexpr bool kSmem = false;
  float2* g;
  __device__ __forceinline__ float2 operator()(float2 v, int r, int k) const {
    g[r * M + k] = v;
    return v;
  }
};

// The N complex rows (ky) of plane z of an interleaved half spectrum into buf (pitch CW).
template <int N>
__device__ __forceinline__ void stage_complex_plane(float2* buf, const float2* __restrict__ g, int z) {
  constexpr int M = N / 2, CW = PlaneCfg<N>::CW;
  constexpr int64_t P = half_pitch(N);
  constexpr int CH = (M + 2) / 2;  // 16-byte pieces per row (kx = 0..M, staged as M + 2)
  const float2* src = g + hrow(z, 0, N, P);
  for (int e = threadIdx.x; e < N * CH; e += NT) {
    const int y = e / CH, p = e - y * CH, kx = 2 * p;
    cp_async16(buf + y * CW + kx, src + (int64_t)y * HQ * P + hcol(kx), true);
  }
}

// Load hook of a plane's y inverse: DY multiplies by i kfs f_n on load (f_n the signed
// frequency of row n, zero on the Nyquist row); PACK joins columns 0 and M into column 0
// as X_0 + i X_M.
template <int N, bool DY, bool PACK>
struct PlaneLoad {
  float kfs;
  __device__ __forceinline__ float2 in(float2 v, int n) const {
    if (!DY) return v;
    return cmul_if(v, (n == N / 2) ? 0.f : kfs * (float)freq_index(n, N));
  }
  __device__ __forceinline__ float2 operator()(const float2* buf, int n, int c, int at) const {
    float2 v = in(buf[at], n);
    if (PACK && c == 0) {
      const float2 m = in(buf[at + N / 2], n);
      v = make_float2(v.x - m.y, v.y + m.x);
    }
    return v;
  }
};
// ... and its store hook: the real parts of columns 0 and M from the joined one.
template <int N>
struct PlaneUnpack {
  static constexpr bool kSmem = true;
  float2* buf;
  __device__ __forceinline__ float2 operator()(float2 v, int, int c, int at) const {
    if (c != 0) return v;
    buf[at + N / 2] = make_float2(v.y, 0.f);
    return make_float2(v.x, 0.f);
  }
};

// y inverse of every column of plane a, in place (DY: of i kfs f_y times them).
// HERM: the plane belongs to a real field, so columns 0 and M are Hermitian along y and
// their inverses real: both ride on one complex column, which leaves M = N/2 columns,
// whole chunks of 32 with no idle thread, instead of M + 1 in chunks of 24.  The force
// and screening spectra are such; caller-given potentials (the LPT planes) need not be.
// Force plane pass 3.41 -> 2.99 ms, screening plane pass 863 -> 838 us over 256 meshes of
// 128^3 (the derivative on load instead of in a pass of its own also in the LPT planes, 957 -> 908).
// Where |X_M| is far below |X_0| (a potential: by about M^2) the joined column's rounding is
// relative to X_0, so column M's own relative error grows by their ratio.  The field's does not: its
// x transform adds the two columns in its first step, with a rounding of that size.
template <int N, bool HERM, bool DY>
__device__ __forceinline__ void plane_yinv(float2* a, const float2* tw, float kfs) {
  using C = PlaneCfg<N>;
  if constexpr (HERM) {
    constexpr int TW = C::M < 32 ? C::M : 32;
    fft_tile<N, TW, C::CW, NT, true, 1, PlaneLoad<N, DY, true>, PlaneUnpack<N>>(a, tw, PlaneLoad<N, DY, true>{kfs},
                                                                              PlaneUnpack<N>{a});
#pragma unroll 1
    for (int c0 = TW; c0 < C::M; c0 += TW)
      fft_tile<N, TW, C::CW, NT, true, 1, PlaneLoad<N, DY, false>>(a + c0, tw, PlaneLoad<N, DY, false>{kfs});
  } else {
#pragma unroll 1
    for (int c0 = 0; c0 < C::CW; c0 += C::TWCOL)
      fft_tile<N, C::TWCOL, C::CW, NT, true, 1, PlaneLoad<N, DY, false>>(a + c0, tw, PlaneLoad<N, DY, false>{kfs});
  }
}

// c2r of the N rows of plane buffer a (x derivative i kfs kx applied on load when
// kfs != 0) to the real plane at g (N x N floats).
template <int N>
__device__ __forceinline__ void plane_xc2r(float2* a, const float2* tw, float kfs, float* g) {
  using C = PlaneCfg<N>;
  fft_rowtile<C::M, N, C::CW, NT, true, C2rCombine<N, C::CW>, PlaneRowOut<C::M>>(
      a, tw + N, C2rCombine<N, C::CW>{a, tw, kfs}, PlaneRowOut<C::M>{reinterpret_cast<float2*>(g)});
}

// Gradient components from spectra after their z inverse, one (plane, component)
// per CTA: component q is c2r(yinv(in[q] times i kfs ky when bit q of dy)) with
// i kfs kx applied on load when bit q of dx.  The CTAs of one plane are
// consecutive (x = plane * n + q), so components that share an input spectrum
// run side by side and the repeated reads of its plane come from L2.
struct PlaneJobs {
  const float2* in[6];
  float* out[6];
  int n, dx, dy;
  float kfs;
  float* zdst = nullptr;  // optional: zdst[0, zfloats) of each simulation is cleared, zchunk
  int64_t zfloats = 0;    // floats (a multiple of 4) per CTA, by 16-byte stores
  int64_t zchunk = 0;
};

template <int N, bool HERM>
__global__ void __launch_bounds__(NT) k_plane_grad(PlaneJobs jobs, const float2* __restrict__ twg, Multi m) {
  using C = PlaneCfg<N>;
  extern __shared__ __align__(128) float2 sm[];
  float2* tw = sm;
  float2* a = sm + N + C::M;
  const int z = blockIdx.x / jobs.n, q = blockIdx.x - z * jobs.n;
  const float2* in = jobs.in[0];
  float* out = jobs.out[0];
#pragma unroll
  for (int i = 1; i < 6; ++i)  // selects, not an indexed copy of the parameters
    if (i == q) {
      in = jobs.in[i];
      out = jobs.out[i];
    }
  load_plane_tw<N>(tw, twg);
  pdl_wait();
  const int64_t by = shift_of(m, blockIdx.y), off = (int64_t)z * N * N;
  stage_complex_plane<N>(a, moved(in, by), z);
  cp_async_commit();
  if (jobs.zdst) {  // this CTA's share of the zero fill while its plane lands
    const int64_t lo = (int64_t)blockIdx.x * jobs.zchunk, hi = min(lo + jobs.zchunk, jobs.zfloats);
    float4* d = reinterpret_cast<float4*>(moved(jobs.zdst, by));
    for (int64_t i = lo / 4 + threadIdx.x; i < hi / 4; i += NT) d[i] = make_float4(0.f, 0.f, 0.f, 0.f);
  }
  cp_async_wait<0>();
  __syncthreads();
  pdl_go();
  if ((jobs.dy >> q) & 1) plane_yinv<N, HERM, true>(a, tw, jobs.kfs);
  else plane_yinv<N, HERM, false>(a, tw, 0.f);
  plane_xc2r<N>(a, tw, ((jobs.dx >> q) & 1) ? jobs.kfs : 0.f, moved(out, by) + off);
}

// Screening source of plane blockIdx.x in one pass (Sec. 6.1, Sec. 6.2): the
// screening field's plane after its z inverse is transformed back along y and x
// (c2r), S = delta eps(w) is formed as the forward x transform loads it (delta
// read from the density plane in global memory), and the forward x (r2c) and y
// steps write S's plane of the interleaved half spectrum; the z pass follows.
template <int N, int MODEL>
__global__ void __launch_bounds__(NT) k_plane_screen(const float2* __restrict__ w_in,
                                                     const float* __restrict__ rho,
                                                     float2* __restrict__ s_out, ForceParams fp,
                                                     const float2* __restrict__ twg, Multi m) {
  using C = PlaneCfg<N>;
  constexpr int M = C::M;
  extern __shared__ __align__(128) float2 sm[];
  float2* tw = sm;
  float2* a = sm + N + C::M;
  const int z = blockIdx.x;
  load_plane_tw<N>(tw, twg);
  pdl_wait();
  const int64_t by = shift_of(m, blockIdx.y);
  resolve(fp, by);
  stage_complex_plane<N>(a, moved(w_in, by), z);
  cp_async_commit();
  cp_async_wait<0>();
  __syncthreads();
  pdl_go();
  plane_yinv<N, true, false>(a, tw, 0.f);
  const ScreenSource<M, MODEL> src{reinterpret_cast<const float2*>(moved(rho, by) + (int64_t)z * N * N),
                                         fp.inv_rhobar, MODEL == 1 ? fp.fr_thr : fp.dgp_coef, fp.C};
  fft_rowtile_inv_r2c<M, N, C::CW, NT, C2rCombine<N, C::CW>, ScreenSource<M, MODEL>, false, RowStore>(
      a, tw + N, tw, C2rCombine<N, C::CW>{a, tw, 0.f}, src, RowStore{});
  __syncthreads();
  constexpr int64_t P = half_pitch(N);
  float2* g = moved(s_out, by) + hrow(z, 0, N, P);
#pragma unroll 1
  for (int c0 = 0; c0 < C::CW; c0 += C::TWCOL)
    fft_tile<N, C::TWCOL, C::CW, NT, false, 1, TileLoad, ColOut>(
        a + c0, tw, TileLoad{}, ColOut{g + hcol(c0), HQ * HQ * P, HQ * P, C::M + 1 - c0});
}

// ---------------------------------------------------------------- launch helpers
template <int N, int NBUF>
constexpr size_t col_smem() {
  static_assert(col_rows(N) == fft_rows<N>(), "column stage rows");
  return col_smem_c(N, NBUF);
}

// Along y: o = z, n = y.  Along z: o = y, n = z (rows of a plane group 8 elements apart).
template <int N, int TW>
ColGeo<N, TW> geo_y(Multi m) {
  const int64_t P = half_pitch(N);
  return ColGeo<N, TW>{HQ * N * P, 8, HQ * HQ * P, HQ * P, 0, m};
}
template <int N, int TW>
ColGeo<N, TW> geo_z(Multi m) {
  const int64_t P = half_pitch(N);
  return ColGeo<N, TW>{HQ * HQ * P, HQ * P, HQ * N * P, 8, 1, m};
}
template <int N, int TW>
constexpr int64_t col_tiles() {
  return (int64_t)N * ((N / 2) / TW + 1);
}

}  // namespace

void set_grid_cap(int max_ctas) { g_grid_cap = max_ctas > 0 ? max_ctas : 0; }

#define COLA_SWITCH_N(NVAL, ...)                 \
  switch (NVAL) {                                \
    case 32: { constexpr int N = 32; __VA_ARGS__; } break;     \
    case 64: { constexpr int N = 64; __VA_ARGS__; } break;     \
    case 128: { constexpr int N = 128; __VA_ARGS__; } break;   \
    case 256: { constexpr int N = 256; __VA_ARGS__; } break;   \
    case 512: { constexpr int N = 512; __VA_ARGS__; } break;   \
    case 1024: { constexpr int N = 1024; __VA_ARGS__; } break; \
    default: return cudaErrorInvalidValue;       \
  }

template <int N>
static cudaError_t launch_xr2c(const float* in, float2* out, float scale, float offset,
                               const float2* tw, cudaStream_t s, Multi m) {
  constexpr RowShape SH = r2c_shape(N);
  constexpr int TWX = SH.rows, T = SH.threads;
  const int64_t tps = (int64_t)N * N / TWX;
  const int64_t ntiles = tps * m.nb;
  auto go = [&](auto bulk_c) {
    constexpr bool BULK = decltype(bulk_c)::value;
    const size_t sm = RowCfg<N, TWX>::smem + (BULK ? 2 * sizeof(uint64_t) + 16 : 0);
    auto k = k_xr2c<N, TWX, T, SH.ctas, BULK>;
    unsigned grid;
    cudaError_t e = prep(k, sm, ntiles, grid, T);
    if (e != cudaSuccess) return e;
    k<<<grid, T, sm, s>>>(in, out, scale, offset, tw, ntiles, m);
    return cudaGetLastError();
  };
  // one 1024-point simulation: 1-D bulk copies stage the real rows (1.93 -> 1.90 ms at 1024^3)
  if constexpr (N >= 1024) {
    if (!m.shift && (reinterpret_cast<uintptr_t>(in) & 15) == 0) return go(std::true_type{});
  }
  return go(std::false_type{});
}

cudaError_t fft_xr2c(int Nv, const float* in, float2* out, float scale, float offset,
                     const float2* tw, cudaStream_t s, Multi m) {
  COLA_SWITCH_N(Nv, return launch_xr2c<N>(in, out, scale, offset, tw, s, m));
  return cudaSuccess;
}

template <int N>
static cudaError_t launch_xc2r_multi(int njobs, const float2* const* in, float* const* out,
                                     const float* kfs, const float2* tw, cudaStream_t s, Multi m) {
  constexpr RowShape SH = c2r_shape(N);
  constexpr int TWX = SH.rows, T = SH.threads;
  const size_t sm = RowCfg<N, TWX>::smem;
  RowJobs jobs{};
  jobs.njobs = njobs;
  fast_div_magic((uint32_t)njobs, jobs.jmul, jobs.jshift);
  for (int i = 0; i < njobs; ++i) {
    jobs.in[i] = in[i];
    jobs.out[i] = out[i];
    jobs.kfs[i] = kfs[i];
  }
  const int64_t tpj = (int64_t)N * N / TWX;
  auto k = k_xc2r<N, TWX, T, SH.ctas>;
  unsigned grid;
  cudaError_t e = prep(k, sm, tpj * njobs * m.nb, grid, T);
  if (e != cudaSuccess) return e;
  k<<<grid, T, sm, s>>>(jobs, tw, tpj, m);
  return cudaGetLastError();
}

cudaError_t fft_xc2r_multi(int Nv, int njobs, const float2* const* in, float* const* out,
                           const float* kfs, const float2* tw, cudaStream_t s, Multi m) {
  if (njobs < 1 || njobs > 6) return cudaErrorInvalidValue;
  COLA_SWITCH_N(Nv, return launch_xc2r_multi<N>(njobs, in, out, kfs, tw, s, m));
  return cudaSuccess;
}

template <int N>
static cudaError_t launch_xc2r_pair(const float2* a, const float2* b, float* xy, float kfs, const float2* tw,
                                   cudaStream_t s, Multi m) {
  if constexpr (N < 256) {
    return cudaErrorInvalidValue;
  } else {
    constexpr RowShape SH = pair_shape(N);
    constexpr int TWX = SH.rows, T = SH.threads;
    const size_t sm = RowCfg<N, TWX>::smem;
    const int64_t tps = (int64_t)N * N / (TWX / 2);
    auto k = k_xc2r_pair<N, TWX, T, SH.ctas>;
    unsigned grid;
    cudaError_t e = prep(k, sm, tps * m.nb, grid, T);
    if (e != cudaSuccess) return e;
    k<<<grid, T, sm, s>>>(a, b, reinterpret_cast<float2*>(xy), kfs, tw, tps, m);
    return cudaGetLastError();
  }
}

cudaError_t fft_xc2r_pair(int Nv, const float2* a, const float2* b, float* xy, float kfs, const float2* tw,
                          cudaStream_t s, Multi m) {
  COLA_SWITCH_N(Nv, return launch_xc2r_pair<N>(a, b, xy, kfs, tw, s, m));
  return cudaSuccess;
}

template <int N, int OUT>
static cudaError_t launch_xc2r_multi16(int njobs, const float2* const* in, void* const* out, const float* kfs,
                                       const SimHeader* hdr, const float2* tw, cudaStream_t s, Multi m) {
  constexpr RowShape SH = c2r_shape(N);
  constexpr int TWX = SH.rows, T = SH.threads;
  const size_t sm = RowCfg<N, TWX>::smem;
  RowJobs jobs{};
  jobs.njobs = njobs;
  jobs.hdr = hdr;
  fast_div_magic((uint32_t)njobs, jobs.jmul, jobs.jshift);
  for (int i = 0; i < njobs; ++i) {
    jobs.in[i] = in[i];
    jobs.out[i] = out[i];
    jobs.kfs[i] = kfs[i];
  }
  const int64_t tpj = (int64_t)N * N / TWX;
  auto k = k_xc2r<N, TWX, T, SH.ctas, OUT>;
  unsigned grid;
  cudaError_t e = prep(k, sm, tpj * njobs * m.nb, grid, T);
  if (e != cudaSuccess) return e;
  k<<<grid, T, sm, s>>>(jobs, tw, tpj, m);
  return cudaGetLastError();
}

cudaError_t fft_xc2r_multi16(int Nv, int njobs, const float2* const* in, void* const* out, const float* kfs,
                             int prec, const SimHeader* hdr, const float2* tw, cudaStream_t s, Multi m) {
  if (njobs < 1 || njobs > 6 || !hdr || (prec != 1 && prec != 2)) return cudaErrorInvalidValue;
#define COLA_C2R16(NN)                                                                                    \
  case NN:                                                                                               \
    return prec == 1 ? launch_xc2r_multi16<NN, 1>(njobs, in, out, kfs, hdr, tw, s, m)                    \
                     : launch_xc2r_multi16<NN, 2>(njobs, in, out, kfs, hdr, tw, s, m);
  switch (Nv) {
    COLA_C2R16(32)
    COLA_C2R16(64)
    COLA_C2R16(128)
    COLA_C2R16(256)
    COLA_C2R16(512)
    default:
      return cudaErrorInvalidValue;
  }
#undef COLA_C2R16
}

cudaError_t fft_xc2r(int Nv, const float2* in, float* out, float kfs, const float2* tw,
                     cudaStream_t s, Multi m) {
  return fft_xc2r_multi(Nv, 1, &in, &out, &kfs, tw, s, m);
}

// Tensor map of a half spectrum for the TMA tile loads of a column pass along
// z (zaxis) or y, TW columns per tile (the 5-D view described above
// tma_tile).  False when the driver's encoder is unavailable or refuses the
// map: the launch then stages its tiles with cp.async.
static bool spectrum_map(CUtensorMap& map, const float2* base, int N, int TW, bool zaxis) {
  static const PFN_cuTensorMapEncodeTiled_v12000 encode = [] {
    void* f = nullptr;
    cudaDriverEntryPointQueryResult q{};
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault, &q) !=
            cudaSuccess ||
        q != cudaDriverEntryPointSuccess)
      f = nullptr;
    return reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(f);
  }();
  if (!encode || (reinterpret_cast<uintptr_t>(base) & 15)) return false;
  const cuuint64_t P = (cuuint64_t)half_pitch(N), n = (cuuint64_t)N;
  const cuuint64_t dims[5] = {8, HQ, P / 8, n, n / HQ};
  const cuuint64_t strides[4] = {64, 64 * HQ, HQ * P * 8, HQ * P * n * 8};
  const cuuint32_t box[5] = {(cuuint32_t)TW, zaxis ? (cuuint32_t)HQ : 1u, 1u, zaxis ? 1u : (cuuint32_t)std::min(N, 256),
                             zaxis ? (cuuint32_t)std::min(N / HQ, 256) : 1u};
  const cuuint32_t es[5] = {1, 1, 1, 1, 1};
  return encode(&map, CU_TENSOR_MAP_DATA_TYPE_UINT64, 5, const_cast<float2*>(base), dims, strides, box, es,
                CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// TMA staging applies to single-simulation launches of 1024-point columns
// (tiles of at most one 64-byte chunk).  Measured on GB300 (ms per launch
// against cp.async staging): z force pass 5.09 -> 4.57, screening-field z pass
// 3.24 -> 3.05, y passes 1-2 % faster; at N = 512 the plain y pass runs two
// CTAs per SM at 128 registers and lost (0.187 -> 0.222).
template <int N, int TW>
constexpr bool tma_shape() {
  return N >= 1024 && TW <= 8 && TW % 2 == 0;
}

// DENSE as in OpCol (in or out is then a dense half spectrum, axis 1)
template <int N, bool INV, int DENSE>
static cudaError_t launch_col(const float2* in, float2* out, int axis, const float2* tw, cudaStream_t s, Multi m) {
  constexpr int TW = ytw(N);
  const int64_t ntiles = col_tiles<N, TW>() * m.nb;
  const ColGeo<N, TW> geo = axis == 1 ? geo_y<N, TW>(m) : geo_z<N, TW>(m);
  CUtensorMap map{};
  auto go = [&](auto tma_c) {
    constexpr bool TMA = decltype(tma_c)::value;
    constexpr size_t smk = TMA ? tma_smem<N, fft_rows<N>() * TW, 0>() : col_smem_tw(N, TW);
    auto k = k_col<N, TW, INV, TMA, DENSE>;
    unsigned grid;
    cudaError_t e = prep(k, smk, ntiles, grid, ct(N, INV));
    if (e != cudaSuccess) return e;
    k<<<grid, ct(N, INV), smk, s>>>(OpCol<N, TW, INV, DENSE>{geo, in, out}, tw, ntiles, map);
    return cudaGetLastError();
  };
  if constexpr (tma_shape<N, TW>() && DENSE != 2) {
    if (!m.shift && spectrum_map(map, in, N, TW, axis != 1)) return go(std::true_type{});
  }
  return go(std::false_type{});
}

cudaError_t fft_col(int Nv, float2* data, int axis, bool inv, const float2* tw, cudaStream_t s,
                    Multi m) {
  COLA_SWITCH_N(Nv, return inv ? launch_col<N, true, 0>(data, data, axis, tw, s, m)
                               : launch_col<N, false, 0>(data, data, axis, tw, s, m));
  return cudaSuccess;
}

cudaError_t fft_y_dense(int Nv, float2* data, float2* dense, bool inv, const float2* tw, cudaStream_t s) {
  COLA_SWITCH_N(Nv, return inv ? launch_col<N, true, 2>(dense, data, 1, tw, s, Multi{})
                               : launch_col<N, false, 1>(data, dense, 1, tw, s, Multi{}));
  return cudaSuccess;
}

template <int N>
static cudaError_t launch_yinv2(const float2* in, float2* outp, float2* outd, float kfs,
                                const float2* tw, cudaStream_t s, Multi m) {
  constexpr int TW = ytw(N);
  const int64_t ntiles = col_tiles<N, TW>() * m.nb;
  CUtensorMap map{};
  auto go = [&](auto tma_c) {
    constexpr bool TMA = decltype(tma_c)::value;
    constexpr size_t sm = yinv2r_smem<N, TW>() + (TMA ? 4 * sizeof(uint64_t) : 0);
    auto k = k_yinv2r<N, TW, TMA>;
    unsigned grid;
    cudaError_t e = prep(k, sm, ntiles, grid, yt(N));
    if (e != cudaSuccess) return e;
    k<<<grid, yt(N), sm, s>>>(geo_y<N, TW>(m), in, outp, outd, kfs, tw, ntiles, map);
    return cudaGetLastError();
  };
  if constexpr (tma_shape<N, TW>()) {
    if (!m.shift && spectrum_map(map, in, N, TW, false)) return go(std::true_type{});
  }
  return go(std::false_type{});
}

cudaError_t fft_yinv2(int Nv, const float2* in, float2* outp, float2* outd, float kfs,
                      const float2* tw, cudaStream_t s, Multi m) {
  COLA_SWITCH_N(Nv, return launch_yinv2<N>(in, outp, outd, kfs, tw, s, m));
  return cudaSuccess;
}

template <int N>
static cudaError_t launch_zsf(const float2* in, float2* dk_out, float2* w_out,
                              const ForceParams& fp, const float2* tw, cudaStream_t s, Multi m) {
  constexpr int TW = ztw(N), T = zt(N);
  constexpr size_t sm = col_smem_tw(N, TW);
  const int64_t ntiles = col_tiles<N, TW>() * m.nb;
  CUtensorMap map{};
  const bool tma = tma_shape<N, TW>() && !m.shift && spectrum_map(map, in, N, TW, true);
  auto go = [&](auto model, auto tma_c) {
    constexpr int MODEL = decltype(model)::value;
    constexpr bool TMA = decltype(tma_c)::value;
    constexpr size_t smk = TMA ? tma_smem<N, fft_rows<N>() * TW, 0>() : sm;
    auto k = k_z_screen_field<N, TW, MODEL, TMA, T>;
    unsigned grid;
    cudaError_t e = prep(k, smk, ntiles, grid, T);
    if (e != cudaSuccess) return e;
    return launch_pdl(dependent_launch(m, N, kDepTransform, s), k, dim3(grid), T, smk, s,
                      OpZScreenField<N, TW, MODEL, T>{geo_z<N, TW>(m), in, dk_out, w_out, fp}, tw, ntiles, map);
  };
  auto pick = [&](auto tma_c) {
    if (fp.model == 1) return go(std::integral_constant<int, 1>{}, tma_c);
    if (fp.filter == 0) return go(std::integral_constant<int, 2>{}, tma_c);
    return go(std::integral_constant<int, 3>{}, tma_c);
  };
  if constexpr (tma_shape<N, TW>()) {
    if (tma) return pick(std::true_type{});
  }
  return pick(std::false_type{});
}

cudaError_t mesh_z_screen_field(int Nv, const float2* in, float2* dk_out, float2* w_out,
                                const ForceParams& fp, const float2* tw, cudaStream_t s, Multi m) {
  if (fp.model != 1 && fp.model != 2) return cudaErrorInvalidValue;
  COLA_SWITCH_N(Nv, return launch_zsf<N>(in, dk_out, w_out, fp, tw, s, m));
  return cudaSuccess;
}

template <int N>
static cudaError_t launch_xscreen(const float2* w_in, const float* rho, float2* s_out,
                                  const ForceParams& fp, const float2* tw, cudaStream_t s, Multi m) {
  constexpr RowShape SH = screen_shape(N);
  constexpr int TWX = SH.rows, T = SH.threads;
  constexpr size_t sm = xscreen_smem<N, TWX>();
  const int64_t tps = (int64_t)N * N / TWX;
  const int64_t ntiles = tps * m.nb;
  unsigned grid;
  if (fp.model == 1) {
    auto k = k_x_screen<N, TWX, T, SH.ctas, 1>;
    cudaError_t e = prep(k, sm, ntiles, grid, T);
    if (e != cudaSuccess) return e;
    k<<<grid, T, sm, s>>>(w_in, rho, s_out, fp, tw, ntiles, m);
  } else {
    auto k = k_x_screen<N, TWX, T, SH.ctas, 2>;
    cudaError_t e = prep(k, sm, ntiles, grid, T);
    if (e != cudaSuccess) return e;
    k<<<grid, T, sm, s>>>(w_in, rho, s_out, fp, tw, ntiles, m);
  }
  return cudaGetLastError();
}

cudaError_t mesh_x_screen_source(int Nv, const float2* w_in, const float* rho, float2* s_out,
                                 const ForceParams& fp, const float2* tw, cudaStream_t s, Multi m) {
  if (fp.model != 1 && fp.model != 2) return cudaErrorInvalidValue;
  COLA_SWITCH_N(Nv, return launch_xscreen<N>(w_in, rho, s_out, fp, tw, s, m));
  return cudaSuccess;
}

template <int N, bool SCR>
static cudaError_t launch_zforce_t(const float2* in, const float2* dk, float2* phi,
                                   float2* phiz, const ForceParams& fp,
                                   const float2* tw, cudaStream_t s, Multi m) {
  constexpr int TW = ztw(N), T = zt(N);
  constexpr size_t sm = zforce_smem<N, TW>();
  const int64_t ntiles = col_tiles<N, TW>() * m.nb;
  CUtensorMap map{}, dmap{};
  const bool tma = tma_shape<N, TW>() && !m.shift && spectrum_map(map, in, N, TW, true) &&
                   (!SCR || spectrum_map(dmap, dk, N, TW, true));
  auto go = [&](auto tma_c) {
    constexpr bool TMA = decltype(tma_c)::value;
    constexpr size_t smk = TMA ? tma_smem<N, fft_rows<N>() * TW, N * TW>() : sm;
    auto k = k_z_force<N, TW, SCR, TMA, T>;
    unsigned grid;
    cudaError_t e = prep(k, smk, ntiles, grid, T);
    if (e != cudaSuccess) return e;
    return launch_pdl(dependent_launch(m, N, kDepTransform, s), k, dim3(grid), T, smk, s,
                      OpZForce<N, TW, SCR, T>{geo_z<N, TW>(m), in, dk, phi, phiz, fp}, tw, ntiles, map, dmap);
  };
  if constexpr (tma_shape<N, TW>()) {
    if (tma) return go(std::true_type{});
  }
  return go(std::false_type{});
}

cudaError_t mesh_z_force(int Nv, const float2* in, const float2* dk, float2* phi_out,
                         float2* phiz_out, const ForceParams& fp, const float2* tw, cudaStream_t s,
                         Multi m) {
  const bool two = fp.screened && fp.model == 1;  // S and delta(k)
  if (two && dk == nullptr) return cudaErrorInvalidValue;
  COLA_SWITCH_N(Nv, return two ? launch_zforce_t<N, true>(in, dk, phi_out, phiz_out, fp, tw, s, m)
                               : launch_zforce_t<N, false>(in, dk, phi_out, phiz_out, fp, tw, s, m));
  return cudaSuccess;
}

template <int N, int PREC>
static cudaError_t launch_lpt_t(const void* p1, const void* p2, float2* o0, float2* o1,
                                float2* o2, float2* o3, const LptParams& lp, const float2* tw,
                                cudaStream_t s, Multi m, float* zero_dst, int64_t zero_floats,
                                bool* zeroed) {
  constexpr int TW = col_tw(N, 4);
  // the zero fill rides along where the pass runs one CTA per SM (N >= 512: room for the
  // 16 KB zero region) on 16-byte aligned memory
  const bool zf = zero_dst && zero_floats > 0 && N >= 512 && (zero_floats % 4) == 0 &&
                  (reinterpret_cast<uintptr_t>(zero_dst) & 15) == 0;
  using Op = OpLptZ<N, TW, PREC>;
  // one simulation at N >= 512 (one CTA per SM either way): the table row also goes to shared
  // memory if it fits there (about 4500 nodes); a longer one is read from global memory
  size_t sm = col_smem<N, 4>() + (zf ? Op::kZero : 0);
  const size_t row = (size_t)lp.nk * sizeof(float4);
  const int tab_smem = N >= 512 && !m.shift && sm + row <= smem_most() ? 1 : 0;
  if (tab_smem) sm += row;
  const int64_t ntiles = col_tiles<N, TW>() * m.nb;
  auto k = k_lpt_z<N, TW, PREC>;
  unsigned grid;
  cudaError_t e = prep(k, sm, ntiles, grid);
  if (e != cudaSuccess) return e;
  Op op{geo_z<N, TW>(m), p1, p2, o0, o1, o2, o3, lp, tab_smem};
  if (zf) {
    op.zdst = reinterpret_cast<char*>(zero_dst);
    op.zbytes = zero_floats * (int64_t)sizeof(float);
    const int64_t tps = col_tiles<N, TW>();
    op.zchunk = ((op.zbytes + tps - 1) / tps + 15) / 16 * 16;
  }
  e = launch_pdl(dependent_launch(m, N, kDepTransform, s), k, dim3(grid), NT, sm, s, op, tw, ntiles);
  if (e == cudaSuccess && zeroed) *zeroed = zf;
  return e;
}

template <int N, int PREC>
static cudaError_t launch_lpt8(const void* p1, const void* p2, float2* o0, float2* o1, float2* o2, float2* o3,
                               const LptParams& lp, const float2* tw, cudaStream_t s, Multi m) {
  const size_t sm = LptZ8<N>::smem;
  const int64_t ntiles = col_tiles<N, 8>() * m.nb;
  auto k = k_lpt_z8<N, PREC>;
  unsigned grid;
  cudaError_t e = prep(k, sm, ntiles, grid);
  if (e != cudaSuccess) return e;
  k<<<grid, NT, sm, s>>>(geo_z<N, 8>(m), static_cast<const uint32_t*>(p1), static_cast<const uint32_t*>(p2), o0, o1,
                         o2, o3, lp, tw, ntiles);
  return cudaGetLastError();
}
template <int N>
static cudaError_t launch_lptr(const void* p1, const void* p2, float2* o0, float2* o1, float2* o2, float2* o3,
                               const LptParams& lp, const float2* tw, cudaStream_t s, Multi m) {
  constexpr size_t sm = LptZr<N>::smem;
  constexpr int TW = LptZr<N>::TW, T = LptZr<N>::T;
  const int64_t ntiles = col_tiles<N, TW>() * m.nb;
  auto k = k_lpt_zr<N>;
  unsigned grid;
  cudaError_t e = prep(k, sm, ntiles, grid, T);
  if (e != cudaSuccess) return e;
  return launch_pdl(dependent_launch(m, N, kDepTransform, s), k, dim3(grid), T, sm, s, geo_z<N, TW>(m),
                    static_cast<const float2*>(p1), static_cast<const float2*>(p2), o0, o1, o2, o3, lp, tw, ntiles);
}
template <int N>
static cudaError_t launch_lpt(const void* p1, const void* p2, float2* o0, float2* o1, float2* o2,
                              float2* o3, const LptParams& lp, const float2* tw,
                              cudaStream_t s, Multi m, float* zd, int64_t zn, bool* zeroed) {
  // 16-bit seeds, ms per launch with 4-column tiles (k_lpt_z) -> 8-column tiles: N = 256 0.180 ->
  // 0.143, N = 512 1.55 -> 1.44 (FP32 seeds at 512 the other way, 1.40 -> 1.46)
  if constexpr (N == 256 || N == 512) {
    if (lp.seed_prec == 1) return launch_lpt8<N, 1>(p1, p2, o0, o1, o2, o3, lp, tw, s, m);
    if (lp.seed_prec == 2) return launch_lpt8<N, 2>(p1, p2, o0, o1, o2, o3, lp, tw, s, m);
  }
  if (lp.seed_prec == 1) return launch_lpt_t<N, 1>(p1, p2, o0, o1, o2, o3, lp, tw, s, m, zd, zn, zeroed);
  if (lp.seed_prec == 2) return launch_lpt_t<N, 2>(p1, p2, o0, o1, o2, o3, lp, tw, s, m, zd, zn, zeroed);
  if constexpr (N <= 256) {
    // three tiles and more per resident CTA (4 per SM), or the short chain of k_lpt_z
    if (N == 256 || col_tiles<N, LptZr<N>::TW>() * m.nb >= 12 * (int64_t)sm_count())
      return launch_lptr<N>(p1, p2, o0, o1, o2, o3, lp, tw, s, m);
  }
  if constexpr (N != 256) return launch_lpt_t<N, 0>(p1, p2, o0, o1, o2, o3, lp, tw, s, m, zd, zn, zeroed);
  else return cudaErrorInvalidValue;
}

cudaError_t lpt_z(int Nv, const void* phi1, const void* phi2, float2* o0, float2* o1, float2* o2,
                  float2* o3, const LptParams& lp, const float2* tw, cudaStream_t s, Multi m,
                  float* zero_dst, int64_t zero_floats, bool* zeroed) {
  if (zeroed) *zeroed = false;
  if (Nv > 512) return cudaErrorInvalidValue;  // four double-buffered 4-column tiles exceed shared memory
  COLA_SWITCH_N(Nv, return launch_lpt<N>(phi1, phi2, o0, o1, o2, o3, lp, tw, s, m, zero_dst, zero_floats, zeroed));
  return cudaSuccess;
}

template <int N>
static cudaError_t launch_plane_r2c(const float* in, float2* out, float scale, float offset,
                                    const float2* tw, cudaStream_t s, Multi m) {
  if constexpr (N > 128) {
    return cudaErrorInvalidValue;
  } else {
    constexpr size_t sm = PlaneCfg<N>::smem;
    auto k = k_plane_r2c<N>;
    if (sm > 48 * 1024) {
      cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
      if (e != cudaSuccess) return e;
    }
    return launch_pdl(dependent_launch(m, N, kDepTransform, s), k, dim3(N, m.nb), NT, sm, s, in, out, scale, offset, tw, m);
  }
}

cudaError_t fft_plane_r2c(int Nv, const float* in, float2* out, float scale, float offset, const float2* tw,
                          cudaStream_t s, Multi m) {
  COLA_SWITCH_N(Nv, return launch_plane_r2c<N>(in, out, scale, offset, tw, s, m));
  return cudaSuccess;
}

template <int N, bool HERM>
static cudaError_t launch_plane_grad(const PlaneJobs& jobs, const float2* tw, cudaStream_t s, Multi m) {
  if constexpr (N > 128) {
    return cudaErrorInvalidValue;
  } else {
    constexpr size_t sm = PlaneCfg<N>::smem;
    auto k = k_plane_grad<N, HERM>;
    if (sm > 48 * 1024) {
      cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
      if (e != cudaSuccess) return e;
    }
    return launch_pdl(dependent_launch(m, N, kDepTransform, s), k, dim3(jobs.n * N, m.nb), NT, sm, s, jobs, tw, m);
  }
}

template <bool HERM>
static cudaError_t plane_grad(int Nv, const PlaneJobs& jobs, const float2* tw, cudaStream_t s, Multi m) {
  if (jobs.n < 1 || jobs.n > 6) return cudaErrorInvalidValue;
  COLA_SWITCH_N(Nv, return launch_plane_grad<N, HERM>(jobs, tw, s, m));
  return cudaSuccess;
}

cudaError_t fft_plane_force(int Nv, const float2* phi, const float2* phiz, float* fx, float* fy, float* fz,
                            float kfs, const float2* tw, cudaStream_t s, Multi m) {
  const PlaneJobs jobs{{phi, phi, phiz}, {fx, fy, fz}, 3, 1, 2, kfs};
  return plane_grad<true>(Nv, jobs, tw, s, m);
}

cudaError_t fft_plane_lpt(int Nv, const float2* const* lc, float* const* out, float kfs, const float2* tw,
                          cudaStream_t s, Multi m, float* zero_dst, int64_t zero_floats, bool* zeroed) {
  PlaneJobs jobs{{lc[0], lc[0], lc[1], lc[2], lc[2], lc[3]},
                 {out[0], out[1], out[2], out[3], out[4], out[5]},
                 6,
                 0b001001,
                 0b010010,
                 kfs};
  const bool zf = zero_dst && zero_floats > 0 && (zero_floats % 4) == 0 &&
                  (reinterpret_cast<uintptr_t>(zero_dst) & 15) == 0;
  if (zf) {
    const int64_t ctas = (int64_t)jobs.n * Nv;
    jobs.zdst = zero_dst;
    jobs.zfloats = zero_floats;
    jobs.zchunk = (zero_floats + 4 * ctas - 1) / (4 * ctas) * 4;
  }
  const cudaError_t e = plane_grad<false>(Nv, jobs, tw, s, m);
  if (e == cudaSuccess && zeroed) *zeroed = zf;
  return e;
}

template <int N>
static cudaError_t launch_plane_screen(const float2* w_in, const float* rho, float2* s_out,
                                       const ForceParams& fp, const float2* tw, cudaStream_t s, Multi m) {
  if constexpr (N > 128) {
    return cudaErrorInvalidValue;
  } else {
    constexpr size_t sm = PlaneCfg<N>::smem;
    auto k = fp.model == 1 ? k_plane_screen<N, 1> : k_plane_screen<N, 2>;
    if (sm > 48 * 1024) {
      cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
      if (e != cudaSuccess) return e;
    }
    return launch_pdl(dependent_launch(m, N, kDepTransform, s), k, dim3(N, m.nb), NT, sm, s, w_in, rho, s_out, fp, tw, m);
  }
}

cudaError_t fft_plane_screen(int Nv, const float2* w_in, const float* rho, float2* s_out, const ForceParams& fp,
                             const float2* tw, cudaStream_t s, Multi m) {
  if (fp.model != 1 && fp.model != 2) return cudaErrorInvalidValue;
  COLA_SWITCH_N(Nv, return launch_plane_screen<N>(w_in, rho, s_out, fp, tw, s, m));
  return cudaSuccess;
}

cudaError_t wait_probe(double seconds, int* timed_out) {
  if (!(seconds > 0) || seconds > 10) return cudaErrorInvalidValue;
  k_wait_probe<<<1, 32, 0, cudaStreamPerThread>>>((uint64_t)(seconds * 1e9));
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess)
    e = cudaMemcpyFromSymbolAsync(timed_out, g_wait_probe, sizeof(int), 0, cudaMemcpyDeviceToHost,
                                  cudaStreamPerThread);
  if (e == cudaSuccess) e = cudaStreamSynchronize(cudaStreamPerThread);
  return e;
}

cudaError_t tile_load_failures(unsigned* dst, cudaStream_t s) {
  return cudaMemcpyFromSymbolAsync(dst, g_tile_load_failures, sizeof(unsigned), 0, cudaMemcpyDeviceToHost, s);
}

}  // namespace cola
