// Shared-memory FFT building blocks for sm_103a.
//
// A tile of TW independent columns of length L (power of two) lives in shared
// memory as buf[n * PITCH + c] (float2, c = column, n = element).  A transform
// is two in-register DFT passes of radix R1, R2 <= 32 (L = R1 R2, the
// "four-step" factorisation) with one twiddle multiplication between them, so
// each element makes two round trips through shared memory.  Consecutive
// threads handle consecutive columns.
//
// Twiddles come from a table tw[m] = exp(-2 pi i m / T) of the tile's transform
// table length T (host-computed in double precision, rounded to float); a
// length-L transform reads it with stride T / L.  INV selects exp(+...) (the
// unnormalised inverse).
//
// The in-register DFTs are radix-2 decimation in time (inputs in bit-reversed
// positions, placed there at compile time by the loads; outputs in natural
// order): a twiddled butterfly a +- w b is two fused multiply-adds per component
// for a + w b and one for 2a - (a + w b), issued as paired (two-component)
// FMAs; the decimation-in-frequency form (subtract, then multiply by w) takes
// more.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace cola {

// Additions, subtractions and scalings of complex values use the paired
// single-precision instructions of this architecture (two components per
// instruction, each rounded exactly as the scalar operation).  The complex
// multiply stays scalar: its paired form (a multiply and an FMA on swapped
// operands) measured no faster.
__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 csub(float2 a, float2 b) { return __fadd2_rn(a, make_float2(-b.x, -b.y)); }
__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
  return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
// a conj(w) with the roundings spelled out
__device__ __forceinline__ float2 cmul_conj(float2 a, float2 w) {
  return make_float2(fmaf(a.x, w.x, a.y * w.y), fmaf(a.y, w.x, -(a.x * w.y)));
}
__device__ __forceinline__ float2 cconj(float2 a) { return make_float2(a.x, -a.y); }
__device__ __forceinline__ float2 cscale(float2 a, float s) { return __fmul2_rn(a, make_float2(s, s)); }
// multiply by +i
__device__ __forceinline__ float2 cmul_i(float2 a) { return make_float2(-a.y, a.x); }
// i f a, each product rounded on its own.  cscale(cmul_i(a), f) may fuse with the additions
// of a transform that follows; this gives the value that a product stored in a pass of its
// own has (the LPT fields depend on it bit for bit where they are kept in 16 bits).
__device__ __forceinline__ float2 cmul_if(float2 a, float f) {
  return make_float2(__fmul_rn(-f, a.y), __fmul_rn(f, a.x));
}
// multiply by -i (forward) or +i (inverse)
template <bool INV>
__device__ __forceinline__ float2 rot_q(float2 a) {
  return INV ? make_float2(-a.y, a.x) : make_float2(a.y, -a.x);
}

template <bool INV>
__device__ __forceinline__ void dft2(float2& a, float2& b) {
  float2 t = a;
  a = cadd(t, b);
  b = csub(t, b);
}

template <bool INV>
__device__ __forceinline__ void dft4(float2& v0, float2& v1, float2& v2, float2& v3) {
  float2 t0 = cadd(v0, v2), t1 = csub(v0, v2), t2 = cadd(v1, v3), t3 = rot_q<INV>(csub(v1, v3));
  v0 = cadd(t0, t2);
  v2 = csub(t0, t2);
  v1 = cadd(t1, t3);
  v3 = csub(t1, t3);
}

// cos(2 pi m / 32) for m = 0..8 (standard values; sin(2 pi m/32) = cos32(8 - m)).
__host__ __device__ constexpr float cos32(int m) {
  return m == 0 ? 1.0f
       : m == 1 ? 0.98078528040323044913f
       : m == 2 ? 0.92387953251128675613f
       : m == 3 ? 0.83146961230254523708f
       : m == 4 ? 0.70710678118654752440f
       : m == 5 ? 0.55557023301960222474f
       : m == 6 ? 0.38268343236508977173f
       : m == 7 ? 0.19509032201612826785f
       : 0.0f;
}

// a * exp(-/+ 2 pi i m / 32), m in [0, 16) a compile-time constant after unrolling.
template <bool INV>
__device__ __forceinline__ float2 w32mul(float2 a, int m) {
  if (m == 0) return a;
  if (m == 8) return rot_q<INV>(a);
  const float c = m <= 8 ? cos32(m) : -cos32(16 - m);
  const float s = m <= 8 ? cos32(8 - m) : cos32(m - 8);
  return INV ? make_float2(a.x * c - a.y * s, a.y * c + a.x * s)
             : make_float2(a.x * c + a.y * s, a.y * c - a.x * s);
}

// Decimation-in-time butterfly (a, b) <- (a + w b, a - w b) with
// w = exp(-/+ 2 pi i m / 32), m in [0, 16) a compile-time constant after
// unrolling: m = 0 and 8 are additions, the others two paired FMAs for a + w b
// and one for 2a - (a + w b) (the same per-component FMAs as the scalar form).
template <bool INV>
__device__ __forceinline__ void bfly_tw(float2& a, float2& b, int m) {
  if (m == 0) {
    dft2<INV>(a, b);
    return;
  }
  if (m == 8) {
    const float2 wb = rot_q<INV>(b), t = a;
    a = cadd(t, wb);
    b = csub(t, wb);
    return;
  }
  const float c = m <= 8 ? cos32(m) : -cos32(16 - m);
  const float s = m <= 8 ? cos32(8 - m) : cos32(m - 8);  // sin(2 pi m / 32) >= 0
  // forward w b = (c br + s bi, c bi - s br); inverse (c br - s bi, c bi + s br)
  const float sg = INV ? -s : s;
  // x = (c br + (sg bi + ar), c bi + (-sg br + ai)), b <- 2a - x: paired FMAs
  const float2 t = __ffma2_rn(make_float2(sg, -sg), make_float2(b.y, b.x), a);
  const float2 x = __ffma2_rn(make_float2(c, c), b, t);
  b = __ffma2_rn(make_float2(2.f, 2.f), a, make_float2(-x.x, -x.y));
  a = x;
}

// 8-point DFT, natural order in and out: two 4-point DFTs of the even and odd
// inputs and one decimation-in-time layer.
template <bool INV>
__device__ __forceinline__ void dft8(float2* v) {
  float2 e0 = v[0], e1 = v[2], e2 = v[4], e3 = v[6];
  float2 o0 = v[1], o1 = v[3], o2 = v[5], o3 = v[7];
  dft4<INV>(e0, e1, e2, e3);
  dft4<INV>(o0, o1, o2, o3);
  bfly_tw<INV>(e0, o0, 0);
  bfly_tw<INV>(e1, o1, 4);
  bfly_tw<INV>(e2, o2, 8);
  bfly_tw<INV>(e3, o3, 12);
  v[0] = e0;
  v[1] = e1;
  v[2] = e2;
  v[3] = e3;
  v[4] = o0;
  v[5] = o1;
  v[6] = o2;
  v[7] = o3;
}

// In-register DFT of R = 2..32 points on the strided view v[0], v[S], ...,
// v[(R-1)S], in place.  R <= 8: natural order.  R = 16, 32: radix-2
// decimation in time, so input n must sit at position pos_of<R>(n) (placed
// there at compile time by the caller) and output k ends at position k.
template <int R>
__host__ __device__ constexpr int pos_of(int n) {
  if constexpr (R <= 8) {
    return n;
  } else {
    return (n % 2 == 0) ? pos_of<R / 2>(n / 2) : R / 2 + pos_of<R / 2>((n - 1) / 2);
  }
}

template <bool INV, int S>
__device__ __forceinline__ void dft8s(float2* v) {
  float2 t[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) t[i] = v[i * S];
  dft8<INV>(t);
#pragma unroll
  for (int i = 0; i < 8; ++i) v[i * S] = t[i];
}

template <int R, bool INV, int S = 1>
__device__ __forceinline__ void dftR(float2* v) {
  if constexpr (R == 1) {
  } else if constexpr (R == 2) {
    dft2<INV>(v[0], v[S]);
  } else if constexpr (R == 4) {
    dft4<INV>(v[0], v[S], v[2 * S], v[3 * S]);
  } else if constexpr (R == 8) {
    dft8s<INV, S>(v);
  } else {
    static_assert(R == 16 || R == 32, "radix");
    // even inputs in the first half, odd in the second (pos_of), each half a
    // DFT of R / 2 points in natural order, then one butterfly layer
    dftR<R / 2, INV, S>(v);
    dftR<R / 2, INV, S>(v + (R / 2) * S);
#pragma unroll
    for (int k = 0; k < R / 2; ++k) bfly_tw<INV>(v[k * S], v[(k + R / 2) * S], k * (32 / R));
  }
}

// 32-point DFT shared by a thread pair (lanes l and l ^ 16 of a full warp):
// the thread with half = 0 holds x[0..15] in v, its partner x[16..31].  One
// radix-2 decimation-in-frequency step exchanges the halves by shuffle (half 0
// forms a[n] = x[n] + x[n + 16], half 1 b[n] = (x[n] - x[n + 16]) w32^n), then
// each runs a 16-point DFT: half h ends with X[2k + h] at v[k].
template <bool INV>
__device__ __forceinline__ void dft32_pair(float2 (&v)[16], int half) {
  const float sg = half ? -1.f : 1.f;
  float2 u[16];
#pragma unroll
  for (int n = 0; n < 16; ++n) {
    const float ox = __shfl_xor_sync(0xffffffffu, v[n].x, 16);
    const float oy = __shfl_xor_sync(0xffffffffu, v[n].y, 16);
    const float2 t = make_float2(fmaf(sg, v[n].x, ox), fmaf(sg, v[n].y, oy));
    const float2 tw = w32mul<INV>(t, n);
    u[pos_of<16>(n)] = half ? tw : t;
  }
  dftR<16, INV>(u);
#pragma unroll
  for (int k = 0; k < 16; ++k) v[k] = u[k];
}

__host__ __device__ constexpr int ilog2(int n) { return n <= 1 ? 0 : 1 + ilog2(n / 2); }

// L = R1 R2 with R1 <= R2 <= 32.
template <int L>
struct Split {
  static constexpr int p = ilog2(L);
  static constexpr int R1 = 1 << (p / 2);
  static constexpr int R2 = L / R1;
  static_assert(R2 <= 32 && R1 * R2 == L, "transform length");
};

// Rows of shared memory a length-L column-tile transform needs: L, plus R2
// padding rows for the intermediate.
template <int L>
__host__ __device__ constexpr int fft_rows() {
  return L + Split<L>::R2;
}

// Length-L transform of the TW columns of a shared-memory tile (four-step):
// step 1: for each n2 < R2, DFT_R1 over x[R2 n1 + n2], times w_L^(n2 k1);
// step 2: for each k1 < R1, DFT_R2 over n2 gives X[k1 + R1 k2].
// The intermediate Y[n2][k1] goes to row n2 (R1 + 1) + k1, one padding row
// per R1 (the tile needs fft_rows<L>() rows): with a row pitch that is a
// multiple of 8 the 16 lanes of a half-warp hit 16 different bank pairs, and
// every address is a per-thread base plus a compile-time offset.  tw has
// L * TWS entries; the caller synchronises before the call; returns after a
// barrier.
//
// Hooks (defaults: the tile itself): step 1 reads element n of column c as
// ld(buf, n, c, at) and step 2 writes X[n] as st(X[n], n, c, at), at = n PITCH
// + c, so a k-space operation fuses into the first load or the last store
// (reading or writing another array at the same offset).  A store hook with
// kSmem = false writes the outputs itself (e.g. straight to HBM) and the tile
// is left holding the intermediate.
struct TileLoad {
  __device__ __forceinline__ float2 operator()(const float2* buf, int, int, int at) const { return buf[at]; }
};
struct TileStore {
  static constexpr bool kSmem = true;
  __device__ __forceinline__ float2 operator()(float2 v, int, int, int) const { return v; }
};

template <int L, int TW, int PITCH, int NT, bool INV, int TWS = 1, class Load = TileLoad,
          class Store = TileStore>
__device__ __forceinline__ void fft_tile(float2* __restrict__ buf, const float2* __restrict__ tw,
                                         Load ld = Load(), Store st = Store()) {
  constexpr int R1 = Split<L>::R1, R2 = Split<L>::R2;
  constexpr int U1 = TW * R2, P1 = (U1 + NT - 1) / NT;
  constexpr int U2 = TW * R1, P2 = (U2 + NT - 1) / NT;
  static_assert(PITCH % 8 == 0, "column tiles: row pitch a multiple of 8");
  const int tid = threadIdx.x;
  {
    float2 v[P1][R1];
#pragma unroll
    for (int i = 0; i < P1; ++i) {
      const int u = tid + i * NT;
      if ((U1 % NT) == 0 || u < U1) {
        const int c = u % TW, n2 = u / TW;
#pragma unroll
        for (int n1 = 0; n1 < R1; ++n1)
          v[i][pos_of<R1>(n1)] = ld(buf, R2 * n1 + n2, c, (R2 * n1 + n2) * PITCH + c);
        dftR<R1, INV>(v[i]);
        if (n2 > 0) {
#pragma unroll
          for (int k1 = 1; k1 < R1; ++k1) {
            float2 w = tw[n2 * k1 * TWS];
            if (INV) w.y = -w.y;
            v[i][k1] = cmul(v[i][k1], w);
          }
        }
      }
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < P1; ++i) {
      const int u = tid + i * NT;
      if ((U1 % NT) == 0 || u < U1) {
        const int c = u % TW, n2 = u / TW;
        float2* y = buf + n2 * (R1 + 1) * PITCH + c;
#pragma unroll
        for (int k1 = 0; k1 < R1; ++k1) y[k1 * PITCH] = v[i][k1];
      }
    }
  }
  __syncthreads();
  {
    float2 y[P2][R2];
#pragma unroll
    for (int i = 0; i < P2; ++i) {
      const int u = tid + i * NT;
      if ((U2 % NT) == 0 || u < U2) {
        const int c = u % TW, k1 = u / TW;
        const float2* yr = buf + k1 * PITCH + c;
#pragma unroll
        for (int n2 = 0; n2 < R2; ++n2) y[i][pos_of<R2>(n2)] = yr[n2 * (R1 + 1) * PITCH];
        dftR<R2, INV>(y[i]);
      }
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < P2; ++i) {
      const int u = tid + i * NT;
      if ((U2 % NT) == 0 || u < U2) {
        const int c = u % TW, k1 = u / TW;
#pragma unroll
        for (int k2 = 0; k2 < R2; ++k2) {
          const int n = k1 + R1 * k2;
          const float2 o = st(y[i][k2], n, c, n * PITCH + c);
          if constexpr (Store::kSmem) buf[n * PITCH + c] = o;
        }
      }
    }
  }
  __syncthreads();
}

// A forward transform whose outputs feed an inverse one (the k-space operations of
// the z passes) stays in registers in between: after step 2 thread (c, k1) holds
// X[k1 + R1 k2], and those are the inputs n = n2 + R2' n1 of the inverse
// transform's first-step items n2 = k1 + R1 h, h < R2' / R1 (R1', R2' its split).
// So the operation, the inverse's first DFTs and their twiddles follow on the
// same registers: per point and warp 8 shared-memory wavefronts for the two
// transforms instead of 12 (16 with the operation in a pass of its own), and 5
// barriers instead of 8.  Screening-field pass 2.85 -> 2.35 ms at 1024^3.

// Radix of the forward transform's first step: the split's own, or the larger of
// the two where the middle would otherwise have fewer items than threads.
template <int L, int TW, int NT>
__host__ __device__ constexpr int fused_r1() {
  return Split<L>::R1 < Split<L>::R2 && TW * Split<L>::R1 < NT ? Split<L>::R2 : Split<L>::R1;
}

// Step 1 of a column transform (split R1 x R2) up to its intermediate in the tile;
// the caller synchronises before step 2.
template <int R1, int R2, int TW, int PITCH, int NT, bool INV, class Load>
__device__ __forceinline__ void col_step1(float2* __restrict__ buf, const float2* __restrict__ tw, Load ld) {
  constexpr int U = TW * R2, P = (U + NT - 1) / NT;
  float2 v[P][R1];
#pragma unroll
  for (int i = 0; i < P; ++i) {
    const int u = threadIdx.x + i * NT;
    if ((U % NT) == 0 || u < U) {
      const int c = u % TW, n2 = u / TW;
#pragma unroll
      for (int n1 = 0; n1 < R1; ++n1)
        v[i][pos_of<R1>(n1)] = ld(buf, R2 * n1 + n2, c, (R2 * n1 + n2) * PITCH + c);
      dftR<R1, INV>(v[i]);
      if (n2 > 0) {
#pragma unroll
        for (int k1 = 1; k1 < R1; ++k1) {
          float2 w = tw[n2 * k1];
          if (INV) w.y = -w.y;
          v[i][k1] = cmul(v[i][k1], w);
        }
      }
    }
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < P; ++i) {
    const int u = threadIdx.x + i * NT;
    if ((U % NT) == 0 || u < U) {
      const int c = u % TW, n2 = u / TW;
      float2* y = buf + n2 * (R1 + 1) * PITCH + c;
#pragma unroll
      for (int k1 = 0; k1 < R1; ++k1) y[k1 * PITCH] = v[i][k1];
    }
  }
}

// Step 2 of the forward transform: the item's X[k1 + R1 k2] into y[k2].
template <int R1, int R2, int PITCH>
__device__ __forceinline__ void col_fwd2(float2 (&y)[R2], const float2* __restrict__ buf, int c, int k1) {
  const float2* yr = buf + k1 * PITCH + c;
#pragma unroll
  for (int n2 = 0; n2 < R2; ++n2) y[pos_of<R2>(n2)] = yr[n2 * (R1 + 1) * PITCH];
  dftR<R2, false>(y);
}

// First step of the inverse transform (split IR1 x IR2) on the R2 forward outputs x
// of item (c, k1): the intermediate's values into v (items h = 0.., IR1 each).
template <int R1, int R2, int IR1, int IR2>
__device__ __forceinline__ void col_inv1(float2 (&v)[R2], const float2 (&x)[R2], const float2* __restrict__ tw,
                                         int k1) {
  constexpr int H = IR2 / R1;
  static_assert(IR2 % R1 == 0 && H * IR1 == R2, "splits");
#pragma unroll
  for (int h = 0; h < H; ++h) {
    float2 t[IR1];
#pragma unroll
    for (int n1 = 0; n1 < IR1; ++n1) t[pos_of<IR1>(n1)] = x[h + H * n1];
    dftR<IR1, true>(t);
    const int n2 = k1 + R1 * h;
    v[h * IR1] = t[0];
#pragma unroll
    for (int k = 1; k < IR1; ++k) v[h * IR1 + k] = n2 > 0 ? cmul(t[k], cconj(tw[n2 * k])) : t[k];
  }
}

// ... and from v into the tile (intermediate rows n2 (IR1 + 1) + k).
template <int R1, int R2, int IR1, int IR2, int PITCH>
__device__ __forceinline__ void col_inv1_store(float2* __restrict__ buf, const float2 (&v)[R2], int c, int k1) {
#pragma unroll
  for (int h = 0; h < IR2 / R1; ++h) {
    float2* y = buf + (k1 + R1 * h) * (IR1 + 1) * PITCH + c;
#pragma unroll
    for (int k = 0; k < IR1; ++k) y[k * PITCH] = v[h * IR1 + k];
  }
}

// Last step of an inverse transform from the tile's intermediate to the store hook
// (one that writes the outputs itself); no barrier.
template <int R1, int R2, int TW, int PITCH, int NT, class Store>
__device__ __forceinline__ void col_inv2(const float2* __restrict__ buf, Store st) {
  static_assert(!Store::kSmem, "outputs leave from registers");
  constexpr int U = TW * R1, P = (U + NT - 1) / NT;
#pragma unroll
  for (int i = 0; i < P; ++i) {
    const int u = threadIdx.x + i * NT;
    if ((U % NT) == 0 || u < U) {
      const int c = u % TW, k1 = u / TW;
      const float2* yr = buf + k1 * PITCH + c;
      float2 y[R2];
#pragma unroll
      for (int n2 = 0; n2 < R2; ++n2) y[pos_of<R2>(n2)] = yr[n2 * (R1 + 1) * PITCH];
      dftR<R2, true>(y);
#pragma unroll
      for (int k2 = 0; k2 < R2; ++k2) {
        const int n = k1 + R1 * k2;
        st(y[k2], n, c, n * PITCH + c);
      }
    }
  }
}

// Forward transform of the tile's TW columns, x = mid(X[n], n, c, at) on every value,
// inverse transform of x to st.  The caller synchronises before the call and before it reuses the tile.
template <int L, int TW, int PITCH, int NT, class Mid, class Store>
__device__ __forceinline__ void fft_tile_fwd_inv(float2* __restrict__ buf, const float2* __restrict__ tw, Mid mid,
                                                 Store st) {
  constexpr int R1 = fused_r1<L, TW, NT>(), R2 = L / R1, IR1 = Split<L>::R1, IR2 = Split<L>::R2;
  constexpr int U = TW * R1, P = (U + NT - 1) / NT;
  static_assert(PITCH % 4 == 0, "column tiles: row pitch a multiple of 4");
  col_step1<R1, R2, TW, PITCH, NT, false>(buf, tw, TileLoad{});
  __syncthreads();
  float2 v[P][R2];
#pragma unroll
  for (int i = 0; i < P; ++i) {
    const int u = threadIdx.x + i * NT;
    if ((U % NT) == 0 || u < U) {
      const int c = u % TW, k1 = u / TW;
      float2 y[R2];
      col_fwd2<R1, R2, PITCH>(y, buf, c, k1);
#pragma unroll
      for (int k2 = 0; k2 < R2; ++k2) y[k2] = mid(y[k2], k1 + R1 * k2, c, (k1 + R1 * k2) * PITCH + c);
      col_inv1<R1, R2, IR1, IR2>(v[i], y, tw, k1);
    }
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < P; ++i) {
    const int u = threadIdx.x + i * NT;
    if ((U % NT) == 0 || u < U) col_inv1_store<R1, R2, IR1, IR2, PITCH>(buf, v[i], u % TW, u / TW);
  }
  __syncthreads();
  col_inv2<IR1, IR2, TW, PITCH, NT>(buf, st);
}

// The same with two inverse transforms, of x = mid(X) to st and of grad(x, n) to st2, one
// after the other; x stays in registers in between.  mid.ready() runs in every thread before
// the barrier ahead of mid, after() once all of mid's reads are done.
template <int L, int TW, int PITCH, int NT, class Mid, class Grad, class After, class Store>
__device__ __forceinline__ void fft_tile_fwd_inv2(float2* __restrict__ buf, const float2* __restrict__ tw, Mid mid,
                                                  Grad grad, After after, Store st, Store st2) {
  constexpr int R1 = fused_r1<L, TW, NT>(), R2 = L / R1, IR1 = Split<L>::R1, IR2 = Split<L>::R2;
  constexpr int U = TW * R1;
  static_assert(PITCH % 4 == 0, "column tiles: row pitch a multiple of 4");
  static_assert(U <= NT, "one middle item per thread");
  col_step1<R1, R2, TW, PITCH, NT, false>(buf, tw, TileLoad{});
  mid.ready();
  __syncthreads();
  const int c = threadIdx.x % TW, k1 = threadIdx.x / TW;
  const bool on = U == NT || threadIdx.x < U;
  float2 x[R2], v[R2];
  if (on) {
    col_fwd2<R1, R2, PITCH>(x, buf, c, k1);
#pragma unroll
    for (int k2 = 0; k2 < R2; ++k2) x[k2] = mid(x[k2], k1 + R1 * k2, c, (k1 + R1 * k2) * PITCH + c);
    col_inv1<R1, R2, IR1, IR2>(v, x, tw, k1);
  }
  __syncthreads();
  after();
  if (on) col_inv1_store<R1, R2, IR1, IR2, PITCH>(buf, v, c, k1);
  __syncthreads();
  col_inv2<IR1, IR2, TW, PITCH, NT>(buf, st);
  if (on) {
#pragma unroll
    for (int k2 = 0; k2 < R2; ++k2) x[k2] = grad(x[k2], k1 + R1 * k2);
    col_inv1<R1, R2, IR1, IR2>(v, x, tw, k1);
  }
  __syncthreads();
  if (on) col_inv1_store<R1, R2, IR1, IR2, PITCH>(buf, v, c, k1);
  __syncthreads();
  col_inv2<IR1, IR2, TW, PITCH, NT>(buf, st2);
}

// Inverse transforms of the tile's columns to st and of i kfs f_n times them (f_n the
// signed frequency, zero on the Nyquist row) to st2.  The first step reads each value
// once and forms both transforms' intermediates, the derivative's in buf2
// (fft_rows<L>() rows, free).  The caller synchronises before the call and before it
// reuses the buffers.
template <int L, int TW, int PITCH, int NT, class Store>
__device__ __forceinline__ void fft_tile_inv_deriv(float2* __restrict__ buf, float2* __restrict__ buf2,
                                                   const float2* __restrict__ tw, float kfs, Store st, Store st2) {
  constexpr int R1 = Split<L>::R1, R2 = Split<L>::R2;
  constexpr int U = TW * R2, P = (U + NT - 1) / NT;
  static_assert(PITCH % 8 == 0, "column tiles: row pitch a multiple of 8");
  float2 v[P][R1];
#pragma unroll
  for (int i = 0; i < P; ++i) {
    const int u = threadIdx.x + i * NT;
    if ((U % NT) == 0 || u < U) {
      const int c = u % TW, n2 = u / TW;
      float2 d[R1];
#pragma unroll
      for (int n1 = 0; n1 < R1; ++n1) {
        const int n = R2 * n1 + n2;
        const float2 x = buf[n * PITCH + c];
        const float f = n == L / 2 ? 0.f : kfs * (float)(n < L / 2 ? n : n - L);
        v[i][pos_of<R1>(n1)] = x;
        d[pos_of<R1>(n1)] = cmul_if(x, f);
      }
      dftR<R1, true>(d);
      dftR<R1, true>(v[i]);
      if (n2 > 0) {
#pragma unroll
        for (int k1 = 1; k1 < R1; ++k1) {
          const float2 w = tw[n2 * k1];
          d[k1] = cmul_conj(d[k1], w);
          v[i][k1] = cmul_conj(v[i][k1], w);
        }
      }
      float2* y = buf2 + n2 * (R1 + 1) * PITCH + c;
#pragma unroll
      for (int k1 = 0; k1 < R1; ++k1) y[k1 * PITCH] = d[k1];
    }
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < P; ++i) {
    const int u = threadIdx.x + i * NT;
    if ((U % NT) == 0 || u < U) {
      float2* y = buf + u / TW * (R1 + 1) * PITCH + u % TW;
#pragma unroll
      for (int k1 = 0; k1 < R1; ++k1) y[k1 * PITCH] = v[i][k1];
    }
  }
  __syncthreads();
  col_inv2<R1, R2, TW, PITCH, NT>(buf, st);
  col_inv2<R1, R2, TW, PITCH, NT>(buf2, st2);
}

// Row pitch (complex values) of a row-major tile transformed in place by
// fft_rowtile<L>: at least L + R2 - 1 (room for the padded intermediate) and
// 8 mod 16, so that the half-warps of both steps hit distinct bank pairs.
template <int L>
__host__ __device__ constexpr int rowtile_pitch() {
  return ((L + Split<L>::R2 - 1 - 8 + 15) / 16) * 16 + 8;
}

// Load hook of fft_rowtile's first step: element n of row c as pre(x, c, n).
struct NoPre {
  __device__ __forceinline__ float2 operator()(float2 v, int, int) const { return v; }
};

// Length-L transforms of the TW rows of a row-major shared-memory tile, in
// place: row c holds x[n] at buf[c * CW + n] (CW = rowtile_pitch<L>()).  Same
// four-step factorisation as fft_tile, with the element index as the fast
// thread index (consecutive lanes touch consecutive elements of one row):
// step 1 (thread = (c, n2)): DFT_R1 over x[R2 n1 + n2] (each value passed
// through pre() as it is loaded), times w_L^(n2 k1), intermediate at
// n2 (R1 + 1) + k1; step 2 (thread = (c, k1)): DFT_R2 gives X[k1 + R1 k2].
// w1 holds w_L^(n2 k1) at w1[k1 R2 + n2] (k1 >= 1; row_twiddle<L> gives the
// entry): consecutive lanes read consecutive entries.  Read from the table
// exp(-2 pi i m / T) instead, at m = n2 k1 T / L, the lanes of one load sit
// k1 T / L entries apart, up to 16 lanes on one bank pair, which took a third
// of the shared-memory wavefronts of the row passes (ncu, 512-point rows: r2c
// 24 per point and warp, LSU pipe 81 % busy).  At 512^3 / 1024^3 (ms): x r2c
// 1.86 -> 1.61, screening x 3.83 -> 3.45, force x c2r 5.20 -> 4.42, LPT x
// 1.17 -> 1.01.
// Each warp owns TW 32 / NT consecutive rows (RowMap), so the steps are ordered by
// warp barriers alone and the warps of a CTA drift apart: while one computes another
// loads.  The caller makes the warp's rows visible to it before the call and
// synchronises the warp before it reuses them.
// Store hook of fft_rowtile's last step: output k of row c as st(X[k], c, k);
// with kSmem = false the hook writes the output itself and the tile keeps the
// intermediate.
struct RowStore {
  static constexpr bool kSmem = true;
  __device__ __forceinline__ float2 operator()(float2 v, int, int) const { return v; }
};

// Index m (of exp(-2 pi i m / L)) of entry i = k1 R2 + n2 of a row transform's
// first-step twiddles.
template <int L>
__host__ __device__ constexpr int row_twiddle(int i) {
  return (i / Split<L>::R2) * (i % Split<L>::R2);
}

// Item idx = lane + 32 i of a warp's rows with R items per row: tile row c, item q.
// With fewer than 32 items in all, lanes repeat them (the same values, written twice).
template <int TW, int NT, int R>
struct RowMap {
  static constexpr int RW = TW * 32 / NT, U = RW * R, P = (U + 31) / 32;
  static_assert(RW * NT == TW * 32 && (U % 32 == 0 || 32 % U == 0), "whole rows per warp");
  int c0, idx0;
  __device__ __forceinline__ RowMap() {
    c0 = (threadIdx.x >> 5) * RW;
    idx0 = (threadIdx.x & 31) % (U < 32 ? U : 32);
  }
  __device__ __forceinline__ int c(int i) const { return c0 + (idx0 + 32 * i) / R; }
  __device__ __forceinline__ int q(int i) const { return (idx0 + 32 * i) % R; }
};

// Step 1 of the row transforms, with the warp barriers that separate it from step 2.
template <int L, int TW, int CW, int NT, bool INV, class Pre>
__device__ __forceinline__ void row_step1(float2* __restrict__ buf, const float2* __restrict__ w1, Pre pre) {
  constexpr int R1 = Split<L>::R1, R2 = Split<L>::R2;
  using Map = RowMap<TW, NT, R2>;
  static_assert(CW >= L + R2 - 1, "row pitch too small for the intermediate");
  const Map mp;
  float2 v[Map::P][R1];
#pragma unroll
  for (int i = 0; i < Map::P; ++i) {
    const int c = mp.c(i), n2 = mp.q(i);
    const float2* x = buf + c * CW + n2;
#pragma unroll
    for (int n1 = 0; n1 < R1; ++n1) v[i][pos_of<R1>(n1)] = pre(x[R2 * n1], c, R2 * n1 + n2);
    dftR<R1, INV>(v[i]);
    if (n2 > 0) {
#pragma unroll
      for (int k1 = 1; k1 < R1; ++k1) {
        float2 w = w1[k1 * R2 + n2];
        if (INV) w.y = -w.y;
        v[i][k1] = cmul(v[i][k1], w);
      }
    }
  }
  __syncwarp();
#pragma unroll
  for (int i = 0; i < Map::P; ++i) {
    float2* y = buf + mp.c(i) * CW + mp.q(i) * (R1 + 1);
#pragma unroll
    for (int k1 = 0; k1 < R1; ++k1) y[k1] = v[i][k1];
  }
  __syncwarp();
}

// PAIR32 (the forward and the chained row transforms): for L = 16 x 32 with one row per warp the
// radix-32 step runs on lane pairs (dft32_pair).
template <int L, int TW, int NT, bool PAIR32>
__host__ __device__ constexpr bool row_pairs() {
  return PAIR32 && Split<L>::R1 == 16 && Split<L>::R2 == 32 && TW * 32 == NT;
}

template <int L, int TW, int CW, int NT, bool INV, class Pre = NoPre, class Store = RowStore>
__device__ __forceinline__ void fft_rowtile(float2* __restrict__ buf, const float2* __restrict__ w1,
                                            Pre pre = Pre(), Store st = Store()) {
  constexpr int R1 = Split<L>::R1, R2 = Split<L>::R2;
  row_step1<L, TW, CW, NT, INV, Pre>(buf, w1, pre);
  using Map = RowMap<TW, NT, R1>;
  const Map mp;
  float2 y[Map::P][R2];
#pragma unroll
  for (int i = 0; i < Map::P; ++i) {
    const float2* yr = buf + mp.c(i) * CW + mp.q(i);
#pragma unroll
    for (int n2 = 0; n2 < R2; ++n2) y[i][pos_of<R2>(n2)] = yr[n2 * (R1 + 1)];
    dftR<R2, INV>(y[i]);
  }
  if constexpr (Store::kSmem) __syncwarp();
#pragma unroll
  for (int i = 0; i < Map::P; ++i) {
    const int c = mp.c(i), k1 = mp.q(i);
#pragma unroll
    for (int k2 = 0; k2 < R2; ++k2) {
      const float2 o = st(y[i][k2], c, k1 + R1 * k2);
      if constexpr (Store::kSmem) buf[c * CW + k1 + R1 * k2] = o;
    }
  }
}

// Forward row transform of real rows packed as z[n] = x[2n] + i x[2n+1] (L
// complex values), with the split into the half spectrum of the 2L reals
//   X[k] = (Z[k] + conj Z[L-k])/2 - i/2 w^k (Z[k] - conj Z[L-k]),  k = 0..L,
// w = exp(-2 pi i / 2L) from twr, done in the registers of step 2: thread (c,
// k1) holds Z[k1 + R1 k2], and Z[L - k] of k1 > 0 is entry R2 - 1 - k2 of lane
// R1 - k1 of the same row, one shuffle away (k1 = 0: the thread's own entry
// (R2 - k2) mod R2).  X leaves through st(X[k], c, k), where consecutive lanes
// hold consecutive k.  Writing Z back to the tile and reading the pairs from
// there costs 8 shared-memory wavefronts per point and warp, this 3 (two
// shuffles, one broadcast twiddle read), and one barrier less: x r2c 1.61 ->
// 1.30 ms and screening x 3.45 -> 3.14 ms at 1024^3, x r2c plane pass 1.21 ->
// 1.06 ms over 256 meshes of 128^3.
template <int L, int TW, int CW, int NT, bool PAIR32, class Store>
__device__ __forceinline__ void row_r2c_step2(float2* __restrict__ buf, const float2* __restrict__ twr, Store st) {
  constexpr int R1 = Split<L>::R1, R2 = Split<L>::R2;
  static_assert(R1 <= 32, "a row's partner lanes within the warp");
  const int lane = threadIdx.x & 31;
  auto emit = [&](float2 zk, float2 zm, int c, int k) {
    const float2 b = cconj(zm), E = cscale(cadd(zk, b), 0.5f), D = csub(zk, b);
    const float2 X = cadd(E, cmul(twr[k], make_float2(0.5f * D.y, -0.5f * D.x)));  // O = (-i/2) D
    const float2 o = st(X, c, k);
    if constexpr (Store::kSmem) buf[c * CW + k] = o;
  };
  if constexpr (row_pairs<L, TW, NT, PAIR32>()) {
    // a row per warp; half h of lane (k1, h) holds Z[k1 + 16 (2k + h)] at y[k]
    const int half = lane >> 4, c = threadIdx.x >> 5, k1 = lane & 15;
    float2 y[16];
    const float2* yr = buf + c * CW + k1 + 16 * half * (R1 + 1);
#pragma unroll
    for (int j = 0; j < 16; ++j) y[j] = yr[j * (R1 + 1)];
    dft32_pair<false>(y, half);
    if constexpr (Store::kSmem) __syncwarp();
    const int partner = k1 ? ((1 - half) << 4) | (16 - k1) : lane;
    const bool own = k1 == 0 && half == 0;
#pragma unroll
    for (int k = 0; k < 16; ++k) {
      float2 zm = make_float2(__shfl_sync(0xffffffffu, y[15 - k].x, partner),
                              __shfl_sync(0xffffffffu, y[15 - k].y, partner));
      if (own) zm = y[(16 - k) & 15];
      emit(y[k], zm, c, k1 + 16 * (2 * k + half));
    }
    if (own) emit(y[0], y[0], c, L);
  } else {
    using Map = RowMap<TW, NT, R1>;
    const Map mp;
    float2 y[Map::P][R2];
#pragma unroll
    for (int i = 0; i < Map::P; ++i) {
      const float2* yr = buf + mp.c(i) * CW + mp.q(i);
#pragma unroll
      for (int n2 = 0; n2 < R2; ++n2) y[i][pos_of<R2>(n2)] = yr[n2 * (R1 + 1)];
      dftR<R2, false>(y[i]);
    }
    if constexpr (Store::kSmem) __syncwarp();
#pragma unroll
    for (int i = 0; i < Map::P; ++i) {
      const int c = mp.c(i), k1 = mp.q(i);
      const int partner = (lane & ~(R1 - 1)) | ((R1 - k1) & (R1 - 1));
#pragma unroll
      for (int k2 = 0; k2 < R2; ++k2) {
        float2 zm = make_float2(__shfl_sync(0xffffffffu, y[i][R2 - 1 - k2].x, partner),
                                __shfl_sync(0xffffffffu, y[i][R2 - 1 - k2].y, partner));
        if (k1 == 0) zm = y[i][(R2 - k2) % R2];
        emit(y[i][k2], zm, c, k1 + R1 * k2);
      }
      if (k1 == 0) emit(y[i][0], y[i][0], c, L);
    }
  }
}

template <int L, int TW, int CW, int NT, class Pre, bool PAIR32, class Store>
__device__ __forceinline__ void fft_rowtile_r2c(float2* __restrict__ buf, const float2* __restrict__ w1,
                                                const float2* __restrict__ twr, Pre pre, Store st) {
  row_step1<L, TW, CW, NT, false, Pre>(buf, w1, pre);
  row_r2c_step2<L, TW, CW, NT, PAIR32, Store>(buf, twr, st);
}

// Inverse row transform, x = mid(z[n], c, n) on every value, forward real transform
// of x (fft_rowtile_r2c).  As in the column passes (fft_tile_fwd_inv) the values a
// thread holds after the inverse are inputs of its own first-step items of the
// forward transform, n2 = k1 + R1 h, so they stay in registers in between (PAIR32:
// the thread's 16 values are the item n2 = k1 + 16 half): 6 shared-memory
// wavefronts per point and warp and three barriers less.
template <int L, int TW, int CW, int NT, class Pre, class Mid, bool PAIR32, class Store>
__device__ __forceinline__ void fft_rowtile_inv_r2c(float2* __restrict__ buf, const float2* __restrict__ w1,
                                                    const float2* __restrict__ twr, Pre pre, Mid mid, Store st) {
  constexpr int R1 = Split<L>::R1, R2 = Split<L>::R2, H = R2 / R1;
  row_step1<L, TW, CW, NT, true, Pre>(buf, w1, pre);
  if constexpr (row_pairs<L, TW, NT, PAIR32>()) {
    const int n2 = threadIdx.x & 31, half = n2 >> 4, c = threadIdx.x >> 5, k1 = n2 & 15;
    float2 y[16], v[16];
    const float2* yr = buf + c * CW + k1 + 16 * half * (R1 + 1);
#pragma unroll
    for (int j = 0; j < 16; ++j) y[j] = yr[j * (R1 + 1)];
    dft32_pair<true>(y, half);
#pragma unroll
    for (int n1 = 0; n1 < 16; ++n1) v[pos_of<16>(n1)] = mid(y[n1], c, n2 + 32 * n1);
    dftR<16, false>(v);
    if (n2 > 0) {
#pragma unroll
      for (int k = 1; k < 16; ++k) v[k] = cmul(v[k], w1[k * R2 + n2]);
    }
    __syncwarp();
    float2* o = buf + c * CW + n2 * (R1 + 1);
#pragma unroll
    for (int k = 0; k < 16; ++k) o[k] = v[k];
  } else {
    using Map = RowMap<TW, NT, R1>;
    const Map mp;
    float2 v[Map::P][R2];
#pragma unroll
    for (int i = 0; i < Map::P; ++i) {
      const int c = mp.c(i), k1 = mp.q(i);
      const float2* yr = buf + c * CW + k1;
      float2 y[R2];
#pragma unroll
      for (int n2 = 0; n2 < R2; ++n2) y[pos_of<R2>(n2)] = yr[n2 * (R1 + 1)];
      dftR<R2, true>(y);
#pragma unroll
      for (int k2 = 0; k2 < R2; ++k2) y[k2] = mid(y[k2], c, k1 + R1 * k2);
#pragma unroll
      for (int h = 0; h < H; ++h) {
        const int n2 = k1 + R1 * h;
        float2 t[R1];
#pragma unroll
        for (int n1 = 0; n1 < R1; ++n1) t[pos_of<R1>(n1)] = y[h + H * n1];
        dftR<R1, false>(t);
        v[i][h * R1] = t[0];
#pragma unroll
        for (int k = 1; k < R1; ++k) v[i][h * R1 + k] = n2 > 0 ? cmul(t[k], w1[k * R2 + n2]) : t[k];
      }
    }
    __syncwarp();
#pragma unroll
    for (int i = 0; i < Map::P; ++i) {
      const int c = mp.c(i), k1 = mp.q(i);
#pragma unroll
      for (int h = 0; h < H; ++h) {
        float2* o = buf + c * CW + (k1 + R1 * h) * (R1 + 1);
#pragma unroll
        for (int k = 0; k < R1; ++k) o[k] = v[i][h * R1 + k];
      }
    }
  }
  __syncwarp();
  row_r2c_step2<L, TW, CW, NT, PAIR32, Store>(buf, twr, st);
}

// Out-of-line copy for kernels that run several transforms per tile: each
// call gets its own register allocation instead of one inlined body per call.
template <int L, int TW, int PITCH, int NT, bool INV, int TWS = 1, class Load = TileLoad,
          class Store = TileStore>
__device__ __noinline__ void fft_tile_call(float2* buf, const float2* tw, Load ld = Load(),
                                           Store st = Store()) {
  fft_tile<L, TW, PITCH, NT, INV, TWS, Load, Store>(buf, tw, ld, st);
}

// Signed frequency index of position n in a length-N transform.
__device__ __forceinline__ int freq_index(int n, int N) { return n < (N >> 1) ? n : n - N; }

}  // namespace cola
