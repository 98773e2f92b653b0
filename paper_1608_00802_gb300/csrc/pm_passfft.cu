// The mesh transforms of 512^3 fp32 meshes as five passes over memory (cloud-in-cell; other sizes have the x-y
// kernels, the plane kernels or cuFFT):
//   x  forward : each row of N reals -> N/2 complex, X[0] + i X[N/2] packed first  (rho -> tmp)
//   y  forward : 8 columns of a z-plane per block, the packed column split          (tmp -> spectrum)
//   z          : 16 columns of the half spectrum per block, Green multiplication, W_g partial, back (in place)
//   y  inverse : the columns packed again                                           (spectrum -> tmp)
//   x  inverse : each row back to N reals                                           (tmp, in place)
// tmp is the potential's mesh: N/2 complex values are a row of it.  A plane (1 MB) does not fit the cluster that
// the 256^2 x-y kernels use, and cuFFT's passes are far from the copy rate: 996 us for its 2D pair plus 504 for
// the four-step z kernel at one block of 128 registers per SM (a pass over memory takes 160 us).  So each pass here
// does as little as it can per value and leaves room for many threads: the five passes take 1193 us.  The
// potential's error against float64 (particle density, of the largest |phi|): 4.7e-7 -> 4.0e-7.  (384^3 by the
// same passes: 535 us against 987 by cuFFT's 3D pair and the Green pass, but in one of 80 jobs the
// displacements ended 2e-2 of the largest away from cuFFT's, in 7 of 80 more than 1e-4: the quantum force amplifies any
// other rounding next to nearly empty nodes.  Which of the two is nearer to float64 over such jobs has not been
// measured; 384^3 keeps cuFFT.)
//
// Rows: 16 threads a row (two rows a warp: the exchanges need no block barrier), H = N/2 = 16 Q points in two
// steps, n = j + 16 m and k = k1 + Q k2: thread j a Q-point DFT over m (Q = 16) and the twiddle, thread
// k1 < Q a 16-point DFT over j.  Columns: N = 8 * 8 * C points in three steps (C = 8), n = j + 8 C m,
// j = j' + C m', k = k1 + 8 (k2 + 8 k3): thread j an 8-point DFT over m and W_N^{j k1}, thread (k1, j') an
// 8-point DFT over m' and W_{8C}^{j' k2}, thread (k1, k2) a C-point DFT over j'; eight values and ~40
// registers a thread.  Slots of the exchange tile are padded by one in C, so that the third step's stride of
// C slots does not meet one bank group (the z kernel's slots are whole bank rows).  Inverses run the same steps
// backwards with conjugate twiddles.
#include "pm_kernels.cuh"

namespace pm {
namespace {

__device__ __forceinline__ float2 conj2(float2 a) { return make_float2(a.x, -a.y); }

// ---------------------------------------------------------------- rows
constexpr int PX_ROWS = 16, PX_THREADS = PX_ROWS * 16;
template <int N>
struct RowShape {
  static constexpr int H = N / 2, Q = H / 16, ROW = H + H / 16 + 1;  // padded row of complex values
};
__device__ __forceinline__ int px_pad(int n) { return n + (n >> 4); }

template <int N>
__global__ void __launch_bounds__(PX_THREADS, 4) k_x_r2c(const float* __restrict__ in, float2* __restrict__ out,
                                                         const float2* __restrict__ tw) {
  constexpr int H = RowShape<N>::H, Q = RowShape<N>::Q, ROW = RowShape<N>::ROW;
  __shared__ float2 S[PX_ROWS * ROW];
  const int j = threadIdx.x & 15;
  const uint32_t row = blockIdx.x * PX_ROWS + (threadIdx.x >> 4);  // (N^2 rows: a multiple of PX_ROWS)
  const float2* src = reinterpret_cast<const float2*>(in) + size_t(row) * H;
  float2* s = S + (threadIdx.x >> 4) * ROW;
  {
    float2 a[Q];
#pragma unroll
    for (int m = 0; m < Q; ++m) a[m] = __ldcs(src + j + 16 * m);
    dft_reg<Q, false>(a);
#pragma unroll
    for (int k1 = 0; k1 < Q; ++k1) s[px_pad(j + 16 * k1)] = cmul(a[bitrev<Q>(k1)], __ldg(tw + 2 * j * k1));
  }
  __syncwarp();
  float2 b[16];
  if (j < Q) {
#pragma unroll
    for (int i = 0; i < 16; ++i) b[i] = s[px_pad(i + 16 * j)];
    dft_reg<16, false>(b);
  }
  __syncwarp();
  if (j < Q) {
#pragma unroll
    for (int k2 = 0; k2 < 16; ++k2) s[px_pad(j + Q * k2)] = b[bitrev<16>(k2)];
  }
  __syncwarp();
  // X[k] = E + W^k O from Z[k] and Z[H - k]; X[0] and X[H], both real, packed
  float2* dst = out + size_t(row) * H;
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    const int k = j + 16 * i;
    const float2 z = s[px_pad(k)], zp = s[px_pad(k ? H - k : 0)];
    const float ex = 0.5f * (z.x + zp.x), ey = 0.5f * (z.y - zp.y), ox = 0.5f * (z.y + zp.y), oy = -0.5f * (z.x - zp.x);
    const float2 wo = cmul(make_float2(ox, oy), __ldg(tw + k));
    dst[k] = k ? make_float2(ex + wo.x, ey + wo.y) : make_float2(ex + ox, ex - ox);
  }
}

// in place: a row's values are read before any of them is written (__syncwarp between them)
template <int N>
__global__ void __launch_bounds__(PX_THREADS, 4) k_x_c2r(float2* mesh, const float2* __restrict__ tw) {
  constexpr int H = RowShape<N>::H, Q = RowShape<N>::Q, ROW = RowShape<N>::ROW;
  __shared__ float2 S[PX_ROWS * ROW];
  const int j = threadIdx.x & 15;
  const uint32_t row = blockIdx.x * PX_ROWS + (threadIdx.x >> 4);
  float2* io = mesh + size_t(row) * H;
  float2* s = S + (threadIdx.x >> 4) * ROW;
  float2 x[Q];
#pragma unroll
  for (int m = 0; m < Q; ++m) x[m] = __ldcs(io + j + 16 * m);
#pragma unroll
  for (int m = 0; m < Q; ++m) s[px_pad(j + 16 * m)] = x[m];
  __syncwarp();
  // Z[k] = (X[k] + X*[H-k]) + i W^-k (X[k] - X*[H-k]); k = 0 from the packed value
#pragma unroll
  for (int m = 0; m < Q; ++m) {
    const int k = j + 16 * m;
    const float2 xp = s[px_pad(k ? H - k : 0)];
    const float2 d = cmul(make_float2(x[m].x - xp.x, x[m].y + xp.y), conj2(__ldg(tw + k)));
    x[m] = k ? make_float2(x[m].x + xp.x - d.y, x[m].y - xp.y + d.x) : make_float2(x[m].x + x[m].y, x[m].x - x[m].y);
  }
  dft_reg<Q, true>(x);
  __syncwarp();
#pragma unroll
  for (int k1 = 0; k1 < Q; ++k1) s[px_pad(j + 16 * k1)] = cmul(x[bitrev<Q>(k1)], conj2(__ldg(tw + 2 * j * k1)));
  __syncwarp();
  if (j < Q) {
    float2 b[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) b[i] = s[px_pad(i + 16 * j)];
    dft_reg<16, true>(b);
#pragma unroll
    for (int k2 = 0; k2 < 16; ++k2) io[j + Q * k2] = b[bitrev<16>(k2)];  // (x[2n], x[2n + 1]), n = k1 + Q k2
  }
}

// ---------------------------------------------------------------- columns
constexpr int PC_COLS = 8;
template <int N>
struct ColShape {
  static constexpr int C = N / 64, BC = 8 * C, THREADS = PC_COLS * BC, MINB = 1536 / THREADS;
  static constexpr int SLOTS = N + N / C;  // padded by one slot in C
  static constexpr size_t smem() { return size_t(SLOTS) * PC_COLS * sizeof(float2); }
};
template <int N>
__device__ __forceinline__ int pc_slot(int s) {
  return (s + s / ColShape<N>::C) * PC_COLS;
}

// the first two steps of a column's transform from its values a[m] = x[j + BC m] (thread (c, j)): the tile
// T holds the values of the third step
template <int N>
__device__ __forceinline__ void cols_forward(float2 (&a)[8], float2* T, const float2* __restrict__ tw, int c, int j) {
  constexpr int C = ColShape<N>::C, BC = ColShape<N>::BC;
  dft_reg<8, false>(a);
#pragma unroll
  for (int k1 = 0; k1 < 8; ++k1) T[pc_slot<N>(k1 * BC + j) + c] = cmul(a[bitrev<8>(k1)], __ldg(tw + j * k1));
  __syncthreads();
  const int k1 = j / C, jp = j - k1 * C;
#pragma unroll
  for (int m = 0; m < 8; ++m) a[m] = T[pc_slot<N>(k1 * BC + jp + C * m) + c];
  dft_reg<8, false>(a);
#pragma unroll
  for (int k2 = 0; k2 < 8; ++k2) T[pc_slot<N>(k1 * BC + k2 * C + jp) + c] = cmul(a[bitrev<8>(k2)], __ldg(tw + 8 * jp * k2));
  __syncthreads();
}
// the last two steps of the inverse, from the tile that the first one filled: a[bitrev(m)] = x[j + BC m]
template <int N>
__device__ __forceinline__ void cols_inverse(float2 (&a)[8], float2* T, const float2* __restrict__ tw, int c, int j) {
  constexpr int C = ColShape<N>::C, BC = ColShape<N>::BC;
  __syncthreads();
  const int k1 = j / C, jp = j - k1 * C;
#pragma unroll
  for (int k2 = 0; k2 < 8; ++k2) a[k2] = T[pc_slot<N>(k1 * BC + k2 * C + jp) + c];
  dft_reg<8, true>(a);
#pragma unroll
  for (int m = 0; m < 8; ++m)
    T[pc_slot<N>(k1 * BC + jp + C * m) + c] = cmul(a[bitrev<8>(m)], conj2(__ldg(tw + (jp + C * m) * k1)));
  __syncthreads();
#pragma unroll
  for (int i = 0; i < 8; ++i) a[i] = T[pc_slot<N>(i * BC + j) + c];
  dft_reg<8, true>(a);
}

// y forward: tmp [z][y][H] -> spec [z][ky][H + 1]
template <int N>
__global__ void __launch_bounds__(ColShape<N>::THREADS, ColShape<N>::MINB) k_y_forward(const float2* __restrict__ in,
                                                                                       float2* __restrict__ spec,
                                                                                       const float2* __restrict__ tw) {
  constexpr int H = N / 2, NH = H + 1, C = ColShape<N>::C, BC = ColShape<N>::BC;
  extern __shared__ __align__(16) unsigned char pc_smem[];
  float2* T = reinterpret_cast<float2*>(pc_smem);
  const int c = threadIdx.x & 7, j = threadIdx.x >> 3;
  const int z = blockIdx.x / (H / PC_COLS), col0 = int(blockIdx.x % (H / PC_COLS)) * PC_COLS;
  const float2* src = in + size_t(z) * N * H + col0 + c;
  float2 a[8];
#pragma unroll
  for (int m = 0; m < 8; ++m) a[m] = __ldcs(src + (j + BC * m) * H);
  cols_forward<N>(a, T, tw, c, j);
  float2* dst = spec + size_t(z) * N * NH + col0 + c;
  const bool packed = col0 == 0;  // this block's first column is A + i B, the columns 0 and N/2
  for (int t = j; t < 64; t += BC) {
    const int k1 = t >> 3, k2 = t & 7;
    float2 b[C];
#pragma unroll
    for (int i = 0; i < C; ++i) b[i] = T[pc_slot<N>(k1 * BC + k2 * C + i) + c];
    dft_reg<C, false>(b);
#pragma unroll
    for (int k3 = 0; k3 < C; ++k3) {
      const int ky = k1 + 8 * (k2 + 8 * k3);
      const float2 v = b[bitrev<C>(k3)];
      if (!packed || c) dst[ky * NH] = v;
      // (the slots this thread has read are its own: the packed column waits there for its mirror)
      if (packed && c == 0) T[pc_slot<N>(k1 * BC + k2 * C + k3)] = v;
    }
  }
  if (packed) {
    __syncthreads();
    for (int ky = threadIdx.x; ky < N; ky += ColShape<N>::THREADS) {
      auto at = [&](int k) { return T[pc_slot<N>((k & 7) * BC + ((k >> 3) & 7) * C + (k >> 6))]; };
      const float2 y = at(ky), ym = at(ky ? N - ky : 0);
      float2* o = spec + (size_t(z) * N + ky) * NH;
      o[0] = make_float2(0.5f * (y.x + ym.x), 0.5f * (y.y - ym.y));
      o[H] = make_float2(0.5f * (y.y + ym.y), -0.5f * (y.x - ym.x));
    }
  }
}

// y inverse: spec [z][ky][H + 1] -> tmp [z][y][H]
template <int N>
__global__ void __launch_bounds__(ColShape<N>::THREADS, ColShape<N>::MINB) k_y_inverse(const float2* __restrict__ spec,
                                                                                       float2* __restrict__ out,
                                                                                       const float2* __restrict__ tw) {
  constexpr int H = N / 2, NH = H + 1, C = ColShape<N>::C, BC = ColShape<N>::BC;
  extern __shared__ __align__(16) unsigned char pc_smem[];
  float2* T = reinterpret_cast<float2*>(pc_smem);
  const int c = threadIdx.x & 7, j = threadIdx.x >> 3;
  const int z = blockIdx.x / (H / PC_COLS), col0 = int(blockIdx.x % (H / PC_COLS)) * PC_COLS;
  const float2* src = spec + size_t(z) * N * NH + col0 + c;
  const bool packed = col0 + c == 0;
  for (int t = j; t < 64; t += BC) {
    const int k1 = t >> 3, k2 = t & 7;
    float2 b[C];
#pragma unroll
    for (int k3 = 0; k3 < C; ++k3) {
      const int ky = k1 + 8 * (k2 + 8 * k3);
      b[k3] = __ldcs(src + ky * NH);
      if (packed) {  // A + i B
        const float2 h = __ldcs(src + ky * NH + H);
        b[k3] = make_float2(b[k3].x - h.y, b[k3].y + h.x);
      }
    }
    dft_reg<C, true>(b);
#pragma unroll
    for (int i = 0; i < C; ++i)
      T[pc_slot<N>(k1 * BC + k2 * C + i) + c] = cmul(b[bitrev<C>(i)], conj2(__ldg(tw + 8 * i * k2)));
  }
  float2 a[8];
  cols_inverse<N>(a, T, tw, c, j);
  float2* dst = out + size_t(z) * N * H + col0 + c;
#pragma unroll
  for (int m = 0; m < 8; ++m) dst[(j + BC * m) * H] = a[bitrev<8>(m)];
}

// ---------------------------------------------------------------- z
// z: 16 columns of the flattened (ky, kx) half plane per block, in place: phi^ = G rho^ with k_green's arithmetic
// and Parseval partial of W_g.  A thread carries two adjacent columns through every step as pairs (re0, re1),
// (im0, im1) in 64-bit registers: the packed fp32 instructions (add, sub, mul, fma .f32x2) do both columns at
// once, a pair of values is one 16-byte access of memory or shared memory, and twiddles and addresses serve two.
// With one column a thread and 8 columns a block the kernel was bound by its instructions and by 64-byte
// segments: 400 -> 327 us (two passes over memory take 160).  Pairs in blocks of 8 columns take 369; the y passes
// do not gain by pairs, because a spectrum row starts on 8 bytes only (inverse 235 -> 295, forward 235 -> 239), nor
// does the z kernel of 256^3 (33 -> 37).
using u64 = unsigned long long;
__device__ __forceinline__ u64 pk2(float a, float b) {
  u64 d;
  asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(a), "f"(b));
  return d;
}
__device__ __forceinline__ float2 un2(u64 a) {
  float2 d;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(d.x), "=f"(d.y) : "l"(a));
  return d;
}
__device__ __forceinline__ u64 add2(u64 a, u64 b) {
  u64 d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ u64 sub2(u64 a, u64 b) {
  u64 d;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ u64 mul2(u64 a, u64 b) {
  u64 d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ u64 fma2(u64 a, u64 b, u64 c) {
  u64 d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
struct C2 {  // two complex values of adjacent columns
  u64 re, im;
};
__device__ __forceinline__ C2 c2_of(float4 v) { return {pk2(v.x, v.z), pk2(v.y, v.w)}; }
__device__ __forceinline__ float4 c2_float4(C2 v) {
  const float2 r = un2(v.re), i = un2(v.im);
  return make_float4(r.x, i.x, r.y, i.y);
}
__device__ __forceinline__ C2 c2_ld(const ulonglong2* p) {
  const ulonglong2 v = *p;
  return {v.x, v.y};
}
__device__ __forceinline__ void c2_st(ulonglong2* p, C2 v) { *p = make_ulonglong2(v.re, v.im); }
// times w = (wx, wx), (wy, wy), or its conjugate
template <bool CONJ>
__device__ __forceinline__ C2 c2_mul(C2 a, ulonglong2 w) {
  if (CONJ) return {fma2(a.im, w.y, mul2(a.re, w.x)), sub2(mul2(a.im, w.x), mul2(a.re, w.y))};
  return {sub2(mul2(a.re, w.x), mul2(a.im, w.y)), fma2(a.re, w.y, mul2(a.im, w.x))};
}
// times exp(-+2 pi i t / 8) (forward: minus) of u - v
template <bool INV>
__device__ __forceinline__ C2 c2_diff8(C2 u, C2 v, int t) {
  if (t == 0) return {sub2(u.re, v.re), sub2(u.im, v.im)};
  if (t == 2) return INV ? C2{sub2(v.im, u.im), sub2(u.re, v.re)} : C2{sub2(u.im, v.im), sub2(v.re, u.re)};
  const C2 d = {sub2(u.re, v.re), sub2(u.im, v.im)};
  const u64 h = pk2(0.707106769f, 0.707106769f), mh = pk2(-0.707106769f, -0.707106769f);
  if (t == 1)
    return INV ? C2{mul2(sub2(d.re, d.im), h), mul2(add2(d.re, d.im), h)}
               : C2{mul2(add2(d.re, d.im), h), mul2(sub2(d.im, d.re), h)};
  return INV ? C2{mul2(add2(d.re, d.im), mh), mul2(sub2(d.re, d.im), h)}
             : C2{mul2(sub2(d.im, d.re), h), mul2(add2(d.re, d.im), mh)};
}
// DFT of M = 2, 4, 8 points (as dft_reg: natural order in, bit-reversed out)
template <int M, bool INV>
__device__ __forceinline__ void c2_dft_pow2(C2* a) {
#pragma unroll
  for (int len = M; len >= 2; len >>= 1) {
    const int half = len >> 1;
#pragma unroll
    for (int b = 0; b < M; b += len) {
#pragma unroll
      for (int j = 0; j < half; ++j) {
        const C2 u = a[b + j], v = a[b + j + half];
        a[b + j] = {add2(u.re, v.re), add2(u.im, v.im)};
        a[b + j + half] = c2_diff8<INV>(u, v, j * (8 / len));
      }
    }
  }
}
constexpr int ZC_COLS = 16, ZC_PAIRS = ZC_COLS / 2;
template <int N>
struct ZShape {
  static constexpr int C = N / 64, BC = 8 * C, THREADS = ZC_PAIRS * BC, MINB = 1024 / THREADS;
  // the exchange tile [slot][pair] (a quarter warp's 16-byte accesses are one slot: no padding), the twiddles as
  // (wx, wx, wy, wy), the Green table
  static constexpr size_t smem() { return size_t(N) * (ZC_PAIRS * 16 + 16 + 4); }
};

__device__ __forceinline__ void load_twiddles(ulonglong2* w, const float2* __restrict__ tw, int n) {
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    const float2 t = __ldg(tw + i);
    w[i] = make_ulonglong2(pk2(t.x, t.x), pk2(t.y, t.y));
  }
}

// the first two steps of the columns' transforms from their values a[m] = x[j + BC m] (thread (c, j)): the tile
// T holds the values of the third step
template <int N>
__device__ __forceinline__ void zc_forward(C2 (&a)[8], ulonglong2* T, const ulonglong2* w, int c, int j) {
  constexpr int C = ZShape<N>::C, BC = ZShape<N>::BC;
  c2_dft_pow2<8, false>(a);
  c2_st(T + j * ZC_PAIRS + c, a[0]);
#pragma unroll
  for (int k1 = 1; k1 < 8; ++k1) c2_st(T + (k1 * BC + j) * ZC_PAIRS + c, c2_mul<false>(a[bitrev<8>(k1)], w[j * k1]));
  __syncthreads();
  const int k1 = j / C, jp = j - k1 * C;
  ulonglong2* t = T + (k1 * BC + jp) * ZC_PAIRS + c;
#pragma unroll
  for (int m = 0; m < 8; ++m) a[m] = c2_ld(t + C * m * ZC_PAIRS);
  c2_dft_pow2<8, false>(a);
  c2_st(t, a[0]);
#pragma unroll
  for (int k2 = 1; k2 < 8; ++k2) c2_st(t + k2 * C * ZC_PAIRS, c2_mul<false>(a[bitrev<8>(k2)], w[8 * jp * k2]));
  __syncthreads();
}
// the last two steps of the inverse, from the tile that the first one filled: a[bitrev(m)] = x[j + BC m]
template <int N>
__device__ __forceinline__ void zc_inverse(C2 (&a)[8], ulonglong2* T, const ulonglong2* w, int c, int j) {
  constexpr int C = ZShape<N>::C, BC = ZShape<N>::BC;
  __syncthreads();
  const int k1 = j / C, jp = j - k1 * C;
  ulonglong2* t = T + (k1 * BC + jp) * ZC_PAIRS + c;
#pragma unroll
  for (int k2 = 0; k2 < 8; ++k2) a[k2] = c2_ld(t + k2 * C * ZC_PAIRS);
  c2_dft_pow2<8, true>(a);
#pragma unroll
  for (int m = 0; m < 8; ++m) c2_st(t + C * m * ZC_PAIRS, c2_mul<true>(a[bitrev<8>(m)], w[(jp + C * m) * k1]));
  __syncthreads();
#pragma unroll
  for (int i = 0; i < 8; ++i) a[i] = c2_ld(T + (i * BC + j) * ZC_PAIRS + c);
  c2_dft_pow2<8, true>(a);
}

template <int N>
__global__ void __launch_bounds__(ZShape<N>::THREADS, ZShape<N>::MINB) k_z_green(float2* spec, const float2* __restrict__ tw,
                                                                                 const float* __restrict__ s2g, float coef,
                                                                                 double* part) {
  constexpr int H = N / 2, NH = H + 1, C = ZShape<N>::C, BC = ZShape<N>::BC;
  constexpr size_t PLANE = size_t(N) * NH;
  extern __shared__ __align__(16) unsigned char pc_smem[];
  ulonglong2 *T = reinterpret_cast<ulonglong2*>(pc_smem), *W = T + N * ZC_PAIRS;
  float* s2 = reinterpret_cast<float*>(W + N);
  const int c = threadIdx.x & 7, j = threadIdx.x >> 3;
  const uint32_t col = blockIdx.x * ZC_COLS + 2 * c;
  C2 a[8];
  {
    const float4* src = reinterpret_cast<const float4*>(spec + col);
#pragma unroll
    for (int m = 0; m < 8; ++m) a[m] = c2_of(__ldcs(src + (j + BC * m) * (PLANE / 2)));
  }
  load_twiddles(W, tw, N);
  for (int i = threadIdx.x; i < N; i += ZShape<N>::THREADS) s2[i] = __ldg(s2g + i);
  __syncthreads();
  zc_forward<N>(a, T, W, c, j);
  // (ky, kx) of the two columns
  const uint32_t ky0 = col / NH, kx0 = col - ky0 * NH, kx1 = kx0 + 1 == NH ? 0 : kx0 + 1, ky1 = kx1 ? ky0 : ky0 + 1;
  const float sx0 = s2[kx0], sx1 = s2[kx1], sy0 = s2[ky0], sy1 = s2[ky1];
  const u64 w2 = pk2((kx0 == 0 || kx0 == H) ? 1.0f : 2.0f, (kx1 == 0 || kx1 == H) ? 1.0f : 2.0f);
  u64 wsum = pk2(0.0f, 0.0f);
  for (int t = j; t < 64; t += BC) {
    const int k1 = t >> 3, k2 = t & 7;
    ulonglong2* s = T + (k1 * BC + k2 * C) * ZC_PAIRS + c;
    C2 b[C], d[C];
#pragma unroll
    for (int i = 0; i < C; ++i) b[i] = c2_ld(s + i * ZC_PAIRS);
    c2_dft_pow2<C, false>(b);
#pragma unroll
    for (int k3 = 0; k3 < C; ++k3) {
      const int kz = k1 + 8 * (k2 + 8 * k3);
      const C2 v = b[bitrev<C>(k3)];
      const float sz = s2[kz];
      const float syz0 = sy0 + sz, syz1 = sy1 + sz;
      const float sum0 = syz0 + sx0, sum1 = syz1 + sx1;
      const u64 g = pk2((col == 0 && kz == 0) ? 0.0f : coef * __frcp_rn(sum0), coef * __frcp_rn(sum1));
      wsum = fma2(mul2(w2, g), fma2(v.re, v.re, mul2(v.im, v.im)), wsum);
      d[k3] = {mul2(v.re, g), mul2(v.im, g)};
    }
    c2_dft_pow2<C, true>(d);
#pragma unroll
    for (int i = 0; i < C; ++i) c2_st(s + i * ZC_PAIRS, c2_mul<true>(d[bitrev<C>(i)], W[8 * i * k2]));
  }
  zc_inverse<N>(a, T, W, c, j);
  float4* dst = reinterpret_cast<float4*>(spec + col);
#pragma unroll
  for (int m = 0; m < 8; ++m) dst[(j + BC * m) * (PLANE / 2)] = c2_float4(a[bitrev<8>(m)]);
  const float2 ws = un2(wsum);
  float acc[1] = {ws.x + ws.y};
  block_sum_store<1>(acc, part, gridDim.x);
}

template <int N>
cudaError_t z_prepare() {
  static DeviceOnce once;
  return once([](int&) {
    const void* const fns[] = {(const void*)k_z_green<N>};
    return raise_smem(fns, ZShape<N>::smem());
  });
}

template <int N>
cudaError_t pass_potential(const float* rho, float* phi, float2* spec, const float2* tw, const float* s2, float coef,
                           double* part, cudaStream_t s, int stage) {
  using S = ColShape<N>;
  constexpr unsigned rows = unsigned(N) * N / PX_ROWS, planes = unsigned(N) * (N / 2 / PC_COLS);
  float2* tmp = reinterpret_cast<float2*>(phi);
  if (stage == 0) {
    k_x_r2c<N><<<rows, PX_THREADS, 0, s>>>(rho, tmp, tw);
    k_y_forward<N><<<planes, S::THREADS, S::smem(), s>>>(tmp, spec, tw);
  } else if (stage == 1) {
    using Z = ZShape<N>;
    const cudaError_t e = z_prepare<N>();
    if (e != cudaSuccess) return e;
    k_z_green<N><<<unsigned(pass_fft_tiles(N)), Z::THREADS, Z::smem(), s>>>(spec, tw, s2, coef, part);
  } else {
    k_y_inverse<N><<<planes, S::THREADS, S::smem(), s>>>(spec, tmp, tw);
    k_x_c2r<N><<<rows, PX_THREADS, 0, s>>>(tmp, tw);
  }
  return cudaGetLastError();
}

}  // namespace

bool pass_fft_supported(int n) { return n == 512; }
int pass_fft_tiles(int n) { return n * (n / 2 + 1) / ZC_COLS; }

cudaError_t launch_pass_fft(int stage, const float* rho, float* phi, void* spec, const float2* tw, const float* s2, int n,
                            double coef, double* part, cudaStream_t s) {
  switch (n) {
    case 512: return pass_potential<512>(rho, phi, static_cast<float2*>(spec), tw, s2, float(coef), part, s, stage);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace pm
