// The x and y transforms of the z-planes of 64^3 and 128^3 fp32 meshes, one CTA per plane and direction,
// before and after the z kernel.  A plane's half spectrum (16 and 64 KB) fits one SM's shared memory, so the
// rows and the columns are transformed there without a second pass.  These meshes are bound by the number
// and the latency of the launches, not by bytes: a 64^3 solve was seven kernels (cuFFT's 3D pair and the
// Green pass, 18 us and six gaps) and is three, 8.7 us.
//
// Forward: 8 threads a row, H = N/2 = 8 Q points in two steps (n = j + 8 m, k = k1 + Q k2), in place in the
// tile; the column threads form X[k] = E[k] + W^k O[k] from Z[k] and Z[H - k] as they load, X[0] + i X[H]
// packed in column 0; N = P 8 points in two steps (thread j < P an 8-point DFT over the rows j + P m and the
// twiddle, thread k1 < 8 a P-point DFT); column 0 is split into kx = 0 and kx = N/2 at the end.  Inverse: the
// same backwards.  Layouts and normalisation are those of the batched 2D R2C and C2R.
#include "pm_kernels.cuh"

namespace pm {
namespace {

template <int N>
struct Plane {
  static constexpr int H = N / 2, NH = H + 1, Q = H / 8, P = N / 8, THREADS = N * 8;
  static constexpr int ROW = H + 8;  // row stride: two rows of a half warp on different banks
  static constexpr size_t smem() { return size_t(N) * ROW * sizeof(float2); }
};
__device__ __forceinline__ float2 conj_of(float2 a) { return make_float2(a.x, -a.y); }

template <int N, bool PACKED>
__global__ void __launch_bounds__(Plane<N>::THREADS, 1) k_plane_r2c(const float* __restrict__ rho, float2* __restrict__ spec,
                                                                    const float2* __restrict__ tw, size_t ms) {
  constexpr int H = Plane<N>::H, NH = Plane<N>::NH, Q = Plane<N>::Q, P = Plane<N>::P, ROW = Plane<N>::ROW;
  if constexpr (PACKED) {  // member blockIdx.y of a packed group
    const size_t o = size_t(blockIdx.y) * ms;
    rho = moff(rho, o), spec = moff(spec, o);
  }
  extern __shared__ __align__(16) unsigned char pl_smem[];
  float2* T = reinterpret_cast<float2*>(pl_smem);
  const int z = blockIdx.x;
  {
    const int j = threadIdx.x & 7, r = threadIdx.x >> 3;
    const float2* src = reinterpret_cast<const float2*>(rho) + (size_t(z) * N + r) * H;
    float2* s = T + r * ROW;
    float2 a[Q];
#pragma unroll
    for (int m = 0; m < Q; ++m) a[m] = __ldg(src + j + 8 * m);
    dft_reg<Q, false>(a);
#pragma unroll
    for (int k1 = 0; k1 < Q; ++k1) s[j + 8 * k1] = cmul(a[bitrev<Q>(k1)], __ldg(tw + 2 * j * k1));
    __syncwarp();
    float2 b[8];
    if (j < Q) {
#pragma unroll
      for (int i = 0; i < 8; ++i) b[i] = s[i + 8 * j];
      dft_reg<8, false>(b);
    }
    __syncwarp();
    if (j < Q) {
#pragma unroll
      for (int k2 = 0; k2 < 8; ++k2) s[j + Q * k2] = b[bitrev<8>(k2)];
    }
  }
  __syncthreads();
  const int c = threadIdx.x % H, j = threadIdx.x / H;  // column and its thread (j < 16)
  {
    float2 a[8];
    if (j < P) {
      const float2 w = __ldg(tw + c);
      const int cm = c ? H - c : 0;
#pragma unroll
      for (int m = 0; m < 8; ++m) {
        const float2 *row = T + (j + P * m) * ROW, u = row[c], v = row[cm];
        const float ex = 0.5f * (u.x + v.x), ey = 0.5f * (u.y - v.y), ox = 0.5f * (u.y + v.y), oy = -0.5f * (u.x - v.x);
        const float2 wo = cmul(make_float2(ox, oy), w);
        a[m] = c ? make_float2(ex + wo.x, ey + wo.y) : make_float2(ex + ox, ex - ox);
      }
      dft_reg<8, false>(a);
    }
    __syncthreads();  // every column has read its mirror
    if (j < P) {
#pragma unroll
      for (int k1 = 0; k1 < 8; ++k1) T[(j + P * k1) * ROW + c] = cmul(a[bitrev<8>(k1)], __ldg(tw + j * k1));
    }
  }
  __syncthreads();
  float2* dst = spec + size_t(z) * N * NH;
  if (j < 8) {
    float2 b[P];
#pragma unroll
    for (int i = 0; i < P; ++i) b[i] = T[(i + P * j) * ROW + c];
    dft_reg<P, false>(b);
#pragma unroll
    for (int k2 = 0; k2 < P; ++k2) {
      const float2 v = b[bitrev<P>(k2)];
      if (c)
        dst[(j + 8 * k2) * NH + c] = v;
      else
        T[(k2 + P * j) * ROW] = v;  // (slots that this thread alone has read)
    }
  }
  __syncthreads();
  if (threadIdx.x < N) {  // column 0: A + i B
    const int ky = threadIdx.x, km = ky ? N - ky : 0;
    const float2 y = T[((ky >> 3) + P * (ky & 7)) * ROW], ym = T[((km >> 3) + P * (km & 7)) * ROW];
    dst[ky * NH] = make_float2(0.5f * (y.x + ym.x), 0.5f * (y.y - ym.y));
    dst[ky * NH + H] = make_float2(0.5f * (y.y + ym.y), -0.5f * (y.x - ym.x));
  }
}

template <int N, bool PACKED>
__global__ void __launch_bounds__(Plane<N>::THREADS, 1) k_plane_c2r(const float2* __restrict__ spec, float* __restrict__ phi,
                                                                    const float2* __restrict__ tw, size_t ms) {
  constexpr int H = Plane<N>::H, NH = Plane<N>::NH, Q = Plane<N>::Q, P = Plane<N>::P, ROW = Plane<N>::ROW;
  if constexpr (PACKED) {
    const size_t o = size_t(blockIdx.y) * ms;
    spec = moff(spec, o), phi = moff(phi, o);
  }
  extern __shared__ __align__(16) unsigned char pl_smem[];
  float2* T = reinterpret_cast<float2*>(pl_smem);
  const int z = blockIdx.x;
  {
    const int c = threadIdx.x % H, j = threadIdx.x / H;
    const float2* src = spec + size_t(z) * N * NH;
    if (j < 8) {
      float2 b[P];
#pragma unroll
      for (int k2 = 0; k2 < P; ++k2) {
        const float2* at = src + (j + 8 * k2) * NH;
        b[k2] = __ldg(at + c);
        if (c == 0) {
          const float2 h = __ldg(at + H);
          b[k2] = make_float2(b[k2].x - h.y, b[k2].y + h.x);  // A + i B
        }
      }
      dft_reg<P, true>(b);
#pragma unroll
      for (int i = 0; i < P; ++i) T[(i + P * j) * ROW + c] = cmul(b[bitrev<P>(i)], conj_of(__ldg(tw + i * j)));
    }
    __syncthreads();
    if (j < P) {
      float2 a[8];
#pragma unroll
      for (int k1 = 0; k1 < 8; ++k1) a[k1] = T[(j + P * k1) * ROW + c];
      dft_reg<8, true>(a);
#pragma unroll
      for (int m = 0; m < 8; ++m) T[(j + P * m) * ROW + c] = a[bitrev<8>(m)];  // row j + P m
    }
  }
  __syncthreads();
  const int j = threadIdx.x & 7, r = threadIdx.x >> 3;
  float2* s = T + r * ROW;
  float2 x[Q];
#pragma unroll
  for (int m = 0; m < Q; ++m) {
    const int k = j + 8 * m;
    const float2 u = s[k], v = s[k ? H - k : 0];
    const float2 d = cmul(make_float2(u.x - v.x, u.y + v.y), conj_of(__ldg(tw + k)));
    x[m] = k ? make_float2(u.x + v.x - d.y, u.y - v.y + d.x) : make_float2(u.x + u.y, u.x - u.y);
  }
  dft_reg<Q, true>(x);
  __syncwarp();  // the row's values are read
#pragma unroll
  for (int k1 = 0; k1 < Q; ++k1) s[j + 8 * k1] = cmul(x[bitrev<Q>(k1)], conj_of(__ldg(tw + 2 * j * k1)));
  __syncwarp();
  if (j < Q) {
    float2 b[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) b[i] = s[i + 8 * j];
    dft_reg<8, true>(b);
    float2* dst = reinterpret_cast<float2*>(phi) + (size_t(z) * N + r) * H;
#pragma unroll
    for (int k2 = 0; k2 < 8; ++k2) dst[j + Q * k2] = b[bitrev<8>(k2)];  // (x[2n], x[2n + 1]), n = k1 + Q k2
  }
}

template <int N>
cudaError_t plane_prepare() {
  static DeviceOnce once;
  return once([](int&) {
    const void* const fns[] = {(const void*)k_plane_r2c<N, false>, (const void*)k_plane_r2c<N, true>,
                               (const void*)k_plane_c2r<N, false>, (const void*)k_plane_c2r<N, true>};
    return raise_smem(fns, Plane<N>::smem());
  });
}

template <int N>
cudaError_t plane_fft(bool inverse, float* mesh, float2* spec, const float2* tw, cudaStream_t s, int nm, size_t ms) {
  const cudaError_t e = plane_prepare<N>();
  if (e != cudaSuccess) return e;
  const dim3 g(N, unsigned(nm));
  constexpr int T = Plane<N>::THREADS;
  constexpr size_t sm = Plane<N>::smem();
  if (inverse)
    nm > 1 ? k_plane_c2r<N, true><<<g, T, sm, s>>>(spec, mesh, tw, ms) : k_plane_c2r<N, false><<<g, T, sm, s>>>(spec, mesh, tw, 0);
  else
    nm > 1 ? k_plane_r2c<N, true><<<g, T, sm, s>>>(mesh, spec, tw, ms) : k_plane_r2c<N, false><<<g, T, sm, s>>>(mesh, spec, tw, 0);
  return cudaGetLastError();
}

}  // namespace

bool plane_fft_supported(int n) { return n == 64 || n == 128; }

cudaError_t launch_plane_fft(bool inverse, float* mesh, void* spec, const float2* tw, int n, cudaStream_t s, int nm,
                             size_t ms) {
  switch (n) {
    case 64: return plane_fft<64>(inverse, mesh, static_cast<float2*>(spec), tw, s, nm, ms);
    case 128: return plane_fft<128>(inverse, mesh, static_cast<float2*>(spec), tw, s, nm, ms);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace pm
