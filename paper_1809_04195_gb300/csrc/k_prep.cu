// Plan-time kernels: coil-map preparation, the space-time kernel Psi (Sec. IV.B) and
// the projection of per-echo k-space onto the basis (re-sort and project, Sec. III.A).
#include "launch.h"
#include "t2sh_device.cuh"

namespace t2sh {

constexpr int kPsiThreads = 64;  // many small CTAs: these kernels are bound by latency

// S'_{c,m}(y, z) = (-1)^(y+z) S_{c,m}(y, z): the image-side half of the FFT centring
// (FFTmod, Sec. IV.A) folded into the maps once.  Also the per-pixel largest
// eigenvalue of S(p)^H S(p) (C x M), max-reduced over all pixels into *lam_bits
// (float bits; non-negative floats order like their bit patterns).
__global__ void __launch_bounds__(kThreads) k_maps_prep(Geom g, const float2* in, float2* out,
                                                      unsigned* lam_bits) {
  const int N = g.ny * g.nz;
  const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;  // over S * N pixels
  float lam = 0.0f;
  if (idx < (long long)g.S * N) {
    const int s = (int)(idx / N);
    const int n = (int)(idx - (long long)s * N);
    const int y = n / g.nz, z = n - y * g.nz;
    const float sg = parity_sign(y + z);
    double a = 0.0, d = 0.0, br = 0.0, bi = 0.0;
    for (int c = 0; c < g.C; ++c) {
      const long long base = ((long long)(s * g.C + c) * g.M) * N + n;
      const float2 s0 = in[base];
      out[base] = cscale(s0, sg);
      a += (double)s0.x * s0.x + (double)s0.y * s0.y;
      if (g.M > 1) {
        const float2 s1 = in[base + N];
        out[base + N] = cscale(s1, sg);
        d += (double)s1.x * s1.x + (double)s1.y * s1.y;
        br += (double)s0.x * s1.x + (double)s0.y * s1.y;  // conj(s0) s1
        bi += (double)s0.x * s1.y - (double)s0.y * s1.x;
      }
    }
    double l = a;
    if (g.M > 1) {
      const double h = 0.5 * (a - d);
      l = 0.5 * (a + d) + sqrt(h * h + br * br + bi * bi);
    }
    lam = (float)l;
  }
  // warp max then one atomic per warp
  for (int o = 16; o > 0; o >>= 1) lam = fmaxf(lam, __shfl_xor_sync(0xffffffffu, lam, o));
  if ((threadIdx.x & 31) == 0 && lam > 0.0f) atomicMax(lam_bits, __float_as_uint(lam));
}

// Largest eigenvalue of the real symmetric K x K matrix acc (upper triangle): its eigenvector v in
// float32 (Jacobi on the matrix scaled by its trace, so the pivots are in the normal range), then
// in float64 w = A v and w.w / v.w.  That quotient errs by the square of v's error (1e-13 of the
// trace; where the two largest eigenvalues agree to 1e-6, by less than a float32 rounding), and a
// full float64 Jacobi per point costs 20 times the rest of the kernel on a chip whose float64 rate
// is 1/60 of float32: 64x48, T = 32: 263 -> 22 us; 256x160, T = 80: 527 -> 41 us.
template <int KC>
__device__ __forceinline__ float sym_lam_max(const double (&acc)[KC][KC]) {
  double tr = 0.0;
#pragma unroll
  for (int k = 0; k < KC; ++k) tr += acc[k][k];
  if (!(tr > 0.0)) return 0.f;
  const double inv = 1.0 / tr;
  float ar[KC][KC], ai[KC][KC], vr[KC][KC], vi[KC][KC];
#pragma unroll
  for (int k = 0; k < KC; ++k)
#pragma unroll
    for (int l = k; l < KC; ++l) {
      ar[k][l] = ar[l][k] = (float)(acc[k][l] * inv);
      ai[k][l] = ai[l][k] = 0.f;
    }
  herm_jacobi_rounds<float, KC>(ar, ai, vr, vi, KC == 4 ? 6 : 9);
  float m = ar[0][0], v[KC];
#pragma unroll
  for (int k = 0; k < KC; ++k) v[k] = vr[k][0];
#pragma unroll
  for (int i = 1; i < KC; ++i) {
    const bool up = ar[i][i] > m;
    m = up ? ar[i][i] : m;
#pragma unroll
    for (int k = 0; k < KC; ++k) v[k] = up ? vr[k][i] : v[k];
  }
  double ww = 0.0, vw = 0.0;
#pragma unroll
  for (int k = 0; k < KC; ++k) {
    double w = 0.0;
#pragma unroll
    for (int l = 0; l < KC; ++l) w += (k <= l ? acc[k][l] : acc[l][k]) * (double)v[l];
    ww += w * w;
    vw += (double)v[k] * w;
  }
  return vw > 0.0 ? (float)(ww / vw) : 0.f;
}

__device__ __forceinline__ void warp_max_bits(float lam, unsigned* bits) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) lam = fmaxf(lam, __shfl_xor_sync(0xffffffffu, lam, o));
  if ((threadIdx.x & 31) == 0 && lam > 0.0f) atomicMax(bits, __float_as_uint(lam));
}

// acc += the outer products of the basis rows in `word` (bit i: echo t0 + i), in float64
template <int KC>
__device__ __forceinline__ void psi_add(double (&acc)[KC][KC], const float* sphi, int K, int t0, unsigned word) {
  while (word) {
    const float* ph = sphi + (t0 + __ffs(word) - 1) * K;
    word &= word - 1;
    double d[KC];
#pragma unroll
    for (int k = 0; k < KC; ++k) d[k] = k < K ? (double)ph[k] : 0.0;
#pragma unroll
    for (int k = 0; k < KC; ++k)
#pragma unroll
      for (int l = k; l < KC; ++l)
        if (l < K) acc[k][l] += d[k] * d[l];
  }
}

// the 32 echoes t0 .. t0 + 31 of point n as a bit word
__device__ __forceinline__ unsigned mask_word(const uint8_t* __restrict__ mask, int T, int N, int t0, int n) {
  unsigned word = 0;
  const int m = min(32, T - t0);
#pragma unroll 16
  for (int i = 0; i < m; ++i) word |= (mask[(long long)(t0 + i) * N + n] ? 1u : 0u) << i;
  return word;
}

// Psi(n)_{kl} = sum_t Phi_{tk} P_t(n) Phi_{tl} in float64, stored as float32 upper
// triangle (p = 0.. for k <= l, row by row) scaled by 1/N so the unnormalised
// DFT pair needs no other scaling, SoA [P][ny][nz].  Also the sampling pattern as bit words
// bits[T / 32][n] (nullable) and lambda_max(Psi(n)) max-reduced into *lam_bits.
// A thread adds only its own samples: a warp takes as many steps as its densest point has
// samples, not T.
template <int KC>
__global__ void __launch_bounds__(kPsiThreads) k_psi_build(Geom g, const float* __restrict__ phi,
                                                      const uint8_t* __restrict__ mask, float* __restrict__ psi,
                                                      unsigned* __restrict__ bits, unsigned* lam_bits) {
  extern __shared__ float sphi[];  // [T][K]
  for (int i = threadIdx.x; i < g.T * g.K; i += blockDim.x) sphi[i] = phi[i];
  __syncthreads();
  const int N = g.ny * g.nz;
  const int n = blockIdx.x * blockDim.x + threadIdx.x;
  float lam = 0.0f;
  if (n < N) {
    double acc[KC][KC];
#pragma unroll
    for (int k = 0; k < KC; ++k)
#pragma unroll
      for (int l = 0; l < KC; ++l) acc[k][l] = 0.0;
    for (int t0 = 0; t0 < g.T; t0 += 32) {
      const unsigned word = mask_word(mask, g.T, N, t0, n);
      if (bits) bits[(long long)(t0 >> 5) * N + n] = word;
      psi_add<KC>(acc, sphi, g.K, t0, word);
    }
    const double inv_n = 1.0 / (double)N;
    int p = 0;
#pragma unroll
    for (int k = 0; k < KC; ++k)
#pragma unroll
      for (int l = k; l < KC; ++l)
        if (l < g.K) {
          psi[(long long)p * N + n] = (float)(acc[k][l] * inv_n);
          ++p;
        }
    lam = sym_lam_max<KC>(acc);
  }
  warp_max_bits(lam, lam_bits);
}

// Place of (image k, point n = y nz + z) of per-coil data in a layout of t
struct TePlace {
  long long base;
  int step;  // image stride
  int rot;   // slot of image 0 (with slot rotation, K = 4), or -1
  __device__ __forceinline__ TePlace(const Geom& g, const TLayout& lt, long long sc, int n) {
    const int N = g.ny * g.nz;
    rot = -1;
    if (lt.W) {
      const int y = n / g.nz, z = n - y * g.nz;
      base = (sc * N + (long long)y * g.nz) * g.K + (z / lt.W) * (g.K * lt.W) + z % lt.W;
      step = lt.W;
      if (lt.trb) rot = y % lt.trb + y / lt.trb;
    } else {
      base = sc * g.K * (long long)N + n;
      step = N;
    }
  }
  __device__ __forceinline__ long long at(int k) const {
    return base + (long long)(rot >= 0 ? (k + rot) & 3 : k) * step;
  }
};

__device__ __forceinline__ float2 ld_sample(const float2* p) {
  float2 v;
  asm volatile("ld.global.L1::no_allocate.L2::64B.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "l"(p));
  return v;
}

// ytil[s][c][k][n] = sum_t Phi_{tk} P_t(n) y[s][c][t][n], in any layout of t.  A thread walks
// the set bits of its point only, NS samples of NP (slice, coil) planes at a time, so eight
// independent loads are in flight instead of one behind one mask byte.  The samples are
// scattered 8-byte values (5 % of the plane), so the kernel is bound by what DRAM fetches for them:
// with the default 128-byte fetches 54 % of the whole array (2.0 GB of 3.8, 342 us), with 64-byte
// ones 281 us.  240x128, C = 8, T = 80 at 5 %, 24 slices: 785 us before.
template <int KC, int NP, int NS>
__global__ void __launch_bounds__(kThreads) k_project(Geom g, TLayout lt, const float* __restrict__ phi,
                                                    const unsigned* __restrict__ bits,
                                                    const float2* y, float2* __restrict__ out) {
  extern __shared__ float sphi[];
  for (int i = threadIdx.x; i < g.T * g.K; i += blockDim.x) sphi[i] = phi[i];
  __syncthreads();
  pdl_wait();
  pdl_trigger();
  const int N = g.ny * g.nz;
  const int n = blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= N) return;
  const long long nsc = (long long)g.S * g.C, plane = (long long)g.T * N;
  for (long long sc0 = (long long)blockIdx.y * NP; sc0 < nsc; sc0 += (long long)gridDim.y * NP) {
    const int np = (int)min((long long)NP, nsc - sc0);
    float2 acc[NP][KC];
#pragma unroll
    for (int i = 0; i < NP; ++i)
#pragma unroll
      for (int k = 0; k < KC; ++k) acc[i][k] = make_float2(0.f, 0.f);
    const float2* yb = y + sc0 * plane + n;
    for (int t0 = 0; t0 < g.T; t0 += 32) {
      unsigned word = bits[(long long)(t0 >> 5) * N + n];
      while (word) {
        int t[NS];
        float2 v[NS][NP];
#pragma unroll
        for (int u = 0; u < NS; ++u) {
          t[u] = word ? t0 + __ffs(word) - 1 : -1;
          word &= word - 1;
#pragma unroll
          for (int i = 0; i < NP; ++i)
            v[u][i] = t[u] >= 0 && i < np ? ld_sample(yb + i * plane + (long long)t[u] * N) : make_float2(0.f, 0.f);
        }
#pragma unroll
        for (int u = 0; u < NS; ++u) {
          if (t[u] >= 0) {
            const float* ph = sphi + t[u] * g.K;
#pragma unroll
            for (int k = 0; k < KC; ++k)
              if (k < g.K) {
                const float f = ph[k];
#pragma unroll
                for (int i = 0; i < NP; ++i) {
                  acc[i][k].x = fmaf(f, v[u][i].x, acc[i][k].x);
                  acc[i][k].y = fmaf(f, v[u][i].y, acc[i][k].y);
                }
              }
          }
        }
      }
    }
#pragma unroll
    for (int i = 0; i < NP; ++i) {
      if (i < np) {
        const TePlace pl(g, lt, sc0 + i, n);
#pragma unroll
        for (int k = 0; k < KC; ++k)
          if (k < g.K) out[pl.at(k)] = acc[i][k];
      }
    }
  }
}

// y[s][c][t][n] = P_t(n) sum_k Phi_{tk} v_k(n) for every echo, v (in any layout of t) the
// transformed and scaled coefficients of the coil.  A pure streaming write (the T echoes are K / T
// times the input): one thread owns two neighbouring points and writes 16 bytes per echo, whole
// 512-byte runs per warp, so it is bound by HBM writes.  256x160, C = 12, T = 80, 8 slices
// (2.5 GB): 400 us, 0.93 of the measured copy bandwidth; 745 us when the column pass wrote the
// echoes itself in 64-byte runs, 445 us with the column pass now.  Where the points and planes give an SM
// fewer than eight CTAs, the echoes are shared out too, in chunks of 32 down to 8 (blockIdx.z): A x of one
// slice of 64x48, K = 4, C = 8, T = 32 10.0 -> 9.0 us, of 260x240, M = 2, C = 7, T = 80 64 -> 56 us.  WIDE: y is 16-byte aligned; an
// array that starts at an odd value of another takes 8-byte stores.
template <int KC, bool WIDE>
__global__ void __launch_bounds__(kThreads) k_expand_te(Geom g, TLayout lt, const float* __restrict__ phi,
                                                      const unsigned* __restrict__ bits,
                                                      const float2* v, float2* __restrict__ y, int tc) {
  extern __shared__ float sphi[];
  for (int i = threadIdx.x; i < g.T * g.K; i += blockDim.x) sphi[i] = phi[i];
  __syncthreads();
  pdl_wait();
  pdl_trigger();
  const int N = g.ny * g.nz;
  const int n = 2 * (blockIdx.x * blockDim.x + threadIdx.x);  // nz is even: both points share a row
  if (n >= N) return;
  const long long nsc = (long long)g.S * g.C;
  const int tlo = blockIdx.z * tc, thi = min(g.T, tlo + tc);  // this CTA's echoes
  for (long long sc = blockIdx.y; sc < nsc; sc += gridDim.y) {
    const TePlace pl(g, lt, sc, n);
    float4 a[KC];
#pragma unroll
    for (int k = 0; k < KC; ++k)
      a[k] = k < g.K ? *reinterpret_cast<const float4*>(v + pl.at(k)) : make_float4(0.f, 0.f, 0.f, 0.f);
    float2* yb = y + (sc * g.T + tlo) * (long long)N + n;
    for (int t0 = tlo; t0 < thi; t0 += 32) {  // tc is a multiple of 32 or divides it: no chunk leaves its word
      uint2 b = *reinterpret_cast<const uint2*>(bits + (long long)(t0 >> 5) * N + n);
      b.x >>= t0 & 31;
      b.y >>= t0 & 31;
      const int m = min(32, thi - t0);
#pragma unroll 4
      for (int i = 0; i < m; ++i) {
        float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
        const float* ph = sphi + (t0 + i) * g.K;
        if ((b.x >> i) & 1u) {
#pragma unroll
          for (int k = 0; k < KC; ++k)
            if (k < g.K) {
              o.x = fmaf(ph[k], a[k].x, o.x);
              o.y = fmaf(ph[k], a[k].y, o.y);
            }
        }
        if ((b.y >> i) & 1u) {
#pragma unroll
          for (int k = 0; k < KC; ++k)
            if (k < g.K) {
              o.z = fmaf(ph[k], a[k].z, o.z);
              o.w = fmaf(ph[k], a[k].w, o.w);
            }
        }
        if constexpr (WIDE) {
          __stcs(reinterpret_cast<float4*>(yb), o);
        } else {
          __stcs(yb, make_float2(o.x, o.y));
          __stcs(yb + 1, make_float2(o.z, o.w));
        }
        yb += N;
      }
    }
  }
}

cudaError_t launch_maps_prep(const Geom& g, const float2* maps_in, float2* maps_out, unsigned* lam_bits,
                             cudaStream_t st) {
  const long long tot = (long long)g.S * g.ny * g.nz;
  const unsigned grid = (unsigned)((tot + kThreads - 1) / kThreads);
  k_maps_prep<<<grid, kThreads, 0, st>>>(g, maps_in, maps_out, lam_bits);
  return cudaGetLastError();
}

cudaError_t launch_psi_build(const Geom& g, const float* phi, const uint8_t* mask, float* psi, unsigned* bits,
                             unsigned* lam_bits, cudaStream_t st) {
  const int N = g.ny * g.nz;
  const unsigned grid = (unsigned)((N + kPsiThreads - 1) / kPsiThreads);
  const size_t sm = sizeof(float) * g.T * g.K;
  if (g.K <= 4) k_psi_build<4><<<grid, kPsiThreads, sm, st>>>(g, phi, mask, psi, bits, lam_bits);
  else k_psi_build<8><<<grid, kPsiThreads, sm, st>>>(g, phi, mask, psi, bits, lam_bits);
  return cudaGetLastError();
}

template <int KC, int NP, int NS>
static cudaError_t project_go(const Geom& g, const TLayout& lt, const float* phi, const unsigned* bits, const float2* y,
                              float2* out, cudaStream_t st) {
  const int N = g.ny * g.nz;
  const long long planes = ((long long)g.S * g.C + NP - 1) / NP;
  dim3 grid((N + kThreads - 1) / kThreads, (unsigned)(planes < 65535 ? planes : 65535));
  return launch_pdl(k_project<KC, NP, NS>, grid, kThreads, sizeof(float) * g.T * g.K, st, g, lt, phi, bits, y, out);
}

cudaError_t launch_project(const Geom& g, const TLayout& lt, const float* phi, const unsigned* bits, const float2* y_te,
                           float2* y_proj, cudaStream_t st) {
  int nsm = 0;
  const cudaError_t e = sm_count(&nsm);
  if (e != cudaSuccess) return e;
  // four planes per thread read the bit words once for four; where that leaves SMs without a few
  // CTAs each, the k-space centre (every echo sampled) is the critical path: one plane per thread
  // and eight samples at a time
  const long long ctas = (long long)((g.ny * g.nz + kThreads - 1) / kThreads) * (((long long)g.S * g.C + 3) / 4);
  if (ctas >= 6LL * nsm)
    return g.K <= 4 ? project_go<4, 4, 2>(g, lt, phi, bits, y_te, y_proj, st)
                    : project_go<8, 4, 2>(g, lt, phi, bits, y_te, y_proj, st);
  return g.K <= 4 ? project_go<4, 1, 8>(g, lt, phi, bits, y_te, y_proj, st)
                  : project_go<8, 1, 8>(g, lt, phi, bits, y_te, y_proj, st);
}

cudaError_t launch_expand_te(const Geom& g, const TLayout& lt, const float* phi, const unsigned* bits, const float2* v,
                             float2* y_te, cudaStream_t st) {
  const int N2 = g.ny * g.nz / 2;
  const long long nsc = (long long)g.S * g.C;
  int nsm = 0;
  const cudaError_t e = sm_count(&nsm);
  if (e != cudaSuccess) return e;
  const long long ctas = (long long)((N2 + kThreads - 1) / kThreads) * nsc;
  int tc = (g.T + 31) / 32 * 32;
  while (tc > 8 && ctas * ((g.T + tc - 1) / tc) < 8LL * nsm) tc = tc > 32 ? 32 : tc / 2;
  dim3 grid((N2 + kThreads - 1) / kThreads, (unsigned)(nsc < 65535 ? nsc : 65535), (g.T + tc - 1) / tc);
  const size_t sm = sizeof(float) * g.T * g.K;
  const bool wide = ((uintptr_t)y_te & 15) == 0;
  auto kern = g.K <= 4 ? (wide ? k_expand_te<4, true> : k_expand_te<4, false>)
                       : (wide ? k_expand_te<8, true> : k_expand_te<8, false>);
  return launch_pdl(kern, grid, kThreads, sm, st, g, lt, phi, bits, v, y_te, tc);
}

}  // namespace t2sh
