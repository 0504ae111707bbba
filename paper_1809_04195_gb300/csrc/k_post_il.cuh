// TE images (see k_post.cu for the steps and the weights) for the line lengths of T2SH_POST_LENGTHS,
// N = RI RT, with the three transforms of a coil line chained through registers:
//   A  item j < RT:  S x at z = j + RT r (r < RI), DFT_RI                        -> exchange 1
//   B  item k1 < RI: twiddle, DFT_RT -> frequencies k1 + RI k2; homodyne weights and band mask on
//                    them, two IDFT_RT, conjugate twiddles                       -> exchange 2, 3
//   C  item j < RT:  two IDFT_RI -> h, l at z = j + RT r; their square in the phase of l is added to
//                    the thread's own sums over the coils
// CTA = (slice, band of 4 G rows), the row fastest, so exchanges have no bank conflicts (inner runs
// padded to odd, lines four apart modulo 16) and a warp's loads and stores are whole sectors.  The
// coil loop has two barriers; the next coil's map rows stream in by cp.async.  Bound by instruction
// issue (three line transforms per coil, echo and row): three echoes of the knee scan (320 slices of
// 256x160, C = 12) 23.6 -> 2.14 ms.
#pragma once

#include <algorithm>

#define T2SH_PACKED_ADD 1
#include "t2sh_device.cuh"

// length, RI, RT (RI <= RT: the image side keeps RI values of every map set and 2 RI of h and l)
#define T2SH_POST_LENGTHS_A(X)                                                                                   \
  X(48, 6, 8) X(64, 8, 8) X(80, 8, 10) X(100, 10, 10) X(120, 10, 12) X(144, 12, 12) X(160, 10, 16) X(200, 10, 20) \
  X(234, 13, 18) X(260, 13, 20) X(300, 15, 20) X(54, 6, 9)
#define T2SH_POST_LENGTHS_B(X)                                                                                   \
  X(50, 5, 10) X(72, 8, 9) X(90, 9, 10) X(104, 8, 13) X(128, 8, 16) X(150, 10, 15) X(162, 9, 18) X(208, 13, 16)   \
  X(240, 15, 16) X(270, 15, 18) X(320, 16, 20) X(60, 6, 10)
#define T2SH_POST_LENGTHS_C(X)                                                                                   \
  X(52, 4, 13) X(78, 6, 13) X(96, 8, 12) X(108, 9, 12) X(130, 10, 13) X(156, 12, 13) X(180, 12, 15) X(192, 12, 16) \
  X(216, 12, 18) X(256, 16, 16) X(288, 16, 18)

namespace t2sh {

namespace {

template <int N, int RI, int RT, int MC>
struct PostIl {
  static_assert(RI * RT == N && RI <= RT, "N = RI RT");
  static constexpr int G = RT % 8 == 0 ? 1 : 2;  // groups of four rows; two where one leaves a warp part empty
  static constexpr int ROWS = 4 * G;
  static constexpr int THREADS = (4 * RT * G + 31) / 32 * 32;
  static constexpr int SA = RI | 1, SC = RT | 1;  // exchange 1 [RT][RI], exchanges 2 and 3 [RI][RT]
  static constexpr int pad4(int n) { return n + ((4 - n % 16) + 16) % 16; }
  static constexpr int LA = pad4(RT * SA), LC = pad4(RI * SC);
  static constexpr int REGS = MC == 2 || RT >= 13 ? 160 : 128;  // 2.38 ms at 128 registers (N = 160), 2.16 at 160
  static constexpr int MINB = 65536 / (REGS * THREADS) > 0 ? 65536 / (REGS * THREADS) : 1;
  static constexpr size_t smem =
      sizeof(float2) * ((size_t)N + ROWS * (LA + 2 * LC) + 2 * (size_t)MC * ROWS * N);
};

template <int N, int RI, int RT, int MC>
__global__ void __launch_bounds__(PostIl<N, RI, RT, MC>::THREADS, PostIl<N, RI, RT, MC>::MINB)
    k_post_il(Geom g, const float2* __restrict__ tw_g, const float2* __restrict__ maps, const float* __restrict__ phi,
              const float2* __restrict__ alpha, PostArgs pa, float* __restrict__ out) {
  using P = PostIl<N, RI, RT, MC>;
  constexpr int ROWS = P::ROWS, SA = P::SA, SC = P::SC, LA = P::LA, LC = P::LC;
  extern __shared__ float2 smem[];
  const int K = g.K;
  const long long NN = (long long)g.ny * N;
  const int s = blockIdx.y, y0 = blockIdx.x * ROWS, rb = min(ROWS, g.ny - y0);
  // row 4 grp + (tid & 3) of the band; image-side item ji < RT, frequency-side item jf < RI
  const int i = threadIdx.x >> 2;
  const int gi = i / RT, ji = i - gi * RT, gf = i / RI, jf = i - gf * RI;
  const bool in_i = gi < P::G, in_f = gf < P::G;
  const int ri = 4 * (in_i ? gi : 0) + (threadIdx.x & 3), rf = 4 * (in_f ? gf : 0) + (threadIdx.x & 3);
  const bool on = in_i && ri < rb;
  float2* tw = smem;
  float2* e1 = tw + N;                   // [ROWS][LA]
  float2* e2 = e1 + ROWS * LA;           // [ROWS][LC], h
  float2* e3 = e2 + ROWS * LC;           // [ROWS][LC], l
  float2* mst = e3 + ROWS * LC;          // map rows x2 [MC][ROWS][N]
  for (int e = threadIdx.x; e < N; e += P::THREADS) tw[e] = tw_g[e];
  auto issue = [&](int c, int buf) {
    const float2* mp = maps + (long long)(s * g.C + c) * MC * NN + (long long)y0 * N;
    float2* md = mst + buf * MC * ROWS * N;
#pragma unroll
    for (int m = 0; m < MC; ++m)
      for (int e = threadIdx.x; e < rb * (N / 2); e += P::THREADS)  // the band's rows are contiguous
        cp_async16(md + m * ROWS * N + 2 * e, mp + (long long)m * NN + 2 * e);
  };
  const float inv_n = 1.f / (float)N;
  const long long img = (long long)s * MC * K * NN + (long long)(y0 + ri) * N + ji;
  for (int ti = 0; ti < pa.nte; ++ti) {
    const float* ph = phi + (size_t)pa.te[ti] * K;
    float2 x[MC][RI];  // the echo's image at this thread's points
#pragma unroll
    for (int m = 0; m < MC; ++m)
#pragma unroll
      for (int q = 0; q < RI; ++q) x[m][q] = make_float2(0.f, 0.f);
    if (on) {
      for (int k = 0; k < K; ++k) {
        const float f = ph[k];
#pragma unroll
        for (int m = 0; m < MC; ++m)
#pragma unroll
          for (int q = 0; q < RI; ++q) {
            const float2 a = alpha[img + (long long)(m * K + k) * NN + RT * q];
            x[m][q].x = fmaf(f, a.x, x[m][q].x);
            x[m][q].y = fmaf(f, a.y, x[m][q].y);
          }
      }
    }
    float acc[RI];
#pragma unroll
    for (int q = 0; q < RI; ++q) acc[q] = 0.f;
    issue(0, 0);
    cp_async_commit();
    cp_async_wait<0>();
    __syncthreads();
    for (int c = 0; c < g.C; ++c) {
      const int buf = c & 1;
      if (c + 1 < g.C) issue(c + 1, buf ^ 1);  // last read before the previous coil's second barrier
      cp_async_commit();
      if (in_i) {
        const float2* mrow = mst + (buf * MC * ROWS + ri) * N + ji;
        float2 v[RI];
#pragma unroll
        for (int q = 0; q < RI; ++q) {
          v[q] = make_float2(0.f, 0.f);
#pragma unroll
          for (int m = 0; m < MC; ++m) cfma(v[q], mrow[m * ROWS * N + RT * q], x[m][q]);
        }
        dft_r<RI, false>(v);
        float2* w = e1 + ri * LA + ji * SA;
#pragma unroll
        for (int q = 0; q < RI; ++q) w[q] = v[q];
      }
      __syncthreads();
      if (in_f) {
        const float2* r = e1 + rf * LA + jf;
        float2 h[RT], l[RT];
#pragma unroll
        for (int q = 0; q < RT; ++q) h[q] = r[q * SA];
#pragma unroll
        for (int q = 1; q < RT; ++q) h[q] = twiddle_mul<false>(h[q], tw[q * jf]);
        dft_r<RT, false>(h);
#pragma unroll
        for (int q = 0; q < RT; ++q) {
          const int d = jf + RI * q - N / 2;  // frequency
          const float hw = d < -pa.w ? 0.f : (d <= pa.w ? 1.f : 2.f);
          const bool band = d >= -pa.w && d <= pa.w;
          l[q] = band ? h[q] : make_float2(0.f, 0.f);
          h[q] = cscale(h[q], hw);
        }
        dft_r<RT, true>(h);
        dft_r<RT, true>(l);
#pragma unroll
        for (int q = 1; q < RT; ++q) {
          const float2 t = tw[q * jf];
          h[q] = twiddle_mul<true>(h[q], t);
          l[q] = twiddle_mul<true>(l[q], t);
        }
        float2 *wh = e2 + rf * LC + jf * SC, *wl = e3 + rf * LC + jf * SC;
#pragma unroll
        for (int q = 0; q < RT; ++q) {
          wh[q] = h[q];
          wl[q] = l[q];
        }
      }
      cp_async_wait<0>();
      __syncthreads();  // exchanges 2 and 3 are written, the next coil's maps are here
      if (in_i) {
        const float2 *rh = e2 + ri * LC + ji, *rl = e3 + ri * LC + ji;
        float2 h[RI], l[RI];
#pragma unroll
        for (int q = 0; q < RI; ++q) {
          h[q] = rh[q * SC];
          l[q] = rl[q * SC];
        }
        dft_r<RI, true>(h);
        dft_r<RI, true>(l);
#pragma unroll
        for (int q = 0; q < RI; ++q) {
          const float l2 = l[q].x * l[q].x + l[q].y * l[q].y;
          const float o = (l2 > 0.f ? (h[q].x * l[q].x + h[q].y * l[q].y) * rsqrtf(l2) : h[q].x) * inv_n;
          acc[q] = fmaf(o, o, acc[q]);
        }
      }
    }
    if (on) {
      float* o = out + ((long long)s * pa.nte + ti) * NN + (long long)(y0 + ri) * N + ji;
#pragma unroll
      for (int q = 0; q < RI; ++q) o[RT * q] = sqrtf(acc[q]);
    }
    // the next echo's first map copy lands in buffer 0, read last before this echo's final barriers
  }
}

template <int N, int RI, int RT, int MC>
cudaError_t post_il_go(const Geom& g, const float2* tw, const float2* maps, const float* phi, const float2* alpha,
                       const PostArgs& pa, float* out, cudaStream_t st) {
  using P = PostIl<N, RI, RT, MC>;
  if (P::smem > 220 * 1024) return cudaErrorNotSupported;
  const cudaError_t e = smem_optin((const void*)k_post_il<N, RI, RT, MC>, (int)P::smem);
  if (e != cudaSuccess) return e;
  dim3 grid((g.ny + P::ROWS - 1) / P::ROWS, g.S);
  k_post_il<N, RI, RT, MC><<<grid, P::THREADS, P::smem, st>>>(g, tw, maps, phi, alpha, pa, out);
  return cudaGetLastError();
}

}  // namespace

#define T2SH_POST_PART(name, LENGTHS)                                                                          \
  cudaError_t name(const Geom& g, const float2* tw, const float2* maps, const float* phi, const float2* alpha, \
                   const PostArgs& pa, float* out, cudaStream_t st) {                                          \
    switch (g.nz) {                                                                                            \
      LENGTHS(T2SH_POST_CASE)                                                                                  \
      default: return cudaErrorNotSupported;                                                                   \
    }                                                                                                          \
  }
#define T2SH_POST_CASE(n, ri, rt)                                                              \
  case n:                                                                                      \
    return g.M == 1 ? post_il_go<n, ri, rt, 1>(g, tw, maps, phi, alpha, pa, out, st)           \
                    : post_il_go<n, ri, rt, 2>(g, tw, maps, phi, alpha, pa, out, st);

}  // namespace t2sh
