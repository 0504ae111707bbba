// Row (kz) passes on the interleaved per-coil intermediate t[s][c][y][z / 4][slot][z % 4] of
// k_col_il.cuh (four basis images), for the line lengths of T2SH_ROW_LENGTHS: N = RI RT.
//
// CTA = (slice, band of RB rows), the coil loop inside (Algorithm 1 puts it
// outermost): the image rows stay in registers and only t goes to memory.  A line is transformed
// in two register stages with one shared-memory exchange, RI items of radix RT on the side of t
// and RT items of radix RI on the image side:
//   forward  A: item j < RT forms S x at z = j + RT r (r < RI), DFT_RI
//            B: item j < RI: twiddle, DFT_RT                       -> t at z = j + RI k
//   adjoint  A: item j < RI: IDFT_RT of t at z = j + RI r
//            B: item j < RT: twiddle, IDFT_RI, conj(S) and the sum over coils at z = j + RT k
// The basis image is the fastest thread index in every stage: a half-warp is four columns of all
// four images, so on the side of t it touches exactly one 128-byte line per access (t is bound by
// the number of lines a load touches as much as by bytes), the map values of the image side are
// broadcast, and with the four lines' exchange windows starting four (mod 16) apart no stage has
// bank conflicts.  The adjoint requests the next coil's t one coil ahead.
//
// Bound by HBM (maps and t once each, image rows once).  Knee scan (320 slices of 256x160, C = 12,
// 6.71 GB per launch): forward 1.11 -> 0.99 ms, adjoint 1.15 -> 1.01 ms against the planar passes,
// 0.98 of the measured copy bandwidth; Table I (M = 2, 7.19 GB): 1.39 -> 1.04 and 1.48 -> 1.18 ms.
// The adjoint's loads in flight wait in L1, so the SM's split is set to what the resident CTAs'
// shared memory needs: after a column pass that leaves 28 KB of L1, 1.59 ms (M = 2, 240 points)
// against 1.18, 1.28 against 1.05 (160 points).
// Reading t with half-warps of one image (four lines per load instead of one) took 1.43 ms, and
// storing it as runs of R1 columns (partial sectors) 1.30 ms.
#pragma once

#include <algorithm>

// packed two-lane complex additions in the butterflies: fewer issue slots
#define T2SH_PACKED_ADD 1
#include "launch.h"
#include "t2sh_device.cuh"

namespace t2sh {

namespace {

// length, RI, RT, rows of a CTA: multiples of four from 48 to 320 that are two radices of at most 20,
// RI a multiple of four so that a half-warp's columns on the side of t are one aligned chunk.  The
// rows are four digits, forward and adjoint with one map set, then with two: each the fastest of one
// to four at 60 slices of 128 x 192 points' worth of lines, C = 10.  One row where the items of both
// sides fill their warps or the registers limit the CTAs, two or three where 4 RI or 4 RT leaves a warp
// part empty: 144 points 5.8 -> 6.1 TB/s forward, 72 points 4.6 -> 6.0, 52 points 2.8 -> 4.9, 256 points
// 6.0 with one row and with two.  Balanced radices for short lines, which use more threads of a warp
// on the image side: 48 = 8 x 6 5.9 and 5.3 TB/s (forward, adjoint), 16 x 3 3.0 and 2.5; 64 = 8 x 8
// 6.5 and 5.7, 16 x 4 3.8 and 3.2; 160 = 8 x 20 is slower than 16 x 10 (5.7 and 6.1).
#define T2SH_ROW_LENGTHS(X) \
  X(48, 8, 6, 1111) X(52, 4, 13, 2222) X(60, 12, 5, 2222) X(64, 8, 8, 2121) X(72, 8, 9, 2233)               \
  X(80, 8, 10, 3233) X(96, 8, 12, 2222) X(100, 20, 5, 2211) X(104, 8, 13, 2222) X(108, 12, 9, 2222)         \
  X(120, 12, 10, 2222) X(128, 16, 8, 1222) X(144, 12, 12, 2222) X(156, 12, 13, 2211) X(160, 16, 10, 1211)   \
  X(180, 12, 15, 1111) X(192, 16, 12, 1111) X(200, 20, 10, 2212) X(208, 16, 13, 1111) X(216, 12, 18, 2222)  \
  X(240, 16, 15, 1111) X(256, 16, 16, 1111) X(260, 20, 13, 2211) X(288, 16, 18, 2212) X(300, 20, 15, 2212)  \
  X(320, 16, 20, 2211)

constexpr int row_rows(int n, bool adj, int mc) {
  int d = 1111;
#define X(len, ri, rt, r) d = n == len ? r : d;
  T2SH_ROW_LENGTHS(X)
#undef X
  return d / (mc == 1 ? (adj ? 100 : 1000) : (adj ? 1 : 10)) % 10;
}

template <int N, int RI_, int RT_, int MODE, int MC>
struct RowIl {
  static constexpr int RI = RI_, RT = RT_;
  static_assert(RI * RT == N && RI % 4 == 0, "N = RI RT");
  // exchange [RT items][RI] (forward) or [RI items][RT] (adjoint), the inner run padded to odd
  static constexpr int S = (MODE == ROW_FWD ? RI : RT) | 1;
  static constexpr int L0 = (MODE == ROW_FWD ? RT : RI) * S;
  static constexpr int LINE = L0 + ((4 - L0 % 16) + 16) % 16;
  static constexpr int J = RI > RT ? RI : RT;
  // MINB holds the registers to 80 (forward), 96 or 128; 144 for the adjoint of two map sets at radix
  // 16 and more on both sides, which otherwise spills (288 points 4.2 -> 4.5 TB/s, 320 points 4.2 -> 5.0,
  // 256 points 5.2 -> 5.4; 240 points 5.3 with 128 and 5.1 with 144).
  static constexpr int RB = row_rows(N, MODE == ROW_ADJ, MC);
  static constexpr int THREADS = (4 * J * RB + 31) / 32 * 32;
  static constexpr int REGS = MC == 2 ? (RI > 16 ? 168 : MODE == ROW_ADJ && RI == 16 && RT >= 16 ? 144 : 128) : MODE == ROW_FWD ? (RI > 16 || RT > 16 ? 96 : 80)
                                                                               : RT <= 10 && RI <= 16 ? 96 : 128;
  static constexpr int MINB = 65536 / (REGS * THREADS) > 0 ? 65536 / (REGS * THREADS) : 1;
  static constexpr size_t smem = sizeof(float2) * ((size_t)N + 4 * RB * LINE + 2 * (size_t)MC * RB * N);
};

// barrier among all threads of the cluster, shared-memory writes before it visible after it
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// *p in the shared memory of CTA `rank` of the cluster
__device__ __forceinline__ float2 cluster_lds2(const float2* p, int rank) {
  unsigned a;
  float2 v;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_u32(p)), "r"(rank));
  asm volatile("ld.shared::cluster.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(a) : "memory");
  return v;
}

// CTAs that share a band's coils: as many as keep the whole plan's launch within one wave of resident CTAs (a
// launch over some of its slices takes the same number: it sets the order of the sum over the coils), more
// than four only within half a wave, and at most eight, the portable size of the cluster in which the
// adjoint sums over the coils.  One slice of 64 x 48, C = 8: forward 4.6 -> 2.3 us, adjoint 5.6 -> 4.2,
// a 50-iteration solve 1.22 -> 1.11 ms (1.14 with four CTAs); two slices with M = 2: 1.26 ms with four,
// 1.35 with eight.  Beyond one wave the sum costs the adjoint more than a fuller last wave gives (32
// slices of 192 x 192: 148 -> 167 us with a split by waves).
inline int row_split(long long ctas, long long resident, int C) {
  for (int n = std::min(8, C); n > 1; --n) {
    const int cs = (C + n - 1) / n;
    if ((C + cs - 1) / cs == n && ctas * n <= (n > 4 ? resident / 2 : resident)) return n;  // every CTA has a coil
  }
  return 1;
}

template <int N, int RI, int RT, int MODE, int MC>
__global__ void __launch_bounds__(RowIl<N, RI, RT, MODE, MC>::THREADS, RowIl<N, RI, RT, MODE, MC>::MINB)
    k_row_il(Geom g, int trb, int cs, const float2* __restrict__ tw_g, const float2* __restrict__ maps,
             const float2* x, float2* t, float2* __restrict__ out) {
  using R = RowIl<N, RI, RT, MODE, MC>;
  constexpr int LINE = R::LINE, S = R::S, RB = R::RB;
  extern __shared__ float2 smem[];
  const int NN = g.ny * N;
  const int s = blockIdx.y, y0 = blockIdx.x * RB;
  const int rb = min(RB, g.ny - y0);
  const int c0 = blockIdx.z * cs, c1 = min(g.C, c0 + cs);  // this CTA's coils
  // basis image k, item i of the band: t-side items (jt < RI, row rt), image-side items (ji < RT, row ri)
  const int k = threadIdx.x & 3, i = threadIdx.x >> 2;
  const int rt = i / RI, jt = i - rt * RI;
  const int ri = i / RT, ji = i - ri * RT;
  constexpr bool ALL_T = 4 * RI * RB == R::THREADS;  // every thread has an item on the side of t
  const bool in_t = ALL_T || rt < RB, on_t = rt < rb, on_i = ri < rb;
  float2* tw = smem;
  float2* ex = tw + N;               // [RB][4][LINE]
  float2* mst = ex + 4 * RB * LINE;  // map rows x2 [MC][RB][N]
  for (int e = threadIdx.x; e < N; e += R::THREADS) tw[e] = tw_g[e];

  auto issue = [&](int c, int buf) {
    constexpr int H = N / 2;  // 16-byte copies per row
    const float2* mp = maps + (long long)(s * g.C + c) * MC * NN + (long long)y0 * N;
    float2* md = mst + buf * MC * RB * N;
    for (int e = threadIdx.x; e < MC * RB * H; e += R::THREADS) {
      const int line = e / H, col = 2 * (e - line * H);
      const int m = line / RB, row = line - m * RB;
      if (row < rb) cp_async16(md + line * N + col, mp + (long long)m * NN + row * N + col);
    }
  };
  issue(c0, 0);  // the plan's maps: not written by any kernel of the solve
  cp_async_commit();

  // t-side address of coil c0: row, slot and the thread's column within its line of t
  const int yt = y0 + (in_t ? rt : 0);
  const int slot = trb ? (k + yt % trb + yt / trb) & 3 : k;
  float2* tp = t + ((long long)(s * g.C + c0) * g.ny + yt) * (4 * N) + slot * 4 + (jt >> 2) * 16 + (jt & 3);
  const long long tcoil = 4LL * NN;
  const float2* exi = ex + ((ri < RB ? ri : 0) * 4 + k) * LINE;
  float2* ext = ex + ((in_t ? rt : 0) * 4 + k) * LINE;
  const long long img = (long long)s * MC * 4 * NN + (long long)k * NN + (long long)(y0 + ri) * N + ji;

  pdl_wait();
  pdl_trigger();
  if constexpr (MODE == ROW_FWD) {
    float2 xr[MC][RI];
#pragma unroll
    for (int m = 0; m < MC; ++m)
#pragma unroll
      for (int q = 0; q < RI; ++q)
        xr[m][q] = on_i ? x[img + (long long)m * 4 * NN + RT * q] : make_float2(0.f, 0.f);
    float2* exw = const_cast<float2*>(exi) + ji * S;
    for (int c = c0; c < c1; ++c) {
      const int buf = (c - c0) & 1;
      cp_async_wait<0>();
      __syncthreads();  // coil c's maps are here, and nobody is in the previous coil any more
      if (c + 1 < c1) issue(c + 1, buf ^ 1);
      cp_async_commit();
      if (ri < RB) {
        const float2* mrow = mst + (buf * MC * RB + ri) * N + ji;
        float2 a[RI];
#pragma unroll
        for (int q = 0; q < RI; ++q) {
          float2 v = make_float2(0.f, 0.f);
#pragma unroll
          for (int m = 0; m < MC; ++m) cfma(v, mrow[m * RB * N + RT * q], xr[m][q]);
          a[q] = v;
        }
        dft_r<RI, false>(a);
#pragma unroll
        for (int q = 0; q < RI; ++q) exw[q] = a[q];
      }
      __syncthreads();
      if (in_t) {
        float2 b[RT];
#pragma unroll
        for (int q = 0; q < RT; ++q) b[q] = ext[q * S + jt];
#pragma unroll
        for (int q = 1; q < RT; ++q) b[q] = twiddle_mul<false>(b[q], tw[q * jt]);
        dft_r<RT, false>(b);
        if (on_t) {
#pragma unroll
          for (int q = 0; q < RT; ++q) tp[q * (4 * RI)] = b[q];
        }
      }
      tp += tcoil;
    }
  } else {
    float2 acc[MC][RI];
#pragma unroll
    for (int m = 0; m < MC; ++m)
#pragma unroll
      for (int q = 0; q < RI; ++q) acc[m][q] = make_float2(0.f, 0.f);
    float2 tn[RT];
#pragma unroll
    for (int q = 0; q < RT; ++q) tn[q] = on_t ? tp[q * (4 * RI)] : make_float2(0.f, 0.f);
    for (int c = c0; c < c1; ++c) {
      const int buf = (c - c0) & 1;
      cp_async_wait<0>();
      __syncthreads();  // coil c's maps are here, and nobody is in the previous coil any more
      if (c + 1 < c1) issue(c + 1, buf ^ 1);
      cp_async_commit();
      float2 a[RT];
#pragma unroll
      for (int q = 0; q < RT; ++q) a[q] = tn[q];
      tp += tcoil;
      if (c + 1 < c1) {
#pragma unroll
        for (int q = 0; q < RT; ++q) tn[q] = on_t ? tp[q * (4 * RI)] : make_float2(0.f, 0.f);
      }
      if (in_t) {
        dft_r<RT, true>(a);
#pragma unroll
        for (int q = 0; q < RT; ++q) ext[jt * S + q] = a[q];
      }
      __syncthreads();
      if (ri < RB) {
        float2 b[RI];
#pragma unroll
        for (int q = 0; q < RI; ++q) b[q] = exi[q * S + ji];
#pragma unroll
        for (int q = 1; q < RI; ++q) b[q] = twiddle_mul<true>(b[q], tw[q * ji]);
        dft_r<RI, true>(b);
        const float2* mrow = mst + (buf * MC * RB + ri) * N + ji;
#pragma unroll
        for (int m = 0; m < MC; ++m)
#pragma unroll
          for (int q = 0; q < RI; ++q) cfmac(acc[m][q], mrow[m * RB * N + RT * q], b[q]);
      }
    }
    if (gridDim.z == 1) {
      if (on_i) {
#pragma unroll
        for (int m = 0; m < MC; ++m)
#pragma unroll
          for (int q = 0; q < RI; ++q) out[img + (long long)m * 4 * NN + RT * q] = acc[m][q];
      }
    } else {
      // the cluster's CTAs hold the sums over their coils: each leaves its own in shared memory, in
      // the order [map set][row][column][image], and adds up a share of all of them
      static_assert(LINE >= N, "the sums fit in the exchange and the map rows");
      cp_async_wait<0>();
      __syncthreads();
      if (ri < RB) {
#pragma unroll
        for (int m = 0; m < MC; ++m)
#pragma unroll
          for (int q = 0; q < RI; ++q) ex[((m * RB + ri) * N + ji + RT * q) * 4 + k] = acc[m][q];
      }
      cluster_sync();
      const int ns = gridDim.z;
      for (int e = blockIdx.z * R::THREADS + threadIdx.x; e < MC * RB * N * 4; e += ns * R::THREADS) {
        float2 v = cluster_lds2(ex + e, 0);
        for (int r = 1; r < ns; ++r) {
          const float2 w = cluster_lds2(ex + e, r);
          v.x += w.x;
          v.y += w.y;
        }
        const int pos = (e >> 2) % N, row = (e >> 2) / N % RB, m = (e >> 2) / (N * RB);
        if (row < rb) out[((long long)(s * MC + m) * 4 + (e & 3)) * NN + (long long)(y0 + row) * N + pos] = v;
      }
      cluster_sync();  // nobody leaves while its sums are read
    }
  }
  cp_async_wait<0>();
}

template <int N, int RI, int RT, int MODE, int MC>
cudaError_t row_il_go(const Geom& g, int trb, const float2* tw, const float2* maps, const float2* x, float2* t,
                      float2* out, cudaStream_t st) {
  using R = RowIl<N, RI, RT, MODE, MC>;
  const cudaError_t e = smem_optin((const void*)k_row_il<N, RI, RT, MODE, MC>, (int)R::smem,
                                   R::MINB * ((int)R::smem + 1024));
  if (e != cudaSuccess) return e;
  int nsm = 0;
  const cudaError_t es = sm_count(&nsm);
  if (es != cudaSuccess) return es;
  const int nb = (g.ny + R::RB - 1) / R::RB;
  const int ns = row_split((long long)nb * g.Sp, (long long)nsm * R::MINB, g.C);
  const int cs = (g.C + ns - 1) / ns;
  return launch_pdl_cluster(k_row_il<N, RI, RT, MODE, MC>, dim3(nb, g.S, ns), MODE == ROW_ADJ ? ns : 1, R::THREADS,
                            R::smem, st, g, trb, cs, tw, maps, x, t, out);
}

}  // namespace

// compiled once per direction (T2SH_ROW_MODE), so that the unrolled kernels build in parallel
#define T2SH_ROW_NAME2(m) launch_row_il_##m
#define T2SH_ROW_NAME(m) T2SH_ROW_NAME2(m)
cudaError_t T2SH_ROW_NAME(T2SH_ROW_MODE)(const Geom& g, int trb, const float2* tw, const float2* maps, const float2* x,
                                         float2* t, float2* out, cudaStream_t st) {
  switch (g.nz) {
#define X(n, ri, rt, r)                                                                                   \
  case n:                                                                                                \
    return g.M == 1 ? row_il_go<n, ri, rt, T2SH_ROW_MODE, 1>(g, trb, tw, maps, x, t, out, st)            \
                    : row_il_go<n, ri, rt, T2SH_ROW_MODE, 2>(g, trb, tw, maps, x, t, out, st);
    T2SH_ROW_LENGTHS(X)
#undef X
    default: return cudaErrorNotSupported;
  }
}

#if T2SH_ROW_FIRST
cudaError_t launch_row_il_ROW_ADJ(const Geom& g, int trb, const float2* tw, const float2* maps, const float2* x,
                                  float2* t, float2* out, cudaStream_t st);

bool row_il_supported(const Geom& g) {
  if (g.K != 4 || g.M > 2) return false;
  switch (g.nz) {
#define X(n, ri, rt, r) case n:
    T2SH_ROW_LENGTHS(X)
#undef X
    return true;
    default: return false;
  }
}

cudaError_t launch_row_il(const Geom& g, RowMode mode, int trb, const float2* tw_z, const float2* maps,
                          const float2* x, float2* t, float2* out, cudaStream_t st) {
  if (!row_il_supported(g)) return cudaErrorNotSupported;
  return mode == ROW_FWD ? launch_row_il_ROW_FWD(g, trb, tw_z, maps, x, t, out, st)
                         : launch_row_il_ROW_ADJ(g, trb, tw_z, maps, x, t, out, st);
}
#endif

}  // namespace t2sh
