// Row (kz) passes on the interleaved per-coil intermediate t[s][c][y][z / 4][slot][z % 4] of
// k_col_il.cu (four basis images), for line lengths N = 16 R1.
//
// CTA = (slice, band of RB rows), 64 RB threads, the coil loop inside (Algorithm 1 puts it
// outermost): the image rows stay in registers and only t goes to memory.  A line is transformed
// in two register stages with one shared-memory exchange, 16 items of radix R1 on the side of t
// and R1 items of radix 16 on the image side:
//   forward  A: item j < R1 forms S x at z = j + R1 r (r < 16), DFT_16
//            B: item j < 16: twiddle, DFT_R1                       -> t at z = j + 16 k
//   adjoint  A: item j < 16: IDFT_R1 of t at z = j + 16 r
//            B: item j < R1: twiddle, IDFT_16, conj(S) and the sum over coils at z = j + R1 k
// The basis image is the fastest thread index in every stage: a half-warp is four columns of all
// four images, so on the side of t it touches exactly one 128-byte line per access (t is bound by
// the number of lines a load touches as much as by bytes), the map values of the image side are
// broadcast, and with the four lines' exchange windows starting four (mod 16) apart no stage has
// bank conflicts.  The adjoint requests the next coil's t one coil ahead.
//
// Bound by HBM (maps and t once each, image rows once).  Knee scan (320 slices of 256x160, C = 12,
// 6.71 GB per launch): forward 1.12 -> 1.01 ms, adjoint 1.15 -> 1.02 ms against the planar passes,
// 0.97 of the measured copy bandwidth; Table I (M = 2, 7.19 GB): 1.39 -> 1.04 and 1.48 -> 1.22 ms.
// Reading t with half-warps of one image (four lines per load instead of one) took 1.43 ms, and
// storing it as runs of R1 columns (partial sectors) 1.30 ms.
#include <algorithm>

// packed two-lane complex additions in the butterflies: fewer issue slots
#define T2SH_PACKED_ADD 1
#include "t2sh_device.cuh"

namespace t2sh {

namespace {

template <int N, int MODE, int MC>
struct RowIl {
  static constexpr int R1 = N / 16;
  static constexpr int SA = (R1 % 2) ? R1 : R1 + 1;  // [16 items][R1] exchange stride (adjoint)
  static constexpr int SB = 17;                      // [R1 items][16] exchange stride (forward)
  static constexpr int S = MODE == ROW_FWD ? SB : SA;
  static constexpr int L0 = MODE == ROW_FWD ? R1 * SB : 16 * SA;
  static constexpr int LINE = L0 + ((4 - L0 % 16) + 16) % 16;
  // One-row bands (64 threads) where the 4 R1 image-side items fill their warps or lines are
  // short, two-row bands otherwise: adjoint at N = 160 1.02 ms with two rows, 1.09 with one (40
  // items leave the second warp three quarters empty); forward with two map sets at N = 240
  // 1.04 ms with one row, 1.09 with two.  MINB holds the registers to 80 (forward), 96 or 128.
  static constexpr int RB = (MODE == ROW_FWD || R1 <= 4 || R1 == 8 || R1 >= 15) ? 1 : 2;
  static constexpr int THREADS = 64 * RB;
  static constexpr int MINB = (MC == 2 ? 8 : MODE == ROW_FWD ? 12 : R1 <= 10 ? 10 : 8) / RB;
  static constexpr size_t smem = sizeof(float2) * ((size_t)N + 4 * RB * LINE + 2 * (size_t)MC * RB * N);
};

template <int N, int MODE, int MC>
__global__ void __launch_bounds__(RowIl<N, MODE, MC>::THREADS, RowIl<N, MODE, MC>::MINB)
    k_row_il(Geom g, int trb, const float2* __restrict__ tw_g, const float2* __restrict__ maps,
             const float2* __restrict__ x, float2* __restrict__ t, float2* __restrict__ out) {
  using R = RowIl<N, MODE, MC>;
  constexpr int R1 = R::R1, LINE = R::LINE, S = R::S, RB = R::RB;
  extern __shared__ float2 smem[];
  const int NN = g.ny * N;
  const int s = blockIdx.y, y0 = blockIdx.x * RB;
  const int rb = min(RB, g.ny - y0);
  // basis image k, item i of the band: t-side items (jt < 16, row rt), image-side items (ji < R1, row ri)
  const int k = threadIdx.x & 3, i = threadIdx.x >> 2;
  const int jt = i & 15, rt = i >> 4;
  const int ri = i / R1, ji = i - ri * R1;
  const bool on_t = rt < rb, on_i = ri < rb;
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
  issue(0, 0);
  cp_async_commit();

  // t-side address of coil 0: row, slot and the thread's column within its line of t
  const int yt = y0 + rt;
  float2* tp = t + ((long long)s * g.C * g.ny + yt) * (4 * N) + ((k + yt % trb + yt / trb) & 3) * 4 + (jt >> 2) * 16 + (jt & 3);
  const long long tcoil = 4LL * NN;
  const float2* exi = ex + ((ri < RB ? ri : 0) * 4 + k) * LINE;
  float2* ext = ex + (rt * 4 + k) * LINE;
  const long long img = (long long)s * MC * 4 * NN + (long long)k * NN + (long long)(y0 + ri) * N + ji;

  if constexpr (MODE == ROW_FWD) {
    float2 xr[MC][16];
#pragma unroll
    for (int m = 0; m < MC; ++m)
#pragma unroll
      for (int q = 0; q < 16; ++q)
        xr[m][q] = on_i ? x[img + (long long)m * 4 * NN + R1 * q] : make_float2(0.f, 0.f);
    float2* exw = const_cast<float2*>(exi) + ji * S;
    for (int c = 0; c < g.C; ++c) {
      const int buf = c & 1;
      cp_async_wait<0>();
      __syncthreads();  // coil c's maps are here, and nobody is in the previous coil any more
      if (c + 1 < g.C) issue(c + 1, buf ^ 1);
      cp_async_commit();
      if (ri < RB) {
        const float2* mrow = mst + (buf * MC * RB + ri) * N + ji;
        float2 a[16];
#pragma unroll
        for (int q = 0; q < 16; ++q) {
          float2 v = make_float2(0.f, 0.f);
#pragma unroll
          for (int m = 0; m < MC; ++m) cfma(v, mrow[m * RB * N + R1 * q], xr[m][q]);
          a[q] = v;
        }
        dft16<false>(a);
#pragma unroll
        for (int q = 0; q < 16; ++q) exw[q] = a[q];
      }
      __syncthreads();
      float2 b[R1];
#pragma unroll
      for (int q = 0; q < R1; ++q) b[q] = ext[q * S + jt];
#pragma unroll
      for (int q = 1; q < R1; ++q) b[q] = twiddle_mul<false>(b[q], tw[q * jt]);
      dft_r<R1, false>(b);
      if (on_t) {
#pragma unroll
        for (int q = 0; q < R1; ++q) tp[q * 64] = b[q];
      }
      tp += tcoil;
    }
  } else {
    float2 acc[MC][16];
#pragma unroll
    for (int m = 0; m < MC; ++m)
#pragma unroll
      for (int q = 0; q < 16; ++q) acc[m][q] = make_float2(0.f, 0.f);
    float2 tn[R1];
#pragma unroll
    for (int q = 0; q < R1; ++q) tn[q] = on_t ? tp[q * 64] : make_float2(0.f, 0.f);
    for (int c = 0; c < g.C; ++c) {
      const int buf = c & 1;
      cp_async_wait<0>();
      __syncthreads();  // coil c's maps are here, and nobody is in the previous coil any more
      if (c + 1 < g.C) issue(c + 1, buf ^ 1);
      cp_async_commit();
      float2 a[R1];
#pragma unroll
      for (int q = 0; q < R1; ++q) a[q] = tn[q];
      tp += tcoil;
      if (c + 1 < g.C) {
#pragma unroll
        for (int q = 0; q < R1; ++q) tn[q] = on_t ? tp[q * 64] : make_float2(0.f, 0.f);
      }
      dft_r<R1, true>(a);
#pragma unroll
      for (int q = 0; q < R1; ++q) ext[jt * S + q] = a[q];
      __syncthreads();
      if (ri < RB) {
        float2 b[16];
#pragma unroll
        for (int q = 0; q < 16; ++q) b[q] = exi[q * S + ji];
#pragma unroll
        for (int q = 1; q < 16; ++q) b[q] = twiddle_mul<true>(b[q], tw[q * ji]);
        dft16<true>(b);
        const float2* mrow = mst + (buf * MC * RB + ri) * N + ji;
#pragma unroll
        for (int m = 0; m < MC; ++m)
#pragma unroll
          for (int q = 0; q < 16; ++q) cfmac(acc[m][q], mrow[m * RB * N + R1 * q], b[q]);
      }
    }
    if (on_i) {
#pragma unroll
      for (int m = 0; m < MC; ++m)
#pragma unroll
        for (int q = 0; q < 16; ++q) out[img + (long long)m * 4 * NN + R1 * q] = acc[m][q];
    }
  }
  cp_async_wait<0>();
}

template <int N, int MODE, int MC>
cudaError_t row_il_go(const Geom& g, int trb, const float2* tw, const float2* maps, const float2* x, float2* t,
                      float2* out, cudaStream_t st) {
  using R = RowIl<N, MODE, MC>;
  const cudaError_t e = smem_optin((const void*)k_row_il<N, MODE, MC>, (int)R::smem);
  if (e != cudaSuccess) return e;
  dim3 grid((g.ny + R::RB - 1) / R::RB, g.S);
  k_row_il<N, MODE, MC><<<grid, R::THREADS, R::smem, st>>>(g, trb, tw, maps, x, t, out);
  return cudaGetLastError();
}

template <int N>
cudaError_t row_il_n(const Geom& g, RowMode mode, int trb, const float2* tw, const float2* maps, const float2* x,
                     float2* t, float2* out, cudaStream_t st) {
  if (mode == ROW_FWD)
    return g.M == 1 ? row_il_go<N, ROW_FWD, 1>(g, trb, tw, maps, x, t, out, st)
                    : row_il_go<N, ROW_FWD, 2>(g, trb, tw, maps, x, t, out, st);
  return g.M == 1 ? row_il_go<N, ROW_ADJ, 1>(g, trb, tw, maps, x, t, out, st)
                  : row_il_go<N, ROW_ADJ, 2>(g, trb, tw, maps, x, t, out, st);
}

}  // namespace

bool row_il_supported(const Geom& g) {
  if (g.K != 4 || g.M > 2) return false;
  for (int n : {48, 64, 96, 128, 160, 192, 240, 256})
    if (g.nz == n) return true;
  return false;
}

cudaError_t launch_row_il(const Geom& g, RowMode mode, int trb, const float2* tw_z, const float2* maps,
                          const float2* x, float2* t, float2* out, cudaStream_t st) {
  if (!row_il_supported(g)) return cudaErrorNotSupported;
  switch (g.nz) {
    case 48: return row_il_n<48>(g, mode, trb, tw_z, maps, x, t, out, st);
    case 64: return row_il_n<64>(g, mode, trb, tw_z, maps, x, t, out, st);
    case 96: return row_il_n<96>(g, mode, trb, tw_z, maps, x, t, out, st);
    case 128: return row_il_n<128>(g, mode, trb, tw_z, maps, x, t, out, st);
    case 160: return row_il_n<160>(g, mode, trb, tw_z, maps, x, t, out, st);
    case 192: return row_il_n<192>(g, mode, trb, tw_z, maps, x, t, out, st);
    case 240: return row_il_n<240>(g, mode, trb, tw_z, maps, x, t, out, st);
    default: return row_il_n<256>(g, mode, trb, tw_z, maps, x, t, out, st);
  }
}

}  // namespace t2sh
