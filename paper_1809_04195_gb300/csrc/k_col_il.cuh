// Column (ky) passes on the interleaved per-coil intermediate, four basis images (K = 4).
//
// Layout of t:  t[s][c][y][z / 4][slot][z % 4], slot = (k + y mod RB + y div RB) mod 4.  The four
// basis images of four neighbouring columns are one 128-byte line, so a column tile (N rows of
// one line each) is a plain two-dimensional tensor-map box, every DRAM sector of it is used, and
// the rotation of the slots with the row, which the row passes apply for free, makes every
// shared-memory access below conflict free without padding.
//
// Transform: N = RA RB, decimation in frequency forward and in time backward, in place:
//   A   item j < RB:  DFT_RA over q of rows j + RB q             -> the same rows
//   B   item k1 < RA: twiddle, DFT_RB over j of rows j + RB k1   -> frequencies k1 + RA k2 in
//       registers, the 4 x 4 space-time kernel Psi on them, IDFT_RB, conjugate twiddle
//                                                                -> the same rows
//   A'  item j < RB:  IDFT_RA over q of rows j + RB q            -> global memory
// A thread owns one column w and two basis images (pair kp) of its item's rows; Psi takes the
// other two from the neighbouring lane.  The transform never reorders the column: frequencies
// stay where stage B leaves them, and Psi is read in that order.  A tile has three barriers among
// its own 64 ... 160 threads.
//
// Bound by shared-memory wavefronts (77 % of the L1 data pipe while active at 256 points), issue and HBM
// together.  Knee scan (320 slices of 256x160, C = 12, 10.1 GB per launch): 2.52 -> 1.69 ms against the
// 8-column planar tiles of k_col_tma.cu, 0.88 of the measured copy bandwidth; 260-point columns of
// Table I (8.05 GB): 2.51 -> 1.72 ms.  What it saves: the two exchanges around Psi (a frequency's four
// images sit in two neighbouring lanes), two of five barriers, and the barriers join 128 threads instead
// of 512, so the four groups of an SM drift apart and hide each other's stalls.  Psi stays in shared
// memory for a whole run of slices and coils instead of being copied per tile.  Where RB is even the two
// lanes of a point take half of its frequencies each, which reads ten floats of Psi per point instead of
// sixteen: 200 slices of 256x160 1.08 -> 1.06 ms, 60 slices of 288x96 0.28 -> 0.26, and of 320x96 0.39 ->
// 0.30, where the shared memory that this frees holds a spare buffer.  With all four images in one thread the code outgrew the instruction cache (2.58 ms, a
// third of the stalls "no instruction"); five groups at 96 registers took 1.91 ms at 256 points and
// 0.26 instead of 0.17 at 192.
#pragma once

#include <cuda.h>

#include <algorithm>

// packed two-lane complex additions: 1.77 -> 1.75 ms at 256 points, 1.94 -> 1.86 ms at 260 (before spare buffers)
#define T2SH_PACKED_ADD 1

#include "launch.h"
#include "t2sh_device.cuh"

// length, RA, RB: even products of 2, 3, 5 and 13 from 48 to 320 that are two radices of at most 20
#define T2SH_IL_LENGTHS_A(X) X(256, 16, 16) X(48, 8, 6) X(100, 10, 10) X(144, 12, 12) X(54, 9, 6) X(234, 18, 13)
#define T2SH_IL_LENGTHS_B(X) X(240, 16, 15) X(64, 8, 8) X(180, 15, 12) X(72, 9, 8) X(130, 13, 10) X(288, 18, 16)
#define T2SH_IL_LENGTHS_C(X) X(192, 16, 12) X(96, 12, 8) X(200, 20, 10) X(80, 10, 8) X(156, 13, 12) X(50, 10, 5)
#define T2SH_IL_LENGTHS_D(X) X(160, 16, 10) X(128, 16, 8) X(216, 18, 12) X(90, 10, 9) X(150, 15, 10) X(52, 13, 4)
#define T2SH_IL_LENGTHS_E(X) X(260, 20, 13) X(108, 12, 9) X(60, 10, 6) X(208, 16, 13) X(320, 20, 16) X(162, 18, 9)
#define T2SH_IL_LENGTHS_F(X) X(300, 20, 15) X(120, 12, 10) X(78, 13, 6) X(104, 13, 8) X(270, 18, 15)
#define T2SH_IL_LENGTHS(X) \
  T2SH_IL_LENGTHS_A(X) T2SH_IL_LENGTHS_B(X) T2SH_IL_LENGTHS_C(X) T2SH_IL_LENGTHS_D(X) T2SH_IL_LENGTHS_E(X) \
  T2SH_IL_LENGTHS_F(X)

namespace t2sh {

namespace {

// The two radices of a column length, the larger one first (stage B keeps RA items busy).
template <int N> struct IlRadix;
#define T2SH_IL_LENGTH(n, ra, rb) \
  template <> struct IlRadix<n> { static constexpr int RA = ra, RB = rb; };
T2SH_IL_LENGTHS(T2SH_IL_LENGTH)
#undef T2SH_IL_LENGTH

template <int N>
struct Il : IlRadix<N> {
  static constexpr int RA = IlRadix<N>::RA, RB = IlRadix<N>::RB;
  static_assert(RA * RB == N && RA >= RB, "N = RA RB");
  static constexpr int GT = (8 * RA + 31) / 32 * 32;  // threads of a group
  static constexpr int TILE = N * 128;                // bytes
  static constexpr int BOX = N <= 256 ? N : N / 2;    // rows of one tensor-map box
  static_assert(N % BOX == 0 && BOX <= 256, "whole boxes");
  // an even RB: the two lanes of a point take half of the frequencies each in Psi (ten floats a point)
  static constexpr bool HALF = RB % 2 == 0;
  static constexpr size_t psi_bytes = (size_t)N * 4 * (HALF ? 40 : 64);
  static constexpr int TWS = (N + 15) / 16 * 16 + 8;  // between the lanes' tables, half the banks apart
  static constexpr int TW = HALF ? TWS + N : N;        // roots of unity
  // `bufs` tile buffers, Psi of a tile's columns, roots of unity, a barrier and a tile number per buffer
  static constexpr size_t smem(int bufs) { return (size_t)bufs * TILE + psi_bytes + TW * 8 + 16 * 12; }
  static constexpr size_t smem_adj(int groups) { return (size_t)groups * TILE + N * 8; }
  // groups of a CTA, which share the Psi block of their columns: 512 threads at 128 registers,
  // or what fits in shared memory
  static constexpr int GS = (int)((232448 - psi_bytes - TW * 8 - 192) / TILE);
  static constexpr int G = 512 / GT < GS ? 512 / GT : GS;
  // Tile buffers: one per group, and up to as many spare ones where a CTA has fewer than four groups
  // to hide a tile's way from memory.  260 points (three groups, one spare buffer; 288 slices of
  // 260x240) 1.85 -> 1.72 ms; with four groups spare buffers gave nothing (192 points 0.232 and
  // 0.237 ms, 256 points 1.71 and 1.73 ms).
  static constexpr int NB = G >= 4 || GS <= G ? G : 2 * G < GS ? 2 * G : GS;
  static constexpr int THREADS = G * GT;
  static_assert(G >= 1 && NB >= G && NB <= 16 && smem(NB) <= 232448, "shared memory");
  static constexpr int E = RA <= 16 ? 2 : 1;  // basis images held in registers while the next tile is requested
  static constexpr bool FULL = 8 * RA == GT;  // every thread has an item in stage B
};

__device__ __forceinline__ void tma_load_2d(void* dst, const void* tmap, unsigned long long* bar, int x, int y) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];" ::
          "r"(smem_u32(dst)),
      "l"(tmap), "r"(smem_u32(bar)), "r"(x), "r"(y)
      : "memory");
}

// wait until *seq has reached `tile`; false if it has not within the bounded wait
__device__ __forceinline__ bool seq_wait_bounded(const volatile int* seq, int tile) {
  if (*seq >= tile) return true;
  const unsigned long long t0 = global_ns();
  while (*seq < tile)
    if (global_ns() - t0 > kWaitNs) return false;
  return true;
}

// barrier among the GT threads of group `grp`
template <int GT>
__device__ __forceinline__ void group_sync(int grp) {
  if constexpr (GT == 32) __syncwarp();
  else asm volatile("bar.sync %0, %1;" ::"r"(grp + 1), "n"(GT) : "memory");
}

__device__ __forceinline__ float2 lds2(const unsigned char* p, int off) { return *reinterpret_cast<const float2*>(p + off); }
__device__ __forceinline__ void sts2(unsigned char* p, int off, float2 v) { *reinterpret_cast<float2*>(p + off) = v; }

// the value in the neighbouring lane, which holds the other two basis images of the point
__device__ __forceinline__ float2 shfl_xor2(float2 v) {
  return make_float2(__shfl_xor_sync(0xffffffffu, v.x, 4), __shfl_xor_sync(0xffffffffu, v.y, 4));
}

// A thread's place in its group: column w, basis pair kp, item j
struct IlItem {
  int w, kp, j;
  bool onb;  // has an item in stage B (the others shadow item 0 and write nothing)
};
template <int N>
__device__ __forceinline__ IlItem il_item(int gt) {
  const int j = gt >> 3;
  const bool onb = Il<N>::FULL || j < Il<N>::RA;
  return {gt & 3, (gt >> 2) & 1, onb ? j : 0, onb};
}

// IDFT_RA of the NK basis images in c (the thread's images i0 ..), to rows j + RB q of t
template <int RA, int RB, int NK>
__device__ __forceinline__ void il_store(float2 (&c)[NK][RA], int i0, float2* gp, const int (&gs)[4], int rowlen,
                                         bool on) {
#pragma unroll
  for (int i = 0; i < NK; ++i) dft_r<RA, true>(c[i]);
  if (!on) return;
#pragma unroll
  for (int q = 0; q < RA; ++q) {
    float2* row = gp + q * RB * rowlen;
#pragma unroll
    for (int i = 0; i < NK; ++i) row[gs[(i0 + i + q) & 3]] = c[i][q];
  }
}

// Normal-operator column pass, in place on t.  CTAs walk contiguous runs of the (column tile,
// slice x coil) list in column-tile-major order: Psi of four columns stays in shared memory for
// all slices and coils of the run.  Tile p of a run belongs to group p mod ngroups and lands in
// buffer p mod nbuf; the group that has read tile p requests tile p + nbuf into its buffer.  So with
// spare buffers a tile is on its way while the group that will take it still works on its last one.
// seq[b] is the tile last requested into buffer b: a group looks there before it waits for the
// buffer's barrier, whose phase alone would not tell this tile from the one two visits earlier.
template <int N>
__global__ void __launch_bounds__(Il<N>::THREADS, 1)
    k_col_il(Geom g, const __grid_constant__ CUtensorMap tm, const float2* __restrict__ tw_g,
             const float* __restrict__ psi, float2* t, int nsc, int ntiles, int ngroups, int nbuf) {
  using L = Il<N>;
  constexpr int RA = L::RA, RB = L::RB, GT = L::GT, E = L::E;
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  const int grp = threadIdx.x / GT, gt = threadIdx.x - grp * GT;
  unsigned char* buf = smem_raw + (size_t)grp * L::TILE;
  // Psi by point.  HALF: [k2 mod RB / 2][k1][k2 div RB / 2][w], images a, b of the lane that takes the
  // frequency and c, d of the other: (aa, ab, bb, ac), (ad, bc, bd, cc), (cd, dd).  Otherwise
  // [k2][k1][kp][w]: the pair's own block (aa, ab, bb, -), and its block with the other pair (ac, ad, bc, bd)
  constexpr int NP = L::HALF ? N * 4 : N * 8;
  float4* pso = reinterpret_cast<float4*>(smem_raw + (size_t)nbuf * L::TILE);
  float4* psx = pso + NP;
  float2* psz = reinterpret_cast<float2*>(psx + NP);  // HALF only
  // [j][k1]: w_N^(j k1); HALF: [kp][j][k1], for kp = 1 times (-1)^j, which turns the frequencies by RB / 2
  float2* tws = reinterpret_cast<float2*>(smem_raw + (size_t)nbuf * L::TILE + L::psi_bytes);
  unsigned long long* bar = reinterpret_cast<unsigned long long*>(tws + L::TW);
  volatile int* seq = reinterpret_cast<volatile int*>(bar + 16);
  for (int i = threadIdx.x; i < N; i += blockDim.x) {
    const float2 v = tw_g[(i / RA) * (i % RA)];
    tws[i] = v;
    if (L::HALF) tws[L::TWS + i] = (i / RA) % 2 ? make_float2(-v.x, -v.y) : v;
  }
  const int nz = g.nz;
  const int rowlen = 4 * nz;
  if (threadIdx.x < nbuf) {
    mbar_init(bar + threadIdx.x, 1);
    seq[threadIdx.x] = -1;
    fence_mbar_init();
  }
  const IlItem it = il_item<N>(gt);
  const bool wa = (gt & ~31) / 8 < RB;  // some thread of the warp has an item in stages A and A'
  const bool on = it.onb && it.j < RB;            // this thread has an item in stages A and A'
  const int ja = RA == RB || on ? it.j : 0;  // idle threads read item 0 there and write nothing
  // address bases by slot: image 2 kp + i of row j + RB q is at pa[(i + q) & 3] + q RB rows, of row
  // j + RB k1 at pb[(i + j) & 3] + j rows
  unsigned char* pa[4];
  unsigned char* pb[4];
  int gs[4];
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    pa[m] = buf + ja * 128 + ((m + 2 * it.kp + ja) & 3) * 32 + it.w * 8;
    pb[m] = buf + it.j * RB * 128 + ((m + 2 * it.kp + it.j) & 3) * 32 + it.w * 8;
    gs[m] = ((m + 2 * it.kp + ja) & 3) * 4;
  }
  const float2* tw = tws + (L::HALF ? it.kp * L::TWS : 0) + it.j;
  const int lo = (int)((long long)ntiles * blockIdx.x / gridDim.x),
            hi = (int)((long long)ntiles * (blockIdx.x + 1) / gridDim.x);
  int b = grp;  // the group's next buffer
  unsigned phase = 0;
  bool dead = false;  // a bounded wait ran out: nothing is requested or waited for any more

  auto request = [&](int tile, int buffer) {  // one thread
    const int zt = tile / nsc, sc = tile - zt * nsc;
    mbar_expect_tx(bar + buffer, L::TILE);
#pragma unroll
    for (int h = 0; h < N / L::BOX; ++h)
      tma_load_2d(smem_raw + (size_t)buffer * L::TILE + h * L::BOX * 128, &tm, bar + buffer, zt * 16, sc * N + h * L::BOX);
    __threadfence_block();
    seq[buffer] = tile;
  };

  int tile = lo + grp;
  for (int seg = lo; seg < hi;) {
    const int zt = seg / nsc;
    const int end = min(hi, (zt + 1) * nsc);
    __syncthreads();  // the barriers are set up, and nobody reads the previous columns' Psi any more
    for (int e = threadIdx.x; e < N * 4; e += blockDim.x) {
      const int w = e & 3, pos = e >> 2, k2 = pos / RA, k1 = pos - k2 * RA;
      const float* pp = psi + (long long)(k1 + RA * k2) * nz + zt * 4 + w;
      const long long NN = (long long)N * nz;
      // upper triangle, row by row: 00 01 02 03 11 12 13 22 23 33
      const float p02 = pp[2 * NN], p03 = pp[3 * NN], p12 = pp[5 * NN], p13 = pp[6 * NN];
      if constexpr (L::HALF) {
        const bool up = k2 >= RB / 2;  // the lane of images 2 and 3 takes it
        const int e1 = ((k2 - (up ? RB / 2 : 0)) * RA + k1) * 8 + (up ? 4 : 0) + w;
        const float p00 = pp[0], p01 = pp[NN], p11 = pp[4 * NN], p22 = pp[7 * NN], p23 = pp[8 * NN], p33 = pp[9 * NN];
        pso[e1] = up ? make_float4(p22, p23, p33, p02) : make_float4(p00, p01, p11, p02);
        psx[e1] = up ? make_float4(p12, p03, p13, p00) : make_float4(p03, p12, p13, p22);
        psz[e1] = up ? make_float2(p01, p11) : make_float2(p23, p33);
      } else {
        pso[pos * 8 + w] = make_float4(pp[0], pp[NN], pp[4 * NN], 0.f);
        pso[pos * 8 + 4 + w] = make_float4(pp[7 * NN], pp[8 * NN], pp[9 * NN], 0.f);
        psx[pos * 8 + w] = make_float4(p02, p03, p12, p13);
        psx[pos * 8 + 4 + w] = make_float4(p02, p12, p03, p13);
      }
    }
    if (seg == lo) {  // the first columns' Psi (the plan's) is copied before t is touched
      pdl_wait();
      pdl_trigger();
      if (threadIdx.x == 0)
        for (int i = 0; i < nbuf && lo + i < hi; ++i) request(lo + i, i);
    }
    __syncthreads();
    for (; tile < end; tile += ngroups) {
      if (!dead && !(seq_wait_bounded(seq + b, tile) && mbar_wait_bounded(bar + b, phase))) {
        dead = true;
        if (g.err) atomicExch(g.err, 1);
      }
      if (wa) {
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          float2 a[RA];
#pragma unroll
          for (int q = 0; q < RA; ++q) a[q] = lds2(pa[(k + q) & 3], q * RB * 128);
          dft_r<RA, false>(a);
          if (on) {
#pragma unroll
            for (int q = 0; q < RA; ++q) sts2(pa[(k + q) & 3], q * RB * 128, a[q]);
          }
        }
      }
      group_sync<GT>(grp);
      {
        float2 b[2][RB];
#pragma unroll
        for (int k = 0; k < 2; ++k) {
#pragma unroll
          for (int j = 0; j < RB; ++j) b[k][j] = lds2(pb[(k + j) & 3], j * 128);
#pragma unroll
          for (int j = 1; j < RB; ++j) b[k][j] = twiddle_mul<false>(b[k][j], tw[j * RA]);
          dft_r<RB, false>(b[k]);
        }
        if constexpr (L::HALF) {
          // register r holds frequency k2 = r in the lane of images 0 and 1 and r + RB / 2 (mod RB) in that of
          // 2 and 3, so each lane takes the frequencies of its lower registers, with the other lane's upper ones
          constexpr int H = RB / 2;
#pragma unroll
          for (int r = 0; r < H; ++r) {
            const int e = (r * RA + it.j) * 8 + it.kp * 4 + it.w;
            const float4 po = pso[e], px = psx[e];
            const float2 pz = psz[e];
            const float2 va = b[0][r], vb = b[1][r], vc = shfl_xor2(b[0][r + H]), vd = shfl_xor2(b[1][r + H]);
            b[0][r].x = fmaf(px.x, vd.x, fmaf(po.w, vc.x, fmaf(po.y, vb.x, po.x * va.x)));
            b[0][r].y = fmaf(px.x, vd.y, fmaf(po.w, vc.y, fmaf(po.y, vb.y, po.x * va.y)));
            b[1][r].x = fmaf(px.z, vd.x, fmaf(px.y, vc.x, fmaf(po.z, vb.x, po.y * va.x)));
            b[1][r].y = fmaf(px.z, vd.y, fmaf(px.y, vc.y, fmaf(po.z, vb.y, po.y * va.y)));
            float2 yc, yd;
            yc.x = fmaf(pz.x, vd.x, fmaf(px.w, vc.x, fmaf(px.y, vb.x, po.w * va.x)));
            yc.y = fmaf(pz.x, vd.y, fmaf(px.w, vc.y, fmaf(px.y, vb.y, po.w * va.y)));
            yd.x = fmaf(pz.y, vd.x, fmaf(pz.x, vc.x, fmaf(px.z, vb.x, px.x * va.x)));
            yd.y = fmaf(pz.y, vd.y, fmaf(pz.x, vc.y, fmaf(px.z, vb.y, px.x * va.y)));
            b[0][r + H] = shfl_xor2(yc);
            b[1][r + H] = shfl_xor2(yd);
          }
        } else {
#pragma unroll
          for (int k2 = 0; k2 < RB; ++k2) {
            const int e = (k2 * RA + it.j) * 8 + it.kp * 4 + it.w;
            const float4 po = pso[e], px = psx[e];
            const float2 va = b[0][k2], vb = b[1][k2];
            float2 vc, vd;  // the other pair, from the lane that holds it
            vc.x = __shfl_xor_sync(0xffffffffu, va.x, 4);
            vc.y = __shfl_xor_sync(0xffffffffu, va.y, 4);
            vd.x = __shfl_xor_sync(0xffffffffu, vb.x, 4);
            vd.y = __shfl_xor_sync(0xffffffffu, vb.y, 4);
            b[0][k2].x = fmaf(px.y, vd.x, fmaf(px.x, vc.x, fmaf(po.y, vb.x, po.x * va.x)));
            b[0][k2].y = fmaf(px.y, vd.y, fmaf(px.x, vc.y, fmaf(po.y, vb.y, po.x * va.y)));
            b[1][k2].x = fmaf(px.w, vd.x, fmaf(px.z, vc.x, fmaf(po.z, vb.x, po.y * va.x)));
            b[1][k2].y = fmaf(px.w, vd.y, fmaf(px.z, vc.y, fmaf(po.z, vb.y, po.y * va.y)));
          }
        }
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          dft_r<RB, true>(b[k]);
#pragma unroll
          for (int j = 1; j < RB; ++j) b[k][j] = twiddle_mul<true>(b[k][j], tw[j * RA]);
#pragma unroll
          for (int j = 0; j < RB; ++j)
            if (L::FULL || it.onb) sts2(pb[(k + j) & 3], j * 128, b[k][j]);
        }
      }
      group_sync<GT>(grp);
      const int sc = tile - zt * nsc;
      float2* gp = t + ((long long)sc * N + ja) * rowlen + zt * 16 + it.w;
#pragma unroll
      for (int k = 0; k < 2 - E; ++k) {
        float2 c[1][RA];
#pragma unroll
        for (int q = 0; q < RA; ++q) c[0][q] = lds2(pa[(k + q) & 3], q * RB * 128);
        if (wa) il_store<RA, RB, 1>(c, k, gp, gs, rowlen, on);
      }
      float2 c[E][RA];
#pragma unroll
      for (int k = 0; k < E; ++k)
#pragma unroll
        for (int q = 0; q < RA; ++q) c[k][q] = lds2(pa[(2 - E + k + q) & 3], q * RB * 128);
      fence_proxy_async_smem();
      group_sync<GT>(grp);  // the buffer is read: the next tile lands while this one is finished
      if (gt == 0 && tile + nbuf < hi && !dead) request(tile + nbuf, b);
      int step = ngroups;
      b += ngroups;
      if (b >= nbuf) {
        b -= nbuf;
        step -= nbuf;
        phase ^= 1;
      }
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        pa[m] += step * L::TILE;
        pb[m] += step * L::TILE;
      }
      if (wa) il_store<RA, RB, E>(c, 2 - E, gp, gs, rowlen, on);
    }
    seg = end;
  }
  // copies in flight are given one more bounded wait before the CTA leaves
  if (__syncthreads_or(dead) && threadIdx.x < nbuf && seq[threadIdx.x] >= 0)
    mbar_wait_bounded(bar + threadIdx.x, ((seq[threadIdx.x] - lo) / nbuf) & 1);
}

// A^H y column pass: IDFT_y of the projected k-space column scaled by gsign (-1)^(ky + kz) /
// sqrt(ny nz), to the interleaved t.  The values go straight from global memory to registers
// (64 loads in flight per thread), then stages B' and A' as above.  IN_IL: the k-space itself has
// t's layout and may be t (a tile is read whole before it is written).
template <int N, bool IN_IL>
__global__ void __launch_bounds__(Il<N>::THREADS, 1)
    k_col_il_adj(Geom g, const float2* __restrict__ tw_g, const float2* in, float2* t, long long ntiles, int ngroups) {
  using L = Il<N>;
  constexpr int RA = L::RA, RB = L::RB, GT = L::GT;
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  const int grp = threadIdx.x / GT, gt = threadIdx.x - grp * GT;
  unsigned char* buf = smem_raw + (size_t)grp * L::TILE;
  const int nz = g.nz;
  const int rowlen = 4 * nz;
  const IlItem it = il_item<N>(gt);
  const bool wa = (gt & ~31) / 8 < RB;  // some thread of the warp has an item in stages A and A'
  const bool on = it.onb && it.j < RB;            // this thread has an item in stages A and A'
  const int ja = RA == RB || on ? it.j : 0;  // idle threads read item 0 there and write nothing
  unsigned char* pa[4];
  unsigned char* pb[4];
  int gs[4];
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    pa[m] = buf + ja * 128 + ((m + 2 * it.kp + ja) & 3) * 32 + it.w * 8;
    pb[m] = buf + it.j * RB * 128 + ((m + 2 * it.kp + it.j) & 3) * 32 + it.w * 8;
    gs[m] = ((m + 2 * it.kp + ja) & 3) * 4;
  }
  float2* tws = reinterpret_cast<float2*>(smem_raw + (size_t)ngroups * L::TILE);
  for (int i = threadIdx.x; i < N; i += blockDim.x) tws[i] = tw_g[(i / RA) * (i % RA)];
  const float2* tw = tws + it.j;
  __syncthreads();
  pdl_wait();
  pdl_trigger();
  // tiles in slice-and-coil-major order: neighbouring groups read neighbouring columns
  const int ntz = nz / 4;
  const long long step = (long long)gridDim.x * ngroups;
  for (long long tile = (long long)blockIdx.x * ngroups + grp; tile < ntiles; tile += step) {
    const long long sc = tile / ntz;
    const int zt = (int)(tile - sc * ntz);
    {
      const float scale = g.gsign * g.inv_sqrt_n * parity_sign(it.j + it.w);  // of frequency k1; 4 zt is even
      float2 b[2][RB];
#pragma unroll
      for (int k2 = 0; k2 < RB; ++k2) {
        const int f = it.j + RA * k2;
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          const int kk = 2 * it.kp + k;
          if (IN_IL)
            b[k][k2] = in[(sc * N + f) * rowlen + zt * 16 + ((kk + f % RB + f / RB) & 3) * 4 + it.w];
          else
            b[k][k2] = in[((sc * 4 + kk) * N + f) * nz + zt * 4 + it.w];
          if (RA % 2 && k2 % 2) b[k][k2] = make_float2(-b[k][k2].x, -b[k][k2].y);
        }
      }
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        dft_r<RB, true>(b[k]);
#pragma unroll
        for (int j = 1; j < RB; ++j) b[k][j] = twiddle_mul<true>(b[k][j], tw[j * RA]);
#pragma unroll
        for (int j = 0; j < RB; ++j)
          if (L::FULL || it.onb) sts2(pb[(k + j) & 3], j * 128, cscale(b[k][j], scale));
      }
    }
    group_sync<GT>(grp);
    if (wa) {
      float2* gp = t + (sc * N + ja) * rowlen + zt * 16 + it.w;
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        float2 c[1][RA];
#pragma unroll
        for (int q = 0; q < RA; ++q) c[0][q] = lds2(pa[(k + q) & 3], q * RB * 128);
        il_store<RA, RB, 1>(c, k, gp, gs, rowlen, on);
      }
    }
    group_sync<GT>(grp);
  }
}

// Forward column pass of A: DFT_y of t, centring signs and scale.  PROJ: then Psi N, to planar
// k-space `out` [S][C][K][ny][nz]; otherwise in place, row f of t holding frequency f (a tile is
// read whole before it is written).
template <int N, bool PROJ>
__global__ void __launch_bounds__(Il<N>::THREADS, 1)
    k_col_il_fwd(Geom g, const float2* __restrict__ tw_g, const float* __restrict__ psi, const float2* t, float2* out,
                 long long ntiles, int ngroups) {
  using L = Il<N>;
  constexpr int RA = L::RA, RB = L::RB, GT = L::GT;
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  const int grp = threadIdx.x / GT, gt = threadIdx.x - grp * GT;
  unsigned char* buf = smem_raw + (size_t)grp * L::TILE;
  const int nz = g.nz;
  const int rowlen = 4 * nz;
  const IlItem it = il_item<N>(gt);
  const bool wa = (gt & ~31) / 8 < RB;
  const bool on = it.j < RB;
  const int ja = RA == RB || on ? it.j : 0;
  unsigned char* pa[4];
  unsigned char* pb[4];
  int gs[4];
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    pa[m] = buf + ja * 128 + ((m + 2 * it.kp + ja) & 3) * 32 + it.w * 8;
    pb[m] = buf + it.j * RB * 128 + ((m + 2 * it.kp + it.j) & 3) * 32 + it.w * 8;
    gs[m] = ((m + 2 * it.kp + ja) & 3) * 4;
  }
  float2* tws = reinterpret_cast<float2*>(smem_raw + (size_t)ngroups * L::TILE);
  for (int i = threadIdx.x; i < N; i += blockDim.x) tws[i] = tw_g[(i / RA) * (i % RA)];
  const float2* tw = tws + it.j;
  __syncthreads();
  pdl_wait();
  pdl_trigger();
  const int ntz = nz / 4;
  const float scale0 = g.gsign * g.inv_sqrt_n * parity_sign(it.j + it.w);  // of frequency k1; 4 zt is even
  const long long step = (long long)gridDim.x * ngroups;
  for (long long tile = (long long)blockIdx.x * ngroups + grp; tile < ntiles; tile += step) {
    const long long sc = tile / ntz;
    const int zt = (int)(tile - sc * ntz);
    if (wa) {
      const float2* gp = t + (sc * N + ja) * rowlen + zt * 16 + it.w;
      float2 a[2][RA];
#pragma unroll
      for (int k = 0; k < 2; ++k)
#pragma unroll
        for (int q = 0; q < RA; ++q) a[k][q] = gp[(long long)(q * RB) * rowlen + gs[(k + q) & 3]];
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        dft_r<RA, false>(a[k]);
        if (on) {
#pragma unroll
          for (int q = 0; q < RA; ++q) sts2(pa[(k + q) & 3], q * RB * 128, a[k][q]);
        }
      }
    }
    group_sync<GT>(grp);
    float2 b[2][RB];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
#pragma unroll
      for (int j = 0; j < RB; ++j) b[k][j] = lds2(pb[(k + j) & 3], j * 128);
#pragma unroll
      for (int j = 1; j < RB; ++j) b[k][j] = twiddle_mul<false>(b[k][j], tw[j * RA]);
      dft_r<RB, false>(b[k]);
    }
    group_sync<GT>(grp);  // the buffer is read: the next tile may be written
#pragma unroll
    for (int k2 = 0; k2 < RB; ++k2) {
      const int f = it.j + RA * k2;
      const float scale = RA % 2 && k2 % 2 ? -scale0 : scale0;
      const float2 va = cscale(b[0][k2], scale), vb = cscale(b[1][k2], scale);
      if constexpr (PROJ) {
        float2 vc, vd;  // the other pair, from the lane that holds it
        vc.x = __shfl_xor_sync(0xffffffffu, va.x, 4);
        vc.y = __shfl_xor_sync(0xffffffffu, va.y, 4);
        vd.x = __shfl_xor_sync(0xffffffffu, vb.x, 4);
        vd.y = __shfl_xor_sync(0xffffffffu, vb.y, 4);
        const float2 v[4] = {it.kp ? vc : va, it.kp ? vd : vb, it.kp ? va : vc, it.kp ? vb : vd};
        const float* pp = psi + (long long)f * nz + zt * 4 + it.w;
        const long long NN = (long long)N * nz;
        // rows 2 kp and 2 kp + 1 of the upper triangle 00 01 02 03 11 12 13 22 23 33
        const float n = (float)(N * nz);
        const float p02 = pp[2 * NN] * n, p03 = pp[3 * NN] * n, p12 = pp[5 * NN] * n, p13 = pp[6 * NN] * n;
        const float d0 = pp[(it.kp ? 7 : 0) * NN] * n, d1 = pp[(it.kp ? 8 : 1) * NN] * n,
                    d2 = pp[(it.kp ? 9 : 4) * NN] * n;
        const float r0[4] = {it.kp ? p02 : d0, it.kp ? p12 : d1, it.kp ? d0 : p02, it.kp ? d1 : p03};
        const float r1[4] = {it.kp ? p03 : d1, it.kp ? p13 : d2, it.kp ? d1 : p12, it.kp ? d2 : p13};
        float2 u0 = cscale(v[0], r0[0]), u1 = cscale(v[0], r1[0]);
#pragma unroll
        for (int l = 1; l < 4; ++l) {
          u0 = make_float2(fmaf(r0[l], v[l].x, u0.x), fmaf(r0[l], v[l].y, u0.y));
          u1 = make_float2(fmaf(r1[l], v[l].x, u1.x), fmaf(r1[l], v[l].y, u1.y));
        }
        float2* o = out + ((sc * 4 + 2 * it.kp) * N + f) * nz + zt * 4 + it.w;
        if (L::FULL || it.onb) {
          o[0] = u0;
          o[NN] = u1;
        }
      } else {
        float2* o = out + (sc * N + f) * rowlen + zt * 16 + it.w;
        const int rot = 2 * it.kp + f % RB + f / RB;
        if (L::FULL || it.onb) {
          o[(rot & 3) * 4] = va;
          o[((rot + 1) & 3) * 4] = vb;
        }
      }
    }
  }
}

// groups per CTA: all of them once the tiles fill the chip, fewer while SMs would stay idle
template <int N>
int il_groups(long long ntiles, int nsm) {
  const long long per = (ntiles + nsm - 1) / nsm;
  return (int)std::max<long long>(1, std::min<long long>(Il<N>::G, per));
}

template <int N>
cudaError_t il_normal(const Geom& g, const float2* tw, const float* psi, float2* t, cudaStream_t st) {
  using L = Il<N>;
  TmaEncodeFn enc = tma_encode_fn();
  if (!enc) return cudaErrorNotSupported;
  const long long nsc = (long long)g.S * g.C, ntiles = nsc * (g.nz / 4);
  if (nsc * N > 0x7fffffffLL || ntiles + nsc > 0x7fffffffLL) return cudaErrorNotSupported;
  CUtensorMap tm;
  const cuuint64_t d[2] = {(cuuint64_t)(4 * g.nz), (cuuint64_t)(nsc * N)};
  const cuuint64_t s[1] = {(cuuint64_t)g.nz * 32};
  const cuuint32_t b[2] = {16, (cuuint32_t)L::BOX}, es[2] = {1, 1};
  if (enc(&tm, CU_TENSOR_MAP_DATA_TYPE_INT64, 2, t, d, s, b, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
          CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
          CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
    return cudaErrorNotSupported;
  int nsm = 0;
  cudaError_t e = smem_optin((const void*)k_col_il<N>, (int)L::smem(L::NB));
  if (e == cudaSuccess) e = sm_count(&nsm);
  if (e != cudaSuccess) return e;
  const int ng = il_groups<N>(ntiles, nsm);
  const int grid = (int)std::min<long long>(nsm, (ntiles + ng - 1) / ng);
  const int nbuf = (int)std::max<long long>(ng, std::min<long long>(L::NB, (ntiles + grid - 1) / grid));
  return launch_pdl(k_col_il<N>, dim3(grid), ng * L::GT, L::smem(nbuf), st, g, tm, tw, psi, t, (int)nsc, (int)ntiles, ng,
                    nbuf);
}

template <int N, bool IN_IL>
cudaError_t il_adj(const Geom& g, const float2* tw, const float2* in, float2* t, cudaStream_t st) {
  using L = Il<N>;
  const long long nsc = (long long)g.S * g.C, ntiles = nsc * (g.nz / 4);
  int nsm = 0;
  cudaError_t e = smem_optin((const void*)k_col_il_adj<N, IN_IL>, (int)L::smem_adj(L::G));
  if (e == cudaSuccess) e = sm_count(&nsm);
  if (e != cudaSuccess) return e;
  const int ng = il_groups<N>(ntiles, nsm);
  const int grid = (int)std::min<long long>(nsm, (ntiles + ng - 1) / ng);
  return launch_pdl(k_col_il_adj<N, IN_IL>, dim3(grid), ng * L::GT, L::smem_adj(ng), st, g, tw, in, t, ntiles, ng);
}

template <int N, bool PROJ>
cudaError_t il_fwd(const Geom& g, const float2* tw, const float* psi, const float2* t, float2* out, cudaStream_t st) {
  using L = Il<N>;
  const long long nsc = (long long)g.S * g.C, ntiles = nsc * (g.nz / 4);
  int nsm = 0;
  cudaError_t e = smem_optin((const void*)k_col_il_fwd<N, PROJ>, (int)L::smem_adj(L::G));
  if (e == cudaSuccess) e = sm_count(&nsm);
  if (e != cudaSuccess) return e;
  const int ng = il_groups<N>(ntiles, nsm);
  const int grid = (int)std::min<long long>(nsm, (ntiles + ng - 1) / ng);
  return launch_pdl(k_col_il_fwd<N, PROJ>, dim3(grid), ng * L::GT, L::smem_adj(ng), st, g, tw, psi, t, out, ntiles, ng);
}

template <int N>
cudaError_t il_go(const Geom& g, IlPass pass, const float2* tw, const float* psi, const float2* in, float2* t,
                  cudaStream_t st) {
  switch (pass) {
    case IL_NORMAL: return il_normal<N>(g, tw, psi, t, st);
    case IL_ADJ_PLANAR: return il_adj<N, false>(g, tw, in, t, st);
    case IL_ADJ: return il_adj<N, true>(g, tw, in, t, st);
    case IL_FWD_PROJ: return il_fwd<N, true>(g, tw, psi, in, t, st);
    case IL_FWD_RAW: return il_fwd<N, false>(g, tw, psi, in, t, st);
  }
  return cudaErrorInvalidValue;
}

}  // namespace

}  // namespace t2sh
