// Chebyshev transforms along z (Sec. 3.2.1) as float64-accurate matrix products on the tensor
// cores: tcgen05 MMAs with bf16 operands staged in shared memory and fp32 accumulators in tensor
// memory (the exact split of ch_tc.cuh).
//
// The transform of one line is a product with a fixed Nz x Nz matrix B (rows = outputs):
//   forward (samples at z_k = cos(pi k / N) -> coefficients)
//     a_n = sum_k W_nk f_k,  W_nk = e_k cos(pi n k / N) / (cbar_n N),
//     e_k = 1 at k = 0, N and 2 otherwise, cbar_n = 2 at n = 0, N and 1 otherwise;
//   backward (coefficients -> samples)  f_j = sum_n cos(pi n j / N) a_n.
// Real and imaginary parts are separate rows of the left operand.
//
// Folding.  cos(pi n (N-k) / N) = (-1)^n cos(pi n k / N) and e_k = e_{N-k}, so with H = N / 2
//   even outputs need only s_k = x_k + x_{N-k}, odd ones only d_k = x_k - x_{N-k}, k < H
// (both matrices are symmetric in this way), plus (-1)^m x_H for output n = 2m.  The sums and
// differences are exact in fixed point, the middle element is added to the recombined integer
// (it is the row's value times one weight), and the last output n = N, sum_k w_k (-1)^k x_k, is
// summed exactly by the producers; the MMAs then do two H x H products of K = H instead of one
// (N+1) x (N+1) product of K = N + 1.  All weights share one power-of-two scale 2^q.
//
// Tiles and data flow.  A tile is 128 rows (re and im of 64 lines of one field).  Its passes are
// (output slice of NT columns, parity, K group): the accumulators of a pass live in tensor memory.
// Persistent CTAs (one per SM) have four kinds of warps, so the scan, the conversion, the MMAs and
// the epilogue of different passes and tiles overlap:
//   scan (3 warps): the rows' scales of the next tile (the rows' first, cold read, after an L2
//     prefetch of the tile one further ahead) and the middle elements' terms;
//   producers (8 warps): per K stage of 16 (one MMA k-step) a thread converts four pairs
//     (x_k, x_{N-k}) of the real and imaginary rows of one line to fixed point, writes the eight
//     digit planes of the sums to the stage's shared buffer and keeps the differences (and, with
//     several slices, the sums) in a per-CTA buffer in global memory (L2), read back by the same
//     thread for the later passes; thread 0 also issues the bulk copy of the stage's matrix digits;
//   issuer (1 thread): the MMAs of each stage as it fills;
//   epilogue (8 warps): drains a pass's accumulators, recombines and stores.
// Twenty warps keep 96 registers each (seventeen would not allow more: five on one sub-partition).
#include <math.h>
#include <stdint.h>
#include <stdlib.h>
#include <string.h>

#include <algorithm>
#include <vector>

#include "ch_internal.h"
#include "ch_tc.cuh"

namespace chf {

namespace {

using namespace tc;

constexpr int kPW = 8, kEW = 8, kSW = 3;          // producer, epilogue and scan warps
constexpr int kThreads = 32 * (kPW + kEW + 1 + kSW);   // epilogue 0..7, producers, issuer, scan
constexpr int kStages = 4;                        // K stages in flight
constexpr int kRB = 3;                            // tiles whose row scales are held
constexpr int kStageBytes = kABytes + b_stage_bytes(kNTMax);
// per stage full, bfull, empty; accfull, accfree, rowfull[kRB], rowfree[kRB], fin
constexpr int kBars = 3 * kStages + 3 + 2 * kRB;
// stages, row scales and middle terms, barriers, the tensor-memory address
constexpr size_t kSmem = (size_t)kStages * kStageBytes +
                         kRB * kRows * (sizeof(long long) + sizeof(int)) + (size_t)(kBars + 1) * 8;
// one pass's stage block kept in global memory: four fixed-point values of two rows per thread
constexpr size_t kKeepStage = (size_t)kPW * 32 * 8 * sizeof(long long);

template <typename TO> __device__ __forceinline__ TO times(TO v, double f) { return v; }
template <> __device__ __forceinline__ double times<double>(double v, double f) { return v * f; }

// Row of a tile: lines in blocks of eight, the real parts of a block in rows 16 b .. + 7, the
// imaginary ones in 16 b + 8 .. + 15 (a producer half-warp, eight lines x two K groups of four,
// then stores 128 contiguous bytes).
__device__ __forceinline__ int tile_row(int l, int part) { return (l >> 3) * 16 + part * 8 + (l & 7); }

// the bit patterns of one complex element
template <typename T> struct CBits { typename FBits<T>::U re, im; };
__device__ __forceinline__ CBits<double> ld_cplx(const double* p) {
  const double2 v = *reinterpret_cast<const double2*>(p);
  return {FBits<double>::bits(v.x), FBits<double>::bits(v.y)};
}
__device__ __forceinline__ CBits<float> ld_cplx(const float* p) {
  const float2 v = *reinterpret_cast<const float2*>(p);
  return {FBits<float>::bits(v.x), FBits<float>::bits(v.y)};
}
__device__ __forceinline__ CBits<df> ld_cplx(const df* p) {
  const float4 v = *reinterpret_cast<const float4*>(p);
  return {FBits<df>::bits(df(v.x, v.y)), FBits<df>::bits(df(v.z, v.w))};
}

// One pass's outputs of one thread: columns m0 .. m0 + CW - 1 of its row, four at a time, from the
// eight accumulators at tensor-memory address tb; dst: output column m0 (columns 4 scalars apart).
// Arguments as in the kernel.
template <typename TO, int NMAG>
__device__ __forceinline__ void epilogue_pass(uint32_t tb, int NT, int CW, int m0, int H, int c,
                                              int kc, int par, bool rowok, bool nan, bool safe,
                                              int ex, long long mid, bool halve0, long long* part,
                                              TO* dst, uint32_t barAccFree, int lane) {
  for (int c0 = 0; c0 < CW; c0 += 4) {
    uint32_t v[kDiags][4];
    tmem_ldx4(tb + (uint32_t)c0, NT, v);
    if (c0 + 4 >= CW) {   // all read: the accumulators are free for the next pass
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncwarp();
      if (lane == 0)
        asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(barAccFree) : "memory");
    }
    long long T[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) T[e] = recombine<NMAG>(v, e);
    if (kc > 1) {
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        if (c > 0) T[e] += part[(c0 + e) * kEW * 32];
        if (c + 1 < kc) part[(c0 + e) * kEW * 32] = T[e];
      }
      if (c + 1 < kc) continue;
    }
    if (par == 0) {
      // (-1)^m x_H Y (m0 + c0 is a multiple of four); the forward weight of n = 0 is half
      const long long t0 = (halve0 && m0 + c0 == 0) ? mid / 2 : mid;
      T[0] += t0;
      T[1] -= mid;
      T[2] += mid;
      T[3] -= mid;
    }
    TO r[4];
    if (safe) {
#pragma unroll
      for (int e = 0; e < 4; ++e)
        r[e] = (e & 1) ? scaled_alu<TO>(T[e], ex) : scaled<TO>(T[e], ex);
    } else {
#pragma unroll
      for (int e = 0; e < 4; ++e) r[e] = nan ? qnan<TO>() : scaled_any<TO>(T[e], ex);
    }
#pragma unroll
    for (int e = 0; e < 4; ++e)
      if (rowok && m0 + c0 + e < H) dst[4 * (c0 + e)] = r[e];
  }
}

// in / out: nf fields of complex lines (re, im interleaved), field stride fsi / fso complex
// elements, line stride Nz = N + 1; dig: the matrix digits, stage blocks of 7 NT rows x 16 K in
// the order slice, parity, stage; keep: keep_bytes per CTA; nst stages per parity in kc groups of
// gst; nmag: accumulators known to stay within 2^22 (8, 3 or 0); q: log2 of the matrix scale;
// ymid: middle weight times 2^q; lastf: factor of output N (forward).  The 2 nsl passes of a tile are
// cut into items of np passes; several items a tile only where all items have a CTA each (launch_t).
template <typename TI, typename TO>
__global__ void __launch_bounds__(kThreads, 1)
    cheb_tc_kernel(const TI* __restrict__ in, long long fsi, TO* __restrict__ out, long long fso,
                   int nlines, int Nz, int tpf, int ntiles, int np, int NT, int nsl, int nst, int kc,
                   int gst, int nmag, const uint16_t* __restrict__ dig, char* __restrict__ keep,
                   long long keep_bytes, int fwd, int q, long long ymid, double lastf,
                   int* __restrict__ err) {
  typedef FBits<TI> F;
  extern __shared__ __align__(1024) unsigned char tsm[];
  unsigned char* stages = tsm;
  long long* sC = reinterpret_cast<long long*>(tsm + (size_t)kStages * kStageBytes);
  int* sE = reinterpret_cast<int*>(sC + kRB * kRows);
  unsigned long long* bars = reinterpret_cast<unsigned long long*>(sE + kRB * kRows);
  uint32_t* sT = reinterpret_cast<uint32_t*>(bars + kBars);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int N = Nz - 1, H = N / 2;
  const uint32_t barFull = su32(bars), barB = barFull + 8 * kStages;
  const uint32_t barEmpty = barFull + 16 * kStages, barAccFull = barFull + 24 * kStages;
  const uint32_t barAccFree = barAccFull + 8, barRow = barAccFull + 16;
  const uint32_t barRowFree = barRow + 8 * kRB, barFin = barRowFree + 8 * kRB;
  if (tid == 0) {
    for (int b = 0; b < kStages; ++b) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(barFull + 8 * b), "r"(kPW));
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(barB + 8 * b));
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(barEmpty + 8 * b));
    }
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(barAccFull));
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(barAccFree), "r"(kEW));
    for (int b = 0; b < kRB; ++b) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(barRow + 8 * b), "r"(kSW));
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(barRowFree + 8 * b),
                   "r"(kEW + kPW));
    }
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(barFin));
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  const bool issuer_warp = warp == kPW + kEW;
  if (issuer_warp) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     su32(sT)),
                 "r"(512));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  const int nparts = 2 * nsl / np, nitems = ntiles * nparts;
  // row scales and middle terms of lines l0 .. l0 + 3 of a tile, a warp's lanes along the lines
  auto scan4 = [&](int tile, int b, int l0) {
    const int fld = tile / tpf;
    const int line0 = (tile - fld * tpf) * (kRows / 2);
    const int nl = min(kRows / 2, nlines - line0);
    const TI* src = in + ((size_t)fld * fsi + (size_t)line0 * Nz) * 2;
    unsigned kr[4] = {0, 0, 0, 0}, ki[4] = {0, 0, 0, 0};
#pragma unroll 2
    for (int k = lane; k < Nz; k += 32) {
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (l0 + i < nl) {
          const CBits<TI> x = ld_cplx(src + ((size_t)(l0 + i) * Nz + k) * 2);
          kr[i] = max(kr[i], F::key(x.re));
          ki[i] = max(ki[i], F::key(x.im));
        }
    }
    unsigned mr = 0, mi = 0;   // lane i < 4: the keys of line l0 + i
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const unsigned a = __reduce_max_sync(0xffffffffu, kr[i]);
      const unsigned c = __reduce_max_sync(0xffffffffu, ki[i]);
      if (lane == i) {
        mr = a;
        mi = c;
      }
    }
    if (lane < 4 && l0 + lane < kRows / 2) {
      const int l = l0 + lane, er = row_scale<TI>(mr), ei = row_scale<TI>(mi);
      long long xr = 0, xi = 0;
      if (l < nl) {
        const CBits<TI> x = ld_cplx(src + ((size_t)l * Nz + H) * 2);
        xr = Fixed<TI, true>::of(x.re, er);
        xi = Fixed<TI, true>::of(x.im, ei);
      }
      const int ro = b * kRows + tile_row(l, 0);
      sE[ro] = er;
      sE[ro + 8] = ei;
      // X_H Y_H / 2^62 (|X_H| < 2^62, Y_H <= 2^54)
      sC[ro] = __mul64hi(xr, ymid * 4);
      sC[ro + 8] = __mul64hi(xi, ymid * 4);
    }
  };
  // the first tile by every warp (scanned by three, it kept the others waiting: a launch of one tile per
  // CTA 13 -> 10 us at N = 16, 19 -> 13 at N = 64)
  if (4 * warp < kRows / 2) scan4(blockIdx.x / nparts, 0, 4 * warp);
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();   // barriers and tensor-memory address visible to every warp
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *sT;
  const uint32_t sBase = su32(stages);
  const uint32_t bbytes = (uint32_t)b_stage_bytes(NT);
  char* kcta = keep + (long long)blockIdx.x * keep_bytes;
  Waiter W;

  if (issuer_warp) {
    if (lane == 0) {
      uint32_t slot = 0, use = 0;   // stage slot and how often it was used
      uint32_t pass = 0;
      bool any = false;
      for (int item = blockIdx.x; item < nitems; item += gridDim.x)
        for (int pp = 0; pp < np; ++pp)
          for (int c = 0; c < kc; ++c, ++pass) {
            if (pass > 0 && !W.wait(barAccFree, (pass - 1) & 1)) goto drain;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const int s0 = c * gst, s1 = min(nst, s0 + gst);
            for (int st = s0; st < s1; ++st) {
              if (!W.wait(barFull + 8 * slot, use & 1) || !W.wait(barB + 8 * slot, use & 1))
                goto drain;
              asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
              const uint32_t sA = sBase + slot * (uint32_t)kStageBytes;
              issue_stage(tmem, sA, sA + (uint32_t)kABytes, NT, st == s0);
              any = true;
              mma_commit(barEmpty + 8 * slot);
              if (++slot == kStages) {
                slot = 0;
                ++use;
              }
            }
            mma_commit(barAccFull);
          }
    drain:
      // however the loop ended, here or in another warp (an epilogue that gave up waits for no MMA):
      // the MMAs in flight finish (bounded) before the tensor memory is released
      if (any) {
        mma_commit(barFin);
        W.ok = mbar_wait(barFin, 0) && W.ok;
      }
    }
    __syncwarp();
  } else if (warp > kPW + kEW) {
    // ---- scan: four lines at a time
    const int sw = warp - (kPW + kEW + 1);
    int ti = 0;
    for (int item = blockIdx.x; item < nitems; item += gridDim.x, ++ti) {
      const int tile = item / nparts;
      if (sw == 0 && lane == 0 && item + (int)gridDim.x < nitems) {
        const int tn = (item + gridDim.x) / nparts, fn = tn / tpf, ln = (tn - fn * tpf) * (kRows / 2);
        const char* a = reinterpret_cast<const char*>(in + ((size_t)fn * fsi + (size_t)ln * Nz) * 2);
        const char* z = a + (size_t)min(kRows / 2, nlines - ln) * Nz * 2 * sizeof(TI);
        const uintptr_t a16 = ((uintptr_t)a + 15) & ~(uintptr_t)15;
        const uintptr_t z16 = (uintptr_t)z & ~(uintptr_t)15;
        if (z16 > a16)
          asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(a16),
                       "r"((uint32_t)(z16 - a16))
                       : "memory");
      }
      const int b = ti % kRB;
      if (ti >= kRB && !W.wait_warp(barRowFree + 8 * b, (ti / kRB - 1) & 1)) break;
      if (ti > 0)
        for (int l0 = 4 * sw; l0 < kRows / 2; l0 += 4 * kSW) scan4(tile, b, l0);
      __syncwarp();
      if (lane == 0)
        asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(barRow + 8 * b) : "memory");
    }
  } else if (warp >= kEW) {
    // ---- producers: thread = (line l of the tile, g): K positions 4 g .. 4 g + 3 of a stage,
    // position 4 g + e holding k = 16 st + g + 4 e
    const int p = tid - 32 * kEW, pw = warp - kEW;
    const int l = pw * 8 + ((lane >> 1) & 7), g = (lane >> 4) * 2 + (lane & 1);
    const int row = tile_row(l, 0);
    const uint32_t oa = (uint32_t)((g >> 1) * (int)kALbo + row * 16 + (g & 1) * 8);
    const uint64_t pol = policy_evict_last();
    longlong2* kp = reinterpret_cast<longlong2*>(kcta) + p;
    uint32_t slot = 0, use = 0;
    int ti = 0;
    // the stage's digit planes of v (biased; 0..3 the real row, 4..7 the imaginary one) and, by
    // one thread, the copy of its matrix digits; false after a wait ran out
    auto put = [&](const unsigned long long (&v)[8], const uint16_t* bsrc) {
      if (use > 0 && !W.wait_warp(barEmpty + 8 * slot, (use & 1) ^ 1)) return false;
      unsigned char* sA = stages + (size_t)slot * kStageBytes;
      if (p == 0) bulk_load(su32(sA) + (uint32_t)kABytes, bsrc, bbytes, barB + 8 * slot, pol);
#pragma unroll
      for (int i = 0; i < kAPlanes; ++i) {
        const int b = 7 - i, sh = b < 4 ? 0 : 32;
        uint32_t w[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) w[e] = (uint32_t)(v[e] >> sh);
        *reinterpret_cast<uint2*>(sA + i * kPlaneBytes + oa) =
            make_uint2(digit_pair(w[0], w[1], b & 3), digit_pair(w[2], w[3], b & 3));
        *reinterpret_cast<uint2*>(sA + i * kPlaneBytes + oa + 128) =
            make_uint2(digit_pair(w[4], w[5], b & 3), digit_pair(w[6], w[7], b & 3));
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncwarp();
      if (lane == 0)
        asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(barFull + 8 * slot)
                     : "memory");
      if (++slot == kStages) {
        slot = 0;
        ++use;
      }
      return true;
    };
    auto keep_at = [&](int par, int st) { return kp + (size_t)(par * nst + st) * (4 * kPW * 32); };
    auto store_keep = [&](longlong2* d, const unsigned long long (&v)[8]) {
#pragma unroll
      for (int i = 0; i < 4; ++i)
        __stcg(d + i * kPW * 32, make_longlong2((long long)v[2 * i], (long long)v[2 * i + 1]));
    };
    const size_t bstride = (size_t)bbytes / 2;   // elements of a stage block
    for (int item = blockIdx.x; item < nitems; item += gridDim.x, ++ti) {
      const int tile = item / nparts, pp0 = (item - tile * nparts) * np;
      const int fld = tile / tpf;
      const int line = (tile - fld * tpf) * (kRows / 2) + l;
      const bool rowok = line < nlines;
      const TI* src = in + ((size_t)fld * fsi + (size_t)(rowok ? line : 0) * Nz) * 2;
      const TI *lo = src + 2 * g, *hi = src + 2 * (N - g);
      CBits<TI> xa[4], xb[4];
      auto load = [&](int st) {
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const int k = 16 * st + 4 * e;
          xa[e] = {0, 0};
          xb[e] = {0, 0};
          if (rowok && k + g < H) {
            xa[e] = ld_cplx(lo + 2 * k);
            xb[e] = ld_cplx(hi - 2 * k);
          }
        }
      };
      load(0);
      const int rbuf = ti % kRB;
      if (!W.wait_warp(barRow + 8 * rbuf, (ti / kRB) & 1)) break;
      const int ere = sE[rbuf * kRows + row], eim = sE[rbuf * kRows + row + 8];
      __syncwarp();
      if (lane == 0)
        asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(barRowFree + 8 * rbuf)
                     : "memory");
      const bool tiny = __any_sync(0xffffffffu, min(ere, eim) < kTinyScale) != 0;
      // first pass: convert, fold, write the sums' (odd passes: the differences') planes, keep what the
      // item's other passes need (all biased)
      WordSums sumr, sumi;
      unsigned long long s0r = 0, s0i = 0;
      bool ok = true;
      for (int st = 0; st < nst && ok; ++st) {
        unsigned long long s[8], d[8];
        if (!tiny) {
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const long long x = Fixed<TI, false>::of(xa[e].re, ere), y = Fixed<TI, false>::of(xb[e].re, ere);
            const long long z = Fixed<TI, false>::of(xa[e].im, eim), w = Fixed<TI, false>::of(xb[e].im, eim);
            s[e] = x + y + kABias;
            d[e] = x - y + kABias;
            s[4 + e] = z + w + kABias;
            d[4 + e] = z - w + kABias;
          }
        } else {
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const long long x = Fixed<TI, true>::of(xa[e].re, ere), y = Fixed<TI, true>::of(xb[e].re, ere);
            const long long z = Fixed<TI, true>::of(xa[e].im, eim), w = Fixed<TI, true>::of(xb[e].im, eim);
            s[e] = x + y + kABias;
            d[e] = x - y + kABias;
            s[4 + e] = z + w + kABias;
            d[4 + e] = z - w + kABias;
          }
        }
        if (st + 1 < nst) load(st + 1);
        if (np > 1) store_keep(keep_at(1, st), d);   // for np = 2 pp0 is even
        if (np > 2) store_keep(keep_at(0, st), s);
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          sumr.add(s[e]);
          sumi.add(s[4 + e]);
        }
        if (st == 0) {
          s0r = s[0];
          s0i = s[4];
        }
        const uint16_t* bsrc = dig + ((size_t)pp0 * nst + st) * bstride;
        ok = pp0 & 1 ? put(d, bsrc) : put(s, bsrc);
      }
      if (!ok) break;
      // the last output n = N: sum_k w_k (-1)^k x_k, (-1)^k = (-1)^g for this thread's k; weights
      // e_k = 2 except k = 0, N (forward) or 1.  High and low words are added apart.
      if (pp0 == 0) {
        const int f2 = fwd ? 2 : 1, sf = g & 1 ? -f2 : f2;
        long long hr = sf * sumr.high(4 * nst), lr = sf * sumr.low(4 * nst);
        long long hm = sf * sumi.high(4 * nst), lm = sf * sumi.low(4 * nst);
        if (g == 0) {
          const int wm = (H & 1) ? -f2 : f2;
          long long xr = 0, xi = 0;
          if (rowok) {
            const CBits<TI> x = ld_cplx(src + 2 * H);
            xr = Fixed<TI, true>::of(x.re, ere);
            xi = Fixed<TI, true>::of(x.im, eim);
          }
          hr += wm * (xr >> 32);
          lr += wm * (long long)(unsigned)xr;
          hm += wm * (xi >> 32);
          lm += wm * (long long)(unsigned)xi;
          if (fwd) {   // s_0 was counted twice
            const long long a = (long long)(s0r - kABias), c = (long long)(s0i - kABias);
            hr -= a >> 32;
            lr -= (long long)(unsigned)a;
            hm -= c >> 32;
            lm -= (long long)(unsigned)c;
          }
        }
#pragma unroll
        for (int off = 1; off <= 16; off <<= 4) {   // the four threads of the line
          hr += __shfl_xor_sync(0xffffffffu, hr, off);
          lr += __shfl_xor_sync(0xffffffffu, lr, off);
          hm += __shfl_xor_sync(0xffffffffu, hm, off);
          lm += __shfl_xor_sync(0xffffffffu, lm, off);
        }
        if (g == 0 && rowok) {
          TO vr = ere == kNanRow ? qnan<TO>()
                                 : words_scaled<TO>(hr, lr, ere - F::EOFF - 62);
          TO vi = eim == kNanRow ? qnan<TO>()
                                 : words_scaled<TO>(hm, lm, eim - F::EOFF - 62);
          if (fwd) {
            vr = times<TO>(vr, lastf);
            vi = times<TO>(vi, lastf);
          }
          TO* o = out + ((size_t)fld * fso + (size_t)line * Nz + N) * 2;
          o[0] = vr;
          o[1] = vi;
        }
      }
      // the later passes: odd, then even and odd of each further slice, from the kept values
      for (int pp = pp0 + 1; pp < pp0 + np && ok; ++pp) {
        const int par = pp & 1;
        longlong2 nx[4];
        auto fetch = [&](int st) {
          const longlong2* s = keep_at(par, st);
#pragma unroll
          for (int i = 0; i < 4; ++i) nx[i] = __ldcg(s + i * kPW * 32);
        };
        fetch(0);
        for (int st = 0; st < nst && ok; ++st) {
          unsigned long long v[8];
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            v[2 * i] = (unsigned long long)nx[i].x;
            v[2 * i + 1] = (unsigned long long)nx[i].y;
          }
          if (st + 1 < nst) fetch(st + 1);
          ok = put(v, dig + ((size_t)pp * nst + st) * bstride);
        }
      }
      if (!ok) break;
    }
    // the copies still in flight finish (bounded) before the CTA ends: all were consumed unless a
    // wait ran out, in this warp or in the issuer
    if (p == 0) {
      const uint64_t dl = gtime() + kWaitNs;
      for (int b = 0; b < kStages; ++b) {
        const uint32_t n = use + (b < (int)slot ? 1u : 0u);   // copies issued to slot b
        if (n > 0 && !mbar_wait_until(barB + 8 * b, (n - 1) & 1, dl)) W.ok = false;
      }
    }
  } else {
    // ---- epilogue: warp w reads tensor-memory lanes 32 (w % 4) .. + 31 (its rows), columns
    // (w / 4) NT / 2 .. + NT / 2 - 1 of each of the eight accumulators
    const int qd = warp & 3, cg = warp >> 2, CW = NT / 2;
    const int row = qd * 32 + lane;
    const int l = (row >> 4) * 8 + (row & 7), part_c = (row >> 3) & 1;
    const uint32_t tb = tmem + ((uint32_t)(qd * 32) << 16) + (uint32_t)(cg * CW);
    // sums over several K groups are kept here between the groups
    long long* part = reinterpret_cast<long long*>(kcta + (size_t)2 * nst * kKeepStage) + tid;
    uint32_t pass = 0;
    int ti = 0;
    for (int item = blockIdx.x; item < nitems; item += gridDim.x, ++ti) {
      const int tile = item / nparts, pp0 = (item - tile * nparts) * np;
      const int fld = tile / tpf, rbuf = ti % kRB;
      const int line = (tile - fld * tpf) * (kRows / 2) + l;
      if (!W.wait_warp(barRow + 8 * rbuf, (ti / kRB) & 1)) break;
      const int me = sE[rbuf * kRows + row];
      const long long mid = sC[rbuf * kRows + row];
      __syncwarp();
      if (lane == 0)
        asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(barRowFree + 8 * rbuf)
                     : "memory");
      const bool rowok = line < nlines, nan = me == kNanRow;
      const int ex = me - F::EOFF - q;   // result = T 2^(E - q)
      const bool safe =
          __all_sync(0xffffffffu, !rowok || (!nan && safe_exp<TO>(ex))) != 0;
      TO* dst = out + ((size_t)fld * fso + (size_t)(rowok ? line : 0) * Nz) * 2 + part_c;
      bool ok = true;
      for (int pp = pp0; pp < pp0 + np && ok; ++pp) {
        const int par = pp & 1, m0 = (pp >> 1) * NT + cg * CW;
        TO* d = dst + 2 * (size_t)(2 * m0 + par);
        for (int c = 0; c < kc; ++c, ++pass) {
          if (!(ok = W.wait_warp(barAccFull, pass & 1))) break;
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          if (nmag == 8)
            epilogue_pass<TO, 8>(tb, NT, CW, m0, H, c, kc, par, rowok, nan, safe, ex, mid, fwd, part,
                                 d, barAccFree, lane);
          else if (nmag == 3)
            epilogue_pass<TO, 3>(tb, NT, CW, m0, H, c, kc, par, rowok, nan, safe, ex, mid, fwd, part,
                                 d, barAccFree, lane);
          else
            epilogue_pass<TO, 0>(tb, NT, CW, m0, H, c, kc, par, rowok, nan, safe, ex, mid, fwd, part,
                                 d, barAccFree, lane);
        }
      }
      if (!ok) break;
    }
  }
  if (!W.ok) atomicOr(err, 1);
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (issuer_warp)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512));
}

template <typename TI, typename TO>
cudaError_t launch_t(const void* in, long long fsi, void* out, long long fso, int nf, int nlines,
                     int Nz, const ChebTc& t, int* err, cudaStream_t s) {
  const int tpf = (nlines + kRows / 2 - 1) / (kRows / 2);
  const long long ntiles = (long long)nf * tpf;
  if (ntiles <= 0) return cudaSuccess;
  // Rule: as many CTAs to a tile as all tiles find an SM each; a tile's passes (two for N <= 128, four
  // up to 256) then run side by side and each CTA converts its rows again
  // (24 tiles, us, one CTA a tile / split: N = 128 30 / 18, N = 192 48 / 21, N = 256 62 / 26).
  int np = 2 * t.nsl;
  while (np % 2 == 0 && ntiles * (2 * t.nsl / np) * 2 <= t.ctas) np /= 2;
  const int grid = (int)std::min<long long>(ntiles * (2 * t.nsl / np), t.ctas);
  cheb_tc_kernel<TI, TO><<<grid, kThreads, kSmem, s>>>(
      (const TI*)in, fsi, (TO*)out, fso, nlines, Nz, tpf, (int)ntiles, np, t.NT, t.nsl, t.nst, t.kc,
      t.gst, t.nmag, t.dig, t.keep, (long long)cheb_tc_keep_bytes(Nz - 1), t.dir == 0 ? 1 : 0, t.q, t.ymid,
      t.dir == 0 ? 0.5 / (double)(Nz - 1) : 1.0, err);
  return cudaGetLastError();
}

uint16_t bf16_bits(float f) {
  uint32_t u;
  memcpy(&u, &f, sizeof u);
  return (uint16_t)(u >> 16);   // exact: a digit has at most eight significant bits
}

}  // namespace

int cheb_tc_tables(int N, int dir, std::vector<uint16_t>& dig, ChebTc* t) {
  if (N < 2 || N % 2 || (N + 16) / 16 * 16 >= 512) return -1;
  const int H = N / 2;
  t->dir = dir;
  t->nsl = (H + kNTMax - 1) / kNTMax;
  t->NT = ((H + t->nsl - 1) / t->nsl + 15) / 16 * 16;
  t->nst = (H + kKS - 1) / kKS;
  t->kc = (t->nst * kKS + kMaxK - 1) / kMaxK;
  t->gst = (t->nst + t->kc - 1) / t->kc;
  // one scale for the whole matrix, its largest weight (1 backward, 2 / N forward) at most 2^54
  t->q = 54;
  if (dir == 0)
    for (int h = H; h > 1; h >>= 1) ++t->q;
  // the weights times 2^q: W_nk = w cos(pi n k / N), w = 2 / N (forward, half of it at n = 0 and at
  // k = 0, where the cosine is 1) or 1; tabulated by angle
  const long double pi = 3.141592653589793238462643383279502884L;
  const long double w = dir == 0 ? 2.0L / (long double)N : 1.0L;
  std::vector<long long> Y(2 * N);
  for (int a = 0; a <= N; ++a) {
    long double c = 0.0L;
    if (2 * a < N) c = cosl(pi * (long double)a / (long double)N);
    else if (2 * a > N) c = -cosl(pi * (long double)(N - a) / (long double)N);
    Y[a] = (long long)llroundl(ldexpl(w * c, t->q));
  }
  for (int a = N + 1; a < 2 * N; ++a) Y[a] = Y[2 * N - a];
  const long long Yh = (long long)llroundl(ldexpl(0.5L * w, t->q));
  const long long Yq = (long long)llroundl(ldexpl(0.25L * w, t->q));
  t->ymid = dir == 0 ? (long long)llroundl(ldexpl(2.0L / (long double)N, t->q)) : 1ll << 54;
  const int NT = t->NT;
  double bound = 0.0, bound3 = 0.0;   // of all accumulators and of the first three
  const size_t block = (size_t)kPlanes * NT * kKS;
  dig.assign((size_t)2 * t->nsl * t->nst * block, 0);
  for (int m = 0; m < H; ++m)
    for (int par = 0; par < 2; ++par) {
      double sum[kPlanes] = {};          // sum_k |digit j|
      for (int k = 0; k < H; ++k) {
        const int st = k / kKS, kk = k % kKS;
        const int pos = 4 * (kk & 3) + (kk >> 2);   // k = 16 st + g + 4 e sits at position 4 g + e
        const int n = 2 * m + par;
        const long long yk = dir == 1 || (n > 0 && k > 0) ? Y[((long long)n * k) % (2 * N)]
                             : n == 0 && k == 0          ? Yq
                                                         : Yh;
        const unsigned long long y = (unsigned long long)yk + kBias;
        uint16_t* b = dig.data() + ((size_t)(2 * (m / NT) + par) * t->nst + st) * block;
        for (int j = 0; j < kPlanes; ++j) {
          const int row = j * NT + m % NT, d = (int)((y >> (8 * (6 - j))) & 255ull) - 128;
          b[((size_t)(pos >> 3) * kPlanes * NT + row) * 8 + (pos & 7)] = bf16_bits((float)d);
          sum[j] += abs(d);
        }
      }
      // |G_d| <= 128 sum_{j <= d} sum_k |b_jk|
      double acc = 0.0;
      for (int j = 0; j < kPlanes; ++j) {
        acc += 128.0 * sum[j];
        if (j == 2) bound3 = std::max(bound3, acc);
      }
      bound = std::max(bound, acc);
    }
  t->nmag = bound <= 4194304.0 ? 8 : (bound3 <= 4194304.0 ? 3 : 0);
  return 0;
}

size_t cheb_tc_keep_bytes(int N) {
  const size_t nst = (N / 2 + kKS - 1) / kKS;
  return 2 * nst * kKeepStage + (size_t)(kNTMax / 2) * kEW * 32 * sizeof(long long);
}

cudaError_t cheb_tc_prepare() {
  static SmemLimit c0, c1, c2, c3, c4;
  cudaError_t e = ensure_smem(cheb_tc_kernel<double, double>, kSmem, &c0);
  if (e == cudaSuccess) e = ensure_smem(cheb_tc_kernel<float, double>, kSmem, &c1);
  if (e == cudaSuccess) e = ensure_smem(cheb_tc_kernel<double, float>, kSmem, &c2);
  if (e == cudaSuccess) e = ensure_smem(cheb_tc_kernel<df, double>, kSmem, &c3);
  if (e == cudaSuccess) e = ensure_smem(cheb_tc_kernel<double, df>, kSmem, &c4);
  return e;
}

cudaError_t launch_cheb_tc(int tin, int tout, const void* in, long long fsi, void* out,
                           long long fso, int nf, int nlines, int Nz, const ChebTc& t, int* err,
                           cudaStream_t s) {
  if (tin == 0 && tout == 0)
    return launch_t<double, double>(in, fsi, out, fso, nf, nlines, Nz, t, err, s);
  if (tin == 1 && tout == 0)
    return launch_t<float, double>(in, fsi, out, fso, nf, nlines, Nz, t, err, s);
  if (tin == 0 && tout == 1)
    return launch_t<double, float>(in, fsi, out, fso, nf, nlines, Nz, t, err, s);
  if (tin == 2 && tout == 0)
    return launch_t<df, double>(in, fsi, out, fso, nf, nlines, Nz, t, err, s);
  if (tin == 0 && tout == 2)
    return launch_t<double, df>(in, fsi, out, fso, nf, nlines, Nz, t, err, s);
  return cudaErrorInvalidValue;
}

// Failure path of the bounded waits, exercised on purpose: one thread runs a loop of `nwaits`
// waits of the transform's shape (the same Waiter, alternating the parities of two mbarriers)
// on barriers that nothing arrives at.  The first wait gives up after kWaitNs and every later
// one returns at once, so the kernel ends after about one bound however long the loop; the
// thread records the failure in err[0] and the number of waits that actually spun in err[1].
// No TMEM and no asynchronous copy is involved, so nothing else is left in flight.
__global__ void __launch_bounds__(32) wait_selftest_kernel(int* __restrict__ err, int nwaits) {
  __shared__ __align__(8) uint64_t bar[2];
  if (threadIdx.x != 0) return;
  const uint32_t b0 = su32(&bar[0]), b1 = su32(&bar[1]);
  asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(b0));
  asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(b1));
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  Waiter W;
  int spun = 0;
  for (int i = 0; i < nwaits; ++i) {
    if (W.ok) ++spun;
    W.wait((i & 1) ? b1 : b0, (uint32_t)((i >> 1) & 1));
  }
  if (!W.ok) atomicOr(&err[0], 1);
  atomicAdd(&err[1], spun);
}

// Eight independent float64 FMA chains per thread (enough to cover the pipe's latency): x <- x
// a + b with |a| < 1, so the values stay bounded; the sum is stored so nothing is dead code.
__global__ void __launch_bounds__(256) fma_probe_kernel(double* __restrict__ out, int iters) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  double x[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) x[i] = 1e-3 * (t + i);
  const double a = 0.999999, b = 1e-6;
  for (int it = 0; it < iters; ++it) {
#pragma unroll
    for (int i = 0; i < 8; ++i) x[i] = fma(x[i], a, b);
  }
  double s = 0.0;
#pragma unroll
  for (int i = 0; i < 8; ++i) s += x[i];
  out[t] = s;
}

cudaError_t launch_fma_probe(double* out, int blocks, int iters, cudaStream_t s) {
  fma_probe_kernel<<<blocks, 256, 0, s>>>(out, iters);
  return cudaGetLastError();
}

cudaError_t launch_wait_selftest(int* err, int nwaits, cudaStream_t s) {
  wait_selftest_kernel<<<1, 32, 0, s>>>(err, nwaits);
  return cudaGetLastError();
}

}  // namespace chf
