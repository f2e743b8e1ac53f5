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
// Persistent CTAs (one per SM) have three kinds of warps, so conversion, MMAs and the epilogue of
// different passes overlap:
//   producers (8 warps): per K stage of 16 (one MMA k-step) a thread converts four pairs
//     (x_k, x_{N-k}) of the real and imaginary rows of one line to fixed point, writes the seven
//     digit planes of the sums to the stage's shared buffer and keeps the differences (and, with
//     several slices, the sums) in a per-CTA buffer in global memory (L2), read back by the same
//     thread for the later passes; thread 0 also issues the bulk copy of the stage's matrix digits;
//   issuer (1 thread): the MMAs of each stage as it fills;
//   epilogue (8 warps): drains a pass's accumulators, recombines and stores.
// What bounds it: integer issue (about 45 instructions per element converted and 25 per output)
// and the shared-memory bandwidth of the MMA operands; the tensor pipe itself needs 0.93 of the
// 16-wide stage's time at NT = 64.
#include <math.h>
#include <stdint.h>
#include <string.h>

#include <algorithm>
#include <vector>

#include "ch_internal.h"
#include "ch_tc.cuh"

namespace chf {

namespace {

using namespace tc;

constexpr int kPW = 8, kEW = 8;                   // producer and epilogue warps
constexpr int kThreads = 32 * (kPW + kEW + 1);    // epilogue 0..7, producers 8..15, issuer 16
constexpr int kStages = 5;                        // K stages in flight
constexpr int kStageBytes = kABytes + b_stage_bytes(kNTMax);
// per stage full, bfull, empty; accfull, accfree, rowfull[2], rowfree[2], fin
constexpr int kBars = 3 * kStages + 7;
// stages, row scales and middle terms (two tiles), barriers, the tensor-memory address
constexpr size_t kSmem = (size_t)kStages * kStageBytes + 2 * kRows * (sizeof(long long) + sizeof(int)) +
                         (size_t)(kBars + 1) * 8;
// one pass's stage block kept in global memory: four fixed-point values of two rows per thread
constexpr size_t kKeepStage = (size_t)kPW * 32 * 8 * sizeof(long long);

template <typename TO> __device__ __forceinline__ TO times(TO v, double f) { return v; }
template <> __device__ __forceinline__ double times<double>(double v, double f) { return v * f; }

// in / out: nf fields of complex lines (re, im interleaved), field stride fsi / fso complex
// elements, line stride Nz = N + 1; dig: the matrix digits, stage blocks of 7 NT rows x 16 K in
// the order slice, parity, stage; keep: keep_bytes per CTA; nst stages per parity in kc groups of
// gst; q: log2 of the matrix scale; ymid: middle weight times 2^q; lastf: factor of output N
// (forward).
template <typename TI, typename TO>
__global__ void __launch_bounds__(kThreads, 1)
    cheb_tc_kernel(const TI* __restrict__ in, long long fsi, TO* __restrict__ out, long long fso,
                   int nlines, int Nz, int tpf, int ntiles, int NT, int nsl, int nst, int kc,
                   int gst, const uint16_t* __restrict__ dig, char* __restrict__ keep,
                   long long keep_bytes, int fwd, int q, long long ymid, double lastf,
                   int* __restrict__ err) {
  typedef FBits<TI> F;
  typedef typename F::U U;
  extern __shared__ __align__(1024) unsigned char tsm[];
  unsigned char* stages = tsm;
  long long* sC = reinterpret_cast<long long*>(tsm + (size_t)kStages * kStageBytes);
  int* sE = reinterpret_cast<int*>(sC + 2 * kRows);
  unsigned long long* bars = reinterpret_cast<unsigned long long*>(sE + 2 * kRows);
  uint32_t* sT = reinterpret_cast<uint32_t*>(bars + kBars);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int N = Nz - 1, H = N / 2;
  const uint32_t barFull = su32(bars), barB = barFull + 8 * kStages;
  const uint32_t barEmpty = barFull + 16 * kStages, barAccFull = barFull + 24 * kStages;
  const uint32_t barAccFree = barAccFull + 8, barRow = barAccFull + 16, barRowFree = barAccFull + 32;
  const uint32_t barFin = barAccFull + 48;
  if (tid == 0) {
    for (int b = 0; b < kStages; ++b) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(barFull + 8 * b), "r"(kPW));
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(barB + 8 * b));
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(barEmpty + 8 * b));
    }
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(barAccFull));
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(barAccFree), "r"(kEW));
    for (int b = 0; b < 2; ++b) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(barRow + 8 * b), "r"(kPW));
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(barRowFree + 8 * b), "r"(kEW));
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
      for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x)
        for (int pp = 0; pp < 2 * nsl; ++pp)
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
      if (!W.ok && any) {
        // a wait ran out: nothing more is issued; wait (bounded) for the MMAs in flight before
        // the tensor memory is released
        mma_commit(barFin);
        mbar_wait_until(barFin, 0, gtime() + kWaitNs);
      }
    }
    __syncwarp();
  } else if (warp >= kEW) {
    // ---- producers: thread = (line l of the tile, g): K positions 4 g .. 4 g + 3 of a stage,
    // position 4 g + e holding k = 16 st + g + 4 e (so the four threads of a line read
    // consecutive elements).  Rows 2 l (re) and 2 l + 1 (im); threads g >= 2 take the im row
    // first, so that a half-warp's 8-byte stores fall on different banks.
    const int p = tid - 32 * kEW, pw = warp - kEW;
    const int l = pw * 8 + (lane >> 2), g = lane & 3, sw = g >> 1;
    const int ra = 2 * l + sw, rb = 2 * l + 1 - sw;
    const uint32_t oa = (uint32_t)(sw * (int)kALbo + ra * 16 + (g & 1) * 8);
    const uint32_t ob = (uint32_t)(sw * (int)kALbo + rb * 16 + (g & 1) * 8);
    const uint64_t pol = policy_evict_last();
    longlong2* kp = reinterpret_cast<longlong2*>(kcta) + p;
    uint32_t slot = 0, use = 0;
    int ti = 0;
    // the stage's digit planes of v (0..3 row a, 4..7 row b) and, by one thread, the copy of its
    // matrix digits; false after a wait ran out
    auto put = [&](const long long (&v)[8], const uint16_t* bsrc) {
      if (use > 0 && !W.wait_warp(barEmpty + 8 * slot, (use & 1) ^ 1)) return false;
      unsigned char* sA = stages + (size_t)slot * kStageBytes;
      if (p == 0) bulk_load(su32(sA) + (uint32_t)kABytes, bsrc, bbytes, barB + 8 * slot, pol);
      uint32_t lo[8], hi[8];
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        const unsigned long long y = (unsigned long long)v[e] + kBias;
        lo[e] = (uint32_t)y;
        hi[e] = (uint32_t)(y >> 32);
      }
#pragma unroll
      for (int i = 0; i < kPlanes; ++i) {
        const int b = 6 - i;
        const uint32_t* w = b < 4 ? lo : hi;
        *reinterpret_cast<uint2*>(sA + i * kPlaneBytes + oa) =
            make_uint2(digit_pair(w[0], w[1], b & 3), digit_pair(w[2], w[3], b & 3));
        *reinterpret_cast<uint2*>(sA + i * kPlaneBytes + ob) =
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
    auto store_keep = [&](longlong2* d, const long long (&v)[8]) {
#pragma unroll
      for (int i = 0; i < 4; ++i) __stcg(d + i * kPW * 32, make_longlong2(v[2 * i], v[2 * i + 1]));
    };
    const size_t bstride = (size_t)bbytes / 2;   // elements of a stage block
    for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x, ++ti) {
      const int fld = tile / tpf;
      const int line = (tile - fld * tpf) * (kRows / 2) + l;
      const bool rowok = line < nlines;
      const TI* src = in + ((size_t)fld * fsi + (size_t)(rowok ? line : 0) * Nz) * 2;
      // the rows' scales (their first, cold read)
      unsigned ka = 0, kb = 0;
      if (rowok) {
#pragma unroll 8
        for (int k = g; k < Nz; k += 4) {
          ka = max(ka, F::key(F::bits(src[2 * k + sw])));
          kb = max(kb, F::key(F::bits(src[2 * k + 1 - sw])));
        }
      }
      // threads g >= 2 hold the rows the other way round
      unsigned kre = sw ? kb : ka, kim = sw ? ka : kb;
#pragma unroll
      for (int off = 1; off < 4; off <<= 1) {
        kre = max(kre, __shfl_xor_sync(0xffffffffu, kre, off));
        kim = max(kim, __shfl_xor_sync(0xffffffffu, kim, off));
      }
      const int ere = row_scale<TI>(kre), eim = row_scale<TI>(kim);
      const int ea = sw ? eim : ere, eb = sw ? ere : eim;
      // the middle element, its integer term for the even outputs, and the row scales
      long long xmr = 0, xmi = 0;
      if (g == 0) {
        if (rowok) {
          xmr = to_fixed<TI>(F::bits(src[2 * H]), ere);
          xmi = to_fixed<TI>(F::bits(src[2 * H + 1]), eim);
        }
      }
      if (ti >= 2 && !W.wait_warp(barRowFree + 8 * (ti & 1), ((ti >> 1) - 1) & 1)) break;
      if (g == 0) {
        // x_H Y_H / 2^54 (|x_H| < 2^54, Y_H <= 2^54)
        sC[(ti & 1) * kRows + 2 * l] = __mul64hi(xmr * 256, ymid * 4);
        sC[(ti & 1) * kRows + 2 * l + 1] = __mul64hi(xmi * 256, ymid * 4);
        sE[(ti & 1) * kRows + 2 * l] = ere;
        sE[(ti & 1) * kRows + 2 * l + 1] = eim;
      }
      __syncwarp();
      if (lane == 0)
        asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(barRow + 8 * (ti & 1))
                     : "memory");
      // first pass: convert, fold, write the sums' planes, keep the differences
      long long suma = 0, sumb = 0, s0a = 0, s0b = 0;
      U xa[4], ya[4], xb[4], yb[4];
      auto load = [&](int st) {
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const int k = 16 * st + g + 4 * e;
          const bool ok = rowok && k < H;
          xa[e] = xb[e] = ya[e] = yb[e] = 0;
          if (ok) {
            xa[e] = F::bits(src[2 * k + sw]);
            xb[e] = F::bits(src[2 * k + 1 - sw]);
            ya[e] = F::bits(src[2 * (N - k) + sw]);
            yb[e] = F::bits(src[2 * (N - k) + 1 - sw]);
          }
        }
      };
      load(0);
      bool ok = true;
      for (int st = 0; st < nst && ok; ++st) {
        long long s[8], d[8];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const long long x = to_fixed<TI>(xa[e], ea), y = to_fixed<TI>(ya[e], ea);
          const long long z = to_fixed<TI>(xb[e], eb), w = to_fixed<TI>(yb[e], eb);
          s[e] = x + y;
          d[e] = x - y;
          s[4 + e] = z + w;
          d[4 + e] = z - w;
          suma += s[e];       // at most 62 values below 2^55 per thread
          sumb += s[4 + e];
        }
        if (st == 0) {
          s0a = s[0];
          s0b = s[4];
        }
        store_keep(keep_at(1, st), d);
        if (nsl > 1) store_keep(keep_at(0, st), s);
        if (st + 1 < nst) load(st + 1);
        ok = put(s, dig + (size_t)st * bstride);
      }
      if (!ok) break;
      // the last output n = N: sum_k w_k (-1)^k x_k, (-1)^k = (-1)^g for this thread's k; weights
      // e_k = 2 except k = 0, N (forward) or 1
      {
        long long tre = sw ? sumb : suma, tim = sw ? suma : sumb;
        if (g & 1) {
          tre = -tre;
          tim = -tim;
        }
        const int m2 = (H & 1) ? -1 : 1;
        // |partial| < 2^61 here; halves of 27 low bits keep the sums over threads in range
        long long hr = tre >> 27, lr = tre & 0x7FFFFFF, hi_ = tim >> 27, li = tim & 0x7FFFFFF;
        if (fwd) {
          hr *= 2; lr *= 2; hi_ *= 2; li *= 2;
        }
        if (g == 0) {
          const int wm = fwd ? 2 * m2 : m2;
          hr += wm * (xmr >> 27); lr += wm * (xmr & 0x7FFFFFF);
          hi_ += wm * (xmi >> 27); li += wm * (xmi & 0x7FFFFFF);
          if (fwd) {   // s_0 counted twice (g = 0: rows in order)
            hr -= s0a >> 27; lr -= s0a & 0x7FFFFFF;
            hi_ -= s0b >> 27; li -= s0b & 0x7FFFFFF;
          }
        }
#pragma unroll
        for (int off = 1; off < 4; off <<= 1) {
          hr += __shfl_xor_sync(0xffffffffu, hr, off);
          lr += __shfl_xor_sync(0xffffffffu, lr, off);
          hi_ += __shfl_xor_sync(0xffffffffu, hi_, off);
          li += __shfl_xor_sync(0xffffffffu, li, off);
        }
        if (g == 0 && rowok) {
          // sum = 2^(E - 54) (h 2^27 + l) = T 2^(E - 51), T = h 2^24 + l / 8
          TO vr = ere == kNanRow ? qnan<TO>()
                                 : scaled<TO>(hr * 16777216ll + ((lr + 4) >> 3), ere - F::EOFF - 51);
          TO vi = eim == kNanRow ? qnan<TO>()
                                 : scaled<TO>(hi_ * 16777216ll + ((li + 4) >> 3), eim - F::EOFF - 51);
          if (fwd) {
            vr = times<TO>(vr, lastf);
            vi = times<TO>(vi, lastf);
          }
          TO* o = out + ((size_t)fld * fso + (size_t)line * Nz + N) * 2;
          o[0] = vr;
          o[1] = vi;
        }
      }
      // the later passes: slice 0 odd, then even and odd of each further slice, from the kept values
      for (int pp = 1; pp < 2 * nsl && ok; ++pp) {
        const int par = pp & 1;
        longlong2 nx[4];
        auto fetch = [&](int st) {
          const longlong2* s = keep_at(par, st);
#pragma unroll
          for (int i = 0; i < 4; ++i) nx[i] = __ldcg(s + i * kPW * 32);
        };
        fetch(0);
        for (int st = 0; st < nst && ok; ++st) {
          long long v[8];
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            v[2 * i] = nx[i].x;
            v[2 * i + 1] = nx[i].y;
          }
          if (st + 1 < nst) fetch(st + 1);
          ok = put(v, dig + ((size_t)pp * nst + st) * bstride);
        }
      }
      if (!ok) break;
    }
    // after a failed wait the copies still in flight finish (bounded) before the CTA ends
    if (!W.ok && p == 0) {
      const uint64_t dl = gtime() + kWaitNs;
      for (int b = 0; b < kStages; ++b) {
        const uint32_t n = use + (b < (int)slot ? 1u : 0u);   // copies issued to slot b
        if (n > 0) mbar_wait_until(barB + 8 * b, (n - 1) & 1, dl);
      }
    }
  } else {
    // ---- epilogue: warp w reads tensor-memory lanes 32 (w % 4) .. + 31 (its rows), columns
    // (w / 4) NT / 2 .. + NT / 2 - 1 of each of the seven accumulators, four at a time
    const int qd = warp & 3, cg = warp >> 2, CW = NT / 2;
    const int row = qd * 32 + lane;
    const uint32_t tb = tmem + ((uint32_t)(qd * 32) << 16) + (uint32_t)(cg * CW);
    // sums over several K groups are kept here between the groups
    long long* part = reinterpret_cast<long long*>(kcta + (size_t)2 * nst * kKeepStage) + tid;
    uint32_t pass = 0;
    int ti = 0;
    for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x, ++ti) {
      const int fld = tile / tpf;
      const int line = (tile - fld * tpf) * (kRows / 2) + (row >> 1);
      if (!W.wait_warp(barRow + 8 * (ti & 1), (ti >> 1) & 1)) break;
      const int me = sE[(ti & 1) * kRows + row];
      const long long mid = sC[(ti & 1) * kRows + row];
      __syncwarp();
      if (lane == 0)
        asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(barRowFree + 8 * (ti & 1))
                     : "memory");
      const bool rowok = line < nlines, nan = me == kNanRow;
      const int ex = me - F::EOFF - q;   // result = T 2^(E - q)
      TO* dst = out + ((size_t)fld * fso + (size_t)(rowok ? line : 0) * Nz) * 2 + (row & 1);
      bool ok = true;
      for (int pp = 0; pp < 2 * nsl && ok; ++pp) {
        const int par = pp & 1, m0 = (pp >> 1) * NT + cg * CW;
        for (int c = 0; c < kc; ++c, ++pass) {
          if (!(ok = W.wait_warp(barAccFull, pass & 1))) break;
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          for (int c0 = 0; c0 < CW; c0 += 4) {
            uint32_t v[7][4];
            tmem_ld7x4(tb + (uint32_t)c0, NT, v);
            if (c0 + 4 >= CW) {   // all read: the accumulators are free for the next pass
              asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
              __syncwarp();
              if (lane == 0)
                asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(barAccFree)
                             : "memory");
            }
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              const int m = m0 + c0 + e;
              if (m < H && rowok) {
                long long T = recombine(v, e);
                if (c > 0) T += part[(c0 + e) * kEW * 32];
                if (c + 1 < kc) {
                  part[(c0 + e) * kEW * 32] = T;
                  continue;
                }
                if (par == 0) {
                  // (-1)^m x_H Y; the forward weight of n = 0 is half the others'
                  const long long t = (fwd && m == 0) ? mid / 2 : mid;
                  T += (m & 1) ? -t : t;
                }
                dst[2 * (size_t)(2 * m + par)] = nan ? qnan<TO>() : scaled<TO>(T, ex);
              }
            }
          }
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
  const int grid = (int)std::min<long long>(ntiles, t.ctas);
  cheb_tc_kernel<TI, TO><<<grid, kThreads, kSmem, s>>>(
      (const TI*)in, fsi, (TO*)out, fso, nlines, Nz, tpf, (int)ntiles, t.NT, t.nsl, t.nst, t.kc,
      t.gst, t.dig, t.keep, (long long)cheb_tc_keep_bytes(Nz - 1), t.dir == 0 ? 1 : 0, t.q, t.ymid,
      t.dir == 0 ? 0.5 / (double)(Nz - 1) : 1.0, err);
  return cudaGetLastError();
}

uint16_t bf16_bits(float f) {
  uint32_t u;
  memcpy(&u, &f, sizeof u);
  return (uint16_t)(u >> 16);   // exact: a digit has at most eight significant bits
}

// weight of input k in output n < N, times 2^q; cs[a] = cos(pi a / N)
long long weight(const std::vector<long double>& cs, int N, int dir, int q, int n, int k) {
  long double v = cs[((long long)n * k) % (2 * N)];
  if (dir == 0) v *= (k == 0 ? 1.0L : 2.0L) / ((n == 0 ? 2.0L : 1.0L) * (long double)N);
  return (long long)llroundl(ldexpl(v, q));
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
  const long double pi = 3.141592653589793238462643383279502884L;
  std::vector<long double> cs(2 * N);   // cos(pi a / N)
  for (int a = 0; a <= N; ++a) {
    if (2 * a == N) cs[a] = 0.0L;
    else if (2 * a < N) cs[a] = cosl(pi * (long double)a / (long double)N);
    else cs[a] = -cosl(pi * (long double)(N - a) / (long double)N);
  }
  for (int a = N + 1; a < 2 * N; ++a) cs[a] = cs[2 * N - a];
  t->ymid = dir == 0 ? (long long)llroundl(ldexpl(2.0L / (long double)N, t->q)) : 1ll << 54;
  const int NT = t->NT;
  const size_t block = (size_t)kPlanes * NT * kKS;
  dig.assign((size_t)2 * t->nsl * t->nst * block, 0);
  for (int m = 0; m < H; ++m)
    for (int par = 0; par < 2; ++par)
      for (int k = 0; k < H; ++k) {
        const int st = k / kKS, kk = k % kKS;
        const int pos = 4 * (kk & 3) + (kk >> 2);   // k = 16 st + g + 4 e sits at position 4 g + e
        const unsigned long long y = (unsigned long long)weight(cs, N, dir, t->q, 2 * m + par, k) + kBias;
        uint16_t* b = dig.data() + ((size_t)(2 * (m / NT) + par) * t->nst + st) * block;
        for (int j = 0; j < kPlanes; ++j) {
          const int row = j * NT + m % NT;
          b[((size_t)(pos >> 3) * kPlanes * NT + row) * 8 + (pos & 7)] =
              bf16_bits((float)((int)((y >> (8 * (6 - j))) & 255ull) - 128));
        }
      }
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
