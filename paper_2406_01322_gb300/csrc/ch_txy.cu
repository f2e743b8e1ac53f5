// Float64 Fourier transforms along y and x (Sec. 3.2.1, with the 3/2-rule padding and truncation)
// as exact-split products on the tensor cores (ch_tc.cuh): dense real cosine and sine matrices of
// the padded lengths, float64-accurate, in place of shared-memory FFTs on the float64 pipe.
//
// GB300 issues about 1.6 float64 operations per clock per SM; a padded line of 192 points costs
// about 12 of them per real sample by FFT, which is what bounded these passes.  As digit products
// the same transforms need no float64 arithmetic: about 50 integer instructions per sample
// converted, 30 per sample produced, and tensor work that stays below both for the lengths used.
//
// Four transforms, n = 0 .. nout - 1 and P the padded length:
//   YB (modes -> samples in y):  f(n), f(P-n) = C +- i S,  C = sum_k s_k cos, S = sum_k d_k sin,
//      s_k = c_k + c_{-k}, d_k = c_k - c_{-k} (s_0 = c_0), k < Ny / 2;
//   YF (samples -> modes in y):  c_n, c_{-n} = C -+ i S,  s_k = f(k) + f(P-k), d_k = f(k) - f(P-k);
//   XB (half spectrum -> real samples in x):  f(n), f(P-n) = E +- O,
//      E = Re c_0 + 2 sum Re c_k cos, O = -2 sum Im c_k sin;
//   XF (real samples -> half spectrum):  Re c_n = sum s_k cos, Im c_n = -sum d_k sin;
// angles 2 pi k n / P.  The sums and differences s, d are exact in fixed point, both products of an
// output are recombined as integers of one scale and added exactly, so every result is rounded
// once.  For even P the sample k = P / 2 of a forward transform enters as (-1)^n times its weight
// (added to the recombined integer), and the output n = P / 2 of a backward transform, an
// alternating sum, is formed exactly by the producers.
//
// Tiles, warps and stages as in the Chebyshev transform (ch_tc.cu): a tile is 64 complex lines
// (re and im rows; YB, YF) or 128 lines (XB, XF), lines neighbouring in memory so that every load
// and store of a warp covers whole sectors; passes are (output slice, cosine or sine product, K
// group).  The recombined cosine products wait in shared memory for the sine ones.
#include <math.h>
#include <stdint.h>
#include <stdlib.h>
#include <string.h>

#include <algorithm>
#include <type_traits>
#include <vector>

#include "ch_internal.h"
#include "ch_tc.cuh"

namespace chf {

namespace {

using namespace tc;

constexpr int kPW = 8, kEW = 8, kSW = 3;               // producer, epilogue and scan warps
constexpr int kThreads = 32 * (kPW + kEW + 1 + kSW);   // epilogue 0..7, producers, issuer, scan
constexpr int kMaxStages = 6;
constexpr int kMaxFields = 9;
constexpr int kMaxSlices = 8;   // transforms of up to 1024 points
// tiles whose row scales are held: the scan runs at most this far ahead (with three, and an L2
// prefetch of a fourth, tiles left L2 before they were converted: 256x256x129 y forward 1.75 ms
// against 1.49)
constexpr int kRB = 2;
constexpr int kBars = 3 * kMaxStages + 4 + 2 * kRB;
constexpr size_t kTail = kRB * kRows * (sizeof(long long) + 2 * sizeof(int)) + (size_t)(kBars + 1) * 8;
// fixed-point values of one pass's stage block kept in global memory, eight per producer thread
constexpr size_t kKeepStage = (size_t)kPW * 32 * 8 * sizeof(long long);

__host__ __device__ constexpr int stage_bytes(int NT) { return kABytes + b_stage_bytes(NT); }

enum { YB = 0, YF = 1, XB = 2, XF = 3 };

struct Args {
  const double* in[kMaxFields];   // input and output of each output field
  double* out[kMaxFields];
  unsigned dmask;             // output fields of i k times the input
  double kscale;              // k of mode 1
  int nlines, tpf, ntiles;    // lines per field, tiles per field, tiles
  // SPLIT: the output slices of a tile are shared by gridDim.y CTAs, cut[blockIdx.y] ..
  // cut[blockIdx.y + 1] - 1
  short cut[kMaxSlices + 1];
  // line l starts at element (l / ld) ihs + (l % ld) ils of the input (complex elements; real
  // samples for XF) and (l / ld) ohs + (l % ld) ols of the output (real samples for XB)
  int ld;
  long long ihs, ils, ohs, ols;
  long long estr, ostr;       // element strides along the transform, in and out
  int n1, P;                  // modes of the full spectrum (Ny; unused for x), transform length
  int lift;                   // XF: outputs n >= 1 times 2^lift
  TxyPlan t;
  char* keep;
  long long keep_bytes;
  int* err;
};

// row of complex line l (YB, YF): lines in blocks of eight, real parts then imaginary parts
__device__ __forceinline__ int tile_row(int l, int part) { return (l >> 3) * 16 + part * 8 + (l & 7); }

__device__ __forceinline__ unsigned dkey(double v) {
  return FBits<double>::key(FBits<double>::bits(v));
}
template <bool TINY> __device__ __forceinline__ long long fix(double v, int maxe) {
  return Fixed<double, TINY>::of(FBits<double>::bits(v), maxe);
}

// outputs of one thread in one pass: columns m0 .. m0 + CW - 1 of its row
template <int MODE, int NMAG>
__device__ __forceinline__ void epilogue_pass(const Args& A, uint32_t tb, int CW, int m0, int grp,
                                              int c, bool rowok, bool nan, bool safe, int ex,
                                              long long mid, int part_c, long long* part,
                                              long long* hold, double* dst, uint32_t barAccFree,
                                              int lane) {
  const int nout = A.t.nout;
  for (int c0 = 0; c0 < CW; c0 += 4) {
    uint32_t v[kDiags][4];
    tmem_ldx4(tb + (uint32_t)c0, A.t.NT, v);
    if (c0 + 4 >= CW) {   // all read: the accumulators are free for the next pass
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncwarp();
      if (lane == 0)
        asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(barAccFree) : "memory");
    }
    long long T[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) T[e] = recombine<NMAG>(v, e);
    if (A.t.kc > 1) {
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        if (c > 0) T[e] += part[(c0 + e) * kEW * 32];
        if (c + 1 < A.t.kc) part[(c0 + e) * kEW * 32] = T[e];
      }
      if (c + 1 < A.t.kc) continue;
    }
    if (grp == 0) {
      if (MODE == YF || MODE == XF) {   // (-1)^n times the middle sample (m0 + c0 is even)
        T[0] += mid;
        T[1] -= mid;
        T[2] += mid;
        T[3] -= mid;
      }
#pragma unroll
      for (int e = 0; e < 4; ++e) hold[(c0 + e) * kEW * 32] = T[e];
      continue;
    }
    double ra[4], rb[4];
    long long a[4], b[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const long long h = hold[(c0 + e) * kEW * 32];
      if (MODE == YB || MODE == YF) {
        // the other part's sine product: re rows take -S_im (YB) or +S_im (YF), im rows the other
        long long o = __shfl_xor_sync(0xffffffffu, T[e], 8);
        if ((part_c == 0) == (MODE == YB)) o = -o;
        a[e] = h + o;
        b[e] = h - o;
      } else if (MODE == XB) {
        a[e] = h + T[e];
        b[e] = h - T[e];
      } else {
        a[e] = h;
        b[e] = T[e];
      }
    }
    if (safe) {
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        ra[e] = scaled<double>(a[e], ex);
        rb[e] = scaled_alu<double>(b[e], ex);
      }
    } else {
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        ra[e] = nan ? qnan<double>() : scaled_any<double>(a[e], ex);
        rb[e] = nan ? qnan<double>() : scaled_any<double>(b[e], ex);
      }
    }
    if (MODE == XF && A.lift && m0 + c0 == 0)
      ra[0] = nan ? qnan<double>() : scaled_any<double>(a[0], ex - A.lift);
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int n = m0 + c0 + e;
      if (!rowok || n >= nout) continue;
      if (MODE == XF) {
        *reinterpret_cast<double2*>(dst + 2 * (size_t)n * A.ostr) = make_double2(ra[e], rb[e]);
      } else if (MODE == XB) {
        // in rows of samples (ostr = 1) on 16-byte boundaries, samples n, n + 1 (n even) in one store
        const bool rows = A.ostr == 1 && ((uintptr_t)dst & 15) == 0;
        if (rows && !(e & 1) && n + 1 < nout)
          *reinterpret_cast<double2*>(dst + n) = make_double2(ra[e], ra[e | 1]);
        else if (!rows || !(e & 1))
          dst[(size_t)n * A.ostr] = ra[e];
        if (n > 0) dst[(size_t)(A.P - n) * A.ostr] = rb[e];
      } else if (MODE == YB) {
        dst[2 * (size_t)n * A.ostr] = ra[e];
        if (n > 0) dst[2 * (size_t)(A.P - n) * A.ostr] = rb[e];
      } else {
        // the y Nyquist row (n1 / 2) is zero
        dst[2 * (size_t)n * A.ostr] = ra[e];
        dst[2 * (size_t)(n > 0 ? A.n1 - n : A.n1 / 2) * A.ostr] = n > 0 ? rb[e] : 0.0;
      }
    }
  }
}

// SPLIT: several CTAs to a tile (its own instantiation: with the passes' bounds at run time in the only
// one, the x line of 128 x 128 x 129 went from 0.81 to 0.84 ms)
template <int MODE, bool SPLIT>
__global__ void __launch_bounds__(kThreads, 1) txy_kernel(const __grid_constant__ Args A) {
  constexpr bool CPX = MODE == YB || MODE == YF;   // rows: re and im of 64 lines; else 128 lines
  constexpr int LPT = CPX ? kRows / 2 : kRows;     // lines per tile
  constexpr int ISC = MODE == XF ? 1 : 2;          // doubles per input element
  constexpr int OSC = MODE == XB ? 1 : 2;
  extern __shared__ __align__(1024) unsigned char tsm[];
  const int NT = A.t.NT, ns = A.t.stages, nst = A.t.nst;
  // this CTA's passes
  const int pp0 = SPLIT ? 2 * A.cut[blockIdx.y] : 0;
  const int pp1 = SPLIT ? 2 * A.cut[blockIdx.y + 1] : 2 * A.t.nsl;
  const int sbytes = stage_bytes(NT);
  unsigned char* stages = tsm;
  // the recombined cosine products of a pass, per epilogue thread (in L2 instead, with room for five
  // stages, the epilogue was slower: y backward 0.20 -> 0.23, x backward 0.28 -> 0.31 ms at 128^3)
  long long* hold0 = reinterpret_cast<long long*>(tsm + (size_t)ns * sbytes);
  long long* sC = hold0 + (NT / 2) * kEW * 32;
  int* sE = reinterpret_cast<int*>(sC + kRB * kRows);
  unsigned* sK = reinterpret_cast<unsigned*>(sE + kRB * kRows);   // largest key of each line
  unsigned long long* bars = reinterpret_cast<unsigned long long*>(sK + kRB * kRows);
  uint32_t* sT = reinterpret_cast<uint32_t*>(bars + kBars);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t barFull = su32(bars), barB = barFull + 8 * kMaxStages;
  const uint32_t barEmpty = barFull + 16 * kMaxStages, barAccFull = barFull + 24 * kMaxStages;
  const uint32_t barAccFree = barAccFull + 8, barRow = barAccFull + 16;
  const uint32_t barRowFree = barRow + 8 * kRB, barFin = barRowFree + 8 * kRB, barKey = barFin + 8;
  for (int i = tid; i < kRB * kRows; i += kThreads) sK[i] = 0;
  if (tid == 0) {
    for (int b = 0; b < kMaxStages; ++b) {
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
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(barKey), "r"(kSW));
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  const bool issuer_warp = warp == kPW + kEW;
  if (issuer_warp) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     su32(sT)),
                 "r"(512));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  // largest keys of elements ja .. jz - 1 of lines 32 gi .. + 31 of a tile, lanes along the lines, U
  // loads in flight per lane
  const int nel = MODE == YB ? A.n1 : MODE == XB ? A.t.nk : A.P;
  constexpr int U = MODE == XF ? 24 : 12;
  auto keys = [&](int tile, int b, int gi, int ja, int jz) {
    const int fld = tile / A.tpf, l = gi * 32 + lane;
    const int line = (tile - fld * A.tpf) * LPT + l;
    const bool ok = line < A.nlines, d = (A.dmask >> fld) & 1;
    const double* src =
        A.in[fld] + (ok ? (line / A.ld) * A.ihs + (line % A.ld) * A.ils : 0) * ISC;
    unsigned key = 0;
#pragma unroll 1
    for (int j0 = ja; j0 < jz; j0 += U) {
      double2 v[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int j = j0 + u;
        v[u] = make_double2(0.0, 0.0);
        if (ok && j < jz && !(MODE == YB && j == A.n1 / 2)) {
          if (MODE == XF) v[u].x = src[(size_t)j * A.estr];
          else v[u] = *reinterpret_cast<const double2*>(src + 2 * (size_t)j * A.estr);
        }
      }
      if (MODE != XF && d) {
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int j = j0 + u;
          const double k = A.kscale * (double)((MODE == YB && j > A.n1 / 2) ? j - A.n1 : j);
          v[u] = make_double2(k * v[u].x, k * v[u].y);
        }
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        key = max(key, dkey(v[u].x));
        if (MODE != XF) key = max(key, dkey(v[u].y));
      }
    }
    if (key) atomicMax(&sK[b * kRows + l], key);
  };
  __syncthreads();   // sK cleared
  {
    // the first tile's keys by every warp: nothing else can begin before they are known (with
    // the same change in the Chebyshev kernel, a 64 x 36 x 145 transform and its inverse 206 -> 129 us)
    constexpr int G = LPT / 32, parts = kThreads / 32 / G;
    const int pt = warp / G;
    if (pt < parts) keys(blockIdx.x, 0, warp % G, nel * pt / parts, nel * (pt + 1) / parts);
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();   // barriers and tensor-memory address visible to every warp
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *sT;
  const uint32_t sBase = su32(stages);
  char* kcta = A.keep + (long long)(SPLIT ? blockIdx.y * gridDim.x + blockIdx.x : blockIdx.x) * A.keep_bytes;
  Waiter W;

  if (issuer_warp) {
    if (lane == 0) {
      uint32_t slot = 0, use = 0, pass = 0;
      bool any = false;
      for (int tile = blockIdx.x; tile < A.ntiles; tile += gridDim.x)
        for (int pp = pp0; pp < pp1; ++pp)
          for (int c = 0; c < A.t.kc; ++c, ++pass) {
            if (pass > 0 && !W.wait(barAccFree, (pass - 1) & 1)) goto drain;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const int s0 = c * A.t.gst, s1 = min(nst, s0 + A.t.gst);
            for (int st = s0; st < s1; ++st) {
              if (!W.wait(barFull + 8 * slot, use & 1) || !W.wait(barB + 8 * slot, use & 1))
                goto drain;
              asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
              const uint32_t sA = sBase + slot * (uint32_t)sbytes;
              issue_stage(tmem, sA, sA + (uint32_t)kABytes, NT, st == s0);
              any = true;
              mma_commit(barEmpty + 8 * slot);
              if ((int)++slot == ns) {
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
    // ---- scan: one scale per line (a complex line's parts share it); each warp takes a third of the
    // elements of every line
    const int sw = warp - (kPW + kEW + 1), st = sw * 32 + lane;
    int ti = 0;
    for (int tile = blockIdx.x; tile < A.ntiles; tile += gridDim.x, ++ti) {
      const int b = ti % kRB;
      if (ti >= kRB && !W.wait_warp(barRowFree + 8 * b, (ti / kRB - 1) & 1)) break;
      const int fld = tile / A.tpf;
      if (ti > 0)
#pragma unroll 1
        for (int gi = 0; gi < LPT / 32; ++gi) keys(tile, b, gi, nel * sw / kSW, nel * (sw + 1) / kSW);
      __syncwarp();
      if (lane == 0)
        asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(barKey) : "memory");
      if (!W.wait_warp(barKey, ti & 1)) break;
      for (int l = st; l < LPT; l += 32 * kSW) {
        const int line = (tile - fld * A.tpf) * LPT + l;
        const bool ok = line < A.nlines && !(A.P & 1);
        const double* mp = A.in[fld] + (ok ? (line / A.ld) * A.ihs + (line % A.ld) * A.ils +
                                                 (long long)(A.P / 2) * A.estr
                                           : 0) * ISC;
        const int sc = row_scale<double>(sK[b * kRows + l]);
        sK[b * kRows + l] = 0;   // for tile ti + kRB, whose scan waits for this one's readers
        if (CPX) {
          long long xr = 0, xi = 0;
          if (MODE == YF && ok) {
            const double2 x = *reinterpret_cast<const double2*>(mp);
            xr = fix<true>(x.x, sc);
            xi = fix<true>(x.y, sc);
          }
          const int ro = b * kRows + tile_row(l, 0);
          sE[ro] = sc;
          sE[ro + 8] = sc;
          sC[ro] = __mul64hi(xr, A.t.ymid * 4);   // X Y / 2^62
          sC[ro + 8] = __mul64hi(xi, A.t.ymid * 4);
        } else {
          const long long x = MODE == XF && ok ? fix<true>(*mp, sc) : 0;
          sE[b * kRows + l] = sc;
          sC[b * kRows + l] = __mul64hi(x, A.t.ymid * 4);
        }
      }
      __syncwarp();
      if (lane == 0)
        asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(barRow + 8 * b) : "memory");
    }
  } else if (warp >= kEW) {
    // ---- producers.  YB, YF: thread = (line l, g), K positions 4 g + e of a stage holding
    // k = 16 st + g + 4 e, both parts.  XB, XF: thread = (line l, hf), positions 8 hf + e holding
    // k = 16 st + hf + 2 e.
    const int p = tid - 32 * kEW, pw = warp - kEW;
    const int l = CPX ? pw * 8 + ((lane >> 1) & 7) : pw * 16 + (lane & 15);
    const int g = CPX ? (lane >> 4) * 2 + (lane & 1) : lane >> 4;
    constexpr int KS = CPX ? 4 : 2, NE = CPX ? 4 : 8;   // k step and values per stage
    const int row = CPX ? tile_row(l, 0) : l;
    const uint32_t oa = CPX ? (uint32_t)((g >> 1) * (int)kALbo + row * 16 + (g & 1) * 8)
                            : (uint32_t)(g * (int)kALbo + row * 16);
    const uint32_t bbytes = (uint32_t)b_stage_bytes(NT);
    const size_t bstride = (size_t)bbytes / 2;   // elements of a stage block
    const uint64_t pol = policy_evict_last();
    longlong2* kp = reinterpret_cast<longlong2*>(kcta) + p;
    uint32_t slot = 0, use = 0;
    int ti = 0;
    // the stage's digit planes of v (biased) and, by one thread, the copy of its matrix digits;
    // false after a wait ran out
    auto put = [&](const unsigned long long (&v)[8], const uint16_t* bsrc) {
      if (use > 0 && !W.wait_warp(barEmpty + 8 * slot, (use & 1) ^ 1)) return false;
      unsigned char* sA = stages + (size_t)slot * sbytes;
      if (p == 0) bulk_load(su32(sA) + (uint32_t)kABytes, bsrc, bbytes, barB + 8 * slot, pol);
#pragma unroll
      for (int i = 0; i < kAPlanes; ++i) {
        const int b = 7 - i, sh = b < 4 ? 0 : 32;
        uint32_t w[8], r[4];
#pragma unroll
        for (int e = 0; e < 8; ++e) w[e] = (uint32_t)(v[e] >> sh);
#pragma unroll
        for (int e = 0; e < 4; ++e) r[e] = digit_pair(w[2 * e], w[2 * e + 1], b & 3);
        if (CPX) {
          *reinterpret_cast<uint2*>(sA + i * kPlaneBytes + oa) = make_uint2(r[0], r[1]);
          *reinterpret_cast<uint2*>(sA + i * kPlaneBytes + oa + 128) = make_uint2(r[2], r[3]);
        } else {
          *reinterpret_cast<uint4*>(sA + i * kPlaneBytes + oa) = make_uint4(r[0], r[1], r[2], r[3]);
        }
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncwarp();
      if (lane == 0)
        asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(barFull + 8 * slot)
                     : "memory");
      if ((int)++slot == ns) {
        slot = 0;
        ++use;
      }
      return true;
    };
    auto keep_at = [&](int grp, int st) { return kp + (size_t)(grp * nst + st) * (4 * kPW * 32); };
    auto store_keep = [&](longlong2* d, const unsigned long long (&v)[8]) {
#pragma unroll
      for (int i = 0; i < 4; ++i)
        __stcg(d + i * kPW * 32, make_longlong2((long long)v[2 * i], (long long)v[2 * i + 1]));
    };
    for (int tile = blockIdx.x; tile < A.ntiles; tile += gridDim.x, ++ti) {
      const int fld = tile / A.tpf;
      const int line = (tile - fld * A.tpf) * LPT + l;
      const bool rowok = line < A.nlines, d = (A.dmask >> fld) & 1;
      const int lh = line / A.ld, ll = line - lh * A.ld;
      const double* src = A.in[fld] + (rowok ? lh * A.ihs + ll * A.ils : 0) * ISC;
      // complex inputs: x (k) and, folded, y (L - k); real ones: two samples per element
      double2 x[8];
      auto load = [&](int st) {
#pragma unroll
        for (int e = 0; e < NE; ++e) {
          const int k = 16 * st + g + KS * e;
          const bool ok = rowok && k < A.t.nk, okm = ok && k > 0;
          if (CPX) {
            const int L = MODE == YB ? A.n1 : A.P;
            x[e] = make_double2(0.0, 0.0);
            x[4 + e] = make_double2(0.0, 0.0);
            if (ok) x[e] = *reinterpret_cast<const double2*>(src + 2 * (size_t)k * A.estr);
            if (okm) x[4 + e] = *reinterpret_cast<const double2*>(src + 2 * (size_t)(L - k) * A.estr);
          } else if (MODE == XB) {
            x[e] = make_double2(0.0, 0.0);
            if (ok) x[e] = *reinterpret_cast<const double2*>(src + 2 * (size_t)k * A.estr);
          } else {
            x[e] = make_double2(0.0, 0.0);
            if (ok) x[e].x = src[(size_t)k * A.estr];
            if (okm) x[e].y = src[(size_t)(A.P - k) * A.estr];
          }
        }
      };
      load(0);
      const int rbuf = ti % kRB;
      if (!W.wait_warp(barRow + 8 * rbuf, (ti / kRB) & 1)) break;
      const int sc = sE[rbuf * kRows + row];
      __syncwarp();
      if (lane == 0)
        asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(barRowFree + 8 * rbuf)
                     : "memory");
      const bool tiny = __any_sync(0xffffffffu, sc < kTinyScale) != 0;
      WordSums sumr, sumi;
      unsigned long long s0 = 0;
      bool ok = true;
      for (int st = 0; st < nst && ok; ++st) {
        if ((MODE == YB || MODE == XB) && d) {   // i k times the mode
#pragma unroll
          for (int e = 0; e < NE; ++e) {
            const double k = A.kscale * (double)(16 * st + g + KS * e);
            x[e] = make_double2(-k * x[e].y, k * x[e].x);
            if (CPX) x[4 + e] = make_double2(k * x[4 + e].y, -k * x[4 + e].x);
          }
        }
        unsigned long long s[8], dd[8];
        auto convert = [&](auto tag) {
          constexpr bool TINY = decltype(tag)::value;
#pragma unroll
          for (int e = 0; e < NE; ++e) {
            if (CPX) {
              const long long a = fix<TINY>(x[e].x, sc), b = fix<TINY>(x[4 + e].x, sc);
              const long long u = fix<TINY>(x[e].y, sc), v = fix<TINY>(x[4 + e].y, sc);
              s[e] = a + b + kABias;
              dd[e] = a - b + kABias;
              s[4 + e] = u + v + kABias;
              dd[4 + e] = u - v + kABias;
            } else {
              const long long a = fix<TINY>(x[e].x, sc), b = fix<TINY>(x[e].y, sc);
              s[e] = MODE == XB ? a + kABias : a + b + kABias;
              dd[e] = MODE == XB ? b + kABias : a - b + kABias;
            }
          }
        };
        if (tiny) convert(std::true_type());
        else convert(std::false_type());
        if (st + 1 < nst) load(st + 1);
        store_keep(keep_at(1, st), dd);
        if (SPLIT ? (int)gridDim.y < A.t.nsl : A.t.nsl > 1) store_keep(keep_at(0, st), s);   // more than one slice
        if (MODE == YB || MODE == XB) {
#pragma unroll
          for (int e = 0; e < NE; ++e) {
            sumr.add(s[e]);
            if (CPX) sumi.add(s[4 + e]);
          }
          if (st == 0) s0 = s[0];
        }
        ok = put(s, A.t.dig + ((size_t)pp0 * nst + st) * bstride);
      }
      if (!ok) break;
      if ((MODE == YB || MODE == XB) && !(A.P & 1) && (!SPLIT || blockIdx.y == 0)) {
        // output n = P / 2: sum_k (-1)^k s_k (YB, and XB of unit weights), 2 sum_k (-1)^k Re c_k -
        // Re c_0 (XB);
        // (-1)^k = (-1)^g.  High and low words are added apart.
        const int f = MODE == XB && !A.t.unit ? 2 : 1;
        const int sf = g & 1 ? -f : f, cnt = NE * nst;
        long long hr = sf * sumr.high(cnt), lr = sf * sumr.low(cnt);
        long long hm = CPX ? sf * sumi.high(cnt) : 0, lm = CPX ? sf * sumi.low(cnt) : 0;
        if (f == 2 && g == 0) {
          const long long z = (long long)(s0 - kABias);
          hr -= z >> 32;
          lr -= (long long)(unsigned)z;
        }
#pragma unroll
        for (int off = CPX ? 1 : 16; off <= 16; off <<= 4) {   // the threads of the line
          hr += __shfl_xor_sync(0xffffffffu, hr, off);
          lr += __shfl_xor_sync(0xffffffffu, lr, off);
          if (CPX) {
            hm += __shfl_xor_sync(0xffffffffu, hm, off);
            lm += __shfl_xor_sync(0xffffffffu, lm, off);
          }
        }
        if (g == 0 && rowok) {
          const int e2 = sc - FBits<double>::EOFF - 62;
          const double vr = sc == kNanRow ? qnan<double>()
                                          : words_scaled<double>(hr, lr, e2);
          double* o = A.out[fld] + (lh * A.ohs + ll * A.ols + (long long)(A.P / 2) * A.ostr) * OSC;
          if (CPX) {
            const double vi = sc == kNanRow ? qnan<double>()
                                            : words_scaled<double>(hm, lm, e2);
            *reinterpret_cast<double2*>(o) = make_double2(vr, vi);
          } else {
            *o = vr;
          }
        }
      }
      for (int pp = pp0 + 1; pp < pp1 && ok; ++pp) {
        longlong2 nx[4];
        auto fetch = [&](int st) {
          const longlong2* s = keep_at(pp & 1, st);
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
          ok = put(v, A.t.dig + ((size_t)pp * nst + st) * bstride);
        }
      }
      if (!ok) break;
    }
    // the copies still in flight finish (bounded) before the CTA ends: all were consumed unless a
    // wait ran out, in this warp or in the issuer
    if (p == 0) {
      const uint64_t dl = gtime() + kWaitNs;
      for (int b = 0; b < ns; ++b) {
        const uint32_t n = use + (b < (int)slot ? 1u : 0u);   // copies issued to slot b
        if (n > 0 && !mbar_wait_until(barB + 8 * b, (n - 1) & 1, dl)) W.ok = false;
      }
    }
  } else {
    // ---- epilogue: warp w reads tensor-memory lanes 32 (w % 4) .. + 31 (its rows), columns
    // (w / 4) NT / 2 .. + NT / 2 - 1 of each of the eight accumulators
    const int qd = warp & 3, cg = warp >> 2, CW = NT / 2;
    const int row = qd * 32 + lane;
    const int l = CPX ? (row >> 4) * 8 + (row & 7) : row, part_c = CPX ? (row >> 3) & 1 : 0;
    const uint32_t tb = tmem + ((uint32_t)(qd * 32) << 16) + (uint32_t)(cg * CW);
    // sums over several K groups are kept here between the groups
    long long* part = reinterpret_cast<long long*>(kcta + (size_t)2 * nst * kKeepStage) + tid;
    uint32_t pass = 0;
    int ti = 0;
    for (int tile = blockIdx.x; tile < A.ntiles; tile += gridDim.x, ++ti) {
      const int fld = tile / A.tpf, rbuf = ti % kRB;
      const int line = (tile - fld * A.tpf) * LPT + l;
      if (!W.wait_warp(barRow + 8 * rbuf, (ti / kRB) & 1)) break;
      const int me = sE[rbuf * kRows + row];
      const long long mid = sC[rbuf * kRows + row];
      __syncwarp();
      if (lane == 0)
        asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(barRowFree + 8 * rbuf)
                     : "memory");
      const bool rowok = line < A.nlines, nan = me == kNanRow;
      const int ex = me - FBits<double>::EOFF - A.t.q + (MODE == XF ? A.lift : 0);   // T 2^(E - q)
      const bool safe =
          __all_sync(0xffffffffu, !rowok || (!nan && safe_exp<double>(ex))) != 0;
      const int lh = line / A.ld, ll = line - lh * A.ld;
      double* dst = A.out[fld] + (rowok ? lh * A.ohs + ll * A.ols : 0) * OSC + part_c;
      bool ok = true;
      for (int pp = pp0; pp < pp1 && ok; ++pp) {
        const int m0 = (pp >> 1) * NT + cg * CW;
        for (int c = 0; c < A.t.kc; ++c, ++pass) {
          if (!(ok = W.wait_warp(barAccFull, pass & 1))) break;
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          if (A.t.nmag == 8)
            epilogue_pass<MODE, 8>(A, tb, CW, m0, pp & 1, c, rowok, nan, safe, ex, mid, part_c, part,
                                   hold0 + tid, dst, barAccFree, lane);
          else
            epilogue_pass<MODE, 0>(A, tb, CW, m0, pp & 1, c, rowok, nan, safe, ex, mid, part_c, part,
                                   hold0 + tid, dst, barAccFree, lane);
        }
      }
      if (!ok) break;
    }
  }
  if (!W.ok) atomicOr(A.err, 1);
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (issuer_warp)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512));
}

// The nine products (in place: seven physical fields u v w phi phi_x phi_y phi_z in, Sxx - Szz,
// Syy - Szz, Sxy, Sxz, Syz, phi^3, u phi, v phi, w phi out) of n samples per field.  About 20
// float64 operations per sample: bound by the float64 pipe and by HBM about equally.
struct Phys9 {
  double* f[9];
};
__global__ void __launch_bounds__(256) products_kernel(const Phys9 p, long long n, double kappa) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x) {
    const double u = p.f[0][i], v = p.f[1][i], w = p.f[2][i], ph = p.f[3][i];
    const double fx = p.f[4][i], fy = p.f[5][i], fz = p.f[6][i];
    const double kx = kappa * fx, ky = kappa * fy, kz = kappa * fz;
    const double wz = fma(w, w, kz * fz);
    p.f[0][i] = fma(-u, u, fma(-kx, fx, wz));
    p.f[1][i] = fma(-v, v, fma(-ky, fy, wz));
    p.f[2][i] = -fma(u, v, kx * fy);
    p.f[3][i] = -fma(u, w, kx * fz);
    p.f[4][i] = -fma(v, w, ky * fz);
    p.f[5][i] = ph * ph * ph;
    p.f[6][i] = u * ph;
    p.f[7][i] = v * ph;
    p.f[8][i] = w * ph;
  }
}

// The assembly's z-independent combinations (launch_ycomb), in place on the nine products' modes:
//   P = kx ky (Sxx' - Syy') + (ky^2 - kx^2) Sxy, Q = i (kx Syz - ky Sxz), C = i (kx Sxz + ky Syz),
//   R = -(kx^2 Sxx' + 2 kx ky Sxy + ky^2 Syy'), F = -i (kx u phi + ky v phi), w phi, phi^3
// (on the kx = ky = 0 line P and Q hold Sxz and Syz).  One thread per mode and z.
__global__ void __launch_bounds__(256) combine_kernel(double2* __restrict__ f, long long fs, int Ny,
                                                      int Nz, double kxs, double kys) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i >= fs) return;
  const long long line = i / Nz;
  const int mx = (int)(line / Ny), j = (int)(line - (long long)mx * Ny);
  const double kx = kxs * mx, ky = kys * (j < Ny / 2 ? j : j - Ny);
  const double2 xx = f[i], yy = f[fs + i], xy = f[2 * fs + i], xz = f[3 * fs + i];
  const double2 yz = f[4 * fs + i], p3 = f[5 * fs + i], uf = f[6 * fs + i], vf = f[7 * fs + i];
  const double2 wf = f[8 * fs + i];
  const double a = kx * ky, b = fma(ky, ky, -kx * kx), c = kx * kx, d = ky * ky, a2 = 2.0 * a;
  if (line == 0) {
    f[i] = xz;
    f[fs + i] = yz;
  } else {
    f[i] = make_double2(fma(b, xy.x, a * (xx.x - yy.x)), fma(b, xy.y, a * (xx.y - yy.y)));
    f[fs + i] = mul_i(make_double2(fma(kx, yz.x, -ky * xz.x), fma(kx, yz.y, -ky * xz.y)));
  }
  f[2 * fs + i] = mul_i(make_double2(fma(kx, xz.x, ky * yz.x), fma(kx, xz.y, ky * yz.y)));
  f[3 * fs + i] = make_double2(-fma(c, xx.x, fma(a2, xy.x, d * yy.x)),
                               -fma(c, xx.y, fma(a2, xy.y, d * yy.y)));
  f[4 * fs + i] = mul_mi(make_double2(fma(kx, uf.x, ky * vf.x), fma(kx, uf.y, ky * vf.y)));
  f[5 * fs + i] = wf;
  f[6 * fs + i] = p3;
}

// Transposed Jacobian of the nine products, point by point: the fields u v w phi phi_x phi_y phi_z
// (p, in) and the product adjoints b (nine fields of n samples) give the fields' adjoints (p, out).
// 33 float64 operations per sample (0.34 ms at 192 x 192 x 129 samples) bound it.
__global__ void __launch_bounds__(256) adj_products_kernel(const Phys9 p,
                                                           const double* __restrict__ b, long long n,
                                                           double kappa) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x) {
    const double u = p.f[0][i], v = p.f[1][i], w = p.f[2][i], ph = p.f[3][i];
    const double fx = p.f[4][i], fy = p.f[5][i], fz = p.f[6][i];
    const double b0 = -2.0 * b[i], b1 = -2.0 * b[n + i], bz = -(b0 + b1);
    const double b2 = b[2 * n + i], b3 = b[3 * n + i], b4 = b[4 * n + i], b5 = b[5 * n + i];
    const double b6 = b[6 * n + i], b7 = b[7 * n + i], b8 = b[8 * n + i];
    p.f[0][i] = fma(u, b0, fma(-v, b2, fma(-w, b3, ph * b6)));
    p.f[1][i] = fma(v, b1, fma(-u, b2, fma(-w, b4, ph * b7)));
    p.f[2][i] = fma(w, bz, fma(-u, b3, fma(-v, b4, ph * b8)));
    p.f[3][i] = fma(3.0 * ph * ph, b5, fma(u, b6, fma(v, b7, w * b8)));
    p.f[4][i] = kappa * fma(fx, b0, fma(-fy, b2, -fz * b3));
    p.f[5][i] = kappa * fma(fy, b1, fma(-fx, b2, -fz * b4));
    p.f[6][i] = kappa * fma(fz, bz, fma(-fx, b3, -fy * b4));
  }
}

// phi += -i kx phi_x on modes (Mx, Q)
__global__ void __launch_bounds__(256) fold_dx_kernel(double2* __restrict__ phi,
                                                      const double2* __restrict__ phix, long long fs,
                                                      int Q, double kxs) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i >= fs) return;
  const double k = kxs * (double)(i / Q);
  const double2 a = phi[i], b = phix[i];
  phi[i] = make_double2(fma(k, b.y, a.x), fma(-k, b.x, a.y));
}

uint16_t bf16_bits(float f) {
  uint32_t u;
  memcpy(&u, &f, sizeof u);
  return (uint16_t)(u >> 16);   // exact: a digit has at most eight significant bits
}

size_t plan_smem(int NT, int ns) {
  return (size_t)ns * stage_bytes(NT) + (size_t)(NT / 2) * kEW * 32 * sizeof(long long) + kTail;
}

template <int MODE> cudaError_t launch_mode(Args& a, int nf, const Txy& x, cudaStream_t s) {
  constexpr int LPT = MODE == YB || MODE == YF ? kRows / 2 : kRows;
  static SmemLimit cur[2];
  cudaError_t e = ensure_smem(txy_kernel<MODE, false>, a.t.smem, &cur[0]);
  if (e == cudaSuccess) e = ensure_smem(txy_kernel<MODE, true>, a.t.smem, &cur[1]);
  if (e != cudaSuccess) return e;
  a.tpf = (a.nlines + LPT - 1) / LPT;
  a.ntiles = a.tpf * nf;
  a.keep = x.keep;
  a.keep_bytes = (long long)x.keep_bytes;
  a.err = x.err;
  if (a.ntiles <= 0) return cudaSuccess;
  // Rule: as many CTAs to a tile as all tiles find an SM each, up to one per output slice (its cosine and
  // sine products meet in shared memory); each converts the tile's rows again.  One CTA a tile / this, us:
  // y backward 16 x 648 x 65 (54 tiles, two CTAs each) 607 / 360, 8 x 648 x 17 (12 tiles, eight) 598 / 163;
  // x backward, products and x forward of 512 x 24 x 9 (21 and 27 tiles) 690 / 263.
  const int parts = std::max(1, std::min(std::min(a.t.nsl, kMaxSlices), x.ctas / a.ntiles));
  if (parts == 1) {
    txy_kernel<MODE, false><<<std::min(a.ntiles, x.ctas), kThreads, a.t.smem, s>>>(a);
  } else {
    for (int i = 0; i <= parts; ++i) a.cut[i] = (short)(i * a.t.nsl / parts);
    txy_kernel<MODE, true><<<dim3(a.ntiles, parts), kThreads, a.t.smem, s>>>(a);
  }
  return cudaGetLastError();
}

}  // namespace

size_t txy_keep_bytes(const TxyPlan& t) {
  return 2 * (size_t)t.nst * kKeepStage + (size_t)(kNTMax / 2) * kEW * 32 * sizeof(long long);
}

int txy_plan(int mode, int n1, int P, double scale, std::vector<uint16_t>& dig, TxyPlan* t) {
  const int half = (P + 1) / 2;   // samples n and P - n share a column: n < half (and P / 2)
  t->nk = mode == YB ? n1 / 2 : mode == XB ? n1 : half;
  t->nout = mode == YF ? n1 / 2 : mode == XF ? n1 : half;
  t->nsl = (t->nout + kNTMax - 1) / kNTMax;
  t->NT = ((t->nout + t->nsl - 1) / t->nsl + 15) / 16 * 16;
  t->nst = (t->nk + kKS - 1) / kKS;
  t->kc = (t->nst * kKS + kMaxK - 1) / kMaxK;
  t->gst = (t->nst + t->kc - 1) / t->kc;
  t->stages = kMaxStages;
  while (t->stages > 2 && plan_smem(t->NT, t->stages) > 226 * 1024) --t->stages;
  t->smem = plan_smem(t->NT, t->stages);
  t->unit = mode == XB && scale == 1.0;
  std::vector<long double> cs, sn;
  circle(P, cs, sn);
  // Matrix scale 2^q: the largest weight at most 2^54 and every recombined integer below 2^63.  Those are
  // 2^-62 of the sums of X_k Y_nk, |X_k| < 0.976 2^62 (twice that for the sums and differences s, d): over
  // an output's row of cosines and its row of sines, added (YB, YF, XB) or apart (XF), and the middle sample's
  // term.  Taken from the rows themselves the sums are 0.64 of the weights' count (with every weight counted
  // as the largest there were one or two bits fewer, and a backward transform of a steep spectrum of 648 or 1024
  // points was off by 6.7e-16 and 7.1e-16 where the FFT is by 3.0e-16 and 3.8e-16; now 2.0e-16 and 3.7e-16).
  const double wmax = mode == XB || mode == YF ? fabs(scale) : 1.0;
  // (one table look-up and one addition a weight, two chains: a grid's plans need up to a million)
  std::vector<double> mag[2] = {std::vector<double>(P), std::vector<double>(P)};
  for (int a = 0; a < P; ++a) {
    const double c = fabs((double)cs[a]), d = fabs((double)sn[a]);
    mag[0][a] = mode == XF ? c : c + d;
    mag[1][a] = d;
  }
  double top = 0.0;
  for (int m = 0; m < (mode == XF ? 2 : 1); ++m) {
    const double* w = mag[m].data();
    for (int n = 0; n < t->nout; ++n) {
      const int n2 = 2 * n >= P ? 2 * n - P : 2 * n;
      double s0 = 0.0, s1 = 0.0;
      int a0 = 0, a1 = n;   // n k mod P for even and odd k
      int k = 0;
      for (; k + 1 < t->nk; k += 2) {
        s0 += w[a0];
        s1 += w[a1];
        a0 += n2;
        a1 += n2;
        a0 -= a0 >= P ? P : 0;
        a1 -= a1 >= P ? P : 0;
      }
      if (k < t->nk) s0 += w[a0];
      top = std::max(top, s0 + s1);
    }
  }
  top = 0.976 * wmax * ((mode == XB ? 1.0 : 2.0) * top + (mode == YF || mode == XF ? 1.0 : 0.0));
  t->q = (int)floor(std::min(54.0 - log2(wmax), 62.99 - log2(top)));
  t->ymid = mode == YF ? (long long)llround(ldexp(scale, t->q)) : mode == XF ? 1ll << t->q : 0;
  // the weights times 2^q by angle 2 pi a / P, of cosine and sine, and at k = 0 (cosine 1, sine 0)
  std::vector<long long> Y[2] = {std::vector<long long>(P), std::vector<long long>(P)};
  const long double w = mode == YF || mode == XB ? (long double)scale : 1.0L;
  const long double ws = mode == XB || mode == XF ? -w : w;
  for (int a = 0; a < P; ++a) {
    Y[0][a] = (long long)llroundl(ldexpl(w * cs[a], t->q));
    Y[1][a] = (long long)llroundl(ldexpl(ws * sn[a], t->q));
  }
  const long long Y0 = mode == XB ? 1ll << t->q : Y[0][0];
  // their digits as bf16, and the sum of the digits' magnitudes; entry P: k = 0
  struct Dig {
    uint16_t d[kPlanes];
    int sum;
  };
  std::vector<Dig> D[2] = {std::vector<Dig>(P + 1), std::vector<Dig>(P + 1)};
  for (int grp = 0; grp < 2; ++grp)
    for (int a = 0; a <= P; ++a) {
      const long long v = a < P ? Y[grp][a] : (grp == 0 ? Y0 : 0);
      const unsigned long long y = (unsigned long long)v + kBias;
      D[grp][a].sum = 0;
      for (int j = 0; j < kPlanes; ++j) {
        const int dgt = (int)((y >> (8 * (6 - j))) & 255ull) - 128;
        D[grp][a].d[j] = bf16_bits((float)dgt);
        D[grp][a].sum += abs(dgt);
      }
    }
  const int NT = t->NT;
  const size_t block = (size_t)kPlanes * NT * kKS;
  dig.assign((size_t)2 * t->nsl * t->nst * block, 0);
  double bound = 0.0;
  for (int n = 0; n < t->nout; ++n)
    for (int grp = 0; grp < 2; ++grp) {
      double acc = 0.0;   // |G_d| <= 128 sum_j sum_k |b_jk|
      uint16_t* b0 = dig.data() + (size_t)(2 * (n / NT) + grp) * t->nst * block + (size_t)(n % NT) * 8;
      int a = 0;          // n k mod P
      for (int k = 0; k < t->nk; ++k, a = a + n >= P ? a + n - P : a + n) {
        const Dig& e = D[grp][k == 0 ? P : a];
        const int st = k / kKS, kk = k % kKS;
        // stage position of k: 4 g + e holds g + 4 e (complex lines), 8 hf + e holds hf + 2 e
        const int pos = mode == YB || mode == YF ? 4 * (kk & 3) + (kk >> 2) : 8 * (kk & 1) + (kk >> 1);
        uint16_t* b = b0 + st * block + (size_t)(pos >> 3) * kPlanes * NT * 8 + (pos & 7);
        for (int j = 0; j < kPlanes; ++j) b[(size_t)j * NT * 8] = e.d[j];
        acc += 128.0 * e.sum;
      }
      bound = std::max(bound, acc);
    }
  t->nmag = bound <= 4194304.0 ? 8 : 0;
  return 0;
}

// y pass of nf fields: dir 1 modes (Mx, Ny, Nz) -> samples (Mx, P, Nz), dir 0 the inverse
// (truncated, times the plan's scale); arguments as in launch_ypass
cudaError_t launch_txy_y(int dir, const GridDev& g, int P, const void* in, void* out, int nf,
                         long long fs_in, long long fs_out, const YMap& map, const Txy& x,
                         const TxyPlan& plan, cudaStream_t s) {
  Args a;
  memset(&a, 0, sizeof a);
  if (nf > kMaxFields) return cudaErrorInvalidValue;
  for (int f = 0; f < nf; ++f) {
    a.in[f] = (const double*)in + 2 * map.src[f] * fs_in;
    a.out[f] = (double*)out + 2 * f * fs_out;
  }
  a.dmask = dir == 1 ? map.dy_mask : 0;
  a.kscale = map.kys;
  a.nlines = g.Mx * g.nz;
  a.ld = g.nz;
  a.ihs = (long long)(dir == 1 ? g.ny : P) * g.nz;
  a.ohs = (long long)(dir == 1 ? P : g.ny) * g.nz;
  a.ils = a.ols = 1;
  a.estr = a.ostr = g.nz;
  a.n1 = g.ny;
  a.P = P;
  a.t = plan;
  return dir == 1 ? launch_mode<YB>(a, nf, x, s) : launch_mode<YF>(a, nf, x, s);
}

cudaError_t launch_txy_ycomb(const GridDev& g, const void* in, void* out9, long long fs_in,
                             long long fs_out, const Txy& x, cudaStream_t s) {
  YMap map;
  for (int f = 0; f < YMap::kMax; ++f) map.src[f] = f;
  map.dy_mask = 0;
  map.kys = 0.0;
  cudaError_t e = launch_txy_y(0, g, g.Py, in, out9, 9, fs_in, fs_out, map, x, x.yf, s);
  if (e != cudaSuccess) return e;
  combine_kernel<<<(unsigned)((fs_out + 255) / 256), 256, 0, s>>>(
      (double2*)out9, fs_out, g.ny, g.nz, 6.283185307179586476925 / g.lx,
      6.283185307179586476925 / g.ly);
  return cudaGetLastError();
}

// x line: six fields (Mx, Py, Nz) -> seven physical fields -> nine products -> nine fields
cudaError_t launch_txy_x(const GridDev& g, const void* in6, void* out9, long long fs, const Txy& x,
                         cudaStream_t s) {
  const int Q = g.Py * g.nz;
  const long long np = (long long)g.Px * Q;
  Args a;
  memset(&a, 0, sizeof a);
  const int src[7] = {0, 1, 2, 3, 3, 4, 5};   // u v w phi (phi -> i kx phi) phi_y phi_z
  for (int f = 0; f < 7; ++f) {
    a.in[f] = (const double*)in6 + 2 * src[f] * fs;
    a.out[f] = x.phys[f];
  }
  a.dmask = 1u << 4;
  a.kscale = 6.283185307179586476925 / g.lx;
  a.nlines = a.ld = Q;
  a.ils = a.ols = 1;
  a.estr = a.ostr = Q;
  a.P = g.Px;
  a.t = x.xb;
  cudaError_t e = launch_mode<XB>(a, 7, x, s);
  if (e != cudaSuccess) return e;
  Phys9 p;
  memcpy(p.f, x.phys, sizeof p.f);
  products_kernel<<<(unsigned)std::min<long long>((np + 255) / 256, (long long)x.ctas * 32), 256, 0, s>>>(
      p, np, g.kappa);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  for (int f = 0; f < 9; ++f) {
    a.in[f] = x.phys[f];
    a.out[f] = (double*)out9 + 2 * f * fs;
  }
  a.dmask = 0;
  a.t = x.xf;
  return launch_mode<XF>(a, 9, x, s);
}

// transposed x line (adjoint of launch_txy_x under the real inner product): the seven physical fields
// of in6 again, the nine product adjoints by the transpose of the truncated forward transform (a
// backward transform of unit weights), the transposed Jacobian point by point, and the transpose of
// the padded backward transform (a forward transform with the modes k >= 1 doubled); phi_x's adjoint
// folds into phi's.  At 128^3 the five launches take 1.3 ms in place of the 3.3 of the FFT kernel.
cudaError_t launch_txy_adj_x(const GridDev& g, const void* in6, void* pb9, void* out6, long long fs,
                             double* adj9, const Txy& x, const TxyPlan& xb1, cudaStream_t s) {
  const int Q = g.Py * g.nz;
  const long long np = (long long)g.Px * Q;
  const double kxs = 6.283185307179586476925 / g.lx;
  Args a;
  memset(&a, 0, sizeof a);
  const int src[7] = {0, 1, 2, 3, 3, 4, 5};
  for (int f = 0; f < 7; ++f) {
    a.in[f] = (const double*)in6 + 2 * src[f] * fs;
    a.out[f] = x.phys[f];
  }
  a.dmask = 1u << 4;
  a.kscale = kxs;
  a.nlines = a.ld = Q;
  a.ils = a.ols = 1;
  a.estr = a.ostr = Q;
  a.P = g.Px;
  a.t = x.xb;
  cudaError_t e = launch_mode<XB>(a, 7, x, s);
  if (e != cudaSuccess) return e;
  for (int f = 0; f < 9; ++f) {
    a.in[f] = (const double*)pb9 + 2 * f * fs;
    a.out[f] = adj9 + f * np;
  }
  a.dmask = 0;
  a.t = xb1;
  if ((e = launch_mode<XB>(a, 9, x, s)) != cudaSuccess) return e;
  Phys9 p;
  memcpy(p.f, x.phys, sizeof p.f);
  adj_products_kernel<<<(unsigned)std::min<long long>((np + 255) / 256, (long long)x.ctas * 32), 256, 0,
                        s>>>(p, adj9, np, g.kappa);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  for (int f = 0; f < 7; ++f) {
    a.in[f] = x.phys[f];
    a.out[f] = f == 4 ? (double*)pb9 : (double*)out6 + 2 * src[f] * fs;
  }
  a.lift = 1;
  a.t = x.xf;
  if ((e = launch_mode<XF>(a, 7, x, s)) != cudaSuccess) return e;
  fold_dx_kernel<<<(unsigned)((fs + 255) / 256), 256, 0, s>>>((double2*)out6 + 3 * fs,
                                                              (const double2*)pb9, fs, Q, kxs);
  return cudaGetLastError();
}

// x transforms between rows of physical samples (Nz, Ny, Nx) and modes (Mx, Ny, Nz) on the unpadded
// grid: dir 0 phys[f] -> spec field f, dir 1 the inverse (field map src, i kx times the input for
// the fields of dmask)
cudaError_t launch_txy_rows(int dir, const GridDev& g, double* const* phys, double2* spec,
                            long long fs, int nf, const int* src, unsigned dmask, const Txy& x,
                            cudaStream_t s) {
  Args a;
  memset(&a, 0, sizeof a);
  if (nf > kMaxFields) return cudaErrorInvalidValue;
  for (int f = 0; f < nf; ++f) {
    double* m = (double*)spec + 2 * (src ? src[f] : f) * fs;
    a.in[f] = dir == 0 ? phys[f] : m;
    a.out[f] = dir == 0 ? m : phys[f];
  }
  a.dmask = dir == 1 ? dmask : 0;
  a.kscale = 6.283185307179586476925 / g.lx;
  a.nlines = g.ny * g.nz;
  a.ld = g.nz;                                        // line = y Nz + z
  const long long rh = g.nx, rl = (long long)g.ny * g.nx, mh = g.nz, ml = 1;
  a.ihs = dir == 0 ? rh : mh;
  a.ils = dir == 0 ? rl : ml;
  a.ohs = dir == 0 ? mh : rh;
  a.ols = dir == 0 ? ml : rl;
  const long long ms = (long long)g.ny * g.nz;
  a.estr = dir == 0 ? 1 : ms;
  a.ostr = dir == 0 ? ms : 1;
  a.P = g.nx;
  a.t = dir == 0 ? x.xfu : x.xbu;
  return dir == 0 ? launch_mode<XF>(a, nf, x, s) : launch_mode<XB>(a, nf, x, s);
}

}  // namespace chf
