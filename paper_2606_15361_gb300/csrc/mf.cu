// DM-scaled boxcar matched filter (Methods, "Matched filtering").
//
// One CTA per DM row. The row segment [F_prev, E_new) of the plane ring (block start times
// [F_prev, F_new) plus the Wmax-1 samples their windows reach) is staged in shared memory as it lies
// in the ring (columns from the 16-byte boundary at or before F_prev); its exact integer sums give mu
// and sigma over the block's start times, and an in-place exclusive scan turns it into prefix
// sums, so every boxcar is P[t+W] - P[t]. Everything works on quads of four consecutive columns
// per lane (one 128-bit shared access).
//
// Decision: a cell is in the mask iff max over the row's widths of
//   SNR(W) = (S_W - mu*W) / (sigma*sqrt(W))          (FP64, this operation order)
// reaches Theta. SNR(S) is monotone in the integer S, so lane j of the last warp finds the
// smallest integer tau_W with SNR(tau_W) >= Theta of width 2^j by a bounded search around
// mu*W + Theta*sigma*sqrt(W); the per-cell test is then the exact integer compare
// S_W >= tau_W. Cells in the mask get their FP64 S/N maximum (ties -> smaller width; FP64 only
// for the widths that FP32 leaves) rounded to float and are appended to the block's cell list
// for peak selection.
// Mode A floors sigma at sigma_min; Mode C scores the integer root counts (S/N does not
// change under the 1/sqrt(N_f) scale).

#include <climits>
#include <cmath>
#include <vector>

#include "bulk.h"
#include "snd_internal.h"

namespace snd {
namespace {

struct MfArgs {
  const int32_t* plane;
  int Lp, ndm;
  long long f_prev, e_prev, e_new;
  int nb;  // start times in this block
  const uint16_t* width_mask;
  int binary;
  double theta, sigma_min;
  float out_scale;  // 1/sqrt(N_f) for the caller's float plane, else 0
  uint32_t* mask;
  int mw;
  MfCell* cells;
  int cell_cap;
  uint32_t* counters;
  void* plane_out;
  int nemit;
  int out_u8;       // caller's plane in uint8 (binary / graded roots are 0..255)
  int pf_rows;      // rows resident at once: row d prefetches row d + pf_rows into L2
  int tau_steps;    // bound of the threshold search, steps each way
  int nowrap;       // every prefix sum of the staged segment is below 2^31 (no wrap-around)
  int stat32;       // a lane's sums of y and y^2 over its groups fit in 32 bits
  long long wait_cycles;  // bound of the staging wait (clock cycles)
};

constexpr uint32_t kAllWidths = (1u << kNumWidthSlots) - 1u;

template <bool A, bool NW = false>
struct WidthSet {  // tag: every width slot of the row is in use (A) or not known to be; prefix
  static constexpr bool kAll = A;     // sums that never wrap (NW)
  static constexpr bool kNoWrap = NW;
};

__device__ __forceinline__ double snr_of(long long s, double mu_w, double den) {
  return __ddiv_rn(__dsub_rn(static_cast<double>(s), mu_w), den);
}

// S/N in FP32 of a window sum: c = (bits of floor(mu W), its fraction, 1 / (sigma sqrt W))
__device__ __forceinline__ float snr32(int s, const float3& c) {
  return (static_cast<float>(s - __float_as_int(c.x)) - c.y) * c.z;
}

// One DM row d of one plan's block (the body of k_mf and of the many-beam k_mf_multi), by NT threads.
//
// What bounds it: shared-memory wavefronts (the threshold reads a quad per width and four start times)
// and the latency of its phases one after the other, so the phases are few and touch shared memory
// little: the copy lands, the quads are read once for the sums and once for the scan, which writes
// them; the segment is never shifted to F_prev's column (the mask words are, at the end). Threads per
// CTA follow the row's length, so that an SM's shared memory is full of threads.
// Stage times before and after (us, with the event pair; before: a shifting pass, 256 threads, FP64 for
// every width of a cell): 2048 rows x 16384 binary 113 -> 104, graded 132 -> 106, float with the caller's
// plane 134 -> 113; 1537 x 10007 82 -> 63; 4096 x 7246 117 -> 95; 128 x 16384 59 -> 32.
template <int NT>
__device__ __forceinline__ void mf_row(const MfArgs& a, const int d) {
  extern __shared__ __align__(16) int32_t smem[];  // G quads: columns ca0 .. of the ring, then prefix sums
  constexpr int NW = NT / 32;
  __shared__ long long red1[NW], red2[NW];
  __shared__ uint32_t wsum[NW];
  __shared__ int tau[kNumWidthSlots];
  __shared__ double s_muw[kNumWidthSlots], s_den[kNumWidthSlots];
  __shared__ float3 s_f32[kNumWidthSlots];
  __shared__ int s_ok;
  __shared__ __align__(8) unsigned long long bar;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int len = static_cast<int>(a.e_new - a.f_prev);
  const int c0 = static_cast<int>(a.f_prev % a.Lp);
  const int r0 = c0 & 3;               // staged column j holds sample j - r0 of the segment
  const int G = ((len + r0) >> 2) + 1; // quads staged: up to the one whose first prefix may be P[len]
  const int nb = a.nb;
  int4* Y4 = reinterpret_cast<int4*>(smem);
  const int32_t* src = a.plane + static_cast<size_t>(d) * a.Lp;
  const int ca0 = c0 - r0;
  // 1. one thread copies the segment (one bulk copy, or two across the ring's wrap point) onto an
  //    mbarrier; every thread waits for it (bounded)
  const uint32_t bs = smem_u32(&bar);
  if (tid == 0) {
    bar_init(bs, 1);
    bar_init_fence();
  }
  __syncthreads();
  const int n1 = min(G, (a.Lp - ca0) >> 2);  // quads before the wrap point
  if (tid == 0) {
    bar_expect(bs, static_cast<uint32_t>(G) * 16u);
    bulk_g2s(smem_u32(Y4), src + ca0, static_cast<uint32_t>(n1) * 16u, bs);
    if (n1 < G) bulk_g2s(smem_u32(Y4 + n1), src, static_cast<uint32_t>(G - n1) * 16u, bs);
  }
  const bool landed = bar_wait(bs, 0, a.wait_cycles);
  if (!__syncthreads_and(landed)) {
    // the wait gave up: report it, let the copies land (normal bound) before the CTA leaves
    if (tid == 0) {
      atomicOr(&a.counters[kCntStatus], kStatusMfTimeout);
      bar_wait(bs, 0, kStageWaitCycles);
    }
    return;
  }
  // 2. one pass over the warp's quads (contiguous per warp), which are zero outside the segment: the
  //    caller's plane (the newly emitted samples [E_prev, E_new)), the exact sums over the block's start
  //    times and the warp's total for the scan
  const int seg = (((G + 31) >> 5) + NW - 1) / NW * 32;
  const int glo = min(G, wid * seg), ghi = min(G, glo + seg);
  auto quad = [&](int g) {
    int4 v = Y4[g];
    const int i = 4 * g - r0;  // sample of the quad's first column
    if (i < 0 || i + 3 >= len) {
      if (i < 0 || i >= len) v.x = 0;
      if (i + 1 < 0 || i + 1 >= len) v.y = 0;
      if (i + 2 < 0 || i + 2 >= len) v.z = 0;
      if (i + 3 >= len) v.w = 0;
    }
    return v;
  };
  if (a.plane_out) {
    // lanes along the row, one column each, so a store instruction covers 32 neighbouring values
    const int j0 = static_cast<int>(a.e_prev - a.f_prev) + r0;  // staged column of the first emitted sample
    const int32_t* y = smem + j0;
    const size_t o = static_cast<size_t>(d) * a.nemit;
    if (a.out_scale != 0.0f) {
      float* out = static_cast<float*>(a.plane_out) + o;
      for (int k = tid; k < a.nemit; k += NT) out[k] = static_cast<float>(y[k]) * a.out_scale;
    } else if (a.out_u8) {
      uint8_t* out = static_cast<uint8_t*>(a.plane_out) + o;
      for (int k = tid; k < a.nemit; k += NT) out[k] = static_cast<uint8_t>(y[k]);
    } else {
      int32_t* out = static_cast<int32_t*>(a.plane_out) + o;
      for (int k = tid; k < a.nemit; k += NT) out[k] = y[k];
    }
  }
  if (nb <= 0) return;
  {
    uint32_t tot = 0;
    long long s1 = 0, s2 = 0;
    // a lane sums y and y^2 in 32 bits where its quads cannot overflow them (a.stat32), else in
    // 64 bits; the warp reduction is in 64 bits either way
    auto pass = [&](auto zero) {
      using Acc = decltype(zero);
      Acc a1 = 0, a2 = 0;
#pragma unroll 2
      for (int g = glo + lane; g < ghi; g += 32) {
        const int4 v = quad(g);
        const int i = 4 * g - r0;
        const Acc x = static_cast<Acc>(v.x), y = static_cast<Acc>(v.y), z = static_cast<Acc>(v.z), w = static_cast<Acc>(v.w);
        const uint32_t gs = static_cast<uint32_t>(v.x) + static_cast<uint32_t>(v.y) + static_cast<uint32_t>(v.z) +
                            static_cast<uint32_t>(v.w);
        tot += gs;
        if (i + 3 < nb) {  // columns before the segment are zero
          a1 += static_cast<Acc>(gs);
          a2 += (x * x + y * y) + (z * z + w * w);
        } else {
          if (i < nb) { a1 += x; a2 += x * x; }
          if (i + 1 < nb) { a1 += y; a2 += y * y; }
          if (i + 2 < nb) { a1 += z; a2 += z * z; }
        }
      }
      s1 = static_cast<long long>(a1);
      s2 = static_cast<long long>(a2);
    };
    if (a.stat32) pass(0u); else pass(0ll);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      tot += __shfl_xor_sync(0xFFFFFFFFu, tot, o);
      s1 += __shfl_down_sync(0xFFFFFFFFu, s1, o);
      s2 += __shfl_down_sync(0xFFFFFFFFu, s2, o);
    }
    if (lane == 0) {
      wsum[wid] = tot;
      red1[wid] = s1;
      red2[wid] = s2;
    }
  }
  __syncthreads();
  const uint32_t wm = a.width_mask[d];
  if (wid == NW - 1) {
    // row statistics (FP64, fixed order) and, lane j, the integer threshold of width 2^j
    long long t1 = 0, t2 = 0;
    for (int w = 0; w < NW; ++w) {
      t1 += red1[w];
      t2 += red2[w];
    }
    const double n = static_cast<double>(nb);
    const double mu = __ddiv_rn(static_cast<double>(t1), n);
    const double var = __dsub_rn(__ddiv_rn(static_cast<double>(t2), n), __dmul_rn(mu, mu));
    double sig = var > 0.0 ? __dsqrt_rn(var) : 0.0;
    if (a.binary && sig < a.sigma_min) sig = a.sigma_min;
    if (lane == 0) s_ok = sig > 0.0;
    if (sig > 0.0 && lane < kNumWidthSlots && ((wm >> lane) & 1)) {
      const double w = static_cast<double>(1 << lane);
      const double mu_w = __dmul_rn(mu, w);
      const double den = __dmul_rn(sig, __dsqrt_rn(w));
      s_muw[lane] = mu_w;
      s_den[lane] = den;
      const double whole = floor(mu_w);
      s_f32[lane] = make_float3(__int_as_float(static_cast<int>(whole)), static_cast<float>(mu_w - whole),
                                static_cast<float>(1.0 / den));
      double est = ceil(__dadd_rn(mu_w, __dmul_rn(a.theta, den)));
      if (est < 0.0) est = 0.0;
      if (est > 2147483000.0) est = 2147483000.0;
      long long sv = static_cast<long long>(est);
      int down = 0, up = 0;
      while (sv > 0 && down < a.tau_steps && snr_of(sv - 1, mu_w, den) >= a.theta) {
        --sv;
        ++down;
      }
      while (up < a.tau_steps && snr_of(sv, mu_w, den) < a.theta) {
        ++sv;
        ++up;
      }
      if (down == a.tau_steps || up == a.tau_steps) atomicOr(&a.counters[kCntStatus], kStatusTauTimeout);
      tau[lane] = static_cast<int>(sv);
    }
  }
  // 3. exclusive scan in place (uint32 wrap-around keeps window sums exact): a lane scans its quad, the
  //    warp scans the quads' sums, the running carry starts at the sum of the warps before
  {
    uint32_t carry = 0;
    for (int w = 0; w < wid; ++w) carry += wsum[w];
    for (int base = glo; base < ghi; base += 32) {
      const int g = base + lane;
      const int4 v = g < ghi ? quad(g) : make_int4(0, 0, 0, 0);
      const uint32_t a0 = static_cast<uint32_t>(v.x);
      const uint32_t a1 = a0 + static_cast<uint32_t>(v.y);
      const uint32_t a2 = a1 + static_cast<uint32_t>(v.z);
      const uint32_t a3 = a2 + static_cast<uint32_t>(v.w);
      uint32_t incl = a3;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t u = __shfl_up_sync(0xFFFFFFFFu, incl, o);
        if (lane >= o) incl += u;
      }
      const uint32_t ex = carry + incl - a3;
      if (g < ghi)
        Y4[g] = make_int4(static_cast<int32_t>(ex), static_cast<int32_t>(ex + a0), static_cast<int32_t>(ex + a1),
                          static_cast<int32_t>(ex + a2));
      carry += __shfl_sync(0xFFFFFFFFu, incl, 31);
    }
  }
  __syncthreads();
  // the row a CTA of the next wave will stage: its segment into L2 (bulk prefetches, one or two
  // across the wrap point) while this row is scored
  if (tid == 0 && d + a.pf_rows < a.ndm) {
    const int32_t* nsrc = a.plane + static_cast<size_t>(d + a.pf_rows) * a.Lp;
    bulk_prefetch_l2(nsrc + ca0, static_cast<uint32_t>(n1) * 16u);
    if (n1 < G) bulk_prefetch_l2(nsrc, static_cast<uint32_t>(G - n1) * 16u);
  }
  const int nbw = (nb + 31) >> 5;
  uint32_t* mrow = a.mask + static_cast<size_t>(d) * a.mw;
  if (!s_ok) {
    for (int q = tid; q < nbw; q += NT) mrow[q] = 0;
    return;
  }
  int tw[kNumWidthSlots];
#pragma unroll
  for (int j = 0; j < kNumWidthSlots; ++j) tw[j] = ((wm >> j) & 1) ? tau[j] : 0x7FFFFFFF;
  const uint32_t* P = reinterpret_cast<const uint32_t*>(smem) + r0;  // P[t]: the sum before sample t
  const uint4* P4 = reinterpret_cast<const uint4*>(smem);
  // 4. threshold: lane m of an iteration tests the start times of quad m against every width of the
  //    row (window ends P[4m + W ...] are quad m + W/4 for W >= 4, quads m and m+1 below).
  //    A cell passes iff max over widths of S_W - tau_W >= 0; S_W < 2^31 and tau_W < 2^31, so
  //    the wrapped difference P[t+W] - P[t] - tau_W read as int32 is exact.
  // hit nibble of quad m (bit e: its column e passes)
  // Without wrap-around (prefix sums below 2^31, the usual case) the test is rearranged as
  // max over W of (P[t+W] - tau_W) >= P[t]: one add-and-max per (start time, width), which
  // the compiler can issue as a single three-input integer instruction.
  auto quad_hits = [&](int m, auto all) -> uint32_t {
    constexpr bool ALL = decltype(all)::kAll;
    constexpr bool NOWRAP = decltype(all)::kNoWrap;
    const uint4 p = P4[m], q = P4[m + 1];
    int h0 = INT_MIN, h1 = INT_MIN, h2 = INT_MIN, h3 = INT_MIN;
    auto upd = [](int& h, uint32_t end, uint32_t start, int tj) {
      if constexpr (NOWRAP) {
        h = max(static_cast<int>(end) + (-tj), h);
      } else {
        h = max(h, static_cast<int>(end - start - static_cast<uint32_t>(tj)));
      }
    };
    if (ALL || (wm & 1u)) {
      upd(h0, p.y, p.x, tw[0]);
      upd(h1, p.z, p.y, tw[0]);
      upd(h2, p.w, p.z, tw[0]);
      upd(h3, q.x, p.w, tw[0]);
    }
    if (ALL || (wm & 2u)) {
      upd(h0, p.z, p.x, tw[1]);
      upd(h1, p.w, p.y, tw[1]);
      upd(h2, q.x, p.z, tw[1]);
      upd(h3, q.y, p.w, tw[1]);
    }
    if (ALL || (wm & 4u)) {
      upd(h0, q.x, p.x, tw[2]);
      upd(h1, q.y, p.y, tw[2]);
      upd(h2, q.z, p.z, tw[2]);
      upd(h3, q.w, p.w, tw[2]);
    }
#pragma unroll
    for (int j = 3; j < kNumWidthSlots; ++j)
      if (ALL || ((wm >> j) & 1u)) {
        const uint4 e = P4[m + (1 << (j - 2))];
        upd(h0, e.x, p.x, tw[j]);
        upd(h1, e.y, p.y, tw[j]);
        upd(h2, e.z, p.z, tw[j]);
        upd(h3, e.w, p.w, tw[j]);
      }
    if constexpr (NOWRAP)
      return (h0 >= static_cast<int>(p.x) ? 1u : 0u) | (h1 >= static_cast<int>(p.y) ? 2u : 0u) |
             (h2 >= static_cast<int>(p.z) ? 4u : 0u) | (h3 >= static_cast<int>(p.w) ? 8u : 0u);
    return (h0 >= 0 ? 1u : 0u) | (h1 >= 0 ? 2u : 0u) | (h2 >= 0 ? 4u : 0u) | (h3 >= 0 ? 8u : 0u);
  };
  // The warps take iterations in turn (a burst's cells, which cost an evaluation each, spread over
  // them). An iteration makes four column words (word k = columns 32 k ..), kept in the mask row until
  // all are there; the mask word of start times 32 q .. is column words q and q + 1 shifted by r0.
  const int tit = (nb + r0 + 127) >> 7;  // iterations over the columns of start times
  for (int it = wid; it < tit; it += NW) {
    const int m = it * 32 + lane;
    const int i = 4 * m - r0;  // start time of the quad's first column
    uint32_t nib = 0;
    if (i + 3 >= 0 && i < nb) {
      // rows with every width (most rows above a small DM) take a copy of the loop with no
      // width tests, so all window loads of the quad can be in flight together
      if (a.nowrap)
        nib = (wm == kAllWidths) ? quad_hits(m, WidthSet<true, true>{}) : quad_hits(m, WidthSet<false, true>{});
      else
        nib = (wm == kAllWidths) ? quad_hits(m, WidthSet<true>{}) : quad_hits(m, WidthSet<false>{});
      if (nb - i < 4) nib &= (1u << (nb - i)) - 1u;  // start times inside the block
      if (i < 0) nib &= ~((1u << -i) - 1u);
    }
    uint32_t word = nib << (4 * (lane & 7));
    word |= __shfl_xor_sync(0xFFFFFFFFu, word, 1);
    word |= __shfl_xor_sync(0xFFFFFFFFu, word, 2);
    word |= __shfl_xor_sync(0xFFFFFFFFu, word, 4);
    const int k = 4 * it + (lane >> 3);
    if ((lane & 7) == 0 && k <= nbw) mrow[k] = word;  // a mask row has a word past its last (96 spare columns)
    while (nib) {
      const int e = __ffs(nib) - 1;
      nib &= nib - 1u;
      const int t = i + e;
      const uint32_t p0 = P[t];
      // The cell's S/N is the FP64 maximum over the widths. FP64 divides are slow here, so FP32 finds
      // the widths that can hold it, those within 1e-4 of its own largest. That leaves no maximum out,
      // whatever Theta is: FP32 gets x = S - mu W, an exact integer less a fraction, to 2^-25 and a
      // relative 2^-22, which is below 4e-5 of an x from 2^-10 on. Where the largest S/N has a smaller x
      // (at least 1 / nb, as mu is a multiple of that), x at any other width with a positive S/N is the
      // same times the widths' ratio, and its S/N at least sqrt 2 below.
      float best32 = -3.0e38f;
#pragma unroll
      for (int j = 0; j < kNumWidthSlots; ++j)
        if ((wm >> j) & 1) best32 = fmaxf(best32, snr32(static_cast<int>(P[t + (1 << j)] - p0), s_f32[j]));
      const float floor32 = best32 - 1e-4f * fabsf(best32);
      double best = -1.0e300;
      int bw = 0;
#pragma unroll 1
      for (int j = 0; j < kNumWidthSlots; ++j) {
        if (!((wm >> j) & 1)) continue;
        const int S = static_cast<int>(P[t + (1 << j)] - p0);
        if (!(snr32(S, s_f32[j]) >= floor32)) continue;
        const double sv = snr_of(S, s_muw[j], s_den[j]);
        if (sv > best) {
          best = sv;
          bw = 1 << j;
        }
      }
      const uint32_t idx = atomicAdd(&a.counters[kCntCells], 1u);
      if (idx < static_cast<uint32_t>(a.cell_cap)) {
        MfCell c;
        c.cell = static_cast<uint32_t>(d) * static_cast<uint32_t>(nb) + static_cast<uint32_t>(t);
        c.snr = __double2float_rn(best);
        c.width = bw;
        a.cells[idx] = c;
      } else {
        atomicOr(&a.counters[kCntStatus], kStatusCellOverflow);
      }
    }
  }
  if (r0 == 0) return;
  __syncthreads();
  for (int q0 = 0; q0 < nbw; q0 += NT) {
    const int q = q0 + tid;
    const uint32_t w = q < nbw ? __funnelshift_r(mrow[q], q + 1 < 4 * tit ? mrow[q + 1] : 0u, r0) : 0u;
    __syncthreads();  // every word of this round is read before one is rewritten
    if (q < nbw) mrow[q] = w;
  }
}

template <int NT>
__global__ void __launch_bounds__(NT, 1152 / NT) k_mf(const __grid_constant__ MfArgs a) { mf_row<NT>(a, blockIdx.x); }

constexpr int kMaxMfBeams = 64;

// Many plans' blocks in one launch: CTA i scores row i - first[b] of the last beam b with
// first[b] <= i.
struct MfMulti {
  int nbeams;
  int first[kMaxMfBeams];
  MfArgs beam[kMaxMfBeams];
};

template <int NT>
__global__ void __launch_bounds__(NT, 1152 / NT) k_mf_multi(const __grid_constant__ MfMulti m) {
  const int i = static_cast<int>(blockIdx.x);
  int lo = 0, hi = m.nbeams - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (m.first[mid] <= i) lo = mid; else hi = mid - 1;
  }
  mf_row<NT>(m.beam[lo], i - m.first[lo]);
}

// Threads per CTA by how many CTAs' rows fit an SM (four and more: 256; three: 384; two: 512; one:
// 1024), or 1024 where the rows are too few to fill the GPU (`alone`: at most one per SM).
enum { kMf256, kMf384, kMf512, kMf1024, kMfShapes };
int mf_shape(int quads, bool alone) {
  const int smem = quads * 16 + 2048;
  if (alone && quads > 1024) return kMf1024;
  if (smem <= 56 * 1024) return kMf256;
  if (smem <= 75 * 1024) return kMf384;
  return smem <= 113 * 1024 ? kMf512 : kMf1024;
}
template <typename F>
cudaError_t mf_dispatch(int shape, F&& f) {
  switch (shape) {
    case kMf256: return f.template go<256>();
    case kMf384: return f.template go<384>();
    case kMf512: return f.template go<512>();
    default: return f.template go<1024>();
  }
}

// Arguments of one plan's block; *quads = the quads of a row's segment.
// Returns false when the block has nothing to do.
bool mf_args(const Plan& p, int64_t e_prev, int64_t e_new, int64_t f_prev, int64_t f_new, void* d_plane_out,
             MfArgs& a, int* quads) {
  const int nb = static_cast<int>(f_new - f_prev);
  const int nemit = static_cast<int>(e_new - e_prev);
  if (nb <= 0 && (d_plane_out == nullptr || nemit <= 0)) return false;
  a = MfArgs{};
  a.plane = p.dp.plane;
  a.Lp = p.Lp;
  a.ndm = p.ndm;
  a.f_prev = f_prev;
  a.e_prev = e_prev;
  a.e_new = e_new;
  a.nb = nb;
  a.width_mask = p.dp.width_mask;
  a.binary = p.mode == SND_MODE_BINARY;
  a.theta = p.det_theta;
  a.sigma_min = p.sigma_min;
  a.out_scale = (p.mode == SND_MODE_FLOAT) ? static_cast<float>(1.0 / std::sqrt(static_cast<double>(p.nchan))) : 0.0f;
  a.mask = p.dp.mask;
  a.mw = p.mw;
  a.cells = p.dp.cells;
  a.cell_cap = p.cell_cap;
  a.counters = p.dp.counters;
  a.plane_out = nemit > 0 ? d_plane_out : nullptr;
  a.nemit = nemit;
  a.out_u8 = p.plane_u8;
  a.tau_steps = p.loop_limit > 0 ? static_cast<int>(p.loop_limit < 64 ? p.loop_limit : 64) : 64;
  const int len = static_cast<int>(e_new - f_prev);
  *quads = ((len + static_cast<int>(f_prev % p.Lp & 3)) >> 2) + 1;  // as mf_row stages them
  {
    // largest root value of the mode times the staged samples bounds every prefix sum
    const double vmax = p.mode == SND_MODE_BINARY ? 1.0 : (p.mode == SND_MODE_GRADED ? p.N : p.nchan);
    a.nowrap = vmax * (len + 8.0) < 2147483647.0 ? 1 : 0;
    // samples a lane of the statistics sums (at least 256 threads)
    const double per_lane = 4.0 * ((*quads + 255) / 256);
    a.stat32 = per_lane * vmax * vmax < 4294967295.0 ? 1 : 0;
  }
  a.wait_cycles = p.wait_limit > 0 ? p.wait_limit : kStageWaitCycles;
  return true;
}

// The launch of one shape: the rows of one plan or of many.
struct MfLaunch {
  MfArgs* one;
  MfMulti* many;
  int rows, smem;
  cudaStream_t s;
  template <int NT>
  cudaError_t go() {
    const void* kern = many ? reinterpret_cast<const void*>(k_mf_multi<NT>) : reinterpret_cast<const void*>(k_mf<NT>);
    int dev = 0, nsm = 0, per_sm = 0;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxDynSmem);
    if (e == cudaSuccess) e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, NT, smem);
    if (e != cudaSuccess) return e;
    const int resident = per_sm > 0 ? nsm * per_sm : rows;  // rows in flight: the next wave's are prefetched
    if (many) {
      for (int b = 0; b < many->nbeams; ++b) many->beam[b].pf_rows = resident;
      k_mf_multi<NT><<<rows, NT, smem, s>>>(*many);
    } else {
      one->pf_rows = resident;
      k_mf<NT><<<rows, NT, smem, s>>>(*one);
    }
    return cudaGetLastError();
  }
};

}  // namespace

cudaError_t launch_mf(const Plan& p, int64_t e_prev, int64_t e_new, int64_t f_prev, int64_t f_new,
                      void* d_plane_out, cudaStream_t s) {
  MfArgs a;
  int quads = 0;
  if (!mf_args(p, e_prev, e_new, f_prev, f_new, d_plane_out, a, &quads)) return cudaSuccess;
  int dev = 0, nsm = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  p.launches += 1;
  return mf_dispatch(mf_shape(quads, p.ndm <= nsm), MfLaunch{&a, nullptr, p.ndm, quads * 16, s});
}

cudaError_t launch_mf_batch(const Plan* const* plans, const ChunkPos* pos, int n, cudaStream_t s) {
  // Blocks are grouped by their rows' shape, so a long-chunk beam does not lower the occupancy of
  // every other beam's rows: a launch per shape in use (more only past 64 beams of one).
  std::vector<MfArgs> args(n);
  std::vector<int> quads(n, 0), live(n, 0);
  for (int i = 0; i < n; ++i)
    live[i] = mf_args(*plans[i], pos[i].e_prev, pos[i].e_new, pos[i].f_prev, pos[i].f_new, nullptr, args[i], &quads[i]);
  for (int c = 0; c < kMfShapes; ++c) {
    for (int i0 = 0; i0 < n;) {
      MfMulti m{};
      int most = 0, rows = 0;
      const Plan* owner = nullptr;
      int i = i0;
      for (; i < n && m.nbeams < kMaxMfBeams; ++i) {
        if (!live[i] || mf_shape(quads[i], false) != c) continue;
        m.beam[m.nbeams] = args[i];
        m.first[m.nbeams] = rows;
        rows += plans[i]->ndm;
        most = most > quads[i] ? most : quads[i];
        if (!owner) owner = plans[i];
        ++m.nbeams;
      }
      i0 = i;
      if (m.nbeams == 0) continue;
      owner->launches += 1;
      const cudaError_t e = mf_dispatch(c, MfLaunch{nullptr, &m, rows, most * 16, s});
      if (e != cudaSuccess) return e;
    }
  }
  return cudaSuccess;
}

}  // namespace snd
