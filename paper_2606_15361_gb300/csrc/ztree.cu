// Labelled-payload Mode C tree with stored partial sums (Methods, "Tree activation modes",
// Mode C; payload x_c(t) = z_c(t) 1[P_c(t) >= u_c] from "Input encoding").
//
// Each node below the root is stored in ST (FP16 or FP32) before its parent reads it, and
// every node adds its children in index order in FP32 starting from 0 (a leaf's children
// are its C channel payloads, already in ST). The root stays FP32; the plane is
// root * fp32(1/sqrt(N_f)). The tree is evaluated per (DM, output time) in "absolute time"
// form: channel c of DM d is read at t + delta_c(d), so the node values equal those of the
// paper's per-node delay lines and the rounding points are exactly the node outputs.
//
// Two forms: k_tree_zs shares each leaf pattern among the DMs of a tile and is used wherever its
// tables fit (see choose_ztree_sharing); k_tree_z sums every leaf per DM and serves the rest: trees
// of one leaf, delay spreads above 16383 samples in a 16-DM tile, windows longer than the ring.
//
// k_tree_z: CTA = 16 trial DMs (one warp each) x 64*NP consecutive output samples; lane L holds the
// sample pairs t0 + 64 j + 2 L, + 1 (slot j). Leaves are processed in groups whose channel
// windows (from a 16-byte aligned ring position at or before the tile's smallest delay per
// channel: tile width + the tile's delay spread) are copied by the TMA engine into one of two
// shared-memory buffers while the previous group is summed from the other. The open nodes of
// every level are per-thread FP32 registers (MAXL levels x 2 NP samples).

#include <cuda_fp16.h>

#include <climits>
#include <cmath>

#include "bulk.h"
#include "snd_internal.h"

namespace snd {
namespace {

struct ZArgs {
  const void* zring;
  int Rz, nchan, ndm, nleaves, C, B, nlev;
  int level_nodes[kMaxLevels];
  const int32_t* delays;  // [ndm][nchan]
  const int32_t* zwb;     // [ndm_tiles][nchan]
  const int32_t* carry;   // [nleaves] levels a finished leaf completes (its carry depth)
  const int32_t* eoff;    // pattern sharing: [ndm_tiles][nleaves + 1] first pattern of each (tile, leaf)
  const int32_t* ent;     // pattern sharing: [patterns][8] (Plan::zent)
  const uint32_t* zdm;    // pattern sharing: [ndm_tiles][nleaves][16] (Plan::zdm)
  int stride;             // pattern sharing: samples of one stored pattern series
  int max_pat;            // pattern sharing: most patterns of one round
  int win, G;             // staged samples per channel, leaves per group
  long long t0;           // first output sample of this call
  int nout;
  float* out;             // plane ring (omode 0, column t mod Lp) or caller plane (omode 1, column t - t0)
  long long ostride;
  int omode, Lp;
  float scale;
  uint32_t* status;        // plan status word (a staging wait that gives up sets kStatusTreeTimeout)
  long long wait_cycles;   // bound of a staging wait (clock cycles)
};

// Two consecutive stored values x = (lo, hi) added to two FP32 sums: lo_sum += lo, hi_sum += hi,
// each rounded once to nearest. FP16: the mixed-precision add of the sm_100 family takes the
// FP16 operand as is (its conversion to FP32 is exact), so each result equals
// fp32(value) + sum rounded once, as an FP32 add of the converted value would give.
__device__ __forceinline__ void add_pair(float& lo_sum, float& hi_sum, uint32_t x, const __half*) {
  asm("{\n .reg .b16 l, h;\n mov.b32 {l, h}, %2;\n add.rn.f32.f16 %0, l, %0;\n add.rn.f32.f16 %1, h, %1;\n}"
      : "+f"(lo_sum), "+f"(hi_sum)
      : "r"(x));
}
__device__ __forceinline__ void add_pair(float& lo_sum, float& hi_sum, uint2 x, const float*) {
  lo_sum = __fadd_rn(lo_sum, __uint_as_float(x.x));
  hi_sum = __fadd_rn(hi_sum, __uint_as_float(x.y));
}
// parent += stored(v): the value rounded to the storage type, added in FP32
__device__ __forceinline__ float add_stored(float parent, float v, const __half*) {
  const __half h = __float2half_rn(v);
  float r;
  asm("add.rn.f32.f16 %0, %1, %2;" : "=f"(r) : "h"(__half_as_ushort(h)), "f"(parent));
  return r;
}
__device__ __forceinline__ float add_stored(float parent, float v, const float*) { return __fadd_rn(parent, v); }

// the pair (window[i], window[i + 1]) of a staged channel window, i = 2 k + odd: one aligned
// load, or for an odd start two aligned words and a byte permute
__device__ __forceinline__ uint32_t load_pair(const __half* w, int k, bool odd) {
  const uint32_t* W = reinterpret_cast<const uint32_t*>(w);
  if (!odd) return W[k];
  return __byte_perm(W[k], W[k + 1], 0x5432);
}
__device__ __forceinline__ uint2 load_pair(const float* w, int k, bool odd) {
  if (!odd) return reinterpret_cast<const uint2*>(w)[k];
  return make_uint2(__float_as_uint(w[2 * k + 1]), __float_as_uint(w[2 * k + 2]));
}
// f(Int<0>{}) .. f(Int<N - 1>{})
template <int I> struct Int { static constexpr int value = I; };
template <int N, int I = 0, typename F>
__device__ __forceinline__ void static_for(F&& f) {
  if constexpr (I < N) {
    f(Int<I>{});
    static_for<N, I + 1>(f);
  }
}
template <typename ST> struct PairT;           // two stored values
template <> struct PairT<__half> { using T = uint32_t; };
template <> struct PairT<float> { using T = uint2; };

// CTA = DT trial DMs (one warp each) x 64 NP consecutive output samples: lane L holds samples
// t0 + 64 j + 2 L and + 1 (pair slot j < NP). Leaves are processed in groups of G; a group's
// channel windows (each from a 16-byte aligned ring position: the tile's smallest delay, the
// tile width and its delay spread) are copied by the TMA engine into one of two shared-memory
// buffers while the previous group is summed from the other, so staging overlaps the adds.
template <typename ST, int MAXL, int NP, int CT>
__global__ void __launch_bounds__(512, 2) k_tree_z(const __grid_constant__ ZArgs a) {
  using P2 = typename PairT<ST>::T;
  constexpr int EPC = 16 / sizeof(ST);  // stored values per 16 bytes
  extern __shared__ __align__(16) unsigned char zsm[];
  __shared__ __align__(8) unsigned long long bars[2];
  const int DT = blockDim.y;
  const int lane = threadIdx.x, wd = threadIdx.y, tid = wd * 32 + lane, nthr = 32 * DT;
  const int tile = blockIdx.y;
  const long long tb = a.t0 + static_cast<long long>(blockIdx.x) * (64 * NP);
  const int d = tile * DT + wd;
  const bool active = d < a.ndm;
  const int GC = a.G * a.C;
  const int WZ = a.win + 2 * EPC;  // staged values per channel: the window, its slack and one chunk
  const size_t bufb = static_cast<size_t>(GC) * WZ * sizeof(ST) + static_cast<size_t>(4) * DT * GC;
  const ST* ring = static_cast<const ST*>(a.zring);
  const int* wb = a.zwb + static_cast<size_t>(tile) * a.nchan;
  const int ngroups = (a.nleaves + a.G - 1) / a.G;
  if (tid == 0) {
    bar_init(smem_u32(&bars[0]), 1);
    bar_init(smem_u32(&bars[1]), 1);
    bar_init_fence();
  }
  __syncthreads();

  // stage group gi into buffer gi & 1: warp 0 issues one bulk copy per channel window (two
  // across the ring's end) after announcing the bytes; every thread fills the DM offsets
  auto issue = [&](int gi) {
    unsigned char* buf = zsm + (gi & 1) * bufb;
    ST* win = reinterpret_cast<ST*>(buf);
    int* drel = reinterpret_cast<int*>(buf + static_cast<size_t>(GC) * WZ * sizeof(ST));
    const int c0 = gi * a.G * a.C, nc = min(a.nchan, (gi + 1) * a.G * a.C) - c0;
    if (wd == 0) {
      const uint32_t bar = smem_u32(&bars[gi & 1]);
      // the buffer was last read by generic loads, before the barrier that ended that group
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      if (lane == 0) bar_expect(bar, static_cast<uint32_t>(nc) * WZ * sizeof(ST));
      __syncwarp();
      for (int cl = lane; cl < nc; cl += 32) {
        const int c = c0 + cl;
        const ST* row = ring + static_cast<size_t>(c) * a.Rz;
        const int r0 = static_cast<int>(((tb + wb[c]) & ~static_cast<long long>(EPC - 1)) % a.Rz);
        const int n1 = min(WZ, a.Rz - r0);
        ST* dst = win + static_cast<size_t>(cl) * WZ;
        bulk_g2s(smem_u32(dst), row + r0, static_cast<uint32_t>(n1 * sizeof(ST)), bar);
        if (n1 < WZ) bulk_g2s(smem_u32(dst + n1), row, static_cast<uint32_t>((WZ - n1) * sizeof(ST)), bar);
      }
    }
    for (int i = tid; i < DT * nc; i += nthr) {
      const int w = i / nc, cl = i - w * nc;
      const int dd = min(tile * DT + w, a.ndm - 1);
      const int c = c0 + cl;
      const int slack = static_cast<int>((tb + wb[c]) & (EPC - 1));
      drel[w * GC + cl] = a.delays[static_cast<size_t>(dd) * a.nchan + c] - wb[c] + slack;
    }
  };

  float acc[MAXL][2 * NP];
  float root[2 * NP];
#pragma unroll
  for (int l = 0; l < MAXL; ++l)
#pragma unroll
    for (int j = 0; j < 2 * NP; ++j) acc[l][j] = 0.0f;
#pragma unroll
  for (int j = 0; j < 2 * NP; ++j) root[j] = 0.0f;

  issue(0);
  __syncthreads();  // group 0's DM offsets
  for (int gi = 0; gi < ngroups; ++gi) {
    if (gi + 1 < ngroups) issue(gi + 1);  // its buffer was released by the last barrier
    const bool ok = bar_wait(smem_u32(&bars[gi & 1]), (gi >> 1) & 1, a.wait_cycles);
    if (__syncthreads_or(!ok)) {
      // a staging wait ran out: report it, and let the copies in flight land (normal bound)
      // before the CTA's shared memory is released
      if (tid == 0) {
        atomicOr(a.status, kStatusTreeTimeout);
        for (int g2 = gi; g2 < gi + 2 && g2 < ngroups; ++g2)
          bar_wait(smem_u32(&bars[g2 & 1]), (g2 >> 1) & 1, kStageWaitCycles);
      }
      return;
    }
    const unsigned char* buf = zsm + (gi & 1) * bufb;
    const ST* win = reinterpret_cast<const ST*>(buf);
    const int* drel = reinterpret_cast<const int*>(buf + static_cast<size_t>(GC) * WZ * sizeof(ST));
    const int k0 = gi * a.G, k1 = min(a.nleaves, k0 + a.G);
    if (active) {
      for (int k = k0; k < k1; ++k) {
        const int cl0 = (k - k0) * a.C;
        const int cn = min(a.C, a.nchan - k * a.C);
        float v[2 * NP];
#pragma unroll
        for (int j = 0; j < 2 * NP; ++j) v[j] = 0.0f;
        auto add_channel = [&](int cl) {
          const int rel = drel[wd * GC + cl];
          const ST* w = win + static_cast<size_t>(cl) * WZ;
          const int kb = (rel >> 1) + lane;
          const bool odd = rel & 1;
          P2 x[NP];
#pragma unroll
          for (int j = 0; j < NP; ++j) x[j] = load_pair(w, kb + 32 * j, odd);
#pragma unroll
          for (int j = 0; j < NP; ++j) add_pair(v[2 * j], v[2 * j + 1], x[j], ring);
        };
        if (CT) {
#pragma unroll
          for (int ci = 0; ci < (CT > 0 ? CT : 1); ++ci) add_channel(cl0 + ci);
        } else {
          for (int ci = 0; ci < cn; ++ci) add_channel(cl0 + ci);
        }
        if (a.nlev == 1) {  // a single leaf is the root: its FP32 sum is not stored
#pragma unroll
          for (int j = 0; j < 2 * NP; ++j) root[j] = v[j];
          continue;
        }
        // the stored leaf goes into its parent's sum (acc[l] holds the open node of level
        // l + 1); when it is the parent's last child the parent is finished, and so on up
        // `depth` levels. depth depends on the leaf only, so the branch is warp-uniform and
        // taken by one leaf in B.
#pragma unroll
        for (int j = 0; j < 2 * NP; ++j) acc[0][j] = add_stored(acc[0][j], v[j], ring);
        const int depth = __ldg(a.carry + k);
        if (depth > 0) {
#pragma unroll
          for (int l = 0; l + 1 < MAXL; ++l) {
            if (l < depth) {
              const bool to_root = (l + 1 == a.nlev - 1);
#pragma unroll
              for (int j = 0; j < 2 * NP; ++j) {
                const float x = acc[l][j];
                acc[l][j] = 0.0f;
                if (to_root) {
                  root[j] = x;
                } else {
                  acc[l + 1][j] = add_stored(acc[l + 1][j], x, ring);
                }
              }
            }
          }
        }
      }
    }
    __syncthreads();  // every reader of this buffer is done: the group after next may refill it
  }
  if (!active) return;
  float* orow = a.out + static_cast<size_t>(d) * a.ostride;
#pragma unroll
  for (int j = 0; j < 2 * NP; ++j) {
    const long long t = tb + 64 * (j >> 1) + 2 * lane + (j & 1);
    if (t - a.t0 >= a.nout) continue;
    const long long col = a.omode ? (t - a.t0) : (t % a.Lp);
    orow[col] = __fmul_rn(root[j], a.scale);
  }
}

template <typename ST, int MAXL, int NP>
cudaError_t run_z(const ZArgs& a, dim3 grid, dim3 block, int smem, cudaStream_t s) {
  // the compile-time 4-channel leaf applies when every leaf has 4 channels
  auto kern = (a.C == 4 && a.nchan % 4 == 0) ? k_tree_z<ST, MAXL, NP, 4> : k_tree_z<ST, MAXL, NP, 0>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxDynSmem);
  if (e != cudaSuccess) return e;
  kern<<<grid, block, smem, s>>>(a);
  return cudaGetLastError();
}

// 32-bit store at a shared-memory byte address plus a constant (lds32's counterpart)
template <int OFF>
__device__ __forceinline__ void sts32(uint32_t addr, uint32_t v) {
  asm volatile("st.shared.b32 [%0 + %1], %2;" ::"r"(addr), "n"(OFF), "r"(v) : "memory");
}

// The same tree with each distinct leaf pattern of a DM tile summed once. Within 16 neighbouring
// trial DMs a leaf's channels keep one of a few relative delays (3.8 of 16 on a 1024-channel,
// 2048-DM grid over 2000 pc cm^-3), and a leaf's stored value depends on that pattern and on the
// leaf's own delay only. So a CTA first sums every pattern of a group of leaves over its tile and
// the delays it serves (phase A), rounds it to the storage type once, as every DM would, and keeps
// the series in shared memory; then each DM adds one stored value per leaf instead of C channels
// (phase B). Operands and order of every addition are those of k_tree_z, so the planes are the same
// bit for bit.
// What bounds it: instruction issue and shared-memory reads, one stored pair per (DM, leaf) in phase
// B and C pairs per pattern in phase A, against C per (DM, leaf) in k_tree_z. A lane carries 2 NP
// outputs of every open level in registers, which is what limits the tile: 16 DMs (one warp each) x
// 64 NP samples on the whole register file of an SM; a longer tile repeats less of the delay span
// per pattern. Each warp stages its share of a group's windows; the copies of group g + 2 start once
// phase A of group g has read its windows, so they have two groups' work to land.
// FP16: lane L holds the sample pairs 64 j + 2 L, + 1 (slots 2 j, 2 j + 1); FP32: the samples 32 j + L.
// 1024 channels, 2048 DMs, 16384 samples: FP16 3.7 ms (k_tree_z 6.5), FP32 4.6 (9.9); B = 2, nine
// levels, FP16 7.7 (20.7). ncu: issue active 63%; of the instructions about 16% are the additions,
// 15% shared loads, the rest selecting pairs, addresses, loops and the nodes above the leaves.
template <typename ST, int MAXL, int NP, int CT>
__global__ void __launch_bounds__(512, 1) k_tree_zs(const __grid_constant__ ZArgs a) {
  constexpr bool HALF = sizeof(ST) == 2;
  constexpr int EPC = 16 / sizeof(ST);
  constexpr int TS = 64 * NP;
  constexpr int DT = 16;
  constexpr int NS = 2 * NP;               // outputs per lane
  constexpr int NL32 = HALF ? NP : NS;     // 32-bit loads that cover them
  extern __shared__ __align__(16) unsigned char zsm[];
  __shared__ __align__(8) unsigned long long bars[2];
  const int lane = threadIdx.x, wd = threadIdx.y;
  const int tile = blockIdx.y;
  const long long tb = a.t0 + static_cast<long long>(blockIdx.x) * TS;
  const int d = tile * DT + wd;
  const bool active = d < a.ndm;
  const int WZ = a.win;
  const ST* ring = static_cast<const ST*>(a.zring);
  const int* wb = a.zwb + static_cast<size_t>(tile) * a.nchan;
  const int* eo = a.eoff + static_cast<size_t>(tile) * (a.nleaves + 1);
  const int ngroups = (a.nleaves + a.G - 1) / a.G;
  // shared memory: 2 x (channel windows | pattern records) | 4 x DM offsets | pattern series
  const uint32_t s0 = smem_u32(zsm);
  const uint32_t winb = static_cast<uint32_t>(a.G * a.C * WZ) * static_cast<uint32_t>(sizeof(ST));
  const uint32_t bufb = winb + static_cast<uint32_t>(a.max_pat) * 32u;
  const uint32_t sdm = s0 + 2 * bufb, sser = sdm + 4u * a.G * (DT * 4u);
  const int tile0 = __ldg(eo);
  if (wd == 0 && lane == 0) {
    bar_init(smem_u32(&bars[0]), DT);  // one arrival per warp
    bar_init(smem_u32(&bars[1]), DT);
    bar_init_fence();
  }
  __syncthreads();

  // Group gi's copies: every warp announces and copies the channel windows wd, wd + 16, ..., warp 0
  // also the pattern records and the DM offsets.
  const int tbr = static_cast<int>(tb % a.Rz);
  auto issue = [&](int gi, int e0, int ne) {
    const int k0 = gi * a.G, k1 = min(a.nleaves, k0 + a.G);
    const int c0 = k0 * a.C, nc = min(a.nchan, k1 * a.C) - c0;
    const uint32_t bar = smem_u32(&bars[gi & 1]);
    const uint32_t buf = s0 + (gi & 1) * bufb;
    // the buffers were last read by generic loads, before the barrier that precedes this call
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    if (lane == 0) {
      const int mine = nc > wd ? (nc - wd + DT - 1) / DT : 0;
      bar_expect(bar, static_cast<uint32_t>(mine) * WZ * static_cast<uint32_t>(sizeof(ST)) +
                          (wd == 0 ? ne * 32u + (k1 - k0) * (DT * 4u) : 0u));
    }
    __syncwarp();
    const int cl = wd + DT * lane;
    if (cl < nc) {
      const ST* row = ring + static_cast<size_t>(c0 + cl) * a.Rz;
      // (tb + delay) rounded down to 16 bytes, modulo the ring (a multiple of 16 bytes above any delay)
      int r0 = (tbr + __ldg(wb + c0 + cl)) & ~(EPC - 1);
      if (r0 >= a.Rz) r0 -= a.Rz;
      const int n1 = min(WZ, a.Rz - r0);
      const uint32_t dst = buf + static_cast<uint32_t>(cl) * WZ * static_cast<uint32_t>(sizeof(ST));
      bulk_g2s(dst, row + r0, static_cast<uint32_t>(n1 * sizeof(ST)), bar);
      if (n1 < WZ) bulk_g2s(dst + n1 * static_cast<uint32_t>(sizeof(ST)), row, static_cast<uint32_t>((WZ - n1) * sizeof(ST)), bar);
    }
    if (wd == 0 && lane == 0) {
      bulk_g2s(buf + winb, a.ent + static_cast<size_t>(e0) * 8, static_cast<uint32_t>(ne) * 32u, bar);
      bulk_g2s(sdm + (gi & 3) * a.G * (DT * 4u), a.zdm + (static_cast<size_t>(tile) * a.nleaves + k0) * DT,
               static_cast<uint32_t>(k1 - k0) * (DT * 4u), bar);
    }
  };
  auto first_of = [&](int gi) { return __ldg(eo + min(a.nleaves, gi * a.G)); };  // group gi's first pattern

  float acc[MAXL - 1][NS];
#pragma unroll
  for (int l = 0; l < MAXL - 1; ++l)
#pragma unroll
    for (int j = 0; j < NS; ++j) acc[l][j] = 0.0f;

  int e0 = tile0, e1 = first_of(1), e2 = first_of(2);
  issue(0, e0, e1 - e0);
  if (ngroups > 1) issue(1, e1, e2 - e1);
  for (int gi = 0; gi < ngroups; ++gi) {
    const int k0 = gi * a.G, k1 = min(a.nleaves, k0 + a.G);
    const int e3 = first_of(gi + 3);
    const bool ok = bar_wait(smem_u32(&bars[gi & 1]), (gi >> 1) & 1, a.wait_cycles);
    // also the end of the previous group's phase B: the series may be rewritten
    if (__syncthreads_or(!ok)) {
      // a staging wait ran out: report it, and let the copies in flight land (normal bound)
      // before the CTA's shared memory is released
      if (wd == 0 && lane == 0) {
        atomicOr(a.status, kStatusTreeTimeout);
        for (int g2 = gi; g2 < gi + 2 && g2 < ngroups; ++g2)
          bar_wait(smem_u32(&bars[g2 & 1]), (g2 >> 1) & 1, kStageWaitCycles);
      }
      return;
    }
    // A. each pattern's stored leaf series, in pieces of 32 words (a word is a pair of FP16 values or
    // one FP32 value): the NL32 pieces that every pattern of the group has are split evenly over the
    // warps, and the warp with a pattern's last one also takes those of its delay span
    const uint32_t swin = s0 + (gi & 1) * bufb;
    const int4* recs = reinterpret_cast<const int4*>(zsm + (gi & 1) * bufb + winb);
    const int pieces = NL32 * (e1 - e0);
    const int last = (wd + 1) * pieces / DT;
    for (int p = wd * pieces / DT; p < last;) {
      const int e = p / NL32, p0 = p - e * NL32;
      const int4 ra = recs[2 * e], rb = recs[2 * e + 1];
      const int off[7] = {ra.x, ra.y, ra.z, ra.w, rb.x, rb.y, rb.z};
      const int k = rb.w >> 16, words = HALF ? (TS + (rb.w & 0xFFFF) + 1) >> 1 : TS + (rb.w & 0xFFFF);
      const int cl0 = (k - k0) * a.C, cn = CT ? CT : min(a.C, a.nchan - k * a.C);
      constexpr int NC = CT ? CT : 7;
      uint32_t at[NC], sel[NC];  // this lane's next word of each channel; which bytes make its pair
#pragma unroll
      for (int ci = 0; ci < NC; ++ci) {
        // bits 28-30: the window's first delay mod 8, whose part below 16 bytes the copy kept
        const int phase = (tbr + (off[ci] >> 28)) & (EPC - 1);
        const int v = ci < cn ? (cl0 + ci) * WZ + (off[ci] & 0x0FFFFFFF) + phase : 0;
        at[ci] = swin + 4u * static_cast<uint32_t>((HALF ? v >> 1 : v) + 32 * p0 + lane);
        sel[ci] = (v & 1) ? 0x5432u : 0x3210u;
      }
      uint32_t out = sser + static_cast<uint32_t>(e) * a.stride * static_cast<uint32_t>(sizeof(ST)) + 4u * (32 * p0 + lane);
      auto piece = [&](auto it) {  // the piece after `it` more
        constexpr int O = 128 * decltype(it)::value;
        if constexpr (HALF) {
          uint32_t x[NC], y[NC];
#pragma unroll
          for (int ci = 0; ci < NC; ++ci)
            if (ci < cn) {
              x[ci] = lds32<O>(at[ci]);
              y[ci] = lds32<O + 4>(at[ci]);
            }
          float v0 = 0.0f, v1 = 0.0f;
#pragma unroll
          for (int ci = 0; ci < NC; ++ci)
            if (ci < cn) add_pair(v0, v1, __byte_perm(x[ci], y[ci], sel[ci]), ring);
          const __half2 hv = __floats2half2_rn(v0, v1);
          sts32<O>(out, *reinterpret_cast<const uint32_t*>(&hv));
        } else {
          uint32_t x[NC];
#pragma unroll
          for (int ci = 0; ci < NC; ++ci)
            if (ci < cn) x[ci] = lds32<O>(at[ci]);
          float v = 0.0f;
#pragma unroll
          for (int ci = 0; ci < NC; ++ci)
            if (ci < cn) v = __fadd_rn(v, __uint_as_float(x[ci]));
          sts32<O>(out, __float_as_uint(v));
        }
      };
      auto advance = [&](uint32_t by) {
#pragma unroll
        for (int ci = 0; ci < NC; ++ci) at[ci] += by;
        out += by;
      };
      const int p1 = min(NL32, p0 + last - p);
      int q = p0;
      for (; q + 4 <= p1; q += 4) {
        static_for<4>(piece);
        advance(512u);
      }
      for (; q < p1; ++q) {
        piece(Int<0>{});
        advance(128u);
      }
      if (p1 == NL32)
        for (int w = 32 * NL32 + lane; w < words; w += 32) {
          piece(Int<0>{});
          advance(128u);
        }
      p += p1 - p0;
    }
    __syncthreads();
    // the windows and records are read: the group after next may land in their place
    if (gi + 2 < ngroups) issue(gi + 2, e2, e3 - e2);
    // B. each DM adds its pattern's stored value of every leaf; finished nodes go up
    if (active) {
      uint32_t sd = sdm + (gi & 3) * a.G * (DT * 4u) + 4u * wd;
      for (int k = k0; k < k1; ++k, sd += DT * 4u) {
        const uint32_t m = lds32<0>(sd);
        const int depth = __ldg(a.carry + k);
        const int q = (static_cast<int>(m >> 14) - (e0 - tile0)) * a.stride + static_cast<int>(m & 16383u);
        const uint32_t w = sser + 4u * static_cast<uint32_t>((HALF ? q >> 1 : q) + lane);
        if constexpr (HALF) {
          if (q & 1) {
            static_for<NP>([&](auto j) {
              constexpr int J = decltype(j)::value;
              add_pair(acc[0][2 * J], acc[0][2 * J + 1], __byte_perm(lds32<128 * J>(w), lds32<128 * J + 4>(w), 0x5432), ring);
            });
          } else {
            static_for<NP>([&](auto j) {
              constexpr int J = decltype(j)::value;
              add_pair(acc[0][2 * J], acc[0][2 * J + 1], lds32<128 * J>(w), ring);
            });
          }
        } else {
          static_for<NS>([&](auto j) {
            constexpr int J = decltype(j)::value;
            acc[0][J] = __fadd_rn(acc[0][J], __uint_as_float(lds32<128 * J>(w)));
          });
        }
        // a leaf that is its parent's last child finishes the parent, and so on up `depth`
        // levels (depth depends on the leaf only, so the branch is warp-uniform); the root ends in
        // acc[0], whose own node is finished by then
        if (depth > 0) {
          constexpr int top = MAXL - 2;
#pragma unroll
          for (int l = 0; l < MAXL - 1; ++l) {
            if (l < depth) {
              const bool to_root = l + 1 == a.nlev - 1;
#pragma unroll
              for (int j = 0; j < NS; ++j) {
                const float x = acc[l][j];
                if (to_root) {
                  acc[0][j] = x;
                } else if (l < top) {
                  acc[l][j] = 0.0f;
                  acc[l < top ? l + 1 : l][j] = add_stored(acc[l < top ? l + 1 : l][j], x, ring);
                }
              }
            }
          }
        }
      }
    }
    e0 = e1;
    e1 = e2;
    e2 = e3;
  }
  if (!active) return;
  // the root's sum to the caller's plane (column t - t0) or the plane ring (column t mod Lp)
  float* orow = a.out + static_cast<size_t>(d) * a.ostride;
  const int n = min(TS, a.nout - static_cast<int>(blockIdx.x) * TS);  // samples of this tile
  const int col0 = a.omode ? static_cast<int>(tb - a.t0) : static_cast<int>(tb % a.Lp);
  const int wrap = a.omode ? INT_MAX : a.Lp;
#pragma unroll
  for (int j = 0; j < NS; ++j) {
    const int i = HALF ? 64 * (j >> 1) + 2 * lane + (j & 1) : 32 * j + lane;
    int col = col0 + i;
    if (col >= wrap) col -= wrap;
    if (i < n) orow[col] = __fmul_rn(acc[0][j], a.scale);
  }
}

template <typename ST, int MAXL, int NP>
cudaError_t run_zs(const ZArgs& a, dim3 grid, int smem, cudaStream_t s) {
  auto kern = (a.C == 4 && a.nchan % 4 == 0) ? k_tree_zs<ST, MAXL, NP, 4> : k_tree_zs<ST, MAXL, NP, 0>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxDynSmem);
  if (e != cudaSuccess) return e;
  kern<<<grid, dim3(32, 16), smem, s>>>(a);
  return cudaGetLastError();
}

// The pattern-sharing launch: of the tile lengths the tree's depth allows, the one with the least
// estimated work, i.e. waves of CTAs (one per SM) times the additions of a CTA plus a round's fixed
// cost; short calls take short tiles so that every SM has one.
template <typename ST>
cudaError_t launch_shared(const Plan& p, ZArgs& a, cudaStream_t s) {
  int dev = 0, nsm = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  const ZGeom& z = p.zgeom;
  ZShape best{};
  double cost = 0.0;
  for (int np = ztree_max_pairs(p.nlev); np >= 2; np -= np > 4 ? 4 : 2) {
    const ZShape sh = ztree_shape(p, np);
    if (sh.group == 0) continue;
    const double ts = 64.0 * np;
    const double ctas = std::ceil(a.nout / ts) * z.ndm_tiles;
    const double per = 16.0 * ts + 0.01 * z.share_pct * (ts + 0.5 * z.sspread) * (p.C + 1) + 4096.0 / sh.group;
    const double c = std::ceil(ctas / nsm) * per;
    if (best.group == 0 || c < cost) {
      best = sh;
      cost = c;
    }
  }
  if (best.group == 0) return cudaErrorInvalidConfiguration;
  a.win = best.win;
  a.stride = best.stride;
  a.G = best.group;
  a.max_pat = z.group_max[best.group - 1];
  const dim3 grid(static_cast<unsigned>((a.nout + 64 * best.np - 1) / (64 * best.np)), z.ndm_tiles);
  if (p.nlev <= 4) {
    if (best.np == 12) return run_zs<ST, 4, 12>(a, grid, best.smem, s);
    if (best.np == 8) return run_zs<ST, 4, 8>(a, grid, best.smem, s);
    return run_zs<ST, 4, 4>(a, grid, best.smem, s);
  }
  if (p.nlev <= 6) return best.np == 8 ? run_zs<ST, 6, 8>(a, grid, best.smem, s) : run_zs<ST, 6, 4>(a, grid, best.smem, s);
  if (p.nlev <= 10) return run_zs<ST, 10, 4>(a, grid, best.smem, s);
  return run_zs<ST, 16, 2>(a, grid, best.smem, s);
}

}  // namespace

cudaError_t launch_tree_z(const Plan& p, int64_t e_prev, int64_t e_new, void* d_plane_out, cudaStream_t s) {
  if (e_new <= e_prev) return cudaSuccess;
  const ZGeom& z = p.zgeom;
  ZArgs a{};
  a.zring = p.dp.zring;
  a.Rz = z.Rz;
  a.nchan = p.nchan;
  a.ndm = p.ndm;
  a.nleaves = p.nleaves;
  a.C = p.C;
  a.B = p.B;
  a.nlev = p.nlev;
  for (int l = 0; l < kMaxLevels; ++l) a.level_nodes[l] = l < p.nlev ? p.level_nodes[l] : 1;
  a.delays = p.dp.delays;
  a.zwb = p.dp.zwb;
  a.carry = p.dp.zcarry;
  a.win = z.win;
  a.G = z.group_leaves;
  a.t0 = e_prev;
  a.nout = static_cast<int>(e_new - e_prev);
  if (d_plane_out) {
    a.out = static_cast<float*>(d_plane_out);
    a.ostride = a.nout;
    a.omode = 1;
  } else {
    a.out = reinterpret_cast<float*>(p.dp.plane);
    a.ostride = p.Lp;
    a.omode = 0;
  }
  a.Lp = p.Lp;
  a.scale = static_cast<float>(1.0 / std::sqrt(static_cast<double>(p.nchan)));
  a.status = p.dp.counters + kCntStatus;
  a.wait_cycles = p.wait_limit > 0 ? p.wait_limit : kStageWaitCycles;
  a.eoff = p.dp.zeoff;
  a.ent = p.dp.zent;
  a.zdm = p.dp.zdm;
  if (z.shared) {
    p.launches += 1;
    return z.fp16 ? launch_shared<__half>(p, a, s) : launch_shared<float>(p, a, s);
  }
  dim3 block(32, z.dms_per_cta);
  dim3 grid(static_cast<unsigned>((a.nout + z.tile_samples - 1) / z.tile_samples), z.ndm_tiles);
  p.launches += 1;
  if (z.fp16) {
    if (z.maxl == 4) return run_z<__half, 4, 4>(a, grid, block, z.smem_bytes, s);
    if (z.maxl == 8) return run_z<__half, 8, 2>(a, grid, block, z.smem_bytes, s);
    return run_z<__half, 16, 1>(a, grid, block, z.smem_bytes, s);
  }
  if (z.maxl == 4) return run_z<float, 4, 4>(a, grid, block, z.smem_bytes, s);
  if (z.maxl == 8) return run_z<float, 8, 2>(a, grid, block, z.smem_bytes, s);
  return run_z<float, 16, 1>(a, grid, block, z.smem_bytes, s);
}

}  // namespace snd
