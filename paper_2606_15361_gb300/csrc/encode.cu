// Delta encoder (Methods, "Input encoding"): per-channel two-pass sigma-clip statistics
// and x_c(t) = 1[z_c(t) > theta], written bit-packed into the mirrored spike ring.
//
// Statistics come from a 256-bin histogram per channel of the chunk, evaluated in a fixed
// FP64 order with explicit round-to-nearest intrinsics (no contraction), so the integer
// level u_c (fire iff P >= u_c) is one well-defined decision:
//   mu0 = S1/n, sigma0 = sqrt(max(0, S2/n - mu0^2)), clip to [mu0 -+ 5 sigma0],
//   S1c = (S1in + n_lo lo) + n_hi hi, S2c = (S2in + n_lo lo^2) + n_hi hi^2,
//   mu = S1c/n, sigma = sqrt(max(0, S2c/n - mu^2)), u = min{v in 0..255 : v > mu + theta sigma}.
//
// Two forms: k_encode does a whole chunk of a block of 32 channels in one launch, with a cluster's
// CTAs holding the samples in shared memory between the statistics and the packing; the labelled
// payload, and chunks too long for that, take k_hist, k_levels and a pack kernel.
//
// Ring layout: ring[c][2R] uint32; absolute sample a lives in word a>>5, bit a&31, stored at
// physical word (a>>5) mod R and again at R + that (the mirror lets any window of < R words
// be read contiguously).

#include <cuda_fp16.h>

#include <algorithm>

#include "snd_internal.h"

namespace snd {
namespace {

constexpr int kHistRowsPerBlock = 2048;
constexpr int kHistWarps = 32;  // warps of a histogram CTA, each over every kHistWarps-th row

// CTA (bx, by) of the histogram: 32 channels x kHistRowsPerBlock samples, kHistWarps warps
__device__ __forceinline__ void hist_cta(const uint8_t* __restrict__ chunk, int nsamp, int nchan,
                                         uint32_t* __restrict__ hist, int bx, int by) {
  constexpr int NT = 32 * kHistWarps;
  __shared__ uint32_t h[256][32];
  const int lane = threadIdx.x, wy = threadIdx.y;
  const int tid = wy * 32 + lane;
  for (int i = tid; i < 256 * 32; i += NT) (&h[0][0])[i] = 0;
  __syncthreads();
  const int c = bx * 32 + lane;
  const int r0 = by * kHistRowsPerBlock;
  const int r1 = min(nsamp, r0 + kHistRowsPerBlock);
  if (c < nchan) {
    // eight rows' loads in flight per lane before their counts are added
    int r = r0 + wy;
    for (; r + 7 * kHistWarps < r1; r += 8 * kHistWarps) {
      uint32_t v[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) v[k] = __ldg(chunk + static_cast<size_t>(r + kHistWarps * k) * nchan + c);
#pragma unroll
      for (int k = 0; k < 8; ++k) atomicAdd(&h[v[k]][lane], 1u);
    }
    for (; r < r1; r += kHistWarps) atomicAdd(&h[__ldg(chunk + static_cast<size_t>(r) * nchan + c)][lane], 1u);
  }
  __syncthreads();
  for (int i = tid; i < 256 * 32; i += NT) {
    const int v = i >> 5, l = i & 31;
    const int cc = bx * 32 + l;
    const uint32_t n = h[v][l];
    if (cc < nchan && n) atomicAdd(&hist[static_cast<size_t>(cc) * 256 + v], n);
  }
}

__global__ void __launch_bounds__(32 * kHistWarps) k_hist(const uint8_t* __restrict__ chunk, int nsamp, int nchan,
                                              uint32_t* __restrict__ hist) {
  hist_cta(chunk, nsamp, nchan, hist, blockIdx.x, blockIdx.y);
}

// One warp per channel; lane l holds bins l, l+32, ..., l+224. Integer sums are exact; the
// FP64 steps run on lane 0 in the fixed order above. For integer v, v < lo <=> v < ceil(lo)
// and v > hi <=> v > floor(hi), and the smallest integer above thr is floor(thr) + 1, so the
// clip bounds and the level are exact integer decisions.
// With ztab set (labelled payload), every lane also writes the payload of its 8 values,
// z = (v - mu)/sigma in FP64 for v >= u (0 below), rounded once to FP16 (zmode bit 0) or FP32;
// with zmode bit 1 (the paper's own 0/1 spike payload) z = 1 for v >= u instead.
__device__ __forceinline__ void levels_warp(uint32_t* __restrict__ hist, int nchan, int nsamp, double theta,
                                            int32_t* __restrict__ levels, void* __restrict__ ztab, int zmode,
                                            const int c, const int lane) {
  if (c >= nchan) return;
  uint32_t* h = hist + static_cast<size_t>(c) * 256;
  long long n[8];
  long long s1 = 0, s2 = 0;
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const int v = lane + 32 * k;
    n[k] = h[v];
    h[v] = 0;  // ready for the next chunk
    s1 += n[k] * v;
    s2 += n[k] * v * v;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    s1 += __shfl_xor_sync(0xFFFFFFFFu, s1, o);
    s2 += __shfl_xor_sync(0xFFFFFFFFu, s2, o);
  }
  const double nf = static_cast<double>(nsamp);
  const double mu0 = __ddiv_rn(static_cast<double>(s1), nf);
  const double var0 = __dsub_rn(__ddiv_rn(static_cast<double>(s2), nf), __dmul_rn(mu0, mu0));
  const double sig0 = var0 > 0.0 ? __dsqrt_rn(var0) : 0.0;
  const double lo = __dsub_rn(mu0, __dmul_rn(5.0, sig0));
  const double hi = __dadd_rn(mu0, __dmul_rn(5.0, sig0));
  const int ilo = static_cast<int>(fmin(fmax(ceil(lo), -1.0), 257.0));    // in range: v >= ilo
  const int ihi = static_cast<int>(fmin(fmax(floor(hi), -1.0), 257.0));   //           v <= ihi
  long long s1in = 0, s2in = 0, nlo = 0, nhi = 0;
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const int v = lane + 32 * k;
    if (v < ilo) {
      nlo += n[k];
    } else if (v > ihi) {
      nhi += n[k];
    } else {
      s1in += n[k] * v;
      s2in += n[k] * v * v;
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    s1in += __shfl_xor_sync(0xFFFFFFFFu, s1in, o);
    s2in += __shfl_xor_sync(0xFFFFFFFFu, s2in, o);
    nlo += __shfl_xor_sync(0xFFFFFFFFu, nlo, o);
    nhi += __shfl_xor_sync(0xFFFFFFFFu, nhi, o);
  }
  // every lane holds the same reduced sums, so every lane evaluates the same FP64 recipe
  const double s1c = __dadd_rn(__dadd_rn(static_cast<double>(s1in), __dmul_rn(static_cast<double>(nlo), lo)),
                               __dmul_rn(static_cast<double>(nhi), hi));
  const double s2c =
      __dadd_rn(__dadd_rn(static_cast<double>(s2in), __dmul_rn(static_cast<double>(nlo), __dmul_rn(lo, lo))),
                __dmul_rn(static_cast<double>(nhi), __dmul_rn(hi, hi)));
  const double mu = __ddiv_rn(s1c, nf);
  const double var = __dsub_rn(__ddiv_rn(s2c, nf), __dmul_rn(mu, mu));
  const double sig = var > 0.0 ? __dsqrt_rn(var) : 0.0;
  int u = 256;
  if (sig > 0.0) {
    const double thr = __dadd_rn(mu, __dmul_rn(theta, sig));
    if (thr < 0.0) {
      u = 0;
    } else if (thr < 255.0) {
      u = static_cast<int>(floor(thr)) + 1;
    }
  }
  if (lane == 0) levels[c] = u;
  if (ztab) {
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const int v = lane + 32 * k;
      const double z = (v >= u) ? ((zmode & 2) ? 1.0 : __ddiv_rn(__dsub_rn(static_cast<double>(v), mu), sig)) : 0.0;
      if (zmode & 1) {
        static_cast<__half*>(ztab)[static_cast<size_t>(c) * 256 + v] = __double2half(z);
      } else {
        static_cast<float*>(ztab)[static_cast<size_t>(c) * 256 + v] = __double2float_rn(z);
      }
    }
  }
}

__global__ void __launch_bounds__(256) k_levels(uint32_t* __restrict__ hist, int nchan, int nsamp, double theta,
                                                int32_t* __restrict__ levels, void* __restrict__ ztab, int zmode) {
  levels_warp(hist, nchan, nsamp, theta, levels, ztab, zmode, (blockIdx.x * blockDim.x + threadIdx.x) >> 5,
              threadIdx.x & 31);
}

// Labelled payload into the ring: zring[c][(t0 + r) mod Rz] = ztab[c][P_c(r)]. A CTA
// transposes 32 channels x 256 samples through shared memory, so both the chunk reads and
// the ring writes are contiguous runs; the 32 payload tables it uses stay in L1.
template <typename ST>
__global__ void __launch_bounds__(256) k_pack_z(const uint8_t* __restrict__ chunk, int nsamp, int nchan,
                                                const ST* __restrict__ ztab, long long t0, ST* __restrict__ zring,
                                                int Rz) {
  __shared__ ST tile[32][257];
  const int lane = threadIdx.x, wy = threadIdx.y;
  const int c0 = blockIdx.x * 32, r0 = blockIdx.y * 256;
  const int c = c0 + lane;
  for (int rl = wy; rl < 256; rl += 8) {
    const int r = r0 + rl;
    if (r < nsamp && c < nchan)
      tile[lane][rl] = __ldg(ztab + static_cast<size_t>(c) * 256 + chunk[static_cast<size_t>(r) * nchan + c]);
  }
  __syncthreads();
  for (int cl = wy; cl < 32; cl += 8) {
    if (c0 + cl >= nchan) break;
    ST* row = zring + static_cast<size_t>(c0 + cl) * Rz;
    for (int rl = lane; rl < 256; rl += 32) {
      const int r = r0 + rl;
      if (r < nsamp) row[static_cast<int>((t0 + r) % Rz)] = tile[cl][rl];
    }
  }
}

// One thread per (channel, ring word). Lanes run over channels, so each row read is a
// contiguous run of bytes. Bits of samples before the chunk keep the ring's old value.
__global__ void __launch_bounds__(256) k_pack(const uint8_t* __restrict__ chunk, int nsamp, int nchan,
                                              const int32_t* __restrict__ levels, long long t0,
                                              long long word0, int nwords, uint32_t* __restrict__ ring,
                                              int R) {
  const int c = blockIdx.x * 32 + threadIdx.x;
  const int q = blockIdx.y * 8 + threadIdx.y;
  if (c >= nchan || q >= nwords) return;
  const long long aw = word0 + q;
  const long long s0 = aw * 32;  // absolute sample of bit 0
  const int u = levels[c];
  uint32_t bits = 0;
#pragma unroll 4
  for (int i = 0; i < 32; ++i) {
    const long long a = s0 + i;
    const long long r = a - t0;
    if (r >= 0 && r < nsamp) {
      const int v = chunk[static_cast<size_t>(r) * nchan + c];
      bits |= static_cast<uint32_t>(v >= u) << i;
    }
  }
  const int phys = static_cast<int>(aw % R);
  uint32_t* row = ring + static_cast<size_t>(c) * 2 * R;
  // keep the bits of samples before the chunk (written by the previous chunk)
  const uint32_t keep = (s0 < t0) ? ((1u << static_cast<int>(t0 - s0)) - 1u) : 0u;
  const uint32_t w = (row[phys] & keep) | bits;
  row[phys] = w;
  row[phys + R] = w;
}

// Warp per (ring word, 32 channels): lane l holds sample 32*aw + l and loads its 32 channel
// bytes with two 16-byte loads; one ballot per channel turns the 32 comparisons into that
// channel's spike word. Requires nchan % 32 == 0 and a 16-byte aligned chunk.
__device__ __forceinline__ void pack32_warp(const uint8_t* __restrict__ chunk, int nsamp, int nchan,
                                            const int32_t* __restrict__ levels, long long t0, long long word0,
                                            int nwords, uint32_t* __restrict__ ring, int R, const int task,
                                            const int lane) {
  const int ncb = nchan >> 5;
  if (task >= nwords * ncb) return;
  const int q = task / ncb, cb = task - q * ncb;
  const int c0 = cb * 32;
  const long long aw = word0 + q;
  const long long r = aw * 32 + lane - t0;
  const bool valid = r >= 0 && r < nsamp;
  uint4 b0 = make_uint4(0, 0, 0, 0), b1 = b0;
  if (valid) {
    const uint4* src = reinterpret_cast<const uint4*>(chunk + static_cast<size_t>(r) * nchan + c0);
    b0 = __ldg(src);
    b1 = __ldg(src + 1);
  }
  const uint32_t wv[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
  const int my_u = levels[c0 + lane];
  uint32_t mine = 0;
#pragma unroll
  for (int j = 0; j < 32; ++j) {
    const int u = __shfl_sync(0xFFFFFFFFu, my_u, j);
    const int v = static_cast<int>((wv[j >> 2] >> (8 * (j & 3))) & 0xFFu);
    const uint32_t word = __ballot_sync(0xFFFFFFFFu, valid && v >= u);
    if (lane == j) mine = word;
  }
  const long long s0 = aw * 32;
  const int phys = static_cast<int>(aw % R);
  uint32_t* row = ring + static_cast<size_t>(c0 + lane) * 2 * R;
  uint32_t w = mine;
  // only the chunk's first word keeps bits of samples before the chunk (previous chunk)
  if (s0 < t0) w |= row[phys] & ((1u << static_cast<int>(t0 - s0)) - 1u);
  row[phys] = w;
  row[phys + R] = w;
}

__global__ void __launch_bounds__(256) k_pack32(const uint8_t* __restrict__ chunk, int nsamp, int nchan,
                                                const int32_t* __restrict__ levels, long long t0, long long word0,
                                                int nwords, uint32_t* __restrict__ ring, int R) {
  pack32_warp(chunk, nsamp, nchan, levels, t0, word0, nwords, ring, R, (blockIdx.x * blockDim.x + threadIdx.x) >> 5,
              threadIdx.x & 31);
}

// One beam's chunk for k_encode. A cluster of S CTAs takes 32 channels; CTA `rank` of it the ring words
// w0 + rank * wpc .. (wpc words), i.e. those words' samples.
struct EncBeam {
  const uint8_t* chunk;
  int nsamp, nchan;
  int32_t* levels;
  double theta;
  long long t0, w0;
  int nwords, wpc;
  uint32_t* ring;
  int R;
  int vec;             // bytes per load: 16, 4 or 1 (what the chunk's address and nchan allow)
  uint32_t* counters;  // the beam's matched-filter / candidate block counters, cleared here
};

constexpr int kMaxEncBeams = 64;
constexpr int kEncCluster = 8;  // most CTAs of a cluster

struct EncMulti {
  int nbeams;
  int first[kMaxEncBeams];  // clusters of the beams before
  EncBeam beam[kMaxEncBeams];
};

// dynamic shared memory of a CTA: the samples and the packed words
__host__ __device__ constexpr int enc_smem(int wpc) { return wpc * 32 * 32 + 32 * (wpc | 1) * 4; }

// static shared memory of a CTA of NT threads
template <int NT>
struct EncShared {
  uint32_t red[NT / 32][4][32];
  // every CTA's totals: sum and sum of squares; count below, count above, sum and sum of squares of both
  uint32_t tot1[kEncCluster][2][32], tot2[kEncCluster][4][32];
  int clip[2][32], lev[32];
};

// Longest chunk of the one-launch encoder: what a CTA may have in shared memory less its static part
// (217,728 bytes: 189 ring words a CTA, 1512 a cluster, 48,384 samples from a word's start).
constexpr int kEncMaxSmem = 227 * 1024 - static_cast<int>(sizeof(EncShared<512>));
// The most dynamic shared memory with which `ctas` CTAs of NT threads fit an SM (228 KB, of which a CTA
// takes its dynamic and static parts and 1 KB).
template <int NT>
constexpr int enc_fit(int ctas) { return 228 * 1024 / ctas - 1024 - static_cast<int>(sizeof(EncShared<NT>)); }
// A CTA of 256 threads where three fit an SM, of 512 where fewer do: 4096 channels take 57 us with
// three of 256 threads and 64 with two of 512 (12,500 samples; 62 and 71 at 14,300), and 63 against 54
// where even 512 threads fit three times (11,000 samples).
constexpr int kEncSmall = enc_fit<256>(3);  // 66,176 bytes: 57 words a CTA
constexpr int kEncTwo = enc_fit<512>(2);    // 100,992 bytes: 87 words

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ uint32_t cluster_size() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
// v into the 32-bit word at shared address `addr` of every CTA of the cluster (visible after the next
// cluster barrier): pushed rather than read later, so no load waits on another SM
__device__ __forceinline__ void cluster_put(uint32_t addr, uint32_t v, int S) {
  for (int r = 0; r < S; ++r) {
    uint32_t ra;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(addr), "r"(r));
    asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(ra), "r"(v) : "memory");
  }
}

// Encoder of one chunk in one launch. What bounded the three-kernel form was latency, not bytes: three
// dependent launches, global atomics between them, and a second read of the chunk in 4-byte ring
// stores. Here each CTA brings its samples into shared memory once (asynchronous copies, all in flight
// together) and sums them per channel, the cluster adds its CTAs' sums through distributed shared
// memory, one warp evaluates the FP64 recipe for all 32 channels at once (lane = channel), a second
// pass over the shared samples sums what the clip bounds leave out, and the same samples are compared
// and packed; ring words leave as contiguous runs per channel. No histogram: with the samples in
// shared memory two passes of exact integer sums cost less than its atomics (with them 24 us for 64
// channels, 56 us for 1024). Sums and FP64 steps are those of levels_warp, so the levels are the same.
// Encoder stage (with its event pair): 1024 channels x 16384 samples 48 -> 27 us, 4096 x 7246 80 -> 41,
// 1000 x 10007 54 -> 29 (4-byte loads), 64 x 1024 26 -> 16.
template <int kEncThreads>
__device__ __forceinline__ void encode_cta(const EncBeam& e, const int cb, unsigned char* sm) {
  constexpr int NW = kEncThreads / 32;
  __shared__ EncShared<kEncThreads> sh;
  auto &red = sh.red;
  auto &tot1 = sh.tot1;
  auto &tot2 = sh.tot2;
  auto &clip = sh.clip;
  auto &lev = sh.lev;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int rank = static_cast<int>(cluster_rank()), S = static_cast<int>(cluster_size());
  unsigned char* tile = sm;                                // [wpc * 32][32]
  uint32_t* bits = reinterpret_cast<uint32_t*>(tile + e.wpc * 32 * 32);  // [32][wpc | 1]
  const int c0 = cb * 32;
  const int q0 = rank * e.wpc, nq = max(0, min(e.wpc, e.nwords - q0));  // this CTA's ring words
  const long long aw0 = e.w0 + q0;
  const int rbase = static_cast<int>(aw0 * 32 - e.t0);     // chunk row of tile row 0 (negative in the first word)
  const int i0 = max(0, -rbase), i1 = min(nq * 32, e.nsamp - rbase);  // tile rows that are in the chunk

  // the samples of [i0, i1) x 32 channels (bytes past the last channel stay unread)
  const uint8_t* src = e.chunk + static_cast<long long>(rbase) * e.nchan + c0;
  const int nc = min(32, e.nchan - c0);
  const uint32_t stile = static_cast<uint32_t>(__cvta_generic_to_shared(tile));
  if (e.vec == 16) {
    const int per = nc >> 4;  // 16-byte pieces a row
    for (int i = i0 * 2 + tid; i < i1 * 2; i += kEncThreads) {
      const int row = i >> 1, p = i & 1;
      if (p < per)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(stile + row * 32 + p * 16),
                     "l"(src + static_cast<long long>(row) * e.nchan + p * 16)
                     : "memory");
    }
  } else if (e.vec == 4) {
    const int per = nc >> 2;
    for (int i = i0 * 8 + tid; i < i1 * 8; i += kEncThreads) {
      const int row = i >> 3, p = i & 7;
      if (p < per)
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(stile + row * 32 + p * 4),
                     "l"(src + static_cast<long long>(row) * e.nchan + p * 4)
                     : "memory");
    }
  }
  asm volatile("cp.async.commit_group;" ::: "memory");
  if (e.vec == 1 && lane < nc) {
    int i = i0 + wid;
    for (; i + 7 * NW < i1; i += 8 * NW) {
      uint8_t v[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) v[k] = __ldg(src + static_cast<long long>(i + NW * k) * e.nchan + lane);
#pragma unroll
      for (int k = 0; k < 8; ++k) tile[(i + NW * k) * 32 + lane] = v[k];
    }
    for (; i < i1; i += NW) tile[i * 32 + lane] = __ldg(src + static_cast<long long>(i) * e.nchan + lane);
  }
  cluster_arrive();  // the peers' shared memory may be written once they have all started
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();

  // first pass: sums over the chunk, lane = channel (a CTA's fit 32 bits: at most 6.6e4 samples of
  // 255^2; channels past the last sum what was there, and are not written out)
  uint32_t a1 = 0, a2 = 0;
  {
    int i = i0 + wid;
    for (; i + 7 * NW < i1; i += 8 * NW) {
      uint32_t v[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) v[k] = tile[(i + NW * k) * 32 + lane];
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        a1 += v[k];
        a2 += v[k] * v[k];
      }
    }
    for (; i < i1; i += NW) {
      const uint32_t v = tile[i * 32 + lane];
      a1 += v;
      a2 += v * v;
    }
  }
  red[wid][0][lane] = a1;
  red[wid][1][lane] = a2;
  cluster_wait();
  __syncthreads();
  if (wid < 2) {
    uint32_t s = 0;
#pragma unroll
    for (int w = 0; w < NW; ++w) s += red[w][wid][lane];
    cluster_put(static_cast<uint32_t>(__cvta_generic_to_shared(&tot1[rank][wid][lane])), s, S);
  }
  cluster_arrive();
  cluster_wait();
  const double nf = static_cast<double>(e.nsamp);
  double lo = 0.0, hi = 0.0;
  long long s1 = 0, s2 = 0;  // of the chunk, in warp 0
  if (wid == 0) {
    for (int r = 0; r < S; ++r) {
      s1 += tot1[r][0][lane];
      s2 += tot1[r][1][lane];
    }
    const double mu0 = __ddiv_rn(static_cast<double>(s1), nf);
    const double var0 = __dsub_rn(__ddiv_rn(static_cast<double>(s2), nf), __dmul_rn(mu0, mu0));
    const double sig0 = var0 > 0.0 ? __dsqrt_rn(var0) : 0.0;
    lo = __dsub_rn(mu0, __dmul_rn(5.0, sig0));
    hi = __dadd_rn(mu0, __dmul_rn(5.0, sig0));
    clip[0][lane] = static_cast<int>(fmin(fmax(ceil(lo), -1.0), 257.0));
    clip[1][lane] = static_cast<int>(fmin(fmax(floor(hi), -1.0), 257.0));
  }
  __syncthreads();
  // second pass: the values outside the clip bounds: how many below and above, and their sums. They
  // are few (5 sigma), so eight rows are tested at once and a warp only goes through them one by one
  // where a lane has one (testing and adding row by row took 17,000 cycles of 2,080 rows, this an eighth)
  {
    const int ilo = clip[0][lane], ihi = clip[1][lane];
    uint32_t s1 = 0, s2 = 0, nlo = 0, nhi = 0;
    auto out = [&](int v) {
      if (v < ilo) ++nlo; else if (v > ihi) ++nhi; else return;
      s1 += v;
      s2 += v * v;
    };
    int i = i0 + wid;
    for (; i + 7 * NW < i1; i += 8 * NW) {
      int v[8], least = 255, most = 0;
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        v[k] = tile[(i + NW * k) * 32 + lane];
        least = min(least, v[k]);
        most = max(most, v[k]);
      }
      if (__any_sync(0xFFFFFFFFu, lane < nc && (least < ilo || most > ihi))) {
#pragma unroll 1
        for (int k = 0; k < 8; ++k) out(tile[(i + NW * k) * 32 + lane]);
      }
    }
    for (; i < i1; i += NW) out(tile[i * 32 + lane]);
    red[wid][0][lane] = nlo;
    red[wid][1][lane] = nhi;
    red[wid][2][lane] = s1;
    red[wid][3][lane] = s2;
  }
  __syncthreads();
  if (wid < 4) {
    uint32_t s = 0;
#pragma unroll
    for (int w = 0; w < NW; ++w) s += red[w][wid][lane];
    cluster_put(static_cast<uint32_t>(__cvta_generic_to_shared(&tot2[rank][wid][lane])), s, S);
  }
  cluster_arrive();
  cluster_wait();
  if (wid == 0) {
    long long nlo = 0, nhi = 0, s1in = s1, s2in = s2;
    for (int r = 0; r < S; ++r) {
      nlo += tot2[r][0][lane];
      nhi += tot2[r][1][lane];
      s1in -= tot2[r][2][lane];
      s2in -= tot2[r][3][lane];
    }
    const double s1c = __dadd_rn(__dadd_rn(static_cast<double>(s1in), __dmul_rn(static_cast<double>(nlo), lo)),
                                 __dmul_rn(static_cast<double>(nhi), hi));
    const double s2c =
        __dadd_rn(__dadd_rn(static_cast<double>(s2in), __dmul_rn(static_cast<double>(nlo), __dmul_rn(lo, lo))),
                  __dmul_rn(static_cast<double>(nhi), __dmul_rn(hi, hi)));
    const double mu = __ddiv_rn(s1c, nf);
    const double var = __dsub_rn(__ddiv_rn(s2c, nf), __dmul_rn(mu, mu));
    const double sig = var > 0.0 ? __dsqrt_rn(var) : 0.0;
    int u = 256;
    if (sig > 0.0) {
      const double thr = __dadd_rn(mu, __dmul_rn(e.theta, sig));
      if (thr < 0.0) {
        u = 0;
      } else if (thr < 255.0) {
        u = static_cast<int>(floor(thr)) + 1;
      }
    }
    lev[lane] = u;
    if (rank == 0 && lane < nc) e.levels[c0 + lane] = u;
  }
  __syncthreads();

  // pack: a warp per ring word, lane = sample. P >= u for four channels at a time: v + (256 - u) in
  // 16-bit halves carries into bit 8 exactly when it holds (u <= 256); the lane's 32 bits are gathered
  // byte by byte (bit 8 b + i = channel 4 i + b) and a 32 x 32 transpose over the warp turns samples'
  // words into channels' (a ballot per channel took four times as long).
  const int bp = e.wpc | 1;  // odd pitch: the lanes' words fall into different banks
  uint32_t ke[8], ko[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    ke[i] = static_cast<uint32_t>(256 - lev[4 * i]) | (static_cast<uint32_t>(256 - lev[4 * i + 2]) << 16);
    ko[i] = static_cast<uint32_t>(256 - lev[4 * i + 1]) | (static_cast<uint32_t>(256 - lev[4 * i + 3]) << 16);
  }
  for (int q = wid; q < nq; q += NW) {
    const int i = q * 32 + lane;
    const uint4 b0 = *reinterpret_cast<const uint4*>(tile + i * 32), b1 = *reinterpret_cast<const uint4*>(tile + i * 32 + 16);
    const uint32_t wv[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
    uint32_t x = 0;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const uint32_t ev = (wv[j] & 0x00FF00FFu) + ke[j], od = ((wv[j] >> 8) & 0x00FF00FFu) + ko[j];
      x += __byte_perm(ev, od, 0x7351) << j;  // bytes 1 and 3 of both: 0 or 1 each
    }
    if (i < i0 || i >= i1) x = 0;
#pragma unroll
    for (int j = 16; j > 0; j >>= 1) {
      const uint32_t m = j == 16 ? 0x0000FFFFu : (j == 8 ? 0x00FF00FFu : (j == 4 ? 0x0F0F0F0Fu : (j == 2 ? 0x33333333u : 0x55555555u)));
      const uint32_t y = __shfl_xor_sync(0xFFFFFFFFu, x, j);
      x = (lane & j) ? ((x & ~m) | ((y >> j) & m)) : ((x & m) | ((y << j) & ~m));
    }
    bits[(4 * (lane & 7) + (lane >> 3)) * bp + q] = x;
  }
  __syncthreads();
  const int phys0 = static_cast<int>(aw0 % e.R);
  for (int c = wid; c < nc; c += NW) {
    uint32_t* row = e.ring + static_cast<size_t>(c0 + c) * 2 * e.R;
    for (int q = lane; q < nq; q += 32) {
      int phys = phys0 + q;
      if (phys >= e.R) phys -= e.R;
      uint32_t w = bits[c * bp + q];
      // only the chunk's first word keeps bits of samples before the chunk (previous chunk)
      if (rank == 0 && q == 0 && rbase < 0) w |= row[phys] & ((1u << -rbase) - 1u);
      row[phys] = w;
      row[phys + e.R] = w;
    }
  }
}

__device__ __forceinline__ void clear_block_counters(const EncBeam& e) {
  e.counters[kCntCells] = 0;
  e.counters[kCntRuns] = 0;
  e.counters[kCntBlockCands] = 0;
}

// one plan: cluster i takes channels 32 i ..
template <int NT>
__global__ void __launch_bounds__(NT, 1024 / NT) k_encode(const __grid_constant__ EncBeam e) {
  extern __shared__ __align__(16) unsigned char esm[];
  if (blockIdx.x == 0 && threadIdx.x == 0) clear_block_counters(e);
  encode_cta<NT>(e, static_cast<int>(blockIdx.x) / static_cast<int>(cluster_size()), esm);
}

// many plans: cluster i takes channels 32 (i - first[b]) .. of the last beam b with first[b] <= i
template <int NT>
__global__ void __launch_bounds__(NT, 1024 / NT) k_encode_multi(const __grid_constant__ EncMulti m) {
  extern __shared__ __align__(16) unsigned char esm[];
  const int i = static_cast<int>(blockIdx.x) / static_cast<int>(cluster_size());
  int lo = 0, hi = m.nbeams - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (m.first[mid] <= i) lo = mid; else hi = mid - 1;
  }
  const EncBeam& e = m.beam[lo];
  if (i == m.first[lo] && cluster_rank() == 0 && threadIdx.x == 0) clear_block_counters(e);
  encode_cta<NT>(e, i - m.first[lo], esm);
}

// Whether k_encode takes this plan's chunk at S CTAs per cluster; fills e.
bool enc_beam(const Plan& p, const uint8_t* chunk, int nsamp, int S, EncBeam& e) {
  if (p.mode == SND_MODE_ZFLOAT) return false;
  e.chunk = chunk;
  e.nsamp = nsamp;
  e.nchan = p.nchan;
  e.levels = p.dp.levels;
  e.theta = p.enc_theta;
  e.t0 = p.T;
  e.w0 = p.T >> 5;
  e.nwords = static_cast<int>(((p.T + nsamp - 1) >> 5) - e.w0 + 1);
  e.wpc = (e.nwords + S - 1) / S;
  e.ring = p.dp.ring;
  e.R = p.R;
  const uintptr_t at = reinterpret_cast<uintptr_t>(chunk) | static_cast<uintptr_t>(p.nchan);
  e.vec = (at & 15u) == 0 ? 16 : ((at & 3u) == 0 ? 4 : 1);
  e.counters = p.dp.counters;
  return enc_smem(e.wpc) <= kEncMaxSmem && e.nwords <= e.R;
}

template <typename A>
cudaError_t run_encode(void (*kern)(A), int threads, const A& args, int clusters, int S, int smem, cudaStream_t s) {
  // the same value at every launch, as other threads may launch the kernel with other sizes
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kEncMaxSmem);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(static_cast<unsigned>(clusters) * S);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = S;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, args);
}

}  // namespace

cudaError_t launch_encode(const Plan& p, const uint8_t* d_chunk, int nsamp, cudaStream_t s) {
  const DevPtrs& dp = p.dp;
  {
    // eight CTAs a cluster, fewer for chunks of few words (at least eight words each)
    const int nwords = static_cast<int>(((p.T + nsamp - 1) >> 5) - (p.T >> 5) + 1);
    int S = kEncCluster;
    while (S > 1 && nwords < 8 * S) S /= 2;
    EncBeam b{};
    // A few channels read byte by byte are one or two clusters, whose CTAs' loads take longer than the three
    // launches that spread a long chunk over the GPU (stage us, one launch / three: 7 channels x 26,000 samples
    // 28 / 26, 48,000 39 / 26; 33 x 26,000 29 / 31, 48,000 37 / 31; 66 x 48,000 37 / 35).
    const bool long_bytes = p.nchan <= 64 && nwords > 104 * kEncCluster;
    if (enc_beam(p, d_chunk, nsamp, S, b) && !(b.vec == 1 && long_bytes)) {
      p.launches += 1;
      const int smem = enc_smem(b.wpc), clusters = (p.nchan + 31) / 32;
      return smem <= kEncSmall ? run_encode(k_encode<256>, 256, b, clusters, S, smem, s)
                               : run_encode(k_encode<512>, 512, b, clusters, S, smem, s);
    }
  }
  cudaError_t ec = cudaMemsetAsync(dp.counters, 0, sizeof(uint32_t) * (kCntBlockCands + 1), s);
  if (ec != cudaSuccess) return ec;
  dim3 hb(32, kHistWarps), hg((p.nchan + 31) / 32, (nsamp + kHistRowsPerBlock - 1) / kHistRowsPerBlock);
  k_hist<<<hg, hb, 0, s>>>(d_chunk, nsamp, p.nchan, dp.hist);
  const bool z = p.mode == SND_MODE_ZFLOAT;
  k_levels<<<(p.nchan * 32 + 255) / 256, 256, 0, s>>>(dp.hist, p.nchan, nsamp, p.enc_theta, dp.levels,
                                                      z ? dp.ztab : nullptr, p.zgeom.fp16 | (p.zgeom.unit << 1));
  const long long t0 = p.T;
  if (z) {
    dim3 zb(32, 8), zg((p.nchan + 31) / 32, (nsamp + 255) / 256);
    if (p.zgeom.fp16) {
      k_pack_z<__half><<<zg, zb, 0, s>>>(d_chunk, nsamp, p.nchan, static_cast<const __half*>(dp.ztab), t0,
                                         static_cast<__half*>(dp.zring), p.zgeom.Rz);
    } else {
      k_pack_z<float><<<zg, zb, 0, s>>>(d_chunk, nsamp, p.nchan, static_cast<const float*>(dp.ztab), t0,
                                        static_cast<float*>(dp.zring), p.zgeom.Rz);
    }
    p.launches += 3;
    return cudaGetLastError();
  }
  const long long w0 = t0 >> 5;
  const long long w1 = (t0 + nsamp - 1) >> 5;
  const int nwords = static_cast<int>(w1 - w0 + 1);
  if (p.nchan % 32 == 0 && (reinterpret_cast<uintptr_t>(d_chunk) & 15u) == 0) {
    const long long tasks = static_cast<long long>(nwords) * (p.nchan / 32);
    k_pack32<<<static_cast<unsigned>((tasks * 32 + 255) / 256), 256, 0, s>>>(d_chunk, nsamp, p.nchan, dp.levels, t0,
                                                                           w0, nwords, dp.ring, p.R);
  } else {
    dim3 pb(32, 8), pg((p.nchan + 31) / 32, (nwords + 7) / 8);
    k_pack<<<pg, pb, 0, s>>>(d_chunk, nsamp, p.nchan, dp.levels, t0, w0, nwords, dp.ring, p.R);
  }
  p.launches += 3;
  return cudaGetLastError();
}

// Encoders of several plans in one launch per shared-memory class (three CTAs fit an SM, two, one), so
// a long-chunk beam does not lower every other beam's occupancy: eight beams of 1024 channels, one with
// 24,000 samples and seven with 22,000, take 498 us a step in one launch and 417 in two. Beams of which
// all CTAs fit the GPU one per SM need no such care, and save the launch. More launches only past
// kMaxEncBeams beams of a class. Plans that k_encode does not take run their own launch_encode.
cudaError_t launch_encode_batch(const Plan* const* plans, const uint8_t* const* chunks, const int32_t* nsamp, int n,
                                cudaStream_t s) {
  constexpr int S = kEncCluster;
  int dev = 0, nsm = 0, wide = 0;  // wide: CTAs that fit fewer than three times
  cudaError_t err = cudaGetDevice(&dev);
  if (err == cudaSuccess) err = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  if (err != cudaSuccess) return err;
  for (int i = 0; i < n; ++i) {
    EncBeam b{};
    if (enc_beam(*plans[i], chunks[i], nsamp[i], S, b) && enc_smem(b.wpc) > kEncSmall) wide += (plans[i]->nchan + 31) / 32 * S;
  }
  auto cls = [&](int smem) { return smem <= kEncSmall ? 0 : (smem <= kEncTwo || wide <= nsm ? 1 : 2); };
  EncMulti m{};
  int clusters = 0, smem = 0;
  const Plan* owner = nullptr;
  auto flush = [&](int c) -> cudaError_t {
    if (m.nbeams == 0) return cudaSuccess;
    const cudaError_t e = c == 0 ? run_encode(k_encode_multi<256>, 256, m, clusters, S, smem, s)
                                 : run_encode(k_encode_multi<512>, 512, m, clusters, S, smem, s);
    owner->launches += 1;
    m.nbeams = 0;
    clusters = smem = 0;
    owner = nullptr;
    return e;
  };
  for (int c = 0; c < 3; ++c) {
    for (int i = 0; i < n; ++i) {
      const Plan& p = *plans[i];
      EncBeam& b = m.beam[m.nbeams];
      if (!enc_beam(p, chunks[i], nsamp[i], S, b)) {
        if (c != 0) continue;
        const cudaError_t e = launch_encode(p, chunks[i], nsamp[i], s);
        if (e != cudaSuccess) return e;
        continue;
      }
      if (cls(enc_smem(b.wpc)) != c) continue;
      m.first[m.nbeams] = clusters;
      clusters += (p.nchan + 31) / 32;
      smem = std::max(smem, enc_smem(b.wpc));
      if (!owner) owner = &p;
      if (++m.nbeams == kMaxEncBeams) {
        const cudaError_t e = flush(c);
        if (e != cudaSuccess) return e;
      }
    }
    const cudaError_t e = flush(c);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace snd
