// K2s, resident form: domain selection (Sec. III-B) for CSR couplings whose
// state fits the chip. Restarts are independent, so a CTA takes RB of them
// and keeps everything they need in shared memory for a whole run of steps:
// theta, m and v, the spins (two buffers: 16 bits per restart and site in the
// form the sums take them, or one bit when that is all the room there is)
// and, when there is room, the couplings. A step then touches no
// global memory and waits for no other CTA: one launch runs all the steps
// that the launch-per-step form takes two launches each for.
//
// What bounds it: instruction issue when RB n is large (about 75 per spin
// update, and 6 per coupling of a site whatever the restarts: the coupling's
// word, its column and value, the neighbour's spins, a multiply-add per pair
// of restarts), the latency of one gather, update and CTA barrier when it is
// small.
//
// Couplings are stored as slices of 32 rows (the rows one warp takes
// together), entry k of the slice's 32 rows side by side, padded with zero
// couplings to the slice's longest row: one conflict-free 32-bit load per
// lane and coupling. Padding adds +-0 to a row's sum, which changes nothing.
//
// Results are those of the launch-per-step form bit for bit. Integer sums are
// exact. In FP32 a thread takes the rows that one warp of that form takes (8
// warps per block of `rpb` rows), in the same order, the 8 partial sums of a
// block are added in warp order, and the blocks' in FP64 in track_kernel's
// order. A dedicated warp turns the partials of step s - 1 into energies and
// bests while the others run step s; every thread keeps the spins of its
// sites at the best step as register bits, as the small tensor-core form does.
#include "ds_internal.cuh"

#include <algorithm>
#include <cmath>

namespace ising {

struct SparseRes {
  int rb = 1;           // restarts per CTA (1, 2, 4 or 8)
  int nt = 32;          // threads that own sites (a tracking warp comes on top)
  int rpb = 8, kr = 1;  // rows per block of partial sums, rows per thread and pass
  int passes = 1;
  int nvb = 1;          // blocks of partial sums
  int slices = 1;
  DevMem ell, off;
  int64_t entries = 0;  // coupling slots, padding included
  bool pack = true;     // spins as 16 bits per restart and site, else as bits
  bool ell_smem = false;
  size_t smem = 0;
};

namespace {

struct SrArgs {
  int n;
  int64_t B, Bp;
  int nt, rpb, kr, passes, nvb, slices;
  int64_t entries;
  // shared-memory offsets in bytes (passed, not derived in the kernel: under
  // register pressure the compiler would derive them again in every step)
  int spins, buffer, part, off_at, ell_at;
  const uint32_t* ell;  // V8: column | value << 24; else pairs (column, FP32 bits)
  const int* off;       // slice offsets in entries of 32 lanes
  int steps;
  long long t0, T;
  StepConsts k;
  const float2* bias;
  float *theta, *m, *v;  // [n][Bp]
  const float* hf;       // null: no field
  const int32_t* hint;
  uint32_t* bits_out;    // the next step's spins, zeroed
  double cq, chs;
  double* best_E;
  long long* best_t;
  int8_t* best_s;
  int64_t bs_ld;
  double* last_E;
  long long* counters;
  double *conv_ring, *conv_init;  // convergence rule, or null
  long long* conv_step;
  unsigned long long* conv_count;
  int* live32;
};

// Shared-memory layout (bytes).
struct SrLayout {
  size_t spins, part, off, ell, total;
  size_t buffer;  // bytes of one spin buffer
  SrLayout(int n, int rb, int nvb, int slices, int64_t entries, int ebytes,
                               bool int_e, bool pack, bool ell_smem) {
    buffer = ((size_t)n * (pack ? 2 * rb : 1) + 15) / 16 * 16;
    spins = 12 * (size_t)n * rb;
    spins = (spins + 15) / 16 * 16;
    part = spins + 2 * buffer;
    // INT: q and h, [2 slots][32 warps][rb]; else [2 slots][nvb][rb]
    const size_t pb = int_e ? (size_t)2 * 2 * 32 * rb * 4 : (size_t)2 * nvb * rb * 4;
    off = part + (pb + 15) / 16 * 16;
    ell = off + (((size_t)slices + 1) * 4 + 15) / 16 * 16;
    total = ell + (ell_smem ? (size_t)entries * ebytes : 0);
  }
};

// Threads of a CTA at most: with 4 or 8 restarts a thread has enough to do at
// half the warps, and needs the registers (64 spill).
__host__ __device__ constexpr int sr_threads(int rb) { return rb >= 4 ? 512 : 1024; }

// The row of thread `tid`, pass p, k-th row (or -1).
__host__ __device__ __forceinline__ int sr_row(int n, int nt, int rpb, int tid, int p, int k) {
  const int vw = p * nt + tid;
  if (rpb == 8) return vw < n ? vw : -1;  // (one row per thread and pass)
  const int w = vw & 7;
  const int64_t row = (int64_t)(vw >> 3) * rpb + w + 8 * k;
  return w + 8 * k < rpb && row < n ? (int)row : -1;
}

// The spins of one site's RB restarts as 16-bit words, two to a register:
// V8 (integer sums) +-1 as s_0 + 65536 s_1, so that adding value x word sums
// both restarts at once; else BF16 +-1, each a shift or a mask away from FP32.
template <int RB, bool V8>
struct SpinWords {
  static constexpr int W = (RB + 1) / 2;
  uint32_t w[W];
  __device__ __forceinline__ explicit SpinWords(uint32_t bits) {
#pragma unroll
    for (int k = 0; k < W; ++k) {
      const uint32_t b0 = (bits >> (2 * k)) & 1u, b1 = (bits >> (2 * k + 1)) & 1u;
      if (V8) w[k] = (2u * b0 - 1u) + (RB > 1 ? (2u * b1 - 1u) << 16 : 0u);
      else w[k] = (b0 ? 0x3F80u : 0xBF80u) | (b1 ? 0x3F800000u : 0xBF800000u);
    }
  }
  __device__ __forceinline__ SpinWords(const uint8_t* buf, int site) {
    if constexpr (RB == 1) w[0] = V8 ? (uint32_t)(int)reinterpret_cast<const int16_t*>(buf)[site]
                                     : reinterpret_cast<const uint16_t*>(buf)[site];
    else if constexpr (RB == 2) w[0] = reinterpret_cast<const uint32_t*>(buf)[site];
    else if constexpr (RB == 4) {
      const uint2 x = reinterpret_cast<const uint2*>(buf)[site];
      w[0] = x.x; w[1] = x.y;
    } else {
      const uint4 x = reinterpret_cast<const uint4*>(buf)[site];
      w[0] = x.x; w[1] = x.y; w[2] = x.z; w[3] = x.w;
    }
  }
  __device__ __forceinline__ void store(uint8_t* buf, int site) const {
    if constexpr (RB == 1) reinterpret_cast<uint16_t*>(buf)[site] = (uint16_t)w[0];
    else if constexpr (RB == 2) reinterpret_cast<uint32_t*>(buf)[site] = w[0];
    else if constexpr (RB == 4) reinterpret_cast<uint2*>(buf)[site] = make_uint2(w[0], w[1]);
    else reinterpret_cast<uint4*>(buf)[site] = make_uint4(w[0], w[1], w[2], w[3]);
  }
};

template <int RB, bool V8, bool PACK>
__device__ __forceinline__ void store_spins(uint8_t* buf, int site, uint32_t bits) {
  if constexpr (PACK) SpinWords<RB, V8>(bits).store(buf, site);
  else buf[site] = (uint8_t)bits;
}

template <int RB, bool V8, bool PACK>
__device__ __forceinline__ SpinWords<RB, V8> load_spins(const uint8_t* buf, int site) {
  if constexpr (PACK) return SpinWords<RB, V8>(buf, site);
  else return SpinWords<RB, V8>((uint32_t)buf[site]);
}

// ELLS: the couplings are in shared memory too (a pointer that may be either
// costs 64-bit address arithmetic and generic loads per coupling).
template <int RB, bool INT_E, bool V8, bool PACK, bool ELLS>
__global__ void __launch_bounds__(sr_threads(RB), 1) sparse_res_kernel(const SrArgs A) {
  extern __shared__ __align__(16) uint8_t smem[];
  __shared__ uint32_t imp[2], alldone[2];
  __shared__ float2 corr[2];  // Adam's bias corrections, slot s mod 2
  // integer energies need no particular order: one row per thread and pass
  const int kr = INT_E ? 1 : A.kr;
  auto row_of = [&](int p, int k) {
    if (!INT_E) return sr_row(A.n, A.nt, A.rpb, (int)threadIdx.x, p, k);
    const int i = p * A.nt + (int)threadIdx.x;
    return i < A.n ? i : -1;
  };
  const int n = A.n, nt = A.nt, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  float* sth = reinterpret_cast<float*>(smem);  // [RB][n]
  float* smm = sth + RB * n;
  float* svv = smm + RB * n;
  uint8_t* sp = smem + A.spins;  // two buffers
  int* pq = reinterpret_cast<int*>(smem + A.part);  // INT: [2][32][RB], then h
  int* ph = pq + 2 * 32 * RB;
  float* bs = reinterpret_cast<float*>(smem + A.part);  // else [2][nvb][RB]
  int* soff = reinterpret_cast<int*>(smem + A.off_at);
  const int64_t b0 = (int64_t)blockIdx.x * RB;
  const bool site = tid < nt;  // (the last warp tracks)
  const int nidx = A.passes * kr;
  const int nwarps = nt / 32;

  // the couplings, offsets and state of this CTA's restarts
  for (int e = tid; e <= A.slices; e += blockDim.x) soff[e] = A.off[e];
  if (ELLS) {
    const uint4* src = reinterpret_cast<const uint4*>(A.ell);
    uint4* dst = reinterpret_cast<uint4*>(smem + A.ell_at);
    for (int64_t e = tid; e < A.entries * (V8 ? 4 : 8) / 16; e += blockDim.x) dst[e] = src[e];
  }
  if (tid < 2) alldone[tid] = 0, imp[tid] = 0;
  // bit idx RB + r of these words: site idx of this thread, restart r. The
  // spins of the step to come, of the last two steps, of the best step, and
  // which sites the best ones were set for
  uint32_t next_bits = 0, prev_bits = 0, prev2_bits = 0, best_bits = 0, any_bits = 0, rep = 0;
  if (site)
    for (int idx = 0; idx < nidx; ++idx) {
      rep |= 1u << (idx * RB);
      const int i = row_of(idx / kr, idx % kr);
      if (i < 0) continue;
      const int64_t g = (int64_t)i * A.Bp + b0;
      uint32_t byte = 0;
#pragma unroll
      for (int r = 0; r < RB; ++r) {
        const float th = A.theta[g + r];
        sth[r * n + i] = th;
        smm[r * n + i] = A.m[g + r];
        svv[r * n + i] = A.v[g + r];
        byte |= (sin_nonneg(th) ? 1u : 0u) << r;
      }
      store_spins<RB, V8, PACK>(sp, i, byte);
      next_bits |= byte << (idx * RB);
    }
  // tracking lane r: restart b0 + r
  const int64_t b = b0 + lane;
  const bool mine = !site && lane < RB && b < A.B;
  double bE = 0.0, lE = 0.0, win[5] = {0, 0, 0, 0, 0}, E1 = 0.0;
  long long bT = 0;
  bool stopped = !mine, was_stopped = !mine;
  if (mine) {
    bE = A.best_E[b];
    lE = A.last_E[b];
    bT = A.best_t[b];
    if (A.conv_step) {
      stopped = was_stopped = A.conv_step[b] != 0;
      E1 = A.conv_init[b];
#pragma unroll
      for (int j = 0; j < 5; ++j) {
        const long long tt = A.t0 - 4 + j;
        if (tt >= 1) win[j] = A.conv_ring[(tt - 1) % 5 * A.B + b];
      }
    }
  }
  __syncthreads();
  if (!site && A.conv_step) {
    const bool all = __all_sync(0xffffffffu, stopped);
    if (lane == 0 && all) alldone[0] = 1;
  }
  __syncthreads();
  const bool retired = alldone[0] != 0;  // every restart stopped before this launch
  __syncthreads();
  if (tid == 0) alldone[0] = 0;

  // Energies and bests of step index e, by the tracking warp.
  auto track = [&](int e) {
    const int slot = e & 1;
    const long long t = A.t0 + e + 1;
    double E = 0.0;
    if (INT_E) {
#pragma unroll
      for (int r = 0; r < RB; ++r) {
        const int q = __reduce_add_sync(0xffffffffu, lane < nwarps ? pq[(slot * 32 + lane) * RB + r] : 0);
        int h = 0;
        if (A.hf) h = __reduce_add_sync(0xffffffffu, lane < nwarps ? ph[(slot * 32 + lane) * RB + r] : 0);
        if (lane == r) E = A.cq * (double)q + A.chs * (double)h;
      }
    } else {
      // (the restarts' FP64 chains side by side: one after another they were
      // the longest part of a step)
      double x[RB];
#pragma unroll
      for (int r = 0; r < RB; ++r) x[r] = 0.0;
      for (int c = lane; c < A.nvb; c += 32)
#pragma unroll
        for (int r = 0; r < RB; ++r) x[r] += (double)bs[(slot * A.nvb + c) * RB + r];
#pragma unroll
      for (int o = 16; o; o >>= 1)
#pragma unroll
        for (int r = 0; r < RB; ++r) x[r] += __shfl_xor_sync(0xffffffffu, x[r], o);
#pragma unroll
      for (int r = 0; r < RB; ++r)
        if (lane == r) E = x[r];
    }
    bool better = false;
    if (!stopped) {
      lE = E;
      better = E < bE;
      if (better) {
        bE = E;
        bT = t;
      }
      if (A.conv_step && t <= A.T) {
        // (conv_update, with the window in registers)
        win[0] = win[1]; win[1] = win[2]; win[2] = win[3]; win[3] = win[4]; win[4] = E;
        if (t == 1) E1 = E;
        if (t >= 5) {
          const double mx = fmax(fmax(fmax(win[0], win[1]), fmax(win[2], win[3])), win[4]);
          const double mn = fmin(fmin(fmin(win[0], win[1]), fmin(win[2], win[3])), win[4]);
          if (mx - mn <= kConvTol * fabs(E - E1)) {
            stopped = true;
            A.conv_step[b] = t;
            atomicAdd(A.conv_count, 1ull);
            atomicSub(&A.live32[b >> 5], 1);
          }
        }
      }
    }
    const uint32_t bits = __ballot_sync(0xffffffffu, better);
    if (lane == 0) imp[slot] = bits;
    if (A.conv_step) {
      const bool all = __all_sync(0xffffffffu, stopped);
      if (lane == 0 && all) alldone[(e + 1) & 1] = 1;
    }
  };

  const float2* bias = A.bias + A.t0 + 1;  // of step index 0
  if (!site && lane == 0) corr[0] = bias[0];
  __syncthreads();
  int s = 0;
  bool early = false;
  if (!retired)
    for (; s < A.steps; ++s) {
      const int cur = s & 1;
      const uint8_t* spc = sp + cur * A.buffer;
      uint8_t* spn = sp + (cur ^ 1) * A.buffer;
      if (!site) {
        if (lane == 0 && s + 1 < A.steps) corr[cur ^ 1] = bias[s + 1];
        if (s >= 1) track(s - 1);
      } else {
        const float2 bcs = corr[cur];
        if (s >= 2) {
          const uint32_t mk = imp[cur] * rep;  // the bests of step s - 2
          best_bits = (best_bits & ~mk) | (prev2_bits & mk);
          any_bits |= mk;
        }
        prev2_bits = prev_bits;
        prev_bits = next_bits;
        next_bits = 0;
        int eq[RB], eh[RB];
#pragma unroll
        for (int r = 0; r < RB; ++r) eq[r] = eh[r] = 0;
        for (int p = 0; p < A.passes; ++p) {
          float ee[RB];
#pragma unroll
          for (int r = 0; r < RB; ++r) ee[r] = 0.f;
          for (int k = 0; k < kr; ++k) {
            const int idx = p * kr + k;
            const int i = row_of(p, k);
            const int sl = idx * nwarps + warp;
            const int cnt = soff[sl + 1] - soff[sl], e0 = soff[sl] * 32 + lane;
            float G[RB];
            int Gi[RB];
            if constexpr (V8) {
              constexpr int W = (RB + 1) / 2;
              int P[W];
#pragma unroll
              for (int w = 0; w < W; ++w) P[w] = 0;
              const uint32_t* en = (ELLS ? reinterpret_cast<const uint32_t*>(smem + A.ell_at) : A.ell) + e0;
#pragma unroll 4
              for (int e = 0; e < cnt; ++e, en += 32) {
                const uint32_t x = *en;
                const int val = (int)x >> 24;
                const SpinWords<RB, V8> y = load_spins<RB, V8, PACK>(spc, (int)(x & 0xFFFFFFu));
#pragma unroll
                for (int w = 0; w < W; ++w) P[w] += (int)y.w[w] * val;
              }
#pragma unroll
              for (int r = 0; r < RB; ++r) {
                const int lo = (int)(int16_t)(P[r / 2] & 0xFFFF);
                Gi[r] = RB == 1 ? P[0] : ((r & 1) ? (P[r / 2] - lo) >> 16 : lo);
                G[r] = (float)Gi[r];
              }
            } else {
#pragma unroll
              for (int r = 0; r < RB; ++r) G[r] = 0.f;
              const uint2* en = reinterpret_cast<const uint2*>(
                  ELLS ? reinterpret_cast<const uint32_t*>(smem + A.ell_at) : A.ell) + e0;
#pragma unroll 4
              for (int e = 0; e < cnt; ++e, en += 32) {
                const uint2 x = *en;
                const SpinWords<RB, V8> y = load_spins<RB, V8, PACK>(spc, (int)x.x);
                const float J = __uint_as_float(x.y);
                // G + J s, one rounding, as G + (s > 0 ? J : -J)
#pragma unroll
                for (int r = 0; r < RB; ++r)
                  G[r] = fmaf(J, __uint_as_float((r & 1) ? y.w[r / 2] & 0xFFFF0000u : y.w[r / 2] << 16), G[r]);
              }
#pragma unroll
              for (int r = 0; r < RB; ++r) Gi[r] = INT_E ? __float2int_rn(G[r]) : 0;
            }
            if (i < 0) continue;
            const uint32_t own = prev_bits >> (idx * RB);
            const float h = A.hf ? __ldg(A.hf + i) : 0.f;
            const int hi = INT_E && A.hf ? __ldg(A.hint + i) : 0;
            uint32_t byte = 0;
#pragma unroll
            for (int r = 0; r < RB; ++r) {
              const bool up = (own >> r) & 1u;
              const float sg = up ? 1.f : -1.f;
              if (INT_E) {
                eq[r] += up ? Gi[r] : -Gi[r];
                eh[r] += up ? hi : -hi;
              } else {
                ee[r] += sg * fmaf(A.k.cq, G[r], A.k.ch * h);
              }
              const float F = fmaf(A.k.cq, G[r], fmaf(A.k.ch, h, -A.k.mu * sg));
              float th = sth[r * n + i], m = smm[r * n + i], v = svv[r * n + i];
              const float g = cos_proj(th) * F;
              th = adam_update(A.k, bcs.x, bcs.y, g, th, m, v);
              sth[r * n + i] = th;
              smm[r * n + i] = m;
              svv[r * n + i] = v;
              byte |= (sin_nonneg(th) ? 1u : 0u) << r;
            }
            store_spins<RB, V8, PACK>(spn, i, byte);
            next_bits |= byte << (idx * RB);
          }
          if (!INT_E) {
            // the 8 rows' sums of a block in warp order
            const int vb = (p * nt + tid) >> 3;
#pragma unroll
            for (int r = 0; r < RB; ++r) {
              float a = __shfl_sync(0xffffffffu, ee[r], lane & ~7);
#pragma unroll
              for (int w = 1; w < 8; ++w) a += __shfl_sync(0xffffffffu, ee[r], (lane & ~7) + w);
              if ((lane & 7) == 0 && vb < A.nvb) bs[(cur * A.nvb + vb) * RB + r] = a;
            }
          }
        }
        if (INT_E) {
#pragma unroll
          for (int r = 0; r < RB; ++r) {
            const int q = __reduce_add_sync(0xffffffffu, eq[r]);
            const int hs = A.hf ? __reduce_add_sync(0xffffffffu, eh[r]) : 0;
            if (lane == 0) {
              pq[(cur * 32 + warp) * RB + r] = q;
              ph[(cur * 32 + warp) * RB + r] = hs;
            }
          }
        }
      }
      __syncthreads();
      // (alldone[cur] is written at step s only, by the tracking of s - 1)
      if (alldone[cur]) {
        early = true;
        break;
      }
    }
  // the last step's energies (none when every restart stopped before it),
  // then the bests of the last two steps
  const int last = early ? s : s - 1;  // index of the last step computed
  if (!retired) {
    if (!site && !early) track(last);
    __syncthreads();
    if (site) {
      if (last >= 1) {
        const uint32_t mk = imp[(last - 1) & 1] * rep;
        best_bits = (best_bits & ~mk) | (prev2_bits & mk);
        any_bits |= mk;
      }
      if (!early) {
        const uint32_t mk = imp[last & 1] * rep;
        best_bits = (best_bits & ~mk) | (prev_bits & mk);
        any_bits |= mk;
      }
    }
  }
  if (site)
    for (int idx = 0; idx < nidx; ++idx) {
      const int i = row_of(idx / kr, idx % kr);
      if (i < 0) continue;
      const int64_t g = (int64_t)i * A.Bp + b0;
#pragma unroll
      for (int r = 0; r < RB; ++r) {
        if (!retired) {
          A.theta[g + r] = sth[r * n + i];
          A.m[g + r] = smm[r * n + i];
          A.v[g + r] = svv[r * n + i];
        }
        if ((any_bits >> (idx * RB + r)) & 1u)
          A.best_s[(b0 + r) * A.bs_ld + i] = ((best_bits >> (idx * RB + r)) & 1u) ? 1 : -1;
      }
      const uint32_t bits = (next_bits >> (idx * RB)) & ((1u << RB) - 1u);
      atomicOr(&A.bits_out[(int64_t)i * (A.Bp / 32) + (b0 >> 5)], bits << (b0 & 31));
    }
  if (mine) {
    A.best_E[b] = bE;
    A.best_t[b] = bT;
    A.last_E[b] = lE;
    if (A.conv_step && !was_stopped) {
      A.conv_init[b] = E1;
      const long long te = A.t0 + A.steps;  // (a restart that stopped never reads its window again)
#pragma unroll
      for (int j = 0; j < 5; ++j)
        if (te - 4 + j >= 1) A.conv_ring[(te - 5 + j) % 5 * A.B + b] = win[j];
    }
  }
  if (blockIdx.x == 0 && tid == 0) A.counters[0] = A.t0 + A.steps;
}

// Restart-steps of a launch under the convergence rule, counted in the slices
// of 128 restarts in which the launch-per-step form retires them.
__global__ void sr_work_kernel(int64_t B, const long long* __restrict__ conv_step, long long t0,
                               long long steps, unsigned long long* work) {
  const int64_t c0 = (int64_t)blockIdx.x * 128, c1 = c0 + 128 < B ? c0 + 128 : B;
  __shared__ long long mx[4];
  const int64_t b = c0 + threadIdx.x;
  long long x = 0;
  if (b < c1) x = conv_step[b] ? conv_step[b] : 0x7fffffffffffffffll;
  for (int o = 16; o; o >>= 1) x = max(x, __shfl_xor_sync(0xffffffffu, x, o));
  if ((threadIdx.x & 31) == 0) mx[threadIdx.x >> 5] = x;
  __syncthreads();
  if (threadIdx.x == 0) {
    x = max(max(mx[0], mx[1]), max(mx[2], mx[3]));
    const long long done = min(max(x - t0, 0ll), steps);
    atomicAdd(work, (unsigned long long)(done * (c1 - c0)));
  }
}

// Longest row of each slice of 32 thread slots (entries of 32 lanes).
__global__ void sr_width_kernel(int n, int nt, int rpb, int kr, int slices,
                                const int32_t* __restrict__ rowptr, int* __restrict__ width) {
  const int lane = threadIdx.x & 31;
  const int sl = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (sl >= slices) return;
  const int idx = sl / (nt / 32), tid = sl % (nt / 32) * 32 + lane;
  const int i = sr_row(n, nt, rpb, tid, idx / kr, idx % kr);
  int d = i >= 0 ? rowptr[i + 1] - rowptr[i] : 0;
  d = __reduce_max_sync(0xffffffffu, d);
  if (lane == 0) {
    width[sl] = d;
    atomicMax(&width[slices + 1], d);  // the longest row of all
  }
}

// Exclusive prefix sums in place, off[slices] the total (one block).
__global__ void __launch_bounds__(1024) sr_scan_kernel(int slices, int* __restrict__ off) {
  __shared__ int part[32];
  __shared__ int carry;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (threadIdx.x == 0) carry = 0;
  __syncthreads();
  for (int base = 0; base < slices; base += 1024) {
    const int e = base + threadIdx.x;
    const int x = e < slices ? off[e] : 0;
    int y = x;
    for (int o = 1; o < 32; o <<= 1) {
      const int z = __shfl_up_sync(0xffffffffu, y, o);
      if (lane >= o) y += z;
    }
    if (lane == 31) part[warp] = y;
    __syncthreads();
    if (warp == 0) {
      int p = part[lane];
      for (int o = 1; o < 32; o <<= 1) {
        const int z = __shfl_up_sync(0xffffffffu, p, o);
        if (lane >= o) p += z;
      }
      part[lane] = p;
    }
    __syncthreads();
    const int before = carry + (warp ? part[warp - 1] : 0);
    if (e < slices) off[e] = before + y - x;
    __syncthreads();
    if (threadIdx.x == 1023) carry = before + y;
    __syncthreads();
  }
  if (threadIdx.x == 0) off[slices] = carry;
}

__global__ void sr_fill_kernel(int n, int nt, int rpb, int kr, int slices, bool v8,
                               const int32_t* __restrict__ rowptr, const int32_t* __restrict__ col,
                               const void* __restrict__ val, const int* __restrict__ off,
                               uint32_t* __restrict__ ell) {
  const int lane = threadIdx.x & 31;
  const int sl = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (sl >= slices) return;
  const int idx = sl / (nt / 32), tid = sl % (nt / 32) * 32 + lane;
  const int i = sr_row(n, nt, rpb, tid, idx / kr, idx % kr);
  const int a = i >= 0 ? rowptr[i] : 0, d = i >= 0 ? rowptr[i + 1] - a : 0;
  const int o0 = off[sl], w = off[sl + 1] - o0;
  for (int k = 0; k < w; ++k) {
    const int64_t e = ((int64_t)o0 + k) * 32 + lane;
    const uint32_t c = k < d ? (uint32_t)col[a + k] : 0u;
    if (v8) {
      const uint32_t x = k < d ? (uint8_t)static_cast<const int8_t*>(val)[a + k] : 0u;
      ell[e] = c | (x << 24);
    } else {
      const float x = k < d ? static_cast<const float*>(val)[a + k] : 0.f;
      reinterpret_cast<uint2*>(ell)[e] = make_uint2(c, __float_as_uint(x));
    }
  }
}

template <int RB, bool INT_E, bool V8, bool PACK>
int sr_launch(ising_ds* ds, const SparseRes* R, const SrArgs& a) {
  auto kern = R->ell_smem ? sparse_res_kernel<RB, INT_E, V8, PACK, true>
                          : sparse_res_kernel<RB, INT_E, V8, PACK, false>;
  ISING_CUDA(ds->ctx, cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                           (int)(ds->ctx->smem_optin - 1024)));
  kern<<<(unsigned)((ds->B + RB - 1) / RB), R->nt + 32, R->smem, ds->ctx->stream>>>(a);
  ISING_CUDA(ds->ctx, cudaGetLastError());
  return ISING_OK;
}

template <int RB, bool PACK>
int sr_launch_rb(ising_ds* ds, const SparseRes* R, const SrArgs& a) {
  if (ds->int_energy)
    return ds->sp_int8 ? sr_launch<RB, true, true, PACK>(ds, R, a) : sr_launch<RB, true, false, PACK>(ds, R, a);
  return ds->sp_int8 ? sr_launch<RB, false, true, PACK>(ds, R, a) : sr_launch<RB, false, false, PACK>(ds, R, a);
}

template <int RB>
int sr_launch_pack(ising_ds* ds, const SparseRes* R, const SrArgs& a) {
  return R->pack ? sr_launch_rb<RB, true>(ds, R, a) : sr_launch_rb<RB, false>(ds, R, a);
}

}  // namespace

static int sparse_res_layout(ising_ds* ds);

// Whether the session runs this form, and its operands. It does when the
// state of RB restarts fits a CTA's shared memory (n RB up to about 16300,
// 14300 with 16-bit spins), with RB the least of 1, 2, 4, 8 that gives every SM at most one CTA, or 8
// (several waves of CTAs then): the launch-per-step form costs at least two
// launches and an L2 round trip per coupling however small the instance.
// Where the operands find no room, the session takes a launch per step.
int sparse_res_setup(ising_ds* ds) {
  const int rc = sparse_res_layout(ds);
  return rc == ISING_ENOMEM ? ISING_OK : rc;
}

static int sparse_res_layout(ising_ds* ds) {
  ising_ctx* ctx = ds->ctx;
  if ((ds->p.flags & ISING_DS_STREAMING) || ds->relaxed()) return ISING_OK;
  const DevInstance& I = ds->inst;
  const int64_t n = ds->n, nnz = I.nnz;
  if (n > kSparseResMaxSpins || nnz > (1 << 24)) return ISING_OK;
  const bool v8 = ds->sp_int8;
  if (ds->int_energy) {
    // energies and fields are added in 32 bits
    if (I.j_absmax * (double)nnz >= 1073741824.0) return ISING_OK;
    if (I.has_h && std::ldexp(I.h_absmax, ds->h_shift) * (double)n >= 1073741824.0) return ISING_OK;
  }
  SparseRes R;
  R.rb = 8;
  for (int c : {4, 2, 1})
    if (ceil_div_i(ds->B, c) <= ctx->sm_count) R.rb = c;
  // a CTA runs until its slowest restart stops: under the convergence rule
  // fewer of them per CTA retire sooner
  if (ds->conv.p) R.rb = std::min(R.rb, 2);
  if (ds->int_energy) {
    R.rpb = 8;
    R.nvb = ceil_div_i(n, 8);
  } else {
    R.rpb = (int)((n + ds->mtiles - 1) / ds->mtiles);
    R.nvb = ds->mtiles;
    // (the launch-per-step form's rows per block; its last blocks may be short)
    if (ceil_div_i(n, R.rpb) != ds->mtiles) return ISING_OK;
  }
  R.kr = ceil_div_i(R.rpb, 8);
  const int vw = R.nvb * 8;
  R.passes = ceil_div_i(vw, sr_threads(R.rb) - 32);
  R.nt = (ceil_div_i(vw, R.passes) + 31) / 32 * 32;
  if (R.passes * R.kr * R.rb > 32) return ISING_OK;  // (a bit per site and restart of a thread)
  R.slices = R.passes * R.kr * (R.nt / 32);
  const size_t limit = ctx->smem_optin - 1024;
  const int ebytes = v8 ? 4 : 8;
  auto bytes = [&](bool pack, bool ell) {
    return SrLayout((int)n, R.rb, R.nvb, R.slices, R.entries, ebytes, ds->int_energy, pack, ell).total;
  };
  if (bytes(false, false) > limit) return ISING_OK;
  ISING_TRY(dev_alloc(ctx, R.off, ((size_t)R.slices + 2) * 4));
  ISING_CUDA(ctx, cudaMemsetAsync(R.off.p, 0, R.off.bytes, ctx->stream));
  const int g = ceil_div_i((int64_t)R.slices * 32, 256);
  sr_width_kernel<<<g, 256, 0, ctx->stream>>>((int)n, R.nt, R.rpb, R.kr, R.slices,
                                              I.rowptr.as<int32_t>(), R.off.as<int>());
  sr_scan_kernel<<<1, 1024, 0, ctx->stream>>>(R.slices, R.off.as<int>());
  ISING_CUDA(ctx, cudaGetLastError());
  int info[2] = {0, 0};  // entries of 32 lanes, longest row
  ISING_CUDA(ctx, cudaMemcpyAsync(info, R.off.as<int>() + R.slices, 8, cudaMemcpyDeviceToHost, ctx->stream));
  ISING_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
  R.entries = (int64_t)info[0] * 32;
  // two restarts' neighbour sums share a word, 16 bits each
  if (v8 && R.rb > 1 && I.j_absmax * (double)info[1] >= 32768.0) return ISING_OK;
  // One restart per CTA walks all couplings on as many SMs as there are restarts,
  // 0.07 ns a slot (0.085 with 8-byte slots), where the launch-per-step form
  // spreads its rows over the whole chip. us per step, that form / this one, with
  // the slots: int8, 8 restarts, 312000 27.4 / 26.7, 486000 33.1 / 40.4; 152
  // restarts 1090000 83.9 / 82.8, 1700000 111 / 127; FP32, 8 restarts, 163000 20.8 /
  // 19.9, 277000 25.5 / 28.2, 4700000 182 / 379; 152 restarts 450000 44.0 / 40.6,
  // 900000 68.7 / 82.9. With two or more restarts per CTA it was never the slower.
  if (R.rb == 1 && R.entries > (v8 ? 250000 + 6000 * ds->B : 150000 + 2600 * ds->B)) return ISING_OK;
  // FP32 energies keep the other form's rows per block: with very many restarts
  // under the convergence rule a CTA has a warp or two and each thread many rows
  // (300 spins of degree 48, 16384 restarts: 45 ms a run against 10; degree 12,
  // 170 slots a thread: 20 against 47 or, where all stop early, 6.6 against 5.2)
  if (R.entries > 6 * (int64_t)R.nt * R.nt) return ISING_OK;
  // a few long rows would pad their slices and leave the other lanes idle
  if (R.entries > 6 * nnz + 32768) return ISING_OK;
  ISING_TRY(dev_alloc(ctx, R.ell, (size_t)R.entries * ebytes));
  sr_fill_kernel<<<g, 256, 0, ctx->stream>>>((int)n, R.nt, R.rpb, R.kr, R.slices, v8,
                                             I.rowptr.as<int32_t>(), I.indices.as<int32_t>(),
                                             ds->sp_val.p, R.off.as<int>(), R.ell.as<uint32_t>());
  ISING_CUDA(ctx, cudaGetLastError());
  R.pack = bytes(true, false) <= limit;
  R.ell_smem = bytes(R.pack, true) <= limit;
  R.smem = bytes(R.pack, R.ell_smem);
  ds->sres = new SparseRes(std::move(R));
  return ISING_OK;
}

// Queues `steps` steps (one launch per 20000).
int sparse_res_run(ising_ds* ds, int64_t steps) {
  ising_ctx* ctx = ds->ctx;
  const SparseRes* R = ds->sres;
  SrArgs a;
  a.n = (int)ds->n;
  a.B = ds->B;
  a.Bp = ds->Bp;
  a.nt = R->nt;
  a.rpb = R->rpb;
  a.kr = R->kr;
  a.passes = R->passes;
  a.nvb = R->nvb;
  a.slices = R->slices;
  a.entries = R->entries;
  a.ell = R->ell.as<uint32_t>();
  const SrLayout L((int)ds->n, R->rb, R->nvb, R->slices, R->entries, ds->sp_int8 ? 4 : 8,
                   ds->int_energy, R->pack, R->ell_smem);
  a.spins = (int)L.spins;
  a.buffer = (int)L.buffer;
  a.part = (int)L.part;
  a.off_at = (int)L.off;
  a.ell_at = (int)L.ell;
  a.off = R->off.as<int>();
  a.T = ds->T;
  a.k = ds->k;
  a.bias = ds->bias.as<float2>();
  a.theta = ds->theta.as<float>();
  a.m = ds->m.as<float>();
  a.v = ds->v.as<float>();
  a.hf = ds->inst.has_h ? ds->hf.as<float>() : nullptr;
  a.hint = ds->hint.as<int32_t>();
  a.cq = ds->inst.cq;
  a.chs = ds->inst.ch * std::ldexp(1.0, -ds->h_shift);
  a.best_E = ds->best_E.as<double>();
  a.best_t = ds->best_t.as<long long>();
  a.best_s = ds->best_s.as<int8_t>();
  a.bs_ld = ds->bs_ld;
  a.last_E = ds->last_E.as<double>();
  a.counters = ds->counters.as<long long>();
  const bool conv = ds->conv.p != nullptr;
  a.conv_ring = conv ? ds->conv_ring() : nullptr;
  a.conv_init = conv ? ds->conv_init() : nullptr;
  a.conv_step = conv ? ds->conv_step() : nullptr;
  a.conv_count = conv ? ds->conv_count() : nullptr;
  a.live32 = conv ? ds->live.as<int>() : nullptr;
  while (steps > 0) {
    const int64_t k = std::min<int64_t>(steps, 20000);
    DevMem& out = ds->spins[(ds->t + k + 1) % 3];
    ISING_CUDA(ctx, cudaMemsetAsync(out.p, 0, out.bytes, ctx->stream));
    a.bits_out = out.as<uint32_t>();
    a.steps = (int)k;
    a.t0 = ds->t;
    switch (R->rb) {
      case 1: ISING_TRY(sr_launch_pack<1>(ds, R, a)); break;
      case 2: ISING_TRY(sr_launch_pack<2>(ds, R, a)); break;
      case 4: ISING_TRY(sr_launch_pack<4>(ds, R, a)); break;
      default: ISING_TRY(sr_launch_pack<8>(ds, R, a)); break;
    }
    if (conv) {
      sr_work_kernel<<<ceil_div_i(ds->B, 128), 128, 0, ctx->stream>>>(
          ds->B, ds->conv_step(), ds->t, k, ds->work.as<unsigned long long>());
      ISING_CUDA(ctx, cudaGetLastError());
    } else {
      ds->work_host += k * ds->B;
    }
    ds->t += k;
    steps -= k;
  }
  return ISING_OK;
}

void sparse_res_release(ising_ds* ds) {
  delete ds->sres;
  ds->sres = nullptr;
}

}  // namespace ising
