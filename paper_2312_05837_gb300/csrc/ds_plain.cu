// K2p: the plain FP32 form of the fused domain-selection step (Sec. III-B)
// on the CUDA cores. G = J S is a tiled SIMT SGEMM over blocks of 128 spins x
// TN restarts; the epilogue does, per element: loss field F = cQ G + cH h - mu s,
// gradient g = cos(theta) F, Adam, projection, rounding of the new spin, and
// the energy partials of the input spins for this block's 128 rows. In the
// relaxed mode the product runs on x = sin(theta) (X), the epilogue takes the
// rounded spins from Sr, writes x_{t+1} and leaves the energies to a
// kModeEnergy pass.
//
// n B n multiply-adds, each output's in order of k (the sums must not depend on
// the tiling). A thread holds 8 rows x 4 restarts: 32 multiply-adds for three
// shared-memory loads. J is symmetric, so the block's 128 columns of row k, which
// are contiguous, stand for its 128 rows of column k: the J tile is copied
// asynchronously without turning it over, three chunks of 16 k deep. TN is the
// width that fills the SMs' waves best: at n = 1500 and 512 restarts, 132 tiles of
// 48 (one per SM) instead of 48 tiles of 128. Measured there: 279 us per step with
// 128 x 128 tiles loaded and used in turn, 102 us now.
// What bounds it there: few warps. A tile of 48 has six, so two of an SM's four
// schedulers hold two and two hold one; the schedulers issue in half of their
// cycles, the FMA pipe is 38 % and the shared-memory pipe 47 % busy, DRAM 3 %
// (ncu). Pairs of rows by fma.rn.f32x2 take their second operand twice from
// shared memory and were slower (110 us, 4 x 4 or 8 x 4 per thread).
#include "ds_internal.cuh"

namespace ising {
namespace {

constexpr int BM = 128, BK = 16;
constexpr int kStages = 3;  // chunks of J in flight or in use

// Shared memory in floats: J chunks [kStages][BK][BM], restart chunks
// [2][BK][TN]; afterwards the products [TN][BM + 4].
template <int TN>
struct PlainTile {
  static constexpr int kThreads = BM / 8 * (TN / 4);
  static constexpr int kA = BK * BM, kB = BK * TN;
  static constexpr int kG = TN * (BM + 4);
  static constexpr int kFloats = kStages * kA + 2 * kB > kG ? kStages * kA + 2 * kB : kG;
};

__device__ __forceinline__ void copy_async(void* dst, const float* src, bool ok, bool wide) {
  const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
  // (size 0 reads nothing and writes zeros)
  if (wide) asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(ok ? 16 : 0) : "memory");
  else asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(d), "l"(src), "r"(ok ? 4 : 0) : "memory");
}

__global__ void to_float_kernel(const void* J, int dt, int64_t count, float* out) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < count;
       e += (int64_t)gridDim.x * blockDim.x)
    out[e] = (float)load_as_double(J, dt, e);
}

template <int MODE, bool INT_E, int TN>
__global__ void __launch_bounds__(PlainTile<TN>::kThreads) plain_step_kernel(
    const float* __restrict__ J, int64_t n, int64_t B, const float* __restrict__ S,
    const float* __restrict__ Sr, float* __restrict__ Xnext,
    float* __restrict__ Snext, float* __restrict__ theta, float* __restrict__ m,
    float* __restrict__ v, const float* __restrict__ hf, const int32_t* __restrict__ hint,
    StepConsts k, const float2* __restrict__ bias, const long long* __restrict__ counters,
    long long* __restrict__ qpart, long long* __restrict__ hpart, float* __restrict__ epart,
    float* __restrict__ Gout, const int* __restrict__ live32, unsigned long long* __restrict__ work) {
  constexpr bool UPDATE = MODE == kModeUpdate || MODE == kModeRelaxed;
  constexpr bool PARTIALS = MODE == kModeUpdate || MODE == kModeEnergy;
  using L = PlainTile<TN>;
  extern __shared__ __align__(16) float smem[];
  float* As = smem;                      // [kStages][BK][BM]
  float* Bs = smem + kStages * L::kA;    // [2][BK][TN]
  const int tid = threadIdx.x;
  const int tx = tid & 15, ty = tid >> 4;
  const int64_t m0 = (int64_t)blockIdx.x * BM, n0 = (int64_t)blockIdx.y * TN;
  const int64_t ne = n0 + TN < B ? n0 + TN : B;
  if (MODE != kModeCoupling) {
    // restarts retire in slices of 128; a tile in two slices needs both
    const int64_t c0 = n0 / 128 * 128, c1 = (ne + 127) / 128 * 128;
    if (restarts_retired(live32, c0, c1 < B ? c1 : B)) return;  // (uniform per block)
    // the slice's restart-steps, by the tile that starts in it first
    if (UPDATE && work && blockIdx.x == 0 && tid == 0)
      for (int64_t c = (n0 + 127) / 128 * 128; c < ne; c += 128) {
        const int64_t e = c + 128 < B ? c + 128 : B;
        if (!restarts_retired(live32, c, e)) atomicAdd(work, (unsigned long long)(e - c));
      }
  }
  const bool wide = (n & 3) == 0;  // rows of J and S start on 16 bytes
  // where this thread's pieces of the next J chunk start (wide copies)
  constexpr int kAq = (BK * BM / 4 + L::kThreads - 1) / L::kThreads;
  const float* asrc[kAq];
#pragma unroll
  for (int q = 0; q < kAq; ++q) {
    const int e = tid + q * L::kThreads;
    asrc[q] = J + (int64_t)(e / (BM / 4)) * n + m0 + e % (BM / 4) * 4;
  }
  auto load_a = [&](int stage, int64_t k0) {
    float* dst = As + stage * L::kA;
    if (wide) {
#pragma unroll
      for (int q = 0; q < kAq; ++q) {
        const int e = tid + q * L::kThreads;
        if (kAq * L::kThreads > BK * BM / 4 && e >= BK * BM / 4) break;
        const bool ok = k0 + e / (BM / 4) < n && m0 + e % (BM / 4) * 4 < n;
        copy_async(dst + 4 * e, ok ? asrc[q] : J, ok, true);
        asrc[q] += BK * n;
      }
    } else {
      for (int e = tid; e < BK * BM; e += L::kThreads) {
        const int kk = e / BM, r = e % BM;
        const bool ok = k0 + kk < n && m0 + r < n;
        copy_async(dst + kk * BM + r, ok ? J + (k0 + kk) * n + m0 + r : J, ok, false);
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  // four consecutive k of one restart per thread and step
  constexpr int kBq = (BK * TN / 4 + L::kThreads - 1) / L::kThreads;
  float4 breg[kBq];
  auto fetch_b = [&](int64_t k0) {
#pragma unroll
    for (int q = 0; q < kBq; ++q) {
      const int e = tid + q * L::kThreads;
      const int b = e / (BK / 4);
      const int64_t kk = k0 + e % (BK / 4) * 4, gb = n0 + b;
      float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
      if (b < TN && gb < B) {
        const float* src = S + gb * n + kk;
        if (wide) {
          if (kk < n) x = *reinterpret_cast<const float4*>(src);
        } else {
          if (kk < n) x.x = src[0];
          if (kk + 1 < n) x.y = src[1];
          if (kk + 2 < n) x.z = src[2];
          if (kk + 3 < n) x.w = src[3];
        }
      }
      breg[q] = x;
    }
  };
  auto store_b = [&](int buf) {
#pragma unroll
    for (int q = 0; q < kBq; ++q) {
      const int e = tid + q * L::kThreads;
      const int b = e / (BK / 4), kk = e % (BK / 4) * 4;
      if (b >= TN) continue;
      float* dst = Bs + buf * L::kB + kk * TN + b;
      dst[0] = breg[q].x;
      dst[TN] = breg[q].y;
      dst[2 * TN] = breg[q].z;
      dst[3 * TN] = breg[q].w;
    }
  };
  // rows 4 tx .. + 3 and 64 + 4 tx .. + 3, restarts 4 ty .. + 3 of the tile
  float acc[8][4];
#pragma unroll
  for (int r = 0; r < 8; ++r)
#pragma unroll
    for (int c = 0; c < 4; ++c) acc[r][c] = 0.f;
  const int chunks = (int)((n + BK - 1) / BK);
  for (int p = 0; p < kStages - 1; ++p) load_a(p, (int64_t)p * BK);
  fetch_b(0);
  for (int c = 0; c < chunks; ++c) {
    store_b(c & 1);
    asm volatile("cp.async.wait_group %0;" ::"n"(kStages - 2) : "memory");
    __syncthreads();  // chunk c has landed; chunk c - 1 is read by no one any more
    load_a((c + kStages - 1) % kStages, (int64_t)(c + kStages - 1) * BK);
    if (c + 1 < chunks) fetch_b((int64_t)(c + 1) * BK);
    const float* Ac = As + c % kStages * L::kA + 4 * tx;
    const float* Bc = Bs + (c & 1) * L::kB + 4 * ty;
    // the operands of kk + 1 are read while those of kk are multiplied
    float4 a0 = *reinterpret_cast<const float4*>(Ac);
    float4 a1 = *reinterpret_cast<const float4*>(Ac + 64);
    float4 b0 = *reinterpret_cast<const float4*>(Bc);
#pragma unroll
    for (int kk = 0; kk < BK; ++kk) {
      const float a[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
      const float b[4] = {b0.x, b0.y, b0.z, b0.w};
      if (kk + 1 < BK) {
        a0 = *reinterpret_cast<const float4*>(Ac + (kk + 1) * BM);
        a1 = *reinterpret_cast<const float4*>(Ac + (kk + 1) * BM + 64);
        b0 = *reinterpret_cast<const float4*>(Bc + (kk + 1) * TN);
      }
#pragma unroll
      for (int r = 0; r < 8; ++r)
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[r][q] = fmaf(a[r], b[q], acc[r][q]);
    }
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();
  // the products to shared memory, [restart][row]
  float* Gs = smem;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    float* row = Gs + (4 * ty + q) * (BM + 4) + 4 * tx;
    *reinterpret_cast<float4*>(row) = make_float4(acc[0][q], acc[1][q], acc[2][q], acc[3][q]);
    *reinterpret_cast<float4*>(row + 64) = make_float4(acc[4][q], acc[5][q], acc[6][q], acc[7][q]);
  }
  __syncthreads();

  const long long t = counters[0] + 1;
  const float2 bc = bias[t];
  for (int col = ty; col < TN; col += L::kThreads / 16) {
    const int64_t b = n0 + col;
    int qs = 0, hs = 0;
    float es = 0.f;
    // all loads first (16 lanes per restart, rows tx + 16 r)
    float s8[8], th8[8], m8[8], v8[8];
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      const int64_t i = m0 + tx + 16 * r;
      s8[r] = 1.f;
      th8[r] = m8[r] = v8[r] = 0.f;
      if (i < n && b < B && MODE != kModeCoupling) {
        const int64_t idx = b * n + i;
        s8[r] = Sr[idx];
        if (UPDATE) {
          th8[r] = theta[idx];
          m8[r] = m[idx];
          v8[r] = v[idx];
        }
      }
    }
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      const int64_t i = m0 + tx + 16 * r;
      if (i < n && b < B) {
        const int64_t idx = b * n + i;
        const float G = Gs[col * (BM + 4) + tx + 16 * r];
        if (MODE == kModeCoupling) {
          Gout[idx] = G;
          continue;
        }
        const float s = s8[r];
        const float h = hf[i];
        if (INT_E) {
          qs += (int)s * __float2int_rn(G);
          hs += (int)s * hint[i];
        } else {
          es += s * fmaf(k.cq, G, k.ch * h);
        }
        if (UPDATE) {
          const float F = fmaf(k.cq, G, fmaf(k.ch, h, -k.mu * s));
          float th = th8[r];
          const float g = cos_proj(th) * F;
          float mm = m8[r], vv = v8[r];
          th = adam_update(k, bc.x, bc.y, g, th, mm, vv);
          theta[idx] = th;
          m[idx] = mm;
          v[idx] = vv;
          Snext[idx] = sin_nonneg(th) ? 1.f : -1.f;
          if (MODE == kModeRelaxed) Xnext[idx] = sin_proj(th);
        }
      }
    }
    // reduce over the 16 lanes (tx) that share this restart
#pragma unroll
    for (int o = 8; o; o >>= 1) {
      if (INT_E) {
        qs += __shfl_xor_sync(0xffffffffu, qs, o);
        hs += __shfl_xor_sync(0xffffffffu, hs, o);
      } else {
        es += __shfl_xor_sync(0xffffffffu, es, o);
      }
    }
    if (PARTIALS && tx == 0 && b < B) {
      const int64_t o = (int64_t)blockIdx.x * B + b;
      if (INT_E) {
        qpart[o] = qs;
        hpart[o] = hs;
      } else {
        epart[o] = es;
      }
    }
  }
}

// Restarts per tile: the busiest SM's share, waves of tiles times the width,
// sets the step's time; the wider of equals (it loads less per product).
int plain_width(const ising_ds* ds) {
  int best = 0;
  int64_t cost = 0;
  for (int w : {128, 96, 64, 48, 32}) {
    const int64_t tiles = (int64_t)ceil_div_i(ds->n, BM) * ceil_div_i(ds->B, w);
    const int64_t c = (tiles + ds->ctx->sm_count - 1) / ds->ctx->sm_count * w;
    if (!best || c < cost) best = w, cost = c;
  }
  return best;
}

}  // namespace

int plain_setup(ising_ds* ds) {
  ising_ctx* ctx = ds->ctx;
  ds->ld = ds->n;
  ds->Bp = ds->B;
  ds->spin_kind = kSpinF32;
  ds->mtiles = ceil_div_i(ds->n, BM);
  const int64_t nn = ds->n * ds->n;
  ISING_TRY(dev_alloc(ctx, ds->Jf, nn * 4));
  int g = (int)std::min<int64_t>((nn + 255) / 256, (int64_t)ctx->sm_count * 16);
  to_float_kernel<<<g, 256, 0, ctx->stream>>>(ds->inst.J.p, ds->inst.j_dtype, nn, ds->Jf.as<float>());
  ISING_CUDA(ctx, cudaGetLastError());
  return ISING_OK;
}

int plain_step(ising_ds* ds, int mode, float* Gout) {
  ising_ctx* ctx = ds->ctx;
  const int64_t t = ds->t + 1;
  const float* S = ds->spins[t % 3].as<float>();
  float* Sn = ds->spins[(t + 1) % 3].as<float>();
  // relaxed mode: the product's operand is x_t, the rounded spins come along
  const bool rel = mode == kModeRelaxed;
  const float* X = rel ? ds->xbuf[t % 2].as<float>() : S;
  float* Xn = rel ? ds->xbuf[(t + 1) % 2].as<float>() : nullptr;
  const int ps = (int)(t % 2);
  const int width = plain_width(ds);
  const dim3 grid(ceil_div_i(ds->n, BM), ceil_div_i(ds->B, width));
#define ISING_PLAIN_W(U, I, W)                                                                \
  do {                                                                                        \
    auto kern = plain_step_kernel<U, I, W>;                                                   \
    const int bytes = PlainTile<W>::kFloats * 4;                                              \
    ISING_CUDA(ctx, cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes)); \
    kern<<<grid, PlainTile<W>::kThreads, bytes, ctx->stream>>>(                               \
      ds->Jf.as<float>(), ds->n, ds->B, X, S, Xn, Sn, ds->theta.as<float>(), ds->m.as<float>(),\
      ds->v.as<float>(), ds->hf.as<float>(), ds->hint.as<int32_t>(), ds->k,                   \
      ds->bias.as<float2>(), ds->counters.as<long long>(), ds->qpart[ps].as<long long>(),     \
      ds->hpart[ps].as<long long>(), ds->epart[ps].as<float>(), Gout,                        \
      ds->live.p ? ds->live.as<int>() : nullptr, ds->work.as<unsigned long long>());          \
  } while (0)
#define ISING_PLAIN(U, I)                                                                     \
  do {                                                                                        \
    switch (width) {                                                                          \
      case 32: ISING_PLAIN_W(U, I, 32); break;                                                \
      case 48: ISING_PLAIN_W(U, I, 48); break;                                                \
      case 64: ISING_PLAIN_W(U, I, 64); break;                                                \
      case 96: ISING_PLAIN_W(U, I, 96); break;                                                \
      default: ISING_PLAIN_W(U, I, 128); break;                                               \
    }                                                                                         \
  } while (0)
  if (mode == kModeUpdate) {
    if (ds->int_energy) ISING_PLAIN(kModeUpdate, true); else ISING_PLAIN(kModeUpdate, false);
  } else if (mode == kModeEnergy) {
    if (ds->int_energy) ISING_PLAIN(kModeEnergy, true); else ISING_PLAIN(kModeEnergy, false);
  } else if (rel) {
    if (ds->int_energy) ISING_PLAIN(kModeRelaxed, true); else ISING_PLAIN(kModeRelaxed, false);
  } else {
    ISING_PLAIN(kModeCoupling, true);
  }
#undef ISING_PLAIN_W
#undef ISING_PLAIN
  ISING_CUDA(ctx, cudaGetLastError());
  return ISING_OK;
}

}  // namespace ising
