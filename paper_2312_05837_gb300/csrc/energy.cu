// K3: energy of rounded spin vectors, E(s) = cQ s^T J s + cH h^T s (Sec. II).
//
// Four forms, all deterministic; integer couplings are exact in each:
//   fixed    dense J: every J_ij becomes a 64-bit integer (itself, or
//            rint(J_ij 2^k) with one scale for the matrix), so s^T J s is summed
//            in integers whatever the order, rounded once at the end;
//   planes   dense J and many vectors: the same integers as digits in FP16
//            planes, their sums on the tensor cores, exact as well;
//   packed   CSR without long rows, many vectors: a lane per vector, spins as bits;
//   general  a warp per row and vector, int64 or FP64: few CSR vectors, dense J
//            whose values spread too widely for one scale, the call without
//            allocation, and spins that are not +-1.
// General form: one block handles 64 rows of one vector; a warp forms (J s)_i
// for 8 rows (lanes stride over the columns of a dense row or the entries of
// a CSR row), then the block adds s_i (J s)_i and h_i s_i over its rows in a
// fixed order. A second kernel adds the block partials of each vector in a
// fixed order.
#include "common.cuh"

#include <algorithm>
#include <atomic>
#include <cmath>
#include <type_traits>

namespace ising {
namespace {

constexpr int kRowsPerBlock = 64;

// The instance as the rows kernel reads it: dense or CSR J with row offsets
// of type Off (the library's own int32 copy, or a caller's int64 offsets),
// and h scaled by 2^h_shift to integers in the exact mode.
template <typename Off>
struct RowsView {
  int64_t n;
  int layout, j_dtype, h_dtype, h_shift;
  const void* J;
  const Off* rowptr;
  const int32_t* indices;
  const void* h;  // nullable
};

template <bool INT, typename Off>
__global__ void __launch_bounds__(256) energy_rows(RowsView<Off> in, const int8_t* __restrict__ spins,
                                                   int64_t nchunks, void* __restrict__ qpart,
                                                   void* __restrict__ hpart) {
  using Acc = typename std::conditional<INT, long long, double>::type;
  const int64_t n = in.n;
  const int64_t vec = blockIdx.y;
  const int8_t* s = spins + vec * n;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  __shared__ Acc sq[8], sh[8];
  Acc q_acc = 0, h_acc = 0;
  for (int r = 0; r < kRowsPerBlock / 8; ++r) {
    int64_t i = (int64_t)blockIdx.x * kRowsPerBlock + warp * (kRowsPerBlock / 8) + r;
    if (i >= n) break;
    Acc dot = 0;
    if (in.layout == ISING_LAYOUT_DENSE) {
      const int64_t base = i * n;
      for (int64_t j = lane; j < n; j += 32) {
        if (INT) dot += (Acc)load_as_int(in.J, in.j_dtype, base + j) * s[j];
        else dot += load_as_double(in.J, in.j_dtype, base + j) * (double)s[j];
      }
    } else {
      for (int64_t k = (int64_t)in.rowptr[i] + lane; k < (int64_t)in.rowptr[i + 1]; k += 32) {
        int32_t j = in.indices[k];
        if (INT) dot += (Acc)load_as_int(in.J, in.j_dtype, k) * s[j];
        else dot += load_as_double(in.J, in.j_dtype, k) * (double)s[j];
      }
    }
    for (int o = 16; o; o >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, o);
    if (lane == 0) {
      q_acc += dot * (Acc)s[i];
      if (in.h) {
        if (INT) h_acc += (Acc)llrint(ldexp(load_as_double(in.h, in.h_dtype, i), in.h_shift)) * s[i];
        else h_acc += load_as_double(in.h, in.h_dtype, i) * (double)s[i];
      }
    }
  }
  if (lane == 0) {
    sq[warp] = q_acc;
    sh[warp] = h_acc;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    Acc a = 0, b = 0;
    for (int w = 0; w < 8; ++w) { a += sq[w]; b += sh[w]; }
    static_cast<Acc*>(qpart)[vec * nchunks + blockIdx.x] = a;
    static_cast<Acc*>(hpart)[vec * nchunks + blockIdx.x] = b;
  }
}

// One warp per vector: lane l adds chunks l, l + 32, ..., then a fixed xor tree
// (a thread per vector walked the chunks of n = 120000 for 120 us).
template <bool INT>
__global__ void __launch_bounds__(256) energy_finish(int64_t count, int64_t nchunks,
                                                     const void* __restrict__ qpart,
                                                     const void* __restrict__ hpart, double cq,
                                                     double ch, int h_shift, double* __restrict__ E,
                                                     int64_t* __restrict__ Q,
                                                     int64_t* __restrict__ H) {
  using Acc = typename std::conditional<INT, long long, double>::type;
  const int lane = threadIdx.x & 31;
  const int64_t v = blockIdx.x * (int64_t)(blockDim.x >> 5) + (threadIdx.x >> 5);
  if (v >= count) return;
  Acc a = 0, b = 0;
  for (int64_t c = lane; c < nchunks; c += 32) {
    a += static_cast<const Acc*>(qpart)[v * nchunks + c];
    b += static_cast<const Acc*>(hpart)[v * nchunks + c];
  }
  for (int o = 16; o; o >>= 1) {
    a += __shfl_xor_sync(0xffffffffu, a, o);
    b += __shfl_xor_sync(0xffffffffu, b, o);
  }
  if (lane != 0) return;
  if (INT) {
    E[v] = cq * (double)a + ch * ldexp((double)b, -h_shift);
    if (Q) Q[v] = (int64_t)a;
    if (H) H[v] = (int64_t)b;
  } else {
    E[v] = cq * (double)a + ch * (double)b;
  }
}

// ---------------------------------------------------------------- fixed form
//
// Bound by the integer pipe. GB300 runs two FP64 lanes per SM and cycle against
// 64 integer ones, and the general form spends three FP64 operations per
// coupling and vector (two conversions and the FMA). Here a coupling is
// converted once for V vectors to I = rint(J_ij 2^k) and every vector adds it
// where its spin is +1 (two predicated 32-bit additions; s^T J s follows from
// 2 sum_{s_j = +1} I - sum_j I). A lane's sums are split into limbs of 24, 24
// and the remaining bits, which the warp reduces with redux.sync, the block in
// shared memory and the grid by 64-bit integer atomics: exact in any order.
// k is chosen so that no lane sum can overflow (53 to 58 bits per coupling).

constexpr int kFixRows = 4;      // rows of one block (its 8 warps share the columns)
constexpr int kFixVectors = 4;   // vectors per pass (1 for a single vector)

// Spins as bits, word w of vector v: spins 32 w .. 32 w + 31 (bit set = +1;
// columns past n are 0). `odd` is raised by any spin that is not +-1.
__global__ void __launch_bounds__(256) pack_rows_kernel(const int8_t* __restrict__ spins,
                                                        int64_t count, int64_t n, int64_t words,
                                                        uint32_t* __restrict__ bits,
                                                        unsigned int* __restrict__ odd) {
  const int lane = threadIdx.x & 31;
  const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
  for (int64_t e = blockIdx.x * (int64_t)(blockDim.x >> 5) + (threadIdx.x >> 5); e < count * words;
       e += warps) {
    const int64_t v = e / words, j = (e - v * words) * 32 + lane;
    const int s = j < n ? spins[v * n + j] : -1;
    const uint32_t w = __ballot_sync(0xffffffffu, s == 1);
    const uint32_t bad = __ballot_sync(0xffffffffu, s != 1 && s != -1);
    if (lane == 0) {
      bits[e] = w;
      if (bad) atomicOr(odd, 1u);
    }
  }
}

// rint(x 2^shift) (ties away from zero for floats, which are handled in
// integer arithmetic: float to 64-bit conversions run at the FP64 rate).
template <typename T>
__device__ __forceinline__ long long to_fixed(T x, int shift, double dscale) {
  if constexpr (std::is_same<T, double>::value) {
    return __double2ll_rn(x * dscale);
  } else if constexpr (std::is_same<T, float>::value) {
    const unsigned int u = __float_as_uint(x), e = (u >> 23) & 0xFFu;
    const unsigned int mant = (u & 0x7FFFFFu) | (e ? 0x800000u : 0u);
    // |x| 2^shift = mant 2^(max(e, 1) - 150 + shift) < 2^58: mant 2^38, shifted
    // right by d in [4, 63] (62 bits; d = 63 rounds to 0)
    const int d = min(38 - ((int)max(e, 1u) - 150 + shift), 63);
    const long long m = (long long)((((unsigned long long)mant << 38) + (1ull << (d - 1))) >> d);
    return (int)u < 0 ? -m : m;
  } else {
    return (long long)x;  // (integer types are never scaled: whole_couplings)
  }
}

// Block: rows 4 blockIdx.x .. + 3, vectors V blockIdx.y .., the blockIdx.z-th
// `span` columns (a multiple of 1024); warp w takes every 8th group of 32 VEC
// columns, lane l of it VEC consecutive ones (VEC = 4 needs n % 4 == 0, so that
// every row starts on a vector boundary).
// limbs[v][3] receives the limbs of s^T I s.
template <typename T, int VEC, int V>
__global__ void __launch_bounds__(256) energy_fixed_kernel(
    int64_t n, int64_t span, const T* __restrict__ J, int shift, double dscale,
    const uint32_t* __restrict__ bits, int64_t words, int64_t count,
    unsigned long long* __restrict__ limbs) {
  extern __shared__ uint32_t sbits[];  // [V][words]
  __shared__ int red[8][kFixRows][V][3];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t i0 = (int64_t)blockIdx.x * kFixRows, v0 = (int64_t)blockIdx.y * V;
  for (int64_t e = threadIdx.x; e < V * words; e += blockDim.x) {
    const int64_t v = e / words;
    sbits[e] = v0 + v < count ? bits[v0 * words + e] : 0u;
  }
  __syncthreads();
  long long acc[kFixRows][V], rs[kFixRows];
#pragma unroll
  for (int r = 0; r < kFixRows; ++r) {
    rs[r] = 0;
#pragma unroll
    for (int v = 0; v < V; ++v) acc[r][v] = 0;
  }
  int64_t g = warp, groups = (n + 32 * VEC - 1) / (32 * VEC);
  if constexpr (std::is_same<T, double>::value) {  // (the only type whose columns are split)
    const int64_t per = span / (32 * VEC);
    g += blockIdx.z * per;
    groups = min(groups, (blockIdx.z + 1) * per);
  }
#pragma unroll 2
  for (; g < groups; g += 8) {
    const int64_t j = (g * 32 + lane) * VEC;
    T x[kFixRows][VEC];
#pragma unroll
    for (int r = 0; r < kFixRows; ++r) {
      const bool ok = i0 + r < n && j < n;
      const T* src = J + (i0 + r) * n + j;
      if constexpr (VEC == 1) {
        x[r][0] = ok ? __ldcs(src) : T(0);
      } else {
        struct alignas(sizeof(T) * VEC <= 16 ? sizeof(T) * VEC : 16) Quad { T q[VEC]; };
        const Quad z = ok ? *reinterpret_cast<const Quad*>(src) : Quad{};
#pragma unroll
        for (int c = 0; c < VEC; ++c) x[r][c] = z.q[c];
      }
    }
    uint32_t w[V];
#pragma unroll
    for (int v = 0; v < V; ++v)
      w[v] = j < n ? sbits[v * words + (j >> 5)] >> (int)(j & 31) : 0u;
#pragma unroll
    for (int c = 0; c < VEC; ++c)
#pragma unroll
      for (int r = 0; r < kFixRows; ++r) {
        const long long I = to_fixed<T>(x[r][c], shift, dscale);
        rs[r] += I;
#pragma unroll
        for (int v = 0; v < V; ++v)
          if ((w[v] >> c) & 1u) acc[r][v] += I;
      }
  }
#pragma unroll
  for (int r = 0; r < kFixRows; ++r)
#pragma unroll
    for (int v = 0; v < V; ++v) {
      const long long S = 2 * acc[r][v] - rs[r];
      const unsigned int lo = __reduce_add_sync(0xffffffffu, (unsigned int)(S & 0xFFFFFF));
      const unsigned int mid = __reduce_add_sync(0xffffffffu, (unsigned int)((S >> 24) & 0xFFFFFF));
      const int hi = __reduce_add_sync(0xffffffffu, (int)(S >> 48));
      if (lane == 0) {
        red[warp][r][v][0] = (int)lo;
        red[warp][r][v][1] = (int)mid;
        red[warp][r][v][2] = hi;
      }
    }
  __syncthreads();
  for (int e = threadIdx.x; e < V * 3; e += blockDim.x) {
    const int v = e / 3, k = e - 3 * v;
    if (v0 + v >= count) continue;
    long long t = 0;
#pragma unroll
    for (int r = 0; r < kFixRows; ++r) {
      const int64_t i = i0 + r;
      if (i >= n) break;
      long long G = 0;
#pragma unroll
      for (int u = 0; u < 8; ++u) G += red[u][r][v][k];
      t += (sbits[v * words + (i >> 5)] >> (int)(i & 31)) & 1u ? G : -G;
    }
    atomicAdd(&limbs[(v0 + v) * 3 + k], (unsigned long long)t);
  }
}

// s^T I s = L0 + 2^24 L1 + 2^48 L2, and h^T s: a block per vector.
template <bool INT>
__global__ void __launch_bounds__(256) energy_fixed_finish(
    int64_t n, const uint32_t* __restrict__ bits, int64_t words,
    const unsigned long long* __restrict__ limbs, const void* __restrict__ h, int h_dtype,
    int h_shift, double cq, double ch, double unscale, double* __restrict__ E,
    int64_t* __restrict__ Q, int64_t* __restrict__ H) {
  using Acc = typename std::conditional<INT, long long, double>::type;
  const int64_t v = blockIdx.x;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  __shared__ Acc sh[8];
  Acc a = 0;
  if (h)
    for (int64_t i = threadIdx.x; i < n; i += blockDim.x) {
      const bool up = (bits[v * words + (i >> 5)] >> (int)(i & 31)) & 1u;
      Acc x;
      if (INT) x = (Acc)llrint(ldexp(load_as_double(h, h_dtype, i), h_shift));
      else x = (Acc)load_as_double(h, h_dtype, i);
      a += up ? x : -x;
    }
  for (int o = 16; o; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
  if (lane == 0) sh[warp] = a;
  __syncthreads();
  if (threadIdx.x != 0) return;
  for (int w = 1; w < 8; ++w) a += sh[w];
  const long long L0 = (long long)limbs[v * 3], L1 = (long long)limbs[v * 3 + 1];
  const long long L2 = (long long)limbs[v * 3 + 2];
  if (INT) {
    const long long q = L0 + (L1 << 24) + (L2 << 48);
    E[v] = cq * (double)q + ch * ldexp((double)a, -h_shift);
    if (Q) Q[v] = q;
    if (H) H[v] = (long long)a;
  } else {
    // carries first, so that the two halves do not overlap
    const long long c1 = L1 + (L0 >> 24), c2 = L2 + (c1 >> 24);
    const double lo = (double)(((c1 & 0xFFFFFF) << 24) | (L0 & 0xFFFFFF));
    E[v] = cq * (fma((double)c2, 0x1p48, lo) * unscale) + ch * (double)a;
  }
}

// The binary scale of the integer forms: 0 for integer couplings; else every
// J_ij becomes rint(J_ij 2^*shift) with b bits (|J| < 2^E, largest b bits), and
// the form is used only where all those roundings together stay below 2^-53
// sum |J_ij|, what rounding each coupling once to FP64 may cost. Each is off by
// at most 2^-(b + 1) 2^E, and sum |J_ij| is at least the count of non-zeros times
// their geometric mean, which the mean exponent bounds below: so FP64 couplings
// need a mean exponent of E - b + 52. FP32 couplings have 24 bits: those above
// 2^(E - b + 24) are exact, and where the mean exponent is at least E - b + 48 at
// most 4 / 15 of the others' number can lie below that, whose roundings add up to
// less than 2^-54 sum |J_ij|.
bool scale_for(const DevInstance& I, int b, int* shift) {
  int ex = 0;
  std::frexp(I.j_absmax, &ex);  // |J| < 2^ex
  const int need = I.j_dtype == ISING_F64 ? 52 : 48;
  if ((double)I.j_expsum < (double)(ex - b + need) * (double)I.j_nonzeros) return false;
  *shift = b - ex;
  return *shift >= -120 && *shift <= 120;  // a float power of two; no result underflows
}

// Columns of one block of the fixed form when `splits` blocks share a row: whole
// groups of every warp and lane.
int64_t split_columns(int64_t n, int splits) { return ((n + splits - 1) / splits + 1023) / 1024 * 1024; }

// Integer couplings that the integer forms add as they are (scale 0): whatever
// the fields, whose sum of a non-dyadic h stays in FP64.
bool whole_couplings(const DevInstance& I) { return I.j_integer && I.j_absmax <= 2147483648.0; }

// b for the fixed form: the most for which no lane's sums overflow, with the
// columns dealt to *splits blocks where FP64 couplings need the bits (n = 8192
// Gaussian: one lane's 32 terms leave 56 bits, two blocks' 16 leave 57).
bool fixed_scale(const DevInstance& I, int* shift, int* splits) {
  *shift = 0;
  *splits = 1;
  if (whole_couplings(I) || I.j_nonzeros == 0) return true;
  for (;; *splits *= 2) {
    const int64_t lane_terms = 4 * ((split_columns(I.n, *splits) + 1023) / 1024);
    int lg = 0;
    while (((int64_t)1 << lg) < lane_terms) ++lg;
    const int b = std::min(58, 61 - lg);
    if (scale_for(I, b, shift)) return true;
    if (b == 58 || I.j_dtype != ISING_F64) return false;
  }
}

template <typename T, int VEC>
int fixed_launch(ising_ctx* ctx, const DevInstance& I, int shift, int splits, const uint32_t* bits,
                 int64_t words, int64_t count, unsigned long long* limbs) {
  const double dsc = std::ldexp(1.0, shift);
  const int V = count == 1 ? 1 : kFixVectors;
  const int64_t span = split_columns(I.n, splits);
  const dim3 grid((unsigned)((I.n + kFixRows - 1) / kFixRows), (unsigned)((count + V - 1) / V),
                  (unsigned)((I.n + span - 1) / span));
  const size_t smem = (size_t)V * words * 4;
  if (V == 1)
    energy_fixed_kernel<T, VEC, 1><<<grid, 256, smem, ctx->stream>>>(
        I.n, span, I.J.as<T>(), shift, dsc, bits, words, count, limbs);
  else
    energy_fixed_kernel<T, VEC, kFixVectors><<<grid, 256, smem, ctx->stream>>>(
        I.n, span, I.J.as<T>(), shift, dsc, bits, words, count, limbs);
  ISING_CUDA(ctx, cudaGetLastError());
  return ISING_OK;
}

template <typename T>
int fixed_launch_t(ising_ctx* ctx, const DevInstance& I, int shift, int splits, const uint32_t* bits,
                   int64_t words, int64_t count, unsigned long long* limbs) {
  // rows of a multiple of four values start on a vector boundary
  return I.n % 4 == 0 ? fixed_launch<T, 4>(ctx, I, shift, splits, bits, words, count, limbs)
                      : fixed_launch<T, 1>(ctx, I, shift, splits, bits, words, count, limbs);
}

// --------------------------------------------------------------- planes form
//
// The integers of the fixed form as digits d_p in [-2^(w - 1), 2^(w - 1)] of base
// 2^w, one FP16 plane per digit: s^T d_p s is a matrix product whose FP32 sums
// are exact while n 2^(w - 1) <= 2^22, so 256 vectors cost the tensor cores 5
// products where the fixed form spends 7 integer instructions per coupling and
// vector. Bound by writing and reading the planes (10 bytes per coupling).

constexpr double kPlaneTerms = 268435456.0;  // coupling-vectors from which the form pays

// Digits of every coupling, and the spins as FP16 +-1.
template <typename T>
__global__ void __launch_bounds__(256) split_digits_kernel(const T* __restrict__ J, int64_t n, int64_t ld,
                                                           int shift, double dscale, int w, int planes,
                                                           uint16_t* __restrict__ out) {
  const long long half = 1ll << (w - 1), mask = (1ll << w) - 1;
  // four columns per thread: one 8-byte store per plane (rows of ld, a multiple
  // of 64, start on a vector boundary; columns from n to ld are never read)
  for (int64_t i = blockIdx.y; i < n; i += gridDim.y)
    for (int64_t k = 4 * (blockIdx.x * (int64_t)blockDim.x + threadIdx.x); k < n;
         k += 4 * (int64_t)gridDim.x * blockDim.x) {
      long long I[4];
#pragma unroll
      for (int c = 0; c < 4; ++c) I[c] = k + c < n ? to_fixed<T>(J[i * n + k + c], shift, dscale) : 0;
      for (int p = 0; p < planes; ++p) {
        uint16_t f[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          // (the last digit takes what is left, at most 2^(w - 1) in magnitude)
          const long long d = p + 1 < planes ? ((I[c] + half) & mask) - half : I[c];
          f[c] = __half_as_ushort(__int2half_rn((int)d));
          I[c] = (I[c] - d) >> w;
        }
        *reinterpret_cast<uint2*>(out + ((int64_t)p * n + i) * ld + k) =
            make_uint2(f[0] | (uint32_t)f[1] << 16, f[2] | (uint32_t)f[3] << 16);
      }
    }
}

__global__ void __launch_bounds__(256) spins_f16_kernel(const int8_t* __restrict__ spins, int64_t count,
                                                        int64_t n, int64_t ld, uint16_t* __restrict__ out) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < count * ld;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t v = e / ld, i = e - v * ld;
    out[e] = i >= n ? 0 : (spins[v * n + i] == 1 ? 0x3C00 : 0xBC00);
  }
}

// sum_p 2^(w p) (sum of plane p's partial rows) in limbs; a warp per vector.
__global__ void __launch_bounds__(256) join_digits_kernel(int64_t count, int64_t rows, int w, int planes,
                                                          const long long* __restrict__ parts,
                                                          unsigned long long* __restrict__ limbs) {
  const int lane = threadIdx.x & 31;
  const int64_t v = blockIdx.x * (int64_t)(blockDim.x >> 5) + (threadIdx.x >> 5);
  if (v >= count) return;
  __int128 acc = 0;
  for (int p = 0; p < planes; ++p) {
    long long q = 0;
    for (int64_t r = lane; r < rows; r += 32) q += parts[((int64_t)p * rows + r) * count + v];
    for (int o = 16; o; o >>= 1) q += __shfl_xor_sync(0xffffffffu, q, o);
    acc += (__int128)q << (w * p);
  }
  if (lane != 0) return;
  limbs[v * 3] = (unsigned long long)(acc & 0xFFFFFF);
  limbs[v * 3 + 1] = (unsigned long long)((acc >> 24) & 0xFFFFFF);
  limbs[v * 3 + 2] = (unsigned long long)(long long)(acc >> 48);
}

// Digit width, planes and scale; false when the form does not apply.
bool plane_scale(const DevInstance& I, int* w, int* planes, int* shift) {
  int lg = 0;
  while (((int64_t)1 << lg) < I.n) ++lg;
  *w = std::min(12, 23 - lg);
  if (*w < 9) return false;  // n <= 16384
  if (whole_couplings(I) || I.j_nonzeros == 0) {
    *shift = 0;
    int bits = 1;
    while (std::ldexp(1.0, bits) <= I.j_absmax) ++bits;
    *planes = (bits + 1 + *w - 1) / *w;
    return true;
  }
  for (*planes = 5; *planes <= 7; ++*planes)
    if (scale_for(I, std::min(58, *w * *planes - 2), shift)) return true;
  return false;
}

template <typename T>
int split_launch(ising_ctx* ctx, const DevInstance& I, int64_t ld, int shift, int w, int planes,
                 uint16_t* out) {
  const dim3 grid((unsigned)std::min<int64_t>((I.n + 1023) / 1024, 64), (unsigned)std::min<int64_t>(I.n, 65535));
  split_digits_kernel<T><<<grid, 256, 0, ctx->stream>>>(I.J.as<T>(), I.n, ld, shift,
                                                        std::ldexp(1.0, shift), w, planes, out);
  ISING_CUDA(ctx, cudaGetLastError());
  return ISING_OK;
}

// --------------------------------------------------------------- packed form
//
// CSR with a warp per row and vector leaves most lanes idle (a row has a few
// entries). Here a lane is a vector: 32 vectors' spins of one site are one
// word, an edge is one broadcast word and one addition per lane.

// Word w of site i: vectors 32 w .. 32 w + 31 (bit set = +1; vectors past
// count are 0).
__global__ void __launch_bounds__(256) pack_sites_kernel(const int8_t* __restrict__ spins,
                                                         int64_t count, int64_t n, int64_t words,
                                                         uint32_t* __restrict__ bits,
                                                         unsigned int* __restrict__ odd) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n * words;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t w = e / n, i = e - w * n;
    uint32_t word = 0;
    bool bad = false;
    const int64_t left = count - 32 * w;
    const int cnt = left < 32 ? (int)left : 32;
    for (int k = 0; k < cnt; ++k) {
      const int s = spins[(32 * w + k) * n + i];
      word |= (s == 1 ? 1u : 0u) << k;
      bad |= s != 1 && s != -1;
    }
    bits[i * words + w] = word;
    if (bad) atomicOr(odd, 1u);
  }
}

constexpr int kPackedRow = 128;  // the longest row of an instance in this form
constexpr int kPackedLevels = 6;  // its 32 groups of four entries in the counter

// (J s)_i of the lane's vector over the row's entries [e0, e1). Integers in
// order; FP64 pairwise, four entries by a tree and the groups of four by a
// binary counter (level l holds the sum of 2^l groups), so that no entry passes
// through more additions than in the general form's lanes and tree: in order,
// the error of rows of 64 entries was 1.6 times that form's.
template <bool INT, typename Acc = typename std::conditional<INT, long long, double>::type>
__device__ __forceinline__ Acc packed_row(const RowsView<int32_t>& in, const uint32_t* __restrict__ bits,
                                          int64_t words, int e0, int e1, int lane) {
  auto term = [&](int e) {
    const uint32_t w = bits[(int64_t)in.indices[e] * words];
    Acc x;
    if constexpr (INT) x = (Acc)load_as_int(in.J, in.j_dtype, e);
    else x = (Acc)load_as_double(in.J, in.j_dtype, e);
    return (w >> lane) & 1u ? x : -x;
  };
  if constexpr (INT) {
    Acc dot = 0;
#pragma unroll 4
    for (int e = e0; e < e1; ++e) dot += term(e);
    return dot;
  } else {
    Acc level[kPackedLevels];
#pragma unroll
    for (int l = 0; l < kPackedLevels; ++l) level[l] = 0;
#pragma unroll 1
    for (int e = e0; e < e1; e += 4) {
      Acc x[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const Acc y = term(e + u < e1 ? e + u : e0);
        x[u] = e + u < e1 ? y : (Acc)0;
      }
      Acc sum = (x[0] + x[1]) + (x[2] + x[3]);
      const int g = (e - e0) >> 2;  // (uniform over the warp)
      bool carry = true;
#pragma unroll
      for (int l = 0; l < kPackedLevels; ++l)
        if (carry) {
          if (l + 1 < kPackedLevels && ((g >> l) & 1)) {
            sum += level[l];
            level[l] = 0;
          } else {
            level[l] += sum;  // (empty, or the last level)
            carry = false;
          }
        }
    }
    Acc dot = level[0];
#pragma unroll
    for (int l = 1; l < kPackedLevels; ++l) dot += level[l];
    return dot;
  }
}

// Block: kRowsPerBlock rows (warp w takes every 8th), 32 vectors (blockIdx.y);
// partials as the general form's, [vector][block].
template <bool INT>
__global__ void __launch_bounds__(256) energy_packed_kernel(RowsView<int32_t> in,
                                                            const uint32_t* __restrict__ bits,
                                                            int64_t words, int64_t count,
                                                            int64_t nchunks, void* __restrict__ qpart,
                                                            void* __restrict__ hpart) {
  using Acc = typename std::conditional<INT, long long, double>::type;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  __shared__ Acc sq[8][32], sh[8][32];
  Acc q = 0, hs = 0;
  const int64_t r0 = (int64_t)blockIdx.x * kRowsPerBlock;
  for (int64_t i = r0 + warp; i < r0 + kRowsPerBlock && i < in.n; i += 8) {
    const Acc dot = packed_row<INT>(in, bits + blockIdx.y, words, in.rowptr[i], in.rowptr[i + 1], lane);
    const bool up = (bits[i * words + blockIdx.y] >> lane) & 1u;
    q += up ? dot : -dot;
    if (in.h) {
      Acc x;
      if (INT) x = (Acc)llrint(ldexp(load_as_double(in.h, in.h_dtype, i), in.h_shift));
      else x = (Acc)load_as_double(in.h, in.h_dtype, i);
      hs += up ? x : -x;
    }
  }
  sq[warp][lane] = q;
  sh[warp][lane] = hs;
  __syncthreads();
  const int64_t v = (int64_t)blockIdx.y * 32 + lane;
  if (warp != 0 || v >= count) return;
  for (int w = 1; w < 8; ++w) { q += sq[w][lane]; hs += sh[w][lane]; }
  static_cast<Acc*>(qpart)[v * nchunks + blockIdx.x] = q;
  static_cast<Acc*>(hpart)[v * nchunks + blockIdx.x] = hs;
}

int pack_grid(ising_ctx* ctx, int64_t warps) {
  return (int)std::max<int64_t>(1, std::min<int64_t>((warps + 7) / 8, (int64_t)ctx->sm_count * 16));
}

}  // namespace

namespace {

int energy_general(ising_ctx* ctx, const DevInstance& inst, bool exact, const int8_t* spins,
                   int64_t count, double* E, int64_t* Q, int64_t* H) {
  const int64_t nchunks = (inst.n + kRowsPerBlock - 1) / kRowsPerBlock;
  DevMem qp, hp;
  ISING_TRY(dev_alloc(ctx, qp, (size_t)(count * nchunks) * 8));
  ISING_TRY(dev_alloc(ctx, hp, (size_t)(count * nchunks) * 8));
  dim3 grid((unsigned)nchunks, (unsigned)count);
  const InstView iv = view(inst);
  RowsView<int32_t> v{iv.n, iv.layout, iv.j_dtype, iv.h_dtype, exact ? inst.h_shift : 0,
                      iv.J, iv.rowptr, iv.indices, iv.h};
  const int fg = ceil_div_i(count, 8);
  if (exact) {
    energy_rows<true><<<grid, 256, 0, ctx->stream>>>(v, spins, nchunks, qp.p, hp.p);
    energy_finish<true><<<fg, 256, 0, ctx->stream>>>(count, nchunks, qp.p, hp.p, inst.cq, inst.ch,
                                                     inst.h_shift, E, Q, H);
  } else {
    energy_rows<false><<<grid, 256, 0, ctx->stream>>>(v, spins, nchunks, qp.p, hp.p);
    energy_finish<false><<<fg, 256, 0, ctx->stream>>>(count, nchunks, qp.p, hp.p, inst.cq, inst.ch,
                                                      0, E, nullptr, nullptr);
  }
  ISING_CUDA(ctx, cudaGetLastError());
  // the scratch buffers are freed when this function returns: wait for the kernels
  ISING_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
  return ISING_OK;
}

// Whether every spin was +-1; `odd` is the flag the packing kernel raised.
int read_odd(ising_ctx* ctx, const unsigned int* odd, bool* ok) {
  unsigned int o = 0;
  ISING_CUDA(ctx, cudaMemcpyAsync(&o, odd, 4, cudaMemcpyDeviceToHost, ctx->stream));
  ISING_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
  *ok = o == 0;
  return ISING_OK;
}

// The limbs of s^T I s by the planes form (spins known to be +-1 or the result
// is thrown away by the caller).
int plane_limbs(ising_ctx* ctx, const DevInstance& inst, int w, int planes, int shift,
                const int8_t* spins, int64_t count, unsigned long long* limbs) {
  const int64_t n = inst.n, ld = (n + 63) / 64 * 64, rows = 4 * ((n + 127) / 128);
  DevMem P, S, parts;
  ISING_TRY(dev_alloc(ctx, P, (size_t)planes * n * ld * 2));
  ISING_TRY(dev_alloc(ctx, S, (size_t)count * ld * 2));
  ISING_TRY(dev_alloc(ctx, parts, (size_t)planes * rows * count * 8));
  uint16_t* out = P.as<uint16_t>();
  switch (inst.j_dtype) {
    case ISING_F64: ISING_TRY(split_launch<double>(ctx, inst, ld, shift, w, planes, out)); break;
    case ISING_F32: ISING_TRY(split_launch<float>(ctx, inst, ld, shift, w, planes, out)); break;
    case ISING_I8: ISING_TRY(split_launch<int8_t>(ctx, inst, ld, shift, w, planes, out)); break;
    default: ISING_TRY(split_launch<int32_t>(ctx, inst, ld, shift, w, planes, out)); break;
  }
  spins_f16_kernel<<<pack_grid(ctx, (count * ld + 31) / 32), 256, 0, ctx->stream>>>(spins, count, n, ld,
                                                                                  S.as<uint16_t>());
  ISING_CUDA(ctx, cudaGetLastError());
  ISING_TRY(tc_plane_energies(ctx, n, ld, count, out, planes, S.p, parts.as<long long>()));
  join_digits_kernel<<<ceil_div_i(count, 8), 256, 0, ctx->stream>>>(count, rows, w, planes,
                                                                    parts.as<long long>(), limbs);
  ISING_CUDA(ctx, cudaGetLastError());
  return ISING_OK;
}

int energy_fixed(ising_ctx* ctx, const DevInstance& inst, bool exact, int shift, int splits,
                 const int8_t* spins, int64_t count, double* E, int64_t* Q, int64_t* H, bool* ok) {
  const int64_t n = inst.n, words = (n + 31) / 32;
  DevMem work;  // limbs [count][3], the flag (8 bytes), bits [count][words]
  ISING_TRY(dev_alloc(ctx, work, (size_t)count * 24 + 8 + (size_t)(count * words) * 4));
  ISING_CUDA(ctx, cudaMemsetAsync(work.p, 0, (size_t)count * 24 + 8, ctx->stream));
  unsigned long long* L = work.as<unsigned long long>();
  unsigned int* odd = reinterpret_cast<unsigned int*>(L + 3 * count);
  uint32_t* bw = reinterpret_cast<uint32_t*>(odd + 2);
  pack_rows_kernel<<<pack_grid(ctx, count * words), 256, 0, ctx->stream>>>(spins, count, n, words, bw, odd);
  ISING_CUDA(ctx, cudaGetLastError());
  int w = 0, planes = 0, pshift = 0, rc = ISING_ENOMEM;  // (or no room for the planes)
  // (from 16 vectors and 2^28 coupling-vectors on: n = 4096 takes 35 us per four
  // vectors in the fixed form and about 200 us for 256 in planes)
  if (count >= 16 && (double)n * (double)n * (double)count >= kPlaneTerms &&
      plane_scale(inst, &w, &planes, &pshift))
    rc = plane_limbs(ctx, inst, w, planes, pshift, spins, count, L);
  if (rc == ISING_OK) shift = pshift;
  else if (rc != ISING_ENOMEM) return rc;
  else switch (inst.j_dtype) {
    case ISING_F64: ISING_TRY(fixed_launch_t<double>(ctx, inst, shift, splits, bw, words, count, L)); break;
    case ISING_F32: ISING_TRY(fixed_launch_t<float>(ctx, inst, shift, splits, bw, words, count, L)); break;
    case ISING_I8: ISING_TRY(fixed_launch_t<int8_t>(ctx, inst, shift, splits, bw, words, count, L)); break;
    default: ISING_TRY(fixed_launch_t<int32_t>(ctx, inst, shift, splits, bw, words, count, L)); break;
  }
  const void* h = inst.has_h ? inst.h.p : nullptr;
  const double unscale = std::ldexp(1.0, -shift);
  if (exact)
    energy_fixed_finish<true><<<(unsigned)count, 256, 0, ctx->stream>>>(
        n, bw, words, L, h, inst.h_dtype, inst.h_shift, inst.cq, inst.ch, unscale, E, Q, H);
  else
    energy_fixed_finish<false><<<(unsigned)count, 256, 0, ctx->stream>>>(
        n, bw, words, L, h, inst.h_dtype, 0, inst.cq, inst.ch, unscale, E, nullptr, nullptr);
  ISING_CUDA(ctx, cudaGetLastError());
  return read_odd(ctx, odd, ok);
}

int energy_packed(ising_ctx* ctx, const DevInstance& inst, bool exact, const int8_t* spins,
                  int64_t count, double* E, int64_t* Q, int64_t* H, bool* ok) {
  const int64_t n = inst.n, words = (count + 31) / 32;
  const int64_t nchunks = (n + kRowsPerBlock - 1) / kRowsPerBlock;
  DevMem bits, qp, hp, odd;
  ISING_TRY(dev_alloc(ctx, bits, (size_t)(n * words) * 4));
  ISING_TRY(dev_alloc(ctx, qp, (size_t)(count * nchunks) * 8));
  ISING_TRY(dev_alloc(ctx, hp, (size_t)(count * nchunks) * 8));
  ISING_TRY(dev_alloc(ctx, odd, 4));
  ISING_CUDA(ctx, cudaMemsetAsync(odd.p, 0, 4, ctx->stream));
  pack_sites_kernel<<<pack_grid(ctx, (n * words + 31) / 32), 256, 0, ctx->stream>>>(
      spins, count, n, words, bits.as<uint32_t>(), odd.as<unsigned int>());
  const InstView iv = view(inst);
  RowsView<int32_t> v{iv.n, iv.layout, iv.j_dtype, iv.h_dtype, exact ? inst.h_shift : 0,
                      iv.J, iv.rowptr, iv.indices, iv.h};
  const dim3 grid((unsigned)nchunks, (unsigned)words);
  const int fg = ceil_div_i(count, 8);
  if (exact) {
    energy_packed_kernel<true><<<grid, 256, 0, ctx->stream>>>(v, bits.as<uint32_t>(), words, count,
                                                              nchunks, qp.p, hp.p);
    energy_finish<true><<<fg, 256, 0, ctx->stream>>>(count, nchunks, qp.p, hp.p, inst.cq, inst.ch,
                                                     inst.h_shift, E, Q, H);
  } else {
    energy_packed_kernel<false><<<grid, 256, 0, ctx->stream>>>(v, bits.as<uint32_t>(), words, count,
                                                               nchunks, qp.p, hp.p);
    energy_finish<false><<<fg, 256, 0, ctx->stream>>>(count, nchunks, qp.p, hp.p, inst.cq, inst.ch,
                                                      0, E, nullptr, nullptr);
  }
  ISING_CUDA(ctx, cudaGetLastError());
  return read_odd(ctx, odd.as<unsigned int>(), ok);
}

}  // namespace

// Which form runs: the fixed form for every dense J that one scale holds (at
// n = 4096 FP32: 256 vectors 23.5 ms in the general form, 2.5 in the fixed, 0.2
// in planes; one vector of n = 1000: 166 -> 6.4 us) but integers where the general
// form is faster (few_integers), the packed form for CSR instances where
// packed_pays, the general form otherwise and whenever a spin is not +-1.
//
// Integer dense J: the general form has two launches and a host read less (about
// 10 us) and adds in 64-bit integers without FP64, but a warp walks a row of n
// (65 ns per 1000 columns and row: 65 n us in all, n in thousands); a row and
// vector costs it 0.1 + 0.8 n ns and the fixed form 0.45 + 0.25 n. us per call,
// general / fixed, int8: n = 128, 16, 300 and 4000 vectors 102 / 109, 103 / 130,
// 188 / 364; n = 256: 106 / 107, 132 / 153, 361 / 629; n = 512, 16, 300 and 1000:
// 125 / 114, 194 / 203, 344 / 398; n = 1000, 1 and 64: 158 / 115, 217 / 158.
bool few_integers(const DevInstance& I, int64_t count) {
  const double n = (double)I.n, c = (double)count;
  return n * c * (0.35 - 0.55e-3 * n) > 65.0 * n - 10000.0 && (count < 16 || n * n * c < kPlaneTerms);
}

// The packed form: a launch and a host read more (about 25 us a call), and a
// warp walks a row alone, but a row of 32 vectors costs one warp instead of 32
// (0.15 ns each with integers, 0.55 in FP64). us per call, general / packed, n
// 20000: int8 of degree 4 and 8, 16, 32 vectors 187 / 188, 213 / 185, 262 / 185;
// of degree 128, 8 and 256 vectors 465 / 525, 1301 / 926; FP64 of degree 64, 8
// and 32 vectors 407 / 609, 737 / 612. n = 1000 of degree 8: int8, 32 and 256
// vectors 173 / 196, 210 / 201; FP64 187 / 197, 310 / 203.
bool packed_pays(const DevInstance& I, bool exact, int64_t count) {
  const int64_t row = std::min<int64_t>(kPackedRow, exact ? count : 2 * count);
  return count >= 8 && I.row_max <= row && (double)I.n * (double)count >= (exact ? 131072.0 : 65536.0);
}

int energy_device(ising_ctx* ctx, const DevInstance& inst, const int8_t* spins, int64_t count,
                  double* E, int64_t* Q, int64_t* H) {
  if (count <= 0) return ISING_OK;
  const bool exact = inst.j_integer && inst.j_absmax < 2147483648.0 && inst.h_dyadic;
  if (count > 65535) return fail(ctx, ISING_EINVAL, "energy: count > 65535 per call");
  bool ok = false;
  int shift = 0, splits = 1, rc = ISING_OK;
  if (inst.layout == ISING_LAYOUT_DENSE) {
    if (!(exact && few_integers(inst, count)) && fixed_scale(inst, &shift, &splits))
      rc = energy_fixed(ctx, inst, exact, shift, splits, spins, count, E, Q, H, &ok);
  } else if (packed_pays(inst, exact, count)) {
    rc = energy_packed(ctx, inst, exact, spins, count, E, Q, H, &ok);
  }
  // (no room for a form's scratch: the general form's is smaller)
  if (rc != ISING_OK && rc != ISING_ENOMEM) return rc;
  return rc == ISING_OK && ok ? ISING_OK : energy_general(ctx, inst, exact, spins, count, E, Q, H);
}

}  // namespace ising

// ---------------------------------------------------------------------------
// Energy with no allocation at all, for callers that cannot allocate device
// memory (a host that hands the library fixed buffers, or code running where
// cudaMalloc is not allowed, such as inside a stream being captured into a
// CUDA graph by someone else). The per-block partial sums live in one
// file-scope device array instead of a cudaMalloc'd buffer.

namespace ising {
namespace {

// Scratch for the no-allocation energy: 2 MiB per device, held by every GPU
// that loads this library until the process exits. One call needs
// count * ceil(n / 64) * 16 bytes of it.
constexpr size_t kNoAllocScratchBytes = size_t(2) << 20;
static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoAllocScratchBytes];

// Device address of g_noalloc_scratch per device, looked up by the first call
// made with that device current (the array's host-side name is not a device
// address). Threads racing on a first call store the same address; the slots
// are atomic so that the race is well defined. A device reset invalidates
// the cached address (the library does not reset devices).
constexpr int kMaxDevices = 64;
std::atomic<void*> g_noalloc_ptr[kMaxDevices];
thread_local char g_noalloc_err[256] = "";

int noalloc_fail(int code, const char* msg) {
  snprintf(g_noalloc_err, sizeof g_noalloc_err, "%s", msg);
  return code;
}

}  // namespace
}  // namespace ising

extern "C" const char* ising_energy_noalloc_error(void) { return ising::g_noalloc_err; }

extern "C" int ising_energy_noalloc(const ising_instance* inst, const int8_t* spins,
                                    int64_t count, double* E_out, void* stream) {
  using namespace ising;
  if (!inst || !spins || !E_out) return noalloc_fail(ISING_EINVAL, "inst, spins and E_out are required");
  if (inst->mem != ISING_MEM_DEVICE)
    return noalloc_fail(ISING_EINVAL, "the instance must be in device memory");
  if (inst->n < 1) return noalloc_fail(ISING_EINVAL, "n must be >= 1");
  if (inst->layout != ISING_LAYOUT_DENSE && inst->layout != ISING_LAYOUT_CSR)
    return noalloc_fail(ISING_EINVAL, "unknown layout");
  if (dtype_size(inst->j_dtype) == 0 || !inst->J) return noalloc_fail(ISING_EINVAL, "bad J");
  if (inst->layout == ISING_LAYOUT_CSR && (!inst->indptr || (!inst->indices && inst->nnz > 0)))
    return noalloc_fail(ISING_EINVAL, "CSR needs indptr and indices");
  if (inst->h && (dtype_size(inst->h_dtype) == 0 || inst->h_dtype == ISING_I8))
    return noalloc_fail(ISING_EINVAL, "h_dtype must be F64, F32 or I32");
  if (count < 0 || count > 65535) return noalloc_fail(ISING_EINVAL, "count must lie in [0, 65535]");
  if (count == 0) return ISING_OK;
  const int64_t nchunks = (inst->n + kRowsPerBlock - 1) / kRowsPerBlock;
  const size_t need = (size_t)count * (size_t)nchunks * 16;
  if (need > kNoAllocScratchBytes)
    return noalloc_fail(ISING_EINVAL,
                        "count * ceil(n / 64) * 16 bytes exceeds the 2 MiB no-allocation scratch");
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) {
    cudaGetLastError();
    return noalloc_fail(ISING_ECUDA, "no current CUDA device");
  }
  void* sp = g_noalloc_ptr[dev].load(std::memory_order_acquire);
  if (!sp) {
    cudaError_t e = cudaGetSymbolAddress(&sp, g_noalloc_scratch);
    if (e != cudaSuccess || !sp) {
      cudaGetLastError();
      return noalloc_fail(ISING_ECUDA, "cudaGetSymbolAddress of the scratch array failed");
    }
    g_noalloc_ptr[dev].store(sp, std::memory_order_release);
  }
  unsigned char* scratch = static_cast<unsigned char*>(sp);
  void* qp = scratch;
  void* hp = scratch + (size_t)count * nchunks * 8;
  const bool exact = (inst->j_dtype == ISING_I8 || inst->j_dtype == ISING_I32) &&
                     (!inst->h || inst->h_dtype == ISING_I32);
  double cq, ch;
  coefficients(inst, &cq, &ch);
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  dim3 grid((unsigned)nchunks, (unsigned)count);
  // integer h (I32) enters the exact sums unscaled
  const RowsView<int64_t> v{inst->n, inst->layout, inst->j_dtype, inst->h_dtype, 0, inst->J,
                            inst->indptr, inst->indices, inst->h};
  if (exact) {
    energy_rows<true><<<grid, 256, 0, st>>>(v, spins, nchunks, qp, hp);
    energy_finish<true><<<(unsigned)((count + 7) / 8), 256, 0, st>>>(
        count, nchunks, qp, hp, cq, ch, 0, E_out, nullptr, nullptr);
  } else {
    energy_rows<false><<<grid, 256, 0, st>>>(v, spins, nchunks, qp, hp);
    energy_finish<false><<<(unsigned)((count + 7) / 8), 256, 0, st>>>(
        count, nchunks, qp, hp, cq, ch, 0, E_out, nullptr, nullptr);
  }
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return noalloc_fail(ISING_ECUDA, cudaGetErrorString(e));
  return ISING_OK;
}
