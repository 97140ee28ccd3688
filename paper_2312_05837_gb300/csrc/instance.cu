// Upload and validation of an Ising instance (Sec. II: J real symmetric with
// zero diagonal, h real). Integer facts about J and h are gathered here so
// that the solver paths can choose exact integer energy accumulation.
#include "common.cuh"

#include <algorithm>
#include <cmath>
#include <type_traits>

namespace ising {
namespace {

struct ValFlags {
  unsigned int bad;             // bit 0 asymmetric, 1 diagonal, 2 CSR order/range, 3 indptr, 4 non-finite
  unsigned int j_nonint;        // some J value is not an integer
  unsigned long long j_absmax;  // bit pattern of max |J| (non-negative double)
  unsigned int h_mask;          // bit k: every h * 2^k is an integer below 2^30
  unsigned long long h_absmax;
  unsigned long long j_nonzeros;  // dense: non-zero J values, and the sum of
  long long j_expsum;             // their binary exponents (floor log2 |J|)
  int row_max;                    // CSR: entries of the longest row
};

// Facts gathered per thread and merged once per warp (a same-address atomic
// per element would serialise millions of updates).
struct LocalFacts {
  unsigned int bad = 0, nonint = 0;
  double absmax = 0.0;
  __device__ void note(double x) {
    if (!isfinite(x)) bad |= 16u;
    if (x != rint(x)) nonint = 1u;
    absmax = fmax(absmax, fabs(x));
  }
  __device__ void flush(ValFlags* f) {
    for (int o = 16; o; o >>= 1) {
      bad |= __shfl_xor_sync(0xffffffffu, bad, o);
      nonint |= __shfl_xor_sync(0xffffffffu, nonint, o);
      absmax = fmax(absmax, __shfl_xor_sync(0xffffffffu, absmax, o));
    }
    if ((threadIdx.x & 31) == 0) {
      if (bad) atomicOr(&f->bad, bad);
      if (nonint) atomicOr(&f->j_nonint, nonint);
      atomicMax(&f->j_absmax, (unsigned long long)__double_as_longlong(absmax));
    }
  }
};

// Facts of one stored type in that type's own arithmetic (GB300 runs FP64 at a
// sixty-fourth of the FP32 rate, so widening every element to FP64 made the
// check compute-bound: 174 us for n = 4096 FP32, against 10 us of traffic).
template <typename T>
struct TypedFacts {
  unsigned int bad = 0, nonint = 0;
  unsigned long long absbits = 0;  // max |x|: its bits (floats), its value (integers)
  unsigned int nonzeros = 0;
  int expsum = 0;
  __device__ void note(T x) {
    if constexpr (sizeof(T) == 8) {
      const unsigned long long u = (unsigned long long)__double_as_longlong(x) & 0x7FFFFFFFFFFFFFFFull;
      const int e = (int)(u >> 52);
      if (e == 0x7FF) bad |= 16u;
      if (!nonint && x != rint(x)) nonint = 1u;
      absbits = u > absbits ? u : absbits;
      if (u) { ++nonzeros; expsum += e ? e - 1023 : -1075; }
    } else if constexpr (std::is_same<T, float>::value) {
      const unsigned int u = __float_as_uint(x) & 0x7FFFFFFFu;
      const int e = (int)(u >> 23);
      if (e == 0xFF) bad |= 16u;
      if (x != rintf(x)) nonint = 1u;
      absbits = u > absbits ? u : absbits;
      if (u) { ++nonzeros; expsum += e ? e - 127 : -150; }
    } else {
      const unsigned int u = x < 0 ? 0u - (unsigned int)x : (unsigned int)x;
      absbits = u > absbits ? u : absbits;
      if (u) { ++nonzeros; expsum += 31 - __clz((int)u); }
    }
  }
  __device__ double absmax() const {
    if constexpr (sizeof(T) == 8) return __longlong_as_double((long long)absbits);
    else if constexpr (std::is_same<T, float>::value) return (double)__uint_as_float((unsigned int)absbits);
    else return (double)absbits;
  }
};

// x == y as the values compare (both zeros are equal; NaN is reported apart).
template <typename T>
__device__ __forceinline__ bool same_value(T x, T y) {
  if constexpr (sizeof(T) == 8) {
    const unsigned long long a = (unsigned long long)__double_as_longlong(x);
    const unsigned long long b = (unsigned long long)__double_as_longlong(y);
    return a == b || ((a | b) << 1) == 0;
  } else {
    return x == y;
  }
}

// Dense: J[i][j] == J[j][i] exactly, J[i][i] == 0, plus value facts. A block
// takes pairs of 32 x 32 tiles mirrored at the diagonal: both are read in row
// order, one is turned over through shared memory, so J is read once (a
// thread per element fetched its mirror image column by column).
template <typename T>
__global__ void __launch_bounds__(256) check_dense(const T* __restrict__ J, int64_t n, ValFlags* f,
                                                   bool structure) {
  __shared__ T tile[32][33];
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const int64_t nt = (n + 31) / 32, pairs = nt * (nt + 1) / 2;
  TypedFacts<T> lf;
  for (int64_t p = blockIdx.x; p < pairs; p += gridDim.x) {
    // p = bi (bi + 1) / 2 + bj, bj <= bi
    int64_t bi = (int64_t)((sqrtf(8.0f * (float)p + 1.0f) - 1.0f) * 0.5f);
    while (bi * (bi + 1) / 2 > p) --bi;
    while ((bi + 1) * (bi + 2) / 2 <= p) ++bi;
    const int64_t bj = p - bi * (bi + 1) / 2;
    T x[4], y[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int r = ty + 8 * k;
      const int64_t i = bi * 32 + r, j = bj * 32 + tx;
      const int64_t i2 = bj * 32 + r, j2 = bi * 32 + tx;
      x[k] = i < n && j < n ? J[i * n + j] : T(0);
      y[k] = i2 < n && j2 < n ? J[i2 * n + j2] : T(0);
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      lf.note(x[k]);
      if (bi != bj) lf.note(y[k]);
      tile[ty + 8 * k][tx] = x[k];
    }
    __syncthreads();
    if (structure) {
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int r = ty + 8 * k;
        if (!same_value(y[k], tile[tx][r])) lf.bad |= 1u;
        if (bi == bj && r == tx && x[k] != T(0)) lf.bad |= 2u;
      }
    }
    __syncthreads();
  }
  // merged once per warp (a same-address atomic per element would serialise
  // millions of updates)
  unsigned int bad = lf.bad, nonint = lf.nonint, nz = lf.nonzeros;
  int es = lf.expsum;
  double mx = lf.absmax();
  for (int o = 16; o; o >>= 1) {
    bad |= __shfl_xor_sync(0xffffffffu, bad, o);
    nonint |= __shfl_xor_sync(0xffffffffu, nonint, o);
    nz += __shfl_xor_sync(0xffffffffu, nz, o);
    es += __shfl_xor_sync(0xffffffffu, es, o);
    mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  }
  if (tx == 0) {
    if (bad) atomicOr(&f->bad, bad);
    if (nonint) atomicOr(&f->j_nonint, nonint);
    if (mx > 0.0) atomicMax(&f->j_absmax, (unsigned long long)__double_as_longlong(mx));
    if (nz) {
      atomicAdd(&f->j_nonzeros, (unsigned long long)nz);
      atomicAdd(reinterpret_cast<unsigned long long*>(&f->j_expsum), (unsigned long long)(long long)es);
    }
  }
}

__global__ void check_indptr(const int64_t* indptr, int64_t n, int64_t nnz, int32_t* rowptr,
                             ValFlags* f) {
  int64_t longest = 0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i <= n;
       i += (int64_t)gridDim.x * blockDim.x) {
    int64_t a = indptr[i];
    if (i == 0 && a != 0) atomicOr(&f->bad, 8u);
    if (i == n && a != nnz) atomicOr(&f->bad, 8u);
    if (i < n && indptr[i + 1] < a) atomicOr(&f->bad, 8u);
    if (i < n && indptr[i + 1] - a > longest) longest = indptr[i + 1] - a;
    rowptr[i] = (int32_t)a;
  }
  const int m = __reduce_max_sync(0xffffffffu, (int)min(longest, (int64_t)INT32_MAX));
  if ((threadIdx.x & 31) == 0 && m > 0) atomicMax(&f->row_max, m);
}

// CSR rows: columns in range, strictly increasing, no diagonal; each (i,j,v)
// has a partner (j,i,v) found by binary search in row j.
__global__ void check_csr(const int64_t* indptr, const int32_t* idx, const void* vals, int dt,
                          int64_t n, ValFlags* f, bool structure) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  const int64_t i0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int64_t trips = (n + stride - 1) / stride;
  LocalFacts lf;
  for (int64_t tr = 0; tr < trips; ++tr) {
    const int64_t i = i0 + tr * stride;
    if (i >= n) continue;
    int64_t a = indptr[i], b = indptr[i + 1];
    int32_t prev = -1;
    for (int64_t k = a; k < b; ++k) {
      int32_t j = idx[k];
      double x = load_as_double(vals, dt, k);
      lf.note(x);
      if (!structure) continue;
      if (j < 0 || j >= n || j <= prev) {
        lf.bad |= 4u;
        break;
      }
      prev = j;
      if (j == i) {
        lf.bad |= 2u;
        continue;
      }
      int64_t lo = indptr[j], hi = indptr[j + 1] - 1;
      bool found = false;
      while (lo <= hi) {
        int64_t mid = (lo + hi) >> 1;
        int32_t c = idx[mid];
        if (c == (int32_t)i) {
          found = (load_as_double(vals, dt, mid) == x);
          break;
        }
        if (c < (int32_t)i) lo = mid + 1; else hi = mid - 1;
      }
      if (!found) lf.bad |= 1u;
    }
  }
  lf.flush(f);
}

__global__ void check_h(const void* h, int dt, int64_t n, ValFlags* f) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  const int64_t i0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int64_t trips = (n + stride - 1) / stride;
  unsigned int bad = 0, mask_all = 0x1FFu;
  double amax = 0.0;
  for (int64_t tr = 0; tr < trips; ++tr) {
    const int64_t i = i0 + tr * stride;
    if (i >= n) continue;
    double x = load_as_double(h, dt, i);
    if (!isfinite(x)) bad |= 16u;
    amax = fmax(amax, fabs(x));
    unsigned int mask = 0;
    for (int k = 0; k <= 8; ++k) {
      double y = ldexp(x, k);
      if (y == rint(y) && fabs(y) < 1073741824.0) mask |= 1u << k;
    }
    mask_all &= mask;
  }
  for (int o = 16; o; o >>= 1) {
    bad |= __shfl_xor_sync(0xffffffffu, bad, o);
    mask_all &= __shfl_xor_sync(0xffffffffu, mask_all, o);
    amax = fmax(amax, __shfl_xor_sync(0xffffffffu, amax, o));
  }
  if ((threadIdx.x & 31) == 0) {
    if (bad) atomicOr(&f->bad, bad);
    atomicAnd(&f->h_mask, mask_all);
    atomicMax(&f->h_absmax, (unsigned long long)__double_as_longlong(amax));
  }
}

int grid_for(ising_ctx* ctx, int64_t work) {
  int64_t g = (work + 255) / 256;
  int64_t cap = (int64_t)ctx->sm_count * 8;
  if (g > cap) g = cap;
  if (g < 1) g = 1;
  return (int)g;
}

}  // namespace

int upload_instance(ising_ctx* ctx, const ising_instance* in, DevInstance* out, bool validate) {
  if (!in) return fail(ctx, ISING_EINVAL, "instance is NULL");
  if (in->n < 1) return fail(ctx, ISING_EINVAL, "n must be >= 1 (got %lld)", (long long)in->n);
  if (in->n > (int64_t)INT32_MAX - 1) return fail(ctx, ISING_EINVAL, "n too large");
  if (in->layout != ISING_LAYOUT_DENSE && in->layout != ISING_LAYOUT_CSR)
    return fail(ctx, ISING_EINVAL, "unknown layout %d", in->layout);
  if (dtype_size(in->j_dtype) == 0) return fail(ctx, ISING_EINVAL, "unknown j_dtype %d", in->j_dtype);
  if (in->h && (dtype_size(in->h_dtype) == 0 || in->h_dtype == ISING_I8))
    return fail(ctx, ISING_EINVAL, "h_dtype must be F64, F32 or I32");
  if (in->convention != ISING_CONV_PHYSICS && in->convention != ISING_CONV_PAPER)
    return fail(ctx, ISING_EINVAL, "unknown convention %d", in->convention);
  if (in->mem != ISING_MEM_HOST && in->mem != ISING_MEM_DEVICE)
    return fail(ctx, ISING_EINVAL, "unknown mem %d", in->mem);
  if (!std::isfinite(in->j_scale)) return fail(ctx, ISING_EINVAL, "j_scale must be finite");
  if (!in->J) return fail(ctx, ISING_EINVAL, "J is NULL");
  const int64_t n = in->n;
  cudaMemcpyKind kind = in->mem == ISING_MEM_HOST ? cudaMemcpyHostToDevice : cudaMemcpyDeviceToDevice;
  cudaStream_t st = ctx->stream;
  out->n = n;
  out->layout = in->layout;
  out->j_dtype = in->j_dtype;
  out->j_scale = in->j_scale;
  out->convention = in->convention;
  coefficients(in, &out->cq, &out->ch);
  const size_t jsz = dtype_size(in->j_dtype);

  DevMem flags;
  ISING_TRY(dev_alloc(ctx, flags, sizeof(ValFlags)));
  ValFlags f0{};
  f0.h_mask = 0x1FFu;
  ISING_CUDA(ctx, cudaMemcpyAsync(flags.p, &f0, sizeof f0, cudaMemcpyHostToDevice, st));
  ValFlags* fd = flags.as<ValFlags>();

  if (in->layout == ISING_LAYOUT_DENSE) {
    if ((uint64_t)n > 46340ull) return fail(ctx, ISING_EINVAL, "dense n too large");
    size_t bytes = (size_t)n * (size_t)n * jsz;
    ISING_TRY(dev_alloc(ctx, out->J, bytes));
    ISING_CUDA(ctx, cudaMemcpyAsync(out->J.p, in->J, bytes, kind, st));
    out->nnz = n * n;
    const int64_t nt = (n + 31) / 32;
    const int g = (int)std::min<int64_t>(nt * (nt + 1) / 2, (int64_t)ctx->sm_count * 8);
    switch (in->j_dtype) {
      case ISING_F64: check_dense<<<g, 256, 0, st>>>(out->J.as<double>(), n, fd, validate); break;
      case ISING_F32: check_dense<<<g, 256, 0, st>>>(out->J.as<float>(), n, fd, validate); break;
      case ISING_I8: check_dense<<<g, 256, 0, st>>>(out->J.as<int8_t>(), n, fd, validate); break;
      default: check_dense<<<g, 256, 0, st>>>(out->J.as<int32_t>(), n, fd, validate); break;
    }
    ISING_CUDA(ctx, cudaGetLastError());
  } else {
    if (!in->indptr || (!in->indices && in->nnz > 0))
      return fail(ctx, ISING_EINVAL, "CSR instance needs indptr and indices");
    if (in->nnz < 0 || in->nnz > (int64_t)INT32_MAX)
      return fail(ctx, ISING_EINVAL, "nnz out of range (%lld)", (long long)in->nnz);
    out->nnz = in->nnz;
    ISING_TRY(dev_alloc(ctx, out->J, (size_t)in->nnz * jsz));
    ISING_TRY(dev_alloc(ctx, out->indptr, (size_t)(n + 1) * 8));
    ISING_TRY(dev_alloc(ctx, out->rowptr, (size_t)(n + 1) * 4));
    ISING_TRY(dev_alloc(ctx, out->indices, (size_t)in->nnz * 4));
    if (in->nnz) {
      ISING_CUDA(ctx, cudaMemcpyAsync(out->J.p, in->J, (size_t)in->nnz * jsz, kind, st));
      ISING_CUDA(ctx, cudaMemcpyAsync(out->indices.p, in->indices, (size_t)in->nnz * 4, kind, st));
    }
    ISING_CUDA(ctx, cudaMemcpyAsync(out->indptr.p, in->indptr, (size_t)(n + 1) * 8, kind, st));
    check_indptr<<<grid_for(ctx, n + 1), 256, 0, st>>>(out->indptr.as<int64_t>(), n, in->nnz,
                                                       out->rowptr.as<int32_t>(), fd);
    ISING_CUDA(ctx, cudaGetLastError());
    ValFlags fh;
    ISING_CUDA(ctx, cudaMemcpyAsync(&fh, fd, sizeof fh, cudaMemcpyDeviceToHost, st));
    ISING_CUDA(ctx, cudaStreamSynchronize(st));
    if (fh.bad & 8u) return fail(ctx, ISING_EINVAL, "CSR indptr is not a valid offset array");
    check_csr<<<grid_for(ctx, n), 256, 0, st>>>(out->indptr.as<int64_t>(),
                                                out->indices.as<int32_t>(), out->J.p,
                                                in->j_dtype, n, fd, validate);
    ISING_CUDA(ctx, cudaGetLastError());
  }
  out->has_h = in->h != nullptr;
  out->h_dtype = in->h ? in->h_dtype : ISING_F64;
  if (in->h) {
    size_t hb = (size_t)n * dtype_size(in->h_dtype);
    ISING_TRY(dev_alloc(ctx, out->h, hb));
    ISING_CUDA(ctx, cudaMemcpyAsync(out->h.p, in->h, hb, kind, st));
    check_h<<<grid_for(ctx, n), 256, 0, st>>>(out->h.p, in->h_dtype, n, fd);
    ISING_CUDA(ctx, cudaGetLastError());
  }
  ValFlags fh;
  ISING_CUDA(ctx, cudaMemcpyAsync(&fh, fd, sizeof fh, cudaMemcpyDeviceToHost, st));
  ISING_CUDA(ctx, cudaStreamSynchronize(st));
  if (fh.bad & 16u) return fail(ctx, ISING_EINVAL, "J or h holds a non-finite value");
  if (fh.bad & 4u) return fail(ctx, ISING_EINVAL, "CSR columns out of range or not strictly increasing");
  if (fh.bad & 2u) return fail(ctx, ISING_EINVAL, "J has a non-zero diagonal");
  if (fh.bad & 1u) return fail(ctx, ISING_EINVAL, "J is not symmetric");
  out->j_integer = fh.j_nonint == 0;
  out->j_absmax = bits_to_double(fh.j_absmax);
  out->j_nonzeros = (int64_t)fh.j_nonzeros;
  out->j_expsum = fh.j_expsum;
  out->row_max = fh.row_max;
  out->h_absmax = in->h ? bits_to_double(fh.h_absmax) : 0.0;
  out->h_dyadic = true;
  out->h_shift = 0;
  if (in->h) {
    out->h_dyadic = fh.h_mask != 0;
    for (int k = 0; k <= 8; ++k)
      if (fh.h_mask & (1u << k)) { out->h_shift = k; break; }
  }
  return ISING_OK;
}

}  // namespace ising
