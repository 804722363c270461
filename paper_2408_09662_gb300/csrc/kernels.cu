// Interpreter kernel, for programs that are too large to compile: W warps walk
// the instruction streams of one group of 32 instances (lane = instance), with
// CTA barriers between the phases that the host laid out (interp.cpp).  Every
// lane of a warp reads the same instruction, so the switch below never diverges
// within a warp.  The work vector lives in shared memory (slot-major, one column
// per lane: conflict-free) and, beyond that, in a global workspace in the
// instance-fastest layout, of which one group's columns stay in L2.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <type_traits>

#include "internal.h"

namespace cusadi {
namespace {

#include "math64.cuh"   // FP64 exp, sin, cos, division, square root on the integer pipe

__device__ __forceinline__ double op_exp(double a) { return cs_exp64(a); }
__device__ __forceinline__ double op_sin(double a) { return cs_sin64(a); }
__device__ __forceinline__ double op_cos(double a) { return cs_cos64(a); }
__device__ __forceinline__ double op_sqrt(double a) { return cs_sqrt64(a); }
__device__ __forceinline__ double op_div(double a, double b) { return cs_div64(a, b); }
__device__ __forceinline__ float op_exp(float a) { return expf(a); }
__device__ __forceinline__ float op_sin(float a) { return sinf(a); }
__device__ __forceinline__ float op_cos(float a) { return cosf(a); }
__device__ __forceinline__ float op_sqrt(float a) { return sqrtf(a); }
__device__ __forceinline__ float op_div(float a, float b) { return a / b; }

template <typename T>
__device__ __forceinline__ T eval_op(uint32_t op, T a, T b, T k) {
  const T Z = T(0), O = T(1);
  switch (op) {
    case ADD: return a + b;
    case SUB: return a - b;
    case MUL: return a * b;
    case DIV: return op_div(a, b);
    case NEG: return -a;
    case EXP: return op_exp(a);
    case LOG: return log(a);
    case POW: return pow(a, b);
    case SQ: return a * a;
    case SQRT: return op_sqrt(a);
    case SIN: return op_sin(a);
    case COS: return op_cos(a);
    case TAN: return tan(a);
    case ATAN: return atan(a);
    case ATAN2: return atan2(a, b);
    case TANH: return tanh(a);
    case FABS: return fabs(a);
    case FMIN: return fmin(a, b);
    case FMAX: return fmax(a, b);
    case FMA_CONST: return fma(k, a, b);
    case IF_ELSE_ZERO: return a != Z ? b : Z;
    case LT: return a < b ? O : Z;
    case LE: return a <= b ? O : Z;
    case EQ: return a == b ? O : Z;
    case NE: return a != b ? O : Z;
    case NOT: return a == Z ? O : Z;
    case AND: return (a != Z && b != Z) ? O : Z;
    case OR: return (a != Z || b != Z) ? O : Z;
    case ASIN: return asin(a);
    case ACOS: return acos(a);
    case SINH: return sinh(a);
    case COSH: return cosh(a);
    case ERF: return erf(a);
    case SIGN: return a > Z ? O : (a < Z ? -O : Z);
    case FLOOR: return floor(a);
    case CEIL: return ceil(a);
    case FMOD: return fmod(a, b);
    case INV: return op_div(O, a);
    case HYPOT: return hypot(a, b);
    case LOG1P: return log1p(a);
    case EXPM1: return expm1(a);
    case COPYSIGN: return copysign(a, b);
    case ASSIGN: return a;
  }
  return Z;
}

__device__ __forceinline__ double flip(double v, uint32_t sign) {
  return __hiloint2double((int)((uint32_t)__double2hiint(v) ^ sign), __double2loint(v));
}
__device__ __forceinline__ float flip(float v, uint32_t sign) {
  return __uint_as_float(__float_as_uint(v) ^ sign);
}
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ double add_rn(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float add_rn(float a, float b) { return __fadd_rn(a, b); }

// a * b rounded on its own, then added to or subtracted from c (or c from it);
// a subtraction is the addition of the negated operand, so the FP64 unit sees two
// instructions whichever it is
template <typename T>
__device__ __forceinline__ T mul_then(uint32_t op, T a, T b, T c) {
  return add_rn(flip(mul_rn(a, b), op == I_SUB_MUL ? 0x80000000u : 0u), flip(c, op == I_MUL_SUB ? 0x80000000u : 0u));
}
template <typename T>
__device__ __forceinline__ T interp_op(uint32_t op, T a, T b, T c) {
  if (op >= I_MUL_ADD) return mul_then(op, a, b, c);
  return eval_op<T>(op, a, b, c);
}

// B: buffer element type; S: work-slot type; MIXED: per-op precision tags.
// A warp stages its stream 32 instructions at a time: one coalesced load per lane,
// issued a batch ahead, then broadcast reads.  Bundles of multiply-adds on work
// slots, most of what linear algebra is made of, have their operands read together
// and are evaluated without decoding; other instructions (about 100 issued each)
// run one after the other.  Measured (GB300, ms; one thread per instance with the
// slots in HBM -> this): LDL^T FP64 n = 47, N = 16,384 16.7 -> 2.81, n = 100, N =
// 8,192 180 -> 15.5, n = 22, N = 65,536 2.36 -> 1.48; random 20k ops FP64, N =
// 16,384 8.6 -> 2.2; MPC mixed 19.8 -> 5.1.  The FP64 unit's share is 1.3 ms of the
// 2.81; barriers between phases and reads of workspace rows make up the rest.
// (Programs of a few dozen ops lose: quadrotor Jacobian FP32, N = 1,000,003, 0.140
// -> 0.155.)
template <typename B, typename S, bool MIXED>
__global__ void __launch_bounds__(512, 1) interp_kernel(
    const uint4* __restrict__ ops, const int32_t* __restrict__ begin, int ways, const S* __restrict__ K,
    const B* __restrict__ X, long long ldx, const B* __restrict__ X2, long long ldx2,
    long long split, B* __restrict__ Y, long long ldy, long long N, S* W,
    long long ldw, unsigned n_shared, int acc, int reduce, S* __restrict__ Wr, long long ldr) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  // one-warp groups come several to a CTA (their streams have no barriers)
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, warp = w % ways, grp = w / ways;
  const long long i0 = ((long long)blockIdx.x * ((blockDim.x >> 5) / ways) + grp) * 32 + lane;
  const bool active = i0 < N;
  const long long ix = active ? i0 : N - 1;  // inactive lanes read a valid column
  uint4* const stage = reinterpret_cast<uint4*>(smem_raw) + w * 64;
  S* const sm = reinterpret_cast<S*>(reinterpret_cast<uint4*>(smem_raw) + (blockDim.x >> 5) * 64) +
                grp * n_shared * 32 + lane;
  S* const gm = W + i0;                      // columns up to the next multiple of 128 exist (ldw)
  auto get = [&](unsigned o) -> S {
    if (o < n_shared) return sm[o * 32];
    const unsigned cls = o >> kOperandShift;
    const long long k = o & kOperandMask;
    if (cls == 0) return gm[(k - n_shared) * ldw];
    if (cls == 3) return K[k];
    const long long col = cls == 2 ? 0 : ix;
    return (S)(k < split ? X[k * ldx + col] : X2[(k - split) * ldx2 + col]);
  };
  auto any = [&](unsigned o) -> S* {         // a work slot of either tier
    return o < n_shared ? sm + o * 32 : gm + (long long)(o - n_shared) * ldw;
  };
  const int end = begin[warp + 1];
  int at = begin[warp];
  uint4 next = at + lane < end ? ops[at + lane] : make_uint4(I_NOP, 0, 0, 0);
  for (int turn = 0; at < end; at += 32, turn ^= 32) {
    stage[turn + lane] = next;
    __syncwarp();
    next = at + 32 + lane < end ? ops[at + 32 + lane] : make_uint4(I_NOP, 0, 0, 0);
    const int m = end - at < 32 ? end - at : 32;
    uint4 ahead = stage[turn];
    for (int t = 0; t < m;) {
      const uint4 o = ahead;
      const unsigned op = o.x & 127u, dst = o.x >> 8;
      if (!MIXED && op >= I_FAST) {          // kBundle multiply-adds on work slots
        const uint4* const d = stage + turn + t;
        t += kBundle;
        ahead = stage[turn + (t & 31)];
        S a[kBundle], b[kBundle], c[kBundle];
        unsigned code[kBundle];
        if (op < I_FAST_FAR) {
#pragma unroll
          for (int j = 0; j < kBundle; ++j) {
            const uint4 e = d[j];
            code[j] = e.x;
            a[j] = sm[e.y * 32];
            b[j] = sm[e.z * 32];
            c[j] = sm[e.w * 32];
          }
#pragma unroll
          for (int j = 0; j < kBundle; ++j)
            sm[(code[j] >> 8) * 32] = mul_then(I_MUL_ADD + (code[j] & 3u), a[j], b[j], c[j]);
        } else {
#pragma unroll
          for (int j = 0; j < kBundle; ++j) {
            const uint4 e = d[j];
            code[j] = e.x;
            a[j] = *any(e.y);
            b[j] = *any(e.z);
            c[j] = *any(e.w);
          }
#pragma unroll
          for (int j = 0; j < kBundle; ++j)
            *any(code[j] >> 8) = mul_then(I_MUL_ADD + (code[j] & 3u), a[j], b[j], c[j]);
        }
        continue;
      }
      ++t;
      ahead = stage[turn + (t & 31)];
      if (op == I_NOP) continue;
      if (op == I_SYNC) {
        __syncthreads();
        continue;
      }
      const S a = get(o.y);
      if (op == I_OUTPUT) {
        if (o.z && reduce) {   // reduced row z - 1: the instance's term, summed later
          if (active) Wr[(long long)(o.z - 1) * ldr + i0] = a;
        } else if (active) {
          B* p = &Y[dst * ldy + i0];
          *p = acc ? *p + (B)a : (B)a;
        }
        continue;
      }
      const S b = get(o.z), c = op >= I_MUL_ADD || op == FMA_CONST ? get(o.w) : S(0);
      S r;
      if (!MIXED || ((o.x >> 7) & 1u)) {
        r = interp_op<S>(op, a, b, c);
      } else {
        r = (S)interp_op<float>(op, (float)a, (float)b, (float)c);
      }
      if (dst < n_shared) sm[dst * 32] = r;
      else gm[(long long)(dst - n_shared) * ldw] = r;
    }
  }
}

template <typename B, typename S, bool MIXED>
int launch(const IOp* ops, const int32_t* begin, int ways, const void* k, const void* X, int64_t ldx,
           const void* X2, int64_t ldx2, int64_t split, void* Y, int64_t ldy, int64_t N, void* W,
           int64_t ldw, int64_t n_shared, int acc, int reduce, void* Wr, int64_t ldr,
           cudaStream_t st) {
  auto kern = interp_kernel<B, S, MIXED>;
  const int groups = ways == 1 && (size_t)n_shared * 128 * sizeof(S) <= 160 * 1024 ? 4 : 1;   // per CTA
  const size_t smem = (size_t)groups * ((size_t)n_shared * 32 * sizeof(S) + (size_t)ways * 64 * sizeof(uint4));
  const long long grid = (N + 32 * groups - 1) / (32 * groups);
  kern<<<(unsigned)grid, 32 * ways * groups, smem, st>>>(reinterpret_cast<const uint4*>(ops), begin, ways, (const S*)k,
                                                (const B*)X, ldx, (const B*)X2, ldx2, split, (B*)Y,
                                                ldy, N, (S*)W, ldw, (unsigned)n_shared, acc, reduce,
                                                (S*)Wr, ldr);
  return (int)cudaGetLastError();
}

// One CTA per reduced row: strided per-thread sums, then a tree, always in the
// same order, so the result has the same bits on every run.
template <typename B, typename S>
__global__ void __launch_bounds__(512) reduce_finish_kernel(const S* __restrict__ Wr, long long ldr,
                                                            long long N, const int64_t* __restrict__ rows,
                                                            B* __restrict__ Y, long long ldy, int accumulate) {
  __shared__ S s_[512];
  const S* __restrict__ P = Wr + (long long)blockIdx.x * ldr;
  S a = 0;
  for (long long j = threadIdx.x; j < N; j += 512) a += P[j];
  s_[threadIdx.x] = a;
  __syncthreads();
  for (int d = 256; d > 0; d >>= 1) {
    if ((int)threadIdx.x < d) s_[threadIdx.x] += s_[threadIdx.x + d];
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    B* p = &Y[rows[blockIdx.x] * ldy];
    *p = (B)(accumulate ? (S)*p + s_[0] : s_[0]);
  }
}

// One CTA per row of Y: S[r] = sum over j < N of Y[r * ldy + j], in the same
// order as reduce_finish_kernel (strided per-thread sums, then a tree).
template <typename T>
__global__ void __launch_bounds__(512) sum_rows_kernel(const T* __restrict__ Y, long long ldy,
                                                       long long N, T* __restrict__ S,
                                                       int accumulate) {
  __shared__ T s_[512];
  const T* __restrict__ P = Y + (long long)blockIdx.x * ldy;
  T a = 0;
  for (long long j = threadIdx.x; j < N; j += 512) a += P[j];
  s_[threadIdx.x] = a;
  __syncthreads();
  for (int d = 256; d > 0; d >>= 1) {
    if ((int)threadIdx.x < d) s_[threadIdx.x] += s_[threadIdx.x + d];
    __syncthreads();
  }
  if (threadIdx.x == 0) S[blockIdx.x] = accumulate ? S[blockIdx.x] + s_[0] : s_[0];
}

}  // namespace

// The shared-memory limit belongs to the kernel, which all functions and threads share:
// it is the device's own, set before the first launch and never lowered to one launch's.
int prepare_interp(int dtype) {
  int dev = 0, most = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (e != cudaSuccess) return (int)e;
  const auto attr = cudaFuncAttributeMaxDynamicSharedMemorySize;
  if (dtype == CUSADI_F64) return (int)cudaFuncSetAttribute(interp_kernel<double, double, false>, attr, most);
  if (dtype == CUSADI_F32) return (int)cudaFuncSetAttribute(interp_kernel<float, float, false>, attr, most);
  return (int)cudaFuncSetAttribute(interp_kernel<float, double, true>, attr, most);
}

int launch_interp(const IOp* ops, const int32_t* begin, int ways, const void* k, int dtype, const void* X,
                  int64_t ldx, const void* X2, int64_t ldx2, int64_t split, void* Y, int64_t ldy,
                  int64_t N, void* W, int64_t ldw, int64_t n_shared, int acc, int reduce,
                  void* Wr, int64_t ldr, void* stream) {
  cudaStream_t st = (cudaStream_t)stream;
  if (dtype == CUSADI_F64)
    return launch<double, double, false>(ops, begin, ways, k, X, ldx, X2, ldx2, split, Y, ldy, N, W, ldw, n_shared, acc, reduce, Wr, ldr, st);
  if (dtype == CUSADI_F32)
    return launch<float, float, false>(ops, begin, ways, k, X, ldx, X2, ldx2, split, Y, ldy, N, W, ldw, n_shared, acc, reduce, Wr, ldr, st);
  return launch<float, double, true>(ops, begin, ways, k, X, ldx, X2, ldx2, split, Y, ldy, N, W, ldw, n_shared, acc, reduce, Wr, ldr, st);
}

// Dense copy of one sparse output argument: dense[k * ldd + i] = y[(off +
// map[k]) * ldy + i] where map[k] >= 0 (a structural non-zero), else 0, k over
// the nrow * ncol entries (row-major).  Bound by HBM: a thread moves four 16-byte
// pieces of one entry's row (single elements where the rows' addresses do not allow
// whole pieces), its index looked up once.  One element and a 64-bit division per
// thread ran at less than half the bandwidth: 6 x 8 FP64, N = 1,000,003: 200 -> 88
// us, 6.7 TB/s.
template <typename T, int V>
struct alignas(V * sizeof(T)) Pack { T v[V]; };

template <typename T, int V>
__global__ void __launch_bounds__(256) densify_kernel(const T* __restrict__ y, int64_t ldy,
                                                      int64_t off, const int32_t* __restrict__ map,
                                                      int64_t n_dense, T* __restrict__ dense,
                                                      int64_t ldd, int64_t N) {
  constexpr int U = 4;
  const int64_t first = ((int64_t)blockIdx.x * U * 256 + threadIdx.x) * V;
  for (int64_t k = blockIdx.y; k < n_dense; k += gridDim.y) {
    const int32_t src = map[k];
    const T* const from = y + (off + src) * ldy;
    T* const to = dense + k * ldd;
    Pack<T, V> p[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int64_t i = first + (int64_t)u * 256 * V;
      if (src >= 0 && i + V <= N) p[u] = *reinterpret_cast<const Pack<T, V>*>(from + i);
      else
        for (int v = 0; v < V; ++v) p[u].v[v] = src >= 0 && i + v < N ? from[i + v] : T(0);
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int64_t i = first + (int64_t)u * 256 * V;
      if (i + V <= N) *reinterpret_cast<Pack<T, V>*>(to + i) = p[u];
      else
        for (int v = 0; v < V && i + v < N; ++v) to[i + v] = p[u].v[v];
    }
  }
}

template <typename T>
int densify(const T* y, int64_t ldy, int64_t off, const int32_t* map, int64_t n_dense, T* dense, int64_t ldd,
            int64_t N, cudaStream_t st) {
  constexpr int V = 16 / (int)sizeof(T);
  const bool whole = (uintptr_t)y % 16 == 0 && (uintptr_t)dense % 16 == 0 && ldy % V == 0 && ldd % V == 0;
  const int64_t per = (int64_t)256 * 4 * (whole ? V : 1);
  const dim3 grid((unsigned)((N + per - 1) / per), (unsigned)std::min<int64_t>(n_dense, 65535));
  if (whole) densify_kernel<T, V><<<grid, 256, 0, st>>>(y, ldy, off, map, n_dense, dense, ldd, N);
  else densify_kernel<T, 1><<<grid, 256, 0, st>>>(y, ldy, off, map, n_dense, dense, ldd, N);
  return (int)cudaGetLastError();
}

int launch_densify(int dtype, const void* y, int64_t ldy, int64_t off, const int32_t* map,
                   int64_t n_dense, void* dense, int64_t ldd, int64_t N, void* stream) {
  if (n_dense <= 0 || N <= 0) return 0;
  cudaStream_t st = (cudaStream_t)stream;
  if (dtype == CUSADI_F64)
    return densify((const double*)y, ldy, off, map, n_dense, (double*)dense, ldd, N, st);
  return densify((const float*)y, ldy, off, map, n_dense, (float*)dense, ldd, N, st);
}

int launch_reduce_finish(int dtype, const void* Wr, int64_t ldr, int64_t N, const int64_t* rows,
                         int64_t n_rows, void* Y, int64_t ldy, int accumulate, void* stream) {
  if (n_rows <= 0 || N <= 0) return 0;
  cudaStream_t st = (cudaStream_t)stream;
  if (dtype == CUSADI_F64)
    reduce_finish_kernel<double, double><<<(unsigned)n_rows, 512, 0, st>>>(
        (const double*)Wr, ldr, N, rows, (double*)Y, ldy, accumulate);
  else if (dtype == CUSADI_F32)
    reduce_finish_kernel<float, float><<<(unsigned)n_rows, 512, 0, st>>>(
        (const float*)Wr, ldr, N, rows, (float*)Y, ldy, accumulate);
  else
    reduce_finish_kernel<float, double><<<(unsigned)n_rows, 512, 0, st>>>(
        (const double*)Wr, ldr, N, rows, (float*)Y, ldy, accumulate);
  return (int)cudaGetLastError();
}

int launch_sum_rows(int dtype, const void* Y, int64_t ldy, int64_t rows, int64_t N, void* S,
                    int accumulate, void* stream) {
  if (rows <= 0) return 0;
  cudaStream_t st = (cudaStream_t)stream;
  if (dtype == CUSADI_F64)
    sum_rows_kernel<double><<<(unsigned)rows, 512, 0, st>>>((const double*)Y, ldy, N, (double*)S,
                                                            accumulate);
  else
    sum_rows_kernel<float><<<(unsigned)rows, 512, 0, st>>>((const float*)Y, ldy, N, (float*)S,
                                                           accumulate);
  return (int)cudaGetLastError();
}

}  // namespace cusadi
