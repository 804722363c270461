// CUDA source generator: one straight-line kernel body per program segment.
//
// CusADi §III-A turns each instruction into one CUDA statement over a global
// work array (Listing 1, Listing 2).  Here each SSA value becomes a local
// variable, so the compiler keeps the work vector in registers; inputs are
// loaded at their first use and outputs stored right after they are computed,
// all instance-fastest so a warp touches 32 consecutive elements per row.
// Programs longer than segment_ops are split into several kernels that pass
// the values live across a cut through a workspace (same SoA layout).
//
// Launch shapes of the one-thread form: R consecutive instances per thread
// (every statement repeated per lane, rows moved as float2/float4/double2
// when the buffers allow), a register cap through the launch bounds, CTA
// barriers every few hundred ops, a register budget that moves the values
// past it to shared-memory slots, workspace rows or re-reads, and pairs of
// out-of-line math calls of the same function issued as one two-argument
// call.  The cooperative form (W warps per 32 instances, its schedule from
// plan_coop in coop.cpp) is generate_coop, further down.
#include <algorithm>
#include <cinttypes>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <set>
#include <sstream>

#include "internal.h"
#include "math64_text.h"   // kMath64Text: csrc/math64.cuh as text (made by the build)

namespace cusadi {

namespace {

std::string lit(double v, bool f64) {
  char buf[64];
  if (f64) {
    if (std::isnan(v)) return "__longlong_as_double(0x7ff8000000000000ll)";
    if (std::isinf(v)) return v > 0 ? "__longlong_as_double(0x7ff0000000000000ll)"
                                    : "__longlong_as_double((long long)0xfff0000000000000ull)";
    std::snprintf(buf, sizeof buf, "%a", v);
    return std::string("(") + buf + ")";
  }
  float f = (float)v;
  if (std::isnan(f)) return "__int_as_float(0x7fc00000)";
  if (std::isinf(f)) return f > 0 ? "__int_as_float(0x7f800000)" : "__int_as_float((int)0xff800000u)";
  std::snprintf(buf, sizeof buf, "%af", (double)f);
  return std::string("(") + buf + ")";
}

struct MathFn {
  const char* d;
  const char* f;
};

MathFn math_name(int op) {
  switch (op) {
    case EXP: return {"exp", "expf"};
    case LOG: return {"log", "logf"};
    case POW: return {"pow", "powf"};
    case SIN: return {"sin", "sinf"};
    case COS: return {"cos", "cosf"};
    case TAN: return {"tan", "tanf"};
    case ATAN: return {"atan", "atanf"};
    case ATAN2: return {"atan2", "atan2f"};
    case TANH: return {"tanh", "tanhf"};
    case ASIN: return {"asin", "asinf"};
    case ACOS: return {"acos", "acosf"};
    case SINH: return {"sinh", "sinhf"};
    case COSH: return {"cosh", "coshf"};
    case ERF: return {"erf", "erff"};
    case FMOD: return {"fmod", "fmodf"};
    case HYPOT: return {"hypot", "hypotf"};
    case LOG1P: return {"log1p", "log1pf"};
    case EXPM1: return {"expm1", "expm1f"};
    case SQRT: return {"sqrt", "sqrtf"};
    case DIV: case INV: return {"div", "div"};
    case FABS: return {"fabs", "fabsf"};
    case FMIN: return {"fmin", "fminf"};
    case FMAX: return {"fmax", "fmaxf"};
    case FLOOR: return {"floor", "floorf"};
    case CEIL: return {"ceil", "ceilf"};
    case COPYSIGN: return {"copysign", "copysignf"};
  }
  return {"?", "?"};
}

struct Gen {
  const Graph& g;
  const CodegenOptions& o;
  std::vector<int> seg_of;          // per node (leaves: -1)
  std::vector<int> last_seg;        // last segment that reads the node
  std::vector<int64_t> ws_slot;     // workspace row of values crossing a cut
  std::vector<std::vector<int64_t>> out_rows;  // per node: output rows it feeds
  std::set<std::pair<int, bool>> calls;        // (op, f64) of out-of-line math used
  std::set<std::pair<int, bool>> calls2;       // (op, f64) of the paired (two-argument) versions
  bool own_f32 = false;                        // own FP32 sin/cos/exp used
  bool own_f64 = false;                        // FP64 math of math64.cuh used
  std::set<std::string> wrappers;              // out-of-line wrappers of math64.cuh functions used

  Gen(const Graph& g_, const CodegenOptions& o_) : g(g_), o(o_) {}

  bool node_f64(int32_t i) const {
    if (o.dtype == CUSADI_F64) return true;
    if (o.dtype == CUSADI_F32) return false;
    return g.nodes[i].f64 != 0;
  }
  const char* ty(bool f64) const { return f64 ? "double" : "float"; }
  bool buf_f64() const { return o.dtype == CUSADI_F64; }
  bool ws_f64() const { return o.dtype != CUSADI_F32; }
  // no value of its own to compute: inputs, constants, multiplies that joined their readers
  bool leaf(int32_t i) const {
    return g.nodes[i].op == INPUT || g.nodes[i].op == CONST || (!g.gone.empty() && g.gone[i]);
  }
};

// Whether op is inlined at its uses (else one out-of-line function per op and
// precision, called from every use).
bool inlined(int op, int inline_math) {
  if (inline_math == 1) return true;
  if (inline_math == 2) return op == EXP || op == EXPM1 || op == LOG || op == LOG1P;
  return false;
}

// FP64 functions that run on the integer pipe (math64.cuh), where the
// straight-line kernels leave it idle; an FP64 instruction occupies its unit 64
// clocks per warp.  Weights in FMAs, library -> ours, from long chains of one op:
// exp 15 -> 1.2, sin/cos 18 -> 4.4, div 7.7 -> 1.9, sqrt 8.2 -> 1.9.
bool own_f64_math(int op) {
  return op == EXP || op == SIN || op == COS || op == DIV || op == INV || op == SQRT;
}

// __launch_bounds__ of a kernel of `threads` threads per CTA: a register cap
// becomes the minimum number of resident CTAs per SM that leaves each thread
// at most that many registers (a plain --maxrregcount is ignored for kernels
// with launch bounds).
std::string launch_bounds(int threads, int maxrregcount) {
  std::string s = "__launch_bounds__(" + std::to_string(threads);
  if (maxrregcount > 0) s += ", " + std::to_string(std::max(1, 65536 / (threads * maxrregcount)));
  return s + ")";
}

// Register cap of a one-thread kernel when the caller names none; 0 leaves it
// to the compiler.  live: 32-bit registers' worth of values live at once; a
// kernel needs about 20 more.
//  * above the 255 a thread can have, the cap is 255: with calls to out-of-line
//    functions the compiler else settles on as few as 32 registers and spills
//    the rest (LQR step, 510 live: 179 KB of spill stores at 32 registers and
//    1.24 ms, 33 KB at 255; MPC mixed 1.65 -> 1.35 ms);
//  * 129 to 168 would hold 12 warps per SM, at most 128 holds 16: cap 128 (FP32
//    random 20k-op program at N = 65,536, 165 registers: 0.61 -> 0.35 ms; FP64
//    cart-pole, 138 registers: 0.075 -> 0.059 ms).
int auto_register_cap(int64_t live) {
  const int64_t need = live + 20;
  if (need > 255) return 255;
  return need > 128 && need <= 168 ? 128 : 0;
}

// out-of-line forms of math64.cuh's functions with several results or arguments
const char* const kRecip = "static __device__ __noinline__ cs_u64 cs_recip_d(double b) { return cs_recip64(b); }\n";
const char* const kDivr = "static __device__ __noinline__ double cs_divr_d(double a, double b, cs_u64 r) "
                          "{ return cs_divr64(a, b, r); }\n";
const char* const kDivr2 = "static __device__ __noinline__ double2 cs_divr2_d(double a, double b, double d, cs_u64 r) "
                           "{ double2 q; cs_divr64x2(a, b, d, r, q.x, q.y); return q; }\n";
const char* const kSincos = "static __device__ __noinline__ double2 cs_sincos_d(double x) "
                            "{ double2 r; cs_sincos64(x, r.x, r.y); return r; }\n";

const char* const kSincosF = "static __device__ __noinline__ float2 cs_sincos_f(float x) "
                             "{ float2 r; sincosf(x, &r.x, &r.y); return r; }\n";

// FP32 division by a constant c > 0 without the compiler's range check and branch,
// which keep it from overlapping one division with the next.  r is 1/c rounded to
// nearest, q the product x r and e the residual q c - x, exact where both are scaled up
// by 2^64 (|x| < 1).  When q is within an ulp of x/c, q - e r rounds x/c to nearest
// (P. Markstein, "Computation of elementary functions on the IBM RISC System/6000
// processor", 1990): |c r - 1| <= 2^-25 makes it so; for other constants q takes in
// l = 1/c - r as well (cs_divc2_f).
// Subnormal quotients: q - e/c lies halfway between two of them or off the half by at
// least 1/C of it, C the integer of c's mantissa.  An odd C below 2^24 leaves no
// halves, and the one rounding of q - e r decides as q - e/c would.  An even C
// (`even`) has halves, and is off by 2/C else: e r is rounded on its own, which keeps
// the halves (|c r - 1| <= 2^-25, or the sum with l: 1 when rounded) and no other.
// Overflow: a product past the largest finite value (c < 1) stays there, and the
// residual decides.  An infinite x, whose residual is a NaN otherwise, stays.
// Bits of x / c for 2^-20 <= c < 2^24 (powers of two: exact_reciprocal).  SRB step FP32,
// 75 such divisions, N = 4,096: 6.49 -> 5.88 us, its adjoint 15.1 -> 13.2, N = 65,536: 9.1
// -> 8.4 and 35.6 -> 30.5.
const char* const kDivc = R"(static __device__ __forceinline__ float cs_divc_f(float x, float c, float r, bool even) {
  const bool t = fabsf(x) < 1.0f, small = c < 1.0f;
  const float S = t ? 0x1p+64f : 1.0f, p = __fmul_rn(x, r);
  const float q = small ? fmaxf(fminf(p, 0x1.fffffep+127f), -0x1.fffffep+127f) : p;
  const float d = fmaf(__fmul_rn(q, S), c, -__fmul_rn(x, S)), e = small ? d : fminf(d, 0x1p+126f);
  return even ? fmaf(__fmul_rn(e, -r), t ? 0x1p-64f : 1.0f, q) : fmaf(e, t ? r * -0x1p-64f : -r, q);
}
)";
const char* const kDivc2 = R"(static __device__ __forceinline__ float cs_divc2_f(float x, float c, float r, float l, bool even) {
  const bool t = fabsf(x) < 1.0f, small = c < 1.0f;
  const float S = t ? 0x1p+64f : 1.0f, a = fabsf(x);
  const float p = fmaf(a, r, __fmul_rn(a, l)), q = small ? fminf(p, 0x1.fffffep+127f) : p;
  const float e = fmaf(__fmul_rn(q, S), c, -__fmul_rn(a, S));
  const float y = even ? fmaf(fmaf(e, -r, __fmul_rn(e, -l)), t ? 0x1p-64f : 1.0f, q) : fmaf(e, t ? r * -0x1p-64f : -r, q);
  return copysignf(a < __int_as_float(0x7f800000) ? y : a, x);
}
)";

// 2^64 / b of b's mantissa in [1, 2) (2^64 - 1 for 1), as cs_recip64 returns
uint64_t recip_of(double b) {
  uint64_t u;
  std::memcpy(&u, &b, 8);
  const uint64_t m = (u & 0xfffffffffffffull) | 1ull << 52;
  if (m == 1ull << 52) return ~0ull;
  return (uint64_t)(((unsigned __int128)1 << 116) / m);
}
// 1/k of a constant power of two, where it is as exact as the division and one multiply;
// 0: k is none, or its reciprocal no normal number
double exact_reciprocal(const Node& b, bool f64) {
  int e;
  const double k = f64 ? b.k : (double)(float)b.k;
  if (b.op != CONST || std::fabs(std::frexp(k, &e)) != 0.5 || std::abs(e - 1) > (f64 ? 1022 : 126)) return 0.0;
  return 1.0 / k;
}
// divisors that the constant form takes: normal, and inside cs_div_far's range
bool const_divisor(const Node& b) {
  const double m = std::fabs(b.k);
  return b.op == CONST && m >= 0x1p-509 && m < 0x1p+513 && exact_reciprocal(b, true) == 0.0;
}

// the function itself, to be inlined where it is named
std::string math_fn(int op, bool f64) {
  MathFn m = math_name(op);
  if (f64 && own_f64_math(op)) return std::string("cs_") + m.d + "64";
  return f64 ? m.d : m.f;
}

std::string call_name(int op, bool f64, bool inl) {
  MathFn m = math_name(op);
  if (inl) return math_fn(op, f64);
  return std::string("cs_") + m.d + (f64 ? "_d" : "_f");
}

// The engine's own single-precision sin, cos and exp (FP32 ops when the
// library's are not inlined): Cody & Waite argument reduction with an FMA per
// step and near-minimax polynomials; constants from csrc/gen_math_coeffs.py.
// sin/cos take the fast path for |x| <= 128 * pi/2, where the 17-bit leading
// parts of pi/2 make j * part exact; anything else (and inf/NaN) goes to the
// library function.  Branch-free apart from that rare fallback.
bool own_f32_math(int op) { return op == SIN || op == COS || op == EXP; }

const char* kOwnMathF32 = R"(static __device__ __noinline__ float cs_sin_slow(float a) { return sinf(a); }
static __device__ __noinline__ float cs_cos_slow(float a) { return cosf(a); }
static __device__ __forceinline__ void cs_sincos_core(float x, float& s, float& c, int& q) {
  const float j = rintf(x * 0x1.45f306p-1f);
  float r = fmaf(-j, 0x1.922p+0f, x);
  r = fmaf(-j, -0x1.2aefp-18f, r);
  r = fmaf(-j, 0x1.68c234p-39f, r);
  q = (int)j;
  const float t = r * r;
  s = fmaf(r * t, fmaf(t, fmaf(t, -0x1.9943ep-13f, 0x1.11073ap-7f), -0x1.555546p-3f), r);
  c = fmaf(t, fmaf(t, fmaf(t, fmaf(t, 0x1.99169ep-16f, -0x1.6c07f2p-10f), 0x1.55553cp-5f), -0x1p-1f), 1.0f);
}
static __device__ __forceinline__ float cs_own_sin_f(float x) {
  if (!(fabsf(x) <= 201.0f)) return cs_sin_slow(x);
  float s, c; int q;
  cs_sincos_core(x, s, c, q);
  const float v = (q & 1) ? c : s;
  return (q & 2) ? -v : v;
}
static __device__ __forceinline__ float cs_own_cos_f(float x) {
  if (!(fabsf(x) <= 201.0f)) return cs_cos_slow(x);
  float s, c; int q;
  cs_sincos_core(x, s, c, q);
  const float v = (q & 1) ? s : c;
  return ((q + 1) & 2) ? -v : v;
}
static __device__ __forceinline__ float cs_own_exp_f(float x) {
  const float xc = x < -104.0f ? -104.0f : (x > 89.0f ? 89.0f : x);
  const float k = rintf(xc * 0x1.715476p+0f);
  float r = fmaf(-k, 0x1.62e4p-1f, xc);
  r = fmaf(-k, 0x1.7f7d1cp-20f, r);
  float p = fmaf(r, 0x1.6a2448p-10f, 0x1.1239d4p-7f);
  p = fmaf(r, p, 0x1.5558f2p-5f);
  p = fmaf(r, p, 0x1.555492p-3f);
  p = fmaf(r, p, 0x1.fffffcp-2f);
  p = fmaf(r * r, p, r) + 1.0f;
  const int ki = (int)k, k1 = ki >> 1, k2 = ki - k1;
  return (p * __int_as_float((k1 + 127) << 23)) * __int_as_float((k2 + 127) << 23);
}
)";

// Own math as generated: mode 1 inlines sin/cos/exp at every use, mode 2 makes
// them out-of-line functions (one copy of the code, a call per use).
std::string own_math_source(int mode) {
  std::string t = kOwnMathF32;
  if (mode == 2) {
    const std::string a = "__forceinline__ float cs_own_", b = "__noinline__ float cs_own_";
    for (size_t p = t.find(a); p != std::string::npos; p = t.find(a, p + b.size())) t.replace(p, a.size(), b);
  }
  return t;
}

// Accesses of NL consecutive instances of one row by one thread (NL = 2 or 4):
// one vector load/store when `full` (the caller checked alignment and that all
// NL instances are inside the batch), else one element at a time, the lanes
// past the batch's end reading lane 0's element and storing nothing.
const char* kLaneAccess = R"(template <typename T> struct cs_vec2;
template <> struct cs_vec2<float> { typedef float2 t; };
template <> struct cs_vec2<double> { typedef double2 t; };
template <typename T>
static __device__ __forceinline__ void cs_ld2(const T* __restrict__ p, bool full, int m, T& a, T& b) {
  if (full) { const typename cs_vec2<T>::t v = *reinterpret_cast<const typename cs_vec2<T>::t*>(p); a = v.x; b = v.y; }
  else { a = p[0]; b = m > 1 ? p[1] : a; }
}
template <typename T>
static __device__ __forceinline__ void cs_st2(T* __restrict__ p, bool full, int m, T a, T b) {
  if (full) { typename cs_vec2<T>::t v; v.x = a; v.y = b; *reinterpret_cast<typename cs_vec2<T>::t*>(p) = v; }
  else { p[0] = a; if (m > 1) p[1] = b; }
}
static __device__ __forceinline__ void cs_ld4(const float* __restrict__ p, bool full, int m, float& a, float& b,
                                              float& c, float& d) {
  if (full) { const float4 v = *reinterpret_cast<const float4*>(p); a = v.x; b = v.y; c = v.z; d = v.w; }
  else { a = p[0]; b = m > 1 ? p[1] : a; c = m > 2 ? p[2] : a; d = m > 3 ? p[3] : a; }
}
static __device__ __forceinline__ void cs_st4(float* __restrict__ p, bool full, int m, float a, float b, float c,
                                              float d) {
  if (full) *reinterpret_cast<float4*>(p) = make_float4(a, b, c, d);
  else { p[0] = a; if (m > 1) p[1] = b; if (m > 2) p[2] = c; if (m > 3) p[3] = d; }
}
static __device__ __forceinline__ void cs_ld4(const double* __restrict__ p, bool full, int m, double& a, double& b,
                                              double& c, double& d) {
  if (full) { cs_ld2(p, true, 2, a, b); cs_ld2(p + 2, true, 2, c, d); }
  else { a = p[0]; b = m > 1 ? p[1] : a; c = m > 2 ? p[2] : a; d = m > 3 ? p[3] : a; }
}
static __device__ __forceinline__ void cs_st4(double* __restrict__ p, bool full, int m, double a, double b,
                                              double c, double d) {
  if (full) { cs_st2(p, true, 2, a, b); cs_st2(p + 2, true, 2, c, d); }
  else { p[0] = a; if (m > 1) p[1] = b; if (m > 2) p[2] = c; if (m > 3) p[3] = d; }
}
)";

// C expression of node i, in precision f, with its operands' expressions (operands()).
std::string op_expr(Gen& G, int64_t i, bool f, const std::string& A, const std::string& B, const std::string& C,
                    const CodegenOptions& o) {
  const Node& x = G.g.nodes[i];
  const char* T = G.ty(f);
  const int32_t m = G.g.fused.empty() ? -1 : G.g.fused[i];
  if (m >= 0) {   // contract() joined a multiply: the compiler contracts nothing itself
    const std::string& F = G.g.nodes[m].op == SQ ? A : B;
    return std::string(f ? "fma(" : "fmaf(") + (x.op == SUB && x.b == m ? "-" : "") + A + ", " + F + ", " +
           (x.op == SUB && x.a == m ? "-" : "") + C + ")";
  }
  std::string Z = std::string("(") + T + ")0", One = std::string("(") + T + ")1";
  std::string e;
  const MathFn fn = math_name(x.op);
  const char* mn = f ? fn.d : fn.f;
  if (x.op == DIV) {
    const double r = exact_reciprocal(G.g.nodes[x.b], f);
    if (r != 0.0) return A + " * " + lit(r, f);
  }
  if (f && own_f64_math(x.op)) {
    const int op = x.op == INV ? (int)DIV : (int)x.op;
    const bool inl = inlined(op, o.inline_math);
    if (op == DIV && const_divisor(G.g.nodes[x.op == INV ? x.a : x.b])) {
      const double b = G.g.nodes[x.op == INV ? x.a : x.b].k;
      G.own_f64 = true;
      if (!inl) G.wrappers.insert(kDivr);
      char r[32];
      std::snprintf(r, sizeof r, "0x%016" PRIx64 "ull", recip_of(b));
      return std::string(inl ? "cs_divr64(" : "cs_divr_d(") + (x.op == INV ? One : A) + ", " + lit(b, true) + ", " + r + ")";
    }
    if (!inl) G.calls.insert({op, true});
    G.own_f64 = true;
    return call_name(op, true, inl) + "(" + (x.op == INV ? One + ", " : "") + A + (x.op == DIV ? ", " + B : "") + ")";
  }
  switch (x.op) {
    case ADD: e = A + " + " + B; break;
    case SUB: e = A + " - " + B; break;
    case MUL: e = A + " * " + B; break;
    case DIV: {
      e = A + " / " + B;
      const Node& b = G.g.nodes[x.b];
      const float c = std::fabs((float)b.k);
      if (!f && b.op == CONST && c >= 0x1p-20f && c < 0x1p+24f) {
        const float r = (float)(1.0 / (double)c);
        const double off = (double)c * r - 1.0;          // c r is exact in double
        const bool one = std::fabs(off) <= 0x1p-25;
        uint32_t bits;
        std::memcpy(&bits, &c, 4);
        G.wrappers.insert(one ? kDivc : kDivc2);
        e = std::string(b.k < 0 ? "-" : "") + (one ? "cs_divc_f(" : "cs_divc2_f(") + A + ", " + lit(c, false) + ", " +
            lit(r, false) + (one ? "" : ", " + lit(-off / (double)c, false)) + (bits & 1 ? ", false)" : ", true)");
      }
      break;
    }
    case NEG: e = "-" + A; break;
    case SQ: e = A + " * " + A; break;
    case INV: e = One + " / " + A; break;
    case SQRT: case FABS: case FLOOR: case CEIL: e = std::string(mn) + "(" + A + ")"; break;
    case FMIN: case FMAX: case COPYSIGN: e = std::string(mn) + "(" + A + ", " + B + ")"; break;
    case FMA_CONST: e = std::string(f ? "fma(" : "fmaf(") + lit(x.k, f) + ", " + A + ", " + B + ")"; break;
    case IF_ELSE_ZERO: e = "(" + A + " != " + Z + " ? " + B + " : " + Z + ")"; break;
    case LT: e = "(" + A + " < " + B + " ? " + One + " : " + Z + ")"; break;
    case LE: e = "(" + A + " <= " + B + " ? " + One + " : " + Z + ")"; break;
    case EQ: e = "(" + A + " == " + B + " ? " + One + " : " + Z + ")"; break;
    case NE: e = "(" + A + " != " + B + " ? " + One + " : " + Z + ")"; break;
    case NOT: e = "(" + A + " == " + Z + " ? " + One + " : " + Z + ")"; break;
    case AND: e = "((" + A + " != " + Z + " && " + B + " != " + Z + ") ? " + One + " : " + Z + ")"; break;
    case OR: e = "((" + A + " != " + Z + " || " + B + " != " + Z + ") ? " + One + " : " + Z + ")"; break;
    case SIGN: e = "(" + A + " > " + Z + " ? " + One + " : (" + A + " < " + Z + " ? -" + One + " : " + Z + "))"; break;
    default:
      if (!f && o.inline_math != 1 && o.own_math && own_f32_math(x.op)) {
        G.own_f32 = true;
        e = std::string(x.op == SIN ? "cs_own_sin_f(" : (x.op == COS ? "cs_own_cos_f(" : "cs_own_exp_f(")) + A + ")";
      } else if (op_call(x.op)) {
        const bool inl = inlined(x.op, o.inline_math);
        if (!inl) G.calls.insert({x.op, f});
        e = call_name(x.op, f, inl) + "(" + A + (op_arity(x.op) == 2 ? ", " + B : "") + ")";
      } else {
        e = "/* unsupported op */ " + Z;
      }
  }
  return e;
}

}  // namespace

std::string finish_source(CodegenResult& R, const std::string& prefix, const char* tin,
                          const char* tw);

CodegenResult generate(const Graph& g, const CodegenOptions& o) {
  CodegenResult R;
  Gen G(g, o);
  const int64_t n = (int64_t)g.nodes.size();
  G.seg_of.assign(n, -1);
  G.last_seg.assign(n, -1);
  G.out_rows.assign(n, {});
  for (size_t r = 0; r < g.out.size(); ++r) G.out_rows[g.out[r]].push_back((int64_t)r);

  // segment cuts by op count
  std::vector<std::pair<int64_t, int64_t>> segs;
  {
    int64_t start = 0, ops = 0;
    for (int64_t i = 0; i < n; ++i) {
      if (G.leaf(i)) continue;
      if (o.segment_ops > 0 && ops >= o.segment_ops) {
        segs.push_back({start, i});
        start = i;
        ops = 0;
      }
      ++ops;
    }
    segs.push_back({start, n});
  }
  const int nseg = (int)segs.size();
  for (int s = 0; s < nseg; ++s)
    for (int64_t i = segs[s].first; i < segs[s].second; ++i)
      if (!G.leaf(i)) G.seg_of[i] = s;
  for (int64_t i = 0; i < n; ++i) {
    const Node& x = g.nodes[i];
    if (G.leaf(i)) continue;
    for (int32_t a : operands(g, i))
      if (a >= 0 && !G.leaf(a)) G.last_seg[a] = std::max(G.last_seg[a], G.seg_of[i]);
  }
  // workspace rows for values read in a later segment; a row is free again for
  // values defined after the segment of its last reader
  G.ws_slot.assign(n, -1);
  {
    std::vector<std::vector<int64_t>> release(nseg + 1);
    std::vector<int64_t> free_rows;
    int64_t rows = 0;
    for (int s = 0; s < nseg; ++s) {
      for (int64_t r : release[s > 0 ? s - 1 : nseg]) free_rows.push_back(r);
      if (s > 0) release[s - 1].clear();
      for (int64_t i = segs[s].first; i < segs[s].second; ++i) {
        if (G.leaf(i) || G.last_seg[i] <= s) continue;
        int64_t r;
        if (!free_rows.empty()) { r = free_rows.back(); free_rows.pop_back(); }
        else r = rows++;
        G.ws_slot[i] = r;
        release[G.last_seg[i]].push_back(r);
      }
    }
    R.ws_rows = rows;
  }
  for (uint8_t f : g.out_reduce) R.has_reduce |= (f != 0);
  std::vector<int64_t> reduce_k(g.out_reduce.size(), -1);
  for (size_t r = 0; r < g.out_reduce.size(); ++r)
    if (g.out_reduce[r]) {
      reduce_k[r] = (int64_t)R.reduce_rows.size();
      R.reduce_rows.push_back((int64_t)r);
    }

  const char* tin = G.buf_f64() ? "double" : "float";
  const char* tw = G.ws_f64() ? "double" : "float";
  // Register budget (spill_values > 0, one instance per thread): per segment, a
  // linear scan over the values' live ranges in statement order keeps at most
  // spill_values of them in registers; when a value finds the budget full,
  // whichever of it and the live register values is read last leaves the
  // registers for its whole life (M. Poletto and V. Sarkar, "Linear scan
  // register allocation", TOPLAS 1999).  An input or a value carried from an
  // earlier kernel is then re-read from its buffer at each use; a computed value
  // is stored once to a shared-memory slot (spill_shared_kb per CTA), or beyond
  // those to a workspace row, and re-read at each use.  Accesses go through
  // volatile pointers so that the compiler does not keep the value in a register.
  enum { SP_REG = 0, SP_SMEM = 1, SP_WS = 2, SP_RELOAD = 3 };
  // where each value lives in the segment being generated (a value carried into
  // a later segment is placed afresh there)
  std::vector<uint8_t> sp_kind(n, SP_REG);
  std::vector<int64_t> sp_idx(n, -1);
  const bool spill = o.spill_values > 0 && !o.device_fn && std::max(1, o.inst_per_thread) == 1;
  const int64_t sp_cap_sm = (int64_t)o.spill_shared_kb * 1024 / ((int64_t)o.block * (G.ws_f64() ? 8 : 4));
  const int64_t sp_ws_base = R.ws_rows;   // spill rows follow the carried rows
  // fills sp_kind / sp_idx for segment s; returns (shared slots, workspace rows) used
  auto spill_segment = [&](int s) -> std::pair<int64_t, int64_t> {
    std::fill(sp_kind.begin(), sp_kind.end(), (uint8_t)SP_REG);
    std::fill(sp_idx.begin(), sp_idx.end(), (int64_t)-1);
    // positions: materialised operands of op i at 2i, its result at 2i + 1
    std::vector<int64_t> def(n, -1), end(n, -1), order;
    for (int64_t i = segs[s].first; i < segs[s].second; ++i) {
      if (G.leaf(i)) continue;
      const Node& x = g.nodes[i];
      for (int32_t a : {x.a, x.b}) {
        if (a < 0 || g.nodes[a].op == CONST) continue;
        const bool outside = g.nodes[a].op == INPUT || G.seg_of[a] != s;
        if (outside && def[a] < 0) { def[a] = 2 * i; order.push_back(a); }
        end[a] = std::max(end[a], 2 * i + 1);
      }
      def[i] = 2 * i + 1;
      end[i] = std::max(end[i], def[i]);
      order.push_back(i);
    }
    std::set<std::pair<int64_t, int64_t>> active;   // (end, value) in registers
    std::vector<int64_t> spilled;
    for (int64_t v : order) {
      while (!active.empty() && active.begin()->first <= def[v]) active.erase(active.begin());
      if ((int64_t)active.size() < o.spill_values) { active.insert({end[v], v}); continue; }
      auto last = std::prev(active.end());
      if (last->first > end[v]) {
        spilled.push_back(last->second);
        active.erase(last);
        active.insert({end[v], v});
      } else {
        spilled.push_back(v);
      }
    }
    // memory slots of the spilled computed values: shared first, then workspace rows
    std::sort(spilled.begin(), spilled.end(), [&](int64_t a, int64_t c) { return def[a] < def[c]; });
    std::set<std::pair<int64_t, int64_t>> live_sm, live_ws;   // (end, slot)
    std::vector<int64_t> free_sm, free_ws;
    int64_t next_sm = 0, next_ws = 0;
    for (int64_t v : spilled) {
      if (def[v] % 2 == 0) { sp_kind[v] = SP_RELOAD; continue; }   // input / carried value
      while (!live_sm.empty() && live_sm.begin()->first <= def[v]) { free_sm.push_back(live_sm.begin()->second); live_sm.erase(live_sm.begin()); }
      while (!live_ws.empty() && live_ws.begin()->first <= def[v]) { free_ws.push_back(live_ws.begin()->second); live_ws.erase(live_ws.begin()); }
      int64_t k;
      if (!free_sm.empty() || next_sm < sp_cap_sm) {
        if (!free_sm.empty()) { k = free_sm.back(); free_sm.pop_back(); } else k = next_sm++;
        sp_kind[v] = SP_SMEM; sp_idx[v] = k; live_sm.insert({end[v], k});
      } else {
        if (!free_ws.empty()) { k = free_ws.back(); free_ws.pop_back(); } else k = next_ws++;
        sp_kind[v] = SP_WS; sp_idx[v] = sp_ws_base + k; live_ws.insert({end[v], k});
      }
    }
    return {next_sm, next_ws};
  };
  if (spill) {   // sizes: the most any segment needs (the segments run one after the other)
    int64_t sm = 0, ws = 0;
    for (int s = 0; s < nseg; ++s) {
      auto u = spill_segment(s);
      sm = std::max(sm, u.first);
      ws = std::max(ws, u.second);
    }
    R.ws_rows += ws;
    R.smem_bytes = sm * o.block * (G.ws_f64() ? 8 : 4);
  }
  // Lanes: a kernel thread evaluates NL consecutive instances i .. i + NL - 1,
  // op by op in turn; their inputs and outputs move as one vector access when
  // the buffers allow it.  A kernel thread past the end of the batch still runs
  // (CTA barriers need it) on the last thread's instances, storing nothing.
  const int NL = o.device_fn ? 1 : std::max(1, o.inst_per_thread);
  int cap = o.maxrregcount;
  if (cap == 0 && !o.device_fn && !spill) {
    int64_t words = o.dtype == CUSADI_F64 ? 2 : 1;   // MIXED: most values are single
    cap = auto_register_cap(max_live(g) * words * NL);
  }
  cap = std::max(cap, 0);   // -1: none, and no rule either
  R.register_cap = cap;
  const bool clamped = o.adjoint || NL > 1 || (o.sync_every > 0 && !o.device_fn);
  R.inst_per_thread = NL;
  auto vname = [&](int64_t i, int r) {
    return NL == 1 ? "v" + std::to_string(i) : "v" + std::to_string(i) + "_" + std::to_string(r);
  };
  // a comma-separated list of the NL lane names of node i
  auto lanes = [&](int64_t i) {
    std::string l;
    for (int r = 0; r < NL; ++r) l += (r ? ", " : "") + vname(i, r);
    return l;
  };

  // Paired calls: an out-of-line unary math call (sin, cos, exp, ...) is issued
  // together with a later call of the same function whose argument is already
  // computed, as one call of a two-argument version: half the call overhead, and
  // the two evaluations inside it are independent work the compiler can overlap.
  const bool pairing = o.pair_calls > 0 && NL == 1 && !spill && o.inline_math != 1;
  auto pairable = [&](int64_t i) {
    const Node& x = g.nodes[i];
    if (G.leaf(i) || !op_call(x.op) || op_arity(x.op) != 1 || inlined(x.op, o.inline_math)) return false;
    return !( !G.node_f64((int32_t)i) && o.own_math && own_f32_math(x.op));
  };
  std::vector<int64_t> partner(n, -1);
  std::vector<uint8_t> hoisted(n, 0);
  // sin and cos of one argument: one call for both (the later one moves up to
  // the earlier).  Divisors of at least three FP64 divisions of a segment: one
  // reciprocal, then short divisions (math64.cuh).
  const bool own64 = o.inline_math != 1;
  std::vector<int64_t> trig(n, -1);            // per argument: its first sin or cos in the segment
  std::vector<int32_t> n_div(n, 0);            // per divisor: divisions of the segment
  std::vector<uint8_t> have_recip(n, 0);
  auto divisor = [&](int64_t i) -> int32_t {
    const Node& x = g.nodes[i];
    if ((x.op != DIV && x.op != INV) || !G.node_f64((int32_t)i)) return -1;
    const int32_t b = x.op == INV ? x.a : x.b;
    return g.nodes[b].op == CONST || (spill && sp_kind[b] != SP_REG) ? -1 : b;
  };
  // a division by a reciprocal: its divisor's node (constants by node, too), else -1
  const int64_t kDivPairWindow = 64;
  // FP32 sin and cos of one argument share a call when they are at most this far apart:
  // a value kept longer costs a register (20,000 random ops, N = 16,384: 320 us
  // whatever the distance, 316 at 64); pair_calls pairs calls in its own way (349 us
  // at N = 65,536 and 128 registers, 378 with both).
  const int64_t kSincosWindow = 64;
  std::vector<int64_t> waits(n, -1);           // division evaluated with a later one
  std::vector<int64_t> first_use(n, INT64_MAX);
  for (int64_t i = n - 1; i >= 0; --i)
    for (int32_t a : operands(g, i))
      if (a >= 0 && !G.leaf(i)) first_use[a] = i;
  auto short_div = [&](int64_t i) -> int32_t {
    const Node& x = g.nodes[i];
    if (G.leaf(i) || (x.op != DIV && x.op != INV) || !G.node_f64((int32_t)i)) return -1;
    const int32_t b = x.op == INV ? x.a : x.b;
    if (const_divisor(g.nodes[b])) return b;
    return divisor(i) >= 0 && n_div[b] >= 3 ? b : -1;
  };
  // is node a's value there where node i is evaluated (a division that waits for a
  // later one is not, whatever its index)
  auto ready_at = [&](int32_t a, int64_t i, int s) {
    return a < 0 || G.leaf(a) || G.seg_of[a] != s || (a < i && waits[a] < i);
  };
  for (int s = 0; s < nseg; ++s) {
    if (spill) spill_segment(s);
    std::fill(trig.begin(), trig.end(), (int64_t)-1);
    std::fill(n_div.begin(), n_div.end(), 0);
    std::fill(have_recip.begin(), have_recip.end(), (uint8_t)0);
    for (int64_t i = segs[s].first; own64 && i < segs[s].second; ++i) {
      const Node& x = g.nodes[i];
      const bool f64 = G.node_f64((int32_t)i);
      if ((x.op == SIN || x.op == COS) && (f64 || (o.own_math == 0 && o.pair_calls == 0)) && g.nodes[x.a].op != CONST) {
        const int64_t f = trig[x.a];
        if (f < 0 || (!f64 && i - f > kSincosWindow)) trig[x.a] = i;
        else if (g.nodes[f].op != x.op && G.node_f64((int32_t)f) == f64 && partner[f] < 0) { partner[f] = i; hoisted[i] = 1; }
      }
      const int32_t b = divisor(i);
      if (b >= 0) ++n_div[b];
    }
    // two quotients by one divisor in one call: the later one moves up where its
    // numerator is ready, else the earlier one waits where nothing needs it yet
    for (int64_t i = segs[s].first; own64 && NL == 1 && !spill && i < segs[s].second; ++i) {
      const int32_t b = short_div(i);
      if (b < 0 || partner[i] >= 0 || hoisted[i] || waits[i] >= 0) continue;
      const int64_t lim = std::min<int64_t>(segs[s].second, i + 1 + kDivPairWindow);
      for (int64_t j = i + 1; j < lim; ++j) {
        if (short_div(j) != b || partner[j] >= 0 || hoisted[j]) continue;   // in a pair already
        const int32_t a = g.nodes[j].op == INV ? -1 : g.nodes[j].a;
        const bool ready = ready_at(a, i, s);
        if (ready) { partner[i] = j; hoisted[j] = 1; }
        else if (first_use[i] > j) { partner[j] = i; waits[i] = j; }
        if (ready || first_use[i] > j) break;
      }
    }
    if (pairing) {
      for (int64_t i = segs[s].first; i < segs[s].second; ++i) {
        if (!pairable(i) || hoisted[i] || partner[i] >= 0) continue;
        const int64_t lim = std::min<int64_t>(segs[s].second, i + 1 + o.pair_calls);
        for (int64_t j = i + 1; j < lim; ++j) {
          if (!pairable(j) || hoisted[j] || partner[j] >= 0 || g.nodes[j].op != g.nodes[i].op ||
              G.node_f64((int32_t)j) != G.node_f64((int32_t)i))
            continue;
          if (!ready_at(g.nodes[j].a, i, s)) continue;
          partner[i] = j;
          hoisted[j] = 1;
          break;
        }
      }
    }
    std::ostringstream body;
    std::vector<uint8_t> have(n, 0);   // leaf or ws value materialised in this segment
    std::vector<uint8_t> decl_buf(n, 0);  // lanes declared with the buffer's type, not the op's
    G.calls.clear();
    G.calls2.clear();
    G.own_f32 = false;
    G.own_f64 = false;
    G.wrappers.clear();
    auto operand = [&](int32_t i, bool want_f64, int r) -> std::string {
      const Node& x = g.nodes[i];
      bool f = G.node_f64(i);
      if (x.op == CONST) return lit(x.k, want_f64);
      if (spill && sp_kind[i] != SP_REG) {
        // read at each use from where the value lives
        const char* W2 = G.ty(want_f64);
        if (sp_kind[i] == SP_SMEM)
          return std::string("((") + W2 + ")cs_sp[" + std::to_string(sp_idx[i]) + " * blockDim.x])";
        if (sp_kind[i] == SP_WS)
          return std::string("((") + W2 + ")Wv[" + std::to_string(sp_idx[i]) + "ll * ldw])";
        if (x.op == INPUT) {
          const bool second = o.split >= 0 && x.io >= o.split;
          const int64_t row = second ? x.io - o.split : x.io;
          const std::string base = second ? (x.bcast ? "X2b" : "X2") : (x.bcast ? "Xb" : "X");
          return std::string("((") + W2 + ")((const volatile " + tin + "*)" + base + ")[" + std::to_string(row) +
                 (second ? "ll * ldx2])" : "ll * ldx])");
        }
        return std::string("((") + W2 + ")Wv[" + std::to_string(G.ws_slot[i]) + "ll * ldw])";
      }
      if (x.op == INPUT) {
        if (!have[i]) {
          have[i] = 1;
          const bool second = o.split >= 0 && x.io >= o.split;
          const int64_t row = second ? x.io - o.split : x.io;
          const std::string src = std::string(second ? (x.bcast ? "X2b[" : "X2[") : (x.bcast ? "Xb[" : "X[")) +
                                  std::to_string(row) + (second ? "ll * ldx2]" : "ll * ldx]");
          if (NL == 1 || x.bcast) {
            // a broadcast row holds one value for every instance: all lanes share it
            body << "  const " << G.ty(f) << " v" << i << " = (" << G.ty(f) << ")" << src << ";\n";
          } else {
            decl_buf[i] = 1;
            body << "  " << tin << " " << lanes(i) << ";\n"
                 << "  cs_ld" << NL << "(&" << src << ", full, m, " << lanes(i) << ");\n";
          }
        }
        std::string name = (NL == 1 || x.bcast) ? "v" + std::to_string(i) : vname(i, r);
        const bool df = decl_buf[i] ? G.buf_f64() : f;
        if (df != want_f64) return std::string("(") + G.ty(want_f64) + ")" + name;
        return name;
      }
      if (G.seg_of[i] != s) {
        if (!have[i]) {
          have[i] = 1;
          if (NL == 1) {
            body << "  const " << G.ty(f) << " v" << i << " = (" << G.ty(f) << ")W["
                 << G.ws_slot[i] << "ll * ldw];\n";
          } else {
            decl_buf[i] = 1;   // workspace columns are padded to 32: always whole vectors
            body << "  " << tw << " " << lanes(i) << ";\n"
                 << "  cs_ld" << NL << "(&W[" << G.ws_slot[i] << "ll * ldw], true, " << NL << ", "
                 << lanes(i) << ");\n";
          }
        }
      }
      const bool df = decl_buf[i] ? G.ws_f64() : f;
      if (df != want_f64) return std::string("(") + G.ty(want_f64) + ")" + vname(i, r);
      return vname(i, r);
    };
    // stores of output row r of node i (values v[lane])
    auto store_out = [&](int64_t r, const std::vector<std::string>& v) {
      if (o.adjoint) {
        for (int l = 0; l < NL; ++l) {
          const std::string guard = NL == 1 ? "active" : "active && m > " + std::to_string(l);
          const std::string off = NL == 1 ? "" : " + " + std::to_string(l);
          const std::string plain = "if (" + guard + ") { " + tin + "* p_ = &Y[" + std::to_string(r) +
                                    "ll * ldy" + off + "]; *p_ = acc ? *p_ + (" + tin + ")" + v[l] + " : (" +
                                    tin + ")" + v[l] + "; }";
          if (g.out_reduce[r]) {
            // the instance's term goes to the workspace (a coalesced store); the
            // finishing kernel sums each such row over the instances
            body << "  if (reduce) {\n    if (" << guard << ") Wp[" << reduce_k[r] << "ll * ldw" << off
                 << "] = (" << tw << ")" << v[l] << ";\n  } else " << plain << "\n";
          } else {
            body << "  " << plain << "\n";
          }
        }
      } else if (NL == 1) {
        body << "  " << (clamped ? "if (active) " : "") << "Y[" << r << "ll * ldy] = (" << tin << ")" << v[0] << ";\n";
      } else {
        body << "  if (active) cs_st" << NL << "(&Y[" << r << "ll * ldy], full, m";
        for (int l = 0; l < NL; ++l) body << ", (" << tin << ")" << v[l];
        body << ");\n";
      }
      if (o.debug_checks && !o.device_fn)   // count non-finite results (cusadi_debug_count)
        for (int l = 0; l < NL; ++l)
          body << "  if (active" << (NL == 1 ? "" : " && m > " + std::to_string(l)) << " && !isfinite((double)("
               << v[l] << "))) atomicAdd(&cs_dbg, 1u);\n";
    };
    auto lane_values = [&](int64_t i, bool f) {
      std::vector<std::string> v;
      for (int l = 0; l < NL; ++l) v.push_back(G.leaf(i) ? operand((int32_t)i, f, l) : vname(i, l));
      return v;
    };
    // outputs fed directly by inputs or constants are written by segment 0
    if (s == 0) {
      for (int64_t i = 0; i < n; ++i) {
        if (!G.leaf(i) || G.out_rows[i].empty()) continue;
        std::vector<std::string> v = lane_values(i, G.node_f64((int32_t)i));
        for (int64_t r : G.out_rows[i]) store_out(r, v);
      }
    }
    // where node i's value goes beside its register: spill slot, workspace row, outputs
    auto keep = [&](int64_t i) {
      const bool f = G.node_f64((int32_t)i);
      if (spill && sp_kind[i] == SP_SMEM)
        body << "  cs_sp[" << sp_idx[i] << " * blockDim.x] = (" << tw << ")v" << i << ";\n";
      else if (spill && sp_kind[i] == SP_WS)
        body << "  Wv[" << sp_idx[i] << "ll * ldw] = (" << tw << ")v" << i << ";\n";
      if (G.ws_slot[i] >= 0) {
        if (NL == 1) {
          body << "  if (active) W[" << G.ws_slot[i] << "ll * ldw] = (" << tw << ")v" << i << ";\n";
        } else {
          body << "  if (active) cs_st" << NL << "(&W[" << G.ws_slot[i] << "ll * ldw], true, " << NL;
          for (int l = 0; l < NL; ++l) body << ", (" << tw << ")" << vname(i, l);
          body << ");\n";
        }
      }
      if (!G.out_rows[i].empty()) {
        std::vector<std::string> v = lane_values(i, f);
        for (int64_t r : G.out_rows[i]) store_out(r, v);
      }
    };
    int64_t since_sync = 0;
    for (int64_t i = segs[s].first; i < segs[s].second; ++i) {
      if (G.leaf(i)) continue;
      const Node& x = g.nodes[i];
      const bool f = G.node_f64((int32_t)i);
      const char* T = G.ty(f);
      const std::array<int32_t, 3> reads = operands(g, i);
      if (waits[i] >= 0) continue;   // evaluated with a later division
      const bool two_div = partner[i] >= 0 && short_div(i) >= 0;
      const bool sincos = partner[i] >= 0 && !two_div && g.nodes[partner[i]].op != x.op;
      const int32_t dv = own64 ? divisor(i) : -1;
      if (two_div) {
        const int64_t j = partner[i];
        const int32_t b = short_div(i);
        auto numerator = [&](int64_t k) { return g.nodes[k].op == INV ? std::string("1.0") : operand(g.nodes[k].a, true, 0); };
        const std::string A = numerator(i), Aj = numerator(j), B = operand(b, true, 0);
        G.own_f64 = true;
        G.wrappers.insert(kDivr2);
        std::string r = "r" + std::to_string(b);
        if (g.nodes[b].op == CONST) {
          char h[32];
          std::snprintf(h, sizeof h, "0x%016" PRIx64 "ull", recip_of(g.nodes[b].k));
          r = h;
        } else if (!have_recip[b]) {
          G.wrappers.insert(kRecip);
          body << "  const cs_u64 " << r << " = cs_recip_d(" << B << ");\n";
          have_recip[b] = 1;
        }
        body << "  const double2 p" << i << " = cs_divr2_d(" << A << ", " << Aj << ", " << B << ", " << r << ");\n"
             << "  const double v" << i << " = p" << i << ".x, v" << j << " = p" << i << ".y;\n";
      } else if (sincos) {
        const int64_t j = partner[i];
        if (f) G.own_f64 = true;
        G.wrappers.insert(f ? kSincos : kSincosF);
        for (int l = 0; l < NL; ++l) {
          const std::string A = operand(x.a, f, l);
          body << "  const " << T << "2 p" << vname(i, l) << " = cs_sincos_" << (f ? "d(" : "f(") << A << ");\n"
               << "  const " << T << " " << vname(i, l) << " = p" << vname(i, l) << (x.op == SIN ? ".x" : ".y") << ", "
               << vname(j, l) << " = p" << vname(i, l) << (x.op == SIN ? ".y" : ".x") << ";\n";
        }
      } else if (pairing && partner[i] >= 0) {
        const int64_t j = partner[i];
        std::string A = operand(x.a, f, 0), Aj = operand(g.nodes[j].a, f, 0);
        G.calls2.insert({x.op, f});
        MathFn m = math_name(x.op);
        body << "  const " << T << "2 p" << i << " = cs_" << m.d << "2" << (f ? "_d" : "_f") << "(" << A
             << ", " << Aj << ");\n"
             << "  const " << T << " v" << i << " = p" << i << ".x;\n"
             << "  const " << T << " v" << j << " = p" << i << ".y;\n";
      } else if (hoisted[i]) {       // computed with its partner
      } else if (dv >= 0 && n_div[dv] >= 3) {
        G.own_f64 = true;
        G.wrappers.insert(kRecip);
        G.wrappers.insert(kDivr);
        const bool shared = NL == 1 || (g.nodes[dv].op == INPUT && g.nodes[dv].bcast);
        for (int l = 0; l < NL; ++l) {
          const std::string A = x.op == INV ? "1.0" : operand(x.a, true, l), B = operand(dv, true, l);
          const std::string r = "r" + std::to_string(dv) + (shared ? "" : "_" + std::to_string(l));
          if (!have_recip[dv] && (l == 0 || !shared)) body << "  const cs_u64 " << r << " = cs_recip_d(" << B << ");\n";
          body << "  const double " << vname(i, l) << " = cs_divr_d(" << A << ", " << B << ", " << r << ");\n";
        }
        have_recip[dv] = 1;
      } else {
        for (int l = 0; l < NL; ++l) {
          std::string e[3];
          for (int k = 0; k < 3; ++k)
            if (reads[k] >= 0) e[k] = operand(reads[k], f, l);
          body << "  const " << T << " " << vname(i, l) << " = " << op_expr(G, i, f, e[0], e[1], e[2], o) << ";\n";
        }
      }
      keep(i);
      if (two_div && waits[partner[i]] == i) keep(partner[i]);
      if (o.sync_every > 0 && !o.device_fn && ++since_sync >= o.sync_every) {
        body << "  __syncthreads();\n";
        since_sync = 0;
      }
    }

    std::ostringstream src;
    src << "// Generated straight-line kernel: segment " << s << " of " << nseg
        << (o.adjoint ? " (adjoint)" : "") << ", dtype "
        << (o.dtype == CUSADI_F64 ? "f64" : (o.dtype == CUSADI_F32 ? "f32" : "mixed"));
    if (NL > 1) src << ", " << NL << " instances per thread";
    if (o.sync_every > 0 && !o.device_fn) src << ", CTA barrier every " << o.sync_every << " ops";
    src << "\n";
    if (NL > 1) src << kLaneAccess;
    if (G.own_f32) src << own_math_source(o.own_math);
    if (G.own_f64) src << kMath64Text;
    for (const std::string& w : G.wrappers) src << w;
    if (o.debug_checks && !o.device_fn) src << "__device__ unsigned int cs_dbg;   // non-finite results\n";
    {
      for (auto& c : G.calls) {
        const char* t = c.second ? "double" : "float";
        bool bin = op_arity(c.first) == 2;
        src << "static __device__ __noinline__ " << t << " " << call_name(c.first, c.second, false) << "("
            << t << " a" << (bin ? std::string(", ") + t + " b" : "") << ") { return "
            << math_fn(c.first, c.second) << "(a" << (bin ? ", b" : "") << "); }\n";
      }
      for (auto& c : G.calls2) {   // two independent evaluations per call
        MathFn m = math_name(c.first);
        const char* t = c.second ? "double" : "float";
        const std::string fn = math_fn(c.first, c.second);
        src << "static __device__ __noinline__ " << t << "2 cs_" << m.d << "2" << (c.second ? "_d" : "_f")
            << "(" << t << " a, " << t << " b) { " << t << "2 r; r.x = " << fn << "(a); r.y = " << fn
            << "(b); return r; }\n";
      }
    }
    std::string name = o.prefix + "_" + std::to_string(s);
    if (o.device_fn) {
      // one instance per call; the caller owns the index and the bounds check
      src << "extern \"C\" __device__ void " << name << "(\n"
          << "    const " << tin << "* __restrict__ X, long long ldx, const " << tin
          << "* __restrict__ X2, long long ldx2, " << tin
          << "* __restrict__ Y, long long ldy,\n    " << tw
          << "* __restrict__ W, long long ldw, long long i) {\n"
          << "  const bool active = true;\n  const int acc = 0, reduce = 0;\n"
          << "  const " << tin << "* __restrict__ Xb = X;\n"
          << "  const " << tin << "* __restrict__ X2b = X2;\n"
          << "  " << tin << "* __restrict__ Yb = Y;\n"
          << "  X += i; X2 += i; Y += i; W += i;\n"
          << "  (void)Xb; (void)X2b; (void)Yb; (void)W; (void)ldw; (void)ldx2; (void)acc; (void)reduce; (void)active;\n"
          << body.str() << "}\n";
      Segment S;
      S.begin = segs[s].first;
      S.end = segs[s].second;
      S.name = name;
      S.source = src.str();
      R.segs.push_back(std::move(S));
      continue;
    }
    src << "extern \"C\" __global__ void " << launch_bounds(o.block, cap) << " " << name << "(\n"
        << "    const " << tin << "* __restrict__ X, long long ldx, const " << tin
        << "* __restrict__ X2, long long ldx2, " << tin
        << "* __restrict__ Y, long long ldy,\n    long long N, " << tw
        << "* __restrict__ W, long long ldw, int acc, int reduce, int vec) {\n";
    if (NL == 1) {
      src << "  const long long i0 = (long long)blockIdx.x * blockDim.x + threadIdx.x;\n";
      if (clamped) {
        src << "  const bool active = i0 < N;\n"
            << "  const long long i = active ? i0 : N - 1;\n";
      } else {
        src << "  if (i0 >= N) return;\n  const bool active = true;\n  const long long i = i0;\n";
      }
    } else {
      // m: instances of this thread inside the batch; full: whole vector accesses
      src << "  const long long i0 = ((long long)blockIdx.x * blockDim.x + threadIdx.x) * " << NL << ";\n"
          << "  const bool active = i0 < N;\n"
          << "  const long long i = active ? i0 : (N - 1) / " << NL << " * " << NL << ";\n"
          << "  const int m = N - i < " << NL << " ? (int)(N - i) : " << NL << ";\n"
          << "  const bool full = vec != 0 && m == " << NL << ";\n";
    }
    src << "  const " << tin << "* __restrict__ Xb = X;\n"
        << "  const " << tin << "* __restrict__ X2b = X2;\n"
        << "  " << tin << "* __restrict__ Yb = Y;\n";
    if (spill)   // values kept out of registers: shared slots and workspace rows, never cached
      src << "  extern __shared__ __align__(16) unsigned char cs_smem[];\n"
          << "  volatile " << tw << "* const cs_sp = reinterpret_cast<volatile " << tw
          << "*>(cs_smem) + threadIdx.x;\n"
          << "  volatile " << tw << "* const Wv = W + i;\n"
          << "  (void)cs_sp; (void)Wv;\n";
    if (o.adjoint && R.has_reduce)
      src << "  " << tw << "* __restrict__ Wp = W + " << R.ws_rows << "ll * ldw + i;  // reduced-row terms\n";
    src << "  X += i; X2 += i; Y += i; W += i;\n"
        << "  (void)Xb; (void)X2b; (void)Yb; (void)W; (void)ldw; (void)ldx2; (void)acc; (void)reduce; (void)active; (void)vec;\n"
        << body.str() << "}\n";
    Segment S;
    S.begin = segs[s].first;
    S.end = segs[s].second;
    S.name = name;
    S.source = src.str();
    R.segs.push_back(std::move(S));
  }
  if (R.has_reduce) R.segs[0].source += finish_source(R, o.prefix, tin, tw);
  return R;
}

// One CTA per reduced row adds the row's N per-instance terms in a fixed order
// (strided per thread, then a tree), so the sum is the same on every run; it
// then writes, or adds to, the row's column 0.
std::string finish_source(CodegenResult& R, const std::string& prefix, const char* tin,
                          const char* tw) {
  {
    std::ostringstream z;
    R.finish_kernel = prefix + "_finish";
    z << "static __device__ const long long cs_reduce_row[] = {";
    for (size_t k = 0; k < R.reduce_rows.size(); ++k) z << (k ? ", " : "") << R.reduce_rows[k];
    z << "};\n"
      << "extern \"C\" __global__ void __launch_bounds__(512) " << R.finish_kernel << "(const " << tw
      << "* __restrict__ W, long long ldw, long long N, " << tin << "* __restrict__ Y, long long ldy, "
      << "int accumulate) {\n"
      << "  __shared__ " << tw << " s_[512];\n"
      << "  const " << tw << "* __restrict__ P = W + (" << R.ws_rows << "ll + blockIdx.x) * ldw;\n"
      << "  " << tw << " a = 0;\n"
      << "  for (long long j = threadIdx.x; j < N; j += 512) a += P[j];\n"
      << "  s_[threadIdx.x] = a;\n"
      << "  __syncthreads();\n"
      << "  for (int d = 256; d > 0; d >>= 1) {\n"
      << "    if ((int)threadIdx.x < d) s_[threadIdx.x] += s_[threadIdx.x + d];\n"
      << "    __syncthreads();\n"
      << "  }\n"
      << "  if (threadIdx.x == 0) {\n"
      << "    " << tin << "* p = &Y[cs_reduce_row[blockIdx.x] * ldy];\n"
      << "    *p = (" << tin << ")(accumulate ? (" << tw << ")*p + s_[0] : s_[0]);\n"
      << "  }\n}\n";
    return z.str();
  }
}

}  // namespace cusadi

namespace cusadi {

// Cooperative kernels: the CTA's warps split one program; lane l of every warp
// works on instance 32 * blockIdx.x + l.  The code is laid out phase by phase:
// one `if (warp == w)` block per warp with work in that phase, then a
// __syncthreads() at function scope, so every thread executes the same barrier
// instructions.  (Per-warp regions with a non-aligned barrier.sync gave wrong
// results at 6-8 warps with ~160 KB of shared slots on GB300, so that layout
// is not used.)  Values read by another warp are staged in shared memory
// (overflow: workspace rows); values a warp needs in a later phase are
// declared at function scope.
CodegenResult generate_coop(const Graph& g, const CodegenOptions& o, const CoopPlan& plan) {
  CodegenResult R;
  Gen G(g, o);
  const int64_t n = (int64_t)g.nodes.size();
  const int W = plan.ways;
  const int NG = o.device_fn ? 1 : std::max(1, o.coop_groups);   // groups of 32 instances per CTA
  G.out_rows.assign(n, {});
  for (size_t r = 0; r < g.out.size(); ++r) G.out_rows[g.out[r]].push_back((int64_t)r);
  // segments: runs of whole phases of at most ~segment_ops ops
  std::vector<int64_t> ops_in_phase(plan.n_phases, 0);
  for (int64_t i = 0; i < n; ++i)
    if (!G.leaf(i)) ops_in_phase[plan.phase[i]]++;
  std::vector<std::pair<int, int>> segs;  // [first phase, last phase + 1)
  {
    int start = 0;
    int64_t acc = 0;
    for (int q = 0; q < plan.n_phases; ++q) {
      if (o.segment_ops > 0 && acc > 0 && acc + ops_in_phase[q] > o.segment_ops) {
        segs.push_back({start, q});
        start = q;
        acc = 0;
      }
      acc += ops_in_phase[q];
    }
    segs.push_back({start, plan.n_phases});
  }
  const int nseg = (int)segs.size();
  std::vector<int> seg_of_phase(plan.n_phases, 0);
  for (int s = 0; s < nseg; ++s)
    for (int q = segs[s].first; q < segs[s].second; ++q) seg_of_phase[q] = s;
  G.seg_of.assign(n, -1);
  G.last_seg.assign(n, -1);
  for (int64_t i = 0; i < n; ++i)
    if (!G.leaf(i)) G.seg_of[i] = seg_of_phase[plan.phase[i]];
  for (int64_t i = 0; i < n; ++i) {
    if (G.leaf(i)) continue;
    for (int32_t a : operands(g, i))
      if (a >= 0 && !G.leaf(a)) G.last_seg[a] = std::max(G.last_seg[a], G.seg_of[i]);
  }
  std::vector<int> slot, gslot;
  int n_gslots = 0;
  const bool sm64 = o.dtype != CUSADI_F32;
  // shared-memory budget for cross-warp values (CUSADI_COOP_SHARED_KB overrides
  // it, so tests can force the workspace overflow path on small programs)
  int budget_kb = o.coop_shared_kb;
  if (const char* e = std::getenv("CUSADI_COOP_SHARED_KB")) budget_kb = std::max(0, std::atoi(e));
  const int max_slots = (int)((budget_kb * 1024) / (32 * (sm64 ? 8 : 4)));
  const int n_slots = assign_coop_slots(g, plan, G.seg_of, max_slots, slot, gslot, n_gslots);
  // workspace rows for values crossing kernels (same interval reuse as generate)
  G.ws_slot.assign(n, -1);
  {
    std::vector<std::vector<int64_t>> release(nseg + 1);
    std::vector<int64_t> free_rows;
    int64_t rows = 0;
    std::vector<std::vector<int64_t>> defs(nseg);
    for (int64_t i = 0; i < n; ++i)
      if (!G.leaf(i)) defs[G.seg_of[i]].push_back(i);
    for (int s = 0; s < nseg; ++s) {
      if (s > 0) {
        for (int64_t r : release[s - 1]) free_rows.push_back(r);
        release[s - 1].clear();
      }
      for (int64_t i : defs[s]) {
        if (G.last_seg[i] <= s) continue;
        int64_t r;
        if (!free_rows.empty()) { r = free_rows.back(); free_rows.pop_back(); }
        else r = rows++;
        G.ws_slot[i] = r;
        release[G.last_seg[i]].push_back(r);
      }
    }
    R.ws_rows = rows;
  }
  // cross-warp values that did not fit in shared memory use rows after those
  const int64_t g_base = R.ws_rows;
  R.ws_rows += n_gslots;
  const char* tin = G.buf_f64() ? "double" : "float";
  const char* tw = G.ws_f64() ? "double" : "float";
  const bool sm_f64 = sm64;  // shared slots hold the widest type in use
  const char* tsm = sm_f64 ? "double" : "float";
  // adjoint outputs: accumulate or overwrite; a reduced (broadcast) row's term
  // goes to its workspace row, summed over the instances by the finishing kernel
  for (uint8_t f : g.out_reduce) R.has_reduce |= (f != 0);
  std::vector<int64_t> reduce_k(g.out_reduce.size(), -1);
  for (size_t r = 0; r < g.out_reduce.size(); ++r)
    if (g.out_reduce[r]) {
      reduce_k[r] = (int64_t)R.reduce_rows.size();
      R.reduce_rows.push_back((int64_t)r);
    }
  auto store_out = [&](std::ostringstream& body, int64_t r, const std::string& v) {
    if (o.debug_checks && !o.device_fn)   // count non-finite results (cusadi_debug_count)
      body << "    if (active && !isfinite((double)(" << v << "))) atomicAdd(&cs_dbg, 1u);\n";
    if (!o.adjoint) {
      body << "    if (active) Y[" << r << "ll * ldy] = (" << tin << ")" << v << ";\n";
      return;
    }
    const std::string plain = std::string("if (active) { ") + tin + "* p_ = &Y[" + std::to_string(r) +
                              "ll * ldy]; *p_ = acc ? *p_ + (" + tin + ")" + v + " : (" + tin + ")" + v + "; }";
    if (!g.out_reduce[r]) {
      body << "    " << plain << "\n";
      return;
    }
    body << "    if (reduce) { if (active) Wp[" << reduce_k[r] << "ll * ldw] = (" << tw << ")" << v
         << "; } else " << plain << "\n";
  };
  // nodes per (segment, warp, phase) in topological order
  for (int s = 0; s < nseg; ++s) {
    std::vector<std::vector<std::vector<int64_t>>> work(W, std::vector<std::vector<int64_t>>(segs[s].second - segs[s].first));
    for (int64_t i = 0; i < n; ++i)
      if (!G.leaf(i) && G.seg_of[i] == s) work[plan.owner[i]][plan.phase[i] - segs[s].first].push_back(i);
    std::ostringstream regions;
    G.calls.clear();
    G.own_f32 = false;
    G.own_f64 = false;
    G.wrappers.clear();
    const int nph_seg = segs[s].second - segs[s].first;
    // phase-major layout: every warp reaches the same __syncthreads() (aligned
    // barrier); a value used by its own warp in a later phase is declared once
    // at function scope, everything else is local to its phase block
    std::vector<int> last_own_phase(n, -1);
    for (int64_t i = 0; i < n; ++i) {
      if (G.leaf(i) || G.seg_of[i] != s) continue;
      for (int32_t a : operands(g, i))
        if (a >= 0 && !G.leaf(a) && G.seg_of[a] == s && plan.owner[a] == plan.owner[i])
          last_own_phase[a] = std::max(last_own_phase[a], plan.phase[i]);
    }
    std::ostringstream decls;
    std::vector<std::ostringstream> phase_code(nph_seg);
    std::vector<std::vector<std::string>> phase_warp(nph_seg, std::vector<std::string>(W));
    for (int w = 0; w < W; ++w) {
      std::ostringstream body;
      std::vector<uint8_t> have(n, 0);
      auto operand = [&](int32_t i, bool want_f64) -> std::string {
        const Node& x = g.nodes[i];
        bool f = G.node_f64(i);
        if (x.op == CONST) return lit(x.k, want_f64);
        // a value this warp loads (input, another warp's value, an earlier
        // kernel's value) gets its own name; in the phase-major layout it is
        // declared at function scope because later phases may use it again
        const bool loaded = x.op == INPUT || G.seg_of[i] != s || plan.owner[i] != w;
        std::string name = "v" + std::to_string(i) + (loaded ? "_" + std::to_string(w) : "");
        if (!have[i]) {
          std::string lhs;
          if (loaded) {
            decls << "  " << G.ty(f) << " " << name << ";\n";
            lhs = "    " + name;
          } else {
            lhs = std::string("    const ") + G.ty(f) + " " + name;
          }
          if (x.op == INPUT) {
            const bool second = o.split >= 0 && x.io >= o.split;   // adjoint: y_bar rows
            const int64_t row = second ? x.io - o.split : x.io;
            body << lhs << " = (" << G.ty(f) << ")"
                 << (second ? (x.bcast ? "X2b[" : "X2[") : (x.bcast ? "Xb[" : "X[")) << row
                 << (second ? "ll * ldx2];\n" : "ll * ldx];\n");
          } else if (G.seg_of[i] != s) {
            body << lhs << " = (" << G.ty(f) << ")W[" << G.ws_slot[i] << "ll * ldw];\n";
          } else if (plan.owner[i] != w) {
            if (slot[i] >= 0)
              body << lhs << " = (" << G.ty(f) << ")cs_x[" << slot[i] << " * 32 + lane];\n";
            else
              body << lhs << " = (" << G.ty(f) << ")W[" << g_base + gslot[i] << "ll * ldw];\n";
          }
          have[i] = 1;
        }
        if (f != want_f64) return std::string("(") + G.ty(want_f64) + ")" + name;
        return name;
      };
      const int nph = nph_seg;
      for (int q = 0; q < nph; ++q) {
        for (int64_t i : work[w][q]) {
          const bool f = G.node_f64((int32_t)i);
          const char* T = G.ty(f);
          const std::array<int32_t, 3> reads = operands(g, i);
          std::string e[3];
          for (int k = 0; k < 3; ++k)
            if (reads[k] >= 0) e[k] = operand(reads[k], f);
          const std::string value = op_expr(G, i, f, e[0], e[1], e[2], o);
          const bool persists = plan.phase[i] < last_own_phase[i];
          if (persists) {
            decls << "  " << T << " v" << i << ";\n";
            body << "    v" << i << " = " << value << ";\n";
          } else {
            body << "    const " << T << " v" << i << " = " << value << ";\n";
          }
          have[i] = 1;
          if (slot[i] >= 0) body << "    cs_x[" << slot[i] << " * 32 + lane] = (" << tsm << ")v" << i << ";\n";
          if (gslot[i] >= 0) body << "    if (active) W[" << g_base + gslot[i] << "ll * ldw] = (" << tw << ")v" << i << ";\n";
          if (G.ws_slot[i] >= 0) body << "    if (active) W[" << G.ws_slot[i] << "ll * ldw] = (" << tw << ")v" << i << ";\n";
          for (int64_t r : G.out_rows[i]) store_out(body, r, "v" + std::to_string(i));
        }
        phase_warp[q][w] = body.str();
        body.str("");
        body.clear();
      }
      if (s == 0 && w == 0) {
        // outputs fed directly by inputs or constants
        for (int64_t i = 0; i < n; ++i) {
          if (!G.leaf(i) || G.out_rows[i].empty()) continue;
          std::string v = operand((int32_t)i, G.node_f64((int32_t)i));
          for (int64_t r : G.out_rows[i]) store_out(body, r, v);
        }
      }
      if (!body.str().empty()) phase_warp[nph - 1][w] += body.str();
    }
    {
      regions << decls.str();
      for (int q = 0; q < nph_seg; ++q) {
        bool first = true;
        for (int w = 0; w < W; ++w) {
          if (phase_warp[q][w].empty()) continue;
          regions << (first ? "  if (warp == " : "  else if (warp == ") << w << ") {\n" << phase_warp[q][w] << "  }\n";
          first = false;
        }
        if (q + 1 < nph_seg) regions << "  __syncthreads();\n";
      }
    }
    std::ostringstream src;
    src << "// Generated cooperative kernel: segment " << s << " of " << nseg << ", " << W
        << " warps per 32 instances, " << (segs[s].second - segs[s].first) << " phases\n";
    if (G.own_f32) src << own_math_source(o.own_math);
    if (G.own_f64) src << kMath64Text;
    for (const std::string& w : G.wrappers) src << w;
    if (o.debug_checks && !o.device_fn) src << "__device__ unsigned int cs_dbg;   // non-finite results\n";
    {
      for (auto& c : G.calls) {
        const char* t = c.second ? "double" : "float";
        bool bin = op_arity(c.first) == 2;
        src << "static __device__ __noinline__ " << t << " " << call_name(c.first, c.second, false) << "("
            << t << " a" << (bin ? std::string(", ") + t + " b" : "") << ") { return "
            << math_fn(c.first, c.second) << "(a" << (bin ? ", b" : "") << "); }\n";
      }
    }
    std::string name = o.prefix + "_" + std::to_string(s);
    if (o.device_fn) {
      // one group of 32 instances (first .. first + count - 1) per call, made
      // by every thread of the calling CTA of 32 * W threads (the barriers
      // need all of them); the barrier on entry orders this segment after the
      // previous one's workspace writes and shared-slot reads
      src << "extern \"C\" __device__ void " << name << "(\n"
          << "    const " << tin << "* __restrict__ X, long long ldx, " << tin
          << "* __restrict__ Y, long long ldy, " << tw << "* __restrict__ W, long long ldw,\n"
          << "    long long first, int count, unsigned char* __restrict__ cs_smem) {\n"
          << "  " << tsm << "* __restrict__ cs_x = reinterpret_cast<" << tsm << "*>(cs_smem);\n"
          << "  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;\n"
          << "  const bool active = lane < count;\n"
          << "  const long long i = first + (active ? lane : count - 1);\n"
          << "  const " << tin << "* __restrict__ Xb = X;\n"
          << "  X += i; Y += i; W += i;\n"
          << "  (void)Xb; (void)W; (void)ldw; (void)cs_x;\n"
          << "  __syncthreads();\n"
          << regions.str() << "}\n";
      Segment S;
      S.begin = segs[s].first;
      S.end = segs[s].second;
      S.name = name;
      S.source = src.str();
      R.segs.push_back(std::move(S));
      continue;
    }
    // NG groups of 32 instances per CTA: warp w of every group runs role w % W
    // on group w / W, each group with its own block of shared slots
    src << "extern \"C\" __global__ void " << launch_bounds(32 * W * NG, o.maxrregcount) << " " << name << "(\n"
        << "    const " << tin << "* __restrict__ X, long long ldx, const " << tin
        << "* __restrict__ X2, long long ldx2, " << tin << "* __restrict__ Y, long long ldy,\n    long long N, "
        << tw << "* __restrict__ W, long long ldw, int acc, int reduce, int vec) {\n"
        << "  extern __shared__ __align__(16) unsigned char cs_smem[];\n"
        << "  const int lane = threadIdx.x & 31, warp = (threadIdx.x >> 5) % " << W
        << ", grp = (threadIdx.x >> 5) / " << W << ";\n"
        << "  " << tsm << "* __restrict__ cs_x = reinterpret_cast<" << tsm << "*>(cs_smem) + grp * "
        << std::max(n_slots, 1) * 32 << ";\n"
        << "  const long long i0 = ((long long)blockIdx.x * " << NG << " + grp) * 32 + lane;\n"
        << "  const bool active = i0 < N;\n"
        << "  const long long i = active ? i0 : N - 1;\n"
        << "  const " << tin << "* __restrict__ Xb = X;\n"
        << "  const " << tin << "* __restrict__ X2b = X2;\n";
    if (R.has_reduce) src << "  " << tw << "* __restrict__ Wp = W + " << R.ws_rows << "ll * ldw + i;  // reduced-row terms\n";
    src << "  X += i; X2 += i; Y += i; W += i;\n"
        << "  (void)Xb; (void)X2b; (void)ldx2; (void)W; (void)ldw; (void)acc; (void)reduce; (void)cs_x; (void)vec;\n"
        << regions.str() << "}\n";
    Segment S;
    S.begin = segs[s].first;
    S.end = segs[s].second;
    S.name = name;
    S.source = src.str();
    R.segs.push_back(std::move(S));
  }
  R.coop_ways = W;
  R.coop_groups = NG;
  R.smem_bytes = (int64_t)NG * std::max(n_slots, 1) * 32 * (sm_f64 ? 8 : 4);
  if (R.has_reduce && !o.device_fn) R.segs[0].source += finish_source(R, o.prefix, tin, tw);
  return R;
}

}  // namespace cusadi
