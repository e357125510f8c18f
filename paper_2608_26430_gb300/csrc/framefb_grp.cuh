// Group-transform kernel of libframefb: the whole adapter pass (Sec. 3.1
// update, Lemma 1 gradient of Appendix A) for k = 16, k*rho = d frames on the
// CUDA cores, one thread per 32-coordinate group and token pair.  It serves
// fp32 activations and the bf16 shapes that the tcgen05 kernels do not fill
// (framefb_grp.cu says which).  Included by framefb_grp.cu only.
//
// Phi is block diagonal: a group's 16 complex coordinates times the realified
// DFT_16 / 4 (Sec. 3.2 construction), so a thread transforms its group in
// registers (radix 4 x 4, exact fp32) and only coefficients go through shared
// memory.  A unit is a few token pairs of one matrix.  Per unit u a CTA runs
//   phase A   synthesis of unit u - 1 (groups of RZ / RG added into the rows of
//             Y / dX) beside the analysis of unit u (V = X Phi_in, U = dY
//             Phi_out): neither touches the other's buffers, so the memory
//             latency of one hides behind the arithmetic of the other;
//   phase B   the coefficient SpMM of unit u (framefb_pair.cuh), run sums into
//             RZ / RG, dC in registers.
// The rows of the next unit are prefetched to L2 in phase B.
//
// BIG: plans of more than 16 entries per column (8192-entry supports) or of more
// coefficients than whole buffers hold.  The buffers hold only the coefficients
// that the support names (the popcount of the group's mask below a coefficient is
// its slot), so that pairs of 14336-wide rows fit where the support leaves most
// of them out (Zipf rows; 8192 uniform entries name too many), and the coefficient
// values and dC sums sit in shared memory.
//
// Bound: latency: two phases with a barrier between them, one or two CTAs per SM.
// Per token pair, fused: 768^2 in fp32 2.7 k shared-memory and L1 wavefronts and 0.9 k
// issue cycles in 4.0 k cycles; a 4096 -> 14336 BIG pair 20 k wavefronts (6 k of them
// bank conflicts) and 11 k issue cycles in 46 k; a third of the warps' waiting is for
// global loads, a fifth at the barriers.  Measured (fused pass, against the kernels
// that ran before): fp32, 8 matrices of 768^2, 2048 tokens 203 -> 105 us; a
// LLaMA-3-8B-shaped layer, Zipf supports, 16384 tokens 5.90 -> 4.08 ms.
#pragma once
#include "framefb_pair.cuh"

namespace ffb {
namespace grp {

using namespace pair;

// Bounded by construction: this kernel waits on nothing but CTA barriers.
constexpr int kMaxMats = 160;  // matrices of a launch

// Buffers of a token pair (float2 offsets), side 0 the input side (X, V, RG,
// dX), side 1 the output side (dY, U, RZ, Y): A[s] V or U, B[s] RG or RZ.
struct Shape {
  int32_t G[2];
  int32_t A[2], B[2];
  int32_t pair;  // float2 per token pair
  int32_t PP;    // token pairs per unit
};

struct Mat {
  const void* in[2];  // X, dY
  void* out[2];       // dX, Y
  int64_t ld[2];      // elements
  const uint8_t* plan;
  const float* c_val;
  int32_t N, ubeg, ntiles, shape;
  float seff;         // s / 16
  int32_t cost;       // of one unit, relative
  int64_t cbeg;       // cost of the units before ubeg
};

// Matrix that holds position x of a list whose matrices begin at first(j).
template <typename First, typename T>
__host__ __device__ __forceinline__ int32_t matrix_at(int32_t nmats, T x, First first) {
  int32_t lo = 0, hi = nmats - 1;
  while (lo < hi) {
    const int32_t mid = (lo + hi + 1) >> 1;
    if (first(mid) <= x)
      lo = mid;
    else
      hi = mid - 1;
  }
  return lo;
}

// First unit of CTA c of `grid`: the units are split at equal cost.  (A CTA whose
// share lies inside one unit has none.)
template <typename L>
__host__ __device__ __forceinline__ int32_t first_unit(const L& a, int32_t c, int32_t grid) {
  const int64_t x = a.total_cost * c / grid;
  const int32_t j = matrix_at(a.nmats, x, [&](int32_t i) { return a.m[i].cbeg; });
  return a.m[j].ubeg + static_cast<int32_t>((x - a.m[j].cbeg + a.m[j].cost - 1) / a.m[j].cost);
}

struct Launch {
  int32_t nmats, total_units, stride, mode;
  int32_t oPlan, oMask;  // shared memory (bytes): plan columns, group masks; pair buffers at 0
  int64_t total_cost;    // sum over the matrices of ntiles * cost
  float* partial;        // [(grid + nmats) * stride] dC partial sums, slot = cta + matrix
  Shape sh[kMaxMats];    // distinct geometries
  Mat m[kMaxMats];
};

// DFT_16 in place: X_q = sum_r x_r e^{S 2 pi i q r / 16}, output q in slot
// 4 (q mod 4) + q / 4.
template <int S>
__device__ __forceinline__ void dft16(C2 (&x)[16]) {
#pragma unroll
  for (int j = 0; j < 4; ++j) dft4<S>(x[j], x[4 + j], x[8 + j], x[12 + j]);
  constexpr float c1 = 0.92387953251128674f, s1 = 0.38268343236508977f;  // e^{i pi / 8}
  auto w = [](float c, float s) { return C2{pk(c, c), pk(S > 0 ? s : -s, S > 0 ? s : -s)}; };
  x[5] = cmul(x[5], w(c1, s1));
  x[9] = rot8<S, 1>(x[9]);
  x[13] = cmul(x[13], w(s1, c1));
  x[6] = rot8<S, 1>(x[6]);
  {  // * (i S)
    const C2 z{0ull, 0ull};
    x[10] = addi<S>(z, x[10]);
  }
  x[14] = rot8<S, 3>(x[14]);
  x[7] = cmul(x[7], w(s1, c1));
  x[11] = rot8<S, 3>(x[11]);
  x[15] = cmul(x[15], w(-c1, -s1));
#pragma unroll
  for (int j = 0; j < 4; ++j) dft4<S>(x[4 * j], x[4 * j + 1], x[4 * j + 2], x[4 * j + 3]);
}
__device__ __forceinline__ constexpr int slot16(int q) { return 4 * (q & 3) + (q >> 2); }

// float4 of complex coefficient i of group g in a buffer: the low bits
// permuted by the group, so that lanes on neighbouring groups hit distinct banks.
__device__ __forceinline__ int at_group(int g, int i) { return 16 * g + (i ^ (g & 7)); }
// float2 of frame column x (group-major)
__device__ __forceinline__ uint32_t col_slot(uint32_t x) {
  const uint32_t g = x >> 5, c = x & 31;
  return 32 * g + 2 * ((c >> 1) ^ (g & 7)) + (c & 1);
}

// ---------------------------------------------------------------------------
// one group of a token's row: 32 elements; quarter q = elements 8q .. 8q + 7
// ---------------------------------------------------------------------------
__device__ __forceinline__ void ld256(const void* p, bool wide, uint4& a, uint4& b) {
  if (wide) {
    asm volatile("ld.global.v8.u32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(a.x), "=r"(a.y), "=r"(a.z), "=r"(a.w), "=r"(b.x), "=r"(b.y), "=r"(b.z), "=r"(b.w)
                 : "l"(p));
  } else {
    a = reinterpret_cast<const uint4*>(p)[0];
    b = reinterpret_cast<const uint4*>(p)[1];
  }
}
__device__ __forceinline__ void st256(void* p, bool wide, const uint4& a, const uint4& b) {
  if (wide) {
    asm volatile("st.global.v8.u32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"l"(p), "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w),
                 "r"(b.x), "r"(b.y), "r"(b.z), "r"(b.w)
                 : "memory");
  } else {
    reinterpret_cast<uint4*>(p)[0] = a;
    reinterpret_cast<uint4*>(p)[1] = b;
  }
}

// Elements per 32-byte access, and its complex coordinates as floats.
template <typename Elem>
struct Io;
template <>
struct Io<__nv_bfloat16> {
  static constexpr int kPer = 16;
  static __device__ __forceinline__ void unpack(const uint4& a, const uint4& b, float (&v)[16]) {
    const uint32_t w[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      v[2 * i] = __uint_as_float(w[i] << 16);
      v[2 * i + 1] = __uint_as_float(w[i] & 0xFFFF0000u);
    }
  }
  static __device__ __forceinline__ void pack(const float (&v)[16], uint4& a, uint4& b) {
    uint32_t w[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) w[i] = pack_bf16(v[2 * i], v[2 * i + 1]);
    a = make_uint4(w[0], w[1], w[2], w[3]);
    b = make_uint4(w[4], w[5], w[6], w[7]);
  }
};
template <>
struct Io<float> {
  static constexpr int kPer = 8;
  static __device__ __forceinline__ void unpack(const uint4& a, const uint4& b, float (&v)[8]) {
    const uint32_t w[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = __uint_as_float(w[i]);
  }
  static __device__ __forceinline__ void pack(const float (&v)[8], uint4& a, uint4& b) {
    a = make_uint4(__float_as_uint(v[0]), __float_as_uint(v[1]), __float_as_uint(v[2]), __float_as_uint(v[3]));
    b = make_uint4(__float_as_uint(v[4]), __float_as_uint(v[5]), __float_as_uint(v[6]), __float_as_uint(v[7]));
  }
};

// The current matrix, in shared memory.
template <typename Elem>
struct Cur {
  int32_t G[2], A[2], B[2];
  int32_t pair;
  float seff;
  const Elem* in[2];
  Elem* out[2];
  int64_t ld[2];
  int32_t wide_in[2], wide_out[2];  // 32-byte aligned rows
};

// Group g of the token pair (t, t + 1) of a row matrix as 16 complex pairs.
template <typename Elem>
__device__ __forceinline__ void load_rows(const Elem* row, int64_t ld, bool two, bool wide, C2 (&x)[16]) {
  constexpr int PER = Io<Elem>::kPer, Q = 32 / PER;
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    uint4 a0, b0, a1 = make_uint4(0, 0, 0, 0), b1 = a1;
    ld256(row + q * PER, wide, a0, b0);
    if (two) ld256(row + ld + q * PER, wide, a1, b1);
    float u[PER], v[PER];
    Io<Elem>::unpack(a0, b0, u);
    Io<Elem>::unpack(a1, b1, v);
#pragma unroll
    for (int i = 0; i < PER / 2; ++i) x[q * PER / 2 + i] = C2{pk(u[2 * i], v[2 * i]), pk(u[2 * i + 1], v[2 * i + 1])};
  }
}

// row += seff * x (x in slot16 order) for both tokens of the pair.
template <typename Elem>
__device__ __forceinline__ void add_rows(Elem* row, int64_t ld, bool two, bool wide, float seff, const C2 (&x)[16]) {
  constexpr int PER = Io<Elem>::kPer, Q = 32 / PER;
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    uint4 a[2], b[2];
#pragma unroll
    for (int t = 0; t < 2; ++t)
      if (t == 0 || two) ld256(row + t * ld + q * PER, wide, a[t], b[t]);
    float d0[PER], d1[PER];
#pragma unroll
    for (int i = 0; i < PER / 2; ++i) {
      const C2 z = x[slot16(q * PER / 2 + i)];
      unpk(z.re, d0[2 * i], d1[2 * i]);
      unpk(z.im, d0[2 * i + 1], d1[2 * i + 1]);
    }
#pragma unroll
    for (int t = 0; t < 2; ++t) {
      if (t == 1 && !two) break;
      float y[PER];
      Io<Elem>::unpack(a[t], b[t], y);
#pragma unroll
      for (int i = 0; i < PER; ++i) y[i] = fmaf(seff, t == 0 ? d0[i] : d1[i], y[i]);
      uint4 ra, rb;
      Io<Elem>::pack(y, ra, rb);
      st256(row + t * ld + q * PER, wide, ra, rb);
    }
  }
}

// ---------------------------------------------------------------------------
// A thread's share of a plan column, in shared memory (a group's transform
// takes half the registers; plan words beside it would spill): five arrays of
// one uint4 per four entries and thread,
//   0: V offset | RZ target << 16, 1: its coefficient value,
//   2: U offset | RG target << 16, 3: its value, 4: V offset of the column,
// offsets and targets in bytes.  The dC sums stay in registers.
// ---------------------------------------------------------------------------
struct Cols {
  uint32_t zcarry, gcarry;  // targets of the runs that a column's first half leaves open
  int hZ, hG;               // entries per thread
};
__host__ __device__ constexpr int cols_bytes(int NT, int KE) { return 5 * KE * NT * 4; }

template <int KE, int NT>
__device__ __forceinline__ uint4 get_cols(const uint8_t* sp, int a, int i0) {
  return reinterpret_cast<const uint4*>(sp)[(a * (KE / 4) + i0 / 4) * NT + threadIdx.x];
}

template <int KE, int H, int NT>
__device__ __forceinline__ void load_cols(Cols& ch, uint8_t* sp, int mode, const uint8_t* plan, const float* c_val, int col,
                                          int half) {
  const bool F = mode & kF, D = mode & kD, C = mode & kC;
  const FfbPlanHeader& h = *reinterpret_cast<const FfbPlanHeader*>(plan);
  auto tab = [&](int32_t off) { return reinterpret_cast<const int32_t*>(plan + off); };
  ch.hZ = F ? half_of<H>(h.EZ) : 0;
  ch.hG = D || C ? half_of<H>(h.EG) : 0;
  const int K[2] = {h.n, h.m};
  auto word = [&](uint32_t w, int ts) {  // store target of side ts
    const uint32_t t = w >> 16;
    const uint32_t o = t == FFB_NO_STORE ? t : 8u * (static_cast<int>(t) < K[ts] ? col_slot(t) : t);
    return 8u * col_slot(w & 0x7FFFu) | (o << 16);
  };
  bool openZ = false, openG = false;
  uint32_t firstZ = FFB_NO_STORE, firstG = FFB_NO_STORE;
  auto put = [&](int a, int i, uint32_t x) {
    reinterpret_cast<uint32_t*>(sp)[((a * (KE / 4) + i / 4) * NT + threadIdx.x) * 4 + (i & 3)] = x;
  };
#pragma unroll
  for (int i = 0; i < KE; ++i) {
    uint32_t zw = FFB_NO_STORE << 16, gw = FFB_NO_STORE << 16, gb = 0;
    float zc = 0.f, gc = 0.f;
    const int ez = half * ch.hZ + i, eg = half * ch.hG + i;
    if (i < ch.hZ && ez < h.EZ) {
      zw = word(static_cast<uint32_t>(ld_g(tab(h.off_zb) + ez * kColumns + col)), 1);
      const int32_t qi = ld_g(tab(h.off_zq) + ez * kColumns + col);
      zc = qi >= 0 ? ld_g(c_val + qi) : 0.f;
      openZ = qi >= 0 && (zw >> 16) == FFB_NO_STORE;
      if (firstZ == FFB_NO_STORE) firstZ = zw >> 16;
    }
    if (i < ch.hG && eg < h.EG) {
      gw = word(static_cast<uint32_t>(ld_g(tab(h.off_ga) + eg * kColumns + col)), 0);
      gb = 8u * col_slot(static_cast<uint32_t>(ld_g(tab(h.off_gb) + eg * kColumns + col)));
      const int32_t qi = ld_g(tab(h.off_gq) + eg * kColumns + col);
      gc = (D && qi >= 0) ? ld_g(c_val + qi) : 0.f;
      openG = qi >= 0 && (gw >> 16) == FFB_NO_STORE;
      if (firstG == FFB_NO_STORE) firstG = gw >> 16;
      if (!D) gw |= FFB_NO_STORE << 16;
    }
    put(0, i, zw);
    put(1, i, __float_as_uint(zc));
    put(2, i, gw);
    put(3, i, __float_as_uint(gc));
    put(4, i, gb);
  }
  ch.zcarry = ch.gcarry = FFB_NO_STORE;
  if constexpr (H == 2) {
    const uint32_t open = __shfl_xor_sync(0xffffffffu, (openZ ? 1u : 0u) | (openG ? 2u : 0u), 16);
    if (half == 1) {
      if (open & 1u) ch.zcarry = firstZ;
      if ((open & 2u) && D) ch.gcarry = firstG;
    }
  }
}

// U[a] V[b] of both tokens.  Summed before it goes to the dC sum: a chain of one
// rounding per pair instead of two (8 matrices of 768^2 fp32, 2048 tokens: dC against
// fp64 1.81e-7 -> 1.61e-7 relative, the one-phase kernel 1.72e-7).
__device__ __forceinline__ float pair_dot(float2 u, float2 v) { return fmaf(u.x, v.x, u.y * v.y); }

// The coefficient SpMM of one token pair: run sums of c V[b] -> RZ (F), of
// c U[a] -> RG (D), dC += U[a] V[b] (C).
template <int KE, int H, int NT>
__device__ __forceinline__ void spmm_cols(const Cols& ch, float (&dc)[KE], const uint8_t* sp, bool F, bool D, bool C,
                                          const float2* V, const float2* U, float2* RG, float2* RZ) {
  if (D || C) {
    float2 acc = make_float2(0.f, 0.f);
#pragma unroll
    for (int i0 = 0; i0 < KE; i0 += 4) {
      if (i0 >= ch.hG) continue;
      const uint4 w4 = get_cols<KE, NT>(sp, 2, i0), c4 = get_cols<KE, NT>(sp, 3, i0), b4 = get_cols<KE, NT>(sp, 4, i0);
      const uint32_t w[4] = {w4.x, w4.y, w4.z, w4.w}, gb[4] = {b4.x, b4.y, b4.z, b4.w};
      const float gc[4] = {__uint_as_float(c4.x), __uint_as_float(c4.y), __uint_as_float(c4.z), __uint_as_float(c4.w)};
      float2 ub[4], vb[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        ub[e] = at(U, w[e] & 0xFFFFu);
        vb[e] = C ? at(V, gb[e]) : make_float2(0.f, 0.f);
      }
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        dc[i0 + e] += pair_dot(ub[e], vb[e]);
        acc.x = fmaf(gc[e], ub[e].x, acc.x);
        acc.y = fmaf(gc[e], ub[e].y, acc.y);
        const uint32_t t = w[e] >> 16;
        if (t != FFB_NO_STORE) {
          at(RG, t) = acc;
          acc = make_float2(0.f, 0.f);
        }
      }
    }
    if constexpr (H == 2) {
      const float cx = __shfl_xor_sync(0xffffffffu, acc.x, 16), cy = __shfl_xor_sync(0xffffffffu, acc.y, 16);
      if (ch.gcarry != FFB_NO_STORE) {
        float2& o = at(RG, ch.gcarry);
        o = make_float2(cx + o.x, cy + o.y);
      }
    }
  }
  if (F) {
    float2 acc = make_float2(0.f, 0.f);
#pragma unroll
    for (int i0 = 0; i0 < KE; i0 += 4) {
      if (i0 >= ch.hZ) continue;
      const uint4 w4 = get_cols<KE, NT>(sp, 0, i0), c4 = get_cols<KE, NT>(sp, 1, i0);
      const uint32_t w[4] = {w4.x, w4.y, w4.z, w4.w};
      const float zc[4] = {__uint_as_float(c4.x), __uint_as_float(c4.y), __uint_as_float(c4.z), __uint_as_float(c4.w)};
      float2 vz[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) vz[e] = at(V, w[e] & 0xFFFFu);
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        acc.x = fmaf(zc[e], vz[e].x, acc.x);
        acc.y = fmaf(zc[e], vz[e].y, acc.y);
        const uint32_t t = w[e] >> 16;
        if (t != FFB_NO_STORE) {
          at(RZ, t) = acc;
          acc = make_float2(0.f, 0.f);
        }
      }
    }
    if constexpr (H == 2) {
      const float cx = __shfl_xor_sync(0xffffffffu, acc.x, 16), cy = __shfl_xor_sync(0xffffffffu, acc.y, 16);
      if (ch.zcarry != FFB_NO_STORE) {
        float2& o = at(RZ, ch.zcarry);
        o = make_float2(cx + o.x, cy + o.y);
      }
    }
  }
}

// ---------------------------------------------------------------------------
// BIG plans: KE = 16 entries per thread (two threads per column of up to 32).
//   z: V slot (13 bits) | RZ target (12) << 13 | low 7 bits of gb << 25
//   g: U slot (12) | RG target (13) << 12 | high 6 bits of gb << 25
// (all ones in a target: no store).  Coefficient values of both paths and the
// dC sums: arrays of one float4 per four entries and thread.
// ---------------------------------------------------------------------------
constexpr int kBigE = 16;
constexpr uint32_t kNoZ = 0xFFFu, kNoG = 0x1FFFu;
constexpr int kBigU = 4094, kBigV = 8190;  // slots (with overflow) of the two sides
struct Big {
  uint32_t z[kBigE], g[kBigE];
  uint32_t zcarry, gcarry;
  int hZ, hG;
  __device__ __forceinline__ uint32_t gb(int e) const { return (z[e] >> 25) | ((g[e] >> 25) << 7); }
};
__host__ __device__ constexpr int big_bytes(int NT) { return 3 * kBigE * NT * 4; }

template <int NT, typename Slot, typename Over>
__device__ __forceinline__ void load_big(Big& ch, uint8_t* sp, int mode, const uint8_t* plan, const float* c_val, int col,
                                         int half, Slot slot, Over over) {
  const bool F = mode & kF, D = mode & kD, C = mode & kC;
  const FfbPlanHeader& h = *reinterpret_cast<const FfbPlanHeader*>(plan);
  auto tab = [&](int32_t off) { return reinterpret_cast<const int32_t*>(plan + off); };
  ch.hZ = F ? half_of<2>(h.EZ) : 0;
  ch.hG = D || C ? half_of<2>(h.EG) : 0;
  const int K[2] = {h.n, h.m};
  auto target = [&](uint32_t t, int sd) {
    return static_cast<int>(t) < K[sd] ? slot(sd, t) : over(sd, t - K[sd]);
  };
  bool openZ = false, openG = false;
  uint32_t firstZ = kNoZ, firstG = kNoG;
  float* arr = reinterpret_cast<float*>(sp);
  auto put = [&](int a, int i, float x) { arr[((a * (kBigE / 4) + i / 4) * NT + threadIdx.x) * 4 + (i & 3)] = x; };
#pragma unroll
  for (int i = 0; i < kBigE; ++i) {
    uint32_t z = kNoZ << 13, g = kNoG << 12;
    float zc = 0.f, gc = 0.f;
    const int ez = half * ch.hZ + i, eg = half * ch.hG + i;
    if (i < ch.hZ && ez < h.EZ) {
      const uint32_t w = static_cast<uint32_t>(ld_g(tab(h.off_zb) + ez * kColumns + col));
      const int32_t qi = ld_g(tab(h.off_zq) + ez * kColumns + col);
      const uint32_t t = (w >> 16) == FFB_NO_STORE ? kNoZ : target(w >> 16, 1);
      // (padding entries carry column 0: slot 0 of the buffer, with value 0)
      z = (qi >= 0 ? slot(0, w & 0x7FFFu) : 0u) | (t << 13);
      zc = qi >= 0 ? ld_g(c_val + qi) : 0.f;
      openZ = qi >= 0 && t == kNoZ;
      if (firstZ == kNoZ) firstZ = t;
    }
    if (i < ch.hG && eg < h.EG) {
      const uint32_t w = static_cast<uint32_t>(ld_g(tab(h.off_ga) + eg * kColumns + col));
      const int32_t qi = ld_g(tab(h.off_gq) + eg * kColumns + col);
      const uint32_t t = (w >> 16) == FFB_NO_STORE || !D ? kNoG : target(w >> 16, 0);
      const uint32_t b = qi >= 0 ? slot(0, static_cast<uint32_t>(ld_g(tab(h.off_gb) + eg * kColumns + col))) : 0u;
      g = (qi >= 0 ? slot(1, w & 0x7FFFu) : 0u) | (t << 12) | ((b >> 7) << 25);
      z |= (b & 127u) << 25;
      gc = (D && qi >= 0) ? ld_g(c_val + qi) : 0.f;
      openG = D && qi >= 0 && t == kNoG;
      if (firstG == kNoG) firstG = t;
    }
    ch.z[i] = z;
    ch.g[i] = g;
    put(0, i, zc);
    put(1, i, gc);
    put(2, i, 0.f);
  }
  const uint32_t open = __shfl_xor_sync(0xffffffffu, (openZ ? 1u : 0u) | (openG ? 2u : 0u), 16);
  ch.zcarry = half == 1 && (open & 1u) ? firstZ : kNoZ;
  ch.gcarry = half == 1 && (open & 2u) ? firstG : kNoG;
}

template <int NT>
__device__ __forceinline__ void spmm_big(const Big& ch, uint8_t* sp, bool F, bool D, bool C, const float2* V,
                                         const float2* U, float2* RG, float2* RZ) {
  float4* arr = reinterpret_cast<float4*>(sp) + threadIdx.x;
  if (D || C) {
    float2 acc = make_float2(0.f, 0.f);
#pragma unroll
    for (int i0 = 0; i0 < kBigE; i0 += 4) {
      if (i0 >= ch.hG) continue;
      const float4 gc4 = arr[(kBigE / 4 + i0 / 4) * NT];
      float4 dc4 = arr[(2 * (kBigE / 4) + i0 / 4) * NT];
      const float gc[4] = {gc4.x, gc4.y, gc4.z, gc4.w};
      float dc[4] = {dc4.x, dc4.y, dc4.z, dc4.w};
      float2 ub[4], vb[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        ub[e] = U[ch.g[i0 + e] & 0xFFFu];
        vb[e] = C ? V[ch.gb(i0 + e)] : make_float2(0.f, 0.f);
      }
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        dc[e] += pair_dot(ub[e], vb[e]);
        acc.x = fmaf(gc[e], ub[e].x, acc.x);
        acc.y = fmaf(gc[e], ub[e].y, acc.y);
        const uint32_t t = (ch.g[i0 + e] >> 12) & kNoG;
        if (t != kNoG) {
          RG[t] = acc;
          acc = make_float2(0.f, 0.f);
        }
      }
      if (C) arr[(2 * (kBigE / 4) + i0 / 4) * NT] = make_float4(dc[0], dc[1], dc[2], dc[3]);
    }
    const float cx = __shfl_xor_sync(0xffffffffu, acc.x, 16), cy = __shfl_xor_sync(0xffffffffu, acc.y, 16);
    if (ch.gcarry != kNoG) {
      float2& o = RG[ch.gcarry];
      o = make_float2(cx + o.x, cy + o.y);
    }
  }
  if (F) {
    float2 acc = make_float2(0.f, 0.f);
#pragma unroll
    for (int i0 = 0; i0 < kBigE; i0 += 4) {
      if (i0 >= ch.hZ) continue;
      const float4 zc4 = arr[(i0 / 4) * NT];
      const float zc[4] = {zc4.x, zc4.y, zc4.z, zc4.w};
      float2 vz[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) vz[e] = V[ch.z[i0 + e] & 0x1FFFu];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        acc.x = fmaf(zc[e], vz[e].x, acc.x);
        acc.y = fmaf(zc[e], vz[e].y, acc.y);
        const uint32_t t = (ch.z[i0 + e] >> 13) & kNoZ;
        if (t != kNoZ) {
          RZ[t] = acc;
          acc = make_float2(0.f, 0.f);
        }
      }
    }
    const float cx = __shfl_xor_sync(0xffffffffu, acc.x, 16), cy = __shfl_xor_sync(0xffffffffu, acc.y, 16);
    if (ch.zcarry != kNoZ) {
      float2& o = RZ[ch.zcarry];
      o = make_float2(cx + o.x, cy + o.y);
    }
  }
}

// ---------------------------------------------------------------------------
template <typename Elem, int NT, int KE, bool BIG>
__global__ void __launch_bounds__(NT, NT == 512 ? 1 : 2) fft_tile_kernel(const __grid_constant__ Launch args) {
  chain_wait();
  chain_next();
  static_assert(!BIG || (NT == 512 && KE == kBigE), "big plans: two threads per column");
  constexpr int H = NT / kColumns;
  extern __shared__ __align__(128) uint8_t smem[];
  __shared__ Cur<Elem> cur_s;
  const int mode = args.mode;
  const bool F = mode & kF, D = mode & kD, C = mode & kC;
  const int kAna = (F || C ? 1 : 0) | (D || C ? 2 : 0), kSyn = (D ? 1 : 0) | (F ? 2 : 0);
  const int tid = threadIdx.x, lane = tid & 31;
  const int half = H == 2 ? lane >> 4 : 0;
  const int col = H == 2 ? (tid >> 5) * 16 + (lane & 15) : tid;
  float2* pairs = reinterpret_cast<float2*>(smem);
  uint8_t* sp = smem + args.oPlan;
  uint32_t* masks = reinterpret_cast<uint32_t*>(smem + args.oMask);  // side 0's groups, then side 1's
  uint32_t* bases = nullptr;                                        // BIG: first slot of each group

  const int u_begin = first_unit(args, blockIdx.x, gridDim.x);
  const int u_end = blockIdx.x + 1 == gridDim.x ? args.total_units : first_unit(args, blockIdx.x + 1, gridDim.x);
  if (u_begin >= u_end) {
    // no unit: the dC reduction still sums this CTA's slot of a matrix with units
    // on both sides of it
    if (C && u_begin < args.total_units) {
      const int k = matrix_at(args.nmats, u_begin, [&](int32_t i) { return args.m[i].ubeg; });
      if (u_begin > args.m[k].ubeg) {
        float* dst = args.partial + static_cast<size_t>(blockIdx.x + k) * args.stride;
        const int nnz = reinterpret_cast<const FfbPlanHeader*>(args.m[k].plan)->nnz;
        for (int q = tid; q < nnz; q += NT) dst[q] = 0.f;
      }
    }
    return;
  }

  // slots of frame columns in the pair buffers
  int G0 = 0, G1 = 0, cnt0 = 0, cnt1 = 0;
  auto slot = [&](int sd, uint32_t x) -> uint32_t {
    if constexpr (BIG) {
      const int g = (sd ? G0 : 0) + (x >> 5);
      return bases[g] + __popc(masks[g] & ((1u << (x & 31)) - 1u));
    } else {
      return col_slot(x);
    }
  };
  auto over = [&](int sd, uint32_t o) -> uint32_t { return (sd ? cnt1 : cnt0) + o; };

  // analysis of group task r of a pair's input rows, synthesis likewise
  auto analyse = [&](int p, int r, int64_t t0, int ntok) {
    const int sd = kAna == 2 || r >= (kAna & 1 ? G0 : 0) ? 1 : 0;
    const int g = kAna == 3 && sd ? r - G0 : r;
    const uint32_t mask = masks[(sd ? G0 : 0) + g];
    if (mask == 0u) return;  // no coefficient of this group is read
    C2 x[16];
    load_rows<Elem>(cur_s.in[sd] + (t0 + 2 * p) * cur_s.ld[sd] + 32 * g, cur_s.ld[sd], 2 * p + 1 < ntok, cur_s.wide_in[sd], x);
    dft16<1>(x);
    float2* A = pairs + p * cur_s.pair + cur_s.A[sd];
    if constexpr (BIG) {
      float2* a = A + bases[(sd ? G0 : 0) + g];
#pragma unroll
      for (int c = 0; c < 32; ++c) {
        const C2 z = x[slot16(c >> 1)];
        if (mask >> c & 1u) *reinterpret_cast<f2*>(a++) = c & 1 ? z.im : z.re;
      }
    } else {
      float4* a = reinterpret_cast<float4*>(A);
#pragma unroll
      for (int i = 0; i < 16; ++i) sts_c(a + at_group(g, i), x[slot16(i)]);
    }
  };
  auto synthesise = [&](int p, int r, int64_t t0, int ntok) {
    const int sd = kSyn == 2 || r >= (kSyn & 1 ? G0 : 0) ? 1 : 0;
    const int g = kSyn == 3 && sd ? r - G0 : r;
    const uint32_t mask = masks[(sd ? G0 : 0) + g];
    if (mask == 0u) return;  // no run sum falls in this group
    C2 x[16];
    const float2* B = pairs + p * cur_s.pair + cur_s.B[sd];
    if constexpr (BIG) {
      const float2* b = B + bases[(sd ? G0 : 0) + g];
#pragma unroll
      for (int c = 0; c < 32; ++c) {
        f2 v = 0ull;
        if (mask >> c & 1u) v = *reinterpret_cast<const f2*>(b++);
        if (c & 1)
          x[c >> 1].im = v;
        else
          x[c >> 1].re = v;
      }
    } else {
      const float4* b = reinterpret_cast<const float4*>(B);
#pragma unroll
      for (int i = 0; i < 16; ++i) x[i] = lds_c(b + at_group(g, i));
    }
    dft16<-1>(x);
    add_rows<Elem>(cur_s.out[sd] + (t0 + 2 * p) * cur_s.ld[sd] + 32 * g, cur_s.ld[sd], 2 * p + 1 < ntok, cur_s.wide_out[sd],
                   cur_s.seff, x);
  };
  // tasks [0, ns): synthesis of the pairs of unit (ts0, ts), [ns, ns + na): analysis of (ta0, ta)
  auto phase = [&](int64_t ts0, int ts, int64_t ta0, int ta) {
    const int gs = (kSyn & 1 ? G0 : 0) + (kSyn & 2 ? G1 : 0), ga = (kAna & 1 ? G0 : 0) + (kAna & 2 ? G1 : 0);
    const int ns = ((ts + 1) >> 1) * gs, na = ((ta + 1) >> 1) * ga;
    int t = tid;
    asm volatile("" : "+r"(t));
    for (; t < ns + na; t += NT) {
      if (t < ns) {
        const int p = t / gs;
        synthesise(p, t - p * gs, ts0, ts);
      } else {
        const int p = (t - ns) / ga;
        analyse(p, t - ns - p * ga, ta0, ta);
      }
    }
  };

  using Chunk = std::conditional_t<BIG, Big, Cols>;
  Chunk ch{};
  float dc[BIG ? 1 : KE];
  int cur = -1, j = matrix_at(args.nmats, u_begin, [&](int32_t i) { return args.m[i].ubeg; });
  int nfZ = 0, nfix = 0, PP = 1;
  const uint8_t* plan = nullptr;
  auto flush = [&](int mat) {
    if (!C) return;
    float* dst = args.partial + static_cast<size_t>(blockIdx.x + mat) * args.stride;
    if constexpr (BIG) {
      const FfbPlanHeader& h = *reinterpret_cast<const FfbPlanHeader*>(plan);
      const int32_t* gq = reinterpret_cast<const int32_t*>(plan + h.off_gq);
      const float* arr = reinterpret_cast<const float*>(sp);
      for (int i = 0; i < ch.hG; ++i) {
        const int e = half * ch.hG + i;
        if (e < h.EG) {
          const int32_t qi = ld_g(gq + e * kColumns + col);
          if (qi >= 0) dst[qi] = arr[((2 * (kBigE / 4) + i / 4) * NT + tid) * 4 + (i & 3)];
        }
      }
    } else {
      flush_dc(plan, dst, dc, ch.hG, col, half);
    }
  };

  int64_t tp0 = 0;  // the previous unit (of the same matrix): first token, tokens
  int tp = 0;
  for (int u = u_begin; u < u_end; ++u) {
    while (u >= args.m[j].ubeg + args.m[j].ntiles) ++j;
    if (j != cur) {
      if (cur >= 0) {
        phase(tp0, tp, 0, 0);
        tp = 0;
        flush(cur);
        __syncthreads();
      }
      cur = j;
      const Mat& M = args.m[j];
      const Shape& sh = args.sh[M.shape];
      plan = M.plan;
      const FfbPlanHeader& h = *reinterpret_cast<const FfbPlanHeader*>(plan);
      nfZ = F ? h.nfixZ : 0;
      nfix = nfZ + (D ? h.nfixG : 0);
      G0 = sh.G[0];
      G1 = sh.G[1];
      PP = sh.PP;
      if (tid < 2) {
        cur_s.G[tid] = sh.G[tid];
        cur_s.A[tid] = sh.A[tid];
        cur_s.B[tid] = sh.B[tid];
        cur_s.in[tid] = static_cast<const Elem*>(M.in[tid]);
        cur_s.out[tid] = static_cast<Elem*>(M.out[tid]);
        cur_s.ld[tid] = M.ld[tid];
        const bool rows32 = (M.ld[tid] * sizeof(Elem)) % 32 == 0;
        cur_s.wide_in[tid] = rows32 && (reinterpret_cast<uintptr_t>(M.in[tid]) & 31u) == 0;
        cur_s.wide_out[tid] = rows32 && (reinterpret_cast<uintptr_t>(M.out[tid]) & 31u) == 0;
        cur_s.pair = sh.pair;
        cur_s.seff = M.seff;
      }
      const uint32_t* gm = reinterpret_cast<const uint32_t*>(plan + h.off_gmask);
      const uint32_t* zm = reinterpret_cast<const uint32_t*>(plan + h.off_zmask);
      for (int g = tid; g < G0 + G1; g += NT) masks[g] = g < G0 ? ld_g(gm + g) : ld_g(zm + (g - G0));
      // run-sum slots that no run writes read as zero
      for (int x = tid; x < PP * sh.pair; x += NT) pairs[x] = make_float2(0.f, 0.f);
      __syncthreads();
      if constexpr (BIG) {
        bases = masks + G0 + G1;
        if (tid < 32) {  // exclusive prefix sums of the masks' popcounts, per side
          for (int sd = 0; sd < 2; ++sd) {
            const int o = sd ? G0 : 0, n = sd ? G1 : G0;
            uint32_t run = 0;
            for (int g = lane; g < (n + 31) / 32 * 32; g += 32) {
              const uint32_t c = g < n ? __popc(masks[o + g]) : 0u;
              uint32_t inc = c;
#pragma unroll
              for (int d = 1; d < 32; d *= 2) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, inc, d);
                if (lane >= d) inc += y;
              }
              if (g < n) bases[o + g] = run + inc - c;
              run += __shfl_sync(0xffffffffu, inc, 31);
            }
            if (lane == 0) bases[G0 + G1 + sd] = run;
          }
        }
        __syncthreads();
        cnt0 = bases[G0 + G1];
        cnt1 = bases[G0 + G1 + 1];
        load_big<NT>(ch, sp, mode, plan, M.c_val, col, half, slot, over);
      } else {
        load_cols<KE, H, NT>(ch, sp, mode, plan, M.c_val, col, half);
#pragma unroll
        for (int i = 0; i < KE; ++i) dc[i] = 0.f;
      }
    }
    const int64_t t0 = 2 * static_cast<int64_t>(PP) * (u - args.m[j].ubeg);
    const int ntok = static_cast<int>(min(static_cast<int64_t>(2 * PP), args.m[j].N - t0));
    const int npair = (ntok + 1) >> 1;

    phase(tp0, tp, t0, ntok);
    __syncthreads();

    // rows towards L2, one 128-byte line per thread and turn: this unit's
    // output rows and the next unit's input rows
    {
      const int64_t left = args.m[j].N - t0 - ntok;
      const int nin = static_cast<int>(min(static_cast<int64_t>(2 * PP), left > 0 ? left : 0));
#pragma unroll
      for (int w = 0; w < 4; ++w) {
        const int sd = w & 1;
        const bool in = w >= 2;
        if (!(((in ? kAna : kSyn) >> sd) & 1)) continue;
        const int lines = (sd ? G1 : G0) * (32 * static_cast<int>(sizeof(Elem))) / 128 + 1;  // rows may start inside a line
        const int rows = in ? nin : ntok;
        const Elem* base = in ? cur_s.in[sd] + (t0 + ntok) * cur_s.ld[sd] : cur_s.out[sd] + t0 * cur_s.ld[sd];
        const int bytes = (sd ? G1 : G0) * 32 * static_cast<int>(sizeof(Elem));
        for (int x = tid; x < lines * rows; x += NT) {
          const int r = x / lines, o = min(128 * (x - r * lines), bytes - 1);
          asm volatile("prefetch.global.L2 [%0];" ::"l"(reinterpret_cast<const uint8_t*>(base + r * cur_s.ld[sd]) + o));
        }
      }
    }

    for (int p = 0; p < npair; ++p) {
      float2* b = pairs + p * cur_s.pair;
      if constexpr (BIG)
        spmm_big<NT>(ch, sp, F, D, C, b + cur_s.A[0], b + cur_s.A[1], b + cur_s.B[0], b + cur_s.B[1]);
      else
        spmm_cols<KE, H, NT>(ch, dc, sp, F, D, C, b + cur_s.A[0], b + cur_s.A[1], b + cur_s.B[0], b + cur_s.B[1]);
    }
    __syncthreads();
    if (kSyn && nfix > 0) {
      const FfbPlanHeader& h = *reinterpret_cast<const FfbPlanHeader*>(plan);
      const int n = h.n, m = h.m;
      fix_runs<NT>(plan, nfZ, nfix, npair, pairs + cur_s.B[0], pairs + cur_s.B[1], cur_s.pair, [&](int sd, uint32_t x) -> uint32_t {
        const uint32_t K = sd ? m : n;
        return x < K ? slot(sd, x) : BIG ? over(sd, x - K) : x;
      });
      __syncthreads();
    }
    tp0 = t0;
    tp = kSyn ? ntok : 0;
  }
  phase(tp0, tp, 0, 0);
  if (cur >= 0) flush(cur);
}

}  // namespace grp
}  // namespace ffb
