// Device code shared by the token-pair kernels of libframefb (framefb_row.cuh,
// framefb_grp.cuh): fp32x2 arithmetic on token pairs, the plan shares, the
// coefficient SpMM, the dC reduction.
//
// Every value is a token pair: complex element i of a buffer is the float4
// (re t0, re t1, im t0, im t1), so one fp32x2 instruction serves both tokens,
// a coefficient (column 2i + s) is one float2, and the SpMM gathers both
// tokens with one 8-byte access.
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

#include "framefb_ptx.cuh"
#include "plan_layout.h"

namespace ffb {
namespace pair {

enum { kF = 1, kD = 2, kC = 4 };
constexpr int kColumns = 256;  // plan columns (FRAMEFB_THREADS)

// ---------------------------------------------------------------------------
// token-pair arithmetic
// ---------------------------------------------------------------------------
using f2 = uint64_t;
struct C2 {
  f2 re, im;
};

__device__ __forceinline__ f2 pk(float a, float b) {
  f2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void unpk(f2 x, float& a, float& b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(x)); }
__device__ __forceinline__ f2 add2(f2 a, f2 b) {
  f2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f2 sub2(f2 a, f2 b) {
  f2 r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f2 mul2(f2 a, f2 b) {
  f2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) {
  f2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ C2 cadd(C2 a, C2 b) { return C2{add2(a.re, b.re), add2(a.im, b.im)}; }
__device__ __forceinline__ C2 csub(C2 a, C2 b) { return C2{sub2(a.re, b.re), sub2(a.im, b.im)}; }
// x * w, w = (c c, s s)
__device__ __forceinline__ C2 cmul(C2 x, C2 w) {
  return C2{sub2(mul2(x.re, w.re), mul2(x.im, w.im)), fma2(x.im, w.re, mul2(x.re, w.im))};
}
// a + i S b, S = +1 or -1
template <int S>
__device__ __forceinline__ C2 addi(C2 a, C2 b) {
  return S > 0 ? C2{sub2(a.re, b.im), add2(a.im, b.re)} : C2{add2(a.re, b.im), sub2(a.im, b.re)};
}

template <int S>
__device__ __forceinline__ void dft4(C2& a, C2& b, C2& c, C2& d) {
  const C2 t0 = cadd(a, c), t1 = csub(a, c), t2 = cadd(b, d), t3 = csub(b, d);
  a = cadd(t0, t2);
  c = csub(t0, t2);
  b = addi<S>(t1, t3);
  d = addi<-S>(t1, t3);
}
// x * e^{S 2 pi i q / 8}, q = 1 or 3
template <int S, int Q>
__device__ __forceinline__ C2 rot8(C2 x) {
  const f2 h = pk(0.70710678118654752f, 0.70710678118654752f), nh = pk(-0.70710678118654752f, -0.70710678118654752f);
  if (Q == 1)  // (1 + i S) / sqrt 2
    return S > 0 ? C2{mul2(sub2(x.re, x.im), h), mul2(add2(x.re, x.im), h)}
                 : C2{mul2(add2(x.re, x.im), h), mul2(sub2(x.im, x.re), h)};
  return S > 0 ? C2{mul2(add2(x.re, x.im), nh), mul2(sub2(x.re, x.im), h)}  // (-1 + i S) / sqrt 2
               : C2{mul2(sub2(x.im, x.re), h), mul2(add2(x.re, x.im), nh)};
}

__device__ __forceinline__ C2 lds_c(const float4* p) {
  const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(p);
  return C2{v.x, v.y};
}
__device__ __forceinline__ void sts_c(float4* p, C2 x) { *reinterpret_cast<ulonglong2*>(p) = make_ulonglong2(x.re, x.im); }

// This thread's share of a plan column: KE entries of each path.
// zw: V slot | RZ store target << 16; gw: U slot | RG store target << 16, as
// byte offsets into the buffers (so a buffer holds at most 8191 float2).
// zcarry / gcarry: where the run that the column's first half leaves open is
// stored by the second half (FFB_NO_STORE: none).  The coefficient values of
// both paths and the V slots of the column path are registers for KE = 4; for
// KE = 8 they sit in shared memory (three arrays of one float4 per four
// entries and thread): with all six arrays in registers the transforms'
// registers spilled to local memory, and those loads bounded the kernel.
constexpr int kMaxSlots = 8191;
template <int KE>
struct Share {
  static constexpr bool kSm = KE > 4;
  uint32_t zw[KE], gw[KE];
  uint32_t gb[kSm ? 1 : KE];
  float zc[kSm ? 1 : KE], gc[kSm ? 1 : KE];
  uint32_t zcarry, gcarry;
  int hZ, hG;
};
__host__ __device__ constexpr int plan_bytes(int NT, int KE) { return KE > 4 ? 3 * KE * NT * 4 : 0; }

// entries i0 .. i0 + 3 of array a (0 zc, 1 gc, 2 gb) of this thread
template <int KE, int NT>
__device__ __forceinline__ void get_plan(const uint8_t* sp, int a, int i0, uint32_t (&v)[4]) {
  const uint4 x = reinterpret_cast<const uint4*>(sp)[(a * (KE / 4) + i0 / 4) * NT + threadIdx.x];
  v[0] = x.x;
  v[1] = x.y;
  v[2] = x.z;
  v[3] = x.w;
}

// Entries per thread of a column of E entries with H threads per column.  With
// two, the first takes whole blocks of four: the loops walk blocks, and an entry
// past its share, inside the block, would add 0 x (the gathered value) to the run
// that it passes on to the second half, which is not 0 for an infinity or a NaN.
// (Entries past the end of a column follow its last store and reach nothing.)
template <int H>
__device__ __forceinline__ int half_of(int E) {
  return H == 2 ? ((E + 1) / 2 + 3) & ~3 : E;
}

// slot(side, x): index of frame column x of a side (0 input, 1 output) in its
// buffers (float2); overflow slots (x >= the side's columns) stay as they are.
template <int KE, int H, int NT, typename Slot>
__device__ __forceinline__ void load_share(Share<KE>& ch, uint8_t* sp, int mode, const uint8_t* plan, const float* c_val,
                                           int col, int half, Slot slot) {
  const bool F = mode & kF, D = mode & kD, C = mode & kC;
  const FfbPlanHeader& h = *reinterpret_cast<const FfbPlanHeader*>(plan);
  auto tab = [&](int32_t off) { return reinterpret_cast<const int32_t*>(plan + off); };
  ch.hZ = F ? half_of<H>(h.EZ) : 0;
  ch.hG = D || C ? half_of<H>(h.EG) : 0;
  const int K[2] = {h.n, h.m};
  // gather index of side sd | store target of side ts << 16
  auto word = [&](uint32_t w, int sd, int ts) {
    const uint32_t t = w >> 16;
    return 8u * slot(sd, w & 0x7FFFu) |
           ((t == FFB_NO_STORE ? t : 8u * (static_cast<int>(t) < K[ts] ? slot(ts, t) : t)) << 16);
  };
  bool openZ = false, openG = false;  // the last entry of the share continues
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
      zw = word(static_cast<uint32_t>(ld_g(tab(h.off_zb) + ez * kColumns + col)), 0, 1);
      const int32_t qi = ld_g(tab(h.off_zq) + ez * kColumns + col);
      zc = qi >= 0 ? ld_g(c_val + qi) : 0.f;
      const uint32_t tg = zw >> 16;
      openZ = qi >= 0 && tg == FFB_NO_STORE;
      if (firstZ == FFB_NO_STORE) firstZ = tg;
    }
    if (i < ch.hG && eg < h.EG) {
      gw = word(static_cast<uint32_t>(ld_g(tab(h.off_ga) + eg * kColumns + col)), 1, 0);
      gb = 8u * slot(0, static_cast<uint32_t>(ld_g(tab(h.off_gb) + eg * kColumns + col)));
      const int32_t qi = ld_g(tab(h.off_gq) + eg * kColumns + col);
      gc = (D && qi >= 0) ? ld_g(c_val + qi) : 0.f;
      const uint32_t tg = gw >> 16;
      openG = qi >= 0 && tg == FFB_NO_STORE;
      if (!D) gw |= FFB_NO_STORE << 16;
      if (firstG == FFB_NO_STORE) firstG = tg;
    }
    ch.zw[i] = zw;
    ch.gw[i] = gw;
    if constexpr (Share<KE>::kSm) {
      put(0, i, __float_as_uint(zc));
      put(1, i, __float_as_uint(gc));
      put(2, i, gb);
    } else {
      ch.zc[i] = zc;
      ch.gc[i] = gc;
      ch.gb[i] = gb;
    }
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

// float2 at a byte offset
__device__ __forceinline__ float2& at(float2* base, uint32_t bytes) {
  return *reinterpret_cast<float2*>(reinterpret_cast<uint8_t*>(base) + bytes);
}
__device__ __forceinline__ const float2& at(const float2* base, uint32_t bytes) {
  return *reinterpret_cast<const float2*>(reinterpret_cast<const uint8_t*>(base) + bytes);
}

// The coefficient SpMM of one token pair over this thread's share: run sums of
// c V[b] -> RZ (F), of c U[a] -> RG (D), dC += U[a] V[b] (C).  sp: the share's
// arrays in shared memory (KE = 8).
template <int KE, int H, int NT>
__device__ __forceinline__ void spmm(const Share<KE>& ch, float (&dc)[KE], const uint8_t* sp, bool F, bool D, bool C,
                                     const float2* V, const float2* U, float2* RG, float2* RZ) {
  if (D || C) {
    float2 acc = make_float2(0.f, 0.f);
#pragma unroll
    for (int i0 = 0; i0 < KE; i0 += 4) {  // four entries' gathers in flight
      if (i0 >= ch.hG) continue;
      float2 ub[4], vb[4];
      uint32_t gb[4], gc[4];
      if constexpr (Share<KE>::kSm) {
        get_plan<KE, NT>(sp, 2, i0, gb);
        get_plan<KE, NT>(sp, 1, i0, gc);
      } else {
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          gb[e] = ch.gb[e];
          gc[e] = __float_as_uint(ch.gc[e]);
        }
      }
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        ub[e] = at(U, ch.gw[i0 + e] & 0xFFFFu);
        vb[e] = C ? at(V, gb[e]) : make_float2(0.f, 0.f);
      }
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        dc[i0 + e] = fmaf(ub[e].x, vb[e].x, fmaf(ub[e].y, vb[e].y, dc[i0 + e]));
        const float c = __uint_as_float(gc[e]);
        acc.x = fmaf(c, ub[e].x, acc.x);
        acc.y = fmaf(c, ub[e].y, acc.y);
        const uint32_t tg = ch.gw[i0 + e] >> 16;
        if (tg != FFB_NO_STORE) {
          at(RG, tg) = acc;
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
      float2 vz[4];
      uint32_t zc[4];
      if constexpr (Share<KE>::kSm) {
        get_plan<KE, NT>(sp, 0, i0, zc);
      } else {
#pragma unroll
        for (int e = 0; e < 4; ++e) zc[e] = __float_as_uint(ch.zc[e]);
      }
#pragma unroll
      for (int e = 0; e < 4; ++e) vz[e] = at(V, ch.zw[i0 + e] & 0xFFFFu);
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const float c = __uint_as_float(zc[e]);
        acc.x = fmaf(c, vz[e].x, acc.x);
        acc.y = fmaf(c, vz[e].y, acc.y);
        const uint32_t tg = ch.zw[i0 + e] >> 16;
        if (tg != FFB_NO_STORE) {
          at(RZ, tg) = acc;
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

// Rows (columns) split between plan columns: add the overflow pieces.  RG, RZ:
// the buffers of pair 0, `pair` float2 between pairs; slot(side, t): index of
// store target t, overflow slots included.
template <int NT, typename Slot>
__device__ __forceinline__ void fix_runs(const uint8_t* plan, int nfZ, int nfix, int npair, float2* RG, float2* RZ, int pair,
                                         Slot slot) {
  const FfbPlanHeader& h = *reinterpret_cast<const FfbPlanHeader*>(plan);
  const int4* fz = reinterpret_cast<const int4*>(plan + h.off_fixZ);
  const int4* fg = reinterpret_cast<const int4*>(plan + h.off_fixG);
  for (int w = threadIdx.x; w < nfix * npair; w += NT) {
    const int p = w / nfix, i = w - p * nfix;
    const bool z = i < nfZ;
    const int4 it = z ? ld_g(fz + i) : ld_g(fg + (i - nfZ));
    float2* R = (z ? RZ : RG) + p * pair;
    const uint32_t dst = slot(z ? 1 : 0, static_cast<uint32_t>(it.x));
    float2 a = R[dst];
    for (int c = 0; c < it.z; ++c) {
      const float2 o = R[slot(z ? 1 : 0, static_cast<uint32_t>(it.y + c))];
      a.x += o.x;
      a.y += o.y;
    }
    R[dst] = a;
  }
}

// dC partial sums of this thread's entries to the CTA's slot of a matrix.
template <int KE>
__device__ __forceinline__ void flush_dc(const uint8_t* plan, float* dst, const float (&dc)[KE], int hG, int col, int half) {
  const FfbPlanHeader& h = *reinterpret_cast<const FfbPlanHeader*>(plan);
  const int32_t* gq = reinterpret_cast<const int32_t*>(plan + h.off_gq);
#pragma unroll
  for (int i = 0; i < KE; ++i) {
    const int e = half * hG + i;
    if (i < hG && e < h.EG) {
      const int32_t qi = ld_g(gq + e * kColumns + col);
      if (qi >= 0) dst[qi] = dc[i];
    }
  }
}

// dC_q = seff * sum over the CTAs that visited the matrix, in a fixed order:
// kLanes interleaved sums, then a tree over them.
constexpr int kReduceMats = 160;
struct ReduceMat {
  float* dC;
  int32_t c0, c1, nnz;  // CTAs [c0, c1] visited the matrix
  float seff;
};
struct Reduce {
  const float* partial;
  int32_t stride, pad;
  ReduceMat m[kReduceMats];
};
constexpr int kLanes = 8;

static __global__ void __launch_bounds__(256) pair_reduce_kernel(const __grid_constant__ Reduce r) {
  chain_wait();
  chain_next();
  const int j = blockIdx.y;
  const ReduceMat& M = r.m[j];
  // lane l of a group of 8 warps' lanes: entry q = 32 x block + lane, part = warp
  __shared__ float s[kLanes][32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int q = blockIdx.x * 32 + lane;
  float a = 0.f;
  if (q < M.nnz)
    for (int c = M.c0 + w; c <= M.c1; c += kLanes) a += r.partial[static_cast<size_t>(c + j) * r.stride + q];
  s[w][lane] = a;
  __syncthreads();
  if (w == 0 && q < M.nnz) {
    const float x = ((s[0][lane] + s[1][lane]) + (s[2][lane] + s[3][lane])) +
                    ((s[4][lane] + s[5][lane]) + (s[6][lane] + s[7][lane]));
    M.dC[q] = M.seff * x;
  }
}

}  // namespace pair
}  // namespace ffb
