// Row-transform kernel of libframefb: the whole adapter pass (Sec. 3.1
// update, Lemma 1 gradient of Appendix A) for frames with rho = 2, k*rho = d
// (the paper's own regime): Phi is one realified DFT of size k = d / 2, so the
// transforms run as fast Fourier transforms in fp32 on chip instead of dense
// contractions.  Included by framefb_row.cu only.
//
// A row of d features is k complex values; its frame coefficients are their
// inverse DFT (Sec. 3.2 construction), the synthesis the forward DFT.  A unit
// is a few token pairs of one matrix; a CTA takes a contiguous range of units
// and runs, per unit, with a CTA barrier between passes:
//   analysis    V = X Phi_in, U = dY Phi_out: Stockham passes of radix 2..8
//               over both sides at once; the rows were landed in shared memory
//               one unit ahead by bulk copies;
//   SpMM        run sums of c V[b] -> RZ, of c U[a] -> RG; dC += U[a] V[b];
//               plan columns in registers, H threads per column;
//   synthesis   Stockham passes over RZ / RG, the last one adds into the rows
//               of Y / dX (prefetched to L2 before the SpMM).
// (Token pairs: framefb_pair.cuh.)
//
// Bound: shared memory.  At d = 4096 a token pair moves about 15 k wavefronts
// (four transforms of four passes and the SpMM's gathers; 3 k of them bank
// conflicts), against 10 k issue cycles and 80 KB of DRAM traffic; the pair takes
// 23 k cycles, one CTA of 512 threads per SM.  Measured (fused pass): 4 matrices of 4096^2, 8192 tokens
// 1.21 ms against 6.90 ms as dense contractions; 24 of 768^2, 4096 tokens
// 0.57 ms against 2.99 ms.  dC against the fp64 oracle: 3e-7 relative (1.7e-5
// before: bf16 hi + lo frames).
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "framefb_pair.cuh"

namespace ffb {
namespace row {

using namespace pair;

// Bounded waits of the row kernel that gave up (see framefb_wait_timeouts).
__device__ unsigned int g_row_timeouts;

constexpr int kMaxShapes = 8;   // distinct geometries of a launch
constexpr int kMaxMats = 96;    // matrices of a launch

// Passes of a DFT_K: radix of pass q, product of the earlier radices (a power
// of two: an odd factor comes last), passes.
template <int K>
struct Plan;
template <>
struct Plan<128> {
  static constexpr int np = 3, r[4] = {8, 4, 4, 1};
};
template <>
struct Plan<256> {
  static constexpr int np = 3, r[4] = {8, 8, 4, 1};
};
template <>
struct Plan<384> {
  static constexpr int np = 3, r[4] = {8, 8, 6, 1};
};
template <>
struct Plan<512> {
  static constexpr int np = 3, r[4] = {8, 8, 8, 1};
};
template <>
struct Plan<1024> {
  static constexpr int np = 4, r[4] = {8, 8, 4, 4};
};
template <>
struct Plan<1536> {
  static constexpr int np = 4, r[4] = {8, 8, 8, 3};
};
template <>
struct Plan<2048> {
  static constexpr int np = 4, r[4] = {8, 8, 8, 4};
};
template <int K>
constexpr int ns_of(int q) {
  int n = 1;
  for (int i = 0; i < q; ++i) n *= Plan<K>::r[i];
  return n;
}
// The first pass writes element (j, r) to r (K / 8 + 1) + j: its stores and
// the next pass's loads are then free of bank conflicts.
__host__ __device__ constexpr int scratch_of(int k) { return k + 8; }  // float4 of a buffer
inline __host__ __device__ int passes_of(int k) {  // 0: a size the kernel does not take
  return k == 128 || k == 256 || k == 384 || k == 512 ? 3 : k == 1024 || k == 1536 || k == 2048 ? 4 : 0;
}

// Twiddle table e^{2 pi i t / k}: the entries the passes read (k over the
// smallest radix after the first).
inline __host__ __device__ int twiddles_of(int k) {
  return k == 384 || k == 512 ? 64 : k == 1536 || k == 2048 ? 512 : k / 4;
}

// Geometry of a matrix.  Buffers of a token pair (float2 offsets from the
// pair's base), side 0 the input side (X, V, RG, dX), side 1 the output side
// (dY, U, RZ, Y): A[s] holds the analysis result (V or U), B[s] the run sums
// (RG or RZ); both serve as the passes' scratch.
struct Shape {
  int32_t k[2];   // DFT sizes (d = 2 k)
  int32_t A[2], B[2];
  int32_t pair;   // float2 per token pair
  int32_t PP;     // token pairs per unit
  int32_t tw[2];  // twiddle tables (float2 offsets)
};

struct Mat {
  const void* in[2];  // X, dY
  void* out[2];       // dX, Y
  int64_t ld[2];      // elements
  const uint8_t* plan;
  const float* c_val;
  int32_t N, ubeg, ntiles, shape;
  float seff;         // s / sqrt(k_in k_out)
  int32_t pad;
};

struct Launch {
  int32_t nmats, total_units, stride, mode;
  int32_t stage1;            // byte offset of the dY rows in the stage
  int32_t oPairs, oTw, oPlan, oBar; // shared memory (bytes): pair buffers, twiddles, plan columns, mbarrier
  float* partial;            // [(grid + nmats) * stride] dC partial sums, slot = cta + matrix
  Shape sh[kMaxShapes];
  Mat m[kMaxMats];
};

// DFT of R values in place, natural order: X_q = sum_r x_r e^{S 2 pi i q r / R}
template <int R, int S>
struct Dft;

template <int S>
struct Dft<4, S> {
  static __device__ __forceinline__ void run(C2 (&x)[4]) { dft4<S>(x[0], x[1], x[2], x[3]); }
};

template <int S>
struct Dft<8, S> {
  static __device__ __forceinline__ void run(C2 (&x)[8]) {
    // 2 x 4: even and odd inputs
    dft4<S>(x[0], x[2], x[4], x[6]);
    dft4<S>(x[1], x[3], x[5], x[7]);
    const C2 e0 = x[0], e1 = x[2], e2 = x[4], e3 = x[6];
    const C2 o0 = x[1], o1 = rot8<S, 1>(x[3]), o2 = x[5], o3 = rot8<S, 3>(x[7]);
    x[0] = cadd(e0, o0);
    x[4] = csub(e0, o0);
    x[1] = cadd(e1, o1);
    x[5] = csub(e1, o1);
    x[2] = addi<S>(e2, o2);
    x[6] = addi<-S>(e2, o2);
    x[3] = cadd(e3, o3);
    x[7] = csub(e3, o3);
  }
};

// odd sizes: symmetric and antisymmetric halves of the inputs
template <int R>
struct OddTab;
template <>
struct OddTab<3> {
  static __host__ __device__ constexpr float c(int) { return -0.5f; }
  static __host__ __device__ constexpr float s(int) { return 0.86602540378443865f; }
};
template <int R, int S>
__device__ __forceinline__ void dft_odd(C2 (&x)[R]) {
  constexpr int H = R / 2;
  C2 t[H], u[H];
#pragma unroll
  for (int i = 0; i < H; ++i) {
    t[i] = cadd(x[i + 1], x[R - 1 - i]);
    u[i] = csub(x[i + 1], x[R - 1 - i]);
  }
  const C2 x0 = x[0];
#pragma unroll
  for (int i = 0; i < H; ++i) x[0] = cadd(x[0], t[i]);
#pragma unroll
  for (int q = 1; q <= H; ++q) {
    C2 a = x0, b{0ull, 0ull};
#pragma unroll
    for (int i = 1; i <= H; ++i) {
      int e = (q * i) % R;
      const bool neg = e > H;
      if (neg) e = R - e;
      const float c = OddTab<R>::c(e), s = neg ? -OddTab<R>::s(e) : OddTab<R>::s(e);
      const f2 cc = pk(c, c), ss = pk(s, s);
      a = C2{fma2(t[i - 1].re, cc, a.re), fma2(t[i - 1].im, cc, a.im)};
      b = C2{fma2(u[i - 1].re, ss, b.re), fma2(u[i - 1].im, ss, b.im)};
    }
    x[q] = addi<S>(a, b);
    x[R - q] = addi<-S>(a, b);
  }
}
template <int S>
struct Dft<3, S> {
  static __device__ __forceinline__ void run(C2 (&x)[3]) { dft_odd<3, S>(x); }
};
// 6 = 2 x 3 with coprime index maps (no twiddles): input r = 3 r1 + 2 r2 mod 6,
// output q with q mod 2 = q1, q mod 3 = q2
template <int S>
struct Dft<6, S> {
  static __device__ __forceinline__ void run(C2 (&x)[6]) {
    C2 a[3] = {cadd(x[0], x[3]), cadd(x[2], x[5]), cadd(x[4], x[1])};
    C2 b[3] = {csub(x[0], x[3]), csub(x[2], x[5]), csub(x[4], x[1])};
    dft_odd<3, S>(a);
    dft_odd<3, S>(b);
    x[0] = a[0];
    x[4] = a[1];
    x[2] = a[2];
    x[3] = b[0];
    x[1] = b[1];
    x[5] = b[2];
  }
};

// x[r] *= w^r: the powers by complex products, at most three deep
template <int R>
__device__ __forceinline__ void twiddle(C2 (&x)[R], float c, float s) {
  C2 p[R];
  p[1] = C2{pk(c, c), pk(s, s)};
#pragma unroll
  for (int r = 2; r < R; ++r) p[r] = cmul(p[r / 2], p[r - r / 2]);
#pragma unroll
  for (int r = 1; r < R; ++r) x[r] = cmul(x[r], p[r]);
}

// ---------------------------------------------------------------------------
// rows of activations: complex coordinate e of a row
// ---------------------------------------------------------------------------
using W = uint32_t;  // two bf16
__device__ __forceinline__ float w_re(W w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float w_im(W w) { return __uint_as_float(w & 0xFFFF0000u); }
__device__ __forceinline__ W w_axpy(W y, float s, float a, float b) {
  return pack_bf16(fmaf(s, a, w_re(y)), fmaf(s, b, w_im(y)));
}

// The current matrix, in shared memory.
struct Cur {
  int32_t A[2], B[2];
  int32_t tw[2];
  int32_t pair;
  float seff;
  W* out[2];       // dX, Y
  int64_t ldw[2];  // words per row
};

// Pass Q of the DFT_K of the sides in `sides` (bit 0 input side, bit 1 output
// side, 3 both) over the unit's np token pairs.  ANA: inverse DFT of the
// staged rows into A; else forward DFT of B, added into the output rows.
template <int K, int Q, bool ANA, int NT>
__device__ __forceinline__ void pass(const Cur& cur, int oPairs, int stage1, int oTw, int sides, int npair, int64_t t0,
                                     int ntok) {
  extern __shared__ __align__(128) uint8_t smem[];
  using P = Plan<K>;
  constexpr int R = P::r[Q], np = P::np, nb = K / R, Ns = ns_of<K>(Q), S = ANA ? 1 : -1;
  constexpr bool EDGE = ANA ? Q == 0 : Q == np - 1;
  constexpr int rs = K / 8 + 1;  // first-pass output stride
  // both sides: one half of the CTA each where it has a whole DFT's
  // butterflies to do, else interleaved
  constexpr bool kHalves = NT == 512 && K >= 1024;
  const bool halves = kHalves && sides == 3;
  const int cnt = (sides == 3 && !halves ? 2 : 1) * npair * nb;
  // opaque: the index arithmetic of the many passes must not be hoisted out of
  // the unit loop, where it would only be spilled
  int t = threadIdx.x;
  asm volatile("" : "+r"(t));
  const int half = t / (NT / 2);
  if (halves) t -= half * (NT / 2);
  for (; t < cnt; t += halves ? NT / 2 : NT) {
    // (pair, side, butterfly)
    const int ps = t / nb, j = t - ps * nb;
    const int sd = halves ? half : sides == 3 ? ps & 1 : sides >> 1;
    const int p = sides == 3 && !halves ? ps >> 1 : ps;
    const int jl = j & (Ns - 1);
    const int base = oPairs + 8 * p * cur.pair;
    const int A = base + 8 * cur.A[sd], B = base + 8 * cur.B[sd];  // bytes
    const bool two = 2 * p + 1 < ntok;
    C2 x[R];
    W y0[EDGE ? R : 1], y1[EDGE ? R : 1];
    W *o0 = nullptr, *o1 = nullptr;
    if constexpr (!ANA && EDGE) {
      // the rows this butterfly adds into: loaded before the work
      const int64_t ld = cur.ldw[sd];
      o0 = cur.out[sd] + (t0 + 2 * p) * ld + jl;
      o1 = o0 + ld;
#pragma unroll
      for (int r = 0; r < R; ++r) y0[r] = o0[r * Ns];
      if (two) {
#pragma unroll
        for (int r = 0; r < R; ++r) y1[r] = o1[r * Ns];
      }
    }
    if constexpr (ANA && EDGE) {
      const W* r0 = reinterpret_cast<const W*>(smem + (sd ? stage1 : 0)) + 2 * p * K + j;  // row 2 p, K words each
      const W* r1 = r0 + K;
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const W a = r0[r * nb];
        const W c = two ? r1[r * nb] : 0u;
        x[r] = C2{pk(w_re(a), w_re(c)), pk(w_im(a), w_im(c))};
      }
    } else {
      // analysis pass q reads what pass q - 1 wrote, ending in A; synthesis
      // starts in B and alternates
      constexpr int step = Q == 1 ? nb / 8 : nb;
      float4* src = reinterpret_cast<float4*>(smem + ((ANA ? ((np - Q) & 1) == 0 : (Q & 1) != 0) ? A : B)) +
                    (Q == 1 ? (j & 7) * rs + (j >> 3) : j);
#pragma unroll
      for (int r = 0; r < R; ++r) x[r] = lds_c(src + r * step);
      // run-sum slots that no run writes read as zero in every unit: the last
      // analysis pass clears B behind itself
      if constexpr (ANA && Q == np - 1) {
#pragma unroll
        for (int r = 0; r < R; ++r) src[r * step] = make_float4(0.f, 0.f, 0.f, 0.f);
      }
    }
    if constexpr (Q > 0) {
      const float2 w = reinterpret_cast<const float2*>(smem + oTw)[cur.tw[sd] + jl * (K / (Ns * R))];
      twiddle<R>(x, w.x, S > 0 ? w.y : -w.y);
    }
    Dft<R, S>::run(x);
    if constexpr (!ANA && EDGE) {
      const float sc = cur.seff;
#pragma unroll
      for (int r = 0; r < R; ++r) {
        float a0, a1, b0, b1;
        unpk(x[r].re, a0, a1);
        unpk(x[r].im, b0, b1);
        o0[r * Ns] = w_axpy(y0[r], sc, a0, b0);
        if (two) o1[r * Ns] = w_axpy(y1[r], sc, a1, b1);
      }
    } else {
      constexpr int step = Q == 0 ? rs : Ns;
      float4* dst = reinterpret_cast<float4*>(smem + ((ANA ? ((np - 1 - Q) & 1) == 0 : (Q & 1) == 0) ? A : B)) +
                    (Q == 0 ? j : (j - jl) * R + jl);
#pragma unroll
      for (int r = 0; r < R; ++r) sts_c(dst + r * step, x[r]);
    }
  }
}

template <int K, bool ANA, int NT>
__device__ __forceinline__ void pass_q(int q, const Cur& cur, int oPairs, int stage1, int oTw, int sides, int npair,
                                       int64_t t0, int ntok) {
  if (q == 0)
    pass<K, 0, ANA, NT>(cur, oPairs, stage1, oTw, sides, npair, t0, ntok);
  else if (q == 1)
    pass<K, 1, ANA, NT>(cur, oPairs, stage1, oTw, sides, npair, t0, ntok);
  else if (q == 2)
    pass<K, 2, ANA, NT>(cur, oPairs, stage1, oTw, sides, npair, t0, ntok);
  else if constexpr (Plan<K>::np == 4)
    pass<K, 3, ANA, NT>(cur, oPairs, stage1, oTw, sides, npair, t0, ntok);
}

// Pass q of the transforms of size k over `sides`.
template <int K, bool ANA, int NT>
__device__ __forceinline__ void pass_k(int k, int q, const Cur& cur, int oPairs, int stage1, int oTw, int sides, int npair,
                                       int64_t t0, int ntok) {
  if constexpr (K > 0) {
    pass_q<K, ANA, NT>(q, cur, oPairs, stage1, oTw, sides, npair, t0, ntok);
    return;
  }
  switch (k) {
    case 128: pass_q<128, ANA, NT>(q, cur, oPairs, stage1, oTw, sides, npair, t0, ntok); break;
    case 256: pass_q<256, ANA, NT>(q, cur, oPairs, stage1, oTw, sides, npair, t0, ntok); break;
    case 384: pass_q<384, ANA, NT>(q, cur, oPairs, stage1, oTw, sides, npair, t0, ntok); break;
    case 512: pass_q<512, ANA, NT>(q, cur, oPairs, stage1, oTw, sides, npair, t0, ntok); break;
    case 1024: pass_q<1024, ANA, NT>(q, cur, oPairs, stage1, oTw, sides, npair, t0, ntok); break;
    case 1536: pass_q<1536, ANA, NT>(q, cur, oPairs, stage1, oTw, sides, npair, t0, ntok); break;
    default: pass_q<2048, ANA, NT>(q, cur, oPairs, stage1, oTw, sides, npair, t0, ntok); break;
  }
}

// ---------------------------------------------------------------------------
// NT threads: H = NT / 256 threads per plan column (the two halves of a
// column sit 16 lanes apart, so that the half-warps of a gather are the same
// 16 plan columns as with one thread per column).
// ---------------------------------------------------------------------------
// K: the DFT size of both sides of every matrix of the launch, or 0 for any.
template <int NT, int KE, int K>
__global__ void __launch_bounds__(NT, NT == 512 ? 1 : 2) row_kernel(const __grid_constant__ Launch args) {
  chain_wait();
  chain_next();
  constexpr int H = NT / kColumns;
  extern __shared__ __align__(128) uint8_t smem[];
  __shared__ Cur cur_s;
  const int mode = args.mode;
  const bool F = mode & kF, D = mode & kD, C = mode & kC;
  const int kAna = (F || C ? 1 : 0) | (D || C ? 2 : 0), kSyn = (D ? 1 : 0) | (F ? 2 : 0);
  const int tid = threadIdx.x, lane = tid & 31;
  const int half = H == 2 ? lane >> 4 : 0;
  const int col = H == 2 ? (tid >> 5) * 16 + (lane & 15) : tid;
  uint64_t* bar = reinterpret_cast<uint64_t*>(smem + args.oBar);
  float2* tw = reinterpret_cast<float2*>(smem + args.oTw);
  float2* pairs = reinterpret_cast<float2*>(smem + args.oPairs);

  const int64_t units = args.total_units;
  const int64_t u_begin = (static_cast<int64_t>(blockIdx.x) * units) / gridDim.x;
  const int64_t u_end = (static_cast<int64_t>(blockIdx.x + 1) * units) / gridDim.x;
  if (u_begin >= u_end) return;

  if (tid == 0) {
    mbar_init(bar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();

  auto slot = [](int, uint32_t x) { return x; };  // buffers in the order of the frame columns
  auto next_mat = [&](int j, int64_t u) {
    while (u >= args.m[j].ubeg + args.m[j].ntiles) ++j;
    return j;
  };
  // rows of unit u (matrix j) into the stage: one bulk copy per row
  auto issue = [&](int j, int64_t u) {
    const Mat& M = args.m[j];
    const Shape& sh = args.sh[M.shape];
    const int64_t t0 = 2 * static_cast<int64_t>(sh.PP) * (u - M.ubeg);
    const int ntok = static_cast<int>(min(static_cast<int64_t>(2 * sh.PP), M.N - t0));
    uint32_t bytes[2];
    for (int sd = 0; sd < 2; ++sd) bytes[sd] = (kAna >> sd) & 1 ? 4u * sh.k[sd] : 0u;
    mbar_arrive_expect_tx(bar, ntok * (bytes[0] + bytes[1]));
    for (int sd = 0; sd < 2; ++sd) {
      if (!bytes[sd]) continue;
      for (int i = 0; i < ntok; ++i)
        asm volatile(
            "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                smem_u32(smem + (sd ? args.stage1 : 0) + i * bytes[sd])),
            "l"(static_cast<const uint16_t*>(M.in[sd]) + (t0 + i) * M.ld[sd]), "r"(bytes[sd]), "r"(smem_u32(bar))
            : "memory");
    }
  };
  int j = next_mat(0, u_begin);
  if (tid == 0) issue(j, u_begin);

  Share<KE> ch{};
  float dc[KE];
  int cur = -1, cur_shape = -1, nfZ = 0, nfix = 0;
  int k0 = 0, k1 = 0, PP = 1;
  const uint8_t* plan = nullptr;
  uint32_t phase = 0;
  bool failed = false;

  auto flush = [&](int mat) {  // dC partial sums of this thread's entries to the CTA's slot of the matrix
    if (C) flush_dc(plan, args.partial + static_cast<size_t>(blockIdx.x + mat) * args.stride, dc, ch.hG, col, half);
  };

  // Barrier between passes.  With a side per half of the CTA the sides share
  // nothing until the SpMM, so each half waits for itself only: one half's
  // shared-memory traffic then runs beside the other's arithmetic.
  constexpr bool kHalves = NT == 512 && K >= 1024;
  auto pass_bar = [&](int sides) {
    if (kHalves && sides == 3)
      asm volatile("bar.sync %0, %1;" ::"r"(1 + tid / (NT / 2)), "n"(NT / 2) : "memory");
    else
      __syncthreads();
  };

  for (int64_t u = u_begin; u < u_end; ++u) {
    j = next_mat(j, u);
    if (j != cur) {
      __syncthreads();  // every thread is past the previous unit
      if (cur >= 0) flush(cur);
      cur = j;
      const Mat& M = args.m[j];
      const Shape& sh = args.sh[M.shape];
      plan = M.plan;
      const FfbPlanHeader& h = *reinterpret_cast<const FfbPlanHeader*>(plan);
      nfZ = F ? h.nfixZ : 0;
      nfix = nfZ + (D ? h.nfixG : 0);
      load_share<KE, H, NT>(ch, smem + args.oPlan, mode, plan, M.c_val, col, half, slot);
#pragma unroll
      for (int i = 0; i < KE; ++i) dc[i] = 0.f;
      if (tid < 2) {
        cur_s.A[tid] = sh.A[tid];
        cur_s.B[tid] = sh.B[tid];
        cur_s.tw[tid] = sh.tw[tid];
        cur_s.out[tid] = static_cast<W*>(M.out[tid]);
        cur_s.ldw[tid] = M.ld[tid] >> 1;
        cur_s.pair = sh.pair;
        cur_s.seff = M.seff;
      }
      if (M.shape != cur_shape) {
        cur_shape = M.shape;
        k0 = K > 0 ? K : sh.k[0];
        k1 = K > 0 ? K : sh.k[1];
        PP = sh.PP;
        for (int sd = 0; sd < 2; ++sd) {
          if (sd == 1 && sh.tw[1] == sh.tw[0]) continue;
          // omega^i = e^{2 pi i / k}: the angle's rounding error corrected to first order
          const float kf = static_cast<float>(sh.k[sd]);
          for (int i = tid; i < twiddles_of(sh.k[sd]); i += NT) {
            const float a = 2.f * static_cast<float>(i);
            const float f = a / kf, e = fmaf(-f, kf, a) / kf * 3.14159265358979f;
            float sn, cs;
            sincospif(f, &sn, &cs);
            tw[sh.tw[sd] + i] = make_float2(fmaf(-e, sn, cs), fmaf(e, cs, sn));
          }
        }
      }
      __syncthreads();
    }
    const int64_t t0 = 2 * static_cast<int64_t>(PP) * (u - args.m[j].ubeg);
    const int ntok = static_cast<int>(min(static_cast<int64_t>(2 * PP), args.m[j].N - t0));
    const int npair = (ntok + 1) >> 1;
    const int np0 = passes_of(k0), np1 = passes_of(k1), npm = max(np0, np1);

    // ---- analysis: transforms of different lengths end together
    failed = !(mbar_test_wait(bar, phase) || mbar_wait_bounded(bar, phase));
    phase ^= 1u;
    if (failed && tid == 0) atomicAdd(&g_row_timeouts, 1u);
    for (int t = 0; t < npm; ++t) {
      // one job for both sides where they have the same size, else one each
#pragma unroll 1
      for (int sd = 0; sd < (K > 0 || k0 == k1 ? 1 : 2); ++sd) {
        const int sides = K > 0 || k0 == k1 ? kAna : kAna & (1 << sd), q = t - (npm - (sd ? np1 : np0));
        if (sides && q >= 0) pass_k<K, true, NT>(sd ? k1 : k0, q, cur_s, args.oPairs, args.stage1, args.oTw, sides, npair, t0, ntok);
      }
      if (t == 0 && (kSyn & ~kAna)) {
        // a side with a synthesis but no analysis: its run sums start from zero
        const int sd = (kSyn & ~kAna) >> 1, d = 2 * (sd ? k1 : k0);
        for (int p = 0; p < npair; ++p)
          for (int x = tid; x < d; x += NT) pairs[p * cur_s.pair + cur_s.B[sd] + x] = make_float2(0.f, 0.f);
      }
      if (t + 1 < npm) pass_bar(kAna);
    }
    if (__syncthreads_or(failed)) {
      failed = true;
      break;
    }
    if (tid == 0 && u + 1 < u_end) issue(next_mat(j, u + 1), u + 1);  // the stage is free

    // ---- the output rows towards L2, one 128-byte line per thread and turn
    for (int sd = 0; sd < 2; ++sd) {
      if (!((kSyn >> sd) & 1)) continue;
      const int lines = (sd ? k1 : k0) >> 5;  // 128-byte lines of a row (4 k bytes)
      for (int x = tid; x < lines * ntok; x += NT) {
        const int r = x / lines;
        asm volatile("prefetch.global.L2 [%0];" ::"l"(cur_s.out[sd] + (t0 + r) * cur_s.ldw[sd] + 32 * (x - r * lines)));
      }
    }

    // ---- coefficient SpMM
    for (int p = 0; p < npair; ++p) {
      float2* base = pairs + p * cur_s.pair;
      spmm<KE, H, NT>(ch, dc, smem + args.oPlan, F, D, C, base + cur_s.A[0], base + cur_s.A[1], base + cur_s.B[0],
                      base + cur_s.B[1]);
    }
    __syncthreads();
    if (kSyn) {
      if (nfix > 0) {
        fix_runs<NT>(plan, nfZ, nfix, npair, pairs + cur_s.B[0], pairs + cur_s.B[1], cur_s.pair, slot);
        __syncthreads();
      }
      // ---- synthesis: both sides start together
      for (int t = 0; t < npm; ++t) {
#pragma unroll 1
        for (int sd = 0; sd < (K > 0 || k0 == k1 ? 1 : 2); ++sd) {
          const int sides = K > 0 || k0 == k1 ? kSyn : kSyn & (1 << sd);
          if (sides && t < (sd ? np1 : np0))
            pass_k<K, false, NT>(sd ? k1 : k0, t, cur_s, args.oPairs, args.stage1, args.oTw, sides, npair, t0, ntok);
        }
        pass_bar(kSyn);
      }
      if (kSyn != kAna) __syncthreads();  // (halves of the CTA go their own way only from one pass to the next)
    }
  }
  if (failed) {
    // the copies of this unit may still be in flight (no others are)
    if (tid == 0) mbar_wait_bounded(bar, phase ^ 1u);
    __syncthreads();
    return;
  }
  if (cur >= 0) flush(cur);
}

}  // namespace row
}  // namespace ffb
