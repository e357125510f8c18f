// Launchers of the group-transform path of libframefb (framefb_grp.cuh): which
// structured matrices it takes, validation, the shared-memory map, launches.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstddef>
#include <cstring>
#include <memory>
#include <new>
#include <string>
#include <vector>

#include "framefb.h"
#include "framefb_dense.h"
#include "framefb_grp.cuh"
#include "framefb_grp.h"
#include "framefb_launch.h"
#include "plan_internal.h"
#include "plan_layout.h"

namespace ffb_host {

namespace {

namespace fg = ffb::grp;
namespace fp = ffb::pair;

static_assert(sizeof(fg::Launch) <= 32764 && sizeof(fp::Reduce) <= 32764, "launch parameters exceed the parameter space");
static_assert(fg::kMaxMats <= fp::kReduceMats, "one reduction per launch");

inline size_t rup(size_t x, size_t a) { return (x + a - 1) / a * a; }
inline bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

const FfbPlanHeader* header_of(const framefb_plan* p) {
  if (!p || p->image.size() < sizeof(FfbPlanHeader)) return nullptr;
  const FfbPlanHeader* h = reinterpret_cast<const FfbPlanHeader*>(p->image.data());
  if (h->magic != FFB_PLAN_MAGIC || h->version != FFB_PLAN_VERSION || h->P != fp::kColumns) return nullptr;
  if (static_cast<size_t>(h->total_bytes) > p->image.size() || h->layout != FFB_LAYOUT_GROUPS) return nullptr;
  return h;
}

// A kernel variant: threads per CTA, plan entries per thread and path, big
// plans (compacted buffers).
struct Variant {
  int nt, ke;
  bool big;
  bool operator==(const Variant& o) const { return nt == o.nt && ke == o.ke && big == o.big; }
};

constexpr size_t kSmemSm = 228 * 1024;          // shared memory of an SM
constexpr size_t kSmemCta = 227 * 1024 - 256;   // of a CTA, less the static part
constexpr int kMaxPairs = 8;
// relative cost of a group's transform and of a support entry (per pair)
constexpr int kGroupCost = 16, kEntryCost = 1;

size_t budget(const Variant& v) { return v.nt == 512 ? kSmemCta : kSmemSm / 2 - 1024 - 256; }

// Columns of a side in the support (set bits of the plan's group masks).
int32_t named(const FfbPlanHeader* h, int sd) {
  const uint8_t* base = reinterpret_cast<const uint8_t*>(h);
  const uint32_t* m = reinterpret_cast<const uint32_t*>(base + (sd ? h->off_zmask : h->off_gmask));
  int32_t n = 0;
  for (int32_t g = 0; g < (sd ? h->Gm : h->Gn); ++g) n += __builtin_popcount(m[g]);
  return n;
}

// Buffers of a token pair of a matrix on a variant; false when slots exceed
// the variant's fields.
bool shape_of(const FfbPlanHeader* h, const Variant& v, fg::Shape& sh) {
  std::memset(&sh, 0, sizeof(sh));
  int32_t off = 0;
  for (int sd = 0; sd < 2; ++sd) {
    const int32_t d = sd ? h->m : h->n, ovf = sd ? h->ovfZ : h->ovfG;
    const int32_t slots = v.big ? named(h, sd) : d;
    if (v.big ? slots + ovf > (sd ? fg::kBigU : fg::kBigV) : slots + ovf > fp::kMaxSlots) return false;
    sh.G[sd] = d / FFB_GROUP;
    sh.A[sd] = off;
    off += static_cast<int32_t>(rup(std::max(slots, 1), 2));
    sh.B[sd] = off;
    off += static_cast<int32_t>(rup(std::max(slots + ovf, 1), 2));
  }
  sh.pair = off;
  return true;
}

// Shared memory of a launch: the largest of its shapes.
struct Regions {
  size_t pairs = 0, masks = 0;
  void take(const fg::Shape& sh, int pp, const Variant& v) {
    pairs = std::max(pairs, rup(static_cast<size_t>(pp) * sh.pair * 8, 16));
    masks = std::max(masks, rup(4 * static_cast<size_t>((v.big ? 2 : 1) * (sh.G[0] + sh.G[1]) + 2), 16));
  }
  size_t plan(const Variant& v) const { return v.big ? fg::big_bytes(v.nt) : fg::cols_bytes(v.nt, v.ke); }
  size_t bytes(const Variant& v) const { return pairs + masks + plan(v); }
};

// The kernel variant of a plan (nt = 0: none fits): two CTAs of 256 threads
// per SM where a unit fits half an SM and a column has at most 8 entries, else
// one CTA of 512 threads, with compacted buffers for columns of up to 32.
Variant variant(const FfbPlanHeader* h) {
  const int e = std::max(h->EZ, h->EG);
  for (const Variant& v : {Variant{256, 4, false}, Variant{256, 8, false}, Variant{512, 8, false}, Variant{512, fg::kBigE, true}}) {
    if (e > v.ke * (v.nt / fp::kColumns)) continue;
    fg::Shape sh;
    if (!shape_of(h, v, sh)) continue;
    Regions r;
    r.take(sh, 1, v);
    if (r.bytes(v) <= budget(v)) return v;
  }
  return Variant{0, 0, false};
}

void* kernel_ptr(const Variant& v, framefb_dtype dt) {
  const Variant big{512, fg::kBigE, true};
  if (dt == FRAMEFB_BF16)  // (plans with whole buffers run on the tcgen05 kernels)
    return v == big ? reinterpret_cast<void*>(fg::fft_tile_kernel<__nv_bfloat16, 512, fg::kBigE, true>) : nullptr;
  if (v == Variant{256, 4, false}) return reinterpret_cast<void*>(fg::fft_tile_kernel<float, 256, 4, false>);
  if (v == Variant{256, 8, false}) return reinterpret_cast<void*>(fg::fft_tile_kernel<float, 256, 8, false>);
  if (v == Variant{512, 8, false}) return reinterpret_cast<void*>(fg::fft_tile_kernel<float, 512, 8, false>);
  return v == big ? reinterpret_cast<void*>(fg::fft_tile_kernel<float, 512, fg::kBigE, true>) : nullptr;
}

struct Prepared {
  fg::Launch* args;
  fp::Reduce* red;
  int grid, nnz_max;
  Variant v;
  int64_t slots;  // CTAs that are resident
  size_t smem, ws_bytes;
};

// Matrices of a launch of big plans: the dC sums of 8192 entries each (a slot per CTA
// and matrix) then fit the library's static workspace.
constexpr int kMaxBig = 96;
static_assert((152 + kMaxBig) * 8192 * 4 + 256 <= FRAMEFB_STATIC_WS_BYTES, "static workspace");

// One launch: as many matrices as the parameters hold, of one variant.
struct Chunk {
  std::vector<const framefb_mat*> mats;
  Variant v;
};

std::vector<Chunk> chunks_of(const framefb_mat* mats, int32_t nmats) {
  std::vector<Variant> kinds;
  std::vector<Variant> of(nmats);
  for (int32_t j = 0; j < nmats; ++j) {
    // (matrices of one plan come in runs)
    of[j] = j > 0 && mats[j].plan == mats[j - 1].plan ? of[j - 1] : variant(header_of(mats[j].plan));
    if (of[j].nt && std::find(kinds.begin(), kinds.end(), of[j]) == kinds.end()) kinds.push_back(of[j]);
  }
  std::vector<Chunk> out;
  for (const Variant& v : kinds) {
    Regions all;  // of one pair of each matrix of the chunk
    bool open = false;
    const framefb_plan* plan = nullptr;
    fg::Shape sh;
    for (int32_t j = 0; j < nmats; ++j) {
      if (!(of[j] == v)) continue;
      if (mats[j].plan != plan) shape_of(header_of(plan = mats[j].plan), v, sh);
      Regions with = all;
      with.take(sh, 1, v);
      if (!open || static_cast<int>(out.back().mats.size()) == (v.big ? kMaxBig : fg::kMaxMats) || with.bytes(v) > budget(v)) {
        out.push_back(Chunk{{}, v});
        with = Regions();
        with.take(sh, 1, v);
        open = true;
      }
      all = with;
      out.back().mats.push_back(&mats[j]);
    }
  }
  return out;
}

framefb_status prepare(const Chunk& ch, int32_t ops, framefb_dtype dt, Prepared& P) {
  // (the matrices' entries are filled below, the rest is never read)
  std::memset(P.args, 0, offsetof(fg::Launch, m));
  std::memset(P.red, 0, offsetof(fp::Reduce, m));
  fg::Launch& A = *P.args;
  P.v = ch.v;
  void* fn = kernel_ptr(ch.v, dt);
  if (!fn) return FRAMEFB_EINVAL;
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return FRAMEFB_ECUDA;
  const int per = ch.v.nt == 512 ? 1 : 2;
  const int nm = static_cast<int>(ch.mats.size());
  // pairs per unit: what fits, but no more than one unit per CTA takes.  (Rounded
  // up: with units of one pair and up to two per CTA, some CTAs walked two units one
  // after the other: 256^2 fp32, 3000 entries, 512 tokens, forward 15.7 us, 11.9 so.)
  const int64_t slots = static_cast<int64_t>(sms) * per;
  int64_t pairs = 0;
  for (const framefb_mat* M : ch.mats) pairs += (M->N + 1) / 2;
  const int64_t spread = std::max<int64_t>(1, (pairs + slots - 1) / slots);
  int nsh = 0;
  Regions reg;
  for (int j = 0; j < nm; ++j) {
    if (j > 0 && ch.mats[j]->plan == ch.mats[j - 1]->plan) {
      A.m[j].shape = A.m[j - 1].shape;
      continue;
    }
    fg::Shape sh;
    if (!shape_of(header_of(ch.mats[j]->plan), ch.v, sh)) return FRAMEFB_EINVAL;
    int s = 0;  // (plans of one geometry share it)
    while (s < nsh && std::memcmp(&A.sh[s], &sh, sizeof(sh)) != 0) ++s;
    if (s == nsh) {
      A.sh[nsh++] = sh;
      reg.take(sh, 1, ch.v);
    }
    A.m[j].shape = s;
  }
  if (reg.bytes(ch.v) > budget(ch.v)) return FRAMEFB_EUNSUPPORTED;
  const size_t room = budget(ch.v) - reg.masks - reg.plan(ch.v);
  for (int i = 0; i < nsh; ++i) {
    fg::Shape& sh = A.sh[i];
    const int64_t fit = static_cast<int64_t>(room / (static_cast<size_t>(sh.pair) * 8));
    sh.PP = static_cast<int32_t>(std::max<int64_t>(1, std::min<int64_t>({kMaxPairs, spread, fit})));
    reg.take(sh, sh.PP, ch.v);
  }
  P.smem = reg.bytes(ch.v);
  A.oPlan = static_cast<int32_t>(reg.pairs);
  A.oMask = static_cast<int32_t>(reg.pairs + reg.plan(ch.v));
  int64_t units = 0;
  int32_t nnz_max = 0;
  for (int j = 0; j < nm; ++j) {
    const framefb_mat& M = *ch.mats[j];
    const FfbPlanHeader& h = *header_of(M.plan);
    fg::Mat& K = A.m[j];
    const fg::Shape& sh = A.sh[K.shape];
    K.in[0] = M.X;
    K.in[1] = M.dY;
    K.out[0] = M.dX;
    K.out[1] = M.Y;
    K.ld[0] = M.ldx;
    K.ld[1] = M.ldy;
    K.plan = static_cast<const uint8_t*>(M.plan_dev);
    K.c_val = M.c_val;
    K.N = M.N;
    K.ubeg = static_cast<int32_t>(units);
    K.ntiles = (M.N + 2 * sh.PP - 1) / (2 * sh.PP);
    K.seff = static_cast<float>(static_cast<double>(M.scale) / 16.0);
    units += K.ntiles;
    if (units > INT32_MAX / 2) return FRAMEFB_EUNSUPPORTED;
    nnz_max = std::max(nnz_max, h.nnz);
  }
  // The units are split over the CTAs at equal cost: groups to transform and
  // entries to gather, per pair; one unit per CTA where there are no more of them.
  for (int j = 0; j < nm; ++j) {
    const FfbPlanHeader& h = *header_of(ch.mats[j]->plan);
    fg::Mat& K = A.m[j];
    K.cost = units <= slots ? 1 : A.sh[K.shape].PP * (2 * (h.Gn + h.Gm) * kGroupCost + h.nnz * kEntryCost) / 64 + 1;
    K.cbeg = A.total_cost;
    A.total_cost += static_cast<int64_t>(K.cost) * K.ntiles;
  }
  A.nmats = nm;
  A.mode = ops;
  A.total_units = static_cast<int32_t>(units);
  A.stride = (nnz_max + 63) & ~63;
  P.nnz_max = nnz_max;
  int per_sm = 0;
  if (allow_shared(fn, dev, P.smem) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, ch.v.nt, P.smem) != cudaSuccess)
    return FRAMEFB_ECUDA;
  if (per_sm < 1) return FRAMEFB_EUNSUPPORTED;
  // (With a unit for every CTA at equal shares the largest unit's cost bounded the
  // grid: 4096 -> 256 beside two small ones, 128 tokens, forward, 24.5 us, 10.6 so.)
  P.grid = static_cast<int>(std::min<int64_t>({slots, static_cast<int64_t>(sms) * per_sm, units}));
  P.slots = slots;
  P.ws_bytes = 0;
  if (ops & FRAMEFB_OP_GRAD_COEFF) {
    P.ws_bytes = static_cast<size_t>(P.grid + nm) * A.stride * sizeof(float) + 256;
    P.red->stride = A.stride;
    // CTA of a unit: the last one whose share begins at or before the unit
    auto cta_of = [&](const fg::Mat& K, int32_t u) {
      const int64_t at = K.cbeg + static_cast<int64_t>(u - K.ubeg) * K.cost;
      return static_cast<int32_t>(((at + 1) * P.grid + A.total_cost - 1) / A.total_cost - 1);
    };
    for (int j = 0; j < nm; ++j) {
      fp::ReduceMat& R = P.red->m[j];
      R.dC = ch.mats[j]->dC;
      R.nnz = header_of(ch.mats[j]->plan)->nnz;
      R.seff = A.m[j].seff;
      R.c0 = cta_of(A.m[j], A.m[j].ubeg);
      R.c1 = cta_of(A.m[j], A.m[j].ubeg + A.m[j].ntiles - 1);
    }
  }
  return FRAMEFB_OK;
}

// Launch parameters live on the heap: too large for the stack of some callers.
struct Buffers {
  std::unique_ptr<fg::Launch> a{new fg::Launch};
  std::unique_ptr<fp::Reduce> r{new fp::Reduce};
  Prepared prep() {
    Prepared p{};
    p.args = a.get();
    p.red = r.get();
    return p;
  }
};


bool frame_ok(const framefb_dev_frame* f, int32_t d) {
  return f && f->dft_groups && f->k == 16 && f->d == d && f->ncols == d && f->rho * 16 == d && f->val && f->colptr && f->rowidx;
}

framefb_status check_mat(const framefb_mat& M, int32_t ops, framefb_dtype dt) {
  const bool F = ops & FRAMEFB_OP_FORWARD, D = ops & FRAMEFB_OP_BACKWARD_DX, C = ops & FRAMEFB_OP_GRAD_COEFF;
  const FfbPlanHeader* h = header_of(M.plan);
  if (!h || M.N < 0 || M.n <= 0 || M.m <= 0 || h->n != M.n || h->m != M.m) return FRAMEFB_EINVAL;
  if (!frame_ok(M.fin, M.n) || !frame_ok(M.fout, M.m)) return FRAMEFB_EINVAL;
  if (!M.plan_dev || !aligned16(M.plan_dev) || !std::isfinite(M.scale)) return FRAMEFB_EINVAL;
  if ((F || D) && h->nnz > 0 && !M.c_val) return FRAMEFB_EINVAL;
  if (C && h->nnz > 0 && !M.dC) return FRAMEFB_EINVAL;
  if (M.N == 0) return FRAMEFB_OK;
  const int64_t esz = dt == FRAMEFB_BF16 ? 2 : 4;
  const bool needX = F || C, needdY = D || C;
  if ((needX || D) && (M.ldx < M.n || (M.ldx * esz) % 16)) return FRAMEFB_EINVAL;
  if ((needdY || F) && (M.ldy < M.m || (M.ldy * esz) % 16)) return FRAMEFB_EINVAL;
  if (needX && (!M.X || !aligned16(M.X))) return FRAMEFB_EINVAL;
  if (needdY && (!M.dY || !aligned16(M.dY))) return FRAMEFB_EINVAL;
  if (F && (!M.Y || !aligned16(M.Y))) return FRAMEFB_EINVAL;
  if (D && (!M.dX || !aligned16(M.dX))) return FRAMEFB_EINVAL;
  return FRAMEFB_OK;
}

}  // namespace

// The path takes
//   * fp32: every structured plan that fits a variant with whole buffers.  Fused
//     pass, the one-phase FFT kernel -> this one: 8 matrices of 768^2, 2048 tokens
//     203 -> 104 us; 4096^2, 1000 entries, 256 tokens 34 -> 22; 96 of 256^2, 512
//     tokens 440 -> 123; 8 tokens of one of 256^2 the same 13 us.
//   * fp32 with compacted buffers (BIG), where it is the faster one.  Columns of up
//     to 16 entries come here for their wide sides only (8192, 14336 features), and
//     the transforms of mostly unnamed coordinates gain nothing: 14336 -> 4096, 1000
//     entries, fused, 8 / 256 / 2000 tokens 24 / 42 / 185 us there, 32 / 35 / 196
//     here.  Longer columns: passes with dX and dC (4096^2, 8192 entries, 8 / 1024
//     tokens 64 / 173 -> 54 / 99; 4096 -> 14336 57 / 335 -> 52 / 153; an input side
//     of more than 256 groups from 160 tokens, 14336 -> 4096 at 128 / 202 tokens 62 /
//     109 against 69 / 70); a forward pass on 8192 features and more of both sides
//     (4096^2 31 / 57 -> 21 / 41, but 4096 -> 1024, 1024 tokens 35 -> 41); dX or dC
//     alone there from 768 tokens (4096^2, 512 / 1024 / 2000 tokens, dX 31 / 56 / 107
//     against 36 / 48 / 66).
//   * bf16: plans beyond the tcgen05 kernels with a side of more than 128
//     groups (the LLaMA-3 MLP shapes), whole: the tcgen05 kernel would run them
//     in parts or not at all.  8192 Zipf entries, fused, 64 / 1024 / 4096 tokens:
//     4096 -> 14336 (five parts) 112 / 193 / 412 -> 43 / 99 / 248 us, 4096 -> 5120
//     74 / 125 / 263 -> 38 / 74 / 199;
//     14336 -> 4096 (contraction path) 61 / 218 / 660 -> 61 / 109 / 265 us, so
//     that side from 128 tokens.  Narrower big plans stay in parts (4096^2, 8192
//     tokens 289 us against 340 here).
constexpr int32_t kMinTokensWideIn = 128;
constexpr int32_t kBigGroups = 256;      // of both sides: a forward pass, dX or dC alone
constexpr int32_t kBigTokensWideIn = 160, kBigTokensOne = 768;

GrpKind grp_kind(const framefb_plan* plan) {
  const FfbPlanHeader* h = header_of(plan);
  const Variant v = h ? variant(h) : Variant{0, 0, false};
  return v.nt == 0 ? GrpKind::none : v.big ? GrpKind::big : GrpKind::whole;
}

bool grp_takes(GrpKind kind, const framefb_mat& M, int32_t ops, framefb_dtype dt) {
  if (kind == GrpKind::none || M.N < 1) return false;
  if (kind == GrpKind::whole) return dt == FRAMEFB_F32;
  const FfbPlanHeader* h = header_of(M.plan);
  if (dt == FRAMEFB_BF16) return h->Gm > 128 || (h->Gn > 128 && M.N >= kMinTokensWideIn);
  const bool D = ops & FRAMEFB_OP_BACKWARD_DX, C = ops & FRAMEFB_OP_GRAD_COEFF;
  if (static_cast<size_t>(ffb_tile_layout(*h, ops, 1, C).total) * 4 > 227 * 1024) return true;  // too large for the other
  if (std::max(h->EZ, h->EG) <= 16) return false;
  if (D && C) return h->Gn <= 256 || M.N >= kBigTokensWideIn;
  return h->Gn + h->Gm >= kBigGroups && (ops == FRAMEFB_OP_FORWARD || M.N >= kBigTokensOne);
}

struct GrpLaunches {
  struct One {
    Buffers b;
    Prepared P{};
    void* fn = nullptr;
    unsigned mats = 0;
    bool reduce = false;
  };
  std::vector<One> list;
};

framefb_status grp_check(const framefb_mat* mats, int32_t nmats, int32_t ops, framefb_dtype dt, size_t* ws_need,
                         GrpReady* keep) {
  *ws_need = 0;
  if (nmats == 0) return FRAMEFB_OK;
  int64_t pairs = 0, slots = 0;
  int32_t stride = 0;
  bool big = false;
  std::vector<framefb_mat> wide;  // unpadded, with an input side that fewer tokens send to the contraction path
  try {
    for (int32_t j = 0; j < nmats; ++j) {
      const framefb_status s = check_mat(mats[j], ops, dt);
      if (s != FRAMEFB_OK) return s;
      const FfbPlanHeader* h = header_of(mats[j].plan);
      pairs += (mats[j].N + 1) / 2;
      stride = std::max(stride, (h->nnz + 63) & ~63);
      if (dt == FRAMEFB_BF16 && h->Gn > 128 && mats[j].ldx == mats[j].n && mats[j].ldy == mats[j].m) wide.push_back(mats[j]);
    }
  } catch (const std::bad_alloc&) {
    return FRAMEFB_ENOMEM;
  }
  // (asked for at every token count, as on the contraction path)
  const framefb_status ds = dense_check(wide.data(), static_cast<int32_t>(wide.size()), ops, dt, ws_need);
  if (ds != FRAMEFB_OK) return ds;
  try {
    auto all = std::make_shared<GrpLaunches>();
    for (const Chunk& c : chunks_of(mats, nmats)) {
      if (keep || all->list.empty()) all->list.emplace_back();
      GrpLaunches::One& l = all->list.back();
      l.P = l.b.prep();
      const framefb_status s = prepare(c, ops, dt, l.P);
      if (s != FRAMEFB_OK) return s;
      *ws_need = std::max(*ws_need, l.P.ws_bytes);
      slots = std::max(slots, l.P.slots);
      big = big || l.P.v.big;
      l.fn = kernel_ptr(l.P.v, dt);
      l.mats = static_cast<unsigned>(c.mats.size());
      l.reduce = (ops & FRAMEFB_OP_GRAD_COEFF) && l.P.nnz_max > 0;
    }
    // What a query reports covers any smaller token count too: more tokens can make
    // fewer, larger units, and calls of few tokens take other kernels, with a CTA per
    // SM, where the plan is a big one.
    if (!keep && (ops & FRAMEFB_OP_GRAD_COEFF))
      *ws_need = std::max(*ws_need, static_cast<size_t>((big ? slots : std::min(slots, pairs)) + nmats) * stride * sizeof(float) + 256);
    if (keep) *keep = std::move(all);
  } catch (const std::bad_alloc&) {
    return FRAMEFB_ENOMEM;
  }
  return FRAMEFB_OK;
}

framefb_status grp_run(const GrpReady& ready, void* ws, cudaStream_t st) {
  if (!ready) return FRAMEFB_OK;
  for (const GrpLaunches::One& l : ready->list) {
    const Prepared& P = l.P;
    P.args->partial = static_cast<float*>(ws);
    P.red->partial = static_cast<const float*>(ws);
    void* kargs[] = {P.args};
    if (launch_chained(l.fn, dim3(P.grid), dim3(P.v.nt), kargs, P.smem, st) != cudaSuccess) return FRAMEFB_ECUDA;
    if (l.reduce) {
      void* rargs[] = {P.red};
      if (launch_chained(reinterpret_cast<void*>(fp::pair_reduce_kernel), dim3((P.nnz_max + 31) / 32, l.mats),
                         dim3(32 * fp::kLanes), rargs, 0, st) != cudaSuccess)
        return FRAMEFB_ECUDA;
    }
  }
  return FRAMEFB_OK;
}

}  // namespace ffb_host
