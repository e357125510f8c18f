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
#define FFB_GRP(N, E, B)                                                                             \
  if (v == Variant{N, E, B})                                                                         \
    return dt == FRAMEFB_BF16 ? reinterpret_cast<void*>(fg::fft_tile_kernel<__nv_bfloat16, N, E, B>)    \
                              : reinterpret_cast<void*>(fg::fft_tile_kernel<float, N, E, B>);
  FFB_GRP(256, 4, false)
  FFB_GRP(256, 8, false)
  FFB_GRP(512, 8, false)
  FFB_GRP(512, fg::kBigE, true)
#undef FFB_GRP
  return nullptr;
}

struct Prepared {
  fg::Launch* args;
  fp::Reduce* red;
  int grid, nnz_max;
  Variant v;
  size_t smem, ws_bytes, ws_cover;  // (workspace this launch takes, and what a query reports)
};

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
      if (!open || static_cast<int>(out.back().mats.size()) == fg::kMaxMats || with.bytes(v) > budget(v)) {
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
  P.ws_bytes = P.ws_cover = 0;
  if (ops & FRAMEFB_OP_GRAD_COEFF) {
    // (more tokens can make fewer, larger units: what is asked for covers the
    // grid of any smaller count)
    auto bytes = [&](int64_t ctas) { return static_cast<size_t>(ctas + nm) * A.stride * sizeof(float) + 256; };
    P.ws_bytes = bytes(P.grid);
    P.ws_cover = bytes(std::min(slots, pairs));
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
//   * fp32: every structured plan that fits a variant (the one-phase FFT kernel
//     keeps the others).  Fused pass, that kernel -> this one: 8 matrices of
//     768^2, 2048 tokens 203 -> 107 us; 2 of 3072^2, 1000 tokens 85 -> 63 us; 8 of
//     256^2, 4096 tokens 277 -> 90 us; 8 tokens of one of 256^2 the same 21 us.
//   * bf16: plans beyond the tcgen05 kernels with a side of more than 128
//     groups (the LLaMA-3 MLP shapes), whole: the tcgen05 kernel would run them
//     in parts or not at all.  8192 Zipf entries, fused, 64 / 1024 / 4096 tokens:
//     4096 -> 14336 (five parts) 115 / 194 / 408 -> 49 / 102 / 249 us;
//     14336 -> 4096 (contraction path) 61 / 220 / 664 -> 61 / 112 / 268 us, so
//     that side from 128 tokens.  Narrower big plans stay in parts (4096^2, 8192
//     tokens 289 us against 340 here).
constexpr int32_t kMinTokensWideIn = 128;

bool grp_takes(const framefb_mat& M, int32_t ops, framefb_dtype dt) {
  (void)ops;
  const FfbPlanHeader* h = header_of(M.plan);
  if (!h || M.N < 1) return false;
  const Variant v = variant(h);
  if (v.nt == 0) return false;
  if (dt == FRAMEFB_F32) return true;
  return v.big && (h->Gm > 128 || (h->Gn > 128 && M.N >= kMinTokensWideIn));
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
  for (int32_t j = 0; j < nmats; ++j) {
    framefb_status s = check_mat(mats[j], ops, dt);
    if (s != FRAMEFB_OK) return s;
    // the workspace asked for covers fewer tokens too, where the contraction
    // path takes these plans (kMinTokensWideIn)
    if (dt == FRAMEFB_BF16 && header_of(mats[j].plan)->Gn > 128 && mats[j].ldx == mats[j].n && mats[j].ldy == mats[j].m) {
      size_t need = 0;
      s = dense_check(&mats[j], 1, ops, dt, &need);
      if (s != FRAMEFB_OK) return s;
      *ws_need = std::max(*ws_need, need);
    }
  }
  try {
    auto all = std::make_shared<GrpLaunches>();
    for (const Chunk& c : chunks_of(mats, nmats)) {
      if (keep || all->list.empty()) all->list.emplace_back();
      GrpLaunches::One& l = all->list.back();
      l.P = l.b.prep();
      const framefb_status s = prepare(c, ops, dt, l.P);
      if (s != FRAMEFB_OK) return s;
      *ws_need = std::max(*ws_need, keep ? l.P.ws_bytes : l.P.ws_cover);
      l.fn = kernel_ptr(l.P.v, dt);
      l.mats = static_cast<unsigned>(c.mats.size());
      l.reduce = (ops & FRAMEFB_OP_GRAD_COEFF) && l.P.nnz_max > 0;
    }
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
