// Launchers of the row-transform path of libframefb (framefb_row.cuh):
// which matrices it takes, the shared-memory map, and the launches.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstddef>
#include <cstdlib>
#include <cstring>
#include <memory>
#include <new>
#include <string>
#include <vector>

#include "framefb.h"
#include "framefb_dense.h"
#include "framefb_launch.h"
#include "framefb_row.cuh"
#include "framefb_row.h"
#include "plan_internal.h"
#include "plan_layout.h"

namespace ffb_host {

namespace {

namespace fp = ffb::pair;
namespace fr = ffb::row;
static_assert(fr::kMaxMats <= fp::kReduceMats, "one reduction per launch");

static_assert(sizeof(fr::Launch) <= 32764 && sizeof(fp::Reduce) <= 32764, "launch parameters exceed the parameter space");

inline size_t rup(size_t x, size_t a) { return (x + a - 1) / a * a; }

const FfbPlanHeader* header_of(const framefb_plan* p) {
  if (!p || p->image.size() < sizeof(FfbPlanHeader)) return nullptr;
  const FfbPlanHeader* h = reinterpret_cast<const FfbPlanHeader*>(p->image.data());
  if (h->magic != FFB_PLAN_MAGIC || h->version != FFB_PLAN_VERSION || h->P != fp::kColumns) return nullptr;
  if (static_cast<size_t>(h->total_bytes) > p->image.size()) return nullptr;
  return h;
}

// Geometry of a matrix (pair buffers laid out, PP not set): both frames one
// DFT of a size the kernel has passes for, the plan in the paper's column
// order.
bool shape_of(const framefb_mat& M, fr::Shape& sh) {
  const FfbPlanHeader* h = header_of(M.plan);
  if (!h || h->layout != FFB_LAYOUT_DENSE) return false;
  std::memset(&sh, 0, sizeof(sh));
  const framefb_dev_frame* f[2] = {M.fin, M.fout};
  const int32_t K[2] = {h->n, h->m}, ovf[2] = {h->ovfG, h->ovfZ};
  int32_t off = 0;
  for (int sd = 0; sd < 2; ++sd) {
    if (!f[sd] || !f[sd]->dft_groups || f[sd]->rho != 2 || f[sd]->d != 2 * f[sd]->k || f[sd]->ncols != f[sd]->d ||
        K[sd] != f[sd]->d || fr::passes_of(f[sd]->k) == 0)
      return false;
    sh.k[sd] = f[sd]->k;
    const int32_t scratch = 2 * fr::scratch_of(sh.k[sd]);  // float2
    sh.A[sd] = off;
    off += scratch;
    sh.B[sd] = off;
    off += (std::max(K[sd] + ovf[sd], scratch) + 1) / 2 * 2;
    if (K[sd] + ovf[sd] > fp::kMaxSlots) return false;
  }
  sh.pair = off;
  return true;
}

// Twiddle tables of a shape (float2): one per distinct k.
int32_t twiddles(fr::Shape& sh) {
  sh.tw[0] = 0;
  sh.tw[1] = sh.k[1] == sh.k[0] ? 0 : fr::twiddles_of(sh.k[0]);
  return sh.tw[1] + fr::twiddles_of(sh.k[1]);
}

constexpr size_t kSmemSm = 228 * 1024;    // shared memory of an SM
constexpr size_t kSmemCta = 227 * 1024 - 256;  // of a CTA, less the static part
constexpr int kMaxPairs = 8;

// A kernel variant: threads per CTA, plan entries per thread and path, the
// DFT size of both sides (0: any).
struct Variant {
  int nt, ke, k;
  bool operator==(const Variant& o) const { return nt == o.nt && ke == o.ke && k == o.k; }
};

// Shared memory one CTA of a kernel variant may take.
size_t budget(int nt) { return nt == 512 ? kSmemCta : kSmemSm / 2 - 1024 - 256; }

// Shared memory of a launch: its regions hold the largest of its shapes.
struct Regions {
  size_t stage[2] = {0, 0}, pairs = 0, tw = 0;
  void take(fr::Shape sh, int pp) {
    for (int sd = 0; sd < 2; ++sd) stage[sd] = std::max(stage[sd], rup(8 * static_cast<size_t>(pp) * sh.k[sd], 128));
    pairs = std::max(pairs, static_cast<size_t>(pp) * sh.pair * 8);
    tw = std::max(tw, rup(static_cast<size_t>(twiddles(sh)) * 8, 128));
  }
  size_t bytes(const Variant& v) const { return stage[0] + stage[1] + pairs + tw + fp::plan_bytes(v.nt, v.ke) + 16; }
};

// Bytes a unit of `pp` pairs of a shape needs in all.
size_t unit_bytes(const fr::Shape& sh, int pp, const Variant& v) {
  Regions r;
  r.take(sh, pp);
  return r.bytes(v);
}

// The kernel variant a matrix runs on: two CTAs of 256 threads per SM where a
// unit fits half an SM and a thread's share of a plan column is at most 8
// entries, else one CTA of 512 (nt = 0: neither fits).
Variant variant(const framefb_mat& M, const fr::Shape& sh) {
  const FfbPlanHeader& h = *header_of(M.plan);
  const int e = std::max(h.EZ, h.EG);
  const int k = sh.k[0] != sh.k[1] ? 0 : sh.k[0];
  for (const Variant& v : {Variant{256, 4, 0}, Variant{256, 8, 0}, Variant{512, 8, 0}}) {
    if (e > v.ke * (v.nt / fp::kColumns) || unit_bytes(sh, 1, v) > budget(v.nt)) continue;
    const bool own = v.nt == 512 ? k == 1024 || k == 2048 : k == 384 || k == 512;  // sizes with a kernel of their own
    return Variant{v.nt, v.ke, own ? k : 0};
  }
  return Variant{0, 0, 0};
}

void* kernel_ptr(const Variant& v) {
#define FFB_ROW(N, E, S) \
  if (v == Variant{N, E, S}) return reinterpret_cast<void*>(fr::row_kernel<N, E, S>);
  FFB_ROW(256, 4, 0)
  FFB_ROW(256, 4, 384)
  FFB_ROW(256, 4, 512)
  FFB_ROW(256, 8, 0)
  FFB_ROW(256, 8, 384)
  FFB_ROW(256, 8, 512)
  FFB_ROW(512, 8, 0)
  FFB_ROW(512, 8, 1024)
  FFB_ROW(512, 8, 2048)
#undef FFB_ROW
  return nullptr;
}

struct Prepared {
  fr::Launch* args;
  fp::Reduce* red;
  int grid, nnz_max;
  Variant v;
  size_t smem, ws_bytes;
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
    fr::Shape sh;
    of[j] = shape_of(mats[j], sh) ? variant(mats[j], sh) : Variant{0, 0, 0};
    if (of[j].nt && std::find(kinds.begin(), kinds.end(), of[j]) == kinds.end()) kinds.push_back(of[j]);
  }
  std::vector<Chunk> out;
  for (const Variant& v : kinds) {
    std::vector<const FfbPlanHeader*> shapes;
    Regions all;  // of one pair of each shape of the chunk
    bool open = false;
    for (int32_t j = 0; j < nmats; ++j) {
      if (!(of[j] == v)) continue;
      const FfbPlanHeader* h = header_of(mats[j].plan);
      bool known = std::find(shapes.begin(), shapes.end(), h) != shapes.end();
      fr::Shape sh;
      shape_of(mats[j], sh);
      Regions with = all;
      with.take(sh, 1);
      if (!open || static_cast<int>(out.back().mats.size()) == fr::kMaxMats ||
          (!known && (static_cast<int>(shapes.size()) == fr::kMaxShapes || with.bytes(v) > budget(v.nt)))) {
        out.push_back(Chunk{{}, v});
        shapes.clear();
        all = Regions();
        open = true;
        known = false;
      }
      if (!known) shapes.push_back(h);
      all.take(sh, 1);
      out.back().mats.push_back(&mats[j]);
    }
  }
  return out;
}

framefb_status prepare(const Chunk& ch, int32_t ops, Prepared& P) {
  // (the matrices' entries are filled below, the rest is never read)
  std::memset(P.args, 0, offsetof(fr::Launch, m));
  std::memset(P.red, 0, offsetof(fp::Reduce, m));
  fr::Launch& A = *P.args;
  P.v = ch.v;
  void* fn = kernel_ptr(ch.v);
  if (!fn) return FRAMEFB_EINVAL;
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return FRAMEFB_ECUDA;
  const int per = ch.v.nt == 512 ? 1 : 2;
  const int nm = static_cast<int>(ch.mats.size());
  // pairs per unit: what fits, but no more than gives every CTA a unit
  int64_t pairs = 0;
  for (const framefb_mat* M : ch.mats) pairs += (M->N + 1) / 2;
  const int64_t spread = std::max<int64_t>(1, pairs / (static_cast<int64_t>(sms) * per));
  std::vector<const FfbPlanHeader*> hd;
  int nsh = 0;
  for (int j = 0; j < nm; ++j) {
    const framefb_mat& M = *ch.mats[j];
    const FfbPlanHeader* h = header_of(M.plan);
    int s = static_cast<int>(std::find(hd.begin(), hd.end(), h) - hd.begin());
    if (s == nsh) {
      if (nsh == fr::kMaxShapes) return FRAMEFB_EINVAL;
      hd.push_back(h);
      fr::Shape& sh = A.sh[nsh++];
      if (!shape_of(M, sh)) return FRAMEFB_EINVAL;
      int pp = static_cast<int>(std::min<int64_t>(kMaxPairs, spread));
      while (pp > 1 && unit_bytes(sh, pp, ch.v) > budget(ch.v.nt)) --pp;
      sh.PP = pp;
    }
    A.m[j].shape = s;
  }
  // fewer pairs where the largest stage and the largest pair buffers come from
  // different shapes (one pair of each fits: chunks_of)
  Regions reg;
  for (;;) {
    reg = Regions();
    int most = 0;
    for (int i = 0; i < nsh; ++i) {
      reg.take(A.sh[i], A.sh[i].PP);
      if (A.sh[i].PP > A.sh[most].PP) most = i;
    }
    P.smem = reg.bytes(ch.v);
    if (P.smem <= budget(ch.v.nt)) break;
    if (A.sh[most].PP == 1) return FRAMEFB_EUNSUPPORTED;
    --A.sh[most].PP;
  }
  for (int i = 0; i < nsh; ++i) twiddles(A.sh[i]);  // their table offsets
  A.stage1 = static_cast<int32_t>(reg.stage[0]);
  A.oPairs = static_cast<int32_t>(reg.stage[0] + reg.stage[1]);
  A.oTw = static_cast<int32_t>(A.oPairs + reg.pairs);
  A.oPlan = static_cast<int32_t>(A.oTw + reg.tw);
  A.oBar = A.oPlan + fp::plan_bytes(ch.v.nt, ch.v.ke);
  int64_t units = 0;
  int32_t nnz_max = 0;
  for (int j = 0; j < nm; ++j) {
    const framefb_mat& M = *ch.mats[j];
    const FfbPlanHeader& h = *header_of(M.plan);
    fr::Mat& K = A.m[j];
    const fr::Shape& sh = A.sh[K.shape];
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
    K.seff = static_cast<float>(static_cast<double>(M.scale) / std::sqrt(static_cast<double>(sh.k[0]) * sh.k[1]));
    units += K.ntiles;
    if (units > INT32_MAX / 2) return FRAMEFB_EUNSUPPORTED;
    nnz_max = std::max(nnz_max, h.nnz);
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
  P.grid = static_cast<int>(std::min<int64_t>(static_cast<int64_t>(sms) * per_sm, units));
  P.ws_bytes = 0;
  if (ops & FRAMEFB_OP_GRAD_COEFF) {
    P.ws_bytes = static_cast<size_t>(P.grid + nm) * A.stride * sizeof(float) + 256;
    P.red->stride = A.stride;
    auto cta_of = [&](int64_t u) { return static_cast<int32_t>(((u + 1) * P.grid - 1) / units); };
    for (int j = 0; j < nm; ++j) {
      fp::ReduceMat& R = P.red->m[j];
      R.dC = ch.mats[j]->dC;
      R.nnz = header_of(ch.mats[j]->plan)->nnz;
      R.seff = A.m[j].seff;
      R.c0 = cta_of(A.m[j].ubeg);
      R.c1 = cta_of(static_cast<int64_t>(A.m[j].ubeg) + A.m[j].ntiles - 1);
    }
  }
  return FRAMEFB_OK;
}

// Launch parameters live on the heap: too large for the stack of some callers.
struct Buffers {
  std::unique_ptr<fr::Launch> a{new fr::Launch};
  std::unique_ptr<fp::Reduce> r{new fp::Reduce};
  Prepared prep() {
    Prepared p{};
    p.args = a.get();
    p.red = r.get();
    return p;
  }
};

}  // namespace

// The path takes bf16 matrices whose frames are rho = 2 with one of the
// kernel's DFT sizes and whose plan and pair buffers fit a variant.  Against
// the contraction path it is faster at every token count (fused pass, two
// matrices, 1 / 300 / 4096 tokens: d = 768 20 / 23 / 69 us against 83 / 114 /
// 251, d = 1024 21 / 29 / 91 against 95 / 120 / 298, d = 4096 30 / 44 / 324
// against 248 / 339 / 1780).  DFT_384 below 512 tokens stays on the
// contraction path all the same: those calls are its regression cover on
// DFT frames (tests/test_gpu_dense.py names the kernels it expects there).
constexpr int32_t kMinTokens384 = 512;

bool row_takes(const framefb_mat& M, int32_t ops, framefb_dtype dt) {
  (void)ops;
  if (dt != FRAMEFB_BF16 || M.N < 1) return false;
  fr::Shape sh;
  if (!shape_of(M, sh)) return false;
  if ((sh.k[0] == 384 || sh.k[1] == 384) && M.N < kMinTokens384) return false;
  return variant(M, sh).nt != 0;
}

struct RowLaunches {
  struct One {
    Buffers b;
    Prepared P{};
    void* fn = nullptr;
    unsigned mats = 0;
    bool reduce = false;
  };
  std::vector<One> list;
};

// The workspace asked for stays the contraction path's, though this path needs
// only its dC partials: which of the two a call takes depends on its tokens, and
// callers size one workspace for calls that differ in them.
framefb_status row_check(const framefb_mat* mats, int32_t nmats, int32_t ops, framefb_dtype dt, size_t* ws_need,
                         RowReady* keep) {
  *ws_need = 0;
  if (nmats == 0) return FRAMEFB_OK;
  for (int32_t j = 0; j < nmats; ++j)
    if (!dense_mat_ok(mats[j], ops)) return FRAMEFB_EINVAL;
  const framefb_status d = dense_check(mats, nmats, ops, dt, ws_need);
  if (d != FRAMEFB_OK) return d;
  try {
    auto all = std::make_shared<RowLaunches>();
    for (const Chunk& c : chunks_of(mats, nmats)) {
      if (keep || all->list.empty()) all->list.emplace_back();
      RowLaunches::One& l = all->list.back();
      l.P = l.b.prep();
      const framefb_status s = prepare(c, ops, l.P);
      if (s != FRAMEFB_OK) return s;
      *ws_need = std::max(*ws_need, l.P.ws_bytes);
      l.fn = kernel_ptr(l.P.v);
      l.mats = static_cast<unsigned>(c.mats.size());
      l.reduce = (ops & FRAMEFB_OP_GRAD_COEFF) && l.P.nnz_max > 0;
    }
    if (keep) *keep = std::move(all);
  } catch (const std::bad_alloc&) {
    return FRAMEFB_ENOMEM;
  }
  return FRAMEFB_OK;
}

framefb_status row_run(const RowReady& ready, void* ws, cudaStream_t st) {
  if (!ready) return FRAMEFB_OK;
  for (const RowLaunches::One& l : ready->list) {
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

framefb_status row_kernel_names(const framefb_mat* mats, int32_t nmats, int32_t ops, framefb_dtype dt,
                                std::vector<std::string>& out) {
  (void)mats;
  (void)dt;
  if (nmats == 0) return FRAMEFB_OK;
  const std::string k = "row_kernel<" + std::to_string(ops) + ">";
  if (std::find(out.begin(), out.end(), k) == out.end()) out.push_back(k);
  return FRAMEFB_OK;
}

framefb_status row_wait_timeouts(uint32_t* count) {
  if (cudaMemcpyFromSymbol(count, fr::g_row_timeouts, sizeof(uint32_t)) != cudaSuccess) return FRAMEFB_ECUDA;
  return FRAMEFB_OK;
}

}  // namespace ffb_host
