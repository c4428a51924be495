// Fusion planner (host) and the fused-segment tile kernel.
//
// The planner groups a circuit into segments; all gates of a segment are
// applied to each tile while it sits in shared memory, so a segment costs
// one HBM read and one HBM write of the state however many gates it holds.
// This is the single-GPU counterpart of the paper's observation that gates
// on local qubits need no data exchange (Sec. 2): a segment's tile qubits
// play the role of the local qubits, and choosing them per segment lets the
// "non-local" gates become local too.
#include <algorithm>
#include <iterator>
#include <mutex>
#include <string>
#include <type_traits>
#include <unordered_map>

#include "arith.cuh"
#include "jit.h"
#include "lqs_internal.cuh"
#include "tile.cuh"
#include "tile_ops.cuh"

// Dense work per segment: a compiled segment is straight-line code, and one
// whose dense updates add up past this weight (3 per two-qubit dense op, 1
// per one-qubit dense op; diagonal and permutation ops are free) spends more
// in instruction fetch than a further pass costs.  30-qubit 10-layer ansatz,
// complex128: caps of 8 / 12 / 16 / 24 / 40 ran 451 / 418 / 426 / 453 / 510 ms.
// Two-qubit ops weigh 3, so that a segment takes four: with 4 (three to a
// segment) U4 windows on 24 qubits ran 4.46 ms, a U4 brick circuit 4.87, 200
// random gates 7.75; with 3 4.34, 4.74, 7.54.
#ifndef LQS_SEGMENT_DENSE_CAP
#define LQS_SEGMENT_DENSE_CAP 12
#endif
// complex64 segments carry float32 arithmetic, several times less code per op;
// their two-qubit ops weigh 4
#ifndef LQS_SEGMENT_DENSE_CAP_C64
#define LQS_SEGMENT_DENSE_CAP_C64 64
#endif
// The float64 policy is bound by its pipe, not by instruction fetch: caps of
// 12 / 16 / 24 ran 24-qubit circuits of 4 layers RX + RZ in 28.6 / 28.7 / 28.2 ms,
// U4 windows 32.7 / 32.6 / 32.4, a 10-layer ansatz 26.7 / 27.2 / 26.3.  Searched
// plans helped the ansatz (25.0 ms) and cost the universal circuit 18% (18.6 ->
// 21.9): fewer passes, more diagonal products.
#ifndef LQS_SEGMENT_DENSE_CAP_F64
#define LQS_SEGMENT_DENSE_CAP_F64 24
#endif

namespace lqs {

// ---------------------------------------------------------------------------
// configuration
// ---------------------------------------------------------------------------
int resolve_cfg(int n, int dtype, const lqs_fuse_cfg* cfg, PlanCfg& pc, int* arith) {
  const int kmax = dtype == LQS_C64 ? 14 : 13;  // tile <= 128 KiB of shared memory
  pc.k = reg_tile_qubits(dtype);                  // the register-tile kernel's shape
  pc.b = dtype == LQS_C64 ? 5 : 4;
  pc.max_ops = kMaxTileOps;
  if (dtype == LQS_C64) pc.dense2_weight = 4;
  int ar = LQS_ARITH_AUTO;
  if (cfg) {
    if (cfg->tile_qubits) pc.k = cfg->tile_qubits;
    if (cfg->low_qubits) pc.b = cfg->low_qubits;
    if (cfg->max_ops) pc.max_ops = std::min<int>(cfg->max_ops, kMaxTileOps);
    ar = cfg->arith;
    if (ar != LQS_ARITH_AUTO && ar != LQS_ARITH_F64 && ar != LQS_ARITH_DF)
      return set_error(LQS_ERR_ARG, "cfg.arith must be LQS_ARITH_AUTO, LQS_ARITH_F64 or LQS_ARITH_DF");
  }
  if (pc.k < 3 || pc.k > kmax)
    return set_error(LQS_ERR_ARG, "tile_qubits must be in [3, " + std::to_string(kmax) + "]");
  const int bmin = dtype == LQS_C64 ? 1 : 0;  // bulk copies move multiples of 16 bytes
  if (pc.b < std::max(bmin, 1) || pc.b > pc.k - 2)
    return set_error(LQS_ERR_ARG, "low_qubits must be in [1, tile_qubits - 2]");
  if (pc.max_ops < 1) return set_error(LQS_ERR_ARG, "max_ops must be positive");
  ar = current_arith(ar);
  const bool f64 = dtype == LQS_C128 && ar == LQS_ARITH_F64;
  // multi-tile states whose segments run as compiled code
  if (n > reg_tile_qubits(dtype) && jit_enabled_for(n))
    pc.dense_cap = dtype == LQS_C64 ? LQS_SEGMENT_DENSE_CAP_C64 : f64 ? LQS_SEGMENT_DENSE_CAP_F64 : LQS_SEGMENT_DENSE_CAP;
  // complex128 only: another order of commuting gates rounds differently, far
  // below double precision but by up to the last float32 bit in complex64,
  // whose energies and gradients are to stay what program order gives.  Not for
  // the float64 policy either: its float64 pipe is the bound, and searched plans
  // trade passes for more diagonal products (LQS_SEGMENT_DENSE_CAP_F64)
  pc.search = dtype == LQS_C128 && !f64 && pc.dense_cap > 0 && pc.k == reg_tile_qubits(dtype);
  if (n <= pc.k) {  // the whole state is one tile
    pc.k = n;
    pc.b = n;
  }
  if (arith) *arith = ar;
  return LQS_OK;
}

static int coef_count(const KOp& o) {
  switch (o.kind) {
    case K_PHASE: return 1;
    case K_DIAG1: return 2;
    case K_ANTI1: return 2;
    case K_SWAP: return 0;
    case K_DENSE1: return 4;
    case K_DENSE1R: return 4;
    case K_DENSE2: return 16;
    case K_DIAG2: return 4;
  }
  return 0;
}

// ---------------------------------------------------------------------------
// planner
// ---------------------------------------------------------------------------
//
// A segment executes remaining ops that (1) commute with all earlier ops it
// leaves behind and (2) have their non-diagonal targets in the segment's tile.
// Diagonal ops and controls need no tile qubit.  Ops on disjoint wires
// commute; searched plans also let ops pass each other when every wire they
// share is one that both leave in the Z basis (controls, diagonal targets).
static int dense_weight(const KOp& o, int w2) {
  return o.kind == K_DENSE2 ? w2 : (o.kind == K_DENSE1 || o.kind == K_DENSE1R) ? 1 : 0;
}


namespace {
struct POp {
  uint64_t x, z;  // wires it must keep its order on / may pass other z wires on
  uint64_t t;     // qubits it needs in the tile
  int nc, dense;
};

// Of the first `look` remaining ops (indices `rem`, in order) those that one
// segment with tile Q executes; with `grow`, Q gains qubits in program order
// while it holds fewer than k.  Returns the weight of the executed
// ops.
int fill_segment(const std::vector<POp>& ops, const std::vector<int>& rem, size_t look, const PlanCfg& pc, int k,
                 uint64_t all, bool grow, uint64_t& Q, std::vector<int>* out) {
  uint64_t bx = 0, bz = 0;  // wires of the ops left behind
  int n_ops = 0, ncoef = 0, dense = 0, weight = 0;
  for (size_t j = 0; j < look && n_ops < pc.max_ops; ++j) {
    const int i = rem[j];
    const POp& o = ops[(size_t)i];
    if (!(o.x & (bx | bz)) && !(o.z & bx)) {
      const uint64_t need = o.t & ~Q;
      if ((!need || (grow && __builtin_popcountll(Q | need) <= k)) &&
          ncoef + o.nc <= kMaxTileCoef && (pc.dense_cap <= 0 || dense + o.dense <= pc.dense_cap || !n_ops)) {
        Q |= need;
        ++n_ops;
        ncoef += o.nc;
        dense += o.dense;
        weight += o.t ? 8 : 1;
        if (out) out->push_back(i);
        continue;
      }
    }
    bx |= o.x;
    bz |= o.z;
    if (bx == all) break;
  }
  return weight;
}

// One plan.  Without search each segment takes qubits in program order.  With
// it every window of neighbouring qubits is tried too, and the tile that
// executes the most is improved by exchanging one qubit at a time.  Layers
// with a CNOT ladder advance in skewed windows this way (half the qubits per
// layer, two to five layers per pass): 30-qubit 10-layer ansatz, complex128 33
// -> 27 passes (21 with a dense cap of 16) and 444 -> 418 ms; 24-qubit
// universal circuit 55 -> 23 and 6.29 -> 5.43 ms.  Tiles are weighed on the ops
// just ahead (1024: eleven layers of 30 qubits), so that the time of the search
// is proportional to the circuit's length.  The scan ends early only where every
// wire is blocked, and one that is only a control never is: 16000 ops on 30
// qubits with such a wire took 1.35 s on all ops, 0.24 s now.
constexpr size_t kLookAhead = 1024;
int make_plan(int n, const std::vector<POp>& ops, const PlanCfg& pc, bool search, std::vector<Segment>& segs) {
  const int k = std::min(pc.k, n), b = std::min(pc.b, k);
  const uint64_t all = n >= 64 ? ~0ull : ((1ull << n) - 1);
  const uint64_t low = b >= 64 ? ~0ull : ((1ull << b) - 1);
  auto padded = [&](uint64_t Q) {
    for (int q = b; q < n && __builtin_popcountll(Q) < k; ++q) Q |= 1ull << q;
    return Q;
  };
  std::vector<int> rem(ops.size());
  for (size_t i = 0; i < ops.size(); ++i) rem[i] = (int)i;
  segs.clear();
  while (!rem.empty()) {
    Segment seg;
    uint64_t Q = low;
    const size_t look = search ? std::min(rem.size(), kLookAhead) : rem.size();
    int best = fill_segment(ops, rem, look, pc, k, all, true, Q, search ? nullptr : &seg.ops);
    Q = padded(Q);
    if (search) {
      auto weigh = [&](uint64_t T) { return fill_segment(ops, rem, look, pc, k, all, false, T, nullptr); };
      best = std::max(best, weigh(Q));
      for (int s = b; s + (k - b) <= n; ++s) {
        const uint64_t T = low | (((1ull << (k - b)) - 1) << s);
        const int w = weigh(T);
        if (w > best) best = w, Q = T;
      }
      for (int round = 0; round < 4; ++round) {
        uint64_t top = Q;
        for (int i = b; i < n; ++i) {
          if (!((Q >> i) & 1)) continue;
          for (int j = b; j < n; ++j) {
            if ((Q >> j) & 1) continue;
            const uint64_t T = (Q & ~(1ull << i)) | (1ull << j);
            const int w = weigh(T);
            if (w > best) best = w, top = T;
          }
        }
        if (top == Q) break;
        Q = top;
      }
    }
    seg.qmask = Q;
    if (search) fill_segment(ops, rem, rem.size(), pc, k, all, false, Q, &seg.ops);
    if (seg.ops.empty()) return set_error(LQS_ERR_ARG, "internal: planner made no progress");
    std::vector<int> left;
    left.reserve(rem.size() - seg.ops.size());
    std::set_difference(rem.begin(), rem.end(), seg.ops.begin(), seg.ops.end(), std::back_inserter(left));
    rem.swap(left);
    segs.push_back(std::move(seg));
  }
  return LQS_OK;
}

// Plans with a search cost 2-20 ms of host time (300-900 ops), so they are
// kept by structure: everything the plan depends on, never an address.  At most
// 32 MiB of them (about 28 bytes per op), all given back at once when full.
constexpr size_t kMaxSearchedBytes = 32u << 20;
std::mutex g_search_mu;
size_t g_searched_bytes = 0;
std::unordered_map<std::string, std::vector<Segment>> g_searched;
}  // namespace

int plan_segments(int n, const std::vector<KOp>& ops, const PlanCfg& pc, std::vector<Segment>& segs) {
  std::vector<POp> po(ops.size());
  auto set_pass = [&](bool commute) {
    for (size_t i = 0; i < ops.size(); ++i) {
      const uint64_t t = ops[i].tile_mask(), w = ops[i].wire_mask();
      po[i] = POp{commute ? t : w, commute ? w & ~t : 0, t, coef_count(ops[i]), dense_weight(ops[i], pc.dense2_weight)};
    }
  };
  set_pass(false);
  if (!pc.search) return make_plan(n, po, pc, false, segs);
  std::string key;
  const int hdr[5] = {n, pc.k, pc.b, pc.max_ops, pc.dense_cap};
  key.append(reinterpret_cast<const char*>(hdr), sizeof hdr);
  for (const POp& o : po) {
    const uint64_t rec[3] = {o.x, o.t, (uint64_t)o.nc << 32 | (uint64_t)o.dense};
    key.append(reinterpret_cast<const char*>(rec), sizeof rec);
  }
  {
    std::lock_guard<std::mutex> lk(g_search_mu);
    auto it = g_searched.find(key);
    if (it != g_searched.end()) {
      segs = it->second;
      return LQS_OK;
    }
  }
  LQS_TRY(make_plan(n, po, pc, false, segs));
  if (segs.size() > 1) {
    std::vector<Segment> alt;
    set_pass(true);
    LQS_TRY(make_plan(n, po, pc, true, alt));
    if (alt.size() < segs.size()) segs.swap(alt);
  }
  size_t bytes = key.size() + 64;
  for (const Segment& s : segs) bytes += sizeof s + s.ops.size() * sizeof s.ops[0];
  if (bytes > kMaxSearchedBytes) return LQS_OK;
  std::lock_guard<std::mutex> lk(g_search_mu);
  if (g_searched_bytes + bytes > kMaxSearchedBytes) {
    g_searched.clear();
    g_searched_bytes = 0;
  }
  if (g_searched.emplace(std::move(key), segs).second) g_searched_bytes += bytes;
  return LQS_OK;
}

// ---------------------------------------------------------------------------
// tile program construction
// ---------------------------------------------------------------------------
static TileGeom make_tile_geom(int n, uint64_t Q, int k, int b, size_t amp_bytes) {
  TileGeom G{};
  G.n = n;
  G.k = k;
  G.b = b;
  G.r = 0;
  for (int q = b; q < n; ++q)
    if ((Q >> q) & 1) G.h[G.r++] = q;
  G.ntiles = 1ull << (n - k);
  G.row_bytes = (uint32_t)(amp_bytes << b);
  return G;
}

static int local_pos(const TileGeom& G, int q) {
  if (q < 0) return -1;
  if (q < G.b) return q;
  for (int m = 0; m < G.r; ++m)
    if (G.h[m] == q) return G.b + m;
  return -1;
}

template <class A>
static typename A::C cc(const KOp& op, int i) { return A::cconst(op.m[2 * i], op.m[2 * i + 1]); }

template <class A>
int add_tile_op(TileProg<A>& P, const KOp& o, int gslot) {
  if (P.nops >= kMaxTileOps) return set_error(LQS_ERR_ARG, "internal: tile program full");
  const TileGeom& G = P.g;
  TOp t{};
  t.kind = (uint8_t)o.kind;
  t.special = (uint8_t)o.special;
  t.gen = (uint8_t)o.gen;
  t.gslot = (int16_t)gslot;
  t.l0 = (int8_t)local_pos(G, o.t0);
  t.l1 = (int8_t)local_pos(G, o.t1);
  if (!o.diagonal() && ((o.t0 >= 0 && t.l0 < 0) || (o.t1 >= 0 && t.l1 < 0)))
    return set_error(LQS_ERR_ARG, "internal: non-diagonal target outside the tile");
  if (o.t0 >= 0 && t.l0 < 0) t.e0 = 1ull << o.t0;
  if (o.t1 >= 0 && t.l1 < 0) t.e1 = 1ull << o.t1;
  int fix[6], nfix = 0;
  for (int q = 0; q < G.n; ++q) {
    if (!((o.cmask >> q) & 1)) continue;
    const int lp = local_pos(G, q);
    if (lp >= 0) {
      t.lcmask |= 1u << lp;
      fix[nfix++] = lp;
    } else {
      t.ecmask |= 1ull << q;
    }
  }
  // diagonal ops with a local target enumerate pairs (K_DIAG1) over it; K_DIAG2
  // and K_PHASE enumerate single amplitudes
  const bool pair_target = o.kind != K_PHASE && o.kind != K_DIAG2 && !(o.kind == K_DIAG1 && t.l0 < 0);
  if (pair_target) {
    if (t.l0 >= 0) fix[nfix++] = t.l0;
    if (t.l1 >= 0 && o.kind != K_DIAG1) fix[nfix++] = t.l1;
  }
  if (nfix > 4) return set_error(LQS_ERR_ARG, "internal: more than 4 fixed tile bits");
  std::sort(fix, fix + nfix);
  t.nfix = (uint8_t)nfix;
  for (int i = 0; i < nfix; ++i) t.fix[i] = (uint8_t)fix[i];
  const int nc = coef_count(o);
  if (P.ncoef + nc > kMaxTileCoef) return set_error(LQS_ERR_ARG, "internal: tile coefficient pool full");
  t.coef = (int16_t)P.ncoef;
  for (int i = 0; i < nc; ++i) P.coef[P.ncoef + i] = (o.kind == K_DENSE1R) ? A::cconst(o.m[i], 0.0) : cc<A>(o, i);
  P.ncoef += nc;
  // an uncontrolled real 2x2 with m11 = s m00 and m10 = -s m01 (s = +1:
  // rotations such as RY, special 1; s = -1: reflections such as H, special 2)
  // is g times an orthogonal matrix: compiled segments apply it in a cheaper
  // form (the interpreter ignores the mark).  Special 3: the Hadamard pattern
  // m00 = m01 = m10 = -m11 > 0, sums and differences only.
  if (o.kind == K_DENSE1R && o.cmask == 0) {
    if (o.m[3] == o.m[0] && o.m[2] == -o.m[1]) t.special = 1;
    else if (o.m[0] > 0.0 && o.m[1] == o.m[0] && o.m[2] == o.m[0] && o.m[3] == -o.m[0]) t.special = 3;
    else if (o.m[3] == -o.m[0] && o.m[2] == o.m[1]) t.special = 2;
  }
  P.op[P.nops++] = t;
  return LQS_OK;
}

template <class A>
void init_prog(TileProg<A>& P, int n, uint64_t Q, int k, int b) {
  P.g = make_tile_geom(n, Q, k, b, (size_t)A::kAmpBytes);
  P.nops = 0;
  P.ncoef = 0;
  P.ngrad = 0;
  P.nfold = 0;
}

// ---------------------------------------------------------------------------
// the fused kernel: persistent CTAs, one tile in shared memory per CTA
// ---------------------------------------------------------------------------
template <class A>
__global__ void __launch_bounds__(kTileThreads) k_fused(typename A::S* __restrict__ psi,
                                                        const __grid_constant__ TileProg<A> P, int* status) {
  using S = typename A::S;
  using W = typename A::W;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  const TileGeom& G = P.g;
  const uint32_t nt = 1u << G.k;
  S* buf = reinterpret_cast<S*>(smem_raw);
  W* T = reinterpret_cast<W*>(smem_raw);
  uint64_t* bar = reinterpret_cast<uint64_t*>(smem_raw + (size_t)nt * sizeof(S));
  if (threadIdx.x == 0) {
    mbar_init(bar, 1);
    fence_mbar_init();
  }
  __syncthreads();
  uint32_t phase = 0;
  bool ok = true;
  for (uint64_t t = blockIdx.x; t < G.ntiles; t += gridDim.x) {
    const uint64_t base = tile_base(G, t);
    if (threadIdx.x < 32) tile_load_issue(G, buf, psi, base, bar);
    ok = __syncthreads_and(mbar_wait(bar, phase));
    phase ^= 1u;
    if (!ok) break;
    if constexpr (!std::is_same<S, W>::value) {
      for (uint32_t j = threadIdx.x; j < nt; j += blockDim.x) {
        const S s = buf[j];
        T[j] = A::load(s);
      }
      __syncthreads();
    }
    for (int i = 0; i < P.nops; ++i) {
      tile_apply<A>(T, P.op[i], P.coef, base, G.k);
      __syncthreads();
    }
    if constexpr (!std::is_same<S, W>::value) {
      for (uint32_t j = threadIdx.x; j < nt; j += blockDim.x) {
        const W w = T[j];
        buf[j] = A::store(w);
      }
    }
    fence_proxy_async();
    __syncthreads();
    if (threadIdx.x < 32) tile_store_issue(G, psi, buf, base);
  }
  if (threadIdx.x < 32) bulk_wait0();
  if (!ok) {
    if (threadIdx.x == 0) {
      flag_timeout(status, 1);
      mbar_wait(bar, phase ^ 1u);  // let the load in flight land before the CTA exits (bounded)
    }
  }
}

template <class A>
static int launch_fused_t(SV* sv, const std::vector<KOp>& ops, const Segment& seg, const PlanCfg& pc, int arith) {
  const int n = sv->n, k = std::min(pc.k, n), b = std::min(pc.b, k);
  static thread_local TileProg<A> P;  // ~14 KB: keep it off the stack
  init_prog(P, n, seg.qmask, k, b);
  for (int i : seg.ops) LQS_TRY(add_tile_op(P, ops[i], -1));
  const size_t smem = ((size_t)sizeof(typename A::S) << k) + 16;
  static bool attr_done = false;
  if (!attr_done) {
    LQS_CUDA_TRY(cudaFuncSetAttribute(k_fused<A>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024));
    attr_done = true;
  }
  int per_sm = 0;
  LQS_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_fused<A>, kTileThreads, smem));
  per_sm = std::max(per_sm, 1);
  const uint64_t grid = std::min<uint64_t>(P.g.ntiles, (uint64_t)std::max(sv->sms, 1) * per_sm);
  double flops = 0.0;
  for (int i : seg.ops) flops += kop_touched_fraction(ops[i]) * kop_flops_per_amp(ops[i]);
  const std::string pname = std::string("k_fused/") + arith_tag(sv->dtype, arith);
  ProfScope ps(sv->stream, pname.c_str(), 2.0 * (double)sv->bytes(), flops * (double)sv->N());
  k_fused<A><<<(unsigned)grid, kTileThreads, smem, sv->stream>>>(static_cast<typename A::S*>(sv->d), P, sv->d_status);
  count_launch();
  LQS_CUDA_TRY(cudaGetLastError());
  return LQS_OK;
}

int launch_segment(SV* sv, const std::vector<KOp>& ops, const Segment& seg, const PlanCfg& pc, int arith,
                   unsigned fmt) {
  const int k = std::min(pc.k, sv->n), b = std::min(pc.b, k);
  if (fmt) return launch_fused_reg(sv, ops, seg, k, b, arith, fmt);  // checked by seg_split_capable
  // A lone gate is cheaper as a plain pass: it only touches the amplitudes it changes.
  if (seg.ops.size() == 1) return launch_gate(sv, ops[seg.ops[0]], arith);
  if (k == reg_tile_qubits(sv->dtype)) {
    const int rc = launch_fused_reg(sv, ops, seg, k, b, arith);
    if (rc != LQS_ERR_UNSUPPORTED) return rc;
    // the register program (gates plus layout changes) overflowed: split the
    // segment in two, keeping the order of its gates
    Segment lo, hi;
    lo.qmask = hi.qmask = seg.qmask;
    lo.ops.assign(seg.ops.begin(), seg.ops.begin() + seg.ops.size() / 2);
    hi.ops.assign(seg.ops.begin() + seg.ops.size() / 2, seg.ops.end());
    LQS_TRY(launch_segment(sv, ops, lo, pc, arith));
    return launch_segment(sv, ops, hi, pc, arith);
  }
  if (sv->dtype == LQS_C64) return launch_fused_t<ArF32>(sv, ops, seg, pc, arith);
  if (arith == LQS_ARITH_F64) return launch_fused_t<ArF64>(sv, ops, seg, pc, arith);
  return launch_fused_t<ArDF>(sv, ops, seg, pc, arith);
}

// Mirrors launch_segment's routing and splitting without launching: each
// register-tile program the segment will run is noted for the segment
// compiler (and queued for compilation when the mode asks, or `force`).
int jit_collect(int n, int dtype, int arith, const std::vector<KOp>& ops, const Segment& seg, const PlanCfg& pc,
                bool force, std::vector<void*>& todo) {
  if (seg.ops.size() == 1) return LQS_OK;
  const int k = std::min(pc.k, n), b = std::min(pc.b, k);
  if (k != reg_tile_qubits(dtype)) return LQS_OK;
  const int rc = note_reg_prog(n, dtype, arith, ops, seg, k, b, force, todo);
  if (rc != LQS_ERR_UNSUPPORTED) return rc;
  Segment lo, hi;
  lo.qmask = hi.qmask = seg.qmask;
  lo.ops.assign(seg.ops.begin(), seg.ops.begin() + seg.ops.size() / 2);
  hi.ops.assign(seg.ops.begin() + seg.ops.size() / 2, seg.ops.end());
  LQS_TRY(jit_collect(n, dtype, arith, ops, lo, pc, force, todo));
  return jit_collect(n, dtype, arith, ops, hi, pc, force, todo);
}

// explicit instantiations used by the measurement kernels
template int add_tile_op<ArF32>(TileProg<ArF32>&, const KOp&, int);
template int add_tile_op<ArF64>(TileProg<ArF64>&, const KOp&, int);
template int add_tile_op<ArDF>(TileProg<ArDF>&, const KOp&, int);
template void init_prog<ArF32>(TileProg<ArF32>&, int, uint64_t, int, int);
template void init_prog<ArF64>(TileProg<ArF64>&, int, uint64_t, int, int);
template void init_prog<ArDF>(TileProg<ArDF>&, int, uint64_t, int, int);

}  // namespace lqs

namespace lqs {

// One thread waits, with the kernels' bounded wait, on a shared-memory barrier
// that expects one arrival and never gets it; the wait gives up and flags the
// status exactly as a tile load that never landed would.  No copy is issued.
__global__ void k_wait_for_nothing(int* status) {
  __shared__ __align__(8) uint64_t bar;
  mbar_init(&bar, 1);
  fence_mbar_init();
  if (!mbar_wait(&bar, 0)) flag_timeout(status, 16);
}

}  // namespace lqs

extern "C" int lqs_check_bounded_wait(lqs_sv* h) {
  void* dptr = nullptr;
  int n = 0, dtype = 0;
  LQS_TRY(lqs_sv_info(h, &dptr, &n, &dtype));  // validates the handle
  lqs::SV* sv = reinterpret_cast<lqs::SV*>(h);
  lqs::k_wait_for_nothing<<<1, 1, 0, sv->stream>>>(sv->d_status);
  LQS_CUDA_TRY(cudaGetLastError());
  lqs::count_launch();
  return LQS_OK;
}
