// Jump-forward forced spans (GRID Sec. 6.1, step 6 of the per-token hot
// path): while a row's mask admits exactly one token id, that token is
// forced; it is appended to the row's span and the row is advanced by it,
// without sampling.  Everything runs on the device: a decoding step per span
// position (the mask step fed with the forced tokens), whose packing kernel
// finds each row's next forced token or stops the row.  A row that has stopped
// is left out of the later steps, whose blocks for it end at once: most rows
// stop at the first position, and masking them anew at each of max_span
// positions cost 480 us of nine whole steps (32 SQL rows, V = 32,000,
// max_span 8) where this takes 120 us.

#include <cstring>

#include "grid_state.cuh"

namespace grid {
namespace {

// aux layout (B ints each): tok, stop
__global__ void k_force_init(int32_t* __restrict__ span, int32_t* __restrict__ span_len, int32_t* __restrict__ aux,
                             int B, int max_span) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < B * max_span) span[i] = -1;
  if (i < B) {
    span_len[i] = 0;
    aux[i] = -1;
    aux[B + i] = 0;
  }
}

}  // namespace
}  // namespace grid

using namespace grid;

extern "C" int grid_forced_span(const grid_spec* s, grid_configs* c, int32_t max_span, uint32_t* d_mask,
                                int32_t* d_span, int32_t* d_span_len, int32_t* d_status, uint8_t* d_records,
                                void* stream) {
  if (!s || !c || !d_mask || (!d_span && max_span > 0) || !d_span_len || !d_status || max_span < 0 || max_span > 4096)
    return set_error(GRID_E_INVALID_ARG, "grid_forced_span: bad arguments");
  const bool audit = c->c.hs != nullptr;
  if (audit != (d_records != nullptr) && max_span > 0)
    return set_error(GRID_E_INVALID_ARG, audit ? "grid_forced_span: audit is on: pass the records of the forced tokens"
                                               : "grid_forced_span: records given but audit is not enabled");
  cudaStream_t st = (cudaStream_t)stream;
  const int B = c->B;
  const MaskScratch m{c->ctx, c->rng, c->sel, c->verd0, c->verd1, c->A2, c->vcbits,
                      c->surv, c->vsurv, c->cap, c->vcap, c->words_v};
  const int n = std::max(B * std::max(max_span, 1), B);
  k_force_init<<<(n + 255) / 256, 256, 0, st>>>(d_span, d_span_len, c->aux, B, max_span);
  GRID_CUDA(cudaGetLastError());
  int rc;
  for (int pos = 0; pos <= max_span; ++pos) {
    // the step at span position pos, fed with the tokens that the step before forced (rows without one are left out)
    const AdvArgs adv{c->c, c->aux, 1, 0, c->aux + B};
    const ForceArgs force{d_span, d_span_len, c->aux, c->aux + B, pos, max_span};
    if ((rc = launch_masks(s, c->c, m, B, d_mask, d_status, st, nullptr, FusedLogits(), pos > 0 ? &adv : nullptr,
                           pos < max_span ? &force : nullptr)))
      return rc;
    // every interior token of a span is audited (kind 1), at the configuration
    // its mask was computed at, before the advance
    if (audit && pos < max_span &&
        (rc = audit_append(s, c, d_mask, c->aux, 1u, d_records + (size_t)pos * 80, (long long)max_span * 80, st)))
      return rc;
  }
  GRID_CUDA(cudaGetLastError());
  return GRID_OK;
}

// ---------------------------------------------------------------------------
// Token-denominated reserve (GRID Sec. 5, Prop. 9, Termination; Sec. 6.1
// step 3): per row, the cheapest legal completion of the output plus EOS,
// counted in vocabulary tokens, so that a decoding loop whose remaining
// budget falls to that count plus a safety margin writes it instead of
// sampling.  The cost model is the paper's: every terminal of a completion
// is written as a fixed rendering (a blank and the terminal's lexeme, split
// greedily into vocabulary tokens), so a completion costs the sum of its
// terminals' rendering lengths; the pending lexeme is either ended as it
// stands (by the blank, or by the state's separator byte) or first extended,
// byte by byte, to the shortest lexeme of one terminal.  The cheapest
// terminal completion of a stack is found exactly over the LR(0) items:
// completing kernel item [A -> alpha . beta] of the top state costs beta's
// cheapest yield and leaves the stack with alpha popped and the goto on A
// pushed; every completion decomposes into such steps, and they only lower
// the stack (or keep its height, for |alpha| = 1), so one pass over the
// heights from the top down, with a fixpoint at each height, settles all
// costs.

namespace grid {
namespace {

constexpr uint32_t kInf = 0x3FFFFFFFu;
constexpr int kReserveEntries = 4096;  // search entries per row
constexpr int kMaxExt = 64;            // bytes of a pending-lexeme extension

struct REnt {
  int32_t level, state, cost, parent, item, next;
};

// The stack base[0:keep] ++ ovl[0:m].
struct VStack {
  const uint16_t* base;
  int keep;
  const uint16_t* ovl;
  int m;
  __device__ int at(int i) const { return i < keep ? base[i] : ovl[i - keep]; }
  __device__ int size() const { return keep + m; }
};

// The cheapest terminal completion of `vs` (in rendering tokens), or kInf;
// on success goal_e / goal_item name its last step.
template <class T>
__device__ uint32_t reserve_search(const T& t, const ReserveTables& rt, const VStack& vs, REnt* ent,
                                   int32_t* head, int& goal_e, int& goal_item, bool& overflow) {
  const int kmax = vs.size() - 1;
  goal_e = goal_item = -1;
  if (kmax >= t.D) {  // one level head per stack position: D of them
    overflow = true;
    return kInf;
  }
  for (int k = 0; k <= kmax; ++k) head[k] = -1;
  int cnt = 0;
  overflow = false;
  auto insert = [&](int level, int state, uint32_t cost, int parent, int item) -> bool {
    for (int e = head[level]; e >= 0; e = ent[e].next)
      if (ent[e].state == state) {
        if (cost >= (uint32_t)ent[e].cost) return false;
        ent[e].cost = (int32_t)cost;
        ent[e].parent = parent;
        ent[e].item = item;
        return true;
      }
    if (cnt >= rt.E) {
      overflow = true;
      return false;
    }
    ent[cnt] = REnt{level, state, (int32_t)cost, parent, item, head[level]};
    head[level] = cnt++;
    return true;
  };
  insert(kmax, vs.at(kmax), 0u, -1, -1);
  uint32_t best = kInf;
  goal_e = goal_item = -1;
  for (int k = kmax; k >= 0; --k) {
    // steps that keep the height (|alpha| = 1), to a fixpoint; the goal
    for (int round = 0; round <= t.S; ++round) {
      bool changed = false;
      for (int e = head[k]; e >= 0; e = ent[e].next) {
        const int s = ent[e].state;
        const uint32_t c0 = (uint32_t)ent[e].cost;
        for (int i = rt.item_off[s]; i < rt.item_off[s + 1]; ++i) {
          const uint32_t ic = rt.item_cost[i];
          if (ic >= kInf) continue;
          const int p = rt.item_p[i], d = rt.item_d[i];
          const uint32_t c = c0 + ic;
          if (p == 0) {  // S' -> . start at height 0, S' -> start . at height 1: the sentence is complete
            if (((d == 0 && k == 0) || (d == 1 && k == 1)) && c < best) {
              best = c;
              goal_e = e;
              goal_item = i;
            }
            continue;
          }
          if (d != 1 || k < 1) continue;
          const int g = t.gto(vs.at(k - 1) * t.NNT + t.lhs(p));
          if (g >= t.S) continue;
          if (insert(k, g, c, e, i)) changed = true;
        }
      }
      if (!changed) break;
    }
    // steps that lower the stack (|alpha| >= 2)
    for (int e = head[k]; e >= 0; e = ent[e].next) {
      const int s = ent[e].state;
      const uint32_t c0 = (uint32_t)ent[e].cost;
      for (int i = rt.item_off[s]; i < rt.item_off[s + 1]; ++i) {
        const int p = rt.item_p[i], d = rt.item_d[i];
        const uint32_t ic = rt.item_cost[i];
        if (p == 0 || d < 2 || d > k || ic >= kInf) continue;
        const int g = t.gto(vs.at(k - d) * t.NNT + t.lhs(p));
        if (g >= t.S) continue;
        insert(k - d + 1, g, c0 + ic, e, i);
      }
    }
  }
  return best;
}

// The tokens rendering terminal x (one warp lane writes).
__device__ void put_terminal(const ReserveTables& rt, int x, int32_t* out, int cap, int& n) {
  for (int j = rt.rend_off[x]; j < rt.rend_off[x + 1]; ++j) {
    if (n < cap) out[n] = rt.rend_tok[j];
    ++n;
  }
}

struct ReserveArgs {
  int32_t* scratch;
  size_t scratch_ints;
  int32_t *d_cost, *d_tokens;
  int cap;
  int32_t* d_status;
  const int32_t* d_budget;
  int safety;
  int32_t* d_fire;
};

// One thread per row: evaluates the ways to end the pending lexeme (option 0:
// as it stands; option 1 + tau: extended to tau's shortest lexeme) and keeps
// the cheapest, then writes its tokens.  For rows whose search is larger than
// the warps' shared memory (k_reserve).
template <class T>
__device__ __noinline__ void reserve_serial(const T& t, const T& ts, const ReserveTables& rt,
                                            const DevConfigs& c, const ReserveArgs& ra, int b) {
  int32_t* const scratch = ra.scratch;
  const size_t scratch_ints = ra.scratch_ints;
  int32_t *const d_cost = ra.d_cost, *const d_tokens = ra.d_tokens, *const d_status = ra.d_status,
               *const d_fire = ra.d_fire;
  const int32_t* const d_budget = ra.d_budget;
  const int cap = ra.cap, safety = ra.safety;
  REnt* ent = reinterpret_cast<REnt*>(scratch + (size_t)b * scratch_ints);
  int32_t* head = scratch + (size_t)b * scratch_ints + (size_t)rt.E * (sizeof(REnt) / 4);
  int32_t* out = d_tokens + (size_t)b * cap;
  const int depth = c.depth[b], q = c.q[b], lx = c.lx[b];
  const uint16_t* base = c.stack + (size_t)b * t.D;
  int status = GRID_ST_OK, n = 0;
  uint32_t total_best = kInf;
  if (c.flags[b] & 1) {
    status = GRID_ST_COMPLETE;
  } else {
    const int mc = max_chain_of(t);
    const uint32_t pc0 = lx >= 0 ? t.lx_pcats[lx] : 0u, wc0 = lx >= 0 ? t.lx_wcats[lx] : 0u;
    const Bits4 live0 = q == kStart ? Bits4::zero() : live_prime(ts, q, pc0);
    uint16_t lo[kMaxOvl], ls[kMaxOvl];
    uint8_t y[kMaxExt];
    int best_opt = -1;
    bool any_overflow = false;
    // builds option `opt` into (vs, y, ylen, sep); false when it does not apply
    auto build = [&](int opt, VStack& vs, int& ylen, int& sep) -> bool {
      ylen = 0;
      sep = ' ';
      if (q == kStart) {
        if (opt != 0) return false;
        vs = VStack{base, depth, lo, 0};
        return true;
      }
      int q2 = q, lx2 = lx;
      uint32_t pc = pc0, wc = wc0;
      if (opt > 0) {  // extend the lexeme to terminal tau's shortest lexeme
        const int tau = opt - 1;
        if (tau >= t.n_term || t.ign.has(tau) || !live0.has(tau)) return false;
        int cat = -1;
        for (int k = 0; k < t.n_cat; ++k)
          if (t.cat_term[k] == tau) cat = k;
        int len;
        if (cat >= 0) {
          if (lx < 0) return false;
          len = rt.lx_wdist[(size_t)lx * rt.NC + cat];
          if (len == 0xFFFF) return false;
        } else {
          len = rt.dfa_tdist[(size_t)q * t.T1 + tau];
          if (len == 0xFF) return false;
        }
        if (len == 0 || len > kMaxExt) return false;  // len 0: the lexeme as it stands (option 0)
        for (int i = 0; i < len; ++i) {
          const int by = cat >= 0 ? rt.lx_wbyte[(size_t)lx2 * rt.NC + cat] : rt.dfa_tbyte[(size_t)q2 * t.T1 + tau];
          const int nq = ts.nxt(q2 * ts.C + ts.cls(by));
          if (nq == kDead) return false;
          q2 = nq;
          lx2 = lex_step(ts, q2, lx2, by, pc, wc);
          if (cat >= 0 && lx2 < 0) return false;
          y[ylen++] = (uint8_t)by;
        }
      } else if (opt != 0) {
        return false;
      }
      sep = rt.sep_byte[q2];
      if (sep < 0) return false;
      Walker w;
      walker_init(w, LArr{lo, 1}, LArr{ls, 1}, kMaxOvl, base, depth, nullptr, 0, q2, lx2, pc, wc, nullptr, nullptr);
      if (emit(ts, w, mc) <= 0) return false;
      vs = VStack{base, w.keep, lo, w.m};
      return true;
    };
    auto total_of = [&](uint32_t C, int ylen, int sep) -> uint32_t {
      if (C >= kInf) return kInf;
      // the blank that ends the lexeme comes with the first rendering; another
      // separator is a token of its own, needed only before a rendering
      return (uint32_t)ylen + ((C > 0 && sep != ' ') ? 1u : 0u) + C + 1u;
    };
    for (int opt = 0; opt <= t.n_term; ++opt) {
      VStack vs;
      int ylen, sep;
      if (!build(opt, vs, ylen, sep)) continue;
      bool ok = true;
      for (int i = 0; i < ylen && ok; ++i) ok = rt.byte_tok[y[i]] >= 0;
      if (!ok) continue;
      int ge, gi;
      bool of;
      const uint32_t C = reserve_search(ts, rt, vs, ent, head, ge, gi, of);
      any_overflow |= of;
      if (C > 0 && C < kInf && sep != ' ' && rt.byte_tok[sep] < 0) continue;
      const uint32_t tot = total_of(C, ylen, sep);
      if (tot < total_best) {
        total_best = tot;
        best_opt = opt;
      }
    }
    if (best_opt < 0) {
      status = any_overflow ? GRID_ST_BOUND : GRID_ST_NONVIABLE;
    } else {
      // the chosen option again, and its tokens
      VStack vs;
      int ylen, sep, ge, gi;
      bool of;
      build(best_opt, vs, ylen, sep);
      const uint32_t C = reserve_search(ts, rt, vs, ent, head, ge, gi, of);
      for (int i = 0; i < ylen; ++i) {
        if (n < cap) out[n] = rt.byte_tok[y[i]];
        ++n;
      }
      if (C > 0 && sep != ' ') {
        if (n < cap) out[n] = rt.byte_tok[sep];
        ++n;
      }
      // the steps in order: reverse the parent chain from the goal entry
      int prev = -1, cur = ge;
      while (cur >= 0) {
        const int nx = ent[cur].parent;
        ent[cur].parent = prev;
        prev = cur;
        cur = nx;
      }
      auto put_item = [&](int i) {
        const int p = rt.item_p[i], d = rt.item_d[i];
        for (int j = rt.prod_off[p] + d; j < rt.prod_off[p + 1]; ++j) {
          const int X = rt.prod_rhs[j];
          if (X < t.T1) {
            put_terminal(rt, X, out, cap, n);
          } else {
            for (int k = rt.ny_off[X - t.T1]; k < rt.ny_off[X - t.T1 + 1]; ++k) put_terminal(rt, rt.ny[k], out, cap, n);
          }
        }
      };
      for (int e = prev; e >= 0; e = ent[e].parent)  // prev: the start entry, which has no step
        if (ent[e].item >= 0) put_item(ent[e].item);
      put_item(gi);
      if (n < cap) out[n] = t.eos;
      ++n;
      if (n > cap) status = GRID_ST_BOUND;
    }
  }
  for (int i = n; i < cap; ++i) out[i] = -1;
  d_cost[b] = status == GRID_ST_OK || (status == GRID_ST_BOUND && total_best < kInf) ? (int32_t)total_best : -1;
  if (status == GRID_ST_COMPLETE) d_cost[b] = 0;
  d_status[b] = status;
  if (d_fire) d_fire[b] = (status == GRID_ST_OK && d_budget && d_budget[b] <= (int)total_best + safety) ? 1 : 0;
}

// ---- the same search on the warps of a block, in shared memory
//
// One warp per way to end the pending lexeme.  What bounds a search is its
// chain of entries: each is visited in the order of the serial search (an
// entry's place in its level's list, and the first of equal costs, decide
// which completion is written), its items one per lane.  Of the lanes that
// reach one state the cheapest, then the first, is inserted, at the place of
// the first of them.  An entry is visited again only after its cost fell: any
// other visit would insert nothing.
constexpr int kRsvWarps = 8;
constexpr int kRsvEnt = 384;     // entries per warp (more: reserve_serial)
constexpr int kRsvDepth = 1024;  // stack entries (more: reserve_serial)
constexpr int kRsvNone = 0xFFFF;

struct RsvWarp {
  int32_t cost[kRsvEnt], done[kRsvEnt];  // done: the cost an entry was visited with
  uint16_t state[kRsvEnt], next[kRsvEnt], parent[kRsvEnt], item[kRsvEnt];
  uint16_t head[kRsvDepth + kMaxOvl];
  uint16_t lo[kMaxOvl], ls[kMaxOvl];
  uint8_t y[kMaxExt];
};

// k_reserve's dynamic shared memory, for the largest staged tables
constexpr int kRsvSmem = kMaxStage + kRsvWarps * (int)sizeof(RsvWarp);
static_assert(kRsvSmem + 4096 <= 227 * 1024 && sizeof(RsvWarp) % 16 == 0, "the warps' search spaces fit");

// A way to end the pending lexeme: the stack base[0:keep] ++ lo[0:m] it
// leaves, its extension's length and the separator.
struct RsvOption {
  bool ok;
  int keep, m, ylen, sep;
};

struct RsvGoal {
  uint32_t cost;
  int e, item;
  bool full;  // more entries than a warp holds
};

__device__ __forceinline__ int rsv_at(const uint16_t* base, const RsvOption& o, const RsvWarp& w, int i) {
  return i < o.keep ? base[i] : w.lo[i - o.keep];
}

// reserve_search on one warp.
template <class T>
__device__ RsvGoal rsv_search(const T& t, const ReserveTables& rt, const uint16_t* base, const RsvOption& o,
                              RsvWarp& w, int lane) {
  RsvGoal goal{kInf, -1, -1, false};
  const int kmax = o.keep + o.m - 1;
  int cnt = 0;
  for (int k = lane; k <= kmax; k += 32) w.head[k] = kRsvNone;
  __syncwarp();
  // the same in every lane; lane 0 writes
  auto insert = [&](int level, int state, uint32_t cost, int parent, int item) -> bool {
    const int h = w.head[level];
    int e = h;
    while (e != kRsvNone && w.state[e] != state) e = w.next[e];
    if (e != kRsvNone) {
      if (cost >= (uint32_t)w.cost[e]) return false;
      __syncwarp();
      if (lane == 0) {
        w.cost[e] = (int32_t)cost;
        w.parent[e] = (uint16_t)parent;
        w.item[e] = (uint16_t)item;
      }
    } else {
      if (cnt == kRsvEnt) {
        goal.full = true;
        return false;
      }
      __syncwarp();
      if (lane == 0) {
        w.cost[cnt] = (int32_t)cost;
        w.done[cnt] = -1;
        w.state[cnt] = (uint16_t)state;
        w.next[cnt] = (uint16_t)h;
        w.parent[cnt] = (uint16_t)parent;
        w.item[cnt] = (uint16_t)item;
        w.head[level] = (uint16_t)cnt;
      }
      ++cnt;
    }
    __syncwarp();
    return true;
  };
  // the lanes' candidates (key: level << 16 | state, or -1), in item order
  auto insert_all = [&](int key, uint32_t c, int e, int item) -> bool {
    bool changed = false;
    uint32_t todo = __ballot_sync(0xffffffffu, key >= 0);
    while (todo) {
      const int k0 = __shfl_sync(0xffffffffu, key, __ffs(todo) - 1);
      const uint32_t same = __ballot_sync(0xffffffffu, key == k0);
      const uint32_t low = __reduce_min_sync(0xffffffffu, key == k0 ? c : 0xFFFFFFFFu);
      const int l = __ffs(__ballot_sync(0xffffffffu, key == k0 && c == low)) - 1;
      changed |= insert(k0 >> 16, k0 & 0xFFFF, low, e, __shfl_sync(0xffffffffu, item, l));
      todo &= ~same;
    }
    return changed;
  };
  insert(kmax, rsv_at(base, o, w, kmax), 0u, kRsvNone, kRsvNone);
  for (int k = kmax; k >= 0 && !goal.full; --k) {
    const int below = k >= 1 ? rsv_at(base, o, w, k - 1) : 0;
    // steps that keep the height (|alpha| = 1), to a fixpoint; the goal
    for (int round = 0; round <= t.S; ++round) {
      bool changed = false;
      for (int e = w.head[k]; e != kRsvNone; e = w.next[e]) {
        const int s = w.state[e];
        const uint32_t c0 = (uint32_t)w.cost[e];
        if (w.done[e] == (int32_t)c0) continue;
        __syncwarp();
        if (lane == 0) w.done[e] = (int32_t)c0;
        __syncwarp();
        const int i1 = __ldg(&rt.item_off[s + 1]);
        for (int i0 = __ldg(&rt.item_off[s]); i0 < i1; i0 += 32) {
          const int i = i0 + lane;
          uint32_t c = kInf;
          int p = -1, d = 0, key = -1;
          if (i < i1) {
            const uint32_t ic = __ldg(&rt.item_cost[i]);
            p = __ldg(&rt.item_p[i]);
            d = __ldg(&rt.item_d[i]);
            if (ic < kInf) c = c0 + ic;
          }
          // S' -> . start at height 0, S' -> start . at height 1: the sentence is complete
          const bool fin = c < kInf && p == 0 && ((d == 0 && k == 0) || (d == 1 && k == 1));
          if (__any_sync(0xffffffffu, fin)) {
            const uint32_t low = __reduce_min_sync(0xffffffffu, fin ? c : 0xFFFFFFFFu);
            const int l = __ffs(__ballot_sync(0xffffffffu, fin && c == low)) - 1;
            if (low < goal.cost) {
              goal.cost = low;
              goal.e = e;
              goal.item = i0 + l;
            }
          }
          if (c < kInf && p > 0 && d == 1 && k >= 1) {
            const int g = t.gto(below * t.NNT + t.lhs(p));
            if (g < t.S) key = (k << 16) | g;
          }
          changed |= insert_all(key, c, e, i);
        }
      }
      if (!changed) break;
    }
    // steps that lower the stack (|alpha| >= 2)
    for (int e = w.head[k]; e != kRsvNone; e = w.next[e]) {
      const int s = w.state[e];
      const uint32_t c0 = (uint32_t)w.cost[e];
      const int i1 = __ldg(&rt.item_off[s + 1]);
      for (int i0 = __ldg(&rt.item_off[s]); i0 < i1; i0 += 32) {
        const int i = i0 + lane;
        uint32_t ic = kInf;
        int key = -1;
        if (i < i1) {
          ic = __ldg(&rt.item_cost[i]);
          const int p = __ldg(&rt.item_p[i]), d = __ldg(&rt.item_d[i]);
          if (p != 0 && d >= 2 && d <= k && ic < kInf) {
            const int g = t.gto(rsv_at(base, o, w, k - d) * t.NNT + t.lhs(p));
            if (g < t.S) key = ((k - d + 1) << 16) | g;
          }
        }
        insert_all(key, c0 + ic, e, i);
      }
    }
  }
  return goal;
}

// One block per row (the trigger and the tokens of the cheapest way are
// written by the warp that found it).  One thread per row, with the entries
// and the level heads in global memory, took 1,220 us for 32 SQL rows of up
// to 2,000 tokens; this takes 130 us.
template <bool ST>
__global__ void __launch_bounds__(kRsvWarps * 32) k_reserve(TabT<ST> t, ReserveTables rt, DevConfigs c, ReserveArgs ra) {
  __shared__ __align__(16) uint16_t s_stk[kRsvDepth];
  __shared__ unsigned long long s_best;  // total << 32 | option of the cheapest way
  __shared__ int s_slow;  // the row is reserve_serial's from the start
  __shared__ int s_full;  // a way's search needs more entries than a warp holds
  stage_tables(t);
  const auto& ts = t;
  const int b = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  RsvWarp& w = reinterpret_cast<RsvWarp*>(smem + ((t.blob_bytes + 15) & ~15))[warp];
  const int depth = c.depth[b], q = c.q[b], lx = c.lx[b];
  const bool complete = c.flags[b] & 1;
  const uint16_t* gbase = c.stack + (size_t)b * t.D;
  if (threadIdx.x == 0) {
    s_best = ~0ull;
    s_full = 0;
    s_slow = !complete && (depth > kRsvDepth || depth + kMaxOvl > t.D || t.S >= kRsvNone || rt.n_items >= kRsvNone);
  }
  if (depth <= kRsvDepth)
    for (int i = threadIdx.x; i < depth; i += blockDim.x) s_stk[i] = gbase[i];
  __syncthreads();
  const uint16_t* base = s_stk;
  const int mc = max_chain_of(t);
  const uint32_t pc0 = lx >= 0 ? t.lx_pcats[lx] : 0u, wc0 = lx >= 0 ? t.lx_wcats[lx] : 0u;
  const Bits4 live0 = q == kStart || complete ? Bits4::zero() : live_prime(ts, q, pc0).andnot(ts.ign);
  // way `opt`, by lane 0
  auto build = [&](int opt) -> RsvOption {
    RsvOption o{false, depth, 0, 0, ' '};
    if (q == kStart) {
      o.ok = true;
      return o;
    }
    int q2 = q, lx2 = lx;
    uint32_t pc = pc0, wc = wc0;
    if (opt > 0) {  // extend the lexeme to terminal tau's shortest lexeme
      const int tau = opt - 1;
      int cat = -1;
      for (int k = 0; k < t.n_cat; ++k)
        if (t.cat_term[k] == tau) cat = k;
      int len;
      if (cat >= 0) {
        if (lx < 0) return o;
        len = rt.lx_wdist[(size_t)lx * rt.NC + cat];
        if (len == 0xFFFF) return o;
      } else {
        len = rt.dfa_tdist[(size_t)q * t.T1 + tau];
        if (len == 0xFF) return o;
      }
      if (len == 0 || len > kMaxExt) return o;  // len 0: the lexeme as it stands (option 0)
      for (int i = 0; i < len; ++i) {
        const int by = cat >= 0 ? rt.lx_wbyte[(size_t)lx2 * rt.NC + cat] : rt.dfa_tbyte[(size_t)q2 * t.T1 + tau];
        const int nq = ts.nxt(q2 * ts.C + ts.cls(by));
        if (nq == kDead || rt.byte_tok[by] < 0) return o;
        q2 = nq;
        lx2 = lex_step(ts, q2, lx2, by, pc, wc);
        if (cat >= 0 && lx2 < 0) return o;
        w.y[o.ylen++] = (uint8_t)by;
      }
    }
    o.sep = rt.sep_byte[q2];
    if (o.sep < 0) return o;
    Walker x;
    walker_init(x, LArr{w.lo, 1}, LArr{w.ls, 1}, kMaxOvl, base, depth, nullptr, 0, q2, lx2, pc, wc, nullptr, nullptr);
    if (emit(ts, x, mc) <= 0) return o;
    o.keep = x.keep;
    o.m = x.m;
    o.ok = true;
    return o;
  };
  auto total_of = [&](const RsvOption& o, uint32_t C) -> uint32_t {
    // the blank that ends the lexeme comes with the first rendering; another
    // separator is a token of its own, needed only before a rendering
    if (C >= kInf || (C > 0 && o.sep != ' ' && rt.byte_tok[o.sep] < 0)) return kInf;
    return (uint32_t)o.ylen + ((C > 0 && o.sep != ' ') ? 1u : 0u) + C + 1u;
  };
  RsvOption mine{false, 0, 0, 0, 0};  // the way that this warp looked at last
  RsvGoal goal{kInf, -1, -1, false};
  int mine_opt = -1;
  // its cost, to every lane: kInf where it leads nowhere or `goal` is full
  auto look = [&](int opt) -> uint32_t {
    RsvOption o{false, 0, 0, 0, 0};
    mine_opt = -1;
    goal.full = false;
    __syncwarp();
    if (lane == 0) o = build(opt);
    o.ok = __shfl_sync(0xffffffffu, (int)o.ok, 0);
    o.keep = __shfl_sync(0xffffffffu, o.keep, 0);
    o.m = __shfl_sync(0xffffffffu, o.m, 0);
    o.ylen = __shfl_sync(0xffffffffu, o.ylen, 0);
    o.sep = __shfl_sync(0xffffffffu, o.sep, 0);
    if (!o.ok) return kInf;
    mine = o;
    mine_opt = opt;
    goal = rsv_search(ts, rt, base, o, w, lane);
    return goal.full ? kInf : total_of(o, goal.cost);
  };
  // What the warps tell each other is written between the barrier above and
  // the one below, and read after the latter alone: s_slow is not written
  // again, s_full and s_best are not read here.
  if (!complete && !s_slow) {
    auto offer = [&](int opt) {
      const uint32_t tot = look(opt);
      if (lane == 0 && goal.full) atomicExch(&s_full, 1);
      if (lane == 0 && tot < kInf) atomicMin(&s_best, ((unsigned long long)tot << 32) | (unsigned)opt);
    };
    int at = 0;  // the ways in order: 0, then 1 + tau of the live terminals
    if (warp == at++ % kRsvWarps) offer(0);
    Bits4 rest = live0;
    while (rest.any()) {
      const int tau = rest.lowest();
      rest.clear_lowest();
      if (warp == at++ % kRsvWarps && tau < t.n_term) offer(1 + tau);
    }
  }
  __syncthreads();
  if (s_slow || s_full) {
    if (threadIdx.x == 0) reserve_serial(t, ts, rt, c, ra, b);
    return;
  }
  const int cap = ra.cap;
  int32_t* out = ra.d_tokens + (size_t)b * cap;
  const unsigned long long best = s_best;
  int status = GRID_ST_OK;
  const uint32_t total = best == ~0ull ? kInf : (uint32_t)(best >> 32);
  if (complete || total >= kInf) {
    if (warp != 0) return;
    status = complete ? GRID_ST_COMPLETE : GRID_ST_NONVIABLE;
    for (int i = lane; i < cap; i += 32) out[i] = -1;
  } else {
    const int opt = (int)(uint32_t)best;
    const int owner = opt == 0 ? 0 : [&] {
      int at = 1;
      Bits4 rest = live0;
      while (rest.lowest() != opt - 1) {
        rest.clear_lowest();
        ++at;
      }
      return at % kRsvWarps;
    }();
    if (warp != owner) return;
    if (mine_opt != opt) look(opt);  // a later way of this warp took its place
    // the steps in order, in head[]: the parent chain from the goal entry, reversed, then the goal's item
    int len = 0;
    for (int e = goal.e; e != kRsvNone; e = w.parent[e]) len += w.item[e] != kRsvNone;
    __syncwarp();
    uint16_t* steps = reinterpret_cast<uint16_t*>(w.done);  // (the visits are over) 2 kRsvEnt entries
    if (lane == 0) {
      int k = len;
      for (int e = goal.e; e != kRsvNone; e = w.parent[e])
        if (w.item[e] != kRsvNone) steps[--k] = w.item[e];
      steps[len] = (uint16_t)goal.item;
    }
    __syncwarp();
    int n = mine.ylen;
    for (int i = lane; i < n && i < cap; i += 32) out[i] = rt.byte_tok[w.y[i]];
    if (goal.cost > 0 && mine.sep != ' ') {
      if (lane == 0 && n < cap) out[n] = rt.byte_tok[mine.sep];
      ++n;
    }
    // an item's rendering is item_cost tokens: a lane writes one item at a time
    for (int k0 = 0; k0 <= len; k0 += 32) {
      const int i = k0 + lane <= len ? steps[k0 + lane] : -1;
      const int own = i >= 0 ? (int)rt.item_cost[i] : 0;
      int at = own;
      for (int d = 1; d < 32; d <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, at, d);
        if (lane >= d) at += v;
      }
      const int sum = __shfl_sync(0xffffffffu, at, 31);
      at += n - own;
      if (i >= 0) {
        const int p = rt.item_p[i], d = rt.item_d[i];
        for (int j = rt.prod_off[p] + d; j < rt.prod_off[p + 1]; ++j) {
          const int X = rt.prod_rhs[j];
          if (X < t.T1) {
            put_terminal(rt, X, out, cap, at);
          } else {
            for (int k = rt.ny_off[X - t.T1]; k < rt.ny_off[X - t.T1 + 1]; ++k) put_terminal(rt, rt.ny[k], out, cap, at);
          }
        }
      }
      n += sum;
    }
    if (lane == 0 && n < cap) out[n] = t.eos;
    ++n;
    if (n > cap) status = GRID_ST_BOUND;
    for (int i = n + lane; i < cap; i += 32) out[i] = -1;
  }
  if (lane != 0) return;
  ra.d_cost[b] = complete ? 0 : (total < kInf ? (int32_t)total : -1);
  ra.d_status[b] = status;
  if (ra.d_fire)
    ra.d_fire[b] = (status == GRID_ST_OK && ra.d_budget && ra.d_budget[b] <= (int)total + ra.safety) ? 1 : 0;
}

}  // namespace

size_t reserve_scratch_bytes(const grid_spec* s) {
  return (size_t)kReserveEntries * sizeof(REnt) + (size_t)s->t.D * 4;
}

int build_reserve_tables(grid_spec* s, cudaStream_t st, std::vector<std::vector<uint8_t>>& keep) {
  const HostGrammar& h = s->g->h;
  const HostVocab& hv = s->v->h;
  ReserveTables& rt = s->rt;
  Arena& a = s->mem;
  const int T1 = h.T1, NNT = h.NNT, P = h.P, NS = hv.NS;
  auto is_ign = [&](int t) { return (h.ignored[t >> 5] >> (t & 31)) & 1u; };
  // the smallest id of every distinct spelling; exact lookup of a byte string
  std::vector<int32_t> id_of(std::max(1, NS), -1);
  for (int id = hv.V - 1; id >= 0; --id)
    if (hv.spell_of_id[id] >= 0) id_of[hv.spell_of_id[id]] = id;
  int maxlen = 1;
  for (int sp = 0; sp < NS; ++sp) maxlen = std::max(maxlen, hv.spell_off[sp + 1] - hv.spell_off[sp]);
  auto find = [&](const uint8_t* p, int n) {
    int lo = 0, hi = NS;
    while (lo < hi) {  // first spelling not below p[0:n] (bytes unsigned, shorter first)
      const int mid = (lo + hi) / 2;
      const int off = hv.spell_off[mid], len = hv.spell_off[mid + 1] - off;
      int cmp = std::memcmp(hv.spell_bytes.data() + off, p, (size_t)std::min(len, n));
      if (cmp == 0) cmp = len < n ? -1 : (len > n ? 1 : 0);
      if (cmp < 0)
        lo = mid + 1;
      else
        hi = mid;
    }
    if (lo < NS) {
      const int off = hv.spell_off[lo], len = hv.spell_off[lo + 1] - off;
      if (len == n && std::memcmp(hv.spell_bytes.data() + off, p, (size_t)n) == 0) return lo;
    }
    return -1;
  };
  std::vector<int32_t> byte_tok(256, -1);
  for (int b = 0; b < 256; ++b) {
    const uint8_t x = (uint8_t)b;
    const int sp = find(&x, 1);
    if (sp >= 0) byte_tok[b] = id_of[sp];
  }
  // renderings: " " + lexeme, split greedily (longest spelling first)
  std::vector<int32_t> rend_off(1, 0), rend_tok;
  std::vector<uint32_t> tcost(T1, kInf);
  for (int tau = 0; tau < T1; ++tau) {
    if (tau < h.n_term && !is_ign(tau) && !h.render_lex[tau].empty()) {
      const std::string str = " " + h.render_lex[tau];
      const uint8_t* p = reinterpret_cast<const uint8_t*>(str.data());
      const int n = (int)str.size();
      std::vector<int32_t> toks;
      bool ok = true;
      for (int i = 0; i < n && ok;) {
        ok = false;
        for (int L = std::min(maxlen, n - i); L >= 1; --L) {
          const int sp = find(p + i, L);
          if (sp >= 0) {
            toks.push_back(id_of[sp]);
            i += L;
            ok = true;
            break;
          }
        }
      }
      if (ok) {
        tcost[tau] = (uint32_t)toks.size();
        rend_tok.insert(rend_tok.end(), toks.begin(), toks.end());
      }
    }
    rend_off.push_back((int32_t)rend_tok.size());
  }
  // cheapest yield of every nonterminal, settled in order of cost (a
  // production is used only once all its nonterminals are settled, so every
  // yield is finite and well founded)
  std::vector<uint32_t> mcost(NNT, kInf);
  std::vector<int> bestp(NNT, -1), order;
  std::vector<char> settled(NNT, 0);
  for (;;) {
    uint32_t best = kInf;
    int bA = -1, bP = -1;
    for (int p = 0; p < P; ++p) {
      const int A = h.plhs[p];
      if (settled[A]) continue;
      uint32_t sum = 0;
      bool ok = true;
      for (int j = h.prod_off[p]; j < h.prod_off[p + 1] && ok; ++j) {
        const int X = h.prod_rhs[j];
        const uint32_t cx = X < T1 ? tcost[X] : (settled[X - T1] ? mcost[X - T1] : kInf);
        if (cx >= kInf) ok = false;
        sum = std::min<uint32_t>(kInf, sum + cx);
      }
      if (ok && sum < best) {
        best = sum;
        bA = A;
        bP = p;
      }
    }
    if (bA < 0) break;
    settled[bA] = 1;
    mcost[bA] = best;
    bestp[bA] = bP;
    order.push_back(bA);
  }
  std::vector<std::vector<int32_t>> yield(NNT);
  size_t ytotal = 0;
  for (int A : order) {
    const int p = bestp[A];
    for (int j = h.prod_off[p]; j < h.prod_off[p + 1]; ++j) {
      const int X = h.prod_rhs[j];
      if (X < T1)
        yield[A].push_back(X);
      else
        yield[A].insert(yield[A].end(), yield[X - T1].begin(), yield[X - T1].end());
    }
    ytotal += yield[A].size();
    if (ytotal > (1u << 24)) return set_error(GRID_E_TOO_LARGE, "grid_specialize: cheapest yields too long");
  }
  std::vector<int32_t> ny_off(1, 0), ny;
  for (int A = 0; A < NNT; ++A) {
    ny.insert(ny.end(), yield[A].begin(), yield[A].end());
    ny_off.push_back((int32_t)ny.size());
  }
  std::vector<uint32_t> item_cost(h.kitem_p.size(), kInf);
  for (size_t i = 0; i < h.kitem_p.size(); ++i) {
    const int p = h.kitem_p[i], d = h.kitem_d[i];
    uint32_t sum = 0;
    for (int j = h.prod_off[p] + d; j < h.prod_off[p + 1]; ++j) {
      const int X = h.prod_rhs[j];
      sum = std::min<uint32_t>(kInf, sum + (X < T1 ? tcost[X] : mcost[X - T1]));
    }
    item_cost[i] = sum;
  }
  Upload up;
  up.add(h.kitem_off, &rt.item_off);
  up.add(h.kitem_p, &rt.item_p);
  up.add(h.kitem_d, &rt.item_d);
  up.add(item_cost, &rt.item_cost, false);
  up.add(h.prod_off, &rt.prod_off);
  up.add(h.prod_rhs, &rt.prod_rhs);
  up.add(ny_off, &rt.ny_off, false);
  up.add(ny, &rt.ny, false);
  up.add(rend_off, &rt.rend_off, false);
  up.add(rend_tok, &rt.rend_tok, false);
  up.add(h.sep_byte, &rt.sep_byte);
  up.add(byte_tok, &rt.byte_tok, false);
  up.add(h.dfa_tdist, &rt.dfa_tdist);
  up.add(h.dfa_tbyte, &rt.dfa_tbyte);
  up.add(h.lx_wdist, &rt.lx_wdist);
  up.add(h.lx_wbyte, &rt.lx_wbyte);
  if (int rc = up.commit(a, st, keep)) return rc;
  rt.NC = std::max(1, h.n_cat);
  rt.n_items = (int)h.kitem_p.size();
  rt.E = kReserveEntries;
  rt.ok = 1;
  return GRID_OK;
}

}  // namespace grid

extern "C" int grid_reserve(const grid_spec* s, const grid_configs* c, int32_t* d_cost, int32_t* d_tokens, int32_t cap,
                            int32_t* d_status, const int32_t* d_budget, int32_t safety, int32_t* d_fire, void* stream) {
  if (!s || !c || !d_cost || !d_tokens || cap <= 0 || !d_status || (d_budget && !d_fire))
    return set_error(GRID_E_INVALID_ARG, "grid_reserve: bad arguments");
  if (!s->rt.ok) return set_error(GRID_E_INVALID_ARG, "grid_reserve: the spec has no reserve tables");
  const size_t dyn = ((s->t.blob_bytes + 15) & ~15) + kRsvWarps * sizeof(RsvWarp);
  const ReserveArgs ra{c->rscratch, reserve_scratch_bytes(s) / 4, d_cost, d_tokens, cap, d_status, d_budget, safety,
                       d_fire};
  auto launch = [&](auto kern, const auto& t) -> int {
    GRID_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kRsvSmem));
    kern<<<c->B, kRsvWarps * 32, dyn, (cudaStream_t)stream>>>(t, s->rt, c->c, ra);
    return GRID_OK;
  };
  if (int rc = s->t.blob_bytes ? launch(k_reserve<true>, TabT<true>(s->t)) : launch(k_reserve<false>, TabT<false>(s->t)))
    return rc;
  GRID_CUDA(cudaGetLastError());
  return GRID_OK;
}
