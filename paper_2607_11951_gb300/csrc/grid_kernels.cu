// libgrid device side for sm_103a: table upload, CI precompute, configurations
// and the kernels of the cold full-vocabulary mask.
//
// Specialization (grid_specialize, Sec. 4.2 / cold-schema specialization), for
// every precomputed lexer state (the start state and each state where no
// lexicon category is live) and every distinct spelling:
//   k_lex_hash, k_ids, k_spell16   the identifier trie's hash, the alias lists,
//                 the spellings' first bytes
//   k_classify    the spelling's class: a CI class id (its verdict is a
//                 function of the allowed set alone), always / never viable,
//                 a verdict class (its stack-dependent events fit one record),
//                 or byte-walked CD (more events than a record holds)
//   k_events      the event records of the verdict-class spellings, class ids
//                 with equal terminal sets rewritten to one class
//   k_vc_merge, k_vc_gather, k_vc_rank, k_vc_place   equal records become the
//                 table's verdict classes, in the order of their events
//   k_compact     per lexer state: the list of its byte-walked spellings
//   k_scatter_vc, k_permute   class codes and verdict-class indices re-indexed
//                 by token id (coalesced in k_pack)
//
// Mask step (grid_masks, Def. 4):
//   k_row    one block per row: the forced emission of the pending lexeme
//            (what every token whose first byte ends the lexeme must go
//            through) -> sigma', and the EOS gate (Sec. 3.2); the first bytes
//            that end the lexeme; one lane per terminal tau and context runs
//            tau's reduce chain (A0 = A(sigma), A1 = A(sigma') are the ballots)
//            and, for allowed tau, the allowed set after shifting tau (walks
//            simulate nothing before their second shift); then, for rows
//            without a table, the live first-byte ranges that continue the
//            lexeme, and the class selections
//   k_filter per row and context: the byte-walked spellings and the verdict
//            classes whose first stack-dependent emission can succeed
//   k_walk   persistent; per row: each surviving verdict class evaluated once
//            against the row's stack, and the byte walks: lanes walk token
//            bytes through the DFA and the identifier trie, emissions pick the
//            highest-priority parser-viable candidate on a copy-on-write
//            overlay (Sec. 4.1); first-byte subtrees of the trie in which no
//            spelling can survive are never entered; a walked spelling's
//            verdict is set for each of its ids (alias ids share a spelling
//            and so a verdict) in an id-indexed bitmap with the mask's layout
//   k_pack   per token id: CI class selection | verdict class | walked verdict
//            | EOS gate, packed into the id-order mask; with logits
//            (grid_masks_apply) the -inf fill of the word's sectors as well;
//            with a mask cache, the context-independent bits of a hit read
//            from the cache entry (or stored into the entry the row claimed)
// Decoding step (grid_advance_masks): the same kernels, k_row feeding each
// row's tokens on warp 0 of its block before it prepares the row.
// Parser step (grid_advance):  k_advance, k_advance_one.   Masked logits:  k_apply.
//
// Every loop is bounded; hitting a bound writes GRID_ST_BOUND.  No kernel traps.

#include <cuda_runtime.h>

#include <algorithm>
#include <array>
#include <cstring>
#include <mutex>
#include <string>
#include <type_traits>
#include <unordered_map>
#include <utility>
#include <vector>

#include "grid_state.cuh"

namespace grid {
namespace {

constexpr int kWalkWarps = 24;   // warps per k_walk block, at most (one block per SM)
constexpr int kSpan = 32;        // CD list entries per walk item (one warp batch)
constexpr int kStackWin = 1024;  // stacks up to this depth are copied to shared memory in k_row/k_advance
constexpr int kFilterPer = 4;    // records per k_filter thread
constexpr int kRangeSpan = 32;   // continuing first-byte ranges are walked in items of (up to) this many spellings
constexpr int kWalkWin = 512;    // k_walk mirrors row stacks up to this depth per warp
constexpr int kRowWarps = 6;     // k_row: warps per row block
constexpr int kRowJobWarps = kRowWarps - 1;  // k_row: warps 1 .. compute the allowed sets
// Class codes as k_pack reads them: CI class ids 0..ncls-1, then these five
// (so that one bit test of the row's class selection covers CI, always and
// never, and only verdict-class and walked tokens need a second lookup).
constexpr int kPackCodes = 5;  // ncls + 0 always, +1 never, +2 n/a, +3 verdict class, +4 walked;
                               // with vc_inline, 32 nselw + v: verdict class v of the code's table
constexpr int kWalkRowsCached = 256;  // rows whose queue bounds k_walk keeps in shared memory
constexpr int kStagedSets = 512; // classes whose terminal sets are staged with the tables, at most
constexpr int kLaneOvl = 32;     // overlay / scratch entries per walk lane (shared memory)
constexpr int kMaxRows = 65535;  // rows of one configurations object (a grid dimension of the mask kernels)

// ---------------------------------------------------------------------------
__global__ void k_reset(DevConfigs c, int B, int D) {
  int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= B) return;
  c.stack[(size_t)b * D] = 0;
  if (c.hs) c.hs[(size_t)b * D] = 0;  // H(root) = 0
  c.depth[b] = 1;
  c.q[b] = kStart;
  c.lx[b] = 0;
  c.flags[b] = 0;
}

// ---------------- specialization ----------------
template <bool ST>
__global__ void k_classify(TabT<ST> t, uint16_t* __restrict__ cls_sp, uint16_t* __restrict__ key_sp,
                           int32_t* __restrict__ counts) {
  stage_tables(t);
  const auto& ts = t;
  const int tbl = blockIdx.y;
  const int q0 = t.tbl_q[tbl];
  const int lx0 = q0 == kStart ? 0 : -1;
  int ncd = 0, nvc = 0;
  uint16_t rec[kRecLen];
  for (int s = blockIdx.x * blockDim.x + threadIdx.x; s < t.NS; s += gridDim.x * blockDim.x) {
    const int off = t.spell_off[s];
    const int len = t.spell_off[s + 1] - off;
    const uint8_t* by = t.spell_bytes + off;
    uint16_t code, key = 0xFFFF;
    if (!t.ci_on)
      code = kClsCD;
    else if (q0 != kStart && ts.nxt(q0 * ts.C + ts.cls(by[0])) == kDead)
      code = kClsNA;
    else
      code = classify(ts, q0, lx0, by, len, key, rec);
    cls_sp[(size_t)tbl * t.NS + s] = code;
    key_sp[(size_t)tbl * t.NS + s] = key;
    ncd += code == kClsCD;
    nvc += code == kClsVC;
  }
  ncd = __reduce_add_sync(0xffffffffu, ncd);
  nvc = __reduce_add_sync(0xffffffffu, nvc);
  if ((threadIdx.x & 31) == 0) {
    if (ncd) atomicAdd(&counts[2 * tbl], ncd);
    if (nvc) atomicAdd(&counts[2 * tbl + 1], nvc);
  }
}

// Event records of the kClsVC spellings, appended per table in any order:
// slot -> (table, spelling, record).
template <bool ST>
__global__ void k_events(TabT<ST> t, const uint16_t* __restrict__ cls_sp, const int32_t* __restrict__ vc_base,
                         int32_t* __restrict__ fill, int32_t* __restrict__ slot_tbl, int32_t* __restrict__ slot_sp,
                         uint16_t* __restrict__ slot_rec) {
  stage_tables(t);
  const auto& ts = t;
  const int tbl = blockIdx.y;
  const int q0 = t.tbl_q[tbl];
  const int lx0 = q0 == kStart ? 0 : -1;
  uint16_t rec[kRecLen];
  for (int s = blockIdx.x * blockDim.x + threadIdx.x; s < t.NS; s += gridDim.x * blockDim.x) {
    if (cls_sp[(size_t)tbl * t.NS + s] != kClsVC) continue;
    const int off = t.spell_off[s];
    uint16_t key;
    for (int k = 0; k < kRecLen; ++k) rec[k] = 0;
    classify(ts, q0, lx0, t.spell_bytes + off, t.spell_off[s + 1] - off, key, rec);
    const int slot = vc_base[tbl] + atomicAdd(&fill[tbl], 1);
    slot_tbl[slot] = tbl;
    slot_sp[slot] = s;
    for (int k = 0; k < kRecLen; ++k)  // class ids of equal terminal sets become one class
      slot_rec[(size_t)slot * kRecLen + k] = k > 0 && k < 2 + rec[0] && rec[k] < kClsFirstCode ? t.cls_map[rec[k]] : rec[k];
  }
}

// Per lexer state q and mask word wi, the ids whose first byte ends a pending
// lexeme in state q (every id at the start state): the split of a row's ids
// between sigma' and sigma that k_pack applies one word at a time.
__global__ void k_killw(Tables t, uint32_t* __restrict__ out) {
  const int wi = blockIdx.x * blockDim.x + threadIdx.x;
  const int q = blockIdx.y;
  if (wi >= t.W) return;
  uint32_t w = 0u;
  for (int j = 0; j < 32; ++j) {
    const int id = 32 * wi + j;
    const int by = id < t.Vp ? t.first_byte_by_id[id] : 0;
    if (q == kStart || q == kDead || t.next[q * t.C + t.byte_class[by]] == kDead) w |= 1u << j;
  }
  out[(size_t)q * t.W + wi] = w;
}

// ---- tables made on the device from what was uploaded: each replaces a host
// loop over the vocabulary or the identifier trie (50,000 identifiers and
// V = 151,936: the trie's hash 5.9 ms, the merge of the event records 10.3 ms,
// the sixteen-byte heads and the alias lists 0.8 ms of 22 ms).

// Identifier-trie edges into the open-addressing hash (entries cleared to
// 0xFF bytes, load factor <= 1/2), a node per thread.
__global__ void k_lex_hash(const int32_t* __restrict__ cstart, const uint8_t* __restrict__ cbyte,
                           const int32_t* __restrict__ cnode, const uint32_t* __restrict__ pcats,
                           const uint32_t* __restrict__ wcats, int LN, uint4* __restrict__ tab, uint32_t mask,
                           int shift) {
  const int n = blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= LN) return;
  for (int e = cstart[n]; e < cstart[n + 1]; ++e) {
    const uint32_t key = (uint32_t)n * 256u + cbyte[e];
    const int child = cnode[e];
    uint32_t h = (key * 0x9E3779B1u) >> shift;
    for (uint32_t i = 0; i <= mask; ++i) {
      if (atomicCAS(&tab[h].x, kHashEmpty, key) == kHashEmpty) {
        tab[h].y = (uint32_t)child;
        tab[h].z = pcats[child];
        tab[h].w = wcats[child];
        break;
      }
      h = (h + 1u) & mask;
    }
  }
}

// The list of each spelling's ids (aliases, in any order); specials, EOS and
// padding ids have no spelling.
__global__ void k_ids(const int32_t* __restrict__ spell_of_id, int Vp, int32_t* __restrict__ id_of_spell,
                      int32_t* __restrict__ next_alias) {
  const int id = blockIdx.x * blockDim.x + threadIdx.x;
  if (id >= Vp) return;
  const int sp = spell_of_id[id];
  next_alias[id] = sp >= 0 ? atomicExch(&id_of_spell[sp], id) : -1;
}

// The first 16 bytes of each spelling, zero padded.
__global__ void k_spell16(const int32_t* __restrict__ spell_off, const uint8_t* __restrict__ bytes, int NS,
                          uint4* __restrict__ out) {
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= NS) return;
  const int off = spell_off[s], len = min(16, spell_off[s + 1] - off);
  uint32_t w[4] = {0u, 0u, 0u, 0u};
#pragma unroll
  for (int i = 0; i < 16; ++i)
    if (i < len) w[i >> 2] |= (uint32_t)bytes[off + i] << (8 * (i & 3));
  out[s] = make_uint4(w[0], w[1], w[2], w[3]);
}

// ---- the event records' merge into verdict classes
struct Rec {
  uint4 a, b;
  __device__ __forceinline__ bool operator==(const Rec& o) const {
    return a.x == o.a.x && a.y == o.a.y && a.z == o.a.z && a.w == o.a.w && b.x == o.b.x && b.y == o.b.y &&
           b.z == o.b.z && b.w == o.b.w;
  }
};
static_assert(sizeof(Rec) == kRecLen * 2, "an event record is two 16-byte words");

// A record's place in its table's order: the events one after the other (each
// + 1; 0 after the last, so that a record comes before those it starts), then
// the final class.
struct RecKey {
  unsigned long long k[4];
  __device__ __forceinline__ bool operator<(const RecKey& o) const {
    if (k[0] != o.k[0]) return k[0] < o.k[0];
    if (k[1] != o.k[1]) return k[1] < o.k[1];
    if (k[2] != o.k[2]) return k[2] < o.k[2];
    return k[3] < o.k[3];
  }
};

__device__ __forceinline__ RecKey rec_key(const uint16_t* r) {
  RecKey x;
#pragma unroll
  for (int w = 0; w < 4; ++w) {
    unsigned long long v = 0;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int e = 4 * w + j;
      const unsigned long long f = e < kMaxEv ? (e < r[0] ? r[2 + e] + 1ull : 0ull) : (e == kMaxEv ? r[1] : 0ull);
      v = (v << 16) | f;
    }
    x.k[w] = v;
  }
  return x;
}

// Equal records of one table find one slot (rep): an open-addressing table of
// slots (cleared to -1, at least twice as large), the first to claim an entry
// stands for its record and takes the next place in its table.
__global__ void k_vc_merge(const int32_t* __restrict__ slot_tbl, const Rec* __restrict__ rec, int nslot,
                           int32_t* __restrict__ tab, uint32_t mask, int32_t* __restrict__ rep,
                           int32_t* __restrict__ place, int32_t* __restrict__ count) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= nslot) return;
  const Rec r = rec[i];
  const int tbl = slot_tbl[i];
  uint32_t h = (uint32_t)tbl;
  const uint32_t w[8] = {r.a.x, r.a.y, r.a.z, r.a.w, r.b.x, r.b.y, r.b.z, r.b.w};
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    h = (h ^ w[k]) * 0x9E3779B1u;
    h ^= h >> 15;
  }
  h &= mask;
  for (uint32_t n = 0; n <= mask; ++n) {
    const int cur = atomicCAS(&tab[h], -1, i);
    if (cur == -1) {
      rep[i] = i;
      place[i] = atomicAdd(&count[tbl], 1);
      return;
    }
    if (slot_tbl[cur] == tbl && rec[cur] == r) {
      rep[i] = cur;
      return;
    }
    h = (h + 1u) & mask;
  }
}

// The distinct records, table by table (in any order within it), with their keys.
__global__ void k_vc_gather(const int32_t* __restrict__ slot_tbl, const Rec* __restrict__ rec, int nslot,
                            const int32_t* __restrict__ rep, const int32_t* __restrict__ place,
                            const int32_t* __restrict__ vc_off, int32_t* __restrict__ src, RecKey* __restrict__ key,
                            int32_t* __restrict__ rank) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= nslot || rep[i] != i) return;
  const int at = vc_off[slot_tbl[i]] + place[i];
  src[at] = i;
  key[at] = rec_key(reinterpret_cast<const uint16_t*>(rec + i));
  rank[at] = 0;
}

// Each record's rank in its table: the number of smaller keys, counted over
// the table's keys in tiles; grid (records / 256, tables, parts of the tiles).
// Quadratic in a table's records, of which there are at most as many as
// spellings: with 150,000 of them in the start state's table a specialization
// takes 18.7 ms (4.2 ms with 60,000), 164 ms when the host merged and sorted them.
__global__ void __launch_bounds__(256) k_vc_rank(const RecKey* __restrict__ key, const int32_t* __restrict__ vc_off,
                                                 int32_t* __restrict__ rank) {
  __shared__ RecKey s_key[256];
  const int a = vc_off[blockIdx.y], n = vc_off[blockIdx.y + 1] - a;
  const int p = blockIdx.x * 256 + threadIdx.x;
  if ((int)blockIdx.x * 256 >= n) return;
  const RecKey own = key[a + min(p, n - 1)];
  int less = 0;
  for (int t0 = blockIdx.z * 256; t0 < n; t0 += gridDim.z * 256) {
    __syncthreads();
    if (t0 + (int)threadIdx.x < n) s_key[threadIdx.x] = key[a + t0 + threadIdx.x];
    __syncthreads();
    const int m = min(256, n - t0);
    for (int j = 0; j < m; ++j) less += s_key[j] < own ? 1 : 0;
  }
  if (p < n && less) atomicAdd(&rank[a + p], less);
}

// The records in their order, and each one's index for its slots (place, reused).
__global__ void k_vc_place(const Rec* __restrict__ rec, const int32_t* __restrict__ slot_tbl,
                           const int32_t* __restrict__ src, const int32_t* __restrict__ rank, int n,
                           const int32_t* __restrict__ vc_off, Rec* __restrict__ out, uint16_t* __restrict__ first,
                           int32_t* __restrict__ place) {
  const int at = blockIdx.x * blockDim.x + threadIdx.x;
  if (at >= n) return;
  const int i = src[at], to = vc_off[slot_tbl[i]] + rank[at];
  const Rec r = rec[i];
  out[to] = r;
  first[to] = (uint16_t)(r.a.y & 0xFFFFu);
  place[i] = rank[at];
}

__global__ void k_scatter_vc(const int32_t* __restrict__ slot_tbl, const int32_t* __restrict__ slot_sp,
                             const int32_t* __restrict__ rep, const int32_t* __restrict__ place, int nslot, int NS,
                             uint32_t* __restrict__ vc_sp) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < nslot) vc_sp[(size_t)slot_tbl[i] * NS + slot_sp[i]] = (uint32_t)place[rep[i]];
}

// Per table the list of its byte-walked spellings and their keys (runs of
// neighbours in any order; grid.y: tables).
__global__ void k_compact(const uint16_t* __restrict__ cls_sp, const uint16_t* __restrict__ key_sp, int NS,
                          const int32_t* __restrict__ cd_off, const uint16_t* __restrict__ cls_map,
                          int32_t* __restrict__ fill, int32_t* __restrict__ cd_list, uint16_t* __restrict__ cd_key) {
  const int tbl = blockIdx.y, lane = threadIdx.x & 31;
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  const bool f = s < NS && cls_sp[(size_t)tbl * NS + s] == kClsCD;
  const uint32_t bal = __ballot_sync(0xffffffffu, f);
  if (!bal) return;
  int at = 0;
  if (lane == 0) at = cd_off[tbl] + atomicAdd(&fill[tbl], __popc(bal));
  at = __shfl_sync(0xffffffffu, at, 0) + __popc(bal & ((1u << lane) - 1u));
  if (f) {
    const uint16_t k = key_sp[(size_t)tbl * NS + s];
    cd_list[at] = s;
    cd_key[at] = k == 0xFFFF ? k : cls_map[k];
  }
}

__global__ void k_permute(Tables t, const uint16_t* __restrict__ cls_sp, const uint32_t* __restrict__ vc_sp,
                          uint16_t* __restrict__ cls_by_id, uint32_t* __restrict__ vc_by_id,
                          uint8_t* __restrict__ fb_by_id) {
  const int id = blockIdx.x * blockDim.x + threadIdx.x;
  if (id >= t.Vp) return;
  const int s = t.spell_of_id[id];  // -1 for EOS, specials and the padding ids
  fb_by_id[id] = s >= 0 ? t.spell_bytes[t.spell_off[s]] : 0;
  for (int k = 0; k < t.n_tbl; ++k) {
    const uint16_t c = s >= 0 ? cls_sp[(size_t)k * t.NS + s] : kClsNA;
    uint16_t code = c < kClsFirstCode ? t.cls_map[c] : c;  // the k_pack code of c
    if (c >= kClsFirstCode)
      code = (uint16_t)(t.ncls + (c == kClsAcc ? 0 : c == kClsRej ? 1 : c == kClsNA ? 2 : c == kClsVC ? 3 : 4));
    if (c == kClsVC && t.vc_inline) code = (uint16_t)(32 * t.nselw + vc_sp[(size_t)k * t.NS + s]);
    cls_by_id[(size_t)k * t.Vp + id] = code;
    if (vc_by_id) vc_by_id[(size_t)k * t.Vp + id] = c == kClsVC ? vc_sp[(size_t)k * t.NS + s] : 0xFFFFFFFFu;
  }
}

// ---------------- mask step ----------------
// Class selections for the allowed sets AI0 and AI1 (with the ignored
// terminals), word w0, by a warp: bit c = the set of class c meets them.
template <class T>
__device__ __forceinline__ void select_word(const T& t, const Bits4 AI0, const Bits4 AI1, int w0, int lane,
                                            uint32_t& v0, uint32_t& v1) {
  const int c = w0 * 32 + lane;
  Bits4 set = Bits4::zero();
  if (c < t.ncls) set = t.set4(c);
  const bool all = c == t.ncls;  // the code "always"
  v0 = __ballot_sync(0xffffffffu, all || (set & AI0).any());
  v1 = __ballot_sync(0xffffffffu, all || (set & AI1).any());
}

// The configuration one warp leaves after feeding its row's tokens (lane 0's
// values; `win`: the warp's shared-memory window holds the row's stack).
struct AdvOut {
  int depth, q, lx, flags, status;
  uint32_t pc, wc;
  bool win;
  int keep;  // entries below it are the incoming stack's (the node hashes from here on are new)
};

// Rolling node hashes (Sec. 6.4) of the entries keep .. depth - 1 of row b's
// stack, by one warp: the entries' symbols are loaded together, the hashes
// chain from the parent of entry `keep`.  Only the entries that are left are
// hashed, once the tokens are fed, away from the chain that the mask waits
// for: hashing each push as it was made, on the lane that feeds the tokens,
// cost k_row 51 us of 76 at 32 rows (24 without hashes).
template <class T>
__device__ __forceinline__ void hash_nodes(const T& t, uint64_t* __restrict__ hs, const uint16_t* stack, int keep,
                                           int depth, int lane) {
  if (keep >= depth) return;
  uint64_t hp = hs[keep - 1];
  for (int i0 = keep; i0 < depth; i0 += 32) {
    const uint32_t sym = i0 + lane < depth ? t.acc_sym[stack[i0 + lane]] : 0u;
    const int n = min(32, depth - i0);
    for (int i = 0; i < n; ++i) {
      hp = node_hash_quad(lane, hp, __shfl_sync(0xffffffffu, sym, i));
      if (lane == 0) hs[i0 + i] = hp;
    }
  }
}

// Advance of row b (Sec. 3.1 parser step, Sec. 4.1 byte walk) by one warp, in
// three parts.  advance_load: the lanes copy the row's stack for an
// out-of-place advance and mirror it in `win` (kStackWin entries, 16-byte
// accesses when the row stride allows them); the first 256 entries are read
// before the depth is known.  parse_batch, over the batches that lex_batch
// made, feeds the tokens while the stack fits the window and the grammar's
// chains have a bound (Tables::chain_rate).  advance_serial feeds what is left
// on lane 0 (a token that is refused, EOS, a stack beyond the window).
//
// A token that is fed costs the chain of its table look-ups, so nothing but
// the stack's own steps stays serial: feeding every byte on lane 0, with the
// token's spelling loaded when its turn came and each reduce chain run twice
// (once for a set of terminals, once for the one that shifts), took 3.9 us a
// token (2,000 tokens, 32 SQL rows: 7.8 ms; 1.8 ms this way).
constexpr int kAdvSpec = 32;  // 16-byte stack accesses issued per lane before the depth is known

// What the parts share, in shared memory: of a token, of a batch.
struct FeedShared {
  uint16_t undo[kStackWin];
  uint16_t scr[kChainNs * 32];
  uint16_t lo[kMaxOvl], ls[kMaxOvl];  // lane 0's overlay and scratch
};
struct AdvShared {
  LexBatch lex;
  FeedShared f;
};

struct AdvRow {
  int depth, flags;
  LexState s;
  bool win;
};

// The row's configuration (every lane gets it) and its pending lexeme's categories.
template <class T>
__device__ __forceinline__ AdvRow advance_config(const T& t, const DevConfigs& c, int b, int lane) {
  int cf = 0;
  if (lane < 4) {
    const int32_t* f = lane == 0 ? c.depth : lane == 1 ? c.q : lane == 2 ? c.lx : c.flags;
    cf = f[b];
  }
  uint32_t cpc = 0u, cwc = 0u;  // category bits of the pending lexeme's trie node (lane 2)
  if (lane == 2 && cf >= 0) {
    cpc = t.lx_pcats[cf];
    cwc = t.lx_wcats[cf];
  }
  AdvRow r;
  r.depth = __shfl_sync(0xffffffffu, cf, 0);
  r.s.q = __shfl_sync(0xffffffffu, cf, 1);
  r.s.lx = __shfl_sync(0xffffffffu, cf, 2);
  r.flags = __shfl_sync(0xffffffffu, cf, 3);
  r.s.pc = __shfl_sync(0xffffffffu, cpc, 2);
  r.s.wc = __shfl_sync(0xffffffffu, cwc, 2);
  r.win = r.depth <= kStackWin;
  return r;
}

template <class T>
__device__ __forceinline__ AdvRow advance_load(const T& t, const DevConfigs& cin, const DevConfigs& cout, int b,
                                               int copy, int lane, uint16_t* win) {
  const uint16_t* src = (copy ? cin.stack : cout.stack) + (size_t)b * t.D;
  uint16_t* stack = cout.stack + (size_t)b * t.D;
  const bool vec = t.D % 8 == 0;  // rows start on 16-byte boundaries: 8 entries per access
  const uint4* s4 = reinterpret_cast<const uint4*>(src);
  uint4 sv = make_uint4(0u, 0u, 0u, 0u);
  if (vec && lane < kAdvSpec && lane * 8 < t.D) sv = s4[lane];
  const AdvRow r = advance_config(t, copy ? cin : cout, b, lane);
  if (vec) {
    const int n8 = (r.depth + 7) >> 3;  // (n8 * 8 <= D: the last access stays inside the row)
    uint4* d4 = reinterpret_cast<uint4*>(stack);
    uint4* w4 = reinterpret_cast<uint4*>(win);
    if (lane < n8) {
      if (copy) d4[lane] = sv;
      if (r.win) w4[lane] = sv;
    }
    for (int i = lane + kAdvSpec; i < n8; i += 32) {
      const uint4 v = s4[i];
      if (copy) d4[i] = v;
      if (r.win) w4[i] = v;
    }
  } else {
    for (int i = lane; i < r.depth; i += 32) {
      const uint16_t v = src[i];
      if (copy) stack[i] = v;
      if (r.win) win[i] = v;
    }
  }
  if (copy && cout.hs) {  // the node hashes travel with the stack
    const uint64_t* hsrc = cin.hs + (size_t)b * t.D;
    uint64_t* hdst = cout.hs + (size_t)b * t.D;
    for (int i = lane; i < r.depth; i += 32) hdst[i] = hsrc[i];
  }
  __syncwarp();
  return r;
}

// Whether the warp feeds the row's tokens in batches (else they are
// advance_serial's; a single token is feed_one's).
template <class T>
__device__ __forceinline__ bool feed_fits(const T& t, const AdvRow& r, int n_steps) {
  return n_steps > 1 && t.chain_rate > 0 && r.win && !(r.flags & 1);
}

__device__ __forceinline__ Feed feed_begin(const AdvRow& r, uint16_t* win, FeedShared& sh) {
  return Feed{win, sh.undo, sh.scr, kStackWin, r.depth, r.depth, r.depth, 0, r.depth, false, r.s};
}

// After the last batch (`fed`: parse_batch went through all of them, `end` is
// the lexer's state there): the test of the last token, the stack written
// back, and the row as advance_serial goes on with it at token f.tok.
template <class T>
__device__ __forceinline__ void feed_end(const T& ts, Feed& f, bool fed, const LexState& end, int n_steps,
                                         AdvRow& r, uint16_t* stack, int lane, int max_chain) {
  if (fed && (!f.any || (f.depth <= ts.D && feed_live(ts, f, end.q, end.pc, lane, max_chain) == 1))) {
    f.tok = n_steps;
    f.s = end;
  } else {
    feed_back(f, lane);
  }
  for (int i = f.wlow + lane; i < f.depth; i += 32) stack[i] = f.win[i];
  r.depth = f.depth;
  r.s = f.s;
  __syncwarp();
}

// Lane 0 only: tokens k0 .. n_steps - 1, one after the other (`first`: token 0,
// loaded ahead).
template <class T>
__device__ __forceinline__ void advance_serial(const T& t, const T& ts, const DevConfigs& cout,
                                               const int32_t* __restrict__ tokens, int k0, int n_steps, int b,
                                               uint16_t* win, FeedShared& sh, const AdvRow& r, int keep,
                                               const LexToken& first, AdvOut& out) {
  uint16_t* stack = cout.stack + (size_t)b * t.D;
  const LArr lo{sh.lo, 1}, ls{sh.ls, 1};
  int depth = r.depth, q = r.s.q, lx = r.s.lx, flags = r.flags;
  uint32_t pc = r.s.pc, wcat = r.s.wc;
  bool use_win = r.win;
  int status = GRID_ST_OK;
  const int mc = max_chain_of(t);
  Walker w;
#pragma unroll 1
  for (int k = k0; k < n_steps; ++k) {
    const int tok = tokens[(size_t)b * n_steps + k];
    if (tok < 0) continue;
    if (flags & 1) {
      status = GRID_ST_COMPLETE;
      break;
    }
    if (tok >= t.V) {
      status = GRID_ST_TOKEN_NOT_ALLOWED;
      break;
    }
    walker_init(w, lo, ls, kMaxOvl, use_win ? win : stack, depth, nullptr, 0, q, lx, pc, wcat, nullptr, nullptr);
    if (tok == t.eos) {
      const int e = eos_gate(ts, w, mc);
      if (e < 0) {
        status = GRID_ST_BOUND;
        break;
      }
      if (e == 0) {
        status = GRID_ST_TOKEN_NOT_ALLOWED;
        break;
      }
      flags |= 1;
      continue;
    }
    const LexToken x = k == 0 ? first : lex_fetch(t, &tokens[(size_t)b * n_steps + k], 0, 1, 0);
    if (x.st != 1) {
      status = GRID_ST_TOKEN_NOT_ALLOWED;
      break;
    }
    const int e = walk_bytes(ts, w, x.sp, mc);
    if (e < 0) {
      status = GRID_ST_BOUND;
      break;
    }
    if (e == 0) {
      status = GRID_ST_TOKEN_NOT_ALLOWED;
      break;
    }
    if (w.keep + w.m > t.D) {
      status = GRID_ST_STACK_OVERFLOW;
      break;
    }
#pragma unroll 1
    for (int i = 0; i < w.m; ++i) stack[w.keep + i] = w.ovl[i];
    if (w.m > 0) keep = min(keep, w.keep);
    if (use_win && w.keep + w.m <= kStackWin) {
#pragma unroll 1
      for (int i = 0; i < w.m; ++i) win[w.keep + i] = w.ovl[i];
    } else {
      use_win = false;
    }
    depth = w.keep + w.m;
    q = w.q;
    lx = w.lx;
    pc = w.pc;
    wcat = w.wc;
  }
  out = AdvOut{depth, q, lx, flags, status, pc, wcat, use_win, keep};
}

// The same as a call, where it is seldom reached: its code is not in the way of
// the rest's.  The call reads the tables' descriptor from a copy in local
// memory; k_advance, where every token of a row may come this way (a grammar
// without CI classes, a stack beyond the window), has it inline: a prompt of 400
// tokens fed this way 1,319 us, through the call 1,610.
template <class T>
__device__ __noinline__ void advance_rest(const T& t, const T& ts, const DevConfigs& cout,
                                          const int32_t* __restrict__ tokens, int k0, int n_steps, int b,
                                          uint16_t* win, FeedShared& sh, const AdvRow& r, int keep,
                                          const LexToken& first, AdvOut& out) {
  advance_serial(t, ts, cout, tokens, k0, n_steps, b, win, sh, r, keep, first, out);
}

// Token k of a row, by its warp: feed_one, and `row` and `out` are the row after
// it; else advance_rest, which feeds the tokens after it too (false; `out` is
// lane 0's).
template <class T>
__device__ __forceinline__ bool advance_one(const T& t, const DevConfigs& cout, const int32_t* __restrict__ tokens,
                                            int k, int n_steps, int b, uint16_t* win, FeedShared& sh, AdvRow& row,
                                            const LexToken& x, int lane, AdvOut& out) {
  const int mc = max_chain_of(t);
  uint16_t* stack = cout.stack + (size_t)b * t.D;
  if (x.st == 1 && row.win && !(row.flags & 1)) {
    Feed f = feed_begin(row, win, sh);
    LexState s = row.s;
    if (feed_one(t, f, s, x.sp, lane, mc)) {
      for (int i = f.wlow + lane; i < f.depth; i += 32) stack[i] = win[i];
      row.depth = f.depth;
      row.s = s;
      out = AdvOut{f.depth, s.q, s.lx, row.flags, GRID_ST_OK, s.pc, s.wc, true, min(out.keep, f.wlow)};
      return true;
    }
    feed_back(f, lane);
  }
  if (lane == 0) advance_rest(t, t, cout, tokens, k, n_steps, b, win, sh, row, out.keep, x, out);
  return false;
}

// The configuration that the advance leaves, by lane 0.
__device__ __forceinline__ void advance_store(const DevConfigs& cout, int b, const AdvOut& o) {
  cout.depth[b] = o.depth;
  cout.q[b] = o.q;
  cout.lx[b] = o.lx;
  cout.flags[b] = o.flags;
}

// One block per row (kRowWarps warps), plus clearing blocks after the rows.
// Phase 1, every warp at once: warp 0 finds the first bytes that continue the
// pending lexeme and what can follow each (rows without a CI table); the job
// warps make the forced emission of the pending lexeme (sigma -> sigma', what
// every token whose first byte ends the lexeme must go through), the allowed
// sets of both contexts (A0 and A1), the EOS gate (Sec. 3.2) and, for every
// allowed terminal, the allowed set after its shift (A2: walks and verdict
// classes simulate nothing before their second shift).  Phase 2: warp 0 lays
// out the live ones of the continuing first-byte ranges, warps 1 .. 5 select
// the contexts' CI classes.  Then
// thread 0 writes the row's context for the later kernels and, with a mask
// cache, looks the row's key up (k_pack reads a ready entry) or claims an
// empty slot for it (k_pack fills it).
// Clearing blocks zero both verdict bitmaps and the verdict-class bits.
// With ADV the row's tokens are fed first (by warp 0, from
// adv.cin into c), and the row is masked in the configuration that leaves:
// the advance of one row and the mask preparation of another overlap, and
// the stack window is taken from the advance.  The row's status is then the
// advance's error, if its token was refused, else the mask step's.
// ADV: 0 no tokens, 1 one token per row, 2 several (its own instance, so that
// the usual step does not carry the batch feed's code).
template <int ADV, bool ST>
__global__ void __launch_bounds__(kRowWarps * 32, 2) k_row(TabT<ST> t, DevConfigs c, RowCtx* __restrict__ ctx,
                                                        RowRanges* __restrict__ rng, uint32_t* __restrict__ A2,
                                                        uint32_t* __restrict__ sel, uint32_t* __restrict__ verd0,
                                                        uint32_t* __restrict__ verd1, uint32_t* __restrict__ vcbits,
                                                        int n_vcbits, int B, int words_v, CacheDev cache,
                                                        AdvArgs adv) {
  __shared__ __align__(16) uint16_t s_stk[kStackWin];
  __shared__ uint16_t s_ovl1[kMaxOvl];
  __shared__ __align__(16) uint16_t s_ovl2[kRowJobWarps][kMaxOvl * 32];
  __shared__ uint16_t s_scr[kRowJobWarps][kMaxOvl * 32];
  __shared__ uint16_t s_em[kRowJobWarps][kMaxOvl];
  __shared__ __align__(16) uint32_t s_A0[4], s_A1[4];
  __shared__ LexToken s_own;
  __shared__ uint4 s_lv[256];   // rows without a table: live' after each continuing byte
  __shared__ uint8_t s_by[256]; // the continuing bytes
  __shared__ int s_row[8];  // complete, depth, q, lx, emit_ok, keep1, m1, eos_ok
  __shared__ uint32_t s_pc[2];
  __shared__ int s_status, s_total0, s_nrng, s_adv[3];
  if ((int)blockIdx.x >= B) {
    // clearing blocks: zero both verdict bitmaps and the verdict-class bits of every row
    pdl_wait();
    const size_t n = (size_t)B * words_v;
    const size_t n4 = n >> 2;
    const size_t stride = (size_t)(gridDim.x - B) * blockDim.x;
    const size_t first = (size_t)(blockIdx.x - B) * blockDim.x + threadIdx.x;
    const uint4 z = make_uint4(0u, 0u, 0u, 0u);
    for (size_t i = first; i < n4; i += stride) {
      reinterpret_cast<uint4*>(verd0)[i] = z;
      reinterpret_cast<uint4*>(verd1)[i] = z;
    }
    for (size_t i = (n4 << 2) + first; i < n; i += stride) {
      verd0[i] = 0u;
      verd1[i] = 0u;
    }
    for (size_t i = first; i < (size_t)n_vcbits; i += stride) vcbits[i] = 0u;
    return;
  }
  stage_tables(t);
  const auto& ts = t;
  pdl_wait();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int b = blockIdx.x;
  RowCtx& r = ctx[b];
  if (ADV && adv.skip && adv.skip[b]) {  // a row that is done with: its mask and status stay as they are
    if (threadIdx.x == 0) r.complete = 2;
    return;
  }
  const uint16_t* base = c.stack + (size_t)b * t.D;
  const bool vec = ADV == 0 && t.D % 8 == 0 && kStackWin / 8 <= kRowWarps * 32;
  uint4 sv = make_uint4(0u, 0u, 0u, 0u);
  if (ADV) {
    // the row's tokens, on warp 0 (its shared state in the job warps' area,
    // which phase 1 uses only after the barrier below)
    AdvOut o;
    AdvShared& sh = *reinterpret_cast<AdvShared*>(s_ovl2);
    static_assert(sizeof(AdvShared) <= sizeof(s_ovl2), "the advance's shared state overlays the job warps' area");
    const int32_t* toks = adv.tokens + (size_t)b * adv.n_steps;
    AdvRow row;
    if (ADV == 1) {
      // the token with its spelling, and the configuration with its stack: two chains of loads on two warps
      if (warp == 1) {
        const LexToken own = lex_fetch(t, toks, 0, adv.n_steps, lane);
        if (lane == 0) s_own = own;
      } else if (warp == 0) {
        row = advance_load(t, adv.cin, c, b, adv.copy, lane, s_stk);
      }
      __syncthreads();
      if (warp == 0) {
        o = AdvOut{row.depth, row.s.q, row.s.lx, row.flags, GRID_ST_OK, row.s.pc, row.s.wc, row.win, row.depth};
        if (s_own.st != 0) advance_one(t, c, adv.tokens, 0, adv.n_steps, b, s_stk, sh.f, row, s_own, lane, o);
      }
    } else if (warp == 0) {
      const LexToken own = lex_fetch(t, toks, 0, adv.n_steps, lane);
      row = advance_load(t, adv.cin, c, b, adv.copy, lane, s_stk);
      int k0 = 0, keep = row.depth;
      if (feed_fits(t, row, adv.n_steps)) {
        Feed f = feed_begin(row, s_stk, sh.f);
        LexState carry = row.s;
        bool fed = true;
        for (int k = 0; k < adv.n_steps && fed; k = sh.lex.next) {
          const LexToken mine = k == 0 ? own : lex_fetch(t, toks, k, adv.n_steps, lane);
          lex_batch(t, ts, mine, k, adv.n_steps, lane, carry, sh.lex);
          fed = parse_batch(ts, f, sh.lex, k, lane, max_chain_of(t));
          __syncwarp();
        }
        feed_end(ts, f, fed, carry, adv.n_steps, row, c.stack + (size_t)b * t.D, lane, max_chain_of(t));
        k0 = f.tok;
        keep = f.wlow;
      }
      o = AdvOut{row.depth, row.s.q, row.s.lx, row.flags, GRID_ST_OK, row.s.pc, row.s.wc, row.win, keep};
      if (lane == 0 && k0 < adv.n_steps)
        advance_rest(t, ts, c, adv.tokens, k0, adv.n_steps, b, s_stk, sh.f, row, keep, own, o);
    }
    if (threadIdx.x == 0) {
      advance_store(c, b, o);
      s_row[0] = o.flags & 1;
      s_row[1] = o.depth;
      s_row[2] = o.q;
      s_row[3] = o.lx;
      s_pc[0] = o.pc;
      s_pc[1] = o.wc;
      s_adv[0] = o.status;
      s_adv[1] = o.win ? 1 : 0;
      s_adv[2] = o.keep;
      s_status = GRID_ST_OK;
      s_total0 = 0;
      s_nrng = 0;
    }
  } else {
    // the stack window is read before the depth is known (one 16-byte access
    // per thread), in parallel with the configuration
    if (vec && (int)threadIdx.x < kStackWin / 8 && (int)threadIdx.x * 8 < t.D)
      sv = reinterpret_cast<const uint4*>(base)[threadIdx.x];
    if (threadIdx.x == 0) {
      const int lx = c.lx[b];
      s_row[0] = c.flags[b] & 1;
      s_row[1] = c.depth[b];
      s_row[2] = c.q[b];
      s_row[3] = lx;
      s_pc[0] = lx >= 0 ? t.lx_pcats[lx] : 0u;
      s_pc[1] = lx >= 0 ? t.lx_wcats[lx] : 0u;
      s_adv[0] = GRID_ST_OK;
      s_adv[1] = 0;
      s_status = GRID_ST_OK;
      s_total0 = 0;
      s_nrng = 0;
    }
  }
  if (threadIdx.x < 4) s_A0[threadIdx.x] = s_A1[threadIdx.x] = 0u;
  __syncthreads();
  const int complete = s_row[0], depth = s_row[1], q = s_row[2], lx = s_row[3];
  const uint32_t pc0 = s_pc[0], wc0 = s_pc[1];
  if (depth <= kStackWin) {  // the reduce chains below read the stack top repeatedly
    if (ADV && s_adv[1]) {
      // the advance left the row's stack in the window
    } else if (vec) {
      if ((int)threadIdx.x < ((depth + 7) >> 3)) reinterpret_cast<uint4*>(s_stk)[threadIdx.x] = sv;
    } else {
      for (int i = threadIdx.x; i < depth; i += blockDim.x) s_stk[i] = base[i];
    }
    base = s_stk;
  }
  if (!ADV || !s_adv[1]) __syncthreads();
  const int mc = max_chain_of(t);
  const int tbl0 = (q != kStart && t.ci_on) ? ts.tblq(q) : -1;
  int status = GRID_ST_OK;
  // ---- phase 1: all at once
  const bool ranged = q != kStart && tbl0 < 0 && !complete;  // the spellings that go on are those of first-byte ranges
  int lo_r[8], hi_r[8];  // warp 0, a ranged row: spellings by first byte 32 j + lane
  uint32_t cw[8];        // and which of the bytes continue the lexeme
  if (warp == 0) {
    if (ranged) {
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        lo_r[j] = t.first_of_byte[j * 32 + lane];
        hi_r[j] = t.first_of_byte[j * 32 + lane + 1];
      }
      // what can follow the lexeme on each continuing byte that starts a
      // spelling, a byte per lane: known before the allowed set is
      int nc = 0;
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const bool go = hi_r[j] > lo_r[j] && ts.nxt(q * ts.C + ts.cls(j * 32 + lane)) != kDead;
        cw[j] = __ballot_sync(0xffffffffu, go);
        if (go) s_by[nc + __popc(cw[j] & ((1u << lane) - 1u))] = (uint8_t)(j * 32 + lane);
        nc += __popc(cw[j]);
      }
      __syncwarp();
      for (int i = lane; i < nc; i += 32) {
        const int by = s_by[i];
        uint32_t pc2 = 0u, wc2 = 0u;
        const int q2 = ts.nxt(q * ts.C + ts.cls(by));
        lex_step(ts, q2, lx, by, pc2, wc2);
        const Bits4 L = live_prime(ts, q2, pc2);
        s_lv[by] = make_uint4(L.x, L.y, L.z, L.w);
      }
      __syncwarp();
    }
    if (ADV && c.hs) hash_nodes(t, c.hs + (size_t)b * t.D, base, s_adv[2], depth, lane);
  } else if (!complete) {
    // job warps: 32 terminals of one context each, one per lane: tau is
    // allowed iff its reduce chain reaches SHIFT (A0 / A1 are the ballots),
    // and then the allowed set after that shift (A2) comes from one set
    // simulation.  In sigma' (first: its jobs are the longer ones) a warp
    // begins with the forced emission of the pending lexeme, what every token
    // whose first byte ends the lexeme must go through: its candidates' chains
    // run on the lanes, and the first in priority order that reaches SHIFT (or
    // is ignored) is shifted; and $end's lane finds the EOS gate (Sec. 3.2).
    // Emission and terminals share one copy of the chain's code: a third of
    // the issue slots of this kernel went by waiting for instructions.
    const int nw = (t.T1 + 31) >> 5;
    uint16_t* const em = s_em[warp - 1];
    const LArr scr{s_scr[warp - 1] + lane, 32}, ovl{s_ovl2[warp - 1] + lane, 32};
#pragma unroll 1
    for (int job = warp - 1; job < 2 * nw; job += kRowJobWarps) {
      const int cx = job < nw ? 1 : 0, w0 = cx ? job : job - nw;
      bool has = cx == 1 || q != kStart;
      int keep = depth, m = 0;  // the context: base[0:keep] ++ em[0:m]
      int pick_keep = depth, pick_m = 0;
      bool emitting = cx == 1 && q != kStart, picked = false, bound = false;
      Bits4 K = Bits4::zero();
      if (emitting) {
        K = cands(ts, q, wc0);
        if (K.any() && ts.ign.has(K.lowest())) {
          emitting = false;  // an ignored lexeme: the stack stays
        } else if (!K.any()) {
          emitting = has = false;
        }
      }
      int tau = 32 * w0 + lane, a = 0, ko = 0, mo = 0, ns = 0;
#pragma unroll 1
      for (;;) {
        const int kw = K.x ? 0 : (K.y ? 1 : (K.z ? 2 : 3));
        const bool run = emitting ? ((K.word(kw) >> lane) & 1u) && !ts.ign.has(32 * kw + lane)
                                  : has && tau < (cx ? t.T1 : t.n_term) && !ts.ign.has(tau);
        a = 0;
        if (run)
          a = simulate(ts, base, keep, (const uint16_t*)em, m, emitting ? 32 * kw + lane : tau, scr, kMaxOvl, ko, mo,
                       ns, mc);
        if (!emitting) break;
        bound |= __any_sync(0xffffffffu, a < 0);
        const uint32_t ok = __ballot_sync(0xffffffffu, a > 0 && a != kAccept), ig = K.word(kw) & ts.ign.word(kw);
        if (!picked && (ok | ig)) {
          picked = true;
          const int l = __ffs(ok | ig) - 1;
          if ((ok >> l) & 1u) {
            pick_keep = __shfl_sync(0xffffffffu, ko, l);
            const int pns = __shfl_sync(0xffffffffu, ns, l);
            pick_m = pns + 1;
            if (pick_m > kMaxOvl) {
              bound = true;
              pick_m = 0;
            } else if (lane == l) {
#pragma unroll 1
              for (int i = 0; i < pns; ++i) em[i] = scr[i];
              em[pns] = (uint16_t)(a - 1);
            }
            __syncwarp();
          }
        }
        if (kw == 0) K.x = 0u;
        else if (kw == 1) K.y = 0u;
        else if (kw == 2) K.z = 0u;
        else K.w = 0u;
        if (!K.any()) {
          emitting = false;
          has = picked && !bound;
          if (bound) status = GRID_ST_BOUND;
          if (has) {
            keep = pick_keep;
            m = pick_m;
          }
        }
      }
      if (a < 0) status = GRID_ST_BOUND;
      const bool allowed = a > 0 && a != kAccept;
      if (cx == 1 && (t.n_term >> 5) == w0) {
        const bool eos = __any_sync(0xffffffffu, tau == t.n_term && a == kAccept);
        if (lane == 0) s_row[7] = eos;
      }
      if (allowed) {
        Bits4 An = Bits4::zero();
        if (mo + ns + 1 <= kMaxOvl) {
          // the stack after the shift: base[0:ko] ++ em[0:mo] ++ scr[0:ns] ++ (a-1)
#pragma unroll 1
          for (int i = 0; i < mo; ++i) ovl[i] = em[i];
#pragma unroll 1
          for (int i = 0; i < ns; ++i) ovl[mo + i] = scr[i];
          ovl[mo + ns] = (uint16_t)(a - 1);
          bool over = false;
          An = simulate_set(ts, base, ko, ovl, mo + ns + 1, t.par, scr, kMaxOvl, mc, over);
          if (over) status = GRID_ST_BOUND;
        } else {
          status = GRID_ST_BOUND;
        }
        reinterpret_cast<uint4*>(A2)[((size_t)b * 2 + cx) * t.T1 + tau] = make_uint4(An.x, An.y, An.z, An.w);
      }
      const uint32_t word = __ballot_sync(0xffffffffu, allowed);
      if (lane == 0) (cx ? s_A1 : s_A0)[w0] = word;
      if (cx == 1 && w0 == 0) {
        if (lane == 0) {
          s_row[4] = has;
          s_row[5] = keep;
          s_row[6] = m;
        }
        for (int i = lane; i < m; i += 32) s_ovl1[i] = em[i];
      }
      __syncwarp();
    }
  }
  status = __reduce_max_sync(0xffffffffu, status);
  if (lane == 0 && status != GRID_ST_OK) atomicMax(&s_status, status);
  __syncthreads();
  const int emit_ok = complete ? 0 : s_row[4], keep1 = complete ? depth : s_row[5], m1 = complete ? 0 : s_row[6];
  const Bits4 A0 = Bits4::load(s_A0), A1 = Bits4::load(s_A1);
  // ---- phase 2: ranges (warp 0), class selections (the other warps)
  if (!complete) {
    if (warp == 0 && ranged) {
      // continuing first-byte ranges (rows without a CI table for q).  A first
      // byte whose lexeme has no live terminal in A0 u I (category terminals
      // counted only while the lexeme is a prefix of one of their words)
      // rejects every spelling it starts: liveness only shrinks along the
      // lexeme, and any later emission picks among its live terminals.
      int total0 = 0, nrng = 0;
      RowRanges& R = rng[b];
      const Bits4 AI = A0 | ts.ign;
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        if (!cw[j]) continue;
        bool cont = (cw[j] >> lane) & 1u;
        if (cont) {
          const uint4 v = s_lv[j * 32 + lane];
          cont = (Bits4{v.x, v.y, v.z, v.w} & AI).any();
        }
        const int chunks = cont ? (hi_r[j] - lo_r[j] + kRangeSpan - 1) / kRangeSpan : 0;
        const uint32_t bal = __ballot_sync(0xffffffffu, cont);
        int incl = chunks;
        for (int d = 1; d < 32; d <<= 1) {
          int v = __shfl_up_sync(0xffffffffu, incl, d);
          if (lane >= d) incl += v;
        }
        if (cont) {
          const int k = nrng + __popc(bal & ((1u << lane) - 1u));
          R.lo[k] = lo_r[j];
          R.hi[k] = hi_r[j];
          R.cpre[k] = total0 + incl - chunks;
        }
        total0 += __shfl_sync(0xffffffffu, incl, 31);
        nrng += __popc(bal);
      }
      if (lane == 0) {
        R.cpre[nrng] = total0;
        s_total0 = total0;
        s_nrng = nrng;
      }
    } else if (warp >= 1 && t.ci_on) {
      // both contexts' selection words, one at a time per warp 1 ..
      const Bits4 AI0 = A0 | ts.ign, AI1 = A1 | ts.ign;
      const int nw = t.nselw;
      for (int w0 = warp - 1; w0 < nw; w0 += kRowWarps - 1) {
        uint32_t v0, v1;
        select_word(ts, AI0, AI1, w0, lane, v0, v1);
        if (lane == 0 && tbl0 >= 0) sel[(size_t)b * 2 * nw + w0] = v0;
        if (lane == 0 && emit_ok) sel[((size_t)b * 2 + 1) * nw + w0] = v1;
      }
    }
  }
  __syncthreads();
  // ---- the row's context for the later kernels
  if (threadIdx.x == 0) {
    // configuration-keyed cache of the context-independent part (Sec. 4.3):
    // key = (kind, lexer state, emit_ok, A(sigma), A(sigma')); the CD residue
    // is never cached.  A ready entry with this key is read; an empty slot is
    // claimed and filled by k_pack; any other slot is left alone.
    int chit = -1, cfill = -1;
    if (cache.n && !complete) {
      uint32_t key[11];
      key[0] = (q != kStart && tbl0 < 0) ? 1u : 0u;
      key[1] = (uint32_t)q;
      key[2] = (uint32_t)emit_ok;
      for (int k = 0; k < 4; ++k) {
        key[3 + k] = s_A0[k];
        key[7 + k] = emit_ok ? s_A1[k] : 0u;
      }
      unsigned long long hsh = 1469598103934665603ull;  // FNV-1a over the key words
      for (int k = 0; k < 11; ++k) {
        hsh ^= key[k];
        hsh *= 1099511628211ull;
      }
      const int slot = (int)(hsh & (unsigned long long)(cache.n - 1));
      uint32_t* h = cache.hdr + (size_t)slot * 16;
      atomicAdd(&cache.stats[0], 1ull);
      const uint32_t state = *(volatile uint32_t*)h;
      if (state == 2u) {
        bool same = true;
        for (int k = 0; k < 11; ++k) same &= ((volatile uint32_t*)h)[1 + k] == key[k];
        if (same) {
          chit = slot;
          atomicAdd(&cache.stats[1], 1ull);
        }
      } else if (state == 0u && atomicCAS(h, 0u, 1u) == 0u) {
        for (int k = 0; k < 11; ++k) h[1 + k] = key[k];
        cfill = slot;
        atomicAdd(&cache.stats[2], 1ull);
      }
    }
    r.chit = chit;
    r.cfill = cfill;
    for (int k = 0; k < 4; ++k) {
      r.A0[k] = s_A0[k];
      r.A1[k] = emit_ok ? s_A1[k] : 0u;
    }
    r.q = q;
    r.lx = lx;
    r.pc0 = pc0;
    r.wc0 = wc0;
    r.depth = depth;
    r.tbl0 = tbl0;
    r.emit_ok = emit_ok;
    r.eos_ok = complete ? 0 : s_row[7];
    r.complete = complete;
    r.pack_done = 0ull;
    r.keep1 = keep1;
    r.m1 = m1;
    r.work0 = 0;
    r.nrange = s_total0;
    r.nsurv[0] = 0;
    r.nsurv[1] = 0;
    r.nvs[0] = 0;
    r.nvs[1] = 0;
    r.nrng = s_nrng;
    r.fcnt = 0;
    r.fid = 0x7FFFFFFF;
  }
  for (int i = threadIdx.x; i < m1; i += blockDim.x) r.ovl1[i] = s_ovl1[i];
  if (threadIdx.x == 0) r.status = s_adv[0] != GRID_ST_OK ? s_adv[0] : (complete ? GRID_ST_COMPLETE : s_status);
}

// grid = (blocks, B, 2 or 3), 256 threads, kFilterPer records per
// thread (few blocks, all resident at once): compact, per row and context,
// what the walk has to evaluate.
//  - blocks x < cd_blocks: the byte-walked CD spellings that a walk could
//    admit: the class of the first stack-dependent emission must be selected
//    for the context's allowed set and, for sigma', the first byte must end
//    the pending lexeme; survivors go to surv[(b*2 + cx) * cap ...].
//  - the other blocks: the verdict classes whose first event's class is
//    selected (any other record fails at its first emission); survivors go to
//    vsurv[(b*2 + cx) * vcap ...].
// Both lists are in any order.
//  - z = 2, rows without a table (the pending lexeme may be an identifier),
//    context sigma: the spellings of the row's continuing first-byte ranges, a range
//    item per warp, as far as they stay inside the pending lexeme.  Most die
//    there within a few bytes; one that ends there is viable (its last test is
//    the walk's), and its ids' verdicts are set here; one that ends the lexeme
//    goes to the row's unused verdict-class list, for k_walk to walk from the
//    start.  Walked as they came, 32 of a range to a warp, nearly every warp
//    waited for one long walk among 31 short ones: 70% of k_walk's time at
//    256 SQL rows (50,000 items of 13,500 cycles).
constexpr int kScanList = 1024;  // entries of a verdict-class list, at least, for the scan to use it

// Whether the row's range spellings are in its list, of scan_cap entries (-1:
// no scan in this step); else k_walk goes through the ranges.
__device__ __forceinline__ bool scanned(const RowCtx& r, int scan_cap) { return r.nsurv[0] <= scan_cap; }

__device__ __forceinline__ void scan_ranges(const TabT<false>& t, RowCtx& r, const RowRanges& R, int32_t* list,
                                            int vcap, uint32_t* verd, int warp, int warps, int lane,
                                            unsigned long long* work) {
  const Bits4 AI = Bits4{r.A0[0], r.A0[1], r.A0[2], r.A0[3]} | t.ign;
  const int items = r.nrange, nrng = r.nrng;
  const LexState s0{r.q, r.lx, r.pc0, r.wc0};
  int steps = 0, count = 0;
  for (int c = warp; c < items; c += warps) {
    int a = 0, z = nrng;  // range a with cpre[a] <= c < cpre[a + 1]
    while (z - a > 1) {
      const int mid = (a + z) >> 1;
      if (R.cpre[mid] <= c)
        a = mid;
      else
        z = mid;
    }
    const int sp_i = R.lo[a] + (c - R.cpre[a]) * kRangeSpan + lane;
    int res = 0;  // 0 rejected, 1 viable, 2 ends the pending lexeme
    if (sp_i < R.hi[a]) {
      const Spell sp = load_spell(t, sp_i);
      LexState s = s0;
      res = 1;
      int seen = 0;
#pragma unroll 1
      for (int i = 0; i < sp.len; ++i) {
        const int b = sp.at(i);
        const int nq = t.nxt(s.q * t.C + t.cls(b));
        if (nq == kDead) {
          res = 2;
          break;
        }
        ++seen;
        s.q = nq;
        s.lx = lex_step(t, s.q, s.lx, b, s.pc, s.wc);
        if (!(live_prime(t, s.q, s.pc) & AI).any()) {
          res = 0;
          break;
        }
      }
      if (res != 2) {  // decided here (k_walk counts the others)
        steps += seen;
        ++count;
      }
      if (res == 1)
        for (int id = t.id_of_spell[sp_i]; id >= 0; id = t.next_alias[id]) atomicOr(&verd[id >> 5], 1u << (id & 31));
    }
    const uint32_t bal = __ballot_sync(0xffffffffu, res == 2);
    if (bal) {
      int at = 0;
      if (lane == 0) at = atomicAdd(&r.nsurv[0], __popc(bal));
      at = __shfl_sync(0xffffffffu, at, 0) + __popc(bal & ((1u << lane) - 1u));
      if (res == 2 && at < vcap) list[at] = sp_i;
    }
  }
  if (work) {
    if (steps) atomicAdd(&work[0], (unsigned long long)steps);
    if (count) atomicAdd(&work[5], (unsigned long long)count);
  }
}

__global__ void __launch_bounds__(256) k_filter(TabT<false> t, RowCtx* __restrict__ ctx,
                                                const uint32_t* __restrict__ sel, int32_t* __restrict__ surv, int cap,
                                                int32_t* __restrict__ vsurv, int vcap, int cd_blocks,
                                                const RowRanges* __restrict__ rng, uint32_t* __restrict__ verd0,
                                                int words_v, unsigned long long* __restrict__ work) {
  __shared__ int s_warp[8];
  __shared__ int s_base;
  pdl_wait();
  const int b = blockIdx.y, cx = blockIdx.z;
  RowCtx& r = ctx[b];
  const int q = r.q, tbl0 = r.tbl0;
  if (r.complete) return;
  if (cx == 1 && !r.emit_ok) return;
  if (cx == 0 && (q == kStart || tbl0 < 0)) return;
  if (cx == 2) {
    if (q != kStart && tbl0 < 0)
      scan_ranges(t, r, rng[b], vsurv + (size_t)b * 2 * vcap, vcap, verd0 + (size_t)b * words_v,
                  blockIdx.x * 8 + (threadIdx.x >> 5), gridDim.x * 8, threadIdx.x & 31, work);
    return;
  }
  const int tb = cx ? 0 : tbl0;
  const bool vc = (int)blockIdx.x >= cd_blocks;
  const int bx = vc ? (int)blockIdx.x - cd_blocks : (int)blockIdx.x;
  const int len = vc ? t.vc_off[tb + 1] - t.vc_off[tb] : t.cd_off[tb + 1] - t.cd_off[tb];
  const int i0 = bx * (int)blockDim.x * kFilterPer + threadIdx.x;  // records i0 + j * blockDim.x
  if (i0 - (int)threadIdx.x >= len) return;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t* csel = sel + ((size_t)b * 2 + cx) * t.nselw;
  bool pass[kFilterPer];
  int sv[kFilterPer];
#pragma unroll
  for (int j = 0; j < kFilterPer; ++j) {
    const int i = i0 + j * (int)blockDim.x;
    pass[j] = false;
    sv[j] = -1;
    if (i < len) {
      if (vc) {
        sv[j] = i;
        const uint16_t k = t.vc_first[t.vc_off[tb] + i];
        pass[j] = (csel[k >> 5] >> (k & 31)) & 1u;
      } else {
        const int s = t.cd_list[t.cd_off[tb] + i];
        sv[j] = s;
        const uint16_t k = t.cd_key[t.cd_off[tb] + i];
        pass[j] = k == 0xFFFF || ((csel[k >> 5] >> (k & 31)) & 1u);
        if (pass[j] && cx == 1 && q != kStart) {
          const int b0 = (int)(__ldg(&t.spell16[s]).x & 0xFFu);
          pass[j] = t.next[q * t.C + t.byte_class[b0]] == kDead;
        }
      }
    }
  }
  uint32_t bal[kFilterPer];
  int cnt = 0;
#pragma unroll
  for (int j = 0; j < kFilterPer; ++j) {
    bal[j] = __ballot_sync(0xffffffffu, pass[j]);
    cnt += __popc(bal[j]);
  }
  if (lane == 0) s_warp[warp] = cnt;
  __syncthreads();
  if (threadIdx.x == 0) {
    int tot = 0;
    for (int k = 0; k < (int)(blockDim.x >> 5); ++k) {
      const int c = s_warp[k];
      s_warp[k] = tot;
      tot += c;
    }
    s_base = tot ? atomicAdd(vc ? &r.nvs[cx] : &r.nsurv[cx], tot) : 0;
  }
  __syncthreads();
  int at = s_base + s_warp[warp];
  int32_t* out = vc ? vsurv + ((size_t)b * 2 + cx) * vcap : surv + ((size_t)b * 2 + cx) * cap;
#pragma unroll
  for (int j = 0; j < kFilterPer; ++j) {
    if (pass[j]) out[at + __popc(bal[j] & ((1u << lane) - 1u))] = sv[j];
    at += __popc(bal[j]);
  }
}

// Ends of the first three queue segments of a row (x, y, z) and its length
// (w).  Segments: [sigma walked CD spellings, or ranges][sigma' verdict
// classes][sigma' walked CD spellings][sigma verdict classes].  The byte
// walks come first: their items are the longest, and starting them early
// keeps them off the end of the kernel.
__device__ __forceinline__ int4 row_queue(const RowCtx& x, int scan_cap) {
  if (x.complete) return make_int4(0, 0, 0, 0);
  const int ed = x.tbl0 >= 0 || scanned(x, scan_cap) ? (x.nsurv[0] + kSpan - 1) / kSpan : x.nrange;
  const int ea = ed + ((x.nvs[1] + 31) >> 5);
  const int eb = ea + (x.nsurv[1] + kSpan - 1) / kSpan;
  return make_int4(ed, ea, eb, eb + ((x.nvs[0] + 31) >> 5));
}

// Persistent walk.  Every row owns one work queue of items, in four segments:
// the spellings that continue the pending lexeme under sigma (its table's
// byte-walked list, or its continuing first-byte ranges when the state has no
// table), the verdict classes of the start state's table under sigma' (the
// context of tokens whose first byte ends the pending lexeme), the start
// state's byte-walked spellings under sigma', and the verdict classes of the
// pending lexer state's table under sigma.  A block's warps start on one row, blocks
// on different ones, and drain a row's queue item by item; to find work a warp
// examines 32 rows at once (one per lane), from its current row on, and stops
// when no queue has items left.
// A warp keeps the current row's context (allowed sets, sigma' overlay, stack
// mirror) until it moves to another row.
//
// Verdict-class items: 32 of the records that k_filter kept for the row and
// context, one per lane, each evaluated once against the row's stack; an
// accepted record sets its bit in vcbits (cleared by k_row), which k_pack
// reads back per token id.
// List items: up to kSpan spellings that k_filter kept (byte-walked ones whose
// first stack-dependent emission can succeed and, for sigma', whose first byte
// ends the pending lexeme; or, of a row whose ranges it scanned, those that end
// the pending lexeme).  Range items (up to kRangeSpan spellings of one live first-byte
// range; k_row already dropped the first-byte subtrees in which no spelling
// can survive): the range's items interleave, lane j of item i walking
// spelling lo + i + j * (items of the range).  Both kinds share one call of
// walk_bytes, one spelling per lane.
// With COUNT, each lane also counts its work (lexer steps, ACTION and GOTO
// lookups, verdict-class events) in registers and adds the totals to
// work[0..3] when it is done (and the records and spellings it evaluated to
// work[4..5]); the plain instance has no counting code.
struct WalkWarp {
  uint32_t A[2][4];                 // the cached row's A0 and A1
  uint16_t lane[2 * kLaneOvl * 32];  // the lanes' overlays and scratch
  uint16_t win[kWalkWin];           // the row's stack
  uint16_t ovl[kMaxOvl];            // sigma's overlay
};
static_assert(sizeof(WalkWarp) % 16 == 0, "the warps' parts start on 16-byte boundaries");
// k_walk's dynamic shared memory, at most: the tables, then a WalkWarp per warp (24 beside up to 99 KB of tables, 22
// beside the largest that are staged)
constexpr int kWalkSmem = 227 * 1024 - 5120;
static_assert(kWalkSmem - kMaxStage >= 20 * (int)sizeof(WalkWarp), "the largest tables leave room for the warps");

template <bool COUNT, bool ST>
__global__ void __launch_bounds__(kWalkWarps * 32, 1) k_walk(TabT<ST> t, RowCtx* __restrict__ ctx,
                                                             const RowRanges* __restrict__ rng, const uint16_t* stacks,
                                                             const int32_t* __restrict__ surv, int cap,
                                                             const uint32_t* __restrict__ A2,
                                                             uint32_t* __restrict__ verd0,
                                                             uint32_t* __restrict__ verd1, uint32_t* __restrict__ vcbits,
                                                             int vcw, const int32_t* __restrict__ vsurv, int vcap,
                                                             int words_v, int B, int scan_cap,
                                                             unsigned long long* __restrict__ work) {
  WalkWarp& sw = reinterpret_cast<WalkWarp*>(smem + t.blob_bytes)[threadIdx.x >> 5];
  __shared__ int4 s_seg[kWalkRowsCached];
  stage_tables(t);
  const auto& ts = t;
  pdl_wait();
  const int lane = threadIdx.x & 31;
  const int mc = max_chain_of(t);
  const LArr lo{sw.lane + lane, 32}, ls{sw.lane + kLaneOvl * 32 + lane, 32};
  uint32_t cnt[6] = {0u, 0u, 0u, 0u, 0u, 0u};  // the walk's work units, then records and spellings evaluated
  uint32_t* const ctr = COUNT ? cnt : nullptr;
  // queue length and segment ends of every row
  const bool cached = B <= kWalkRowsCached;
  if (cached) {
    for (int i = threadIdx.x; i < B; i += blockDim.x) {
      const int4 e = row_queue(ctx[i], scan_cap);
      s_seg[i] = e;
    }
  }
  __syncthreads();
  // a block's warps start on one row, so that its context, lists and A2 are in the SM's L1 (a step of 256 SQL rows: -4%)
  int row = (int)((long long)blockIdx.x * B / gridDim.x);
  if (B <= (int)gridDim.x) row = blockIdx.x % B;
  int cur = -1;  // row whose context is cached below
  // the lane's walk of that row's last item met a bound: reported before the next one (at the walks themselves, a step
  // of 256 SQL rows took 235 us, here 232)
  bool met = false;
  int tbl0 = -1, depth = 0, q = 0, lx = 0, keep1 = 0, m1 = 0, nrng = 0;
  uint32_t pc0 = 0, wc0 = 0;
  const uint16_t* base = stacks;
  for (;;) {
    if (met) atomicCAS(&ctx[cur].status, GRID_ST_OK, GRID_ST_BOUND);
    met = false;
    // next item of the current row; once that queue is drained, of the first
    // row from there on with items left (32 rows examined at once, one per lane)
    int cidx = -1;
    int4 seg = make_int4(0, 0, 0, 0);
    {
      int got = 0;
      const int4 e = cached ? s_seg[row] : row_queue(ctx[row], scan_cap);
      if (lane == 0 && e.w > 0) got = atomicAdd(&ctx[row].work0, 1);
      got = __shfl_sync(0xffffffffu, got, 0);
      if (e.w > 0 && got < e.w) {
        cidx = got;
        seg = e;
      }
    }
    for (int off = 0; off < B && cidx < 0; off += 32) {
      int rr = row + off + lane;
      rr = rr >= B ? rr - B : rr;
      int4 e = make_int4(0, 0, 0, 0);
      bool has = false;
      if (off + lane < B) {
        e = cached ? s_seg[rr] : row_queue(ctx[rr], scan_cap);
        has = e.w > 0 && *((volatile const int32_t*)&ctx[rr].work0) < e.w;
      }
      uint32_t bal = __ballot_sync(0xffffffffu, has);
      while (bal) {  // warp-uniform
        const int l = __ffs(bal) - 1;
        bal &= bal - 1;
        const int rl = __shfl_sync(0xffffffffu, rr, l);
        const int tl = __shfl_sync(0xffffffffu, e.w, l);
        int got = 0;
        if (lane == 0) got = atomicAdd(&ctx[rl].work0, 1);
        got = __shfl_sync(0xffffffffu, got, 0);
        if (got < tl) {
          cidx = got;
          row = rl;
          seg = make_int4(__shfl_sync(0xffffffffu, e.x, l), __shfl_sync(0xffffffffu, e.y, l),
                          __shfl_sync(0xffffffffu, e.z, l), tl);
          break;
        }
      }
    }
    const int ed = seg.x, ea = seg.y, eb = seg.z;
    if (cidx < 0) break;
    RowCtx& r = ctx[row];
    if (cur != row) {
      cur = row;
      tbl0 = r.tbl0;
      depth = r.depth;
      q = r.q;
      lx = r.lx;
      pc0 = r.pc0;
      wc0 = r.wc0;
      keep1 = r.keep1;
      m1 = r.m1;
      nrng = r.nrng;
      __syncwarp();
      if (lane < 4) {
        sw.A[0][lane] = r.A0[lane];
        sw.A[1][lane] = r.A1[lane];
      }
      for (int i = lane; i < m1 && i < kMaxOvl; i += 32) sw.ovl[i] = r.ovl1[i];
      base = stacks + (size_t)row * t.D;
      if (depth <= kWalkWin) {  // mirror the row's stack: reduce chains read its top repeatedly
        for (int i = lane; i < depth; i += 32) sw.win[i] = base[i];
        base = sw.win;
      }
      __syncwarp();
    }
    // ---- the item: context and source
    const bool c1 = cidx >= ed && cidx < eb;
    const bool is_vc = (cidx >= ed && cidx < ea) || cidx >= eb;
    if (c1 && m1 > kLaneOvl) {  // sigma' overlay larger than a walk lane holds: flag the row
      met = lane == 0;
      continue;
    }
    const uint32_t* Ac = sw.A[c1 ? 1 : 0];
    const uint32_t* A2row = A2 + ((size_t)row * 2 + (c1 ? 1 : 0)) * t.T1 * 4;
    const int ckeep = c1 ? keep1 : depth, cm = c1 ? m1 : 0;
    const int cq = c1 ? kStart : q, clx = c1 ? 0 : lx;
    const uint32_t cpc = c1 ? t.root_pc : pc0, cwc = c1 ? t.root_wc : wc0;
    if (is_vc) {  // 32 surviving verdict classes of the context's table, one per lane
      const int tb = c1 ? 0 : tbl0;
      const int cxi = c1 ? 1 : 0;
      const int item = c1 ? cidx - ed : cidx - eb;
      const int k = item * 32 + lane;
      int res = 0, v = 0;
      if (k < r.nvs[cxi]) {
        if (COUNT) ++cnt[4];
        v = vsurv[((size_t)row * 2 + cxi) * vcap + k];
        Walker w;
        walker_init(w, lo, ls, kLaneOvl, base, ckeep, sw.ovl, cm, cq, clx, cpc, cwc, Ac, A2row, ctr);
        res = eval_record(ts, w, ts.vc_rec + (size_t)(t.vc_off[tb] + v) * kRecLen, mc);
        met |= res < 0;
      }
      if (res > 0) atomicOr(&vcbits[((size_t)row * 2 + cxi) * vcw + (v >> 5)], 1u << (v & 31));
      continue;
    }
    uint32_t* vb = (c1 ? verd1 : verd0) + (size_t)row * words_v;
    const int32_t* list = nullptr;
    int p0, p1, step = 1;
    if (c1 || tbl0 >= 0 || scanned(r, scan_cap)) {  // survivors of k_filter
      const int n = c1 ? r.nsurv[1] : r.nsurv[0];
      list = c1 || tbl0 >= 0 ? surv + ((size_t)row * 2 + (c1 ? 1 : 0)) * cap : vsurv + (size_t)row * 2 * vcap;
      p0 = (c1 ? cidx - ea : cidx) * kSpan;
      p1 = min(n, p0 + kSpan);
    } else {
      const int c0 = cidx;
      const RowRanges& R = rng[row];
      int a = 0, z = nrng;  // range k with cpre[k] <= c0 < cpre[k+1]
      while (z - a > 1) {
        const int mid = (a + z) >> 1;
        if (R.cpre[mid] <= c0)
          a = mid;
        else
          z = mid;
      }
      // the range's items interleave: item i takes spellings lo + i,
      // lo + i + n, lo + i + 2n, ... (n items), so that runs of costly
      // neighbours (long multi-word continuations of one prefix) spread
      // over many warps instead of lengthening one
      step = R.cpre[a + 1] - R.cpre[a];
      p0 = R.lo[a] + (c0 - R.cpre[a]);
      p1 = R.hi[a];
    }
    // ---- one spelling per lane, one walk call site
    {
      int sp_i = -1;
      bool go = false;
      if (list) {
        const int i = p0 + lane;
        go = i < p1;
        if (go) sp_i = list[i];
      } else {
        sp_i = p0 + lane * step;
        go = sp_i < p1;
      }
      if (go) {
        if (COUNT) ++cnt[5];
        const Spell sp = load_spell(ts, sp_i);
        Walker w;
        walker_init(w, lo, ls, kLaneOvl, base, ckeep, sw.ovl, cm, cq, clx, cpc, cwc, Ac, A2row, ctr);
        const int res = walk_bytes(ts, w, sp, mc);
        met |= res < 0;
        if (res > 0)  // the verdict of every id with this spelling, in the mask's layout
          for (int id = t.id_of_spell[sp_i]; id >= 0; id = t.next_alias[id]) atomicOr(&vb[id >> 5], 1u << (id & 31));
      }
    }
  }
  if (COUNT)
    for (int k = 0; k < 6; ++k)
      if (cnt[k]) atomicAdd(&work[k], (unsigned long long)cnt[k]);
}

// -inf over the rejected ones of elements [e0, e1) of a row of logits, by the
// `step` threads of which this is number `tid`; bit e of `word` (element e's
// accept bit is bit e & 31 of word(e >> 5)).  One 256-bit access per 32-byte
// sector of memory (8 fp32 or 16 bf16), so that every store writes a whole
// sector and a warp's store covers 1 KB of contiguous bytes.  A sector whose
// tokens are all rejected is written without being read; a mixed sector is
// read, blended and written; a fully accepted sector is not touched.  Each
// thread takes kBatch sectors at a time: their accept bits loaded
// together, then the rejected sectors stored (they wait on nothing), then the
// mixed sectors read together and stored, so that a thread waits on two rounds
// of loads per batch instead of two per sector.  Where the elements start off
// a sector boundary (SHIFTED) a sector's bits come from two words, and only
// the elements before the first and after the last whole sector are stored one
// by one: stored element by element throughout, 256 rows of 151,937 bf16
// logits took 199 us, this way 18.
constexpr int kApplyBatch = 4;
template <typename T, bool SHIFTED, int kBatch, typename Word>
__device__ __forceinline__ void apply_span(T* row, int e0, int e1, const Word& word, int tid, int step) {
  constexpr int E = 32 / sizeof(T);  // elements per sector
  constexpr uint32_t sfull = (1u << E) - 1u;
  constexpr uint32_t fill = sizeof(T) == 4 ? 0xFF800000u : 0xFF80FF80u;  // -inf in every element of a word
  const int o = SHIFTED ? min(e1, e0 + (int)(((32u - (uint32_t)(uintptr_t)(row + e0)) & 31u) / sizeof(T))) : e0;
  const int nsec = (e1 - o) / E;
  for (int s0 = tid; s0 < nsec; s0 += kBatch * step) {
    uint32_t sb[kBatch];
#pragma unroll
    for (int u = 0; u < kBatch; ++u) {  // the sectors' accept bits
      const int e = o + (s0 + u * step) * E;
      const bool in = s0 + u * step < nsec;
      if (SHIFTED) {
        const uint32_t lo = in ? word(e >> 5) : 0u, hi = in ? word((e + E - 1) >> 5) : 0u;
        sb[u] = in ? __funnelshift_r(lo, hi, e & 31) & sfull : sfull;
      } else {
        sb[u] = in ? (word(e >> 5) >> (e & 31)) & sfull : sfull;
      }
    }
#pragma unroll
    for (int u = 0; u < kBatch; ++u) {  // rejected sectors first: written without a read
      const int e = o + (s0 + u * step) * E;
      if (s0 + u * step < nsec && sb[u] == 0u)
        asm volatile("st.global.v8.b32 [%0], {%1,%1,%1,%1,%1,%1,%1,%1};" ::"l"(row + e), "r"(fill) : "memory");
    }
    uint32_t v[kBatch][8];
#pragma unroll
    for (int u = 0; u < kBatch; ++u) {  // mixed sectors: read
      const int e = o + (s0 + u * step) * E;
      if (s0 + u * step < nsec && sb[u] != 0u && sb[u] != sfull)
        asm volatile("ld.global.v8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                     : "=r"(v[u][0]), "=r"(v[u][1]), "=r"(v[u][2]), "=r"(v[u][3]), "=r"(v[u][4]), "=r"(v[u][5]),
                       "=r"(v[u][6]), "=r"(v[u][7])
                     : "l"(row + e)
                     : "memory");
    }
#pragma unroll
    for (int u = 0; u < kBatch; ++u) {  // mixed sectors: blend and store
      if (s0 + u * step >= nsec || sb[u] == sfull || sb[u] == 0u) continue;
      T* p = row + o + (s0 + u * step) * E;
      uint32_t w[8];
      if (sizeof(T) == 4) {
#pragma unroll
        for (int k = 0; k < 8; ++k) w[k] = ((sb[u] >> k) & 1u) ? v[u][k] : fill;
      } else {
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          const uint32_t lo = (sb[u] >> (2 * k)) & 1u, hi = (sb[u] >> (2 * k + 1)) & 1u;
          w[k] = (lo ? (v[u][k] & 0xFFFFu) : 0xFF80u) | (hi ? (v[u][k] & 0xFFFF0000u) : 0xFF800000u);
        }
      }
      asm volatile("st.global.v8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"l"(p), "r"(w[0]), "r"(w[1]), "r"(w[2]),
                   "r"(w[3]), "r"(w[4]), "r"(w[5]), "r"(w[6]), "r"(w[7])
                   : "memory");
    }
  }
  // the elements outside whole sectors, fewer than E at either end
  if (tid < 2 * E) {
    const int e = tid < E ? e0 + tid : o + nsec * E + tid - E;
    if (tid < E ? e < o : e < e1) {
      if (!((word(e >> 5) >> (e & 31)) & 1u)) {
        if (sizeof(T) == 4)
          reinterpret_cast<uint32_t*>(row)[e] = 0xFF800000u;
        else
          reinterpret_cast<uint16_t*>(row)[e] = 0xFF80u;
      }
    }
  }
}

// grid = (ceil(W / kPackWords), B), kPackWords threads: thread (b, wi) makes
// mask word wi of row b, the 32 token ids 32 wi .. 32 wi + 31 (the id tables
// are padded to a multiple of 32 ids, so each thread reads its ids' class
// codes with 16-byte loads).  Per id: the first byte decides the context (it
// ends the pending lexeme: sigma' and the start state's table; otherwise sigma
// and the pending state's table, or the walk when the state has none), and the
// class code is the place of the id's bit in the context's bit array, the
// class selections followed by the verdict-class bits, which the block stages
// in shared memory; the walks' verdicts come as a word.  Large batches are
// bound by the instructions per id and by the four blocks that 64 registers
// leave an SM: one look-up per id instead of three with the selects between
// them took a step of 256 SQL rows (bf16 logits) from 251 to 234 us, of 32
// rows from 66 to 62.5; without the bound on registers (76 to 95 of them) it
// was 270 and 68.  The last block of a row writes its status (EMPTY_MASK for a
// viable row with no bit set).
//
// With APPLY (1 = fp32, 2 = bf16 logits) the block then masks the logits of its
// ids (Sec. 2 masked decoding, as grid_apply_mask; apply_span).
constexpr int kPackWords = 256;
constexpr int kMaxPack = 96 * 1024;  // bytes of a row's bit arrays, at most
//
// With FORCE (a step of grid_forced_span) the last block of a row also finds
// the row's forced token: where the step's status is OK and the mask holds
// exactly one bit, that id is appended to the span and is the next step's
// token; any other row stops.  Rows that stopped before are left alone.
template <int APPLY, bool CACHE, bool FORCE = false>
__global__ void __launch_bounds__(kPackWords, 4) k_pack(Tables t, RowCtx* __restrict__ ctx, const uint32_t* __restrict__ sel,
                                                     const uint32_t* __restrict__ vcbits, int vcw,
                                                     const uint32_t* __restrict__ verd0,
                                                     const uint32_t* __restrict__ verd1, int words_v,
                                                     uint32_t* __restrict__ mask, int32_t* __restrict__ d_status,
                                                     void* __restrict__ logits, long long stride, int vec_ok,
                                                     CacheDev cache, ForceArgs force) {
  extern __shared__ __align__(16) uint32_t s_dyn[];  // per context: class selections (nselw) | verdict-class bits (vcw)
  __shared__ int s_any, s_cnt, s_id;
  const int b = blockIdx.y;
  const int wi = blockIdx.x * kPackWords + threadIdx.x;
  const bool have = wi < t.W;
  const int nw = t.nselw, len = nw + vcw;
  const int code_vc = t.ncls + 3, code_walk = t.ncls + 4;
  // spec tables only, read before the wait on the walks: the start state's class codes
  uint4 c04[4];
  if (have) {
    const uint4* c = reinterpret_cast<const uint4*>(t.cls_by_id) + 4 * wi;
#pragma unroll
    for (int k = 0; k < 4; ++k) c04[k] = c[k];
  }
  if (threadIdx.x == 0) {
    s_any = 0;
    if (FORCE) {
      s_cnt = 0;
      s_id = 0x7FFFFFFF;
    }
  }
  pdl_wait();
  const RowCtx& rc = ctx[b];
  const int complete = rc.complete, tb = rc.tbl0, emit_ok = rc.emit_ok, q = rc.q;
  const int hit = CACHE ? rc.chit : -1, fill = CACHE ? rc.cfill : -1;
  const bool eos_ok = rc.eos_ok != 0 && !complete;
  if (complete == 2) return;
  // The contexts' bit arrays, indexed by class code: a context that k_row did
  // not prepare (a completed row, sigma' without a forced emission, sigma
  // without a table) has no bit set, so that no id asks for its context again.
  {
    const bool c0 = !complete && tb >= 0, c1 = !complete && emit_ok;
    const uint32_t* vb = vcbits + (size_t)b * 2 * vcw;
    for (int i = threadIdx.x; i < len; i += kPackWords) {
      uint32_t x0 = 0u, x1 = 0u;
      if (i < nw) {
        if (t.ci_on && c0) x0 = sel[(size_t)b * 2 * nw + i];
        if (t.ci_on && c1) x1 = sel[((size_t)b * 2 + 1) * nw + i];
      } else {
        if (c0) x0 = vb[i - nw];
        if (c1) x1 = vb[vcw + i - nw];
      }
      s_dyn[i] = x0;
      s_dyn[len + i] = x1;
    }
  }
  uint32_t killw = 0u, m = 0u;
  uint4 ct4[4];
  if (have && !complete) {
    // bit j: id 32 wi + j's first byte ends the pending lexeme (context sigma')
    killw = t.killw[(size_t)q * t.W + wi];
    // the walks' verdicts (set for walked ids alone, whose codes have no bit in the arrays)
    m = verd0[(size_t)b * words_v + wi] & ~killw;
    if (emit_ok) m |= verd1[(size_t)b * words_v + wi] & killw;
    if (tb >= 0) {
      const uint4* c = reinterpret_cast<const uint4*>(t.cls_by_id + (size_t)tb * t.Vp) + 4 * wi;
#pragma unroll
      for (int k = 0; k < 4; ++k) ct4[k] = c[k];
    }
  }
  __syncthreads();
  if (have && !complete) {
    const uint32_t c0w[16] = {c04[0].x, c04[0].y, c04[0].z, c04[0].w, c04[1].x, c04[1].y, c04[1].z, c04[1].w,
                              c04[2].x, c04[2].y, c04[2].z, c04[2].w, c04[3].x, c04[3].y, c04[3].z, c04[3].w};
    uint32_t ctw[16];
#pragma unroll
    for (int k = 0; k < 16; ++k) ctw[k] = code_walk | ((uint32_t)code_walk << 16);
    if (tb >= 0) {
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        ctw[4 * k] = ct4[k].x;
        ctw[4 * k + 1] = ct4[k].y;
        ctw[4 * k + 2] = ct4[k].z;
        ctw[4 * k + 3] = ct4[k].w;
      }
    }
    uint32_t dep = 0u;  // the residue: ids decided per row, in a context that exists
    if (t.vc_inline) {
#pragma unroll
      for (int j = 0; j < 32; ++j) {
        const bool cx = (killw >> j) & 1u;
        const uint32_t code = ((cx ? c0w[j >> 1] : ctw[j >> 1]) >> ((j & 1) * 16)) & 0xFFFFu;
        if (CACHE && (int)code >= code_vc && (!cx || emit_ok)) dep |= 1u << j;
        m |= ((s_dyn[(cx ? len : 0) + (code >> 5)] >> (code & 31)) & 1u) << j;
      }
    } else {
#pragma unroll
      for (int j = 0; j < 32; ++j) {
        const bool cx = (killw >> j) & 1u;
        uint32_t code = ((cx ? c0w[j >> 1] : ctw[j >> 1]) >> ((j & 1) * 16)) & 0xFFFFu;
        if (CACHE && (int)code >= code_vc && (!cx || emit_ok)) dep |= 1u << j;
        if ((int)code == code_vc)  // the verdict class, looked up
          code = 32 * nw + t.vc_by_id[(size_t)(cx ? 0 : tb) * t.Vp + 32 * wi + j];
        m |= ((s_dyn[(cx ? len : 0) + (code >> 5)] >> (code & 31)) & 1u) << j;
      }
    }
    if (CACHE) {
      if (fill >= 0) {
        cache.ci[(size_t)fill * t.W + wi] = m & ~dep;
        cache.sel[(size_t)fill * t.W + wi] = dep;
      }
      // a cache hit gives the context-independent bits; only the residue ids are decided here
      if (hit >= 0) m = cache.ci[(size_t)hit * t.W + wi] | (m & cache.sel[(size_t)hit * t.W + wi]);
    }
    const int ej = t.eos - 32 * wi;
    if (ej >= 0 && ej < 32 && eos_ok) m |= 1u << ej;  // the EOS gate is stack-dependent: never cached
  }
  if (have) {
    mask[(size_t)b * t.W + wi] = m;
    if (m) s_any = 1;
    if (FORCE && m) {
      atomicAdd(&s_cnt, __popc(m));
      atomicMin(&s_id, 32 * wi + __ffs(m) - 1);
    }
  }
  if (APPLY) {
    using T = typename std::conditional<APPLY == 1, uint32_t, uint16_t>::type;
    T* row = reinterpret_cast<T*>(logits) + (size_t)b * stride;
    if (APPLY == 2 && vec_ok) {
      // a thread's word is two bf16 sectors of its own: written from the
      // register (256 SQL rows: 247 us a step, 255 us through shared memory)
      if (have) {
        uint32_t v[2][8];
#pragma unroll
        for (int u = 0; u < 2; ++u) {  // mixed whole sectors: read
          const int e = 32 * wi + 16 * u;
          const uint32_t sb = (m >> (16 * u)) & 0xFFFFu;
          if (e + 16 <= t.V && sb != 0u && sb != 0xFFFFu)
            asm volatile("ld.global.v8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                         : "=r"(v[u][0]), "=r"(v[u][1]), "=r"(v[u][2]), "=r"(v[u][3]), "=r"(v[u][4]), "=r"(v[u][5]),
                           "=r"(v[u][6]), "=r"(v[u][7])
                         : "l"(row + e)
                         : "memory");
        }
#pragma unroll
        for (int u = 0; u < 2; ++u) {  // blend and store
          const int e = 32 * wi + 16 * u;
          const uint32_t sb = (m >> (16 * u)) & 0xFFFFu;
          if (e >= t.V || sb == 0xFFFFu) continue;
          if (e + 16 <= t.V) {
            uint32_t w[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) {
              const uint32_t lo = (sb >> (2 * k)) & 1u, hi = (sb >> (2 * k + 1)) & 1u;
              w[k] = sb == 0u ? 0xFF80FF80u
                              : (lo ? (v[u][k] & 0xFFFFu) : 0xFF80u) | (hi ? (v[u][k] & 0xFFFF0000u) : 0xFF800000u);
            }
            asm volatile("st.global.v8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"l"(row + e), "r"(w[0]), "r"(w[1]),
                         "r"(w[2]), "r"(w[3]), "r"(w[4]), "r"(w[5]), "r"(w[6]), "r"(w[7])
                         : "memory");
          } else {
            for (int k = 0; e + k < t.V; ++k)
              if (!((sb >> k) & 1u)) row[e + k] = (T)0xFF80u;
          }
        }
      }
    } else {
      // the logits of the block's ids, by their bits in shared memory:
      // consecutive threads take consecutive sectors, whatever word they
      // packed (32 SQL rows, fp32: 68.5 -> 65 us a step; 27 rows of 32,001
      // fp32 logits, off the sector boundaries: 50.9 -> 46.2 us)
      __syncthreads();
      s_dyn[threadIdx.x] = m;  // (the selections were read)
      __syncthreads();
      const int wb = blockIdx.x * kPackWords;
      auto word = [&](int w) { return s_dyn[w - wb]; };
      const int e1 = min(t.V, 32 * (wb + kPackWords));
      constexpr int kEach = 32 * (int)sizeof(T) / 32;  // sectors per thread of a whole block
      if (vec_ok)
        apply_span<T, false, kEach>(row, 32 * wb, e1, word, threadIdx.x, kPackWords);
      else
        apply_span<T, true, kEach>(row, 32 * wb, e1, word, threadIdx.x, kPackWords);
    }
  }
  if (CACHE && fill >= 0) __threadfence();  // the entry's words before its readiness
  __syncthreads();
  // one atomic per block counts the block for its row and carries whether it
  // set a bit; the row's last block writes the status (and marks a cache
  // entry the row filled ready: all blocks have written their words)
  if (threadIdx.x == 0) {
    if (FORCE && s_cnt) {
      atomicAdd(&ctx[b].fcnt, s_cnt);
      atomicMin(&ctx[b].fid, s_id);
      __threadfence();
    }
    const unsigned long long old = atomicAdd(&ctx[b].pack_done, 1ull + (s_any ? (1ull << 32) : 0ull));
    if ((uint32_t)old == gridDim.x - 1) {
      int st = atomicAdd(&ctx[b].status, 0);
      if (st == GRID_ST_OK && (old >> 32) == 0ull && !s_any) st = GRID_ST_EMPTY_MASK;
      d_status[b] = st;
      if (FORCE) {
        __threadfence();
        const bool one = st == GRID_ST_OK && atomicAdd(&ctx[b].fcnt, 0) == 1;
        const int id = atomicMin(&ctx[b].fid, 0x7FFFFFFF);
        if (one) {
          force.span[(size_t)b * force.max_span + force.pos] = id;
          force.span_len[b] = force.pos + 1;
        }
        force.tok[b] = one ? id : -1;
        force.stop[b] = one ? 0 : 1;
      }
      if (CACHE && fill >= 0) {
        __threadfence();
        atomicExch(cache.hdr + (size_t)fill * 16, 2u);
      }
    }
  }
}

// What a row's advance leaves, by its warp (`out` is lane 0's).
template <class T>
__device__ __forceinline__ void advance_done(const T& t, const DevConfigs& cout, const AdvOut& out,
                                             int32_t* __restrict__ d_status, int b, int lane) {
  if (lane == 0) {
    advance_store(cout, b, out);
    d_status[b] = out.status;
  }
  if (cout.hs) {
    __syncwarp();
    hash_nodes(t, cout.hs + (size_t)b * t.D, cout.stack + (size_t)b * t.D, __shfl_sync(0xffffffffu, out.keep, 0),
               __shfl_sync(0xffffffffu, out.depth, 0), lane);
  }
}

// Several tokens per row, a block of two warps per row: warp 1 lexes the next
// batch of tokens while warp 0 parses the last one.
template <bool ST>
__global__ void __launch_bounds__(64, 3) k_advance(TabT<ST> t, DevConfigs cin, DevConfigs cout,
                                                const int32_t* __restrict__ tokens, int n_steps,
                                                int32_t* __restrict__ d_status, int B, int copy) {
  __shared__ __align__(16) uint16_t s_stk[kStackWin];
  __shared__ AdvShared sh;
  __shared__ LexBatch s_lex1;  // with sh.lex: the batch being parsed and the one being made
  __shared__ int s_stop[2];    // set while batch j is parsed, read before batch j + 1 is: j odd, j even
  stage_tables(t);
  const auto& ts = t;
  pdl_wait();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int b = blockIdx.x;
  const int mc = max_chain_of(t);
  const int32_t* toks = tokens + (size_t)b * n_steps;
  AdvRow row;
  Feed f;
  LexToken own;
  bool fed = true;
  own = lex_fetch(t, toks, 0, n_steps, lane);
  if (warp == 0) {
    row = advance_load(t, cin, cout, b, copy, lane, s_stk);
    f = feed_begin(row, s_stk, sh.f);
    if (lane == 0) {
      s_stop[0] = 0;
      s_stop[1] = feed_fits(t, row, n_steps) ? 0 : 1;
    }
    fed = feed_fits(t, row, n_steps);
  } else {
    row = advance_config(t, copy ? cin : cout, b, lane);
  }
  LexState carry = row.s;
  for (int k = 0, j = 0, next; k < n_steps; k = next, ++j) {
    LexBatch& L = j & 1 ? s_lex1 : sh.lex;
    if (warp == 1 && feed_fits(t, row, n_steps)) {
      const LexToken mine = k == 0 ? own : lex_fetch(t, toks, k, n_steps, lane);
      lex_batch(t, ts, mine, k, n_steps, lane, carry, L);
    }
    __syncthreads();
    next = L.next;
    if (((volatile int*)s_stop)[(j + 1) & 1]) break;
    if (warp == 0) {
      fed = parse_batch(ts, f, L, k, lane, mc);
      carry = L.end;
      if (lane == 0) s_stop[j & 1] = fed ? 0 : 1;
    }
  }
  if (warp != 0) return;
  int k0 = 0, keep = row.depth;
  if (feed_fits(t, row, n_steps)) {
    feed_end(ts, f, fed, carry, n_steps, row, cout.stack + (size_t)b * t.D, lane, mc);
    k0 = f.tok;
    keep = f.wlow;
  }
  AdvOut out{row.depth, row.s.q, row.s.lx, row.flags, GRID_ST_OK, row.s.pc, row.s.wc, row.win, keep};
  if (lane == 0 && k0 < n_steps)
    advance_serial(t, ts, cout, tokens, k0, n_steps, b, s_stk, sh.f, row, keep, own, out);
  advance_done(t, cout, out, d_status, b, lane);
}

// One token per row, or a few in large batches: a warp per row, in large batches
// several rows in a block, so that the tables are staged once for them (one
// token, a row a block and eight: 1,024 SQL rows 17.4 and 13.2 us, 4,096 rows
// 43.4 and 20.4; 32 expression rows in a graph 3.3 and 3.7).
constexpr int kOneRows = 8;  // rows of a block, at most
constexpr int kFewTokens = 8;  // tokens of a row that k_advance_one is given, at most
struct OneShared {
  uint16_t win[kStackWin];
  FeedShared f;
};
static_assert(sizeof(OneShared) % 16 == 0, "the rows' parts start on 16-byte boundaries");

template <bool ST>
__global__ void __launch_bounds__(kOneRows * 32) k_advance_one(TabT<ST> t, DevConfigs cin, DevConfigs cout,
                                                               const int32_t* __restrict__ tokens, int n_steps,
                                                               int32_t* __restrict__ d_status, int B, int copy) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  OneShared& sh = reinterpret_cast<OneShared*>(smem + t.blob_bytes)[warp];
  stage_tables(t);
  pdl_wait();
  const int b = blockIdx.x * (blockDim.x >> 5) + warp;
  if (b >= B) return;
  const LexToken own = lex_fetch(t, tokens + (size_t)b * n_steps, 0, n_steps, lane);  // lane k: token k
  AdvRow row = advance_load(t, cin, cout, b, copy, lane, sh.win);
  AdvOut out{row.depth, row.s.q, row.s.lx, row.flags, GRID_ST_OK, row.s.pc, row.s.wc, row.win, row.depth};
#pragma unroll 1
  for (int k = 0; k < n_steps; ++k) {
    LexToken x;
    x.st = __shfl_sync(0xffffffffu, own.st, k);
    if (x.st == 0) continue;
    x.sp.len = __shfl_sync(0xffffffffu, own.sp.len, k);
    x.sp.head = make_uint4(__shfl_sync(0xffffffffu, own.sp.head.x, k), __shfl_sync(0xffffffffu, own.sp.head.y, k),
                           __shfl_sync(0xffffffffu, own.sp.head.z, k), __shfl_sync(0xffffffffu, own.sp.head.w, k));
    x.sp.all = reinterpret_cast<const uint8_t*>(__shfl_sync(0xffffffffu, (unsigned long long)own.sp.all, k));
    if (!advance_one(t, cout, tokens, k, n_steps, b, sh.win, sh.f, row, x, lane, out)) break;
  }
  advance_done(t, cout, out, d_status, b, lane);
}

// In-place -inf fill (apply_span), grid = (blocks per row, B): few, long-lived
// blocks (block scheduling, not memory, bounds a grid of one short block per
// 256 sectors).
template <typename T, bool SHIFTED>
__global__ void __launch_bounds__(256) k_apply(const uint32_t* __restrict__ mask, T* __restrict__ logits, int B,
                                               int V, int W, long long stride) {
  pdl_wait();
  const uint32_t* mrow = mask + (size_t)blockIdx.y * W;
  apply_span<T, SHIFTED, kApplyBatch>(logits + (size_t)blockIdx.y * stride, 0, V, [&](int w) { return mrow[w]; },
                         blockIdx.x * blockDim.x + threadIdx.x, gridDim.x * blockDim.x);
}

// Launch with programmatic stream serialization: the kernel may begin (stage
// its tables) while the previous kernel in the stream drains; it waits for
// that kernel's results with griddepcontrol.wait (pdl_wait).
template <typename... KArgs, typename... Args>
static cudaError_t launch_pdl(void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                              Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, std::forward<Args>(args)...);
}

size_t align16(size_t x) { return (x + 15) & ~size_t(15); }

}  // namespace
}  // namespace grid

using namespace grid;

int grid::g_sms = 152;  // SM count of the current device, set by grid_specialize

// The dynamic shared-memory cap is a per-function attribute shared by every
// spec in the process, so it is raised once to the largest staged block
// allowed instead of to this spec's size.
static int set_smem_limits() {
  const int dyn = std::max(kMaxStage + kOneRows * (int)sizeof(OneShared), kMaxPack);
  const void* kernels[] = {
      (const void*)k_classify<true>, (const void*)k_events<true>, (const void*)k_advance<true>,
      (const void*)k_advance_one<true>,
      (const void*)k_row<0, true>, (const void*)k_row<1, true>, (const void*)k_row<2, true>,
      // k_pack: one row's class selections and verdict-class bits, two contexts
      (const void*)k_pack<0, false>, (const void*)k_pack<1, false>, (const void*)k_pack<2, false>,
      (const void*)k_pack<0, true>, (const void*)k_pack<1, true>, (const void*)k_pack<2, true>,
      (const void*)k_pack<0, false, true>};
  for (const void* k : kernels) GRID_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, dyn));
  const void* walks[] = {(const void*)k_walk<false, true>, (const void*)k_walk<true, true>,
                         (const void*)k_walk<false, false>, (const void*)k_walk<true, false>};
  for (const void* k : walks)
    GRID_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, kWalkSmem));
  return GRID_OK;
}

// Bounds of the reduce chains under one lookahead (Tables::chain_rate,
// chain_base), 0 where none is shown.  A chain's reductions are the nodes of
// parse trees: nodes of empty yield; nodes over one symbol that is not empty
// beside empty ones; and nodes over two or more such symbols, each of which
// leaves fewer of them on the stack (at most one per stack entry).  Between
// two of the last kind, at one place of the stack, no nonterminal comes twice
// (the grammar would be ambiguous, and its tables would conflict), so a run of
// the second kind is a path in the graph of its productions.  What a chain
// pushes is one symbol and empty ones on top of it: a path in the goto graph
// over nullable nonterminals.
static void chain_bounds(const HostGrammar& h, Tables& t) {
  t.chain_rate = t.chain_base = 0;
  const int T1 = h.T1, N = h.NNT;
  constexpr int kBig = 1 << 12;
  // eps[A]: the most nodes of an empty tree of A (-1: A is not nullable)
  std::vector<int> eps(N, -1);
  for (int round = 0; round <= N + 1; ++round) {
    bool changed = false;
    for (int p = 0; p < h.P; ++p) {
      int sum = 1;
      for (int j = h.prod_off[p]; j < h.prod_off[p + 1] && sum > 0; ++j) {
        const int X = h.prod_rhs[j];
        sum = X < T1 || eps[X - T1] < 0 ? 0 : std::min(kBig, sum + eps[X - T1]);
      }
      if (sum > eps[h.plhs[p]] && sum > 0) {
        eps[h.plhs[p]] = sum;
        changed = true;
      }
    }
    if (!changed) break;
    if (round == N + 1) return;  // empty trees without a bound
  }
  // up[A]: the most steps of a run of second-kind nodes (and their empty parts) that ends in A
  std::vector<int> up(N, 0);
  int emax = 0, longest = 0;
  for (int round = 0; round <= N + 1; ++round) {
    bool changed = false;
    for (int p = 0; p < h.P; ++p) {
      int sum = 0, solid = 0;
      for (int j = h.prod_off[p]; j < h.prod_off[p + 1]; ++j) {
        const int X = h.prod_rhs[j];
        if (X >= T1 && eps[X - T1] > 0)
          sum = std::min(kBig, sum + eps[X - T1]);
        else
          ++solid;
      }
      emax = std::max(emax, sum);
      if (solid > 1) continue;
      for (int j = h.prod_off[p]; j < h.prod_off[p + 1]; ++j) {  // the symbol that is not empty
        const int X = h.prod_rhs[j];
        if (solid == 1 && X >= T1 && eps[X - T1] > 0) continue;
        const int v = std::min(kBig, (X < T1 ? 0 : up[X - T1]) + 1 + sum);
        if (v > up[h.plhs[p]]) {
          up[h.plhs[p]] = v;
          changed = true;
        }
      }
    }
    if (!changed) break;
    if (round == N + 1) return;
  }
  for (int A = 0; A < N; ++A) longest = std::max(longest, up[A]);
  // the longest path over nullable gotos
  std::vector<int> len(h.S, 0);
  int path = 0;
  for (int round = 0; round <= h.S + 1; ++round) {
    bool changed = false;
    for (int s = 0; s < h.S; ++s)
      for (int A = 0; A < N; ++A) {
        const int g = h.go[(size_t)s * N + A];
        if (eps[A] < 0 || g >= h.S || len[g] + 1 <= len[s]) continue;
        len[s] = len[g] + 1;
        path = std::max(path, len[s]);
        changed = true;
      }
    if (!changed) break;
    if (path + 2 >= kLaneOvl || round == h.S + 1) return;
  }
  const int rate = 1 + emax + longest + 1, base = (path + 1) * (emax + 1);
  if (path + 2 >= kLaneOvl || emax >= kBig || longest >= kBig) return;
  t.chain_rate = rate;
  t.chain_base = base;
}

// The distinct terminal sets of the CI class ids (four words each, in the order
// of their first id) and each id's set: events and final tests use nothing else
// of a class, so that ids with equal sets are one class from there on.
static void class_sets(const HostGrammar& h, std::vector<uint32_t>& sets, std::vector<uint16_t>& map) {
  const int n = (2 * h.Q) << h.n_cat;
  map.resize(n);
  std::unordered_map<std::string, uint16_t> seen;
  for (int c = 0; c < n; ++c) {
    const int hi = c >> h.n_cat, kind = hi / h.Q, q = hi - kind * h.Q;
    const uint32_t* v = (kind ? h.acc : h.live).data() + (size_t)q * 4;
    uint32_t w[4];
    for (int k = 0; k < 4; ++k) w[k] = v[k] & ~h.catmask[k];
    for (int k = 0; k < h.n_cat; ++k) {
      const int tau = h.cat_term[k];
      if ((c >> k) & 1) w[tau >> 5] |= v[tau >> 5] & (1u << (tau & 31));
    }
    const auto it = seen.emplace(std::string(reinterpret_cast<const char*>(w), 16), (uint16_t)(sets.size() / 4));
    if (it.second) sets.insert(sets.end(), w, w + 4);
    map[c] = it.first->second;
  }
}

// Tables::ev_list and Tables::live_any.
static void lexeme_tables(const HostGrammar& h, std::vector<uint64_t>& ev, std::vector<uint32_t>& live) {
  const int sets = 1 << h.n_cat;
  ev.assign((size_t)h.Q * sets, 0);
  live.assign(((size_t)h.Q * sets + 31) / 32, 0u);
  for (int q = 0; q < h.Q; ++q)
    for (int c = 0; c < sets; ++c) {
      auto has = [&](const std::vector<uint32_t>& set, int tau) {
        if (!((set[q * 4 + (tau >> 5)] >> (tau & 31)) & 1u)) return false;
        if (!((h.catmask[tau >> 5] >> (tau & 31)) & 1u)) return true;
        for (int k = 0; k < h.n_cat; ++k)
          if (h.cat_term[k] == tau && ((c >> k) & 1)) return true;
        return false;
      };
      uint64_t list = 0;
      int n = 0;
      bool ign = false;
      for (int tau = 0; tau < h.n_term; ++tau) {
        if (has(h.live, tau)) live[((size_t)q * sets + c) >> 5] |= 1u << ((q * sets + c) & 31);
        if (ign || !has(h.acc, tau)) continue;
        ign = (h.ignored[tau >> 5] >> (tau & 31)) & 1u;
        if (!ign && n < kLexCand) list |= (uint64_t)tau << (8 * n);
        n += ign ? 0 : 1;
      }
      ev[(size_t)q * sets + c] = n > kLexCand ? (uint64_t)0x7F << 56 : list | ((uint64_t)(n | (ign ? 0x80 : 0)) << 56);
    }
}

// grid_specialize's work.  The caller frees what it leaves, after success and
// after every error: what only the specialization needs is tmp's and keep's
// (the host buffers of copies in flight); after an error, the spec too.
static int specialize(const grid_grammar* g, const grid_vocab* v, cudaStream_t st, grid_spec* s, Arena& tmp,
                      std::vector<std::vector<uint8_t>>& keep) {
  const HostGrammar& h = g->h;
  const HostVocab& hv = v->h;
  s->g = g;
  s->v = v;
  Tables& t = s->t;
  std::memset(&t, 0, sizeof(t));
  t.n_term = h.n_term;
  t.T1 = h.T1;
  t.S = h.S;
  t.NNT = h.NNT;
  t.P = h.P;
  t.Q = h.Q;
  t.C = h.C;
  t.n_cat = h.n_cat;
  t.LN = h.LN;
  t.NS = hv.NS;
  t.V = hv.V;
  t.eos = hv.eos;
  t.W = (hv.V + 31) / 32;
  t.D = h.max_depth;
  chain_bounds(h, t);
  t.ign = Bits4{h.ignored[0], h.ignored[1], h.ignored[2], h.ignored[3]};
  t.cm = Bits4{h.catmask[0], h.catmask[1], h.catmask[2], h.catmask[3]};
  for (int c = 0; c < h.n_cat; ++c) t.cat_term[c] = h.cat_term[c];
  uint32_t par[4] = {0u, 0u, 0u, 0u};
  for (int tau = 0; tau < h.n_term; ++tau) par[tau >> 5] |= 1u << (tau & 31);
  t.par = Bits4{par[0] & ~h.ignored[0], par[1] & ~h.ignored[1], par[2] & ~h.ignored[2], par[3] & ~h.ignored[3]};
  // per LALR state: the terminals that shift, and the terminals grouped by
  // the production they reduce by (for simulating a set of terminals at once)
  std::vector<uint32_t> shift_mask((size_t)h.S * 4, 0u), red_mask;
  // reduce actions carry their production's length and left-hand side
  // (-(1 + (plen << 10 | lhs))), so that a reduce step needs no second lookup
  int max_plen = 0;
  for (int pr = 0; pr < h.P; ++pr) max_plen = std::max(max_plen, (int)h.plen[pr]);
  if (h.NNT >= 1024 || max_plen >= 32)
    return set_error(GRID_E_TOO_LARGE, "grammar exceeds the packed reduce encoding (1024 nonterminals, "
                                       "right-hand sides of 31 symbols)");
  std::vector<int16_t> action16(h.action.size());
  for (size_t i = 0; i < h.action.size(); ++i) {
    const int a = h.action[i];
    action16[i] = a >= 0 ? (int16_t)a : (int16_t)(-(1 + ((h.plen[-a - 1] << 10) | h.plhs[-a - 1])));
  }
  std::vector<uint32_t> red_off(h.S + 1, 0);
  std::vector<uint16_t> red_p;
  for (int st = 0; st < h.S; ++st) {
    std::vector<std::pair<int, std::array<uint32_t, 4>>> groups;
    for (int tau = 0; tau < h.T1; ++tau) {
      const int a = h.action[(size_t)st * h.T1 + tau];
      if (a > 0 && a != kAccept) {
        shift_mask[(size_t)st * 4 + (tau >> 5)] |= 1u << (tau & 31);
      } else if (a < 0) {
        const int pr = -a - 1;
        auto it = std::find_if(groups.begin(), groups.end(), [&](const auto& g) { return g.first == pr; });
        if (it == groups.end()) {
          groups.push_back({pr, {0u, 0u, 0u, 0u}});
          it = groups.end() - 1;
        }
        it->second[tau >> 5] |= 1u << (tau & 31);
      }
    }
    for (const auto& g : groups) {
      red_p.push_back((uint16_t)((h.plen[g.first] << 10) | h.plhs[g.first]));
      for (int w = 0; w < 4; ++w) red_mask.push_back(g.second[w]);
    }
    red_off[st + 1] = (uint32_t)red_p.size();
  }
  // lexeme tables, where the class ids fit (the bound of ci_on below)
  std::vector<uint64_t> ev_list;
  std::vector<uint32_t> live_any;
  const long n_ids = (long)(2 * h.Q) << h.n_cat;  // CI class ids
  t.ci_on = n_ids < (long)kClsFirstCode ? 1 : 0;
  std::vector<uint32_t> sets;
  std::vector<uint16_t> cls_map;
  if (t.ci_on) {
    lexeme_tables(h, ev_list, live_any);
    class_sets(h, sets, cls_map);
  } else {
    t.chain_rate = 0;
  }
  s->n_classes = t.ci_on ? (int)n_ids : 0;
  s->has_cats = h.n_cat > 0;
  t.ncls = (int)(sets.size() / 4);
  t.nselw = (t.ncls + kPackCodes + 31) / 32;
  std::vector<uint32_t> cat_live((h.Q + 31) / 32, 0u);
  for (int q = 0; q < h.Q; ++q)
    for (int w = 0; w < 4; ++w)
      if (h.live[q * 4 + w] & h.catmask[w]) cat_live[q >> 5] |= 1u << (q & 31);
  // precomputed lexer states: the start state and every state at which no
  // lexicon category is live (there the lexicon node cannot matter)
  std::vector<int32_t> tq{kStart};
  std::vector<int16_t> tbl_of_q(h.Q, -1);
  tbl_of_q[kStart] = 0;
  if (t.ci_on) {
    for (int q = 2; q < h.Q; ++q) {
      if (!((cat_live[q >> 5] >> (q & 31)) & 1u) && tq.size() < 4096) {
        tbl_of_q[q] = (int16_t)tq.size();
        tq.push_back(q);
      }
    }
  }
  t.n_tbl = (int)tq.size();
  // staged block: byte classes, DFA, acc/live, ACTION, GOTO, left-hand
  // sides, shift masks and reduce groups, live lexemes, states
  // with live categories, tables of states, class sets (where they are few
  // and there is room: the kernels find them in global memory too)
  constexpr int kSec = 15;
  std::vector<size_t> off(kSec + 1, 0);
  const size_t sizes[kSec] = {256, h.next.size() * 2, h.acc.size() * 4, h.live.size() * 4, action16.size() * 2,
                              h.go.size() * 2, h.plhs.size() * 2, shift_mask.size() * 4,
                              red_off.size() * 4, red_p.size() * 2, red_mask.size() * 4, live_any.size() * 4,
                              cat_live.size() * 4, tbl_of_q.size() * 2, sets.size() * 4};
  const void* srcs[kSec] = {h.byte_class, h.next.data(), h.acc.data(), h.live.data(), action16.data(),
                            h.go.data(), h.plhs.data(), shift_mask.data(), red_off.data(),
                            red_p.data(), red_mask.data(), live_any.data(), cat_live.data(),
                            tbl_of_q.data(), sets.data()};
  for (int k = 0; k < kSec; ++k) off[k + 1] = align16(off[k] + sizes[k]);
  const bool stage_sets = !sets.empty() && t.ncls <= kStagedSets && off[kSec] <= (size_t)kMaxStage;
  if (!stage_sets) off[kSec] = off[kSec - 1];
  std::vector<uint8_t> blob(off[kSec], 0);
  for (int k = 0; k < (stage_sets ? kSec : kSec - 1); ++k)
    if (sizes[k]) std::memcpy(blob.data() + off[k], srcs[k], sizes[k]);
  Arena& a = s->mem;
  int rc;
  // id-indexed tables are padded to Vp ids (a multiple of 32), so that the
  // ids of one mask word are read with 16-byte loads
  t.Vp = (hv.V + 31) & ~31;
  std::vector<int32_t> spell_of_id_p(hv.spell_of_id);
  spell_of_id_p.resize(t.Vp, -1);
  // identifier-trie edges -> open-addressing hash (load factor <= 1/2)
  int hash_bits = 4;
  while ((size_t(1) << hash_bits) < 2 * h.lx_cbyte.size() + 2) ++hash_bits;
  t.lx_hmask = (1u << hash_bits) - 1u;
  t.lx_hshift = 32 - hash_bits;
  t.root_pc = h.LN > 0 ? h.lx_pcats[0] : 0u;
  t.root_wc = h.LN > 0 ? h.lx_wcats[0] : 0u;
  const uint8_t* dblob = nullptr;
  const int32_t *lx_cstart = nullptr, *lx_cnode = nullptr;
  const uint8_t* lx_cbyte = nullptr;
  uint4 *lx_hash = nullptr, *spell16 = nullptr;
  int32_t *id_of_spell = nullptr, *next_alias = nullptr;
  // Copies in flight read and write this function's arrays: from here on every
  // exit waits for the stream first.
  auto done = [&](int code) {
    cudaStreamSynchronize(st);
    return code;
  };
#define GRID_DONE(call)                       \
  do {                                        \
    const int code_ = [&]() -> int {          \
      GRID_CUDA(call);                        \
      return GRID_OK;                         \
    }();                                      \
    if (code_ != GRID_OK) return done(code_); \
  } while (0)
  {
    Upload up, up_tmp;
    up.add(blob, &dblob);
    up.add(ev_list, &t.ev_list);
    up.add(sets, &t.cls_sets);
    up.add(cls_map, &t.cls_map);
    up.add(tq, &t.tbl_q);
    up.add(h.acc_sym, &t.acc_sym);
    up.add(hv.first_of_byte, &t.first_of_byte);
    up.add(h.lx_pcats, &t.lx_pcats);
    up.add(h.lx_wcats, &t.lx_wcats);
    up.add(hv.spell_off, &t.spell_off);
    up.add(hv.spell_bytes, &t.spell_bytes);
    up.add(spell_of_id_p, &t.spell_of_id);
    up.reserve((size_t)t.lx_hmask + 1, &lx_hash);
    up.reserve(std::max(1, t.NS), &spell16);
    up.reserve(std::max(1, t.NS), &id_of_spell);
    up.reserve(t.Vp, &next_alias);
    up_tmp.add(h.lx_cstart, &lx_cstart);
    up_tmp.add(h.lx_cbyte, &lx_cbyte);
    up_tmp.add(h.lx_cnode, &lx_cnode);
    if ((rc = up.commit(a, st, keep)) || (rc = up_tmp.commit(tmp, st, keep))) return done(rc);
  }
  t.lx_hash = lx_hash;
  t.spell16 = spell16;
  t.id_of_spell = id_of_spell;
  t.next_alias = next_alias;
  t.blob = dblob;
  t.blob_bytes = off[kSec] <= (size_t)kMaxStage ? (int)off[kSec] : 0;
  t.o_class = (int)off[0];
  t.o_next = (int)off[1];
  t.o_acc = (int)off[2];
  t.o_live = (int)off[3];
  t.o_action = (int)off[4];
  t.o_go = (int)off[5];
  t.o_lhs = (int)off[6];
  t.o_shift = (int)off[7];
  t.o_roff = (int)off[8];
  t.o_rp = (int)off[9];
  t.o_red = (int)off[10];
  t.o_lany = (int)off[11];
  t.o_catq = (int)off[12];
  t.o_tblq = (int)off[13];
  t.o_sets = stage_sets ? (int)off[14] : -1;
  t.byte_class = dblob + off[0];
  t.next = reinterpret_cast<const uint16_t*>(dblob + off[1]);
  t.acc = reinterpret_cast<const uint32_t*>(dblob + off[2]);
  t.live = reinterpret_cast<const uint32_t*>(dblob + off[3]);
  t.action = reinterpret_cast<const int16_t*>(dblob + off[4]);
  t.go = reinterpret_cast<const uint16_t*>(dblob + off[5]);
  t.plhs = reinterpret_cast<const uint16_t*>(dblob + off[6]);
  t.shift_mask = reinterpret_cast<const uint32_t*>(dblob + off[7]);
  t.red_off = reinterpret_cast<const uint32_t*>(dblob + off[8]);
  t.red_p = reinterpret_cast<const uint16_t*>(dblob + off[9]);
  t.red_mask = reinterpret_cast<const uint32_t*>(dblob + off[10]);
  t.live_any = reinterpret_cast<const uint32_t*>(dblob + off[11]);
  t.cat_live = reinterpret_cast<const uint32_t*>(dblob + off[12]);
  t.tbl_of_q = reinterpret_cast<const int16_t*>(dblob + off[13]);
  GRID_DONE(cudaMemsetAsync(lx_hash, 0xFF, ((size_t)t.lx_hmask + 1) * 16, st));
  GRID_DONE(cudaMemsetAsync(id_of_spell, 0xFF, (size_t)std::max(1, t.NS) * 4, st));
  k_lex_hash<<<(h.LN + 255) / 256 + 1, 256, 0, st>>>(lx_cstart, lx_cbyte, lx_cnode, t.lx_pcats, t.lx_wcats, h.LN,
                                                    lx_hash, t.lx_hmask, t.lx_hshift);
  k_ids<<<(t.Vp + 255) / 256, 256, 0, st>>>(t.spell_of_id, t.Vp, id_of_spell, next_alias);
  k_spell16<<<(t.NS + 255) / 256 + 1, 256, 0, st>>>(t.spell_off, t.spell_bytes, t.NS, spell16);
  {
    Blake2b fb;
    fb.init(16);
    fb.update("GRIDspec", 8);
    fb.update(h.fingerprint, 16);
    fb.update(hv.fingerprint, 16);
    fb.final(s->fingerprint);
  }
  if ((rc = set_smem_limits())) return done(rc);
  int dev = 0;
  cudaGetDevice(&dev);
  s->device = dev;
  cudaDeviceGetAttribute(&s->sms, cudaDevAttrMultiProcessorCount, dev);
  g_sms = s->sms;
  // CI classification on the device
  uint16_t *cls_sp = nullptr, *key_sp = nullptr, *cls_by_id = nullptr;
  int32_t* counts_d = nullptr;  // per table: walked spellings, verdict-class spellings; then the fills of both lists
  uint32_t *vc_by_id = nullptr, *vc_sp = nullptr;
  uint8_t* fb = nullptr;
  {
    Upload up;
    up.reserve((size_t)t.n_tbl * t.NS, &cls_sp);
    up.reserve((size_t)t.n_tbl * t.NS, &key_sp);
    up.reserve((size_t)t.n_tbl * t.NS, &vc_sp);
    up.reserve((size_t)t.n_tbl * 5, &counts_d);
    if ((rc = up.commit(tmp, st, keep))) return done(rc);
    up.reserve((size_t)t.n_tbl * t.Vp, &cls_by_id);
    up.reserve((size_t)t.Vp, &fb);
    if ((rc = up.commit(a, st, keep))) return done(rc);
  }
  t.cls_by_id = cls_by_id;
  t.first_byte_by_id = fb;
  int32_t *cd_fill = counts_d + 2 * t.n_tbl, *vc_fill = counts_d + 3 * t.n_tbl, *vc_count = counts_d + 4 * t.n_tbl;
  GRID_DONE(cudaMemsetAsync(counts_d, 0, (size_t)t.n_tbl * 20, st));
  const dim3 cgrid(std::max(1, std::min((t.NS + 255) / 256, 4 * s->sms)), t.n_tbl);
  if (t.blob_bytes)
    k_classify<true><<<cgrid, 256, t.blob_bytes, st>>>(TabT<true>(t), cls_sp, key_sp, counts_d);
  else
    k_classify<false><<<cgrid, 256, 0, st>>>(TabT<false>(t), cls_sp, key_sp, counts_d);
  // the reserve's tables are laid out while the device classifies
  if ((rc = build_reserve_tables(s, st, keep))) return done(rc);
  std::vector<int32_t> counts2(2 * t.n_tbl);
  GRID_DONE(cudaMemcpyAsync(counts2.data(), counts_d, t.n_tbl * 8, cudaMemcpyDeviceToHost, st));
  GRID_DONE(cudaStreamSynchronize(st));
  std::vector<int32_t> counts(t.n_tbl), cdoff(t.n_tbl + 1, 0), vcbase(t.n_tbl + 1, 0);
  for (int k = 0; k < t.n_tbl; ++k) {
    counts[k] = counts2[2 * k];
    cdoff[k + 1] = cdoff[k] + counts2[2 * k];
    vcbase[k + 1] = vcbase[k] + counts2[2 * k + 1];
  }
  // CD spellings walked byte by byte (more than kMaxEv events), and the event
  // records of the verdict-class spellings -> distinct records per table
  const int nslot = vcbase.back();
  int32_t* cd_list = nullptr;
  uint16_t* cd_key = nullptr;
  const int32_t* vcbase_d = nullptr;
  int32_t *slot_tbl = nullptr, *slot_sp = nullptr, *rep = nullptr, *place = nullptr, *tab = nullptr;
  Rec* slot_rec = nullptr;
  uint32_t tab_mask = 1;
  while (tab_mask < 2u * (uint32_t)nslot) tab_mask = 2 * tab_mask + 1;
  {
    Upload up;
    up.add(vcbase, &vcbase_d);
    up.reserve(nslot, &slot_tbl);
    up.reserve(nslot, &slot_sp);
    up.reserve(nslot, &slot_rec);
    up.reserve(nslot, &rep);
    up.reserve(nslot, &place);
    up.reserve((size_t)tab_mask + 1, &tab);
    if ((rc = up.commit(tmp, st, keep))) return done(rc);
    up.add(cdoff, &t.cd_off);
    up.reserve(cdoff.back(), &cd_list);
    up.reserve(cdoff.back(), &cd_key);
    if ((rc = up.commit(a, st, keep))) return done(rc);
  }
  t.cd_list = cd_list;
  t.cd_key = cd_key;
  k_compact<<<dim3((t.NS + 255) / 256 + 1, t.n_tbl), 256, 0, st>>>(cls_sp, key_sp, t.NS, t.cd_off, t.cls_map, cd_fill,
                                                                   cd_list, cd_key);
  const int sgrid = (nslot + 255) / 256;
  std::vector<int32_t> n_distinct(t.n_tbl, 0);
  if (nslot > 0) {
    uint16_t* rec16 = reinterpret_cast<uint16_t*>(slot_rec);
    if (t.blob_bytes)
      k_events<true><<<cgrid, 256, t.blob_bytes, st>>>(TabT<true>(t), cls_sp, vcbase_d, vc_fill, slot_tbl, slot_sp, rec16);
    else
      k_events<false><<<cgrid, 256, 0, st>>>(TabT<false>(t), cls_sp, vcbase_d, vc_fill, slot_tbl, slot_sp, rec16);
    GRID_DONE(cudaMemsetAsync(tab, 0xFF, ((size_t)tab_mask + 1) * 4, st));
    k_vc_merge<<<sgrid, 256, 0, st>>>(slot_tbl, slot_rec, nslot, tab, tab_mask, rep, place, vc_count);
    GRID_DONE(cudaMemcpyAsync(n_distinct.data(), vc_count, t.n_tbl * 4, cudaMemcpyDeviceToHost, st));
  }
  GRID_DONE(cudaStreamSynchronize(st));
  std::vector<int32_t> vcoff(t.n_tbl + 1, 0);
  for (int k = 0; k < t.n_tbl; ++k) {
    vcoff[k + 1] = vcoff[k] + n_distinct[k];
    s->max_vc = std::max(s->max_vc, n_distinct[k]);
  }
  s->vcw = (s->max_vc + 31) / 32;
  // each table's records in the order of their event sequences: a walk item
  // evaluates 32 neighbouring records on one row's stack, and records that
  // share their first events take the same path through them, so the warp's
  // lanes stay together
  Rec* recs = nullptr;
  uint16_t* firsts = nullptr;
  RecKey* keys = nullptr;
  int32_t *src = nullptr, *rank = nullptr;
  const int n_vc = vcoff.back();
  {
    Upload up;
    up.add(vcoff, &t.vc_off);
    up.reserve(n_vc, &recs);
    up.reserve(n_vc, &firsts);
    if ((rc = up.commit(a, st, keep))) return done(rc);
    up.reserve(n_vc, &keys);
    up.reserve(n_vc, &src);
    up.reserve(n_vc, &rank);
    if ((rc = up.commit(tmp, st, keep))) return done(rc);
  }
  t.vc_rec = reinterpret_cast<const uint16_t*>(recs);
  t.vc_first = firsts;
  if (nslot > 0) {
    k_vc_gather<<<sgrid, 256, 0, st>>>(slot_tbl, slot_rec, nslot, rep, place, t.vc_off, src, keys, rank);
    k_vc_rank<<<dim3((s->max_vc + 255) / 256, t.n_tbl, 8), 256, 0, st>>>(keys, t.vc_off, rank);
    k_vc_place<<<(n_vc + 255) / 256, 256, 0, st>>>(slot_rec, slot_tbl, src, rank, n_vc, t.vc_off, recs, firsts, place);
    k_scatter_vc<<<sgrid, 256, 0, st>>>(slot_tbl, slot_sp, rep, place, nslot, t.NS, vc_sp);
  }
  // verdict-class indices ride in the 16-bit class codes when they fit;
  // otherwise k_pack looks them up per id (the rule counts the class ids as
  // they are before equal sets share one, so that a spec's facts stay what
  // they are)
  t.vc_inline = s->n_classes + kPackCodes + s->max_vc <= 0xFFFF && 32 * t.nselw + s->max_vc <= 0xFFFF ? 1 : 0;
  if (!t.vc_inline && (rc = a.alloc((size_t)t.n_tbl * t.Vp * 4, (void**)&vc_by_id))) return done(rc);
  t.vc_by_id = vc_by_id;
  k_permute<<<(t.Vp + 255) / 256, 256, 0, st>>>(t, cls_sp, vc_sp, cls_by_id, vc_by_id, fb);
  {
    uint32_t* killw = nullptr;
    if ((rc = a.alloc((size_t)t.Q * t.W * 4, (void**)&killw))) return done(rc);
    k_killw<<<dim3((t.W + 255) / 256, t.Q), 256, 0, st>>>(t, killw);
    t.killw = killw;
  }
  GRID_DONE(cudaGetLastError());
  GRID_DONE(cudaStreamSynchronize(st));
  s->n_vc = vcoff.back();
  if ((size_t)(2 * std::max(1, t.nselw) + 2 * std::max(1, s->vcw)) * 4 > (size_t)kMaxPack)
    return set_error(GRID_E_TOO_LARGE, "grid_specialize: the class selections and verdict-class bits of one "
                                       "row exceed the packing kernel's shared memory");
  s->max_cd = *std::max_element(counts.begin(), counts.end());
  s->walk_items = (float)t.NS / 32;
  if (t.ci_on) {
    long shifts = 0;
    for (int q = 0; q < h.S; ++q)
      for (int tau = 0; tau < h.n_term; ++tau) shifts += h.action[(size_t)q * h.T1 + tau] > 0;
    s->walk_items *= (float)shifts / ((float)h.S * (float)h.n_term);
  }
  int per_sm = 0;
  if (t.blob_bytes)
    GRID_DONE(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_advance<true>, 64, t.blob_bytes));
  else
    GRID_DONE(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_advance<false>, 64, 0));
  s->adv_fit = per_sm * s->sms;
  GRID_DONE(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_row<1, true>, kRowWarps * 32, t.blob_bytes));
  s->row_pair = per_sm > 1;
  return GRID_OK;
#undef GRID_DONE
}

extern "C" int grid_specialize(const grid_grammar* g, const grid_vocab* v, void* stream, grid_spec** out) {
  if (!g || !v || !out) return set_error(GRID_E_INVALID_ARG, "grid_specialize: bad arguments");
  *out = nullptr;
  auto* s = new grid_spec();
  Arena tmp;
  std::vector<std::vector<uint8_t>> keep;
  const int rc = specialize(g, v, (cudaStream_t)stream, s, tmp, keep);
  tmp.release();
  if (rc == GRID_OK)
    *out = s;
  else
    grid_spec_free(s);
  return rc;
}

extern "C" int grid_spec_info(const grid_spec* s, int64_t out[8]) {
  if (!s || !out) return set_error(GRID_E_INVALID_ARG, "grid_spec_info: bad arguments");
  const Tables& t = s->t;
  std::vector<int32_t> off(t.n_tbl + 1);
  GRID_CUDA(cudaMemcpy(off.data(), t.cd_off, (t.n_tbl + 1) * 4, cudaMemcpyDeviceToHost));
  out[0] = t.n_tbl;
  out[1] = s->n_classes;
  out[2] = off[1] - off[0];
  out[3] = off[t.n_tbl];
  out[4] = t.blob_bytes;
  out[5] = s->n_vc;
  out[6] = (t.ci_on ? 1 : 0) | (t.vc_inline ? 2 : 0);
  out[7] = t.NS;
  return GRID_OK;
}

extern "C" void grid_spec_free(grid_spec* s) {
  if (!s) return;
  s->mem.release();
  delete s;
}

extern "C" int grid_configs_create(const grid_spec* s, int32_t B, grid_configs** out) {
  if (!s || !out || B <= 0) return set_error(GRID_E_INVALID_ARG, "grid_configs_create: bad arguments");
  if (B > kMaxRows)
    return set_error(GRID_E_TOO_LARGE, "grid_configs_create: more than " + std::to_string(kMaxRows) + " rows");
  *out = nullptr;
  auto* c = new grid_configs();
  c->B = B;
  c->D = s->t.D;
  c->words_v = s->t.W;
  c->cap = std::max(1, s->max_cd);
  c->vcap = std::max(1, s->max_vc);
  Arena& a = c->mem;
  int rc;
  if ((rc = a.alloc((size_t)B * c->D * sizeof(uint16_t), (void**)&c->c.stack)) ||
      (rc = a.alloc(B * 4, (void**)&c->c.depth)) || (rc = a.alloc(B * 4, (void**)&c->c.q)) ||
      (rc = a.alloc(B * 4, (void**)&c->c.lx)) || (rc = a.alloc(B * 4, (void**)&c->c.flags)) ||
      (rc = a.alloc(B * sizeof(RowCtx), (void**)&c->ctx)) ||
      (rc = a.alloc(B * sizeof(RowRanges), (void**)&c->rng)) ||
      (rc = a.alloc((size_t)B * 2 * std::max(1, s->t.nselw) * 4, (void**)&c->sel)) ||
      (rc = a.alloc((size_t)B * c->words_v * 4, (void**)&c->verd0)) ||
      (rc = a.alloc((size_t)B * c->words_v * 4, (void**)&c->verd1)) ||
      (rc = a.alloc((size_t)B * 2 * s->t.T1 * 16, (void**)&c->A2)) ||
      (rc = a.alloc((size_t)B * 2 * std::max(1, s->vcw) * 4, (void**)&c->vcbits)) ||
      (rc = a.alloc((size_t)B * 2 * std::max(1, s->max_cd) * 4, (void**)&c->surv)) ||
      (rc = a.alloc((size_t)B * 2 * c->vcap * 4, (void**)&c->vsurv)) ||
      (rc = a.alloc((size_t)B * 2 * 4, (void**)&c->aux)) ||
      (rc = a.alloc((size_t)B * reserve_scratch_bytes(s), (void**)&c->rscratch))) {
    grid_configs_free(c);
    return rc;
  }
  k_reset<<<(B + 127) / 128, 128>>>(c->c, B, c->D);
  cudaError_t e = cudaDeviceSynchronize();
  if (e != cudaSuccess) {
    grid_configs_free(c);
    return set_error(GRID_E_CUDA, std::string("grid_configs_create: ") + cudaGetErrorString(e));
  }
  *out = c;
  return GRID_OK;
}

extern "C" void grid_configs_free(grid_configs* c) {
  if (!c) return;
  c->mem.release();
  delete c;
}

extern "C" int grid_configs_reset(const grid_spec* s, grid_configs* c, void* stream) {
  if (!s || !c) return set_error(GRID_E_INVALID_ARG, "grid_configs_reset: bad arguments");
  k_reset<<<(c->B + 127) / 128, 128, 0, (cudaStream_t)stream>>>(c->c, c->B, c->D);
  GRID_CUDA(cudaGetLastError());
  return audit_reset(s, c, (cudaStream_t)stream);  // a fresh chain for every row, when audit is on
}

int grid::launch_advance(const grid_spec* s, const DevConfigs& in, const DevConfigs& out, int B,
                         const int32_t* d_tokens, int32_t n_steps, int32_t* d_status, int copy, cudaStream_t st) {
  const TabT<true> ts(s->t);
  const TabT<false> tg(s->t);
  auto launch = [&](auto kern, const auto& t, int blocks, int threads, size_t dyn) {
    return launch_pdl(kern, dim3(blocks), dim3(threads), t.blob_bytes + dyn, st, t, in, out, d_tokens, n_steps,
                      d_status, B, copy);
  };
  // Several tokens go to a block per row while the blocks of all rows are on the SMs at once.  In larger batches each
  // wave of blocks would stage the tables anew: there a few tokens are fed one after the other by a warp per row (2
  // tokens, 4,096 SQL rows: 73 us as one block per row, 27 this way), and more of them in blocks that read the tables
  // from global memory, of which more fit (16 tokens: 255 us staged, 129; within one wave, 256 rows: 36 and 48),
  // unless the tables are so small that staging them costs nothing (expression grammar, 16 tokens, 4,096 rows: 80 us
  // staged, 85).
  const bool wave = B <= s->adv_fit;
  if (n_steps <= 1 || (n_steps <= kFewTokens && !wave)) {
    const int rows = std::min(kOneRows, (B + s->sms - 1) / s->sms);  // of a block: one until every SM has its block
    const size_t dyn = rows * sizeof(OneShared);
    const int blocks = (B + rows - 1) / rows;
    GRID_CUDA(s->t.blob_bytes ? launch(k_advance_one<true>, ts, blocks, rows * 32, dyn)
                              : launch(k_advance_one<false>, tg, blocks, rows * 32, dyn));
  } else {
    const bool staged = s->t.blob_bytes > 0 && (wave || s->t.blob_bytes <= 16 * 1024);
    GRID_CUDA(staged ? launch(k_advance<true>, ts, B, 64, 0) : launch(k_advance<false>, tg, B, 64, 0));
  }
  GRID_CUDA(cudaGetLastError());
  return GRID_OK;
}

extern "C" int grid_advance(const grid_spec* s, const grid_configs* in, grid_configs* out,
                            const int32_t* d_tokens, int32_t n_steps, int32_t* d_status, void* stream) {
  if (!s || !in || !out || !d_tokens || !d_status || n_steps < 0 || in->B != out->B || in->D != out->D)
    return set_error(GRID_E_INVALID_ARG, "grid_advance: bad arguments");
  if ((in->c.hs != nullptr) != (out->c.hs != nullptr))
    return set_error(GRID_E_INVALID_ARG, "grid_advance: audit must be enabled on both configurations or on neither");
  return launch_advance(s, in->c, out->c, in->B, d_tokens, n_steps, d_status, in != out ? 1 : 0,
                        (cudaStream_t)stream);
}

// Warps per k_walk block.  A walk waits for its look-ups, so a large batch
// wants every warp that fits (24, by shared memory and 80 registers: 256 SQL
// rows 291 us a step, 514 us with 8 warps, 337 us with 16), a small one the
// shortest start, and room for the next kernel's blocks beside it (one
// expression row 24.1 us with 4 warps, 27.1 us with 24; one SQL row 38.3 and
// 42.1).  Between them by the walk items that may come up: a row's spellings go
// as far as its state shifts their first terminal, the share of terminals that
// a state shifts on average (every spelling where the grammar has no CI
// classes).  That gives 235 items a row for 152,000 SQL tokens (counted: 196),
// 7 for a grammar of 60 keywords (7), 46 to 60 for random grammars and 20,000
// tokens (51 to 88).  Per step with 8, 12, 16 and 24 warps: 8 SQL rows 51.1,
// 48.0, 46.3, 47.6 us; 64 rows of a random grammar 79.4, 69.3, 65.2, 60.4 us;
// 16 rows without CI classes 51.4, 47.5, 45.3, 44.0 us.
static int walk_warps(const grid_spec* s, int B) {
  const float n = (float)B * s->walk_items / (float)s->sms;  // items per SM
  const int room = (kWalkSmem - s->t.blob_bytes) / (int)sizeof(WalkWarp);
  if (n < (B == 1 ? 2.f : 1.f)) return 4;
  return n < 4.f ? 8 : n < 8.f ? 12 : n < 16.f ? 16 : std::min(kWalkWarps, room);
}

// The four kernels of one mask step on `st`; `ev` (5 events or NULL) is
// recorded before the first kernel and after each.
int grid::launch_masks(const grid_spec* s, const DevConfigs& c, const MaskScratch& m, int B, uint32_t* d_mask,
                       int32_t* d_status, cudaStream_t st, const cudaEvent_t* ev, const FusedLogits& lg,
                       const AdvArgs* adv, const ForceArgs* force) {
  const Tables& t = s->t;
  const int vcw = std::max(1, s->vcw);
  const int n_vcbits = B * 2 * vcw;
  const size_t zero_words = (size_t)B * m.words_v * 2 + n_vcbits;
  const int zero_blocks = std::min(128, (int)((zero_words / 8 + kRowWarps * 32 * 4 - 1) / (kRowWarps * 32 * 4)) + 1);
  if (ev) GRID_CUDA(cudaEventRecord(ev[0], st));
  const TabT<true> ts(t);  // the tables as the kernels that stage them take them, or
  const TabT<false> tg(t);  // that read a block too large to stage from global memory
  // Tables so large that k_row has one block on an SM are staged for batches of one row per SM alone: beyond them the
  // blocks wait for one another's SM (tables of 96 KB, 256 rows: 54 us staged, 47 from global memory; 152 rows 36 and
  // 38; tables of 52 KB leave two blocks, 512 rows: 149 and 160).
  const bool staged = t.blob_bytes > 0 && (B <= s->sms || s->row_pair);
  auto row = [&](auto kern, const auto& tab) {
    return launch_pdl(kern, dim3(B + zero_blocks), dim3(kRowWarps * 32), tab.blob_bytes, st, tab, c, m.ctx, m.rng,
                      m.A2, m.sel, m.verd0, m.verd1, m.vcbits, n_vcbits, B, m.words_v, m.cache,
                      adv ? *adv : AdvArgs{});
  };
  if (staged)
    GRID_CUDA(!adv ? row(k_row<0, true>, ts) : adv->n_steps <= 1 ? row(k_row<1, true>, ts) : row(k_row<2, true>, ts));
  else
    GRID_CUDA(!adv ? row(k_row<0, false>, tg) : adv->n_steps <= 1 ? row(k_row<1, false>, tg) : row(k_row<2, false>, tg));
  if (ev) GRID_CUDA(cudaEventRecord(ev[1], st));
  const int cd_blocks = (s->max_cd + 256 * kFilterPer - 1) / (256 * kFilterPer);
  const int vc_blocks = (s->max_vc + 256 * kFilterPer - 1) / (256 * kFilterPer);
  // the scan of the ranges in k_filter: where the walks fill the SMs for long (256 SQL rows: 290 -> 248 us a step,
  // 128 rows 163 -> 157), not where a step waits for the longest of them (32 rows 72 -> 95 us: what is left of the
  // ranges then packs 32 long walks into a warp)
  const bool scan = s->has_cats && m.vcap >= kScanList && (long)B * ((t.NS + 1023) / 1024) / s->sms >= 100;
  const int scan_blocks = scan ? std::min((t.NS / kRangeSpan + 256 + 7) / 8, std::max(1, 32 * s->sms / B)) : 0;
  GRID_CUDA(launch_pdl(k_filter, dim3(std::max({1, cd_blocks + vc_blocks, scan_blocks}), B, scan ? 3 : 2), dim3(256), 0,
                       st, tg, m.ctx,
                       (const uint32_t*)m.sel, m.surv, m.cap, m.vsurv, m.vcap, cd_blocks, (const RowRanges*)m.rng,
                       m.verd0, m.words_v, s->walk_work));
  if (ev) GRID_CUDA(cudaEventRecord(ev[2], st));
  const int ww = walk_warps(s, B);
  auto walk = [&](auto kern, const auto& tab) {
    return launch_pdl(kern, dim3(s->sms), dim3(ww * 32), tab.blob_bytes + ww * sizeof(WalkWarp), st, tab, m.ctx,
                      (const RowRanges*)m.rng, (const uint16_t*)c.stack, (const int32_t*)m.surv, m.cap,
                      (const uint32_t*)m.A2, m.verd0, m.verd1, m.vcbits, vcw, (const int32_t*)m.vsurv, m.vcap,
                      m.words_v, B, scan ? m.vcap : -1, s->walk_work);
  };
  if (s->walk_work)  // the measured instance, which counts its work
    GRID_CUDA(staged ? walk(k_walk<true, true>, ts) : walk(k_walk<true, false>, tg));
  else
    GRID_CUDA(staged ? walk(k_walk<false, true>, ts) : walk(k_walk<false, false>, tg));
  if (ev) GRID_CUDA(cudaEventRecord(ev[3], st));
  const dim3 pgrid((t.W + kPackWords - 1) / kPackWords, B);
  const size_t psmem = std::max<size_t>((size_t)2 * (t.nselw + vcw), kPackWords) * 4;
  const int esz = lg.dtype == GRID_DTYPE_F32 ? 4 : 2;
  const int vec_ok = lg.p && ((uintptr_t)lg.p % 32 == 0) && ((lg.stride * esz) % 32 == 0);  // 32-byte sectors
  auto pack = [&](auto kern) {
    return launch_pdl(kern, pgrid, dim3(kPackWords), psmem, st, t, m.ctx, (const uint32_t*)m.sel,
                      (const uint32_t*)m.vcbits, vcw, (const uint32_t*)m.verd0, (const uint32_t*)m.verd1, m.words_v,
                      d_mask, d_status, lg.p, (long long)lg.stride, lg.p ? vec_ok : 0, m.cache,
                      force ? *force : ForceArgs{});
  };
  const bool cached = m.cache.n > 0;
  const int mode = !lg.p ? 0 : (lg.dtype == GRID_DTYPE_F32 ? 1 : 2);
  cudaError_t pe;
  if (force)  // (a span's step has neither logits nor a cache)
    pe = pack(k_pack<0, false, true>);
  else if (mode == 0)
    pe = cached ? pack(k_pack<0, true>) : pack(k_pack<0, false>);
  else if (mode == 1)
    pe = cached ? pack(k_pack<1, true>) : pack(k_pack<1, false>);
  else
    pe = cached ? pack(k_pack<2, true>) : pack(k_pack<2, false>);
  GRID_CUDA(pe);
  if (ev) GRID_CUDA(cudaEventRecord(ev[4], st));
  GRID_CUDA(cudaGetLastError());
  return GRID_OK;
}

extern "C" int grid_masks(const grid_spec* s, const grid_configs* c, uint32_t* d_mask, int32_t* d_status,
                          void* stream) {
  if (!s || !c || !d_mask || !d_status) return set_error(GRID_E_INVALID_ARG, "grid_masks: bad arguments");
  const MaskScratch m{c->ctx, c->rng, c->sel, c->verd0, c->verd1, c->A2, c->vcbits,
                      c->surv, c->vsurv, c->cap, c->vcap, c->words_v};
  return launch_masks(s, c->c, m, c->B, d_mask, d_status, (cudaStream_t)stream, c->ev[0] ? c->ev : nullptr);
}

extern "C" int grid_masks_apply(const grid_spec* s, const grid_configs* c, uint32_t* d_mask, int32_t* d_status,
                                void* d_logits, int32_t dtype, int64_t row_stride, void* stream) {
  if (!s || !c || !d_mask || !d_status || !d_logits || row_stride < s->t.V ||
      (dtype != GRID_DTYPE_F32 && dtype != GRID_DTYPE_BF16))
    return set_error(GRID_E_INVALID_ARG, "grid_masks_apply: bad arguments");
  const MaskScratch m{c->ctx, c->rng, c->sel, c->verd0, c->verd1, c->A2, c->vcbits,
                      c->surv, c->vsurv, c->cap, c->vcap, c->words_v};
  FusedLogits lg;
  lg.p = d_logits;
  lg.dtype = dtype;
  lg.stride = row_stride;
  return launch_masks(s, c->c, m, c->B, d_mask, d_status, (cudaStream_t)stream, c->ev[0] ? c->ev : nullptr, lg);
}

// ---------------------------------------------------------------------------
// Configuration-keyed mask cache (Sec. 4.3, Def. T1 key, Prop. OBL-KEY1).
struct grid_cache {
  const grid_spec* s = nullptr;
  CacheDev d;
  Arena mem;
};

extern "C" int grid_cache_create(const grid_spec* s, int32_t n_entries, grid_cache** out) {
  if (!s || !out || n_entries <= 0 || (n_entries & (n_entries - 1)) || n_entries > (1 << 20))
    return set_error(GRID_E_INVALID_ARG, "grid_cache_create: n_entries must be a power of two in 1 .. 2^20");
  *out = nullptr;
  auto* c = new grid_cache();
  c->s = s;
  c->d.n = n_entries;
  const size_t W = s->t.W;
  int rc;
  if ((rc = c->mem.alloc((size_t)n_entries * 16 * 4, (void**)&c->d.hdr)) ||
      (rc = c->mem.alloc((size_t)n_entries * W * 4, (void**)&c->d.ci)) ||
      (rc = c->mem.alloc((size_t)n_entries * W * 4, (void**)&c->d.sel)) ||
      (rc = c->mem.alloc(4 * 8, (void**)&c->d.stats))) {
    c->mem.release();
    delete c;
    return rc;
  }
  cudaError_t e = cudaMemset(c->d.hdr, 0, (size_t)n_entries * 16 * 4);
  if (e == cudaSuccess) e = cudaMemset(c->d.stats, 0, 4 * 8);
  if (e == cudaSuccess) e = cudaDeviceSynchronize();
  if (e != cudaSuccess) {
    c->mem.release();
    delete c;
    return set_error(GRID_E_CUDA, std::string("grid_cache_create: ") + cudaGetErrorString(e));
  }
  *out = c;
  return GRID_OK;
}

extern "C" void grid_cache_free(grid_cache* c) {
  if (!c) return;
  c->mem.release();
  delete c;
}

extern "C" int grid_cache_clear(grid_cache* c, void* stream) {
  if (!c) return set_error(GRID_E_INVALID_ARG, "grid_cache_clear: bad arguments");
  GRID_CUDA(cudaMemsetAsync(c->d.hdr, 0, (size_t)c->d.n * 16 * 4, (cudaStream_t)stream));
  GRID_CUDA(cudaMemsetAsync(c->d.stats, 0, 4 * 8, (cudaStream_t)stream));
  return GRID_OK;
}

extern "C" int grid_cache_stats(const grid_cache* c, int64_t out[4]) {
  if (!c || !out) return set_error(GRID_E_INVALID_ARG, "grid_cache_stats: bad arguments");
  unsigned long long st[3];
  std::vector<uint32_t> hdr((size_t)c->d.n * 16);
  GRID_CUDA(cudaMemcpy(st, c->d.stats, 3 * 8, cudaMemcpyDeviceToHost));
  GRID_CUDA(cudaMemcpy(hdr.data(), c->d.hdr, hdr.size() * 4, cudaMemcpyDeviceToHost));
  int64_t ready = 0;
  for (int i = 0; i < c->d.n; ++i) ready += hdr[(size_t)i * 16] == 2u;
  out[0] = (int64_t)st[0];
  out[1] = (int64_t)st[1];
  out[2] = (int64_t)st[2];
  out[3] = ready;
  return GRID_OK;
}

extern "C" int grid_masks_cached(const grid_spec* s, const grid_configs* c, grid_cache* cache, uint32_t* d_mask,
                                 int32_t* d_status, void* d_logits, int32_t dtype, int64_t row_stride, void* stream) {
  if (!s || !c || !cache || !d_mask || !d_status || cache->s != s ||
      (d_logits && (row_stride < s->t.V || (dtype != GRID_DTYPE_F32 && dtype != GRID_DTYPE_BF16))))
    return set_error(GRID_E_INVALID_ARG, "grid_masks_cached: bad arguments (the cache must belong to the spec)");
  MaskScratch m{c->ctx, c->rng, c->sel, c->verd0, c->verd1, c->A2, c->vcbits,
                c->surv, c->vsurv, c->cap, c->vcap, c->words_v};
  m.cache = cache->d;
  FusedLogits lg;
  lg.p = d_logits;
  lg.dtype = dtype;
  lg.stride = row_stride;
  return launch_masks(s, c->c, m, c->B, d_mask, d_status, (cudaStream_t)stream, c->ev[0] ? c->ev : nullptr, lg);
}

extern "C" int grid_advance_masks(const grid_spec* s, const grid_configs* in, grid_configs* out, grid_cache* cache,
                                  const int32_t* d_tokens, int32_t n_steps, uint32_t* d_mask, int32_t* d_status,
                                  void* d_logits, int32_t dtype, int64_t row_stride, void* stream) {
  if (!s || !in || !out || !d_tokens || !d_mask || !d_status || n_steps < 0 || in->B != out->B || in->D != out->D)
    return set_error(GRID_E_INVALID_ARG, "grid_advance_masks: bad arguments");
  if (cache && cache->s != s)
    return set_error(GRID_E_INVALID_ARG, "grid_advance_masks: the cache must belong to the spec");
  if (d_logits && (row_stride < s->t.V || (dtype != GRID_DTYPE_F32 && dtype != GRID_DTYPE_BF16)))
    return set_error(GRID_E_INVALID_ARG, "grid_advance_masks: bad logits arguments");
  if ((in->c.hs != nullptr) != (out->c.hs != nullptr))
    return set_error(GRID_E_INVALID_ARG,
                     "grid_advance_masks: audit must be enabled on both configurations or on neither");
  MaskScratch m{out->ctx, out->rng, out->sel, out->verd0, out->verd1, out->A2, out->vcbits,
                out->surv, out->vsurv, out->cap, out->vcap, out->words_v};
  if (cache) m.cache = cache->d;
  FusedLogits lg;
  lg.p = d_logits;
  lg.dtype = dtype;
  lg.stride = row_stride;
  const AdvArgs adv{in->c, d_tokens, n_steps, in != out ? 1 : 0, nullptr};
  return launch_masks(s, out->c, m, out->B, d_mask, d_status, (cudaStream_t)stream, out->ev[0] ? out->ev : nullptr,
                      lg, &adv);
}

extern "C" int grid_spec_set_work_counters(grid_spec* s, unsigned long long* d_counters) {
  if (!s) return set_error(GRID_E_INVALID_ARG, "grid_spec_set_work_counters: bad arguments");
  s->walk_work = d_counters;
  return GRID_OK;
}

extern "C" int grid_configs_set_events(grid_configs* c, void* const* events, int32_t n_events) {
  if (!c || (n_events != 0 && n_events != kMaskKernels + 1) || (n_events && !events))
    return set_error(GRID_E_INVALID_ARG, "grid_configs_set_events: pass 0 or 5 events");
  for (int i = 0; i <= kMaskKernels; ++i) {
    c->ev[i] = n_events ? static_cast<cudaEvent_t>(events[i]) : nullptr;
    if (n_events && !c->ev[i]) {
      for (int k = 0; k <= kMaskKernels; ++k) c->ev[k] = nullptr;
      return set_error(GRID_E_INVALID_ARG, "grid_configs_set_events: null event");
    }
  }
  return GRID_OK;
}

// ---------------------------------------------------------------------------
// grid_masks_static: the mask step without any allocation.
//
// Some callers cannot allocate device memory when they need a mask: a serving
// engine whose own pool has reserved the device memory up front (a driver
// allocation would fail, or fragment the pool), or one that cannot afford the
// device-wide synchronization that freeing memory implies in the middle of a
// decoding step.  Such a caller keeps the parser configurations in device
// memory it already owns and passes them in; the scratch of the step (row
// contexts, class selections, survivor lists, verdict bitmaps) comes from the
// fixed array below instead of from a grid_configs.  The array is part of the
// library's device image: the CUDA runtime reserves it on every device where
// the library's kernels are loaded and keeps it until the process exits.
constexpr size_t kStaticScratchBytes = size_t(8) << 20;
constexpr int kStaticMaxDevices = 64;
static __device__ __align__(256) uint8_t g_static_scratch[kStaticScratchBytes];

namespace {
// In host code `g_static_scratch` names a host-side shadow of the array, not
// device memory; kernels get the device address found at set-up.
std::mutex g_static_mu;
uint8_t* g_static_dev[kStaticMaxDevices] = {};

// Offsets of the step's buffers inside the array (each 256-byte aligned),
// sized exactly as grid_configs_create sizes the same buffers.
struct StaticCarve {
  size_t ctx, rng, sel, verd0, verd1, A2, vcbits, surv, vsurv, total;
};

StaticCarve carve_static(const grid_spec* s, int B, int words_v) {
  StaticCarve c{};
  size_t at = 0;
  auto take = [&](size_t bytes) {
    const size_t o = at;
    at += (std::max<size_t>(bytes, 16) + 255) & ~size_t(255);
    return o;
  };
  c.ctx = take((size_t)B * sizeof(RowCtx));
  c.rng = take((size_t)B * sizeof(RowRanges));
  c.sel = take((size_t)B * 2 * std::max(1, s->t.nselw) * 4);
  c.verd0 = take((size_t)B * words_v * 4);
  c.verd1 = take((size_t)B * words_v * 4);
  c.A2 = take((size_t)B * 2 * s->t.T1 * 16);
  c.vcbits = take((size_t)B * 2 * std::max(1, s->vcw) * 4);
  c.surv = take((size_t)B * 2 * std::max(1, s->max_cd) * 4);
  c.vsurv = take((size_t)B * 2 * std::max(1, s->max_vc) * 4);
  c.total = at;
  return c;
}
}  // namespace

extern "C" int grid_masks_static(const grid_spec* s, const uint16_t* d_stack, const int32_t* d_depth,
                                 const int32_t* d_dfa_state, const int32_t* d_lex_node, const int32_t* d_flags,
                                 int32_t B, int32_t stack_stride, uint32_t* d_mask, int32_t* d_status,
                                 void* stream) {
  if (!s || !d_stack || !d_depth || !d_dfa_state || !d_lex_node || !d_flags || !d_mask || !d_status || B <= 0)
    return set_error(GRID_E_INVALID_ARG, "grid_masks_static: bad arguments");
  const Tables& t = s->t;
  if (B > kMaxRows)
    return set_error(GRID_E_TOO_LARGE, "grid_masks_static: more than " + std::to_string(kMaxRows) + " rows");
  if (stack_stride != t.D)
    return set_error(GRID_E_INVALID_ARG, "grid_masks_static: stack_stride " + std::to_string(stack_stride) +
                                             " differs from the grammar's max_depth " + std::to_string(t.D));
  int dev = 0;
  GRID_CUDA(cudaGetDevice(&dev));
  if (dev != s->device)
    return set_error(GRID_E_INVALID_ARG, "grid_masks_static: the spec lives on device " + std::to_string(s->device) +
                                             ", the current device is " + std::to_string(dev));
  if (dev < 0 || dev >= kStaticMaxDevices)
    return set_error(GRID_E_INVALID_ARG, "grid_masks_static: device ordinal " + std::to_string(dev) +
                                             " is beyond the " + std::to_string(kStaticMaxDevices) + " supported");
  const int words_v = t.W;
  const StaticCarve cv = carve_static(s, B, words_v);
  if (cv.total > kStaticScratchBytes)
    return set_error(GRID_E_TOO_LARGE, "grid_masks_static: B=" + std::to_string(B) + " needs " +
                                           std::to_string(cv.total) + " bytes of scratch with this spec, more than "
                                           "the " + std::to_string(kStaticScratchBytes) +
                                           "-byte static area; use grid_masks with a grid_configs instead");
  uint8_t* area = nullptr;
  {
    std::lock_guard<std::mutex> lock(g_static_mu);
    if (!g_static_dev[dev]) {  // set-up, once per device
      void* p = nullptr;
      const cudaError_t e = cudaGetSymbolAddress(&p, g_static_scratch);
      if (e != cudaSuccess || !p)
        return set_error(GRID_E_CUDA, std::string("grid_masks_static: cudaGetSymbolAddress: ") +
                                          cudaGetErrorString(e));
      g_static_dev[dev] = static_cast<uint8_t*>(p);
    }
    area = g_static_dev[dev];
  }
  const MaskScratch m{reinterpret_cast<RowCtx*>(area + cv.ctx),
                      reinterpret_cast<RowRanges*>(area + cv.rng),
                      reinterpret_cast<uint32_t*>(area + cv.sel),
                      reinterpret_cast<uint32_t*>(area + cv.verd0),
                      reinterpret_cast<uint32_t*>(area + cv.verd1),
                      reinterpret_cast<uint32_t*>(area + cv.A2),
                      reinterpret_cast<uint32_t*>(area + cv.vcbits),
                      reinterpret_cast<int32_t*>(area + cv.surv),
                      reinterpret_cast<int32_t*>(area + cv.vsurv),
                      std::max(1, s->max_cd),
                      std::max(1, s->max_vc),
                      words_v};
  // the kernels only read the configurations
  const DevConfigs c{const_cast<uint16_t*>(d_stack), const_cast<int32_t*>(d_depth),
                     const_cast<int32_t*>(d_dfa_state), const_cast<int32_t*>(d_lex_node),
                     const_cast<int32_t*>(d_flags)};
  // What must start at zero is cleared by k_row itself on every call: the
  // verdict bitmaps and verdict-class bits (its clearing blocks) and each
  // row's queue, survivor and completion counters.  The other buffers are
  // written before they are read within the call, so the previous call's
  // contents do not matter.
  return launch_masks(s, c, m, B, d_mask, d_status, (cudaStream_t)stream, nullptr);
}

extern "C" int grid_apply_mask(const uint32_t* d_mask, void* d_logits, int32_t dtype, int32_t B, int32_t V,
                               int64_t row_stride, void* stream) {
  if (!d_mask || !d_logits || B <= 0 || V <= 0 || row_stride < V ||
      (dtype != GRID_DTYPE_F32 && dtype != GRID_DTYPE_BF16))
    return set_error(GRID_E_INVALID_ARG, "grid_apply_mask: bad arguments");
  cudaStream_t st = (cudaStream_t)stream;
  const int W = (V + 31) / 32;
  const int esz = dtype == GRID_DTYPE_F32 ? 4 : 2;
  if (B > 65535) return set_error(GRID_E_TOO_LARGE, "grid_apply_mask: more than 65535 rows in one call");
  const int sectors = (V * esz + 31) / 32;  // 32-byte sectors per row
  const int per_row = std::max(1, std::min((sectors + 255) / 256, (g_sms * 4 + B - 1) / B));
  const dim3 grid(per_row, B);
  const bool shifted = (uintptr_t)d_logits % 32 != 0 || (row_stride * esz) % 32 != 0;  // rows off the sector boundaries
  auto apply = [&](auto kern, auto* p) {
    return launch_pdl(kern, grid, dim3(256), 0, st, d_mask, p, B, V, W, (long long)row_stride);
  };
  if (dtype == GRID_DTYPE_F32)
    GRID_CUDA(shifted ? apply(k_apply<uint32_t, true>, (uint32_t*)d_logits)
                      : apply(k_apply<uint32_t, false>, (uint32_t*)d_logits));
  else
    GRID_CUDA(shifted ? apply(k_apply<uint16_t, true>, (uint16_t*)d_logits)
                      : apply(k_apply<uint16_t, false>, (uint16_t*)d_logits));
  GRID_CUDA(cudaGetLastError());
  return GRID_OK;
}

extern "C" int grid_configs_export(const grid_configs* c, int32_t row, int32_t* stack, int32_t cap,
                                   int32_t* depth, int32_t* dfa_state, int32_t* lex_node, int32_t* flags) {
  if (!c || row < 0 || row >= c->B || !depth || !dfa_state || !lex_node || !flags || cap < 0 || (cap && !stack))
    return set_error(GRID_E_INVALID_ARG, "grid_configs_export: bad arguments");
  GRID_CUDA(cudaMemcpy(depth, c->c.depth + row, 4, cudaMemcpyDeviceToHost));
  GRID_CUDA(cudaMemcpy(dfa_state, c->c.q + row, 4, cudaMemcpyDeviceToHost));
  GRID_CUDA(cudaMemcpy(lex_node, c->c.lx + row, 4, cudaMemcpyDeviceToHost));
  GRID_CUDA(cudaMemcpy(flags, c->c.flags + row, 4, cudaMemcpyDeviceToHost));
  int n = std::min(*depth, cap);
  if (n > 0) {
    std::vector<uint16_t> tmp(n);
    GRID_CUDA(cudaMemcpy(tmp.data(), c->c.stack + (size_t)row * c->D, n * 2, cudaMemcpyDeviceToHost));
    for (int i = 0; i < n; ++i) stack[i] = tmp[i];
  }
  return GRID_OK;
}
