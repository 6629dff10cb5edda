// Device-side data structures and per-lane routines of the mask path.
//
// A configuration kappa = (sigma, rho) (GRID Def. 1) is, on the device, the
// row's stack of LALR(1) states (uint16, bottom first) plus the scan state of
// the pending lexeme: the lexer DFA state q and the node lx of the identifier
// trie (-1 once the lexeme left every lexicon word).  While a token is tried,
// the row stack is never written: a lane works on the virtual stack
// base[0:keep] ++ ovl[0:m] (copy-on-write top of stack), and a simulated
// reduce chain additionally pushes into scr[0:ns].
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

#include "grid_internal.h"

namespace grid {

constexpr int kMaxOvl = 48;  // per-token overlay / scratch entries per lane

// CI class codes (Sec. 4.2).  Codes below kClsFirstCode are class ids
// ((kind * Q + q) << n_cat | cats): kind 0 = the verdict is "the live set of
// (q, cats) meets A u I" (token ends inside one lexeme), kind 1 = "the
// candidate set of (q, cats) meets A u I" (one boundary, then ignored bytes).
constexpr uint16_t kClsFirstCode = 0xFFFB;  // class ids are below this value
constexpr uint16_t kClsVC = 0xFFFB;   // context-dependent, decided by its verdict class (event record)
constexpr uint16_t kClsNA = 0xFFFC;   // spelling does not continue this lexer state
constexpr uint16_t kClsAcc = 0xFFFD;  // viable for every allowed set
constexpr uint16_t kClsRej = 0xFFFE;  // viable for no allowed set
constexpr uint16_t kClsCD = 0xFFFF;   // context-dependent, too many events: walked byte by byte

// Event record of a context-dependent spelling (GRID Sec. 4.2, verdict-
// equivalence grouping): rec[0] = number of stack-dependent emissions n,
// rec[1] = the final test (a live class id, or kClsAcc when the trailing
// lexeme is live for an ignored terminal), rec[2 .. 2+n) = the candidate
// classes of the emissions in order.  Spellings with equal records have equal
// verdicts at every stack; each distinct record is a verdict class.
constexpr int kRecLen = 16;
constexpr int kMaxEv = kRecLen - 2;

// A set of at most 128 terminals held in four registers.  Word access goes
// through selects, never through a runtime-indexed array (which would live
// in local memory).
struct Bits4 {
  uint32_t x, y, z, w;
  __host__ __device__ __forceinline__ static Bits4 zero() { return Bits4{0u, 0u, 0u, 0u}; }
  // (p is 16-byte aligned)
  __device__ __forceinline__ static Bits4 load(const uint32_t* p) {
    const uint4 v = *reinterpret_cast<const uint4*>(p);
    return Bits4{v.x, v.y, v.z, v.w};
  }
  __device__ __forceinline__ uint32_t word(int i) const { return i == 0 ? x : (i == 1 ? y : (i == 2 ? z : w)); }
  __device__ __forceinline__ bool has(int t) const { return (word(t >> 5) >> (t & 31)) & 1u; }
  __device__ __forceinline__ void set(int t) {
    const uint32_t b = 1u << (t & 31);
    const int i = t >> 5;
    x |= i == 0 ? b : 0u;
    y |= i == 1 ? b : 0u;
    z |= i == 2 ? b : 0u;
    w |= i == 3 ? b : 0u;
  }
  __device__ __forceinline__ bool any() const { return (x | y | z | w) != 0u; }
  __device__ __forceinline__ int count() const { return __popc(x) + __popc(y) + __popc(z) + __popc(w); }
  __device__ __forceinline__ Bits4 operator&(const Bits4& o) const { return Bits4{x & o.x, y & o.y, z & o.z, w & o.w}; }
  __device__ __forceinline__ Bits4 operator|(const Bits4& o) const { return Bits4{x | o.x, y | o.y, z | o.z, w | o.w}; }
  __device__ __forceinline__ Bits4 andnot(const Bits4& o) const {
    return Bits4{x & ~o.x, y & ~o.y, z & ~o.z, w & ~o.w};
  }
  __device__ __forceinline__ int lowest() const {
    return x ? __ffs(x) - 1 : (y ? 31 + __ffs(y) : (z ? 63 + __ffs(z) : (w ? 95 + __ffs(w) : -1)));
  }
  __device__ __forceinline__ void clear_lowest() {
    if (x)
      x &= x - 1u;
    else if (y)
      y &= y - 1u;
    else if (z)
      z &= z - 1u;
    else
      w &= w - 1u;
  }
};

struct Tables {
  int n_term, T1, S, NNT, P, Q, C, n_cat, LN;
  int NS, V, eos, W, D;
  int Vp;     // V rounded up to a multiple of 32: the row length of the id-indexed tables
  Bits4 ign;  // ignored terminals (the set I)
  Bits4 cm;   // category terminals
  Bits4 par;  // the terminals that the parser sees (not ignored, without $end)
  int cat_term[32];
  // staged block: these arrays (and live_any) live contiguously in `blob`
  const uint8_t* blob;
  int blob_bytes;  // 0 = too large to stage in shared memory
  const uint8_t* byte_class;
  const uint16_t* next;
  const uint32_t* acc;
  const uint32_t* live;
  const int16_t* action;
  const uint16_t* go;
  const uint16_t* plhs;
  const uint32_t* shift_mask;  // S * 4: terminals whose action is SHIFT
  const uint32_t* red_off;     // S + 1: reduce groups of state s are red_off[s] .. red_off[s+1]
  const uint16_t* red_p;       // each reduce group's production as plen << 10 | lhs
  const uint32_t* red_mask;    // 4 per reduce group: its lookahead terminals
  // identifier trie
  const uint32_t* lx_pcats;
  const uint32_t* lx_wcats;
  // open-addressing hash of the identifier-trie edges: key = node * 256 + byte,
  // entry = {key, child, child's prefix categories, child's word categories}
  const uint4* lx_hash;
  uint32_t lx_hmask;
  int lx_hshift;
  uint32_t root_pc, root_wc;
  // vocabulary trie
  const int32_t* spell_off;
  const uint8_t* spell_bytes;
  const uint4* spell16;  // first 16 bytes of each spelling, zero padded (one load per walk)
  const int32_t* spell_of_id;
  const int32_t* id_of_spell;  // NS: the first of each spelling's ids (a list in any order)
  const int32_t* next_alias;   // Vp: the next id of the spelling's list, -1 after the last
  const int32_t* first_of_byte;
  const uint8_t* first_byte_by_id;
  const uint32_t* killw;       // Q * W: bit j of word (q, wi): id 32 wi + j's first byte ends a lexeme at q
  // CI tables (one per lexer state in the precomputed set; table 0 = start state)
  int ci_on;
  int n_tbl;
  int ncls;                   // distinct terminal sets of the CI class ids: the classes that the step works with
  int nselw;
  const int16_t* tbl_of_q;
  const int32_t* tbl_q;
  const uint16_t* cls_by_id;  // n_tbl * V
  const int32_t* cd_off;      // n_tbl + 1
  const int32_t* cd_list;     // spelling indices per table, in any order
  const uint16_t* cd_key;     // per cd_list entry: class of its first stack-dependent emission
  // verdict classes: table k owns records vc_off[k] .. vc_off[k+1] of vc_rec
  const int32_t* vc_off;
  const uint16_t* vc_rec;     // kRecLen per verdict class
  const uint16_t* vc_first;   // class id of each verdict class's first event
  const uint32_t* vc_by_id;   // n_tbl * V: verdict class (within its table) of kClsVC spellings, or NULL
                              // when the class codes carry it (vc_inline)
  int vc_inline;              // 1: a verdict-class id's code is 32 nselw + its class index
  const uint32_t* cls_sets;   // ncls * 4: terminal set of every class (staged too where o_sets >= 0)
  const uint16_t* cls_map;    // class of every CI class id
  const uint32_t* acc_sym;    // S: the symbol entering each state (audit node hash)
  // a chain on a stack of d entries takes at most (d + 1) * chain_rate + chain_base steps, and pushes fewer
  // entries than a walk's scratch holds (chain_bounds; chain_rate 0: not shown, tokens are fed by one lane)
  int chain_rate, chain_base;
  // per lexer state q and category bits c, at q << n_cat | c (lexeme_tables):
  const uint64_t* ev_list;  // the emission's candidates (LexBatch::ev; 0: none, count 0x7F: more than it holds)
  const uint32_t* live_any; // bit set: a lexeme there is live
  const uint32_t* cat_live; // bit per lexer state: a lexicon category is live there
  // byte offsets of the staged block's arrays in it
  int o_class, o_next, o_acc, o_live, o_action, o_go, o_lhs, o_shift, o_roff, o_rp, o_red, o_lany, o_catq, o_tblq, o_sets;
};

extern __shared__ __align__(16) uint8_t smem[];

// The tables as a kernel's parameter reads them: where the block is staged,
// from its place in dynamic shared memory.  The parameter stays in constant
// memory and the offsets are operands of the address arithmetic, with 32-bit
// shared-memory loads; a descriptor in shared memory, rebased onto the block,
// cost a look-up of the pointer and a generic 64-bit load per access, and its
// copying by each block.
template <bool STAGED>
struct TabT : Tables {
  TabT() = default;
  explicit TabT(const Tables& t) : Tables(t) {
    if (!STAGED) blob_bytes = 0;
  }
  template <typename E>
  __device__ __forceinline__ E get(const E* p, int o, int i) const {
    return STAGED ? reinterpret_cast<const E*>(smem + o)[i] : p[i];
  }
  __device__ __forceinline__ Bits4 get4(const uint32_t* p, int o, int i) const {
    const uint4 v = STAGED ? reinterpret_cast<const uint4*>(smem + o)[i] : reinterpret_cast<const uint4*>(p)[i];
    return Bits4{v.x, v.y, v.z, v.w};
  }
  __device__ __forceinline__ int cls(int b) const { return get(byte_class, o_class, b); }
  __device__ __forceinline__ int nxt(int i) const { return get(next, o_next, i); }
  __device__ __forceinline__ int act(int i) const { return get(action, o_action, i); }
  __device__ __forceinline__ int gto(int i) const { return get(go, o_go, i); }
  __device__ __forceinline__ int lhs(int p) const { return get(plhs, o_lhs, p); }
  __device__ __forceinline__ uint32_t roff(int s) const { return get(red_off, o_roff, s); }
  __device__ __forceinline__ int rp(int e) const { return get(red_p, o_rp, e); }
  __device__ __forceinline__ Bits4 acc4(int q) const { return get4(acc, o_acc, q); }
  __device__ __forceinline__ Bits4 live4(int q) const { return get4(live, o_live, q); }
  __device__ __forceinline__ Bits4 shift4(int s) const { return get4(shift_mask, o_shift, s); }
  __device__ __forceinline__ Bits4 red4(int e) const { return get4(red_mask, o_red, e); }
  __device__ __forceinline__ Bits4 set4(int c) const {
    if (STAGED && o_sets >= 0) {
      const uint4 v = reinterpret_cast<const uint4*>(smem + o_sets)[c];
      return Bits4{v.x, v.y, v.z, v.w};
    }
    return Bits4::load(cls_sets + c * 4);
  }
  __device__ __forceinline__ int tblq(int q) const { return get(tbl_of_q, o_tblq, q); }
  __device__ __forceinline__ bool cat_live_at(int q) const { return (get(cat_live, o_catq, q >> 5) >> (q & 31)) & 1u; }
  __device__ __forceinline__ bool live_any_at(int i) const { return (get(live_any, o_lany, i >> 5) >> (i & 31)) & 1u; }
};

// Work counters of a walk, kept in the lane's registers when the walk is
// measured and absent (a null pointer the compiler sees) otherwise:
// [0] lexer steps (trie node visits), [1] ACTION lookups (one per reduce
// chain step, for a terminal or a set of terminals), [2] GOTO lookups,
// [3] verdict-class events evaluated.
__device__ __forceinline__ void count_work(uint32_t* ctr, int k) {
  if (ctr) ++ctr[k];
}

// Membership test in a 4-word set stored in memory.
__device__ __forceinline__ bool bit4(const uint32_t* m, int t) { return (m[t >> 5] >> (t & 31)) & 1u; }

// Copy the staged block into shared memory (at the start of the kernel's
// dynamic shared memory, where TabT<true> reads it) with one bulk asynchronous
// copy (the block is 16-byte aligned and a multiple of 16 bytes), completion
// tracked by an mbarrier.  The wait is bounded; if it gives up, the block is
// copied again with plain loads (same bytes), so the result never depends on
// the bulk copy finishing.  Every thread of the block must call this.
template <bool STAGED>
__device__ __forceinline__ void stage_tables(const TabT<STAGED>& t) {
  if constexpr (STAGED) {
    __shared__ __align__(8) uint64_t s_bar;
    __shared__ int s_late;
    const uint32_t bar = (uint32_t)__cvta_generic_to_shared(&s_bar);
    if (threadIdx.x == 0) {
      s_late = 0;
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar) : "memory");
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
      asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(t.blob_bytes)
                   : "memory");
      asm volatile(
          "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
              (uint32_t)__cvta_generic_to_shared(smem)),
          "l"(t.blob), "r"(t.blob_bytes), "r"(bar)
          : "memory");
    }
    __syncthreads();
    uint32_t done = 0;
    for (int it = 0; it < (1 << 20) && !done; ++it)
      asm volatile(
          "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], 0;\n selp.u32 %0, 1, 0, p;\n}"
          : "=r"(done)
          : "r"(bar)
          : "memory");
    if (!done) s_late = 1;
    __syncthreads();
    if (s_late) {
      const uint4* src = reinterpret_cast<const uint4*>(t.blob);
      uint4* dst = reinterpret_cast<uint4*>(smem);
      for (int i = threadIdx.x; i < (t.blob_bytes >> 4); i += blockDim.x) dst[i] = src[i];
      __syncthreads();
    }
  }
}

// Programmatic dependent launch: the step's kernels are launched so that each
// may start while its predecessor in the stream finishes; everything a kernel
// does before this wait touches only the spec's read-only tables.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

constexpr uint32_t kHashEmpty = 0xFFFFFFFFu;

// Child of identifier-trie node lx on byte b (-1 if none), with the child's
// prefix / word category bits (0 when there is no child); q is the lexer state
// after the byte.  A trie node spells a prefix of some category's word, so
// that category is live in the state that the prefix leaves: where none is,
// there is no child, and no probe (punctuation, numbers and blanks, each an L2
// access otherwise).  One 16-byte load per probe; the table is at most half
// full, so probing ends at an empty slot.
template <class T>
__device__ __forceinline__ int lex_step(const T& t, int q, int lx, int b, uint32_t& pc, uint32_t& wc) {
  pc = 0u;
  wc = 0u;
  if (lx < 0 || !t.cat_live_at(q)) return -1;
  const uint32_t key = (uint32_t)lx * 256u + (uint32_t)b;
  uint32_t h = (key * 0x9E3779B1u) >> t.lx_hshift;
#pragma unroll 1
  for (uint32_t i = 0; i <= t.lx_hmask; ++i) {
    const uint4 e = __ldg(&t.lx_hash[h]);
    if (e.x == key) {
      pc = e.z;
      wc = e.w;
      return (int)e.y;
    }
    if (e.x == kHashEmpty) return -1;
    h = (h + 1u) & t.lx_hmask;
  }
  return -1;
}

// Terminal set of DFA state q filtered by the lexicon: non-category terminals
// pass, category terminal c passes iff bit c of `cats` is set.
template <class T>
__device__ __forceinline__ Bits4 lex_filter(const T& t, const Bits4 v, uint32_t cats) {
  Bits4 out = v.andnot(t.cm);
#pragma unroll 1
  while (cats) {
    const int c = __ffs(cats) - 1;
    cats &= cats - 1;
    const int term = t.cat_term[c];
    if (v.has(term)) out.set(term);
  }
  return out;
}

// live'(q, r): terminals live at q, category terminals only while r is a
// prefix of one of their words (pc = prefix category bits of r's trie node).
template <class T>
__device__ __forceinline__ Bits4 live_prime(const T& t, int q, uint32_t pc) { return lex_filter(t, t.live4(q), pc); }

// Emission candidates of r: terminals accepting at q, category terminals only
// if r is one of their words (wc = word category bits of r's trie node).
template <class T>
__device__ __forceinline__ Bits4 cands(const T& t, int q, uint32_t wc) { return lex_filter(t, t.acc4(q), wc); }

template <class T>
__device__ __forceinline__ int max_chain_of(const T& t) { return 2 * t.D + 256; }

// A lane's small array: element i lives at p[i * s].  Walk lanes keep their
// overlays in shared memory interleaved across the warp (s = 32, no bank
// conflicts); single-thread users keep them in local arrays (s = 1).
struct LArr {
  uint16_t* p;
  int s;
  __device__ __forceinline__ uint16_t& operator[](int i) const { return p[i * s]; }
};

// Reduce chain of terminal tau on the virtual stack base[0:keep] ++ ovl[0:m]
// (Sec. 3.2, "allowed terminals by simulation").  Returns the ACTION code that
// ends it (> 0: shift to code-1, or kAccept), 0 on error, -1 on a bound.  On
// shift/accept, (keep_o, m_o, scr[0:ns]) is the stack under the pushed state.
template <class T, typename OV>
__device__ __forceinline__ int simulate(const T& t, const uint16_t* base, int keep, OV ovl, int m, int tau,
                                        LArr scr, int cap, int& keep_o, int& m_o, int& ns, int max_chain,
                                        uint32_t* ctr = nullptr) {
  int k = keep, mm = m;
  ns = 0;
  int top = mm ? ovl[mm - 1] : base[k - 1];
#pragma unroll 1
  for (int it = 0; it < max_chain; ++it) {
    if (top >= t.S) return 0;
    count_work(ctr, 1);
    const int a = t.act(top * t.T1 + tau);
    if (a == 0) return 0;
    if (a > 0) {
      keep_o = k;
      m_o = mm;
      return a;
    }
    const int code = -a - 1;  // plen << 10 | lhs
    int n = code >> 10;
    int x = min(n, ns);
    ns -= x;
    n -= x;
    x = min(n, mm);
    mm -= x;
    n -= x;
    k -= n;
    if (k < 1) return 0;
    const int top2 = ns ? scr[ns - 1] : (mm ? ovl[mm - 1] : base[k - 1]);
    if (top2 >= t.S) return 0;
    if (ns >= cap) return -1;
    count_work(ctr, 2);
    top = t.gto(top2 * t.NNT + (code & 1023));
    scr[ns++] = (uint16_t)top;
  }
  return -1;
}

// The terminals of G whose reduce chains on the virtual stack reach SHIFT:
// simulate() for a set of terminals at once.  Terminals travel together while
// they take the same action; where the remaining ones reduce by different
// productions, the group of the first production listed for the state goes
// on and the others are simulated again from the start in a later round
// (they follow the same path up to that state).  After kSetRounds rounds the
// rest is simulated one terminal at a time.  `bound` is set on a bound.
constexpr int kSetRounds = 8;

template <class T, typename OV>
__device__ __forceinline__ Bits4 simulate_set(const T& t, const uint16_t* base, int keep, OV ovl, int m, Bits4 G,
                                              LArr scr, int cap, int max_chain, bool& bound,
                                              uint32_t* ctr = nullptr) {
  Bits4 res = Bits4::zero();
  Bits4 todo = G;
#pragma unroll 1
  for (int round = 0; round < kSetRounds && todo.any(); ++round) {
    Bits4 g = todo;
    todo = Bits4::zero();
    int k = keep, mm = m, ns = 0;
    int it = 0;
    int top = mm ? ovl[mm - 1] : base[k - 1];
#pragma unroll 1
    for (; it < max_chain && g.any(); ++it) {
      if (top >= t.S) break;
      count_work(ctr, 1);
      const Bits4 sh = t.shift4(top);
      res = res | (g & sh);
      g = g.andnot(sh);
      if (!g.any()) break;
      int p = -1;
      Bits4 gp = Bits4::zero();
#pragma unroll 1
      for (uint32_t e = t.roff(top); e < t.roff(top + 1); ++e) {
        const Bits4 x = g & t.red4(e);
        if (!x.any()) continue;
        if (p < 0) {
          p = t.rp(e);
          gp = x;
        } else {
          todo = todo | x;
        }
      }
      if (p < 0) break;  // the rest is an error here
      g = gp;
      int n = p >> 10;  // p: plen << 10 | lhs
      int x = min(n, ns);
      ns -= x;
      n -= x;
      x = min(n, mm);
      mm -= x;
      n -= x;
      k -= n;
      if (k < 1) break;
      const int top2 = ns ? scr[ns - 1] : (mm ? ovl[mm - 1] : base[k - 1]);
      if (top2 >= t.S) break;
      if (ns >= cap) {
        bound = true;
        return res;
      }
      count_work(ctr, 2);
      top = t.gto(top2 * t.NNT + (p & 1023));
      scr[ns++] = (uint16_t)top;
    }
    if (it == max_chain && g.any()) {
      bound = true;
      return res;
    }
  }
#pragma unroll 1
  while (todo.any()) {
    const int tau = todo.lowest();
    todo.clear_lowest();
    int keep_o, m_o, ns;
    const int a = simulate(t, base, keep, ovl, m, tau, scr, cap, keep_o, m_o, ns, max_chain, ctr);
    if (a < 0) {
      bound = true;
      return res;
    }
    if (a > 0 && a != kAccept) res.set(tau);
  }
  return res;
}

// Per-lane walk state.  Acur is the allowed-terminal set of the current
// virtual stack when it is known without simulation: the context's set before
// any shift, and after the first shift of terminal tau the precomputed set
// A2[tau] (if the caller has it); after a second shift it is NULL and the
// reduce chains are simulated.
struct Walker {
  const uint16_t* base;
  int keep, m;
  int q, lx;
  uint32_t pc, wc;  // category bits of trie node lx (0 if lx < 0)
  int nshift;
  bool shifted;
  int pend;  // a first shift not yet applied to the overlay (-1: none)
  const uint32_t* Acur;
  const uint32_t* A2;
  LArr ovl, scr;  // overlay and simulation scratch, `cap` entries each
  int cap;
  uint32_t* ctr;  // work counters (measured walks), or NULL
};

__device__ __forceinline__ void walker_init(Walker& w, LArr ovl_store, LArr scr_store, int cap, const uint16_t* base,
                                            int keep, const uint16_t* ovl, int m, int q, int lx, uint32_t pc,
                                            uint32_t wc, const uint32_t* A, const uint32_t* A2,
                                            uint32_t* ctr = nullptr) {
  w.ctr = ctr;
  w.ovl = ovl_store;
  w.scr = scr_store;
  w.cap = cap;
  w.base = base;
  w.keep = keep;
  w.m = min(m, cap);  // callers pass m <= cap; a larger m would only be a caller bug
#pragma unroll 1
  for (int k = 0; k < w.m; ++k) w.ovl[k] = ovl[k];
  w.q = q;
  w.lx = lx;
  w.pc = pc;
  w.wc = wc;
  w.nshift = 0;
  w.shifted = false;
  w.pend = -1;
  w.Acur = A;
  w.A2 = A2;
}

__device__ __forceinline__ bool commit(Walker& w, int keep_o, int m_o, int ns, int target) {
  if (m_o + ns + 1 > w.cap) return false;
  w.keep = keep_o;
  w.m = m_o;
#pragma unroll 1
  for (int i = 0; i < ns; ++i) w.ovl[w.m++] = w.scr[i];
  w.ovl[w.m++] = (uint16_t)target;
  return true;
}

// Apply a deferred first shift to the overlay.  The terminal is in the
// allowed set of the stack it was deferred at, so it reaches SHIFT.
template <class T>
__device__ __forceinline__ bool materialize(const T& t, Walker& w, int max_chain) {
  int keep_o, m_o, ns;
  const int a = simulate(t, w.base, w.keep, w.ovl, w.m, w.pend, w.scr, w.cap, keep_o, m_o, ns, max_chain, w.ctr);
  w.pend = -1;
  if (a <= 0 || a == kAccept) return false;
  return commit(w, keep_o, m_o, ns, a - 1);
}

// Emission of the pending lexeme (Sec. 2, contextual resolution): the first
// candidate in priority order that is ignored or reaches SHIFT wins and is
// shifted.  While the walker knows the allowed set of its stack (Acur) the
// pick is a set test; a first shift whose successor allowed set is known (A2)
// is only recorded, and applied to the overlay when a later step needs the
// stack itself.  Returns 1 ok, 0 reject, -1 bound.
template <class T>
__device__ __forceinline__ int emit_set(const T& t, Walker& w, Bits4 K, int max_chain) {
#pragma unroll 1
  while (K.any()) {
    const int tau = K.lowest();
    K.clear_lowest();
    if (t.ign.has(tau)) return 1;
    if (w.Acur && !bit4(w.Acur, tau)) continue;
    if (w.Acur && w.nshift == 0 && w.A2) {
      w.pend = tau;
      w.shifted = true;
      w.Acur = w.A2 + tau * 4;
      w.nshift = 1;
      return 1;
    }
    if (w.pend >= 0 && !materialize(t, w, max_chain)) return -1;
    if (!w.Acur && K.count() > 0) {
      // several candidates left: find the first that reaches SHIFT (or is
      // ignored) with one set simulation, then simulate that one to shift it
      bool bound = false;
      Bits4 rest = K;
      rest.set(tau);
      const Bits4 ok =
          simulate_set(t, w.base, w.keep, w.ovl, w.m, rest.andnot(t.ign), w.scr, w.cap, max_chain, bound, w.ctr);
      if (bound) return -1;
      const int pick = (ok | (rest & t.ign)).lowest();
      if (pick < 0) return 0;
      if (t.ign.has(pick)) return 1;
      K = Bits4::zero();
      int keep_o, m_o, ns;
      const int a = simulate(t, w.base, w.keep, w.ovl, w.m, pick, w.scr, w.cap, keep_o, m_o, ns, max_chain, w.ctr);
      if (a <= 0 || a == kAccept || !commit(w, keep_o, m_o, ns, a - 1)) return -1;
      w.shifted = true;
      w.Acur = (w.nshift == 0 && w.A2) ? w.A2 + pick * 4 : nullptr;
      ++w.nshift;
      return 1;
    }
    int keep_o, m_o, ns;
    int a = simulate(t, w.base, w.keep, w.ovl, w.m, tau, w.scr, w.cap, keep_o, m_o, ns, max_chain, w.ctr);
    if (a < 0) return -1;
    if (a > 0 && a != kAccept) {
      if (!commit(w, keep_o, m_o, ns, a - 1)) return -1;
      w.shifted = true;
      w.Acur = (w.nshift == 0 && w.A2) ? w.A2 + tau * 4 : nullptr;
      ++w.nshift;
      return 1;
    }
  }
  return 0;
}

template <class T>
__device__ __forceinline__ int emit(const T& t, Walker& w, int max_chain) {
  return emit_set(t, w, cands(t, w.q, w.wc), max_chain);
}

// Def. 2 trailing liveness for live set L.  1 / 0 / -1.
template <class T>
__device__ __forceinline__ int trailing_set(const T& t, Walker& w, Bits4 L, int max_chain) {
  if ((L & t.ign).any()) return 1;
  if (const uint32_t* A = w.Acur) return (L & Bits4::load(A)).any() ? 1 : 0;
  if (w.pend >= 0 && !materialize(t, w, max_chain)) return -1;
  if (L.count() == 1) {
    int keep_o, m_o, ns;
    const int a =
        simulate(t, w.base, w.keep, w.ovl, w.m, L.lowest(), w.scr, w.cap, keep_o, m_o, ns, max_chain, w.ctr);
    if (a < 0) return -1;
    return a > 0 && a != kAccept ? 1 : 0;
  }
  bool bound = false;
  const Bits4 ok = simulate_set(t, w.base, w.keep, w.ovl, w.m, L, w.scr, w.cap, max_chain, bound, w.ctr);
  if (bound) return -1;
  return ok.any() ? 1 : 0;
}

template <class T>
__device__ __forceinline__ int trailing_live(const T& t, Walker& w, int max_chain) {
  return trailing_set(t, w, live_prime(t, w.q, w.pc), max_chain);
}

// A spelling's bytes: the first 16 come from one 16-byte load into registers,
// longer spellings read the rest from the byte array.
struct Spell {
  uint4 head;
  const uint8_t* all;
  int len;
  __device__ __forceinline__ int at(int i) const {
    if (i < 16) {
      const uint32_t w = i < 8 ? (i < 4 ? head.x : head.y) : (i < 12 ? head.z : head.w);
      return (int)((w >> ((i & 3) * 8)) & 0xFFu);
    }
    return all[i];
  }
};

template <class T>
__device__ __forceinline__ Spell load_spell(const T& t, int s) {
  Spell sp;
  const int off = t.spell_off[s];
  sp.len = t.spell_off[s + 1] - off;
  sp.head = __ldg(&t.spell16[s]);
  sp.all = t.spell_bytes + off;
  return sp;
}

// Walk one token's bytes (Sec. 4.1).  1 = the output stays a viable prefix,
// 0 = rejected, -1 = bound.
template <class T>
__device__ __forceinline__ int walk_bytes(const T& t, Walker& w, const Spell& sp, int max_chain) {
  const int len = sp.len;
#pragma unroll 1
  for (int i = 0; i < len; ++i) {
    count_work(w.ctr, 0);
    const int b = sp.at(i);
    const int c = t.cls(b);
    int nq = t.nxt(w.q * t.C + c);
    if (nq == kDead) {
      if (w.q == kStart) return 0;
      const int e = emit(t, w, max_chain);
      if (e <= 0) return e;
      w.q = kStart;
      w.lx = 0;
      w.pc = t.root_pc;
      w.wc = t.root_wc;
      nq = t.nxt(kStart * t.C + c);
      if (nq == kDead) return 0;
    }
    w.q = nq;
    w.lx = lex_step(t, w.q, w.lx, b, w.pc, w.wc);
    const Bits4 L = live_prime(t, w.q, w.pc);
    const bool any = w.Acur ? (L & (Bits4::load(w.Acur) | t.ign)).any() : L.any();
    if (!any) return 0;
  }
  return trailing_live(t, w, max_chain);
}

// ---- feeding tokens with a warp (grid_advance, the decoding step)
//
// The lexer does not look at the parser: where a lexeme ends, and which
// terminals it can be, follows from the bytes alone, because an emission
// always takes the whole lexeme.  So a warp lexes up to 32 tokens at once
// (lex_batch) and leaves the candidate list of each lexeme that ends in them,
// and the parser (parse_batch) only has to go through the lists: its lanes run
// the reduce chains of a list's candidates side by side, and the first in
// priority order that reaches SHIFT is shifted.
constexpr int kLexBytes = 384;  // bytes of one batch, at most
constexpr int kLexCand = 7;     // candidates of one lexeme, at most (more: the lane-serial feed)
constexpr int kChainNs = 8;     // entries that a chain pushes, at most

struct LexState {
  int q, lx;
  uint32_t pc, wc;
};

// What lex_batch leaves about its tokens.
struct LexBatch {
  uint64_t ev[kLexBytes];  // per lexeme end: candidates in priority order, a byte each; top byte: their count,
                           // | 0x80 if an ignored terminal follows them; 0: the stack stays as it is
  LexState in, out[32], end;     // the lexer's state before the batch, after each token, after the batch
  uint16_t q[kLexBytes];         // per byte: the DFA state after it
  uint16_t start[kLexBytes + 1]; // per lexeme: its first byte in the batch
  uint16_t evo[33];              // per token: the lexeme ends before it
  uint8_t cls[kLexBytes], byte[kLexBytes];
  uint8_t last[kLexBytes];       // token + 1 if the byte is its last
  uint8_t st[32];                // 0: no token, 1: lexed, 2: for the lane-serial feed (EOS, refused, too long)
  int next;                      // the first token after the batch
};

// The lane's token of the batch that starts at token k, loaded ahead of lexing it.
struct LexToken {
  int st;  // as LexBatch::st
  Spell sp;
};

template <class T>
__device__ __forceinline__ LexToken lex_fetch(const T& t, const int32_t* tokens, int k, int n_steps, int lane) {
  const int tok = k + lane < n_steps ? tokens[k + lane] : -1;
  LexToken x;
  x.st = tok < 0 ? 0 : 2;
  x.sp.len = 0;
  if (tok >= 0 && tok < t.V && tok != t.eos) {
    const int s = t.spell_of_id[tok];
    if (s >= 0) {
      x.sp = load_spell(t, s);
      x.st = 1;
    }
  }
  return x;
}

// Lex the next tokens, from number k on, from state `carry`.  The DFA's chain
// through the bytes (two shared-memory look-ups a byte) is all that is serial;
// the walks through the identifier trie (a dependent L2 access a byte) run a
// lexeme per lane, once the DFA has found where the lexemes start.
template <class T>
__device__ __forceinline__ void lex_batch(const T& t, const T& ts, const LexToken& own, int k, int n_steps,
                                          int lane, LexState& carry, LexBatch& L) {
  const Spell& sp = own.sp;
  int st = own.st;
  int at = sp.len;
  for (int d = 1; d < 32 && d < n_steps - k; d <<= 1) {
    const int v = __shfl_up_sync(0xffffffffu, at, d);
    if (lane >= d) at += v;
  }
  const uint32_t over = __ballot_sync(0xffffffffu, at > kLexBytes);
  int n = min(32, n_steps - k);  // tokens of the batch: as many as fit, at least one
  if (over) n = min(n, max(1, __ffs(over) - 1));
  if (lane >= n) st = 0;
  if (at > kLexBytes && st == 1) st = 2;  // (lane 0: a token that never fits)
  const uint32_t act = __ballot_sync(0xffffffffu, st == 1);
  at -= sp.len;
  if (st == 1) {
    for (int i = 0; i < sp.len; ++i) {
      const int b = sp.at(i);
      L.byte[at + i] = (uint8_t)b;
      L.cls[at + i] = ts.cls(b);
      L.last[at + i] = i + 1 == sp.len ? (uint8_t)(lane + 1) : (uint8_t)0;
    }
  }
  const int total = act ? __shfl_sync(0xffffffffu, at + sp.len, 31 - __clz(act)) : 0;
  __syncwarp();
  // the DFA, the same in every lane
  int q = carry.q, kills = 0, bad = total;  // bad: the first byte that a token is refused at
  if (lane == 0) L.start[0] = 0;
  const int row0 = kStart * ts.C;
  for (int i = 0; i < total; ++i) {
    const int c = L.cls[i];
    int nq = ts.nxt(q * ts.C + c);
    if (nq == kDead) {
      if (q != kStart) nq = ts.nxt(row0 + c);
      if (nq == kDead) {
        bad = i;
        break;
      }
      ++kills;
      if (lane == 0) L.start[kills] = (uint16_t)i;
    }
    q = nq;
    if (lane == 0) {
      L.q[i] = (uint16_t)q;
      if (L.last[i]) L.evo[L.last[i]] = (uint16_t)kills;
    }
  }
  __syncwarp();
  // the lexemes, one per lane: the trie, the lexeme's liveness, its candidates
  for (int j = lane; j <= kills; j += 32) {
    const int a = L.start[j], z = j < kills ? L.start[j + 1] : bad;
    LexState s = j == 0 ? carry : LexState{kStart, 0, t.root_pc, t.root_wc};
    int i = a;
    for (; i < z; ++i) {
      s.q = L.q[i];
      s.lx = lex_step(ts, s.q, s.lx, L.byte[i], s.pc, s.wc);
      const int id = (s.q << ts.n_cat) | (int)s.pc;
      if (!ts.live_any_at(id)) break;
      if (L.last[i]) L.out[L.last[i] - 1] = s;
    }
    if (i < z) {
      bad = min(bad, i);
    } else if (j < kills) {
      uint64_t list = __ldg(&t.ev_list[(s.q << t.n_cat) | (int)s.wc]);
      const int cnt = (int)(list >> 56) & 0x7F;
      if (list == 0 || cnt > kLexCand) bad = min(bad, z);
      if (cnt == 0) list = 0;  // an ignored terminal first
      L.ev[j] = list;
    }
  }
  bad = __reduce_min_sync(0xffffffffu, bad);
  if (st == 1 && at + sp.len > bad) st = 2;
  L.st[lane] = (uint8_t)st;
  __syncwarp();
  const uint32_t good = __ballot_sync(0xffffffffu, st == 1);
  const LexState was = carry;
  if (good) carry = L.out[31 - __clz(good)];
  if (lane == 0) {
    L.in = was;
    L.end = carry;
    L.next = k + n;
  }
  __syncwarp();
}

// The parser's side, the same in every lane of the warp.  win[0:depth) is the
// stack.  Tokens before `tok` are accepted; the state at the start of token
// `tok` is (s_depth, s), and undo[low:s_depth) holds what its emissions took
// off the stack.
struct Feed {
  uint16_t* win;
  uint16_t* undo;
  uint16_t* scr;  // kChainNs * 32
  int cap;        // entries of win
  int depth, low, s_depth, tok;
  int wlow;  // entries below it were never written
  bool any;  // a token was fed
  LexState s;
};

// Reduce chain of tau on win[0:depth): simulate() for a stack without overlay.
template <class T>
__device__ __forceinline__ int chain(const T& t, const uint16_t* win, int depth, int tau, uint16_t* scr,
                                     int& keep_o, int& ns_o, int max_chain) {
  int k = depth, ns = 0, bk = depth;
  int top = win[k - 1], bv = top;  // bv = win[bk - 1]
#pragma unroll 1
  for (int it = 0; it < max_chain; ++it) {
    if (top >= t.S) return 0;
    const int a = t.act(top * t.T1 + tau);
    if (a >= 0) {
      keep_o = k;
      ns_o = ns;
      return a;
    }
    const int code = -a - 1;  // plen << 10 | lhs
    const int n = code >> 10, x = min(n, ns);
    ns -= x;
    k -= n - x;
    if (k < 1) return 0;
    if (k != bk) {
      bk = k;
      bv = win[k - 1];
    }
    const int top2 = ns ? scr[(ns - 1) * 32] : bv;
    if (top2 >= t.S) return 0;
    if (ns >= kChainNs) return -1;
    top = t.gto(top2 * t.NNT + (code & 1023));
    scr[ns * 32] = (uint16_t)top;
    ++ns;
  }
  return -1;
}

// Def. 2 trailing liveness of lexer state (q, pc) on win[0:depth), 32 terminals at a time.  1 / 0 / -1.
template <class T>
__device__ __forceinline__ int feed_live(const T& t, const Feed& f, int q, uint32_t pc, int lane, int max_chain) {
  const Bits4 Lv = live_prime(t, q, pc);
  if ((Lv & t.ign).any()) return 1;
  bool ok = false, bound = false;
  for (int w = 0; w < 4; ++w) {
    const uint32_t word = Lv.word(w);
    if (!word) continue;
    int a = 0, k, ns;
    if ((word >> lane) & 1u) a = chain(t, f.win, f.depth, 32 * w + lane, f.scr + lane, k, ns, max_chain);
    ok |= __any_sync(0xffffffffu, a > 0 && a != kAccept);
    bound |= __any_sync(0xffffffffu, a < 0);
  }
  return bound ? -1 : (ok ? 1 : 0);
}

// Shift on win: lane l's chain ended in SHIFT `a` over win[0:ko) ++ its ns
// scratch entries.  False where a token pushes more than an overlay holds or
// the window is full (the lane-serial feed knows what that means).
__device__ __forceinline__ bool feed_shift(Feed& f, int a, int ko, int ns, int l, int lane) {
  ko = __shfl_sync(0xffffffffu, ko, l);
  ns = __shfl_sync(0xffffffffu, ns, l);
  a = __shfl_sync(0xffffffffu, a, l);
  const int low = min(f.low, ko), nd = ko + ns + 1;
  if (nd - low > kMaxOvl || nd > f.cap) return false;
  for (int i = low + lane; i < f.low; i += 32) f.undo[i] = f.win[i];
  __syncwarp();
  if (lane < ns) f.win[ko + lane] = f.scr[lane * 32 + l];
  if (lane == 0) f.win[ko + ns] = (uint16_t)(a - 1);
  __syncwarp();
  f.low = low;
  f.wlow = min(f.wlow, low);
  f.depth = nd;
  return true;
}

// Go through a batch's lists (its token k is number k0 + k).  True if
// every token was fed; false if the feed has to go on lane-serially at token
// f.tok, in the state at its start (the stack is put back by feed_back).
//
// A token is accepted when its own emissions succeed and the lexeme it leaves
// can still become an allowed terminal.  That test is not made where the next
// emission makes it: if the lexeme's emission shifts tau (or an ignored
// terminal), tau was live in the lexeme all along, on the same stack.  What is
// left is the test after the last token, and, where a chain could run into its
// bound (deep stacks of grammars with long chains), the test of every token,
// which would report that bound.
template <class T>
__device__ __forceinline__ bool parse_batch(const T& t, Feed& f, const LexBatch& L, int k0, int lane,
                                            int max_chain) {
  const int own = L.st[lane];
  uint32_t todo = __ballot_sync(0xffffffffu, own != 0);
  const uint32_t good = __ballot_sync(0xffffffffu, own == 1);
  f.any |= todo != 0u;
  while (todo) {
    const int k = __ffs(todo) - 1;
    todo &= todo - 1u;
    if (!((good >> k) & 1u)) return false;
    const uint32_t before = good & ((1u << k) - 1u);
    const int prev = before ? 31 - __clz(before) : -1;  // the token before it
    const int e1 = L.evo[k + 1];
    for (int e = prev < 0 ? 0 : L.evo[prev + 1]; e < e1; ++e) {
      const uint64_t ev = L.ev[e];
      if (ev == 0) continue;
      const int n = (int)(ev >> 56) & 0x7F;
      int a = 0, ko = 0, ns = 0;
      if (lane < n) a = chain(t, f.win, f.depth, (int)(ev >> (8 * lane)) & 0xFF, f.scr + lane, ko, ns, max_chain);
      if (__any_sync(0xffffffffu, a < 0)) return false;
      const uint32_t win = __ballot_sync(0xffffffffu, a > 0 && a != kAccept);
      if (!win && !(ev >> 63)) return false;
      if (k0 + k != f.tok) {  // the tokens before this one are accepted
        if (f.depth > t.D) return false;
        f.tok = k0 + k;
        f.s = prev < 0 ? L.in : L.out[prev];
        f.s_depth = f.low = f.depth;
      }
      if (!win) continue;  // ignored
      const int l = __ffs(win) - 1;
      if (!feed_shift(f, a, ko, ns, l, lane)) return false;
    }
    if ((f.depth + 1) * t.chain_rate + t.chain_base > max_chain &&
        feed_live(t, f, L.out[k].q, L.out[k].pc, lane, max_chain) != 1)
      return false;
  }
  return true;
}

// Feed one token of state `s` to win[0:depth), with the warp: the bytes are the
// same in every lane, a lexeme's candidates run their chains side by side, and
// the lexeme that is left is tested at the end.  False: for the lane-serial
// feed, at the token's start (feed_back).
template <class T>
__device__ __forceinline__ bool feed_one(const T& t, Feed& f, LexState& s, const Spell& sp, int lane, int max_chain) {
  const int len = sp.len;
#pragma unroll 1
  for (int i = 0; i < len; ++i) {
    const int b = sp.at(i);
    const int c = t.cls(b);
    int nq = t.nxt(s.q * t.C + c);
    if (nq == kDead) {
      if (s.q == kStart) return false;
      Bits4 K = cands(t, s.q, s.wc);
      for (;;) {  // the candidates, 32 terminals at a time
        if (!K.any()) return false;
        const int kw = K.x ? 0 : (K.y ? 1 : (K.z ? 2 : 3));
        const uint32_t word = K.word(kw), ig = word & t.ign.word(kw);
        if (ig & (0u - ig) & word & (0u - word)) break;  // an ignored terminal comes first
        int a = 0, ko = 0, ns = 0;
        if (((word & ~ig) >> lane) & 1u) a = chain(t, f.win, f.depth, 32 * kw + lane, f.scr + lane, ko, ns, max_chain);
        if (__any_sync(0xffffffffu, a < 0)) return false;
        const uint32_t ok = __ballot_sync(0xffffffffu, a > 0 && a != kAccept);
        if (!(ok | ig)) {
          if (kw == 0) K.x = 0u;
          else if (kw == 1) K.y = 0u;
          else if (kw == 2) K.z = 0u;
          else K.w = 0u;
          continue;
        }
        const int l = __ffs(ok | ig) - 1;
        if ((ok >> l) & 1u) {
          if (!feed_shift(f, a, ko, ns, l, lane)) return false;
        }
        break;
      }
      s.q = kStart;
      s.lx = 0;
      s.pc = t.root_pc;
      s.wc = t.root_wc;
      nq = t.nxt(kStart * t.C + c);
      if (nq == kDead) return false;
    }
    s.q = nq;
    s.lx = lex_step(t, s.q, s.lx, b, s.pc, s.wc);
    if (!live_prime(t, s.q, s.pc).any()) return false;
  }
  return f.depth <= t.D && feed_live(t, f, s.q, s.pc, lane, max_chain) == 1;
}

// The stack at the start of token f.tok.
__device__ __forceinline__ void feed_back(Feed& f, int lane) {
  __syncwarp();
  for (int i = f.low + lane; i < f.s_depth; i += 32) f.win[i] = f.undo[i];
  f.depth = f.s_depth;
  f.low = f.s_depth;
  __syncwarp();
}

// EOS gate (Sec. 3.2).  1 / 0 / -1.
template <class T>
__device__ __forceinline__ int eos_gate(const T& t, Walker& w, int max_chain) {
  if (w.q != kStart) {
    int e = emit(t, w, max_chain);
    if (e <= 0) return e;
  }
  if (w.pend >= 0 && !materialize(t, w, max_chain)) return -1;
  int keep_o, m_o, ns;
  int a = simulate(t, w.base, w.keep, w.ovl, w.m, t.n_term, w.scr, w.cap, keep_o, m_o, ns, max_chain, w.ctr);
  if (a < 0) return -1;
  return a == kAccept ? 1 : 0;
}

template <class T>
__device__ __forceinline__ int class_id(const T& t, int kind, int q, uint32_t cats) {
  return ((kind * t.Q + q) << t.n_cat) | (int)(cats & ((1u << t.n_cat) - 1u));
}

// Sec. 4.2 CI/CD classification of one spelling from lexer state (q, lx),
// with the stack abstracted away.  Emissions whose first candidate is ignored
// leave the stack alone and are dropped; every other emission, and the final
// liveness test, is a stack-dependent event.
//   no event but the final test      -> CI live class / kClsAcc / kClsRej
//   one emission, then ignored bytes -> CI candidate class (or kClsAcc)
//   otherwise                        -> kClsVC with its event record `rec`
//                                       (kClsCD when it has more than kMaxEv
//                                       emissions; then `first_key` is the
//                                       class of the first one, 0xFFFF if that
//                                       emission always succeeds)
template <class T>
__device__ __forceinline__ uint16_t classify(const T& t, int q, int lx, const uint8_t* bytes, int len,
                                             uint16_t& first_key, uint16_t* rec) {
  first_key = 0xFFFF;
  uint32_t pc = lx == 0 ? t.root_pc : 0u, wc = lx == 0 ? t.root_wc : 0u;
  int n = 0;
  bool first_ign = false, overflow = false;
#pragma unroll 1
  for (int i = 0; i < len; ++i) {
    const int b = bytes[i];
    const int c = t.cls(b);
    int nq = t.nxt(q * t.C + c);
    if (nq == kDead) {
      if (q == kStart) return kClsRej;
      const Bits4 K = cands(t, q, wc);
      const int first = K.lowest();
      if (first < 0) return kClsRej;
      if (!t.ign.has(first)) {
        if (n == 0) first_ign = (K & t.ign).any();
        if (n < kMaxEv)
          rec[2 + n] = (uint16_t)class_id(t, 1, q, wc);
        else
          overflow = true;
        ++n;
      }
      q = kStart;
      lx = 0;
      pc = t.root_pc;
      wc = t.root_wc;
      nq = t.nxt(kStart * t.C + c);
      if (nq == kDead) return kClsRej;
    }
    q = nq;
    lx = lex_step(t, q, lx, b, pc, wc);
  }
  const Bits4 L = live_prime(t, q, pc);
  const bool lign = (L & t.ign).any();
  if (!L.any()) return kClsRej;
  if (n == 0) return lign ? kClsAcc : (uint16_t)class_id(t, 0, q, pc);
  if (n == 1 && lign) return first_ign ? kClsAcc : rec[2];
  if (overflow) {
    first_key = first_ign ? 0xFFFF : rec[2];
    return kClsCD;
  }
  rec[0] = (uint16_t)n;
  rec[1] = lign ? kClsAcc : (uint16_t)class_id(t, 0, q, pc);
  return kClsVC;
}

// An event record in registers: two 16-byte loads, issued together.
struct RecRegs {
  uint4 a, b;
  __device__ __forceinline__ int at(int i) const {
    const uint32_t w = i < 8 ? (i < 4 ? (i < 2 ? a.x : a.y) : (i < 6 ? a.z : a.w))
                             : (i < 12 ? (i < 10 ? b.x : b.y) : (i < 14 ? b.z : b.w));
    return (int)((w >> ((i & 1) * 16)) & 0xFFFFu);
  }
};

// Verdict of an event record at the walker's stack: each event is an emission
// with the recorded candidate set, then the final liveness test.  1 / 0 / -1.
template <class T>
__device__ __forceinline__ int eval_record(const T& t, Walker& w, const uint16_t* rec, int max_chain) {
  RecRegs r;
  r.a = __ldg(reinterpret_cast<const uint4*>(rec));
  r.b = __ldg(reinterpret_cast<const uint4*>(rec) + 1);
  const int n = r.at(0);
#pragma unroll 1
  for (int i = 0; i < n; ++i) {
    count_work(w.ctr, 3);
    const int e = emit_set(t, w, t.set4(r.at(2 + i)), max_chain);
    if (e <= 0) return e;
  }
  const int f = r.at(1);
  if (f == kClsAcc) return 1;
  return trailing_set(t, w, t.set4(f), max_chain);
}

}  // namespace grid
