// One-CTA ASRAL solver with price-guided searches (included by
// asral_solver.cu, which holds the shared prologue).
//
// Same rounds, same results as Solver<T> (Alg. 2 with Alg. 1 and Alg. 4 per
// round); what differs is how much of the Bellman-Ford of Alg. 3 is run.
//
// Prices.  Every center v keeps a price P(v), a lower bound on the cost of
// getting one unit out of v: over every path v -> ... -> u of Gamma, the
// transfer costs plus q_n(u), the penalty one more unit would pay at u (0
// with a vacancy).  The bounds are the feasible potentials of the successive
// shortest path method for min-cost flow (Edmonds and Karp 1972; Tomizawa
// 1971): for every table entry P(u) <= T[u][v] + P(v), and P(v) <= q_n(v).
// All prices start at 0 with an empty table.  When unit d joins center j:
//
//  * Only d's own edges can break the first inequality, so the merge of d's
//    row into T[j] also tests P(j) <= t_d(v) + P(v).  If it holds, no
//    negative cycle passes through j (Alg. 1 applies nothing); if also
//    P(j) >= q_j(last), the penalty j's last unit pays, no negative path
//    starts at j (Alg. 4 applies nothing), and the round ends there.
//  * Otherwise one synchronous Bellman-Ford from j answers both: a label
//    l(v) is expanded only while l(v) + P(v) is below the best value found so
//    far (P(j) + cycle cost for Alg. 1; min l(u) + q_n(u) for Alg. 4).
//    l(v) + P(v) bounds the value of any completion from v, and a completion
//    that only equals a value already found has more hops and is not the one
//    the full Bellman-Ford reports; so every node of the path it reports is
//    expanded, and the sink's label, hop counts and lowest-index parents come
//    out the same.  (Equality matters: with whole-number costs and tight
//    prices most labels are ties.)
//  * After a cycle was applied, Alg. 4 searches again; the bound uses the
//    prices raised by the first search's labels, max(P(v), P(j) + L - l1(v))
//    (L the cycle's cost), less `off`, the most by which those exceed q_n.
//    These bounds are not tested against the rows that the cycle has just
//    changed: the table is that of a minimum-cost flow again, for which the
//    raised prices hold.
//  * The round ends by raising prices: P(v) = max(P(v), D - l1(v), D2 -
//    l2(v)), D the shortest way from d to a paid slot (L + D2 after a
//    cycle, D2 from j).  For a row of T that did not change this keeps both
//    inequalities by l(v) <= l(u) + T[u][v]; the rows that did change are
//    tested entry by entry (broken_rows), and P(v) <= q_n(v) at the centers of
//    the applied paths.  Should one ever fail, the prices are rebuilt from the
//    table by reverse Bellman-Ford sweeps before the next round.
//  * Which of two equally good bounds a lane sees (the value found so far may
//    fall during a sweep) changes neither labels nor hop counts of the path,
//    but how many other labels are expanded: sweep and frontier counters and
//    prices may differ from run to run, results do not.
//
// What this buys (counted on instances of the city shape, 8,000 x 500, and of
// the batched mix, 6,007 x 126): 48 sweeps of 180 labels and 19 sweeps of 52
// per round become 10 sweeps of about 30 labels and 3 of about 16; half of the
// mix's rounds run no sweep at all.  Per call, against the cluster solver on
// the CTAs it did best on: 317 -> 43 to 46 ms for the mix instance, 1,230 -> 268
// to 277 ms for the city, 37 -> 10.5 to 11.5 ms for 2,000 x 20, 540 -> 36 to 38
// ms for 24 mixed instances in one launch (a cluster each before, a CTA each
// now); 1,000,000 x 500, whose largest center holds 112,000 units, 146 -> 56 s.
//
// Bound by the chain of dependent instructions and reads of a round: a warp
// that runs alone issues about one instruction in five cycles, a dependent
// global read takes about half a microsecond.  A round that ends at the tests
// takes about 1 us, a sweep 0.6 to 1.4 us, an applied path 4 to 10 us.
//
// Layout.  A frontier of a dozen labels is too little work to spread over a
// cluster: one CTA runs the whole round.  Thread t owns columns t, t + 512,
// ...; every thread reads the whole frontier list (broadcast loads) and keeps
// its own column's minimum, so a sweep needs one barrier of the ceil(k / 32)
// warps that own a column and no cross-warp reduction.  A label that improved
// is appended to the next list by its own lane's shared-memory atomic; the
// order inside a list does not matter, because only labels and hop counts are
// kept and `follow` looks up the lowest parent of each node of the one path
// that is applied.  The costs of T sit in shared memory as T (int16 or int32)
// when they fit beside the rest, otherwise they are read from the global
// table through L1; its units too, where both fit.
#pragma once

namespace lbdd {

// Bits of a node in a packed (hop, node) key (k <= 8191).
constexpr int kGNodeBits = 13;
constexpr int kGOrd = 64;                       // prefetched (unit, center) pairs
// Centers up to which the lists of affected entries are as long as
// guided_list says; beyond, one row's.  (The layout would hold eight rows' up to
// 1,356 centers with int16 and 1,296 with int32 costs, four up to 2,002 and
// 1,773, at the expense of the L1 that serves the mirror: not measured.)
constexpr int kGWideLists = 800;
// Affected entries that an apply lists at a time.  Where the cost table does
// not fit shared memory anyway there is room for those of eight rows, so that
// most paths go through each phase at once.
__host__ __device__ inline int32_t guided_list(int32_t k, int32_t elem) {
  return (int64_t)elem * k * k > 160 * 1024 ? 8 * k : k > 1024 ? k : 1024;
}

struct GLayout {
  uint32_t pot, lab1, lab2, hop, list, slack, pen, qn, seg, tailp, path, pathu, mid, raff, ppos, cpath, aff,
      ord, misc, ring, base_total, tsm, total, usm, full;
  int nring, aff_rows;
};

// Rows of CM in flight: 8 where they are short, 4 otherwise (they cover the
// DRAM latency of about four rounds that run no search).
__host__ __device__ inline int guided_ring(int32_t k, int32_t elem) {
  return (int64_t)k * elem <= 3072 ? 8 : 4;
}

// Row stride of the cost table in entries (an odd number of words with int16
// costs, so that the rows of one column spread over the banks).
__host__ __device__ inline int32_t guided_stride(int32_t k, int32_t elem) {
  return slice_stride((k + 1) & ~1, elem);
}

__host__ __device__ inline GLayout make_guided_layout(int32_t k, int32_t elem) {
  GLayout L;
  uint32_t o = 0;
  const uint32_t ku = (uint32_t)k, lt = elem == 2 ? 4u : 8u;
  auto take = [&](uint32_t bytes) { const uint32_t at = o; o = align16(o + bytes); return at; };
  L.pot = take(4u * ku);
  L.lab1 = take(lt * ku);
  L.lab2 = take(lt * ku);
  L.hop = take(2u * ku);
  const uint32_t aff = (uint32_t)(k > kGWideLists ? k : guided_list(k, elem));
  L.aff_rows = (int)(aff / ku) < 32 ? (int)(aff / ku) : 32;
  const uint32_t lists = 2u * 2u * lt * (ku + 2);
  L.list = take(lists > 8u * aff ? lists : 8u * aff);   // also the minima of a rescan
  L.slack = take(4u * ku);
  L.pen = take(4u * ku);
  L.qn = take(4u * ku);
  L.seg = take(4u * ku);
  L.tailp = take(4u * ku);
  L.path = take(4u * (ku + 2));
  L.pathu = take(4u * (ku + 2));
  L.mid = take(4u * (ku + 2));
  L.raff = take(4u * (ku + 2));
  L.ppos = take(4u * (ku + 2));
  L.cpath = take(4u * (ku + 2));
  L.aff = take(4u * aff);
  L.ord = take(8u * kGOrd);
  L.misc = take(128u);
  L.nring = guided_ring(k, elem);
  // the prologue's radix sort uses the ring and what follows (17 KB)
  const uint32_t row = align16((uint32_t)elem * ku);
  const uint32_t ringb = (uint32_t)L.nring * row;
  L.ring = take(ringb > 18432u ? ringb : 18432u);
  L.base_total = o;
  L.tsm = take((uint32_t)elem * ku * (uint32_t)guided_stride(k, elem));
  L.total = o;
  L.usm = take(4u * ku * ku);               // the units of T, where they fit too
  L.full = o;
  return L;
}

// Frontier entry: label and byte offset of the node's row of costs (top bit:
// a strict instance's center with a vacancy).
constexpr uint32_t kGVacant = 0x80000000u;
template <typename LT> struct GEnt;
template <> struct __align__(8) GEnt<int32_t> { int32_t l; uint32_t off; };
template <> struct __align__(16) GEnt<int64_t> { int64_t l; uint32_t off, pad; };

// Penalties and prices stay below this in a guided solve (the host checks the
// penalties), so that a label plus either fits 32 bits with int16 costs.
constexpr int32_t kGPenLimit = 1 << 30;
constexpr int32_t kGNever = kGPenLimit + (1 << 29);   // a price or slot out of every bound

// Rounds that scan long member lists for many entries.  One SM gathers them,
// where the full Bellman-Ford kernel shares them between the CTAs of a cluster
// and reads whole rows when most entries of one are affected.  A scan task (32
// lanes times 16 members) takes about 0.1 us on one CTA; past a number of tasks
// per round the other kernel is the faster one:
//  * `wide` tasks, of rows with more than half their entries affected.  Us per
//    round, guided / full: 20 centers, 660 tasks 73 / 54; 64, 1,270 tasks 129 /
//    70; 126, 7,900 tasks 837 / 182; 500, 31,700 tasks 3,375 / 187.
//  * all tasks, from kHeavyK centers on, where the cluster has 16 CTAs: 256,
//    2,500 tasks 315 / 310; 500, 990 tasks 172 / 177, 2,270 tasks 311 / 249;
//    1,000, 2,270 tasks 400 / 298; 1,800, 3,940 tasks 1,129 / 1,352, 4,480 tasks
//    1,897 / 1,639.  (126 centers, 2,040 tasks 242 / 328.)
// (One center takes half of 20,000 to 60,000 units.  Instances of the city shape
// have at most 360 tasks per round.)  What rounds scan beyond the limits adds
// up (a round below them takes the difference off again); past kHeavyRounds
// limits the rounds end and the host runs the next ones on the other kernel.
// Counted where a list took more than one task and looked at every kHeavyEvery
// rounds: in every apply and round it made the smallest solves 3 to 7 % slower.
constexpr int kHeavyK = 240;
constexpr int kHeavyRounds = 48, kHeavyEvery = 64;
__host__ __device__ inline int64_t heavy_wide(int32_t k) { return 500 + k / 2; }
__host__ __device__ inline int64_t heavy_scans(int32_t k) {
  return k < kHeavyK ? (int64_t)1 << 40 : k < 320 ? 2500 : 1500 + (k > 1200 ? 9 * (int64_t)(k - 1200) / 2 : 0);
}

struct GMisc {
  int32_t paid;       // best value of a path to a paid slot in the last search
  uint32_t sink;      // its hop count << kGNodeBits | node, if paid < ql
  uint32_t next[3];   // parents on the way back, by hop count modulo 3
  int32_t cnt[3];     // list lengths, by sweep modulo 3
  int32_t len, bad, stop, heavy;
  int32_t scans, wide;   // scan tasks since they were looked at: the other rows', the wide ones'
};

template <typename T, bool TSM, bool STRICT>
struct Guided {
  using LT = typename Solver<T>::LT;
  using Ent = GEnt<LT>;
  // Sums of a label, a price and a penalty: 32 bits with int16 costs (labels
  // stay below 2^28, the others below 2^30).
  using PT = LT;
  static constexpr int VPL = 16 / (int)sizeof(T);
  static constexpr int32_t kInf = Solver<T>::kTsInf;
  static constexpr LT kNoLab = Solver<T>::kNoLab;

  const DevInst& I;
  const T* cm;
  int64_t ld;
  int32_t *tc, *td, *pool, *page_tab, *pos;
  int32_t max_pages;
  int32_t n, k, ws;
  int tid, flags;
  int32_t *s_pot, *s_slack, *s_pen, *s_seg, *s_tail, *s_path, *s_pathu, *s_raff, *s_ppos, *s_cpath,
      *s_aff, *s_ord;
  int32_t* s_qn;      // q_n of every center: what one more unit would pay there
  int32_t* s_mid;     // prices of a second search
  LT *s_lab1, *s_lab2;
  uint16_t* s_hop;    // sweep of every label's last change in the last search
  Ent* s_list;        // [2][k + 2]
  GMisc* M;
  unsigned char* s_ring;
  uint32_t ring_row;
  int nring, aff_rows;
  int32_t* s_td;      // [k][k] units of T in shared memory, or null: global only
  T* tt;              // [k][ws] costs of T: shared memory, or the global mirror
  Book* B;

  __device__ Guided(const DevInst& inst, unsigned char* base, const GLayout& L, bool usm, Book* book,
                    int fl)
      : I(inst) {
    cm = static_cast<const T*>(inst.cm);
    ld = inst.ld;
    tc = inst.tc;
    td = inst.td;
    pool = inst.pool;
    page_tab = inst.page_tab;
    pos = inst.pos;
    max_pages = inst.max_pages;
    n = inst.n;
    k = inst.k;
    ws = guided_stride(k, (int32_t)sizeof(T));
    tid = threadIdx.x;
    flags = fl;
    auto i32 = [&](uint32_t at) { return reinterpret_cast<int32_t*>(base + at); };
    s_pot = i32(L.pot);
    s_lab1 = reinterpret_cast<LT*>(base + L.lab1);
    s_lab2 = reinterpret_cast<LT*>(base + L.lab2);
    s_hop = reinterpret_cast<uint16_t*>(base + L.hop);
    s_list = reinterpret_cast<Ent*>(base + L.list);
    s_slack = i32(L.slack);
    s_pen = i32(L.pen);
    s_seg = i32(L.seg);
    s_tail = i32(L.tailp);
    s_path = i32(L.path);
    s_pathu = i32(L.pathu);
    s_mid = i32(L.mid);
    s_qn = i32(L.qn);
    s_raff = i32(L.raff);
    s_ppos = i32(L.ppos);
    s_cpath = i32(L.cpath);
    s_aff = i32(L.aff);
    s_ord = i32(L.ord);
    M = reinterpret_cast<GMisc*>(base + L.misc);
    s_ring = base + L.ring;
    ring_row = align16((uint32_t)sizeof(T) * (uint32_t)k);
    nring = L.nring;
    aff_rows = L.aff_rows;
    tt = TSM ? reinterpret_cast<T*>(base + L.tsm) : static_cast<T*>(inst.mirror);
    s_td = usm ? i32(L.usm) : nullptr;
    B = book;
  }

  __device__ __forceinline__ bool timer() const { return (flags & OPT_PHASE_TIMERS) && tid == 0; }
  __device__ __forceinline__ const T* row(int32_t d) const { return cm + (int64_t)d * ld; }
  __device__ __forceinline__ int32_t edge(int32_t u, int cl) const {
    return (int32_t)tt[(int64_t)u * ws + cl];
  }
  // Cost of the edge u -> column cl in the graph of Alg. 1; in a strict
  // instance a center with a vacancy passes a dummy unit on for nothing
  // (Alg. 5), members or not.
  __device__ __forceinline__ bool vacant(int32_t u) const { return STRICT && s_slack[u] < 0; }
  __device__ __forceinline__ int32_t arc(int32_t u, int cl) const {
    const int32_t t = edge(u, cl);
    return vacant(u) ? min(t, 0) : t;
  }
  // Best unit of entry (u, cl).  In global memory equal costs lower it by
  // reductions at L2, so it is read past L1.
  __device__ __forceinline__ int32_t unit(int32_t u, int cl) const {
    return s_td ? s_td[u * k + cl] : __ldcg(td + (int64_t)u * k + cl);
  }
  // What sits in shared memory is written back when the launch ends.
  __device__ __forceinline__ void set_entry(int32_t u, int cl, int32_t t, int32_t d) {
    if (!TSM) tc[(int64_t)u * k + cl] = t;
    if (s_td) s_td[u * k + cl] = d;
    else td[(int64_t)u * k + cl] = d;
    tt[(int64_t)u * ws + cl] = (T)(t == kTInf ? kInf : t);
  }
  // q_c(x), x >= 1: penalty of the x-th allotment beyond capacity (Def. 4).
  __device__ __forceinline__ int32_t qval(int32_t c, int32_t x) const {
    return __ldg(I.pen + (int64_t)c * I.Q + min(max(x, 1), I.Q) - 1);
  }
  // One unit more (+1) or less (-1) at c.
  __device__ __forceinline__ void shift_load(int32_t c, int32_t by) {
    const int32_t x = s_slack[c] + by;
    s_slack[c] = x;
    if (I.Q > 1) s_pen[c] = qval(c, x + 1);
    s_qn[c] = x >= 0 ? s_pen[c] : 0;
  }

  // ------------------------------------------------------- member lists --
  // Page of entry idx of c's list; the last page's id is kept in shared memory.
  __device__ __forceinline__ int32_t page_of(int32_t c, int32_t idx, int32_t len) const {
    const int32_t p = idx >> kPageShift;
    return p == (len - 1) >> kPageShift ? s_tail[c] : page_tab[(int64_t)c * max_pages + p];
  }
  __device__ __forceinline__ int32_t* mslot(int32_t c, int32_t idx, int32_t len) const {
    return pool + (int64_t)page_of(c, idx, len) * kPageWords + (idx & (kPage - 1));
  }
  // One thread at a time calls these two.  `own` is CM(d, c).
  __device__ void list_append(int32_t c, int32_t d, int32_t own) {
    const int32_t idx = s_seg[c];
    if (idx < 0 || idx >= n) { B->err0 = ST_ERR_INVARIANT; return; }
    if ((idx & (kPage - 1)) == 0) {
      if (B->free_top <= 0) { B->err0 = ST_ERR_INVARIANT; return; }
      const int32_t page = I.free_stack[--B->free_top];
      page_tab[(int64_t)c * max_pages + (idx >> kPageShift)] = page;
      s_tail[c] = page;
    }
    int32_t* slot = pool + (int64_t)s_tail[c] * kPageWords + (idx & (kPage - 1));
    slot[0] = d;
    slot[kPage] = own;
    pos[d] = idx;
    s_seg[c] = idx + 1;
  }
  // last_id, last_own: the list's last member, which takes the place.
  __device__ void list_remove_at(int32_t c, int32_t idx, int32_t last_id, int32_t last_own) {
    const int32_t len = s_seg[c], last = len - 1;
    if (idx < 0 || idx > last || B->free_top >= I.npages || (uint32_t)last_id >= (uint32_t)n) {
      B->err0 = ST_ERR_INVARIANT;
      return;
    }
    if (idx != last) {
      int32_t* to = mslot(c, idx, len);
      to[0] = last_id;
      to[kPage] = last_own;
      pos[last_id] = idx;
    }
    if ((last & (kPage - 1)) == 0) {
      I.free_stack[B->free_top++] = s_tail[c];
      if (last > 0) s_tail[c] = page_tab[(int64_t)c * max_pages + ((last - 1) >> kPageShift)];
    }
    s_seg[c] = last;
  }

  // ------------------------------------------------------------- search --
  __device__ __forceinline__ void group_sync(int nthr) const {
    if (nthr == 32) __syncwarp();
    else asm volatile("bar.sync 1, %0;" ::"r"(nthr) : "memory");
  }
  static __device__ __forceinline__ int32_t clamp32(int64_t x) {
    return (int32_t)max((int64_t)INT32_MIN, min((int64_t)INT32_MAX, x));
  }
  static __device__ __forceinline__ LT relax(LT l, int32_t t, LT b) {
    if constexpr (sizeof(LT) == 4) return __viaddmin_s32(l, t, b);
    else return min(b, l + (LT)t);
  }
  // The cost at byte offset `at` of the table, in shared memory or in the mirror.
  __device__ __forceinline__ int32_t cost_at(uint32_t at) const {
    int32_t t;
    if constexpr (TSM) {
      if constexpr (sizeof(T) == 2)
        asm volatile("ld.shared.s16 %0, [%1];" : "=r"(t) : "r"(at) : "memory");
      else
        asm volatile("ld.shared.s32 %0, [%1];" : "=r"(t) : "r"(at) : "memory");
    } else {
      t = (int32_t)*reinterpret_cast<const T*>(reinterpret_cast<const unsigned char*>(tt) + at);
    }
    return t;
  }
  static __device__ __forceinline__ Ent entry(uint32_t at) {
    Ent e;
    if constexpr (sizeof(LT) == 4) {
      asm volatile("ld.shared.v2.b32 {%0, %1}, [%2];" : "=r"(e.l), "=r"(e.off) : "r"(at) : "memory");
    } else {
      uint32_t lo, hi;
      asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];"
                   : "=r"(lo), "=r"(hi), "=r"(e.off), "=r"(e.pad) : "r"(at) : "memory");
      e.l = (int64_t)(((uint64_t)hi << 32) | lo);
    }
    return e;
  }
  // Pruned synchronous Bellman-Ford from j into `lab` and s_hop.  cyc: look
  // for a cycle through j (lab[j] holds its value); np: for a path to a paid
  // slot cheaper than ql (M->paid its value, M->sink its last node).  `price`
  // holds the bounds.  Every thread calls it.
  //
  // A sweep is a dependent chain of a few warps, so its cost is the number of
  // instructions on that chain (about five cycles each for a lone warp), not
  // its bytes.  It keeps only the least label per column: which predecessor
  // gave it is looked up for the few nodes of the path that is applied
  // (follow), by label and hop count; an edge costs one load and one
  // add-and-minimum.  A lane owns one column, in registers up to 512 centers.
  // The infinite entry of a frontier node's row (its own column) never beats
  // the node's own label; nodes without members are never on the list.
  __device__ void search(int32_t j, bool cyc, bool np, LT* lab, const int32_t* price, int32_t ql) {
    constexpr LT kFixed = std::numeric_limits<LT>::min();   // a label nothing improves
    const int32_t pj = s_pot[j];
    const uint32_t tbase = TSM ? smem_u32(tt) : 0u;
    const uint32_t rowb = (uint32_t)ws * (uint32_t)sizeof(T);
    const uint32_t lbase = smem_u32(s_list), lsize = (uint32_t)(k + 2) * (uint32_t)sizeof(Ent);
    for (int cl = tid; cl < k; cl += kThreads) lab[cl] = cyc || cl != j ? kNoLab : kFixed;
    if (tid == 0) {
      M->paid = INT32_MAX;
      M->sink = ~0u;
      M->next[0] = M->next[1] = M->next[2] = ~0u;
      M->cnt[1] = 0;
      Ent e;
      e.l = 0;
      e.off = (tbase + (uint32_t)j * rowb) | (vacant(j) ? kGVacant : 0u);
      s_list[0] = e;
    }
    __syncthreads();
    const int nthr = min(kThreads, (k + 31) & ~31);
    if (tid < nthr) {
      // frontier nodes in flight: shared memory or L2 latency
      constexpr int U = TSM ? 8 : 16;
      const int lane = tid & 31;
      const bool single = k <= nthr;
      int sweep = 1, m = 1, par = 0, c3 = 1;   // par: list read; c3: counter of the next list
      LT b = kFixed;
      int32_t qv = kGNever, pv = kGNever;
      for (;; ++sweep) {
        const uint32_t in = lbase + (uint32_t)par * lsize;
        Ent* out = s_list + (par ^ 1) * (k + 2);
        const int c3n = c3 == 2 ? 0 : c3 + 1;
        if (tid == 0) {
          M->cnt[c3n] = 0;
          if (timer()) front_stat(m);
        }
        const LT bc = cyc ? (LT)pj + min((LT)-1, lab[j] - 1) : kFixed;
        const int32_t paid = M->paid;
        const int32_t bp = np ? min(ql, paid) - 1 : INT32_MIN;
        unsigned bits = 0;
        for (int cl = tid, c0 = 0; c0 < k; c0 += nthr, cl += nthr) {
          if (!single || sweep == 1) {
            const bool real = cl < k && cl != j;
            b = cl < k ? lab[cl] : kFixed;
            qv = real ? s_qn[cl] : kGNever;
            // a center without members has no edges (its row is infinite)
            pv = real && (s_seg[cl] > 0 || vacant(cl)) ? price[cl] : kGNever;
          }
          const LT old = b;
          const uint32_t colb = (uint32_t)min(cl, k - 1) * (uint32_t)sizeof(T);
          LT b2 = b;
          // N nodes from `at`; the last batch repeats the last node
          auto batch = [&](auto size, uint32_t at, uint32_t last) {
            constexpr int N = decltype(size)::value;
            Ent e[N];
            int32_t t[N];
#pragma unroll
            for (int q = 0; q < N; ++q) e[q] = entry(min(at + q * (uint32_t)sizeof(Ent), last));
#pragma unroll
            for (int q = 0; q < N; ++q) {
              t[q] = cost_at((STRICT ? e[q].off & ~kGVacant : e[q].off) + colb);
              if (STRICT && (e[q].off & kGVacant)) t[q] = min(t[q], 0);
            }
#pragma unroll
            for (int q = 0; q < N; q += 2) {
              b = relax(e[q].l, t[q], b);
              b2 = relax(e[q + 1].l, t[q + 1], b2);
            }
          };
          const uint32_t last = in + (uint32_t)(m - 1) * (uint32_t)sizeof(Ent);
          uint32_t at = in;
          int left = m;
          for (; left > U / 2; left -= U, at += U * (uint32_t)sizeof(Ent))
            batch(std::integral_constant<int, U>(), at, last);
          if (left > 0) batch(std::integral_constant<int, U / 2>(), at, last);
          b = min(b, b2);
          const bool up = b < old;
          if (up) {
            lab[cl] = b;
            s_hop[cl] = (uint16_t)sweep;
          }
          int32_t now = bp;
          if (np) {
            const int32_t vm = __reduce_min_sync(0xffffffffu, up ? clamp_sum(b, qv) : INT32_MAX);
            if (vm < paid && lane == 0) atomicMin(&M->paid, vm);
            now = min(bp, vm - 1);
          }
          // (unsigned: a label that is not reached wraps, and is not used)
          const LT key = (LT)((std::make_unsigned_t<LT>)b + (std::make_unsigned_t<LT>)(LT)pv);
          const bool push = up && (key <= (LT)now || key <= bc);
          if (nthr == 32) bits = __ballot_sync(0xffffffffu, push);
          if (push) {
            const int at = nthr == 32 ? __popc(bits & ((1u << lane) - 1u)) : atomicAdd(&M->cnt[c3], 1);
            Ent ne;
            ne.l = b;
            ne.off = (tbase + (uint32_t)cl * rowb) | (vacant(cl) ? kGVacant : 0u);
            out[at] = ne;
          }
        }
        group_sync(nthr);
        m = nthr == 32 ? __popc(bits) : M->cnt[c3];
        c3 = c3n;
        par ^= 1;
        if (m == 0) break;
        if (sweep > k + 1) {   // labels settle within k + 1 sweeps
          if (tid == 0) M->bad = 1;
          break;
        }
      }
      if (np && M->paid < ql) {   // fewest hops, then lowest node, among the best slots
        const int32_t best = M->paid;
        uint32_t hu = ~0u;
        for (int cl = tid; cl < k; cl += nthr)
          if (cl != j && lab[cl] != kNoLab && (int64_t)lab[cl] + s_qn[cl] == best)
            hu = min(hu, ((uint32_t)s_hop[cl] << kGNodeBits) | (uint32_t)cl);
        hu = __reduce_min_sync(0xffffffffu, hu);
        if (lane == 0 && hu != ~0u) atomicMin(&M->sink, hu);
      }
      if (tid == 0) {
        B->bf_calls++;
        B->bf_sweeps += sweep;
        B->bf_max = max(B->bf_max, (int64_t)sweep);
      }
    }
    __syncthreads();
  }
  static __device__ __forceinline__ int32_t clamp_sum(LT a, int32_t b) {
    if constexpr (sizeof(LT) == 4) return a + b;
    else return clamp32(a + b);
  }

  __device__ __forceinline__ void front_stat(int m) {
    B->front_sum += m;
    B->front_hist[m <= 1 ? 0 : m <= 4 ? 1 : m <= 16 ? 2 : m <= 64 ? 3 : m <= 256 ? 4 : 5]++;
  }

  // -------------------------------------------------------------- apply --
  // The canonical shortest path that ends at node `last` (the cycle through
  // j if last < 0), backwards into s_pathu: the parent of a node v with label
  // l and hop count h is the lowest-index u with l(u) + T[u][v] = l and
  // hop(u) = h - 1.  One warp up to kFollowWarp centers (two strided passes and
  // no barrier), else thread = node and a barrier per hop (one warp up to 192
  // centers measured slower at 126).  Returns its length, -1 if there is
  // none (the one-warp form: to warp 0 only).
  static constexpr int kFollowWarp = 64;
  __device__ __forceinline__ bool precedes(int u, int32_t v, int h, LT l, int32_t j,
                                           const LT* lab) const {
    return s_hop[u] == h - 1 && u != j && u != v && lab[u] != kNoLab && lab[u] + (LT)arc(u, v) == l;
  }
  __device__ int follow(int32_t j, int32_t last, const LT* lab) {
    const bool alone = k <= kFollowWarp;
    int32_t v = last < 0 ? j : last;
    int h = s_hop[v], m = 0, slot = 0;
    LT l = lab[v];
    if (last >= 0) {
      if (tid == 0) s_pathu[0] = v;
      m = 1;
    }
    for (; h > 1; --h) {
      uint32_t best = ~0u;
      for (int u = tid; u < k; u += alone ? 32 : kThreads)
        if (precedes(u, v, h, l, j, lab)) { best = (uint32_t)u; break; }
      if (alone) {
        best = __reduce_min_sync(0xffffffffu, best);
      } else {
        if (best != ~0u) atomicMin(&M->next[slot], best);
        __syncthreads();
        best = M->next[slot];
        slot = slot == 2 ? 0 : slot + 1;
        // the slot after the next one: read before the last barrier
        if (tid == 0) M->next[slot == 2 ? 0 : slot + 1] = ~0u;
      }
      if (best == ~0u) return -1;
      v = (int32_t)best;
      l = lab[v];
      if (tid == 0) s_pathu[m] = v;
      ++m;
    }
    if (l != (LT)arc(j, v)) return -1;
    if (tid == 0) s_pathu[m] = j;
    return m + 1 < 2 ? -1 : m + 1;
  }

  __device__ __forceinline__ int32_t arriving(bool npath, int m, int i) const {
    return i > 0 ? s_pathu[i - 1] : (npath ? -1 : s_pathu[m - 1]);
  }

  // Applies the transfers of the path that follow() finds (Alg. 1 and Alg. 4,
  // "if cost < 0" branch): every center on it hands its best unit for the
  // next center on; for a cycle the last one hands to j, for a path the last
  // center only gains and j only loses a unit.  Then the rows of T of those
  // centers: an entry whose best unit was not the leaving one keeps its
  // minimum over the remaining members and takes the arriving unit in; the
  // others ("affected") are recomputed over the member list.
  //
  // What an apply costs is its chain of global latencies, so everything that
  // can be in flight together is: after the affected entries are listed
  // (shared memory only, where the units fit), the warps share the arriving
  // units' rows and the members of the affected entries, while warp 0 loads
  // what it needs to move the units.  Member lists change only afterwards:
  // the scan of a list skips the leaving unit and adds the arriving one.
  // Returns the length of the path (s_path), -1 if there is none.
  __device__ int apply(int32_t j, bool npath, int32_t last, const LT* lab, int64_t cost) {
    const uint64_t t0 = timer() ? clock_cycles() : 0;
    const int lane = tid & 31, warp = tid >> 5;
    int m = 0;
    if (k > kFollowWarp || warp == 0) m = follow(j, last, lab);
    if (tid < 32) {
      __syncwarp();
      if (lane == 0) M->len = m;
      for (int i = lane; i < m; i += 32) s_path[i] = s_pathu[m - 1 - i];
      __syncwarp();
      for (int i = lane; i < m; i += 32) {
        const int32_t to = (i + 1 < m) ? s_path[i + 1] : (npath ? -1 : j);
        // a dummy unit moves where the edge's cost came from a vacancy
        const bool dummy = STRICT && vacant(s_path[i]) && edge(s_path[i], to) > 0;
        int32_t x = to >= 0 && !dummy ? unit(s_path[i], to) : -1;
        if (to >= 0 && !dummy && (uint32_t)x >= (uint32_t)n) { x = -1; B->err0 = ST_ERR_INVARIANT; }
        s_pathu[i] = x;
        s_raff[i] = 0;
      }
    }
    __syncthreads();
    m = M->len;
    if (m < 0) return m;
    // what moving the units takes, in flight while the rows are updated.
    // Warp 0, lane = center of the path: position of its leaving unit,
    // CM(arriving unit, center).  Paths: warp 1 takes j's unit out (position,
    // and j's last member, which takes its place), warp 2 puts the last
    // arriving unit in; where a page of the pool is freed or taken, warp 1
    // does both.
    int32_t at = -1, own = 0, last_id = 0, last_own = 0;
    bool pages = false;
    if (warp == 0) {
      if (lane < m) {
        const int32_t x_out = s_pathu[lane], x_in = arriving(npath, m, lane);
        if (x_out >= 0) at = pos[x_out];
        if (x_in >= 0) own = (int32_t)row(x_in)[s_path[lane]];
      }
      for (int i = lane + 32; i < m; i += 32) s_ppos[i] = s_pathu[i] >= 0 ? pos[s_pathu[i]] : -1;
    } else if (npath && warp <= 2) {
      const int32_t term = s_path[m - 1], x_in = s_pathu[m - 2];
      pages = ((s_seg[j] - 1) & (kPage - 1)) == 0 || (s_seg[term] & (kPage - 1)) == 0;
      if (x_in >= 0) own = (int32_t)row(x_in)[term];
      if (warp == 1) {
        at = s_pathu[0] >= 0 ? pos[s_pathu[0]] : -1;
        const int32_t* sl = mslot(j, s_seg[j] - 1, s_seg[j]);
        last_id = sl[0];
        last_own = sl[kPage];
      }
    }
    const int chunk = aff_rows;   // rows whose affected entries fit s_aff
    const int nblk = (k + 31) >> 5;
    for (int i0 = 0; i0 < m; i0 += chunk) {
      const int i1 = min(m, i0 + chunk), units = (i1 - i0) * nblk;
      list_affected(i0, units, nblk);
      __syncthreads();
      const uint64_t t1 = timer() ? clock_cycles() : 0;
      if (timer() && i0 == 0) B->t_apply += t1 - t0;
      // lane = row: entries, list length, log2 of the entries per warp, tasks
      const int i = i0 + lane;
      const int na = i < i1 ? s_raff[i] : 0;
      const int len = na > 0 ? s_seg[s_path[i]] : 0;
      // (at least two entries' lanes: a part then stays within a page)
      const int le = na > 16 ? 5 : na > 8 ? 4 : na > 4 ? 3 : na > 2 ? 2 : 1;
      static_assert((kScanU << 4) <= kPage, "a part of a member list lies in one page");
      const int parts = na > 0 ? max(1, (len + (kScanU << (5 - le)) - 1) / (kScanU << (5 - le))) : 0;
      const bool split = __any_sync(0xffffffffu, parts > 1);
      if (warp == 0) {
        const int rows = __reduce_add_sync(0xffffffffu, len);
        if (lane == 0) B->col_rows += rows;
      }
      {
        int incl = ((na + 31) >> 5) * parts;
        const int mine = incl;
        if (__any_sync(0xffffffffu, na > 0)) {
#pragma unroll
          for (int off = 1; off < 32; off <<= 1) {
            const int o = __shfl_up_sync(0xffffffffu, incl, off);
            if (lane >= off) incl += o;
          }
        }
        const int tasks = __shfl_sync(0xffffffffu, incl, 31);
        // scan tasks first, then batches of kMergeU blocks of 32 columns
        const int items = tasks + (units + kMergeU - 1) / kMergeU;
        for (int t = warp; t < items; t += kWarps) {
          if (t < tasks) {
            const int r = __popc(__ballot_sync(0xffffffffu, incl <= t));
            const int na_r = __shfl_sync(0xffffffffu, na, r), len_r = __shfl_sync(0xffffffffu, len, r);
            const int le_r = __shfl_sync(0xffffffffu, le, r);
            const int parts_r = __shfl_sync(0xffffffffu, parts, r);
            const int t0r = t - __shfl_sync(0xffffffffu, incl - mine, r);
            const int blk = t0r / parts_r;
            scan_task(npath, m, i0, r, na_r, len_r, le_r, parts_r, blk, t0r - blk * parts_r);
          } else {
            merge_task(npath, m, i0, units, nblk, (t - tasks) * kMergeU);
          }
        }
      }
      __syncthreads();
      if (split) {
        for (int r = warp; r < i1 - i0; r += kWarps) {
          const int na_r = __shfl_sync(0xffffffffu, na, r);
          const int parts_r = __shfl_sync(0xffffffffu, parts, r);
          if (parts_r > 1) {
            for (int e = lane; e < na_r; e += 32)
              put_entry(s_path[i0 + r], s_aff[r * k + e], best_of(r * k + e));
            // (see heavy_scans)
            if (lane == 0) atomicAdd(2 * na_r > k ? &M->wide : &M->scans, ((na_r + 31) >> 5) * parts_r);
          }
        }
      }
      if (split || i1 < m) __syncthreads();
      if (timer()) B->t_rescan += clock_cycles() - t1;
    }
    move_units(j, npath, m, cost, at, own, last_id, last_own, pages);
    return m;
  }

  static constexpr int kScanU = 16;   // members in flight per lane
  static constexpr int kMergeU = 4;   // column blocks in flight per warp

  // The affected entries of rows i0...: s_aff[row][...] columns, their number
  // in s_raff, their running minima reset.
  __device__ void list_affected(int i0, int units, int nblk) {
    if (s_td) list_affected_by<1>(i0, units, nblk);
    else list_affected_by<kMergeU>(i0, units, nblk);
  }
  // U blocks of 32 entries in flight per warp (the units' latency).
  template <int U>
  __device__ __forceinline__ void list_affected_by(int i0, int units, int nblk) {
    const int lane = tid & 31;
    const int dr = kWarps / nblk, db = kWarps - dr * nblk;
    int w = tid >> 5;
    int r = w / nblk, blk = w - r * nblk;
#pragma unroll 1
    while (w < units) {
      int32_t bd[U], rr[U], vv[U];
#pragma unroll
      for (int q = 0; q < U; ++q) {
        rr[q] = w < units ? r : -1;
        vv[q] = blk * 32 + lane;
        bd[q] = -1;
        if (rr[q] >= 0 && vv[q] < k && s_pathu[i0 + r] >= 0)
          bd[q] = U == 1 ? s_td[s_path[i0 + r] * k + vv[q]]
                         : __ldcg(td + (int64_t)s_path[i0 + r] * k + vv[q]);
        w += kWarps;
        r += dr;
        blk += db;
        if (blk >= nblk) { blk -= nblk; ++r; }
      }
#pragma unroll
      for (int q = 0; q < U; ++q) {
        if (rr[q] < 0) break;
        const int i = i0 + rr[q];
        const bool hit = bd[q] >= 0 && bd[q] == s_pathu[i] && vv[q] != s_path[i];
        if (hit) {
          const int at = rr[q] * k + atomicAdd(&s_raff[i], 1);
          s_aff[at] = vv[q];
          best_of(at) = ~0ull;
        }
      }
    }
  }
  // 64-bit running minimum of a listed entry (the frontier lists' space).
  __device__ __forceinline__ unsigned long long& best_of(int e) const {
    return reinterpret_cast<unsigned long long*>(s_list)[e];
  }
  static __device__ __forceinline__ unsigned long long entry_key(int32_t t, int32_t d) {
    return ((unsigned long long)((uint32_t)t ^ 0x80000000u) << 32) | (uint32_t)d;
  }
  __device__ __forceinline__ void put_entry(int32_t c, int32_t v, unsigned long long best) {
    if (best == ~0ull) set_entry(c, v, kTInf, -1);
    else set_entry(c, v, (int32_t)((uint32_t)(best >> 32) ^ 0x80000000u), (int32_t)(uint32_t)best);
  }

  // A block of at most 32 affected entries of row i0 + r over one part of its
  // center's member list: lane = (entry, member of sixteen in flight), with as
  // many lanes per entry as the block leaves, so that few entries of a long
  // list (a large center) still fill the warps and many entries of a short
  // one read neighbouring columns of the same rows.  Lists of more than one
  // part meet in the entry's running minimum.
  __device__ void scan_task(bool npath, int m, int i0, int r, int na, int len, int le, int parts,
                            int blk, int part) {
    constexpr int U = kScanU;
    const int lane = tid & 31;
    const int e = (blk << 5) + (lane & ((1 << le) - 1)), sub = lane >> le;
    const int step = 32 >> le;
    const int32_t c = s_path[i0 + r], x_out = s_pathu[i0 + r];
    const int32_t v = e < na ? s_aff[r * k + e] : 0;
    const int32_t base = part * U * step + sub;
    unsigned long long best = ~0ull;
    if (e < na && part == 0 && sub == 0) {
      const int32_t x_in = arriving(npath, m, i0 + r);
      if (x_in >= 0) best = entry_key((int32_t)row(x_in)[v] - (int32_t)row(x_in)[c], x_in);
    }
    if (e < na && base < len) {
      // a part is a power of two of at most a page's entries: one page
      const int32_t* sl = mslot(c, base, len);
      const int left = (len - base + step - 1) >> (5 - le);
      const T* cv = cm + v;
      int32_t id[U], ow[U], x[U];
#pragma unroll
      for (int q = 0; q < U; ++q) {
        const int32_t at = (q < left ? q : 0) << (5 - le);   // past the end: the first again
        id[q] = sl[at];
        ow[q] = sl[at + kPage];
      }
#pragma unroll
      for (int q = 0; q < U; ++q) {
        if ((uint32_t)id[q] >= (uint32_t)n) id[q] = x_out;   // guard: corrupt entry
        x[q] = (int32_t)cv[(int64_t)id[q] * ld];
      }
#pragma unroll
      for (int q = 0; q < U; ++q)
        if (id[q] != x_out) best = min(best, entry_key(x[q] - ow[q], id[q]));
    }
    for (int s = 1 << le; s < 32; s <<= 1)
      best = min(best, (unsigned long long)__shfl_xor_sync(0xffffffffu, best, s));
    if (e < na && sub == 0) {
      if (parts > 1) atomicMin(&best_of(r * k + e), best);
      else put_entry(c, v, best);
    }
  }

  // The arriving units into the entries that are not affected: kMergeU blocks
  // of 32 columns from block w of rows i0....
  __device__ void merge_task(bool npath, int m, int i0, int units, int nblk, int w) {
    const int lane = tid & 31;
    int r = w / nblk, blk = w - r * nblk;
    int32_t ct[kMergeU], ow[kMergeU], bd[kMergeU], rr[kMergeU], vv[kMergeU];
#pragma unroll
    for (int q = 0; q < kMergeU; ++q) {
      rr[q] = -1;
      vv[q] = blk * 32 + lane;
      ct[q] = ow[q] = bd[q] = 0;
      if (w + q < units && vv[q] < k) {
        const int i = i0 + r;
        const int32_t c = s_path[i], x_in = arriving(npath, m, i);
        if (x_in >= 0 && vv[q] != c) {
          rr[q] = r;
          const T* rx = row(x_in);
          ct[q] = (int32_t)rx[vv[q]];
          ow[q] = (int32_t)rx[c];
          bd[q] = unit(c, vv[q]);
        }
      }
      if (++blk == nblk) { blk = 0; ++r; }
    }
#pragma unroll
    for (int q = 0; q < kMergeU; ++q) {
      if (rr[q] < 0) continue;
      const int i = i0 + rr[q];
      const int32_t c = s_path[i], x_out = s_pathu[i];
      if (x_out >= 0 && bd[q] == x_out) continue;   // affected
      const int32_t x_in = arriving(npath, m, i);
      const int32_t t = ct[q] - ow[q];
      const int32_t e = edge(c, vv[q]);
      const int32_t bt = e == kInf ? kTInf : e;
      if (lex_less(t, x_in, bt, bd[q])) set_entry(c, vv[q], t, x_in);
    }
  }

  // Member lists, allotment, loads and objective, by a few warps at once (see
  // apply for who holds what); the others may already prepare the next search.
  __device__ void move_units(int32_t j, bool npath, int m, int64_t cost, int32_t at, int32_t own,
                             int32_t last_id, int32_t last_own, bool pages) {
    const int lane = tid & 31, warp = tid >> 5;
    if (warp == 0) {
      for (int b = 0; b < m; b += 32) {
        const int i = b + lane;
        int32_t c = 0, x_out = -1, x_in = -1;
        if (i < m) {
          c = s_path[i];
          x_out = s_pathu[i];
          x_in = arriving(npath, m, i);
          if (b > 0) {   // (warps 1 and 2 may have written the positions meanwhile)
            at = s_ppos[i];
            own = x_in >= 0 ? (int32_t)row(x_in)[c] : 0;
          }
          if (x_out >= 0) I.assign[x_out] = (i + 1 < m) ? s_path[i + 1] : j;
          s_ppos[i] = at;
        }
        if (x_out >= 0 && x_in >= 0) {
          if (at >= 0 && at < s_seg[c]) {
            int32_t* slot = mslot(c, at, s_seg[c]);
            slot[0] = x_in;
            slot[kPage] = own;
          } else {
            s_ppos[i] = -1;
            B->err0 = ST_ERR_INVARIANT;
          }
        }
      }
      __syncwarp();
      for (int i = lane; i < m; i += 32) {   // positions, once all old ones were read
        const int32_t x_in = arriving(npath, m, i);
        if (s_pathu[i] >= 0 && x_in >= 0 && s_ppos[i] >= 0) pos[x_in] = s_ppos[i];
      }
      __syncwarp();
      if (STRICT && lane == 0) {
        // centers that only lose or only gain a real unit: a dummy is on the
        // other side of their pair of edges
        for (int i = 0; i < m; ++i) {
          const int32_t c = s_path[i], x_out = s_pathu[i], x_in = arriving(npath, m, i);
          if (x_out >= 0 && x_in < 0) {
            const int32_t* sl = mslot(c, s_seg[c] - 1, s_seg[c]);
            list_remove_at(c, s_ppos[i], sl[0], sl[kPage]);
            shift_load(c, -1);
          } else if (x_out < 0 && x_in >= 0) {
            list_append(c, x_in, (int32_t)row(x_in)[c]);
            shift_load(c, 1);
          }
        }
      }
    } else if (npath && warp <= 2 && lane == 0) {
      if (warp == 1) {
        list_remove_at(j, at, last_id, last_own);
        shift_load(j, -1);
      }
      if (warp == (pages ? 1 : 2)) {
        const int32_t term = s_path[m - 1];
        if (s_pathu[m - 2] >= 0) list_append(term, s_pathu[m - 2], own);
        else B->err0 = ST_ERR_INVARIANT;
        shift_load(term, 1);
      }
    } else if (warp == 3 && lane == 0) {
      if (npath) B->paths++;
      else B->cycles++;
      B->moves += npath ? m - 1 : m;
      B->delta += cost;
    }
  }

  // Thread 0: the levels after the rounds before round q (see heavy_scans).
  __device__ __forceinline__ void count_scans(int32_t q) {
    const int64_t rounds = q - B->level_q;
    B->level = max((int64_t)0, B->level + M->scans + M->wide - rounds * B->scans_limit);
    B->level_wide = max((int64_t)0, B->level_wide + M->wide - rounds * B->wide_limit);
    B->level_q = q;
    M->scans = M->wide = 0;
    M->heavy = B->level > kHeavyRounds * B->scans_limit || B->level_wide > kHeavyRounds * B->wide_limit;
  }

  // Rows list[0..m) of T against the prices: sets M->bad if an entry breaks
  // P(u) <= T[u][v] + P(v), or a price exceeds q_n.
  __device__ bool broken_rows(const int32_t* list, int m) {
    const int kp = (k + 31) & ~31;
    const int total = m * kp;
    bool bad = false;
    for (int it = tid; it < total; it += kThreads) {
      const int i = it / kp, v = it % kp;
      const int32_t c = list[i];
      if (v < k && v != c) {
        const int32_t t = arc(c, v);
        if (t != kInf && (PT)s_pot[c] > (PT)t + s_pot[v]) bad = true;
      } else if (v == c && !STRICT && s_pot[c] > s_qn[c]) {
        bad = true;
      }
    }
    return bad;
  }

  // Prices from the table: P = q_n lowered by whole sweeps until every entry
  // holds (reverse Bellman-Ford; exact distances to a paid slot).
  __device__ bool rebuild_prices() {
    const int lane = tid & 31, warp = tid >> 5;
    bool room = false;
    for (int v = tid; v < k; v += kThreads) room |= vacant(v);
    room = __syncthreads_or(room) != 0;
    for (int v = tid; v < k; v += kThreads)
      s_pot[v] = !STRICT ? s_qn[v] : room && !vacant(v) ? kGPenLimit - 1 : 0;
    __syncthreads();
    for (int sweep = 0; sweep <= k + 1; ++sweep) {
      bool any = false;
      for (int u = warp; u < k; u += kWarps) {
        int64_t best = INT64_MAX;
        for (int v = lane; v < k; v += 32) {
          const int32_t t = v != u ? arc(u, v) : kInf;
          if (t != kInf) best = min(best, (int64_t)t + s_pot[v]);
        }
        for (int off = 16; off > 0; off >>= 1)
          best = min(best, (int64_t)__shfl_xor_sync(0xffffffffu, best, off));
        if (best < s_pot[u]) {
          any = true;
          __syncwarp();
          if (lane == 0) s_pot[u] = clamp32(best);
        }
        __syncwarp();
      }
      if (__syncthreads_or(any) == 0) return true;
    }
    return false;   // a negative cycle in Gamma: Lemmas 1/2 broken
  }

  // P(v) up to d1 - l1(v) and, after a second search, d2 - l2(v); P(j) up to d2.
  __device__ void raise_prices(int32_t j, PT d2, PT d1, bool second) {
    for (int v = tid; v < k; v += kThreads) {
      PT p = s_pot[v];
      if (v == j) {
        p = max(p, d2);
      } else {
        if (s_lab1[v] != kNoLab) p = max(p, d1 - (PT)s_lab1[v]);
        if (second && s_lab2[v] != kNoLab) p = max(p, d2 - (PT)s_lab2[v]);
      }
      s_pot[v] = (int32_t)p;
    }
  }

  // ----------------------------------------------------------- the loop --
  __device__ __forceinline__ void load_order(int64_t r, int64_t r_end, int slot) {
    const int32_t d = r < r_end ? I.order[r] : -1;
    const int32_t j = !STRICT && (uint32_t)d < (uint32_t)n ? I.smin[d] : -1;
    s_ord[2 * slot] = d;
    s_ord[2 * slot + 1] = (uint32_t)j < (uint32_t)k ? j : -1;
  }
  __device__ __forceinline__ void fetch_row(int32_t q, int32_t count) {
    if (q < count) {
      const int32_t d = s_ord[2 * (q & (kGOrd - 1))];
      if ((uint32_t)d < (uint32_t)n) {
        unsigned char* dst = s_ring + (uint32_t)(q & (nring - 1)) * ring_row;
        const unsigned char* src = reinterpret_cast<const unsigned char*>(row(d));
        for (uint32_t b = 16u * (uint32_t)tid; b < ring_row; b += 16u * kThreads)
          asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst + b)),
                       "l"(src + b) : "memory");
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  }

  // Alg. 5: the cheapest center with a vacancy, lowest index on equal cost
  // (-1: none).  Every thread calls it; the row is in shared memory.
  __device__ int32_t strict_target(const T* r) {
    int32_t bv = INT32_MAX, bj = INT32_MAX;
    for (int v = tid; v < k; v += kThreads)
      if (vacant(v) && (int32_t)r[v] < bv) { bv = (int32_t)r[v]; bj = v; }
    const int32_t wv = __reduce_min_sync(0xffffffffu, bv);
    const int32_t wj = __reduce_min_sync(0xffffffffu, bv == wv ? bj : INT32_MAX);
    if ((tid & 31) == 0) {
      s_aff[2 * (tid >> 5)] = wv;
      s_aff[2 * (tid >> 5) + 1] = wj;
    }
    __syncthreads();
    bv = (tid & 31) < kWarps ? s_aff[2 * (tid & 31)] : INT32_MAX;
    bj = (tid & 31) < kWarps ? s_aff[2 * (tid & 31) + 1] : INT32_MAX;
    const int32_t mv = __reduce_min_sync(0xffffffffu, bv);
    const int32_t mj = __reduce_min_sync(0xffffffffu, bv == mv ? bj : INT32_MAX);
    return mj == INT32_MAX ? -1 : mj;
  }

  __device__ void run_rounds(uint64_t deadline) {
    const uint64_t tstart = tid == 0 ? gtimer_ns() : 0;
    const uint64_t cstart = tid == 0 ? clock_cycles() : 0;
    const int64_t r_begin = I.ctl[CTL_ROUNDS];
    const int64_t r_end = min((int64_t)n, I.ctl[CTL_TARGET]);
    const int32_t count = (int32_t)max((int64_t)0, r_end - r_begin);
    for (int v = tid; v < k; v += kThreads) {
      const int32_t ld = I.load[v], sg = I.seg_size[v];
      s_slack[v] = ld - __ldg(I.cap + v);
      s_pen[v] = qval(v, s_slack[v] + 1);
      s_qn[v] = s_slack[v] >= 0 ? s_pen[v] : 0;
      s_seg[v] = sg;
      s_tail[v] = sg > 0 ? page_tab[(int64_t)v * max_pages + ((sg - 1) >> kPageShift)] : 0;
      s_pot[v] = I.pot[v];
    }
    if (tid == 0) {
      B->delta = I.ctl[CTL_DELTA];
      B->free_top = I.ctl[CTL_FREE_TOP];
      B->cycles = B->paths = B->bf_calls = B->bf_sweeps = B->bf_max = B->moves = B->skipped = B->rows = 0;
      B->t_merge = B->t_relax = B->t_sync = B->t_gather = B->t_apply = B->t_rescan = 0;
      B->t_rloop = B->t_rred = 0;
      B->err0 = 0;
      B->npath_reused = 0;
      B->col_rows = 0;
      B->front_sum = 0;
      for (int h = 0; h < 6; ++h) B->front_hist[h] = 0;
      M->scans = M->wide = 0;
      B->level = I.ctl[CTL_LEVEL];
      B->level_wide = I.ctl[CTL_LEVEL_WIDE];
      M->bad = 0;
      M->stop = 0;
      B->level_q = 0;
      B->scans_limit = flags & OPT_NO_EXIT ? (int64_t)1 << 40 : heavy_scans(k);
      B->wide_limit = flags & OPT_NO_EXIT ? (int64_t)1 << 40 : heavy_wide(k);
      M->heavy = 0;
    }
    if (TSM || I.ctl[CTL_MIRROR] == 0)
      for (int64_t u = 0; u < k; ++u)
        for (int cl = tid; cl < ws; cl += kThreads) {
          const int32_t t = cl < k ? tc[u * k + cl] : kTInf;
          tt[u * ws + cl] = (T)(t == kTInf ? kInf : t);
        }
    if (s_td)
      for (int64_t i = tid; i < (int64_t)k * k; i += kThreads) s_td[i] = td[i];
    if (tid < kGOrd) load_order(r_begin + tid, r_end, tid);
    __syncthreads();
    bool prices_ok = I.ctl[CTL_POT] != 0;
    int64_t status = ST_OK;
    int32_t q = 0;
    for (int i = 0; i + 1 < nring; ++i) fetch_row(i, count);
    const int32_t look = (deadline ? kQuantumCheck : kHeavyEvery) - 1;
    static_assert((kQuantumCheck & (kQuantumCheck - 1)) == 0 && kHeavyEvery % kQuantumCheck == 0, "");
    for (; q < count; ++q) {
      if ((q & look) == 0) {   // (at once inside a stretch of the other kernel)
        if (tid == 0) {
          if (q % kHeavyEvery == 0) count_scans(q);
          M->stop = M->heavy || (deadline && q > 0 && gtimer_ns() >= deadline);
        }
        __syncthreads();
        if (M->stop) break;
      }
      if (!prices_ok) {
        if (!rebuild_prices()) { status = ST_ERR_INVARIANT; break; }
        prices_ok = true;
      }
      const uint64_t tm0 = timer() ? clock_cycles() : 0;
      fetch_row(q + nring - 1, count);
      if (q > 0 && q % 32 == 0 && tid >= kThreads - 32) {
        const int32_t at = q + 32 + (tid & 31);
        load_order(r_begin + at, r_end, at & (kGOrd - 1));
      }
      const int32_t d = s_ord[2 * (q & (kGOrd - 1))];
      int32_t j = s_ord[2 * (q & (kGOrd - 1)) + 1];
      if (d < 0 || (!STRICT && j < 0)) { status = ST_ERR_INVARIANT; break; }   // uniform guard
      if (nring == 8) asm volatile("cp.async.wait_group 7;" ::: "memory");
      else asm volatile("cp.async.wait_group 3;" ::: "memory");
      __syncthreads();
      // Alg. 2, allotment: d joins j; its edges enter row j of T
      const T* r = reinterpret_cast<const T*>(s_ring + (uint32_t)(q & (nring - 1)) * ring_row);
      if (STRICT) {
        j = strict_target(r);
        if (j < 0) { status = ST_ERR_INVARIANT; break; }
      }
      const int32_t own = (int32_t)r[j];
      const bool over = !STRICT && s_slack[j] >= 0;
      const int32_t ql = over ? s_pen[j] : 0;   // q_j(load - cap + 1), paid by d
      const int32_t pj = s_pot[j];
      bool viol = false;
      for (int cl = tid; cl < k; cl += kThreads) {
        if (cl == j) continue;
        const int32_t t = (int32_t)r[cl] - own;
        const int32_t e = edge(j, cl);
        const int32_t bt = e == kInf ? kTInf : e;
        // equal costs take the lower unit: in global memory a reduction that
        // nobody waits for
        if (t < bt) {
          set_entry(j, cl, t, d);
        } else if (t == bt) {
          if (s_td) s_td[j * k + cl] = min(s_td[j * k + cl], d);
          else atomicMin(reinterpret_cast<unsigned*>(td + (int64_t)j * k + cl), (unsigned)d);
        }
        viol |= (PT)t + s_pot[cl] < (PT)pj;
      }
      viol = __syncthreads_or(viol) != 0;
      if (tid == kThreads - 32) {
        I.assign[d] = j;
        list_append(j, d, own);
        shift_load(j, 1);
        B->delta += own + ql;
      }
      if (timer()) B->t_merge += clock_cycles() - tm0;
      if (!viol) {
        if (tid == 0) B->skipped++;
        if (!over || pj >= ql) continue;
      }
      // Alg. 1 and Alg. 4 at j: one search for both, and a second one for
      // Alg. 4 if a cycle was applied
      if (STRICT) __syncthreads();   // j's vacancy counts the allotment
      PT cycv = 0, d1 = 0;
      int mc = 0, m2 = 0;
      bool failed = false;
      for (int stage = 0; stage < 2; ++stage) {
        const uint64_t ts0 = timer() ? clock_cycles() : 0;
        LT* lab = stage ? s_lab2 : s_lab1;
        search(j, stage == 0 && viol, over, lab, stage ? s_mid : s_pot, ql);
        if (timer()) B->t_relax += clock_cycles() - ts0;
        const uint32_t sink = M->sink;
        const PT paid = over ? (PT)min(M->paid, kGNever) : (PT)kGNever;   // exact below ql
        if (stage == 0 && viol) cycv = min((PT)0, (PT)lab[j]);
        const bool cycle = stage == 0 && cycv < 0;
        const bool path = !cycle && over && paid < ql;
        if (stage == 0) d1 = paid;
        if (!cycle) {
          // prices up to the cheapest paid slot, over the labels of both searches
          const PT d2 = over ? min(paid, (PT)ql) : (PT)pj;
          raise_prices(j, d2, d2 + cycv, stage == 1);
          if (stage == 0 && over && tid == 0) B->npath_reused++;
        }
        if (M->bad) { failed = true; break; }
        if (!cycle && !path) break;
        const int m = apply(j, path, path ? (int32_t)(sink & ((1u << kGNodeBits) - 1)) : -1, lab,
                            cycle ? cycv : paid - ql);
        if (m < 0) { failed = true; break; }
        if (path) {
          m2 = m;
          break;
        }
        mc = m;
        for (int i = tid; i < mc; i += kThreads) s_cpath[i] = s_path[i];
        if (!over) {
          raise_prices(j, pj, pj + cycv, false);
          break;
        }
        // bounds for the second search: prices raised by the first labels,
        // less the most by which those exceed q_n
        const PT dt = pj + cycv, off = max((PT)0, dt - d1);
        for (int v = tid; v < k; v += kThreads) {
          PT p = s_pot[v];
          if (v != j && s_lab1[v] != kNoLab) p = max(p, dt - (PT)s_lab1[v]);
          s_mid[v] = (int32_t)max(p - off, (PT)-kGPenLimit);
        }
      }
      if (failed) { status = ST_ERR_INVARIANT; break; }
      __syncthreads();   // prices, loads and rows are final
      const bool bad = broken_rows(s_cpath, mc) | broken_rows(s_path, m2);
      if (__syncthreads_or(bad)) prices_ok = false;   // rebuilt before the next round
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();
    for (int v = tid; v < k; v += kThreads) {
      I.pot[v] = s_pot[v];
      I.load[v] = s_slack[v] + __ldg(I.cap + v);
      I.seg_size[v] = s_seg[v];
    }
    if (s_td)
      for (int64_t i = tid; i < (int64_t)k * k; i += kThreads) td[i] = s_td[i];
    if (TSM)
      for (int64_t u = 0; u < k; ++u)
        for (int cl = tid; cl < k; cl += kThreads) {
          const int32_t t = tt[u * ws + cl];
          tc[u * k + cl] = t == kInf ? kTInf : t;
        }
    if (tid == 0) {
      I.ctl[CTL_POT] = prices_ok && status == ST_OK ? 1 : 0;
      if (count > 0) I.ctl[CTL_MIRROR] = TSM ? 0 : 1;
      I.ctl[CTL_ROUNDS] = r_begin + q;
      I.ctl[CTL_GUIDED] += q;
      const int ended = M->heavy;
      count_scans(q);
      I.ctl[CTL_LEVEL] = B->level;
      I.ctl[CTL_LEVEL_WIDE] = B->level_wide;
      if (ended && r_begin + q < r_end) I.ctl[CTL_HEAVY] = 1;
      I.ctl[CTL_DELTA] = B->delta;
      I.ctl[CTL_FREE_TOP] = B->free_top;
      I.ctl[CTL_STATUS] = status != ST_OK ? status : B->err0;
      I.ctl[CTL_CYCLES] += B->cycles;
      I.ctl[CTL_PATHS] += B->paths;
      I.ctl[CTL_BF_CALLS] += B->bf_calls;
      I.ctl[CTL_BF_SWEEPS] += B->bf_sweeps;
      I.ctl[CTL_BF_MAX] = max(I.ctl[CTL_BF_MAX], B->bf_max);
      I.ctl[CTL_MOVES] += B->moves;
      I.ctl[CTL_NCYC_SKIPPED] += B->skipped;
      I.ctl[CTL_ROWS_SCANNED] += B->rows;
      I.ctl[CTL_T_TOTAL] += gtimer_ns() - tstart;
      I.ctl[CTL_T_CYCLES] += clock_cycles() - cstart;
      I.ctl[CTL_T_MERGE] += B->t_merge;
      I.ctl[CTL_T_RELAX] += B->t_relax;
      I.ctl[CTL_T_APPLY] += B->t_apply;
      I.ctl[CTL_T_RESCAN] += B->t_rescan;
      I.ctl[CTL_TSM_ON] = TSM ? 1 : 0;
      I.ctl[CTL_NPATH_REUSED] += B->npath_reused;
      I.ctl[CTL_COL_ROWS] += B->col_rows;
      I.ctl[CTL_FRONT_SUM] += B->front_sum;
      for (int h = 0; h < 6; ++h) I.ctl[CTL_FRONT_HIST + h] += B->front_hist[h];
    }
    __syncthreads();
  }
};

}  // namespace lbdd
