// Body of the group-resident kernel (gpo_fused.cu includes it once per capacity, each
// time inside its own namespace after defining kMaxN (largest group), kThreads (a
// multiple of 128, at least 256), kMinBlocks (CTAs per SM the launch bounds ask for),
// kRingBytes (the tile ring) and kTmemCols (accumulator columns, a power of two >= 32
// that holds every segment of a one-pass group of kMaxN states, or 512)).

constexpr int kMaxSlots = 8;                    // k-slices in flight at most (mbarrier pairs)
constexpr int kPlaceBytes = kRingBytes - 96 * 128;  // slices lie below this: the MMA of a group's last
                                                    // 128-row block reads its A operand up to 96 rows
                                                    // past the slice (rows that feed unused lanes)
constexpr int kBoxBytes = kTileM * 128;         // 128 rows x 128 bytes
constexpr int kTailRows = 32;                   // rows of the second tensor map's box
constexpr int kGThreads = kThreads - 64;        // warps 2..: group work
constexpr int kEpiThreads = kThreads - 128;     // warps 4..: accumulator drain
constexpr int kReps = kEpiThreads / 128;        // drain warps per accumulator lane quarter
constexpr int kWarpEdges = 256;                 // linked pairs listed per epilogue warp and group
constexpr int kEdgeList = kWarpEdges * (kEpiThreads / 32);
// Groups of two passes wait for the second one's MMAs after draining the first: the token scatter
// of the group before is put there (deferred_tokens) where that wait is longer than the scatter.
// Not before a group of one pass, or with narrow rows: the scatter by the drain warps alone then
// only delays the drain.  Put off / at once, us: 512 groups of 370 states (nearly all of two
// passes) d = 64 141 / 135, 256 169 / 165, 384 183 / 180, 512 193 / 194, 768 233 / 238, 1024
// 253 / 262, 2048 403 / 413; 512 of 320 d = 512 169 / 171, 1024 219 / 228; 512 of 256 states
// (one pass, put off whatever follows) d = 1024 173 / 168, 512 branching ones of 200 222 / 217.
constexpr bool kDeferTokens = kMaxN > 2 * kTileM;
constexpr int kDeferD = 512;                    // narrowest rows for which the scatter is put off
constexpr int kBarGroup = 1;                    // named barrier of the group warps
constexpr int kBarEpi = 2;                      // named barrier of the drain warps
constexpr int kBarSetup = 3;                    // named barrier of warps 2 and 3 (early set-up)
static_assert(kMaxN <= 3 * kTileM, "row blocks of a group");
static_assert(kThreads % 128 == 0 && kThreads >= 256 && kGThreads >= kMaxN, "fused kernel shape");

struct Seg {
  int b, c0, len, tcol;  // row block, first column (local), columns, TMEM column
};

struct Plan {
  int npass;
  int nseg[2];
  Seg seg[2][4];
};

__device__ __forceinline__ int r16(int x) { return (x + 15) & ~15; }

// Byte offset in the ring of the next k-slice of `bytes`: right after the previous
// one, or back at 0 if it would reach past kPlaceBytes.  Producer and MMA warp
// place the same sequence of slices with this rule.
__device__ __forceinline__ int ring_place(int head, int bytes) { return head + bytes <= kPlaceBytes ? head : 0; }
__device__ __forceinline__ int r32(int x) { return (x + 31) & ~31; }

// Segments of the upper triangle: row block b against columns [128 b, n) in
// chunks of at most 256 (one MMA each).  Each segment owns a multiple of 32
// TMEM columns (the epilogue reads 32 columns at a time).  One pass if they
// fit 512 TMEM columns, else pass 0 = blocks >= 1 (at most 256 + 128 columns)
// and pass 1 = block 0 (at most 256 + 128), so that the norms of every column
// a pass needs come from its own or an earlier pass.
// The roles that run in single lanes (producer, MMA issuer) and the drain's plan in shared memory
// take all of this without local arrays: those would lie in local memory, for which the
// statistics' streaming loads leave no place in the few KB of L1 beside the tile ring, so that
// every k-slice of those roles waited for L2 (128 groups of 256 states 55.2 -> 52.3 us, 512 of
// 320 252 -> 243).

// Passes of a group with n states.
__device__ __forceinline__ int plan_passes(int n) {
  int tot = 0;
  for (int b = 0; b * kTileM < n; ++b)
    for (int c0 = b * kTileM; c0 < n; c0 += kTileN) tot += r32(min(kTileN, n - c0));
  return tot <= kTmemCols ? 1 : 2;
}
// Row blocks [b0, b1) of a pass (fewer where the group ends before).
__device__ __forceinline__ void pass_blocks(int npass, int pass, int& b0, int& b1) {
  b0 = npass == 2 && pass == 0 ? 1 : 0;
  b1 = npass == 2 && pass == 1 ? 1 : 3;
}

__device__ __forceinline__ void make_plan(int n, Plan& pl) {
  pl.npass = plan_passes(n);
  for (int pass = 0; pass < pl.npass; ++pass) {
    int b0, b1, m = 0, col = 0;
    pass_blocks(pl.npass, pass, b0, b1);
    for (int b = b0; b < b1 && b * kTileM < n; ++b)
      for (int c0 = b * kTileM; c0 < n; c0 += kTileN) {
        Seg& sg = pl.seg[pass][m++];  // at most 4: two of block 0, one each of blocks 1 and 2
        sg.b = b;
        sg.c0 = c0;
        sg.len = min(kTileN, n - c0);
        sg.tcol = col;
        col += r32(sg.len);
      }
    pl.nseg[pass] = m;
  }
}

// The group's rollout and state ranges; false if they are out of range.  Tree layout:
// the rollouts are the group's leaves and the states come from group_state_off.
__device__ __forceinline__ bool group_range(const gpo_batch& b, const Sizes& sz, int g, int& r0, int& nr, int& s0,
                                            int& n) {
  const int a = b.group_rollout_off[g], c = b.group_rollout_off[g + 1];
  if (a < 0 || c < a || c > sz.R) return false;
  const int x = b.parent ? b.group_state_off[g] : b.rollout_step_off[a];
  const int y = b.parent ? b.group_state_off[g + 1] : b.rollout_step_off[c];
  if (x < 0 || y < x || y > sz.N) return false;
  r0 = a;
  nr = c - a;
  s0 = x;
  n = y - x;
  return true;
}

// Group handled here (all roles agree, they read the same inputs).
__device__ __forceinline__ bool group_active(const gpo_batch& b, const Sizes& sz, int g, int& r0, int& nr, int& s0,
                                             int& n) {
  return group_range(b, sz, g, r0, nr, s0, n) && n > 0 && n <= kMaxN && n <= sz.maxn && nr > 0 && nr <= n;
}

struct __align__(16) GroupSmem {
  int lab[kMaxN];
  union {
    int roll[kMaxN];     // chain layout: rollout of each state (local)
    int par[kMaxN];      // tree layout: parent of each state (local, -1 = the prompt root)
  };
  int dep[kMaxN];
  int slen[kMaxN];
  union {
    int rstart[kMaxN + 1];  // chain layout: local state offsets of the rollouts
    int cown[kMaxN + 1];    // tree layout: c_own, rewards of the subtree's leaves
  };
  float n2[kMaxN];
  alignas(16) float rn[kMaxN];  // 1 / |z_i| (0 for a zero row), read four at a time
  float thr[kMaxN];      // kappa |z_i| (+inf for a zero row or a row that is not tested)
  int rend[kMaxN];       // end (local, exclusive) of the rollout (tree: of the subtree) of state i;
                         // the columns right of i that are not its descendants are [rend, n)
  float eadv[kMaxN], ecor[kMaxN], eeff[kMaxN];
  union {
    int64_t tok0[kMaxN + 1];   // chain layout: token offsets of the rollouts
    int town[2 * kMaxN + 2];   // tree layout: t_own, leaves of the subtree
  };
  int64_t tstart[kMaxN];
  uint8_t rew[kMaxN];
  uint8_t emask[kMaxN];
  unsigned long long esum[3];  // exploration efficiency: token sums
  int flags;             // bit 0: group invalid
  int overflow;          // some warp found more pairs than its part of elist holds
  int nstat[2];          // group_eta_stats: rows with a dot, rows with the norm alone (group_row_stats:
                         // the next block of 8 rows)
  bool wait_ahead;       // the CTA's next group has two passes
  int put_off;           // scatter put off: states of the group, its first token,
  int64_t dbase;
  uint32_t dts[kDeferTokens ? kMaxN + 1 : 1];  // of each state relative to it (they follow one another),
  float dval[kDeferTokens ? kMaxN : 1];        // and each state's advantage
  uint16_t slist[kMaxN]; // those rows: with a dot from the front, the norm alone from the end
  Plan plan;
  uint32_t elist[kEdgeList];  // linked pairs of the group, kWarpEdges per epilogue warp: i | j << 16
  alignas(16) unsigned char X[group_scratch_sep_bytes(kMaxN)];  // group-math sums (separate layout)
};
// Tree layout: the group math's sums (tree_scratch) take elist and X, free once the drain
// has built the classes; during the set-up elist holds the scan's warp totals.
constexpr size_t kTreeXOff = offsetof(GroupSmem, elist);
static_assert(offsetof(GroupSmem, X) + sizeof(GroupSmem::X) - kTreeXOff >= tree_scratch_bytes(kMaxN),
              "tree scratch does not fit");

struct __align__(8) Ctl {
  uint64_t full[kMaxSlots];
  uint64_t empty[kMaxSlots];
  uint64_t tfull;
  uint64_t tempty;
  uint64_t drain;
  int slice_off[kMaxSlots];  // the producer's: offsets of the slices in flight
  uint32_t tmem_base;
};

constexpr uint32_t kCtlOff = (sizeof(GroupSmem) + 15) & ~15u;
constexpr uint32_t kTilesOff = kCtlOff + ((sizeof(Ctl) + 15) & ~15u);
static_assert(kTilesOff + 1023 + kRingBytes <= 232448, "fused kernel exceeds 227 KB of shared memory");

__device__ __forceinline__ void bar_group() { asm volatile("bar.sync %0, %1;" ::"n"(kBarGroup), "n"(kGThreads) : "memory"); }
__device__ __forceinline__ void bar_epi() { asm volatile("bar.sync %0, %1;" ::"n"(kBarEpi), "n"(kEpiThreads) : "memory"); }
__device__ __forceinline__ void bar_setup() { asm volatile("bar.sync %0, %1;" ::"n"(kBarSetup), "n"(64) : "memory"); }

// Bits a..31 of a word (all for a <= 0, none for a >= 32).
__device__ __forceinline__ uint32_t bits_from(int a) { return a <= 0 ? 0xFFFFFFFFu : (a >= 32 ? 0u : 0xFFFFFFFFu << a); }

template <int kBar, int kCount>
__device__ __forceinline__ bool bar_any(bool flag) {
  uint32_t out;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.u32 p, %1, 0;\n\t"
      "bar.red.or.pred q, %2, %3, p;\n\t"
      "selp.u32 %0, 1, 0, q;\n\t}"
      : "=r"(out)
      : "r"((uint32_t)flag), "n"(kBar), "n"(kCount)
      : "memory");
  return out != 0;
}

__device__ __forceinline__ float pick(const uint32_t (&r)[32], int j) {
  float v = 0.f;
#pragma unroll
  for (int k = 0; k < 32; ++k)
    if (k == j) v = __uint_as_float(r[k]);
  return v;
}

// The compensated row statistics that the group's eta's ask for (where group_row_stats has
// not computed every row's; all group threads, one state each: thread gt has state gt; need:
// eta(p(v), v) of that state is read).  The rows are known only once the classes are, when they
// have just been streamed and lie in L2, and they are few: 0.2 to 0.45 of a chain batch's states (a step whose score differs from its
// parent's, below a parent whose class has several edges), 0.85 of a branching one's.  Two
// lists, the rows with a dot (|z_v|^2 and <z_{p(v)}, z_v>) from the front of slist and the
// parents that need |z|^2 alone from its end; a half-warp per row (half_warp_row_sums,
// biases from the Gram diagonal), every row's norm once.  Bound by the latency of its loads
// and dependent sums at 14 warps per SM (a third of the issue slots used).  Results as float
// pairs: |z|^2 in (rn, thr), free once the pairs are tested, the dot in (ecor, eeff).
// Whole call, against the statistics of all rows (a CTA's first group while it streams in,
// the groups after it in a launch of their own before): 512 groups of 320 states 244 -> 219 us
// (other shapes at rest_stats_first in gpo_api.cu).
template <class Par>
__device__ __forceinline__ void group_eta_stats(const gpo_batch& b, const Sizes& sz, const Ws& ws, GroupSmem* gs,
                                                int g, int s0, int n, bool need, Par par, int gt, int wg, int lane,
                                                const Status& st) {
  int* mark = reinterpret_cast<int*>(gs->eadv);  // zeroed with the set-up
  const int pl = need ? par(gt) : -1;
  if (pl >= 0) mark[pl] = 1;
  bar_group();
  const bool alone = gt < n && !need && mark[gt] != 0;
  const uint32_t md = __ballot_sync(0xffffffffu, need), ma = __ballot_sync(0xffffffffu, alone);
  int bd = 0, ba = 0;
  if (lane == 0) {
    if (md) bd = atomicAdd(&gs->nstat[0], __popc(md));
    if (ma) ba = atomicAdd(&gs->nstat[1], __popc(ma));
  }
  bd = __shfl_sync(0xffffffffu, bd, 0);
  ba = __shfl_sync(0xffffffffu, ba, 0);
  const uint32_t below = (1u << lane) - 1u;
  if (need) gs->slist[bd + __popc(md & below)] = (uint16_t)gt;  // together at most n rows: the lists never meet
  if (alone) gs->slist[kMaxN - 1 - (ba + __popc(ma & below))] = (uint16_t)gt;
  bar_group();

  const int nd = gs->nstat[0], na = gs->nstat[1];
  const int pd = (nd + 1) >> 1, pa = (na + 1) >> 1;  // two rows per warp and step
  const int hw = lane >> 4, hl = lane & 15;
  const int64_t rs = sz.stride / 8;  // row stride in 16-byte chunks
  const uint4* Z = reinterpret_cast<const uint4*>(b.emb);
#pragma unroll 1
  for (int k = wg; k < pd + pa; k += kGThreads / 32) {
    const bool wd = k < pd;  // (warp-uniform)
    const int e = 2 * (wd ? k : k - pd) + hw;
    bool live = e < (wd ? nd : na);
    const int i = live ? (int)gs->slist[wd ? e : kMaxN - 1 - e] : 0;
    live = live && GPO_BOUNDS(st, s0 + i, sz.N, kWhereStats);
    float2 n2, dot;
    if (wd) {
      const int q = live ? par(i) : 0;  // the parent, or -1: the prompt embedding
      live = live && GPO_BOUNDS(st, q >= 0 ? s0 + q : 0, sz.N, kWhereStats);
      const uint4* y = q >= 0 ? Z + (int64_t)(s0 + q) * rs : reinterpret_cast<const uint4*>(b.root_emb) + (int64_t)g * rs;
      half_warp_row_sums<true>(Z + (int64_t)(s0 + i) * rs, y, sz.d, gs->n2[i], q >= 0 ? gs->n2[q] : ws.x_root_n2[g].x,
                               hl, live, n2, dot);
    } else {
      half_warp_row_sums<false>(Z + (int64_t)(s0 + i) * rs, nullptr, sz.d, gs->n2[i], 0.f, hl, live, n2, dot);
    }
    if (live && hl == 0) {
      gs->rn[i] = n2.x;
      gs->thr[i] = n2.y;
      if (wd) {
        gs->ecor[i] = dot.x;
        gs->eeff[i] = dot.y;
      }
    }
  }
  bar_group();
}

// Compensated |z_v|^2 and <z_{p(v)}, z_v> of every state of a group into ws.x_n2 / ws.x_dot
// (float pairs), by the group warps while the producer streams the same rows: for a CTA's
// first group, when they would otherwise wait for the stream, of a branching batch or with
// rows of d < kEarlyD.  All rows' statistics then take no longer than the stream and what
// follows it, while group_eta_stats is a serial step after the classes; with wider rows its
// third of a chain batch's rows is the less.  These statistics / group_eta_stats, us a call:
//   groups x states   d = 64    256       512       768       896       1024      1280      1536      2048
//   128 x 256         27 / 35   31 / 37   39 / 41   45 / 50   49 / 52   52 / 53   60 / 61   68 / 65   103 / 87
//   128 x 340         33 / 43   39 / 45   52 / 51   63 / 65   69 / 68   77 / 71   90 / 83   102 / 91  128 / 112
//   256 x 56          19 / 24   21 / 25   25 / 26   29 / 29   31 / 30   33 / 32   38 / 37   41 / 38   50 / 45
//   256 x 112         23 / 31   27 / 31   33 / 33   40 / 40   43 / 42   46 / 42   53 / 49   59 / 52   73 / 62
//   16 x 56           19 / 23   20 / 23   21 / 24   23 / 26   25 / 27   25 / 28   28 / 31   31 / 34   36 / 40
// A branching batch reads 0.85 of its eta's: 128 groups of 200 d = 64 40 / 52, 1024 67 / 74, 2048
// 94 / 103.  The calling warps claim blocks of 8 rows from gs->nstat[0] until none is
// left, so that warps that join late or run slower take fewer (eight_rows_sums).  Parents: with `early` (chain
// layout, before the group's set-up) the previous state for every state but the group's first
// (the set-up fixes the rollouts' first states afterwards: their parent is the prompt root);
// otherwise from the group layout in shared memory.
constexpr int kEarlyD = 1024;
__device__ __forceinline__ void group_row_stats(const gpo_batch& b, const Sizes& sz, const Ws& ws, GroupSmem* gs,
                                                int g, int s0, int n, bool tree, bool early, int lane, const Status& st) {
  const int r = lane >> 2, c = lane & 3;
  const int64_t rs = sz.stride / 8;  // row stride in 16-byte chunks
  const uint4* Z = reinterpret_cast<const uint4*>(b.emb);
  const uint4* RZ = reinterpret_cast<const uint4*>(b.root_emb);
  auto claim = [&]() {
    int k = 0;
    if (lane == 0) k = atomicAdd(&gs->nstat[0], 1);
    return __shfl_sync(0xffffffffu, k, 0);
  };
  for (int blk = claim(); blk * 8 < n; blk = claim()) {
    const int i = blk * 8 + r;  // local row of this lane
    const bool live = i < n;
    // parent: >= 0 a local row, -2 the prompt embedding, -1 none (eta 0)
    int pl = -1;
    if (live) {
      if (early) {
        pl = i - 1;
      } else {
        pl = tree ? gs->par[i] : (gs->dep[i] > 1 ? i - 1 : -1);
        if (pl < 0) pl = b.root_emb ? -2 : -1;
      }
    }
    const bool from_left = pl >= 0 && pl == i - 1 && r > 0;
    // (debug build) the rows this lane reads; the whole warp skips the block if any is out of
    // range, since the sums below shuffle across all its lanes
    const bool rows_ok =
        GPO_BOUNDS(st, s0 + (live ? i : 0), sz.N, kWhereStats) && GPO_BOUNDS(st, pl >= 0 ? s0 + pl : 0, sz.N, kWhereStats);
    if (!__all_sync(0xffffffffu, rows_ok)) continue;
    const uint4* zb = Z + (int64_t)(s0 + (live ? i : 0)) * rs;
    const uint4* pb = pl >= 0 ? Z + (int64_t)(s0 + pl) * rs : (pl == -2 ? RZ + (int64_t)g * rs : nullptr);
    float2 n2, dot;
    eight_rows_sums<false>(zb, pb, live, from_left, sz.d, c, 0.f, 0.f, n2, dot);
    if (pl == -1) dot = make_float2(0.f, 0.f);
    if (live && c == 0 && GPO_BOUNDS(st, s0 + i, sz.N, kWhereStats)) {
      ws.x_n2[s0 + i] = n2;
      ws.x_dot[s0 + i] = dot;
    }
  }
}

// Tree-layout set-up of group g (Sec. 4.2 branching rollouts: parents precede their
// children, depth-first pre-order): checks, depth, subtree end, own terminal statistics
// (Sec. 4.3: c_own / t_own of a state = the rewards / the number of the leaves of its
// subtree, the leaves in state order being the group's rollouts) and the first token of
// every edge.  One state per group thread (kGThreads >= kMaxN); every group thread calls
// it.  An invalid group gets bit 0 of gs->flags (visible to all on return).
__device__ __forceinline__ void tree_setup(const gpo_batch& b, const Sizes& sz, GroupSmem* gs, int g, int r0, int nr,
                                           int s0, int n, int gt, int wg, int lane, const Status& st) {
  const int64_t t0 = b.group_token_off[g], t1 = b.group_token_off[g + 1];
  const int i = gt;
  int pp = -1;
  bool bad = gt == 0 && (t0 < 0 || t1 < t0 || t1 > sz.T);
  if (i < n) {
    pp = b.parent[s0 + i];
    const int L = b.step_len[s0 + i];
    gs->lab[i] = i;
    gs->slen[i] = L;
    gs->par[i] = pp;
    gs->rend[i] = i + 1;
    gs->cown[i] = 0;
    gs->town[i] = 0;
    gs->eadv[i] = 0.f;  // (the marks of group_eta_stats)
    bad = bad || pp < -1 || pp >= i || L < 1;
  }
  bad = bar_any<kBarGroup, kGThreads>(bad);
  bool bad2 = false;
  if (!bad && i < n) {
    if (pp >= 0) {  // pre-order: p(v) lies on the path from the root to the state before v
      int x = i - 1;
      while (x > pp) x = gs->par[x];
      bad2 = x != pp;
    }
    int d = 1;
    for (int x = pp; x >= 0; x = gs->par[x]) {  // par[x] < x: at most i steps
      ++d;
      atomicMax(&gs->rend[x], i + 1);
    }
    gs->dep[i] = d;
  }
  bad = bar_any<kBarGroup, kGThreads>(bad2) || bad;
  if (bad) {
    if (gt == 0) {
      report(st, GPO_ERR_SHAPE, 2, g);
      atomicOr(&gs->flags, 1);
    }
    bar_group();
    return;
  }
  // leaf index and first token: block-wide scans of (is leaf, step length) in state order
  const bool leaf = i < n && gs->rend[i] == i + 1;
  int lc = leaf ? 1 : 0;
  long long tc = i < n ? gs->slen[i] : 0;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, lc, o);
    const long long z = __shfl_up_sync(0xffffffffu, tc, o);
    if (lane >= o) {
      lc += y;
      tc += z;
    }
  }
  int* wl = reinterpret_cast<int*>(gs->X);             // warp totals (X is free until the group math)
  long long* wt = reinterpret_cast<long long*>(gs->X + 64);
  if (lane == 31) {
    wl[wg] = lc;
    wt[wg] = tc;
  }
  bar_group();
  int lbase = 0, ltot = 0;
  long long tbase = 0, ttot = 0;
  for (int w = 0; w < kGThreads / 32; ++w) {
    if (w < wg) {
      lbase += wl[w];
      tbase += wt[w];
    }
    ltot += wl[w];
    ttot += wt[w];
  }
  if (gt == 0 && (ltot != nr || ttot != t1 - t0)) {
    report(st, GPO_ERR_SHAPE, 2, g);
    atomicOr(&gs->flags, 1);
  }
  if (i < n) gs->tstart[i] = t0 + tbase + tc - gs->slen[i];
  if (leaf) {
    const int li = lbase + lc - 1;  // < ltot
    if (li < nr) {
      const int rw = b.reward[r0 + li];
      if (rw > 1) {
        report(st, GPO_ERR_BAD_REWARD, 2, r0 + li);
        atomicOr(&gs->flags, 1);
      } else {
        for (int x = i; x >= 0; x = gs->par[x]) {
          atomicAdd(&gs->cown[x], rw);
          atomicAdd(&gs->town[x], 1);
        }
      }
    }
  }
  bar_group();
}

// A half-warp (hl = its lane) writes x to dst[ts, te), dst 16-byte aligned: whole 16-byte chunks,
// then the at most 3 + 3 tokens of the partial first and last one (which neighbour other states'
// tokens) with scalar stores.
__device__ __forceinline__ void half_warp_span(float* dst, int64_t ts, int64_t te, float x, int hl) {
  const int64_t qa = (ts + 3) >> 2, qb = te >> 2;
  const int64_t h1 = qa <= qb ? 4 * qa : te;  // head [ts, h1)
  const int64_t t0 = qa <= qb ? 4 * qb : te;  // tail [t0, te)
  const int64_t tp = hl < 4 ? ts + hl : t0 + (hl - 4);
  const float4 v = make_float4(x, x, x, x);
  for (int64_t c = qa + hl; c < qb; c += 16) __stcs(reinterpret_cast<float4*>(dst) + c, v);
  if (hl < 4 ? tp < h1 : (hl < 8 && tp < te)) dst[tp] = x;
}

// The token scatter that the group before put off, by the drain warps (thread tid of them).
__device__ __forceinline__ void deferred_tokens(const gpo_outputs& o, const Sizes& sz, const GroupSmem* gs, int tid,
                                                const Status& st) {
  const int64_t base = gs->dbase;
  const int n = gs->put_off;
#pragma unroll 1
  for (int i = tid >> 4; i < n; i += kEpiThreads / 16) {
    const int64_t ts = base + gs->dts[i], te = base + gs->dts[i + 1];
    if (!GPO_BOUNDS(st, ts, sz.T, kWhereTokens) || !GPO_BOUNDS(st, te - 1, sz.T, kWhereTokens)) continue;
    half_warp_span(o.adv, ts, te, gs->dval[i], tid & 15);
  }
}

__global__ void __launch_bounds__(kThreads, kMinBlocks)
    fused_kernel(const __grid_constant__ CUtensorMap zmap, const __grid_constant__ CUtensorMap zmap32, gpo_batch b,
                 gpo_outputs o, Sizes sz, Ws ws, Params p) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  // group state, barriers, then the tiles on a 1024-byte boundary (128B swizzle).  Every
  // pointer is smem_raw plus an offset, so the compiler keeps the shared address space
  // (plain shared loads, stores and atomics rather than generic ones).
  GroupSmem* gs = reinterpret_cast<GroupSmem*>(smem_raw);
  Ctl* ctl = reinterpret_cast<Ctl*>(smem_raw + kCtlOff);
  const uint32_t sbase = smem_u32(smem_raw);
  unsigned char* tiles = smem_raw + (((sbase + kTilesOff + 1023u) & ~1023u) - sbase);
  const Status st{ws.status, ws.tag};
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int KT = (sz.d + kTileK - 1) / kTileK;
  const float kappa = p.kappa_f;

  const bool tree = b.parent != nullptr;
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    sign_status(st);
    if (b.group_rollout_off[0] != 0 || b.group_rollout_off[sz.G] != sz.R) report(st, GPO_ERR_SHAPE, 2, 0);
    if (tree) {
      if (b.group_state_off[0] != 0 || b.group_state_off[sz.G] != sz.N) report(st, GPO_ERR_SHAPE, 2, 1);
      if (b.group_token_off[0] != 0 || b.group_token_off[sz.G] != sz.T) report(st, GPO_ERR_SHAPE, 2, 2);
    } else {
      if (b.rollout_step_off[0] != 0 || b.rollout_step_off[sz.R] != sz.N) report(st, GPO_ERR_SHAPE, 2, 1);
      if (b.rollout_token_off[0] != 0 || b.rollout_token_off[sz.R] != sz.T) report(st, GPO_ERR_SHAPE, 2, 2);
    }
  }
  if (threadIdx.x == 0) {
    for (int s = 0; s < kMaxSlots; ++s) {
      mbar_init(&ctl->full[s], 1);
      mbar_init(&ctl->empty[s], 1);
    }
    mbar_init(&ctl->tfull, 1);
    mbar_init(&ctl->tempty, kEpiThreads / 32);
    mbar_init(&ctl->drain, 1);
    fence_mbar_init();
    gs->nstat[0] = gs->nstat[1] = 0;
    gs->put_off = 0;
    tma_prefetch_desc(&zmap);
    tma_prefetch_desc(&zmap32);
  }
  if (warp == 1) {
    tmem_alloc(&ctl->tmem_base, kTmemCols);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = ctl->tmem_base;

  if (warp == 0) {
    // ---------------------------------------------------------------- TMA producer (lane 0)
    if (lane == 0) {
    // A k-slice (64 embedding elements of the rows a pass reads) takes exactly its bytes
    // of the ring; slice `seq` signals mbarrier pair seq % kMaxSlots.  The slices in flight
    // form one run in ring order, from the oldest one's offset o to head (wrapping to 0 at
    // most once), so a new slice at `off` is free to write when fewer than kMaxSlots are in
    // flight and: the run does not wrap (o < head) and the slice follows head, or wraps to
    // end by o; or the run wraps (o >= head) and the slice follows head and ends by o.
    // Otherwise wait for the oldest slice's consumption and look again.
    int head = 0;
    uint32_t seq = 0, oldest = 0;  // slices issued; oldest slice not yet seen consumed
    bool ok = true;
    // L2 policy: pass 0 of a two-pass group keeps its rows, which pass 1 reads again; the others have
    // none, since group_eta_stats reads the rows after the last pass.  (Evict-first on pass 1 made
    // those reads go to DRAM: 512 groups of 320 states read 557 MB for 337 MB of rows and took
    // 231 us, 224 without it.)
    const uint64_t keep = l2_policy_evict_last();
    for (int g = sz.g0 + (int)blockIdx.x; g < sz.g1 && ok; g += gridDim.x) {
      int r0, nr, s0, n;
      if (!group_active(b, sz, g, r0, nr, s0, n)) continue;
      const int npass = plan_passes(n);
      const int rows = r32(n);  // rows [0, r32(n)) of the group; the MMAs read no further
      for (int pass = 0; pass < npass && ok; ++pass) {
        const int row0 = npass == 2 && pass == 0 ? kTileM : 0;  // pass 0 of two never reads block 0
        const int bytes = (rows - row0) * 128;
        const bool again = npass == 2 && pass == 0;  // pass 1 reads these rows again
        for (int k = 0; k < KT && ok; ++k) {
          const int off = ring_place(head, bytes);
          while (oldest < seq) {
            const int o = ctl->slice_off[oldest % kMaxSlots];
            const bool busy = seq - oldest >= (uint32_t)kMaxSlots ||
                              (o < head ? (off != head && off + bytes > o) : (off != head || head + bytes > o));
            if (!busy) break;
            if (!mbar_wait(&ctl->empty[oldest % kMaxSlots], (oldest / kMaxSlots) & 1u, st, 20)) {
              ok = false;
              break;
            }
            ++oldest;
          }
          if (!ok) break;
          const int bi = (int)(seq % kMaxSlots);
          unsigned char* t = tiles + off;
          mbar_arrive_expect_tx(&ctl->full[bi], (uint32_t)bytes);
          for (int r = row0; r < rows;) {  // 128-row boxes, then 32-row boxes for the tail
            const bool big = rows - r >= kTileM;
            if (again)
              tma_load_2d_hint(t + (r - row0) * 128, big ? &zmap : &zmap32, &ctl->full[bi], k * kTileK, s0 + r, keep);
            else
              tma_load_2d(t + (r - row0) * 128, big ? &zmap : &zmap32, &ctl->full[bi], k * kTileK, s0 + r);
            r += big ? kTileM : kTailRows;
          }
          ctl->slice_off[bi] = off;
          head = off + bytes;
          ++seq;
        }
      }
    }
    for (uint32_t j = oldest; j < seq; ++j)  // copies still landing in shared memory
      mbar_wait(&ctl->full[j % kMaxSlots], (j / kMaxSlots) & 1u, st, 21, 200000000ull, false);
    }
    __syncwarp();
  } else if (warp == 1) {
    // ---------------------------------------------------------------- MMA issuer (lane 0)
    if (lane == 0) {
    int head = 0;
    uint32_t seq = 0;  // slices consumed (the producer's sequence)
    int u = 0;         // accumulator uses (passes) so far
    bool ok = true;
    // GPO_FLAG_DEBUG_TIMEOUT: the first wait runs out (nothing arrives on `drain` before the
    // commit below), and the CTA winds down as after any timeout
    if (p.debug_timeout) {
      mbar_wait(&ctl->drain, 0, st, 27, kDebugTimeoutNs);  // returns false: reports GPO_ERR_TIMEOUT
      ok = false;
    }
    for (int g = sz.g0 + (int)blockIdx.x; g < sz.g1 && ok; g += gridDim.x) {
      int r0, nr, s0, n;
      if (!group_active(b, sz, g, r0, nr, s0, n)) continue;
      const int npass = plan_passes(n);
      const int rows = r32(n);
      for (int pass = 0; pass < npass && ok; ++pass, ++u) {
        const int row0 = npass == 2 && pass == 0 ? kTileM : 0;
        int b0, b1;  // the pass's segments as make_plan has them, walked
        pass_blocks(npass, pass, b0, b1);
        const int bytes = (rows - row0) * 128;
        if (!mbar_wait(&ctl->tempty, ((uint32_t)u & 1u) ^ 1u, st, 22)) {
          ok = false;
          break;
        }
        tc_fence_after();
        for (int k = 0; k < KT; ++k) {
          const int off = ring_place(head, bytes);
          head = off + bytes;
          const int bi = (int)(seq % kMaxSlots);
          if (!mbar_wait(&ctl->full[bi], (seq / kMaxSlots) & 1u, st, 23)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t t = smem_u32(tiles + off);
          uint32_t dt = tmem;
          for (int b = b0; b < b1 && b * kTileM < n; ++b) {
            const uint64_t ad = smem_desc_k128(t + (uint32_t)((b * kTileM - row0) * 128));
            for (int c0 = b * kTileM; c0 < n; c0 += kTileN) {
              const int len = min(kTileN, n - c0);
              const uint64_t bd = smem_desc_k128(t + (uint32_t)((c0 - row0) * 128));
              const uint32_t idesc = idesc_bf16_f32(kTileM, r16(len));
#pragma unroll
              for (int kk = 0; kk < kTileK / 16; ++kk)
                mma_bf16_ss(dt, ad + 2u * kk, bd + 2u * kk, idesc, (k | kk) != 0);
              dt += (uint32_t)r32(len);
            }
          }
          mma_commit(&ctl->empty[bi]);
          ++seq;
        }
        if (ok) mma_commit(&ctl->tfull);
      }
    }
    mma_commit(&ctl->drain);
    mbar_wait(&ctl->drain, 0, st, 24, 200000000ull, false);
    }
    __syncwarp();
  } else if (warp >= 2) {
    // ---------------------------------------------------------------- group warps
    const int gt = threadIdx.x - 64;  // 0..447
    const bool epi = warp >= 4;
    const int q = warp & 3;           // TMEM lane quarter of an epilogue warp
    const int wg = warp - 2;          // 0..13
    int u = 0;
    for (int g = sz.g0 + (int)blockIdx.x; g < sz.g1; g += gridDim.x) {
      int r0 = 0, nr = 0, s0 = 0, n = 0;
      const bool in_range = group_range(b, sz, g, r0, nr, s0, n);
      if (!(in_range && n > 0 && n <= kMaxN && n <= sz.maxn && nr > 0 && nr <= n)) {
        if (gt == 0) {
          // tree layout: states need leaves, and an empty group has no tokens
          const bool tree_bad = tree && in_range &&
                                ((nr == 0 && n > 0) || (n == 0 && b.group_token_off[g + 1] != b.group_token_off[g]));
          if (!in_range || nr > n || (nr > 0 && n == 0) || tree_bad) report(st, GPO_ERR_SHAPE, 2, g);
          else if (n > kMaxN || n > sz.maxn) report(st, GPO_ERR_UNSUPPORTED, 2, g);
          else if (n == 0) {  // a group without states: Eff 0 (no tokens)
            if (o.group_eff) o.group_eff[g] = 0.f;
            if (o.group_eff_graph) o.group_eff_graph[g] = 0.f;
          }
        }
        continue;
      }
      if (gt == 0) {
        make_plan(n, gs->plan);
        gs->flags = 0;
        gs->overflow = 0;
      }

      // ---- compensated row statistics of every row (group_row_stats), for a CTA's first group
      //      where they pay.  Chain layout without prompt embeddings: the drain warps start at
      //      once (every state's parent taken as the state before it; a rollout's first state
      //      then has eta 0 whatever its dot) while warps 2 and 3 lay out the group, then
      //      join them; otherwise all group warps after the set-up.
      const bool first = g < sz.g0 + (int)gridDim.x;
      const bool stats_here = p.mode == 0 && (tree || sz.d < kEarlyD) && first;
      const bool early = stats_here && !tree && b.root_emb == nullptr;
      if (early && epi) group_row_stats(b, sz, ws, gs, g, s0, n, false, true, lane, st);

      if (tree) {
        tree_setup(b, sz, gs, g, r0, nr, s0, n, gt, wg, lane, st);
      } else if (!early || !epi) {
      // ---- validate the group and lay out its states (Sec. 4.2 chain layout): all group
      //      threads, or warps 2 and 3 alone while the drain warps read the statistics
      const int tid = gt, nt = early ? 64 : kGThreads;  // warps 2 and 3: gt = 0..63
      auto sync = [&] {
        if (early) bar_setup();
        else bar_group();
      };
      for (int r = tid; r <= nr; r += nt) {
        gs->rstart[r] = b.rollout_step_off[r0 + r] - s0;
        gs->tok0[r] = b.rollout_token_off[r0 + r];
      }
      for (int r = tid; r < nr; r += nt) gs->rew[r] = b.reward[r0 + r];
      group_scratch_zero(gs->X, n, tid, nt);  // read after the drain
      for (int i = tid; i < n; i += nt) {
        gs->lab[i] = i;
        gs->slen[i] = b.step_len[s0 + i];
        gs->roll[i] = 0;
        gs->dep[i] = 1;
        gs->eadv[i] = 0.f;  // (the marks of group_eta_stats)
      }
      sync();
      for (int r = tid; r < nr; r += nt) {
        const int a = gs->rstart[r], e = gs->rstart[r + 1];
        bool bad = !(a >= 0 && e > a && e <= n) || gs->rew[r] > 1;
        if (gs->rew[r] > 1) report(st, GPO_ERR_BAD_REWARD, 2, r0 + r);
        int64_t t = gs->tok0[r];
        if (!bad) {
          for (int i = a; i < e; ++i) {
            gs->roll[i] = r;
            gs->dep[i] = i - a + 1;
            gs->rend[i] = e;
            gs->tstart[i] = t;
            if (gs->slen[i] < 1) bad = true;
            t += gs->slen[i];
          }
          if (t != gs->tok0[r + 1] || gs->tok0[r] < 0 || gs->tok0[r + 1] > sz.T) bad = true;
        }
        if (bad) {
          if (gs->rew[r] <= 1) report(st, GPO_ERR_SHAPE, 2, r0 + r);
          atomicOr(&gs->flags, 1);
        }
      }
      if (early) group_row_stats(b, sz, ws, gs, g, s0, n, false, true, lane, st);  // join the drain warps
      }
      bar_group();  // set-up (and with `early` the row statistics) complete
      const bool valid = (gs->flags & 1) == 0;
      if (!early && valid && stats_here) group_row_stats(b, sz, ws, gs, g, s0, n, tree, false, lane, st);
      if (valid && p.mode == 0 && b.root_emb && wg == 0) {  // |prompt embedding|^2, one warp
        float2 n2, dot;
        exact_pair_sums<true>(b.root_emb, (int64_t)g * sz.stride, nullptr, 0, false, sz.d, lane, n2, dot);
        if (lane == 0) {
          if (!isfinite(n2.x)) report(st, GPO_ERR_NONFINITE, 3, sz.N + g);
          ws.x_root_n2[g] = n2;
        }
      }

      // ---- eta(p(v), v) of every state from the finished statistics, by warps 2 and 3 while
      //      the drain warps test the pairs (with `early`: no prompt embedding, a rollout's
      //      first state has eta 0); the group math takes it from ecor / eeff, which it
      //      overwrites only with its own outputs, state by state, after reading it
      if (early && valid && !epi) {
        for (int i = gt; i < n; i += 64) {
          const float2 e = gs->dep[i] == 1 ? make_float2(0.f, 0.f)
                                           : ff_eta(ws.x_dot[s0 + i], ws.x_n2[s0 + i - 1], ws.x_n2[s0 + i]);
          gs->ecor[i] = e.x;
          gs->eeff[i] = e.y;
        }
      }

      if (kDeferTokens && gt == 0) {  // (read after the drain)
        int r2, nr2, s2, n2;
        gs->wait_ahead = sz.d >= kDeferD && g + (int64_t)gridDim.x < sz.g1 &&
                         group_active(b, sz, g + (int)gridDim.x, r2, nr2, s2, n2) && plan_passes(n2) == 2;
      }

      // ---- drain the accumulator pass by pass (warps 4..15)
      bool fail = false;
      if (epi) {
        const Plan& pl = gs->plan;
        const int te = threadIdx.x - 128;     // 0..383
        const int t128 = q * 32 + lane;       // accumulator lane = row within a 128-row block
        const int rep = (warp - 4) >> 2;      // which of the quarter's kReps warps
        const int ew = warp - 4;              // epilogue warp 0..11: owns elist[ew * kWarpEdges, ...)
        uint32_t* wlist = gs->elist + ew * kWarpEdges;
        int wcount = 0;                       // pairs this warp found in the group (warp-uniform)
        for (int pass = 0; pass < pl.npass; ++pass, ++u) {
          if (kDeferTokens && gs->put_off && pass == pl.npass - 1) deferred_tokens(o, sz, gs, te, st);
          const bool got = mbar_wait(&ctl->tfull, (uint32_t)u & 1u, st, 25);
          if (bar_any<kBarEpi, kEpiThreads>(!got)) {
            fail = true;
            break;
          }
          tc_fence_after();
          const int nseg = pl.nseg[pass];
          // squared norms (for the threshold test) from the diagonal of the diagonal segments
          // of this pass (row block b is read by the quarter's warp b % 3)
#pragma unroll 1
          for (int si = 0; si < nseg; ++si) {
            const Seg sg = pl.seg[pass][si];
            if (sg.c0 != sg.b * kTileM || sg.b % kReps != rep || q * 32 >= sg.len) continue;
            const int i = sg.b * kTileM + t128;
            const uint32_t base = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)sg.tcol;
            uint32_t r[32];
            tmem_ld_32x32b_x32(base + (uint32_t)(q * 32), r);
            tmem_wait_ld();
            const float dg = pick(r, lane);
            if (i < n) {
              gs->n2[i] = dg;
              if (!isfinite(dg)) report(st, GPO_ERR_NONFINITE, 2, s0 + i);
            }
          }
          bar_epi();
#pragma unroll 1
          for (int si = 0; si < nseg; ++si) {
            const Seg sg = pl.seg[pass][si];
            if (sg.c0 != sg.b * kTileM || sg.b % kReps != rep) continue;
            const int i = sg.b * kTileM + t128;
            if (i < n) {
              const float n2i = gs->n2[i];
              gs->rn[i] = n2i > 0.f ? 1.0f / sqrtf(n2i) : 0.f;
              gs->thr[i] = n2i > 0.f && valid ? kappa * sqrtf(n2i) : __int_as_float(0x7f800000);
            }
          }
          bar_epi();
          // linked pairs: comparable (different rollout [, same depth]) with sim >= kappa,
          // tested as acc / |z_j| - kappa |z_i| >= 0 (one fma per pair).  In the chain layout
          // the columns j > i outside i's rollout are exactly j >= rend(i), so one bit mask per
          // 32-column chunk keeps j in [rend(i), n).  The quarter's chunks that hold a column
          // right of some row of the warp are dealt round-robin to its three warps.  Each pair
          // found goes to the edge list (or, past its capacity, straight into the forest).
          {
            int dealt = 0;
#pragma unroll 1
            for (int si = 0; si < nseg; ++si) {
              const Seg sg = pl.seg[pass][si];
              const int rowbase = sg.b * kTileM + q * 32;
              const int i = rowbase + lane;
              const bool vrow = i < n;
              const float thr = vrow ? gs->thr[i] : __int_as_float(0x7f800000);
              const int re = vrow ? gs->rend[i] : n;
              const int di = vrow ? gs->dep[i] : -1;
              const int nch = (sg.len + 31) >> 5;
#pragma unroll 1
              for (int ch = 0; ch < nch; ++ch) {
                const int cbase = sg.c0 + ch * 32;
                if (cbase + 31 <= rowbase) continue;  // no column right of any row of this warp
                if (dealt++ % kReps != rep) continue;
                uint32_t r[32];
                tmem_ld_32x32b_x32(tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(sg.tcol + ch * 32), r);
                tmem_wait_ld();
                // bit j of `miss` = sign of acc_j / |z_j| - kappa |z_i| (one fma, exact product):
                // set when the pair is below the threshold
                // (four partial masks keep the or-chains short)
                uint32_t mp[4] = {0u, 0u, 0u, 0u};
                const float4* rn4 = reinterpret_cast<const float4*>(gs->rn + cbase);
#pragma unroll
                for (int j4 = 0; j4 < 8; ++j4) {
                  const float4 c = rn4[j4];
                  const float cc[4] = {c.x, c.y, c.z, c.w};
#pragma unroll
                  for (int t = 0; t < 4; ++t) {
                    const int j = 4 * j4 + t;
                    mp[t] |= (__float_as_uint(fmaf(__uint_as_float(r[j]), cc[t], -thr)) >> 31) << j;
                  }
                }
                const uint32_t miss = (mp[0] | mp[1]) | (mp[2] | mp[3]);
                uint32_t mk = vrow ? ~miss & bits_from(re - cbase) & ~bits_from(n - cbase) : 0u;
                if (p.rule == GPO_MERGE_SAME_DEPTH && mk) {
                  uint32_t m2 = 0u;
                  for (uint32_t t = mk; t; t &= t - 1u) {
                    const int j = __ffs(t) - 1;
                    if (gs->dep[cbase + j] == di) m2 |= 1u << j;
                  }
                  mk = m2;
                }
                // this warp's part of the edge list: one pair per lane per step, slots by ballot
                for (uint32_t act = __ballot_sync(0xffffffffu, mk != 0); act;
                     act = __ballot_sync(0xffffffffu, mk != 0)) {
                  const int slot = wcount + __popc(act & ((1u << lane) - 1u));
                  if (mk) {
                    const int j = cbase + __ffs(mk) - 1;
                    mk &= mk - 1u;
                    if (slot < kWarpEdges) wlist[slot] = (uint32_t)i | ((uint32_t)j << 16);
                    else uf_union(gs->lab, i, j);
                  }
                  wcount += __popc(act);
                }
              }
            }
          }
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(&ctl->tempty);  // accumulator free for the next pass
          // classes = connected components of the linked pairs (Alg. S.1) in the label forest
          // lab (lab[x] <= x, within x's class).  Rounds of hooking over every listed pair of
          // the group (the larger of the two current labels is pointed at the smaller) and
          // shortcutting (lab[x] = lab[lab[x]]) until no pair has unequal labels and every
          // label is a root: then each class's label is its smallest member.  The rounds
          // revisit the pairs of earlier passes, whose links a hook may re-point.  If the list
          // overflowed (pairs united directly), the listed pairs are united the same way
          // instead (root-to-root links, which never re-point a link).
          if (lane == 0 && wcount > kWarpEdges) gs->overflow = 1;
          bar_epi();
          const int nw = min(wcount, kWarpEdges);  // this warp's listed pairs
          if (!gs->overflow) {
            bool conv = false;
#pragma unroll 1
            for (int round = 0; round <= kMaxN && !conv; ++round) {
              bool ch = false;
              for (int e = lane; e < nw; e += 32) {
                const uint32_t ij = wlist[e];
                const int lu = gs->lab[ij & 0xFFFFu], lv = gs->lab[ij >> 16];
                if (lu != lv) {
                  atomicMin(&gs->lab[max(lu, lv)], min(lu, lv));
                  ch = true;
                }
              }
              for (int x = te; x < n; x += kEpiThreads) {
                const int l = gs->lab[x], ll = gs->lab[l];
                if (ll != l) {
                  gs->lab[x] = ll;
                  ch = true;
                }
              }
              conv = !bar_any<kBarEpi, kEpiThreads>(ch);
            }
            if (!conv) {  // not reached in practice; the unions below are correct from any state
              for (int e0 = 0; e0 < nw; e0 += 32) {
                if (e0 + lane < nw) {
                  const uint32_t ij = wlist[e0 + lane];
                  uf_union(gs->lab, (int)(ij & 0xFFFFu), (int)(ij >> 16));
                }
                __syncwarp();
              }
            }
          } else {
            for (int e0 = 0; e0 < nw; e0 += 32) {
              if (e0 + lane < nw) {
                const uint32_t ij = wlist[e0 + lane];
                uf_union(gs->lab, (int)(ij & 0xFFFFu), (int)(ij >> 16));
              }
              __syncwarp();
            }
          }
        }
      }
      if (bar_any<kBarGroup, kGThreads>(fail)) break;
      if (kDeferTokens && gt == 0) gs->put_off = 0;

      // ---- next-layer budgets of a branching group (gpo_layer_budget)
      if (valid && p.mode == 1) {
        auto active = [&](int i) { return p.active == nullptr || p.active[s0 + i] != 0; };
        auto put = [&](int i, int label, int bud) {
          p.budget[s0 + i] = bud;
          if (o.class_id) o.class_id[s0 + i] = s0 + label;
        };
        group_budget(n, gs->lab, gs->dep, p.layer, p.b_next, reinterpret_cast<int*>(gs->n2),
                     reinterpret_cast<int*>(gs->esum), reinterpret_cast<int*>(gs->elist), gt, kGThreads,
                     active, [] { bar_group(); }, put);
      }
      // ---- graph reward and dual-group advantage of every edge
      else if (valid) {
        // eta(p(v), v) from the compensated row statistics: of every row, in the workspace, or of
        // the rows that ask for it
        const bool all_rows = stats_here || (!first && p.rest_stats);
        auto par = [&](int i) { return tree ? gs->par[i] : (gs->dep[i] == 1 ? -1 : i - 1); };
        auto etas = [&](const bool (&need)[1]) {
          if (!all_rows) group_eta_stats(b, sz, ws, gs, g, s0, n, need[0], par, gt, wg, lane, st);
        };
        auto eta = [&](int i) -> float2 {
          if (early) return make_float2(gs->ecor[i], gs->eeff[i]);
          const int q = par(i);  // -1: the prompt embedding
          const float2 nq = q < 0 ? ws.x_root_n2[g] : (all_rows ? ws.x_n2[s0 + q] : make_float2(gs->rn[q], gs->thr[q]));
          return all_rows ? ff_eta(ws.x_dot[s0 + i], nq, ws.x_n2[s0 + i])
                          : ff_eta(make_float2(gs->ecor[i], gs->eeff[i]), nq, make_float2(gs->rn[i], gs->thr[i]));
        };
        const bool has_root = b.root_emb != nullptr;
        auto out = [&](int i, int label, float S, float acor, float E, float dual, unsigned char mask) {
          gs->eadv[i] = dual;
          gs->ecor[i] = acor;
          gs->eeff[i] = E;
          gs->emask[i] = mask;
          const int v = s0 + i;
          if (!GPO_BOUNDS(st, v, sz.N, kWhereStateOut)) return;
          if (o.edge_adv) o.edge_adv[v] = dual;
          if (o.class_id) o.class_id[v] = s0 + label;
          if (o.node_score) o.node_score[v] = S;
          if (o.edge_cor) o.edge_cor[v] = acor;
          if (o.edge_eff) o.edge_eff[v] = E;
          if (o.edge_eff_mask) o.edge_eff_mask[v] = mask;
        };
        if (tree) {
          group_advantages_tree<1>(n, nr, gs->lab, gs->par, gs->dep, gs->rend, gs->cown, gs->town,
                                   tree_scratch(smem_raw + kTreeXOff, n), p, gt, kGThreads, [] { bar_group(); },
                                   has_root, etas, eta, out);
        } else {
          group_advantages<1, true>(n, nr, gs->lab, gs->roll, gs->dep, gs->rstart, gs->rew,
                                    group_scratch_sep(gs->X, n), p, gt, kGThreads, [] { bar_group(); }, has_root, etas,
                                    eta, out);
        }
        // ---- exploration efficiency, Eq. (eq1) (the threshold norms' array is free here)
        if (o.group_eff || o.group_eff_graph) {
          auto own = [&](int i) { return tree ? gs->cown[i] > 0 : gs->rew[gs->roll[i]] != 0; };
          auto len = [&](int i) { return gs->slen[i]; };
          group_efficiency(n, gs->lab, reinterpret_cast<int*>(gs->n2), gs->esum, gt, kGThreads, own, par, len,
                           [] { bar_group(); }, [](bool f) { return bar_any<kBarGroup, kGThreads>(f); },
                           o.group_eff ? o.group_eff + g : nullptr, o.group_eff_graph ? o.group_eff_graph + g : nullptr);
        }
        // ---- every token of an edge carries the edge's advantage (Sec. 4.5), state-major, a
        //      half-warp per state.  With a group of two passes to follow on this CTA it is put off
        //      to that group's last wait for its MMAs: it waits ~13 us for the second one
        //      (320 states of 2 KB), the scatter is ~6.5 us of stores, and the next group starts that
        //      much earlier (kDeferD).  The drain warps do it: with
        //      warps 2 and 3 as well, a second copy of the code, 128 groups of 256 states lose more
        //      (51.3 -> 52.0) than these gain, and those two alone take longer than the wait (268).
        //      Only in the instance whose groups can take two passes; the per-token components
        //      go out at once.  Streaming stores: they take no place in L2 from the rows that are
        //      still to be read (256 groups of 56 states with every output 53.4 -> 49.8 us).
        const bool more = o.adv_cor || o.adv_eff || o.eff_mask;
        const bool later = kDeferTokens && !more && gs->wait_ahead &&
                           gs->tstart[n - 1] + gs->slen[n - 1] - gs->tstart[0] <= 0xFFFFFFFFll;
        if (later) {
          const int64_t base = gs->tstart[0];
          if (gt == 0) {
            gs->dbase = base;
            gs->put_off = n;
          }
          for (int i = gt; i < n; i += kGThreads) {
            gs->dts[i] = (uint32_t)(gs->tstart[i] - base);
            gs->dval[i] = gs->eadv[i];
            if (i == n - 1) gs->dts[n] = (uint32_t)(gs->tstart[i] + gs->slen[i] - base);
          }
        } else {
          const int hl = gt & 15;
#pragma unroll 1
          for (int i = gt >> 4; i < n; i += kGThreads / 16) {
            const int64_t ts = gs->tstart[i], te = ts + gs->slen[i];
            const float x = gs->eadv[i];
            const int64_t qa = (ts + 3) >> 2, qb = te >> 2;
            const int64_t h1 = qa <= qb ? 4 * qa : te;  // head [ts, h1)
            const int64_t t0 = qa <= qb ? 4 * qb : te;  // tail [t0, te)
            const int64_t tp = hl < 4 ? ts + hl : t0 + (hl - 4);
            const bool scal = hl < 4 ? tp < h1 : (hl < 8 && tp < te);
            // (debug build) every store below lies in the state's span [ts, te)
            if (!GPO_BOUNDS(st, ts, sz.T, kWhereTokens) || !GPO_BOUNDS(st, te - 1, sz.T, kWhereTokens)) continue;
            {
              const float4 v = make_float4(x, x, x, x);
              for (int64_t c = qa + hl; c < qb; c += 16) __stcs(reinterpret_cast<float4*>(o.adv) + c, v);
              if (scal) o.adv[tp] = x;
            }
            if (more) {
              if (o.adv_cor) {
                const float y = gs->ecor[i];
                const float4 v = make_float4(y, y, y, y);
                for (int64_t c = qa + hl; c < qb; c += 16) __stcs(reinterpret_cast<float4*>(o.adv_cor) + c, v);
                if (scal) o.adv_cor[tp] = y;
              }
              if (o.adv_eff) {
                const float y = gs->eeff[i];
                const float4 v = make_float4(y, y, y, y);
                for (int64_t c = qa + hl; c < qb; c += 16) __stcs(reinterpret_cast<float4*>(o.adv_eff) + c, v);
                if (scal) o.adv_eff[tp] = y;
              }
              if (o.eff_mask) {
                const uint8_t m = gs->emask[i];
                const uint32_t v = 0x01010101u * m;
                for (int64_t c = qa + hl; c < qb; c += 16) __stcs(reinterpret_cast<uint32_t*>(o.eff_mask) + c, v);
                if (scal) o.eff_mask[tp] = m;
              }
            }
          }
        }
      }
      if (gt == 0) gs->nstat[0] = gs->nstat[1] = 0;  // for the next group
      bar_group();
    }
  }

  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 1) tmem_dealloc(tmem, kTmemCols);
}

size_t fused_smem() { return (size_t)kTilesOff + 1023 + (size_t)kRingBytes; }
