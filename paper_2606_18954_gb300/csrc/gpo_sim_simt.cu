// Cosine-similarity merge on the CUDA cores (fp32 embeddings; also selectable for bf16 to
// cross-check the tensor-core kernel): GraphPO Sec. 4.2, pairs of states of one group that
// are not ancestor-related and have cosine >= kappa are linked.  fp32 fused multiply-add
// accumulation.
//
// One CTA per 64 x 32 tile of a work item (a 128-row block against up to 256 columns: two row
// halves by eight column chunks, fewer where no group has states for them; tiles left of a
// diagonal item's diagonal are empty).  Two
// parts of 64 threads, each half of every stage's k: thread (ti, tj) = (t / 8, t % 8) of a part
// owns the outputs of rows ti + 8 a and columns tj + 8 c (a < 8, c < NC), per four elements of
// k one 16-byte chunk of each of its 8 rows and NC columns and 32 NC fma; the second part's
// sums are added to the first's through shared memory.  Rows are staged as they lie in memory,
// kKc elements at a time (row stride kKc + 4 floats: eight consecutive rows fall in eight
// different 16-byte bank groups), in two buffers filled by cp.async while the other one is
// multiplied.  NC = 2 or 4 column chunks of 8 by the tile's valid columns, so that a group of a
// few states more than a multiple of 32 does not pay whole tiles for them.  The linked pairs of
// a tile are united in shared memory, then one union per non-root state in the batch's label
// forest (ws.lab).
//
// Bound by issue (69 % of the slots while an SM has work, 65 % of the instructions fma):
// 64 groups of 257 states, d = 1024 take 184 us, of which the 2.83 G fma of their upper-triangle
// tiles are 70 us of the fp32 pipe at 2070 MHz.  Before, one CTA of 256 threads per item with scalar loads
// transposed into shared memory: 795 us.  The same tile with 64 threads and whole k, one wave
// of long CTAs: 238 us; with four parts 205 us; packed f32x2 fma 256 us.
#include "gpo_internal.cuh"

namespace gpo {

namespace {

constexpr int kTile = 64, kCols = 32;  // rows and columns of a CTA's tile
constexpr int kPart = 64;              // threads of one part
constexpr int kParts = 2;              // parts: each half of every stage's k
constexpr int kThreads = kParts * kPart;
constexpr int kKc = 32;                // k elements of a stage
constexpr int kLd = kKc + 4;           // row stride in shared memory (floats)
static_assert(kTileM == 2 * kTile && kTileN == 8 * kCols && kTile == 2 * kCols, "tiles of a work item");

struct SimtSmem {
  alignas(16) float A[2][kTile * kLd];
  alignas(16) float B[2][kCols * kLd];
  float rrn[kTile], crn[kCols];        // 1 / |z| of the rows and columns
  int rend[kTile];                     // first comparable column right of the row (state index)
  int rdep[kTile], cdep[kCols];        // depths
  int lp[kTile + kCols];               // label forest of the tile's rows, then columns
};

__device__ __forceinline__ int find_root(const int* p, int x) {
  const volatile int* vp = p;
  while (true) {
    const int y = vp[x];
    if (y == x) return x;
    x = y;
  }
}

// Hook the larger root under the smaller one; parent[x] <= x always holds.
__device__ __forceinline__ void unite(int* p, int a, int b) {
  while (true) {
    a = find_root(p, a);
    b = find_root(p, b);
    if (a == b) return;
    if (a > b) {
      const int t = a;
      a = b;
      b = t;
    }
    if (atomicCAS(&p[b], b, a) == b) return;
  }
}

// 16 bytes from global to shared memory, of which `bytes` are read and the rest zeros.
__device__ __forceinline__ void cp_async16(float* dst, const void* src, int bytes) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_u32(dst)), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int kLeft>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(kLeft) : "memory");
}

// Elements [k0, k0 + kKc) of rows [row0, row0 + nrows) into dst (zeros past d; rows past
// nrows are not written, their outputs are not read).
template <bool kBf16>
__device__ __forceinline__ void stage_rows(float* dst, const void* emb, int64_t stride, int d, int row0, int nrows,
                                           int k0) {
  constexpr int kCh = kKc / 4;  // 16-byte chunks of a staged row
  for (int e = threadIdx.x; e < nrows * kCh; e += kThreads) {
    const int r = e / kCh, k = k0 + 4 * (e % kCh);
    const int valid = max(0, min(4, d - k));
    float* to = dst + r * kLd + 4 * (e % kCh);
    const int64_t at = (int64_t)(row0 + r) * stride + (valid > 0 ? k : 0);
    if (kBf16) {
      const uint16_t* from = reinterpret_cast<const uint16_t*>(emb) + at;
      float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
      if (valid == 4) {  // 8-byte aligned: rows on 16 bytes, k a multiple of 4
        const uint2 w = *reinterpret_cast<const uint2*>(from);
        v = make_float4(__uint_as_float(w.x << 16), __uint_as_float(w.x & 0xFFFF0000u), __uint_as_float(w.y << 16),
                        __uint_as_float(w.y & 0xFFFF0000u));
      } else if (valid > 0) {
        v.x = __uint_as_float((uint32_t)from[0] << 16);
        if (valid > 1) v.y = __uint_as_float((uint32_t)from[1] << 16);
        if (valid > 2) v.z = __uint_as_float((uint32_t)from[2] << 16);
      }
      *reinterpret_cast<float4*>(to) = v;
    } else {
      cp_async16(to, reinterpret_cast<const float*>(emb) + at, 4 * valid);
    }
  }
}

// The tile's products (8 NC columns), pair test and links in sm.lp.
template <bool kBf16, int NC>
__device__ __forceinline__ void tile_links(SimtSmem& sm, const gpo_batch& b, const Sizes& sz, int row0, int nr,
                                           int col0, int nc, float kappa, int rule) {
  const int t = threadIdx.x % kPart, part = threadIdx.x / kPart, ti = t >> 3, tj = t & 7;
  const int cr = col0 - row0;                    // columns that are rows of the tile too
  const bool shared = cr + nc <= nr;             // are read from A
  float acc[8][NC];
#pragma unroll
  for (int a = 0; a < 8; ++a)
#pragma unroll
    for (int c = 0; c < NC; ++c) acc[a][c] = 0.f;
  auto stage = [&](int k0, int buf) {
    stage_rows<kBf16>(sm.A[buf], b.emb, sz.stride, sz.d, row0, nr, k0);
    if (!shared) stage_rows<kBf16>(sm.B[buf], b.emb, sz.stride, sz.d, col0, nc, k0);
    cp_async_commit();
  };
  const int nk = (sz.d + kKc - 1) / kKc;
  stage(0, 0);
#pragma unroll 1
  for (int s = 0; s < nk; ++s) {
    const int buf = s & 1;
    if (s + 1 < nk) stage((s + 1) * kKc, buf ^ 1);
    else cp_async_commit();  // (an empty group, so that the wait below always leaves one)
    cp_async_wait<1>();
    __syncthreads();
    const int kp = part * (kKc / kParts);
    const float* A = sm.A[buf] + ti * kLd + kp;
    const float* B = (shared ? sm.A[buf] + cr * kLd : sm.B[buf]) + tj * kLd + kp;
#pragma unroll 1
    for (int k = 0; k < kKc / kParts; k += 4) {
      float4 x[8], y[NC];
#pragma unroll
      for (int a = 0; a < 8; ++a) x[a] = *reinterpret_cast<const float4*>(A + 8 * a * kLd + k);
#pragma unroll
      for (int c = 0; c < NC; ++c) y[c] = *reinterpret_cast<const float4*>(B + 8 * c * kLd + k);
#pragma unroll
      for (int a = 0; a < 8; ++a)
#pragma unroll
        for (int c = 0; c < NC; ++c) {
          float s4 = acc[a][c];
          s4 = fmaf(x[a].x, y[c].x, s4);
          s4 = fmaf(x[a].y, y[c].y, s4);
          s4 = fmaf(x[a].z, y[c].z, s4);
          s4 = fmaf(x[a].w, y[c].w, s4);
          acc[a][c] = s4;
        }
    }
    __syncthreads();  // the buffer is refilled two stages on
  }
  // the other parts' sums, added to the first's in part order
  float* ps = &sm.A[0][0];
  static_assert(sizeof(sm.A) >= sizeof(float) * 8 * 4 * kPart * (kParts - 1), "partial sums");
  if (part > 0) {
#pragma unroll
    for (int a = 0; a < 8; ++a)
#pragma unroll
      for (int c = 0; c < NC; ++c) ps[(((part - 1) * 8 + a) * NC + c) * kPart + t] = acc[a][c];
  }
  __syncthreads();
  if (part > 0) return;
#pragma unroll
  for (int q = 0; q < kParts - 1; ++q)
#pragma unroll
    for (int a = 0; a < 8; ++a)
#pragma unroll
      for (int c = 0; c < NC; ++c) acc[a][c] += ps[((q * 8 + a) * NC + c) * kPart + t];
#pragma unroll
  for (int a = 0; a < 8; ++a) {
    const int r = ti + 8 * a;
    if (r >= nr) continue;
    const float rn = sm.rrn[r];
    const int re = sm.rend[r], di = sm.rdep[r];
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      const int q = tj + 8 * c;
      // comparable: right of the row and past its own rollout (tree layout: its subtree)
      if (q >= nc || col0 + q < re) continue;
      if (rule == GPO_MERGE_SAME_DEPTH && sm.cdep[q] != di) continue;
      if (acc[a][c] * rn * sm.crn[q] >= kappa) unite(sm.lp, r, cr + q < kTile ? cr + q : kTile + q);
    }
  }
}

template <bool kBf16>
__global__ void __launch_bounds__(kThreads)
    sim_simt_kernel(gpo_batch b, Sizes sz, Ws ws, float kappa, int rule, int first) {
  extern __shared__ __align__(16) unsigned char simt_smem[];
  SimtSmem& sm = *reinterpret_cast<SimtSmem*>(simt_smem);
  const Status st{ws.status, ws.tag};
  const int it = first + (int)blockIdx.z;
  const int nitems = (int)*((volatile uint32_t*)&st.p[kStItems]);
  if (nitems < 0 && it == first) plan_fault(st);
  if (it >= nitems || aborted(st)) return;
  const Item item = ws.items[it];
  const GroupInfo gi = ws.groups[item.group];
  const int send = gi.s0 + gi.n;
  const int row0 = item.row0 + kTile * (int)blockIdx.x, col0 = item.col0 + kCols * (int)blockIdx.y;
  const int nr = min(kTile, send - row0), nc = min(kCols, item.col0 + item.ncols - col0);
  if (nr <= 0 || nc <= 0 || col0 < row0) return;
  const bool tree = ws.tree_end != nullptr;
  {
    const int x = threadIdx.x;
    static_assert(kThreads >= kTile, "one row per thread");
    if (x < kTile) sm.lp[x] = x;
    if (x < nr) {
      const int2 mt = ws.state_meta[row0 + x];
      sm.rrn[x] = ws.rn[row0 + x];
      sm.rdep[x] = mt.y;
      sm.rend[x] = tree ? ws.tree_end[row0 + x] : b.rollout_step_off[mt.x + 1];
    }
    if (x < kCols) {
      sm.lp[kTile + x] = kTile + x;
      if (x < nc) {
        sm.crn[x] = ws.rn[col0 + x];
        sm.cdep[x] = ws.state_meta[col0 + x].y;
      }
    }
  }
  if (nc > 16) tile_links<kBf16, 4>(sm, b, sz, row0, nr, col0, nc, kappa, rule);
  else tile_links<kBf16, 2>(sm, b, sz, row0, nr, col0, nc, kappa, rule);
  __syncthreads();
  // (a column that is a row of the tile has the row's slot)
  for (int x = threadIdx.x; x < kTile + kCols; x += kThreads) {
    const int root = find_root(sm.lp, x);
    if (root == x) continue;
    const int v = x < kTile ? row0 + x : col0 + (x - kTile);
    const int u = root < kTile ? row0 + root : col0 + (root - kTile);
    if (GPO_BOUNDS(st, v, sz.N, kWhereEdges) && GPO_BOUNDS(st, u, sz.N, kWhereEdges)) unite(ws.lab, u, v);
  }
}

}  // namespace

cudaError_t setup_sim_simt() {
  cudaError_t e = cudaFuncSetAttribute(sim_simt_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)sizeof(SimtSmem));
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(sim_simt_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)sizeof(SimtSmem));
  return e;
}

cudaError_t launch_sim_simt(const LaunchCtx& lc, const gpo_batch& b, const Sizes& sz, const Ws& ws,
                            const Params& p) {
  if (ws.max_items < 1) return cudaSuccess;
  // A block per tile that some group has states for (row halves x column chunks x items): with all
  // 16 the blocks of the others, which end at once, were most of the time of small groups (16384
  // branching groups of at most 6 states 817 -> 119 us, 2048 of 12 111 -> 25 us; the same as one
  // dimension, with divisions by halves and chunks, costs 4 groups of 257 states 28.3 -> 30.3 us).
  // As many launches as the grid's third dimension asks for (the debug build has a limit that
  // its tests pass).
#ifdef GPO_DEBUG
  constexpr int kItems = 8;
#else
  constexpr int kItems = 65535;
#endif
  const unsigned halves = sz.maxn > kTile ? 2 : 1, chunks = (unsigned)min(kTileN, sz.maxn + kCols - 1) / kCols;
  for (int first = 0; first < ws.max_items; first += kItems) {
    const dim3 grid(halves, chunks, (unsigned)min(ws.max_items - first, kItems));
    if (b.emb_dtype == GPO_EMB_BF16)
      sim_simt_kernel<true><<<grid, kThreads, sizeof(SimtSmem), lc.stream>>>(b, sz, ws, (float)p.kappa, p.rule, first);
    else
      sim_simt_kernel<false><<<grid, kThreads, sizeof(SimtSmem), lc.stream>>>(b, sz, ws, (float)p.kappa, p.rule, first);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace gpo
