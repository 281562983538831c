// Many small graphs prepared together: Algorithm 1 lines 1-4 (graph,
// max/min pivots, d_ip, regions and counts, PivotMDS and the rescale) for a
// whole batch of independent layouts, feeding ssm_batch_iterate.
//
// Graphs are handed out largest first from an atomic counter.  k_prep_pivots,
// a block per graph, builds the CSR (degrees, scatter, rows sorted and
// deduplicated by one thread each, long ones by a warp), then runs the searches
// of max/min sp in shared memory; the running minimum names the regions, whose eccentricities
// and the count-table length close the launch.  k_prep_dist searches from the
// pivots, 32 of a graph at a time.  The host reads the lengths once for the
// whole batch and places the tables.  k_prep_gram forms the exact integer
// Gram matrices Delta^T Delta of the squared distances; k_prep_layout, a block
// per graph, fills the cumulative counts, forms the FP64 matrix
// B = 1/4 J (G - s s^T / n) J and its top two eigenpairs (Householder
// reduction, bisection, inverse iteration), projects, signs and rescales the
// layout.  Sums are of whole numbers or in a fixed order: results do not
// depend on timing.
#include <algorithm>
#include <vector>

#include "block_search.cuh"
#include "common.cuh"

namespace ssm {

constexpr int kPrepMaxN = 12288;
constexpr int kPrepMaxK = 100;
constexpr int kPrepThreads = 512;
constexpr int kPrepShortRow = 48;
constexpr int kDistThreads = 1024;
constexpr int kDistMany = 8;  // nodes of a warp in a level above which the next level looks through all chunks

struct PrepDev {
  int32_t n, k;
  int64_t m_in, edge_off;
  int64_t node_off, row_off, col_off, piv_off, dip_off, cnt_off_off;
};

struct PrepArgs {
  int32_t G;
  const PrepDev *desc;
  const int32_t *order;
  const int32_t *src, *dst;
  int32_t *tmp;  // 2 m_in words per graph at col_off: 16-bit neighbours, as scattered, then compact rows
  int32_t *rowptr, *colidx, *pivots, *region;
  uint16_t *dip;
  int32_t *ecc;        // [sum k]
  int64_t *lens;       // [G] count-table lengths
  int64_t *medges;     // [G] edges after deduplication
  int64_t ubytes, dbytes;  // dynamic shared memory of the two kernels
  unsigned *ctr;       // tasks handed out: pivots, layout, distances
  int32_t *status;
};

// shared memory of a graph's searches from its pivots, without its neighbour lists
__host__ __device__ constexpr int64_t dist_node_bytes(int64_t n) { return 12 * n + 4 * (n + 1) + (n + 31) / 32 * 64; }

// exclusive block scan of a[0..len) in place, total returned; s_part holds a
// word per warp and one more
__device__ int block_exclusive_scan(int *a, int len, int *s_part) {
  const int per = (len + kPrepThreads - 1) / kPrepThreads;
  const int b = threadIdx.x * per, e = min(len, b + per);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int t = 0;
  for (int i = b; i < e; ++i) t += a[i];
  int inc = t;
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += y;
  }
  if (lane == 31) s_part[warp] = inc;
  __syncthreads();
  if (warp == 0) {
    const int v = lane < kPrepThreads / 32 ? s_part[lane] : 0;
    int w = v;
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, w, o);
      if (lane >= o) w += y;
    }
    if (lane < kPrepThreads / 32) s_part[lane] = w - v;
    if (lane == 31) s_part[kPrepThreads / 32] = w;
  }
  __syncthreads();
  int acc = s_part[warp] + inc - t;
  for (int i = b; i < e; ++i) {
    const int v = a[i];
    a[i] = acc;
    acc += v;
  }
  const int total = s_part[kPrepThreads / 32];
  __syncthreads();
  return total;
}

// the rows of more than kPrepShortRow entries sorted and deduplicated, their new
// lengths in key: a warp per row, a bit per neighbour in the warp's part of `bits`
// (2 n + 64 bytes for 16 warps)
__device__ __noinline__ void sort_long_rows(int n, const int *off, uint16_t *col, int *key, unsigned *bits) {
  const int lane = threadIdx.x & 31, words = (n + 31) / 32;
  bits += (threadIdx.x >> 5) * words;
  for (int i0 = 32 * (threadIdx.x >> 5); i0 < n; i0 += blockDim.x) {
    const int il = min(i0 + lane, n - 1);
    for (unsigned m = __ballot_sync(0xffffffffu, i0 + lane < n && off[il + 1] - off[il] > kPrepShortRow); m; m &= m - 1u) {
      const int i = i0 + __ffs(m) - 1, len = off[i + 1] - off[i];
      uint16_t *row = col + off[i];
      for (int w = lane; w < words; w += 32) bits[w] = 0u;
      __syncwarp();
      for (int a = lane; a < len; a += 32) atomicOr(bits + (row[a] >> 5), 1u << (row[a] & 31));
      __syncwarp();
      const int per = (words + 31) / 32, w0 = min(words, lane * per), w1 = min(words, w0 + per);
      int c = 0;
      for (int w = w0; w < w1; ++w) c += __popc(bits[w]);
      int inc = c;
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
      }
      int u = inc - c;
      for (int w = w0; w < w1; ++w)
        for (unsigned b = bits[w]; b; b &= b - 1u) row[u++] = (uint16_t)(32 * w + __ffs(b) - 1);
      if (lane == 31) key[i] = inc;
      __syncwarp();
    }
  }
}

// CSR, max/min pivots, regions, eccentricities and table lengths of one graph
// per block.  The searches are chains of short levels (10 to 30 nodes wide
// after the first few pivots): block_search, the offsets in shared memory and
// the neighbours too where they fit.  512 graphs of 64 to 8192 nodes, k = 100: a
// batch takes as long as its largest graph (1,700 levels), 1.53 ms; with a lane
// per node, neighbours in global memory and a queue atomic per node a level
// took 4,500 cycles, and the searches below were part of the same block: 18.4 ms.
__global__ void __launch_bounds__(kPrepThreads) k_prep_pivots(PrepArgs A) {
  extern __shared__ __align__(16) unsigned char psm[];
  __shared__ int s_part[kPrepThreads / 32 + 1], s_ecc[kPrepMaxK];
  __shared__ int s_task, s_len[3], s_hub[kBsMaxHubs];
  __shared__ unsigned s_key[2];
  const int lane = threadIdx.x & 31;
  for (;;) {
    if (threadIdx.x == 0) s_task = (int)atomicAdd(A.ctr, 1u);
    __syncthreads();
    const int task = s_task;
    __syncthreads();
    if (task >= A.G) break;
    const int gi = A.order[task];
    const PrepDev D = A.desc[gi];
    const int n = D.n, k = D.k;
    const int32_t *src = A.src + D.edge_off, *dst = A.dst + D.edge_off;
    int32_t *rowptr = A.rowptr + D.row_off;
    int32_t *colidx = A.colidx + D.col_off;
    int *key = reinterpret_cast<int *>(psm);                // [n + 1] degrees and cursors, then (distance, pivot)
    int *off = key + (n + 1);                               // [n + 1] row offsets
    uint16_t *qa = reinterpret_cast<uint16_t *>(off + (n + 1));  // [n] queues
    uint16_t *qb = qa + n;                                  // [n]
    // neighbours as 16-bit numbers, rows at off[]; then the rows without
    // duplicates and gaps, for the searches from the pivots
    uint16_t *const tmp = reinterpret_cast<uint16_t *>(A.tmp + D.col_off);
    uint16_t *const packed = tmp + 2 * D.m_in;
    uint16_t *const col = block_search_bytes(n) + 4 * D.m_in <= A.ubytes ? qb + n : tmp;
    // ---- CSR: degrees, scatter, rows sorted and deduplicated
    for (int i = threadIdx.x; i <= n; i += blockDim.x) off[i] = 0;
    __syncthreads();
    for (int64_t e = threadIdx.x; e < D.m_in; e += blockDim.x) {
      const int u = src[e], v = dst[e];
      if (u < 0 || u >= n || v < 0 || v >= n) {
        dev_fail(A.status, SSM_E_GRAPH);
        continue;
      }
      if (u == v) continue;
      atomicAdd(off + u, 1);
      atomicAdd(off + v, 1);
    }
    __syncthreads();
    block_exclusive_scan(off, n + 1, s_part);
    for (int i = threadIdx.x; i <= n; i += blockDim.x) key[i] = off[i];  // cursors
    __syncthreads();
    for (int64_t e = threadIdx.x; e < D.m_in; e += blockDim.x) {
      const int u = src[e], v = dst[e];
      if (u < 0 || u >= n || v < 0 || v >= n || u == v) continue;
      col[atomicAdd(key + u, 1)] = (uint16_t)v;
      col[atomicAdd(key + v, 1)] = (uint16_t)u;
    }
    __syncthreads();
    // rows up to kPrepShortRow: insertion sort by one thread; longer ones: a bit
    // per neighbour, by one warp, the bits in the queues' memory (of 32 nodes or
    // fewer: in a register).  A star of 12,288 nodes by insertion: 60 to 95 ms, as
    // the scatter happens to order the row; now 0.5 with the rest of this kernel
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
      uint16_t *row = col + off[i];
      const int len = off[i + 1] - off[i];
      if (n > 32 && len > kPrepShortRow) continue;
      if (n <= 32) {
        unsigned bits = 0u;
        for (int a = 0; a < len; ++a) bits |= 1u << row[a];
        int u = 0;
        for (; bits; bits &= bits - 1u) row[u++] = (uint16_t)(__ffs(bits) - 1);
        key[i] = u;
        continue;
      }
      for (int a = 1; a < len; ++a) {
        const uint16_t x = row[a];
        int b = a - 1;
        while (b >= 0 && row[b] > x) {
          row[b + 1] = row[b];
          --b;
        }
        row[b + 1] = x;
      }
      int u = 0;
      for (int a = 0; a < len; ++a) {
        const uint16_t x = row[a];
        if (u == 0 || row[u - 1] != x) row[u++] = x;
      }
      key[i] = u;
    }
    if (n > 32) sort_long_rows(n, off, col, key, reinterpret_cast<unsigned *>(qa));
    if (threadIdx.x == 0) key[n] = 0;
    __syncthreads();
    const int m2 = block_exclusive_scan(key, n + 1, s_part);
    for (int i = threadIdx.x; i <= n; i += blockDim.x) rowptr[i] = key[i];
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
      const uint16_t *row = col + off[i];
      const int o = key[i], len = key[i + 1] - o;
      for (int a = 0; a < len; ++a) {
        const uint16_t x = row[a];
        colidx[o + a] = x;
        packed[o + a] = x;
      }
    }
    if (threadIdx.x == 0) A.medges[gi] = m2 / 2;
    __syncthreads();
    // ---- max/min sp (start node 0): each search lowers the running minimum
    // in place and only continues from nodes the new pivot is strictly
    // closer to (the minimum is 1-Lipschitz along edges, so nothing beyond
    // them can change); the first search reaches everything.  A node's key is
    // distance * 128 + pivot: only a strictly smaller distance lowers it, so
    // that at the end it names the region (ties to the lowest pivot index).
    const bool gaps = m2 != off[n];
    if (gaps) {  // the compact rows instead
      __syncthreads();
      for (int i = threadIdx.x; i <= n; i += blockDim.x) off[i] = key[i];
      if (col != tmp)
        for (int t = threadIdx.x; t < m2; t += blockDim.x) col[t] = packed[t];
    }
    const uint16_t *const nbr = gaps && col == tmp ? packed : col;
    __syncthreads();
    for (int i = threadIdx.x; i < n; i += blockDim.x) key[i] = kBsInf;
    if (threadIdx.x < 3) s_len[threadIdx.x] = 0;
    if (threadIdx.x < 2) s_key[threadIdx.x] = 0u;
    __syncthreads();
    const BlockSearch B{key, off, nbr, qa, qb, s_len, s_hub};
    const bool hubs = block_search_hubs(off, n);
    int slot = 0;
    for (int a = 0; a < k; ++a) {
      int p = 0;
      if (a > 0) {
        unsigned best = 0u;
        for (int i = threadIdx.x; i < n; i += blockDim.x)
          best = max(best, ((unsigned)(key[i] >> 7) << 16) | (0xFFFFu - (unsigned)i));
        best = __reduce_max_sync(0xffffffffu, best);
        if (lane == 0) atomicMax(s_key + (a & 1), best);
        __syncthreads();
        p = (int)(0xFFFFu - (s_key[a & 1] & 0xFFFFu));
      }
      if (threadIdx.x == 0) {
        A.pivots[D.piv_off + a] = p;
        s_key[(a + 1) & 1] = 0u;
      }
      if (hubs) block_search<true>(B, p, 7, a, slot);
      else block_search<false>(B, p, 7, a, slot);
      if (a == 0)
        for (int i = threadIdx.x; i < n; i += blockDim.x)
          if (key[i] == kBsInf) dev_fail(A.status, SSM_E_DISCONNECTED);
    }
    // ---- regions and eccentricities
    for (int a = threadIdx.x; a < k; a += blockDim.x) s_ecc[a] = 0;
    __syncthreads();
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
      const int c = key[i] == kBsInf ? 0 : key[i];  // (the status then refuses the batch)
      A.region[D.node_off + i] = c & 127;
      atomicMax(s_ecc + (c & 127), c >> 7);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      int64_t len = 0;
      for (int a = 0; a < k; ++a) {
        A.ecc[D.piv_off + a] = s_ecc[a];
        len += s_ecc[a] + 1;
      }
      A.lens[gi] = len;
    }
    __syncthreads();
  }
}

// d_ip: breadth-first searches from up to 32 pivots of one graph at once, a
// bit per pivot in a node's words.  The unit of work is (graph, word of
// pivots), so that a large graph's searches run on several SMs: as one block's
// work they were the longest chain of a batch.  A level takes two barriers.
// First every warp looks through those of its nodes' chunks (of 32, dealt out in
// turn) that are marked for bits that came in, moves them to `reach` and lists
// the nodes; then four lanes per listed node store its distances, pass the bits on
// to neighbours that do not have them (shared-memory reductions that return
// nothing) and mark their chunks, or, in a warp with many nodes, all chunks.  The
// work of a level is the nodes that changed, so that long thin graphs pay for
// their two or three nodes per level (path of 12,288 nodes, k = 100: 15 ms, with a
// look through all chunks in every level 21).
// 1.7 ms for the batch at k_prep_pivots, 2.3 with 512 threads; a queue of single
// (pivot, node) pairs in global memory took 18 M cycles (9 ms) of the largest
// graph's block alone.
__global__ void __launch_bounds__(kDistThreads) k_prep_dist(PrepArgs A) {
  extern __shared__ __align__(16) unsigned char psm[];
  __shared__ int s_task;
  __shared__ unsigned s_mark[(kPrepMaxN + 1023) / 1024];  // bit w of word j: chunk 32 j + w, warp w's j-th
  __shared__ int s_all[2];                                 // all of them, by parity of the level
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, sub = threadIdx.x & 3;
  constexpr int kMarks = (kPrepMaxN + 1023) / 1024;
  static_assert(kDistThreads == 1024 && kMarks <= 32, "a chunk's bit is its warp's");
  constexpr int kWarps = kDistThreads / 32, kWords = (kPrepMaxK + 31) / 32;
  for (;;) {
    if (threadIdx.x == 0) s_task = (int)atomicAdd(A.ctr + 2, 1u);
    __syncthreads();
    const int task = s_task;
    __syncthreads();
    if (task >= A.G * kWords) break;
    const int gi = A.order[task / kWords], word = task % kWords;
    const PrepDev D = A.desc[gi];
    const int n = D.n, k = min(32, D.k - 32 * word);
    if (k <= 0) continue;
    unsigned *reach = reinterpret_cast<unsigned *>(psm);  // [n] bits that have come in
    unsigned *nxt = reach + n;                            // [n] bits of the next level
    unsigned *cur = nxt + n;                              // [n] bits of this level
    int *off = reinterpret_cast<int *>(cur + n);          // [n + 1]
    uint16_t *list = reinterpret_cast<uint16_t *>(off + n + 1);  // [(n + 31) / 32 * 32] each warp's nodes of a level
    const int chunks = (n + 31) / 32;
    const uint16_t *packed = reinterpret_cast<const uint16_t *>(A.tmp + D.col_off) + 2 * D.m_in;
    const int32_t *rowptr = A.rowptr + D.row_off;
    const int m2 = rowptr[n];
    const bool fits = dist_node_bytes(n) + 2 * (int64_t)m2 <= A.dbytes;
    uint16_t *col = list + chunks * 32;
    for (int i = threadIdx.x; i < n; i += kDistThreads) {
      reach[i] = 0u;
      nxt[i] = 0u;
    }
    for (int i = threadIdx.x; i <= n; i += kDistThreads) off[i] = rowptr[i];
    if (fits)
      for (int t = threadIdx.x; t < m2; t += kDistThreads) col[t] = packed[t];
    const uint16_t *const nbr = fits ? col : packed;
    if (threadIdx.x < kMarks) s_mark[threadIdx.x] = 0u;
    if (threadIdx.x < 2) s_all[threadIdx.x] = 0;
    __syncthreads();
    auto mark = [&](int u) {
      unsigned *m = s_mark + (u >> 10);
      const unsigned bit = 1u << ((u >> 5) & 31);
      if (!(*reinterpret_cast<volatile unsigned *>(m) & bit)) atomicOr(m, bit);
    };
    if (threadIdx.x < k) {
      const int p = A.pivots[D.piv_off + 32 * word + threadIdx.x];
      atomicOr(nxt + p, 1u << threadIdx.x);
      mark(p);
    }
    // a warp's part of the list: as many places as it has nodes
    uint16_t *const mine = list + 32 * ((chunks / kWarps) * warp + min(warp, chunks % kWarps));
    uint16_t *const dip = A.dip + D.dip_off + (int64_t)(32 * word) * n;
    for (int level = 0;; ++level) {
      __syncthreads();
      int cnt = 0;
      const bool marked = lane < kMarks && (s_mark[lane] >> warp & 1u);
      if (marked) atomicAnd(s_mark + lane, ~(1u << warp));
      auto take = [&](int c) {
        const int i = 32 * c + lane;
        const unsigned in = i < n ? nxt[i] : 0u;
        const unsigned m = __ballot_sync(0xffffffffu, in != 0u);
        if (in) {
          nxt[i] = 0u;
          cur[i] = in;
          reach[i] |= in;
          mine[cnt + __popc(m & ((1u << lane) - 1u))] = (uint16_t)i;
        }
        cnt += __popc(m);
      };
      if (s_all[level & 1]) {
        for (int c = warp; c < chunks; c += kWarps) take(c);
      } else {
        for (unsigned b = __ballot_sync(0xffffffffu, marked); b; b &= b - 1u) take(32 * (__ffs(b) - 1) + warp);
      }
      if (!__syncthreads_or(cnt)) break;
      if (threadIdx.x == 0) s_all[level & 1] = 0;
      const bool many = cnt > kDistMany;
      if (many && lane == 0) s_all[(level + 1) & 1] = 1;
      for (int t0 = 0; t0 < cnt; t0 += 8) {
        const int t = t0 + (lane >> 2);
        if (t >= cnt) continue;
        const int v = mine[t];
        const unsigned bits = cur[v];
        const int e = off[v + 1];
        for (int j = off[v] + sub; j < e; j += 4) {
          const int u = nbr[j];
          const unsigned add = bits & ~reach[u];
          if (add) {
            atomicOr(nxt + u, add);
            if (!many) mark(u);
          }
        }
        for (unsigned b = bits & (0x11111111u << sub); b; b &= b - 1u)
          dip[(int64_t)(__ffs(b) - 1) * n + v] = (uint16_t)level;
      }
    }
  }
}

// ------------------------------------------------------------------ layout
struct LayoutDev {
  int32_t n, k;
  int64_t m;
  int64_t node_off, row_off, col_off, piv_off, dip_off, cnt_off_off, cnt_base;
  int64_t gram_off;  // words
};

struct LayoutArgs {
  int32_t G;
  const LayoutDev *desc;
  const int32_t *order, *task0;  // task0 [G + 1]: first Gram task by place in the order
  const int32_t *rowptr, *colidx, *region, *ecc;
  const uint16_t *dip;
  unsigned long long *gram;  // per graph: column sums [k], then 32-bit parts (low, high) of the sums per pair
  int32_t *cnt_off;
  uint32_t *cnt;
  float2 *pos;
  double *eig;  // [2 G] or null
  unsigned *ctr;
  int32_t *status;
};

static int64_t gram_words(int64_t k) { return k + 2 * k * k; }

// The exact Gram matrix Delta^T Delta of the squared distances, over the whole
// GPU: the unit of work is kGramNodes nodes of one graph, so that one large
// graph's products are spread over the SMs (as part of the graph's own block
// they were 4.6 M cycles of the longest chain of a batch).  A thread owns an
// 8 x 8 tile of pivot pairs (91 tiles of the upper triangle at k = 100) in 64
// registers pairs: per node 4 loads of 16 bytes and 64 multiply-adds of 32 x 32
// bits, which bound it (0.9 ms for 512 graphs of 64 to 8192 nodes, 5 G
// products).  A unit's sums (512 products below 2^55) are exact in
// 64 bits; their 32-bit halves are added to the graph's sums by atomics, whole
// numbers, so the order does not show.
constexpr int kGramNodes = 512, kGramStage = 32, kGramThreads = 96, kGramLd = (kPrepMaxK + 7) / 8 * 8;
__global__ void __launch_bounds__(kGramThreads) k_prep_gram(LayoutArgs L) {
  __shared__ __align__(16) uint32_t st[kGramStage][kGramLd];
  // this block's graph: the last place in the order whose tasks start here or before
  int lo = 0, hi = L.G;
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (L.task0[mid] <= (int)blockIdx.x) lo = mid; else hi = mid;
  }
  const LayoutDev D = L.desc[L.order[lo]];
  const int n = D.n, k = D.k, T = (k + 7) / 8, k8 = 8 * T;
  const int n0 = ((int)blockIdx.x - L.task0[lo]) * kGramNodes, n1 = min(n, n0 + kGramNodes);
  const uint16_t *dip = L.dip + D.dip_off;
  unsigned long long *sums = L.gram + D.gram_off;
  int ta = -1, tb = 0;
  if ((int)threadIdx.x < T * (T + 1) / 2) {
    int p = threadIdx.x;
    for (ta = 0; p >= T - ta; ++ta) p -= T - ta;
    tb = ta + p;
  }
  unsigned long long acc[8][8];
#pragma unroll
  for (int x = 0; x < 8; ++x)
#pragma unroll
    for (int y = 0; y < 8; ++y) acc[x][y] = 0ull;
  unsigned long long cs[(kGramLd + kGramThreads - 1) / kGramThreads] = {};
  for (int i0 = n0; i0 < n1; i0 += kGramStage) {
    __syncthreads();
    for (int e = threadIdx.x; e < k8 * kGramStage; e += kGramThreads) {
      const int a = e / kGramStage, t = e % kGramStage;
      const uint32_t d = a < k && i0 + t < n1 ? dip[(int64_t)a * n + i0 + t] : 0u;
      st[t][a] = d * d;
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < (kGramLd + kGramThreads - 1) / kGramThreads; ++q) {
      const int a = threadIdx.x + q * kGramThreads;
      if (a < k8)
        for (int t = 0; t < kGramStage; ++t) cs[q] += st[t][a];
    }
    if (ta < 0) continue;
#pragma unroll 1
    for (int t = 0; t < kGramStage; ++t) {
      uint32_t va[8], vb[8];
      *reinterpret_cast<uint4 *>(va) = *reinterpret_cast<const uint4 *>(&st[t][8 * ta]);
      *reinterpret_cast<uint4 *>(va + 4) = *reinterpret_cast<const uint4 *>(&st[t][8 * ta + 4]);
      *reinterpret_cast<uint4 *>(vb) = *reinterpret_cast<const uint4 *>(&st[t][8 * tb]);
      *reinterpret_cast<uint4 *>(vb + 4) = *reinterpret_cast<const uint4 *>(&st[t][8 * tb + 4]);
#pragma unroll
      for (int x = 0; x < 8; ++x)
#pragma unroll
        for (int y = 0; y < 8; ++y) acc[x][y] += (unsigned long long)va[x] * vb[y];
    }
  }
#pragma unroll
  for (int q = 0; q < (kGramLd + kGramThreads - 1) / kGramThreads; ++q) {
    const int a = threadIdx.x + q * kGramThreads;
    if (a < k) atomicAdd(sums + a, cs[q]);
  }
  if (ta < 0) return;
#pragma unroll
  for (int x = 0; x < 8; ++x)
#pragma unroll
    for (int y = 0; y < 8; ++y) {
      const int a = 8 * ta + x, b = 8 * tb + y;
      if (a > b || b >= k) continue;
      unsigned long long *o = sums + k + 2 * ((int64_t)a * k + b);
      atomicAdd(o, acc[x][y] & 0xFFFFFFFFull);
      if (acc[x][y] >> 32) atomicAdd(o + 1, acc[x][y] >> 32);
    }
}

// fixed-order block sum of one double per thread
__device__ double block_sum_d(double v, double *s_red) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) s_red[threadIdx.x >> 5] = v;
  __syncthreads();
  double t = 0.0;
  for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += s_red[w];
  __syncthreads();
  return t;
}
__device__ __forceinline__ double warp_sum_d(double v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// 1 / sqrt(s) for a normal s > 0, from FP32's reciprocal square root by two
// Newton steps (2^-22 -> 2^-43 -> FP64 rounding); the exponent is halved apart
__device__ __forceinline__ double rsqrt_newton(double s) {
  const int h = (__double2hiint(s) >> 21) - 511;  // half the exponent (of 2^0: 0)
  const double t = __hiloint2double(__double2hiint(s) - (h << 21), __double2loint(s));  // in [1/2, 2)
  double y = (double)rsqrtf((float)t);
  y = fma(0.5 * y, fma(-t * y, y, 1.0), y);
  y = fma(0.5 * y, fma(-t * y, y, 1.0), y);
  return __hiloint2double(__double2hiint(y) - (h << 20), __double2loint(y));
}

// PivotMDS and the rescale of one graph per block.  FP64 runs at a 64th of
// FP32's rate here and a dependent step takes 60 cycles or more, so the
// eigen-solve is a chain of FP64 latencies: the matrix holds the reflectors
// in the rows it no longer needs (81 KB, two blocks per SM fill each other's
// gaps), only a triangle is updated, four threads share a row of a product,
// square roots are two Newton steps, loops over k are a warp's, and the node
// loop of the projection is integer arithmetic.  2.5 ms for 512 graphs of 64 to
// 8192 nodes, k = 100 (with the Gram and an FP64 projection in the block, one
// block per SM and single-thread loops over k: 6.5 ms).
constexpr int kLayLd = kPrepMaxK + 1;  // odd: columns and rows without bank conflicts
__global__ void __launch_bounds__(kPrepThreads, 2) k_prep_layout(LayoutArgs L) {
  extern __shared__ __align__(16) unsigned char lsm[];
  double *Am = reinterpret_cast<double *>(lsm);  // [kPrepMaxK][kLayLd]
  __shared__ double s_red[kPrepThreads / 32];
  __shared__ double s_rm[kPrepMaxK], s_gm;
  __shared__ int s_off[kPrepMaxK + 1];
  __shared__ double s_dg[kPrepMaxK], s_e[kPrepMaxK], s_p[4][kPrepMaxK], s_w[kPrepMaxK], s_lam[2];
  __shared__ double s_y[2][kPrepMaxK], s_fd[2][kPrepMaxK], s_fu[2][kPrepMaxK], s_fu2[2][kPrepMaxK], s_fl[2][kPrepMaxK];
  __shared__ double s_e2[kPrepMaxK];
  __shared__ int s_piv[2][kPrepMaxK];
  __shared__ int s_task;
  __shared__ double s_sig[2], s_kap[2];
  __shared__ int4 s_fix[kPrepMaxK];  // (low, high) parts of an eigenvector pair's entries in fixed point
  __shared__ int s_done;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  constexpr int kWarps = kPrepThreads / 32;
  for (;;) {
    if (threadIdx.x == 0) s_task = (int)atomicAdd(L.ctr, 1u);
    __syncthreads();
    const int task = s_task;
    __syncthreads();
    if (task >= L.G) break;
    const int gi = L.order[task];
    const LayoutDev D = L.desc[gi];
    const int n = D.n, k = D.k;
    const uint16_t *dip = L.dip + D.dip_off;
    const int32_t *region = L.region + D.node_off;
    const int32_t *ecc = L.ecc + D.piv_off;
    // ---- Section 3's counts: cnt_off, histograms, prefix sums
    if (threadIdx.x == 0) {
      int acc = 0;
      for (int a = 0; a < k; ++a) {
        s_off[a] = acc;
        acc += ecc[a] + 1;
      }
      s_off[k] = acc;
    }
    __syncthreads();
    uint32_t *cnt = L.cnt + D.cnt_base;
    for (int a = threadIdx.x; a <= k; a += blockDim.x) L.cnt_off[D.cnt_off_off + a] = s_off[a];
    for (int t = threadIdx.x; t < s_off[k]; t += blockDim.x) cnt[t] = 0u;
    __syncthreads();
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
      const int a = region[i];
      atomicAdd(cnt + s_off[a] + dip[(int64_t)a * n + i], 1u);
    }
    __syncthreads();
    for (int a = threadIdx.x; a < k; a += blockDim.x) {
      uint32_t acc = 0;
      for (int t = s_off[a]; t < s_off[a + 1]; ++t) {
        acc += cnt[t];
        cnt[t] = acc;
      }
    }
    // B = G - s s^T / n, then 1/4 J B J
    const unsigned long long *col = L.gram + D.gram_off, *pairs = col + k;
    const double inv_n = 1.0 / (double)n;
    for (int e = threadIdx.x; e < k * k; e += kPrepThreads) {
      const int a = e / k, b = e % k;
      if (a > b) continue;
      const unsigned long long plo = pairs[2 * e], phi = pairs[2 * e + 1];
      const unsigned __int128 g128 = ((unsigned __int128)phi << 32) + plo;
      const double g = (double)(unsigned long long)(g128 >> 64) * 18446744073709551616.0 + (double)(unsigned long long)g128;
      const double v = g - ((double)col[a] * (double)col[b]) * inv_n;
      Am[a * kLayLd + b] = v;
      Am[b * kLayLd + a] = v;
    }
    __syncthreads();
    for (int a = warp; a < k; a += kWarps) {
      double r = 0.0;
      for (int b = lane; b < k; b += 32) r += Am[a * kLayLd + b];
      r = warp_sum_d(r);
      if (lane == 0) s_rm[a] = r / (double)k;
    }
    __syncthreads();
    if (warp == 0) {
      double g = 0.0;
      for (int a = lane; a < k; a += 32) g += s_rm[a];
      g = warp_sum_d(g);
      if (lane == 0) s_gm = g / (double)k;
    }
    __syncthreads();
    for (int e = threadIdx.x; e < k * k; e += kPrepThreads) {
      const int a = e / k, b = e % k;
      if (a > b) continue;
      const double v = 0.25 * (Am[a * kLayLd + b] - s_rm[a] - s_rm[b] + s_gm);
      Am[a * kLayLd + b] = v;
      Am[b * kLayLd + a] = v;
    }
    __syncthreads();
    // ---- top-2 eigenpairs: Householder reduction of B to a tridiagonal T
    // (Q^T B Q = T; row j keeps the unit reflector of step j in its entries
    // j + 1 .. k - 1), the two largest eigenvalues of T by Sturm-count
    // bisection, their eigenvectors by inverse iteration on T, and back
    // through the reflectors
    for (int j = 0; j + 2 < k; ++j) {
      double *hv = Am + j * kLayLd;
      if (warp == 0) {  // the reflector of row j (the matrix is symmetric)
        double sig = 0.0;
        for (int r = j + 2 + lane; r < k; r += 32) sig = fma(hv[r], hv[r], sig);
        sig = warp_sum_d(sig);
        const double x0 = hv[j + 1];
        // a row that is tridiagonal already (or whose square vanishes): H = I
        const bool none = !(sig >= 1e-290);
        double v0 = 0.0, vinv = 0.0, e = x0;
        if (!none) {
          const double s2 = fma(x0, x0, sig);
          const double nrm = s2 * rsqrt_newton(s2);
          e = x0 >= 0.0 ? -nrm : nrm;
          v0 = x0 - e;
          vinv = rsqrt_newton(fma(v0, v0, sig));
        }
        __syncwarp();
        for (int r = j + 1 + lane; r < k; r += 32) hv[r] = (r == j + 1 ? v0 : hv[r]) * vinv;
        if (lane == 0) s_e[j] = e;
      }
      __syncthreads();
      if (hv[j + 1] == 0.0) continue;  // H = I (the same decision in every thread)
      // p = A v over the trailing block, a quarter of the sum per thread
      for (int r = j + 1 + (threadIdx.x & 127); r < k; r += 128) {
        double t = 0.0;
        for (int c = j + 1 + (threadIdx.x >> 7); c < k; c += kPrepThreads / 128) t = fma(Am[c * kLayLd + r], hv[c], t);
        s_p[threadIdx.x >> 7][r] = t;
      }
      __syncthreads();
      // warp 0: K = v . p, w = 2 (p - K v)
      if (warp == 0) {
        double kk = 0.0, p[(kPrepMaxK + 31) / 32];
#pragma unroll
        for (int q = 0; q < (kPrepMaxK + 31) / 32; ++q) {
          const int r = j + 1 + lane + 32 * q;
          p[q] = r < k ? (s_p[0][r] + s_p[1][r]) + (s_p[2][r] + s_p[3][r]) : 0.0;
          if (r < k) kk = fma(hv[r], p[q], kk);
        }
        kk = warp_sum_d(kk);
#pragma unroll
        for (int q = 0; q < (kPrepMaxK + 31) / 32; ++q) {
          const int r = j + 1 + lane + 32 * q;
          if (r < k) s_w[r] = 2.0 * fma(-kk, hv[r], p[q]);
        }
      }
      __syncthreads();
      // A -= v w^T + w v^T, the lower triangle and its mirror image: a warp
      // takes a short and a long row
      const int M = k - j - 1;
      for (int h = warp; 2 * h < M; h += kWarps)
        for (int side = 0; side < (2 * h == M - 1 ? 1 : 2); ++side) {
          const int r = j + 1 + (side == 0 ? h : M - 1 - h);
          const double vr = hv[r], wr = s_w[r];
          for (int c = j + 1 + lane; c <= r; c += 32) {
            const double v = fma(-wr, hv[c], fma(-vr, s_w[c], Am[r * kLayLd + c]));
            Am[r * kLayLd + c] = v;
            Am[c * kLayLd + r] = v;
          }
        }
      __syncthreads();
    }
    for (int a = threadIdx.x; a < k; a += kPrepThreads) s_dg[a] = Am[a * kLayLd + a];
    if (threadIdx.x == 0) s_e[k - 2] = Am[(k - 1) * kLayLd + (k - 2)];
    __syncthreads();
    // eigenvalues number k-1 and k-2 (ascending) by bisection on Sturm counts,
    // 32 points per step evaluated by the lanes of warp 0 (the largest) and
    // warp 1 (the second); each step of the count's recurrence takes 1/q from
    // an FP32 reciprocal and one Newton step in FP64 (relative error near
    // 2^-46: only the signs of the q are used, and GB300's FP64 division is
    // the slow part of this loop)
    for (int a = threadIdx.x; a + 1 < k; a += blockDim.x) s_e2[a] = s_e[a] * s_e[a];
    __syncthreads();
    if (threadIdx.x < 64) {
      const int lane = threadIdx.x & 31, want = threadIdx.x >> 5;
      double lo = 0.0, hi = 0.0;
      for (int a = 0; a < k; ++a) {
        const double r = (a > 0 ? fabs(s_e[a - 1]) : 0.0) + (a + 1 < k ? fabs(s_e[a]) : 0.0);
        lo = a == 0 ? s_dg[a] - r : fmin(lo, s_dg[a] - r);
        hi = a == 0 ? s_dg[a] + r : fmax(hi, s_dg[a] + r);
      }
      const int idx = k - 1 - want;  // ascending index of the eigenvalue
      double a0 = lo - 1e-12 * (fabs(lo) + fabs(hi)), b0 = hi + 1e-12 * (fabs(lo) + fabs(hi));
      for (int it = 0; it < 40 && b0 - a0 > 4e-16 * fmax(fabs(a0), fabs(b0)); ++it) {
        const double x = a0 + (b0 - a0) * (double)(lane + 1) / 33.0;
        int cnt = 0;  // eigenvalues below x
        double q = s_dg[0] - x;
        cnt += q < 0.0;
        for (int a = 1; a < k; ++a) {
          double r;
          const unsigned aq = (unsigned)__double2hiint(q) & 0x7FFFFFFFu;
          if (aq - 0x39B00000u < 0x0C900000u) {  // 2^-100 <= |q| < 2^101
            const double r0 = (double)__frcp_rn((float)q);
            r = r0 * fma(-q, r0, 2.0);
          } else {
            r = 1.0 / (q == 0.0 ? 1e-300 : q);
          }
          q = fma(-s_e2[a - 1], r, s_dg[a] - x);
          cnt += (unsigned)__double2hiint(q) >> 31;  // its sign (no q here is -0)
        }
        // the smallest lane point with more than idx eigenvalues below it
        const unsigned above = __ballot_sync(0xffffffffu, cnt > idx);
        const int first = above ? __ffs(above) - 1 : 32;
        const double nb = first < 32 ? a0 + (b0 - a0) * (double)(first + 1) / 33.0 : b0;
        const double na = first > 0 ? a0 + (b0 - a0) * (double)first / 33.0 : a0;
        a0 = na;
        b0 = nb;
      }
      if (lane == 0) s_lam[want] = 0.5 * (a0 + b0);
    }
    __syncthreads();
    // inverse iteration on T - lambda I (tridiagonal LU with partial
    // pivoting, factored once, two solves), one warp per eigenvalue (the
    // recurrences on its first lane); the second vector is then made
    // orthogonal to the first
    if (warp < 2) {
      const int want = warp;
      double *y = s_y[want];
      double *dd = s_fd[want], *du = s_fu[want], *du2 = s_fu2[want], *dl = s_fl[want];
      int *piv = s_piv[want];
      const double lam = s_lam[want];
      const double pert = 1e-14 * (fabs(lam) + 1e-300);
      for (int a = lane; a < k; a += 32) {
        y[a] = 1.0 + 0.01 * (double)((a * 37) % 11);
        dd[a] = s_dg[a] - lam;
        du[a] = a + 1 < k ? s_e[a] : 0.0;
        dl[a] = a + 1 < k ? s_e[a] : 0.0;
        du2[a] = 0.0;
      }
      __syncwarp();
      if (lane == 0) {
        for (int a = 0; a + 1 < k; ++a) {
          if (fabs(dd[a]) >= fabs(dl[a])) {
            if (dd[a] == 0.0) dd[a] = pert;
            const double f = dl[a] / dd[a];
            dl[a] = f;
            dd[a + 1] -= f * du[a];
            piv[a] = 0;
          } else {
            const double f = dd[a] / dl[a];
            dd[a] = dl[a];
            dl[a] = f;
            const double t = du[a];
            du[a] = dd[a + 1];
            dd[a + 1] = t - f * dd[a + 1];
            if (a + 2 < k) {
              du2[a] = du[a + 1];
              du[a + 1] = -f * du[a + 1];
            }
            piv[a] = 1;
          }
        }
        if (dd[k - 1] == 0.0) dd[k - 1] = pert;
      }
      __syncwarp();
      for (int a = lane; a < k; a += 32) dd[a] = 1.0 / dd[a];  // reciprocals for the solves
      __syncwarp();
      for (int it = 0; it < 2; ++it) {
        if (lane == 0) {
          double ya = y[0];
          for (int a = 0; a + 1 < k; ++a) {
            const double yb = y[a + 1];
            if (piv[a] == 0) {
              y[a] = ya;
              ya = fma(-dl[a], ya, yb);
            } else {
              y[a] = yb;
              ya = fma(-dl[a], yb, ya);
            }
          }
          double y1 = ya * dd[k - 1], y2 = 0.0;
          y[k - 1] = y1;
          for (int a = k - 2; a >= 0; --a) {
            const double t = fma(-du[a], y1, fma(-du2[a], y2, y[a])) * dd[a];
            y2 = y1;
            y1 = t;
            y[a] = t;
          }
        }
        __syncwarp();
        double nr = 0.0;
        for (int a = lane; a < k; a += 32) nr = fma(y[a], y[a], nr);
        nr = warp_sum_d(nr);
        nr = nr > 0.0 ? 1.0 / sqrt(nr) : 0.0;
        for (int a = lane; a < k; a += 32) y[a] *= nr;
        __syncwarp();
      }
    }
    __syncthreads();
    if (warp == 0) {
      double dt = 0.0, nr = 0.0;
      for (int a = lane; a < k; a += 32) dt = fma(s_y[1][a], s_y[0][a], dt);
      dt = warp_sum_d(dt);
      for (int a = lane; a < k; a += 32) {
        s_y[1][a] = fma(-dt, s_y[0][a], s_y[1][a]);
        nr = fma(s_y[1][a], s_y[1][a], nr);
      }
      nr = warp_sum_d(nr);
      nr = nr > 0.0 ? 1.0 / sqrt(nr) : 0.0;
      for (int a = lane; a < k; a += 32) s_y[1][a] *= nr;
      if (lane == 0) {
        s_done = s_lam[0] > 0.0;
        if (L.eig) {
          L.eig[2 * gi] = s_lam[0];
          L.eig[2 * gi + 1] = s_lam[1];
        }
      }
    }
    __syncthreads();
    // z = H_0 H_1 ... H_{k-3} y, the reflectors applied last to first, a warp
    // per vector; each is then signed so that its largest-magnitude entry
    // (lowest index on a tie) is positive
    if (warp < 2) {
      double *y = s_y[warp];
      for (int j = k - 3; j >= 0; --j) {
        const double *hv = Am + j * kLayLd;
        double dt = 0.0;
        for (int r = j + 1 + lane; r < k; r += 32) dt = fma(hv[r], y[r], dt);
        dt = -2.0 * warp_sum_d(dt);
        for (int r = j + 1 + lane; r < k; r += 32) y[r] = fma(dt, hv[r], y[r]);
        __syncwarp();
      }
      double big = -1.0;
      int at = 0;
      for (int a = lane; a < k; a += 32)
        if (fabs(y[a]) > big) {
          big = fabs(y[a]);
          at = a;
        }
      for (int o = 16; o > 0; o >>= 1) {
        const double ob = __shfl_xor_sync(0xffffffffu, big, o);
        const int oa = __shfl_xor_sync(0xffffffffu, at, o);
        if (ob > big || (ob == big && oa < at)) {
          big = ob;
          at = oa;
        }
      }
      const double sgn = y[at] < 0 ? -1.0 : 1.0;
      __syncwarp();
      // fixed point for the node loop: round(v 2^54) = high 2^27 + low, |v| <= 1
      // (a NaN or an infinity, of a matrix that was none, fails the batch)
      double sg = 0.0, cv = 0.0, cb = 0.0;
      bool bad = false;
      for (int a = lane; a < k; a += 32) {
        const double v = sgn * y[a], cbar = (double)col[a] * inv_n;
        y[a] = v;
        sg += v;
        cv = fma(cbar, v, cv);
        cb += cbar;
        bad |= !(fabs(v) <= 1.0 + 1e-9);
        const long long f = __double2ll_rn(v * 18014398509481984.0);
        int *o = reinterpret_cast<int *>(s_fix + a) + 2 * warp;
        o[0] = (int)(f & 0x7FFFFFF);
        o[1] = (int)(f >> 27);
      }
      sg = warp_sum_d(sg);
      cv = warp_sum_d(cv);
      cb = warp_sum_d(cb);
      if (__any_sync(0xffffffffu, bad) && lane == 0) dev_fail(L.status, SSM_E_NUMERIC);
      if (lane == 0) {
        s_sig[warp] = sg;
        s_kap[warp] = cv - cb / (double)k * sg;
      }
    }
    __syncthreads();
    if (!s_done) dev_fail(L.status, SSM_E_NUMERIC);
    // ---- x_i = -1/2 (sum_a d_ia^2 v_a - rbar_i sigma - kappa): whole
    // numbers, exact (d^2 < 2^28, 100 terms: below 2^63), then FP64
    float2 *pos = L.pos + D.node_off;
    for (int i = threadIdx.x; i < n; i += kPrepThreads) {
      long long xl = 0, xh = 0, yl = 0, yh = 0;
      unsigned long long rs = 0;
#pragma unroll 4
      for (int a = 0; a < k; ++a) {
        const int d = (int)dip[(int64_t)a * n + i];
        const int dd = d * d;
        const int4 f = s_fix[a];
        rs += (unsigned)dd;
        xl += (long long)dd * f.x;
        xh += (long long)dd * f.y;
        yl += (long long)dd * f.z;
        yh += (long long)dd * f.w;
      }
      const double x = fma((double)xh, 134217728.0, (double)xl) * 0x1p-54;
      const double y = fma((double)yh, 134217728.0, (double)yl) * 0x1p-54;
      const double rbar = (double)rs / (double)k;
      pos[i] = make_float2((float)(-0.5 * (x - rbar * s_sig[0] - s_kap[0])),
                           (float)(-0.5 * (y - rbar * s_sig[1] - s_kap[1])));
    }
    __syncthreads();
    // ---- rescale: sum_E ||x_i - x_j|| = m (lengths from the FP32 positions)
    const int32_t *rowptr = L.rowptr + D.row_off;
    const int32_t *colidx = L.colidx + D.col_off;
    double len = 0.0;
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
      const float2 xi = pos[i];
      for (int t = rowptr[i]; t < rowptr[i + 1]; ++t) {
        const int j = colidx[t];
        if (j <= i) continue;
        const float2 xj = pos[j];
        const float dx = xi.x - xj.x, dy = xi.y - xj.y;
        len += (double)sqrtf(dx * dx + dy * dy);
      }
    }
    len = block_sum_d(len, s_red);
    const bool okl = len > 0.0 && isfinite(len);
    if (!okl && threadIdx.x == 0) dev_fail(L.status, SSM_E_NUMERIC);
    const double sc = okl ? (double)D.m / len : 1.0;
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
      const float2 x = pos[i];
      pos[i] = make_float2((float)((double)x.x * sc), (float)((double)x.y * sc));
    }
    __syncthreads();
  }
}

// the workspace of both calls: descriptors, order, counter and lengths
// first (the layout call uses only this prefix), then the scatter area
struct PrepWs {
  PrepDev *pd;
  LayoutDev *ld;
  int32_t *order;
  unsigned *ctr;  // [3]
  int32_t *task0;  // [G + 1]
  unsigned long long *gram;
  int64_t *lens;  // [2 G]: table lengths, then edge counts
  int32_t *tmp;
};

// gram: words of the Gram sums; cap < 0: the prefix only (what the layout call uses)
static void carve_prep(Carver &c, PrepWs &w, int32_t G, int64_t gram, int64_t cap) {
  w.pd = c.take<PrepDev>((size_t)G);
  w.ld = c.take<LayoutDev>((size_t)G);
  w.order = c.take<int32_t>((size_t)G);
  w.ctr = c.take<unsigned>(3);
  w.task0 = c.take<int32_t>((size_t)G + 1);
  w.gram = c.take<unsigned long long>((size_t)gram);
  w.lens = c.take<int64_t>(2 * (size_t)G);
  w.tmp = cap >= 0 ? c.take<int32_t>((size_t)std::max<int64_t>(cap, 1)) : nullptr;
}

// what a batch asks for: its largest graph, with the neighbour lists where a
// block's shared memory holds them
static void prep_smem(int32_t G, const ssm_batch_input *in, int64_t &pivots, int64_t &dist) {
  const int64_t cap = 227 * 1024 - 2048;
  pivots = dist = 0;
  for (int32_t g = 0; g < G; ++g) {
    const int64_t p = block_search_bytes(in[g].n), d = dist_node_bytes(in[g].n), nb = 4 * in[g].m_in;
    pivots = std::max(pivots, p + nb <= cap ? p + nb : p);
    dist = std::max(dist, d + nb <= cap ? d + nb : d);
  }
}

static size_t layout_smem() { return (size_t)kPrepMaxK * kLayLd * sizeof(double); }

}  // namespace ssm

// =========================================================== C ABI
SSM_API size_t ssm_batch_prepare_workspace(int32_t G, const ssm_batch_input *in) {
  if (G < 1 || !in) return 0;
  int64_t cap = 0, gram = 0;
  for (int32_t g = 0; g < G; ++g) {
    cap += 2 * std::max<int64_t>(0, in[g].m_in);
    gram += ssm::gram_words(std::max(in[g].k, 0));
  }
  ssm::Carver c(nullptr, 0);
  ssm::PrepWs w;
  ssm::carve_prep(c, w, G, gram, cap);
  return c.size();
}

SSM_API int ssm_batch_pivots(int32_t G, const ssm_batch_input *in, const int32_t *src, const int32_t *dst,
                             ssm_batch_graph *out, int32_t *rowptr, int32_t *colidx, int32_t *pivots, uint16_t *dip,
                             int32_t *region, int32_t *ecc, int64_t *m_out, int32_t *status, void *ws,
                             size_t ws_bytes, cudaStream_t s) {
  using namespace ssm;
  if (G < 1 || !in || !out || !rowptr || !colidx || !pivots || !dip || !region || !ecc || !status || !ws)
    return fail(SSM_E_ARG, "ssm_batch_pivots: null pointer or G < 1");
  std::vector<PrepDev> pd((size_t)G);
  std::vector<int32_t> order((size_t)G);
  int64_t node = 0, row = 0, col = 0, piv = 0, dipo = 0, offo = 0, edges = 0, gram = 0;
  for (int32_t g = 0; g < G; ++g) {
    const ssm_batch_input &x = in[g];
    if (x.n < 1 || x.n > kPrepMaxN) return fail(SSM_E_ARG, "ssm_batch_pivots: graph %d has n = %d (1..%d)", g, x.n, kPrepMaxN);
    if (x.k < 2 || x.k > x.n || x.k > kPrepMaxK)
      return fail(SSM_E_ARG, "ssm_batch_pivots: graph %d has k = %d (2..min(n, %d))", g, x.k, kPrepMaxK);
    if (x.m_in < 0 || 2 * x.m_in >= ((int64_t)1 << 31)) return fail(SSM_E_ARG, "ssm_batch_pivots: graph %d edge count", g);
    if (x.m_in > 0 && (!src || !dst)) return fail(SSM_E_ARG, "ssm_batch_pivots: null edge arrays");
    PrepDev &d = pd[(size_t)g];
    d.n = x.n; d.k = x.k; d.m_in = x.m_in; d.edge_off = x.edge_off;
    d.node_off = node; d.row_off = row; d.col_off = col; d.piv_off = piv; d.dip_off = dipo; d.cnt_off_off = offo;
    ssm_batch_graph &o = out[g];
    o.n = x.n; o.k = x.k; o.cnt_len = 0; o.reserved = 0;
    o.node_off = node; o.row_off = row; o.col_off = col; o.piv_off = piv; o.dip_off = dipo; o.cnt_off_off = offo;
    o.cnt_base = 0;
    node += x.n; row += x.n + 1; col += 2 * x.m_in; piv += x.k; dipo += (int64_t)x.k * x.n; offo += x.k + 1;
    edges = std::max(edges, x.edge_off + x.m_in);
    gram += gram_words(x.k);
    order[(size_t)g] = g;
  }
  std::stable_sort(order.begin(), order.end(), [&](int32_t a, int32_t b) {
    return (int64_t)pd[(size_t)a].n * pd[(size_t)a].k > (int64_t)pd[(size_t)b].n * pd[(size_t)b].k;
  });
  Carver c(ws, ws_bytes);
  PrepWs w;
  carve_prep(c, w, G, gram, col);
  if (!c.ok) return fail(SSM_E_NOMEM, "ssm_batch_pivots: workspace %zu bytes, need %zu", ws_bytes, c.size());
  SSM_TRY_CUDA(cudaMemcpyAsync(w.pd, pd.data(), pd.size() * sizeof(PrepDev), cudaMemcpyHostToDevice, s));
  SSM_TRY_CUDA(cudaMemcpyAsync(w.order, order.data(), order.size() * sizeof(int32_t), cudaMemcpyHostToDevice, s));
  SSM_TRY_CUDA(cudaMemsetAsync(w.ctr, 0, 3 * sizeof(unsigned), s));
  PrepArgs A;
  A.G = G; A.desc = w.pd; A.order = w.order; A.src = src; A.dst = dst; A.tmp = w.tmp;
  A.rowptr = rowptr; A.colidx = colidx; A.pivots = pivots; A.region = region; A.dip = dip; A.ecc = ecc;
  A.lens = w.lens; A.medges = w.lens + G; A.ctr = w.ctr; A.status = status;
  prep_smem(G, in, A.ubytes, A.dbytes);
  SSM_TRY_CUDA(allow_dynamic_smem((const void *)k_prep_pivots));
  SSM_TRY_CUDA(allow_dynamic_smem((const void *)k_prep_dist));
  int per_sm = 0, per_sm_d = 0;
  SSM_TRY_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_prep_pivots, kPrepThreads, (size_t)A.ubytes));
  SSM_TRY_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm_d, k_prep_dist, kDistThreads, (size_t)A.dbytes));
  if (per_sm < 1 || per_sm_d < 1)
    return fail(SSM_E_ARG, "ssm_batch_pivots: %lld bytes of shared memory do not fit", (long long)std::max(A.ubytes, A.dbytes));
  const int64_t words = (kPrepMaxK + 31) / 32;
  note_launch(), k_prep_pivots<<<std::min(G, per_sm * num_sms()), kPrepThreads, (size_t)A.ubytes, s>>>(A);
  SSM_TRY_CUDA(cudaGetLastError());
  note_launch(), k_prep_dist<<<(int)std::min<int64_t>(G * words, per_sm_d * num_sms()), kDistThreads, (size_t)A.dbytes, s>>>(A);
  SSM_TRY_CUDA(cudaGetLastError());
  std::vector<int64_t> h(2 * (size_t)G);
  int32_t hst = 0;
  SSM_TRY_CUDA(cudaMemcpyAsync(h.data(), w.lens, h.size() * sizeof(int64_t), cudaMemcpyDeviceToHost, s));
  SSM_TRY_CUDA(cudaMemcpyAsync(&hst, status, sizeof hst, cudaMemcpyDeviceToHost, s));
  SSM_TRY_CUDA(cudaStreamSynchronize(s));
  if (hst) return fail(hst, "ssm_batch_pivots: %s", ssm_status_string(hst));
  int64_t base = 0;
  for (int32_t g = 0; g < G; ++g) {
    if (h[(size_t)g] < in[g].k || h[(size_t)g] >= ((int64_t)1 << 30))
      return fail(SSM_E_DISCONNECTED, "ssm_batch_pivots: graph %d has no valid count table (disconnected?)", g);
    out[g].cnt_len = (int32_t)h[(size_t)g];
    out[g].cnt_base = base;
    base += h[(size_t)g];
    if (m_out) m_out[g] = h[(size_t)G + g];
  }
  return SSM_OK;
}

SSM_API int ssm_batch_layout_init(int32_t G, const ssm_batch_graph *graphs, const int64_t *m, const int32_t *rowptr,
                                  const int32_t *colidx, const uint16_t *dip, const int32_t *region,
                                  const int32_t *ecc, int32_t *cnt_off, uint32_t *cnt, float *pos, double *eig,
                                  int32_t *status, void *ws, size_t ws_bytes, cudaStream_t s) {
  using namespace ssm;
  if (G < 1 || !graphs || !m || !rowptr || !colidx || !dip || !region || !ecc || !cnt_off || !cnt || !pos ||
      !status || !ws)
    return fail(SSM_E_ARG, "ssm_batch_layout_init: null pointer or G < 1");
  std::vector<LayoutDev> ld((size_t)G);
  std::vector<int32_t> order((size_t)G), task0((size_t)G + 1);
  int64_t gram = 0, tasks = 0;
  for (int32_t g = 0; g < G; ++g) {
    const ssm_batch_graph &x = graphs[g];
    if (x.n < 1 || x.n > kPrepMaxN || x.k < 2 || x.k > kPrepMaxK || x.k > x.n || x.cnt_len < x.k)
      return fail(SSM_E_ARG, "ssm_batch_layout_init: graph %d has n = %d, k = %d, cnt_len = %d", g, x.n, x.k, x.cnt_len);
    if (m[g] < 1) return fail(SSM_E_ARG, "ssm_batch_layout_init: graph %d has no edges", g);
    LayoutDev &d = ld[(size_t)g];
    d.n = x.n; d.k = x.k; d.m = m[g];
    d.node_off = x.node_off; d.row_off = x.row_off; d.col_off = x.col_off; d.piv_off = x.piv_off;
    d.dip_off = x.dip_off; d.cnt_off_off = x.cnt_off_off; d.cnt_base = x.cnt_base;
    d.gram_off = gram;
    gram += gram_words(x.k);
    order[(size_t)g] = g;
  }
  std::stable_sort(order.begin(), order.end(), [&](int32_t a, int32_t b) {
    const LayoutDev &x = ld[(size_t)a], &y = ld[(size_t)b];
    return (int64_t)x.n * x.k * x.k > (int64_t)y.n * y.k * y.k;
  });
  for (int32_t q = 0; q < G; ++q) {
    task0[(size_t)q] = (int32_t)tasks;
    tasks += (ld[(size_t)order[(size_t)q]].n + kGramNodes - 1) / kGramNodes;
  }
  task0[(size_t)G] = (int32_t)tasks;
  Carver c(ws, ws_bytes);
  PrepWs w;
  carve_prep(c, w, G, gram, -1);
  if (!c.ok) return fail(SSM_E_NOMEM, "ssm_batch_layout_init: workspace %zu bytes, need %zu", ws_bytes, c.size());
  LayoutDev *dd = w.ld;
  int32_t *dorder = w.order;
  unsigned *ctr = w.ctr + 1;
  SSM_TRY_CUDA(cudaMemcpyAsync(dd, ld.data(), ld.size() * sizeof(LayoutDev), cudaMemcpyHostToDevice, s));
  SSM_TRY_CUDA(cudaMemcpyAsync(dorder, order.data(), order.size() * sizeof(int32_t), cudaMemcpyHostToDevice, s));
  SSM_TRY_CUDA(cudaMemcpyAsync(w.task0, task0.data(), task0.size() * sizeof(int32_t), cudaMemcpyHostToDevice, s));
  SSM_TRY_CUDA(cudaMemsetAsync(ctr, 0, sizeof(unsigned), s));
  SSM_TRY_CUDA(cudaMemsetAsync(w.gram, 0, (size_t)gram * sizeof(unsigned long long), s));
  LayoutArgs L;
  L.G = G; L.desc = dd; L.order = dorder; L.task0 = w.task0; L.gram = w.gram; L.rowptr = rowptr; L.colidx = colidx; L.region = region; L.ecc = ecc;
  L.dip = dip; L.cnt_off = cnt_off; L.cnt = cnt; L.pos = reinterpret_cast<float2 *>(pos); L.eig = eig; L.ctr = ctr;
  L.status = status;
  const size_t smem = layout_smem();
  SSM_TRY_CUDA(allow_dynamic_smem((const void *)k_prep_layout));
  int per_sm = 0;
  SSM_TRY_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_prep_layout, kPrepThreads, smem));
  if (per_sm < 1) return fail(SSM_E_ARG, "ssm_batch_layout_init: %zu bytes of shared memory do not fit", smem);
  const int blocks = std::max(1, std::min(G, per_sm * num_sms()));
  note_launch(), k_prep_gram<<<(int)tasks, kGramThreads, 0, s>>>(L);
  SSM_TRY_CUDA(cudaGetLastError());
  note_launch(), k_prep_layout<<<blocks, kPrepThreads, smem, s>>>(L);
  SSM_TRY_CUDA(cudaGetLastError());
  return SSM_OK;
}
