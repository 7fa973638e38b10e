// Contact LCP of a step (Sec. 3.2, Eq. 3.7; Sec. 3.3.3, Alg. 3) on one GPU.
//
//   0 <= -V + B lambda   perp   lambda >= 0,      B = J M J^T
//
// One row per contact volume: a candidate vesicle pair (with its periodic
// image) that has contacts; V its volume (the library's volumes are >= 0 for
// interference, the paper's constraint V >= 0 has the opposite sign, which B
// does not see).  J = dV/dX1 (the gradient rows of stiv_stiv_grad, summed
// per vertex); M block-diagonal, M_ii = m_i I + t_i (1 1^T (x) I_3) per
// vesicle (a local part and a rigid translation), a stand-in with the block
// structure of the locally implicit scheme's A^-1 G.
//
// Assembly (Alg. 3):
//   bounds_kernel   contact range of every candidate pair (contacts are
//                   sorted by pair)
//   rows_kernel     rows = pairs with contacts; q = -V
//   row_sides_kernel per row and side (side 0: the pair's first vesicle, 1: its
//                   second) the gradient of each vertex: a row's contacts are
//                   contiguous, so one CTA sorts their points by vertex in shared
//                   memory and sums the runs in contact order, fixed association
//                   (deterministic)
//   ves_count, ves_scan, ves_fill, ves_rank
//                   the rows of each vesicle, ascending
//   bcount_kernel   per row, the rows sharing a vesicle (union of its two
//                   vesicles' lists)
//   bcol_kernel     the columns and the row of every nonzero
//   bval_kernel     B(j, k) = sum over shared vesicles i (ascending) of
//                   m_i g_j|i . g_k|i + t_i (sum g_j|i) . (sum g_k|i), a join
//                   on the vertex ids of i; one warp per nonzero
// Solve: min-map Newton (Phi = min(lambda, B lambda + q)) in FP64, the Newton
// system on the active set by Jacobi-preconditioned conjugate gradients in
// FP32 (B_AA is symmetric positive definite), Armijo line search on
// |Phi|^2 / 2; one CTA, all iterations in one launch.
#include "stiv_internal.cuh"

#include <math.h>

namespace {

constexpr int RT = 1024;   // threads of the single-CTA kernels

__device__ __forceinline__ int64_t ncontacts(const int64_t* counts, int64_t cap) {
  int64_t n = counts[STIV_C_VF] + counts[STIV_C_EE];
  return n < cap ? n : cap;
}

__global__ void bounds_kernel(const int64_t* counts, int64_t ccap, const int32_t* pair, int32_t* pstart,
                              int32_t* pend) {
  int64_t n = ncontacts(counts, ccap);
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x) {
    int p = pair[k];
    if (k == 0 || pair[k - 1] != p) pstart[p] = (int32_t)k;
    if (k == n - 1 || pair[k + 1] != p) pend[p] = (int32_t)(k + 1);
  }
}

// Block-wide exclusive scan (RT threads); sh: RT / 32 ints.
__device__ int block_scan(int v, int* sh, int& total) {
  int lane = threadIdx.x & 31, w = threadIdx.x >> 5, x = v;
  for (int off = 1; off < 32; off <<= 1) {
    int y = __shfl_up_sync(0xffffffffu, x, off);
    if (lane >= off) x += y;
  }
  if (lane == 31) sh[w] = x;
  __syncthreads();
  int s = sh[lane];
  static_assert(RT / 32 == 32, "one warp total per lane");
  for (int off = 1; off < 32; off <<= 1) {
    int y = __shfl_up_sync(0xffffffffu, s, off);
    if (lane >= off) s += y;
  }
  total = __shfl_sync(0xffffffffu, s, 31);
  int pre = w ? __shfl_sync(0xffffffffu, s, w - 1) : 0;
  __syncthreads();
  return pre + x - v;
}

// A row of more than LONG_ROW contacts is cut into segments of SEG_C contacts for
// row_sides_kernel; the segments after the first are listed (in any order, a row's
// own in a run).
constexpr int LONG_ROW = 2048;
constexpr int SEG_C = 1024;
struct seg_list {
  int32_t* count;    // segments listed (cleared before)
  int32_t* row;      // [ccap / SEG_C + 1]  the row of each
  int32_t* first;    // [rcap]  long rows: place of the row's second segment
  int32_t* done;     // [2 rcap]  long rows: segments finished per side
  int64_t rcap;      // a listed segment's slot in sbeg and scnt: 2 (rcap + place) + side
};
__host__ __device__ inline int row_segments(int len) { return len > LONG_ROW ? (len + SEG_C - 1) / SEG_C : 1; }

// dims: [0] rows, [1] nnz, [2] status (1: rows over capacity, 2: nonzeros
// over capacity), [3] entries (4 x contacts), [4] 2 x rows
__global__ void __launch_bounds__(RT) rows_kernel(const int64_t* counts, int64_t pcap, int64_t ccap,
                                                  const int32_t* pstart, const int32_t* pend, const double* Vp,
                                                  int64_t rcap, int32_t* row_pair, double* q, int64_t* dims,
                                                  seg_list segs) {
  __shared__ int sh[RT / 32];
  int64_t np = counts[STIV_C_PAIRS] < pcap ? counts[STIV_C_PAIRS] : pcap;
  int base = 0;
  for (int64_t p0 = 0; p0 < np; p0 += RT) {
    int64_t p = p0 + threadIdx.x;
    int has = (p < np && pend[p] > pstart[p]) ? 1 : 0;
    int tot;
    int ex = block_scan(has, sh, tot);
    if (has && base + ex < rcap) {
      row_pair[base + ex] = (int32_t)p;
      q[base + ex] = -Vp[p];
      const int more = row_segments(pend[p] - pstart[p]) - 1;
      if (more) {
        const int at = atomicAdd(segs.count, more);
        segs.first[base + ex] = at;
        segs.done[2 * (base + ex)] = 0;
        segs.done[2 * (base + ex) + 1] = 0;
        for (int k = 0; k < more; ++k) segs.row[at + k] = base + ex;
      }
    }
    base += tot;
  }
  if (threadIdx.x == 0) {
    dims[0] = base < rcap ? base : rcap;
    dims[2] = base > rcap ? 1 : 0;
    dims[3] = 4 * ncontacts(counts, ccap);
    dims[4] = 2 * dims[0];
  }
}

constexpr int ST = 256;      // threads of a row-side CTA
constexpr int CH = 2048;     // points sorted at a time
constexpr int SD = 128;      // digits of the sort (7 bits)
// shared memory of row_sides_kernel: its own arrays (33 KB at most) and one 16-bit
// entry per vertex (nv)
constexpr size_t SIDE_SMEM = 2 * 4 * CH + 4 * CH + 4 * (ST / 32) * SD + 2 * (CH + 1) + 256;
constexpr size_t side_table_bytes(int nv) { return sizeof(uint16_t) * (size_t)((nv + 7) & ~7); }

// Exclusive scan over an ST-thread CTA; *total = the sum.  wsum: ST / 32 ints.
__device__ __forceinline__ int cta_scan(int v, int* wsum, int* total) {
  int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  int x = v;
  for (int off = 1; off < 32; off <<= 1) {
    int y = __shfl_up_sync(0xffffffffu, x, off);
    if (lane >= off) x += y;
  }
  if (lane == 31) wsum[w] = x;
  __syncthreads();
  int pre = 0, tot = 0;
  for (int q = 0; q < ST / 32; ++q) { int s = wsum[q]; pre += q < w ? s : 0; tot += s; }
  __syncthreads();
  *total = tot;
  return pre + x - v;
}

// Joins the segments of a long row's side, each its vertices and sums, into one
// list at the first one's place: segment by segment, a vertex seen before adds to
// its entry, another one takes the next.  In place: an entry moves to no place
// after its own, and a batch is read before it is written.  Returns the entries.
__device__ __noinline__ int join_segments(const seg_list& segs, int64_t row, int side, int nseg, int nv, uint16_t* tab,
                                          int* wsum, const int32_t* sbeg, const int32_t* scnt, int32_t* ukey,
                                          double* ug) {
  for (int q = threadIdx.x; q < nv; q += ST) tab[q] = 0xFFFF;
  __syncthreads();
  const int64_t base = __ldcg(&sbeg[2 * row + side]), more = segs.rcap + segs.first[row] - 1;
  int unique = 0;
  for (int sg = 0; sg < nseg; ++sg) {
    const int64_t slot = 2 * (sg ? more + sg : row) + side, lo = __ldcg(&sbeg[slot]);
    const int cnt = __ldcg(&scnt[slot]);
    for (int i0 = 0; i0 < cnt; i0 += ST) {
      const int i = i0 + threadIdx.x;
      const bool in = i < cnt;
      int v = 0;
      double g[3] = {0.0, 0.0, 0.0};
      if (in) {
        v = __ldcg(&ukey[lo + i]);
        for (int c = 0; c < 3; ++c) g[c] = __ldcg(&ug[3 * (lo + i) + c]);
      }
      const bool fresh = in && tab[v] == 0xFFFF;
      int add;
      const int u = unique + cta_scan(fresh ? 1 : 0, wsum, &add);   // barriers: all of the batch is read
      if (fresh) {
        tab[v] = (uint16_t)u;
        ukey[base + u] = v;
        for (int c = 0; c < 3; ++c) ug[3 * (base + u) + c] = g[c];
      } else if (in) {   // a vertex once per segment: no other thread adds to its entry
        double* d = ug + 3 * (base + tab[v]);
        for (int c = 0; c < 3; ++c) d[c] += g[c];
      }
      unique += add;
      __syncthreads();
    }
  }
  return unique;
}

// The unique vertices of row r's side s and the sum of their gradient rows, at
// [sbeg[2 r + s], + scnt[2 r + s]) of ukey and ug (a row's points start at four
// times its first contact, side 1's after side 0's).  The points are taken in
// chunks of at most CH in contact order, each sorted by vertex (stable: vertex <<
// 12 | place); a run's sum goes to a new entry or onto the one an earlier chunk
// made (tab: vertex -> entry).  Four lanes sum a run, strided, then by halves: a
// fixed order.
//
// The global alternative (a keyed entry per point, a radix sort of all of them by
// row, side and vertex, a gather and a segmented scan over all entries: 25
// launches) took 0.42 ms of device time at 1440 vesicles (2.5M points), this
// kernel 0.15 ms, bound by the latency of its short phases.  A row in one CTA takes
// 21 ns a contact, so that a pair that interpenetrates deeply would hold the
// assembly (55,202 contacts of two vesicles at p = 31: 1264 us, 266 in the global
// form): a row of more than LONG_ROW contacts goes in segments to as many CTAs, and
// the one that finishes last joins them (no CTA waits for another): 258 us, and 225
// -> 115 for 7050 contacts (global 190); shorter rows, up to 1620 contacts at 1440
// vesicles, are as they were (213 us).
__global__ void __launch_bounds__(ST, 6) row_sides_kernel(const int64_t* dims, const int32_t* row_pair, const int32_t* pstart,
                                                       const int32_t* pend, const int32_t* ci, const int32_t* gves,
                                                       const int32_t* gvid, const double* grad, int nv, bool vec,
                                                       seg_list segs, int32_t* sbeg, int32_t* scnt, int32_t* ukey,
                                                       double* ug) {
  extern __shared__ uint16_t tab[];          // [nv rounded up to 8]
  __shared__ uint32_t item[2][CH];           // vertex << 12 | place in the chunk
  __shared__ int32_t src[CH];                // by place: gradient row
  __shared__ int32_t cnt[ST / 32][SD];
  __shared__ uint16_t start[CH + 1];         // runs
  __shared__ int wsum[ST / 32];
  __shared__ bool last;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int nlist = *segs.count;             // the listed segments first: their rows take longest
  const int64_t nitem = 2 * (dims[0] + nlist);
  for (int64_t it = blockIdx.x; it < nitem; it += gridDim.x) {
    const int side = (int)(it & 1), unit = (int)(it >> 1);
    const int row = unit < nlist ? segs.row[unit] : unit - nlist;
    const int p = row_pair[row], vi = ci[p];
    const int k0 = pstart[p], k1 = pend[p], nseg = row_segments(k1 - k0);
    const int seg = unit < nlist ? unit - segs.first[row] + 1 : 0;
    const int ka = nseg > 1 ? k0 + seg * SEG_C : k0, ke = nseg > 1 ? min(ka + SEG_C, k1) : k1;
    for (int q = threadIdx.x; q < nv; q += ST) tab[q] = 0xFFFF;
    int64_t base = 4 * (int64_t)k0;
    if (side || seg) {   // after the points of side 0 (side 1) and those of earlier segments
      int c = 0, before = 0, tot;
#pragma unroll 4
      for (int k = k0 + threadIdx.x; k < (side ? k1 : ka); k += ST) {
        int m = 0;
        if (vec) {
          int4 a = ((const int4*)gves)[k];
          m = (a.x == vi) + (a.y == vi) + (a.z == vi) + (a.w == vi);
        } else {
          for (int q = 0; q < 4; ++q) m += gves[4 * (int64_t)k + q] == vi;
        }
        c += m;
        before += k < ka ? m : 0;
      }
      cta_scan(c, wsum, &tot);
      base += tot;         // side 0: of the segments before; side 1: of the row
      if (side && seg) {
        cta_scan(before, wsum, &tot);
        base += 4 * (int64_t)(ka - k0) - tot;
      }
    }
    int unique = 0, n = 0;
    for (int kb = ka; kb < ke; kb += ST) {
      // the points of the next ST contacts on this side
      const int64_t k = kb + threadIdx.x;
      int vs[4], vd[4], c = 0, tot;
      unsigned mine = 0;
      if (k < ke) {
        if (vec) {
          int4 a = ((const int4*)gves)[k], b = ((const int4*)gvid)[k];
          vs[0] = a.x; vs[1] = a.y; vs[2] = a.z; vs[3] = a.w;
          vd[0] = b.x; vd[1] = b.y; vd[2] = b.z; vd[3] = b.w;
        } else {
          for (int q = 0; q < 4; ++q) { vs[q] = gves[4 * k + q]; vd[q] = gvid[4 * k + q]; }
        }
        for (int q = 0; q < 4; ++q)
          if ((vs[q] == vi) == (side == 0)) { mine |= 1u << q; ++c; }
      }
      int at = n + cta_scan(c, wsum, &tot);
      for (int q = 0; q < 4; ++q)
        if (mine >> q & 1u) {
          item[0][at] = ((uint32_t)vd[q] << 12) | (uint32_t)at;
          src[at] = (int32_t)(4 * k + q);
          ++at;
        }
      n += tot;
      __syncthreads();
      if (kb + ST < ke && n + 4 * ST <= CH) continue;
      // sort the n points by vertex
      int cur = 0;
      for (int shift = 12; shift < 26 && (nv - 1) >> (shift - 12); shift += 7) {
        for (int q = lane; q < SD; q += 32) cnt[w][q] = 0;
        __syncwarp();
        uint32_t x[CH / ST];
        int rank[CH / ST];
#pragma unroll
        for (int q = 0; q < CH / ST; ++q) {
          const int i = w * (CH / (ST / 32)) + q * 32 + lane;
          const bool valid = i < n;
          x[q] = valid ? item[cur][i] : 0;
          if (__any_sync(0xffffffffu, valid)) {
            const unsigned dig = (x[q] >> shift) & (SD - 1);
            const unsigned peers = digit_peers<7>(dig, valid), below = peers & ((1u << lane) - 1u);
            const int o = valid ? cnt[w][dig] : 0;
            __syncwarp();
            if (valid && !below) cnt[w][dig] = o + __popc(peers);
            rank[q] = o + __popc(below);
            __syncwarp();
          }
        }
        __syncthreads();
        int run = 0;
        if (threadIdx.x < SD)
          for (int q = 0; q < ST / 32; ++q) { int o = cnt[q][threadIdx.x]; cnt[q][threadIdx.x] = run; run += o; }
        int first = cta_scan(run, wsum, &tot);
        if (threadIdx.x < SD)
          for (int q = 0; q < ST / 32; ++q) cnt[q][threadIdx.x] += first;
        __syncthreads();
#pragma unroll
        for (int q = 0; q < CH / ST; ++q)
          if (w * (CH / (ST / 32)) + q * 32 + lane < n) item[1 - cur][cnt[w][(x[q] >> shift) & (SD - 1)] + rank[q]] = x[q];
        cur = 1 - cur;
        __syncthreads();
      }
      const uint32_t* a = item[cur];
      // runs of one vertex
      unsigned head = 0;
      for (int q = 0; q < CH / ST; ++q) {
        const int i = threadIdx.x * (CH / ST) + q;
        if (i < n && (i == 0 || (a[i] >> 12) != (a[i - 1] >> 12))) head |= 1u << q;
      }
      int runs;
      int o = cta_scan(__popc(head), wsum, &runs);
      for (int q = 0; q < CH / ST; ++q)
        if (head >> q & 1u) start[o++] = (uint16_t)(threadIdx.x * (CH / ST) + q);
      if (threadIdx.x == 0) start[runs] = (uint16_t)n;
      __syncthreads();
      // entries: new ones after the earlier chunks', in vertex order
      for (int r0 = 0; r0 < runs; r0 += ST) {
        const int r = r0 + threadIdx.x;
        const int v = r < runs ? (int)(a[start[r]] >> 12) : 0;
        const bool fresh = r < runs && tab[v] == 0xFFFF;
        int add;
        const int u = unique + cta_scan(fresh ? 1 : 0, wsum, &add);
        if (fresh) { tab[v] = (uint16_t)u; ukey[base + u] = v; }
        if (r < runs) item[1 - cur][r] = (uint32_t)tab[v] | (fresh ? 0x80000000u : 0u);
        unique += add;
      }
      __syncthreads();
      for (int r = threadIdx.x >> 2; r < ((runs + 7) & ~7); r += ST / 4) {   // whole warps
        double s0 = 0.0, s1 = 0.0, s2 = 0.0;
        if (r < runs)
          for (int i = start[r] + (lane & 3); i < start[r + 1]; i += 4) {
            const double* g = grad + 3 * (int64_t)src[a[i] & 0xFFFu];
            s0 += g[0]; s1 += g[1]; s2 += g[2];
          }
        for (int off = 2; off > 0; off >>= 1) {
          s0 += __shfl_xor_sync(0xffffffffu, s0, off);
          s1 += __shfl_xor_sync(0xffffffffu, s1, off);
          s2 += __shfl_xor_sync(0xffffffffu, s2, off);
        }
        if (r < runs && (lane & 3) < 3) {
          const uint32_t e = item[1 - cur][r];
          double* d = ug + 3 * (base + (e & 0xFFFFu)) + (lane & 3);
          const double v = (lane & 3) == 0 ? s0 : ((lane & 3) == 1 ? s1 : s2);
          *d = e >> 31 ? v : *d + v;
        }
      }
      n = 0;
      __syncthreads();
    }
    const int64_t slot = 2 * (int64_t)(unit < nlist ? segs.rcap + unit : row) + side;
    if (threadIdx.x == 0) { sbeg[slot] = (int32_t)base; scnt[slot] = unique; }
    if (nseg > 1) {
      __threadfence();
      __syncthreads();
      if (threadIdx.x == 0) last = atomicAdd(&segs.done[2 * row + side], 1) == nseg - 1;
      __syncthreads();
      if (last) {
        __threadfence();
        unique = join_segments(segs, row, side, nseg, nv, tab, wsum, sbeg, scnt, ukey, ug);
        if (threadIdx.x == 0) scnt[2 * row + side] = unique;
      }
    }
    __syncthreads();
  }
}

// The rows of every vesicle: counted, laid out by a scan (vstart [n_ves + 1]),
// filled in any order and ranked (a vesicle has a row at most once).
__global__ void ves_count_kernel(const int64_t* dims, const int32_t* row_pair, const int32_t* ci, const int32_t* cj,
                                 int32_t* vcnt) {
  int64_t n = dims[0];
  for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < n; r += (int64_t)gridDim.x * blockDim.x) {
    int p = row_pair[r];
    atomicAdd(&vcnt[ci[p]], 1);
    atomicAdd(&vcnt[cj[p]], 1);
  }
}

__global__ void __launch_bounds__(RT) ves_scan_kernel(int n, int32_t* vcnt, int32_t* vstart) {
  __shared__ int sh[RT / 32];
  int base = 0;
  for (int v0 = 0; v0 < n; v0 += RT) {
    int v = v0 + threadIdx.x, tot;
    int ex = block_scan(v < n ? vcnt[v] : 0, sh, tot);
    if (v < n) { vstart[v] = base + ex; vcnt[v] = base + ex; }   // vcnt: the fill position from here on
    base += tot;
  }
  if (threadIdx.x == 0) vstart[n] = base;
}

__global__ void ves_fill_kernel(const int64_t* dims, const int32_t* row_pair, const int32_t* ci, const int32_t* cj,
                                int32_t* vpos, int32_t* lst) {
  int64_t n = dims[0];
  for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < n; r += (int64_t)gridDim.x * blockDim.x) {
    int p = row_pair[r];
    lst[atomicAdd(&vpos[ci[p]], 1)] = (int32_t)r;
    lst[atomicAdd(&vpos[cj[p]], 1)] = (int32_t)r;
  }
}

// One warp per vesicle: each row's place is the number of smaller ones.
__global__ void ves_rank_kernel(int n, const int32_t* vstart, const int32_t* lst, int32_t* out) {
  int lane = threadIdx.x & 31;
  int w0 = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5), nw = (int)((gridDim.x * blockDim.x) >> 5);
  for (int v = w0; v < n; v += nw) {
    int lo = vstart[v], len = vstart[v + 1] - lo;
    for (int i = lane; i < len; i += 32) {
      int x = lst[lo + i], r = 0;
      for (int q = 0; q < len; ++q) r += lst[lo + q] < x;
      out[lo + r] = x;
    }
  }
}

// Rows sharing a vesicle with row r, ascending, without repeats: a merge of
// the sorted row lists of its two vesicles.  f(s) is called for each, in order.
template <class F>
__device__ void for_neighbours(const int32_t* lst, int a0, int a1, int b0, int b1, F f) {
  int i = a0, j = b0, last = -1;
  while (i < a1 || j < b1) {
    int s;
    if (j >= b1 || (i < a1 && lst[i] <= lst[j])) s = lst[i++];
    else s = lst[j++];
    if (s != last) { f(s); last = s; }
  }
}

__global__ void bcount_kernel(const int64_t* dims, const int32_t* row_pair, const int32_t* ci, const int32_t* cj,
                              const int32_t* vrow, const int32_t* vstart, int32_t* bcnt) {
  int64_t n = dims[0];
  for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < n; r += (int64_t)gridDim.x * blockDim.x) {
    int p = row_pair[r], vi = ci[p], vj = cj[p];
    int c = 0;
    for_neighbours(vrow, vstart[vi], vstart[vi + 1], vstart[vj], vstart[vj + 1], [&](int) { ++c; });
    bcnt[r] = c;
  }
}

__global__ void __launch_bounds__(RT) bscan_kernel(int64_t* dims, const int32_t* bcnt, int64_t nnz_cap,
                                                   int64_t* row_ptr) {
  __shared__ int sh[RT / 32];
  int64_t n = dims[0];
  int64_t base = 0;
  for (int64_t r0 = 0; r0 < n; r0 += RT) {
    int64_t r = r0 + threadIdx.x;
    int c = r < n ? bcnt[r] : 0;
    int tot;
    int ex = block_scan(c, sh, tot);
    if (r < n) row_ptr[r] = base + ex;
    base += tot;
  }
  if (threadIdx.x == 0) {
    row_ptr[n] = base;
    dims[1] = base;
    if (base > nnz_cap) dims[2] |= 2;
  }
}

// Entries of row x on one side of its pair (0: first vesicle, 1: second).
__device__ __forceinline__ void side_range(const int32_t* sbeg, const int32_t* scnt, int64_t x, int side, int64_t& lo,
                                           int64_t& hi) {
  lo = sbeg[2 * x + side];
  hi = lo + scnt[2 * x + side];
}

// Columns of B (thread per row): the rows sharing a vesicle with row r,
// ascending, and the row of every nonzero.
__global__ void bcol_kernel(const int64_t* dims, const int32_t* row_pair, const int32_t* ci, const int32_t* cj,
                            const int32_t* vrow, const int32_t* vstart, const int64_t* row_ptr,
                            int64_t nnz_cap, int32_t* col, int32_t* nzrow) {
  int64_t n = dims[0];
  for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < n; r += (int64_t)gridDim.x * blockDim.x) {
    int p = row_pair[r], vi = ci[p], vj = cj[p];
    int64_t o = row_ptr[r];
    for_neighbours(vrow, vstart[vi], vstart[vi + 1], vstart[vj], vstart[vj + 1], [&](int s) {
      if (o < nnz_cap) { col[o] = s; nzrow[o] = (int32_t)r; }
      ++o;
    });
  }
}

// One warp per nonzero: B(r, s) = sum over the vesicles v common to rows r
// and s (ascending) of m_v g_r|v . g_s|v + t_v (sum g_r|v) . (sum g_s|v).
// The dot product over v's vertices is a join on the vertex id: row B's
// entries (B = max(r, s)) are scattered into the warp's vertex-index table in
// shared memory (nvtab slots, -1 = absent, reset after use) and the lanes,
// over row A's entries (A = min(r, s)), look their vertex up (on the diagonal
// every entry is its own match).  Sums are reduced in a fixed order and
// depend on (A, B) only: B(r, s), s >= r, is written to (s, r) as well, B is
// symmetric bit for bit.
__global__ void bval_kernel(const int64_t* dims, const int32_t* row_pair, const int32_t* ci, const int32_t* cj,
                            const int32_t* sbeg, const int32_t* scnt, const int32_t* ukey, const double* ug,
                            const double* m_ves, const double* t_ves, int nvtab, int64_t nnz_cap,
                            const int64_t* row_ptr, const int32_t* col, const int32_t* nzrow, double* val) {
  extern __shared__ int32_t vtab_all[];
  int lane = threadIdx.x & 31;
  int32_t* tab = vtab_all + (size_t)(threadIdx.x >> 5) * nvtab;
  for (int i = lane; i < nvtab; i += 32) tab[i] = -1;
  __syncwarp();
  int64_t nnz = dims[1] < nnz_cap ? dims[1] : nnz_cap;
  int64_t w0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5, nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t k = w0; k < nnz; k += nw) {
    int r = nzrow[k], s = col[k];
    if (s < r) continue;   // written with (s, r)
    int p = row_pair[r], vi = ci[p], vj = cj[p];
    int ps = row_pair[s], si = ci[ps], sj = cj[ps];
    int64_t rA = s < r ? s : r, rB = s < r ? r : s;
    int aI = s < r ? si : vi, bI = s < r ? vi : si;   // first vesicles of rows A and B
    double acc = 0.0;
    for (int t = 0; t < 2; ++t) {
      int v = t ? vj : vi;   // vi < vj: ascending
      if (v != si && v != sj) continue;
      int64_t a0, a1, b0, b1;
      side_range(sbeg, scnt, rA, v == aI ? 0 : 1, a0, a1);
      side_range(sbeg, scnt, rB, v == bI ? 0 : 1, b0, b1);
      double part = 0.0, sa[3] = {0.0, 0.0, 0.0}, sb[3] = {0.0, 0.0, 0.0};
      if (rA == rB) {
#pragma unroll 4
        for (int64_t i = a0 + lane; i < a1; i += 32) {
          double x = ug[3 * i], y = ug[3 * i + 1], z = ug[3 * i + 2];
          part += x * x + y * y + z * z;
          sa[0] += x; sa[1] += y; sa[2] += z;
        }
      } else {
#pragma unroll 4
        for (int64_t i = b0 + lane; i < b1; i += 32) {
          tab[ukey[i]] = (int32_t)(i - b0);
          for (int d = 0; d < 3; ++d) sb[d] += ug[3 * i + d];
        }
        __syncwarp();
#pragma unroll 4
        for (int64_t i = a0 + lane; i < a1; i += 32) {
          int32_t jb = tab[ukey[i]];   // vertex id (the sides may differ)
          if (jb >= 0) {
            int64_t lo = b0 + jb;
            part += ug[3 * i] * ug[3 * lo] + ug[3 * i + 1] * ug[3 * lo + 1] + ug[3 * i + 2] * ug[3 * lo + 2];
          }
          for (int d = 0; d < 3; ++d) sa[d] += ug[3 * i + d];
        }
        __syncwarp();
        for (int64_t i = b0 + lane; i < b1; i += 32) tab[ukey[i]] = -1;
        __syncwarp();
      }
      for (int off = 16; off > 0; off >>= 1) part += __shfl_xor_sync(0xffffffffu, part, off);
      acc += (m_ves ? m_ves[v] : 1.0) * part;
      if (t_ves) {   // rigid translation: (sum of g_A over v's points) . (sum of g_B)
        for (int off = 16; off > 0; off >>= 1)
          for (int d = 0; d < 3; ++d) {
            sa[d] += __shfl_xor_sync(0xffffffffu, sa[d], off);
            sb[d] += __shfl_xor_sync(0xffffffffu, sb[d], off);
          }
        bool dg = rA == rB;
        double b0s = dg ? sa[0] : sb[0], b1s = dg ? sa[1] : sb[1], b2s = dg ? sa[2] : sb[2];
        acc += t_ves[v] * (sa[0] * b0s + sa[1] * b1s + sa[2] * b2s);
      }
    }
    if (lane == 0) {
      val[k] = acc;
      if (s > r) {   // (s, r): among row s's columns
        int64_t lo = row_ptr[s], hi = row_ptr[s + 1];
        if (hi > nnz) hi = nnz;
        while (lo < hi) { int64_t mid = (lo + hi) >> 1; if (col[mid] < r) lo = mid + 1; else hi = mid; }
        if (lo < nnz && nzrow[lo] == s && col[lo] == r) val[lo] = acc;
      }
    }
  }
}

// ---------------------------------------------------------------------------
// min-map Newton, one CTA
// ---------------------------------------------------------------------------
// The solve runs on one SM, and GB300's FP64 pipe is narrow (about two FP64
// FMAs per clock per SM), so it is an inexact Newton method: the outer loop
// (Phi, the merit, the Armijo line search, the right-hand side of the Newton
// system and the free part of the direction, dx_F = -x_F) is FP64, and the
// Newton system on the active set is solved by a Jacobi-preconditioned CG in
// FP32 (B rounded to FP32) to a relative residual of 1e-6.  Convergence is
// decided by the FP64 residual max |Phi| <= tol.
struct solve_args {
  const int64_t* dims;
  const int64_t* row_ptr;
  const int32_t* col;
  const double* val;
  float* valf;    // B's values in FP32
  const double* q;
  double* x;      // lambda
  double* w;      // B x
  double* dx;     // Newton direction
  double* xn;
  float* y;       // CG iterate: dx on the active set
  float* r;
  float* pv;
  float* Ap;
  float* dinv;    // 1 / B_ii (Jacobi preconditioner)
  unsigned char* act;
  double tol;
  int max_newton, max_cg;
  double* info;   // [0] Newton iterations, [1] max |Phi|, [2] CG iterations, [3] status
};

// Block reductions in a fixed order: butterfly within each warp, then warp 0
// over the RT / 32 partial results.  sh holds >= 2 * (RT / 32) + 2 values.
template <class T>
__device__ void block_sum2(T& a, T& b, T* sh) {
  for (int off = 16; off > 0; off >>= 1) {
    a += __shfl_xor_sync(0xffffffffu, a, off);
    b += __shfl_xor_sync(0xffffffffu, b, off);
  }
  int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (lane == 0) { sh[w] = a; sh[RT / 32 + w] = b; }
  __syncthreads();
  if (w == 0) {
    a = sh[lane]; b = sh[RT / 32 + lane];
    for (int off = 16; off > 0; off >>= 1) {
      a += __shfl_xor_sync(0xffffffffu, a, off);
      b += __shfl_xor_sync(0xffffffffu, b, off);
    }
    if (lane == 0) { sh[2 * (RT / 32)] = a; sh[2 * (RT / 32) + 1] = b; }
  }
  __syncthreads();
  a = sh[2 * (RT / 32)]; b = sh[2 * (RT / 32) + 1];
  __syncthreads();
}
__device__ double block_max(double v, double* sh) {
  for (int off = 16; off > 0; off >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, off));
  int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (lane == 0) sh[w] = v;
  __syncthreads();
  if (w == 0) {
    v = sh[lane];
    for (int off = 16; off > 0; off >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, off));
    if (lane == 0) sh[RT / 32] = v;
  }
  __syncthreads();
  double r = sh[RT / 32];
  __syncthreads();
  return r;
}

// psi = |Phi(x)|^2 / 2 with Phi = min(x, B x + q), y = B x (FP64); res = max |Phi|
__device__ double merit(const solve_args& a, int64_t n, const double* x, double* y, double* sh, double& res) {
  double s = 0.0, m = 0.0;
  for (int64_t i = threadIdx.x; i < n; i += RT) {
    double t = 0.0;
    for (int64_t k = a.row_ptr[i]; k < a.row_ptr[i + 1]; ++k) t += a.val[k] * x[a.col[k]];
    y[i] = t;
    double ph = fmin(x[i], t + a.q[i]);
    s += ph * ph;
    m = fmax(m, fabs(ph));
  }
  res = block_max(m, sh);
  double z = 0.0;
  block_sum2(s, z, sh);
  return 0.5 * s;
}

// Ap = B_AA pv on the active set (FP32), 0 elsewhere; returns pv . Ap
__device__ float spmv_active(const solve_args& a, int64_t n, float* shf) {
  float d = 0.0f, z = 0.0f;
  for (int64_t i = threadIdx.x; i < n; i += RT) {
    float t = 0.0f;
    if (a.act[i]) {
      for (int64_t k = a.row_ptr[i]; k < a.row_ptr[i + 1]; ++k) {
        int j = a.col[k];
        if (a.act[j]) t += a.valf[k] * a.pv[j];
      }
      d += a.pv[i] * t;
    }
    a.Ap[i] = t;
  }
  block_sum2(d, z, shf);
  return d;
}

constexpr size_t SOLVE_SMEM = 220 * 1024;   // dynamic shared memory of the solve CTA

__device__ __forceinline__ size_t al16(size_t x) { return (x + 15) & ~(size_t)15; }

// When the vectors, q and B (FP64 and FP32 values) fit in the CTA's shared
// memory (smem_bytes) they are staged there and every iteration runs out of
// it; otherwise the handle's global scratch holds them.
__global__ void __launch_bounds__(RT) solve_kernel(solve_args g, size_t smem_bytes) {
  extern __shared__ __align__(16) unsigned char dsm[];
  __shared__ double sh[2 * (RT / 32) + 2];
  __shared__ float shf[2 * (RT / 32) + 2];
  solve_args a = g;
  int64_t n = g.dims[0], nnz = g.dims[1];
  if (g.dims[2]) {   // matrix over capacity
    if (threadIdx.x == 0) { g.info[0] = 0; g.info[1] = -1; g.info[2] = 0; g.info[3] = 1; }
    return;
  }
  size_t need = 4 * al16(8 * (size_t)n) + 5 * al16(4 * (size_t)n) + al16((size_t)n) + al16(8 * (size_t)(n + 1)) +
                al16(4 * (size_t)nnz) + al16(8 * (size_t)nnz) + al16(4 * (size_t)nnz) + al16(8 * (size_t)n);
  bool in_smem = need <= smem_bytes;
  if (in_smem) {
    unsigned char* p = dsm;
    auto take = [&](size_t bytes) { unsigned char* r = p; p += al16(bytes); return r; };
    a.x = (double*)take(8 * n); a.w = (double*)take(8 * n); a.dx = (double*)take(8 * n);
    a.xn = (double*)take(8 * n);
    a.y = (float*)take(4 * n); a.r = (float*)take(4 * n); a.pv = (float*)take(4 * n);
    a.Ap = (float*)take(4 * n); a.dinv = (float*)take(4 * n);
    a.act = take(n);
    double* qs = (double*)take(8 * n);
    int64_t* rp = (int64_t*)take(8 * (n + 1));
    int32_t* cs = (int32_t*)take(4 * nnz);
    double* vs = (double*)take(8 * nnz);
    a.valf = (float*)take(4 * nnz);
    for (int64_t i = threadIdx.x; i <= n; i += RT) rp[i] = g.row_ptr[i];
    for (int64_t k = threadIdx.x; k < nnz; k += RT) { cs[k] = g.col[k]; vs[k] = g.val[k]; }
    for (int64_t i = threadIdx.x; i < n; i += RT) qs[i] = g.q[i];
    a.row_ptr = rp; a.col = cs; a.val = vs; a.q = qs;
    __syncthreads();
  }
  for (int64_t k = threadIdx.x; k < nnz; k += RT) a.valf[k] = (float)a.val[k];
  for (int64_t i = threadIdx.x; i < n; i += RT) {
    a.x[i] = 0.0;
    double d = 0.0;
    for (int64_t k = a.row_ptr[i]; k < a.row_ptr[i + 1]; ++k)
      if (a.col[k] == i) d = a.val[k];
    a.dinv[i] = d > 0.0 ? (float)(1.0 / d) : 1.0f;
  }
  __syncthreads();
  long long cg_total = 0;
  int it = 0;
  double res = 0.0;
  double psi = merit(a, n, a.x, a.w, sh, res);   // w = B x
  for (it = 0;; ++it) {
    if (res <= a.tol || it == a.max_newton) break;
    // active set; dx_F = -x_F
    for (int64_t i = threadIdx.x; i < n; i += RT) {
      bool ac = a.w[i] + a.q[i] < a.x[i];
      a.act[i] = ac;
      a.dx[i] = ac ? 0.0 : -a.x[i];
    }
    __syncthreads();
    // rhs_A = -(B x + q)_A - B_{A,F} dx_F (FP64, then FP32); PCG from y = 0
    float rz = 0.0f, rr = 0.0f;
    for (int64_t i = threadIdx.x; i < n; i += RT) {
      float ri = 0.0f;
      if (a.act[i]) {
        double s = 0.0;
        for (int64_t k = a.row_ptr[i]; k < a.row_ptr[i + 1]; ++k) {
          int j = a.col[k];
          if (!a.act[j]) s += a.val[k] * a.dx[j];
        }
        ri = (float)(-(a.w[i] + a.q[i]) - s);
      }
      a.r[i] = ri;
      a.y[i] = 0.0f;
      float z = ri * a.dinv[i];
      a.pv[i] = z;
      rz += ri * z; rr += ri * ri;
    }
    block_sum2(rz, rr, shf);
    float rr0 = rr;
    for (int k = 0; k < a.max_cg && rr > 1e-12f * rr0 && rr > 0.0f; ++k) {
      float pAp = spmv_active(a, n, shf);
      if (!(pAp > 0.0f)) break;
      float al = rz / pAp, rzn = 0.0f, rn = 0.0f;
      for (int64_t i = threadIdx.x; i < n; i += RT)
        if (a.act[i]) {
          a.y[i] += al * a.pv[i];
          float ri = a.r[i] - al * a.Ap[i];
          a.r[i] = ri;
          rzn += ri * ri * a.dinv[i];
          rn += ri * ri;
        }
      block_sum2(rzn, rn, shf);
      float be = rzn / rz;
      for (int64_t i = threadIdx.x; i < n; i += RT) a.pv[i] = a.act[i] ? a.r[i] * a.dinv[i] + be * a.pv[i] : 0.0f;
      __syncthreads();
      rz = rzn; rr = rn;
      ++cg_total;
    }
    for (int64_t i = threadIdx.x; i < n; i += RT)
      if (a.act[i]) a.dx[i] = (double)a.y[i];
    __syncthreads();
    // Armijo line search on psi along x + t dx (FP64); w = B xn of the accepted step
    double t = 1.0, pn = psi, rn = res;
    for (int h = 0; h < 40; ++h) {
      for (int64_t i = threadIdx.x; i < n; i += RT) a.xn[i] = a.x[i] + t * a.dx[i];
      __syncthreads();
      pn = merit(a, n, a.xn, a.w, sh, rn);
      if (pn <= (1.0 - 2.0e-4 * t) * psi) break;
      t *= 0.5;
    }
    for (int64_t i = threadIdx.x; i < n; i += RT) a.x[i] = a.xn[i];
    __syncthreads();
    psi = pn; res = rn;
  }
  if (in_smem)
    for (int64_t i = threadIdx.x; i < n; i += RT) g.x[i] = a.x[i];
  if (threadIdx.x == 0) { g.info[0] = it; g.info[1] = res; g.info[2] = (double)cg_total; g.info[3] = res <= a.tol ? 0 : 2; }
}

size_t al256(size_t x) { return (x + 255) & ~(size_t)255; }

}  // namespace

extern "C" int stiv_lcp_matrix(stiv_handle* h, void* stream, int32_t n_ves, int32_t p_max, const stiv_pairs* cand,
                               const stiv_contacts* ct, const int64_t* counts_dev, const double* V_pair_dev,
                               const double* grad_dev, const int32_t* g_ves_dev, const int32_t* g_vid_dev,
                               const double* m_ves_dev, const double* t_ves_dev, const stiv_lcp* lcp) {
  if (!h || !cand || !ct || !counts_dev || !V_pair_dev || !grad_dev || !g_ves_dev || !g_vid_dev || !lcp)
    return STIV_ERR_ARG;
  if (n_ves < 1 || p_max < 1 || p_max > STIV_MAX_P || lcp->row_capacity < 1 || lcp->nnz_capacity < 1 ||
      lcp->row_capacity >= ((int64_t)1 << 30) || !lcp->row_pair || !lcp->q || !lcp->row_ptr || !lcp->col ||
      !lcp->val || !lcp->dims || !cand->i || !cand->j || !ct->pair)
    return STIV_ERR_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  int64_t pcap = cand->capacity, ccap = ct->capacity, rcap = lcp->row_capacity;
  int64_t E = 4 * ccap;
  if (E >= ((int64_t)1 << 31)) return STIV_ERR_ARG;
  const int nv = stiv_nverts(2 * p_max);
  // scratch (handle-owned, grown on demand); pstart, pend, vcnt and the segments'
  // count (after vcnt) are cleared together
  size_t o = 0;
  size_t o_ps = o; o = al256(o + sizeof(int32_t) * pcap);
  size_t o_pe = o; o = al256(o + sizeof(int32_t) * pcap);
  size_t o_vc = o; o = al256(o + sizeof(int32_t) * ((size_t)n_ves + 1));
  const size_t clear = o;
  size_t o_sd = o; o = al256(o + sizeof(int32_t) * 2 * rcap);
  const int64_t scap = ccap / SEG_C + 1;   // listed segments: a long row has less than its contacts / SEG_C
  size_t o_sr = o; o = al256(o + sizeof(int32_t) * scap);
  size_t o_sf = o; o = al256(o + sizeof(int32_t) * rcap);
  size_t o_sb = o; o = al256(o + sizeof(int32_t) * 2 * (rcap + scap));
  size_t o_sc = o; o = al256(o + sizeof(int32_t) * 2 * (rcap + scap));
  size_t o_bc = o; o = al256(o + sizeof(int32_t) * rcap);
  size_t o_nr = o; o = al256(o + sizeof(int32_t) * lcp->nnz_capacity);
  size_t o_uk = o; o = al256(o + sizeof(int32_t) * E);
  size_t o_ug = o; o = al256(o + sizeof(double) * 3 * E);
  size_t o_l1 = o; o = al256(o + sizeof(int32_t) * 2 * rcap);
  size_t o_l2 = o; o = al256(o + sizeof(int32_t) * 2 * rcap);
  size_t o_vs = o; o = al256(o + sizeof(int32_t) * (n_ves + 1));
  if (o > h->lcp_ws_bytes) {
    if (h->lcp_ws) { STIV_CUDA(h, cudaFree(h->lcp_ws)); h->lcp_ws = nullptr; h->lcp_ws_bytes = 0; }
    STIV_CUDA(h, cudaMalloc(&h->lcp_ws, o));
    h->lcp_ws_bytes = o;
  }
  char* w = (char*)h->lcp_ws;
  int32_t* pstart = (int32_t*)(w + o_ps); int32_t* pend = (int32_t*)(w + o_pe);
  int32_t* vcnt = (int32_t*)(w + o_vc);
  seg_list segs;
  segs.count = vcnt + n_ves; segs.row = (int32_t*)(w + o_sr); segs.first = (int32_t*)(w + o_sf);
  segs.done = (int32_t*)(w + o_sd); segs.rcap = rcap;
  int32_t* sbeg = (int32_t*)(w + o_sb); int32_t* scnt = (int32_t*)(w + o_sc);
  int32_t* bcnt = (int32_t*)(w + o_bc);
  int32_t* nzrow = (int32_t*)(w + o_nr);
  int32_t* ukey = (int32_t*)(w + o_uk);
  double* ug = (double*)(w + o_ug);
  int32_t* lst = (int32_t*)(w + o_l1); int32_t* vrow = (int32_t*)(w + o_l2);
  int32_t* vstart = (int32_t*)(w + o_vs);
  int sms = 152;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, h->device);
  // one vertex-index table per warp: as many warps per CTA as 96 KB holds
  int nvtab = nv;
  int bw = (int)((96 * 1024) / (sizeof(int32_t) * (size_t)nvtab));
  bw = bw < 1 ? 1 : (bw > 8 ? 8 : bw);
  size_t bsmem = sizeof(int32_t) * (size_t)nvtab * bw;
  // both limits before the first launch, so that no call is refused halfway (a
  // table of order 32 beside row_sides_kernel's own arrays passes 48 KB)
  STIV_SMEM(h, row_sides_kernel, side_table_bytes(nv), SIDE_SMEM, side_table_bytes(stiv_nverts(2 * STIV_MAX_P)));
  STIV_SMEM(h, bval_kernel, bsmem, 0, 96 * 1024);
  STIV_PROF_N(h, st, "lcp_matrix", 11);
  STIV_CUDA(h, cudaMemsetAsync(w, 0, clear, st));
  // every kernel reads what the ones before it wrote: none is launched after one
  // that was refused
  bounds_kernel<<<sms * 4, 256, 0, st>>>(counts_dev, ccap, ct->pair, pstart, pend);
  STIV_LAUNCH(h);
  rows_kernel<<<1, RT, 0, st>>>(counts_dev, pcap, ccap, pstart, pend, V_pair_dev, rcap, lcp->row_pair, lcp->q,
                                lcp->dims, segs);
  STIV_LAUNCH(h);
  row_sides_kernel<<<sms * 6, ST, side_table_bytes(nv), st>>>(
      lcp->dims, lcp->row_pair, pstart, pend, cand->i, g_ves_dev, g_vid_dev, grad_dev, nv,
      (((uintptr_t)g_ves_dev | (uintptr_t)g_vid_dev) & 15) == 0, segs, sbeg, scnt, ukey, ug);
  STIV_LAUNCH(h);
  ves_count_kernel<<<sms, 256, 0, st>>>(lcp->dims, lcp->row_pair, cand->i, cand->j, vcnt);
  STIV_LAUNCH(h);
  ves_scan_kernel<<<1, RT, 0, st>>>(n_ves, vcnt, vstart);
  STIV_LAUNCH(h);
  ves_fill_kernel<<<sms, 256, 0, st>>>(lcp->dims, lcp->row_pair, cand->i, cand->j, vcnt, lst);
  STIV_LAUNCH(h);
  ves_rank_kernel<<<sms, 256, 0, st>>>(n_ves, vstart, lst, vrow);
  STIV_LAUNCH(h);
  bcount_kernel<<<sms, 256, 0, st>>>(lcp->dims, lcp->row_pair, cand->i, cand->j, vrow, vstart, bcnt);
  STIV_LAUNCH(h);
  bscan_kernel<<<1, RT, 0, st>>>(lcp->dims, bcnt, lcp->nnz_capacity, lcp->row_ptr);
  STIV_LAUNCH(h);
  bcol_kernel<<<sms, 256, 0, st>>>(lcp->dims, lcp->row_pair, cand->i, cand->j, vrow, vstart, lcp->row_ptr,
                                   lcp->nnz_capacity, lcp->col, nzrow);
  STIV_LAUNCH(h);
  bval_kernel<<<sms * 4, 32 * bw, bsmem, st>>>(lcp->dims, lcp->row_pair, cand->i, cand->j, sbeg, scnt, ukey, ug,
                                               m_ves_dev, t_ves_dev, nvtab, lcp->nnz_capacity, lcp->row_ptr, lcp->col, nzrow,
                                               lcp->val);
  STIV_LAUNCH(h);
  return STIV_OK;
}

extern "C" int stiv_lcp_solve(stiv_handle* h, void* stream, const stiv_lcp* lcp, double tol, int32_t max_newton,
                              int32_t max_cg, double* lambda_dev, double* info_dev) {
  if (!h || !lcp || !lambda_dev || !info_dev || !lcp->dims || !lcp->row_ptr || !lcp->col || !lcp->val || !lcp->q)
    return STIV_ERR_ARG;
  if (!(tol > 0.0) || max_newton < 1 || max_cg < 1 || lcp->row_capacity < 1 || lcp->nnz_capacity < 1)
    return STIV_ERR_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  int64_t n = lcp->row_capacity, nz = lcp->nnz_capacity;
  size_t o = 0;
  size_t o_w = o; o = al256(o + sizeof(double) * n);
  size_t o_dx = o; o = al256(o + sizeof(double) * n);
  size_t o_xn = o; o = al256(o + sizeof(double) * n);
  size_t o_y = o; o = al256(o + sizeof(float) * n);
  size_t o_r = o; o = al256(o + sizeof(float) * n);
  size_t o_p = o; o = al256(o + sizeof(float) * n);
  size_t o_ap = o; o = al256(o + sizeof(float) * n);
  size_t o_di = o; o = al256(o + sizeof(float) * n);
  size_t o_act = o; o = al256(o + n);
  size_t o_vf = o; o = al256(o + sizeof(float) * nz);
  if (o > h->lcp_ws2_bytes) {
    if (h->lcp_ws2) { STIV_CUDA(h, cudaFree(h->lcp_ws2)); h->lcp_ws2 = nullptr; h->lcp_ws2_bytes = 0; }
    STIV_CUDA(h, cudaMalloc(&h->lcp_ws2, o));
    h->lcp_ws2_bytes = o;
  }
  char* w = (char*)h->lcp_ws2;
  solve_args a;
  a.dims = lcp->dims; a.row_ptr = lcp->row_ptr; a.col = lcp->col; a.val = lcp->val; a.q = lcp->q;
  a.x = lambda_dev; a.w = (double*)(w + o_w); a.dx = (double*)(w + o_dx); a.xn = (double*)(w + o_xn);
  a.y = (float*)(w + o_y); a.r = (float*)(w + o_r); a.pv = (float*)(w + o_p); a.Ap = (float*)(w + o_ap);
  a.dinv = (float*)(w + o_di);
  a.act = (unsigned char*)(w + o_act);
  a.valf = (float*)(w + o_vf);
  a.tol = tol; a.max_newton = max_newton; a.max_cg = max_cg; a.info = info_dev;
  STIV_PROF(h, st, "lcp_solve");
  size_t smem = SOLVE_SMEM;
  if (cudaFuncSetAttribute(solve_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SOLVE_SMEM) != cudaSuccess) {
    cudaGetLastError();
    smem = 0;   // everything in global scratch
  }
  solve_kernel<<<1, RT, smem, st>>>(a, smem);
  STIV_LAUNCH(h);
  return STIV_OK;
}
