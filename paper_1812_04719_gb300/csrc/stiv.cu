// Contact volumes (Eq. 3.2, App. A) and their gradient with respect to the
// end-of-step positions X1 (Sec. 3.1.2, Sec. 3.3.2), per contact and summed
// per vesicle pair (Alg. 2); the adjoint of the upsampling back to SH
// coefficients; ordering of the contact list.
//
// Per contact, with positions Y = X0 + tau D at the contact time tau and
// D = X1 - X0:
//   V = 1/2 (1 - tau) sqrt((eps dt)^2 |m|^2 + (D_rel . m)^2)
// which is Eq. 3.2, (t - tau_I) sqrt(eps^2 + (U . n)^2) |t|, with t - tau_I =
// (1 - tau) dt, U = D_rel / dt the velocity of the contact point relative to
// the opposite primitive, n = m / |m| and |t| = |m| / 2.  VF: m = (x1-x0) x
// (x2-x0), D_rel = D_p - sum_k beta_k D_k.  EE: m = d1 x d2 (same weight),
// D_rel = D_q(u) - D_p(s).
//
// The gradient is reverse mode written out by hand: V depends on X1 through
// D, through Y, through the weights (beta or s, u: least-squares solutions
// of the inside test) and through tau, an implicit function of X1 via
// f(tau) = 0 (Eq. 3.1): d tau / dX1_q = -tau (df/dY_q) / f'(tau) (stiv_one).
#include "stiv_internal.cuh"

#include <math.h>

namespace {

__device__ __forceinline__ d3 mk(double x, double y, double z) { return {x, y, z}; }
__device__ __forceinline__ d3 operator+(d3 a, d3 b) { return {a.x + b.x, a.y + b.y, a.z + b.z}; }
__device__ __forceinline__ d3 operator-(d3 a, d3 b) { return {a.x - b.x, a.y - b.y, a.z - b.z}; }
__device__ __forceinline__ d3 operator-(d3 a) { return {-a.x, -a.y, -a.z}; }
__device__ __forceinline__ d3 operator*(double s, d3 a) { return {s * a.x, s * a.y, s * a.z}; }
__device__ __forceinline__ double dot(d3 a, d3 b) { return fma(a.z, b.z, fma(a.y, b.y, a.x * b.x)); }
__device__ __forceinline__ d3 cross(d3 a, d3 b) {
  return {fma(a.y, b.z, -(a.z * b.y)), fma(a.z, b.x, -(a.x * b.z)), fma(a.x, b.y, -(a.y * b.x))};
}

__device__ __forceinline__ d3 axpy(double s, d3 a, d3 b) { return {fma(s, a.x, b.x), fma(s, a.y, b.y), fma(s, a.z, b.z)}; }

// V and dV/dX1 (g, with VAR also dV/dX0, g0) of one contact.
//
// Both kinds are the same expression of three difference vectors at tau: a, b
// the triangle's edges from its first vertex (VF) or the two edges (EE), c from
// that vertex to the vertex (VF) or from the first edge's first point to the
// second's (EE).  With the weights (w1, w2) = (b1, b2) (VF) or (s, -u) (EE) the
// relative displacement is Dr = c' - w1 a' - w2 b' (' the differences'
// displacements), (w1, w2) the least-squares solution of c ~ w1 a + w2 b, and f =
// c . (a x b).  So the adjoints are formed for a, b and c and distributed over
// the points at the end: x = P, Q, H, G with c = P - Q, a = H - Q, b = G - Q (VF:
// xp, x0, x1, x2) or G - P (EE: q0, p0, p1, q1).
//
// Reverse mode: adjoints of the vectors at tau (ab, bb, w), of their
// displacements and of tau (taub); with Y = X0 + tau D, D = X1 - X0 and tau
// moving along f(tau; X) = 0, dV/dX1 = Db + tau Yb - taub tau fY / f' and dV/dX0 =
// -Db + (1 - tau) Yb - taub (1 - tau) fY / f'.  dm2 = d_m^2 > 0: tau is a root of
// g = f^2 - d_m^2 |m|^2 (Eq. 3.1, degree six) and fY, f' are those of g.  vabs: U_k
// read as the absolute velocity of the contact point (the literal reading: VF
// the vertex's displacement, EE that of the point p(s) on the first edge).
// VAR = false compiles the common case (relative velocity, d_m = 0, no X0 rows)
// without the variants' code.
//
// Bound by the FP64 pipe: the library is built without contraction, so every
// multiply-add is written as one; with both kinds on one path about 260 FP64
// instructions per contact instead of 406: 0.55 -> 0.31 ms at 1440 vesicles (636k
// contacts).
template <bool VAR>
__device__ __forceinline__ double stiv_one(bool ee, const d3* x0, const d3* x1, double tau, double w1, double w2,
                                           double e2, int vabs, double dm2, bool want, d3* g, bool want0, d3* g0) {
  if (!VAR) { vabs = 0; dm2 = 0.0; want0 = false; }
  // displacements and positions at tau per point (rounded as the contact test's
  // positions are), then the vectors
  d3 D[4], Y[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) { D[q] = x1[q] - x0[q]; Y[q] = axpy(tau, D[q], x0[q]); }
  const d3 Yb = {ee ? Y[0].x : Y[1].x, ee ? Y[0].y : Y[1].y, ee ? Y[0].z : Y[1].z};
  const d3 Db = {ee ? D[0].x : D[1].x, ee ? D[0].y : D[1].y, ee ? D[0].z : D[1].z};
  const d3 a = Y[2] - Y[1], b = Y[3] - Yb, c = Y[0] - Y[1];
  const d3 da = D[2] - D[1], db = D[3] - Db, dc = D[0] - D[1];
  const double q2 = ee ? -w2 : w2;
  const d3 m = cross(a, b);
  d3 Dr;
  if (VAR && vabs) Dr = ee ? axpy(w1, da, D[1]) : D[0];
  else Dr = axpy(-w1, da, axpy(-q2, db, dc));
  const double dm = dot(Dr, m);
  const double Q = fma(dm, dm, e2 * dot(m, m));
  const double rS = rsqrt(Q);            // 1 / sqrt(Q): no division in the adjoint below
  const double S = Q > 0.0 ? Q * rS : 0.0;
  const double rest = 1.0 - tau, half = 0.5 * rest;
  const double V = half * S;
  if (!want && !want0) return V;
  const double qb = half * rS;           // 2 dV/dQ
  const double be = qb * dm;
  const d3 mb = axpy(qb * e2, m, be * Dr), Drb = be * m;
  double z1, z2;
  {
    const double daa = dot(a, a), dab = dot(a, b), dbb = dot(b, b);
    const double iden = 1.0 / fma(daa, dbb, -(dab * dab));
    double h1 = -dot(Drb, da), h2 = -dot(Drb, db);
    if (VAR && vabs) { h1 = ee ? -h1 : 0.0; h2 = 0.0; }
    z1 = fma(dbb, h1, -(dab * h2)) * iden;
    z2 = fma(daa, h2, -(dab * h1)) * iden;
  }
  // least squares (w1, w2) = M^-1 G^T c, G = [a b]
  const d3 w = axpy(z1, a, z2 * b);
  const d3 res = axpy(-w1, a, axpy(-q2, b, c));
  const d3 ab = axpy(z1, res, axpy(-w1, w, cross(b, mb)));
  const d3 bb = axpy(z2, res, axpy(-q2, w, cross(mb, a)));
  // df/dY of f = c . (a x b)
  d3 fc = m, fa = cross(b, c), fb = cross(c, a);
  if (VAR && dm2 > 0.0) {   // d|m|^2 / da = 2 b x m, db = 2 m x a
    const double f2 = 2.0 * dot(c, m);
    fc = f2 * fc;
    fa = axpy(-2.0 * dm2, cross(b, m), f2 * fa);
    fb = axpy(-2.0 * dm2, cross(m, a), f2 * fb);
  }
  const double taub = fma(-0.5, S, dot(w, dc) + (dot(ab, da) + dot(bb, db)));
  const double fp = dot(fc, dc) + (dot(fa, da) + dot(fb, db));
  // to the vectors, then to the points; e1: the sign of Drb and the weight of
  // the adjoints at tau
  auto rows = [&](double at, double e1, d3* o) {
    const double kap = -(taub * at / fp);
    d3 Gc = axpy(kap, fc, at * w), Ga = axpy(kap, fa, at * ab), Gb = axpy(kap, fb, at * bb), ex = {0.0, 0.0, 0.0};
    if (VAR && vabs) {
      ex = e1 * Drb;   // of the point itself
      if (ee) Ga = axpy(e1 * w1, Drb, Ga);
    } else {
      Gc = e1 > 0.0 ? Gc + Drb : Gc - Drb;
      Ga = axpy(-e1 * w1, Drb, Ga);
      Gb = axpy(-e1 * q2, Drb, Gb);
    }
    const d3 sub = {ee ? Gb.x : 0.0, ee ? Gb.y : 0.0, ee ? Gb.z : 0.0};
    const d3 P = Gc - sub;
    const d3 R = -((Gc + Ga) + (Gb - sub));
    o[0] = P; o[1] = R; o[2] = Ga; o[3] = Gb;
    if (VAR && vabs) o[ee ? 1 : 0] = o[ee ? 1 : 0] + ex;
  };
  if (want) rows(tau, 1.0, g);
  if (VAR && want0) rows(rest, -1.0, g0);
  return V;
}

struct stiv_args {
  const int32_t* pv;
  const int64_t* voff;
  const void* X;
  int mixed;
  double L[3];
  const int32_t* ci; const int32_t* cj; const int32_t* cs;
  const int32_t* pair; const int32_t* type; const int32_t* a; const int32_t* b; const double* tau; const double* w;
  const int64_t* counts;
  int64_t cap;
  double e2;
  double dm2;      // d_m^2 (0: the cubic of Eq. 3.1)
  int vabs;
  double* Vc;
  double* grad;
  double* grad0;   // dV/dX0 rows (or NULL)
  int32_t* gves;
  int32_t* gvid;
  bool vec;        // the row and id arrays allow 16-byte stores
};

// X0 and X1 of vertex k of a vesicle at base (its vertices, order nv), shifted
// by sh where the axis' bit of mask is set (the pair's periodic image).
__device__ __forceinline__ void vpos(const stiv_args& A, size_t base, int nv, int k, int mask, const double* sh, d3& p0,
                                     d3& p1) {
  double x[6];
#pragma unroll
  for (int c = 0; c < 6; ++c) {
    size_t idx = base + (size_t)c * nv + k;
    x[c] = A.mixed ? (double)((const float*)A.X)[idx] : ((const double*)A.X)[idx];
  }
#pragma unroll
  for (int c = 0; c < 3; ++c)
    if ((mask >> c) & 1) { x[c] = x[c] + sh[c]; x[3 + c] = x[3 + c] + sh[c]; }
  p0 = {x[0], x[1], x[2]};
  p1 = {x[3], x[4], x[5]};
}

__device__ __forceinline__ int64_t n_contacts(const int64_t* counts, int64_t cap) {
  int64_t n = counts[STIV_C_VF] + counts[STIV_C_EE];
  return n < cap ? n : cap;
}

// One contact's four rows (12 doubles): 16-byte stores where the caller's array
// allows (A.vec), else one by one.
__device__ __forceinline__ void put_rows(double* out, int64_t k, const d3* r, bool vec) {
  double v[12];
#pragma unroll
  for (int q = 0; q < 4; ++q) { v[3 * q] = r[q].x; v[3 * q + 1] = r[q].y; v[3 * q + 2] = r[q].z; }
  if (vec) {
    double2* o = (double2*)(out + 12 * k);
#pragma unroll
    for (int q = 0; q < 6; ++q) o[q] = make_double2(v[2 * q], v[2 * q + 1]);
  } else {
#pragma unroll
    for (int q = 0; q < 12; ++q) out[12 * k + q] = v[q];
  }
}

// VAR: the variants (absolute velocity, d_m > 0, X0 rows) in an instance of
// their own.
template <bool VAR>
__global__ void __launch_bounds__(128, 4) stiv_kernel(stiv_args A) {
  int64_t n = n_contacts(A.counts, A.cap);
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x) {
    const int r = A.pair[k], ty = A.type[k], pa = A.a[k], pb = A.b[k];
    const int vi = A.ci[r], vj = A.cj[r], code = A.cs[r];
    const int Pi = 2 * A.pv[vi], Pj = 2 * A.pv[vj];
    const size_t bi = A.voff[vi], bj = A.voff[vj];
    const double tau = A.tau[k], w1 = A.w[2 * k], w2 = A.w[2 * k + 1];
    double sh[3];
    int mask = 0;
    {
      int s1[3] = {code / 9 - 1, (code / 3) % 3 - 1, code % 3 - 1};
#pragma unroll
      for (int c = 0; c < 3; ++c) { sh[c] = s1[c] * A.L[c]; mask |= s1[c] != 0 ? 1 << c : 0; }
    }
    // the points P, Q, H, G of stiv_one: vertex ids, and whether on vesicle j
    const bool ee = ty == 2;
    int id[4], on;
    if (!ee) {
      int tv[3];
      stiv_tri_verts(ty == 0 ? Pj : Pi, pb, tv);
      id[0] = pa; id[1] = tv[0]; id[2] = tv[1]; id[3] = tv[2];
      on = ty == 0 ? 0xE : 0x1;
    } else {
      stiv_edge_verts(Pi, pa, &id[1], &id[2]);
      stiv_edge_verts(Pj, pb, &id[0], &id[3]);
      on = 0x9;
    }
    d3 x0[4], x1[4];
    const int nvi = stiv_nverts(Pi), nvj = stiv_nverts(Pj);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const bool j = (on >> q) & 1;
      vpos(A, j ? bj : bi, j ? nvj : nvi, id[q], j ? mask : 0, sh, x0[q], x1[q]);
    }
    d3 g[4], g0[4];
    double V = stiv_one<VAR>(ee, x0, x1, tau, w1, w2, A.e2, A.vabs, A.dm2, A.grad != nullptr, g, A.grad0 != nullptr, g0);
    if (A.Vc) A.Vc[k] = V;
    // output order: VF xp, x0, x1, x2; EE p0, p1, q0, q1
    if (A.grad) {
      d3 o[4] = {ee ? g[1] : g[0], ee ? g[2] : g[1], ee ? g[0] : g[2], g[3]};
      put_rows(A.grad, k, o, A.vec);
      int4 vd = ee ? make_int4(id[1], id[2], id[0], id[3]) : make_int4(id[0], id[1], id[2], id[3]);
      int va = ty == 1 ? vj : vi, vb = ty == 1 ? vi : vj;
      int4 vs = make_int4(va, ee ? va : vb, vb, vb);
      if (A.vec) {
        ((int4*)A.gves)[k] = vs;
        ((int4*)A.gvid)[k] = vd;
      } else {
        A.gves[4 * k] = vs.x; A.gves[4 * k + 1] = vs.y; A.gves[4 * k + 2] = vs.z; A.gves[4 * k + 3] = vs.w;
        A.gvid[4 * k] = vd.x; A.gvid[4 * k + 1] = vd.y; A.gvid[4 * k + 2] = vd.z; A.gvid[4 * k + 3] = vd.w;
      }
    }
    if (VAR && A.grad0) {
      d3 o[4] = {ee ? g0[1] : g0[0], ee ? g0[2] : g0[1], ee ? g0[0] : g0[2], g0[3]};
      put_rows(A.grad0, k, o, A.vec);
    }
  }
}

// First k in [0, n) with pair[k] >= r (n: none), by one warp: 32 probes a step.
__device__ __forceinline__ int64_t warp_lower_bound(const int32_t* pair, int64_t n, int64_t r, int lane) {
  int64_t lo = 0, hi = n;   // pair[lo - 1] < r <= pair[hi]
  while (hi - lo > 0) {
    const int64_t step = (hi - lo + 31) / 32, at = lo + lane * step;
    const bool less = at < hi && pair[at] < r;
    const int k = __popc(__ballot_sync(0xffffffffu, less));   // probes below r
    if (k == 0) { hi = lo; break; }
    const int64_t nlo = lo + (k - 1) * step + 1, nhi = lo + k * step;
    lo = nlo;
    hi = nhi < hi ? nhi : hi;
  }
  return lo;
}

// Per candidate pair: sum of its contacts' V (contacts sorted by pair); one
// warp per pair, fixed summation order.  The range is searched 32 ways first, so
// that the sum's loads do not wait for each other (1440 vesicles: 60 -> 17 us).
__global__ void vpair_kernel(const int32_t* pair, const int64_t* counts, int64_t ccap, const double* Vc,
                             int64_t pcap, double* Vp) {
  int lane = threadIdx.x & 31;
  int64_t np = counts[STIV_C_PAIRS]; if (np > pcap) np = pcap;
  int64_t n = n_contacts(counts, ccap);
  int64_t w0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5, nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t r = w0; r < np; r += nw) {
    const int64_t lo = warp_lower_bound(pair, n, r, lane);
    double s = 0.0;
    if (lo < n && pair[lo] == r) {
      const int64_t hi = warp_lower_bound(pair, n, r + 1, lane);
#pragma unroll 4
      for (int64_t k = lo + lane; k < hi; k += 32) s += Vc[k];
    }
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if (lane == 0) Vp[r] = s;
  }
}

// Contact ordering by (pair, type, a, b): counting sort by pair (the FP64 test
// counts), then each pair's segment sorted by its (type, a, b) key.

// Exclusive scan of the per-pair counts (one CTA); counts pairs with contacts and
// writes the detection's counts (every counter is final here).  The work limit of a
// contact capacity (Q3 primitive pairs left by the sign test) is part of the
// interface (STIV_F_WORK_OVERFLOW in stiv.h): capacities that were refused stay
// refused, and callers that grow by it keep the sizes they had, although the
// separation test keeps most of those pairs off the list.
__global__ void __launch_bounds__(1024) pair_scan_kernel(int64_t* ctr, int64_t pcap, int64_t C, int64_t Q3,
                                                         const int32_t* cnt,
                                                         int32_t* off, int64_t* counts, int* tc_status) {
  __shared__ int32_t wsum[32], wnz[32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  int64_t np = ctr[STIV_C_PAIRS]; if (np > pcap) np = pcap;
  int32_t base = 0, z = 0;
  for (int64_t r0 = 0; r0 < np; r0 += 1024) {
    const int64_t r = r0 + threadIdx.x;
    const int32_t c = r < np ? cnt[r] : 0;
    z += c > 0;
    int32_t x = c;
    for (int o = 1; o < 32; o <<= 1) { int32_t y = __shfl_up_sync(0xffffffffu, x, o); if (lane >= o) x += y; }
    if (lane == 31) wsum[w] = x;
    __syncthreads();
    int32_t t = wsum[lane];
    for (int o = 1; o < 32; o <<= 1) { int32_t y = __shfl_up_sync(0xffffffffu, t, o); if (lane >= o) t += y; }
    const int32_t pre = w ? __shfl_sync(0xffffffffu, t, w - 1) : 0;
    if (r < np) off[r] = base + pre + x - c;
    base += __shfl_sync(0xffffffffu, t, 31);
    __syncthreads();
  }
  for (int o = 16; o > 0; o >>= 1) z += __shfl_down_sync(0xffffffffu, z, o);
  if (lane == 0) wnz[w] = z;
  __syncthreads();
  if (threadIdx.x == 0) {
    off[np] = base;
    z = 0;
    for (int q = 0; q < 32; ++q) z += wnz[q];
    ctr[STIV_C_CPAIRS] = z;
    if (ctr[11] > C) ctr[STIV_C_STATUS] |= STIV_F_CONTACTS_OVERFLOW;
    if (ctr[17] > Q3) ctr[STIV_C_STATUS] |= STIV_F_WORK_OVERFLOW;
    if (tc_status && *tc_status) { ctr[STIV_C_STATUS] |= STIV_F_TIMEOUT; *tc_status = 0; }
    for (int k = 0; k < 8; ++k) counts[k] = ctr[k];
    counts[STIV_C_PATCH] -= ctr[18];   // patch pairs, not their work items
    counts[STIV_C_FLOPS] = ctr[12];
    counts[STIV_C_EXACT] = ctr[13];
    counts[STIV_C_PIECE] = ctr[14];
  }
}

__global__ void pair_scatter_kernel(const int64_t* ctr, int64_t C, const int32_t* rp, const int32_t* rt,
                                    const int32_t* ra, const int32_t* rb, const int32_t* off, int32_t* fill,
                                    unsigned long long* seg) {
  int64_t n = ctr[11]; if (n > C) n = C;
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x) {
    int r = rp[k];
    int slot = off[r] + atomicAdd(&fill[r], 1);
    unsigned key = ((unsigned)rt[k] << 30) | ((unsigned)ra[k] << 15) | (unsigned)rb[k];
    seg[slot] = ((unsigned long long)key << 32) | (unsigned long long)(unsigned)k;
  }
}

constexpr int SEG = 2048;        // entries sorted in shared memory at a time
constexpr int SEG_T = 256;       // threads of a sorting CTA

// Stable radix sort of n <= SEG entries of x[0] by the upper 32 bits, 8 bits a
// pass, warps ranking their own entries (as the library's sort): 4 passes, so the
// result is in x[0] again.
__device__ void radix_smem(unsigned long long (*x)[SEG], int (*cnt)[256], int* wsum, int n) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, rounds = (n + SEG_T - 1) / SEG_T;
  int cur = 0;
  for (int shift = 32; shift < 64; shift += 8) {
    for (int q = lane; q < 256; q += 32) cnt[w][q] = 0;
    __syncwarp();
    int rank[SEG / SEG_T];
#pragma unroll
    for (int q = 0; q < SEG / SEG_T; ++q)
      if (q < rounds) {
        const int i = (w * rounds + q) * 32 + lane;
        const bool valid = i < n;
        const unsigned dig = valid ? (unsigned)(x[cur][i] >> shift) & 0xFFu : 0u;
        const unsigned peers = digit_peers<8>(dig, valid), below = peers & ((1u << lane) - 1u);
        const int c = valid ? cnt[w][dig] : 0;
        __syncwarp();
        if (valid && !below) cnt[w][dig] = c + __popc(peers);
        rank[q] = c + __popc(below);
        __syncwarp();
      }
    __syncthreads();
    int run = 0, tot = 0;
    for (int q = 0; q < SEG_T / 32; ++q) { const int c = cnt[q][threadIdx.x]; cnt[q][threadIdx.x] = run; run += c; }
    int s = run;
    for (int o = 1; o < 32; o <<= 1) { int y = __shfl_up_sync(0xffffffffu, s, o); if (lane >= o) s += y; }
    if (lane == 31) wsum[w] = s;
    __syncthreads();
    for (int q = 0; q < w; ++q) tot += wsum[q];
    const int first = tot + s - run;
    for (int q = 0; q < SEG_T / 32; ++q) cnt[q][threadIdx.x] += first;
    __syncthreads();
#pragma unroll
    for (int q = 0; q < SEG / SEG_T; ++q)
      if (q < rounds) {
        const int i = (w * rounds + q) * 32 + lane;
        if (i < n) {
          const unsigned long long e = x[cur][i];
          x[1 - cur][cnt[w][(unsigned)(e >> shift) & 0xFFu] + rank[q]] = e;
        }
      }
    cur = 1 - cur;
    __syncthreads();
  }
}

// One CTA per pair: sort its segment and write its contacts in order; long
// segments are sorted in chunks and merged (each element placed by binary search
// in the other run).  Bound by the latency of its phases: a radix sort of 256
// threads (5 CTAs per SM) instead of a bitonic one of 1024 (2 per SM), the gather
// in the same kernel: ordering at 1440 vesicles 0.165 -> 0.12 ms with the count
// and the final counts moved into neighbouring kernels (6 launches -> 3).
__global__ void __launch_bounds__(SEG_T) pair_sort_kernel(const int64_t* ctr, int64_t pcap, const int32_t* off,
                                                          unsigned long long* seg, unsigned long long* tmp,
                                                          const int32_t* rt, const int32_t* ra, const int32_t* rb,
                                                          const double* rtau, const double* rw, stiv_contacts out) {
  extern __shared__ unsigned long long sx[];
  unsigned long long (*x)[SEG] = (unsigned long long (*)[SEG])sx;
  __shared__ int cnt[SEG_T / 32][256];
  __shared__ int wsum[SEG_T / 32];
  int64_t np = ctr[STIV_C_PAIRS]; if (np > pcap) np = pcap;
  for (int64_t r = blockIdx.x; r < np; r += gridDim.x) {
    const int o = off[r], len = off[r + 1] - o;
    if (len == 0) continue;
    const unsigned long long* src = x[0];
    if (len <= SEG) {
      for (int i = threadIdx.x; i < len; i += SEG_T) x[0][i] = seg[o + i];
      __syncthreads();
      if (len > 1) radix_smem(x, cnt, wsum, len);
    } else {
      for (int c0 = 0; c0 < len; c0 += SEG) {
        const int cl = min(SEG, len - c0);
        for (int i = threadIdx.x; i < cl; i += SEG_T) x[0][i] = seg[o + c0 + i];
        __syncthreads();
        radix_smem(x, cnt, wsum, cl);
        for (int i = threadIdx.x; i < cl; i += SEG_T) seg[o + c0 + i] = x[0][i];
        __syncthreads();
      }
      unsigned long long* from = seg + o;
      unsigned long long* to = tmp + o;
      for (int wdt = SEG; wdt < len; wdt <<= 1) {
        for (int i = threadIdx.x; i < len; i += SEG_T) {
          int run = i / (2 * wdt), a0 = run * 2 * wdt, a1 = min(a0 + wdt, len), b1 = min(a0 + 2 * wdt, len);
          unsigned long long v = from[i];
          int lo = i < a1 ? a1 : a0, hi = i < a1 ? b1 : a1, l0 = lo;   // rank among the other run's smaller elements
          while (lo < hi) { int mid = (lo + hi) >> 1; if (from[mid] < v) lo = mid + 1; else hi = mid; }
          to[a0 + (i - (i < a1 ? a0 : a1)) + (lo - l0)] = v;
        }
        __syncthreads();
        unsigned long long* t = from; from = to; to = t;
      }
      src = from;
    }
    for (int i = threadIdx.x; i < len; i += SEG_T) {
      const int k = (int)(src[i] & 0xFFFFFFFFull);
      const int64_t d = (int64_t)o + i;
      out.pair[d] = (int32_t)r; out.type[d] = rt[k]; out.a[d] = ra[k]; out.b[d] = rb[k];
      out.tau[d] = rtau[k]; out.w[2 * d] = rw[2 * (int64_t)k]; out.w[2 * d + 1] = rw[2 * (int64_t)k + 1];
    }
    __syncthreads();
  }
}

__global__ void scatter_grad_kernel(const int64_t* counts, int64_t cap, const int32_t* pair, const double* wpair,
                                    const double* grad, const int32_t* gves, const int32_t* gvid,
                                    const int32_t* pv, const int64_t* voff, double* gX) {
  int64_t n = n_contacts(counts, cap);
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x) {
    double wgt = wpair ? wpair[pair[k]] : 1.0;
    for (int q = 0; q < 4; ++q) {
      int v = gves[4 * k + q], id = gvid[4 * k + q];
      int nv = stiv_nverts(2 * pv[v]);
      size_t base = voff[v] + (size_t)3 * nv + id;  // X1 block
      for (int c = 0; c < 3; ++c) atomicAdd(&gX[base + (size_t)c * nv], wgt * grad[12 * k + 3 * q + c]);
    }
  }
}

// gcoef = S^T gX for the X1 block; one CTA per (vesicle, coordinate field),
// so that the three fields' phases overlap across CTAs.  S: Legendre step
// then Fourier step, so S^T: Fourier analysis sums per ring, then Legendre
// sums.
//
// Bound by the FP64 pipe, so lanes without work count as much as lanes with: the
// m = 0 sums run with the others (times cos 0 = 1) instead of a loop of their
// own beside every warp, and a thread that takes ring i takes ring P-i with it
// and leaves their sum and difference, so that by Pbar_n^m(-x) = (-1)^(n+m)
// Pbar_n^m(x) the Legendre sums run over half the rings.  1440 vesicles at p = 16:
// 0.44 -> 0.24 ms.
struct adj_args {
  const int32_t* p;
  const int64_t* coef_off;
  const int64_t* vert_off;
  const double* gX;
  double* gcoef;
  const double* leg[STIV_MAX_P + 1];
  const double* trig[STIV_MAX_P + 1];
};

__global__ void __launch_bounds__(256) adjoint_kernel(adj_args a) {
  extern __shared__ double sm[];
  int v = blockIdx.x, f = blockIdx.y;
  if (a.p[v] < 1 || a.p[v] > STIV_MAX_P || !a.leg[a.p[v]]) return;   // order outside [1, p_max]: skipped
  int p = a.p[v], P = 2 * p, nc = (p + 1) * (p + 1), nl = (p + 1) * (p + 2) / 2, ns = 2 * p + 1, W = 2 * P;
  int nv = stiv_nverts(P);
  const int nq = P / 2 + 1, nh = P / 2 + 1;
  double* H = sm;                    // [P+1][ns]   row i < P/2: sum of rings i and P-i, row P-i: their difference
  double* Q = H + (P + 1) * ns;      // [P+1][4][P/2+1] parity combinations of the four symmetric longitudes
  const double* g = a.gX + a.vert_off[v] + (size_t)(3 + f) * nv;
  const double* T = a.trig[p];
  const double* L = a.leg[p];
  double* out = a.gcoef + a.coef_off[v];
  for (int k = threadIdx.x; k < nc; k += blockDim.x) out[f * nc + k] = 0.0;  // X0 block, this field
  // adjoint of the Fourier step.  The forward writes longitudes j, P-j, P+j,
  // 2P-j (j <= P/2, duplicates skipped) from the parity sums Ce, Co, Se, So;
  // their adjoints are the four combinations below.
  for (int task = threadIdx.x; task < (P + 1) * nq; task += blockDim.x) {
    int i = task / nq, j = task - i * nq;
    const double* gr = g + (size_t)i * W;
    int j1 = P - j, j2 = P + j, j3 = (W - j) % W;
    double g0 = gr[j];
    double g1 = (j1 != j) ? gr[j1] : 0.0;
    double g2 = (j2 != j1) ? gr[j2] : 0.0;
    double g3 = (j3 != j && j3 != j2) ? gr[j3] : 0.0;
    double* q = Q + (size_t)i * 4 * nq;
    double s01 = g0 + g1, d01 = g0 - g1, s23 = g2 + g3, d23 = g2 - g3;
    q[0 * nq + j] = s01 + s23;   // cos, even m
    q[1 * nq + j] = d01 - d23;   // cos, odd m
    q[2 * nq + j] = d01 + d23;   // sin, even m
    q[3 * nq + j] = s01 - s23;   // sin, odd m
  }
  __syncthreads();
  for (int task = threadIdx.x; task < nh * ns; task += blockDim.x) {
    int i = task / ns, s = task - i * ns;
    int m = (s + 1) >> 1;
    bool is_sin = s > 0 && (s & 1) == 0;
    const int k = ((is_sin ? 2 : 0) + (m & 1)) * nq;
    const double* qa = Q + (size_t)i * 4 * nq + k;
    const double* qb = Q + (size_t)(P - i) * 4 * nq + k;
    const double* Ts = T + (is_sin ? (p + 1) + m : m);   // m = 0: cos 0 = 1
    double x = 0.0, y = 0.0;
#pragma unroll 2
    for (int j = 0; j < nq; ++j) {
      double c = Ts[(size_t)j * 2 * (p + 1)];
      x = fma(qa[j], c, x);
      y = fma(qb[j], c, y);
    }
    if (i != P - i) {
      H[i * ns + s] = x + y;
      H[(P - i) * ns + s] = x - y;
    } else {
      H[i * ns + s] = x;
    }
  }
  __syncthreads();
  // adjoint of the Legendre step over half the rings (the equator, where odd
  // n + m vanish, with the even ones), and the poles for m = 0
  for (int q = threadIdx.x; q < nc; q += blockDim.x) {
    int n = (int)sqrtf((float)q); while (n * n > q) --n; while ((n + 1) * (n + 1) <= q) ++n;
    int m = q - n * n - n, am = m < 0 ? -m : m;
    int s = m == 0 ? 0 : (m > 0 ? 2 * m - 1 : 2 * am);
    const int e = n * (n + 1) / 2 + am;
    const bool odd = (n + am) & 1;
    const double* Hs = H + s;
    double acc = 0.0;
    for (int i = 0; i < P / 2; ++i) acc = fma(L[(size_t)i * nl + e], Hs[(odd ? P - i : i) * ns], acc);
    if (!odd) acc = fma(L[(size_t)(P / 2) * nl + e], Hs[(P / 2) * ns], acc);
    if (m == 0) {
      acc = fma(L[(size_t)(P + 1) * nl + n * (n + 1) / 2], g[(size_t)W * (P + 1)], acc);
      acc = fma(L[(size_t)(P + 2) * nl + n * (n + 1) / 2], g[(size_t)W * (P + 1) + 1], acc);
    }
    out[3 * nc + f * nc + q] = acc;
  }
}

}  // namespace

int stiv_contact_order(stiv_handle* h, cudaStream_t st, const stiv_pairs* cand, const stiv_contacts* out,
                       detect_ws& w, int64_t* counts) {
  int64_t C = w.C;
  int32_t* rp = w.tmp_i32; int32_t* rt = rp + C; int32_t* ra = rp + 2 * C; int32_t* rb = rp + 3 * C;
  double* rtau = w.tmp_f64; double* rw = w.tmp_f64 + C;
  int64_t pcap = cand->capacity;
  int blocks = (int)((C + 255) / 256); if (blocks > 4096) blocks = 4096; if (blocks < 1) blocks = 1;
  STIV_PROF_N(h, st, "contact_order", 3);
  pair_scan_kernel<<<1, 1024, 0, st>>>(w.ctr, pcap, C, w.Q3, w.pair_cnt, w.pair_off, counts, h->tc_status);
  STIV_LAUNCH(h);
  pair_scatter_kernel<<<blocks, 256, 0, st>>>(w.ctr, C, rp, rt, ra, rb, w.pair_off, w.pair_fill, w.seg);
  STIV_LAUNCH(h);
  const int smem = (int)sizeof(unsigned long long) * 2 * SEG;
  STIV_CUDA(h, cudaFuncSetAttribute(pair_sort_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
  int sblocks = (int)(pcap < 5 * 152 ? pcap : 5 * 152);
  pair_sort_kernel<<<sblocks, SEG_T, smem, st>>>(w.ctr, pcap, w.pair_off, w.seg, w.seg2, rt, ra, rb, rtau, rw, *out);
  STIV_LAUNCH(h);
  return STIV_OK;
}

static int run_stiv(stiv_handle* h, void* stream, const int32_t* p_dev, const int64_t* vert_off_dev,
                    const void* verts_dev, const stiv_pairs* cand, const stiv_contacts* ct, const int64_t* counts_dev,
                    double* Vc, double* Vp, double* grad, int32_t* gves, int32_t* gvid, double* grad0 = nullptr) {
  if (!h || !p_dev || !vert_off_dev || !verts_dev || !cand || !ct || !counts_dev) return STIV_ERR_ARG;
  if (grad && (!gves || !gvid)) return STIV_ERR_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  double* Vtmp = Vc;
  if (!Vtmp && Vp) {
    int rc = stiv_ws_reserve(h, sizeof(double) * (size_t)(ct->capacity > 0 ? ct->capacity : 1));
    if (rc) return rc;
    Vtmp = (double*)h->ws;
  }
  stiv_args A;
  A.pv = p_dev; A.voff = vert_off_dev; A.X = verts_dev; A.mixed = h->prm.precision == STIV_MIXED;
  for (int c = 0; c < 3; ++c) A.L[c] = h->prm.box_L[c];
  A.ci = cand->i; A.cj = cand->j; A.cs = cand->shift;
  A.pair = ct->pair; A.type = ct->type; A.a = ct->a; A.b = ct->b; A.tau = ct->tau; A.w = ct->w;
  A.counts = counts_dev; A.cap = ct->capacity;
  double edt = h->prm.eps * h->prm.dt;
  A.e2 = edt * edt;
  A.vabs = h->prm.velocity == STIV_VEL_ABSOLUTE;
  A.dm2 = h->prm.d_m * h->prm.d_m;
  A.Vc = Vtmp; A.grad = grad; A.gves = gves; A.gvid = gvid; A.grad0 = grad0;
  A.vec = (((uintptr_t)grad | (uintptr_t)gves | (uintptr_t)gvid | (uintptr_t)grad0) & 15) == 0;
  int dev_sms = 152;
  cudaDeviceGetAttribute(&dev_sms, cudaDevAttrMultiProcessorCount, h->device);
  if (Vtmp || grad || grad0) {
    STIV_PROF(h, st, A.grad ? "stiv_grad" : (A.grad0 ? "stiv_grad_x0" : "stiv"));
    if (A.vabs || A.dm2 > 0.0 || A.grad0) stiv_kernel<true><<<dev_sms * 8, 128, 0, st>>>(A);
    else stiv_kernel<false><<<dev_sms * 8, 128, 0, st>>>(A);
    STIV_LAUNCH(h);
  }
  if (Vp) {
    STIV_PROF(h, st, "vpair");
    vpair_kernel<<<dev_sms * 8, 256, 0, st>>>(ct->pair, counts_dev, ct->capacity, Vtmp, cand->capacity, Vp);
    STIV_LAUNCH(h);
  }
  return STIV_OK;
}

extern "C" int stiv_stiv(stiv_handle* h, void* stream, int32_t n_ves, const int32_t* p_dev,
                         const int64_t* vert_off_dev, const void* verts_dev, const stiv_pairs* cand,
                         const stiv_contacts* contacts, const int64_t* counts_dev, double* V_contact_dev,
                         double* V_pair_dev) {
  (void)n_ves;
  return run_stiv(h, stream, p_dev, vert_off_dev, verts_dev, cand, contacts, counts_dev, V_contact_dev, V_pair_dev,
                  nullptr, nullptr, nullptr);
}

extern "C" int stiv_stiv_grad(stiv_handle* h, void* stream, int32_t n_ves, const int32_t* p_dev,
                              const int64_t* vert_off_dev, const void* verts_dev, const stiv_pairs* cand,
                              const stiv_contacts* contacts, const int64_t* counts_dev, double* V_contact_dev,
                              double* V_pair_dev, double* grad_dev, int32_t* g_ves_dev, int32_t* g_vid_dev) {
  (void)n_ves;
  if (!grad_dev) return STIV_ERR_ARG;
  return run_stiv(h, stream, p_dev, vert_off_dev, verts_dev, cand, contacts, counts_dev, V_contact_dev, V_pair_dev,
                  grad_dev, g_ves_dev, g_vid_dev);
}

extern "C" int stiv_stiv_grad_x0(stiv_handle* h, void* stream, int32_t n_ves, const int32_t* p_dev,
                                 const int64_t* vert_off_dev, const void* verts_dev, const stiv_pairs* cand,
                                 const stiv_contacts* contacts, const int64_t* counts_dev, double* grad_x0_dev) {
  (void)n_ves;
  if (!grad_x0_dev) return STIV_ERR_ARG;
  return run_stiv(h, stream, p_dev, vert_off_dev, verts_dev, cand, contacts, counts_dev, nullptr, nullptr, nullptr,
                  nullptr, nullptr, grad_x0_dev);
}

extern "C" int stiv_grad_scatter(stiv_handle* h, void* stream, const int32_t* p_dev, const stiv_contacts* contacts,
                                 const int64_t* counts_dev, const double* weight_pair_dev, const double* grad_dev,
                                 const int32_t* g_ves_dev, const int32_t* g_vid_dev, const int64_t* vert_off_dev,
                                 double* gX_dev) {
  if (!h || !p_dev || !contacts || !counts_dev || !grad_dev || !g_ves_dev || !g_vid_dev || !vert_off_dev || !gX_dev)
    return STIV_ERR_ARG;
  int dev_sms = 152;
  cudaDeviceGetAttribute(&dev_sms, cudaDevAttrMultiProcessorCount, h->device);
  STIV_PROF(h, (cudaStream_t)stream, "grad_scatter");
  scatter_grad_kernel<<<dev_sms * 4, 128, 0, (cudaStream_t)stream>>>(counts_dev, contacts->capacity, contacts->pair,
                                                                     weight_pair_dev, grad_dev, g_ves_dev, g_vid_dev,
                                                                     p_dev, vert_off_dev, gX_dev);
  STIV_LAUNCH(h);
  return STIV_OK;
}

extern "C" int stiv_grad_to_coef(stiv_handle* h, void* stream, int32_t n_ves, int32_t p_max, const int32_t* p_dev,
                                 const int64_t* coef_off_dev, const int64_t* vert_off_dev, const double* gX_dev,
                                 double* gcoef_dev) {
  if (!h || n_ves < 0 || p_max < 1 || p_max > STIV_MAX_P) return STIV_ERR_ARG;
  if (n_ves == 0) return STIV_OK;
  if (!p_dev || !coef_off_dev || !vert_off_dev || !gX_dev || !gcoef_dev) return STIV_ERR_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  if (h->prm.precision == STIV_MIXED)
    return stiv_grad_to_coef_tc(h, st, n_ves, p_max, p_dev, coef_off_dev, vert_off_dev, gX_dev, gcoef_dev);
  adj_args a;
  a.p = p_dev; a.coef_off = coef_off_dev; a.vert_off = vert_off_dev; a.gX = gX_dev; a.gcoef = gcoef_dev;
  for (int p = 0; p <= STIV_MAX_P; ++p) { a.leg[p] = nullptr; a.trig[p] = nullptr; }
  for (int p = 1; p <= p_max; ++p) {
    int rc = stiv_ensure_tables(h, st, p);
    if (rc) return rc;
    a.leg[p] = h->tab[p].leg; a.trig[p] = h->tab[p].trig;
  }
  int Pm = 2 * p_max;
  auto bytes = [](int P) { return sizeof(double) * ((size_t)(P + 1) * (P + 1) + (size_t)(P + 1) * 4 * (P / 2 + 1)); };
  size_t smem = bytes(Pm);
  STIV_SMEM(h, adjoint_kernel, smem, 0, bytes(STIV_MAX_PP));
  STIV_PROF(h, st, "grad_to_coef");
  adjoint_kernel<<<dim3(n_ves, 3), 256, smem, st>>>(a);
  STIV_LAUNCH(h);
  return STIV_OK;
}
