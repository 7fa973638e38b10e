// Narrow phase of Alg. 2 checkContact: every vertex-triangle pair (both
// directions) and edge-edge pair of a candidate vesicle pair whose swept boxes
// overlap is tested with the coplanarity cubic of Eq. 3.1 (d_m = 0), or with
// the degree-six equation of the d_m band (d_m > 0).
//
// The triangulated grid (Sec. 3.1.2, Fig. 3) is cut into patches of 2 x 4 grid
// quads; each primitive belongs to exactly one patch, so each primitive pair
// is examined by exactly one patch pair.
//   patch_pairs_kernel: per candidate vesicle pair, one CTA lists the patch
//     pairs whose FP32 (outward) boxes overlap and some of whose cells (1 x 2
//     quads) meet;
//   narrow_kernel (stages 1-3a): per patch pair, one warp stages both patches
//     in shared memory, finds the primitive pairs whose boxes overlap from bit
//     masks over the vertex slots and filters them; the survivors leave as
//     global pair descriptors;
//   roots_kernel (d_m = 0) or pieces_kernel (d_m > 0) for stage 3b and
//     fp64_kernel (stage 4) work on those lists, so that every stage runs on
//     full warps.  The stages:
//     1. FP32 swept-box test (conservative: never drops an overlapping pair);
//     2. the exact FP64 swept-box test (counts the pairs tested), decided
//        from the FP32 boxes and their error bound, on the FP64 values only
//        for the pairs those do not decide;
//     3. certified FP32 rejection: a pair is dropped only when error-bounded
//        FP32 arithmetic proves that the FP64 test below cannot report a
//        contact (Bernstein bound: no root of the cubic in [0,1]; a direction
//        along which the two primitives stay apart over the whole step; or, on
//        every sub-interval that may hold a root, the point is certainly
//        outside the triangle / the edges certainly miss);
//     4. the FP64 contact test (cubic, root isolation, bisection, inside test)
//        in the fixed arithmetic order, on the survivors only.
// Stage 3 never changes a result: the contact list equals the one obtained by
// running stage 4 on every pair of stage 2 (stiv_params.exact_only = 1).
#include "stiv_internal.cuh"

#include <math.h>

namespace {

constexpr int PSLOT = (STIV_BR + 1) * (STIV_BC + 1);   // slot of the patch's pole; grid slots below it
constexpr int NSLOT = PSLOT + 1;
constexpr int NW = 8;                                  // warps per CTA
constexpr int QCAP = 512;                              // queue entries per warp
constexpr int SOUTH = 1 << 15;                         // patch id flag: the south-pole primitives of a two-pole patch

// Primitives of one patch in terms of its vertex slots (3 rows of 5 grid
// slots, then the pole).  P is even, so every patch spans exactly STIV_BR
// bands and STIV_BC columns; the lists depend only on whether the patch
// touches the north pole (first band), the south pole (last band) and whether
// it owns the pole vertex (first column block).  At P = 2 one patch touches
// both poles; it is examined once with the north pole and all grid
// primitives, and once (SOUTH) with the south pole's primitives alone.  16
// variants, built once per CTA.  The primitives are listed for the lanes that
// stand for them (v, t, e) and given as bit masks over their first slots for
// the lanes that test against all of them (vm, qm, hm, fm).
struct PatchTopo {
  unsigned char v[16];             // vertices owned by the patch: slot
  unsigned short t[32];            // triangles: 3 slots, 4 bits each
  unsigned char e[32];             // edges: 2 slots, 4 bits each
  int nv, nt, ne;
  unsigned vm;                     // owned vertices
  unsigned qm;                     // quads: both triangles, the downward and the diagonal edge at (row, column)
  unsigned hm;                     // edges along a row
  unsigned fm;                     // pole fan (triangles and edges), bits 0-3 by column
  int frow;                        // first slot of the fan's row
};
constexpr int NVAR = 16;
static_assert(STIV_BR == 2 && STIV_BC == 4, "slot and bit layout");

struct WarpSm {
  float4 x[2 * NSLOT], d[2 * NSLOT];    // patch A's slots, then B's: X0 - origin of vesicle i (w: vertex id), X1 - X0
  float4 lo[2 * NSLOT], hi[2 * NSLOT];  // conservative FP32 swept boxes (frame of vesicle i)
  uint4 miss[NSLOT];                    // per slot of B, axis x, y, z: A's slots it misses (low half: A's lo above, high: A's hi below)
  unsigned q[QCAP];                     // primitive pairs: four slots (5 bits each, + 16 on B), kind << 20
};

struct narrow_args {
  const void* X;
  int mixed;
  double L[3];
  const uint64_t* work;
  int64_t W;
  int include_ee;
  int exact_only;
  double dm;                // minimum separation d_m (> 0: the degree-six contact test)
  int nlevel;               // d_m > 0: refinement levels of the piece test (<= NLEVEL)
  const float* vorg;
  const float* fprep;
  int64_t fstride;
  const stiv_pair_info* pinfo;  // per candidate pair: vesicles, orders, offsets, FP32 frame
  // descriptors of primitive pairs: x = pair << 32 | type << 30 | a << 15 | b
  // (primitive ids), y = the 4 vertex ids, 16 bits each, in the order the
  // contact test takes its points (VF: vertex, triangle; EE: p0 < p1, q0 < q1)
  ulonglong2* q3;           // stage 3b input
  ulonglong2* q2;           // stage 4 input
  ulonglong2* q2c;          // stage 4 input whose cubic may have a critical point
  int64_t Q3, Q2;
  int64_t C;  // raw contact capacity
  int32_t* rc_pair; int32_t* rc_type; int32_t* rc_a; int32_t* rc_b;
  double* rc_tau; double* rc_w;
  int32_t* pair_cnt;        // contacts per candidate pair
  int64_t* ctr;
};

__device__ __forceinline__ int slot_of(int rr, int cc) { return rr * (STIV_BC + 1) + cc; }

// Vertex coordinate as stored: double (FP64 form) or float (mixed form).
template <bool MIXED>
__device__ __forceinline__ double vtx(const void* X, size_t i) {
  if (MIXED) return (double)((const float*)X)[i];
  return ((const double*)X)[i];
}

// ---------------------------------------------------------------------------
// staging
// ---------------------------------------------------------------------------
// Topology variant var = first | last << 1 | pole-owner << 2 | south-only << 3
// (see PatchTopo), built by one warp.
__device__ void build_topo(PatchTopo& T, int var, int lane) {
  const int rq = STIV_BR, ncol = STIV_BC;
  bool first = var & 1, last = (var >> 1) & 1, j0 = (var >> 2) & 1, so = (var >> 3) & 1;
  int rown = so ? 0 : rq + (last ? 1 : 0);
  bool north = first && !so, pole = first || last;
  int nvg = rown * ncol, ntq = so ? 0 : 2 * rq * ncol, nfan = pole ? ncol : 0;
  int nh = rown * ncol, nq = so ? 0 : 2 * rq * ncol;
  int frow = north ? 0 : slot_of(rq, 0);
  if (lane == 0) {
    T.nv = nvg + (pole && j0 ? 1 : 0); T.nt = ntq + nfan; T.ne = nh + nq + nfan;
    unsigned rows = 0, quads = 0;
    for (int rr = 0; rr < rown; ++rr) rows |= 0xFu << slot_of(rr, 0);
    if (!so) for (int rr = 0; rr < rq; ++rr) quads |= 0xFu << slot_of(rr, 0);
    T.vm = rows | (pole && j0 ? 1u << PSLOT : 0u);
    T.hm = rows; T.qm = quads; T.fm = pole ? 0xFu : 0u; T.frow = frow;
  }
  for (int k = lane; k < nvg + 1 && k < 16; k += 32)
    T.v[k] = (unsigned char)(k < nvg ? slot_of(k / ncol, k % ncol) : PSLOT);
  for (int k = lane; k < ntq + nfan; k += 32) {
    int s0, s1, s2;
    if (k < ntq) {
      int q = k >> 1, rr = q / ncol, cc = q % ncol;
      s0 = slot_of(rr, cc);
      s1 = (k & 1) == 0 ? slot_of(rr + 1, cc) : slot_of(rr + 1, cc + 1);
      s2 = (k & 1) == 0 ? slot_of(rr + 1, cc + 1) : slot_of(rr, cc + 1);
    } else {
      int cc = k - ntq;
      s0 = PSLOT; s1 = frow + (north ? cc : cc + 1); s2 = frow + (north ? cc + 1 : cc);
    }
    T.t[k] = (unsigned short)(s0 | (s1 << 4) | (s2 << 8));
  }
  for (int k = lane; k < nh + nq + nfan; k += 32) {
    int sa, sb;
    if (k < nh) {
      sa = slot_of(k / ncol, k % ncol); sb = sa + 1;
    } else if (k < nh + nq) {
      int k2 = k - nh, q = k2 >> 1;
      sa = slot_of(q / ncol, q % ncol);
      sb = sa + STIV_BC + 1 + (k2 & 1);
    } else {
      sa = frow + k - nh - nq; sb = PSLOT;
    }
    T.e[k] = (unsigned char)(sa | (sb << 4));
  }
}

// Order-preserving int image of a float (-0 just below +0) and its inverse:
// the warp's integer min / max reductions then give the float min / max.
__device__ __forceinline__ int fkey32(float f) {
  int i = __float_as_int(f);
  return i >= 0 ? i : i ^ 0x7FFFFFFF;
}
__device__ __forceinline__ float fkey_val(int k) { return __int_as_float(k >= 0 ? k : k ^ 0x7FFFFFFF); }

// Bound on the error of a component of the difference of two FP32 frame
// positions of the same vesicle: each is x = fl(xf + off) with xf the
// position relative to the vesicle's origin rounded once (|xf| <= R) and off
// the same float for every point of the vesicle, so off's own error cancels
// and U32 (|xf1| + |xf2| + |x1| + |x2|) remains; R: the larger vesicle
// radius bound of the pair, offm: the largest offset component.  It is at
// most 2 ep (ep = 2^-22 (R_i + R_j + 2 offm)), the bound stage 3a keeps.
__device__ __forceinline__ float same_side_err(float R, float offm) {
  return 1.01f * 5.9604645e-8f * (4.0f * R + 2.0f * offm);
}

// One patch of a patch pair, as its lanes see it.
struct PatchRef {
  int P, I, J, ves, pole;          // pole: vertex id of the pole slot (-1: none)
  const PatchTopo* tp;
};
__device__ __forceinline__ PatchRef patch_ref(const PatchTopo* topo, int P, int ves, int patch) {
  PatchRef r;
  bool so = patch & SOUTH;
  int nbc = stiv_ncol_blocks(P), k = patch & (SOUTH - 1);
  r.P = P; r.ves = ves; r.I = k / nbc; r.J = k % nbc;
  bool f = r.I == 0, l = r.I == stiv_nband_blocks(P) - 1;
  r.pole = f && !so ? 2 * P * (P + 1) : (l ? 2 * P * (P + 1) + 1 : -1);
  r.tp = topo + ((f ? 1 : 0) | (l ? 2 : 0) | (r.J == 0 ? 4 : 0) | (so ? 8 : 0));
  return r;
}

// Stage the two patches of a patch pair (A: of vesicle i, unshifted; B: of
// vesicle j at its periodic image) in one pass over the lanes: lanes 0-14 the
// grid slots of A, lane 15 A's pole, lanes 16-30 and 31 the same for B.  Each
// slot gets its FP32 frame coordinates and a conservative FP32 swept box
// (vesicle j's widened by d_m, rounded up): the box ends lie within m of the
// exact ones.  Returns in gap the margin by which two staged box ends that
// pass each other prove that the exact ones do (3 m on both sides; with
// d_m > 0 plus 2^-21 d_m for the roundings of the widening), and in dmax the
// largest displacement component.
template <bool MIXED, bool DM>
__device__ __forceinline__ void stage_pair(WarpSm& ws, const narrow_args& a, const PatchRef& A, const PatchRef& B,
                                           float4 frame, int lane, float& gap, float& dmax) {
  bool onB = lane >= 16;
  int k = lane & 15;
  int P = onB ? B.P : A.P, W = 2 * P, v = onB ? B.ves : A.ves;
  int r0 = (onB ? B.I : A.I) * STIV_BR, c0 = (onB ? B.J : A.J) * STIV_BC;
  int rr = k / (STIV_BC + 1), col = c0 + k - rr * (STIV_BC + 1);
  if (col >= W) col -= W;
  int vid = k == PSLOT ? (onB ? B.pole : A.pole) : (r0 + rr) * W + col;
  const float4* fp = (const float4*)(a.fprep + (size_t)v * a.fstride) + 2 * (vid >= 0 ? vid : 0);
  float4 x = fp[0], d = fp[1];
  if (MIXED) {   // the staging holds the FP32 vertices themselves: one rounding each, as the FP64 form's staging
    float4 o = ((const float4*)a.vorg)[v];
    d = make_float4(d.x - x.x, d.y - x.y, d.z - x.z, 0.f);
    x = make_float4(x.x - o.x, x.y - o.y, x.z - o.z, 0.f);
  }
  if (onB) { x.x = x.x + frame.x; x.y = x.y + frame.y; x.z = x.z + frame.z; }
  x.w = __int_as_float(vid);
  ws.x[lane] = x;
  ws.d[lane] = d;
  float mx = frame.w + 4.7683716e-7f * (fabsf(x.x) + fabsf(d.x));   // 2^-21 (|x| + |d|)
  float my = frame.w + 4.7683716e-7f * (fabsf(x.y) + fabsf(d.y));
  float mz = frame.w + 4.7683716e-7f * (fabsf(x.z) + fabsf(d.z));
  // positive floats order as their bits
  gap = 6.0f * __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(fmaxf(mx, fmaxf(my, mz)))));
  dmax = __uint_as_float(
      __reduce_max_sync(0xffffffffu, __float_as_uint(fmaxf(fabsf(d.x), fmaxf(fabsf(d.y), fabsf(d.z))))));
  if (DM) {
    float padf = __double2float_ru(a.dm);
    gap += 4.7683716e-7f * padf;
    if (onB) { mx = __fadd_ru(mx, padf); my = __fadd_ru(my, padf); mz = __fadd_ru(mz, padf); }
  }
  float4 lo = make_float4(fminf(x.x, x.x + d.x) - mx, fminf(x.y, x.y + d.y) - my, fminf(x.z, x.z + d.z) - mz, 0.f);
  float4 hi = make_float4(fmaxf(x.x, x.x + d.x) + mx, fmaxf(x.y, x.y + d.y) + my, fmaxf(x.z, x.z + d.z) + mz, 0.f);
  if (vid < 0) {
    lo = make_float4(INFINITY, INFINITY, INFINITY, 0.f);
    hi = make_float4(-INFINITY, -INFINITY, -INFINITY, 0.f);
  }
  ws.lo[lane] = lo;
  ws.hi[lane] = hi;
  __syncwarp();
}

// Which slot boxes of A each slot of B misses, per axis and side, as bits:
// lane k and lane k + 16 take slot k of B against the lower and the upper
// eight slots of A.  A difference of box ends is negative exactly when they
// miss, so its sign bit is shifted into the mask.  Returns whether some
// difference lies in [0, gap): then a pair of boxes may overlap in FP32 and
// not exactly.  (A primitive's box is the union of its slots' boxes, so it
// misses a box on an axis and side exactly when all its slots do.)
__device__ __forceinline__ bool slot_masks(WarpSm& ws, float gap, int lane) {
  int k = lane & 15, h = lane >> 4;
  float4 bl = ws.lo[NSLOT + k], bh = ws.hi[NSLOT + k];
  unsigned lx = 0, ly = 0, lz = 0, hx = 0, hy = 0, hz = 0, near = 0xFFFFFFFFu;
#pragma unroll
  for (int q = 7; q >= 0; --q) {
    float4 al = ws.lo[8 * h + q], ah = ws.hi[8 * h + q];
    unsigned d0 = __float_as_uint(bh.x - al.x), d1 = __float_as_uint(bh.y - al.y), d2 = __float_as_uint(bh.z - al.z);
    unsigned d3 = __float_as_uint(ah.x - bl.x), d4 = __float_as_uint(ah.y - bl.y), d5 = __float_as_uint(ah.z - bl.z);
    lx = __funnelshift_l(d0, lx, 1); ly = __funnelshift_l(d1, ly, 1); lz = __funnelshift_l(d2, lz, 1);
    hx = __funnelshift_l(d3, hx, 1); hy = __funnelshift_l(d4, hy, 1); hz = __funnelshift_l(d5, hz, 1);
    near = min(near, min(min(d0, min(d1, d2)), min(d3, min(d4, d5))));   // negative ones are large as integers
  }
  unsigned wx = lx | (hx << 16), wy = ly | (hy << 16), wz = lz | (hz << 16);
  unsigned ox = __shfl_xor_sync(0xffffffffu, wx, 16), oy = __shfl_xor_sync(0xffffffffu, wy, 16),
           oz = __shfl_xor_sync(0xffffffffu, wz, 16);
  if (h == 0) ws.miss[k] = make_uint4(wx | (ox << 8), wy | (oy << 8), wz | (oz << 8), 0u);
  bool unsure = __any_sync(0xffffffffu, near < __float_as_uint(gap));
  return unsure;
}

__device__ __forceinline__ uint4 and4(uint4 a, uint4 b) { return make_uint4(a.x & b.x, a.y & b.y, a.z & b.z, 0u); }
// Hits (bits 0-15) of primitives whose per-axis misses are w: no axis and side missed.
__device__ __forceinline__ unsigned hits_of(uint4 w) {
  unsigned m = w.x | w.y | w.z;
  return ~(m | (m >> 16)) & 0xFFFFu;
}
__device__ __forceinline__ uint4 shr4(uint4 a, int k) { return make_uint4(a.x >> k, a.y >> k, a.z >> k, 0u); }
// The pole slot's bit of both halves, spread over its half.
__device__ __forceinline__ unsigned pole_half(unsigned w) { return ((w >> PSLOT) & 0x00010001u) * 0xFFFFu; }
__device__ __forceinline__ uint4 pole4(uint4 w) { return make_uint4(pole_half(w.x), pole_half(w.y), pole_half(w.z), 0u); }

__device__ __forceinline__ bool fbox_hit(const float* a, const float* b) {
  return a[0] <= b[3] && b[0] <= a[3] && a[1] <= b[4] && b[1] <= a[4] && a[2] <= b[5] && b[2] <= a[5];
}

// ---------------------------------------------------------------------------
// certified FP32 rejection
// ---------------------------------------------------------------------------
struct f3 { float x, y, z; };
__device__ __forceinline__ f3 fsub(f3 a, f3 b) { return {a.x - b.x, a.y - b.y, a.z - b.z}; }
__device__ __forceinline__ f3 fadd(f3 a, f3 b) { return {a.x + b.x, a.y + b.y, a.z + b.z}; }
__device__ __forceinline__ f3 fcross(f3 u, f3 v) {
  return {fmaf(u.y, v.z, -(u.z * v.y)), fmaf(u.z, v.x, -(u.x * v.z)), fmaf(u.x, v.y, -(u.y * v.x))};
}
__device__ __forceinline__ float fdot(f3 u, f3 v) { return fmaf(u.z, v.z, fmaf(u.y, v.y, u.x * v.x)); }
// Upper bound of the Euclidean norm: s * rsqrtf(s) with rsqrtf's maximum
// error of 2 ulp (2^-22 relative) widened by 2^-20; the rounding of s itself
// is covered by the margins of the callers.
__device__ __forceinline__ float fnorm(f3 u) {
  float s = fdot(u, u);
  return s > 1e-30f ? s * rsqrtf(s) * 1.000001f : 1e-15f;
}
__device__ __forceinline__ f3 fat(f3 x, float t, f3 d) { return {fmaf(t, d.x, x.x), fmaf(t, d.y, x.y), fmaf(t, d.z, x.z)}; }
__device__ __forceinline__ float amax3(f3 u) { return fmaxf(fabsf(u.x), fmaxf(fabsf(u.y), fabsf(u.z))); }

constexpr float U32 = 5.9604645e-8f;   // 2^-24, unit roundoff of float

// Sign of (g1 x g2) . (g3 x g4) over t in [tm - h, tm + h], each g linear in t
// (value gv at tm, rate gd).  eg bounds the error of each component of each
// gv.  |(g1 x g2) . (g3 x g4)| <= |g1||g2||g3||g4|, so the change over the
// interval is at most sum_i h|gd_i| prod_{j != i} max|g_j|.  Returns +1
// (certainly > 0), -1 (certainly < 0) or 0.
// The same test with the bound's ingredients given: M_i >= max |g_i| over the
// interval (plus the input error 2 eg), R_i = h |gd_i| (half width times the
// rate); the norms of the vectors an inside test shares between its forms
// are taken once.
__device__ __forceinline__ int form_sign_m(f3 g0, f3 g1, f3 g2, f3 g3, const float* M, const float* R, const float* G) {
  float val = fdot(fcross(g0, g1), fcross(g2, g3));
  float p01 = M[0] * M[1], p23 = M[2] * M[3];
  float prod = p01 * p23;
  float var = (R[0] + G[0]) * M[1] * p23 + M[0] * (R[1] + G[1]) * p23 + p01 * (R[2] + G[2]) * M[3] + p01 * M[2] * (R[3] + G[3]);
  float rad = (var + 64.0f * U32 * prod) * 1.001f;
  if (val > rad) return 1;
  if (val < -rad) return -1;
  return 0;
}

// For every contact time in [t0, t0 + w], is the point certainly outside the
// triangle / are the edges certainly apart (1), certainly inside (2), or
// undecided (0)?  Points: VF xp, x0, x1, x2; EE p0, p1, q0, q1.
// ep, ed: error bounds of the FP32 positions / displacements per component.
// Each barycentric (VF) or closest-point (EE) numerator is a form
// (g1 x g2) . (g3 x g4) of linear g: |(g1 x g2) . (g3 x g4)| <= prod |g_i|,
// so its change over the interval is at most sum_i h |gd_i| prod_{j != i}
// max |g_j|; form_sign_m certifies its sign.
__device__ int inside_cert(int kind, const f3* x, const f3* d, float t0, float w, float ep, float ed, float es) {
  float h = 0.5f * w + 1e-6f;           // half width, widened past the FP64 root's last ulp
  float tm = t0 + 0.5f * w;
  f3 P[4];
  for (int q = 0; q < 4; ++q) P[q] = fat(x[q], tm, d[q]);
  float pm = fmaxf(fmaxf(amax3(P[0]), amax3(P[1])), fmaxf(amax3(P[2]), amax3(P[3])));
  float eg = 2.0f * (ep + ed) + 4.0f * U32 * pm;  // per component, differences of positions at tm
  float egs = es + 2.0f * ed + 4.0f * U32 * pm;     // the same for two points of one vesicle
  // vector (position difference at tm, rate) -> M, R, G (2 x its error) of form_sign_m
  auto mr = [&](f3 gv, f3 gd, float e, float& M, float& R, float& G) {
    R = h * fnorm(gd);
    G = 2.0f * e;
    M = fnorm(gv) + R + G;
  };
  if (kind == 0) {
    // barycentric weight of T_k ~ ((T_{k+2} - T_{k+1}) x (p - T_{k+1})) . n,  n = (T1 - T0) x (T2 - T0)
    f3 t01 = fsub(P[2], P[1]), t02 = fsub(P[3], P[1]), t12 = fsub(P[3], P[2]);
    f3 q0 = fsub(P[0], P[1]), q1 = fsub(P[0], P[2]), q2 = fsub(P[0], P[3]);
    float Mt01, Rt01, Mt02, Rt02, Mt12, Rt12, Mq0, Rq0, Mq1, Rq1, Mq2, Rq2, Gs, Gc;
    mr(t01, fsub(d[2], d[1]), egs, Mt01, Rt01, Gs);
    mr(t02, fsub(d[3], d[1]), egs, Mt02, Rt02, Gs);
    mr(t12, fsub(d[3], d[2]), egs, Mt12, Rt12, Gs);
    mr(q0, fsub(d[0], d[1]), eg, Mq0, Rq0, Gc);
    mr(q1, fsub(d[0], d[2]), eg, Mq1, Rq1, Gc);
    mr(q2, fsub(d[0], d[3]), eg, Mq2, Rq2, Gc);
    float G[4] = {Gs, Gc, Gs, Gs};
    f3 nt02 = {-t02.x, -t02.y, -t02.z};
    // k = 0: (T2 - T1) x (p - T1); k = 1: (T0 - T2) x (p - T2); k = 2: (T1 - T0) x (p - T0)
    float M0[4] = {Mt12, Mq1, Mt01, Mt02}, R0[4] = {Rt12, Rq1, Rt01, Rt02};
    int sg0 = form_sign_m(t12, q1, t01, t02, M0, R0, G);
    if (sg0 < 0) return 1;
    float M1[4] = {Mt02, Mq2, Mt01, Mt02}, R1[4] = {Rt02, Rq2, Rt01, Rt02};
    int sg1 = form_sign_m(nt02, q2, t01, t02, M1, R1, G);
    if (sg1 < 0) return 1;
    float M2[4] = {Mt01, Mq0, Mt01, Mt02}, R2[4] = {Rt01, Rq0, Rt01, Rt02};
    int sg2 = form_sign_m(t01, q0, t01, t02, M2, R2, G);
    if (sg2 < 0) return 1;
    return (sg0 > 0 && sg1 > 0 && sg2 > 0) ? 2 : 0;
  }
  // EE with m = (p1 - p0) x (q1 - q0):  s ~ ((q0 - p0) x (q1 - q0)) . m,
  // s - 1 ~ ((q0 - p1) x (q1 - q0)) . m,  u ~ ((q0 - p0) x (p1 - p0)) . m,
  // u - 1 ~ ((q1 - p0) x (p1 - p0)) . m   (each divided by |m|^2)
  f3 e1v = fsub(P[1], P[0]), e2v = fsub(P[3], P[2]);
  f3 a0 = fsub(P[2], P[0]), a1 = fsub(P[2], P[1]), a3 = fsub(P[3], P[0]);
  float Me1, Re1, Me2, Re2, Ma0, Ra0, Ma1, Ra1, Ma3, Ra3, Gs, Gc;
  mr(e1v, fsub(d[1], d[0]), egs, Me1, Re1, Gs);
  mr(e2v, fsub(d[3], d[2]), egs, Me2, Re2, Gs);
  mr(a0, fsub(d[2], d[0]), eg, Ma0, Ra0, Gc);
  mr(a1, fsub(d[2], d[1]), eg, Ma1, Ra1, Gc);
  mr(a3, fsub(d[3], d[0]), eg, Ma3, Ra3, Gc);
  float G[4] = {Gc, Gs, Gs, Gs};
  float Ms[4] = {Ma0, Me2, Me1, Me2}, Rs[4] = {Ra0, Re2, Re1, Re2};
  int s0 = form_sign_m(a0, e2v, e1v, e2v, Ms, Rs, G);
  if (s0 < 0) return 1;
  float Ms1[4] = {Ma1, Me2, Me1, Me2}, Rs1[4] = {Ra1, Re2, Re1, Re2};
  int s1 = form_sign_m(a1, e2v, e1v, e2v, Ms1, Rs1, G);
  if (s1 > 0) return 1;
  float Mu[4] = {Ma0, Me1, Me1, Me2}, Ru[4] = {Ra0, Re1, Re1, Re2};
  int u0 = form_sign_m(a0, e1v, e1v, e2v, Mu, Ru, G);
  if (u0 < 0) return 1;
  float Mu1[4] = {Ma3, Me1, Me1, Me2}, Ru1[4] = {Ra3, Re1, Re1, Re2};
  int u1 = form_sign_m(a3, e1v, e1v, e2v, Mu1, Ru1, G);
  if (u1 > 0) return 1;
  return (s0 > 0 && s1 < 0 && u0 > 0 && u1 < 0) ? 2 : 0;
}

// Coefficients of the coplanarity cubic in FP32 and a bound E on the error of
// any value of the cubic (or of its Bernstein coefficients on any sub-interval
// of [0, 1]) against the exact cubic of the FP64 inputs.  Every coefficient is
// a sum of triple products u . (v x w) of difference vectors (six terms each);
// ep / ed bound the input errors of the positions / displacements per
// component.  Each triple product's error is bounded with the magnitudes of
// its own three vectors, so a pair whose displacement differences are small
// (a primitive moving nearly rigidly) keeps a tight bound:  with eu, ev, ew
// the component errors of u, v, w and Au, Av, Aw their largest computed
// components, each of the six terms obeys |xyz - x'y'z'| <= |x - x'||y'||z'|
// + |x||y - y'||z'| + |x||y||z - z'| with |y'| <= Ay + ey, so the product's
// error is at most 6 ((Au + eu)(Av + ev)(Aw + ew) - Au Av Aw + rr Au Av Aw)
// (rr: the relative rounding of the FP32 evaluation per term).
// With d_m > 0 the band test also takes mn = |n0| + |n1| + |n2| (the FP32
// normals' magnitudes) and the largest position / displacement difference
// components A2, Ad2 of the primitive's own pair of vectors (a, b / da, db).
struct cubic32 { float k0, k1, k2, k3, E, ed, mn, A2, Ad2; };

// es: the error bound of the same-vesicle differences a and b (at most 2 ep).
template <bool WM = false>
__device__ __forceinline__ cubic32 cubic_fp32(int kind, const f3* x, const f3* d, float ep, float es) {
  f3 a, b, c, da, db, dc;
  if (kind == 0) {
    a = fsub(x[2], x[1]); b = fsub(x[3], x[1]); c = fsub(x[0], x[1]);
    da = fsub(d[2], d[1]); db = fsub(d[3], d[1]); dc = fsub(d[0], d[1]);
  } else {
    a = fsub(x[1], x[0]); b = fsub(x[3], x[2]); c = fsub(x[2], x[0]);
    da = fsub(d[1], d[0]); db = fsub(d[3], d[2]); dc = fsub(d[2], d[0]);
  }
  f3 n0 = fcross(a, b);
  f3 n1 = fadd(fcross(da, b), fcross(a, db));
  f3 n2 = fcross(da, db);
  cubic32 r;
  r.k0 = fdot(c, n0);
  r.k1 = fdot(dc, n0) + fdot(c, n1);
  r.k2 = fdot(c, n2) + fdot(dc, n1);
  r.k3 = fdot(dc, n2);
  float Aa = amax3(a), Ab = amax3(b), Ac = amax3(c), Ada = amax3(da), Adb = amax3(db), Adc = amax3(dc);
  float A = fmaxf(Aa, fmaxf(Ab, Ac)), Ad = fmaxf(Ada, fmaxf(Adb, Adc));
  float Dm = 0.f;
  for (int q = 0; q < 4; ++q) Dm = fmaxf(Dm, amax3(d[q]));
  float ed = 2.0f * U32 * Dm + 1e-12f;           // |d - D| per component (float rounding of X1 - X0)
  // per component of each difference: both inputs' errors and the rounding of the difference
  // a and b join points of one vesicle, whose common frame offset cancels in
  // the difference (es); c joins the two vesicles (2 ep)
  float ea = es + 2.0f * U32 * Aa, eb = es + 2.0f * U32 * Ab, ec = 2.0f * ep + 2.0f * U32 * Ac;
  float eda = 2.0f * ed + 2.0f * U32 * Ada, edb = 2.0f * ed + 2.0f * U32 * Adb, edc = 2.0f * ed + 2.0f * U32 * Adc;
  float rr = 8.0f * U32;                         // rounding per term
  // The coefficients are sums of the eight triple products u . (v x w) with
  // u in {c, dc}, v in {a, da}, w in {b, db} (k0: c.(a x b); k1: dc.(a x b),
  // c.(da x b), c.(a x db); k2: c.(da x db), dc.(da x b), dc.(a x db); k3:
  // dc.(da x db)).  The sum of their bounds (above) factors over the three
  // choices: with U = Ac + Adc, V = Aa + Ada, W = Ab + Adb and eU, eV, eW the
  // sums of the matching errors, it is 6 ((U + eU)(V + eV)(W + eW) - U V W
  // + rr U V W), evaluated below without cancellation.
  float U = Ac + Adc, V = Aa + Ada, W = Ab + Adb;
  float eU = ec + edc, eV = ea + eda, eW = eb + edb;
  float Esum = 6.f * (eU * (V + eV) * (W + eW) + U * eV * (W + eW) + U * V * eW + rr * U * V * W);
  float S = fabsf(r.k0) + fabsf(r.k1) + fabsf(r.k2) + fabsf(r.k3);
  float M = (A + Ad) * (A + Ad) * (A + Ad);
  r.E = 1.25f * Esum + 64.f * U32 * S + 1e-12f * 48.f * M;
  r.ed = ed;
  if (WM) {
    r.mn = fnorm(n0) + fnorm(n1) + fnorm(n2);
    r.A2 = fmaxf(Aa, Ab);
    r.Ad2 = fmaxf(Ada, Adb);
  }
  return r;
}

__device__ __forceinline__ bool certain_sign4(float c0, float c1, float c2, float c3, float E) {
  return (c0 > E && c1 > E && c2 > E && c3 > E) || (c0 < -E && c1 < -E && c2 < -E && c3 < -E);
}

// The d_m band.  min |f| over an interval is bounded below by the smallest
// Bernstein coefficient of the cubic (all of one sign beyond the error bound
// E); |m(t)| <= |n0| + |n1| + |n2| is bounded above from the FP32 cross
// products with their error bounds (the error model of cubic_fp32); a margin
// of 1e-12 of the squared magnitudes covers the FP64 evaluation of
// g = f^2 - d_m^2 |m|^2.
// Right-hand side of the band test: (d_m max|m|)^2 with its margins.
__device__ float band_rhs(const cubic32& q, float ep, float dm) {
  float A = q.A2, Ad = q.Ad2, ed = q.ed;
  float epd = 2.0f * ep + 2.0f * U32 * A, edd = 2.0f * ed + 2.0f * U32 * Ad;
  float en = 2.0f * ((4.f * epd * A + 4.f * U32 * A * A) + (4.f * edd * A + 4.f * epd * Ad + 8.f * U32 * A * Ad) +
                     (4.f * edd * Ad + 4.f * U32 * Ad * Ad));
  float mmax = q.mn * (1.f + 8.f * U32) + en;
  float S = fabsf(q.k0) + fabsf(q.k1) + fabsf(q.k2) + fabsf(q.k3) + 4.f * q.E;
  float dmm = dm * (1.f + 4.f * U32) * mmax;
  return dmm * dmm * (1.f + 1e-5f) + 1e-12f * (S * S + dmm * dmm);
}

// 1 if the Bernstein coefficients c0..c3 (error E) of the cubic on an
// interval prove |f| > d_m max|m| there (rhs: band_rhs).
__device__ __forceinline__ bool out_of_band(float c0, float c1, float c2, float c3, float E, float rhs) {
  if (!certain_sign4(c0, c1, c2, c3, E)) return false;
  float fmin = fminf(fminf(fabsf(c0), fabsf(c1)), fminf(fabsf(c2), fabsf(c3))) - E;
  return fmin > 0.f && fmin * fmin * (1.f - 1e-5f) > rhs;
}

// ---------------------------------------------------------------------------
// Stage 3a.  The cubic f = c . m, m = a x b, from the difference vectors at
// both ends of the step (index 0: t = 0, 1: t = 1; each moves linearly, so f
// is a blossom): VF a, b the triangle's edges from its first vertex, EE the two
// edges; c from the vertex (the first edge's first point) to that vertex (the
// second edge's first point).  B: the Bernstein coefficients of f on [0, 1],
//   B0 = c0.n00, B1 = (c1.n00 + c0.n01) / 3, B2 = (c1.n01 + c0.n11) / 3, B3 = c1.n11,
// n00 = a0 x b0, n01 = a1 x b0 + a0 x b1, n11 = a1 x b1; E bounds the error of
// each against the exact ones.  With e the error of a component of a
// difference and U, V, W the largest components of c, a, b, each coefficient is
// a mean of triple products of six terms, so its error is at most
// 6 ((U + e)(V + e)(W + e) - U V W + r U V W), the first part written without
// cancellation, r the roundings per term.
// ---------------------------------------------------------------------------
struct blossom {
  f3 a0, b0, c0, a1, b1, c1;
  f3 n00, n01, n11;
  float B0, B1, B2, B3, E, U, V, W;
};

// p, q: first points of the first and second primitive; h: VF second vertex of
// the triangle, EE second point of the first edge; g: last point.
__device__ __forceinline__ blossom blossom_fp32(bool ee, f3 p, f3 q, f3 h, f3 g, f3 dp, f3 dq, f3 dh, f3 dg, float e) {
  blossom r;
  f3 t = ee ? p : q, dt = ee ? dp : dq;
  r.a0 = fsub(h, t); r.b0 = fsub(g, q); r.c0 = fsub(q, p);
  r.a1 = fadd(r.a0, fsub(dh, dt)); r.b1 = fadd(r.b0, fsub(dg, dq)); r.c1 = fadd(r.c0, fsub(dq, dp));
  r.n00 = fcross(r.a0, r.b0);
  r.n01 = fadd(fcross(r.a1, r.b0), fcross(r.a0, r.b1));
  r.n11 = fcross(r.a1, r.b1);
  r.B0 = fdot(r.c0, r.n00);
  r.B1 = (fdot(r.c1, r.n00) + fdot(r.c0, r.n01)) * (1.f / 3.f);
  r.B2 = (fdot(r.c1, r.n01) + fdot(r.c0, r.n11)) * (1.f / 3.f);
  r.B3 = fdot(r.c1, r.n11);
  r.U = fmaxf(amax3(r.c0), amax3(r.c1));
  r.V = fmaxf(amax3(r.a0), amax3(r.a1));
  r.W = fmaxf(amax3(r.b0), amax3(r.b1));
  float Ve = r.V + e, We = r.W + e, UV = r.U * r.V, mx = fmaxf(r.U, fmaxf(r.V, r.W));
  // 7.5 = 1.25 x 6; roundings: 96 U32 per term; the last term covers FP64
  r.E = 7.5f * e * (fmaf(Ve, We, fmaf(r.U, We, UV))) + 4.3e-5f * UV * r.W + 1.3e-9f * mx * mx * mx;
  return r;
}

// Separation certificate: 1 if the FP64 contact test certainly reports neither
// a contact nor a degenerate pair because the two primitives stay apart along
// one direction over the whole step, 0 if undecided.
//
// With C the vectors from the points of the first primitive to those of the
// second at t = 0 and t = 1 (VF: c + {0, a, b}; EE: c + {0, b} - {0, a}), a
// direction v with v . C > 0 for all of them separates the primitives at every
// time, in whatever way both move together: pairs of two vesicles carried along
// by one flow, whose swept boxes overlap over the long common path, are told
// apart here.  v runs through the first NIT iterates towards the point of the
// hull of the C closest to the origin (their mean, then towards the C lowest
// along v).
//
// Why it decides the FP64 test.  Let n = v / |v|, n . C >= delta, and t a time
// at which the test forms the inside weights: f(t) is zero up to rounding there
// (with d_m > 0, |f| <= d_m |m|).  If the weights passed, the least-squares
// residual r, perpendicular to a and b, would be a mean of the C with weights in
// [-tau, 1 + tau], hence n . r >= delta - 12 tau Cm (Cm >= every component of
// the C), while |r| = |f| / |m|.  The guard: the Bernstein coefficients of
// m(0) . m(t) exceed 1e-3 SA SB (SA, SB the larger squared lengths of a and b,
// at most 3 V^2 and 3 W^2), so |m(t)| >= 1e-3 sqrt(SA SB) on [0, 1].  Then the
// determinant |m|^2 of the normal equations is positive in FP64 (relative error
// below 4e-9), their rounding keeps tau below 4e-9 (1 + Cm / min(V, W)) < 1e-5
// (Cm < 1e3 min(V, W) is required), the rounding of f over a bracket of the root
// gives |f| / |m| < 1e-9 Cm, and that of the positions at t less than the error
// e of the FP32 differences (e covers 2^-32 of the coordinates themselves).  So
// delta = 2e-4 Cm beyond the FP32 errors excludes a contact.  With d_m > 0,
// g = f^2 - d_m^2 |m|^2 is zero up to 2.4e-6 Cm^2 |m|^2, so |f| / |m| <= d_m +
// 1.6e-3 sqrt(3) Cm, within delta = 1.00001 d_m + 5e-3 Cm.  A pair is degenerate
// otherwise only when every FP64 coefficient of the polynomial is exactly zero:
// f (with d_m > 0: g) is shown to be away from zero at t = 0 or t = 1.
template <bool DM, int NIT>
__device__ __forceinline__ int separation_reject(bool ee, const blossom& q, float e, float dm) {
  float VW = q.V * q.W, Cm = q.U + q.V + q.W;
  float g0 = fdot(q.n00, q.n00), g1 = 0.5f * fdot(q.n00, q.n01), g2 = fdot(q.n00, q.n11);
  // error of the g: |m(0)| <= 3 V W times that of a x b
  float em = 6.0f * e * (q.V + q.W) + 4e-6f * VW;
  bool ok = fminf(g0, fminf(g1, g2)) > VW * fmaf(9.1e-3f, VW, 6.1f * em) && Cm < 1e3f * fminf(q.V, q.W);
  if (DM) {   // |g| = ||f| - d_m |m|| (|f| + d_m |m|) away from zero
    float m0 = dm * fnorm(q.n00), m1 = dm * fnorm(q.n11), eg = fmaf(dm, em, q.E);
    ok = ok && (fabsf(fabsf(q.B0) - m0) > eg + 0.01f * m0 || fabsf(fabsf(q.B3) - m1) > eg + 0.01f * m1);
  } else {
    ok = ok && (fabsf(q.B0) > q.E || fabsf(q.B3) > q.E);
  }
  if (!ok) return 0;
  float marg = e + (DM ? 1.00001f * dm + 5.1e-3f * Cm : 2.1e-4f * Cm);
  float al = ee ? -0.25f : 1.f / 6.f, be = ee ? 0.25f : 1.f / 6.f;
  f3 v = {fmaf(be, q.b0.x + q.b1.x, fmaf(al, q.a0.x + q.a1.x, 0.5f * (q.c0.x + q.c1.x))),
          fmaf(be, q.b0.y + q.b1.y, fmaf(al, q.a0.y + q.a1.y, 0.5f * (q.c0.y + q.c1.y))),
          fmaf(be, q.b0.z + q.b1.z, fmaf(al, q.a0.z + q.a1.z, 0.5f * (q.c0.z + q.c1.z)))};
#pragma unroll 1
  for (int it = 0;; ++it) {
    float sa0 = fdot(v, q.a0), sb0 = fdot(v, q.b0), sc0 = fdot(v, q.c0);
    float sa1 = fdot(v, q.a1), sb1 = fdot(v, q.b1), sc1 = fdot(v, q.c1);
    // the lowest C at each end: c + fa a + fb b
    float m0 = ee ? fminf(sb0, 0.f) - fmaxf(sa0, 0.f) : fminf(fminf(sa0, sb0), 0.f);
    float m1 = ee ? fminf(sb1, 0.f) - fmaxf(sa1, 0.f) : fminf(fminf(sa1, sb1), 0.f);
    m0 += sc0; m1 += sc1;
    float mn = fminf(m0, m1);
    if (mn > 1.00001f * marg * (fabsf(v.x) + fabsf(v.y) + fabsf(v.z))) return 1;
    if (it + 1 == NIT) return 0;
    bool end = m1 < m0;
    f3 A = end ? q.a1 : q.a0, B = end ? q.b1 : q.b0, C = end ? q.c1 : q.c0;
    float sa = end ? sa1 : sa0, sb = end ? sb1 : sb0;
    float fa = ee ? (sa > 0.f ? -1.f : 0.f) : (sa < 0.f && sa <= sb ? 1.f : 0.f);
    float fb = ee ? (sb < 0.f ? 1.f : 0.f) : (sb < 0.f && sb < sa ? 1.f : 0.f);
    f3 w = fat(fat(C, fa, A), fb, B);
    f3 u = fsub(w, v);
    float t = __fdividef(-fdot(v, u), fmaxf(fdot(u, u), 1e-30f));
    v = fat(v, fminf(fmaxf(t, 0.0f), 1.0f), u);
  }
}

// Stage 3a on one pair: nonzero if the FP64 test certainly finds nothing.  1: the
// cubic keeps one sign over the step (with d_m > 0: keeps |f| above d_m |m|; |m(t)| is
// at most the largest of |n00|, |n01| / 2, |n11|); 2: the first direction
// separates the primitives.
template <bool DM>
__device__ __forceinline__ int reject_fp32(bool ee, const blossom& q, float e, float dm) {
  float lo = fminf(fminf(q.B0, q.B1), fminf(q.B2, q.B3)), hi = fmaxf(fmaxf(q.B0, q.B1), fmaxf(q.B2, q.B3));
  float f = fmaxf(lo, -hi) - q.E;   // > 0: |f| >= this over the step
  if (DM) {
    float VW = q.V * q.W;
    float n2 = fmaxf(fmaxf(fdot(q.n00, q.n00), 0.25f * fdot(q.n01, q.n01)), fdot(q.n11, q.n11));
    float mm = n2 * rsqrtf(fmaxf(n2, 1e-30f)) * 1.000001f + 1e-15f + 6.0f * e * (q.V + q.W) + 4e-6f * VW;
    float dmm = dm * mm * 1.000001f, s = 162.f * q.U * VW;
    if (f > 0.f && f * f * (1.f - 1e-5f) > dmm * dmm * (1.f + 1e-5f) + 1e-12f * (s * s + dmm * dmm)) return 1;
  } else if (f > 0.f) {
    return 1;
  }
  return 2 * separation_reject<DM, 1>(ee, q, e, dm);
}

// ---------------------------------------------------------------------------
// Eq. 3.1 (d_m = 0): earliest contact time of one primitive pair in FP64.
// Comparisons are done on the bit patterns (integer pipe); the arithmetic is
// the fixed FP64 sequence of the method definition.
// ---------------------------------------------------------------------------
enum { KIND_VF = 0, KIND_EE = 1 };

__device__ __forceinline__ bool is_zero(double v) { return (__double_as_longlong(v) << 1) == 0; }
__device__ __forceinline__ bool is_neg(double v) {  // v < 0.0
  long long b = __double_as_longlong(v);
  return b < 0 && (b << 1) != 0;
}
__device__ __forceinline__ bool is_pos(double v) { return __double_as_longlong(v) > 0; }  // v > 0.0, v not NaN

// (lo + hi) * 0.5 rounded as FP64 does it (nearest, ties to even), for
// 0 <= lo < hi, computed on the integer pipe: add the 53-bit significands
// with guard, round and sticky bits, round, halve the exponent.  ok = false
// when the operands or the result leave the normal range; the caller then
// uses the FP64 instructions.
__device__ __forceinline__ double mid_rn(double lo, double hi, bool& ok) {
  const unsigned long long FR = (1ull << 52) - 1, HID = 1ull << 52;
  unsigned long long a = (unsigned long long)__double_as_longlong(lo), b = (unsigned long long)__double_as_longlong(hi);
  int eb = (int)(b >> 52);
  ok = true;
  if (a == 0) {                                 // lo = 0: the sum is hi
    if (eb < 2) { ok = false; return 0.0; }
    return __longlong_as_double((long long)(b - HID));
  }
  int ea = (int)(a >> 52);
  if (ea == 0) { ok = false; return 0.0; }
  unsigned long long ma = (a & FR) | HID, mb = (b & FR) | HID;
  int d = eb - ea;                              // >= 0 because lo < hi
  unsigned long long M = mb << 3;
  if (d < 56) {
    unsigned long long sa = ma << 3, sh = sa >> d;
    M += sh | (unsigned long long)((sh << d) != sa);
  } else {
    M += 1;                                     // lo only sets the sticky bit
  }
  int e = eb;
  if (M >> 56) { M = (M >> 1) | (M & 1); ++e; }
  unsigned low = (unsigned)(M & 7);
  M >>= 3;
  if (low > 4 || (low == 4 && (M & 1))) ++M;
  if (M >> 53) { M >>= 1; ++e; }
  if (e < 2 || e > 2046) { ok = false; return 0.0; }
  return __longlong_as_double((long long)(((unsigned long long)(e - 1) << 52) | (M & FR)));
}

// FP32 image of t in [0, 1] by truncating the significand: |t - m| <= 2^-23 t
// (m = 0 below 2^-126, where |t - m| <= 2^-126).
__device__ __forceinline__ float trunc_f32(double t) {
  unsigned long long b = (unsigned long long)__double_as_longlong(t);
  int e = (int)(b >> 52) - 1023 + 127;
  if (e < 1) return 0.0f;
  return __uint_as_float(((unsigned)e << 23) | (unsigned)((b >> 29) & 0x7FFFFF));
}

// Double-float (unevaluated sum of two floats) arithmetic for the second
// sign tier of the bisection.  two_prod is exact with an FMA; two_sum is
// exact (the library is built without FMA contraction).
struct dflt { float h, l; };
__device__ __forceinline__ dflt two_sum(float a, float b) {
  float s = a + b, bb = s - a;
  return {s, (a - (s - bb)) + (b - bb)};
}
__device__ __forceinline__ dflt fast_two_sum(float a, float b) {  // |a| >= |b|
  float s = a + b;
  return {s, b - (s - a)};
}
__device__ __forceinline__ dflt df_mul(dflt x, dflt y) {
  float p = x.h * y.h, e = fmaf(x.h, y.h, -p);
  e = e + (x.h * y.l + x.l * y.h);
  return fast_two_sum(p, e);
}
__device__ __forceinline__ dflt df_add(dflt x, dflt y) {
  dflt s = two_sum(x.h, y.h);
  return fast_two_sum(s.h, s.l + (x.l + y.l));
}
// m in [2^-74, 1] as a double-float from its bits: the high part keeps 24
// significant bits, the low part the remaining 29 rounded to 24 (|m - h - l|
// <= 2^-47 m); returns false below that range.
__device__ __forceinline__ bool df_of_unit(double m, dflt& r) {
  unsigned long long b = (unsigned long long)__double_as_longlong(m);
  int E = (int)(b >> 52);
  if (E < 949) return false;
  r.h = __uint_as_float(((unsigned)(E - 1023 + 127) << 23) | (unsigned)((b >> 29) & 0x7FFFFF));
  unsigned rem = (unsigned)(b & ((1ull << 29) - 1));
  r.l = __uint2float_rn(rem) * __uint_as_float((unsigned)(E - 1075 + 127) << 23);
  return true;
}

// FP64 operations of the procedure (+ - * / sqrt = 1, fma = 2, negations and
// comparisons 0): the algorithmic work of the exact contact test.  Halvings and
// critical points that are decided without their values count all the same, so
// that the count over the time is no fraction of the FP64 rate.
//
// The bisection takes exactly the FP64 path: every midpoint is the FP64
// midpoint (mid_rn), and every sign is the sign of the FP64 Horner value.
//
// Most halvings need no value at all.  An approximate root r (FP32 Newton steps,
// two steps on FP64 values) and the FP64 values at r - delta and r + delta prove
// the sign of the FP64 value at every midpoint outside: a segment between
// computed critical points is monotone up to 2^-50 S1, so values of the two signs
// beyond 2^-48 (S + S1) (twice the Horner error and that) stay of their sign
// farther out.  From [0, 1] (nearly every pair) the midpoints are dyadic and
// exact as long as the interval is wider than an ulp, so the halvings down to
// the common binary prefix of r - delta and r + delta (43 of some 54) are taken
// at once.  Those left, and all where r - delta and r + delta prove nothing (r
// near a multiple root), are decided by FP64 values: signs from FP32 and
// double-float values there cost more than they save (0.425 -> 0.41 ms at 1440
// vesicles without them).
struct poly32 { float f0, f1, f2, f3, S, S1; bool in_range; };   // FP32 images of the cubic's coefficients

__device__ __forceinline__ poly32 poly_fp32(double k0, double k1, double k2, double k3) {
  poly32 p;
  p.f0 = __double2float_rn(k0); p.f1 = __double2float_rn(k1); p.f2 = __double2float_rn(k2); p.f3 = __double2float_rn(k3);
  float a0 = fabsf(p.f0), a1 = fabsf(p.f1), a2 = fabsf(p.f2), a3 = fabsf(p.f3);
  float mk = fmaxf(fmaxf(a0, a1), fmaxf(a2, a3));
  p.S = ((a0 + a1) + a2) + a3;
  p.S1 = (a1 + 2.0f * a2) + 3.0f * a3;
  p.in_range = mk > 1e-20f && mk < 1e25f;
  return p;
}

// Points l < h in the segment [lo, hi] (in [0, 1]) such that the FP64 value at a
// midpoint <= l has lo's sign and at one >= h the other; li, hi_: the same in
// units of 2^-62, li <= l, h <= hi_.  False when not found.
__device__ __forceinline__ bool root_bounds(const poly32& p, double k0, double k1, double k2, double k3, bool neg_lo,
                                            double lo, double hi, double& l, double& h, long long& li,
                                            long long& hi_) {
  float a = trunc_f32(lo), b = trunc_f32(hi), dv;
  float va = fmaf(fmaf(fmaf(p.f3, a, p.f2), a, p.f1), a, p.f0), vb = fmaf(fmaf(fmaf(p.f3, b, p.f2), b, p.f1), b, p.f0);
  float r = a + (b - a) * __fdividef(va, va - vb);
  r = r > a && r < b ? r : 0.5f * (a + b);
#pragma unroll 1
  for (int it = 0; it < 4; ++it) {   // Newton, kept in the bracket
    float v = fmaf(fmaf(fmaf(p.f3, r, p.f2), r, p.f1), r, p.f0);
    dv = fmaf(fmaf(3.0f * p.f3, r, 2.0f * p.f2), r, p.f1);
    if ((v < 0.0f) == neg_lo) a = r;
    else b = r;
    float rn = r - __fdividef(v, dv);
    r = rn >= a && rn <= b ? rn : 0.5f * (a + b);
  }
  // two steps on FP64 values, in units of 2^-62
  unsigned rb = __float_as_uint(r);
  int ex = (int)(rb >> 23);
  if (ex < 88) return false;
  long long rc = (long long)((rb & 0x7FFFFFu) | 0x800000u) << (ex - 88);   // (1.m) 2^(ex - 127) 2^62
  dv = fmaf(fmaf(3.0f * p.f3, r, 2.0f * p.f2), r, p.f1);
  const float scale = __fdividef(4.6116860e18f, dv);
#pragma unroll
  for (int it = 0; it < 2; ++it) {
    double rd = __longlong_as_double(__double_as_longlong(__ll2double_rn(rc)) - (62ll << 52));
    float corr = __double2float_rn(horner3(k0, k1, k2, k3, rd)) * scale;
    if (!(fabsf(corr) < 4e15f)) return false;   // 1e-3
    rc -= __float2ll_rn(corr);
    if (rc <= 0) return false;
  }
  float Eb = 3.5527137e-15f * (p.S + p.S1);   // 2^-48
  float delta = fabsf(2.0f * Eb * scale) + 65536.0f;   // + 2^-46
  if (!(delta < 4e15f)) return false;
  long long dl = __float2ll_rn(delta);
  li = rc - dl; hi_ = rc + dl;
  if (li <= 0 || hi_ >= (1ll << 62)) return false;
  // to doubles, towards each other, so that they lie inside [li, hi_]
  l = __longlong_as_double(__double_as_longlong(__ll2double_ru(li)) - (62ll << 52));
  h = __longlong_as_double(__double_as_longlong(__ll2double_rd(hi_)) - (62ll << 52));
  if (__double_as_longlong(l) < __double_as_longlong(lo) || __double_as_longlong(h) > __double_as_longlong(hi)) return false;
  float fl = __double2float_rn(horner3(k0, k1, k2, k3, l)), fh = __double2float_rn(horner3(k0, k1, k2, k3, h));
  return neg_lo ? fl < -Eb && fh > Eb : fl > Eb && fh < -Eb;
}

__device__ double bisect64(const poly32& p, double k0, double k1, double k2, double k3, double lo, double hi,
                           double flo, long long& flops) {
  const bool neg_lo = is_neg(flo);
  int it = 0;
  double l, h;   // signs known up to l and from h on
  {
    long long li, hi_;
    if (p.in_range && root_bounds(p, k0, k1, k2, k3, neg_lo, lo, hi, l, h, li, hi_)) {
      if (__double_as_longlong(lo) == 0 && __double_as_longlong(hi) == 0x3FF0000000000000ll) {
        it = __clzll(li ^ hi_) - 2;   // the cell of 2^-it that holds both
        long long c = li >> (62 - it);
        const long long down = (long long)it << 52;
        if (c) lo = __longlong_as_double(__double_as_longlong(__ll2double_rn(c)) - down);
        hi = __longlong_as_double(__double_as_longlong(__ll2double_rn(c + 1)) - down);
        flops += 8 * it;
      }
    } else {
      l = -1.0; h = 2.0;
    }
  }
#pragma unroll 1
  for (; it < 64; ++it) {
    bool ok;
    double mid = mid_rn(lo, hi, ok);
    if (!ok) mid = __dmul_rn(__dadd_rn(lo, hi), 0.5);
    flops += 2;
    // lo, mid, hi are non-negative: compare bit patterns
    long long bm = __double_as_longlong(mid);
    if (!(bm > __double_as_longlong(lo) && bm < __double_as_longlong(hi))) break;
    flops += 6;
    bool neg = neg_lo, done = bm <= __double_as_longlong(l);   // l = -1: a negative pattern
    if (bm >= __double_as_longlong(h)) { neg = !neg_lo; done = true; }
    if (!done) {
      double fm = horner3(k0, k1, k2, k3, mid);
      if (is_zero(fm)) return mid;
      neg = is_neg(fm);
    }
    if (neg == neg_lo) lo = mid;
    else hi = mid;
  }
  return lo;
}

// n / den < 0 for den > 0, decided from the sign of n when the quotient
// cannot underflow to -0: |n| >= 2^-899 and den < 2^171 give |n / den| >
// 2^-1070.
__device__ __forceinline__ bool quot_neg(double n, double den) {
  long long b = __double_as_longlong(n);
  return b < 0 && ((b >> 52) & 0x7FF) >= 124 && (__double_as_longlong(den) >> 52) <= 1193;
}
// n / den rounds above 1 for positive n, den: n exceeds den by more than 8
// units in the last place (then n / den > 1 + 2^-50).
__device__ __forceinline__ bool quot_above1(double n, double den) {
  long long bn = __double_as_longlong(n), bd = __double_as_longlong(den);
  return bn > 0 && bn > bd + 8;
}

// Inside test at the positions Y (VF: xp, x0, x1, x2; EE: p0, q0, p1, q1).
// 1 inside, 0 outside, -1 degenerate.  The weights are the normal equations'
// solution with a = x1 - x0 (p1 - p0), b = x2 - x0 (q1 - q0), c = xp - x0
// (p0 - q0); the two kinds differ in which product of the first numerator is
// rounded, so both take the same instructions on selected operands (in a warp
// that holds both kinds the FP64 work is done once).  A quotient whose sign
// (or excess over 1, of the sum for VF) is decided by its numerator is not
// formed when that already decides "outside": the decision equals that of the
// rounded quotient.
__device__ int inside64(int kind, const d3* Y, double& w1, double& w2) {
  const bool ee = kind != KIND_VF;
  d3 T = {ee ? Y[0].x : Y[1].x, ee ? Y[0].y : Y[1].y, ee ? Y[0].z : Y[1].z};
  d3 a = d3_sub(Y[2], T), b = d3_sub(Y[3], Y[1]), c = d3_sub(Y[0], Y[1]);
  double d00 = d3_dot(a, a), d01 = d3_dot(a, b), d11 = d3_dot(b, b), d20 = d3_dot(c, a), d21 = d3_dot(c, b);
  double den = __fma_rn(d00, d11, -__dmul_rn(d01, d01));
  if (!is_pos(den)) return -1;
  // VF: d11 d20 - d01 d21; EE: d01 d21 - d20 d11
  double u1 = ee ? d01 : d11, u2 = ee ? d21 : d20, v1 = ee ? d20 : d01, v2 = ee ? d11 : d21;
  double n1 = __fma_rn(u1, u2, -__dmul_rn(v1, v2));
  double n2 = __fma_rn(d00, d21, -__dmul_rn(d01, d20));
  if (quot_neg(n1, den) || quot_neg(n2, den)) return 0;
  if (ee) {
    if (quot_above1(n1, den) || quot_above1(n2, den)) return 0;
  } else {
    // 1 - b1 - b2 is rounded twice: 8 ulps beyond are certain
    if (is_pos(n1) && is_pos(n2) && quot_above1(__dadd_rn(n1, n2), den)) return 0;
  }
  double q1 = __ddiv_rn(n1, den);
  double q2 = __ddiv_rn(n2, den);
  w1 = q1; w2 = q2;
  if (is_neg(q1) || is_neg(q2)) return 0;
  if (ee) {
    const long long one = 0x3FF0000000000000ll;
    return __double_as_longlong(q1) <= one || is_zero(q1) ? (__double_as_longlong(q2) <= one || is_zero(q2) ? 1 : 0) : 0;
  }
  double b0 = __dsub_rn(__dsub_rn(1.0, q1), q2);
  return !is_neg(b0) ? 1 : 0;
}

// The rounded quotient n / d when it may lie in (0, 1), else -1: it cannot
// when n is zero, the signs differ, or |n| >= |d| (then n / d >= 1 exactly,
// and so rounded); only the remaining case is divided (an exact quotient in
// (0, 1) may still round to 0 or 1, which the division decides).  Zero or
// NaN d falls in the |n| >= |d| or sign cases exactly as the quotient would
// fall outside (0, 1).
__device__ __forceinline__ double quot01(double n, double d) {
  if (is_zero(n) || is_neg(n) != is_neg(d) || !(fabs(n) < fabs(d))) return -1.0;
  return __ddiv_rn(n, d);
}

// The difference vectors of the cubic from the points (VF: xp, x0, x1, x2; EE:
// p0, q0, p1, q1): a = x1 - x0 (p1 - p0), b = x2 - x0 (q1 - q0), c = xp - x0
// (q0 - p0, the exact negative of p0 - q0).
__device__ __forceinline__ void pair_diffs(bool ee, const d3* X, d3& a, d3& b, d3& c) {
  d3 T = {ee ? X[0].x : X[1].x, ee ? X[0].y : X[1].y, ee ? X[0].z : X[1].z};
  a = d3_sub(X[2], T);
  b = d3_sub(X[3], X[1]);
  c = d3_sub(X[0], X[1]);
  const long long flip = ee ? (long long)0x8000000000000000ull : 0ll;
  c.x = __longlong_as_double(__double_as_longlong(c.x) ^ flip);
  c.y = __longlong_as_double(__double_as_longlong(c.y) ^ flip);
  c.z = __longlong_as_double(__double_as_longlong(c.z) ^ flip);
}

// 0 no contact, 1 contact, 2 degenerate.  Points as for pair_diffs.
__device__ int ccd64(int kind, const d3* X0, const d3* D, double& tau, double& w1, double& w2, long long& flops) {
  flops += 18 + 9 + 21 + 9 + 32;  // differences, cross products (+ sum), 6 dot products + 2 sums
  d3 a, b, c, da, db, dc;
  const bool ee = kind != KIND_VF;
  pair_diffs(ee, X0, a, b, c);
  pair_diffs(ee, D, da, db, dc);
  d3 n0 = d3_cross(a, b);
  d3 n1 = d3_add(d3_cross(da, b), d3_cross(a, db));
  d3 n2 = d3_cross(da, db);
  double k0 = d3_dot(c, n0);
  double k1 = __dadd_rn(d3_dot(dc, n0), d3_dot(c, n1));
  double k2 = __dadd_rn(d3_dot(c, n2), d3_dot(dc, n1));
  double k3 = d3_dot(dc, n2);
  if (is_zero(k0) && is_zero(k1) && is_zero(k2) && is_zero(k3)) return 2;
  poly32 p = poly_fp32(k0, k1, k2, k3);
  flops += 2;
  // Critical points.  When the FP32 images prove that the derivative keeps one
  // sign on [0, 1] (its Bernstein coefficients beyond 1e-5 S1; each root of the
  // stable formula is the root of a quadratic with coefficients a few ulps
  // away), none is computed there; only the discriminant's sign is taken, for
  // the operation count.
  double r[2]; int nr = 0;
  {
    float d1 = p.f1 + p.f2, d2 = (p.f1 + 2.0f * p.f2) + 3.0f * p.f3, m = 1e-5f * p.S1;
    float q4 = 4.0f * p.f2 * p.f2, q12 = 12.0f * p.f3 * p.f1, dsc = q4 - q12;
    bool none = p.in_range && !is_zero(k3) && fminf(p.f1, fminf(d1, d2)) > m;
    none = none || (p.in_range && !is_zero(k3) && fmaxf(p.f1, fmaxf(d1, d2)) < -m);
    if (none && p.S < 1e12f && q4 + fabsf(q12) > 1e-30f && fabsf(dsc) > 1e-5f * (q4 + fabsf(q12))) {
      flops += dsc > 0.0f ? 9 : 4;
    } else {
      double e0 = k1, e1 = __dmul_rn(2.0, k2), e2 = __dmul_rn(3.0, k3);
      if (!is_zero(e2)) {
        double disc = __fma_rn(e1, e1, -__dmul_rn(__dmul_rn(4.0, e2), e0));
        flops += 4;
        if (is_pos(disc)) {
          flops += 5;
          double sq = __dsqrt_rn(disc);
          double q = __dmul_rn(-0.5, __dadd_rn(e1, !is_neg(e1) ? sq : -sq));
          r[0] = quot01(q, e2); r[1] = quot01(e0, q); nr = 2;
        }
      } else if (!is_zero(e1)) {
        r[0] = quot01(-e0, e1); nr = 1;
        flops += 1;
      }
    }
  }
  double cp[2]; int ncp = 0;
  for (int i = 0; i < nr; ++i) if (r[i] > 0.0 && r[i] < 1.0) cp[ncp++] = r[i];
  if (ncp == 2) {
    if (cp[1] < cp[0]) { double t = cp[0]; cp[0] = cp[1]; cp[1] = t; }
    if (cp[1] == cp[0]) ncp = 1;
  }
  // the value at 1, from FP32 when that proves its sign: |f64 - f32| <=
  // gamma_6(2^-53) S + 2^-24 S + gamma_6(2^-24) S (1 + 2^-24) (Horner errors and
  // coefficient rounding) stays below 4.5e-7 S
  double f1v;
  {
    float fs = ((p.f3 + p.f2) + p.f1) + p.f0;
    if (p.in_range && fabsf(fs) > 1.01f * (4.5e-7f * p.S + 1.25e-7f * p.S1)) f1v = fs < 0.0f ? -1.0 : 1.0;
    else f1v = horner3(k0, k1, k2, k3, 1.0);
  }
  double l = 0.0, fl = k0;   // the value at 0 is k0
  bool degen = false;
#pragma unroll 1
  for (int s = 0; s <= ncp; ++s) {
    double rr = s < ncp ? cp[s] : 1.0;
    double fr = s < ncp ? horner3(k0, k1, k2, k3, rr) : f1v, t = l;
    flops += 12;
    bool take = true;
    if (is_zero(fl)) t = l;
    else if (is_zero(fr)) t = rr;
    else if (is_neg(fl) != is_neg(fr)) t = bisect64(p, k0, k1, k2, k3, l, rr, fl, flops);
    else take = false;
    if (take) {
      flops += 24 + 9 + 25 + 3;  // positions, differences, dot products, determinant
      d3 Y[4];
      for (int q = 0; q < 4; ++q) Y[q] = d3_at(X0[q], t, D[q]);
      double u1 = 0.0, u2 = 0.0;
      int in = inside64(kind, Y, u1, u2);
      if (in >= 0) flops += kind == KIND_VF ? 10 : 8;  // numerators, divisions (and 1 - b1 - b2)
      if (in < 0) degen = true;
      if (in == 1) { tau = t; w1 = u1; w2 = u2; return 1; }
    }
    l = rr; fl = fr;
  }
  return degen ? 2 : 0;
}

// ---------------------------------------------------------------------------
// Eq. 3.1 with d_m > 0: g(t) = f(t)^2 - d_m^2 |m(t)|^2 (f the cubic, m the
// normal), degree six.  The roots of the derivatives, found from the linear
// one upward, split [0, 1] into pieces on which each derivative (and finally
// g) is monotone; each piece is taken as in the cubic test, and the first
// piece also at t = 0 when g(0) <= 0.  The fixed FP64 sequence of the method
// definition (plain FP64 instructions, no sign tiers); the stage-4 operation
// count covers the d_m = 0 procedure only.
// ---------------------------------------------------------------------------
__device__ __forceinline__ double horner_n(const double* c, int n, double t) {
  double r = c[n];
  for (int i = n - 1; i >= 0; --i) r = __fma_rn(r, t, c[i]);
  return r;
}

// The bisection of a degree-N polynomial c on [lo, hi] (0 <= lo < hi <= 1),
// taking exactly the FP64 path of the plain procedure: every midpoint is the
// FP64 midpoint, every sign the sign of the FP64 Horner value.  As in the
// cubic's bisection, that sign is read from cheaper evaluations when their
// error bounds prove it.  With S = sum |c_i| and S1 = sum i |c_i|:
//  - FP32 Horner at the truncated midpoint: |f64(mid) - f32| <=
//    gamma_2N(2^-24) S + 2^-24 S + gamma_2N(2^-53) S + 2^-23 S1 (Horner error
//    bounds with room to spare, coefficient rounding, the FP64 value's own
//    error, the midpoint's truncation times max |f'| on [0, 1]) <=
//    (2N + 1.5) 2^-24 S + 1.25e-7 S1 for N <= 6;
//  - double-float Horner: N multiply-add steps at <= 2^-44 relative each, the
//    coefficients' and the midpoint's representation (2^-48 |c_i|, 2^-47 mid
//    times max |f'|) and the FP64 Horner error (< 2^-50 S) stay below
//    2^-40 (S + S1) for N <= 6.
// Above its bound a tier's value has the sign of the FP64 value, which is
// then not zero.  Coefficients outside [1e-25, 1e25] (1e-20 for the
// double-float tier) keep every FP32 term clear of underflow and overflow;
// outside that range only FP64 is used.
template <int N>
__device__ __noinline__ double bisect_tn(const double* c, double lo, double hi, double flo, long long& flops) {
  bool neg_lo = is_neg(flo);
  float fc[N + 1];
  dflt cd[N + 1];
  float S = 0.0f, S1 = 0.0f, mk = 0.0f;
#pragma unroll
  for (int i = 0; i <= N; ++i) {
    fc[i] = __double2float_rn(c[i]);
    float ai = fabsf(fc[i]);
    S = S + ai;
    S1 = S1 + (float)i * ai;
    mk = fmaxf(mk, ai);
    cd[i] = {fc[i], __double2float_rn(__dsub_rn(c[i], (double)fc[i]))};
  }
  float E = 1.01f * ((2.0f * N + 1.5f) * 5.9604645e-8f * S + 1.25e-7f * S1);
  float Edf = 1.01f * 9.094947e-13f * (S + S1);   // 2^-40
  bool use_df = mk > 1e-20f && mk < 1e25f;
  if (!(mk > 1e-25f && mk < 1e25f)) E = INFINITY;
#pragma unroll 1
  for (int it = 0; it < 64; ++it) {
    bool ok;
    double mid = mid_rn(lo, hi, ok);
    if (!ok) mid = __dmul_rn(__dadd_rn(lo, hi), 0.5);
    long long bm = __double_as_longlong(mid);   // lo, mid, hi >= 0: bit patterns order them
    if (!(bm > __double_as_longlong(lo) && bm < __double_as_longlong(hi))) break;
    flops += 2 + 2 * N;
    float m = trunc_f32(mid);
    float fs = fc[N];
#pragma unroll
    for (int i = N - 1; i >= 0; --i) fs = fmaf(fs, m, fc[i]);
    bool neg;
    dflt md;
    bool done = fabsf(fs) > E;
    if (done) {
      neg = fs < 0.0f;
    } else if (use_df && df_of_unit(mid, md)) {
      dflt v = cd[N];
#pragma unroll
      for (int i = N - 1; i >= 0; --i) v = df_add(df_mul(v, md), cd[i]);
      float vv = v.h + v.l;
      neg = vv < 0.0f;
      done = fabsf(vv) > Edf;
    }
    if (!done) {
      double fm = horner_n(c, N, mid);
      if (is_zero(fm)) return mid;
      neg = is_neg(fm);
    }
    if (neg == neg_lo) lo = mid;
    else hi = mid;
  }
  return lo;
}

__device__ __forceinline__ double bisect_n(const double* c, int n, double lo, double hi, double flo,
                                           long long& flops) {
  switch (n) {
    case 2: return bisect_tn<2>(c, lo, hi, flo, flops);
    case 3: return bisect_tn<3>(c, lo, hi, flo, flops);
    case 4: return bisect_tn<4>(c, lo, hi, flo, flops);
    case 5: return bisect_tn<5>(c, lo, hi, flo, flops);
    default: return bisect_tn<6>(c, lo, hi, flo, flops);
  }
}

__device__ __noinline__ int ccd64_dm(int kind, const d3* X0, const d3* D, double dm, double& tau, double& w1,
                                     double& w2, long long& flops) {
  d3 a, b, c, da, db, dc;
  pair_diffs(kind != KIND_VF, X0, a, b, c);
  pair_diffs(kind != KIND_VF, D, da, db, dc);
  d3 n0 = d3_cross(a, b);
  d3 n1 = d3_add(d3_cross(da, b), d3_cross(a, db));
  d3 n2 = d3_cross(da, db);
  double k0 = d3_dot(c, n0);
  double k1 = __dadd_rn(d3_dot(dc, n0), d3_dot(c, n1));
  double k2 = __dadd_rn(d3_dot(c, n2), d3_dot(dc, n1));
  double k3 = d3_dot(dc, n2);
  double q0 = d3_dot(n0, n0);
  double q1 = __dmul_rn(2.0, d3_dot(n0, n1));
  double q2 = __dadd_rn(d3_dot(n1, n1), __dmul_rn(2.0, d3_dot(n0, n2)));
  double q3 = __dmul_rn(2.0, d3_dot(n1, n2));
  double q4 = d3_dot(n2, n2);
  double dd = __dmul_rn(dm, dm);
  // C[k]: the k-th derivative of g, degree 6 - k
  double C[6][7];
  C[0][0] = __dsub_rn(__dmul_rn(k0, k0), __dmul_rn(dd, q0));
  C[0][1] = __dsub_rn(__dmul_rn(2.0, __dmul_rn(k0, k1)), __dmul_rn(dd, q1));
  C[0][2] = __dsub_rn(__dadd_rn(__dmul_rn(2.0, __dmul_rn(k0, k2)), __dmul_rn(k1, k1)), __dmul_rn(dd, q2));
  C[0][3] = __dsub_rn(__dmul_rn(2.0, __dadd_rn(__dmul_rn(k0, k3), __dmul_rn(k1, k2))), __dmul_rn(dd, q3));
  C[0][4] = __dsub_rn(__dadd_rn(__dmul_rn(2.0, __dmul_rn(k1, k3)), __dmul_rn(k2, k2)), __dmul_rn(dd, q4));
  C[0][5] = __dmul_rn(2.0, __dmul_rn(k2, k3));
  C[0][6] = __dmul_rn(k3, k3);
  // differences 18, normals 39, cubic 32, |m|^2 34, d_m^2 1, sextic 28, derivatives 20
  flops += 18 + 39 + 32 + 34 + 1 + 28 + 20;
  bool allz = true;
  for (int i = 0; i <= 6; ++i) allz = allz && is_zero(C[0][i]);
  if (allz) return 2;
  for (int k = 1; k < 6; ++k)
    for (int i = 0; i <= 6 - k; ++i) C[k][i] = __dmul_rn((double)(i + 1), C[k - 1][i + 1]);
  // roots in (0, 1) of C[5] (linear), then C[4], ..., C[1] = g'
  double rts[6], nrt[6];
  int nr = 0;
  if (!is_zero(C[5][1])) {
    double t = __ddiv_rn(-C[5][0], C[5][1]);
    flops += 1;
    if (t > 0.0 && t < 1.0) rts[nr++] = t;
  }
  for (int k = 4; k >= 1; --k) {
    int n = 6 - k, nn = 0;
    for (int sgi = 0; sgi <= nr; ++sgi) {
      double l = sgi == 0 ? 0.0 : rts[sgi - 1], r = sgi == nr ? 1.0 : rts[sgi];
      double fl = horner_n(C[k], n, l), fr = horner_n(C[k], n, r), t;
      flops += 4 * n;
      if (is_zero(fl)) t = l;
      else if (is_zero(fr)) t = r;
      else if (is_neg(fl) != is_neg(fr)) t = bisect_n(C[k], n, l, r, fl, flops);
      else continue;
      if (t > 0.0 && t < 1.0 && (nn == 0 || t > nrt[nn - 1])) nrt[nn++] = t;
    }
    for (int i = 0; i < nn; ++i) rts[i] = nrt[i];
    nr = nn;
  }
  bool degen = false;
  for (int sgi = 0; sgi <= nr; ++sgi) {
    double l = sgi == 0 ? 0.0 : rts[sgi - 1], r = sgi == nr ? 1.0 : rts[sgi];
    double gl = horner_n(C[0], 6, l), gr = horner_n(C[0], 6, r), t;
    flops += 24;
    if (sgi == 0 && (is_neg(gl) || is_zero(gl))) t = l;
    else if (is_zero(gl)) t = l;
    else if (is_zero(gr)) t = r;
    else if (is_neg(gl) != is_neg(gr)) t = bisect_n(C[0], 6, l, r, gl, flops);
    else continue;
    flops += 24 + 9 + 25 + 3;  // positions, differences, dot products, determinant
    d3 Y[4];
    for (int q = 0; q < 4; ++q) Y[q] = d3_at(X0[q], t, D[q]);
    double u1 = 0.0, u2 = 0.0;
    int in = inside64(kind, Y, u1, u2);
    if (in >= 0) flops += kind == KIND_VF ? 10 : 8;  // numerators, divisions (and 1 - b1 - b2)
    if (in < 0) { degen = true; continue; }
    if (in == 1) { tau = t; w1 = u1; w2 = u2; return 1; }
  }
  return degen ? 2 : 0;
}

// ---------------------------------------------------------------------------
// global pair descriptors (stages 3b and 4)
// ---------------------------------------------------------------------------
__device__ __forceinline__ unsigned long long make_desc(int r, int type, int ga, int gb) {
  return ((unsigned long long)(unsigned)r << 32) | ((unsigned long long)type << 30) | ((unsigned long long)ga << 15) |
         (unsigned long long)gb;
}

// The 4 points of a descriptor: vertex id and whether the point belongs to
// vesicle j (periodic image applied).  VF type 0: vertex of i, triangle of j;
// type 1: vertex of j, triangle of i; EE: edge of i, edge of j.
__device__ __forceinline__ void desc_points(ulonglong2 e, int& r, int& type, int& ga, int& gb, int* vid, bool* onj) {
  r = (int)(e.x >> 32); type = (int)((e.x >> 30) & 3); ga = (int)((e.x >> 15) & 0x7FFF); gb = (int)(e.x & 0x7FFF);
  for (int q = 0; q < 4; ++q) vid[q] = (int)((e.y >> (16 * q)) & 0xFFFF);
  onj[0] = type == 1;
  onj[1] = type == 0;
  onj[2] = type != 1;
  onj[3] = type != 1;
}

// FP32 points of a descriptor in the frame of its pair (for stage 3b).
__device__ __forceinline__ void desc_points_f32(const narrow_args& a, ulonglong2 e, int& kind, f3* xq, f3* dq,
                                                float& ep, float& es) {
  int r, ty, ga, gb, vid[4];
  bool onj[4];
  desc_points(e, r, ty, ga, gb, vid, onj);
  const stiv_pair_info* pi = a.pinfo + r;
  float4 fr = pi->frame;
  int vi = pi->vi, vj = pi->vj;
  ep = fr.w;
  es = same_side_err(fmaxf(((const float4*)a.vorg)[vi].w, ((const float4*)a.vorg)[vj].w),
                     fmaxf(fabsf(fr.x), fmaxf(fabsf(fr.y), fabsf(fr.z))));
  kind = ty == 2 ? 1 : 0;
  for (int q = 0; q < 4; ++q) {
    int v = onj[q] ? vj : vi;
    const float4* fp = (const float4*)(a.fprep + (size_t)v * a.fstride) + 2 * (size_t)vid[q];
    float4 x = fp[0], d = fp[1];
    if (a.mixed) {   // FP32 vertices as stored: relative position and displacement, one rounding each
      float4 o = ((const float4*)a.vorg)[v];
      d = make_float4(d.x - x.x, d.y - x.y, d.z - x.z, 0.f);
      x = make_float4(x.x - o.x, x.y - o.y, x.z - o.z, 0.f);
    }
    float o0 = onj[q] ? fr.x : 0.f, o1 = onj[q] ? fr.y : 0.f, o2 = onj[q] ? fr.z : 0.f;
    xq[q] = {x.x + o0, x.y + o1, x.z + o2};
    dq[q] = {d.x, d.y, d.z};
  }
}

// Append a descriptor to a global list (warp-aggregated; lanes with keep).
__device__ __forceinline__ void push_global(ulonglong2* list, int64_t cap, int64_t* count, int64_t* status,
                                            bool keep, ulonglong2 e, int lane) {
  unsigned m = __ballot_sync(0xffffffffu, keep);
  if (!m) return;
  unsigned long long base = 0;
  int leader = __ffs(m) - 1;
  if (lane == leader) base = atomicAdd((unsigned long long*)count, (unsigned long long)__popc(m));
  base = __shfl_sync(0xffffffffu, base, leader);
  if (keep) {
    int64_t k = (int64_t)base + __popc(m & ((1u << lane) - 1u));
    if (k < cap) list[k] = e;
    else atomicOr((unsigned long long*)status, STIV_F_WORK_OVERFLOW);
  }
}

// The exact FP64 swept-box test of a queued primitive pair (slots sl; na of
// them on the first primitive) from the vertex values themselves (FP64, or the
// FP32 values widened), the second vesicle's points at the pair's periodic
// image (added in FP64) and, with d_m > 0, its per-vertex boxes widened by d_m:
// the test that defines the pairs tested, for the rare pair whose FP32 boxes
// and their error bound do not decide it.
template <bool MIXED, bool DM>
__device__ __noinline__ bool exact_box_hit(const WarpSm& ws, const narrow_args& a, int r, int na, const int* sl) {
  const stiv_pair_info& pi = a.pinfo[r];
  int code = pi.code;
  int sB[3] = {code / 9 - 1, (code / 3) % 3 - 1, code % 3 - 1};
  double lo[2][3], hi[2][3];
  for (int side = 0; side < 2; ++side)
    for (int c = 0; c < 3; ++c) { lo[side][c] = INFINITY; hi[side][c] = -INFINITY; }
  for (int q = 0; q < 4; ++q) {
    bool onB = sl[q] >= NSLOT;   // the point belongs to vesicle j (patch B)
    int side = q < na ? 0 : 1;
    int v = __float_as_int(ws.x[sl[q]].w);
    int P = onB ? (pi.Pij >> 16) : (pi.Pij & 0xFFFF);
    int nv = stiv_nverts(P);
    size_t vb = (size_t)(onB ? pi.voff_j : pi.voff_i) + v;
    for (int c = 0; c < 3; ++c) {
      double p0 = vtx<MIXED>(a.X, vb + (size_t)c * nv), p1 = vtx<MIXED>(a.X, vb + (size_t)(3 + c) * nv);
      if (onB && sB[c] != 0) { double shc = sB[c] * a.L[c]; p0 = p0 + shc; p1 = p1 + shc; }
      double l = fmin(p0, p1), h = fmax(p0, p1);
      if (DM && onB) {   // d_m > 0: vesicle j's boxes widened by d_m per vertex (FP64, as computed)
        l = __dsub_rn(l, a.dm);
        h = __dadd_rn(h, a.dm);
      }
      lo[side][c] = fmin(lo[side][c], l);
      hi[side][c] = fmax(hi[side][c], h);
    }
  }
  bool hit = true;
  for (int c = 0; c < 3; ++c) hit = hit && lo[0][c] <= hi[1][c] && lo[1][c] <= hi[0][c];
  return hit;
}

// Whether the exact boxes of a pair whose staged boxes overlap do: certainly
// when the staged ones overlap by gap on every axis, else by the exact test.
template <bool MIXED, bool DM>
__device__ __forceinline__ bool box_hit(const WarpSm& ws, const narrow_args& a, int r, int na, const int* sl, float gap) {
  float4 l0 = ws.lo[sl[0]], h0 = ws.hi[sl[0]], l1 = ws.lo[sl[3]], h1 = ws.hi[sl[3]];
#pragma unroll
  for (int q = 1; q < 3; ++q) {
    float4 l = ws.lo[sl[q]], h = ws.hi[sl[q]];
    if (q < na) {
      l0.x = fminf(l0.x, l.x); l0.y = fminf(l0.y, l.y); l0.z = fminf(l0.z, l.z);
      h0.x = fmaxf(h0.x, h.x); h0.y = fmaxf(h0.y, h.y); h0.z = fmaxf(h0.z, h.z);
    } else {
      l1.x = fminf(l1.x, l.x); l1.y = fminf(l1.y, l.y); l1.z = fminf(l1.z, l.z);
      h1.x = fmaxf(h1.x, h.x); h1.y = fmaxf(h1.y, h.y); h1.z = fmaxf(h1.z, h.z);
    }
  }
  if (h1.x - l0.x >= gap && h1.y - l0.y >= gap && h1.z - l0.z >= gap && h0.x - l1.x >= gap && h0.y - l1.y >= gap &&
      h0.z - l1.z >= gap)
    return true;
  return exact_box_hit<MIXED, DM>(ws, a, r, na, sl);
}

// Global triangle id of the triangle with slots s0, s1, s2 (relative to its
// patch) of a patch.
__device__ __forceinline__ int tri_gid(const PatchRef& R, int s0, int s1, int s2) {
  int W = 2 * R.P, r0 = R.I * STIV_BR, c0 = R.J * STIV_BC;
  if (s0 == PSLOT) {
    bool north = s2 > s1;
    return 4 * R.P * R.P + (north ? 0 : W) + c0 + (north ? s1 : s2 - R.tp->frow);
  }
  int rr = s0 / (STIV_BC + 1), cc = s0 - rr * (STIV_BC + 1);
  return 2 * ((r0 + rr) * W + c0 + cc) + (s1 == s0 + STIV_BC + 1 ? 0 : 1);
}

// Stages 1-3a: one warp per patch pair.
//
// Stage 1 without lists: a lane stands for a vertex, a triangle and an edge of
// patch B, and finds the primitives of A whose boxes meet its own from the slot
// masks, all at once (shifts of the masks stand for A's triangles and edges).
// The hits are counted, laid out in the warp's queue by one scan, and go
// through stages 2 and 3a on full warps; survivors are compacted in place and
// pushed together.
//
// Four CTAs of 8 warps an SM (139 KB of staging): bound by issue slots, 74 %
// of them busy.  4096 vesicles 7.7 ms, with three CTAs 8.3, with five (registers
// spill) 8.0; 1440 of order 16 0.58, 0.62 and 0.62 ms.
template <bool MIXED, bool DM>
__global__ void __launch_bounds__(NW * 32, 4) narrow_kernel(narrow_args a) {
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ PatchTopo topo[NVAR];
  WarpSm& ws = ((WarpSm*)smraw)[threadIdx.x >> 5];
  const int lane = threadIdx.x & 31;
  const unsigned lower = (1u << lane) - 1u;
  for (int var = threadIdx.x >> 5; var < NVAR; var += NW) build_topo(topo[var], var, lane);
  __syncthreads();
  int64_t nwork = a.ctr[STIV_C_PATCH];
  if (nwork > a.W) nwork = a.W;
  long long nprim = 0, nleft = 0;   // pairs whose exact boxes overlap; of them, those the sign test leaves
  long long item = 0;
  if (lane == 0) item = (long long)atomicAdd((unsigned long long*)&a.ctr[10], 1ull);
  item = __shfl_sync(0xffffffffu, item, 0);
  while (item < nwork) {
    // the next item's index is fetched now and read at the end of this one
    long long next = 0;
    if (lane == 0) next = (long long)atomicAdd((unsigned long long*)&a.ctr[10], 1ull);
    uint64_t w = a.work[item];
    const int r = (int)(w >> 32);
    const stiv_pair_info* pi = a.pinfo + r;
    const float4 frame = pi->frame;
    const int Pij = pi->Pij;
    const PatchRef A = patch_ref(topo, Pij & 0xFFFF, pi->vi, (int)((w >> 16) & 0xFFFF));
    const PatchRef B = patch_ref(topo, Pij >> 16, pi->vj, (int)(w & 0xFFFF));
    float gap, dmax;
    stage_pair<MIXED, DM>(ws, a, A, B, frame, lane, gap, dmax);
    const bool unsure = slot_masks(ws, gap, lane);
    __syncwarp();
    // stage 1
    unsigned hv = 0, ht = 0, he = 0, hd = 0;   // hits of this lane's vertex, triangle and edge of B
    {
      const PatchTopo& TA = *A.tp;
      const PatchTopo& TB = *B.tp;
      const unsigned qm = TA.qm, fm = TA.fm;
      const int fr = TA.frow;
      if (lane < TB.nv) {   // against A's triangles: bits 0-8 first of a quad, 10-13 fan; 16-24 second of a quad
        uint4 m = ws.miss[TB.v[lane]];
        uint4 dg = and4(m, shr4(m, STIV_BC + 2));
        hv = (hits_of(and4(dg, shr4(m, STIV_BC + 1))) & qm) | ((hits_of(and4(dg, shr4(m, 1))) & qm) << 16);
        if (fm) hv |= (hits_of(and4(and4(shr4(m, fr), shr4(m, fr + 1)), pole4(m))) & fm) << 10;
      }
      if (lane < TB.nt) {   // against A's vertices
        int t = TB.t[lane];
        ht = hits_of(and4(and4(ws.miss[t & 15], ws.miss[(t >> 4) & 15]), ws.miss[t >> 8])) & TA.vm;
      }
      if (a.include_ee && lane < TB.ne) {   // against A's edges: along a row, down; diagonal, fan
        int t = TB.e[lane];
        uint4 m = and4(ws.miss[t & 15], ws.miss[t >> 4]);
        he = (hits_of(and4(m, shr4(m, 1))) & TA.hm) | ((hits_of(and4(m, shr4(m, STIV_BC + 1))) & qm) << 16);
        hd = hits_of(and4(m, shr4(m, STIV_BC + 2))) & qm;
        if (fm) hd |= (hits_of(and4(shr4(m, fr), pole4(m))) & fm) << 16;
      }
    }
    int cnt = __popc(hv) + __popc(ht) + __popc(he) + __popc(hd), off = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) { int v = __shfl_up_sync(0xffffffffu, off, o); if (lane >= o) off += v; }
    const int total = __shfl_sync(0xffffffffu, off, 31);
    off -= cnt;
    if (lane == 0) nprim += total;
    const float e = 2.0f * frame.w + 4.0f * U32 * dmax + 2e-12f;   // error of a difference component
    for (int base = 0; base < total; base += QCAP) {
      // entries [base, base + QCAP) of the concatenated hits into the queue
      {
        int pos = off - base;
        const PatchTopo& TB = *B.tp;
        const int fr = A.tp->frow;
        auto put = [&](unsigned x) { if (pos >= 0 && pos < QCAP) ws.q[pos] = x; ++pos; };
        unsigned own = NSLOT + (hv ? TB.v[lane] : 0u);
        for (unsigned m = hv; m; m &= m - 1) {
          unsigned b = __ffs(m) - 1, s0, s1, s2;
          if (b >= 16) { s0 = b - 16; s1 = s0 + STIV_BC + 2; s2 = s0 + 1; }
          else if (b < 10) { s0 = b; s1 = s0 + STIV_BC + 1; s2 = s1 + 1; }
          else { s0 = PSLOT; s1 = fr + b - 10 + (fr ? 1 : 0); s2 = fr + b - 10 + (fr ? 0 : 1); }
          put(own | (s0 << 5) | (s1 << 10) | (s2 << 15) | (1u << 20));
        }
        unsigned t = ht ? TB.t[lane] : 0u;
        unsigned tri = ((NSLOT + (t & 15u)) << 5) | ((NSLOT + ((t >> 4) & 15u)) << 10) | ((NSLOT + (t >> 8)) << 15);
        for (unsigned m = ht; m; m &= m - 1) put((__ffs(m) - 1) | tri);
        unsigned ed = he | hd ? TB.e[lane] : 0u;
        ed = ((NSLOT + (ed & 15u)) << 5) | ((NSLOT + (ed >> 4)) << 15) | (2u << 20);
        for (unsigned m = he; m; m &= m - 1) {
          unsigned b = __ffs(m) - 1, s0 = b & 15;
          put(ed | s0 | ((s0 + (b < 16 ? 1 : STIV_BC + 1)) << 10));
        }
        for (unsigned m = hd; m; m &= m - 1) {
          unsigned b = __ffs(m) - 1, s0 = b < 16 ? b : fr + b - 16;
          put(ed | s0 | ((b < 16 ? s0 + STIV_BC + 2 : PSLOT) << 10));
        }
      }
      __syncwarp();
      // stages 2 and 3a: p, q, h, g the slots of blossom_fp32's points (VF: the
      // vertex and the triangle; EE: first points of the two edges, then second)
      const int n = min(total - base, QCAP);
      int kept = 0;
      for (int b0 = 0; b0 < n; b0 += 32) {
        bool keep = b0 + lane < n;
        unsigned en = 0;
        if (keep) {
          en = ws.q[b0 + lane];
          const int p = en & 31, q = (en >> 5) & 31, h = (en >> 10) & 31, g = (en >> 15) & 31;
          const bool ee = (en >> 20) == 2;
          if (unsure) {
            int sl[4] = {p, ee ? h : q, ee ? q : h, g};
            keep = box_hit<MIXED, DM>(ws, a, r, ee ? 2 : 1, sl, gap);
            if (!keep) --nprim;
          }
          if (keep && !a.exact_only) {
            float4 xp = ws.x[p], xq = ws.x[q], xh = ws.x[h], xg = ws.x[g];
            float4 dp = ws.d[p], dq = ws.d[q], dh = ws.d[h], dg = ws.d[g];
            blossom bl = blossom_fp32(ee, {xp.x, xp.y, xp.z}, {xq.x, xq.y, xq.z}, {xh.x, xh.y, xh.z},
                                      {xg.x, xg.y, xg.z}, {dp.x, dp.y, dp.z}, {dq.x, dq.y, dq.z}, {dh.x, dh.y, dh.z},
                                      {dg.x, dg.y, dg.z}, e);
            const int rej = reject_fp32<DM>(ee, bl, e, (float)a.dm);
            keep = rej == 0;
            nleft += rej != 1;
          }
        }
        unsigned m = __ballot_sync(0xffffffffu, keep);
        if (keep) ws.q[kept + __popc(m & lower)] = en;   // below b0 + 32: read by every lane above
        kept += __popc(m);
        __syncwarp();
      }
      // descriptors of the kept pairs: vertex ids in the order the contact test
      // takes its points (EE edge indices are formed by the FP64 stage, for
      // contacts only)
      if (kept) {
        ulonglong2* list = a.exact_only ? a.q2 : a.q3;
        int64_t cap = a.exact_only ? a.Q2 : a.Q3;
        unsigned long long k0 = 0;
        if (lane == 0) k0 = atomicAdd((unsigned long long*)&a.ctr[a.exact_only ? 15 : 14], (unsigned long long)kept);
        k0 = __shfl_sync(0xffffffffu, k0, 0);
        for (int k = lane; k < kept; k += 32) {
          unsigned en = ws.q[k];
          const int p = en & 31, q = (en >> 5) & 31, h = (en >> 10) & 31, g = (en >> 15) & 31, kind = en >> 20;
          unsigned long long v0 = (unsigned)__float_as_int(ws.x[p].w), v1 = (unsigned)__float_as_int(ws.x[q].w),
                             v2 = (unsigned)__float_as_int(ws.x[h].w), v3 = (unsigned)__float_as_int(ws.x[g].w);
          ulonglong2 d;
          if (kind == 2) {
            unsigned long long a0 = v0 < v2 ? v0 : v2, a1 = v0 < v2 ? v2 : v0, b0 = v1 < v3 ? v1 : v3,
                               b1 = v1 < v3 ? v3 : v1;
            d.x = make_desc(r, 2, 0, 0);
            d.y = a0 | (a1 << 16) | (b0 << 32) | (b1 << 48);
          } else {
            const int t = kind == 0 ? NSLOT : 0;
            d.x = make_desc(r, kind, (int)v0, tri_gid(kind == 0 ? B : A, q - t, h - t, g - t));
            d.y = v0 | (v1 << 16) | (v2 << 32) | (v3 << 48);
          }
          if ((int64_t)(k0 + k) < cap) list[k0 + k] = d;
          else atomicOr((unsigned long long*)&a.ctr[STIV_C_STATUS], STIV_F_WORK_OVERFLOW);
        }
      }
      __syncwarp();
    }
    item = __shfl_sync(0xffffffffu, next, 0);
  }
  for (int off = 16; off > 0; off >>= 1) {
    nprim += __shfl_down_sync(0xffffffffu, nprim, off);
    nleft += __shfl_down_sync(0xffffffffu, nleft, off);
  }
  if (lane == 0 && nprim) atomicAdd((unsigned long long*)&a.ctr[STIV_C_PRIM], (unsigned long long)nprim);
  if (lane == 0 && nleft) atomicAdd((unsigned long long*)&a.ctr[17], (unsigned long long)nleft);
}

// ---------------------------------------------------------------------------
// stage 3b, d_m = 0: one lane per descriptor.  Five directions of the separation
// test drop two thirds of the descriptors; the rest collect in the warp's queue
// and take the root test on full warps: where the cubic is certainly monotone on
// [0, 1] it has at most one root, near the FP32 root r.  Every time at which the
// FP64 test can find one has |f| <= E in FP32, so it lies within
// (E + |f(r)|) / min|f'| of r, and the inside certificate on that short interval
// decides nearly every pair.  Cubics that may have a critical point go to the
// FP64 test on a list of their own, so that its warps do the same work.
//
// Bound by instruction issue.  Against 16 pieces of [0, 1], each with its own
// sign and inside certificate and refined twice (0.49 ms at 1440 vesicles on the
// same 4.7M descriptors, 2.0 ms at 4096 on 22.5M), the interval is some 200
// times shorter than a piece: this kernel takes 0.19 and 0.78 ms, and the pairs
// left for the FP64 test fall from 1.05M to 734k (635k of them contacts).
// ---------------------------------------------------------------------------
constexpr int RW = 8;          // warps per CTA
constexpr int NSEP = 5;        // directions of the separation test

// 1: the FP64 contact test certainly finds no contact and nothing degenerate; 2:
// the cubic may have a critical point (not decided here).
__device__ __forceinline__ int root_reject(int kind, const f3* x, const f3* d, float ep, float es) {
  cubic32 q = cubic_fp32(kind, x, d, ep, es);
  if (fabsf(q.k0) <= q.E && fabsf(q.k1) <= q.E && fabsf(q.k2) <= q.E && fabsf(q.k3) <= q.E) return 0;
  // f' in the Bernstein basis, three times the differences of the coefficients of f: error 6 E
  float d0 = q.k1, d1 = q.k1 + q.k2, d2 = (q.k1 + 2.f * q.k2) + 3.f * q.k3;
  float dmin = fmaxf(fminf(d0, fminf(d1, d2)), -fmaxf(d0, fmaxf(d1, d2))) - 6.5f * q.E;
  if (!(dmin > 0.f)) return 2;
  float f0 = q.k0, f1 = ((q.k3 + q.k2) + q.k1) + q.k0;
  if (fminf(f0, f1) > q.E || fmaxf(f0, f1) < -q.E) return 1;   // no root
  float r = __fdividef(f0, f0 - f1), v = 0.f;
#pragma unroll 1
  for (int it = 0; it < 3; ++it) {
    r = fminf(fmaxf(r, 0.f), 1.f);
    v = fmaf(fmaf(fmaf(q.k3, r, q.k2), r, q.k1), r, q.k0);
    if (it < 2) r = r - __fdividef(v, fmaf(fmaf(3.f * q.k3, r, 2.f * q.k2), r, q.k1));
  }
  float S = fabsf(q.k0) + fabsf(q.k1) + fabsf(q.k2) + fabsf(q.k3);
  float del = __fdividef(1.01f * (q.E + fabsf(v) + 8.f * U32 * S), dmin) + 1e-6f;
  float t0 = fmaxf(r - del, 0.f), t1 = fminf(r + del, 1.f);
  return inside_cert(kind, x, d, t0, t1 - t0, ep, q.ed, es) == 1;
}

__global__ void __launch_bounds__(RW * 32, 4) roots_kernel(narrow_args a) {
  __shared__ ulonglong2 queue[RW][64];
  ulonglong2* q = queue[threadIdx.x >> 5];
  const int lane = threadIdx.x & 31;
  const unsigned lower = (1u << lane) - 1u;
  int64_t n3 = a.ctr[14];
  if (n3 > a.Q3) n3 = a.Q3;
  int64_t nb = (n3 + 31) / 32;
  int64_t gw = (int64_t)blockIdx.x * RW + (threadIdx.x >> 5), nw = (int64_t)gridDim.x * RW;
  int nq = 0;
  auto roots = [&](int n) {
    int res = 1;
    ulonglong2 e = make_ulonglong2(0ull, 0ull);
    if (lane < n) {
      e = q[lane];
      int kind;
      f3 xq[4], dq[4];
      float ep, es;
      desc_points_f32(a, e, kind, xq, dq, ep, es);
      res = root_reject(kind, xq, dq, ep, es);
    }
    push_global(a.q2, a.Q2, &a.ctr[15], &a.ctr[STIV_C_STATUS], res == 0, e, lane);
    push_global(a.q2c, a.Q2, &a.ctr[16], &a.ctr[STIV_C_STATUS], res == 2, e, lane);
  };
  for (int64_t b = gw; b < nb; b += nw) {
    int64_t idx = b * 32 + lane;
    bool keep = idx < n3;
    ulonglong2 e = keep ? a.q3[idx] : make_ulonglong2(0ull, 0ull);
    if (keep) {
      int kind;
      f3 xq[4], dq[4];
      float ep, es;
      desc_points_f32(a, e, kind, xq, dq, ep, es);
      float dmx = fmaxf(fmaxf(amax3(dq[0]), amax3(dq[1])), fmaxf(amax3(dq[2]), amax3(dq[3])));
      float ed = 2.0f * ep + 4.0f * U32 * dmx + 2e-12f;
      const bool ee = kind != 0;
      blossom bl = blossom_fp32(ee, xq[0], ee ? xq[2] : xq[1], ee ? xq[1] : xq[2], xq[3], dq[0], ee ? dq[2] : dq[1],
                                ee ? dq[1] : dq[2], dq[3], ed);
      keep = !separation_reject<false, NSEP>(ee, bl, ed, 0.f);
    }
    unsigned m = __ballot_sync(0xffffffffu, keep);
    if (keep) q[nq + __popc(m & lower)] = e;
    nq += __popc(m);
    __syncwarp();
    if (nq >= 32) {
      roots(32);
      ulonglong2 rest = lane + 32 < nq ? q[lane + 32] : make_ulonglong2(0ull, 0ull);
      __syncwarp();
      if (lane + 32 < nq) q[lane] = rest;
      nq -= 32;
      __syncwarp();
    }
  }
  if (nq > 0) roots(nq);
}

// ---------------------------------------------------------------------------
// stage 3b, d_m > 0: the pieces of [0,1] where the point may be in the d_m band,
// certified non-contact.
// A warp takes 32 descriptors; the pieces that need the inside test become
// (descriptor, piece) tasks spread over the lanes, so that every lane runs the
// same test; an undecided piece is split in two, level by level (NLEVEL
// levels), and a half whose cubic certainly keeps one sign is dropped.
// ---------------------------------------------------------------------------
constexpr int PW = 8;          // warps per CTA
constexpr int NPIECE = 16;     // level-0 pieces of [0, 1]
constexpr int NLEVEL = 6;      // most refinement levels (finest piece: 1 / (16 * 32))
constexpr int MAXTASK = 512;
static_assert(NPIECE << (NLEVEL - 1) <= 1024, "piece index fits 10 bits");

struct PieceWarp {
  float x[32][4][3], d[32][4][3];
  float k[32][4], E[32], ep[32], ed[32], es[32];
  float rhs[32];   // band_rhs of each pair
  int kind[32], fail[32];
  unsigned short task[MAXTASK], task2[MAXTASK];
  int ntask2;
};

// A piece is kept when the point may be within d_m of the plane there
// (out_of_band fails); the inside certificate is the cubic's, because the
// degree-six test uses the same inside test at its candidate times.
__global__ void __launch_bounds__(PW * 32, 4) pieces_kernel(narrow_args a) {
  extern __shared__ unsigned char psraw[];
  PieceWarp& W = ((PieceWarp*)psraw)[threadIdx.x >> 5];
  int lane = threadIdx.x & 31;
  int64_t n3 = a.ctr[14];
  if (n3 > a.Q3) n3 = a.Q3;
  int64_t nb = (n3 + 31) / 32;
  int64_t gw = (int64_t)blockIdx.x * PW + (threadIdx.x >> 5), nw = (int64_t)gridDim.x * PW;
  for (int64_t b = gw; b < nb; b += nw) {
    int64_t idx = b * 32 + lane;
    bool valid = idx < n3;
    ulonglong2 e = valid ? a.q3[idx] : make_ulonglong2(0ull, 0ull);
    unsigned mask = 0;
    W.fail[lane] = 0;
    if (valid) {
      int kind;
      f3 xq[4], dq[4];
      float ep, es;
      desc_points_f32(a, e, kind, xq, dq, ep, es);
      bool apart;
      {
        float dmx = fmaxf(fmaxf(amax3(dq[0]), amax3(dq[1])), fmaxf(amax3(dq[2]), amax3(dq[3])));
        float ed = 2.0f * ep + 4.0f * U32 * dmx + 2e-12f;
        const bool ee = kind != 0;
        blossom bl = blossom_fp32(ee, xq[0], ee ? xq[2] : xq[1], ee ? xq[1] : xq[2], xq[3], dq[0], ee ? dq[2] : dq[1],
                                  ee ? dq[1] : dq[2], dq[3], ed);
        apart = separation_reject<true, NSEP>(ee, bl, ed, (float)a.dm);
      }
      cubic32 q = cubic_fp32<true>(kind, xq, dq, ep, es);
      for (int p = 0; p < 4; ++p) {
        W.x[lane][p][0] = xq[p].x; W.x[lane][p][1] = xq[p].y; W.x[lane][p][2] = xq[p].z;
        W.d[lane][p][0] = dq[p].x; W.d[lane][p][1] = dq[p].y; W.d[lane][p][2] = dq[p].z;
      }
      W.k[lane][0] = q.k0; W.k[lane][1] = q.k1; W.k[lane][2] = q.k2; W.k[lane][3] = q.k3;
      W.E[lane] = q.E; W.ep[lane] = ep; W.ed[lane] = q.ed; W.es[lane] = es; W.kind[lane] = kind;
      W.rhs[lane] = band_rhs(q, ep, (float)a.dm);
      if (fabsf(q.k0) <= q.E && fabsf(q.k1) <= q.E && fabsf(q.k2) <= q.E && fabsf(q.k3) <= q.E) {
        W.fail[lane] = 1;   // may vanish identically: FP64 decides (degenerate)
      } else if (!apart) {
        const float w = 1.0f / NPIECE;
#pragma unroll 2
        for (int p = 0; p < NPIECE; ++p) {
          float t0 = p * w;
          float f0 = fmaf(fmaf(fmaf(q.k3, t0, q.k2), t0, q.k1), t0, q.k0);
          float fp1 = fmaf(fmaf(3.f * q.k3, t0, 2.f * q.k2), t0, q.k1);
          float g1 = w * fp1, g2 = w * w * fmaf(3.f * q.k3, t0, q.k2), g3 = w * w * w * q.k3;
          float c1 = f0 + g1 * (1.f / 3.f), c2 = f0 + (2.f * g1 + g2) * (1.f / 3.f), c3 = f0 + g1 + g2 + g3;
          bool keep_p = !out_of_band(f0, c1, c2, c3, q.E, W.rhs[lane]);
          if (keep_p) mask |= 1u << p;
        }
      }
    }
    // task list of this batch: (owner lane, piece) of level 0
    int cnt = __popc(mask), off = cnt;
    for (int o = 1; o < 32; o <<= 1) { int v = __shfl_up_sync(0xffffffffu, off, o); if (lane >= o) off += v; }
    int total = __shfl_sync(0xffffffffu, off, 31);
    off -= cnt;
    for (unsigned m = mask; m; m &= m - 1) {
      int p = __ffs(m) - 1;
      if (off < MAXTASK) W.task[off] = (unsigned short)((lane << 10) | p);
      else W.fail[lane] = 1;
      ++off;
    }
    if (total > MAXTASK) total = MAXTASK;
    // adaptive refinement: a piece that may hold a root and whose inside test
    // is undecided splits in two, down to NLEVEL levels; a half that
    // certainly holds no root is dropped
    unsigned short* cur = W.task;
    unsigned short* nxt = W.task2;
#pragma unroll 1
    for (int level = 0; level < a.nlevel && total > 0; ++level) {
      if (lane == 0) W.ntask2 = 0;
      __syncwarp();
      const float w = (1.0f / NPIECE) * __int_as_float((127 - level) << 23);   // 2^-level / NPIECE
#pragma unroll 1
      for (int t0 = 0; t0 < total; t0 += 32) {
        int t = t0 + lane;
        // a descriptor already bound for the FP64 test needs none of its
        // other pieces decided
        if (t < total && !W.fail[cur[t] >> 10]) {
          int owner = cur[t] >> 10, idx = cur[t] & 1023;
          float tl = idx * w;
          bool may_root = true;
          if (level > 0) {
            float k0 = W.k[owner][0], k1 = W.k[owner][1], k2 = W.k[owner][2], k3 = W.k[owner][3], E = W.E[owner];
            float f0 = fmaf(fmaf(fmaf(k3, tl, k2), tl, k1), tl, k0);
            float fp1 = fmaf(fmaf(3.f * k3, tl, 2.f * k2), tl, k1);
            float g1 = w * fp1, g2 = w * w * fmaf(3.f * k3, tl, k2), g3 = w * w * w * k3;
            float c1 = f0 + g1 * (1.f / 3.f), c2 = f0 + (2.f * g1 + g2) * (1.f / 3.f), c3 = f0 + g1 + g2 + g3;
            may_root = !out_of_band(f0, c1, c2, c3, E, W.rhs[owner]);
          }
          if (may_root) {
            f3 xq[4], dq[4];
            for (int q = 0; q < 4; ++q) {
              xq[q] = {W.x[owner][q][0], W.x[owner][q][1], W.x[owner][q][2]};
              dq[q] = {W.d[owner][q][0], W.d[owner][q][1], W.d[owner][q][2]};
            }
            int res = inside_cert(W.kind[owner], xq, dq, tl, w, W.ep[owner], W.ed[owner], W.es[owner]);
            if (res == 2) {
              W.fail[owner] = 1;                       // a contact: the FP64 test decides its time
            } else if (res == 0) {
              if (level + 1 == a.nlevel) {
                W.fail[owner] = 1;
              } else {
                int k = atomicAdd(&W.ntask2, 2);
                if (k + 1 < MAXTASK) {
                  nxt[k] = (unsigned short)((owner << 10) | (2 * idx));
                  nxt[k + 1] = (unsigned short)((owner << 10) | (2 * idx + 1));
                } else {
                  W.fail[owner] = 1;
                }
              }
            }
          }
        }
      }
      __syncwarp();
      total = min(W.ntask2, MAXTASK);
      unsigned short* tmp = cur; cur = nxt; nxt = tmp;
      __syncwarp();
    }
    __syncwarp();
    push_global(a.q2, a.Q2, &a.ctr[15], &a.ctr[STIV_C_STATUS], valid && W.fail[lane], e, lane);
    __syncwarp();
  }
}

// ---------------------------------------------------------------------------
// stage 4: the FP64 contact test, one descriptor per thread.  Bound by the FP64
// pipe (0.72 busy; about 295 FP64 instructions per warp of pairs, 421 before the
// halvings were taken at once, both kinds shared their instructions and the cubics
// with critical points had warps of their own).  At 1440 vesicles 0.92 -> 0.73 ms
// by the instructions on the same 1.05M pairs, 0.43 ms on the pairs that the root
// test leaves.  The register
// budget is capped (6 blocks of 128 threads per SM, 80 registers, for the
// cubic; 8 blocks, 64 registers, for d_m > 0): the dependent FP64 operations
// need the warps more than the spilled registers cost.
// ---------------------------------------------------------------------------
template <bool MIXED, bool DM>
__global__ void __launch_bounds__(128, DM ? 8 : 6) fp64_kernel(narrow_args a) {
  int lane = threadIdx.x & 31;
  // the two lists one after the other, the second from the next whole warp on
  int64_t n2 = a.ctr[15], n2c = a.ctr[16];
  if (n2 > a.Q2) n2 = a.Q2;
  if (n2c > a.Q2) n2c = a.Q2;
  const int64_t second = (n2 + 31) & ~(int64_t)31, n_all = second + n2c;
  long long ndeg = 0, flops = 0, nexact = 0;
  int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t base = (int64_t)blockIdx.x * blockDim.x; base < n_all; base += stride) {
    int64_t idx = base + threadIdx.x;
    int type = -1, ga = 0, gb = 0, r = 0;
    double tau = 0.0, w1 = 0.0, w2 = 0.0;
    if (idx < n2 || (idx >= second && idx < n_all)) {
      ++nexact;
      int vid[4];
      bool onj[4];
      int ty;
      const ulonglong2 e = idx < n2 ? a.q2[idx] : a.q2c[idx - second];
      desc_points(e, r, ty, ga, gb, vid, onj);
      const stiv_pair_info* pi = a.pinfo + r;
      int code = pi->code, Pij = pi->Pij;
      long long voi = pi->voff_i, voj = pi->voff_j;
      int sB[3] = {code / 9 - 1, (code / 3) % 3 - 1, code % 3 - 1};
      int nvi = stiv_nverts(Pij & 0xFFFF), nvj = stiv_nverts(Pij >> 16);
      d3 X0[4], D[4];   // EE: p0, q0, p1, q1
      for (int k = 0; k < 4; ++k) {
        const int q = ty == 2 ? ((k & 1) << 1) | (k >> 1) : k;
        const bool oj = q == 0 ? onj[0] : q == 1 ? onj[1] : onj[2];
        const int vq = (int)((e.y >> (16 * q)) & 0xFFFF);
        int nv = oj ? nvj : nvi;
        size_t vb = (size_t)(oj ? voj : voi) + vq;
        double p0[3], p1[3];
        for (int c = 0; c < 3; ++c) {
          size_t i0 = vb + (size_t)c * nv, i1 = vb + (size_t)(3 + c) * nv;
          p0[c] = vtx<MIXED>(a.X, i0);
          p1[c] = vtx<MIXED>(a.X, i1);
          if (oj && sB[c] != 0) { double sh = sB[c] * a.L[c]; p0[c] = p0[c] + sh; p1[c] = p1[c] + sh; }
        }
        X0[k] = {p0[0], p0[1], p0[2]};
        D[k] = {__dsub_rn(p1[0], p0[0]), __dsub_rn(p1[1], p0[1]), __dsub_rn(p1[2], p0[2])};
      }
      flops += 12;  // displacements
      int st = DM ? ccd64_dm(ty == 2 ? KIND_EE : KIND_VF, X0, D, a.dm, tau, w1, w2, flops)
                  : ccd64(ty == 2 ? KIND_EE : KIND_VF, X0, D, tau, w1, w2, flops);
      if (st == 1) {
        type = ty;
        if (ty == 2) {   // edge indices of the two edges (their vertex ids are ordered)
          ga = stiv_edge_index(Pij & 0xFFFF, vid[0], vid[1]);
          gb = stiv_edge_index(Pij >> 16, vid[2], vid[3]);
        }
      }
      else if (st == 2) ++ndeg;
    }
    unsigned m = __ballot_sync(0xffffffffu, type >= 0);
    if (m) {
      unsigned long long cb = 0;
      int leader = __ffs(m) - 1;
      if (lane == leader) cb = atomicAdd((unsigned long long*)&a.ctr[11], (unsigned long long)__popc(m));
      cb = __shfl_sync(0xffffffffu, cb, leader);
      if (type >= 0) {
        int64_t k = (int64_t)cb + __popc(m & ((1u << lane) - 1u));
        if (k < a.C) {
          a.rc_pair[k] = r; a.rc_type[k] = type; a.rc_a[k] = ga; a.rc_b[k] = gb;
          a.rc_tau[k] = tau; a.rc_w[2 * k] = w1; a.rc_w[2 * k + 1] = w2;
        }
      }
      // contacts per pair (for their ordering): one addition per warp while its
      // contacts belong to one pair
      const int rl = __shfl_sync(0xffffffffu, r, leader);
      if ((int64_t)cb + __popc(m) <= a.C && __all_sync(0xffffffffu, type < 0 || r == rl)) {
        if (lane == leader) atomicAdd(&a.pair_cnt[rl], __popc(m));
      } else if (type >= 0 && (int64_t)cb + __popc(m & ((1u << lane) - 1u)) < a.C) {   // those stored
        atomicAdd(&a.pair_cnt[r], 1);
      }
      unsigned mee = __ballot_sync(0xffffffffu, type == 2);
      if (lane == leader) {
        if (mee) atomicAdd((unsigned long long*)&a.ctr[STIV_C_EE], (unsigned long long)__popc(mee));
        if (m & ~mee) atomicAdd((unsigned long long*)&a.ctr[STIV_C_VF], (unsigned long long)__popc(m & ~mee));
      }
    }
  }
  for (int off = 16; off > 0; off >>= 1) {
    ndeg += __shfl_down_sync(0xffffffffu, ndeg, off);
    flops += __shfl_down_sync(0xffffffffu, flops, off);
    nexact += __shfl_down_sync(0xffffffffu, nexact, off);
  }
  if (lane == 0) {
    if (ndeg) atomicAdd((unsigned long long*)&a.ctr[STIV_C_DEGEN], (unsigned long long)ndeg);
    if (flops) atomicAdd((unsigned long long*)&a.ctr[12], (unsigned long long)flops);
    if (nexact) atomicAdd((unsigned long long*)&a.ctr[13], (unsigned long long)nexact);
  }
}

// Level 1: the patch pairs of one candidate vesicle pair per CTA.  A's patches
// are kept that meet vesicle j's box, then B's that meet the union of A's
// kept patches, then A's that meet the union of B's; a pair of kept patches
// is emitted when their boxes overlap and some cell of one meets some cell
// of the other (every primitive lies in one cell of its patch).  Dynamic
// shared memory: two lists of mp boxes with their patch ids.
//
// Bound by latency: with one warp per vesicle pair a few deep pairs held the stage
// (a hundred by a hundred patches, 32 at a time); a CTA's warps share them.  1440
// vesicles 0.25 -> 0.14 ms, 4096 1.15 -> 0.52, 64 at 30% 0.13 -> 0.04.  Small orders,
// whose patches fill less than a CTA, pay for it: 9216 vesicles of order 3 (9
// patches) 0.13 -> 0.37 ms.
constexpr int PPT = 128;   // threads of a CTA

struct patch_list {
  float4* lo;              // box (w: patch id)
  float4* hi;
};

__global__ void __launch_bounds__(PPT) patch_pairs_kernel(const int32_t* pv, const double* vbox, const float* pbox,
                                                          double Lx, double Ly, double Lz, const int32_t* ci,
                                                          const int32_t* cj, const int32_t* cs, int64_t cap,
                                                          int64_t W, uint64_t* work, int64_t* ctr, int mp,
                                                          const float* vorg, const int64_t* voff,
                                                          stiv_pair_info* pinfo, double dm) {
  extern __shared__ float4 psm[];
  __shared__ int nlist[3];         // kept patches of A, of B, of A after the second filter
  __shared__ int ubox[2][6];       // union boxes (order-preserving images)
  const patch_list la = {psm, psm + mp}, lb = {psm + 2 * mp, psm + 3 * mp};
  const int lane = threadIdx.x & 31;
  const unsigned lower = (1u << lane) - 1u;
  int64_t npairs = ctr[STIV_C_PAIRS];
  if (npairs > cap) npairs = cap;
  const double L[3] = {Lx, Ly, Lz};
  // append boxes to a list (in any order) and merge them into a union box
  auto keep_box = [&](const patch_list& l, int* n, int* u, bool hit, float4 lo, float4 hi) {
    const unsigned m = __ballot_sync(0xffffffffu, hit);
    if (!m) return;
    int base = 0;
    const int leader = __ffs(m) - 1;
    if (lane == leader) base = atomicAdd(n, __popc(m));
    base = __shfl_sync(0xffffffffu, base, leader);
    if (hit) {
      const int k = base + __popc(m & lower);
      l.lo[k] = lo;
      l.hi[k] = hi;
    }
    if (!u) return;
    const float v[6] = {lo.x, lo.y, lo.z, hi.x, hi.y, hi.z};
#pragma unroll
    for (int c = 0; c < 6; ++c) {
      const int key = fkey32(hit ? v[c] : (c < 3 ? INFINITY : -INFINITY));
      const int e = c < 3 ? __reduce_min_sync(0xffffffffu, key) : __reduce_max_sync(0xffffffffu, key);
      if (lane == c) { if (c < 3) atomicMin(&u[c], e); else atomicMax(&u[c], e); }
    }
  };
  for (int64_t r = blockIdx.x; r < npairs; r += gridDim.x) {
    const int i = ci[r], j = cj[r], code = cs[r];
    const int s[3] = {code / 9 - 1, (code / 3) % 3 - 1, code % 3 - 1};
    const int Pi = 2 * pv[i], Pj = 2 * pv[j];
    __syncthreads();   // the previous pair's lists are read
    if (threadIdx.x < 3) nlist[threadIdx.x] = 0;
    if (threadIdx.x < 12) ubox[threadIdx.x / 6][threadIdx.x % 6] = fkey32(threadIdx.x % 6 < 3 ? INFINITY : -INFINITY);
    if (threadIdx.x == 0) {
      // FP32 frame of the pair: origin of vesicle i; |FP32 position - exact
      // position| per component is bounded by 2^-22 (R_i + R_j + 2 |offset|)
      // (rounding of X0 - origin, of the offset and of the frame change);
      // 2^-32 of the coordinates themselves is added, so that the bound also
      // stands above the FP64 rounding of positions far from the origin
      float o[3], dmax = 0.f, ymax = 0.f;
      for (int c = 0; c < 3; ++c) {
        double d = ((double)vorg[4 * j + c] + s[c] * L[c]) - (double)vorg[4 * i + c];
        o[c] = (float)d;
        dmax = fmaxf(dmax, fabsf(o[c]));
        ymax = fmaxf(ymax, fmaxf(fabsf(vorg[4 * i + c]), fabsf(vorg[4 * j + c])) + (s[c] ? (float)L[c] : 0.f));
      }
      stiv_pair_info p;
      float R = vorg[4 * i + 3] + vorg[4 * j + 3];
      p.frame = make_float4(o[0], o[1], o[2], 2.3841858e-7f * (R + 2.0f * dmax) + 2.3283064e-10f * (ymax + R));
      p.vi = i; p.vj = j; p.code = code; p.Pij = Pi | (Pj << 16);
      p.voff_i = voff[i]; p.voff_j = voff[j];
      pinfo[r] = p;
    }
    const int ni = stiv_npatches(Pi), nj = stiv_npatches(Pj);
    float shlo[3], shhi[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      double sh = s[c] * L[c];
      // d_m > 0: vesicle j's patch boxes widened by d_m (rounded outward)
      shlo[c] = __double2float_rd(__dsub_rd(sh, dm)); shhi[c] = __double2float_ru(__dadd_ru(sh, dm));
    }
    float bj[6];   // vesicle j's box at its image (A's patches are filtered against it)
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      bj[c] = __fadd_rd(__double2float_rd(vbox[6 * j + c]), shlo[c]);
      bj[3 + c] = __fadd_ru(__double2float_ru(vbox[6 * j + 3 + c]), shhi[c]);
    }
    __syncthreads();
    for (int k0 = 0; k0 < ni; k0 += PPT) {
      const int k = k0 + threadIdx.x;
      float4 lo = make_float4(0.f, 0.f, 0.f, 0.f), hi = lo;
      bool hit = false;
      if (k < ni) {
        const float4* b = (const float4*)(pbox + ((size_t)i * mp + k) * STIV_PBOX);
        float4 b0 = b[0], b1 = b[1];   // lo xyz, hi x; hi yz
        lo = make_float4(b0.x, b0.y, b0.z, __int_as_float(k));
        hi = make_float4(b0.w, b1.x, b1.y, 0.f);
        const float box[6] = {lo.x, lo.y, lo.z, hi.x, hi.y, hi.z};
        hit = fbox_hit(box, bj);
      }
      keep_box(la, &nlist[0], ubox[0], hit, lo, hi);
    }
    __syncthreads();
    float ua[6], ub[6];
    for (int c = 0; c < 6; ++c) ua[c] = fkey_val(ubox[0][c]);
    // B's patches against the union of A's kept patches (a patch of B that
    // meets a kept patch of A meets their union), then A's kept patches
    // against the union of B's
    for (int k0 = 0; k0 < nj; k0 += PPT) {
      const int k = k0 + threadIdx.x;
      float4 lo = make_float4(0.f, 0.f, 0.f, 0.f), hi = lo;
      bool hit = false;
      if (k < nj) {
        const float4* b = (const float4*)(pbox + ((size_t)j * mp + k) * STIV_PBOX);
        float4 b0 = b[0], b1 = b[1];
        lo = make_float4(__fadd_rd(b0.x, shlo[0]), __fadd_rd(b0.y, shlo[1]), __fadd_rd(b0.z, shlo[2]), __int_as_float(k));
        hi = make_float4(__fadd_ru(b0.w, shhi[0]), __fadd_ru(b1.x, shhi[1]), __fadd_ru(b1.y, shhi[2]), 0.f);
        const float box[6] = {lo.x, lo.y, lo.z, hi.x, hi.y, hi.z};
        hit = fbox_hit(box, ua);
      }
      keep_box(lb, &nlist[1], ubox[1], hit, lo, hi);
    }
    __syncthreads();
    const int na0 = nlist[0], nb = nlist[1];
    if (na0 == 0 || nb == 0) continue;
    for (int c = 0; c < 6; ++c) ub[c] = fkey_val(ubox[1][c]);
    // in place: an entry moves to a place no later than its own, in rounds
    for (int q0 = 0; q0 < na0; q0 += PPT) {
      const int q = q0 + threadIdx.x;
      float4 lo = make_float4(0.f, 0.f, 0.f, 0.f), hi = lo;
      bool hit = false;
      if (q < na0) {
        lo = la.lo[q]; hi = la.hi[q];
        const float box[6] = {lo.x, lo.y, lo.z, hi.x, hi.y, hi.z};
        hit = fbox_hit(box, ub);
      }
      __syncthreads();
      keep_box(la, &nlist[2], nullptr, hit, lo, hi);
      __syncthreads();
    }
    const int na = nlist[2];
    for (int e0 = 0; e0 < na * nb; e0 += PPT) {
      const int e = e0 + threadIdx.x;
      bool hit = false;
      int pa = 0, pb = 0;
      if (e < na * nb) {
        const int qa = e / nb, qb = e - qa * nb;
        const float4 al = la.lo[qa], ah = la.hi[qa], bl = lb.lo[qb], bh = lb.hi[qb];
        pa = __float_as_int(al.w); pb = __float_as_int(bl.w);
        hit = al.x <= bh.x && bl.x <= ah.x && al.y <= bh.y && bl.y <= ah.y && al.z <= bh.z && bl.z <= ah.z;
        if (hit) {
          // every primitive lies in one of its patch's four cells: some cell
          // of pa must meet some cell of pb (vesicle j's at its image,
          // widened by d_m, rounded outward as the patch boxes)
          const float4* ca = (const float4*)(pbox + ((size_t)i * mp + pa) * STIV_PBOX + STIV_PBOX_CELLS);
          const float4* cb = (const float4*)(pbox + ((size_t)j * mp + pb) * STIV_PBOX + STIV_PBOX_CELLS);
          float bB[4][6];
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            float4 l = cb[2 * q], u = cb[2 * q + 1];
            bB[q][0] = __fadd_rd(l.x, shlo[0]); bB[q][1] = __fadd_rd(l.y, shlo[1]); bB[q][2] = __fadd_rd(l.z, shlo[2]);
            bB[q][3] = __fadd_ru(u.x, shhi[0]); bB[q][4] = __fadd_ru(u.y, shhi[1]); bB[q][5] = __fadd_ru(u.z, shhi[2]);
          }
          bool any = false;
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            float4 l = ca[2 * q], u = ca[2 * q + 1];
            float bA[6] = {l.x, l.y, l.z, u.x, u.y, u.z};
#pragma unroll
            for (int w = 0; w < 4; ++w) any = any || fbox_hit(bA, bB[w]);
          }
          hit = any;
        }
      }
      const unsigned m = __ballot_sync(0xffffffffu, hit);
      // at P = 2 a patch touches both poles: a further item per such patch for
      // its south-pole primitives
      const int sa = Pi == 2 ? 2 : 1, sb = Pj == 2 ? 2 : 1;
      if (m) {
        unsigned long long base = 0;
        const int nm = __popc(m);
        if (lane == 0) {
          base = atomicAdd((unsigned long long*)&ctr[STIV_C_PATCH], (unsigned long long)(nm * sa * sb));
          // the further items, which the reported count leaves out
          if (sa * sb > 1) atomicAdd((unsigned long long*)&ctr[18], (unsigned long long)(nm * (sa * sb - 1)));
        }
        base = __shfl_sync(0xffffffffu, base, 0);
        if (hit)
          for (int z = 0; z < sa * sb; ++z) {
            int64_t k = (int64_t)base + z * nm + __popc(m & lower);
            int qa = pa | (z % sa ? SOUTH : 0), qb = pb | (z / sa ? SOUTH : 0);
            if (k < W) work[k] = ((uint64_t)r << 32) | ((uint64_t)qa << 16) | (uint64_t)qb;
            else atomicOr((unsigned long long*)&ctr[STIV_C_STATUS], STIV_F_WORK_OVERFLOW);
          }
      }
    }
  }
}

}  // namespace

size_t stiv_narrow_smem() { return sizeof(WarpSm) * NW; }

int stiv_narrow_phase(stiv_handle* h, cudaStream_t st, const int32_t* p_dev, const int64_t* voff, const void* X,
                      const stiv_pairs* cand, detect_ws& w, int num_sms, int p_max) {
  const double* L = h->prm.box_L;
  // CTAs per SM: enough to hide the phases of one pair behind those of others
  int blocks = (int)cand->capacity;
  int pp_mult = h->tune[STIV_TUNE_PATCH_BLOCKS] > 0 ? h->tune[STIV_TUNE_PATCH_BLOCKS] : STIV_PATCH_BLOCKS;
  if (cand->capacity > (int64_t)pp_mult * num_sms) blocks = pp_mult * num_sms;
  if (blocks < 1) blocks = 1;
  int mp = stiv_npatches(2 * p_max);
  size_t psmem = (size_t)4 * mp * sizeof(float4);
  STIV_SMEM(h, patch_pairs_kernel, psmem, 1024, 4 * stiv_npatches(STIV_MAX_PP) * sizeof(float4));
  {
    STIV_PROF(h, st, "patch_pairs");
    patch_pairs_kernel<<<blocks, PPT, psmem, st>>>(p_dev, w.vbox, w.pbox, L[0], L[1], L[2], cand->i, cand->j,
                                                   cand->shift, cand->capacity, w.W, w.work, w.ctr, mp, w.vorg,
                                                   voff, w.pinfo, h->prm.d_m);
  }
  STIV_LAUNCH(h);
  narrow_args a;
  bool mixed = h->prm.precision == STIV_MIXED;
  a.X = X; a.mixed = mixed;
  a.pinfo = w.pinfo;
  a.L[0] = L[0]; a.L[1] = L[1]; a.L[2] = L[2];
  a.work = w.work; a.W = w.W; a.include_ee = h->prm.include_ee; a.exact_only = w.exact_only;
  a.dm = h->prm.d_m;
  // five levels by default: at 360 vesicles (p = 15, d_m > 0) pieces and FP64 test
  // take 1.19 ms at 2 levels, 1.06 at 4, 1.04 at 5
  a.nlevel = h->tune[STIV_TUNE_PIECE_LEVELS] > 0 ? h->tune[STIV_TUNE_PIECE_LEVELS] : STIV_PIECE_LEVELS;
  if (a.nlevel > NLEVEL) a.nlevel = NLEVEL;
  if (a.nlevel < 1) a.nlevel = 1;
  a.vorg = w.vorg; a.fprep = w.fprep; a.fstride = w.fstride;
  a.q3 = w.q3; a.q2 = w.q2; a.q2c = w.q2c; a.Q3 = w.Q3; a.Q2 = w.Q2;
  a.C = w.C;
  a.rc_pair = w.tmp_i32; a.rc_type = w.tmp_i32 + w.C; a.rc_a = w.tmp_i32 + 2 * w.C; a.rc_b = w.tmp_i32 + 3 * w.C;
  a.rc_tau = w.tmp_f64; a.rc_w = w.tmp_f64 + w.C;
  a.pair_cnt = w.pair_cnt;
  a.ctr = w.ctr;
  // d_m > 0: widened boxes and the degree-six test, in kernels of their own
  bool dmk = h->prm.d_m > 0.0;
  size_t smem = stiv_narrow_smem();
  auto nk = mixed ? (dmk ? narrow_kernel<true, true> : narrow_kernel<true, false>)
                  : (dmk ? narrow_kernel<false, true> : narrow_kernel<false, false>);
  STIV_CUDA(h, cudaFuncSetAttribute(nk, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  int per_sm = 0;
  STIV_CUDA(h, cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, nk, NW * 32, smem));
  h->max_ctas[0] = per_sm;
  if (h->tune[STIV_TUNE_NARROW_CTAS] > 0 && h->tune[STIV_TUNE_NARROW_CTAS] < per_sm) per_sm = h->tune[STIV_TUNE_NARROW_CTAS];
  if (per_sm < 1) per_sm = 1;
  {
    STIV_PROF(h, st, "narrow");
    nk<<<per_sm * num_sms, NW * 32, smem, st>>>(a);
  }
  STIV_LAUNCH(h);
  if (!w.exact_only) {
    size_t psm2 = dmk ? sizeof(PieceWarp) * PW : 0;
    auto pk = dmk ? pieces_kernel : roots_kernel;
    static_assert(PW == RW, "one block size for both");
    if (dmk) STIV_CUDA(h, cudaFuncSetAttribute(pk, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)psm2));
    int per_sm2 = 0;
    STIV_CUDA(h, cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm2, pk, PW * 32, psm2));
    h->max_ctas[1] = per_sm2;
    if (h->tune[STIV_TUNE_PIECES_CTAS] > 0 && h->tune[STIV_TUNE_PIECES_CTAS] < per_sm2)
      per_sm2 = h->tune[STIV_TUNE_PIECES_CTAS];
    if (per_sm2 < 1) per_sm2 = 1;
    STIV_PROF(h, st, "pieces");
    pk<<<per_sm2 * num_sms, PW * 32, psm2, st>>>(a);
  }
  STIV_LAUNCH(h);
  {
    STIV_PROF(h, st, "fp64");
    auto fk = mixed ? (dmk ? fp64_kernel<true, true> : fp64_kernel<true, false>)
                    : (dmk ? fp64_kernel<false, true> : fp64_kernel<false, false>);
    int fm = h->tune[STIV_TUNE_FP64_BLOCKS] > 0 ? h->tune[STIV_TUNE_FP64_BLOCKS] : STIV_FP64_BLOCKS;
    fk<<<num_sms * fm, 128, 0, st>>>(a);
  }
  STIV_LAUNCH(h);
  return STIV_OK;
}
