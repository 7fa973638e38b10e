// Sec. 3.1.1-3.1.2: spherical-harmonic synthesis of each vesicle's order-p
// series on its order-2p grid (the "upsampled q^up-grid"), plus the swept
// boxes of vesicles and surface patches.
//
// Synthesis per field (vesicle, time, coordinate):
//   ring sums   G_i(m)  = sum_n a_{n,m} Pbar_n^|m|(x_i)          (Legendre step)
//   longitudes  X(i, j) = sum_m G_i(m) {cos|sin}(|m| phi_j)       (Fourier step)
// Both steps use exact symmetries of the grid: Pbar_n^m(-x) = (-1)^(n+m)
// Pbar_n^m(x) pairs ring i with ring P-i, and phi_{P-j} = pi - phi_j,
// phi_{P+j} = pi + phi_j, phi_{2P-j} = 2 pi - phi_j give four outputs from one
// set of parity-split partial sums.  FP64 throughout (fused multiply-adds).
#include "stiv_internal.cuh"

#include <math.h>

namespace {

// Gauss-Legendre node x_i (descending) of order n by Newton's method on P_n.
__device__ double gl_node(int n, int i) {
  double z = cospi((i + 0.75) / (n + 0.5));
  for (int it = 0; it < 100; ++it) {
    double p0 = 1.0, p1 = z;
    for (int k = 2; k <= n; ++k) {
      double p2 = ((2.0 * k - 1.0) * z * p1 - (k - 1.0) * p0) / k;
      p0 = p1; p1 = p2;
    }
    double dp = n * (z * p1 - p0) / (z * z - 1.0);
    double dz = p1 / dp;
    z -= dz;
    if (fabs(dz) <= 1e-16 * fabs(z) + 1e-300) break;
  }
  return z;
}

// Tables for SH order p (mesh order P = 2p): one thread per table row.
__global__ void tables_kernel(int p, double* leg, double* trig, double* theta, double* leg_t, double* trig_t) {
  int P = 2 * p, nl = (p + 1) * (p + 2) / 2;
  int r = blockIdx.x * blockDim.x + threadIdx.x;
  if (r < P + 3) {
    double x;
    if (r <= P) {
      int ih = r <= P / 2 ? r : P - r;       // compute half the nodes, mirror the rest
      x = (2 * ih == P) ? 0.0 : gl_node(P + 1, ih);
      if (r > P / 2) x = -x;
      theta[r] = acos(x);
    } else {
      x = (r == P + 1) ? 1.0 : -1.0;         // north / south pole
    }
    double s = sqrt((1.0 - x) * (1.0 + x));
    double* L = leg + (size_t)r * nl;
    // normalised associated Legendre functions, no Condon-Shortley phase
    L[0] = 0.28209479177387814347;  // 1/sqrt(4 pi)
    for (int m = 1; m <= p; ++m)
      L[m * (m + 1) / 2 + m] = sqrt((2.0 * m + 1.0) / (2.0 * m)) * s * L[(m - 1) * m / 2 + m - 1];
    for (int m = 0; m < p; ++m)
      L[(m + 1) * (m + 2) / 2 + m] = sqrt(2.0 * m + 3.0) * x * L[m * (m + 1) / 2 + m];
    for (int m = 0; m <= p; ++m)
      for (int n = m + 2; n <= p; ++n) {
        double a = sqrt((4.0 * n * n - 1.0) / ((double)(n - m) * (n + m)));
        double b = sqrt(((double)(n - 1 - m) * (n - 1 + m)) / (4.0 * (n - 1) * (n - 1) - 1.0));
        L[n * (n + 1) / 2 + m] = a * (x * L[(n - 1) * n / 2 + m] - b * L[(n - 2) * (n - 1) / 2 + m]);
      }
    // fold the sqrt(2) of the real harmonics with m > 0 into the table
    for (int n = 1; n <= p; ++n)
      for (int m = 1; m <= n; ++m) L[n * (n + 1) / 2 + m] *= 1.41421356237309504880;
    if (r <= P / 2)
      for (int e = 0; e < nl; ++e) leg_t[(size_t)e * (P / 2 + 1) + r] = L[e];
  }
  // trig[j][0][m] = cos(m phi_j), trig[j][1][m] = sin(m phi_j), phi_j = pi j / P, j <= P/2
  int t = blockIdx.x * blockDim.x + threadIdx.x;
  int nt = (P / 2 + 1) * (p + 1);
  if (t < nt) {
    int j = t / (p + 1), m = t % (p + 1);
    int k = (m * j) % (2 * P);  // exact argument reduction
    double sv, cv;
    sincospi((double)k / P, &sv, &cv);
    trig[(size_t)j * 2 * (p + 1) + m] = cv;
    trig[(size_t)j * 2 * (p + 1) + (p + 1) + m] = sv;
    trig_t[(size_t)(2 * m) * (P / 2 + 1) + j] = cv;
    trig_t[(size_t)(2 * m + 1) * (P / 2 + 1) + j] = sv;
  }
}

struct synth_args {
  const int32_t* p;
  const int64_t* coef_off;
  const double* coef;
  const int64_t* vert_off;
  double* verts;
  const double* leg[STIV_MAX_P + 1];
  const double* leg_t[STIV_MAX_P + 1];
  const double* trig_t[STIV_MAX_P + 1];
};

// One CTA per (vesicle, time level) and NF coordinate fields: 3, or 1 (grid z)
// for few vesicles, where the CTAs would leave the chip idle.
//
// Bound by the FP64 pipe (a warp instruction takes it some 20 cycles), so the
// instructions that run for lanes without work count.  In the Legendre step the
// lanes of a warp are rings of one order m (they run the same number of terms;
// with lanes over m half of them waited), in the Fourier step longitudes, three
// fields at a time on one load of the trigonometric values; both read transposed
// tables, lane by lane.  Every sum keeps its terms and their order.  1440
// vesicles at p = 16: 0.60 -> 0.45 ms.
template <int NF>
__global__ void __launch_bounds__(256) synth_kernel(synth_args a) {
  extern __shared__ double sm[];
  int v = blockIdx.x, t = blockIdx.y, f0 = NF == 1 ? blockIdx.z : 0;
  if (a.p[v] < 1 || a.p[v] > STIV_MAX_P || !a.leg[a.p[v]]) return;   // order outside [1, p_max]: skipped
  int p = a.p[v], P = 2 * p, nc = (p + 1) * (p + 1), nl = (p + 1) * (p + 2) / 2, ns = 2 * p + 1;
  int nv = 2 * P * (P + 1) + 2;
  double* C = sm;                        // [NF][nc]
  double* G = sm + NF * nc;              // [NF][P+1][ns]  slot 0: m=0; 2m-1: cos m; 2m: sin m
  const double* coef = a.coef + a.coef_off[v] + (size_t)(t * 3 + f0) * nc;
  for (int k = threadIdx.x; k < NF * nc; k += blockDim.x) C[k] = coef[k];
  __syncthreads();
  const double* L = a.leg[p];
  const double* LT = a.leg_t[p];
  const double* TT = a.trig_t[p];
  // Legendre step over half the rings (parity pairs ring i with ring P-i)
  const int nh = P / 2 + 1, nq = P / 2 + 1;
  for (int task = threadIdx.x; task < NF * nh * ns; task += blockDim.x) {
    int s = task / (NF * nh), rem = task - s * (NF * nh), f = rem / nh, i = rem - f * nh;
    int m = (s + 1) >> 1;
    int sgn = (s == 0) ? 0 : ((s & 1) ? 1 : -1);  // +m cos, -m sin
    const double* Cf = C + f * nc + sgn * m;
    const double* Li = LT + i;
    double E = 0.0, O = 0.0;
    for (int n = m; n <= p; n += 2) {
      E = fma(Cf[n * n + n], Li[(size_t)(n * (n + 1) / 2 + m) * nh], E);
      if (n + 1 <= p) O = fma(Cf[(n + 1) * (n + 2)], Li[(size_t)((n + 1) * (n + 2) / 2 + m) * nh], O);
    }
    G[(f * (P + 1) + i) * ns + s] = E + O;
    if (i != P - i) G[(f * (P + 1) + (P - i)) * ns + s] = E - O;
  }
  __syncthreads();
  // Fourier step: four longitudes per task and field
  size_t base = a.vert_off[v] + (size_t)(t * 3 + f0) * nv;
  for (int task = threadIdx.x; task < (P + 1) * nq; task += blockDim.x) {
    int r = task / nq, j = task - r * nq;
    const double* g = G + (size_t)r * ns;
    const int fs = (P + 1) * ns;
    double Ce[NF], Co[NF], Se[NF], So[NF];
#pragma unroll
    for (int f = 0; f < NF; ++f) { Ce[f] = g[f * fs]; Co[f] = 0.0; Se[f] = 0.0; So[f] = 0.0; }
    for (int m = 1; m <= p; m += 2) {
      double c = TT[(size_t)(2 * m) * nq + j], sn = TT[(size_t)(2 * m + 1) * nq + j];
#pragma unroll
      for (int f = 0; f < NF; ++f) {
        Co[f] = fma(g[f * fs + 2 * m - 1], c, Co[f]);
        So[f] = fma(g[f * fs + 2 * m], sn, So[f]);
      }
      if (m + 1 <= p) {
        c = TT[(size_t)(2 * m + 2) * nq + j]; sn = TT[(size_t)(2 * m + 3) * nq + j];
#pragma unroll
        for (int f = 0; f < NF; ++f) {
          Ce[f] = fma(g[f * fs + 2 * m + 1], c, Ce[f]);
          Se[f] = fma(g[f * fs + 2 * m + 2], sn, Se[f]);
        }
      }
    }
    int W = 2 * P;
    int j1 = P - j, j2 = P + j, j3 = (W - j) % W;
#pragma unroll
    for (int f = 0; f < NF; ++f) {
      double v0 = (Ce[f] + Co[f]) + (Se[f] + So[f]);            // phi_j
      double v1 = (Ce[f] - Co[f]) + (So[f] - Se[f]);            // pi - phi_j
      double v2 = (Ce[f] - Co[f]) + (Se[f] - So[f]);            // pi + phi_j
      double v3 = (Ce[f] + Co[f]) - (Se[f] + So[f]);            // 2 pi - phi_j
      double* X = a.verts + base + (size_t)f * nv + (size_t)r * W;
      X[j] = v0;
      if (j1 != j) X[j1] = v1;
      if (j2 != j1 && j2 < W) X[j2] = v2;
      if (j3 != j && j3 != j2) X[j3] = v3;
    }
  }
  // poles: only m = 0 contributes
  if (threadIdx.x < 2 * NF) {
    int f = threadIdx.x >> 1, pole = threadIdx.x & 1;
    const double* Lr = L + (size_t)(P + 1 + pole) * nl;
    double acc = 0.0;
    for (int n = 0; n <= p; ++n) acc = fma(C[f * nc + n * n + n], Lr[n * (n + 1) / 2], acc);
    a.verts[base + (size_t)f * nv + 2 * P * (P + 1) + pole] = acc;
  }
}

// ---------------------------------------------------------------------------
// Mesh fidelity (Sec. 3.1.2: the q^up-grid triangle mesh must stay within
// alpha d_m of the smooth surface, ||X^{q^up} - X(phi, theta)||_inf; Fig. 6
// estimates the smooth surface on a 4x upsampled grid).  The mesh is read as
// a map from parameter space: on the grid cell [theta_i, theta_{i+1}] x
// [phi_j, phi_{j+1}], with a, b the cell fractions in theta and phi, the
// triangle [(i,j), (i+1,j), (i+1,j+1)] for a >= b and [(i,j), (i+1,j+1),
// (i,j+1)] for a < b (the Fig. 3 split); above ring 0 and below ring P the
// pole fans.  One CTA per (vesicle, time level) takes the largest distance
// between that map and the order-p series over the order-(factor P) grid
// (its Gauss-Legendre rings, phi_k = pi k / (factor P); poles excluded).
// ---------------------------------------------------------------------------

constexpr double kPi = 3.14159265358979323846;

// What the estimate needs of order p and the factor alone (Pf = factor 2p, rings
// r <= Pf), kept in the handle for all orders up to p_max: where each fine ring
// lies on the mesh, the Legendre values of the rings up to the equator and the
// trigonometric values of the longitudes up to pi / 2, both transposed.
struct fid_ring {
  double al, tp;       // fraction between mesh rings cell and cell + 1; in a pole cap from the pole to the first ring
  int zone, cell, tri; // 0 north cap, 1 between rings, 2 south cap; tri: bit sb set when al >= sb / factor
  int pad;
};
__host__ __device__ inline size_t fid_ring_doubles(int p, int factor) {
  return (size_t)(factor * 2 * p + 1) * (sizeof(fid_ring) / sizeof(double));
}
__host__ __device__ inline size_t fid_leg_doubles(int p, int factor) {
  return (size_t)(factor * p + 1) * ((p + 1) * (p + 2) / 2);
}
__host__ __device__ inline size_t fid_trig_doubles(int p, int factor) { return (size_t)(factor * p + 1) * 2 * (p + 1); }
__host__ __device__ inline size_t fid_doubles(int p, int factor) {
  return fid_ring_doubles(p, factor) + fid_leg_doubles(p, factor) + fid_trig_doubles(p, factor);
}

struct fid_args {
  const int32_t* p;
  const int64_t* coef_off;
  const double* coef;
  const int64_t* vert_off;
  const void* verts;
  int mixed;
  int factor;
  const double* theta[STIV_MAX_P + 1];
  const double* tab;              // tables of order p at tab + off[p]: rings, Legendre, trigonometric
  size_t off[STIV_MAX_P + 1];
  double* err;
};

// Gauss-Legendre node x_i (descending) of order n: Newton's method on P_n from
// Tricomi's start (error O(n^-4)), at most 8 steps, stopping once a step is below
// 4e-16 |x|.  The recurrence's coefficients (2k - 1) / k and (k - 1) / k are
// tabulated (c1, c2), so that a step is two dependent operations, no division.
__device__ double fine_node(int n, int i, const double* c1, const double* c2) {
  double z = (1.0 - (1.0 - 1.0 / n) / (8.0 * n * (double)n)) * cospi((i + 0.75) / (n + 0.5));
  for (int it = 0; it < 8; ++it) {
    double p0 = 1.0, p1 = z;
    for (int k = 2; k <= n; ++k) {
      double p2 = fma(c1[k] * z, p1, -(c2[k] * p0));
      p0 = p1; p1 = p2;
    }
    double dz = p1 / (n * (z * p1 - p0) / (z * z - 1.0));
    z -= dz;
    if (fabs(dz) <= 4e-16 * fabs(z)) break;
  }
  return z;
}

// CTA (r, p - 1): fine ring r <= Pf / 2 of order p and its mirror image: node, place on
// the mesh, Legendre values; and longitude r's trigonometric values.
__global__ void __launch_bounds__(64) fid_tables_kernel(fid_args a, double* tab) {
  __shared__ double c1[2 * STIV_MAX_P * 8 + 2], c2[2 * STIV_MAX_P * 8 + 2];
  __shared__ double node;
  const int p = blockIdx.y + 1, P = 2 * p, Pf = a.factor * P, r = blockIdx.x;
  if (r > Pf / 2) return;
  double* base = tab + a.off[p];
  fid_ring* ring = (fid_ring*)base;
  double* leg = base + fid_ring_doubles(p, a.factor);
  double* trig = leg + fid_leg_doubles(p, a.factor);
  const int nq = Pf / 2 + 1, nl = (p + 1) * (p + 2) / 2;
  for (int k = 2 + threadIdx.x; k <= Pf + 1; k += blockDim.x) { c1[k] = (2.0 * k - 1.0) / k; c2[k] = (k - 1.0) / k; }
  for (int m = threadIdx.x; m <= p; m += blockDim.x) {
    double sv, cv;
    sincospi((double)((m * r) % (2 * Pf)) / Pf, &sv, &cv);   // exact argument reduction
    trig[(size_t)(2 * m) * nq + r] = cv;
    trig[(size_t)(2 * m + 1) * nq + r] = sv;
  }
  __syncthreads();
  if (threadIdx.x == 0) node = 2 * r == Pf ? 0.0 : fine_node(Pf + 1, r, c1, c2);
  __syncthreads();
  const double x = node, s = sqrt((1.0 - x) * (1.0 + x));
  // column m of the normalised associated Legendre functions, no Condon-Shortley
  // phase, sqrt(2) folded in for m > 0, by the recurrences of tables_kernel
  for (int m = threadIdx.x; m <= p; m += blockDim.x) {
    double d = 0.28209479177387814347;  // 1/sqrt(4 pi)
    for (int k = 1; k <= m; ++k) d = sqrt((2.0 * k + 1.0) / (2.0 * k)) * s * d;
    const double r2 = m ? 1.41421356237309504880 : 1.0;
    double* L = leg + (size_t)r * nl;
    L[m * (m + 1) / 2 + m] = d * r2;
    if (m < p) {
      double l2 = d, l1 = sqrt(2.0 * m + 3.0) * x * d;
      L[(m + 1) * (m + 2) / 2 + m] = l1 * r2;
      for (int n = m + 2; n <= p; ++n) {
        double ra = sqrt((4.0 * n * n - 1.0) / ((double)(n - m) * (n + m)));
        double rb = sqrt(((double)(n - 1 - m) * (n - 1 + m)) / (4.0 * (n - 1) * (n - 1) - 1.0));
        double l0 = ra * (x * l1 - rb * l2);
        L[n * (n + 1) / 2 + m] = l0 * r2;
        l2 = l1; l1 = l0;
      }
    }
  }
  // where ring r and its mirror image lie on the mesh
  if (threadIdx.x < 2) {
    const int rr = threadIdx.x ? Pf - r : r;
    const double theta = acos(threadIdx.x ? -x : x);
    const double* thc = a.theta[p];
    fid_ring f;
    f.zone = 1; f.cell = 0; f.al = 0.0; f.tp = 0.0; f.pad = 0;
    if (theta < thc[0]) { f.zone = 0; f.tp = theta / thc[0]; }
    else if (theta > thc[P]) { f.zone = 2; f.tp = (kPi - theta) / (kPi - thc[P]); }
    else {
      int i = 0;
      while (i + 1 < P && thc[i + 1] <= theta) ++i;
      f.cell = i;
      f.al = (theta - thc[i]) / (thc[i + 1] - thc[i]);
    }
    f.tri = 0;
    for (int sb = 0; sb < a.factor; ++sb) f.tri |= (f.al >= (double)sb / a.factor) << sb;
    if (rr != r || threadIdx.x == 0) ring[rr] = f;
  }
}

__device__ __forceinline__ double vert_at(const fid_args& a, size_t idx) {
  return a.mixed ? (double)((const float*)a.verts)[idx] : ((const double*)a.verts)[idx];
}

constexpr int FRMAX = 8;   // fine ring pairs per pass at most

// Dynamic shared memory of a CTA at most: 227 KB less the kernel's own arrays.
constexpr size_t FID_SMEM = 226 * 1024;

__host__ __device__ constexpr size_t fid_pass_bytes(int p, int pairs) {
  return sizeof(double) * ((size_t)3 * (p + 1) * (p + 1) + (size_t)6 * pairs * ((2 * p + 1) + (4 * p) * 4));
}

// Pairs of fine rings (r and Pf - r) per pass for order p: as many as keep the
// pass's point tasks (one per ring and longitude quarter) within two rounds of 256
// threads, so that few lanes of the last warp idle, and its rings within the shared
// memory (factor 1 at p = 31: 7 pairs, as 8 would take 239 KB).
__host__ __device__ constexpr int fid_pairs(int p, int factor) {
  int nq = factor * p + 1, r = 256 / nq;
  r = r < 1 ? 1 : (r > FRMAX ? FRMAX : r);
  while (r > 1 && fid_pass_bytes(p, r) > FID_SMEM) --r;
  return r;
}

constexpr bool fid_fits() {   // every order and factor that the entry point takes
  for (int p = 1; p <= STIV_MAX_P; ++p)
    for (int f = 1; f <= 8; ++f)
      if (fid_pass_bytes(p, fid_pairs(p, f)) > FID_SMEM) return false;
  return true;
}
static_assert(fid_fits(), "a pass of fidelity_kernel must fit the shared memory");

// The mesh along one fine ring, per coordinate field and longitude cell j
// (j1 = j + 1 mod 2P), as two lines in the cell fraction b:
//   A + b dA on the triangle (i, j), (i+1, j), (i+1, j+1)  (taken when a_ >= b),
//   B + b dB on the triangle (i, j), (i+1, j+1), (i, j+1)  (when a_ < b),
// with a_ the ring's fraction between mesh rings i and i+1; in the pole caps
// (zone 0 north, 2 south; tp the fraction from the pole to the first ring)
// both lines are the fan triangle's.  out: A, dA, B, dB.
__device__ __forceinline__ void mesh_lines(const fid_args& a, size_t o, int P, int W, int zone, int i, double a_,
                                           double tp, int j, double* out) {
  int j1 = j + 1 == W ? 0 : j + 1;
  if (zone != 1) {
    size_t pole = o + 2 * (size_t)P * (P + 1) + (zone == 2 ? 1 : 0);
    size_t ring = o + (zone == 2 ? (size_t)P * W : 0);
    double N = vert_at(a, pole), x0 = vert_at(a, ring + j), x1 = vert_at(a, ring + j1);
    out[0] = out[2] = fma(tp, x0 - N, N);
    out[1] = out[3] = tp * (x1 - x0);
    return;
  }
  double q = vert_at(a, o + (size_t)i * W + j), rr = vert_at(a, o + (size_t)(i + 1) * W + j);
  double s3 = vert_at(a, o + (size_t)(i + 1) * W + j1), u = vert_at(a, o + (size_t)i * W + j1);
  out[0] = fma(a_, rr - q, q);
  out[1] = s3 - rr;
  out[2] = fma(a_, s3 - u, q);
  out[3] = u - q;
}

// CTA (vesicle, time level, chunk of the ring pairs), a few pairs per pass.  The
// series is evaluated like the synthesis: ring sums G(m) of a ring and its mirror
// image from the even and the odd terms, then per longitude the even and odd
// partial Fourier sums of the three fields, which give the four longitudes phi_k,
// pi - phi_k, pi + phi_k and 2 pi - phi_k (k <= Pf / 2) at once.  The chunks' maxima
// meet in err (cleared before) by an atomic maximum of non-negative bit patterns.
//
// Bound by the FP64 pipe: the points (about 45 operations each at p = 12) are two
// thirds of it.  What depends on the order alone (nodes, Legendre and trigonometric
// values, places on the mesh) is tabulated once per handle instead of per call and
// CTA; chunks fill the chip for few vesicles.  256 vesicles, p = 12, factor 4: 1.53 ->
// 0.83 ms (the nodes alone took 0.23 ms); the FP64 pipe is 0.91 busy.
__global__ void __launch_bounds__(256) fidelity_kernel(fid_args a) {
  extern __shared__ double sm[];
  __shared__ unsigned long long red[256 / 32];
  int v = blockIdx.x, t = blockIdx.y;
  if (a.p[v] < 1 || a.p[v] > STIV_MAX_P || !a.theta[a.p[v]]) {   // order outside [1, p_max]: NaN
    if (threadIdx.x == 0 && blockIdx.z == 0) a.err[2 * (size_t)v + t] = __longlong_as_double(0x7ff8000000000000LL);
    return;
  }
  const int p = a.p[v], P = 2 * p, Pf = a.factor * P, W = 2 * P, nv = 2 * P * (P + 1) + 2;
  const int nc = (p + 1) * (p + 1), nl = (p + 1) * (p + 2) / 2, ns = 2 * p + 1, nq = Pf / 2 + 1;
  const int PR = fid_pairs(p, a.factor), npair = Pf / 2 + 1;   // pair r: rings r and Pf - r (the equator alone)
  double* C = sm;                   // [3][nc]
  double* G = C + 3 * nc;           // [2 PR][3][ns] ring sums (slot 0: m=0; 2m-1: cos m; 2m: sin m); pair k: rings 2k, 2k + 1
  double* ML = G + 2 * PR * 3 * ns; // [2 PR][3][W][4] mesh lines of the current rings (mesh_lines)
  __shared__ double btab[8];
  __shared__ fid_ring info[2 * FRMAX];
  const double* base_t = a.tab + a.off[p];
  const fid_ring* ring = (const fid_ring*)base_t;
  const double* leg = base_t + fid_ring_doubles(p, a.factor);
  const double* trig = leg + fid_leg_doubles(p, a.factor);
  if (threadIdx.x < a.factor) btab[threadIdx.x] = (double)threadIdx.x / a.factor;
  const double* coef = a.coef + a.coef_off[v] + (size_t)t * 3 * nc;
  for (int k = threadIdx.x; k < 3 * nc; k += blockDim.x) C[k] = coef[k];
  size_t base = a.vert_off[v] + (size_t)t * 3 * nv;
  unsigned long long worst2 = 0;   // bit pattern of the largest squared distance
  const int per = (npair + gridDim.z - 1) / gridDim.z, first = blockIdx.z * per, last = min(first + per, npair);
  for (int r0 = first; r0 < last; r0 += PR) {
    const int np = min(PR, last - r0);
    __syncthreads();   // C, btab; info, G and ML are rewritten for the next rings
    if (threadIdx.x < 2 * np) {
      const int r = r0 + (threadIdx.x >> 1);
      info[threadIdx.x] = ring[threadIdx.x & 1 ? Pf - r : r];
    }
    // ring sums: lanes over the fields and rings of one order m run the same terms
    for (int task = threadIdx.x; task < ns * 3 * np; task += blockDim.x) {
      const int sl = task / (3 * np), rem = task - sl * 3 * np, f = rem / np, k = rem - f * np, m = (sl + 1) >> 1;
      const int sgn = sl == 0 ? 0 : ((sl & 1) ? 1 : -1);
      const double* Cf = C + f * nc + sgn * m;
      const double* Lr = leg + (size_t)(r0 + k) * nl + m;
      double E = 0.0, O = 0.0;
      for (int n = m; n <= p; n += 2) {
        E = fma(Cf[n * n + n], Lr[n * (n + 1) / 2], E);
        if (n + 1 <= p) O = fma(Cf[(n + 1) * (n + 2)], Lr[(n + 1) * (n + 2) / 2], O);
      }
      G[((2 * k) * 3 + f) * ns + sl] = E + O;
      G[((2 * k + 1) * 3 + f) * ns + sl] = E - O;
    }
    __syncthreads();
    for (int task = threadIdx.x; task < 2 * np * 3 * W; task += blockDim.x) {
      const int q = task / (3 * W), rem = task - q * 3 * W, f = rem / W, j = rem - f * W;
      const fid_ring& R = info[q];
      mesh_lines(a, base + (size_t)f * nv, P, W, R.zone, R.cell, R.al, R.tp, j, ML + (size_t)task * 4);
    }
    __syncthreads();
    for (int task = threadIdx.x; task < 2 * np * nq; task += blockDim.x) {
      const int k = task / nq, q = task - k * nq;
      if ((k & 1) && 2 * (r0 + (k >> 1)) == Pf) continue;   // the equator's image is itself
      const int tri = info[k].tri;
      const double* g = G + (size_t)k * 3 * ns;
      double Ce[3], Co[3], Se[3], So[3];
#pragma unroll
      for (int f = 0; f < 3; ++f) { Ce[f] = g[f * ns]; Co[f] = 0.0; Se[f] = 0.0; So[f] = 0.0; }
      for (int m = 1; m <= p; m += 2) {
        double c = trig[(size_t)(2 * m) * nq + q], sn = trig[(size_t)(2 * m + 1) * nq + q];
#pragma unroll
        for (int f = 0; f < 3; ++f) {
          Co[f] = fma(g[f * ns + 2 * m - 1], c, Co[f]);
          So[f] = fma(g[f * ns + 2 * m], sn, So[f]);
        }
        if (m + 1 <= p) {
          c = trig[(size_t)(2 * m + 2) * nq + q]; sn = trig[(size_t)(2 * m + 3) * nq + q];
#pragma unroll
          for (int f = 0; f < 3; ++f) {
            Ce[f] = fma(g[f * ns + 2 * m + 1], c, Ce[f]);
            Se[f] = fma(g[f * ns + 2 * m + 2], sn, Se[f]);
          }
        }
      }
      const int kq[4] = {q, Pf - q, Pf + q, (2 * Pf - q) % (2 * Pf)};
#pragma unroll
      for (int w = 0; w < 4; ++w) {
        const int kk = kq[w];
        const bool dup = (w == 1 && kk == kq[0]) || (w == 2 && (kk == kq[1] || kk >= 2 * Pf)) ||
                         (w == 3 && (kk == kq[0] || kk == kq[2]));
        if (dup) continue;
        const int j = kk / a.factor, sb = kk - j * a.factor;
        const double b = btab[sb];
        const int side = (tri >> sb) & 1 ? 0 : 2;
        double d2 = 0.0;
#pragma unroll
        for (int f = 0; f < 3; ++f) {
          const double C0 = w == 0 || w == 3 ? Ce[f] + Co[f] : Ce[f] - Co[f];
          const double S0 = w == 0 || w == 3 ? Se[f] + So[f] : Se[f] - So[f];
          const double val = w == 0 || w == 2 ? C0 + S0 : C0 - S0;   // phi, pi - phi, pi + phi, 2 pi - phi
          const double* l = ML + ((size_t)(k * 3 + f) * W + j) * 4 + side;
          const double e = fma(b, l[1], l[0]) - val;
          d2 = fma(e, e, d2);
        }
        // the maximum on the integer pipe; a NaN is ignored, as fmax ignores it
        const unsigned long long u = (unsigned long long)__double_as_longlong(d2);
        if (u > worst2 && u <= 0x7FF0000000000000ull) worst2 = u;
      }
    }
  }
  for (int off = 16; off > 0; off >>= 1) {
    const unsigned long long o = __shfl_xor_sync(0xffffffffu, worst2, off);
    worst2 = o > worst2 ? o : worst2;
  }
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = worst2;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int q = 1; q < (int)(blockDim.x >> 5); ++q) worst2 = red[q] > worst2 ? red[q] : worst2;
    const double e = sqrt(__longlong_as_double((long long)worst2));
    atomicMax((unsigned long long*)&a.err[2 * (size_t)v + t], (unsigned long long)__double_as_longlong(e));
  }
}

}  // namespace

int stiv_ensure_tables(stiv_handle* h, cudaStream_t st, int p) {
  if (p < 1 || p > STIV_MAX_P) return STIV_ERR_ARG;
  if (h->tab_ready[p]) return STIV_OK;
  int P = 2 * p, nl = (p + 1) * (p + 2) / 2;
  stiv_tables& T = h->tab[p];
  STIV_CUDA(h, cudaMalloc(&T.leg, sizeof(double) * (size_t)(P + 3) * nl));
  STIV_CUDA(h, cudaMalloc(&T.trig, sizeof(double) * (size_t)(P / 2 + 1) * 2 * (p + 1)));
  STIV_CUDA(h, cudaMalloc(&T.theta, sizeof(double) * (P + 1)));
  STIV_CUDA(h, cudaMalloc(&T.leg_t, sizeof(double) * (size_t)nl * (P / 2 + 1)));
  STIV_CUDA(h, cudaMalloc(&T.trig_t, sizeof(double) * (size_t)(P / 2 + 1) * 2 * (p + 1)));
  int n = (P / 2 + 1) * (p + 1) > P + 3 ? (P / 2 + 1) * (p + 1) : P + 3;
  tables_kernel<<<(n + 127) / 128, 128, 0, st>>>(p, T.leg, T.trig, T.theta, T.leg_t, T.trig_t);
  STIV_LAUNCH(h);
  h->tab_ready[p] = true;
  return STIV_OK;
}

static size_t synth_smem(int p, int fields) {
  int P = 2 * p;
  return sizeof(double) * (size_t)fields * ((p + 1) * (p + 1) + (P + 1) * (2 * p + 1));
}

extern "C" int stiv_upsample(stiv_handle* h, void* stream, int32_t n_ves, int32_t p_max, const int32_t* p_dev,
                             const int64_t* coef_off_dev, const double* coef_dev,
                             const int64_t* vert_off_dev, void* verts_dev) {
  if (!h || n_ves < 0 || p_max < 1 || p_max > STIV_MAX_P) return STIV_ERR_ARG;
  if (n_ves == 0) return STIV_OK;
  if (!p_dev || !coef_off_dev || !coef_dev || !vert_off_dev || !verts_dev) return STIV_ERR_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  if (h->prm.precision == STIV_MIXED)
    return stiv_upsample_tc(h, st, n_ves, p_max, p_dev, coef_off_dev, coef_dev, vert_off_dev, (float*)verts_dev);
  synth_args a;
  a.p = p_dev; a.coef_off = coef_off_dev; a.coef = coef_dev; a.vert_off = vert_off_dev;
  a.verts = (double*)verts_dev;
  for (int p = 0; p <= STIV_MAX_P; ++p) { a.leg[p] = nullptr; a.leg_t[p] = nullptr; a.trig_t[p] = nullptr; }
  for (int p = 1; p <= p_max; ++p) {
    int rc = stiv_ensure_tables(h, st, p);
    if (rc) return rc;
    a.leg[p] = h->tab[p].leg; a.leg_t[p] = h->tab[p].leg_t; a.trig_t[p] = h->tab[p].trig_t;
  }
  // one field per CTA where three would leave SMs idle (two vesicles at p = 8:
  // 17.7 -> 16.7 us)
  bool split = 2 * n_ves < 152;
  size_t smem = synth_smem(p_max, split ? 1 : 3);
  STIV_PROF(h, st, "synth");
  if (split) {
    STIV_SMEM(h, synth_kernel<1>, smem, 0, synth_smem(STIV_MAX_P, 1));
    synth_kernel<1><<<dim3(n_ves, 2, 3), 256, smem, st>>>(a);
  } else {
    STIV_SMEM(h, synth_kernel<3>, smem, 0, synth_smem(STIV_MAX_P, 3));
    synth_kernel<3><<<dim3(n_ves, 2), 256, smem, st>>>(a);
  }
  STIV_LAUNCH(h);
  return STIV_OK;
}

extern "C" int stiv_mesh_fidelity(stiv_handle* h, void* stream, int32_t n_ves, int32_t p_max, const int32_t* p_dev,
                                  const int64_t* coef_off_dev, const double* coef_dev, const int64_t* vert_off_dev,
                                  const void* verts_dev, int32_t factor, double* err_dev) {
  if (!h || n_ves < 0 || p_max < 1 || p_max > STIV_MAX_P || factor < 1 || factor > 8) return STIV_ERR_ARG;
  if (n_ves == 0) return STIV_OK;
  if (!p_dev || !coef_off_dev || !coef_dev || !vert_off_dev || !verts_dev || !err_dev) return STIV_ERR_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  fid_args a;
  a.p = p_dev; a.coef_off = coef_off_dev; a.coef = coef_dev; a.vert_off = vert_off_dev; a.verts = verts_dev;
  a.mixed = h->prm.precision == STIV_MIXED; a.factor = factor; a.err = err_dev;
  for (int p = 0; p <= STIV_MAX_P; ++p) a.theta[p] = nullptr;
  for (int p = 1; p <= p_max; ++p) {
    int rc = stiv_ensure_tables(h, st, p);
    if (rc) return rc;
    a.theta[p] = h->tab[p].theta;
  }
  // always raised, and before anything is launched or cleared: the kernel's own
  // arrays count too, so that the line is not at 48 KB of dynamic memory.  To the
  // most of any call, for speed too: with the call's own size 834 instead of 807 us
  // for 256 vesicles of order 12
  STIV_CUDA(h, cudaFuncSetAttribute(fidelity_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)FID_SMEM));
  size_t total = 0, smem = 0;
  for (int p = 0; p <= STIV_MAX_P; ++p) a.off[p] = 0;
  for (int p = 1; p <= p_max; ++p) {
    a.off[p] = total;
    total += fid_doubles(p, factor);
    size_t b = fid_pass_bytes(p, fid_pairs(p, factor));
    smem = b > smem ? b : smem;
  }
  STIV_PROF_N(h, st, "mesh_fidelity", 2);
  // The tables stay valid for the same factor and orders.  Every call waits for
  // the end of the one before (an event: a stream's handle may be that of a
  // destroyed stream, or stand for a stream of each thread), so that it finds
  // them written, and rewrites them only once they have been read.  A captured
  // call makes them in its graph, whose replays overwrite them at any time: from
  // then on every call of the handle makes its own.
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  STIV_CUDA(h, cudaStreamIsCapturing(st, &cap));
  const bool captured = cap != cudaStreamCaptureStatusNone;
  if (captured) h->fid_captured = true;
  else if (h->fid_done) STIV_CUDA(h, cudaStreamWaitEvent(st, h->fid_done, 0));
  else STIV_CUDA(h, cudaEventCreateWithFlags(&h->fid_done, cudaEventDisableTiming));
  const bool made = h->fid_tab && !h->fid_captured && h->fid_factor == factor && h->fid_pmax == p_max;
  if (sizeof(double) * total > h->fid_tab_bytes) {
    h->fid_factor = 0;
    if (h->fid_tab) { STIV_CUDA(h, cudaFree(h->fid_tab)); h->fid_tab = nullptr; h->fid_tab_bytes = 0; }
    STIV_CUDA(h, cudaMalloc(&h->fid_tab, sizeof(double) * total));
    h->fid_tab_bytes = sizeof(double) * total;
  }
  a.tab = h->fid_tab;
  if (!made) {
    h->fid_factor = 0;   // set again once all has been launched
    fid_tables_kernel<<<dim3(factor * p_max + 1, p_max), 64, 0, st>>>(a, h->fid_tab);
    STIV_LAUNCH(h);
  }
  STIV_CUDA(h, cudaMemsetAsync(err_dev, 0, sizeof(double) * 2 * (size_t)n_ves, st));
  // enough chunks for a dozen CTAs per SM, at most one per pass of the largest order
  const int passes = (factor * p_max + fid_pairs(p_max, factor)) / fid_pairs(p_max, factor);
  int chunks = (12 * 152 + 2 * n_ves - 1) / (2 * n_ves);
  chunks = chunks < 1 ? 1 : (chunks > passes ? passes : chunks);
  fidelity_kernel<<<dim3(n_ves, 2, chunks), 256, smem, st>>>(a);
  STIV_LAUNCH(h);
  if (!captured) STIV_CUDA(h, cudaEventRecord(h->fid_done, st));
  h->fid_factor = factor; h->fid_pmax = p_max;
  return STIV_OK;
}
