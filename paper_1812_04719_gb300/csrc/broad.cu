// Space-time bounding boxes (Alg. 2 getBoundingBox) and the bounding-box
// intersection of Alg. 1 (Sec. 3.3.1) on one GPU.
//
//   1. vesicle boxes: exact FP64 min/max of X0 and X1 over all vertices, padded
//      by d_m; patch boxes (4 x 8 grid quads and their vertices) in FP32,
//      rounded outward, for the narrow phase;
//   2. h_m = mean box diagonal (Alg. 1, grid spacing), cell size of a uniform grid
//      (periodic axes: L / floor(L / h_m));
//   3. each box lists the cells it overlaps (an exact cell-range enumeration
//      standing in for the check points of Alg. 1), keyed by the
//      Morton id of the (wrapped) cell;
//   4. stable radix sort by Morton id (Alg. 1, check-point sort; 24-bit keys:
//      at most 256 wrapped cells per axis);
//   5. all box pairs within a cell: the image shift follows from the unwrapped
//      cell coordinates, then bbiCheck in FP64 (Alg. 1, per-cell loop);
//   6. sort + unique (Alg. 1, final step) -> pairs (i < j, shift), ascending.
//
// Up to STIV_BRUTE_MAX vesicles steps 2-6 are replaced by the test of every
// pair of boxes, which gives the same pairs already in order in two launches
// (row_pairs_kernel, emit_pairs_kernel).
#include "stiv_internal.cuh"

#include <math.h>

namespace {

template <typename T>
__device__ __forceinline__ double ld(const void* p, size_t i) { return (double)((const T*)p)[i]; }

__device__ __forceinline__ double vload(const void* X, int mixed, size_t i) {
  return mixed ? (double)((const float*)X)[i] : ((const double*)X)[i];
}

// Order-preserving int64 image of a double (a <= b <=> okey(a) <= okey(b)
// for non-NaN values, -0 just below +0) and its inverse (the map is its own
// inverse): exact FP64 min / max on the integer pipe.
__device__ __forceinline__ long long okey(double v) {
  long long b = __double_as_longlong(v);
  return b ^ ((b >> 63) & 0x7FFFFFFFFFFFFFFFll);
}
__device__ __forceinline__ double okey_val(long long k) {
  return __longlong_as_double(k ^ ((k >> 63) & 0x7FFFFFFFFFFFFFFFll));
}

// x rounded to float toward -inf (up = false) or +inf (up = true), on the
// integer pipe for |x| in the normal float range: the significand truncated
// to 23 bits rounds toward zero, and one unit in the last place more in
// magnitude gives the other direction when bits were dropped (a carry into
// the exponent, up to infinity, is the correct rounding).  Other values take
// the conversion instruction.
__device__ __forceinline__ float d2f_dir(double x, bool up) {
  unsigned long long b = (unsigned long long)__double_as_longlong(x);
  int e = (int)((b >> 52) & 0x7FF) - 1023;
  if (e < -126 || e > 127) return up ? __double2float_ru(x) : __double2float_rd(x);
  unsigned sgn = (unsigned)(b >> 63);
  unsigned f = (sgn << 31) | ((unsigned)(e + 127) << 23) | (unsigned)((b >> 29) & 0x7FFFFF);
  if ((b & 0x1FFFFFFFull) != 0 && (up ? sgn == 0 : sgn != 0)) f += 1;
  return __uint_as_float(f);
}

// One CTA per vesicle.  MIXED (FP32 vertices): the min / max run in FP32,
// which is exact, and widen exactly to FP64, so the boxes are those of the
// FP64 reduction bit for bit without its FP64 instructions.  FP64 vertices:
// the min / max run on order-preserving integer images (exact), and the
// per-vertex FP32 boxes are rounded outward on the integer pipe, so that the
// FP64 pipe only forms the staging differences.
//
// Bound by the latency of its phases more than by HBM (302 MB at 1440 vesicles and
// p = 16, 0.045 ms of copy): 512 threads instead of 256, the reduction by shuffles
// instead of eight barriers, two lanes per patch (a column half each): 0.176 ->
// 0.158 ms.  Vesicles of small orders leave many of the 512 idle: 4096 of orders 8,
// 12 and 16 0.29 -> 0.31 ms, 9216 of order 3 0.13 -> 0.20.
constexpr int BT = 512;
constexpr size_t VB_SMEM = 96 * 1024;   // per-vertex boxes kept in shared memory at most
template <bool MIXED>
__global__ void __launch_bounds__(BT) boxes_kernel(int n, const int32_t* pv, const int64_t* voff, const void* X,
                                                    int mixed, double dm, double Lx, double Ly, double Lz,
                                                    double* vbox, float* pbox, int pstride, float* vorg,
                                                    float* fprep, int64_t fstride, int64_t* ctr, size_t vb_cap,
                                                    int p_max, float* fbox) {
  extern __shared__ float vbs[];   // [6][nv]: swept FP32 box of each vertex (rounded outward), if it fits
  int v = blockIdx.x;
  if (pv[v] < 1 || pv[v] > p_max) {
    // an order outside [1, p_max]: flagged, and an inverted box keeps the
    // vesicle out of every cell (the broad phase skips inverted boxes), so no
    // later kernel reads its mesh
    if (threadIdx.x == 0) atomicOr((unsigned long long*)&ctr[STIV_C_STATUS], STIV_F_BAD_ORDER);
    if (threadIdx.x < 3) {
      vbox[6 * v + threadIdx.x] = INFINITY;
      vbox[6 * v + 3 + threadIdx.x] = -INFINITY;
      fbox[(size_t)threadIdx.x * n + v] = INFINITY;
      fbox[(size_t)(3 + threadIdx.x) * n + v] = -INFINITY;
    }
    if (threadIdx.x < 4) vorg[4 * v + threadIdx.x] = 0.0f;
    return;
  }
  int P = 2 * pv[v], nv = stiv_nverts(P);
  bool use_sm = (size_t)6 * nv <= vb_cap;
  const size_t base = voff[v];
  __shared__ long long red[BT / 32][6];
  double lo[3] = {INFINITY, INFINITY, INFINITY}, hi[3] = {-INFINITY, -INFINITY, -INFINITY};
  bool bad = false;
  if (MIXED) {
    const float* Xf = (const float*)X;
    float flo[3] = {INFINITY, INFINITY, INFINITY}, fhi[3] = {-INFINITY, -INFINITY, -INFINITY};
    for (int k = threadIdx.x; k < nv; k += blockDim.x)
      for (int c = 0; c < 3; ++c) {
        float x0 = Xf[base + (size_t)c * nv + k], x1 = Xf[base + (size_t)(3 + c) * nv + k];
        if (!isfinite(x0) || !isfinite(x1)) bad = true;
        float a = fminf(x0, x1), b = fmaxf(x0, x1);
        flo[c] = fminf(flo[c], a);
        fhi[c] = fmaxf(fhi[c], b);
        if (use_sm) { vbs[c * nv + k] = a; vbs[(3 + c) * nv + k] = b; }
      }
    for (int c = 0; c < 3; ++c) { lo[c] = (double)flo[c]; hi[c] = (double)fhi[c]; }
  }
  long long klo[3], khi[3];
  for (int c = 0; c < 3; ++c) { klo[c] = okey(lo[c]); khi[c] = okey(hi[c]); }
  if (!MIXED) {
    const double* Xd = (const double*)X;
    for (int k = threadIdx.x; k < nv; k += blockDim.x)
      for (int c = 0; c < 3; ++c) {
        double x0 = Xd[base + (size_t)c * nv + k], x1 = Xd[base + (size_t)(3 + c) * nv + k];
        long long b0 = __double_as_longlong(x0), b1 = __double_as_longlong(x1);
        long long k0 = okey(x0), k1 = okey(x1);
        // finite iff the exponent field is not all ones; a NaN is ignored by
        // the min / max, as fmin / fmax ignore it
        if ((~b0 & 0x7FF0000000000000ll) == 0 || (~b1 & 0x7FF0000000000000ll) == 0) bad = true;
        bool n0 = (b0 & 0x7FFFFFFFFFFFFFFFll) > 0x7FF0000000000000ll;
        bool n1 = (b1 & 0x7FFFFFFFFFFFFFFFll) > 0x7FF0000000000000ll;
        if (n0) k0 = k1;
        if (n1) k1 = k0;
        long long ka = k0 < k1 ? k0 : k1, kb = k0 < k1 ? k1 : k0;
        if (!(n0 && n1)) {
          klo[c] = ka < klo[c] ? ka : klo[c];
          khi[c] = kb > khi[c] ? kb : khi[c];
        }
        if (use_sm) {
          vbs[c * nv + k] = d2f_dir(okey_val(ka), false);
          vbs[(3 + c) * nv + k] = d2f_dir(okey_val(kb), true);
        }
      }
  }
  for (int o = 16; o > 0; o >>= 1)
    for (int c = 0; c < 3; ++c) {
      const long long a = __shfl_xor_sync(0xffffffffu, klo[c], o), b = __shfl_xor_sync(0xffffffffu, khi[c], o);
      klo[c] = a < klo[c] ? a : klo[c];
      khi[c] = b > khi[c] ? b : khi[c];
    }
  if ((threadIdx.x & 31) == 0)
    for (int c = 0; c < 3; ++c) { red[threadIdx.x >> 5][c] = klo[c]; red[threadIdx.x >> 5][3 + c] = khi[c]; }
  if (__syncthreads_or(bad) && threadIdx.x == 0) atomicOr((unsigned long long*)&ctr[STIV_C_STATUS], STIV_F_NONFINITE);
  __shared__ float sorg[4];
  __shared__ double vlo_s[3], vhi_s[3];
  int fin = 1;
  if (threadIdx.x < 3) {
    int c = threadIdx.x;
    long long a = red[0][c], b = red[0][3 + c];
    for (int q = 1; q < BT / 32; ++q) {
      a = red[q][c] < a ? red[q][c] : a;
      b = red[q][3 + c] > b ? red[q][3 + c] : b;
    }
    vlo_s[c] = okey_val(a);
    vhi_s[c] = okey_val(b);
    fin = (~__double_as_longlong(vlo_s[c]) & 0x7FF0000000000000ll) != 0 &&
          (~__double_as_longlong(vhi_s[c]) & 0x7FF0000000000000ll) != 0;
  }
  // a box that is not finite on every axis (the vesicle is flagged) is inverted on
  // all of them: infinite ends would meet the inverted boxes above, and the broad
  // phase tells inverted boxes by any one axis
  fin = __syncthreads_and(fin);
  if (threadIdx.x < 3) {
    int c = threadIdx.x;
    double l = vlo_s[c] - dm, u = vhi_s[c] + dm;
    const double bl = fin ? l : INFINITY, bu = fin ? u : -INFINITY;
    vbox[6 * v + c] = bl;
    vbox[6 * v + 3 + c] = bu;
    fbox[(size_t)c * n + v] = __double2float_rd(bl);
    fbox[(size_t)(3 + c) * n + v] = __double2float_ru(bu);
    double L = c == 0 ? Lx : c == 1 ? Ly : Lz;
    if (L > 0.0 && !(u - l < 0.5 * L)) atomicOr((unsigned long long*)&ctr[STIV_C_STATUS], STIV_F_BOX_TOO_SMALL);
    // FP32 frame of this vesicle: origin at the (float-rounded) box centre
    float o = (float)(0.5 * (vlo_s[c] + vhi_s[c]));
    sorg[c] = o;
    vorg[4 * v + c] = o;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    // R bounds |X - o| over the vesicle (both times), rounded up
    double R = 0.0;
    for (int c = 0; c < 3; ++c) R = fmax(R, fmax(vhi_s[c] - (double)sorg[c], (double)sorg[c] - vlo_s[c]));
    vorg[4 * v + 3] = __double2float_ru(R);
  }
  // per-vertex FP32 data (two float4).  FP32 vertices: X0 and X1 as stored,
  // from which the narrow phase takes both the exact keys and the frame
  // coordinates.  FP64 vertices: position at t_n relative to the origin and
  // the displacement X1 - X0, each rounded once.
  float4* f4 = (float4*)(fprep + (size_t)v * fstride);
  if (MIXED) {
    const float* Xf = (const float*)X;
    for (int k = threadIdx.x; k < nv; k += blockDim.x) {
      f4[2 * k] = make_float4(Xf[base + k], Xf[base + (size_t)nv + k], Xf[base + (size_t)2 * nv + k], 0.f);
      f4[2 * k + 1] = make_float4(Xf[base + (size_t)3 * nv + k], Xf[base + (size_t)4 * nv + k],
                                  Xf[base + (size_t)5 * nv + k], 0.f);
    }
  } else
  for (int k = threadIdx.x; k < nv; k += blockDim.x) {
    float xo[3], dd[3];
    for (int c = 0; c < 3; ++c) {
      double x0 = vload(X, mixed, base + (size_t)c * nv + k);
      double x1 = vload(X, mixed, base + (size_t)(3 + c) * nv + k);
      xo[c] = (float)(x0 - (double)sorg[c]);
      dd[c] = (float)(x1 - x0);
    }
    f4[2 * k] = make_float4(xo[0], xo[1], xo[2], 0.f);
    f4[2 * k + 1] = make_float4(dd[0], dd[1], dd[2], 0.f);
  }
  // patch boxes: vertex rows [I*BR, I*BR+BR], columns [J*BC, J*BC+BC]
  // (wrapping), poles; each as the union of its four cells' boxes (band b of
  // the two, column half h), every cell box written beside it.  Per column
  // half, the boxes of its three rows are formed once and merged into its
  // two cells.  P is even, so every patch
  // spans BR bands and BC columns.  From the per-vertex FP32 boxes in shared
  // memory when they fit: rounding outward is monotone, so the result equals
  // rounding the FP64 min / max.
  int nbr = stiv_nband_blocks(P), nbc = stiv_ncol_blocks(P), W = 2 * P;
  __syncthreads();
  // lanes 2 k and 2 k + 1 take the column halves of one patch
  for (int t0 = 0; t0 < 2 * nbr * nbc; t0 += blockDim.x) {
    const int task = t0 + threadIdx.x, patch = task >> 1, h = task & 1;
    const bool on = patch < nbr * nbc;
    int I = on ? patch / nbc : 0, J = on ? patch % nbc : 0;
    int r0 = I * STIV_BR, c0 = J * STIV_BC;
    // per column half: rb[row][lo xyz, hi xyz] of its three rows; pb[pole]:
    // FP32, rounded outward
    float pb[2][6];
    auto vbox_of = [&](int vid, float* o) {
      if (use_sm) {
        for (int c = 0; c < 3; ++c) { o[c] = vbs[c * nv + vid]; o[3 + c] = vbs[(3 + c) * nv + vid]; }
      } else {
        for (int c = 0; c < 3; ++c) {
          double x0 = vload(X, mixed, base + (size_t)c * nv + vid), x1 = vload(X, mixed, base + (size_t)(3 + c) * nv + vid);
          o[c] = __double2float_rd(fmin(x0, x1));
          o[3 + c] = __double2float_ru(fmax(x0, x1));
        }
      }
    };
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      bool has = q == 0 ? I == 0 : I == nbr - 1;
      if (has) vbox_of(W * (P + 1) + q, pb[q]);
      else for (int c = 0; c < 3; ++c) { pb[q][c] = INFINITY; pb[q][3 + c] = -INFINITY; }
    }
    float* B = pbox + ((size_t)v * pstride + patch) * STIV_PBOX;
    float plo[3] = {INFINITY, INFINITY, INFINITY}, phi[3] = {-INFINITY, -INFINITY, -INFINITY};
    {
      float rb[3][6];
#pragma unroll
      for (int rr = 0; rr < 3; ++rr) {
#pragma unroll
        for (int cc = 0; cc <= 2; ++cc) {
          int col = c0 + 2 * h + cc; if (col >= W) col -= W;
          float o[6];
          vbox_of((r0 + rr) * W + col, o);
#pragma unroll
          for (int c = 0; c < 3; ++c) {
            rb[rr][c] = cc == 0 ? o[c] : fminf(rb[rr][c], o[c]);
            rb[rr][3 + c] = cc == 0 ? o[3 + c] : fmaxf(rb[rr][3 + c], o[3 + c]);
          }
        }
      }
#pragma unroll
      for (int b = 0; b < 2; ++b) {
        float lo[3], hi[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          lo[c] = fminf(fminf(rb[b][c], rb[b + 1][c]), pb[b][c]);
          hi[c] = fmaxf(fmaxf(rb[b][3 + c], rb[b + 1][3 + c]), pb[b][3 + c]);
          plo[c] = fminf(plo[c], lo[c]);
          phi[c] = fmaxf(phi[c], hi[c]);
        }
        if (on) {
          float4* C = (float4*)(B + STIV_PBOX_CELLS) + 2 * (2 * b + h);
          C[0] = make_float4(lo[0], lo[1], lo[2], 0.f);
          C[1] = make_float4(hi[0], hi[1], hi[2], 0.f);
        }
      }
    }
    for (int c = 0; c < 3; ++c) {
      plo[c] = fminf(plo[c], __shfl_xor_sync(0xffffffffu, plo[c], 1));
      phi[c] = fmaxf(phi[c], __shfl_xor_sync(0xffffffffu, phi[c], 1));
    }
    if (on && h == 0) {
      ((float4*)B)[0] = make_float4(plo[0], plo[1], plo[2], phi[0]);
      ((float4*)B)[1] = make_float4(phi[1], phi[2], 0.f, 0.f);
    }
  }
}

// grid[0..2] origin, [3..5] cell size, [6..8] cells per axis, [9..11] periodic flag, [12] h_m
__global__ void __launch_bounds__(1024) grid_kernel(int n, const double* vbox, double Lx, double Ly, double Lz,
                                                    double* grid) {
  __shared__ double sdiag[1024], slo[3][1024], shi[3][1024];
  __shared__ int scnt[1024];
  double d = 0.0, lo[3] = {INFINITY, INFINITY, INFINITY}, hi[3] = {-INFINITY, -INFINITY, -INFINITY};
  int nvalid = 0;
  for (int v = threadIdx.x; v < n; v += 1024) {
    if (!(vbox[6 * v] <= vbox[6 * v + 3])) continue;   // inverted: a vesicle left out (bad order)
    ++nvalid;
    double e0 = vbox[6 * v + 3] - vbox[6 * v], e1 = vbox[6 * v + 4] - vbox[6 * v + 1], e2 = vbox[6 * v + 5] - vbox[6 * v + 2];
    d += sqrt(e0 * e0 + e1 * e1 + e2 * e2);
    for (int c = 0; c < 3; ++c) { lo[c] = fmin(lo[c], vbox[6 * v + c]); hi[c] = fmax(hi[c], vbox[6 * v + 3 + c]); }
  }
  sdiag[threadIdx.x] = d;
  scnt[threadIdx.x] = nvalid;
  for (int c = 0; c < 3; ++c) { slo[c][threadIdx.x] = lo[c]; shi[c][threadIdx.x] = hi[c]; }
  __syncthreads();
  for (int s = 512; s > 0; s >>= 1) {
    if (threadIdx.x < s) {
      sdiag[threadIdx.x] += sdiag[threadIdx.x + s];
      scnt[threadIdx.x] += scnt[threadIdx.x + s];
      for (int c = 0; c < 3; ++c) {
        slo[c][threadIdx.x] = fmin(slo[c][threadIdx.x], slo[c][threadIdx.x + s]);
        shi[c][threadIdx.x] = fmax(shi[c][threadIdx.x], shi[c][threadIdx.x + s]);
      }
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    double hm = sdiag[0] / (scnt[0] > 0 ? scnt[0] : 1);
    if (!(hm > 0.0)) hm = 1.0;
    for (int c = 0; c < 3; ++c)
      if (!(slo[c][0] <= shi[c][0])) { slo[c][0] = 0.0; shi[c][0] = 0.0; }   // no valid box
    double L[3] = {Lx, Ly, Lz};
    for (int c = 0; c < 3; ++c) {
      if (L[c] > 0.0) {
        double G = floor(L[c] / hm);
        if (G < 1.0) G = 1.0;
        if (G > 256.0) G = 256.0;
        // whole boxes below the lowest vesicle: unwrapped cells count from there
        grid[c] = floor(slo[c][0] / L[c]) * L[c]; grid[3 + c] = L[c] / G; grid[6 + c] = G; grid[9 + c] = 1.0;
      } else {
        double ext = shi[c][0] - slo[c][0];
        double h = hm;
        if (ext / h > 255.0) h = ext / 255.0;
        double G = floor(ext / h) + 1.0;
        if (!(G >= 1.0)) G = 1.0;   // an extent past the doubles
        grid[c] = slo[c][0]; grid[3 + c] = h; grid[6 + c] = G; grid[9 + c] = 0.0;
      }
    }
    grid[12] = hm;
  }
}

// Cells u0 <= u <= u1 of a box on axis c.  Returns false when a periodic axis' cells
// leave the range that a record holds (then clamped, as the records written are
// those counted whatever the box).
constexpr int UMAX = 500;
__device__ __forceinline__ bool cell_range(const double* grid, const double* box, int c, int& u0, int& u1) {
  double o = grid[c], h = grid[3 + c];
  const double slack = 1e-6;  // cells; covers rounding of the divisions
  u0 = (int)floor((box[c] - o) / h - slack);
  u1 = (int)floor((box[3 + c] - o) / h + slack);
  if (grid[9 + c] == 0.0) {  // free axis: clamp to the grid
    int G = (int)grid[6 + c];
    u0 = max(0, min(u0, G - 1));
    u1 = max(0, min(u1, G - 1));
    return true;
  }
  const bool fits = u0 >= -UMAX && u1 <= UMAX;
  u0 = min(max(u0, -UMAX), UMAX);
  u1 = min(max(u1, -UMAX), UMAX);
  return fits;
}

__global__ void cell_count_kernel(int n, const double* vbox, const double* grid, int32_t* cnt, int64_t* ctr) {
  int v = blockIdx.x * blockDim.x + threadIdx.x;
  if (v >= n) return;
  if (!(vbox[6 * v] <= vbox[6 * v + 3])) { cnt[v] = 0; return; }   // inverted box: no cells
  int c = 1;
  bool fits = true;
  for (int a = 0; a < 3; ++a) {
    int u0, u1;
    fits = cell_range(grid, vbox + 6 * v, a, u0, u1) && fits;
    c *= (u1 - u0 + 1);   // at most (2 UMAX + 1)^3 < 2^31
  }
  if (!fits) atomicOr((unsigned long long*)&ctr[STIV_C_STATUS], STIV_F_BOX_TOO_SMALL);
  cnt[v] = c;
}

// Exclusive scan of n+1 ints (last = total), one CTA; sums above 2^31 - 1 stay there
// (more than any list holds).
__global__ void __launch_bounds__(1024) scan1_kernel(const int32_t* in, int n, int32_t* out) {
  __shared__ int64_t part[1024];
  const int64_t top = 0x7FFFFFFF;
  int per = (n + 1023) / 1024;
  int lo = threadIdx.x * per, hi = min(lo + per, n);
  int64_t s = 0;
  for (int i = lo; i < hi; ++i) s += in[i];
  part[threadIdx.x] = s;
  __syncthreads();
  for (int off = 1; off < 1024; off <<= 1) {
    int64_t v = threadIdx.x >= off ? part[threadIdx.x - off] : 0;
    __syncthreads();
    part[threadIdx.x] += v;
    __syncthreads();
  }
  int64_t run = threadIdx.x ? part[threadIdx.x - 1] : 0;
  for (int i = lo; i < hi; ++i) { out[i] = (int32_t)(run < top ? run : top); run += in[i]; }
  if (threadIdx.x == 1023) out[n] = (int32_t)(part[1023] < top ? part[1023] : top);
}

__device__ __forceinline__ uint32_t spread10(uint32_t x) {
  x &= 0x3FF;
  x = (x | (x << 16)) & 0x030000FF;
  x = (x | (x << 8)) & 0x0300F00F;
  x = (x | (x << 4)) & 0x030C30C3;
  x = (x | (x << 2)) & 0x09249249;
  return x;
}

__global__ void cell_emit_kernel(int n, const double* vbox, const double* grid, const int32_t* off, int64_t R,
                                 uint64_t* key, int32_t* val, int32_t* rbox, int32_t* rcell, int64_t* ctr) {
  int v = blockIdx.x * blockDim.x + threadIdx.x;
  if (v >= n) return;
  int lo[3], hi[3], G[3];
  for (int a = 0; a < 3; ++a) { cell_range(grid, vbox + 6 * v, a, lo[a], hi[a]); G[a] = (int)grid[6 + a]; }
  int64_t r = off[v];
  if (v == n - 1) ctr[8] = off[n];
  if (!(vbox[6 * v] <= vbox[6 * v + 3])) return;   // inverted box: no cells
  for (int x = lo[0]; x <= hi[0]; ++x)
    for (int y = lo[1]; y <= hi[1]; ++y)
      for (int z = lo[2]; z <= hi[2]; ++z, ++r) {
        if (r >= R) { atomicOr((unsigned long long*)&ctr[STIV_C_STATUS], STIV_F_WORK_OVERFLOW); return; }
        int w[3] = {x, y, z};
        for (int a = 0; a < 3; ++a) w[a] = ((w[a] % G[a]) + G[a]) % G[a];
        key[r] = spread10(w[0]) | (spread10(w[1]) << 1) | (spread10(w[2]) << 2);
        val[r] = (int32_t)r;
        rbox[r] = v;
        rcell[r] = (x + 512) | ((y + 512) << 10) | ((z + 512) << 20);
      }
}

__device__ __forceinline__ bool bbi(const double* a, const double* b) {
  return a[0] <= b[3] && b[0] <= a[3] && a[1] <= b[4] && b[1] <= a[4] && a[2] <= b[5] && b[2] <= a[5];
}

// Alg. 1, per-cell loop: every record against the later records of its cell.
__global__ void cell_pairs_kernel(const int64_t* nrec_dev, int64_t R, const uint64_t* key, const int32_t* val,
                                  const int32_t* rbox, const int32_t* rcell, const double* vbox,
                                  const double* grid, double Lx, double Ly, double Lz, int64_t Q,
                                  uint64_t* pkey, int32_t* pval, int64_t* ctr, int nb) {
  const int64_t nrec = *nrec_dev;
  if (nrec > R) return;   // not all are there: flagged, to be run again
  int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= nrec) return;
  double L[3] = {Lx, Ly, Lz};
  int G[3] = {(int)grid[6], (int)grid[7], (int)grid[8]};
  int ra = val[k];
  int ba = rbox[ra], ca = rcell[ra];
  for (int64_t q = k + 1; q < nrec && key[q] == key[k]; ++q) {
    int rb = val[q];
    int bb = rbox[rb], cb = rcell[rb];
    if (bb == ba) continue;
    int s[3];
    bool ok = true;
    for (int a = 0; a < 3; ++a) {
      int du = ((ca >> (10 * a)) & 0x3FF) - ((cb >> (10 * a)) & 0x3FF);
      if (L[a] > 0.0) {
        s[a] = du / G[a];
        if (s[a] * G[a] != du || s[a] < -1 || s[a] > 1) ok = false;
      } else {
        s[a] = 0;
        if (du != 0) ok = false;
      }
    }
    if (!ok) continue;
    int i = ba, j = bb;
    if (i > j) { i = bb; j = ba; s[0] = -s[0]; s[1] = -s[1]; s[2] = -s[2]; }
    double bj[6];
    for (int a = 0; a < 3; ++a) {
      bj[a] = vbox[6 * j + a]; bj[3 + a] = vbox[6 * j + 3 + a];
      if (s[a] != 0) { double sh = s[a] * L[a]; bj[a] = bj[a] + sh; bj[3 + a] = bj[3 + a] + sh; }
    }
    if (!bbi(vbox + 6 * i, bj)) continue;
    int code = 9 * (s[0] + 1) + 3 * (s[1] + 1) + (s[2] + 1);
    unsigned long long slot = atomicAdd((unsigned long long*)&ctr[9], 1ull);
    if ((int64_t)slot < Q) {
      pkey[slot] = ((uint64_t)i << (nb + 5)) | ((uint64_t)j << 5) | (uint64_t)code;
      pval[slot] = 0;
    } else {
      atomicOr((unsigned long long*)&ctr[STIV_C_STATUS], STIV_F_WORK_OVERFLOW);
    }
  }
}

// Alg. 1, final step: unique sorted keys -> output pair list; one CTA.
__global__ void __launch_bounds__(1024) unique_pairs_kernel(const int64_t* nkey_dev, int64_t Q, const uint64_t* key,
                                                            int64_t cap, int32_t* oi, int32_t* oj, int32_t* os,
                                                            int64_t* ctr, int nb) {
  __shared__ int32_t part[1024];
  int64_t n = *nkey_dev; if (n > Q) n = Q;
  int64_t per = (n + 1023) / 1024;
  int64_t lo = threadIdx.x * per, hi = lo + per < n ? lo + per : n;
  int32_t c = 0;
  for (int64_t k = lo; k < hi; ++k) c += (k == 0 || key[k] != key[k - 1]);
  part[threadIdx.x] = c;
  __syncthreads();
  for (int off = 1; off < 1024; off <<= 1) {
    int32_t v = threadIdx.x >= off ? part[threadIdx.x - off] : 0;
    __syncthreads();
    part[threadIdx.x] += v;
    __syncthreads();
  }
  int64_t run = threadIdx.x ? part[threadIdx.x - 1] : 0;
  for (int64_t k = lo; k < hi; ++k) {
    if (k == 0 || key[k] != key[k - 1]) {
      if (run < cap) {
        uint64_t x = key[k];
        oi[run] = (int32_t)(x >> (nb + 5));
        oj[run] = (int32_t)((x >> 5) & ((1ull << nb) - 1));
        os[run] = (int32_t)(x & 31);
      }
      ++run;
    }
  }
  if (threadIdx.x == 1023) {
    int64_t total = part[1023];
    ctr[STIV_C_PAIRS] = total;
    if (total > cap) atomicOr((unsigned long long*)&ctr[STIV_C_STATUS], STIV_F_PAIRS_OVERFLOW);
  }
}

// ---------------------------------------------------------------------------
// All pairs of boxes.  Unit u = (row i, chunk of RCHUNK j's), one warp each,
// row-major, so that the units' hits in order are the pairs in order.  Per lane
// one j: FP32 boxes rounded outward decide, axis by axis, which images may
// overlap (one box's images shifted instead of the other's, widened by 1e-12 of
// the coordinates to cover the FP64 roundings), then bbiCheck in FP64 as below
// for the grid.  A row's first hits are kept, so that the second kernel tests
// again only the rare unit with more.
//
// The n^2 / 2 tests take about 70 instructions per 32; the grid takes 26
// launches (two radix sorts among them), bound by their latency.  Measured, the
// two kernels against the grid: 64 vesicles 0.017 / 0.17 ms, 1024 0.026 / 0.24,
// 4096 0.107 / 0.29, 8192 0.357 / 0.366, 16384 1.22 / 0.53: the line lies at
// 8192 (STIV_BRUTE_MAX).
// ---------------------------------------------------------------------------
constexpr int RCHUNK = STIV_ROW_CHUNK;
constexpr int RKEEP = STIV_ROW_KEEP;
constexpr int RSUM = STIV_ROW_SUM;

struct rows_args {
  int n, nchunk;
  const double* vbox;
  const float* fbox;      // [6][n]
  double L[3];
  int32_t* cnt;           // hits per unit
  int32_t* sum;           // hits per RSUM units (cleared before)
  uint32_t* keep;         // [unit][RKEEP]  j << 5 | shift code
};

// The hits of unit (i, chunk): put(k, j << 5 | code) for the k-th.  Returns their number.
template <class F>
__device__ __forceinline__ int scan_unit(const rows_args& a, int i, int chunk, int lane, F put) {
  int j0 = chunk * RCHUNK, j1 = min(j0 + RCHUNK, a.n);
  if (j1 <= i + 1) return 0;
  float lo[3][3], hi[3][3];   // i's box moved by -s L, per axis and image s
  bool per[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    double l = a.vbox[6 * (size_t)i + c], u = a.vbox[6 * (size_t)i + 3 + c];
    per[c] = a.L[c] > 0.0;
    double w = 1e-12 * (fmax(fabs(l), fabs(u)) + a.L[c]);
#pragma unroll
    for (int s = 0; s < 3; ++s) {
      double d = (s - 1) * a.L[c];
      bool on = s == 1 || per[c];
      lo[c][s] = on ? __double2float_rd(l - d - w) : INFINITY;
      hi[c][s] = on ? __double2float_ru(u - d + w) : -INFINITY;
    }
  }
  int total = 0;
  for (int jb = max(j0, (i + 1) & ~31); jb < j1; jb += 32) {
    int j = jb + lane;
    unsigned mk[3] = {0, 0, 0};
    if (j > i && j < j1) {
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        float bl = a.fbox[(size_t)c * a.n + j], bu = a.fbox[(size_t)(3 + c) * a.n + j];
#pragma unroll
        for (int s = 0; s < 3; ++s) mk[c] |= (lo[c][s] <= bu && bl <= hi[c][s]) ? 1u << s : 0u;
      }
    }
    unsigned code = 0;   // bit 9 sx + 3 sy + sz
    if (mk[0] && mk[1] && mk[2]) {
      const double* A = a.vbox + 6 * (size_t)i;
      const double* B = a.vbox + 6 * (size_t)j;
      unsigned ex[3] = {0, 0, 0};
      for (int c = 0; c < 3; ++c)
        for (int s = 0; s < 3; ++s) {
          if (!((mk[c] >> s) & 1)) continue;
          double b0 = B[c], b3 = B[3 + c];
          if (s != 1) { double sh = (s - 1) * a.L[c]; b0 = b0 + sh; b3 = b3 + sh; }
          if (A[c] <= b3 && b0 <= A[3 + c]) ex[c] |= 1u << s;
        }
      for (int sx = 0; sx < 3; ++sx)
        for (int sy = 0; sy < 3; ++sy)
          if ((ex[0] >> sx) & (ex[1] >> sy) & 1) code |= ex[2] << (9 * sx + 3 * sy);
    }
    unsigned any = __ballot_sync(0xffffffffu, code != 0);
    if (any) {
      int c = __popc(code), off = c;
      for (int o = 1; o < 32; o <<= 1) { int v = __shfl_up_sync(0xffffffffu, off, o); if (lane >= o) off += v; }
      int k = total + off - c;
      for (unsigned m = code; m; m &= m - 1) put(k++, ((uint32_t)j << 5) | (uint32_t)(__ffs(m) - 1));
      total += __shfl_sync(0xffffffffu, off, 31);
    }
  }
  return total;
}

__global__ void __launch_bounds__(256) row_pairs_kernel(rows_args a) {
  int lane = threadIdx.x & 31;
  int64_t u = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
  if (u >= (int64_t)a.n * a.nchunk) return;
  uint32_t* keep = a.keep + u * RKEEP;
  int c = scan_unit(a, (int)(u / a.nchunk), (int)(u % a.nchunk), lane,
                    [&](int k, uint32_t x) { if (k < RKEEP) keep[k] = x; });
  if (lane == 0) {
    a.cnt[u] = c;
    if (c) atomicAdd(&a.sum[u / RSUM], c);
  }
}

// Every CTA sums the counts before its units (whole groups, then the rest of
// its own group), then its warps write their hits.
__global__ void __launch_bounds__(256) emit_pairs_kernel(rows_args a, int64_t cap, int32_t* oi, int32_t* oj,
                                                         int32_t* os, int64_t* ctr) {
  __shared__ int wsum[8], ucnt[8];
  int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  int64_t units = (int64_t)a.n * a.nchunk, u0 = (int64_t)blockIdx.x * 8, u = u0 + w;
  int s = 0;
  int64_t g0 = u0 / RSUM;
  for (int64_t k = threadIdx.x; k < g0; k += 256) s += a.sum[k];
  for (int64_t k = g0 * RSUM + threadIdx.x; k < u0; k += 256) s += a.cnt[k];
  for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
  if (lane == 0) { wsum[w] = s; ucnt[w] = u < units ? a.cnt[u] : 0; }
  __syncthreads();
  int base = 0, total = 0;
  for (int q = 0; q < 8; ++q) { base += wsum[q] + (q < w ? ucnt[q] : 0); total += wsum[q] + ucnt[q]; }
  if (u0 + 8 >= units && threadIdx.x == 0) {
    ctr[STIV_C_PAIRS] = total;
    if (total > cap) atomicOr((unsigned long long*)&ctr[STIV_C_STATUS], STIV_F_PAIRS_OVERFLOW);
  }
  if (u >= units) return;
  int i = (int)(u / a.nchunk);
  auto put = [&](int k, uint32_t x) {
    int64_t at = (int64_t)base + k;
    if (at < cap) { oi[at] = i; oj[at] = (int32_t)(x >> 5); os[at] = (int32_t)(x & 31); }
  };
  if (ucnt[w] <= RKEEP) {
    for (int k = lane; k < ucnt[w]; k += 32) put(k, a.keep[u * RKEEP + k]);
  } else {
    scan_unit(a, i, (int)(u % a.nchunk), lane, put);
  }
}

}  // namespace

// Host side of steps 1-6.  ws: scratch views prepared by the caller.
int stiv_broad_phase(stiv_handle* h, cudaStream_t st, int n, int p_max, const int32_t* p_dev, const int64_t* voff,
                     const void* X, const stiv_pairs* cand, detect_ws& w, int64_t* ctr) {
  int mixed = h->prm.precision == STIV_MIXED;
  const double* L = h->prm.box_L;
  {
  STIV_PROF(h, st, "boxes");
  // per-vertex boxes in shared memory up to 96 KB (orders up to P = 44)
  size_t nv_max = (size_t)(w.fstride / 8);
  size_t vb_cap = 6 * nv_max * sizeof(float) <= VB_SMEM ? 6 * nv_max : 0;
  size_t bsmem = vb_cap * sizeof(float);
  auto bk = mixed ? boxes_kernel<true> : boxes_kernel<false>;
  STIV_SMEM(h, bk, bsmem, 4096, VB_SMEM);
  bk<<<n, BT, bsmem, st>>>(n, p_dev, voff, X, mixed, h->prm.d_m, L[0], L[1], L[2], w.vbox, w.pbox,
                                      w.pstride, w.vorg, w.fprep, w.fstride, ctr, vb_cap, p_max, w.fbox);
  }
  STIV_LAUNCH(h);
  if (n <= h->all_pairs) {
    rows_args a;
    a.n = n; a.nchunk = stiv_row_chunks(n); a.vbox = w.vbox; a.fbox = w.fbox;
    for (int c = 0; c < 3; ++c) a.L[c] = L[c];
    a.cnt = w.row_cnt; a.sum = w.row_sum; a.keep = w.row_keep;
    unsigned blocks = (unsigned)(((int64_t)n * a.nchunk + 7) / 8);
    STIV_PROF_N(h, st, "pairs", 2);
    row_pairs_kernel<<<blocks, 256, 0, st>>>(a);
    STIV_LAUNCH(h);
    emit_pairs_kernel<<<blocks, 256, 0, st>>>(a, cand->capacity, cand->i, cand->j, cand->shift, ctr);
    STIV_LAUNCH(h);
    return STIV_OK;
  }
  {
  STIV_PROF_N(h, st, "cells", 4);
  grid_kernel<<<1, 1024, 0, st>>>(n, w.vbox, L[0], L[1], L[2], w.grid);
  STIV_LAUNCH(h);
  cell_count_kernel<<<(n + 127) / 128, 128, 0, st>>>(n, w.vbox, w.grid, w.cell_count, ctr);
  STIV_LAUNCH(h);
  scan1_kernel<<<1, 1024, 0, st>>>(w.cell_count, n, w.cell_off);
  STIV_LAUNCH(h);
  cell_emit_kernel<<<(n + 127) / 128, 128, 0, st>>>(n, w.vbox, w.grid, w.cell_off, w.R, w.rec_key, w.rec_val,
                                                    w.rec_box, w.rec_cell, ctr);
  }
  STIV_LAUNCH(h);
  // records: ctr[8] = count; sort by Morton id (wrapped cells < 256 per axis: 24 bits)
  int rc;
  {
  STIV_PROF_N(h, st, "sort_cells", stiv_sort_kernels(24));
  rc = stiv_sort_pairs_impl(st, w.R, 24, w.rec_key, w.rec_val, w.rec_key2, w.rec_val2, w.rec_key, w.rec_val,
                            w.sort_scratch, w.sort_scratch_bytes, &ctr[8]);
  }
  // candidate keys i << (nb + 5) | j << 5 | shift code: nb bits per vesicle index
  int nb = 1;
  while ((1 << nb) < n) ++nb;
  int pair_bits = 2 * nb + 5;
  if (rc) return rc;
  {
  STIV_PROF(h, st, "cell_pairs");
  cell_pairs_kernel<<<(unsigned)((w.R + 127) / 128), 128, 0, st>>>(&ctr[8], w.R, w.rec_key2, w.rec_val2, w.rec_box,
                                                                   w.rec_cell, w.vbox, w.grid, L[0], L[1], L[2],
                                                                   w.Q, w.pkey, w.pval, ctr, nb);
  }
  STIV_LAUNCH(h);
  {
    STIV_PROF_N(h, st, "sort_pairs", stiv_sort_kernels(pair_bits));
    rc = stiv_sort_pairs_impl(st, w.Q, pair_bits, w.pkey, w.pval, w.pkey2, w.pval2, w.pkey3, w.pval3,
                              w.sort_scratch, w.sort_scratch_bytes, &ctr[9]);
  }
  if (rc) return rc;
  {
    STIV_PROF(h, st, "unique_pairs");
    unique_pairs_kernel<<<1, 1024, 0, st>>>(&ctr[9], w.Q, w.pkey2, cand->capacity, cand->i, cand->j, cand->shift,
                                            ctr, nb);
  }
  STIV_LAUNCH(h);
  return STIV_OK;
}
