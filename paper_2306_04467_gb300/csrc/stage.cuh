// Per-thread work of one S2O4 stage of the compact two-layer GKS
// (arXiv 2306.04467), shared by the CUDA kernels in gks2l.cu. Each function
// handles one unit of work (a cell-variable, an edge Gauss point of one layer,
// or a cell) and is written as plain host/device code so the arithmetic of a
// unit does not depend on the launch shape.
//
// Deviation form. Every instance carries two FP64 reference values, R2 (a
// depth of the upper layer) and R1 (a water level eta1 = h1 + B of the lower
// layer): the area-weighted means of the state when it was set, rounded to
// 2^-32. The kernels read and write only deviations from them, of type R
// (double in the FP64 form, float in the FP32 form): the cell mirrors
// dq = (h2 - R2, h2U2, h2V2, eta1 - R1, h1U1, h1V1) and gradients
// dg = grad(h2, h2U2, h2V2, h1, h1U1, h1V1), the state's own gradients (so a
// state read out and set again is the same bit for bit); the reconstruction
// sees grad eta1 = grad h1 + grad B of each cell. At rest (eta1 and h2 constant,
// Sec. 3.2) every deviation vanishes, so the well-balanced cancellation
// between the interface flux and the cell sources holds in any precision: the
// reference pressure G (R1 - B)^2 / 2 of the lower layer is integrated around
// the cell exactly (B is linear, 2-point Gauss is exact) and combined with the
// bottom source analytically, leaving -G (eta1_j - R1) grad B_j. FP64 is kept
// for the cell averages, the mass fluxes and the state update, which keeps
// each layer's mass exactly conserved.
#pragma once
#include <cmath>
#include <cstdint>
#include <cstring>

#ifndef __CUDACC__
#define __host__
#define __device__
#define __forceinline__ inline
#endif

namespace gks2l {

#ifndef __CUDACC__
using std::isfinite;
#endif

constexpr int NV = 6;        // h2, h2U2, h2V2, h1 (as eta1 = h1 + B), h1U1, h1V1
constexpr int NSLOT = 9;
constexpr int NCOL = 17;
constexpr int NCOEF = 10;    // per variable: c0 (value offset) + 9 Taylor coefficients
// Side record of one cell for one layer: three slots of 12 values, one per
// variable of the layer (level, x- and y-discharge), each the 10 deviation
// coefficients, the cell-average deviation, then a constant: 1/h_s in slot 0,
// the bottom slope in slots 1-2 (lower layer; zero in the upper). An edge
// point reads its layer's record and slot 0 (the level) of the other layer's.
// In memory the records of a tile of 32 cells are one block, vector by vector:
// [tile][layer][16-byte vector][cell in tile]. A warp of the edge kernels asks
// for the same vector of a few neighbouring cells at a time, so it finds
// several of them in a 128-byte line where a record of its own lies in two
// lines for itself: k_iface<float> 145 -> 123 us, k_edge<float> 333 -> 300 us
// (1.04 M triangles; the fused k_edgef, bound by issue, 287 -> 295 us).
constexpr int NREC = 36;

// Device view of the workspace. R-typed arrays are stored as void* and cast.
struct Dev {
  int nt, ne, ninst;
  int cs;                   // stride of per-cell arrays (nt rounded up to 32)
  // per cell
  const int *inst;
  const double *area, *dX;
  const void *hsR, *ihsR;   // sqrt|Omega| and its inverse, type R
  const void *epsA;         // weno_eps * |Omega|, type R
  const void *bgR;          // [cell][2] grad B, type R
  const double *bmean;
  const int *st_cell;
  const int8_t *st_xf;
  const int *tile_xf;       // per tile of 32 cells: whether any of its stencils has an image transform
  const void *ops;          // per tile of 32 cells: the reconstruction's operator rows
  const void *plane;        // [(f*2+d)][cell] plane operator, type R
  const int *cedge;         // [f][cell]: edge id, or ~edge when the cell is the R side
  const double *fsl;        // [f][cell]: sign * |Gamma| / |Omega| (double, mass sums)
  const void *fslR;         // the same, type R (the other residuals; fsl itself in the double form)
  const int *inst_first;
  double *avg;              // state averages [v][cell] (FP64)
  void *dq, *dg;            // deviation mirrors [pair][cell][2] and gradients [pair][cell][2][2], type R
  void *hrefc;              // R1 - B_j per cell, type R
  double *Wn, *Ln, *Ltn;    // W* between a step's stages (avg keeps W^n), and the stage-1 L and
                            // L_t (rows of the layer depths only, 0 and 3), FP64
  void *incR;               // [4][cell] stage-1 part of the stage-2 momentum increment, type R
  void *srec;               // side records [tile][layer][vector][32][16 bytes], type R (lower layer first)
  void *omg;                // omega_H / gamma_H of eta1 [0] and h2 [1], type R
  const void *mlp;          // gate network, packed image (MlpDev)
  unsigned *gate_mask;      // per tile of 32 cells: bit i = cell i takes the linear weights
  unsigned *gate_next;      // the gate's mask for the next reconstruction (k_update copies it over)
  // positivity option (not in the paper): per layer (0 lower, 1 upper) and
  // cell, whether the edge states' velocities are bounded, and the cell's
  // average depth
  unsigned char *pos_flag;  // [2][cs]
  void *pos_hbar;           // [2][cs], type R
                            // (written by one reconstruction for the next)
  float *wdev;              // [6][cell] max_k |omega_k / gamma_k - 1| (harvesting; scratch)
  // per edge
  // (one aligned vector for what a thread takes at once: an edge's results
  // were read by the update as 78 single values per cell, now as 30 vectors:
  // k_update<float> 38 -> 31 us at 181 k triangles, 158 -> 152 at 1.04 M)
  const int *eg;            // [edge][4] L cell, R cell, the R side's transform, instance
  const void *en;           // [edge][2] unit normal from L to R, type R
  const double *eb;         // [point][edge] B at the Gauss points
  const void *exi;          // [point][edge][4] Gauss point in the L and the R side's scaled frame, type R
  void *hrefe;              // [2][edge] R1 - B at the Gauss points, type R
  void *hc;                 // [2][edge] edge-centre blended level deviations, type R
  double *ept;              // [edge][layer][point][side][4] double form: the sides' level deviation, velocity
                            // along n and t, inverse root of the depth, from k_iface for k_edge (scratch)
  int *wl;                  // [2 * edge] (edge << 1 | layer) units left to the deferred edge pass (scratch)
  int *wl_count;            // their number (zeroed before each fused edge launch)
  // Gauss-point sums (weights 1/2), deviations, by layer (0 lower), type R but for eM
  void *eF;                 // [layer][edge][4] F (2), F_t (2) of the discharge
  double *eM;               // [layer][edge][2] F, F_t of the depth in FP64, converted once per
                            // edge for the cells' FP64 mass sums
  void *eWt, *eWn;          // [layer][edge][4] W_t and the stage-1 W^n (3, and one unused)
  void *eO;                 // [layer][edge][2] the L and the R side's own level deviation, mean
                            // over the two Gauss points (the interlayer source's point values)
  // per instance
  double *ref;              // [inst*2]: R2, R1
  void *refR;               // the same, type R
  double *dt, *t;
  void *dtR;                // [2][inst] dt and 1/dt (0 for a stopped instance), type R
  unsigned long long *dtbits;
  unsigned *ref_done;       // blocks of the reference-level reduction that have finished (wraps to 0)
  double *mass;             // [inst*2 + layer]
  int *status;
  unsigned long long *gate_count;
  const double *xf;         // [code*4] 2x2 linear parts of image transforms
};
// The kernels' next argument, Par, starts on 16 bytes, and its constants come by
// vector loads: at 8 bytes off k_edge<float> spills two of its 96 registers, 291 us in
// place of 283 (1.04 M triangles). Not by alignas, which has the compiler load the
// pointers themselves in pairs too: k_update<float> 886 us in place of 866 (8 M).
static_assert(sizeof(Dev) % 16 == 0, "an even number of pointers");

struct Par {
  double g, chi, cfl, eps, eps_num, gam_hi, weno_eps;
  float gf, chif, epsf, eps_numf, gam_hif;   // the same in single precision
  double ig2, rg, cphi;                      // 2/G, 1/sqrt(G), sqrt(G/(4 pi)): the double form's edge solution
  int use_gate;                              // learned gate active
  float *logit_out;                          // gate logits per cell (device order), or null
  int all_active;                            // reconstruct every instance (harvesting)
  int mask_now;                              // the gate writes the mask in use, not the next one
  int harvest;                               // record the weights' departure from linear
  int staging_polls;                         // > 0: operator staging polls at most this many - 1 times
  double pos_floor;                          // positivity option (not in the paper): 0 = off
};

// a parameter in the form's precision
template <typename R> __host__ __device__ __forceinline__ R pv(double d, float f);
template <> __host__ __device__ __forceinline__ double pv<double>(double d, float) { return d; }
template <> __host__ __device__ __forceinline__ float pv<float>(double, float f) { return f; }

// erf(x) of the single form given ex = e^{-x^2}, which the caller has formed
// already (the double form's is half_erf): the rational approximation 7.1.26 of Abramowitz
// and Stegun (Handbook of Mathematical Functions, after Hastings),
// erf(|x|) = 1 - P(t) e^{-x^2}, P(t) = a1 t + ... + a5 t^5, t = 1/(1 + p|x|),
// absolute error at most 1.5e-7, with P re-expanded about t = 1 in
// s = 1 - t = p|x| t: P = b0 + b1 s + ... + b5 s^5, b_m = (-1)^m sum_k
// C(k, m) a_k, and b0 (= sum a_k = 1 - 1e-9) taken as 1, a change far inside
// that bound. Then erf(|x|) = (1 - e^{-x^2}) - e^{-x^2} s (b1 + ... + b5 s^4)
// has no cancellation at small |x|: it is exact at zero and proportional to x
// for tiny x (relative error 6e-6, the approximation's own slope), so the tiny
// velocities of a state near rest keep their size in the half-space moments'
// erf terms, which enter the deviation h-bar - h_b directly.
template <typename R> __host__ __device__ __forceinline__ R erf_ex(R x, R ex);
template <> __host__ __device__ __forceinline__ float erf_ex<float>(float x, float ex) {
  const float ax = x < 0.f ? -x : x;
  const float t = 1.f / (1.f + 0.3275911f * ax);
  const float s = 0.3275911f * ax * t;
  float q = -1.061405429f;
  q = q * s + 3.853875118f;
  q = q * s - 6.222859923f;
  q = q * s + 5.874886615f;
  q = q * s - 3.44449638f;
  const float e = (1.f - ex) - ex * s * q;
  return x < 0.f ? -e : e;
}
template <typename R> __host__ __device__ __forceinline__ R r_exp(R x);
template <> __host__ __device__ __forceinline__ double r_exp<double>(double x) { return exp(x); }
// single precision on the device: the hardware exponential (a few ulp; the
// arguments here are O(1) Maxwellian exponents and -delta/tau)
template <> __host__ __device__ __forceinline__ float r_exp<float>(float x) {
#ifdef __CUDA_ARCH__
  return __expf(x);
#else
  return expf(x);
#endif
}
template <typename R> __host__ __device__ __forceinline__ R r_expm1(R x);
template <> __host__ __device__ __forceinline__ double r_expm1<double>(double x) { return expm1(x); }
template <> __host__ __device__ __forceinline__ float r_expm1<float>(float x) { return expm1f(x); }
template <typename R> __host__ __device__ __forceinline__ R r_sqrt(R x);
template <> __host__ __device__ __forceinline__ double r_sqrt<double>(double x) { return sqrt(x); }
template <> __host__ __device__ __forceinline__ float r_sqrt<float>(float x) { return sqrtf(x); }
__host__ __device__ __forceinline__ double r_rsqrt(double x) {
#ifdef __CUDA_ARCH__
  return rsqrt(x);
#else
  return 1 / sqrt(x);
#endif
}
template <typename R> __host__ __device__ __forceinline__ R r_abs(R x) { return x < 0 ? -x : x; }

// the bits of a double as a signed integer (> 0: positive, nonzero, and
// finite or NaN), and a finiteness test on them
__host__ __device__ __forceinline__ long long dbits(double x) {
#ifdef __CUDA_ARCH__
  return __double_as_longlong(x);
#else
  long long b;
  std::memcpy(&b, &x, sizeof b);
  return b;
#endif
}
// whether an instance is still advancing (its dt, zero once it has stopped), off the FP64 pipe
__host__ __device__ __forceinline__ bool running(const Dev &d, int inst) { return dbits(d.dt[inst]) > 0; }
__host__ __device__ __forceinline__ bool finite_bits(double x) { return ((dbits(x) >> 52) & 0x7ff) != 0x7ff; }

template <typename R>
__host__ __device__ __forceinline__ void monos(R x, R y, R m[10], R mx[10], R my[10]) {
  const R h = (R)0.5, s = (R)(1.0 / 6.0);
  R xx = x * x, yy = y * y, xy = x * y;
  const R one = (R)1, zero = (R)0;
  m[0] = one; m[1] = x; m[2] = y; m[3] = h * xx; m[4] = xy; m[5] = h * yy;
  m[6] = xx * x * s; m[7] = h * xx * y; m[8] = h * x * yy; m[9] = yy * y * s;
  mx[0] = zero; mx[1] = one; mx[2] = zero; mx[3] = x; mx[4] = y; mx[5] = zero;
  mx[6] = h * xx; mx[7] = xy; mx[8] = h * yy; mx[9] = zero;
  my[0] = zero; my[1] = zero; my[2] = one; my[3] = zero; my[4] = x; my[5] = y;
  my[6] = zero; my[7] = h * xx; my[8] = xy; my[9] = h * yy;
}

template <typename R>
__host__ __device__ __forceinline__ void rot2(const double *M, R v[2]) {
  R a = v[0], b = v[1];
  v[0] = (R)M[0] * a + (R)M[1] * b;
  v[1] = (R)M[2] * a + (R)M[3] * b;
}

// ------------------------------------------------------------------ cell data
// The mirrors hold the variables in pairs, the levels (h2, eta1) and the two
// layers' discharges (x, y): a thread that works on a pair gathers a cell's
// two deviations by one load and their gradients by another, and a mirrored
// discharge or its gradient tensor is at hand whole.
constexpr int NPAIR = 3;
__host__ __device__ __forceinline__ int pair_of(int v) { return v == 0 || v == 3 ? 0 : (v < 3 ? 1 : 2); }
__host__ __device__ __forceinline__ int comp_of(int v) { return v == 0 || v == 3 ? v / 3 : (v < 3 ? v - 1 : v - 4); }
__host__ __device__ __forceinline__ int var_of(int pair, int comp) {
  return pair == 0 ? 3 * comp : (pair == 1 ? 1 : 4) + comp;
}
// n consecutive values (n * sizeof(R) a multiple of their 8- or 16-byte load)
template <typename R, int n> __host__ __device__ __forceinline__ void load_n(const R *p, R *w) {
  for (int i = 0; i < n; i++) w[i] = p[i];
}
template <typename R, int n> __host__ __device__ __forceinline__ void store_n(R *p, const R *w) {
  for (int i = 0; i < n; i++) p[i] = w[i];
}
#ifdef __CUDACC__
template <> __device__ __forceinline__ void load_n<float, 2>(const float *p, float *w) {
  const float2 t = *reinterpret_cast<const float2 *>(p);
  w[0] = t.x; w[1] = t.y;
}
template <> __device__ __forceinline__ void load_n<float, 4>(const float *p, float *w) {
  const float4 t = *reinterpret_cast<const float4 *>(p);
  w[0] = t.x; w[1] = t.y; w[2] = t.z; w[3] = t.w;
}
template <> __device__ __forceinline__ void load_n<double, 2>(const double *p, double *w) {
  const double2 t = *reinterpret_cast<const double2 *>(p);
  w[0] = t.x; w[1] = t.y;
}
template <> __device__ __forceinline__ void load_n<double, 4>(const double *p, double *w) {
  load_n<double, 2>(p, w);
  load_n<double, 2>(p + 2, w + 2);
}
template <> __device__ __forceinline__ void store_n<float, 2>(float *p, const float *w) {
  *reinterpret_cast<float2 *>(p) = make_float2(w[0], w[1]);
}
template <> __device__ __forceinline__ void store_n<float, 4>(float *p, const float *w) {
  *reinterpret_cast<float4 *>(p) = make_float4(w[0], w[1], w[2], w[3]);
}
template <> __device__ __forceinline__ void store_n<double, 2>(double *p, const double *w) {
  *reinterpret_cast<double2 *>(p) = make_double2(w[0], w[1]);
}
template <> __device__ __forceinline__ void store_n<double, 4>(double *p, const double *w) {
  store_n<double, 2>(p, w);
  store_n<double, 2>(p + 2, w + 2);
}
#endif
template <typename R> __host__ __device__ __forceinline__ R *dq_at(const Dev &d, int pair, int c) {
  return (R *)d.dq + ((size_t)pair * d.cs + c) * 2;
}
template <typename R> __host__ __device__ __forceinline__ R *dg_at(const Dev &d, int pair, int c) {
  return (R *)d.dg + ((size_t)pair * d.cs + c) * 4;
}

// A pair's deviations (q) and gradients (g: of the first, then the second, the
// level eta1's as stored plus the cell's grad B) seen through transform xf.
template <typename R>
__host__ __device__ __forceinline__ void image_q(const Dev &d, int pair, int xf, R q[2]) {
  if (pair != 0 && xf != 0) rot2<R>(d.xf + 4 * xf, q);
}
template <typename R>
__host__ __device__ __forceinline__ void load_g(const Dev &d, int pair, int c, R g[4]) {
  load_n<R, 4>(dg_at<R>(d, pair, c), g);
  if (pair == 0) {
    R b[2];
    load_n<R, 2>((const R *)d.bgR + 2 * (size_t)c, b);
    g[2] += b[0];
    g[3] += b[1];
  }
}
template <typename R>
__host__ __device__ __forceinline__ void image_g(const Dev &d, int pair, int xf, R g[4]) {
  if (xf == 0) return;
  const double *M = d.xf + 4 * xf;
  if (pair == 0) {
    rot2<R>(M, g);
    rot2<R>(M, g + 2);
    return;
  }
  // discharge gradient tensor T_ik = d m_i / d x_k -> M T M^T
  const R T[2][2] = {{g[0], g[1]}, {g[2], g[3]}};
  for (int row = 0; row < 2; row++)
    for (int k = 0; k < 2; k++) {
      R s = 0;
      for (int a = 0; a < 2; a++)
        for (int b2 = 0; b2 < 2; b2++) s += (R)M[2 * row + a] * T[a][b2] * (R)M[2 * k + b2];
      g[2 * row + k] = s;
    }
}

// --------------------------------------------------- compact reconstruction
// Operator rows of one cell: element k of row r is at base[r * stride + idx]
// (a tile staged in shared memory: stride = tile width, idx = cell in the tile).
template <typename R> struct CellOps {
  const R *lsq, *p1, *bq, *mm;
  int stride, idx;
};

// One cell and VP variables, a pair (VP = 2) or one of it (VP = 1, comp): P3
// least squares (Eq. Recons-system), three P1 candidates on {cell, face
// neighbour}, smoothness indicators and WENO-Z weights, combined polynomial
// written as deviations in the Taylor basis. Three steps: gather the
// right-hand side, solve the P3 fit, then combine (where the troubled-cell
// gate can choose the linear weights).

// right-hand side: stencil average differences, then h-scaled gradients of
// the cell and its three face neighbours. st: the stencil's cells (-1: none);
// xfs: whether any stencil of the tile is seen through a transform. With VP = 2
// also the averages (nq) and gradients (g) of the cell and its face neighbours
// themselves, for the gate's features
template <typename R>
__host__ __device__ __forceinline__ void gather_one(const Dev &d, int j, int pair, int comp, const int st[NSLOT],
                                                    bool xfs, R rhs[NCOL], R &q0) {
  q0 = dq_at<R>(d, pair, j)[comp];
  const R hs = ((const R *)d.hsR)[j];
#pragma unroll
  for (int s = 0; s < NSLOT; s++) {
    const int c = st[s] >= 0 ? st[s] : j;
    R t = dq_at<R>(d, pair, c)[comp];
    const int xf = xfs && pair != 0 ? d.st_xf[(size_t)s * d.cs + j] : 0;
    if (xf != 0) {
      R m[2];
      load_n<R, 2>(dq_at<R>(d, pair, c), m);
      image_q<R>(d, pair, xf, m);
      t = comp == 0 ? m[0] : m[1];
    }
    rhs[s] = st[s] >= 0 ? t - q0 : (R)0;
  }
#pragma unroll
  for (int m = 0; m < 4; m++) {
    const int c = m == 0 ? j : st[m - 1];
    R g[2];
    load_n<R, 2>(dg_at<R>(d, pair, c) + 2 * comp, g);
    if (pair == 0 && comp == 1) {
      R b[2];
      load_n<R, 2>((const R *)d.bgR + 2 * (size_t)c, b);
      g[0] += b[0];
      g[1] += b[1];
    }
    const int xf = xfs && m > 0 ? d.st_xf[(size_t)(m - 1) * d.cs + j] : 0;
    if (xf != 0) {
      if (pair == 0) {
        rot2<R>(d.xf + 4 * xf, g);
      } else {
        R T[4];
        load_n<R, 4>(dg_at<R>(d, pair, c), T);
        image_g<R>(d, pair, xf, T);
        g[0] = comp == 0 ? T[0] : T[2];
        g[1] = comp == 0 ? T[1] : T[3];
      }
    }
    rhs[9 + 2 * m] = hs * g[0];
    rhs[10 + 2 * m] = hs * g[1];
  }
}
template <typename R, int VP>
__host__ __device__ __forceinline__ void recon_gather(const Dev &d, int j, int pair, int comp, const int st[NSLOT],
                                                      bool xfs, R rhs[VP][NCOL], R q0[VP], R nq[4][2], R g[4][4]) {
  if (VP == 1) {
    gather_one<R>(d, j, pair, comp, st, xfs, rhs[0], q0[0]);
    return;
  }
  R q[2], t[NSLOT][2];
  load_n<R, 2>(dq_at<R>(d, pair, j), q);
#pragma unroll
  for (int s = 0; s < NSLOT; s++) load_n<R, 2>(dq_at<R>(d, pair, st[s] >= 0 ? st[s] : j), t[s]);
  load_g<R>(d, pair, j, g[0]);
#pragma unroll
  for (int f = 0; f < 3; f++) load_g<R>(d, pair, st[f], g[1 + f]);
  const R hs = ((const R *)d.hsR)[j];
  if (xfs) {
#pragma unroll
    for (int s = 0; s < NSLOT; s++) {
      const int xf = d.st_xf[(size_t)s * d.cs + j];
      image_q<R>(d, pair, xf, t[s]);
      if (s < 3) image_g<R>(d, pair, xf, g[1 + s]);
    }
  }
  for (int i = 0; i < 2; i++) {
    nq[0][i] = q[i];
    for (int f = 0; f < 3; f++) nq[1 + f][i] = t[f][i];
  }
#pragma unroll
  for (int i = 0; i < VP; i++) {
    q0[i] = q[i];
#pragma unroll
    for (int s = 0; s < NSLOT; s++) rhs[i][s] = st[s] >= 0 ? t[s][i] - q0[i] : (R)0;
#pragma unroll
    for (int m = 0; m < 4; m++) {
      rhs[i][9 + 2 * m] = hs * g[m][2 * i];
      rhs[i][10 + 2 * m] = hs * g[m][2 * i + 1];
    }
  }
}

// P3 least-squares coefficients a = M rhs; each operator entry is read once
// for the thread's variables
template <typename R, int VP>
__host__ __device__ __forceinline__ void recon_p3(const CellOps<R> &o, const R rhs[VP][NCOL], R a[VP][9]) {
  const int S = o.stride, I = o.idx;
#pragma unroll
  for (int r = 0; r < 9; r++) {
    R s[VP] = {};
#pragma unroll
    for (int c = 0; c < NCOL; c++) {
      const R m = o.lsq[(r * NCOL + c) * S + I];
      for (int i = 0; i < VP; i++) s[i] += m * rhs[i][c];
    }
    for (int i = 0; i < VP; i++) a[i][r] = s[i];
  }
}

// t / a and t / b from one reciprocal (in FP64 5 pipe slots against 8 for each
// division), or by division where the product a b leaves the normal range
template <typename R>
__host__ __device__ __forceinline__ void ratios2(R t, R a, R b, R r[2]) {
  const R ab = a * b;
  // 2^-960 <= ab < 2^960 by the exponent's bits (off the FP64 pipe)
  const int ex = (int)((dbits((double)ab) >> 52) & 0x7ff);
  if (ex > 63 && ex < 1983) {
    const R i = t * ((R)1 / ab);
    r[0] = i * b;
    r[1] = i * a;
  } else {
    r[0] = t / a;
    r[1] = t / b;
  }
}

// The variables' slots of the side records (12 values each, see NREC).
template <typename R, int VP>
__host__ __device__ __forceinline__ void recon_finish(const Dev &d, const Par &p, const CellOps<R> &o, int j, int pair,
                                                      int comp, const R rhs[VP][NCOL], const R a[VP][9],
                                                      const R q0[VP], bool linear, R rec[VP][12]) {
  const int N = d.cs, S = o.stride, I = o.idx;
  const R gh = pv<R>(p.gam_hi, p.gam_hif), gl = ((R)1 - gh) * (R)(1.0 / 3.0);
  R fac[VP], wf[VP][3], b[VP][3][2];
  for (int i = 0; i < VP; i++) {
    fac[i] = 1;
    for (int f = 0; f < 3; f++) {
      wf[i][f] = gl;
      b[i][f][0] = b[i][f][1] = 0;
    }
  }
  if (!linear) {
    R beta[VP][4], bh[VP] = {};
#pragma unroll
    for (int f = 0; f < 3; f++) {
#pragma unroll
      for (int k = 0; k < 2; k++) {
        R s[VP] = {};
#pragma unroll
        for (int c = 0; c < 5; c++) {
          const R m = o.p1[((f * 2 + k) * 5 + c) * S + I];
          const int col = c == 0 ? f : (c < 3 ? 8 + c : 8 + 2 * f + c);
          for (int i = 0; i < VP; i++) s[i] += m * rhs[i][col];
        }
        for (int i = 0; i < VP; i++) b[i][f][k] = s[i];
      }
      for (int i = 0; i < VP; i++) beta[i][1 + f] = b[i][f][0] * b[i][f][0] + b[i][f][1] * b[i][f][1];
    }
    int idx = 0;
#pragma unroll
    for (int k = 0; k < 9; k++) {
      R row[VP] = {};
#pragma unroll
      for (int l = k; l < 9; l++) {
        const R m = o.bq[(idx++) * S + I];
        for (int i = 0; i < VP; i++) {
          // double form: a_k times the row's sum, 54 operations in place of 90
          // (with the weights' shared reciprocals k_recon<double> goes from
          // 404 to 344 FP64 operations per cell and variable, 2224 -> 1897 us
          // at 501 k triangles)
          if (sizeof(R) == 8) row[i] += m * a[i][l];
          else bh[i] += m * a[i][k] * a[i][l];
        }
      }
      if (sizeof(R) == 8)
        for (int i = 0; i < VP; i++) bh[i] += a[i][k] * row[i];
    }
    const R gam[4] = {gh, gl, gl, gl};
    const R epsA = ((const R *)d.epsA)[j];
    const int in = d.inst[j];
#pragma unroll
    for (int i = 0; i < VP; i++) {
      const int c = VP == 2 ? i : comp;
      beta[i][0] = bh[i];
      R tz = (r_abs<R>(bh[i] - beta[i][1]) + r_abs<R>(bh[i] - beta[i][2]) + r_abs<R>(bh[i] - beta[i][3])) *
             (R)(1.0 / 3.0);
      // the variable's value (reference + deviation) scales the regulariser
      R Q0 = q0[i];
      if (pair == 0) Q0 += ((const R *)d.refR)[2 * in + c];
      R eps = epsA * (1 + Q0 * Q0);
      if (sizeof(R) == 8) {
        R u[4], ws = 0;
        for (int k = 0; k < 4; k += 2) {
          R r[2];
          ratios2<R>(tz, beta[i][k] + eps, beta[i][k + 1] + eps, r);
          for (int m = 0; m < 2; m++) {
            u[k + m] = 1 + r[m] * r[m];
            ws += gam[k + m] * u[k + m];
          }
        }
        const R iw = 1 / ws;
        fac[i] = u[0] * iw;
        for (int f = 0; f < 3; f++) wf[i][f] = u[1 + f] * (gl * iw);
      } else {
        R w[4], ws = 0;
        for (int k = 0; k < 4; k++) {
          R r = tz / (beta[i][k] + eps);
          w[k] = gam[k] * (1 + r * r);
          ws += w[k];
        }
        R iw = 1 / ws;
        fac[i] = w[0] * iw / gh;
        for (int f = 0; f < 3; f++) wf[i][f] = w[1 + f] * iw;
      }
      if (p.harvest) {
        R dv = r_abs<R>(fac[i] - 1);
        for (int f = 0; f < 3; f++) {
          R df = r_abs<R>(wf[i][f] / gl - 1);
          dv = df > dv ? df : dv;
        }
        d.wdev[(size_t)var_of(pair, c) * N + j] = (float)dv;
      }
    }
  } else if (p.harvest) {
    for (int i = 0; i < VP; i++) d.wdev[(size_t)var_of(pair, VP == 2 ? i : comp) * N + j] = 0.f;
  }
  // R = (w_H / g_H)(P3 - sum g_m P1_m) + sum w_m P1_m
#pragma unroll
  for (int i = 0; i < VP; i++) {
    R *r = rec[i];
    for (int k = 1; k < 10; k++) r[k] = fac[i] * a[i][k - 1];
    for (int f = 0; f < 3; f++) {
      R cf = wf[i][f] - fac[i] * gl;
      r[1] += cf * b[i][f][0];
      r[2] += cf * b[i][f][1];
    }
    r[0] = 0;
    r[10] = q0[i];
    // omega_H / gamma_H of eta1, then of h2
    if (pair == 0) ((R *)d.omg)[(size_t)((VP == 2 ? i : comp) == 1 ? 0 : N) + j] = fac[i];
  }
#pragma unroll
  for (int k = 3; k < 10; k++) {
    const R m = o.mm[(k - 3) * S + I];
    for (int i = 0; i < VP; i++) rec[i][0] -= rec[i][k] * m;
  }
  // the slots' constants: 1/h_s with the level, the bottom slope with the
  // lower layer's discharges
  if (pair == 0) {
    const R ih = ((const R *)d.ihsR)[j];
    for (int i = 0; i < VP; i++) rec[i][11] = ih;
  } else {
    R g[2] = {0, 0};
    if (pair == 2) load_n<R, 2>((const R *)d.bgR + 2 * (size_t)j, g);
    for (int i = 0; i < VP; i++) rec[i][11] = (VP == 2 ? i : comp) == 0 ? g[0] : g[1];
  }
}
// layer (0 lower) and slot of a variable's part of the side records
__host__ __device__ __forceinline__ int slot_of(int pair, int comp, int &layer) {
  layer = pair == 0 ? 1 - comp : (pair == 2 ? 0 : 1);
  return pair == 0 ? 0 : 1 + comp;
}

// ------------------------------------------------- evaluation at an edge point
// Edge-point side data for layer ell (0: lower, reconstructed eta1; 1: upper),
// all deviations of type R.
template <typename R> struct SideVals {
  R d;            // level deviation at the point (eta1 - R1 or h2 - R2)
  R h;            // depth at the point (href + d)
  R mx, my;       // discharge
  R gh[2];        // gradient of the depth
  R glev[2];      // gradient of the level variable
  R gm[2][2];     // discharge gradient tensor d m_i / d x_k
  R goth[2];      // gradient of the other layer's level variable
};

// cell c's reconstruction at scaled point (x, y), seen through transform xf;
// href is the depth of the reference level at the point
// the first n values (a multiple of 12) of cell c's side record of layer ell
constexpr int RTILE = 32;    // cells per tile of the side records
template <typename R, int n>
__host__ __device__ __forceinline__ void load_rec(const Dev &d, int ell, int c, R *w) {
  constexpr int V = 16 / sizeof(R);   // values per vector
  const R *p = (const R *)d.srec + ((size_t)((unsigned)c / RTILE) * 2 + ell) * (NREC * RTILE) + ((unsigned)c % RTILE) * V;
#pragma unroll
  for (int k = 0; k < n / V; k++) {
#ifdef __CUDA_ARCH__
    const uint4 t = *reinterpret_cast<const uint4 *>(p + k * RTILE * V);
    *reinterpret_cast<uint4 *>(w + k * V) = t;
#else
    for (int i = 0; i < V; i++) w[k * V + i] = p[k * RTILE * V + i];
#endif
  }
}

// Operations rounded as written, whatever the compiler does with the code
// around them: where two kernels must form the same value bit for bit.
template <typename R> struct Rn;
template <> struct Rn<float> {
#ifdef __CUDA_ARCH__
  static __device__ __forceinline__ float mul(float a, float b) { return __fmul_rn(a, b); }
  static __device__ __forceinline__ float add(float a, float b) { return __fadd_rn(a, b); }
  static __device__ __forceinline__ float sub(float a, float b) { return __fsub_rn(a, b); }
  static __device__ __forceinline__ float fma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
  static __device__ __forceinline__ float rcp(float a) { return __frcp_rn(a); }
#else
  static float mul(float a, float b) { return a * b; }
  static float add(float a, float b) { return a + b; }
  static float sub(float a, float b) { return a - b; }
  static float fma(float a, float b, float c) { return std::fma(a, b, c); }
  static float rcp(float a) { return 1.0f / a; }
#endif
};
template <> struct Rn<double> {
#ifdef __CUDA_ARCH__
  static __device__ __forceinline__ double mul(double a, double b) { return __dmul_rn(a, b); }
  static __device__ __forceinline__ double add(double a, double b) { return __dadd_rn(a, b); }
  static __device__ __forceinline__ double sub(double a, double b) { return __dsub_rn(a, b); }
  static __device__ __forceinline__ double fma(double a, double b, double c) { return __fma_rn(a, b, c); }
#else
  static double mul(double a, double b) { return a * b; }
  static double add(double a, double b) { return a + b; }
  static double sub(double a, double b) { return a - b; }
  static double fma(double a, double b, double c) { return std::fma(a, b, c); }
#endif
};

// gradient (scaled by ih) of the level polynomial cf at a point's monomial
// derivatives, explicitly rounded: the edge kernels take the other layer's
// level gradient from the lane that formed it as its own, the deferred edge
// pass forms it again, and both get the same bits
template <typename R>
__host__ __device__ __forceinline__ void level_grad(const R *cf, const R mx[10], const R my[10], R ih, R g[2]) {
  using O = Rn<R>;
  R ax = cf[1], ay = cf[2];
  for (int k : {3, 4, 6, 7, 8}) ax = O::fma(cf[k], mx[k], ax);
  for (int k : {4, 5, 7, 8, 9}) ay = O::fma(cf[k], my[k], ay);
  g[0] = O::mul(ax, ih);
  g[1] = O::mul(ay, ih);
}
// 2x2 rotation, explicitly rounded (for the level gradients above)
template <typename R>
__host__ __device__ __forceinline__ void rot2_rn(const double *M, R v[2]) {
  using O = Rn<R>;
  const R a = v[0], b = v[1];
  v[0] = O::fma((R)M[1], b, O::mul((R)M[0], a));
  v[1] = O::fma((R)M[3], b, O::mul((R)M[2], a));
}

// One side of an edge point: cell c's reconstruction of layer ell at scaled
// point (x, y), seen through transform xf; href is the depth of the
// reference level at the point. OTHER: also form the gradient of the other
// layer's level from its record (otherwise the caller takes it from the lane
// that forms it as its own).
template <typename R, bool OTHER = true>
__host__ __device__ inline void side_vals(const Dev &d, int ell, int c, int xf, R x, R y, R href, SideVals<R> &s) {
  R w[NREC];
  load_rec<R, NREC>(d, ell, c, w);
  R m[10], mx[10], my[10];
  monos<R>(x, y, m, mx, my);
  const R ih = w[11];
  R dev[3], gx[3], gy[3];
  for (int i = 0; i < 3; i++) {
    const R *cf = w + 12 * i;
    R a = cf[0] * m[0];
    for (int k = 1; k < 10; k++) a += cf[k] * m[k];
    dev[i] = a;
    if (i == 0) {
      R g[2];
      level_grad<R>(cf, mx, my, ih, g);
      gx[0] = g[0];
      gy[0] = g[1];
    } else {
      R ax = cf[1] * mx[1], ay = cf[2] * my[2];
      for (int k : {3, 4, 6, 7, 8}) ax += cf[k] * mx[k];
      for (int k : {4, 5, 7, 8, 9}) ay += cf[k] * my[k];
      gx[i] = ax * ih;
      gy[i] = ay * ih;
    }
  }
  s.goth[0] = s.goth[1] = 0;
  if (OTHER) {
    R wo[12];
    load_rec<R, 12>(d, 1 - ell, c, wo);
    level_grad<R>(wo, mx, my, ih, s.goth);
  }
  s.d = w[10] + dev[0];
  s.h = href + s.d;
  s.mx = w[22] + dev[1];
  s.my = w[34] + dev[2];
  s.glev[0] = gx[0]; s.glev[1] = gy[0];
  s.gm[0][0] = gx[1]; s.gm[0][1] = gy[1];
  s.gm[1][0] = gx[2]; s.gm[1][1] = gy[2];
  R gb[2] = {0, 0};
  if (ell == 0) { gb[0] = w[23]; gb[1] = w[35]; }
  if (xf != 0) {
    const double *M = d.xf + 4 * xf;
    R mv[2] = {s.mx, s.my};
    rot2<R>(M, mv);
    s.mx = mv[0]; s.my = mv[1];
    rot2_rn<R>(M, s.glev);
    if (OTHER) rot2_rn<R>(M, s.goth);
    rot2<R>(M, gb);
    R G2[2][2] = {{s.gm[0][0], s.gm[0][1]}, {s.gm[1][0], s.gm[1][1]}};
    for (int i2 = 0; i2 < 2; i2++)
      for (int k = 0; k < 2; k++) {
        R acc = (R)M[2 * i2] * G2[0][0] * (R)M[2 * k] + (R)M[2 * i2] * G2[0][1] * (R)M[2 * k + 1];
        acc += (R)M[2 * i2 + 1] * G2[1][0] * (R)M[2 * k];
        acc += (R)M[2 * i2 + 1] * G2[1][1] * (R)M[2 * k + 1];
        s.gm[i2][k] = acc;
      }
  }
  s.gh[0] = s.glev[0] - gb[0];   // depth = level - B for the lower layer
  s.gh[1] = s.glev[1] - gb[1];
}

// the level deviation and the discharges at scaled point (x, y) from a
// loaded side record
template <typename R>
__host__ __device__ __forceinline__ void rec_values(const R *w, R x, R y, R v[3]) {
  const R hh = (R)0.5, s6 = (R)(1.0 / 6.0);
  const R xx = x * x, yy = y * y, xy = x * y;
  const R m[10] = {(R)1, x, y, hh * xx, xy, hh * yy, xx * x * s6, hh * xx * y, hh * x * yy, yy * y * s6};
  for (int i = 0; i < 3; i++) {
    R a = w[12 * i] * m[0];
    for (int k = 1; k < 10; k++) a += w[12 * i + k] * m[k];
    v[i] = w[12 * i + 10] + a;
  }
}

// depth of the reference level at Gauss point q of edge e for layer ell
template <typename R>
__host__ __device__ __forceinline__ R ref_depth(const Dev &d, int ell, int e, int q) {
  if (ell == 0) return ((const R *)d.hrefe)[q * d.ne + e];
  return ((const R *)d.refR)[2 * d.eg[4 * (size_t)e + 3]];
}

// an edge's cells, transform and instance
struct EdgeIds {
  int L, R, xf, inst;
};
__host__ __device__ __forceinline__ EdgeIds edge_ids(const Dev &d, int e) {
#ifdef __CUDA_ARCH__
  const int4 t = reinterpret_cast<const int4 *>(d.eg)[e];
  return {t.x, t.y, t.z, t.w};
#else
  const int *p = d.eg + 4 * (size_t)e;
  return {p[0], p[1], p[2], p[3]};
#endif
}

// ------------------------------------------------ gas-kinetic interface solution
template <typename R> struct Kern {
  R gu, gv, puu, puv, pvv, bu, bv;
};

// Central moments mu_k = <c^k> (k = 0..5, c = u - U) of the normalised 1-D
// Maxwellian over the half line sgn*u > 0, from E = e^{-lam U^2}/(2 sqrt(pi lam))
// (formed by the caller); e0 = mu_0 - 1/2.
template <typename R>
__host__ __device__ __forceinline__ void half_moments_E(R U, R lam, R sgn, R E, R ex, R mu[6], R &e0) {
  const R th = (R)0.5 / lam;
  e0 = sgn * (R)0.5 * erf_ex<R>(r_sqrt<R>(lam) * U, ex);   // ex = e^{-lam U^2}
  mu[0] = (R)0.5 + e0;
  mu[1] = sgn * E;
  R pw = -sgn * U * E;
  mu[2] = th * mu[0] + pw;
  pw *= -U;
  mu[3] = 2 * th * mu[1] + pw;
  pw *= -U;
  mu[4] = 3 * th * mu[2] + pw;
  pw *= -U;
  mu[5] = 4 * th * mu[3] + pw;
}

// both half lines of one Maxwellian (sgn = +1 into mp, -1 into mm), sharing
// its error function and exponential
template <typename R>
__host__ __device__ __forceinline__ void half_moments_pm(R U, R lam, R mp[6], R mm[6]) {
  const R th = (R)0.5 / lam;
  const R ex = r_exp<R>(-lam * U * U);
  const R e0 = (R)0.5 * erf_ex<R>(r_sqrt<R>(lam) * U, ex);
  const R E = ex * (R)0.5 / r_sqrt<R>((R)3.14159265358979323846 * lam);
  for (int sg = 0; sg < 2; sg++) {
    const R sgn = sg == 0 ? (R)1 : (R)-1;
    R *mu = sg == 0 ? mp : mm;
    mu[0] = (R)0.5 + sgn * e0;
    mu[1] = sgn * E;
    R pw = -sgn * U * E;
    mu[2] = th * mu[0] + pw;
    pw *= -U;
    mu[3] = 2 * th * mu[1] + pw;
    pw *= -U;
    mu[4] = 3 * th * mu[2] + pw;
    pw *= -U;
    mu[5] = 4 * th * mu[3] + pw;
  }
}

// Slope + force kernel on a Maxwellian base (h, U, V, lam), written as a
// polynomial in c = u - U: the exact derivative of ln g along n and t, plus
// the force term, whose cubic part combines into (lam/h) |c|^2 (D . c) with
// D = grad h - grad Phi / G (local frame).
template <typename R>
__host__ __device__ __forceinline__ Kern<R> make_kern(R h, R U, R V, R lam, const R dn[3], const R dt[3],
                                                      const R D[2]) {
  Kern<R> K;
  R ih = 1 / h;
  R aun = (dn[1] - U * dn[0]) * ih, avn = (dn[2] - V * dn[0]) * ih;
  R aut = (dt[1] - U * dt[0]) * ih, avt = (dt[2] - V * dt[0]) * ih;
  R al = lam * ih * (dn[0] * U + dt[0] * V);
  R tl = 2 * lam;
  K.gu = tl * (aun * U + aut * V);
  K.gv = tl * (avn * U + avt * V);
  K.puu = al + tl * aun;
  K.pvv = al + tl * avt;
  K.puv = tl * (avn + aut);
  K.bu = lam * ih * D[0];
  K.bv = lam * ih * D[1];
  return K;
}

// moments of the kernel with weights (1, u, v) and (u, u^2, uv), per unit density
template <typename R>
__host__ __device__ __forceinline__ void kern_moments(const Kern<R> &K, const R mu[6], R th, R U, R V, R out[6]) {
  const R n2 = th, n4 = 3 * th * th;
  R T00 = K.gu * mu[1] + K.puu * mu[2] + K.pvv * mu[0] * n2 + K.bu * (mu[3] + mu[1] * n2);
  R T10 = K.gu * mu[2] + K.puu * mu[3] + K.pvv * mu[1] * n2 + K.bu * (mu[4] + mu[2] * n2);
  R T20 = K.gu * mu[3] + K.puu * mu[4] + K.pvv * mu[2] * n2 + K.bu * (mu[5] + mu[3] * n2);
  R T01 = K.gv * mu[0] * n2 + K.puv * mu[1] * n2 + K.bv * (mu[2] * n2 + mu[0] * n4);
  R T11 = K.gv * mu[1] * n2 + K.puv * mu[2] * n2 + K.bv * (mu[3] * n2 + mu[1] * n4);
  out[0] = T00;
  out[1] = U * T00 + T10;
  out[2] = V * T00 + T01;
  out[3] = out[1];
  out[4] = U * U * T00 + 2 * U * T10 + T20;
  out[5] = U * V * T00 + V * T10 + U * T01 + T11;
}

// time integrals over [0, delta] of C1..C5, from e = exp(-delta/tau) and
// em = 1 - e
template <typename R>
__host__ __device__ __forceinline__ void time_ints_e(R tau, R delta, R e, R em, R q[5]) {
  q[0] = delta - tau * em;
  q[1] = -tau * delta * (1 + e) + 2 * tau * tau * em;
  q[2] = (R)0.5 * delta * delta - tau * delta + tau * tau * em;
  q[3] = tau * em;
  q[4] = tau * delta * e - tau * tau * em;
}
// the same over [0, delta] (qd) and [0, delta / 2] (qh); the full interval's
// exponentials follow from the half interval's: e = eh^2, 1 - e = emh (1 + eh)
template <typename R>
__host__ __device__ __forceinline__ void time_ints2(R tau, R delta, R qd[5], R qh[5]) {
  const R xh = (R)0.5 * delta / tau;
  const R emh = -r_expm1<R>(-xh), eh = r_exp<R>(-xh);
  time_ints_e<R>(tau, (R)0.5 * delta, eh, emh, qh);
  time_ints_e<R>(tau, delta, eh * eh, emh * (1 + eh), qd);
}

// One layer at one Gauss point in the single form, local frame (x along the normal from L to R).
// Depths h_l = href + dl, h_r = href + dr. Returns the value and time
// derivative at the stage start of the flux F and of the interface variables
// W (fit of the two time integrals over delta and delta/2), as deviations:
// the normal-momentum flux minus G href^2 / 2 and the depth minus href.
template <typename R>
__host__ __device__ inline void gks_layer(R href, R dl, R dr, R Ul, R Vl, R Ur, R Vr, const R dnl[3],
                                          const R dtl[3], const R Dl[2], const R dnr[3], const R dtr[3],
                                          const R Dr[2], R g, R tau, R delta, R F[3], R Ft[3], R W[3], R Wt[3]) {
  static_assert(sizeof(R) == 4, "the double form's is gks_layer64");
  const R hlR = href + dl, hrR = href + dr;
  const R dlr = dl - dr;                          // h_l - h_r, exact at rest
  const R laml = 1 / (g * hlR), lamr = 1 / (g * hrR);
  const R thl = (R)0.5 * g * hlR, thr = (R)0.5 * g * hrR;
  // E = e^{-lam U^2} / (2 sqrt(pi lam)) = sqrt(G/(4 pi)) sqrt(h) e^{-lam U^2}
  // on each side: one exponential and one square root serve the half-space
  // moments and the depth-difference term below
  const R xl = r_exp<R>(-laml * Ul * Ul), xr = r_exp<R>(-lamr * Ur * Ur);
  const R sl = r_sqrt<R>(hlR), sr = r_sqrt<R>(hrR);
  const R cphi = r_sqrt<R>(g * (R)(0.25 / 3.14159265358979323846));
  const R El = cphi * sl * xl, Er = cphi * sr * xr;
  R mul[6], mur[6], e0l, e0r;
  half_moments_E<R>(Ul, laml, (R)1, El, xl, mul, e0l);
  half_moments_E<R>(Ur, lamr, (R)-1, Er, xr, mur, e0r);
  // W-bar: the t = 0 interface state; h_b = (h_l + h_r)/2, h-bar = h_b + hdev
  const R db = (R)0.5 * (dl + dr);                // h_b - href
  const R hb = href + db;
  const R hdev = hlR * e0l + hrR * e0r;
  // h_l E_l - h_r E_r with h E = sqrt(G/(4 pi)) h^{3/2} e^{-lam U^2}, written
  // through h_l - h_r so that it vanishes exactly for equal depths and velocities
  const R dphi = dlr * (hlR + sl * sr + hrR) / (sl + sr);
  const R ediff = cphi * (hlR * sl * (xl - xr) + dphi * xr);
  const R mbn = (hlR * Ul * mul[0] + hrR * Ur * mur[0]) + ediff;
  const R mbt = hlR * Vl * mul[0] + hrR * Vr * mur[0];
  const R hbR = hb + hdev;
  const R Ub = mbn / hbR, Vb = mbt / hbR;
  const R lamb = 1 / (g * hbR), thb = (R)0.5 * g * hbR;
  R mbp[6], mbm[6];
  half_moments_pm<R>(Ub, lamb, mbp, mbm);
  Kern<R> kbl = make_kern<R>(hbR, Ub, Vb, lamb, dnl, dtl, Dl);
  Kern<R> kbr = make_kern<R>(hbR, Ub, Vb, lamb, dnr, dtr, Dr);
  Kern<R> kl = make_kern<R>(hlR, Ul, Vl, laml, dnl, dtl, Dl);
  Kern<R> kr = make_kern<R>(hrR, Ur, Vr, lamr, dnr, dtr, Dr);
  R P[5][6], a[6], b[6];
  // C2: equilibrium slopes and force, two-sided
  kern_moments<R>(kbl, mbp, thb, Ub, Vb, a);
  kern_moments<R>(kbr, mbm, thb, Ub, Vb, b);
  for (int k = 0; k < 6; k++) P[1][k] = hbR * (a[k] + b[k]);
  // C3: A-bar from compatibility, d = time derivative of (h, hU, hV)
  const R dh = -P[1][0], dm = -P[1][1], dn = -P[1][2];
  P[2][0] = dh; P[2][1] = dm; P[2][2] = dn;
  P[2][3] = dm;
  P[2][4] = 2 * Ub * dm - Ub * Ub * dh + 2 * thb * dh;
  P[2][5] = Vb * dm + Ub * dn - Ub * Vb * dh;
  // C5: free transport of the initial slopes and force
  kern_moments<R>(kl, mul, thl, Ul, Vl, a);
  kern_moments<R>(kr, mur, thr, Ur, Vr, b);
  for (int k = 0; k < 6; k++) P[4][k] = hlR * a[k] + hrR * b[k];
  // C1 (full-space moments of g-bar) and C4 (g^l, g^r on their half spaces):
  // deviations from the bases h_b and G h_b^2 / 2
  P[0][0] = hdev; P[0][1] = mbn; P[0][2] = mbt;
  P[0][3] = mbn;
  P[0][4] = mbn * Ub + g * hb * hdev + (R)0.5 * g * hdev * hdev;
  P[0][5] = mbn * Vb;
  P[3][0] = hdev; P[3][1] = mbn; P[3][2] = mbt;
  P[3][3] = mbn;
  {
    const R m2l = thl * e0l - Ul * El, m2r = thr * e0r + Ur * Er;   // mu_2 - th/2 on each side
    P[3][4] = hlR * (Ul * Ul * mul[0] + 2 * Ul * mul[1] + m2l) + hrR * (Ur * Ur * mur[0] + 2 * Ur * mur[1] + m2r) +
              (R)0.125 * g * dlr * dlr;
  }
  P[3][5] = hlR * Vl * (Ul * mul[0] + mul[1]) + hrR * Vr * (Ur * mur[0] + mur[1]);
  // fitted value and derivative at the stage start
  R qd[5], qh[5];
  time_ints2<R>(tau, delta, qd, qh);
  R kv[5], kd[5];
  const R id = 1 / delta;
  for (int i = 0; i < 5; i++) {
    kv[i] = (4 * qh[i] - qd[i]) * id;
    kd[i] = 4 * (qd[i] - 2 * qh[i]) * id * id;
  }
  R f[3], ft[3], w[3], wt[3];
  for (int k = 0; k < 3; k++) {
    w[k] = kv[0] * P[0][k];
    wt[k] = kd[0] * P[0][k];
    f[k] = kv[0] * P[0][3 + k];
    ft[k] = kd[0] * P[0][3 + k];
  }
  for (int i = 1; i < 5; i++)
    for (int k = 0; k < 3; k++) {
      w[k] += kv[i] * P[i][k];
      wt[k] += kd[i] * P[i][k];
      f[k] += kv[i] * P[i][3 + k];
      ft[k] += kd[i] * P[i][3 + k];
    }
  // bases relative to the reference: h_b - href and G (h_b^2 - href^2) / 2
  W[0] = db + w[0];
  W[1] = w[1];
  W[2] = w[2];
  F[0] = f[0];
  F[1] = (R)0.5 * g * db * (hb + href) + f[1];
  F[2] = f[2];
  for (int k = 0; k < 3; k++) { Wt[k] = wt[k]; Ft[k] = ft[k]; }
}

// Blended level deviation at one point in the single form (Sec. 2.3): d^r + xi (d^l - d^r) with
// xi = erfc((U_n^l + U_n^r)/2)/2, U_n = (m . n) / h on each side. Written
// with explicitly rounded operations so that the interface kernel and the
// fused edge kernel, which both form it, get the same value whatever the
// compiler does with the code around it.
template <typename R>
__host__ __device__ __forceinline__ R blend_level(R dl, R hl, R mxl, R myl, R dr, R hr, R mxr, R myr, R n0, R n1) {
  static_assert(sizeof(R) == 4, "the double form's is blend64");
  using O = Rn<R>;
  const R ul = O::mul(O::fma(mxl, n0, O::mul(myl, n1)), O::rcp(hl));
  const R ur = O::mul(O::fma(mxr, n0, O::mul(myr, n1)), O::rcp(hr));
  const R xi = O::mul((R)0.5, erfcf(O::mul((R)0.5, O::add(ul, ur))));
  return O::fma(xi, O::sub(dl, dr), dr);
}

// ---------------------------------------------------- interface (iface) unit
// Blended level deviation of layer ell at edge e in the single form (Sec. 2.3), the mean over
// the two Gauss points of h-hat = xi h^l + (1 - xi) h^r with
// xi = erfc((U_n^l + U_n^r)/2)/2; the lower layer is blended as the water
// level eta1 (B is continuous). Each side's record is loaded once for both
// points. (Two lanes per unit, one per side, are no faster in FP32: 136 against
// 121 us at 1.04 M triangles; the double form takes them.)
template <typename R>
__host__ __device__ __forceinline__ R iface_unit(const Dev &d, int e, int ell) {
  static_assert(sizeof(R) == 4, "the double form's is iface_unit64");
  const EdgeIds g = edge_ids(d, e);
  R x[2][4], n[2], vl[2][3], vr[2][3];
  for (int q = 0; q < 2; q++) load_n<R, 4>((const R *)d.exi + ((size_t)q * d.ne + e) * 4, x[q]);
  load_n<R, 2>((const R *)d.en + 2 * (size_t)e, n);
  {
    R w[NREC];
    load_rec<R, NREC>(d, ell, g.L, w);
    for (int q = 0; q < 2; q++) rec_values<R>(w, x[q][0], x[q][1], vl[q]);
  }
  {
    R w[NREC];
    load_rec<R, NREC>(d, ell, g.R, w);
    for (int q = 0; q < 2; q++) rec_values<R>(w, x[q][2], x[q][3], vr[q]);
  }
  R v[2];
  for (int q = 0; q < 2; q++) {
    R mr[2] = {vr[q][1], vr[q][2]};
    if (g.xf != 0) rot2<R>(d.xf + 4 * g.xf, mr);
    const R href = ref_depth<R>(d, ell, e, q);
    const R dl = vl[q][0], dr = vr[q][0];
    v[q] = blend_level<R>(dl, href + dl, vl[q][1], vl[q][2], dr, href + dr, mr[0], mr[1], n[0], n[1]);
  }
  return Rn<R>::mul((R)0.5, Rn<R>::add(v[0], v[1]));
}

// plane gradient (Sec. 2.3) of the blended level `which` for cell c
template <typename R>
__host__ __device__ __forceinline__ void plane_grad(const Dev &d, int c, int which, R g[2]) {
  const int N = d.cs, NE = d.ne;
  const R *pl = (const R *)d.plane, *hc = (const R *)d.hc;
  g[0] = g[1] = 0;
  for (int f = 0; f < 3; f++) {
    int ce = d.cedge[f * N + c];
    int e = ce >= 0 ? ce : ~ce;
    R v = hc[which * NE + e];
    g[0] += pl[(f * 2) * N + c] * v;
    g[1] += pl[(f * 2 + 1) * N + c] * v;
  }
}

// ------------------------------------------------------------- edge unit
// Interface solution of the single form, layer ell at Gauss point q of edge e, global frame:
// out[0..2] = F, out[3..5] = F_t, out[6..8] = W, out[9..11] = W_t (deviations).
// Returns true when out was computed.
// FUSED (runs with the troubled-cell gate, where most cells take the linear
// weights): the unit also returns in *blend the point's blended level
// deviation of layer ell, h-hat - href = d^r + xi (d^l - d^r) with
// xi = erfc((U_n^l + U_n^r)/2)/2 (Sec. 2.3; the edge's blended level is the
// mean over its two points), and computes the solution only where the blend
// weight w of the other layer is 1, where the plane gradients, which need
// every blended level of both cells, carry no weight; elsewhere it returns
// false and the solution is left to a later pass (plain mode, plane
// gradients gathered).
// PAIRED (the edge kernels' thread layout, where the lane two over holds the
// same point and side for the other layer): the other layer's level
// gradient comes from that lane by a shuffle instead of from its record.
// POS (the positivity option, not in the paper): on a side whose cell's
// layer has point depths below half its average, the side velocity is
// bounded by the edge's two cells' average velocities of the layer.
template <typename R, bool FUSED = false, bool PAIRED = false, bool POS = false>
__host__ __device__ inline bool edge_unit(const Dev &d, const Par &p, int e, int ell, int q, R out[12],
                                          R *blend = nullptr, R *own = nullptr) {
  static_assert(sizeof(R) == 4, "the double form's is edge_unit64");
  const EdgeIds g = edge_ids(d, e);
  const int cL = g.L, cR = g.R, xf = g.xf;
  R x[4], n[2];
  load_n<R, 4>((const R *)d.exi + ((size_t)q * d.ne + e) * 4, x);
  load_n<R, 2>((const R *)d.en + 2 * (size_t)e, n);
  const R dt = ((const R *)d.dtR)[g.inst];
  // both stages fit the value and time derivative at their start from the
  // time integrals over dt and dt/2 (the S2O4 construction repeated from the
  // intermediate state, reading R20)
  const R delta = dt;
  const R href = ref_depth<R>(d, ell, e, q);
  SideVals<R> s[2];
#ifdef __CUDA_ARCH__
  constexpr bool SH = PAIRED;
#else
  constexpr bool SH = false;
#endif
  side_vals<R, !SH>(d, ell, cL, 0, x[0], x[1], href, s[0]);
  side_vals<R, !SH>(d, ell, cR, xf, x[2], x[3], href, s[1]);
#ifdef __CUDA_ARCH__
  if (SH) {
    for (int sd = 0; sd < 2; sd++)
      for (int k = 0; k < 2; k++) s[sd].goth[k] = __shfl_xor_sync(0xffffffffu, s[sd].glev[k], 2);
  }
#endif
  // blended derivative of the other layer's level and the well-balance vector
  // D = grad h - grad Phi / G = grad(level) + c (w grad(other) + (1 - w) grad P1)
  const int oth = 1 - ell;  // hc / omg index of the other layer: 0 = eta1, 1 = h2
  const R *om = (const R *)d.omg;
  R w = om[oth * d.cs + cL] < om[oth * d.cs + cR] ? om[oth * d.cs + cL] : om[oth * d.cs + cR];
  w = w < (R)0 ? (R)0 : (w > (R)1 ? (R)1 : w);
  // the plane gradients enter with weight 1 - w (the fused mode computes
  // only units with w = 1)
  R pl[2][2] = {{0, 0}, {0, 0}};
  if (!FUSED) {
#ifdef __CUDA_ARCH__
    // the two lanes of an edge's layer gather one side's each and exchange
    R mine[2], theirs[2];
    plane_grad<R>(d, q == 0 ? cL : cR, oth, mine);
    for (int k = 0; k < 2; k++) theirs[k] = __shfl_xor_sync(0xffffffffu, mine[k], 1);
    for (int k = 0; k < 2; k++) {
      pl[0][k] = q == 0 ? mine[k] : theirs[k];
      pl[1][k] = q == 0 ? theirs[k] : mine[k];
    }
#else
    plane_grad<R>(d, cL, oth, pl[0]);
    plane_grad<R>(d, cR, oth, pl[1]);
#endif
    if (xf != 0) rot2<R>(d.xf + 4 * xf, pl[1]);
  }
  const R cf = ell == 0 ? pv<R>(p.chi, p.chif) : (R)1;
  const R n0 = n[0], n1 = n[1];
  R U[2], V[2], dn[2][3], dtt[2][3], D[2][2];
  for (int sd = 0; sd < 2; sd++) {
    const SideVals<R> &S = s[sd];
    R Dx = S.glev[0] + cf * (w * S.goth[0] + (1 - w) * pl[sd][0]);
    R Dy = S.glev[1] + cf * (w * S.goth[1] + (1 - w) * pl[sd][1]);
    D[sd][0] = Dx * n0 + Dy * n1;
    D[sd][1] = -Dx * n1 + Dy * n0;
    R ih = (R)1 / S.h;
    U[sd] = (S.mx * n0 + S.my * n1) * ih;
    V[sd] = (-S.mx * n1 + S.my * n0) * ih;
    // derivatives along n and t of (h, m_n, m_t)
    const R dir[2][2] = {{n0, n1}, {-n1, n0}};
    R *outv[2] = {dn[sd], dtt[sd]};
    for (int k = 0; k < 2; k++) {
      R ex = dir[k][0], ey = dir[k][1];
      R dhh = S.gh[0] * ex + S.gh[1] * ey;
      R dmx = S.gm[0][0] * ex + S.gm[0][1] * ey;
      R dmy = S.gm[1][0] * ex + S.gm[1][1] * ey;
      outv[k][0] = dhh;
      outv[k][1] = dmx * n0 + dmy * n1;
      outv[k][2] = -dmx * n1 + dmy * n0;
    }
  }
  if (POS) {
    const int N = d.cs, vm = ell == 0 ? 4 : 1;
    const bool bl = d.pos_flag[ell * N + cL] != 0, br = d.pos_flag[ell * N + cR] != 0;
    if (bl || br) {
      const R *hb = (const R *)d.pos_hbar;
      R un[2], ut[2];
      for (int sd = 0; sd < 2; sd++) {
        const int c = sd == 0 ? cL : cR, x = sd == 0 ? 0 : xf;
        R m[2];
        load_n<R, 2>(dq_at<R>(d, pair_of(vm), c), m);
        image_q<R>(d, pair_of(vm), x, m);
        const R mx = m[0], my = m[1];
        const R ih = (R)1 / hb[ell * N + c];
        un[sd] = (mx * n0 + my * n1) * ih;
        ut[sd] = (-mx * n1 + my * n0) * ih;
      }
      const R ulo = un[0] < un[1] ? un[0] : un[1], uhi = un[0] < un[1] ? un[1] : un[0];
      const R tlo = ut[0] < ut[1] ? ut[0] : ut[1], thi = ut[0] < ut[1] ? ut[1] : ut[0];
      for (int sd = 0; sd < 2; sd++) {
        if (!(sd == 0 ? bl : br)) continue;
        U[sd] = U[sd] < ulo ? ulo : (U[sd] > uhi ? uhi : U[sd]);
        V[sd] = V[sd] < tlo ? tlo : (V[sd] > thi ? thi : V[sd]);
      }
    }
  }
  // each side's own level at the point: the interlayer source's values (R16)
  if (own) {
    own[0] = s[0].d;
    own[1] = s[1].d;
  }
  if (FUSED) {
    *blend = blend_level<R>(s[0].d, s[0].h, s[0].mx, s[0].my, s[1].d, s[1].h, s[1].mx, s[1].my, n0, n1);
    if (w < (R)1) return false;
  }
  // collision time (Sec. 4): tau = eps dt + eps_num |(hl^2 - hr^2)/(hl^2 + hr^2)| dt
  const R hl = s[0].h, hr = s[1].h;
  const R jump = r_abs<R>((s[0].d - s[1].d) * (hl + hr) / (hl * hl + hr * hr));
  const R tau = pv<R>(p.eps, p.epsf) * dt + pv<R>(p.eps_num, p.eps_numf) * jump * dt;
  R F[3], Ft[3], W[3], Wt[3];
  gks_layer<R>(href, s[0].d, s[1].d, U[0], V[0], U[1], V[1], dn[0], dtt[0], D[0], dn[1], dtt[1], D[1],
               pv<R>(p.g, p.gf), tau, delta, F, Ft, W, Wt);
  const R *src[4] = {F, Ft, W, Wt};
  for (int k = 0; k < 4; k++) {
    out[3 * k] = src[k][0];
    out[3 * k + 1] = src[k][1] * n0 - src[k][2] * n1;
    out[3 * k + 2] = src[k][1] * n1 + src[k][2] * n0;
  }
  return true;
}

// ------------------------------------------------------------- cell unit
// dX / U_max of a cell (Sec. 4: U_max the larger over the layers of |U| +
// sqrt(G h)) in the form's precision; the update kernel and the kernel that
// starts a newly set state both use it, so a restarted run takes the same
// steps as an uninterrupted one. FP32 form: the reciprocal in single precision
// (dt to ~1e-7 relative), sparing the FP64 pipe a double division.
template <typename R>
__host__ __device__ inline R layer_speed(double h_, double mx, double my, R G) {
  R h = (R)h_, u = (R)mx / h, v = (R)my / h;
  return r_sqrt<R>(u * u + v * v) + r_sqrt<R>(G * h);
}
template <typename R>
__host__ __device__ inline double cfl_ratio(R upper, R lower, double dX) {
  R um = 0;
  um = upper > um ? upper : um;
  um = lower > um ? lower : um;
  if (sizeof(R) == 4) return dX * (double)((R)1 / um);
  return dX / (double)um;
}

#ifdef __CUDACC__
// Flux and source residuals, S2O4 update (Eq. SWE-fully-discrete), interface
// values at the stage end (Eq. S2O3) and Gauss-theorem gradients (Eq. slope-1)
// of a cell: of both its layers (NL = 2), or of one (NL = 1, lay: 0 lower, 1
// upper) with the other layer in the next or previous lane, the two exchanging
// what each needs of the other. All lanes of the warp call; only with `ok` are
// results written. Returns the CFL ratio dX/U_max of the new state (stage 2)
// or 0. Between the stages of a step d.avg keeps W^n and d.Wn holds W*.
template <typename R, int NL>
__device__ __forceinline__ double update_unit(const Dev &d, const Par &p, int j, int lay, int stage, bool ok,
                                              int *flags) {
  const int N = d.cs;
  const size_t NE = (size_t)d.ne;
  const int in = d.inst[j];
  const double dt = d.dt[in];
  // the unit's loads and arithmetic do not wait on dt: a cell of an instance
  // that has stopped (dt = 0) is computed too, and only its writes are dropped
  const bool act = ok && dbits(dt) > 0;
  const R dtr = ((const R *)d.dtR)[in];
  const R cend = stage == 1 ? (R)0.5 * dtr : dtr;
  // by layer (i = 0 .. NL - 1, or the one of the lane): mass residuals in FP64
  // (exact conservation), the rest in R; LF, LFt: the discharge's; mWt, GGt:
  // mean and Gauss-theorem gradient of the depth's W_t; GGn: gradients at the
  // stage end; the interlayer source's point values (R16), this cell's own
  // levels at its six Gauss points: their mean (mO) and Gauss-theorem gradient
  // (GO)
  double LFm[NL] = {}, LFtm[NL] = {};
  R LF[NL][2] = {}, LFt[NL][2] = {}, mWt[NL] = {}, GGt[NL][2] = {}, GGn[NL][3][2] = {}, mO[NL] = {}, GO[NL][2] = {};
#pragma unroll
  for (int f = 0; f < 3; f++) {
    int ce = d.cedge[f * N + j];
    int e = ce >= 0 ? ce : ~ce;
    const int side = ce >= 0 ? 0 : 1;
    const double sl = d.fsl[f * N + j];
    const R slR = ((const R *)d.fslR)[f * N + j];
    R n[2];
    load_n<R, 2>((const R *)d.en + 2 * (size_t)e, n);
    const R snx = slR * n[0], sny = slR * n[1];
#pragma unroll
    for (int i = 0; i < NL; i++) {
      const size_t at = (NL == 2 ? i : lay) * NE + e;
      R F[4], Wt[4], Wn[4];
      double M[2];
      load_n<R, 4>((const R *)d.eF + 4 * at, F);
      load_n<R, 4>((const R *)d.eWt + 4 * at, Wt);
      load_n<R, 4>((const R *)d.eWn + 4 * at, Wn);
      load_n<double, 2>(d.eM + 2 * at, M);
      const R o = ((const R *)d.eO)[2 * at + side];
      mO[i] += o * (R)(1.0 / 3.0);
      GO[i][0] += snx * o; GO[i][1] += sny * o;
      LFm[i] -= sl * M[0];
      LFtm[i] -= sl * M[1];
      mWt[i] += Wt[0] * (R)(1.0 / 3.0);
      GGt[i][0] += snx * Wt[0]; GGt[i][1] += sny * Wt[0];
      for (int k = 0; k < 2; k++) {
        LF[i][k] -= slR * F[k];
        LFt[i][k] -= slR * F[2 + k];
      }
      for (int k = 0; k < 3; k++) {
        R We = Wn[k] + cend * Wt[k];
        GGn[i][k][0] += snx * We; GGn[i][k][1] += sny * We;
      }
    }
  }
  R GOo[NL][2], GGto[NL][2];                       // the other layer's
  for (int i = 0; i < NL; i++)
    for (int k = 0; k < 2; k++) {
      GOo[i][k] = NL == 2 ? GO[NL - 1 - i][k] : __shfl_xor_sync(0xffffffffu, GO[i][k], 1);
      GGto[i][k] = NL == 2 ? GGt[NL - 1 - i][k] : __shfl_xor_sync(0xffffffffu, GGt[i][k], 1);
    }
  const R G = pv<R>(p.g, p.gf), chi = pv<R>(p.chi, p.chif);
  R gb[2], dq0[2], speed[NL], q0[NL], g0[NL][2];   // dq0: the levels' deviations (h2, eta1)
  load_n<R, 2>((const R *)d.bgR + 2 * (size_t)j, gb);
  load_n<R, 2>(dq_at<R>(d, 0, j), dq0);
  const R dt2 = dtr * dtr;
  int fl = 0;
#pragma unroll
  for (int i = 0; i < NL; i++) {
    const int l = NL == 2 ? i : lay, v0 = l == 0 ? 3 : 0;   // the layer and its depth variable
    const R LFh = (R)LFm[i];
    R L[2], Lt[2];
    if (l == 1) {
      // upper layer: -G h2 grad(B + h1) with h1 = eta1 - B at the points; the
      // time derivative by the product rule with the interface solution's W_t (R4)
      const R m2 = ((const R *)d.refR)[2 * in] + mO[i];   // mean of h2 over the 6 Gauss points
      for (int k = 0; k < 2; k++) {
        L[k] = LF[i][k] - G * (dq0[0] - mO[i]) * gb[k] - G * m2 * GOo[i][k];
        Lt[k] = LFt[i][k] - G * (LFh - mWt[i]) * gb[k] - G * mWt[i] * GOo[i][k] - G * m2 * GGto[i][k];
      }
    } else {
      // lower layer: flux reference pressure + bottom source -> -G (eta1 - R1) grad B; interlayer -chi G h1 grad h2
      const R m1 = ((const R *)d.hrefc)[j] + mO[i];       // (R1 - B_j) + the mean level's deviation
      for (int k = 0; k < 2; k++) {
        L[k] = LF[i][k] - G * dq0[1] * gb[k] - chi * G * m1 * GOo[i][k];
        Lt[k] = LFt[i][k] - G * LFh * gb[k] - chi * G * (mWt[i] * GOo[i][k] + m1 * GGto[i][k]);
      }
    }
    // S2O4 (Eq. SWE-fully-discrete): stage 1 W* = W^n + dt/2 L^n + dt^2/8 L_t^n;
    // stage 2 W^{n+1} = W^n + dt L^n + dt^2/6 L_t^n + dt^2/3 L_t^*. The layer
    // depths (exact conservation) in FP64 throughout; the momenta's increments
    // in R (their residuals are R), each added to the FP64 state once
    double nw[3], was[3];
    double *now = (stage == 1 ? d.Wn : d.avg) + (size_t)v0 * N + j;
    double *Ln = d.Ln + (size_t)v0 * N + j, *Ltn = d.Ltn + (size_t)v0 * N + j;
    R *inc = (R *)d.incR + (size_t)(l == 1 ? 0 : 2) * N + j;
    for (int k = 0; k < 3; k++) was[k] = d.avg[(size_t)(v0 + k) * N + j];
    if (stage == 1) {
      if (act) {
        *Ln = LFm[i];
        *Ltn = LFtm[i];
      }
      nw[0] = was[0] + 0.5 * dt * LFm[i] + 0.125 * dt * dt * LFtm[i];
    } else {
      nw[0] = was[0] + dt * *Ln + dt * dt * (1.0 / 6.0) * *Ltn + dt * dt * (1.0 / 3.0) * LFtm[i];
    }
    for (int k = 0; k < 2; k++) {
      if (stage == 1) {
        if (act) inc[(size_t)k * N] = dtr * L[k] + dt2 * (R)(1.0 / 6.0) * Lt[k];
        nw[1 + k] = was[1 + k] + (double)((R)0.5 * dtr * L[k] + (R)0.125 * dt2 * Lt[k]);
      } else {
        nw[1 + k] = was[1 + k] + (double)(inc[(size_t)k * N] + dt2 * (R)(1.0 / 3.0) * Lt[k]);
      }
    }
    // (W* of a cell that has stopped is its state: the one read between stages)
    if (act || (ok && stage == 1))
      for (int k = 0; k < 3; k++) now[(size_t)k * N] = act ? nw[k] : was[k];
    // the level's deviation and gradient (of the lower layer: grad h1 = grad
    // eta1 - grad B, the interface values being water levels)
    const double lev = l == 0 ? nw[0] + d.bmean[j] : nw[0];
    q0[i] = (R)(lev - d.ref[2 * in + 1 - l]);
    for (int k = 0; k < 2; k++) g0[i][k] = l == 0 ? GGn[i][0][k] - gb[k] : GGn[i][0][k];
    if (act) {
      const int pair = l == 1 ? 1 : 2;
      const R q[2] = {(R)nw[1], (R)nw[2]}, g[4] = {GGn[i][1][0], GGn[i][1][1], GGn[i][2][0], GGn[i][2][1]};
      store_n<R, 2>(dq_at<R>(d, pair, j), q);
      store_n<R, 4>(dg_at<R>(d, pair, j), g);
    }
    // health flags by integer tests on the bits (off the FP64 pipe)
    for (int k = 0; k < 3; k++)
      if (!finite_bits(nw[k]) || !isfinite(GGn[i][k][0]) || !isfinite(GGn[i][k][1])) fl |= 2;
    if (!(dbits(nw[0]) > 0)) fl |= 1;
    if (stage == 2) speed[i] = layer_speed<R>(nw[0], nw[1], nw[2], G);
  }
  if (act) {
    if (NL == 2) {
      const R q[2] = {q0[NL - 1], q0[0]}, g[4] = {g0[NL - 1][0], g0[NL - 1][1], g0[0][0], g0[0][1]};
      store_n<R, 2>(dq_at<R>(d, 0, j), q);
      store_n<R, 4>(dg_at<R>(d, 0, j), g);
    } else {
      dq_at<R>(d, 0, j)[1 - lay] = q0[0];
      store_n<R, 2>(dg_at<R>(d, 0, j) + 2 * (1 - lay), g0[0]);
    }
  }
  *flags = act ? fl : 0;
  if (stage != 2) return 0;
  R upper = speed[NL - 1], lower = speed[0];
  if (NL == 1) {
    const R other = __shfl_xor_sync(0xffffffffu, speed[0], 1);
    upper = lay == 1 ? speed[0] : other;
    lower = lay == 1 ? other : speed[0];
  }
  if (!act) return 0;
  return cfl_ratio<R>(upper, lower, d.dX[j]);
}
#endif

}  // namespace gks2l
