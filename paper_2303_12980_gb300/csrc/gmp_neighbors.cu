// Cell-list binning and exact neighbor images on the GPU.
//
// Neighbor set (GMP-Featurizer, Statement of Needs / Overview: molecules,
// clusters and periodic crystals given lattice vectors and positions): all
// (j, n in Z^3, n_k = 0 on non-periodic axes) with
//   d = (x_j - x_i) + ((n1 a1 + n2 a2) + n3 a3),   dx*dx + dy*dy + dz*dz < rc*rc
// where the expression is FP64, evaluated left to right without FMA.  The
// GPU reaches the same decision with far less FP64 work:
//   1. atoms are binned on a grid in (wrapped) fractional coordinates;
//   2. a center scans the rows of bins that its cutoff sphere can touch
//      (periodic axes wrap, giving an image index m); each candidate is
//      pre-screened in FP32 against a rigorous bound on the FP32 error;
//   3. survivors get d and r^2 in double-float arithmetic (about 2^-44
//      relative), which decides every case except a shell of relative width
//      ~1e-9 around rc^2; inside that shell the FP64 expression above is
//      evaluated exactly as written, so the set equals the FP64 one;
//   4. each center's accepted (j, n) records are written in a fixed order,
//      which makes every later sum over a center's neighbors deterministic:
//      grouped by neighbor species, enumeration order within a species
//      (the feature kernels then read the same table rows across a tile),
//      or sorted by (j, n) for the Jacobian and the neighbor-list output.
#include "gmp_internal.cuh"

#include <math.h>
#include <string.h>

#include <algorithm>

namespace {

__device__ __forceinline__ unsigned long long order_key(double v) {
  unsigned long long b = (unsigned long long)__double_as_longlong(v);
  return (b >> 63) ? ~b : (b | 0x8000000000000000ull);
}
__host__ __device__ inline double key_to_double(unsigned long long k) {
  const unsigned long long b = (k >> 63) ? (k & 0x7FFFFFFFFFFFFFFFull) : ~k;
  double v;
  memcpy(&v, &b, sizeof(v));
  return v;
}

__device__ __forceinline__ int floor_div(int a, int b) {  // b > 0
  int q = a / b;
  return (a % b != 0 && ((a < 0) != (b < 0))) ? q - 1 : q;
}

// floor(a / b) for |a| < 2^20 and 1 <= b < 2^24 (both exact in FP32)
// without an integer division: the approximate reciprocal (2 ulp) and the
// rounded product leave the single-precision quotient within a relative
// 2^-21 of a / b, i.e. off by less than |a| / b * 2^-21 < 0.5, so its floor
// is within one of the true one and the remainder test corrects it.
__device__ __forceinline__ int floor_div_small(int a, int b) {
  int q = __float2int_rd(__fmul_rn(__int2float_rn(a), __fdividef(1.0f, __int2float_rn(b))));
  const int r = a - q * b;
  if (r < 0) --q;
  else if (r >= b) ++q;
  return q;
}

__device__ __forceinline__ int32_t pack_wrap(int w0, int w1, int w2) {
  return gmp_pack_shift(w0, w1, w2);
}

// Sort key of a neighbor image: atom first, then n1, n2, n3 (each biased by 512).
__device__ __forceinline__ unsigned long long sort_key(int64_t j, const int* n) {
  return ((unsigned long long)j << 30) | ((unsigned long long)(n[0] + 512) << 20) |
         ((unsigned long long)(n[1] + 512) << 10) | (unsigned long long)(n[2] + 512);
}
__device__ __forceinline__ void sort_key_image(unsigned long long key, int* n) {
  n[0] = (int)((key >> 20) & 1023) - 512;
  n[1] = (int)((key >> 10) & 1023) - 512;
  n[2] = (int)(key & 1023) - 512;
}

// Reference cell of a structure: the cell index of its first atom along
// each periodic axis (0 when it has no atoms or that position is not
// finite).  Atoms and reference points store their cell index relative to
// it, so a structure placed any number of cells away from its cell keeps
// small stored indices; pair image indices, which are differences of the
// stored indices, do not change.
__device__ inline double ref_cell_axis(const GmpStruct& st, const double* __restrict__ atom_pos, int k) {
  if (st.n_atoms <= 0 || !st.periodic[k]) return 0.0;
  const double* x = atom_pos + 3 * st.atom_base;
  const double x0 = x[0], x1 = x[1], x2 = x[2];
  if (!isfinite(x0) || !isfinite(x1) || !isfinite(x2)) return 0.0;
  const double f = floor(x0 * st.Ainv[k] + x1 * st.Ainv[3 + k] + x2 * st.Ainv[6 + k]);
  return fabs(f) < 1e9 ? f : 0.0;
}
__device__ inline void struct_ref_cell(const GmpStruct& st, const double* __restrict__ atom_pos, double (&f0)[3]) {
  for (int k = 0; k < 3; ++k) f0[k] = ref_cell_axis(st, atom_pos, k);
}

// Wraps the fractional coordinate u of a periodic axis into [0, 1) and
// returns the cell index relative to the reference cell f0 (error flag and
// 0 when it does not fit the packed image index).
__device__ inline int wrap_axis(double& u, double f0, uint32_t* err) {
  const double fl = floor(u);
  const double f = fl - f0;
  int w = 0;
  if (fabs(f) > 500.0) {  // image index would not fit the packed shift
    atomicOr(err, GMP_DEV_SHIFT_RANGE);
  } else {
    w = (int)f;
  }
  u -= fl;
  if (u >= 1.0) { u -= 1.0; w += 1; }
  if (u < 0.0) u = 0.0;
  return w;
}

// The double-float split of a position, with the species and the packed wrap.
__device__ __forceinline__ void write_split(int64_t a, const double (&x)[3], int e, const int (&w)[3], float4* xh,
                                            float4* xl) {
  float h[3], l[3];
  for (int k = 0; k < 3; ++k) {
    h[k] = (float)x[k];
    l[k] = (float)(x[k] - (double)h[k]);
  }
  xh[a] = make_float4(h[0], h[1], h[2], __int_as_float(e));
  xl[a] = make_float4(l[0], l[1], l[2], __int_as_float(pack_wrap(w[0], w[1], w[2])));
}

// Position and species of atom a, checked (flagged ones are replaced).
__device__ __forceinline__ int load_atom(int64_t a, const double* __restrict__ pos, const int32_t* __restrict__ species,
                                         int n_el, double (&x)[3], uint32_t* __restrict__ err) {
  for (int k = 0; k < 3; ++k) x[k] = pos[3 * a + k];
  int e = species[a];
  if (e < 0 || e >= n_el) {
    atomicOr(err, GMP_DEV_BAD_SPECIES);
    e = 0;
  }
  if (!isfinite(x[0]) || !isfinite(x[1]) || !isfinite(x[2])) {
    atomicOr(err, GMP_DEV_NONFINITE);
    x[0] = x[1] = x[2] = 0.0;
  }
  return e;
}

// Per atom: checks, fractional coordinates, wrap, double-float split, bbox.
// bbox: 6 keys per structure (min and complemented max of each non-periodic
// fractional axis).
__device__ __forceinline__ void prepare_atom(const GmpStruct* S, const int32_t* __restrict__ struct_of, int64_t a,
                                             const double* __restrict__ pos, const int32_t* __restrict__ species,
                                             int n_el, float4* __restrict__ atom_xh, float4* __restrict__ atom_xl,
                                             GmpD4* __restrict__ atom_u, unsigned long long* bbox,
                                             uint32_t* __restrict__ err) {
  const int s = struct_of[a];
  const GmpStruct& st = S[s];
  double x[3];
  const int e = load_atom(a, pos, species, n_el, x, err);
  double u[3], f0[3];
  int w[3] = {0, 0, 0};
  struct_ref_cell(st, pos, f0);
  for (int k = 0; k < 3; ++k) {
    u[k] = x[0] * st.Ainv[k] + x[1] * st.Ainv[3 + k] + x[2] * st.Ainv[6 + k];
    if (st.periodic[k]) {
      w[k] = wrap_axis(u[k], f0[k], err);
    } else {
      // both slots start at all-ones; the max slot stores the complemented key
      atomicMin(&bbox[6 * s + 2 * k], order_key(u[k]));
      atomicMin(&bbox[6 * s + 2 * k + 1], ~order_key(u[k]));
    }
  }
  write_split(a, x, e, w, atom_xh, atom_xl);
  atom_u[a] = GmpD4{u[0], u[1], u[2], 0.0};
}

// (The first kernel of a call also clears the n_clear words behind the error
// word: counters and sizes of the call, which later kernels use.)
__global__ void k_prepare(const GmpStruct* __restrict__ S, const int32_t* __restrict__ struct_of,
                          int64_t N, const double* __restrict__ pos,
                          const int32_t* __restrict__ species, int n_el,
                          float4* __restrict__ atom_xh, float4* __restrict__ atom_xl,
                          GmpD4* __restrict__ atom_u, unsigned long long* __restrict__ bbox,
                          int64_t n_bins, int32_t* __restrict__ bin_count, int32_t* __restrict__ bin_cursor,
                          uint32_t* __restrict__ err, int n_clear) {
  gmp_let_next_start();
  const unsigned tid = gmp_after_predecessor(threadIdx.x);
  if (blockIdx.x == 0)
    for (int t = tid; t < n_clear; t += blockDim.x) err[1 + t] = 0;
  for (int64_t b = blockIdx.x * (int64_t)blockDim.x + tid; b < n_bins; b += (int64_t)gridDim.x * blockDim.x)
    bin_count[b] = bin_cursor[b] = 0;
  for (int64_t a = blockIdx.x * (int64_t)blockDim.x + tid; a < N;
       a += (int64_t)gridDim.x * blockDim.x)
    prepare_atom(S, struct_of, a, pos, species, n_el, atom_xh, atom_xl, atom_u, bbox, err);
}

// Bin grid and FP32 pre-screen bound of one structure.  bbox: its 6 keys,
// read for non-periodic axes only (a fully periodic structure's grid follows
// from its cell and is made on the host, with the batch description).
// The bins are half a cutoff wide, along axis 0, which the neighbor search
// takes a row at a time, a quarter (a row's ends overshoot the sphere's chord
// by a bin: 508 against 512 us for the neighbor stage of 2,500 small
// structures, 45 against 47 of a 4,096-atom crystal).  One thread runs this
// for a structure, at 1/64 of the FP32 rate in FP64: one division an axis, and
// the bounds, which carry a margin, in FP32.
// In two parts: an axis (they may be taken by different threads), then the rest.
struct GridAxes {
  double w[3], ext[3];  // bin width, extent of the bins
  float uk[3];          // bound on the fractional coordinates
};
__host__ __device__ inline void grid_axis(const GmpStruct& st, const unsigned long long* bbox, GmpGrid& g, GridAxes& x,
                                          int k) {
  const double target = (k == 0 ? 0.25 : 0.5) * st.reach[k];
  if (st.periodic[k]) {
    g.umin[k] = 0.0;
    x.ext[k] = x.w[k] = 1.0;
    const double nbf = target > 0.0 ? floor(1.0 / target) : 1.0;
    g.nb[k] = (int)fmin(fmax(nbf, 1.0), 1024.0);
    g.inv_binw[k] = g.nb[k];
    x.uk[k] = 2.0f;
  } else {
    const double lo = st.n_atoms ? key_to_double(bbox[2 * k]) : 0.0;
    const double hi = st.n_atoms ? key_to_double(~bbox[2 * k + 1]) : 0.0;
    g.umin[k] = lo;
    x.ext[k] = hi - lo;
    x.w[k] = fmax(target, 1e-12);
    g.inv_binw[k] = 1.0 / x.w[k];
    // (fmax: 1 for a NaN, which an extent beyond FP64's range would make here)
    g.nb[k] = (int)fmin(fmax(floor(x.ext[k] * g.inv_binw[k]) + 1.0, 1.0), 1024.0);
    if (g.nb[k] == 1024) {
      x.w[k] = fmax(x.ext[k] / 1023.0, x.w[k]);
      g.inv_binw[k] = 1.0 / x.w[k];
    }
    x.uk[k] = fmaxf(fabsf((float)lo), fabsf((float)hi)) + 1.0f;
  }
}
__host__ __device__ inline void grid_rest(GmpStruct& st, GmpGrid& g, const GridAxes& x, double cutoff) {
  double w[3];
  float uk[3];
  for (int k = 0; k < 3; ++k) {
    w[k] = x.w[k];
    uk[k] = x.uk[k];
  }
  // keep the grid within the reserved bin slots
  while ((int64_t)g.nb[0] * g.nb[1] * g.nb[2] > st.bin_cap) {
    int k = 0;
    if (g.nb[1] > g.nb[k]) k = 1;
    if (g.nb[2] > g.nb[k]) k = 2;
    if (st.periodic[k]) {
      g.nb[k] = (g.nb[k] + 1) / 2;
      g.inv_binw[k] = g.nb[k];
    } else {
      w[k] *= 2.0;
      g.inv_binw[k] *= 0.5;
      g.nb[k] = (int)fmin(fmax(floor(x.ext[k] * g.inv_binw[k]) + 1.0, 1.0), 1024.0);
    }
  }
  // Rigorous two-sided FP32 bounds.  Wrapped Cartesian coordinates are
  // |y_c| <= Y, image shifts |s_c| <= Sh; the FP32 displacement
  // (y_j - y_i) + s has per-component error below 2^-22 (4Y + 4Sh + rc)
  // <= delta = 2^-21 (Y + Sh + rc) (a few roundings of magnitude <= 2Y + Sh
  // each, plus the rounding of the cell to FP32), so | |d32| - |d| | <=
  // sqrt(3) delta, and the three-term FP32 r^2 is within 2^-21 relative of
  // |d32|^2.  Hence FP32 r^2 > (rc + 2 delta)^2 (1 + 2^-20) means |d| > rc
  // and FP32 r^2 < (rc - 2 delta)^2 (1 - 2^-20) means |d| < rc, both by a
  // margin far above the FP64 rounding of the defining expression; only the
  // shell in between needs the exact test.
  // Centers need not be atoms (reference points): along a non-periodic axis
  // a center scans some bin only if its coordinate lies within reach + one
  // bin width of the atoms' range, which the bound on |y| covers.
  // (FP32 sums of at most 10 roundings, a relative 2^-20 at most; coordinates
  // beyond FP32's range leave everything to the exact test.)
  float sk[3], Y = 0.0f, Sh = 0.0f;
  for (int k = 0; k < 3; ++k) {
    const float r = (float)st.reach[k] * 1.000001f;
    uk[k] = fminf(uk[k] + (st.periodic[k] ? 0.0f : r + 2.0f * (float)w[k]), 1e30f);
    sk[k] = ceilf(r) + 2.0f;
  }
  for (int c = 0; c < 3; ++c) {
    float yc = 0.0f, sc = 0.0f;
    for (int k = 0; k < 3; ++k) {
      const float a = fabsf(st.Ahi[3 * k + c]);
      yc += uk[k] * a;
      sc += sk[k] * a;
    }
    Y = fmaxf(Y, yc);
    Sh = fmaxf(Sh, sc);
  }
  const double delta = (double)((Y + Sh + (float)cutoff) * 1.00001f) * 0x1p-21;
  double b = (cutoff + 2.0 * delta);
  g.ortho = 1;
  if (!st.diag) {
    double bk[3];  // |b_k|^2, b_k = column k of Ainv
    for (int k = 0; k < 3; ++k) bk[k] = st.Ainv[k] * st.Ainv[k] + st.Ainv[3 + k] * st.Ainv[3 + k] + st.Ainv[6 + k] * st.Ainv[6 + k];
    for (int k = 0; k < 3; ++k) {
      const int m = k == 2 ? 0 : k + 1;
      const double d = st.Ainv[k] * st.Ainv[m] + st.Ainv[3 + k] * st.Ainv[3 + m] + st.Ainv[6 + k] * st.Ainv[6 + m];
      if (!(d * d <= 1e-18 * bk[k] * bk[m])) g.ortho = 0;
    }
  }
  for (int k = 0; k < 3; ++k) {
    g.rb[k] = (float)(st.reach[k] * g.inv_binw[k]);
    g.h[k] = (float)cutoff / g.rb[k];
  }
  g.inv_h0 = g.rb[0] / (float)cutoff;
  g.pad = 0.0f;
  float p2 = (float)(b * b * (1.0 + 0x1p-20));
  st.prescreen2 = nextafterf(p2, INFINITY);
  const double bi = fmax(cutoff - 2.0 * delta, 0.0);
  float q2 = (float)(bi * bi * (1.0 - 0x1p-20));
  st.inside2 = fmaxf(nextafterf(q2, 0.0f), 0.0f);
}

__host__ __device__ inline void grid_struct(GmpStruct& st, const unsigned long long* bbox, GmpGrid& g, double cutoff) {
  GridAxes x;
  for (int k = 0; k < 3; ++k) grid_axis(st, bbox, g, x, k);
  grid_rest(st, g, x, cutoff);
}

__host__ __device__ inline bool all_periodic(const GmpStruct& st) {
  return st.periodic[0] && st.periodic[1] && st.periodic[2];
}

// The grids that depend on the atoms' range (all: every structure's).
__global__ void k_grid(GmpStruct* __restrict__ S, int n_struct,
                       const unsigned long long* __restrict__ bbox, GmpGrid* __restrict__ G,
                       double cutoff, int all) {
  gmp_let_next_start();
  const unsigned tid = gmp_after_predecessor(threadIdx.x);
  const int s = blockIdx.x * blockDim.x + tid;
  if (s >= n_struct || (!all && all_periodic(S[s]))) return;
  GmpGrid g;
  grid_struct(S[s], bbox + 6 * s, g, cutoff);
  G[s] = g;
}

// Bin, in its structure's grid, of an atom at wrapped fractional coordinates u.
__device__ __forceinline__ int64_t bin_of(const GmpGrid& g, const double* u) {
  int b[3];
  for (int k = 0; k < 3; ++k) {
    double t = floor((u[k] - g.umin[k]) * g.inv_binw[k]);  // as center_place scales
    t = fmin(fmax(t, 0.0), (double)(g.nb[k] - 1));
    b[k] = (int)t;
  }
  return b[0] + (int64_t)g.nb[0] * (b[1] + (int64_t)g.nb[1] * b[2]);
}

// Bin slot of atom a: bin_y = (wrapped FP32 position, packed wrap of the
// atom), bin_je = (atom index, species).
// (wrap = atom_xl[a].w, spec = atom_xh[a].w: packed wrap and species bits)
__device__ __forceinline__ void write_slot(int64_t a, int32_t slot, const float4& y, float spec, float wrap,
                                           float4* __restrict__ bin_y, int2* __restrict__ bin_je) {
  bin_y[slot] = make_float4(y.x, y.y, y.z, wrap);
  bin_je[slot] = make_int2((int32_t)a, __float_as_int(spec));
}

// Slot lists in arbitrary order: slot_atom[bin_start[b] + k] = the k-th
// atom to arrive in bin b.
__global__ void k_bin_scatter(int64_t N, const int32_t* __restrict__ atom_bin,
                              const int32_t* __restrict__ bin_start, int32_t* __restrict__ bin_cursor,
                              int32_t* __restrict__ slot_atom) {
  gmp_let_next_start();
  const unsigned tid = gmp_after_predecessor(threadIdx.x);
  for (int64_t a = blockIdx.x * (int64_t)blockDim.x + tid; a < N;
       a += (int64_t)gridDim.x * blockDim.x) {
    const int32_t bin = atom_bin[a];
    slot_atom[bin_start[bin] + atomicAdd(&bin_cursor[bin], 1)] = (int32_t)a;
  }
}

// Per slot: the atom's rank by index within its bin gives its final slot
// (bins in atom-index order, which makes neighbor enumeration
// deterministic); the bin's slot list is read in parallel, not sorted in
// place.
__global__ void k_bin_place(int64_t N, const int32_t* __restrict__ atom_bin, const int32_t* __restrict__ bin_start,
                            const int32_t* slot_atom, const float4* __restrict__ atom_y,
                            const float4* __restrict__ atom_xh, const float4* __restrict__ atom_xl,
                            float4* __restrict__ bin_y, int2* __restrict__ bin_je) {
  gmp_let_next_start();
  const unsigned tid = gmp_after_predecessor(threadIdx.x);
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + tid; t < N;
       t += (int64_t)gridDim.x * blockDim.x) {
    const int32_t a = slot_atom[t];
    const int32_t bin = atom_bin[a];
    const int32_t b0 = bin_start[bin], b1 = bin_start[bin + 1];
    int32_t rank = 0;
    for (int32_t u = b0; u < b1; ++u) rank += slot_atom[u] < a ? 1 : 0;
    write_slot(a, b0 + rank, atom_y[a], atom_xh[a].w, atom_xl[a].w, bin_y, bin_je);
  }
}

// A center at wrapped fractional coordinates u in the bin grid (units of
// bins; as bin_of scales) and its wrapped FP32 position.
__device__ __forceinline__ void center_place(const GmpStruct& st, const GmpGrid& g, const double* u,
                                             float4& t_out, float4& y_out) {
  float y[3], t[3];
  for (int c = 0; c < 3; ++c) {
    t[c] = (float)((u[c] - g.umin[c]) * g.inv_binw[c]);
    y[c] = (float)(u[0] * st.A[c] + u[1] * st.A[3 + c] + u[2] * st.A[6 + c]);
  }
  t_out = make_float4(t[0], t[1], t[2], 0.0f);
  y_out = make_float4(y[0], y[1], y[2], 0.0f);
}

// Per atom: its bin, its place in the bin grid and its wrapped FP32 position
// (so that the neighbor kernels need no FP64 set-up).
__global__ void k_bin_assign(const GmpStruct* S, const GmpGrid* G,
                             const int32_t* __restrict__ struct_of, int64_t N,
                             const GmpD4* __restrict__ atom_u, int32_t* __restrict__ atom_bin,
                             int32_t* __restrict__ bin_count, float4* __restrict__ atom_t,
                             float4* __restrict__ atom_y) {
  gmp_let_next_start();
  const unsigned tid = gmp_after_predecessor(threadIdx.x);
  for (int64_t a = blockIdx.x * (int64_t)blockDim.x + tid; a < N;
       a += (int64_t)gridDim.x * blockDim.x) {
    const int s = struct_of[a];
    const GmpD4 u4 = atom_u[a];
    const double u[3] = {u4.x, u4.y, u4.z};
    const int32_t bin = (int32_t)(S[s].bin_base + bin_of(G[s], u));
    atom_bin[a] = bin;
    atomicAdd(&bin_count[bin], 1);
    center_place(S[s], G[s], u, atom_t[a], atom_y[a]);
  }
}

// Per reference point: the checks, wrap and double-float split of
// k_prepare and the place of k_bin_assign, in the structure's atom grid.
__global__ void k_point_prepare(const GmpStruct* S, const GmpGrid* G,
                                const int32_t* __restrict__ point_struct, int64_t n, const double* __restrict__ pts,
                                const double* __restrict__ atom_pos, float4* __restrict__ pt_xh,
                                float4* __restrict__ pt_xl, float4* __restrict__ pt_t, float4* __restrict__ pt_y,
                                uint32_t* __restrict__ err) {
  gmp_let_next_start();
  const unsigned tid = gmp_after_predecessor(threadIdx.x);
  for (int64_t a = blockIdx.x * (int64_t)blockDim.x + tid; a < n;
       a += (int64_t)gridDim.x * blockDim.x) {
    const int s = point_struct[a];
    const GmpStruct& st = S[s];
    double x[3] = {pts[3 * a], pts[3 * a + 1], pts[3 * a + 2]};
    if (!isfinite(x[0]) || !isfinite(x[1]) || !isfinite(x[2])) {
      atomicOr(err, GMP_DEV_NONFINITE);
      x[0] = x[1] = x[2] = 0.0;
    }
    double u[3], f0[3];
    int w[3] = {0, 0, 0};
    struct_ref_cell(st, atom_pos, f0);  // the reference cell of the structure's atoms
    for (int k = 0; k < 3; ++k) {
      u[k] = x[0] * st.Ainv[k] + x[1] * st.Ainv[3 + k] + x[2] * st.Ainv[6 + k];
      if (st.periodic[k]) w[k] = wrap_axis(u[k], f0[k], err);
    }
    write_split(a, x, 0, w, pt_xh, pt_xl);
    center_place(st, G[s], u, pt_t[a], pt_y[a]);
  }
}

// Batches of small structures: the whole binning (k_prepare, k_grid,
// k_bin_assign, the scan, k_bin_scatter, k_bin_place) in one launch, a CTA per
// structure, with its coordinates, bin counts, offsets and slot lists in shared
// memory; same outputs as those kernels (bins hold their atoms in index order).
// A structure's atoms and bins are contiguous in the batch, so its bin offsets
// need no scan over the others.  Small structures spend most of the
// multi-kernel binning in launch and tail latency, not work.  Also writes
// struct_of.  Measured on a GB300 (neighbor stage; this kernel / the several):
// one structure of 16 atoms 22 / 27 us, of 256 28 / 28, of 512 38 / 29; 16 of
// 512 53 / 65; 150 of 64 47 / 61; eight batches of 100 structures of 8-256
// atoms 384 / 451.  So it takes batches whose largest structure has up to 256
// atoms, or 512 when the batch holds at least 16 times as many (with larger
// ones the shared memory keeps small structures from filling the chip).
struct StructBins {
  GmpStruct st;
  GmpGrid g;
  double f0[3];                // reference cell (struct_ref_cell)
  unsigned long long bbox[6];  // as prepare_atom's
  GridAxes axes;
  int32_t warp_tot[32];
};
__host__ __device__ inline size_t struct_bins_smem(int n_atoms, int n_bins) {
  return sizeof(StructBins) + (3 * sizeof(double) + 2 * sizeof(int32_t)) * (size_t)n_atoms +
         sizeof(int32_t) * (2 * (size_t)n_bins + 1);
}

__global__ void __launch_bounds__(1024) k_bin_structs(GmpStruct* __restrict__ S, double cutoff, const double* __restrict__ pos,
                                                     const int32_t* __restrict__ species, int n_el,
                                                     GmpGrid* __restrict__ G, int32_t* __restrict__ struct_of,
                                                     float4* atom_xh, float4* atom_xl, int32_t* __restrict__ bin_start,
                                                     float4* __restrict__ bin_y, int2* __restrict__ bin_je,
                                                     float4* __restrict__ atom_t, float4* __restrict__ atom_y,
                                                     uint32_t* __restrict__ err, int n_clear) {
  extern __shared__ __align__(16) unsigned char sm_bins[];
  StructBins& B = *reinterpret_cast<StructBins*>(sm_bins);
  gmp_let_next_start();
  const int tid = (int)gmp_after_predecessor(threadIdx.x), nt = blockDim.x, lane = tid & 31, wid = tid >> 5;
  const int s = blockIdx.x;
  if (s == 0)
    for (int t = tid; t < n_clear; t += nt) err[1 + t] = 0;
  {
    const int32_t* src = reinterpret_cast<const int32_t*>(S + s);
    int32_t* dst = reinterpret_cast<int32_t*>(&B.st);
    for (int t = tid; t < (int)(sizeof(GmpStruct) / 4); t += nt) dst[t] = src[t];
    src = reinterpret_cast<const int32_t*>(G + s);
    dst = reinterpret_cast<int32_t*>(&B.g);
    for (int t = tid; t < (int)(sizeof(GmpGrid) / 4); t += nt) dst[t] = src[t];
    if (tid < 6) B.bbox[tid] = ~0ull;
  }
  __syncthreads();
  const GmpStruct& st = B.st;
  const int n = st.n_atoms;
  const int64_t a0 = st.atom_base;
  const bool open = !all_periodic(st);
  double* const us = reinterpret_cast<double*>(sm_bins + sizeof(StructBins));  // [n][3]
  int32_t* const slot_atom = reinterpret_cast<int32_t*>(us + 3 * (size_t)n);   // [n] atom of each slot
  int32_t* const bin = slot_atom + n;                                          // [n]
  if (tid < 3) B.f0[tid] = ref_cell_axis(st, pos, tid);
  __syncthreads();
  for (int t0 = 0; t0 < n; t0 += nt) {
    const int t = t0 + tid;
    unsigned long long lo[3], hi[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) lo[k] = hi[k] = ~0ull;
    if (t < n) {
      double x[3];
      const int e = load_atom(a0 + t, pos, species, n_el, x, err);
      int w[3] = {0, 0, 0};
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        double u = x[0] * st.Ainv[k] + x[1] * st.Ainv[3 + k] + x[2] * st.Ainv[6 + k];
        if (st.periodic[k]) {
          w[k] = wrap_axis(u, B.f0[k], err);
        } else {
          lo[k] = order_key(u);
          hi[k] = ~lo[k];
        }
        us[3 * t + k] = u;
      }
      write_split(a0 + t, x, e, w, atom_xh, atom_xl);
      struct_of[a0 + t] = s;
    }
    if (open) {
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        if (st.periodic[k]) continue;
        for (int o = 16; o; o >>= 1) {
          lo[k] = min(lo[k], __shfl_xor_sync(0xffffffffu, lo[k], o));
          hi[k] = min(hi[k], __shfl_xor_sync(0xffffffffu, hi[k], o));
        }
        if (lane == 0) {
          atomicMin(&B.bbox[2 * k], lo[k]);
          atomicMin(&B.bbox[2 * k + 1], hi[k]);
        }
      }
    }
  }
  __syncthreads();
  if (open && tid < 32) {
    if (tid < 3) grid_axis(st, B.bbox, B.g, B.axes, tid);
    __syncwarp();
    if (tid == 0) {
      grid_rest(B.st, B.g, B.axes, cutoff);
      G[s] = B.g;
      S[s].prescreen2 = st.prescreen2;
      S[s].inside2 = st.inside2;
    }
  }
  __syncthreads();
  const GmpGrid& g = B.g;
  const int n_bins = g.nb[0] * g.nb[1] * g.nb[2];  // at most bin_cap
  int32_t* const cnt = bin + n;                    // [n_bins] counts, then cursors
  int32_t* const start = cnt + n_bins;             // [n_bins + 1] exclusive offsets
  for (int b = tid; b < n_bins; b += nt) cnt[b] = 0;
  __syncthreads();
  for (int t = tid; t < n; t += nt) {
    const int b = (int)bin_of(g, us + 3 * t);
    bin[t] = b;
    atomicAdd(&cnt[b], 1);
  }
  __syncthreads();
  // exclusive scan of the counts: a contiguous chunk per thread, then the
  // chunk totals across the block
  const int chunk = (n_bins + nt - 1) / nt;
  const int c0 = min(tid * chunk, n_bins), c1 = min(c0 + chunk, n_bins);
  int32_t run = 0;
  for (int b = c0; b < c1; ++b) run += cnt[b];
  int32_t incl = run;
  for (int o = 1; o < 32; o <<= 1) {
    const int32_t v = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += v;
  }
  if (lane == 31) B.warp_tot[wid] = incl;
  __syncthreads();
  int32_t off = incl - run;
  for (int w = 0; w < wid; ++w) off += B.warp_tot[w];
  for (int b = c0; b < c1; ++b) {
    const int32_t c = cnt[b];
    start[b] = off;
    cnt[b] = off;  // cursor
    off += c;
  }
  if (tid == 0) start[n_bins] = n;
  __syncthreads();
  for (int t = tid; t < n; t += nt) slot_atom[atomicAdd(&cnt[bin[t]], 1)] = t;
  __syncthreads();
  // each bin's atoms in index order (insertion sort; a bin holds few atoms)
  for (int b = tid; b < n_bins; b += nt) {
    const int b0 = start[b], b1 = start[b + 1];
    for (int t = b0 + 1; t < b1; ++t) {
      const int32_t v = slot_atom[t];
      int u = t - 1;
      while (u >= b0 && slot_atom[u] > v) {
        slot_atom[u + 1] = slot_atom[u];
        --u;
      }
      slot_atom[u + 1] = v;
    }
  }
  __syncthreads();
  // (the last offset, n, is also the next structure's first: same value)
  for (int b = tid; b <= n_bins; b += nt) bin_start[st.bin_base + b] = (int32_t)a0 + start[b];
  for (int t = tid; t < n; t += nt) {
    const int v = slot_atom[t];
    const int64_t a = a0 + v;
    float4 place, y;
    center_place(st, g, us + 3 * v, place, y);
    atom_t[a] = place;
    atom_y[a] = y;
    write_slot(a, (int32_t)(a0 + t), y, atom_xh[a].w, atom_xl[a].w, bin_y, bin_je);
  }
}

// ------------------------------------------------------------------ scan
template <typename T>
__global__ void k_scan_block(const T* __restrict__ in, T* __restrict__ out, T* __restrict__ sums,
                             int64_t n) {
  __shared__ T sh[1024];
  const int64_t base = (int64_t)blockIdx.x * 1024;
  gmp_let_next_start();
  const int t = gmp_after_predecessor(threadIdx.x);
  T v = (base + t < n) ? in[base + t] : T(0);
  sh[t] = v;
  __syncthreads();
  for (int off = 1; off < 1024; off <<= 1) {
    T add = (t >= off) ? sh[t - off] : T(0);
    __syncthreads();
    sh[t] += add;
    __syncthreads();
  }
  if (base + t < n) out[base + t] = sh[t] - v;  // exclusive
  if (t == 1023) sums[blockIdx.x] = sh[1023];
}

template <typename T>
__global__ void k_scan_add(T* out, const T* offs, int64_t n) {
  gmp_let_next_start();
  const unsigned tid = gmp_after_predecessor(threadIdx.x);
  const int64_t i = (int64_t)blockIdx.x * 1024 + tid;
  if (i < n) out[i] += offs[blockIdx.x];
  if (i == 0) out[n] = offs[gridDim.x];  // the total
}

// The whole scan in one CTA, 4096 values at a time: one launch where the
// block scan, the scan of its sums and the addition take three, each of
// them 3-4 us of latency.  Up to 4 rounds (16384 values, 5 us).
constexpr int64_t kScanOneCta = 16384;
template <typename T>
__global__ void __launch_bounds__(1024) k_scan_one(const T* __restrict__ in, T* __restrict__ out, int64_t n) {
  __shared__ T tot[32];
  gmp_let_next_start();
  const int t = gmp_after_predecessor(threadIdx.x), lane = t & 31, wid = t >> 5;
  T carry = 0;
  for (int64_t base = 0; base < n; base += 4096) {
    const int64_t i0 = base + 4 * t;
    T v[4], run = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      v[k] = run;
      if (i0 + k < n) run += in[i0 + k];
    }
    T incl = run;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const T u = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += u;
    }
    if (lane == 31) tot[wid] = incl;
    __syncthreads();
    T w = tot[lane];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const T u = __shfl_up_sync(0xffffffffu, w, o);
      if (lane >= o) w += u;
    }
    const T before = __shfl_sync(0xffffffffu, w, (wid + 31) & 31);
    const T off = carry + (wid ? before : T(0)) + (incl - run);
#pragma unroll
    for (int k = 0; k < 4; ++k)
      if (i0 + k < n) out[i0 + k] = off + v[k];
    carry += __shfl_sync(0xffffffffu, w, 31);
    __syncthreads();
  }
  if (t == 0) out[n] = carry;
}

// out[0..n] exclusive scan of in[0..n-1]; out[n] = total.  tmp sized by
// gmp_scan_tmp_bytes(n).
template <typename T>
cudaError_t exclusive_scan(const T* in, T* out, int64_t n, void* tmp, cudaStream_t st,
                           int64_t* launches) {
  if (n <= 0) {
    return cudaMemsetAsync(out, 0, sizeof(T), st);
  }
  if (n <= kScanOneCta) {
    GMP_TRY(gmp_launch_next(k_scan_one<T>, 1, 1024, 0, st, in, out, n));
    ++*launches;
    return cudaGetLastError();
  }
  const int64_t nb = (n + 1023) / 1024;
  T* sums = (T*)tmp;
  T* sums_scan = sums + nb + 1;
  void* rest = (void*)(sums_scan + nb + 1);
  GMP_TRY(gmp_launch_next(k_scan_block<T>, (unsigned)nb, 1024, 0, st, in, out, sums, n));
  ++*launches;
  const cudaError_t e = exclusive_scan<T>(sums, sums_scan, nb, rest, st, launches);
  if (e != cudaSuccess) return e;
  GMP_TRY(gmp_launch_next(k_scan_add<T>, (unsigned)nb, 1024, 0, st, out, sums_scan, n));
  ++*launches;
  return cudaGetLastError();
}

// ----------------------------------------------------------- neighbor pass
// The FP64 expression of the neighbor definition, evaluated exactly as written.
__device__ __noinline__ bool fp64_within(const double* __restrict__ pos, const double* __restrict__ xi,
                                         int64_t j, const GmpStruct& st, const int* n, double rc2) {
  double d[3];
  for (int c = 0; c < 3; ++c) {
    double sh = __dadd_rn(__dadd_rn(__dmul_rn((double)n[0], st.A[c]), __dmul_rn((double)n[1], st.A[3 + c])),
                          __dmul_rn((double)n[2], st.A[6 + c]));
    d[c] = __dadd_rn(__dsub_rn(pos[3 * j + c], xi[c]), sh);
  }
  double r2 = __dadd_rn(__dadd_rn(__dmul_rn(d[0], d[0]), __dmul_rn(d[1], d[1])), __dmul_rn(d[2], d[2]));
  return r2 < rc2;
}

__device__ __forceinline__ bool exact_accept(const double* __restrict__ pos, const double* __restrict__ xi, int64_t j,
                                             const float4& xhi, const float4& xli, const float4& xhj,
                                             const float4& xlj, const GmpStruct& st, const int* n,
                                             float rc2hi, float rc2lo, double rc2, float cutoff) {
  gmp_f2 d[3], r2;
  float mag;
  gmp_df_disp<true>(xhi, xli, xhj, xlj, st, n, d, r2, &mag);
  gmp_f2 diff = gmp_df_add(r2, gmp_f2{-rc2hi, -rc2lo});
  // double-float error bound (generous): 2^-36 (mag + rc + 1) (rc + 1) * 16
  const float tol = ldexpf((mag + cutoff + 1.0f) * (cutoff + 1.0f) * 16.0f, -36);
  if (diff.hi < -tol) return true;
  if (diff.hi > tol) return false;
  return fp64_within(pos, xi, j, st, n, rc2);
}

// An image index that does not fit the packed shift.
__device__ __forceinline__ bool out_of_range(const int* n) {
  return abs(n[0]) >= 512 || abs(n[1]) >= 512 || abs(n[2]) >= 512;
}

// Per-warp shared memory: 32 bin segments (float4 + int); in the fill passes also
// keys [max_keys] u64, and to group them by species (FILL 1) species and rank of
// each key [max_keys] u32, per-species counters [n_el] int.
constexpr size_t kSegBytes = 32 * (sizeof(float4) + sizeof(int));
__host__ __device__ inline size_t warp_bytes(int fill, int max_keys, int n_el) {
  if (fill == 0) return kSegBytes;
  return kSegBytes + ((size_t)max_keys * (fill == 1 ? 12 : 8) + (fill == 1 ? (size_t)n_el * 4 : 0) + 15) / 16 * 16;
}

// Warp per center.  The center's cutoff sphere is covered by segments: the
// bins of one row (fixed bins b1, b2 of axes 1 and 2, one image m0 of axis
// 0), whose slots are contiguous.  A lane sets up one segment, 32 at a time:
// a row farther than the cutoff from the center is left out, and with
// orthogonal axes the row is cut to the sphere's chord (bounds on the
// distance between planes, with a slack of kSlack bins that covers the FP32
// rounding of t; the test of each candidate is exact, so the bounds only have
// to keep every neighbor).  The slots of the segments that are not empty are
// then numbered through and taken 32 at a time, a lane's segment found from a
// bit mask of the segments that start among the 32: every lane has a
// candidate, and consecutive lanes read consecutive slots.
// An accepted candidate is kept as (slot, image) and completed afterwards,
// with all lanes busy; a row costs two bin offsets instead of two per bin.
// Bound by instruction issue (60-65%) and the loads' latency; 64 registers, 32
// resident warps per SM (14 words spilled; 80 registers and 24 warps:
// 147 us on the slab of 32,768 atoms, 130 at 64).  Neighbor stage of 2,500 small
// structures / of the alloy slab of 262,144 atoms (GB300): 946 / 1774 us with
// one bin per lane, its slots in turn; 562 / 1004 with groups of 8 lanes walking
// the segments, 4 at a time; 508 / 900 now.
// FILL = 0: count exact neighbors; FILL = 1: write the
// pair records grouped by neighbor species, in enumeration order within a
// species (segments in a fixed order, atoms in index order within a bin:
// deterministic); FILL = 2: sorted by (neighbor atom, image).
constexpr float kSlack = 1e-3f;
template <int FILL>
__global__ void __launch_bounds__(128, 8) k_neighbors(const GmpStruct* S, const GmpGrid* G,
                            const GmpCenters C, int64_t N, float cutoff,
                            float rc2hi, float rc2lo, double rc2, const double* __restrict__ pos,
                            const float4* __restrict__ atom_xh, const float4* __restrict__ atom_xl,
                            const int32_t* __restrict__ bin_start, const float4* __restrict__ bin_y,
                            const int2* __restrict__ bin_je, int n_el,
                            int64_t* __restrict__ counts, const int64_t* __restrict__ offsets,
                            unsigned long long* __restrict__ cursor, int64_t* __restrict__ rng,
                            GmpPair* __restrict__ pairs, int64_t pair_cap, int max_keys,
                            int32_t* __restrict__ maxm, uint32_t* __restrict__ err) {
  extern __shared__ __align__(16) unsigned char sh_fill[];
  constexpr int fill = FILL;
  gmp_let_next_start();
  const unsigned tid = gmp_after_predecessor(threadIdx.x);
  const int lane = tid & 31;
  const int wib = tid >> 5;
  const int64_t i = (int64_t)blockIdx.x * (blockDim.x >> 5) + wib;
  if (i >= N) return;
  unsigned char* wbase = sh_fill + (size_t)wib * warp_bytes(fill, max_keys, n_el);
  float4* seg_sh = reinterpret_cast<float4*>(wbase);          // image shift of the segment, slot of candidate 0
  int* seg_m = reinterpret_cast<int*>(seg_sh + 32);           // packed image (m0, m1, m2)
  const unsigned below = (1u << lane) - 1u;
  int2* keys = reinterpret_cast<int2*>(wbase + kSegBytes);    // accepted: slot, packed image (m0, m1, m2)
  uint32_t* kel = reinterpret_cast<uint32_t*>(keys + max_keys);
  int* ecnt = reinterpret_cast<int*>(kel + max_keys);  // max_keys: a power of 2 >= 32

  const int s = C.sid[i];
  const GmpStruct& st = S[s];
  const GmpGrid& g = G[s];
  const float p2 = st.prescreen2, q2 = st.inside2;
  const float4 xhi = C.xh[i], xli = C.xl[i];
  const double* xi = C.pos + 3 * i;
  int wi[3];
  gmp_unpack_shift(__float_as_int(xli.w), wi);
  const float4 yi = C.y[i];
  int count = 0;   // per lane (count pass) / per warp (fill passes)
  {
    const float4 t4 = C.t[i];
    const float t[3] = {t4.x, t4.y, t4.z};
    int nb[3], lo[3], hi[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      nb[k] = g.nb[k];
      // FP32 bounds as integers (a point far outside the atoms' range
      // saturates and comes out empty after the clamp)
      lo[k] = __float2int_rd(t[k] - g.rb[k] - kSlack);
      hi[k] = __float2int_rd(t[k] + g.rb[k] + kSlack);
      if (!st.periodic[k]) {
        lo[k] = max(lo[k], 0);
        hi[k] = min(hi[k], nb[k] - 1);
      }
    }
    const int im0 = st.periodic[0] ? floor_div(lo[0], nb[0]) : 0;  // images of axis 0
    const int n0 = st.periodic[0] ? floor_div(hi[0], nb[0]) - im0 + 1 : (hi[0] >= lo[0] ? 1 : 0);
    const int n1 = max(hi[1] - lo[1] + 1, 0), n2 = max(hi[2] - lo[2] + 1, 0);
    const int total = n0 * n1 * n2;
    const float rcs = cutoff * cutoff * 1.00001f;
    for (int r0 = 0; r0 < total; r0 += 32) {
      const int cidx = r0 + lane;
      float4 sg = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
      int2 cm = make_int2(0, 0);
      if (cidx < total) {
        // segment (c0, c1, c2); the single-precision quotients hold while
        // the operands are below 2^20 (beyond it a cutoff of over 50 cell
        // widths, whose image count exceeds the per-center limit)
        const bool small = total < (1 << 20);
        const int t01 = small ? floor_div_small(cidx, n0) : cidx / n0;
        const int c2 = small ? floor_div_small(t01, n1) : t01 / n1;
        const int b1 = lo[1] + (t01 - c2 * n1), b2 = lo[2] + c2;
        const float g1 = fmaxf(fmaxf((float)b1 - t[1], t[1] - (float)(b1 + 1)) - kSlack, 0.0f) * g.h[1];
        const float g2 = fmaxf(fmaxf((float)b2 - t[2], t[2] - (float)(b2 + 1)) - kSlack, 0.0f) * g.h[2];
        // squared room left along axis 0 (or, with skew axes, only a bound
        // from each pair of planes alone)
        const float gm = fmaxf(g1, g2);
        const float room = rcs - (g.ortho ? g1 * g1 + g2 * g2 : gm * gm);
        if (room >= 0.0f) {
          const int m0 = im0 + (cidx - t01 * n0);
          int x0 = lo[0], x1 = hi[0], m1 = 0, m2 = 0, w0 = 0;
          if (g.ortho) {
            const float c = __fsqrt_rn(room) * g.inv_h0 + kSlack;
            x0 = max(x0, __float2int_rd(t[0] - c));
            x1 = min(x1, __float2int_rd(t[0] + c));
          }
          if (st.periodic[0]) {
            w0 = m0 * nb[0];
            x0 = max(x0, w0);
            x1 = min(x1, w0 + nb[0] - 1);
          }
          if (st.periodic[1]) m1 = small ? floor_div_small(b1, nb[1]) : floor_div(b1, nb[1]);
          if (st.periodic[2]) m2 = small ? floor_div_small(b2, nb[2]) : floor_div(b2, nb[2]);
          if (x0 <= x1) {
            const int64_t bin = st.bin_base + (int64_t)nb[0] * ((b1 - m1 * nb[1]) + (int64_t)nb[1] * (b2 - m2 * nb[2])) - w0;
            const int first = bin_start[bin + x0];
            cm = make_int2(bin_start[bin + x1 + 1] - first, gmp_pack_shift(m0, m1, m2));
            const float f0 = (float)m0, f1 = (float)m1, f2 = (float)m2;
            sg = make_float4(f0 * st.Ahi[0] + f1 * st.Ahi[3] + f2 * st.Ahi[6],
                             f0 * st.Ahi[1] + f1 * st.Ahi[4] + f2 * st.Ahi[7],
                             f0 * st.Ahi[2] + f1 * st.Ahi[5] + f2 * st.Ahi[8], __int_as_float(first));
          }
        }
      }
      // the candidates of the segments that are not empty, numbered through:
      // lane's segment starts at candidate `start`
      int incl = cm.x;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += v;
      }
      const int start = incl - cm.x, n_cand = __shfl_sync(0xffffffffu, incl, 31);
      const unsigned some = __ballot_sync(0xffffffffu, cm.x > 0);
      if (cm.x > 0) {
        const int at = __popc(some & below);
        sg.w = __int_as_float(__float_as_int(sg.w) - start);
        seg_sh[at] = sg;
        seg_m[at] = cm.y;
      }
      __syncwarp();
      int q0 = -1;  // segments that start before candidate c0, less one
      for (int c0 = 0; c0 < n_cand; c0 += 32) {
        // bit b: a segment starts at candidate c0 + b
        const unsigned heads = __reduce_or_sync(0xffffffffu, cm.x > 0 && (unsigned)(start - c0) < 32u ? 1u << (start - c0) : 0u);
        const int q = q0 + __popc(heads & (below << 1 | 1u));
        q0 += __popc(heads);
        const int cand = c0 + lane;
        int slot = 0, cy = 0;
        bool acc = false;
        if (cand < n_cand) {
          const float4 sh = seg_sh[q];
          cy = seg_m[q];
          slot = __float_as_int(sh.w) + cand;
          const float4 yj = bin_y[slot];
          const float dx = (yj.x - yi.x) + sh.x;
          const float dy = (yj.y - yi.y) + sh.y;
          const float dz = (yj.z - yi.z) + sh.z;
          // three roundings of non-negative terms: within 3 x 2^-24 relative
          const float r2 = __fmaf_rn(dx, dx, __fmaf_rn(dy, dy, __fmul_rn(dz, dz)));
          acc = r2 <= p2;
          // the image index is needed for the boundary shell's exact
          // decision, and in the count pass (whose caller reports it) for
          // its range
          if (acc && (!fill || r2 >= q2)) {
            int wj[3], m[3];
            gmp_unpack_shift(__float_as_int(yj.w), wj);
            gmp_unpack_shift(cy, m);
            const int n[3] = {m[0] + wi[0] - wj[0], m[1] + wi[1] - wj[1], m[2] + wi[2] - wj[2]};
            if (r2 >= q2) {
              const int64_t j = bin_je[slot].x;
              const float4 xhj = atom_xh[j], xlj = atom_xl[j];
              acc = exact_accept(pos, xi, j, xhi, xli, xhj, xlj, st, n, rc2hi, rc2lo, rc2, cutoff);
            }
            if (!fill && acc && out_of_range(n)) {
              atomicOr(err, GMP_DEV_SHIFT_RANGE);  // reported after the count pass
              acc = false;
            }
          }
        }
        if (!fill) {
          count += acc ? 1 : 0;
        } else {
          const unsigned mask = __ballot_sync(0xffffffffu, acc);
          const int slot_k = count + __popc(mask & below);
          if (acc && slot_k < max_keys) keys[slot_k] = make_int2(slot, cy);
          count += __popc(mask);
        }
      }
      __syncwarp();
    }
  }
  if (!fill) {
    for (int o = 16; o; o >>= 1) count += __shfl_xor_sync(0xffffffffu, count, o);
    if (lane == 0) {
      counts[i] = count;
      atomicMax(maxm, count);
    }
    return;
  }
  __syncwarp();
  const int M = count;
  int64_t base;
  if (cursor) {
    // single pass (no count pass before): this center's block is allocated
    // here; its range goes to rng[i], rng[N + i]; a block beyond the
    // capacity guessed from an earlier call is flagged and the caller
    // repeats the build with the two-pass scheme
    unsigned long long b = 0;
    if (lane == 0) {
      b = atomicAdd(cursor, (unsigned long long)M);
      atomicMax(maxm, M);
    }
    base = (int64_t)__shfl_sync(0xffffffffu, b, 0);
    const bool over = base + M > pair_cap || M > max_keys;
    if (lane == 0) {
      rng[i] = over ? 0 : base;
      rng[N + i] = over ? 0 : base + M;
    }
    if (over) {
      // the first to find it closes the work counters: what is queued behind
      // these lists would be thrown away (slabs of 131,072 atoms, lattice constants
      // 3.95 and 3.7 A, in turn through one handle, orders 0-6 x 16 sigmas: the
      // denser one's features 7.4 -> 4.5 ms, with gradients 15.0 -> 8.5; GB300)
      uint32_t before = 0;
      if (lane == 0) before = atomicOr(err, GMP_DEV_CAPACITY);
      if (!(__shfl_sync(0xffffffffu, before, 0) & GMP_DEV_CAPACITY))
        for (int q = lane; q < kCounters; q += 32) atomicMax(reinterpret_cast<int*>(err) + kScalarCounters / 4 + q, kCounterClosed);
      return;
    }
  } else {
    base = offsets[i];
    if (offsets[i + 1] > pair_cap || M > max_keys) {  // capacities fixed in advance (graph replay)
      if (lane == 0) atomicOr(err, GMP_DEV_CAPACITY);
      return;
    }
    if (M != (int)(offsets[i + 1] - base)) {
      if (lane == 0) atomicOr(err, GMP_DEV_TOO_MANY_NEIGHBORS);
      return;
    }
  }
  // image index of an accepted slot's atom from its packed (m0, m1, m2) and
  // wrap; one that does not fit is flagged and replaced, so that the sort keys
  // and records made from it keep naming their atom (10 bits an axis)
  auto image = [&](int m, int wrap, int* n) {
    int wj[3], mm[3];
    gmp_unpack_shift(wrap, wj);
    gmp_unpack_shift(m, mm);
#pragma unroll
    for (int k = 0; k < 3; ++k) n[k] = mm[k] + wi[k] - wj[k];
    if (out_of_range(n)) {
      atomicOr(err, GMP_DEV_SHIFT_RANGE);
      n[0] = n[1] = n[2] = 0;
    }
  };
  unsigned long long* skey = reinterpret_cast<unsigned long long*>(keys);
  if (fill == 2) {
    for (int t = lane; t < M; t += 32) {
      const int2 k = keys[t];
      int n[3];
      image(k.y, __float_as_int(bin_y[k.x].w), n);
      skey[t] = sort_key(bin_je[k.x].x, n);
    }
    __syncwarp();
    // bitonic sort of the M keys (padded to a power of two with ~0)
    int P2 = 1;
    while (P2 < M) P2 <<= 1;
    for (int t = M + lane; t < P2; t += 32) skey[t] = ~0ull;
    __syncwarp();
    for (int k = 2; k <= P2; k <<= 1) {
      for (int jj = k >> 1; jj > 0; jj >>= 1) {
        for (int c = lane; c < P2 / 2; c += 32) {  // comparison c: keys t and t + jj
          const int t = 2 * c - (c & (jj - 1));
          const unsigned long long a = skey[t], b = skey[t + jj];
          if ((a > b) == ((t & k) == 0)) {
            skey[t] = b;
            skey[t + jj] = a;
          }
        }
        __syncwarp();
      }
    }
  }
  const bool by_species = fill == 1 && n_el > 1;
  if (by_species) {
    // destination of key t: species-major, enumeration order within a
    // species (counting sort; lanes of one match group have one species).
    // The key's rank within its species is kept with the species, and its
    // slot makes way for its atom (neither exceeds 16 bits: max_keys records
    // fit the shared memory).
    for (int e = lane; e < n_el; e += 32) ecnt[e] = 0;
    __syncwarp();
    for (int t0 = 0; t0 < M; t0 += 32) {
      const int t = t0 + lane;
      int e = -1;
      if (t < M) {
        const int2 je = bin_je[keys[t].x];
        e = je.y;
        keys[t].x = je.x;
      }
      const unsigned grp = __match_any_sync(0xffffffffu, e);
      const int rank = __popc(grp & ((1u << lane) - 1u));
      int before = 0;
      if (t < M) {
        before = ecnt[e];
        kel[t] = (uint32_t)e << 16 | (uint32_t)(before + rank);
      }
      __syncwarp();
      if (t < M && rank == 0) ecnt[e] = before + __popc(grp);
      __syncwarp();
    }
    // exclusive prefix over the species
    int run = 0;
    for (int e0 = 0; e0 < n_el; e0 += 32) {
      const int e = e0 + lane;
      const int c = e < n_el ? ecnt[e] : 0;
      int incl = c;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += v;
      }
      if (e < n_el) ecnt[e] = run + incl - c;
      run += __shfl_sync(0xffffffffu, incl, 31);
    }
    __syncwarp();
  }
  // records: the double-float displacement, rounded to FP32
  for (int t = lane; t < M; t += 32) {
    int dst = t;
    if (by_species) dst = ecnt[kel[t] >> 16] + (int)(kel[t] & 0xffffu);
    int64_t j;
    int n[3];
    float4 xhj, xlj;
    if (fill == 2) {
      const unsigned long long key = skey[t];
      j = (int64_t)(key >> 30);
      sort_key_image(key, n);
      xhj = atom_xh[j];
      xlj = atom_xl[j];
    } else {
      const int2 k = keys[t];
      j = by_species ? k.x : bin_je[k.x].x;
      xhj = atom_xh[j];
      xlj = atom_xl[j];
      image(k.y, __float_as_int(xlj.w), n);
    }
    gmp_f2 d[3], r2;
    gmp_df_disp(xhi, xli, xhj, xlj, st, n, d, r2);
    float4* dstp = reinterpret_cast<float4*>(pairs + base + dst);
    dstp[0] = make_float4(d[0].hi + d[0].lo, d[1].hi + d[1].lo, d[2].hi + d[2].lo, r2.hi);
    dstp[1] = make_float4(r2.lo, xhj.w, __int_as_float((int32_t)j),
                          __int_as_float(gmp_pack_shift(n[0], n[1], n[2])));
  }
}

__global__ void k_unpack(int64_t P, const GmpPair* __restrict__ pairs, int32_t* __restrict__ nbr_j,
                         int32_t* __restrict__ nbr_shift) {
  gmp_let_next_start();
  const unsigned tid = gmp_after_predecessor(threadIdx.x);
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + tid; t < P;
       t += (int64_t)gridDim.x * blockDim.x) {
    GmpPair p = pairs[t];
    int n[3];
    gmp_unpack_shift(p.shift, n);
    nbr_j[t] = p.j;
    nbr_shift[3 * t] = n[0];
    nbr_shift[3 * t + 1] = n[1];
    nbr_shift[3 * t + 2] = n[2];
  }
}

// Threads per CTA of the per-atom kernels: their FP64 set-up runs at 2 lanes
// per clock and SM, so a batch too small to give every SM 256 atoms is cut
// into one-warp CTAs over more SMs (4096 atoms: 128 SMs instead of 16).
inline int atom_threads(int64_t n, int sm_count) { return n >= 256 * (int64_t)sm_count ? 256 : 32; }

inline unsigned grid_for(int64_t n, int threads, int sm_count) {
  int64_t b = (n + threads - 1) / threads;
  int64_t cap = (int64_t)sm_count * 32;
  if (b > cap) b = cap;
  if (b < 1) b = 1;
  return (unsigned)b;
}

}  // namespace

size_t gmp_scan_tmp_bytes(int64_t n) {
  size_t total = 0;
  while (true) {
    int64_t nb = (n + 1023) / 1024;
    total += 2 * (size_t)(nb + 1) * sizeof(int64_t);
    if (nb <= 1) break;
    n = nb;
  }
  return total + 256;
}

cudaError_t gmp_exclusive_scan_i64(const int64_t* in, int64_t* out, int64_t n, void* tmp,
                                   cudaStream_t stream, int64_t* launches) {
  return exclusive_scan<int64_t>(in, out, n, tmp, stream, launches);
}

void gmp_periodic_grid(GmpStruct& st, GmpGrid& g, double cutoff) {
  memset(&g, 0, sizeof(g));
  if (!all_periodic(st)) return;
  grid_struct(st, nullptr, g, cutoff);
  st.bin_cap = g.nb[0] * g.nb[1] * g.nb[2];  // known: no more are reserved, cleared and scanned
}

cudaError_t gmp_launch_neighbors_prepare(GmpStruct* d_structs, int n_struct,
                                         const int32_t* d_struct_of, int64_t N, double cutoff,
                                         const double* pos, const int32_t* species, int n_el, GmpGridMode mode,
                                         GmpGrid* d_grid, float4* atom_xh, float4* atom_xl,
                                         GmpD4* atom_u, unsigned long long* d_bbox, int64_t n_bins,
                                         int32_t* bin_count, int32_t* bin_cursor, uint32_t* d_err, int n_clear,
                                         cudaStream_t stream, int sm_count, int64_t* launches) {
  if (mode != GmpGridMode::kGiven) {
    const cudaError_t e = cudaMemsetAsync(d_bbox, 0xFF, sizeof(unsigned long long) * 6 * n_struct, stream);
    if (e != cudaSuccess) return e;
  }
  const int nt = atom_threads(N, sm_count);
  GMP_TRY(gmp_launch_next(k_prepare, grid_for(N, nt, sm_count), nt, 0, stream, d_structs, d_struct_of, N, pos,
                          species, n_el, atom_xh, atom_xl, atom_u, d_bbox, n_bins, bin_count, bin_cursor, d_err, n_clear));
  ++*launches;
  if (mode != GmpGridMode::kGiven) {
    GMP_TRY(gmp_launch_next(k_grid, (n_struct + 31) / 32, 32, 0, stream, d_structs, n_struct, d_bbox, d_grid,
                            cutoff, mode == GmpGridMode::kAll ? 1 : 0));
    ++*launches;
  }
  return cudaGetLastError();
}

cudaError_t gmp_launch_bins(const GmpStruct* d_structs, const GmpGrid* d_grid,
                            const int32_t* d_struct_of, int64_t N, int64_t n_bins,
                            int32_t* atom_bin, int32_t* bin_count, int32_t* bin_start,
                            int32_t* bin_cursor, float4* atom_t, float4* atom_y, float4* bin_y, int2* bin_je,
                            const GmpD4* atom_u, const float4* atom_xh, const float4* atom_xl, void* scan_tmp,
                            cudaStream_t stream, int sm_count, int64_t* launches) {
  const int nt = atom_threads(N, sm_count);
  GMP_TRY(gmp_launch_next(k_bin_assign, grid_for(N, nt, sm_count), nt, 0, stream, d_structs, d_grid, d_struct_of, N,
                          atom_u, atom_bin, bin_count, atom_t, atom_y));
  ++*launches;
  cudaError_t e = exclusive_scan<int32_t>(bin_count, bin_start, n_bins, scan_tmp, stream, launches);
  if (e != cudaSuccess) return e;
  // bin_count is free once scanned: it holds the slot lists (room for
  // max(n_bins, N) values)
  GMP_TRY(gmp_launch_next(k_bin_scatter, grid_for(N, 256, sm_count), 256, 0, stream, N, atom_bin, bin_start,
                          bin_cursor, bin_count));
  ++*launches;
  GMP_TRY(gmp_launch_next(k_bin_place, grid_for(N, nt, sm_count), nt, 0, stream, N, atom_bin, bin_start, bin_count,
                          atom_y, atom_xh, atom_xl, bin_y, bin_je));
  ++*launches;
  return cudaGetLastError();
}

bool gmp_bin_structs_fits(int64_t N, int max_atoms, int max_bins) {
  // (at most 2 bins an atom and 8: 26 KB of shared memory at 512 atoms)
  return max_bins <= 2 * max_atoms + 8 && (max_atoms <= 256 || (max_atoms <= 512 && N >= 16 * (int64_t)max_atoms));
}

cudaError_t gmp_launch_bin_structs(GmpStruct* d_structs, int n_struct, int64_t N, int max_atoms, int max_bins,
                                   double cutoff, const double* pos, const int32_t* species, int n_el, GmpGrid* d_grid,
                                   int32_t* d_struct_of, float4* atom_xh, float4* atom_xl, int32_t* bin_start,
                                   float4* bin_y, int2* bin_je, float4* atom_t, float4* atom_y, uint32_t* d_err,
                                   int n_clear, cudaStream_t stream, int sm_count, int64_t* launches) {
  if (!gmp_bin_structs_fits(N, max_atoms, max_bins)) return cudaErrorInvalidValue;
  const size_t smem = struct_bins_smem(max_atoms, max_bins);
  // as many threads as atoms: fewer warps to wait for at each step; with more
  // structures than SMs small CTAs, which leave room for one another
  const int most = n_struct > sm_count ? 128 : 1024;
  const int nt = std::min(most, std::max(64, (max_atoms + 31) / 32 * 32));
  GMP_TRY(gmp_launch_next(k_bin_structs, (unsigned)n_struct, nt, smem, stream, d_structs, cutoff, pos, species, n_el,
                          d_grid, d_struct_of, atom_xh, atom_xl, bin_start, bin_y, bin_je, atom_t, atom_y, d_err,
                          n_clear));
  ++*launches;
  return cudaGetLastError();
}

cudaError_t gmp_launch_point_prepare(const GmpStruct* d_structs, const GmpGrid* d_grid,
                                     const int32_t* point_struct, int64_t n_points, const double* points,
                                     const double* atom_pos, float4* pt_xh, float4* pt_xl, float4* pt_t,
                                     float4* pt_y, uint32_t* d_err, cudaStream_t stream, int sm_count,
                                     int64_t* launches) {
  if (n_points <= 0) return cudaSuccess;
  const int nt = atom_threads(n_points, sm_count);
  GMP_TRY(gmp_launch_next(k_point_prepare, grid_for(n_points, nt, sm_count), nt, 0, stream, d_structs, d_grid,
                          point_struct, n_points, points, atom_pos, pt_xh, pt_xl, pt_t, pt_y, d_err));
  ++*launches;
  return cudaGetLastError();
}

bool gmp_neighbor_keys_fit(int fill, int max_keys, int n_el) { return warp_bytes(fill, max_keys, n_el) <= 227 * 1024; }

cudaError_t gmp_launch_neighbor_pass(int fill, const GmpStruct* d_structs, const GmpGrid* d_grid,
                                     const GmpCenters& C, int64_t N, double cutoff,
                                     const double* pos, const float4* atom_xh, const float4* atom_xl,
                                     const int32_t* bin_start, const float4* bin_y, const int2* bin_je, int n_el,
                                     int64_t* counts, const int64_t* offsets,
                                     GmpPair* pairs, int64_t pair_cap, int max_keys, int32_t* d_maxm,
                                     uint32_t* d_err, cudaStream_t stream, int sm_count, int64_t* launches,
                                     unsigned long long* cursor, int64_t* rng) {
  if (fill < 0 || fill > 2 || (cursor && fill == 0)) return cudaErrorInvalidValue;
  const double rc2 = cutoff * cutoff;
  const float rc2hi = (float)rc2;
  const float rc2lo = (float)(rc2 - (double)rc2hi);
  auto fn = fill == 0 ? k_neighbors<0> : fill == 1 ? k_neighbors<1> : k_neighbors<2>;
  // few centers: one warp per CTA, so that they spread over the SMs
  int warps = N >= 16 * (int64_t)sm_count ? 4 : 1;
  while (warps > 1 && (size_t)warps * warp_bytes(fill, max_keys, n_el) > 96 * 1024) warps >>= 1;
  const size_t smem = (size_t)warps * warp_bytes(fill, max_keys, n_el);
  if (fill) {
    if (smem > 48 * 1024) {
      cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
      if (e != cudaSuccess) return e;
    }
  }
  const unsigned blocks = (unsigned)((N + warps - 1) / warps);
  GMP_TRY(gmp_launch_next(fn, blocks, warps * 32, smem, stream, d_structs, d_grid, C, N, (float)cutoff, rc2hi,
                          rc2lo, rc2, pos, atom_xh, atom_xl, bin_start, bin_y, bin_je, n_el, counts, offsets,
                          cursor, rng, pairs, pair_cap, max_keys, d_maxm, d_err));
  ++*launches;
  return cudaGetLastError();
}

cudaError_t gmp_launch_unpack_neighbors(int64_t P, const GmpPair* pairs, int32_t* nbr_j,
                                        int32_t* nbr_shift, cudaStream_t stream,
                                        int64_t* launches) {
  if (P <= 0) return cudaSuccess;
  GMP_TRY(gmp_launch_next(k_unpack, grid_for(P, 256, 152), 256, 0, stream, P, pairs, nbr_j, nbr_shift));
  ++*launches;
  return cudaGetLastError();
}
