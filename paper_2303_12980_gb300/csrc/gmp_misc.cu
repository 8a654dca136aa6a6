// Small helper kernels: structure ids, Jacobian row counts, the
// order-independent gradient sums and output, strain-derivative sums.
#include "gmp_internal.cuh"

namespace {

__global__ void k_struct_of(const int64_t* __restrict__ atom_off, int n_struct,
                            int32_t* __restrict__ struct_of) {
  for (int s = blockIdx.x; s < n_struct; s += gridDim.x) {
    const int64_t a0 = atom_off[s], a1 = atom_off[s + 1];
    for (int64_t a = a0 + threadIdx.x; a < a1; a += blockDim.x) struct_of[a] = s;
  }
}

// Distinct neighbor atoms per center (lists are sorted by atom), and for
// every pair the rank of its atom among them (the pair's Jacobian row
// within the center's rows).
__global__ void k_jac_count(int64_t N, const int64_t* __restrict__ nbr_beg, const int64_t* __restrict__ nbr_end,
                            const GmpPair* __restrict__ pairs, int64_t* __restrict__ counts,
                            int32_t* __restrict__ local_row) {
  gmp_let_next_start();
  const unsigned tid = gmp_after_predecessor(threadIdx.x);
  const int lane = tid & 31;
  const int64_t i = ((int64_t)blockIdx.x * blockDim.x + tid) >> 5;
  if (i >= N) return;
  const int64_t p0 = nbr_beg[i], p1 = nbr_end[i];
  int c = 0;  // rows so far (warp-uniform)
  for (int64_t base = p0; base < p1; base += 32) {
    const int64_t p = base + lane;
    const bool in = p < p1;
    const bool first = in && (p == p0 || pairs[p - 1].j != pairs[p].j);
    const unsigned m = __ballot_sync(0xffffffffu, first);
    if (in) local_row[p] = c + __popc(m & ((2u << lane) - 1u)) - 1;
    c += __popc(m);
  }
  if (lane == 0) counts[i] = c;
}

// own[j] + the value of j's fixed-point bins, plus acc_in (earlier passes),
// to acc_out or, after the last pass, rounded to grad_pos (bin b counts in
// units of 2^(24 b - 149); added in a fixed order, so the result does not
// depend on the order in which the bins were filled).  Bin 11 holds flags
// of non-finite contributions: NaN if any was NaN or infinities of both
// signs came in, else that infinity.  The bins are left empty for the next
// pass.  One thread per (atom, component).
__global__ void k_grad_bins_finish(int64_t n, unsigned long long* __restrict__ bins,
                                   const double* __restrict__ own, const double* acc_in, double* acc_out,
                                   float* __restrict__ grad_pos) {
  constexpr int kBins = 12;
  constexpr double kBinUnit[11] = {0x1p-149, 0x1p-125, 0x1p-101, 0x1p-77, 0x1p-53, 0x1p-29,
                                   0x1p-5,   0x1p+19,  0x1p+43,  0x1p+67, 0x1p+91};
  gmp_let_next_start();
  const unsigned tid = gmp_after_predecessor(threadIdx.x);
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + tid; t < n; t += (int64_t)gridDim.x * blockDim.x) {
    unsigned long long* bt = bins + t * kBins;
    const unsigned long long fl = bt[11];
    double v;
    if (fl) {
#pragma unroll
      for (int b = 0; b < kBins; ++b) bt[b] = 0;
      v = ((fl & 1ull) || ((fl & 6ull) == 6ull)) ? (double)NAN : ((fl & 2ull) ? (double)INFINITY : -(double)INFINITY);
    } else {
      v = 0.0;
#pragma unroll
      for (int b = 0; b < 11; ++b)  // most are empty; the product is exact
        if (const long long x = (long long)bt[b]) {
          v = __fma_rn((double)x, kBinUnit[b], v);
          bt[b] = 0;
        }
    }
    v = own[t] + v;
    if (acc_in) v = acc_in[t] + v;
    if (grad_pos) grad_pos[t] = (float)v;
    else acc_out[t] = v;
  }
}

// virial[s] = (first) or += the sum over the centers of structure s of
// vir_c[center] (nine values), one warp per structure, lanes over centers in a fixed order.
__global__ void k_virial_reduce(int n_struct, const int64_t* __restrict__ atom_off, const double* __restrict__ vir_c,
                                double* __restrict__ virial, bool first) {
  gmp_let_next_start();
  const unsigned tid = gmp_after_predecessor(threadIdx.x);
  const int lane = tid & 31;
  const int64_t w0 = ((int64_t)blockIdx.x * blockDim.x + tid) >> 5;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t s = w0; s < n_struct; s += nw) {
    const int64_t a0 = atom_off[s], a1 = atom_off[s + 1];
    double acc[9];
#pragma unroll
    for (int v = 0; v < 9; ++v) acc[v] = 0.0;
    for (int64_t a = a0 + lane; a < a1; a += 32)
#pragma unroll
      for (int v = 0; v < 9; ++v) acc[v] += vir_c[9 * a + v];
#pragma unroll
    for (int v = 0; v < 9; ++v) {
      double x = acc[v];
#pragma unroll
      for (int o = 16; o; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
      if (lane == 0) virial[9 * s + v] = first ? x : virial[9 * s + v] + x;
    }
  }
}

}  // namespace

cudaError_t gmp_launch_struct_of(const int64_t* d_atom_off, int n_struct, int32_t* struct_of,
                                 cudaStream_t stream, int64_t* launches) {
  const int blocks = n_struct < 65535 ? n_struct : 65535;
  k_struct_of<<<blocks > 0 ? blocks : 1, 256, 0, stream>>>(d_atom_off, n_struct, struct_of);
  ++*launches;
  return cudaGetLastError();
}

cudaError_t gmp_launch_jacobian_count(int64_t N, const int64_t* nbr_beg, const int64_t* nbr_end, const GmpPair* pairs,
                                      int64_t* counts, int32_t* local_row, cudaStream_t stream, int sm_count,
                                      int64_t* launches) {
  (void)sm_count;
  if (N <= 0) return cudaSuccess;
  const int64_t threads = N * 32;
  GMP_TRY(gmp_launch_next(k_jac_count, (unsigned)((threads + 255) / 256), 256, 0, stream, N, nbr_beg, nbr_end, pairs,
                          counts, local_row));
  ++*launches;
  return cudaGetLastError();
}

cudaError_t gmp_launch_grad_bins_finish(int64_t N, unsigned long long* bins, const double* own,
                                        const double* acc_in, double* acc_out, float* grad_pos, cudaStream_t stream,
                                        int sm_count, int64_t* launches) {
  if (N <= 0) return cudaSuccess;
  const int64_t n = 3 * N;
  // (few values: one-warp CTAs over more SMs, for their FP64 sums)
  const int nt = n >= 256 * (int64_t)sm_count ? 256 : 32;
  int64_t blocks = (n + nt - 1) / nt;
  const int64_t cap = (int64_t)sm_count * 32;
  if (blocks > cap) blocks = cap;
  GMP_TRY(gmp_launch_next(k_grad_bins_finish, (unsigned)blocks, nt, 0, stream, n, bins, own, acc_in, acc_out, grad_pos));
  ++*launches;
  return cudaGetLastError();
}

cudaError_t gmp_launch_virial_reduce(int n_struct, const int64_t* atom_off, const double* vir_c, double* virial, bool first,
                                     cudaStream_t stream, int sm_count, int64_t* launches) {
  if (n_struct <= 0) return cudaSuccess;
  int64_t blocks = ((int64_t)n_struct * 32 + 255) / 256;
  const int64_t cap = (int64_t)sm_count * 8;
  if (blocks > cap) blocks = cap;
  GMP_TRY(gmp_launch_next(k_virial_reduce, (unsigned)blocks, 256, 0, stream, n_struct, atom_off, vir_c, virial, first));
  ++*launches;
  return cudaGetLastError();
}
