// Small-panel kernels of the randomized SVD front end (Algorithm 3) and helpers:
//   * Gram matrices of tall skinny panels (CholeskyQR and the Gram core of the thin SVD)
//   * l x l Cholesky factorisation + triangular inverse in shared memory (fp64)
//   * one-sided Jacobi eigensolver of the l x l core in shared memory, one warp per column
//     pair, rotations through warp shuffles (fp64)
//   * panel x small-matrix products, column scaling, Frobenius partial sums, scaling,
//     the counter-based Gaussian fill.
// All reductions run in a fixed order so that repeated runs are bit-identical.
#include "common.cuh"
#include "panel.cuh"

namespace defl {

// ---------------------------------------------------------------------------------------------
// Gram partials: for panel Y[b, rows, l] (fp32, leading dimension ld), CTA (chunk, batch) writes
// partial[b, chunk, l, l] = sum over its rows of y_r y_r^T  (fp32 products over 32-row groups,
// groups added in fp64).
// ---------------------------------------------------------------------------------------------
constexpr int GRAM_ROWS = 64;    // rows per CTA (256 rows: 35 us for the one panel of n = 1024 it serves)
constexpr int GRAM_SUB = 32;     // rows per fp32 sub-accumulation

__global__ void __launch_bounds__(256) gram_partial_kernel(const float* __restrict__ Y, const float* __restrict__ Y2,
                                                           long long batch_stride, int rows, int l, int ld, int nchunk,
                                                           double* __restrict__ partial) {
  pdl_wait();
  __shared__ float tile[GRAM_SUB][MAX_L + 1];
  __shared__ float tile2[GRAM_SUB][MAX_L + 1];
  const int chunk = blockIdx.x, bz = blockIdx.y, tid = threadIdx.x;
  const float* Yb = Y + (long long)bz * batch_stride;
  const float* Y2b = Y2 ? Y2 + (long long)bz * batch_stride : nullptr;
  const int tx = tid % 16, ty = tid / 16;   // 16 x 16 threads, each a 4 x 4 block of the l x l Gram
  double acc[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = 0.0;
  const int r_begin = chunk * GRAM_ROWS, r_end = min(rows, r_begin + GRAM_ROWS);
  for (int r0 = r_begin; r0 < r_end; r0 += GRAM_SUB) {
    for (int e = tid; e < GRAM_SUB * l; e += 256) {
      const int rr = e / l, c = e % l;
      const int gr = r0 + rr;
      tile[rr][c] = (gr < r_end) ? Yb[(long long)gr * ld + c] : 0.f;
      tile2[rr][c] = Y2b ? ((gr < r_end) ? Y2b[(long long)gr * ld + c] : 0.f) : tile[rr][c];
    }
    __syncthreads();
    float f[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) f[i][j] = 0.f;
    for (int rr = 0; rr < GRAM_SUB; ++rr) {
      float a[4], b[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) a[i] = (ty * 4 + i < l) ? tile[rr][ty * 4 + i] : 0.f;
#pragma unroll
      for (int j = 0; j < 4; ++j) b[j] = (tx * 4 + j < l) ? tile2[rr][tx * 4 + j] : 0.f;
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) f[i][j] = fmaf(a[i], b[j], f[i][j]);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) acc[i][j] += (double)f[i][j];
    __syncthreads();
  }
  double* out = partial + ((long long)bz * nchunk + chunk) * l * l;
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int gi = ty * 4 + i, gj = tx * 4 + j;
      if (gi < l && gj < l) out[gi * l + gj] = acc[i][j];
    }
}

int gram_num_chunks(int rows) { return (rows + GRAM_ROWS - 1) / GRAM_ROWS; }

cudaError_t gram_partial_launch(const float* Y, long long batch_stride, int batch, int rows, int l, int ld,
                                double* partial, cudaStream_t st, long long* launches, const float* Y2) {
  const int nchunk = gram_num_chunks(rows);
  launch_kernel(gram_partial_kernel, dim3(nchunk, batch), 256, 0, st, Y, Y2, batch_stride, rows, l, ld, nchunk, partial);
  if (launches) ++*launches;
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------------------------
// Cholesky of W = sum of partials (l x l, fp64), W = R^T R, output Rinv = R^-1 (upper triangular, fp32, row-major [l,l]).
// A non-positive pivot restarts with W + shift I and sets DEFL_ST_CHOL_SHIFT (bit 1) in status[b].
//
// Symmetric elimination of [W | I] in one l x l array: step j subtracts f_i = W_ij / d_j times row j from every row i > j,
// the columns right of j holding what is left of W, those up to j the unit lower factor's inverse Z as it grows (column j
// becomes -f_i). Then L^-1 = diag(d)^(-1/2) Z and R^-1 is its transpose, so factor and inverse take one sweep of l steps
// with one barrier each, and the only chain per step is barrier, pivot row, reciprocal, one multiply-add.
// Every thread keeps NR consecutive rows of one column in registers; shared memory carries only the pivot row, which is the
// pivot column too (double buffered): with the column published by one lane per group a step took 690 cycles at l = 48, 220 of
// them for that. Of 16 warps (NR >= 5) only the thread that holds the pivot works out its reciprocal, which takes four warps
// of a scheduler 220 cycles (l = 48: 29 -> 23 us); of eight or four warps every thread does, off the path of the stores
// (l = 24: 8.0 -> 7.2 us, 10.6 the other way). The
// steps run in blocks of NR, so that the pivot's place among a thread's rows is known to the compiler and who takes part
// is a comparison of warp-uniform numbers: with rows eight apart the selection took more instructions than the update.
// ---------------------------------------------------------------------------------------------
template <int NR>      // rows per thread, ceil(l / 8)
__global__ void __launch_bounds__(512) chol_inv_kernel(const double* __restrict__ partial, int nchunk, int l, int cw_log2,
                                                       float* __restrict__ Rinv, int* __restrict__ status) {
  constexpr bool OWNER = NR >= 5;
  pdl_wait();
  __shared__ double prow[2][MAX_L], pinv[2], diag[MAX_L], wdiag[MAX_L];
  const int bz = blockIdx.x, tid = threadIdx.x;
  const int c = tid & ((1 << cw_log2) - 1), g = tid >> cw_log2;       // column, group of rows g NR .. g NR + NR - 1
  const double* pb = partial + (long long)bz * nchunk * l * l;
  double w[NR], m[NR];
#pragma unroll
  for (int u = 0; u < NR; ++u) w[u] = 0.0;
  if (c < l) {
#pragma unroll 4
    for (int ch = 0; ch < nchunk; ++ch) {
      const double* pe = pb + (long long)ch * l * l + c;
#pragma unroll
      for (int u = 0; u < NR; ++u) w[u] += (g * NR + u < l) ? pe[(g * NR + u) * l] : 0.0;
    }
#pragma unroll
    for (int u = 0; u < NR; ++u) if (g * NR + u == c) wdiag[c] = w[u];
  }
  double shift = 0.0;
  bool failed = false;
  for (int attempt = 0; attempt < 6; ++attempt) {
    __syncthreads();
    // row j = a NR + u of the array as it stands, and (OWNER) the pivot's reciprocal, by the thread that holds the pivot
    auto publish = [&](int a, int u, int j) {
      if (g == a) {
        prow[j & 1][c] = m[u];
        if (OWNER && c == j) pinv[j & 1] = 1.0 / m[u];
      }
    };
#pragma unroll
    for (int u = 0; u < NR; ++u) m[u] = w[u] + ((g * NR + u == c) ? shift : 0.0);
    publish(0, 0, 0);
    __syncthreads();
    failed = false;
    for (int a = 0; a < 8 && !failed; ++a) {
#pragma unroll
      for (int u = 0; u < NR; ++u) {
        const int j = a * NR + u;
        if (j < l && !failed) {            // (uniform in the block)
          const int buf = j & 1;
          const double d = prow[buf][j], pr = prow[buf][c];       // every thread reads the pivot itself: a bad one is seen by all alike
          double f[NR];
#pragma unroll
          for (int v = 0; v < NR; ++v) f[v] = prow[buf][g * NR + v];      // W_ij = W_ji (rows past l: zeros)
          if (!(d > 0.0) || !isfinite(d)) failed = true;
          else {
            if (tid == 0) diag[j] = d;
            const double inv = OWNER ? pinv[buf] : 1.0 / d;
            // (below the pivot, column j's place becomes Z's)
            const double sc = (c == j) ? inv : inv * pr;
            if (g > a) {
#pragma unroll
              for (int v = 0; v < NR; ++v) m[v] = fma(-f[v], sc, (c == j) ? 0.0 : m[v]);
            } else if (g == a) {
#pragma unroll
              for (int v = u + 1; v < NR; ++v) m[v] = fma(-f[v], sc, (c == j) ? 0.0 : m[v]);
            }
            if (j + 1 < l) publish(u + 1 < NR ? a : a + 1, u + 1 < NR ? u + 1 : 0, j + 1);   // (into the other buffer)
          }
          __syncthreads();
        }
      }
    }
    if (!failed) break;
    // shift as in shifted CholeskyQR: proportional to the trace, growing per attempt
    double trace = 0.0;
    for (int i = 0; i < l; ++i) trace += wdiag[i];
    shift = (shift == 0.0) ? 1e-10 * (trace > 0.0 ? trace : 1.0) : shift * 100.0;
    if (tid == 0 && status) atomicOr(&status[bz], 1);
  }
  __syncthreads();          // (the last failed attempt still reads wdiag)
  // Rinv(c, r) = Z(r, c) / sqrt(d_r): upper triangular; all zeros if every attempt failed
  if (tid < l) wdiag[tid] = failed ? 0.0 : 1.0 / sqrt(diag[tid]);
  __syncthreads();
  float* out = Rinv + (long long)bz * l * l;
#pragma unroll
  for (int u = 0; u < NR; ++u) {
    const int r = g * NR + u;
    if (r < l && c < l) out[c * l + r] = failed ? 0.f : (float)(((c < r) ? m[u] : (c == r ? 1.0 : 0.0)) * wdiag[r]);
  }
}

cudaError_t chol_inv_launch(const double* partial, int nchunk, int batch, int l, float* Rinv, int* status,
                            cudaStream_t st, long long* launches) {
  const int cw_log2 = l <= 16 ? 4 : (l <= 32 ? 5 : 6);       // eight groups of rows x 16, 32 or 64 columns
  const int nr = (l + 7) / 8;
  auto kern = nr <= 1 ? chol_inv_kernel<1> : nr == 2 ? chol_inv_kernel<2> : nr == 3 ? chol_inv_kernel<3>
            : nr == 4 ? chol_inv_kernel<4> : nr == 5 ? chol_inv_kernel<5> : nr == 6 ? chol_inv_kernel<6>
            : nr == 7 ? chol_inv_kernel<7> : chol_inv_kernel<8>;
  launch_kernel(kern, batch, 8 << cw_log2, 0, st, partial, nchunk, l, cw_log2, Rinv, status);
  if (launches) ++*launches;
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------------------------
// Out[b, rows, kout] = In[b, rows, l] * Mtx[b, l(, ldm)] (first kout columns of Mtx). In-place safe.
// ---------------------------------------------------------------------------------------------
constexpr int PA_ROWS = 64;
__global__ void __launch_bounds__(256) panel_apply_kernel(const float* In, long long in_bs, int ld_in,
                                                          const float* __restrict__ Mtx, int ldm, int rows, int l,
                                                          int kout, float* Out, long long out_bs, int ld_out) {
  pdl_wait();
  __shared__ float tile[PA_ROWS][MAX_L + 1];
  __shared__ float mt[MAX_L][MAX_L + 1];
  const int bz = blockIdx.y, tid = threadIdx.x;
  const int r0 = blockIdx.x * PA_ROWS;
  const float* Ib = In + (long long)bz * in_bs;
  const float* Mb = Mtx + (long long)bz * l * ldm;
  for (int e = tid; e < l * kout; e += 256) mt[e / kout][e % kout] = Mb[(e / kout) * ldm + (e % kout)];
  for (int e = tid; e < PA_ROWS * l; e += 256) {
    const int rr = e / l, c = e % l;
    tile[rr][c] = (r0 + rr < rows) ? Ib[(long long)(r0 + rr) * ld_in + c] : 0.f;
  }
  __syncthreads();
  float* Ob = Out + (long long)bz * out_bs;
  for (int e = tid; e < PA_ROWS * kout; e += 256) {
    const int rr = e / kout, c = e % kout;
    if (r0 + rr >= rows) continue;
    float t = 0.f;
    for (int q = 0; q < l; ++q) t = fmaf(tile[rr][q], mt[q][c], t);
    Ob[(long long)(r0 + rr) * ld_out + c] = t;
  }
}

cudaError_t panel_apply_launch(const float* In, long long in_bs, int ld_in, const float* Mtx, int ldm, int batch,
                               int rows, int l, int kout, float* Out, long long out_bs, int ld_out, cudaStream_t st,
                               long long* launches) {
  if (kout <= 0) return cudaSuccess;
  launch_kernel(panel_apply_kernel, dim3((rows + PA_ROWS - 1) / PA_ROWS, batch), 256, 0, st, In, in_bs, ld_in, Mtx, ldm, rows, l,
                                                                                 kout, Out, out_bs, ld_out);
  if (launches) ++*launches;
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------------------------
// One-sided Jacobi eigensolver of the symmetric positive semidefinite core C = sum of partials
// (l x l). Columns of A = C V are rotated pairwise until mutually orthogonal; then ||a_j|| are the
// eigenvalues and the normalised columns the eigenvectors (A = C V = V diag(lambda), so V itself is not carried).
// Eight lanes per column pair (round-robin pairing), dot products by warp shuffles; fp64 throughout.
// Outputs (sorted by decreasing eigenvalue):
//   s[b, l]     = sqrt(eigenvalue)             (singular values of the panel whose Gram this is)
//   E[b, l, l]  = eigenvectors in columns      (fp32)
//   Es[b, l, l] = E diag(1/s)                  (fp32; zero column where s is numerically zero)
// With `signed_input` the matrix is a general symmetric one (Rayleigh quotient of Algorithm 2), sorted by decreasing
// magnitude, s = lambda. It is shifted by 2 ||C||_F first: the columns of C V itself are orthogonal as soon as V spans
// {v(+mu), v(-mu)}, so a pair of eigenvalues of equal magnitude and opposite sign stays mixed in them by an angle up to
// 1e-11 over the relative gap of the magnitudes; the shifted pair is far apart. The eigenvalues are the Rayleigh quotients
// v^T C v with the unshifted matrix (a copy in shared memory): as shifted norms less the shift, 1e-16 ||C||_F is all that
// would be left of a small one beside a large one. One product of C with V for it: 1 us of 50 at l = 16.
// What bounds it is the chain of dependent operations of a round (l - 1 rounds a sweep, one barrier each, half a dozen
// sweeps), not its arithmetic. Only the warps that own pairs take part in the rounds (all of the block loads the partial
// sums and writes the results). Four lanes per pair: a step of a shuffled fp64 sum takes 38 cycles, so two steps and a
// longer local sum beat three. The rotation merely steers the iteration, so its cosine and sine come from two fp32 reciprocal
// square roots (cos 2t = |d| / sqrt(d^2 + g^2), d the difference of the squared norms and g twice the inner product, both over
// the power of two above their sum) and are scaled in fp64 to c^2 + s^2 = 1; tests and angle are worked out side by side,
// without branches. A sweep is the last one when every rotation it made met a cosine below 1e-7 and turned by less than 1e-6: a
// rotation by s of columns whose cosines with a third are c leaves that third at most s c, 1e-13 at a time and 6e-12 over the 63
// rotations a column of the widest core takes part in, below the 1e-11 of the rule that ends only where nothing turns (and takes
// 0.2 sweeps of 10 more). The cosine alone is not enough: values closer than 1e-7 of the shifted norms (the small ones beside
// large ones of a signed core) turn by an angle of order one at any cosine, and mix couplings of that size back in
// (values of 1e6 beside a bulk in [-1, 1], l = 24, restated in fp64: small values off by 2.5e-2 of themselves, 5e-7 with the rule).
// ---------------------------------------------------------------------------------------------
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// four lanes of a warp add up their values (the lanes sub = 0..3 of one column pair)
__device__ __forceinline__ double group4_sum(double v) {
  v += __shfl_xor_sync(0xffffffffu, v, 1);
  v += __shfl_xor_sync(0xffffffffu, v, 2);
  return v;
}

// fp32 reciprocal square root of the hardware's approximation unit (about 1e-7, no special-case handling)
__device__ __forceinline__ float rsqrt_approx(float x) { float r; asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x)); return r; }

// The deflation gate of Algorithms 1 and 2 on the estimated magnitudes s[0..] (descending in magnitude):
//   tau <= 0: window (deflate exactly the requested number);
//   tau > 0 : if |s_window| < tau |s_1| then #{i < kmax : |s_i| > tau |s_1|}, else 0.
__device__ __forceinline__ int gate_count(const float* s, int window, int kmax, float tau) {
  int k = window;
  if (tau > 0.f && window > 0) {
    const float s1 = fabsf(s[0]);
    k = 0;
    if (fabsf(s[window - 1]) < tau * s1)
      for (int i = 0; i < kmax; ++i) if (fabsf(s[i]) > tau * s1) k = i + 1;
  }
  return k;
}

constexpr int JAC_THREADS = 256;
// doubles between columns: at least four per lane row, four more than a multiple of sixteen, so that the eight pairs of a warp,
// neighbouring columns mostly, start in different banks
__host__ __device__ constexpr int jac_stride(int nr) { return (4 * nr - 4 + 15) / 16 * 16 + 4; }

template <int NR>      // rows per lane, ceil(l / 4) rounded up to even
__global__ void __launch_bounds__(JAC_THREADS) jacobi_eig_kernel(const double* __restrict__ partial, int nchunk, int l,
                                                                 int signed_input, float* __restrict__ s_out,
                                                                 float* __restrict__ E, float* __restrict__ Es,
                                                                 int* __restrict__ status, int max_sweeps, int* __restrict__ keff,
                                                                 int window, float tau) {
  extern __shared__ double sm[];
  // column-major: A[c * ls + r], rows l .. 4 NR - 1 and column l (the padding player's) all zero, so that no access of a
  // round needs a test
  constexpr int ls = jac_stride(NR);
  double* A = sm;
  double* C = sm + (l + 1) * ls;      // signed input: the matrix before the shift, stored like A
  __shared__ double lam[MAX_L];       // column norms (eigenvalues of the scaled, shifted matrix), then the eigenvalues
  __shared__ double len[MAX_L];
  __shared__ double nrm2[MAX_L + 1];  // squared column norms of A, carried along by the rotations
  __shared__ int order[MAX_L];
  __shared__ float sorted[MAX_L];
  __shared__ int large[2];            // per parity of the sweep: a rotation with a cosine above 1e-7 or by more than 1e-6 was made
  const int bz = blockIdx.x, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const double* pb = partial + (long long)bz * nchunk * l * l;
  for (int e = tid; e < (l + 1) * ls; e += JAC_THREADS) A[e] = 0.0;
  if (tid < 2) large[tid] = 0;
  if (tid == 0) nrm2[l] = 0.0;
  __syncthreads();
  pdl_wait();
  for (int e0 = tid; e0 < l * l; e0 += 4 * JAC_THREADS) {      // four entries of a thread side by side
    double t[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll 4
    for (int ch = 0; ch < nchunk; ++ch)
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int e = e0 + u * JAC_THREADS;
        t[u] += (e < l * l) ? pb[(long long)ch * l * l + e] : 0.0;
      }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int e = e0 + u * JAC_THREADS;
      if (e < l * l) A[(e % l) * ls + e / l] = t[u];
    }
  }
  __syncthreads();
  // symmetrise (one thread per pair of entries)
  for (int e = tid; e < l * l; e += JAC_THREADS) {
    const int i = e / l, j = e % l;
    if (i < j) { const double a = 0.5 * (A[i * ls + j] + A[j * ls + i]); A[i * ls + j] = a; A[j * ls + i] = a; }
  }
  __syncthreads();
  const int np = (l + 1) & ~1;        // players, padded to even
  const int npairs = np / 2;
  const int grp = tid >> 2, sub = tid & 3;
  // Squared norms of the columns (Frobenius norm for the shift, and for the scale: the matrix is multiplied by the power
  // of two that brings its norm near one, exactly), by `nt` threads in whole warps
  auto column_norms = [&](int nt) {
    for (int j0 = 0; j0 < l; j0 += nt >> 2) {      // (the same trip count for every lane: shuffles inside)
      const int j = j0 + grp;
      double a0 = 0.0, a1 = 0.0;
#pragma unroll
      for (int i = 0; i < NR; i += 2) {
        const double v0 = A[min(j, l) * ls + sub + 4 * i], v1 = A[min(j, l) * ls + sub + 4 * i + 4];
        a0 = fma(v0, v0, a0); a1 = fma(v1, v1, a1);
      }
      const double acc = group4_sum(a0 + a1);
      if (sub == 0 && j < l) nrm2[j] = acc;
    }
  };
  column_norms(JAC_THREADS);
  __syncthreads();
  const double fro = sqrt(warp_sum((lane < l ? nrm2[lane] : 0.0) + (lane + 32 < l ? nrm2[lane + 32] : 0.0)));      // (the same in every warp)
  double scale = 1.0, unscale = 1.0;
  if (fro > 1e-290 && fro < 1e290) {
    const int ex = (int)((__double_as_longlong(fro) >> 52) & 0x7ff);             // fro in [2^(ex-1023), 2^(ex-1022))
    scale = __longlong_as_double((long long)(2046 - ex) << 52);                  // 2^(1023 - ex)
    unscale = __longlong_as_double((long long)ex << 52);
  }
  const double shift = signed_input ? 2.0 * fro * scale : 0.0;
  for (int e = tid; e < l * l; e += JAC_THREADS) {
    const int c = e / l, r = e % l;
    const double v = A[c * ls + r] * scale;
    A[c * ls + r] = v + ((r == c) ? shift : 0.0);
    if (signed_input) C[c * ls + r] = v;
  }
  if (signed_input)
    for (int e = tid; e < l * (ls - l); e += JAC_THREADS) C[(e / (ls - l)) * ls + l + e % (ls - l)] = 0.0;
  __syncthreads();
  const int nt = (npairs * 4 + 31) & ~31;          // threads of the rounds
  if (tid < nt) {
    auto sync = [&]() { asm volatile("bar.sync 1, %0;" ::"r"(nt) : "memory"); };
    int sweep = 0;
    for (; sweep < max_sweeps; ++sweep) {
      // Squared column norms, exact at the start of every sweep. Within the sweep a rotation moves
      // s (2 c gamma - s d) from one column's squared norm to the other's, so a round computes one dot product per pair
      // instead of three.
      column_norms(nt);
      sync();
      if (tid == 0) large[(sweep + 1) & 1] = 0;      // (everybody has looked at the sweep before)
      bool big = false;
      // round-robin: group g > 0 has round + g and round - g modulo np - 1, group 0 the round and the player np - 1; worked out
      // a round ahead. (A pair with the padding player meets the zero column, a group beyond the pairs nothing else: nothing
      // to rotate.)
      int one = grp == 0 ? np - 1 : grp, two = grp == 0 ? 0 : np - 1 - grp;
      if (grp >= npairs) one = two = l;
      for (int round = 0; round < np - 1; ++round) {
        const int p = min(one, two), q = max(one, two);
        if (grp < npairs) {
          if (grp > 0 && ++one == np - 1) one = 0;
          if (++two == np - 1) two = 0;
        }
        double* ap = A + p * ls + sub; double* aq = A + q * ls + sub;
        double x[NR], y[NR];
#pragma unroll
        for (int i = 0; i < NR; ++i) { x[i] = ap[4 * i]; y[i] = aq[4 * i]; }
        const double alpha = nrm2[p], beta = nrm2[q], d = beta - alpha, ab = alpha * beta;
        // 1 / (the power of two above alpha + beta), for the fp32 angle
        const double f = __hiloint2double(0x7fd00000 - (__double2hiint(alpha + beta) & 0x7ff00000), 0);
        const float df = (float)(d * f), adf = fabsf(df);
        double g0 = 0.0, g1 = 0.0;
#pragma unroll
        for (int i = 0; i < NR; i += 2) { g0 = fma(x[i], y[i], g0); g1 = fma(x[i + 1], y[i + 1], g1); }
        const double gamma = group4_sum(g0 + g1), g2 = 2.0 * gamma;
        // rotate when |gamma| > 1e-11 sqrt(alpha beta) (compared in squares): the eigenvalues are then good to about
        // 1e-22 and the vectors to 1e-11 over the relative gap, far beyond the fp32 outputs
        const double gg = gamma * gamma;
        const bool turn = gamma != 0.0 && gg > 1e-22 * ab;
        const float gf = (float)(g2 * f);
        const float h = rsqrt_approx(fmaf(gf, gf, df * df));
        const float xx = fmaf(0.5f * adf, h, 0.5f), ir = rsqrt_approx(xx);
        double c = (double)(xx * ir), sn = (double)(0.5f * copysignf(gf, __int_as_float(__float_as_int(gf) ^ __float_as_int(df))) * h * ir);
        if (turn && !(fabsf(gf) > 1e-18f)) {       // what fp32 cannot hold takes the fp64 formula
          const double zeta = d / g2, t = ((zeta >= 0.0) ? 1.0 : -1.0) / (fabs(zeta) + sqrt(1.0 + zeta * zeta));
          c = 1.0 / sqrt(1.0 + t * t); sn = c * t;
        }
        // c^2 + s^2 = 1 to fp64 rounding: 1 / sqrt(1 - e) = 1 + e/2 + 3/8 e^2 for e of 1e-6
        const double e = 1.0 - fma(c, c, sn * sn), k = fma(fma(0.375, e, 0.5), e, 1.0);
        c *= k; sn *= k;
        if (turn) {
#pragma unroll
          for (int i = 0; i < NR; ++i) { ap[4 * i] = c * x[i] - sn * y[i]; aq[4 * i] = sn * x[i] + c * y[i]; }
          const double moved = sn * fma(2.0 * c, gamma, -sn * d);
          if (sub == 0) { nrm2[p] = alpha - moved; nrm2[q] = beta + moved; }
          big |= gg > 1e-14 * ab || fabs(sn) > 1e-6;
        }
        sync();
      }
      if (big && sub == 0) large[sweep & 1] = 1;
      sync();
      if (!large[sweep & 1]) break;
    }
    if (tid == 0 && sweep >= max_sweeps && status) atomicOr(&status[bz], 2);
  }
  __syncthreads();
  // eigenvalues
  for (int j = warp; j < l; j += JAC_THREADS / 32) {
    const double* aj = A + j * ls;
    const double a0 = (lane < l) ? aj[lane] : 0.0, a1 = (lane + 32 < l) ? aj[lane + 32] : 0.0;
    const double nrm = sqrt(warp_sum(a0 * a0 + a1 * a1));
    if (lane == 0) { len[j] = nrm; lam[j] = nrm * unscale; }
  }
  __syncthreads();
  if (signed_input) {
    // lambda_j = a_j^T C a_j / ||a_j||^2, four lanes per column
    for (int j0 = 0; j0 < l; j0 += JAC_THREADS / 4) {      // (the same trip count for every lane: shuffles inside)
      const int j = min(j0 + grp, l);
      const double* aj = A + j * ls;
      double t[NR];
#pragma unroll
      for (int i = 0; i < NR; ++i) t[i] = 0.0;
      for (int c = 0; c < l; ++c) {
        const double a = aj[c];
#pragma unroll
        for (int i = 0; i < NR; ++i) t[i] = fma(C[c * ls + sub + 4 * i], a, t[i]);
      }
      double acc = 0.0;
#pragma unroll
      for (int i = 0; i < NR; ++i) acc = fma(t[i], aj[sub + 4 * i], acc);
      acc = group4_sum(acc);
      // (a zero matrix has zero columns and no shift)
      if (sub == 0 && j < l) lam[j] = (len[j] <= 1e-150) ? 0.0 : acc / (len[j] * len[j]) * unscale;
    }
    __syncthreads();
  }
  if (tid < l) {
    // (a NaN compares false with everything: it ranks as magnitude -1, after every number, so that `order` is a
    // permutation whatever the input holds)
    double mine = fabs(lam[tid]);
    if (!(mine == mine)) mine = -1.0;
    int rank = 0;
    for (int i = 0; i < l; ++i) {
      double o = fabs(lam[i]);
      if (!(o == o)) o = -1.0;
      if (o > mine || (o == mine && i < tid)) ++rank;
    }
    order[rank] = tid;
  }
  __syncthreads();
  for (int e = tid; e < l * l; e += JAC_THREADS) {
    const int r = e / l, cc = e % l;
    const int src = order[cc];
    // v_j = a_j / ||a_j||; a column that vanished (rank-deficient input) takes its unit vector, which only ever meets a
    // zero singular value
    const double v = (len[src] > 1e-150) ? A[src * ls + r] / len[src] : ((r == src) ? 1.0 : 0.0);
    const double lm = lam[src];
    const double sv = signed_input ? lm : sqrt(lm > 0.0 ? lm : 0.0);
    if (E) E[(long long)bz * l * l + e] = (float)v;
    if (Es) Es[(long long)bz * l * l + e] = (fabs(sv) > 1e-300) ? (float)(v / sv) : 0.f;
    if (r == 0) sorted[cc] = (float)sv;
    if (r == 0 && s_out) s_out[(long long)bz * l + cc] = (float)sv;
  }
  if (keff) {      // the gate on the leading `window` values (a launch of its own took 1.5 us)
    __syncthreads();
    if (tid == 0) keff[bz] = gate_count(sorted, window, window, tau);
  }
}

static const void* jacobi_form(int nr) {
  switch (nr) {
    case 2: return (const void*)jacobi_eig_kernel<2>;
    case 4: return (const void*)jacobi_eig_kernel<4>;
    case 6: return (const void*)jacobi_eig_kernel<6>;
    case 8: return (const void*)jacobi_eig_kernel<8>;
    case 10: return (const void*)jacobi_eig_kernel<10>;
    case 12: return (const void*)jacobi_eig_kernel<12>;
    case 14: return (const void*)jacobi_eig_kernel<14>;
    default: return (const void*)jacobi_eig_kernel<16>;
  }
}

cudaError_t jacobi_eig_launch(const double* partial, int nchunk, int batch, int l, int signed_input, float* s_out,
                              float* E, float* Es, int* status, cudaStream_t st, long long* launches, int max_sweeps, int* keff,
                              int window, float tau) {
  const int nr = (l + 7) / 8 * 2;
  const size_t smem = (size_t)(l + 1 + (signed_input ? l : 0)) * jac_stride(nr) * sizeof(double);
  typedef void (*Form)(const double*, int, int, int, float*, float*, float*, int*, int, int*, int, float);
  launch_kernel((Form)jacobi_form(nr), batch, JAC_THREADS, smem, st, partial, nchunk, l, signed_input, s_out, E, Es, status, max_sweeps > 0 ? max_sweeps : 40, keff,
                window, tau);
  if (launches) ++*launches;
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------------------------
// Frobenius partial sums of a [b, count] array (bf16 or fp32): partial[b, nblk] in fp64.
// ---------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(256) frob_partial_kernel(const void* __restrict__ X, int dtype, long long count,
                                                           int nblk, double* __restrict__ partial) {
  pdl_wait();
  __shared__ double red[8];
  const int bz = blockIdx.y, tid = threadIdx.x;
  const long long per = (count + nblk - 1) / nblk;
  const long long lo = (long long)blockIdx.x * per, hi = min(count, lo + per);
  const long long base = (long long)bz * count;
  double acc = 0.0;
  float f = 0.f;
  int n = 0;
  for (long long i = lo + tid; i < hi; i += 256) {
    const float v = ld_as_float(X, base + i, dtype);
    f = fmaf(v, v, f);
    if (++n == 16) { acc += (double)f; f = 0.f; n = 0; }
  }
  acc += (double)f;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
  if ((tid & 31) == 0) red[tid >> 5] = acc;
  __syncthreads();
  if (tid == 0) {
    double t = 0.0;
    for (int w = 0; w < 8; ++w) t += red[w];
    partial[(long long)bz * nblk + blockIdx.x] = t;
  }
}

cudaError_t frob_partial_launch(const void* X, int dtype, int batch, long long count, int nblk, double* partial,
                                cudaStream_t st, long long* launches) {
  launch_kernel(frob_partial_kernel, dim3(nblk, batch), 256, 0, st, X, dtype, count, nblk, partial);
  if (launches) ++*launches;
  return cudaGetLastError();
}

// rho[b] = sqrt(sum of partials); one warp per matrix, lane-strided sums then a shuffle tree (fixed order);
// inv_rho[b] = 1/rho (0 and status bit 4 when rho is 0 or not finite)
__global__ void rho_finalize_kernel(const double* __restrict__ partial, int nper, int batch, float* __restrict__ rho,
                                    float* __restrict__ inv_rho, float* __restrict__ inv_rho2,
                                    int* __restrict__ status) {
  pdl_wait();
  const int bz = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (bz >= batch) return;
  double t = 0.0;
  for (int i = lane; i < nper; i += 32) t += partial[(long long)bz * nper + i];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
  if (lane != 0) return;
  const double r = sqrt(t);
  const bool ok = (r > 0.0) && isfinite(r);
  if (rho) rho[bz] = (float)r;
  if (inv_rho) inv_rho[bz] = ok ? (float)(1.0 / r) : 0.f;
  if (inv_rho2) inv_rho2[bz] = ok ? (float)(1.0 / t) : 0.f;
  if (!ok && status) atomicOr(&status[bz], 4);
}

cudaError_t rho_finalize_launch(const double* partial, int nper, int batch, float* rho, float* inv_rho,
                                float* inv_rho2, int* status, cudaStream_t st, long long* launches) {
  launch_kernel(rho_finalize_kernel, (batch + 3) / 4, 128, 0, st, partial, nper, batch, rho, inv_rho, inv_rho2, status);
  if (launches) ++*launches;
  return cudaGetLastError();
}

// Frobenius partial sums with 16-byte loads: CTA (blk, batch) sums a contiguous run of whole 16-byte packets (fp32
// sums of at most 64 squares per thread, then fp64), partial[b, nblk]. The leftover elements of a matrix whose
// size is not a whole number of packets go to the last CTA. Needs a 16-byte aligned base and matrix stride.
template <typename T, int V>
__global__ void __launch_bounds__(256) frob_partial_vec_kernel(const T* __restrict__ X, long long count, int nblk,
                                                               double* __restrict__ partial) {
  pdl_wait();
  struct alignas(16) Pack { T v[V]; };
  __shared__ double red[8];
  const int bz = blockIdx.y, tid = threadIdx.x;
  const T* Xb = X + (long long)bz * count;
  const long long nvec = count / V;
  const long long per = (nvec + nblk - 1) / nblk;
  const long long lo = (long long)blockIdx.x * per, hi = min(nvec, lo + per);
  double acc = 0.0;
  const Pack* P = reinterpret_cast<const Pack*>(Xb);
  long long i = lo + tid;
  // four packets per thread in flight
  for (; i + 3 * 256 < hi; i += 4 * 256) {
    Pack q[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) q[u] = P[i + u * 256];
    float f = 0.f;
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
      for (int j = 0; j < V; ++j) { const float v = (float)q[u].v[j]; f = fmaf(v, v, f); }
    acc += (double)f;
  }
  for (; i < hi; i += 256) {
    const Pack q = P[i];
    float f = 0.f;
#pragma unroll
    for (int j = 0; j < V; ++j) { const float v = (float)q.v[j]; f = fmaf(v, v, f); }
    acc += (double)f;
  }
  if (blockIdx.x == nblk - 1) {
    for (long long e = nvec * V + tid; e < count; e += 256) { const float v = (float)Xb[e]; acc += (double)v * (double)v; }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
  if ((tid & 31) == 0) red[tid >> 5] = acc;
  __syncthreads();
  if (tid == 0) {
    double t = 0.0;
    for (int w = 0; w < 8; ++w) t += red[w];
    partial[(long long)bz * nblk + blockIdx.x] = t;
  }
}

cudaError_t frob_partial_vec_launch(const void* X, int dtype, int batch, long long count, int nblk, double* partial,
                                    cudaStream_t st, long long* launches) {
  const int es = (int)dtype_size(dtype);
  const bool aligned = (reinterpret_cast<uintptr_t>(X) & 15) == 0 && ((count * es) & 15) == 0;
  if (!aligned || dtype == F16) return frob_partial_launch(X, dtype, batch, count, nblk, partial, st, launches);
  if (dtype == BF16) launch_kernel(frob_partial_vec_kernel<__nv_bfloat16, 8>, dim3(nblk, batch), 256, 0, st, (const __nv_bfloat16*)X, count, nblk, partial);
  else launch_kernel(frob_partial_vec_kernel<float, 4>, dim3(nblk, batch), 256, 0, st, (const float*)X, count, nblk, partial);
  if (launches) ++*launches;
  return cudaGetLastError();
}

// rho[b] from the identity ||A - U_k diag(s) V_k^T||_F^2 = ||A||_F^2 - sum_{i < keff} s_i^2 (triplets of Algorithm 3):
// one warp per matrix adds the partial sums of ||A||_F^2 (fixed order), lane 0 subtracts the squares in fp64.
// A difference below 1e-6 ||A||_F^2 is below what the fp32 singular values resolve: the residual counts as zero
// (status bit 4, 1/rho = 0), as does a non-finite one.
__global__ void rho_identity_kernel(const double* __restrict__ partial, int nper, int batch, const float* __restrict__ s,
                                    int ld_s, const int* __restrict__ keff, float* __restrict__ rho,
                                    float* __restrict__ inv_rho, float* __restrict__ inv_rho2, int* __restrict__ status) {
  pdl_wait();
  const int bz = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (bz >= batch) return;
  double t = 0.0;
  for (int i = lane; i < nper; i += 32) t += partial[(long long)bz * nper + i];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
  if (lane != 0) return;
  const double total = t;
  const int ke = keff[bz];
  for (int i = 0; i < ke; ++i) { const double v = (double)s[(long long)bz * ld_s + i]; t -= v * v; }
  const bool ok = isfinite(t) && t > 1e-6 * total;
  const double r = ok ? sqrt(t) : 0.0;
  if (rho) rho[bz] = (float)r;
  if (inv_rho) inv_rho[bz] = ok ? (float)(1.0 / r) : 0.f;
  if (inv_rho2) inv_rho2[bz] = ok ? (float)(1.0 / t) : 0.f;
  if (!ok && status) atomicOr(&status[bz], 4);
}

cudaError_t rho_identity_launch(const double* partial, int nper, int batch, const float* s, int ld_s, const int* keff,
                                float* rho, float* inv_rho, float* inv_rho2, int* status, cudaStream_t st,
                                long long* launches) {
  launch_kernel(rho_identity_kernel, (batch + 3) / 4, 128, 0, st, partial, nper, batch, s, ld_s, keff, rho, inv_rho, inv_rho2, status);
  if (launches) ++*launches;
  return cudaGetLastError();
}

// Non-finite results are reported, not returned silently: one CTA per matrix looks at the first 4096 elements and at
// 4096 more spread evenly over the matrix, and raises bit 16 of status[b] when one of them is Inf or NaN. A sample is
// enough: a non-finite entry of an iterate (non-finite input, or a value that left the range of the iterate's
// storage format) reaches the Gram matrix of the next step and from there every entry of the following iterate.
__global__ void __launch_bounds__(1024) finite_probe_kernel(const void* __restrict__ X, int dtype, long long count,
                                                           int* __restrict__ status) {
  pdl_wait();
  const int bz = blockIdx.x, tid = threadIdx.x;
  const long long base = (long long)bz * count;
  const long long stride = max((long long)1, count / 4096);
  // all eight loads of a thread are on their way before the first is looked at
  float v[8];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const long long j = tid + 1024 * i;
    v[i] = (j < count) ? ld_as_float(X, base + j, dtype) : 0.f;
    v[4 + i] = (j * stride < count) ? ld_as_float(X, base + j * stride, dtype) : 0.f;
  }
  bool bad = false;
#pragma unroll
  for (int i = 0; i < 8; ++i) bad |= !isfinite(v[i]);
  if (__syncthreads_or(bad ? 1 : 0) && tid == 0) atomicOr(&status[bz], 16);
}

cudaError_t finite_probe_launch(const void* X, int dtype, int batch, long long count, int* status, cudaStream_t st,
                                long long* launches) {
  if (batch <= 0 || count <= 0) return cudaSuccess;
  launch_kernel(finite_probe_kernel, batch, 1024, 0, st, X, dtype, count, status);
  if (launches) ++*launches;
  return cudaGetLastError();
}

// Out[b, rows, k] = In[b, rows, (ld_in)] * diag(coef): coef_t = c0 * s[b,t] * (use_inv ? inv_rho[b] : 1) + c1
__global__ void scale_cols_kernel(const float* __restrict__ In, long long in_bs, int ld_in, int rows, int k,
                                  const float* __restrict__ s, int ld_s, const float* __restrict__ inv_rho, float c0,
                                  float c1, float* __restrict__ Out, long long out_bs, int ld_out,
                                  const int* __restrict__ keff) {
  pdl_wait();
  const int bz = blockIdx.y;
  const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= (long long)rows * k) return;
  const int r = (int)(e / k), t = (int)(e % k);
  float sc = c0 * s[(long long)bz * ld_s + t] * (inv_rho ? inv_rho[bz] : 1.f) + c1;
  if (keff && t >= keff[bz]) sc = 0.f;     // column not deflated for this matrix (gate)
  Out[(long long)bz * out_bs + (long long)r * ld_out + t] = In[(long long)bz * in_bs + (long long)r * ld_in + t] * sc;
}

cudaError_t scale_cols_launch(const float* In, long long in_bs, int ld_in, int batch, int rows, int k, const float* s,
                              int ld_s, const float* inv_rho, float c0, float c1, float* Out, long long out_bs,
                              int ld_out, cudaStream_t st, long long* launches, const int* keff) {
  if (k <= 0) return cudaSuccess;
  const long long tot = (long long)rows * k;
  launch_kernel(scale_cols_kernel, dim3((unsigned)((tot + 255) / 256), batch), 256, 0, st, In, in_bs, ld_in, rows, k, s, ld_s,
                                                                               inv_rho, c0, c1, Out, out_bs, ld_out, keff);
  if (launches) ++*launches;
  return cudaGetLastError();
}

// Out[b, i] = scale[b] * In[b, i]  (type conversion allowed)
__global__ void scale_kernel(const void* __restrict__ In, int in_dt, void* __restrict__ Out, int out_dt,
                             long long count, const float* __restrict__ scale, int round_tf32, float mult) {
  pdl_wait();
  const int bz = blockIdx.y;
  const float sc = (scale ? scale[bz] : 1.f) * mult;
  const long long base = (long long)bz * count;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < count; i += (long long)gridDim.x * blockDim.x)
  {
    float v = sc * ld_as_float(In, base + i, in_dt);
    if (round_tf32) v = round_to_tf32(v);
    st_from_float(Out, base + i, out_dt, v);
  }
}

cudaError_t scale_launch(const void* In, int in_dt, void* Out, int out_dt, int batch, long long count,
                         const float* scale, cudaStream_t st, long long* launches, int round_tf32, float mult) {
  const int nblk = (int)min((long long)1184, (count + 255) / 256);
  launch_kernel(scale_kernel, dim3(nblk, batch), 256, 0, st, In, in_dt, Out, out_dt, count, scale, round_tf32, mult);
  if (launches) ++*launches;
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------------------------
// Counter-based Gaussian fill (the generator documented in the public header).
// ---------------------------------------------------------------------------------------------
__device__ __forceinline__ unsigned long long mix64(unsigned long long x) {
  x += 0x9E3779B97F4A7C15ull;
  x = (x ^ (x >> 30)) * 0xBF58476D1CE4E5B9ull;
  x = (x ^ (x >> 27)) * 0x94D049BB133111EBull;
  return x ^ (x >> 31);
}

__global__ void fill_gaussian_kernel(void* __restrict__ dst, long long count, int dtype, unsigned long long seed,
                                     long long per_stream, unsigned long long seed_stride) {
  pdl_wait();
  // element e belongs to stream e / per_stream (seed + stream * seed_stride), index e % per_stream
  for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < count;
       e += (long long)gridDim.x * blockDim.x) {
    const unsigned long long stream = per_stream > 0 ? (unsigned long long)(e / per_stream) : 0ull;
    const unsigned long long idx = per_stream > 0 ? (unsigned long long)(e % per_stream) : (unsigned long long)e;
    const unsigned long long hs = mix64(seed + stream * seed_stride);
    const unsigned long long j = idx >> 1;
    const unsigned long long r1 = mix64(hs ^ (2ull * j)), r2 = mix64(hs ^ (2ull * j + 1ull));
    const double u1 = ((double)(r1 >> 11) + 1.0) * (1.0 / 9007199254740992.0);
    const double u2 = (double)(r2 >> 11) * (1.0 / 9007199254740992.0);
    const double rad = sqrt(-2.0 * log(u1));
    double sn, cs;
    sincos(6.283185307179586476925286766559 * u2, &sn, &cs);
    st_from_float(dst, e, dtype, (float)((idx & 1ull) ? rad * sn : rad * cs));
  }
}

cudaError_t fill_gaussian_launch(void* dst, long long count, int dtype, unsigned long long seed, long long per_stream,
                                 unsigned long long seed_stride, cudaStream_t st, long long* launches) {
  if (count <= 0) return cudaSuccess;
  const int nblk = (int)min((long long)2368, (count + 255) / 256);
  launch_kernel(fill_gaussian_kernel, nblk, 256, 0, st, dst, count, dtype, seed, per_stream, seed_stride);
  if (launches) ++*launches;
  return cudaGetLastError();
}

__global__ void fill_int_kernel(int* p, int n, int v) {
  pdl_wait();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) p[i] = v;
}
// a call starts: its matrices' status words and the engine's wait word are zero
__global__ void begin_call_kernel(int* status, int n, int* word) {
  pdl_wait();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) status[i] = 0;
  if (i == 0) *word = 0;
}
cudaError_t begin_call_launch(int* status, int n, int* word, cudaStream_t st, long long* launches) {
  launch_kernel(begin_call_kernel, (n + 255) / 256, 256, 0, st, status, n, word);
  if (launches) ++*launches;
  return cudaGetLastError();
}
cudaError_t fill_int_launch(int* p, int n, int v, cudaStream_t st, long long* launches) {
  if (n <= 0) return cudaSuccess;
  launch_kernel(fill_int_kernel, (n + 255) / 256, 256, 0, st, p, n, v);
  if (launches) ++*launches;
  return cudaGetLastError();
}

}  // namespace defl

namespace defl {
__global__ void or_status_kernel(int* status, int n, const int* word) {
  pdl_wait();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) status[i] |= *word;
}
cudaError_t or_status_launch(int* status, int n, const int* word, cudaStream_t st, long long* launches) {
  if (n <= 0) return cudaSuccess;
  launch_kernel(or_status_kernel, (n + 255) / 256, 256, 0, st, status, n, word);
  if (launches) ++*launches;
  return cudaGetLastError();
}
}  // namespace defl

// ---------------------------------------------------------------------------------------------
// Allocation-free batched Frobenius norm (see defl_frobenius_norms_noalloc in the public header).
// The partial sums that frob_partial_kernel normally writes into context-owned scratch go into a
// fixed file-scope device array instead, so the call needs no cudaMalloc at all.
// ---------------------------------------------------------------------------------------------
#include "../../include/defl.h"
#include <mutex>

namespace defl {
constexpr int NOALLOC_NBLK = 148;   // partial sums per matrix (one per CTA)
static __device__ __align__(256) double g_noalloc_partials[DEFL_NOALLOC_MAX_BATCH * NOALLOC_NBLK];

constexpr int NOALLOC_MAX_DEVICES = 64;
static double* g_noalloc_ptr[NOALLOC_MAX_DEVICES];   // device address of the array, per device
static std::mutex g_noalloc_mutex;
}  // namespace defl

extern "C" int defl_frobenius_norms_noalloc(const void* X, int dtype, int b, long long count, float* norms,
                                            void* cuda_stream) {
  using namespace defl;
  if (!X || !norms || b <= 0 || count <= 0 || (dtype != DEFL_BF16 && dtype != DEFL_F32)) return DEFL_ERR_ARG;
  if (b > DEFL_NOALLOC_MAX_BATCH) return DEFL_ERR_RANK;
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= NOALLOC_MAX_DEVICES) return DEFL_ERR_CUDA;
  double* scratch = nullptr;
  {
    // First call on this device: ask the runtime where this device's copy of the array lives. The
    // array's name is only a host-side handle here; a kernel must be given the looked-up address.
    std::lock_guard<std::mutex> lock(g_noalloc_mutex);
    if (!g_noalloc_ptr[dev]) {
      void* p = nullptr;
      if (cudaGetSymbolAddress(&p, g_noalloc_partials) != cudaSuccess || !p) return DEFL_ERR_CUDA;
      g_noalloc_ptr[dev] = reinterpret_cast<double*>(p);
    }
    scratch = g_noalloc_ptr[dev];
  }
  cudaStream_t st = reinterpret_cast<cudaStream_t>(cuda_stream);
  // every slot read by the second kernel is written by the first, so nothing needs clearing
  launch_kernel(frob_partial_kernel, dim3(NOALLOC_NBLK, b), 256, 0, st, X, dtype, count, NOALLOC_NBLK, scratch);
  if (cudaGetLastError() != cudaSuccess) return DEFL_ERR_CUDA;
  launch_kernel(rho_finalize_kernel, (b + 3) / 4, 128, 0, st, scratch, NOALLOC_NBLK, b, norms, nullptr, nullptr, nullptr);
  if (cudaGetLastError() != cudaSuccess) return DEFL_ERR_CUDA;
  return DEFL_OK;
}

// ---------------------------------------------------------------------------------------------
// Split-precision copies of fp32 panels for the tensor engine: x = hi + lo with hi = bf16(x),
// lo = bf16(x - hi) (about 16 significant bits together).
// ---------------------------------------------------------------------------------------------
namespace defl {

// hi, lo [b, rows, lp] from In [b, rows, l] (leading dimension ld_in); columns l..lp-1 are zero.
__global__ void split_panel_kernel(const float* __restrict__ In, long long in_bs, int ld_in, int rows, int l, int lp,
                                   __nv_bfloat16* __restrict__ hi, __nv_bfloat16* __restrict__ lo) {
  pdl_wait();
  const int bz = blockIdx.y;
  const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= (long long)rows * lp) return;
  const int r = (int)(e / lp), c = (int)(e % lp);
  const float x = (c < l) ? In[(long long)bz * in_bs + (long long)r * ld_in + c] : 0.f;
  const __nv_bfloat16 h = __float2bfloat16_rn(x);
  const long long o = (long long)bz * rows * lp + e;
  hi[o] = h;
  lo[o] = __float2bfloat16_rn(x - __bfloat162float(h));
}

cudaError_t split_panel_launch(const float* In, long long in_bs, int ld_in, int batch, int rows, int l, int lp,
                               __nv_bfloat16* hi, __nv_bfloat16* lo, cudaStream_t st, long long* launches) {
  const long long tot = (long long)rows * lp;
  launch_kernel(split_panel_kernel, dim3((unsigned)((tot + 255) / 256), batch), 256, 0, st, In, in_bs, ld_in, rows, l, lp, hi, lo);
  if (launches) ++*launches;
  return cudaGetLastError();
}

// Out [b, rows, 3*kp] (16-bit) = three column blocks of the (optionally column-scaled) panel In [b, rows, k]:
//   pattern 0: [hi | hi | lo]      pattern 1: [hi | lo | hi]
// so that  Out0 * Out1^T = hi hi^T + hi lo^T + lo hi^T  (the product of the two fp32 panels up to the lo*lo term).
// Column t is scaled by  mult * (c0 * s[b,t] * (inv_rho ? inv_rho[b] : 1) + c1 * (rho ? rho[b] : 1))  (without s: by mult alone).
// The two halves are bf16 or, with `f16`, IEEE half (the type of the product they enter); with `transposed` the
// copy is stored as [b, 3*kp, rows], the layout of an operand whose long side is contiguous.
template <bool F16, bool TRANSPOSED>
__global__ void split_concat3_kernel(const float* __restrict__ In, long long in_bs, int ld_in, int rows, int k, int kp,
                                     const float* __restrict__ s, int ld_s, const float* __restrict__ inv_rho, float c0,
                                     float c1, float mult, int pattern, uint16_t* __restrict__ Out,
                                     const int* __restrict__ keff, const float* __restrict__ rho) {
  pdl_wait();
  const int bz = blockIdx.y;
  const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= (long long)rows * kp) return;
  // consecutive threads walk the contiguous direction of the output
  const int r = TRANSPOSED ? (int)(e % rows) : (int)(e / kp), t = TRANSPOSED ? (int)(e / rows) : (int)(e % kp);
  float x = 0.f;
  if (t < k && !(keff && t >= keff[bz])) {
    x = In[(long long)bz * in_bs + (long long)r * ld_in + t] * mult;
    if (s) x *= c0 * s[(long long)bz * ld_s + t] * (inv_rho ? inv_rho[bz] : 1.f) + c1 * (rho ? rho[bz] : 1.f);
  }
  uint16_t h, lw;
  if (F16) {
    const __half hh = __float2half_rn(x);
    h = __half_as_ushort(hh);
    lw = __half_as_ushort(__float2half_rn(x - __half2float(hh)));
  } else {
    const __nv_bfloat16 hh = __float2bfloat16_rn(x);
    h = __bfloat16_as_ushort(hh);
    lw = __bfloat16_as_ushort(__float2bfloat16_rn(x - __bfloat162float(hh)));
  }
  uint16_t* ob = Out + (long long)bz * rows * (3LL * kp);
  const long long step = TRANSPOSED ? (long long)kp * rows : (long long)kp;      // distance between the three blocks
  uint16_t* o = TRANSPOSED ? ob + (long long)t * rows + r : ob + (long long)r * (3LL * kp) + t;
  o[0] = h;
  o[step] = pattern ? lw : h;
  o[2 * step] = pattern ? h : lw;
}

cudaError_t split_concat3_launch(const float* In, long long in_bs, int ld_in, int batch, int rows, int k, int kp,
                                 const float* s, int ld_s, const float* inv_rho, float c0, float c1, int pattern,
                                 __nv_bfloat16* Out, cudaStream_t st, long long* launches, const int* keff, int f16,
                                 int transposed, float mult, const float* rho) {
  const long long tot = (long long)rows * kp;
  const dim3 grid((unsigned)((tot + 255) / 256), batch);
  uint16_t* o = reinterpret_cast<uint16_t*>(Out);
  if (f16 && transposed) launch_kernel(split_concat3_kernel<true, true>, grid, 256, 0, st, In, in_bs, ld_in, rows, k, kp, s, ld_s, inv_rho, c0, c1, mult, pattern, o, keff, rho);
  else if (f16) launch_kernel(split_concat3_kernel<true, false>, grid, 256, 0, st, In, in_bs, ld_in, rows, k, kp, s, ld_s, inv_rho, c0, c1, mult, pattern, o, keff, rho);
  else if (transposed) launch_kernel(split_concat3_kernel<false, true>, grid, 256, 0, st, In, in_bs, ld_in, rows, k, kp, s, ld_s, inv_rho, c0, c1, mult, pattern, o, keff, rho);
  else launch_kernel(split_concat3_kernel<false, false>, grid, 256, 0, st, In, in_bs, ld_in, rows, k, kp, s, ld_s, inv_rho, c0, c1, mult, pattern, o, keff, rho);
  if (launches) ++*launches;
  return cudaGetLastError();
}

// Row-padded copy of 16-bit matrices: Out [b, rows, ld] from In [b, rows, n], columns n .. ld - 1 zero (ld a multiple of 8).
// Rows of n elements that are not whole 16-byte packets are out of the copy engine's reach; one pass over them puts the
// whole call on the tensor cores. Bound by memory: 16 bytes per store, the eight loads of a thread side by side.
__global__ void __launch_bounds__(256) pad_rows_kernel(const uint16_t* __restrict__ In, uint16_t* __restrict__ Out, long long rows,
                                                       int n, int ld) {
  pdl_wait();
  const int per = ld / 8;
  const long long total = rows * per, stride = (long long)gridDim.x * blockDim.x;
  for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += stride) {
    const long long r = e / per;
    const int c = (int)(e - r * per) * 8;
    uint32_t v[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) v[j] = (c + j < n) ? In[r * n + c + j] : 0;
    reinterpret_cast<uint4*>(Out)[e] = make_uint4(v[0] | (v[1] << 16), v[2] | (v[3] << 16), v[4] | (v[5] << 16), v[6] | (v[7] << 16));
  }
}

cudaError_t pad_rows_launch(const void* In, void* Out, int batch, int rows, int n, int ld, cudaStream_t st, long long* launches) {
  const long long total = (long long)batch * rows * (ld / 8);
  const int nblk = (int)min((long long)148 * 16, (total + 255) / 256);
  launch_kernel(pad_rows_kernel, nblk, 256, 0, st, (const uint16_t*)In, (uint16_t*)Out, (long long)batch * rows, n, ld);
  if (launches) ++*launches;
  return cudaGetLastError();
}

// Matrices whose residual counts as zero (status bit 4: 1/rho = 0) get the padded head alone as filter input,
// X0 = scale * P[:, :keff] W[:, :keff]^T; every other matrix is left untouched (its CTAs return at once).
__global__ void __launch_bounds__(256) zero_residual_entry_kernel(const int* __restrict__ status, const float* __restrict__ P,
                                                                  const float* __restrict__ W, const int* __restrict__ keff,
                                                                  int m, int n, int ld, int k, float scale, void* __restrict__ X0,
                                                                  int dtype) {
  pdl_wait();
  const int bz = blockIdx.y;
  if (!(status[bz] & 4)) return;
  const float* Pb = P + (long long)bz * m * k;
  const float* Wb = W + (long long)bz * n * k;
  const int ke = keff ? min(keff[bz], k) : k;
  const long long tot = (long long)m * n;
  for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < tot; e += (long long)gridDim.x * blockDim.x) {
    const int i = (int)(e / n), j = (int)(e % n);
    float t = 0.f;
    for (int q = 0; q < ke; ++q) t = fmaf(Pb[(long long)i * k + q], Wb[(long long)j * k + q], t);
    st_from_float(X0, ((long long)bz * m + i) * ld + j, dtype, scale * t);
  }
}

cudaError_t zero_residual_entry_launch(const int* status, const float* P, const float* W, const int* keff, int batch, int m,
                                       int n, int ld, int k, float scale, void* X0, int dtype, cudaStream_t st, long long* launches) {
  launch_kernel(zero_residual_entry_kernel, dim3(64, batch), 256, 0, st, status, P, W, keff, m, n, ld, k, scale, X0, dtype);
  if (launches) ++*launches;
  return cudaGetLastError();
}

__global__ void gate_kernel(const float* __restrict__ s, int ld_s, int batch, int window, int kmax, float tau,
                            int* __restrict__ keff) {
  pdl_wait();
  const int bz = blockIdx.x * blockDim.x + threadIdx.x;
  if (bz < batch) keff[bz] = gate_count(s + (long long)bz * ld_s, window, kmax, tau);
}

cudaError_t gate_launch(const float* s, int ld_s, int batch, int window, int kmax, float tau, int* keff, cudaStream_t st,
                        long long* launches) {
  launch_kernel(gate_kernel, (batch + 127) / 128, 128, 0, st, s, ld_s, batch, window, kmax, tau, keff);
  if (launches) ++*launches;
  return cudaGetLastError();
}

}  // namespace defl

// ---------------------------------------------------------------------------------------------
// Fused panel pass for CholeskyQR2 and the triplet products: for panel In[b, rows, l]
//   Out = In * Mtx[:, :kout]   (Mtx null: Out = In), written as fp32 and/or as bf16 hi + lo,
//   and/or the Gram partials of Out (fp32 products over 128-row tiles, tiles added in fp64).
// One CTA walks its share of the rows in 128-row tiles; register-blocked 4 x 8 outputs per thread.
// In-place (Out == In) is safe: a tile is read completely before it is written.
// ---------------------------------------------------------------------------------------------
namespace defl {

constexpr int FUSED_TILE = 128;
constexpr int FUSED_TS = MAX_L + 4;
constexpr size_t FUSED_SMEM = (size_t)(2 * FUSED_TILE + MAX_L) * FUSED_TS * sizeof(float);      // two tiles, the matrix

// Rows are split over CTAs in whole 128-row tiles. The split is chosen so that all CTAs of the launch are resident
// at once (two per SM with this kernel's registers): a fixed 512-row split gave 624 CTAs for 592 places on
// the 48 x 6400-row panels, i.e. a second wave for 32 CTAs, and left two thirds of the GPU idle on 1600-row panels.
// A panel of few matrices spreads over one CTA per tile, the most that fused_max_chunks (which sizes the partials) allows.
int fused_max_chunks(int rows) { return (rows + FUSED_TILE - 1) / FUSED_TILE; }
int fused_num_chunks(int rows, int batch) {
  static int sms = 0;
  if (sms <= 0) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms <= 0)
      sms = 148;
  }
  const int places = sms * 2;
  const int tiles = (rows + FUSED_TILE - 1) / FUSED_TILE;
  int t = 1;
  while (t < tiles && (long long)((tiles + t - 1) / t) * batch > places) ++t;
  return (tiles + t - 1) / t;
}

// acc = tile * ms for rows ty + 32 i and columns 4 tx .. + 3 (NC = 8: 32 + 4 tx .. + 3 too). Rows of ms beyond l and columns
// beyond the ones wanted were zeroed when it was staged, so blocks of four are safe.
template <int NC>
__device__ __forceinline__ void panel_product(float (*tile)[FUSED_TS], float (*ms)[FUSED_TS], int l, int ty, int tx, float (&acc)[4][NC]) {
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < NC; ++j) acc[i][j] = 0.f;
  for (int q = 0; q < l; q += 4) {
    float4 a4[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) a4[i] = *reinterpret_cast<const float4*>(&tile[ty + 32 * i][q]);
#pragma unroll
    for (int qq = 0; qq < 4; ++qq) {
      float b[NC];
#pragma unroll
      for (int h = 0; h < NC / 4; ++h) {
        const float4 b4 = *reinterpret_cast<const float4*>(&ms[q + qq][32 * h + tx * 4]);
        b[4 * h] = b4.x; b[4 * h + 1] = b4.y; b[4 * h + 2] = b4.z; b[4 * h + 3] = b4.w;
      }
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float av = (qq == 0) ? a4[i].x : (qq == 1) ? a4[i].y : (qq == 2) ? a4[i].z : a4[i].w;
#pragma unroll
        for (int j = 0; j < NC; ++j) acc[i][j] = fmaf(av, b[j], acc[i][j]);
      }
    }
  }
}

// (two passes over panels of one batch may share a launch: blockIdx.z)
__global__ void __launch_bounds__(256, 2) panel_fused_kernel(const PanelPass first, const PanelPass second) {
  const PanelPass p = blockIdx.z ? second : first;
  if ((int)blockIdx.x >= p.nchunk) return;
  const float* const In = p.In; const float* const Mtx = p.Mtx; float* const Out = p.Out;
  __nv_bfloat16* const hi = p.hi; __nv_bfloat16* const lo = p.lo; double* const partial = p.partial;
  const long long in_bs = p.in_bs, out_bs = p.out_bs;
  const int ld_in = p.ld_in, rows = p.rows, l = p.l, ldm = p.ldm, kout = p.kout, ld_out = p.ld_out, lp = p.lp, nchunk = p.nchunk;
  extern __shared__ __align__(16) float fsm[];
  // row stride 68 floats: rows stay 16-byte aligned, so register blocks are fetched with 128-bit loads
  float (*tile)[FUSED_TS] = reinterpret_cast<float (*)[FUSED_TS]>(fsm);                              // [128][68], the first of two
  float (*ms)[FUSED_TS] = reinterpret_cast<float (*)[FUSED_TS]>(fsm + 2 * FUSED_TILE * FUSED_TS);    // [64][68]
  const int chunk = blockIdx.x, bz = blockIdx.y, tid = threadIdx.x;
  const float* Ib = In + (long long)bz * in_bs;
  const int wout = Mtx ? kout : l;      // width of Out
  // product: thread (ty, tx) computes rows ty, ty + 32, ty + 64, ty + 96 and columns 4 tx .. 4 tx + 3, 32 + 4 tx .. + 3.
  // A warp's four ty values are then four consecutive tile rows (68 floats apart: different banks) and its eight
  // tx values read 128 contiguous bytes of the staged matrix: one shared-memory wavefront per 16-byte load. (With
  // rows 4 ty + i and columns 8 tx + j the same loads took two wavefronts each, and the product was bound by them.)
  const int ty = tid >> 3, tx = tid & 7;
  // Gram: the upper block triangle of W = In^T In (or Out^T Out) in blocks of 4 rows x 8 columns; the threads form
  // `ngrp` groups of `nblk` (one block each), group g takes the rows g, g + ngrp, ... of every tile. fp32 sums
  // per thread (at most rows-per-CTA / ngrp terms), added up over the groups in fp64 at the end, in a fixed order.
  const int nb4 = (wout + 3) >> 2, nb8 = (wout + 7) >> 3;
  int nblk = 0;
  for (int j = 0; j < nb8; ++j) nblk += min(nb4, 2 * j + 2);
  const int ngrp = min(16, 256 / nblk);
  const int grp = tid / nblk;
  const bool gram_on = partial != nullptr && grp < ngrp;
  int bi = 0, bj = 0;          // this thread's block: rows 4 bi.., columns 8 bj.. of W
  {
    int rem = tid - grp * nblk;
    while (bj < nb8 - 1 && rem >= min(nb4, 2 * bj + 2)) { rem -= min(nb4, 2 * bj + 2); ++bj; }
    bi = rem;
  }
  float g8[4][8];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 8; ++j) g8[i][j] = 0.f;
  const int tiles = (rows + FUSED_TILE - 1) / FUSED_TILE;
  const int chunk_rows = ((tiles + nchunk - 1) / nchunk) * FUSED_TILE;
  const int r_begin = chunk * chunk_rows, r_end = min(rows, r_begin + chunk_rows);
  // Rows of whole 16-byte packets are copied asynchronously, the next tile into the other half of the memory while this one is
  // worked on: with load, product and store taking turns a pass over 48 x 6400 x 48 took 94 us, three times its bytes' time.
  // 16 threads per row (one packet each, up to 64 columns), rows past the end filled with zeros.
  const bool vec = (ld_in & 3) == 0 && (l & 3) == 0 && ((reinterpret_cast<uintptr_t>(Ib) & 15) == 0);
  const int c4 = tid & 15, rr0 = tid >> 4;
  auto fetch = [&](int r0, float (*t)[FUSED_TS]) {
    if (c4 * 4 < l) {
#pragma unroll
      for (int it = 0; it < FUSED_TILE / 16; ++it) {
        const int rr = rr0 + it * 16;
        const bool ok = r0 + rr < r_end;
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;"
                     ::"r"((uint32_t)__cvta_generic_to_shared(&t[rr][c4 * 4])), "l"(Ib + (long long)(ok ? r0 + rr : 0) * ld_in + c4 * 4), "r"(ok ? 16 : 0) : "memory");
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  pdl_wait();
  if (vec) fetch(r_begin, tile);
  if (Mtx) {
    const float* Mb = Mtx + (long long)bz * l * ldm;
#pragma unroll 8
    for (int e = tid; e < MAX_L * MAX_L; e += 256) {
      const int r = e / MAX_L, cc = e % MAX_L;
      ms[r][cc] = (r < l && cc < kout) ? Mb[r * ldm + cc] : 0.f;
    }
  }
  for (int r0 = r_begin; r0 < r_end; r0 += FUSED_TILE) {
    if (vec) {
      asm volatile("cp.async.wait_group 0;" ::: "memory");
      __syncthreads();            // (the tile is there, and everybody is through with the one before)
      if (r0 + FUSED_TILE < r_end) fetch(r0 + FUSED_TILE, tile == reinterpret_cast<float (*)[FUSED_TS]>(fsm) ? tile + FUSED_TILE : tile - FUSED_TILE);
    } else {
      __syncthreads();
      const int lr = (l + 3) & ~3;      // columns l..lr-1 are zeroed: the product walks the row in blocks of four
      for (int e = tid; e < FUSED_TILE * lr; e += 256) {
        const int rr = e / lr, c = e % lr;
        tile[rr][c] = (c < l && r0 + rr < r_end) ? Ib[(long long)(r0 + rr) * ld_in + c] : 0.f;
      }
      __syncthreads();
    }
    if (Mtx && kout <= 32) {
      // (half the columns: the same walk without the second half of a thread's)
      float acc[4][4];
      panel_product<4>(tile, ms, l, ty, tx, acc);
      __syncthreads();
#pragma unroll
      for (int i = 0; i < 4; ++i) *reinterpret_cast<float4*>(&tile[ty + 32 * i][tx * 4]) = make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
      __syncthreads();
    } else if (Mtx) {
      float acc[4][8];
      panel_product<8>(tile, ms, l, ty, tx, acc);
      __syncthreads();
      // (columns wout.. of the tile receive zeros: the staged matrix has zero columns there)
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        *reinterpret_cast<float4*>(&tile[ty + 32 * i][tx * 4]) = make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
        *reinterpret_cast<float4*>(&tile[ty + 32 * i][32 + tx * 4]) = make_float4(acc[i][4], acc[i][5], acc[i][6], acc[i][7]);
      }
      __syncthreads();
    }
    if (Out) {
      float* Ob = Out + (long long)bz * out_bs;
      if ((wout & 3) == 0 && (ld_out & 3) == 0 && ((reinterpret_cast<uintptr_t>(Ob) & 15) == 0)) {
        if (c4 * 4 < wout) {
#pragma unroll
          for (int it = 0; it < FUSED_TILE / 16; ++it) {
            const int rr = rr0 + it * 16;
            if (r0 + rr < r_end)
              *reinterpret_cast<float4*>(Ob + (long long)(r0 + rr) * ld_out + c4 * 4) = *reinterpret_cast<const float4*>(&tile[rr][c4 * 4]);
          }
        }
      } else {
        for (int e = tid; e < FUSED_TILE * wout; e += 256) {
          const int rr = e / wout, c = e % wout;
          if (r0 + rr < r_end) Ob[(long long)(r0 + rr) * ld_out + c] = tile[rr][c];
        }
      }
    }
    if (hi) {
      if ((lp & 3) == 0 && lp <= 64 && ((reinterpret_cast<uintptr_t>(hi) | reinterpret_cast<uintptr_t>(lo)) & 7) == 0) {
        // four values per thread: 8-byte stores of the hi and lo halves (tile columns wout..lp-1 may hold
        // leftovers of the input, so they are masked here)
        if (c4 * 4 < lp) {
#pragma unroll
          for (int it = 0; it < FUSED_TILE / 16; ++it) {
            const int rr = rr0 + it * 16;
            if (r0 + rr >= r_end) continue;
            const float4 x4 = *reinterpret_cast<const float4*>(&tile[rr][c4 * 4]);
            float x[4] = {x4.x, x4.y, x4.z, x4.w};
            __nv_bfloat16 h[4], lw[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              if (c4 * 4 + j >= wout) x[j] = 0.f;
              h[j] = __float2bfloat16_rn(x[j]);
              lw[j] = __float2bfloat16_rn(x[j] - __bfloat162float(h[j]));
            }
            const long long o = ((long long)bz * rows + r0 + rr) * lp + c4 * 4;
            uint2 hv, lv;
            hv.x = (uint32_t)__bfloat16_as_ushort(h[0]) | ((uint32_t)__bfloat16_as_ushort(h[1]) << 16);
            hv.y = (uint32_t)__bfloat16_as_ushort(h[2]) | ((uint32_t)__bfloat16_as_ushort(h[3]) << 16);
            lv.x = (uint32_t)__bfloat16_as_ushort(lw[0]) | ((uint32_t)__bfloat16_as_ushort(lw[1]) << 16);
            lv.y = (uint32_t)__bfloat16_as_ushort(lw[2]) | ((uint32_t)__bfloat16_as_ushort(lw[3]) << 16);
            *reinterpret_cast<uint2*>(hi + o) = hv;
            *reinterpret_cast<uint2*>(lo + o) = lv;
          }
        }
      } else {
        for (int e = tid; e < FUSED_TILE * lp; e += 256) {
          const int rr = e / lp, c = e % lp;
          if (r0 + rr >= r_end) continue;
          const float x = (c < wout) ? tile[rr][c] : 0.f;
          const __nv_bfloat16 h = __float2bfloat16_rn(x);
          const long long o = ((long long)bz * rows + r0 + rr) * lp + c;
          hi[o] = h;
          lo[o] = __float2bfloat16_rn(x - __bfloat162float(h));
        }
      }
    }
    if (gram_on) {
      const int nr = min(FUSED_TILE, r_end - r0);
      for (int rr = grp; rr < nr; rr += ngrp) {
        const float4 a0 = *reinterpret_cast<const float4*>(&tile[rr][bi * 4]);
        const float4 b0 = *reinterpret_cast<const float4*>(&tile[rr][bj * 8]);
        const float4 b1 = *reinterpret_cast<const float4*>(&tile[rr][bj * 8 + 4]);
        const float a[4] = {a0.x, a0.y, a0.z, a0.w};
        const float b[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int j = 0; j < 8; ++j) g8[i][j] = fmaf(a[i], b[j], g8[i][j]);
      }
    }
    if (vec) tile = tile == reinterpret_cast<float (*)[FUSED_TS]>(fsm) ? tile + FUSED_TILE : tile - FUSED_TILE;
  }
  if (partial) {
    // Sum over the groups in fp64 (group order fixed: the result does not depend on timing). Every thread leaves its block
    // in the tile's memory, then one thread per element of W adds up the groups. (Groups taking turns on one shared
    // array, a barrier and 32 dependent updates each, took 10 of the 14 us of a gram pass over a short panel.)
    float4* part = reinterpret_cast<float4*>(fsm);       // [ngrp][nblk][8] quads: at most 256 x 128 bytes
    __syncthreads();
    if (gram_on) {
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int h = 0; h < 2; ++h)
          part[(i * 2 + h) * 256 + tid] = make_float4(g8[i][4 * h], g8[i][4 * h + 1], g8[i][4 * h + 2], g8[i][4 * h + 3]);
    }
    __syncthreads();
    const float* pf = fsm;
    double* out = partial + ((long long)bz * nchunk + chunk) * wout * wout;
    for (int e = tid; e < wout * wout; e += 256) {
      int gi = e / wout, gj = e - gi * wout;
      // blocks below the block diagonal were not computed: take the mirror image
      if ((gi >> 3) > (gj >> 3)) { const int t = gi; gi = gj; gj = t; }
      // block columns before this one hold 2, 4, 6, .. blocks
      const int blk = (gj >> 3) * ((gj >> 3) + 1) + (gi >> 2);
      const float* q = pf + ((gi & 3) * 2 + ((gj >> 2) & 1)) * 1024 + (gj & 3);
      double t = 0.0;
      for (int g = 0; g < ngrp; ++g) t += (double)q[(g * nblk + blk) * 4];
      out[e] = t;
    }
  }
}

cudaError_t panel_prepare() {
  cudaError_t e = cudaSuccess;
  for (int nr = 2; nr <= 16 && e == cudaSuccess; nr += 2) {      // (signed input, the widest core of the form)
    const int l = 4 * nr < MAX_L ? 4 * nr : MAX_L;
    e = cudaFuncSetAttribute(jacobi_form(nr), cudaFuncAttributeMaxDynamicSharedMemorySize, (int)((2 * l + 1) * jac_stride(nr) * sizeof(double)));
  }
  if (e == cudaSuccess) e = cudaFuncSetAttribute(panel_fused_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)FUSED_SMEM);
  return e;
}

PanelPass panel_pass(const float* In, long long in_bs, int ld_in, int batch, int rows, int l, const float* Mtx, int ldm, int kout,
                     float* Out, long long out_bs, int ld_out, __nv_bfloat16* hi, __nv_bfloat16* lo, int lp, double* partial) {
  PanelPass p;
  p.In = In; p.in_bs = in_bs; p.ld_in = ld_in; p.rows = rows; p.l = l; p.Mtx = Mtx; p.ldm = ldm; p.kout = kout;
  p.Out = Out; p.out_bs = out_bs; p.ld_out = ld_out; p.hi = hi; p.lo = lo; p.lp = lp; p.partial = partial;
  p.nchunk = fused_num_chunks(rows, batch);
  return p;
}

cudaError_t panel_fused_launch(const float* In, long long in_bs, int ld_in, int batch, int rows, int l, const float* Mtx,
                               int ldm, int kout, float* Out, long long out_bs, int ld_out, __nv_bfloat16* hi,
                               __nv_bfloat16* lo, int lp, double* partial, cudaStream_t st, long long* launches) {
  const PanelPass p = panel_pass(In, in_bs, ld_in, batch, rows, l, Mtx, ldm, kout, Out, out_bs, ld_out, hi, lo, lp, partial);
  launch_kernel(panel_fused_kernel, dim3(p.nchunk, batch), 256, FUSED_SMEM, st, p, p);
  if (launches) ++*launches;
  return cudaGetLastError();
}

cudaError_t panel_pair_launch(const PanelPass& a, const PanelPass& b, int batch, cudaStream_t st, long long* launches) {
  launch_kernel(panel_fused_kernel, dim3(a.nchunk > b.nchunk ? a.nchunk : b.nchunk, batch, 2), 256, FUSED_SMEM, st, a, b);
  if (launches) ++*launches;
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------------------------
// Momentum of a Muon step, element-wise in fp32: Mom <- mu Mom + Grad, stored in the momentum's type; when `look`
// is given it receives Grad + mu Mom' with Mom' the STORED (rounded) new momentum, i.e. the Nesterov look-ahead
// is a function of the optimizer state as it is kept in memory.
// ---------------------------------------------------------------------------------------------
template <typename T, int V>
__global__ void __launch_bounds__(256) momentum_vec_kernel(T* Mom, const T* __restrict__ Grad, T* look, long long nvec, float mu) {
  pdl_wait();
  // V elements (16 bytes) per thread and trip
  struct alignas(16) Pack { T v[V]; };
  const long long stride = (long long)gridDim.x * blockDim.x;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < nvec; i += stride) {
    const Pack g = reinterpret_cast<const Pack*>(Grad)[i];
    Pack m = reinterpret_cast<const Pack*>(Mom)[i];
    Pack l;
#pragma unroll
    for (int j = 0; j < V; ++j) {
      const float gf = (float)g.v[j];
      m.v[j] = (T)fmaf(mu, (float)m.v[j], gf);
      l.v[j] = (T)fmaf(mu, (float)m.v[j], gf);          // from the momentum as stored
    }
    reinterpret_cast<Pack*>(Mom)[i] = m;
    if (look) reinterpret_cast<Pack*>(look)[i] = l;
  }
}

__global__ void __launch_bounds__(256) momentum_kernel(void* Mom, const void* __restrict__ Grad, void* look, int dtype,
                                                       long long first, long long count, float mu) {
  pdl_wait();
  const long long stride = (long long)gridDim.x * blockDim.x;
  for (long long i = first + (long long)blockIdx.x * blockDim.x + threadIdx.x; i < count; i += stride) {
    const float g = ld_as_float(Grad, i, dtype);
    st_from_float(Mom, i, dtype, fmaf(mu, ld_as_float(Mom, i, dtype), g));
    if (look) st_from_float(look, i, dtype, fmaf(mu, ld_as_float(Mom, i, dtype), g));
  }
}
cudaError_t momentum_launch(void* Mom, const void* Grad, void* look, int dtype, long long count, float mu, cudaStream_t st,
                            long long* launches) {
  if (count <= 0) return cudaSuccess;
  const bool aligned = ((reinterpret_cast<uintptr_t>(Mom) | reinterpret_cast<uintptr_t>(Grad) | reinterpret_cast<uintptr_t>(look)) & 15) == 0;
  const int per = (dtype == BF16) ? 8 : 4;
  const long long nvec = aligned ? count / per : 0;
  if (nvec > 0) {
    const int nblk = (int)min((long long)148 * 16, (nvec + 255) / 256);
    if (dtype == BF16)
      launch_kernel(momentum_vec_kernel<__nv_bfloat16, 8>, nblk, 256, 0, st, (__nv_bfloat16*)Mom, (const __nv_bfloat16*)Grad, (__nv_bfloat16*)look, nvec, mu);
    else
      launch_kernel(momentum_vec_kernel<float, 4>, nblk, 256, 0, st, (float*)Mom, (const float*)Grad, (float*)look, nvec, mu);
    if (launches) ++*launches;
  }
  if (nvec * per < count) {      // the unaligned or leftover part
    launch_kernel(momentum_kernel, 1, 256, 0, st, Mom, Grad, look, dtype, nvec * per, count, mu);
    if (launches) ++*launches;
  }
  return cudaGetLastError();
}

}  // namespace defl
