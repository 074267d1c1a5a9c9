// fp32-FMA product engine: C = epilogue(opA(A) opB(B)) for arbitrary strides and bf16/half/fp32 inputs.
// It is the library's own reference engine (every shape, exact fp32 products) and the engine of
// the fp32 polar path; the large bf16 products normally run on the tensor-core engine instead.
//
// 256 threads per tile in KS groups that each take a slice of every K block; their sums are added up at the end, pairwise
// and in a fixed order (repeated runs are bit-identical). What bounds the small products this engine serves is the trip to
// L2 per K block with few warps to hide it and few tiles to fill the chip, and after that shared-memory reads: so the next
// K block is fetched into registers (16 bytes per load where the strides allow) while the current one is multiplied, shared
// memory is double buffered (one barrier per block), a thread owns 8 x 8 (4 x 8, 8 x 4) outputs, which takes one 16-byte
// read per 16 products (a 4 x 4 block takes one per 8, and was bound by them), and products of few tiles take 32 x 32 tiles.
#include "common.cuh"

namespace defl {

namespace {

constexpr int NT = 256;

template <typename T>
__device__ __forceinline__ float to_f(T v);
template <>
__device__ __forceinline__ float to_f<float>(float v) { return v; }
template <>
__device__ __forceinline__ float to_f<__nv_bfloat16>(__nv_bfloat16 v) { return __bfloat162float(v); }
template <>
__device__ __forceinline__ float to_f<__half>(__half v) { return __half2float(v); }

// four consecutive values in one load (the pointer is aligned to four elements)
__device__ __forceinline__ float4 load_quad(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ float4 load_quad(const __nv_bfloat16* p) {
  const uint2 w = *reinterpret_cast<const uint2*>(p);
  const float2 a = unpack16x2(w.x, false), b = unpack16x2(w.y, false);
  return make_float4(a.x, a.y, b.x, b.y);
}
__device__ __forceinline__ float4 load_quad(const __half* p) {
  const uint2 w = *reinterpret_cast<const uint2*>(p);
  const float2 a = unpack16x2(w.x, true), b = unpack16x2(w.y, true);
  return make_float4(a.x, a.y, b.x, b.y);
}

// How an operand's block travels: 16 bytes (8 for 16-bit types) per load along K or along the rows where that direction is
// contiguous and aligned, single values otherwise.
enum Walk { QUADS_K, QUADS_R, SINGLES_K, SINGLES_R };

// One operand of one K segment, seen as [rows][K] with strides s_r, s_k, and the register image of one of its blocks
// (ROWS x BK): fetched from global memory in one go, stored to shared memory later. A thread keeps its row; successive
// loads of a block step along K by a constant, so a block costs one pointer.
//   QUADS_K    a warp covers eight rows x 16 consecutive K values (64-byte runs; the transposing stores then meet two rows
//              of a bank, not eight)
//   QUADS_R    lanes along the rows, 16-byte stores
//   SINGLES_*  16 lanes along K, or all along the rows
template <typename T, int ROWS, int BK>
struct Block {
  static constexpr int QUADS = ROWS * BK / 4 / NT;
  float q[4 * QUADS];
  const T* p;             // the thread's first value of the next block to fetch
  long long s_r, s_k;
  int left;               // K values from the thread's first K to the end
  int rows_left;          // rows from the thread's row to the end
  int r, k;               // the thread's place within a block
  Walk walk;
  // constant K step between a thread's successive loads of a block
  static constexpr int STEP_QK = NT / 32 / (ROWS / 8) * 16;
  static constexpr int STEP_QR = NT / (ROWS / 4);
  static constexpr int STEP_SR = NT / ROWS;

  __device__ __forceinline__ void start(const void* base, long long off, long long sr, long long sk, int rows,
                                        int K, int row0, int tid) {
    const T* b1 = reinterpret_cast<const T*>(base) + off;
    s_r = sr; s_k = sk;
    const uintptr_t mask = 4 * sizeof(T) - 1;
    const long long other = (sk == 1) ? sr : sk;
    const bool vec = (other & 3) == 0 && (reinterpret_cast<uintptr_t>(b1) & mask) == 0;
    walk = (sk == 1) ? (vec ? QUADS_K : SINGLES_K) : (sr == 1) ? (vec ? QUADS_R : SINGLES_R) : SINGLES_K;
    const int lane = tid & 31, warp = tid >> 5;
    if (walk == QUADS_K) { r = (warp % (ROWS / 8)) * 8 + (lane >> 2); k = (warp / (ROWS / 8)) * 16 + (lane & 3) * 4; }
    else if (walk == QUADS_R) { r = (tid % (ROWS / 4)) * 4; k = tid / (ROWS / 4); }
    else if (walk == SINGLES_K) { r = tid >> 4; k = tid & 15; }
    else { r = tid % ROWS; k = tid / ROWS; }
    rows_left = rows - (row0 + r);
    left = K - k;
    p = b1 + (long long)(row0 + r) * sr + (long long)k * sk;
  }
  __device__ __forceinline__ static float one(const T* a) { return to_f<T>(*a); }
  __device__ __forceinline__ void fetch() {
    if (walk == QUADS_K) {
#pragma unroll
      for (int i = 0; i < QUADS; ++i) {
        const int kk = i * STEP_QK;
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (rows_left > 0 && kk < left) {
          const T* a = p + kk;
          if (kk + 3 < left) v = load_quad(a);
          else { v.x = one(a); if (kk + 1 < left) v.y = one(a + 1); if (kk + 2 < left) v.z = one(a + 2); }
        }
        q[4 * i] = v.x; q[4 * i + 1] = v.y; q[4 * i + 2] = v.z; q[4 * i + 3] = v.w;
      }
    } else if (walk == QUADS_R) {
#pragma unroll
      for (int i = 0; i < QUADS; ++i) {
        const int kk = i * STEP_QR;
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (rows_left > 0 && kk < left) {
          const T* a = p + (long long)kk * s_k;
          if (rows_left > 3) v = load_quad(a);
          else { v.x = one(a); if (rows_left > 1) v.y = one(a + 1); if (rows_left > 2) v.z = one(a + 2); }
        }
        q[4 * i] = v.x; q[4 * i + 1] = v.y; q[4 * i + 2] = v.z; q[4 * i + 3] = v.w;
      }
    } else if (walk == SINGLES_R) {
#pragma unroll
      for (int i = 0; i < 4 * QUADS; ++i) {
        const int kk = i * STEP_SR;
        q[i] = (rows_left > 0 && kk < left) ? one(p + (long long)kk * s_k) : 0.f;
      }
    } else {
      // 16 threads per row: NT / 16 = 16 rows at a time, the next 16 K values after the rows are through
#pragma unroll
      for (int i = 0; i < 4 * QUADS; ++i) {
        const int dr = (16 * i) % ROWS, kk = (16 * i) / ROWS * 16;
        q[i] = (dr < rows_left && kk < left) ? one(p + (long long)dr * s_r + (long long)kk * s_k) : 0.f;
      }
    }
    p += (long long)BK * s_k;
    left -= BK;
  }
  __device__ __forceinline__ void store(float (*s)[ROWS + 4]) const {
    if (walk == QUADS_K) {
#pragma unroll
      for (int i = 0; i < QUADS; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) s[k + i * STEP_QK + j][r] = q[4 * i + j];
    } else if (walk == QUADS_R) {
#pragma unroll
      for (int i = 0; i < QUADS; ++i)
        *reinterpret_cast<float4*>(&s[k + i * STEP_QR][r]) = make_float4(q[4 * i], q[4 * i + 1], q[4 * i + 2], q[4 * i + 3]);
    } else if (walk == SINGLES_R) {
#pragma unroll
      for (int i = 0; i < 4 * QUADS; ++i) s[k + i * STEP_SR][r] = q[i];
    } else {
#pragma unroll
      for (int i = 0; i < 4 * QUADS; ++i) s[k + (16 * i) / ROWS * 16][r + (16 * i) % ROWS] = q[i];
    }
  }
};

// Four consecutive outputs (gi, gj .. gj + 3) of the product.
__device__ __forceinline__ void emit4(const GemmDesc& g, int gi, int gj, const float* acc, bool vec, float alpha, float aux_scale, long long coff, long long xoff, double& sq) {
  if (gi >= g.M || gj >= g.N) return;
  if (vec && gj + 3 < g.N) {
    float x[4] = {0.f, 0.f, 0.f, 0.f}, v[4];
    if (g.epilogue != EPI_STORE) {
      const float4 x4 = *reinterpret_cast<const float4*>(reinterpret_cast<const float*>(g.aux) + xoff + (long long)gi * g.ld_aux + gj);
      x[0] = x4.x; x[1] = x4.y; x[2] = x4.z; x[3] = x4.w;
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      if (g.epilogue == EPI_STORE) v[j] = alpha * acc[j];
      else if (g.epilogue == EPI_POLY) v[j] = g.pb * x[j] + g.pc * acc[j] + ((gi == gj + j) ? g.pa : 0.f);
      else v[j] = aux_scale * x[j] + alpha * acc[j];
      if (g.round_tf32) v[j] = round_to_tf32(v[j]);
    }
    *reinterpret_cast<float4*>(reinterpret_cast<float*>(g.C) + coff + (long long)gi * g.ldc + gj) = make_float4(v[0], v[1], v[2], v[3]);
    return;
  }
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int c = gj + j;
    if (c >= g.N) continue;
    const float a = acc[j];
    float v;
    switch (g.epilogue) {
      case EPI_STORE: v = alpha * a; break;
      case EPI_POLY:
        v = g.pb * ld_as_float(g.aux, xoff + (long long)gi * g.ld_aux + c, g.aux_dtype) + g.pc * a + ((gi == c) ? g.pa : 0.f);
        break;
      case EPI_AUX_PLUS:
        v = aux_scale * ld_as_float(g.aux, xoff + (long long)gi * g.ld_aux + c, g.aux_dtype) + alpha * a;
        break;
      default: {  // EPI_RESID_NORM
        const float r = ld_as_float(g.aux, xoff + (long long)gi * g.ld_aux + c, g.aux_dtype) - a;
        sq += (double)r * (double)r;
        continue;
      }
    }
    if (g.round_tf32) v = round_to_tf32(v);
    if (g.symmetric) {
      if (c >= gi) st_from_float(g.C, coff + (long long)gi * g.ldc + c, g.out_dtype, v);
      if (c > gi) st_from_float(g.C, coff + (long long)c * g.ldc + gi, g.out_dtype, v);
    } else {
      st_from_float(g.C, coff + (long long)gi * g.ldc + c, g.out_dtype, v);
    }
  }
}

template <typename TIn, typename TB, int BM, int BN, int BK, int TM, int TN>
__global__ void __launch_bounds__(NT, 2) gemm_simt_kernel(const GemmDesc g) {
  pdl_wait();
  constexpr int TX = BN / TN, TY = BM / TM;          // threads of one K group
  constexpr int GT = TX * TY, KS = NT / GT;
  constexpr int PARTS = KS / 2;                      // the upper half of the groups hands its sums to the lower half, and again
  constexpr int A_FLOATS = BK * (BM + 4), B_FLOATS = BK * (BN + 4);
  constexpr int RED_FLOATS = PARTS * BM * (BN + 4);
  constexpr int TILE_FLOATS = 2 * (A_FLOATS + B_FLOATS);
  constexpr int OUTS = BM * BN / 4 / NT;             // quads of outputs a thread finishes
  static_assert(OUTS >= 1 && BK % KS == 0, "tile form");
  __shared__ __align__(16) float sm[TILE_FLOATS > RED_FLOATS ? TILE_FLOATS : RED_FLOATS];
  __shared__ double red[NT / 32];
  float (*As)[BK][BM + 4] = reinterpret_cast<float (*)[BK][BM + 4]>(sm);
  float (*Bs)[BK][BN + 4] = reinterpret_cast<float (*)[BK][BN + 4]>(sm + 2 * A_FLOATS);

  const int tn = blockIdx.x, tm = blockIdx.y, bz = blockIdx.z;
  const int row0 = tm * BM, col0 = tn * BN;
  if (g.symmetric && col0 + BN <= row0) return;      // entirely below the diagonal: written as a mirror image
  const int tid = threadIdx.x;
  const int grp = tid / GT, gt = tid % GT;
  const int tx = gt % TX, ty = gt / TX;

  float alpha = g.alpha, aux_scale = g.aux_scale;
  if (g.alpha_dev) alpha *= g.alpha_dev[bz];
  if (g.aux_scale_dev) aux_scale *= g.aux_scale_dev[bz];
  const long long coff = (long long)bz * g.batch_c, xoff = (long long)bz * g.batch_aux;
  // fp32 rows that a thread can take 16 bytes at a time
  const bool vec = !g.symmetric && g.out_dtype == F32 && (g.epilogue == EPI_STORE || g.aux_dtype == F32) &&
                   g.epilogue != EPI_RESID_NORM && (g.ldc & 3) == 0 && (g.batch_c & 3) == 0 &&
                   (reinterpret_cast<uintptr_t>(g.C) & 15) == 0 &&
                   (g.epilogue == EPI_STORE || ((g.ld_aux & 3) == 0 && (g.batch_aux & 3) == 0 &&
                                                (reinterpret_cast<uintptr_t>(g.aux) & 15) == 0));

  // thread (ty, tx): rows 4 ty .. + 3 of every run of 4 TY rows, columns likewise (16-byte shared-memory reads, lanes side by side)
  float acc[TM][TN];
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j) acc[i][j] = 0.f;

  Block<TIn, BM, BK> ra;
  Block<TB, BN, BK> rb;
  for (int seg = 0; seg < g.nseg; ++seg) {
    const int K = g.K[seg];
    ra.start(g.A[seg], (long long)bz * g.batch_a[seg], g.sa_i[seg], g.sa_k[seg], g.M, K, row0, tid);
    rb.start(g.B[seg], (long long)bz * g.batch_b[seg], g.sb_j[seg], g.sb_k[seg], g.N, K, col0, tid);
    ra.fetch();
    rb.fetch();
    if (seg) __syncthreads();                        // the previous segment's last block is still being read
    ra.store(As[0]);
    rb.store(Bs[0]);
    __syncthreads();
    int buf = 0;
    for (int k0 = 0; k0 < K; k0 += BK) {
      const bool more = k0 + BK < K;
      if (more) { ra.fetch(); rb.fetch(); }
      const int depth = min(BK, K - k0);
      auto step = [&](int kk) {
        float a[TM], b[TN];
#pragma unroll
        for (int i = 0; i < TM; i += 4) {
          const float4 a4 = *reinterpret_cast<const float4*>(&As[buf][kk][ty * 4 + i * TY]);
          a[i] = a4.x; a[i + 1] = a4.y; a[i + 2] = a4.z; a[i + 3] = a4.w;
        }
#pragma unroll
        for (int j = 0; j < TN; j += 4) {
          const float4 b4 = *reinterpret_cast<const float4*>(&Bs[buf][kk][tx * 4 + j * TX]);
          b[j] = b4.x; b[j + 1] = b4.y; b[j + 2] = b4.z; b[j + 3] = b4.w;
        }
#pragma unroll
        for (int i = 0; i < TM; ++i)
#pragma unroll
          for (int j = 0; j < TN; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
      };
      if (depth == BK) {
#pragma unroll
        for (int q = 0; q < BK / KS; ++q) step(grp * (BK / KS) + q);
      } else {
        // (a short last block: the groups share what there is)
        for (int kk = grp; kk < depth; kk += KS) step(kk);
      }
      if (more) {
        ra.store(As[buf ^ 1]);
        rb.store(Bs[buf ^ 1]);
        __syncthreads();
        buf ^= 1;
      }
    }
  }

  // The groups' sums meet in shared memory, pairwise and in a fixed order (group q takes up those of q + PARTS, then of
  // q + PARTS / 2, ...), until group 0 leaves the whole product there; every thread finishes whole quads of a row.
  float (*part)[BM][BN + 4] = reinterpret_cast<float (*)[BM][BN + 4]>(sm);
  auto each = [&](int slot, auto&& f) {
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
      for (int j = 0; j < TN; j += 4)
        f(*reinterpret_cast<float4*>(&part[slot][ty * 4 + (i & 3) + (i & ~3) * TY][tx * 4 + j * TX]), i, j);
  };
  auto put = [&](float4& s, int i, int j) { s = make_float4(acc[i][j], acc[i][j + 1], acc[i][j + 2], acc[i][j + 3]); };
#pragma unroll
  for (int half = PARTS; half >= 1; half >>= 1) {
    __syncthreads();
    if (grp >= half && grp < 2 * half) each(grp - half, put);
    __syncthreads();
    if (grp < half)
      each(grp, [&](float4& s, int i, int j) { acc[i][j] += s.x; acc[i][j + 1] += s.y; acc[i][j + 2] += s.z; acc[i][j + 3] += s.w; });
  }
  if (grp == 0) each(0, put);                        // (group 0 alone has read slot 0)
  __syncthreads();
  double sq = 0.0;
#pragma unroll
  for (int i = 0; i < OUTS; ++i) {
    const int e = tid + i * NT, r = e / (BN / 4), c = (e % (BN / 4)) * 4;
    const float4 t = *reinterpret_cast<const float4*>(&part[0][r][c]);
    const float s4[4] = {t.x, t.y, t.z, t.w};
    emit4(g, row0 + r, col0 + c, s4, vec, alpha, aux_scale, coff, xoff, sq);
  }
  if (g.epilogue == EPI_RESID_NORM) {
    // fixed-order block reduction: lanes by shuffle tree, warps summed in index order
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sq += __shfl_down_sync(0xffffffffu, sq, o);
    if ((tid & 31) == 0) red[tid >> 5] = sq;
    __syncthreads();
    if (tid == 0) {
      double t = 0.0;
      for (int w = 0; w < NT / 32; ++w) t += red[w];
      g.partials[(long long)bz * g.partials_per_batch + (long long)tm * gridDim.x + tn] = t;
    }
  }
}

// Rank-k update of a matrix, C = aux_scale aux + alpha A B with A [M, K], B^T [N, K] row-major fp32 and K <= KMAX: one pass
// over `aux` and C, bound by memory. A thread owns four columns (their B values in registers) and RU rows, whose `aux`
// values it fetches before anything else; the rows' A values come from shared memory, the same for all lanes of a warp.
constexpr int RU_ROWS = 4;      // rows per thread; 32 per CTA
template <int KMAX>
__global__ void __launch_bounds__(NT) rank_update_kernel(const GemmDesc g) {
  pdl_wait();
  __shared__ __align__(16) float ua[32][KMAX];
  __shared__ __align__(16) float ub[KMAX][128 + 4];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, bz = blockIdx.z;
  const int row0 = blockIdx.y * 32 + warp * RU_ROWS, col = blockIdx.x * 128 + lane * 4, K = g.K[0];
  const float* X = reinterpret_cast<const float*>(g.aux) + (long long)bz * g.batch_aux;
  const bool on = col < g.N;
  float4 x[RU_ROWS];
#pragma unroll
  for (int i = 0; i < RU_ROWS; ++i)
    x[i] = (on && row0 + i < g.M) ? *reinterpret_cast<const float4*>(X + (long long)(row0 + i) * g.ld_aux + col) : make_float4(0.f, 0.f, 0.f, 0.f);
  const float* A = reinterpret_cast<const float*>(g.A[0]) + (long long)bz * g.batch_a[0];
  const float* B = reinterpret_cast<const float*>(g.B[0]) + (long long)bz * g.batch_b[0];
  for (int e = tid; e < 32 * KMAX; e += NT) {
    const int r = blockIdx.y * 32 + e / KMAX, k = e % KMAX;
    ua[e / KMAX][k] = (r < g.M && k < K) ? A[(long long)r * g.sa_i[0] + k] : 0.f;
  }
  for (int e = tid; e < 128 * KMAX; e += NT) {
    const int c = blockIdx.x * 128 + e / KMAX, k = e % KMAX;
    ub[k][e / KMAX] = (c < g.N && k < K) ? B[(long long)c * g.sb_j[0] + k] : 0.f;
  }
  float alpha = g.alpha, aux_scale = g.aux_scale;
  if (g.alpha_dev) alpha *= g.alpha_dev[bz];
  if (g.aux_scale_dev) aux_scale *= g.aux_scale_dev[bz];
  __syncthreads();
  if (!on) return;
  float b[4][KMAX];
#pragma unroll
  for (int k = 0; k < KMAX; ++k) {
    const float4 b4 = *reinterpret_cast<const float4*>(&ub[k][lane * 4]);
    b[0][k] = b4.x; b[1][k] = b4.y; b[2][k] = b4.z; b[3][k] = b4.w;
  }
  float* C = reinterpret_cast<float*>(g.C) + (long long)bz * g.batch_c;
#pragma unroll
  for (int i = 0; i < RU_ROWS; ++i) {
    if (row0 + i >= g.M) break;
    float t[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int k = 0; k < KMAX; k += 4) {
      const float4 a4 = *reinterpret_cast<const float4*>(&ua[warp * RU_ROWS + i][k]);
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        t[j] = fmaf(a4.x, b[j][k], t[j]); t[j] = fmaf(a4.y, b[j][k + 1], t[j]);
        t[j] = fmaf(a4.z, b[j][k + 2], t[j]); t[j] = fmaf(a4.w, b[j][k + 3], t[j]);
      }
    }
    float v[4] = {aux_scale * x[i].x + alpha * t[0], aux_scale * x[i].y + alpha * t[1], aux_scale * x[i].z + alpha * t[2], aux_scale * x[i].w + alpha * t[3]};
    if (g.round_tf32) {
#pragma unroll
      for (int j = 0; j < 4; ++j) v[j] = round_to_tf32(v[j]);
    }
    *reinterpret_cast<float4*>(C + (long long)(row0 + i) * g.ldc + col) = make_float4(v[0], v[1], v[2], v[3]);
  }
}

bool rank_update_form(const GemmDesc& g) {
  const uintptr_t a = reinterpret_cast<uintptr_t>(g.C) | reinterpret_cast<uintptr_t>(g.aux);
  return g.epilogue == EPI_AUX_PLUS && g.nseg == 1 && g.K[0] <= 16 && !g.symmetric && g.in_dtype == F32 && g.b_dtype == F32 &&
         g.out_dtype == F32 && g.aux_dtype == F32 && g.sa_k[0] == 1 && g.sb_k[0] == 1 && (a & 15) == 0 &&
         ((g.N | g.ldc | g.ld_aux | g.batch_c | g.batch_aux) & 3) == 0 && g.M <= 32 * 65535;
}

// Tile forms. Narrow outputs (panels of at most 16 columns) take 64 x 16, outputs of at most 32 columns 32 x 32; otherwise
// the smaller of two estimates per SM, fitted to B200 timings: a 64 x 64 tile takes 1 us per K block of 32 and CTA on the
// SM, a 32 x 32 tile 0.8 us per K block of 64 (4 x (512 x 384 x 384): 31 us with 32 x 32 tiles; 4 x (128 x 128 x 256): 6.2).
enum SimtForm { FORM_64x64, FORM_32x32, FORM_64x16 };
constexpr int SIMT_SMS = 148;      // (the fit is this chip's)
double simt_estimate(const GemmDesc& g, bool symmetric, int t) {
  const int depth = g.K[0] + (g.nseg == 2 ? g.K[1] : 0);
  const long long tm = (g.M + t - 1) / t, tn = (g.N + t - 1) / t;
  const double per_sm = (double)(((symmetric ? tm * (tm + 1) / 2 : tm * tn) * g.batch + SIMT_SMS - 1) / SIMT_SMS);
  return t == 32 ? 0.8 * per_sm * ((depth + 63) / 64) : per_sm * ((depth + 31) / 32);
}
SimtForm simt_form(const GemmDesc& g) {
  if (g.M > 32 * 65535) return FORM_64x64;            // (the grid's y extent)
  if (g.N <= 16) return FORM_64x16;
  if (g.N <= 32) return FORM_32x32;
  const bool sym = g.symmetric != 0;
  return simt_estimate(g, sym, 32) < simt_estimate(g, sym, 64) ? FORM_32x32 : FORM_64x64;
}

template <typename TIn, typename TB>
void launch_form(const GemmDesc& g, SimtForm f, cudaStream_t st) {
  const int bm = f == FORM_32x32 ? 32 : 64, bn = f == FORM_64x64 ? 64 : (f == FORM_32x32 ? 32 : 16);
  const dim3 grid((g.N + bn - 1) / bn, (g.M + bm - 1) / bm, g.batch);
  if (f == FORM_64x64) launch_kernel(gemm_simt_kernel<TIn, TB, 64, 64, 32, 8, 8>, grid, NT, 0, st, g);
  else if (f == FORM_32x32) launch_kernel(gemm_simt_kernel<TIn, TB, 32, 32, 64, 4, 8>, grid, NT, 0, st, g);
  else launch_kernel(gemm_simt_kernel<TIn, TB, 64, 16, 64, 8, 4>, grid, NT, 0, st, g);
}

}  // namespace

// The mirror stores (two of one value each instead of one of four) cost 5 to 30 % of a small product, so the upper tiles have
// to be clearly fewer: estimated at under 0.72 of all tiles, or at 0.76 with at most two thirds of the tiles to compute, or
// few enough for the smaller tile form. Upper tiles against full, fp32, in graphs: 148 x 64^3 + 30 %, 64 x 128^3 + 31 %,
// 128 x 104^3 + 31 % (full); 64 x 256^3 - 11 %, 64 x 512^3 - 36 %, 128 x 192 x 192 x 768 - 19 %, 24 x 128 x 128 x 512 - 39 % (upper).
bool gemm_simt_symmetric_pays(const GemmDesc& g) {
  if (g.M <= 32 || g.M > 32 * 65535) return false;
  const double f32 = simt_estimate(g, false, 32), f64 = simt_estimate(g, false, 64);
  const double s32 = simt_estimate(g, true, 32), s64 = simt_estimate(g, true, 64);
  const double ratio = fmin(s32, s64) / fmin(f32, f64);
  const long long t = s32 < s64 ? (g.M + 31) / 32 : (g.M + 63) / 64;
  return ratio < 0.72 || (ratio <= 0.76 && 3 * (t * (t + 1) / 2) <= 2 * t * t) || (s32 < s64 && !(f32 < f64));
}

int gemm_simt_partials_per_batch(const GemmDesc& g) {
  const SimtForm f = simt_form(g);
  const int bm = f == FORM_32x32 ? 32 : 64, bn = f == FORM_64x64 ? 64 : (f == FORM_32x32 ? 32 : 16);
  return ((g.M + bm - 1) / bm) * ((g.N + bn - 1) / bn);
}

cudaError_t gemm_simt_launch(const GemmDesc& g, cudaStream_t st, long long* launches) {
  if (g.batch <= 0 || g.M <= 0 || g.N <= 0) return cudaSuccess;
  if (g.b_split == 2) return cudaErrorNotSupported;      // (split panels go to the tensor engine only)
  if (rank_update_form(g)) {
    const dim3 grid((g.N + 127) / 128, (g.M + 31) / 32, g.batch);
    if (g.K[0] <= 8) launch_kernel(rank_update_kernel<8>, grid, NT, 0, st, g);
    else launch_kernel(rank_update_kernel<16>, grid, NT, 0, st, g);
    if (launches) ++*launches;
    return cudaGetLastError();
  }
  const SimtForm f = simt_form(g);
  if (g.in_dtype == F16 || g.b_dtype == F16) {
    // IEEE half operands (iterates of the bf16 path on shapes the tensor engine cannot take): both or neither
    if (g.in_dtype != F16 || g.b_dtype != F16) return cudaErrorNotSupported;
    launch_form<__half, __half>(g, f, st);
  } else if (g.in_dtype == BF16 && g.b_dtype == BF16) launch_form<__nv_bfloat16, __nv_bfloat16>(g, f, st);
  else if (g.in_dtype == BF16) launch_form<__nv_bfloat16, float>(g, f, st);
  else if (g.b_dtype == BF16) launch_form<float, __nv_bfloat16>(g, f, st);
  else launch_form<float, float>(g, f, st);
  if (launches) ++*launches;
  return cudaGetLastError();
}

}  // namespace defl
