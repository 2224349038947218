// FP64-class Gram matrices and rotations of vector blocks wider than 64 columns on the tensor cores (pair
// mode; the projected matrices of Rayleigh-Ritz stay with ozaki_wide.cu), as exact
// fixed-point products (oz8_dev.cuh). Complex data are handled as real matrices of twice the columns
// (the interleaved real view), so every load is a plain contiguous one.
//
//   Gram S = X^+ W: D = X_r^T W_r over the real views; a CTA takes one tile of 128 x 64 entries of D over a
//   range of rows (the K dimension), in chunks of at most 512 rows that share one exponent per column
//   (k_oz_col_exps); Re S_ij = D[2i][2j] + D[2i+1][2j+1], Im S_ij = D[2i][2j+1] - D[2i+1][2j]. A Hermitian
//   result takes only the tiles that meet its upper triangle.
//
//   Rotation X <- X G: A = 128 rows of X, B = 64 columns of the real form of G, K = the columns of X. Results
//   are staged per CTA until the tile is done, so the in-place update never reads what it has written.
//
// Bound: the integer pipe (about 40 instructions to cut a value into digits) beside the tensor cores
// (144 MMAs of 128 x 64 x 16 per 64 entries of K, about 48 clocks each: their operands' shared-memory
// reads). The two overlap: the 64-entry operand rows are used as two halves of 32 entries, and
// while the MMAs of one half run, the 512 threads cut the next 32 entries into the other; the loads of
// the half after that are already in flight. Levels are combined once per 512 entries. Before, cut,
// MMAs and combination ran one after the other for every 64 entries: 18.6 ms a Gram matrix of
// 885 k x 360 and 17.0 / 25.1 ms a triangular / full rotation.
//
// Every wait is bounded; on a timeout the CTA raises the error flag, lets its MMAs in flight land, frees
// its tensor memory and returns.
#include <algorithm>

#include "oefe_internal.h"
#include "oz8_dev.cuh"

namespace {

constexpr int WT = 512;                                            // threads per CTA
constexpr size_t WSMEM = OZ_SMEM;

// largest biased exponent of every column over chunks of `rows` rows
__global__ void k_oz_col_exps(const double* __restrict__ M, long long ld, long long n, int ncol, int rows,
                              int* __restrict__ out) {
  const long long r0 = (long long)blockIdx.x * rows, r1 = min(n, r0 + rows);
  for (int c = threadIdx.x; c < ncol; c += blockDim.x) {
    int m = 0;
    long long r = r0;
    for (; r + 15 < r1; r += 16) {
      double v[16];
#pragma unroll
      for (int u = 0; u < 16; ++u) v[u] = __ldg(M + (r + u) * ld + c);
#pragma unroll
      for (int u = 0; u < 16; ++u) m = max(m, bexp_of(v[u]));
    }
    for (; r < r1; ++r) m = max(m, bexp_of(__ldg(M + r * ld + c)));
    out[(size_t)blockIdx.x * ncol + c] = m;
  }
}

// this thread's row (32 (warp mod 4) + lane) and 16 columns of the accumulated product, stored or added
__device__ __forceinline__ void drain16(uint32_t taddr, const int* sE, const int* sF, double* row0, size_t ld, bool add) {
  const int warp = threadIdx.x >> 5, row = 32 * (warp & 3) + (threadIdx.x & 31), c0 = 16 * (warp >> 2);
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tl = taddr + ((uint32_t)(32 * (warp & 3)) << 16) + c0;
  double* o = row0 + (size_t)row * ld + c0;
#pragma unroll 1
  for (int g = 0; g < 2; ++g) {
    double x[8];
    drain8(tl + 8 * g, sE[row], sF + c0 + 8 * g, x);
#pragma unroll
    for (int j = 0; j < 8; j += 2) {
      double2* p = reinterpret_cast<double2*>(o + 8 * g + j);
      double2 v = make_double2(x[j], x[j + 1]);
      if (add) {
        const double2 old = *p;
        v.x += old.x;
        v.y += old.y;
      }
      *p = v;
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}

struct WGramArgs {
  const double *X, *W;       // real views
  long long ldx, ldw, n;
  int nvr;
  int nI, nJ;                // tiles of 128 rows and 64 columns of D
  bool upper;                // only the tiles (I, J >= 2 I) that meet the upper triangle
  int crows;                 // rows per chunk (a multiple of 64, at most 512)
  long long chunks, cpc;     // chunks, chunks per CTA
  const int *ex, *ew;        // column exponents per chunk
  double* part;              // [block][I][J][128][64]
  int* err;
};

__global__ void __launch_bounds__(WT, 1) k_gram_oz8(const WGramArgs A) {
  extern __shared__ __align__(1024) unsigned char wz_raw[];
  __shared__ int sE[128], sF[ZN];
  __shared__ uint64_t bar[2];
  __shared__ uint32_t tmem_slot;
  __shared__ volatile int s_fail;
  const int tid = threadIdx.x;
  const OzCta C = oz_begin(wz_raw, &tmem_slot, bar, &s_fail);
  Halves H{bar};
  const bool warp0 = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0) == 0;   // (uniform)
  int I = blockIdx.y / A.nJ, J = blockIdx.y % A.nJ;
  if (A.upper) {   // blockIdx.y enumerates the tiles with J >= 2 I row by row
    int y = blockIdx.y;
    I = 0;
    while (y >= A.nJ - 2 * I) {
      y -= A.nJ - 2 * I;
      ++I;
    }
    J = 2 * I + y;
  }
  const long long cb = (long long)blockIdx.x * A.cpc, ce = min(A.chunks, cb + A.cpc);
  double* out = A.part + (((size_t)blockIdx.x * A.nI + I) * A.nJ + J) * 128 * ZN;
  // A: a thread per column and 8 rows of a half (a warp's loads of one row are consecutive columns, its
  // pair order rotated per 8 columns so that stores spread over the banks); B: 4 rows
  const int ar = tid & 127, ag = tid >> 7, bn = tid & 63, bg = tid >> 6;
  const int ca = I * 128 + ar, cw = J * ZN + bn;
  const bool aok = ca < A.nvr, bok = cw < A.nvr;
  const int ash = (ar >> 3) & 3, bsh = (bn >> 3) & 1;
  double a[8], b[4];
  for (long long c = cb; c < ce && !s_fail; ++c) {
    const long long g0 = c * A.crows;
    const int nr = (int)min((long long)A.crows, A.n - g0), steps = 2 * ((nr + 63) / 64);
    if (tid < 128) sE[tid] = aok ? A.ex[c * A.nvr + ca] : 0;
    if (tid < ZN) sF[tid] = bok ? A.ew[c * A.nvr + cw] : 0;
    auto load = [&](int st) {
      const int k0 = 32 * st;
#pragma unroll
      for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          const int k = k0 + 8 * ag + 2 * ((q + ash) & 3) + u;
          a[2 * q + u] = aok && k < nr ? __ldg(A.X + (g0 + k) * A.ldx + ca) : 0.0;
        }
#pragma unroll
      for (int q = 0; q < 2; ++q)
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          const int k = k0 + 4 * bg + 2 * (q ^ bsh) + u;
          b[2 * q + u] = bok && k < nr ? __ldg(A.W + (g0 + k) * A.ldw + cw) : 0.0;
        }
    };
    load(0);
    __syncthreads();
    for (int st = 0; st < steps; ++st) {
      const int h = st & 1;
      const bool ok = H.wait(h, &s_fail);
      if (ok) {
        if (aok) {
          const int bm = sE[ar];
#pragma unroll
          for (int q = 0; q < 4; ++q)
            put_digits(C.sA, ZPA, ar, 32 * h + 8 * ag + 2 * ((q + ash) & 3), fixed54(a[2 * q], bm), fixed54(a[2 * q + 1], bm));
        }
        if (bok) {
          const int bm = sF[bn];
#pragma unroll
          for (int q = 0; q < 2; ++q)
            put_digits(C.sB, ZPB, bn, 32 * h + 4 * bg + 2 * (q ^ bsh), fixed54(b[2 * q], bm), fixed54(b[2 * q + 1], bm));
        }
        if (st + 1 < steps) load(st + 1);
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      if (__syncthreads_or(!ok)) { s_fail = 1; break; }
      if (warp0) issue_half(C.taddr, C.sA, C.sB, h, st == 0, &bar[h]);
      H.out[h] = true;
    }
    if (s_fail) break;
    bool ok = H.wait(0, &s_fail);
    ok = H.wait(1, &s_fail) && ok;
    if (__syncthreads_or(!ok)) { s_fail = 1; break; }
    drain16(C.taddr, sE, sF, out, ZN, c > cb);
    __syncthreads();
  }
  oz_end(C, H, &s_fail, A.err);
}

// S from the partial sums of all blocks; herm: entries below the diagonal are the conjugates of those
// above (i <= j lies in a computed tile: column tile 2j / 64 or j / 64 >= 2 (row tile))
template <typename S>
__global__ void k_gram_oz8_reduce(const double* part, int nbx, int nI, int nJ, int nv, bool upper, S* out) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= nv * nv) return;
  const int r = t / nv, c = t % nv;
  const bool mirror = upper && r > c;
  const int i = mirror ? c : r, j = mirror ? r : c;
  auto D = [&](int ra, int rb) {
    double s = 0.0;
    for (int b = 0; b < nbx; ++b)
      s += part[((((size_t)b * nI + ra / 128) * nJ + rb / ZN) * 128 + ra % 128) * ZN + rb % ZN];
    return s;
  };
  if constexpr (sizeof(S) == sizeof(cd)) {
    const cd v = mkc(D(2 * i, 2 * j) + D(2 * i + 1, 2 * j + 1), D(2 * i, 2 * j + 1) - D(2 * i + 1, 2 * j));
    out[t] = mirror ? cconj(v) : v;
  } else {
    out[t] = D(i, j);
  }
}

// ------------------------------------------------------------------ rotation X <- X G
// The real form of G (row k, column j of the real views): G = herm ? C^+ of a lower triangular C : C
template <typename S>
__global__ void k_rot_form(const S* C, int nv, bool herm, double* G) {
  constexpr int R = sizeof(S) / sizeof(double);
  const long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (t >= (long long)nv * nv) return;
  const int k = (int)(t / nv), j = (int)(t % nv);
  if constexpr (R == 1) {
    G[t] = herm ? (k <= j ? C[(size_t)j * nv + k] : 0.0) : C[t];
  } else {
    const cd g = herm ? (k <= j ? cconj(C[(size_t)j * nv + k]) : mkc(0, 0)) : C[t];
    double* p = G + (size_t)2 * k * 2 * nv + 2 * j;
    p[0] = g.x;
    p[1] = g.y;
    p[2 * nv] = -g.y;
    p[2 * nv + 1] = g.x;
  }
}

struct WRotArgs {
  double* X;                 // real view
  long long ldx, n;
  int nvr, nob;              // real columns, blocks of 64 of them
  bool herm;                 // G upper triangular: no entries below a block's columns
  const double* G;           // nvr x nvr
  const int* eg;             // column exponents of G per 512 rows
  double* stage;             // per CTA: [128][nob 64]
  int* err;
};

__global__ void __launch_bounds__(WT, 1) k_rot_oz8(const WRotArgs A) {
  extern __shared__ __align__(1024) unsigned char wz_raw[];
  __shared__ int sE[128], sF[ZN];
  __shared__ uint64_t bar[2];
  __shared__ uint32_t tmem_slot;
  __shared__ volatile int s_fail;
  const int tid = threadIdx.x;
  const OzCta C = oz_begin(wz_raw, &tmem_slot, bar, &s_fail);
  Halves H{bar};
  const bool warp0 = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0) == 0;   // (uniform)
  const size_t lds = (size_t)A.nob * ZN;
  double* stage = A.stage + (size_t)blockIdx.x * 128 * lds;
  // A: four threads per row of X, 8 consecutive entries of a half each (pair order rotated per row); B: a
  // thread per column of G and 4 rows
  const int ar = tid >> 2, at = tid & 3, bn = tid & 63, bg = tid >> 6;
  const int ash = ar & 3, bsh = (bn >> 3) & 1;
  double a[8], b[4];
  const long long tiles = (A.n + 127) / 128;
  for (long long tile = blockIdx.x; tile < tiles && !s_fail; tile += gridDim.x) {
    const long long r0 = tile * 128;
    const bool aok = r0 + ar < A.n;
    const double* xr = A.X + (r0 + ar) * A.ldx;
    {   // exponents of the rows
      int m = 0;
      if (aok)
        for (int k = 8 * at; k < A.nvr; k += 32) {
          double v[8];
#pragma unroll
          for (int u = 0; u < 8; ++u) v[u] = k + u < A.nvr ? xr[k + u] : 0.0;
#pragma unroll
          for (int u = 0; u < 8; ++u) m = max(m, bexp_of(v[u]));
        }
      m = max(m, __shfl_xor_sync(0xffffffffu, m, 1));
      m = max(m, __shfl_xor_sync(0xffffffffu, m, 2));
      if (at == 0) sE[ar] = m;
    }
    for (int ob = 0; ob < A.nob && !s_fail; ++ob) {
      const int col = ob * ZN + bn;
      const bool bok = col < A.nvr;
      const int kend = A.herm ? min(A.nvr, (ob + 1) * ZN) : A.nvr;
      for (int kb = 0; kb < kend && !s_fail; kb += ZMAXK) {
        const int nk = min(ZMAXK, kend - kb), steps = 2 * ((nk + 63) / 64);
        if (tid < ZN) sF[tid] = bok ? A.eg[(size_t)(kb / ZMAXK) * A.nvr + col] : 0;
        auto load = [&](int st) {
          const int k0 = 32 * st;
#pragma unroll
          for (int q = 0; q < 4; ++q)
#pragma unroll
            for (int u = 0; u < 2; ++u) {
              const int k = k0 + 8 * at + 2 * ((q + ash) & 3) + u;
              a[2 * q + u] = aok && k < nk ? xr[kb + k] : 0.0;
            }
#pragma unroll
          for (int q = 0; q < 2; ++q)
#pragma unroll
            for (int u = 0; u < 2; ++u) {
              const int k = k0 + 4 * bg + 2 * (q ^ bsh) + u;
              b[2 * q + u] = bok && k < nk ? __ldg(A.G + (size_t)(kb + k) * A.nvr + col) : 0.0;
            }
        };
        load(0);
        __syncthreads();
        for (int st = 0; st < steps; ++st) {
          const int h = st & 1;
          const bool ok = H.wait(h, &s_fail);
          if (ok) {
            if (aok) {
              const int bm = sE[ar];
#pragma unroll
              for (int q = 0; q < 4; ++q)
                put_digits(C.sA, ZPA, ar, 32 * h + 8 * at + 2 * ((q + ash) & 3), fixed54(a[2 * q], bm),
                           fixed54(a[2 * q + 1], bm));
            }
            if (bok) {
              const int bm = sF[bn];
#pragma unroll
              for (int q = 0; q < 2; ++q)
                put_digits(C.sB, ZPB, bn, 32 * h + 4 * bg + 2 * (q ^ bsh), fixed54(b[2 * q], bm), fixed54(b[2 * q + 1], bm));
            }
            if (st + 1 < steps) load(st + 1);
          }
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
          if (__syncthreads_or(!ok)) { s_fail = 1; break; }
          if (warp0) issue_half(C.taddr, C.sA, C.sB, h, st == 0, &bar[h]);
          H.out[h] = true;
        }
        if (s_fail) break;
        bool ok = H.wait(0, &s_fail);
        ok = H.wait(1, &s_fail) && ok;
        if (__syncthreads_or(!ok)) { s_fail = 1; break; }
        drain16(C.taddr, sE, sF, stage + (size_t)ob * ZN, lds, kb > 0);
        __syncthreads();
      }
    }
    if (s_fail) break;
    const int nr = (int)min(128ll, A.n - r0);
    for (int r = tid >> 5; r < nr; r += WT / 32)
      for (int c = tid & 31; c < A.nvr; c += 32) A.X[(r0 + r) * A.ldx + c] = stage[(size_t)r * lds + c];
    __syncthreads();
  }
  oz_end(C, H, &s_fail, A.err);
}

size_t a256(size_t x) { return ((x + 255) / 256) * 256; }

}  // namespace

// out = X^+ W (nv x nv) on the tensor cores; herm: the result is known to be Hermitian (only the tiles
// meeting the upper triangle run, the rest is mirrored)
template <typename S>
int gram_oz8(oefe_ctx* c, const S* X, int ldx, const S* W, int ldw, int64_t n, int nv, S* out, bool herm) {
  constexpr int R = sizeof(S) / sizeof(double);
  const int nvr = nv * R, nI = (nvr + 127) / 128, nJ = (nvr + ZN - 1) / ZN;
  int ntile = nI * nJ;
  if (herm) {
    ntile = 0;
    for (int I = 0; I < nI; ++I) ntile += std::max(0, nJ - 2 * I);
  }
  // 512 rows per chunk unless that leaves SMs without one
  int crows = ZMAXK;
  while (crows > 64 && (long long)((n + crows - 1) / crows) * ntile < c->num_sms) crows /= 2;
  WGramArgs A;
  A.chunks = std::max<long long>(1, (n + crows - 1) / crows);
  const int nbx = (int)std::max<long long>(1, std::min<long long>(A.chunks, c->num_sms / std::max(1, ntile)));
  const size_t pb = a256((size_t)nbx * nI * nJ * 128 * ZN * sizeof(double)), eb = a256((size_t)A.chunks * nvr * sizeof(int));
  OEFE_TRY(grow_ozpart(c, pb + 2 * eb));
  int* ex = (int*)((char*)c->d_ozpart + pb);
  int* ew = (int*)((char*)c->d_ozpart + pb + eb);
  A.X = (const double*)X;
  A.W = (const double*)W;
  A.ldx = (long long)ldx * R;
  A.ldw = (long long)ldw * R;
  A.n = n;
  A.nvr = nvr;
  A.nI = nI;
  A.nJ = nJ;
  A.upper = herm;
  A.crows = crows;
  A.cpc = (A.chunks + nbx - 1) / nbx;
  A.ex = ex;
  A.ew = ew;
  A.part = (double*)c->d_ozpart;
  A.err = c->d_status + 2;
  OEFE_CUDA_TRY(c, cudaFuncSetAttribute(k_gram_oz8, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)WSMEM));
  // blocks whose range of chunks is empty (when nbx does not divide them) would leave their tiles unset
  const int used = (int)((A.chunks + A.cpc - 1) / A.cpc);
  OEFE_COUNTED k_oz_col_exps<<<(unsigned)A.chunks, 256, 0, c->stream>>>(A.X, A.ldx, n, nvr, crows, ex);
  OEFE_COUNTED k_oz_col_exps<<<(unsigned)A.chunks, 256, 0, c->stream>>>(A.W, A.ldw, n, nvr, crows, ew);
  OEFE_COUNTED k_gram_oz8<<<dim3(used, ntile), WT, WSMEM, c->stream>>>(A);
  OEFE_COUNTED k_gram_oz8_reduce<S><<<(nv * nv + 255) / 256, 256, 0, c->stream>>>(A.part, used, nI, nJ, nv, herm, out);
  return oz_finish(c, "gram");
}

// X[0:n] <- X G (G = C, or C^+ of a lower triangular C when herm) on the tensor cores
template <typename S>
int rotate_oz8(oefe_ctx* c, S* X, int ldx, int64_t n, int nv, const S* C, bool herm) {
  constexpr int R = sizeof(S) / sizeof(double);
  WRotArgs A;
  A.nvr = nv * R;
  A.nob = (A.nvr + ZN - 1) / ZN;
  const long long tiles = (n + 127) / 128;
  const int grid = (int)std::max<long long>(1, std::min<long long>(tiles, c->num_sms));
  const int gch = (A.nvr + ZMAXK - 1) / ZMAXK;
  const size_t gb = a256((size_t)A.nvr * A.nvr * sizeof(double)), eb = a256((size_t)gch * A.nvr * sizeof(int));
  OEFE_TRY(grow_ozpart(c, gb + eb + (size_t)grid * 128 * A.nob * ZN * sizeof(double)));
  char* base = (char*)c->d_ozpart;
  A.X = (double*)X;
  A.ldx = (long long)ldx * R;
  A.n = n;
  A.herm = herm;
  A.G = (const double*)base;
  A.eg = (const int*)(base + gb);
  A.stage = (double*)(base + gb + eb);
  A.err = c->d_status + 2;
  OEFE_COUNTED k_rot_form<S><<<(unsigned)(((long long)nv * nv + 255) / 256), 256, 0, c->stream>>>(C, nv, herm, (double*)base);
  OEFE_COUNTED k_oz_col_exps<<<gch, 256, 0, c->stream>>>(A.G, A.nvr, A.nvr, A.nvr, ZMAXK, (int*)(base + gb));
  OEFE_CUDA_TRY(c, cudaFuncSetAttribute(k_rot_oz8, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)WSMEM));
  OEFE_COUNTED k_rot_oz8<<<grid, WT, WSMEM, c->stream>>>(A);
  return oz_finish(c, "rotate");
}

template int gram_oz8<double>(oefe_ctx*, const double*, int, const double*, int, int64_t, int, double*, bool);
template int gram_oz8<cd>(oefe_ctx*, const cd*, int, const cd*, int, int64_t, int, cd*, bool);
template int rotate_oz8<double>(oefe_ctx*, double*, int, int64_t, int, const double*, bool);
template int rotate_oz8<cd>(oefe_ctx*, cd*, int, int64_t, int, const cd*, bool);
