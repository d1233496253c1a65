// Action of a molecular Hamiltonian with real tensors on a state
// (operator-action section; the molecular Hamiltonian equation).
//
// Within one spin, a^dag_p a^dag_r a_s a_q = E_pq E_rs - delta_qr E_ps, and
// the two spin orders of the mixed term are the same product of commuting
// one-spin operators, so
//   H = c + sum_pq k_pq (E^a_pq + E^b_pq)
//         + sum_pq E^a_pq [sum_rs V_pqrs E^a_rs + W_pqrs E^b_rs]
//         + sum_pq E^b_pq [sum_rs V_pqrs E^b_rs],
//   k_pq = h_pq - 1/2 sum_r h_prrq,  V = h / 2,  W_pqrs = (h_pqrs + h_rspq) / 2.
// A string of one spin is reached by ne = n (N - n) + n excitations and left
// by as many, so each bracket is needed, and has nonzero terms, for ne of the
// N^2 excitations only.  The products are taken over those lists, per string,
// on the FP32 and FP64 units: N = 12 (6,6) needs 42 of 144 on each side, an
// eighth of the multiply-adds of full N^2 x N^2 products and of the
// intermediates.  (The full products, complex64 on the tensor cores and
// complex128 in FP64, took 5.7 ms at N = 12 (6,6) in complex64 and 8.8 ms at
// N = 10 (5,5) in complex128; now 1.19 and 0.89 ms, bound by the products:
// FP64 rate, and in complex64 the shared-memory reads of the mixed part.)
//   same spin: F[l][s] = sum_k V[pq_l][rs_k] sign_k psi[src_k] + k_{pq_l} psi[s]
//              for the excitations pq_l out of string s, rs_k into it; then
//              out[t] += sum_k sign_k F[l(k)][src_k];
//   mixed:     Y[k][i][j] = sum_l W[pq_l][rs_k] sign_l psi[src_l(i)][j] for the
//              alpha excitations into i and the beta excitations out of j,
//              then the same outer sum along j.
// The alpha same-spin part runs on blocks of columns, the beta one on
// transposed blocks of rows (the rotated spin along rows, so that a warp reads
// neighbouring columns), the mixed one on the same blocks of rows; the block
// size bounds the ne-fold intermediates.
#include <algorithm>

#include "fs_common.cuh"
#include "fs_internal.h"

namespace fs {

// acc += w x, w real.
__device__ __forceinline__ void axpy(float2& acc, float w, float2 x) {
  acc = __ffma2_rn(make_float2(w, w), x, acc);
}
__device__ __forceinline__ void axpy(double2& acc, double w, double2 x) {
  acc.x = fma(w, x.x, acc.x);
  acc.y = fma(w, x.y, acc.y);
}
__device__ __forceinline__ int swap_pq(int pq, int N) {
  const int p = pq / N;
  return (pq - p * N) * N + p;
}

// V = h / 2 and W[pq][rs] = (h_pqrs + h_rspq) / 2 in the state's precision.
template <typename R>
__global__ void k_op_weights(const double* h2, R* V, R* W, int NN) {
  const int64_t n = (int64_t)NN * NN;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int pq = (int)(i / NN), rs = (int)(i - (int64_t)pq * NN);
    const double a = h2[i], b = h2[(int64_t)rs * NN + pq];
    V[i] = (R)(0.5 * a);
    W[i] = (R)(0.5 * (a + b));
  }
}

// Same-spin products of string s = blockIdx.x over columns of X (rows are
// strings): F[l][s][c] for the excitations l out of s, L of them at a time
// (the whole list where the registers allow: every pass reads the ne rows of
// X again).  Their weights, signs folded in, are in shared memory.
//   complex128: a thread owns one column and all L excitations; bound by the
//     FP64 rate (N = 10 (5,5): 0.76 of it).
//   complex64: a thread owns L / 4 excitations of four columns, so that a
//     weight is read for four products (two-lane multiply-adds), from a
//     tile of X in shared memory.  N = 12 (6,6), ne = 42: 232 us; with one
//     column per thread, read from L2 as needed, 320 us.
template <typename R>
__host__ __device__ constexpr int op_rows() {  // rows of X staged at a time
  return sizeof(R) == 4 ? 48 : 32;
}
__device__ __forceinline__ void cp_async_x(float2* dst, const float2* src) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_x(double2* dst, const double2* src) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src) : "memory");
}
template <typename R, int L>
__global__ void __launch_bounds__(128)
    k_op_same(cx_t<R>* F, int64_t fstride, const cx_t<R>* X, int64_t ldx, int64_t col0,
              int64_t ncol, const uint16_t* gpq, const uint32_t* gsrc, int ne, int N,
              const R* V, const __grid_constant__ Mat kmat) {
  using C = cx_t<R>;
  constexpr int LG = sizeof(R) == 4 ? 4 : 1;  // lane groups along l
  constexpr int TL = L / LG, TC = LG;         // excitations and columns of a thread
  constexpr int CW = 32 / LG;                 // columns of a warp per TC
  constexpr int KB = op_rows<R>();
  extern __shared__ __align__(16) unsigned char smraw[];
  C* xs = reinterpret_cast<C*>(smraw);       // [KB][128]: a tile of X
  R* wt = reinterpret_cast<R*>(xs + KB * 128);  // [ne][L]
  uint32_t* src = reinterpret_cast<uint32_t*>(wt + (size_t)ne * L);  // [ne]
  uint32_t* pq = src + ne;                                           // [ne] into s | out of s << 16
  const int64_t s = blockIdx.x;
  const int NN = N * N;
  const int lane = threadIdx.x & 31, lg = lane / CW;
  for (int k = threadIdx.x; k < ne; k += 128) {
    src[k] = gsrc[s * ne + k];
    const int q = gpq[s * ne + k];
    pq[k] = (uint32_t)q | ((uint32_t)swap_pq(q, N) << 16);
  }
  for (int l0 = 0; l0 < ne; l0 += L) {
    __syncthreads();
#pragma unroll 8
    for (int e = threadIdx.x; e < ne * L; e += 128) {
      const int k = e / L, l = l0 + (e - k * L);
      R w = 0;
      if (l < ne) {
        w = V[(int64_t)(pq[l] >> 16) * NN + (pq[k] & 0xFFFFu)];
        if (src[k] >> 31) w = -w;
      }
      wt[e] = w;
    }
    __syncthreads();
    const int lb = lg * TL;  // this thread's first excitation of the pass
    for (int64_t cb = blockIdx.y * 128ll; cb < ncol; cb += gridDim.y * 128ll) {
      C acc[TL][TC];
#pragma unroll
      for (int l = 0; l < TL; ++l)
#pragma unroll
        for (int u = 0; u < TC; ++u) acc[l][u] = mk<R>(0, 0);
      const int cw = (threadIdx.x >> 5) * 32 + lane % CW;  // first column in the tile
      for (int k0 = 0; k0 < ne; k0 += KB) {
        const int nk = min(KB, ne - k0);
        __syncthreads();
        if (cb + threadIdx.x < ncol)
          for (int k = 0; k < nk; ++k)
            cp_async_x(xs + k * 128 + threadIdx.x,
                       X + (int64_t)(src[k0 + k] & 0x7FFFFFFFu) * ldx + col0 + cb + threadIdx.x);
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncthreads();
#pragma unroll 2
        for (int k = 0; k < nk; ++k) {
          C x[TC];
#pragma unroll
          for (int u = 0; u < TC; ++u) x[u] = xs[k * 128 + cw + CW * u];
          const R* w = wt + (k0 + k) * L + lb;
#pragma unroll
          for (int l = 0; l < TL; ++l)
#pragma unroll
            for (int u = 0; u < TC; ++u) axpy(acc[l][u], w[l], x[u]);
        }
      }
#pragma unroll
      for (int u = 0; u < TC; ++u) {
        const int64_t c = cb + cw + CW * u;
        if (c >= ncol) continue;
        const C x = X[s * ldx + col0 + c];
#pragma unroll
        for (int l = 0; l < TL; ++l) {
          if (l0 + lb + l >= ne) break;
          axpy(acc[l][u], (R)kmat.v[pq[l0 + lb + l] >> 16], x);
          F[(l0 + lb + l) * fstride + s * ncol + c] = acc[l][u];
        }
      }
    }
  }
}

// Excitations per pass: the smallest of the compiled widths that covers the
// list in the fewest passes (complex128 at most 32: four registers each).
template <typename R>
static int same_width(int ne) {
  const int most = sizeof(R) == 4 ? 48 : 32;
  const int passes = (ne + most - 1) / most;
  int L = 16;
  while (L < most && passes * L < ne) L += 16;
  return L;
}
template <typename R>
static size_t same_smem(int ne) {
  return (size_t)op_rows<R>() * 128 * sizeof(cx_t<R>) +
         (size_t)ne * (same_width<R>(ne) * sizeof(R) + 8);
}
template <typename R, int L>
static void same_launch(cx_t<R>* F, int64_t fstride, const cx_t<R>* X, int64_t ldx, int64_t col0,
                        int64_t ncol, const Space* sp, int N, const R* V, const Mat& kmat,
                        cudaStream_t st) {
  const size_t smem = same_smem<R>(sp->ne);
  allow_shared_memory(k_op_same<R, L>);
  // four column tiles per CTA: the weights of a string (2000 scattered reads at
  // N = 12) cost as much as one tile's products
  const unsigned ty = (unsigned)std::max<int64_t>(1, std::min<int64_t>((ncol + 511) / 512, 65535));
  k_op_same<R, L><<<dim3((unsigned)sp->dim, ty), 128, smem, st>>>(
      F, fstride, X, ldx, col0, ncol, sp->gpq, sp->gsrc, sp->ne, N, V, kmat);
  FS_CUDA(cudaGetLastError());
}
template <typename R>
static void same_products(cx_t<R>* F, int64_t fstride, const cx_t<R>* X, int64_t ldx, int64_t col0,
                          int64_t ncol, const Space* sp, int N, const R* V, const Mat& kmat,
                          cudaStream_t st) {
  switch (same_width<R>(sp->ne)) {
    case 16: same_launch<R, 16>(F, fstride, X, ldx, col0, ncol, sp, N, V, kmat, st); break;
    case 32: same_launch<R, 32>(F, fstride, X, ldx, col0, ncol, sp, N, V, kmat, st); break;
    default:
      if constexpr (sizeof(R) == 4)
        same_launch<R, 48>(F, fstride, X, ldx, col0, ncol, sp, N, V, kmat, st);
      break;
  }
}

constexpr int kOpL = 16;  // excitations per pass of the mixed products
// Mixed products of alpha string row0 + blockIdx.x: Y[k][ii][j] for the beta
// excitations k out of j (lanes over j).  The row's weights W[pq_l][.],
// signs folded in, are in shared memory (lcap excitations l at a time, two
// side by side); a lane reads its own entry of each, which its neighbours
// mostly share.  Those reads bound the complex64 form.
template <typename R>
__global__ void __launch_bounds__(128)
    k_op_mixed(cx_t<R>* Y, int64_t ystride, const cx_t<R>* X, int64_t db, int64_t row0,
               const uint16_t* apq, const uint32_t* asrc, int nea, const uint16_t* bpq, int neb,
               int N, const R* W, int lcap) {
  using C = cx_t<R>;
  extern __shared__ __align__(16) unsigned char smraw[];
  C* wt = reinterpret_cast<C*>(smraw);  // [lcap / 2][NN], l even in x, odd in y
  const int NN = N * N;
  const int64_t i = row0 + blockIdx.x;
  const uint16_t* pq = apq + i * nea;
  const uint32_t* src = asrc + i * nea;
  for (int64_t j0 = blockIdx.y * 128ll; j0 < db; j0 += gridDim.y * 128ll) {
    const int64_t j = j0 + threadIdx.x;
    for (int k0 = 0; k0 < neb; k0 += kOpL) {
      C acc[kOpL];
      int rs[kOpL];
#pragma unroll
      for (int k = 0; k < kOpL; ++k) {
        acc[k] = mk<R>(0, 0);
        rs[k] = j < db && k0 + k < neb ? swap_pq(bpq[j * neb + k0 + k], N) : 0;
      }
      for (int l0 = 0; l0 < nea; l0 += lcap) {
        const int nl = min(lcap, nea - l0);
        if (nea > lcap || (k0 == 0 && j0 == blockIdx.y * 128ll)) {
          __syncthreads();
          const int np = (nl + 1) / 2;
          for (int e = threadIdx.x; e < np * NN; e += 128) {
            const int h = e / NN, r = e - h * NN, l = l0 + 2 * h;
            auto at = [&](int q) {
              const R w = W[(int64_t)pq[q] * NN + r];
              return (src[q] >> 31) ? -w : w;
            };
            wt[e] = mk<R>(at(l), l + 1 < nea ? at(l + 1) : R(0));
          }
          __syncthreads();
        }
        if (j < db) {
          for (int l = 0; l < nl; l += 2) {
            const C x = X[(int64_t)(src[l0 + l] & 0x7FFFFFFFu) * db + j];
            C y = mk<R>(0, 0);
            if (l + 1 < nl) y = X[(int64_t)(src[l0 + l + 1] & 0x7FFFFFFFu) * db + j];
            const C* w = wt + (l >> 1) * NN;
#pragma unroll
            for (int k = 0; k < kOpL; ++k) {
              const C v = w[rs[k]];
              axpy(acc[k], v.x, x);
              axpy(acc[k], v.y, y);
            }
          }
        }
      }
      if (j < db)
#pragma unroll
        for (int k = 0; k < kOpL; ++k)
          if (k0 + k < neb) Y[(k0 + k) * ystride + (int64_t)blockIdx.x * db + j] = acc[k];
    }
  }
}

// out[row0 + ii][t] = c psi[row0 + ii][t] + sum_k sign_k Y[slot_k][ii][src_k]
// over the beta excitations k into t.
template <typename R>
__global__ void __launch_bounds__(256)
    k_op_gather_cols(cx_t<R>* out, const cx_t<R>* X, int64_t db, int64_t row0, int64_t nrow,
                     const cx_t<R>* Y, int64_t ystride, const uint16_t* gslot,
                     const uint32_t* gsrc, int ne, double constant) {
  const int64_t total = nrow * db;
  const R cst = (R)constant;
  for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < total;
       idx += (int64_t)gridDim.x * blockDim.x) {
    const int64_t ii = idx / db, t = idx - ii * db;
    const cx_t<R> x = X[(row0 + ii) * db + t];
    cx_t<R> acc = mk<R>(cst * x.x, cst * x.y);
    const cx_t<R>* y = Y + ii * db;
#pragma unroll 4
    for (int k = 0; k < ne; ++k) {
      const uint32_t v = gsrc[t * ne + k];
      axpy(acc, (v >> 31) ? R(-1) : R(1), y[gslot[t * ne + k] * ystride + (v & 0x7FFFFFFFu)]);
    }
    out[(row0 + ii) * db + t] = acc;
  }
}

// out[t][col0 + c] += sum_k sign_k F[slot_k][src_k][c] over the excitations k
// into row t.
template <typename R>
__global__ void __launch_bounds__(256)
    k_op_gather_rows(cx_t<R>* out, int64_t ldo, int64_t col0, int64_t ncol, int64_t nrows,
                     const cx_t<R>* F, int64_t fstride, const uint16_t* gslot,
                     const uint32_t* gsrc, int ne) {
  for (int64_t t = blockIdx.x; t < nrows; t += gridDim.x)
    for (int64_t c = blockIdx.y * 256ll + threadIdx.x; c < ncol; c += gridDim.y * 256ll) {
      cx_t<R> acc = out[t * ldo + col0 + c];
#pragma unroll 4
      for (int k = 0; k < ne; ++k) {
        const uint32_t v = gsrc[t * ne + k];
        axpy(acc, (v >> 31) ? R(-1) : R(1),
             F[gslot[t * ne + k] * fstride + (int64_t)(v & 0x7FFFFFFFu) * ncol + c]);
      }
      out[t * ldo + col0 + c] = acc;
    }
}

// The same sums for a transposed block (row t, columns ii), added to
// out[row0 + ii][t] through a 32 x 32 tile.
template <typename R>
__global__ void __launch_bounds__(256)
    k_op_gather_t(cx_t<R>* out, int64_t ldo, int64_t row0, int64_t nrow, int64_t nt,
                  const cx_t<R>* F, int64_t fstride, const uint16_t* gslot, const uint32_t* gsrc,
                  int ne) {
  __shared__ cx_t<R> tile[32][33];
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const int64_t t0 = blockIdx.x * 32ll;
  for (int64_t i0 = blockIdx.y * 32ll; i0 < nrow; i0 += gridDim.y * 32ll) {
    for (int r = ty; r < 32; r += 8) {
      const int64_t t = t0 + r, ii = i0 + tx;
      cx_t<R> acc = mk<R>(0, 0);
      if (t < nt && ii < nrow) {
#pragma unroll 4
        for (int k = 0; k < ne; ++k) {
          const uint32_t v = gsrc[t * ne + k];
          axpy(acc, (v >> 31) ? R(-1) : R(1),
               F[gslot[t * ne + k] * fstride + (int64_t)(v & 0x7FFFFFFFu) * nrow + ii]);
        }
      }
      tile[r][tx] = acc;
    }
    __syncthreads();
    for (int r = ty; r < 32; r += 8) {
      const int64_t ii = i0 + r, t = t0 + tx;
      if (t < nt && ii < nrow) {
        cx_t<R>* o = out + (row0 + ii) * ldo + t;
        const cx_t<R> v = tile[tx][r];
        *o = mk<R>(o->x + v.x, o->y + v.y);
      }
    }
    __syncthreads();
  }
}

template <typename R>
static void molecular_hamiltonian_t(Ctx* ctx, Space* sa, Space* sb, const void* vec_, void* out_,
                                    const double* h1, const double* h2, double constant,
                                    int64_t ws, cudaStream_t st) {
  using C = cx_t<R>;
  constexpr int dt = sizeof(R) == 4 ? FS_C64 : FS_C128;
  const int N = sa->norb, NN = N * N;
  const C* vec = (const C*)vec_;
  C* out = (C*)out_;
  const int64_t da = sa->dim, db = sb->dim;
  build_gather_table(sa, st);
  build_gather_table(sb, st);
  const int nea = sa->ne, neb = sb->ne;
  Mat kmat{};
  for (int p = 0; p < N; ++p)
    for (int q = 0; q < N; ++q) {
      double s = h1[p * N + q];
      for (int r = 0; r < N; ++r) s -= 0.5 * h2[((size_t)(p * N + r) * N + r) * N + q];
      kmat.v[p * N + q] = s;
    }
  const size_t nw = (size_t)NN * NN;
  double* hd = (double*)scratch(ctx, "op_h2", nw * sizeof(double));
  R* V = (R*)scratch(ctx, "op_V", 2 * nw * sizeof(R));
  R* W = V + nw;
  FS_CUDA(cudaMemcpyAsync(hd, h2, nw * sizeof(double), cudaMemcpyHostToDevice, st));
  // block sizes from the workspace budget: rows take the mixed and the beta
  // products and the transposed block, columns the alpha products
  const size_t csz = sizeof(C);
  size_t budget = (size_t)ws;
  if (ws <= 0) {
    size_t fr = 0, tot = 0;
    FS_CUDA(cudaMemGetInfo(&fr, &tot));
    budget = std::min<size_t>((size_t)8 << 30, fr / 4);
  }
  const size_t per_row = (size_t)(2 * neb + 1) * csz * db;
  const size_t per_col = (size_t)std::max(nea, 1) * csz * da;
  const int64_t nr = std::max<int64_t>(1, std::min<int64_t>(da, budget / per_row));
  const int64_t nc = std::max<int64_t>(1, std::min<int64_t>(db, budget / per_col));
  C* buf = (C*)scratch(ctx, "op_F", std::max(nr * per_row, nc * per_col));
  const int sms = ctx->prop.multiProcessorCount;
  const size_t smax = (size_t)ctx->prop.sharedMemPerBlockOptin;
  const int lcap = 2 * (int)std::max<size_t>(1, std::min<size_t>((nea + 1) / 2,
                                                                 (size_t)32 * 1024 / (NN * sizeof(R))));
  const size_t mixed_smem = (size_t)lcap * NN * sizeof(R);
  FS_REQUIRE(same_smem<R>(nea) <= smax && same_smem<R>(neb) <= smax && mixed_smem <= smax, FS_ERR_UNSUPPORTED,
             "operator action: weights exceed shared memory");
  allow_shared_memory(k_op_mixed<R>);
  {
    ProfScope ps("op_weights", st);
    k_op_weights<R><<<(unsigned)std::min<size_t>((nw + 255) / 256, 8 * sms), 256, 0, st>>>(
        hd, V, W, NN);
    FS_CUDA(cudaGetLastError());
  }
  auto ytiles = [](int64_t n, int64_t w) {
    return (unsigned)std::max<int64_t>(1, std::min<int64_t>((n + w - 1) / w, 65535));
  };
  // mixed and beta parts on row blocks; also writes c psi
  for (int64_t i0 = 0; i0 < da; i0 += nr) {
    const int64_t nrow = std::min(nr, da - i0), X = nrow * db;
    C* Y = buf;
    C* G = buf + (size_t)neb * X;
    C* xt = G + (size_t)neb * X;
    if (neb > 0) {
      launch_transpose(vec + i0 * db, xt, nrow, db, dt, st);
      ProfScope ps("op_products", st, 2);
      k_op_mixed<R><<<dim3((unsigned)nrow, ytiles(db, 128)), 128, mixed_smem, st>>>(
          Y, X, vec, db, i0, sa->gpq, sa->gsrc, nea, sb->gpq, neb, N, W, lcap);
      FS_CUDA(cudaGetLastError());
      same_products<R>(G, X, xt, nrow, 0, nrow, sb, N, V, kmat, st);
    }
    ProfScope ps("op_gather", st, neb > 0 ? 2 : 1);
    k_op_gather_cols<R><<<(unsigned)std::min<int64_t>((X + 255) / 256, 32 * sms), 256, 0, st>>>(
        out, vec, db, i0, nrow, Y, X, sb->gslot, sb->gsrc, neb, constant);
    FS_CUDA(cudaGetLastError());
    if (neb > 0) {
      k_op_gather_t<R><<<dim3((unsigned)((db + 31) / 32), ytiles(nrow, 32)), 256, 0, st>>>(
          out, db, i0, nrow, db, G, X, sb->gslot, sb->gsrc, neb);
      FS_CUDA(cudaGetLastError());
    }
  }
  // alpha part on column blocks, added to the output
  for (int64_t j0 = 0; nea > 0 && j0 < db; j0 += nc) {
    const int64_t ncol = std::min(nc, db - j0), X = da * ncol;
    {
      ProfScope ps("op_products", st);
      same_products<R>(buf, X, vec, db, j0, ncol, sa, N, V, kmat, st);
    }
    {
      ProfScope ps("op_gather", st);
      k_op_gather_rows<R><<<dim3((unsigned)std::min<int64_t>(da, 32 * sms), ytiles(ncol, 256)), 256,
                            0, st>>>(out, db, j0, ncol, da, buf, X, sa->gslot, sa->gsrc, nea);
      FS_CUDA(cudaGetLastError());
    }
  }
}

void molecular_hamiltonian(Ctx* ctx, Space* sa, Space* sb, const void* vec, void* out, int dtype,
                           const double* h1, const double* h2, double constant,
                           int64_t workspace_bytes, cudaStream_t st) {
  FS_REQUIRE(sa->norb * sa->norb <= 1024 && sa->norb * sa->norb < 65536, FS_ERR_UNSUPPORTED,
             "operator action supports norb <= 32");
  if (dtype == FS_C64)
    molecular_hamiltonian_t<float>(ctx, sa, sb, vec, out, h1, h2, constant, workspace_bytes, st);
  else
    molecular_hamiltonian_t<double>(ctx, sa, sb, vec, out, h1, h2, constant, workspace_bytes, st);
}

}  // namespace fs
