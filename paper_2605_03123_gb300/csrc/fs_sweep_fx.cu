// Complex128 orbital-rotation sweeps on the tensor cores, in exact
// fixed-point digits (fs_fx.cuh).
//
// The work is that of the window sweeps (fs_sweep.cu): a slab of KV vectors
// of the rotated spin is staged in shared memory, the program's window steps
// of W = 6 adjacent orbitals are applied to it in order, and it is written
// back once with the configuration phases.  A step acts on the C(6, m)
// strings of an orbit as the compound matrix C_m(V) of its 6 x 6 unitary V
// (§2.3), so per class m it is a product X' = X C_m(V)^T over all orbits of
// all vectors of the slab; the diagonal layer of the decomposition is
// multiplied into the last step that covers each orbital, which makes class
// m = 6 (one string, factor det V) part of such steps.
//
// Each vector is held as 64-bit integers scaled by its own 2-norm, which the
// rotations keep, from the first step to the last.  A tile is 128 rows
// (orbit, vector): the sixteen warps gather the rows' amplitudes (the four
// warps of one TMEM lane quarter share a row's strings), cut them into seven
// digits and store those to TMEM as the A operand; 28 digit products against
// the step's images in shared memory accumulate in seven TMEM accumulators;
// the warps read those back, join them and scatter the new amplitudes.
//
// Integers keep an amplitude to some 2^-60 of its vector's norm, FP64
// rotations to 2^-53 of the amplitudes that it is mixed with.  With all
// amplitudes x_j in one range those are at least min |x_j| (the rows of a
// rotation have 2-norm 1), and the digits keep more; a vector with a wide range
// (a determinant and its weakly coupled excitations, a block of a
// block-diagonal rotation that hardly counts) would lose its small ones, and
// integers cannot carry infinities and NaNs.  The CTA sees both when it loads a
// vector (see Range) and rotates such vectors in FP64 instead, one rotation
// after another on the pairs of strings, behind the others.  All vectors of a
// state so, both spins, against the FP64 sweeps: N = 11 (6,5) 0.20 against 0.25
// ms, N = 13 (5,7) 1.33 against 1.55, N = 14 (7,7) 7.9 against 6.5 (two vectors a
// CTA leave the FP64 units waiting at the barrier of each rotation).
//
// Measured (one GB300, one spin, complex128): N = 14 (7,7) 1.52 ms against
// 6.74 ms of the FP64 sweep, which runs at 0.8 of the FP64 rate (2 FMA per
// clock and SM); N = 12 (6,6) 0.105 against 0.80 ms; N = 8 (4,4) 32 + 18
// (images) against 45 us.  Bound by the integer and FP32 instructions of the
// digit cutting and joining (about half of the issue slots used, two thirds
// of the tile rows filled at N = 14) and, behind them, by the products (2250
// of some 5000 clocks of a class 3 tile).
#include <algorithm>
#include <array>
#include <cmath>
#include <type_traits>
#include <vector>

#include "fs_fx.cuh"
#include "fs_common.cuh"
#include "fs_internal.h"

namespace fs {
namespace fx {

constexpr int kThreads = 512;            // the sixteen warps that move data
constexpr int kWarps = kThreads / 32;
constexpr int kCta = kThreads + 32;      // and the one that issues the products
constexpr int kMaxVec = 32;  // vectors per slab
constexpr size_t kStaticBytes = 10 * 1024;  // bound on the kernel's static shared memory
// bytes of one digit's image of class m, and of the classes' seven digits in
// the order 3, 2, 4, 1, 5, then det V as two fixed-point words
__host__ __device__ constexpr int cls(int i) {
  return i == 0 ? 3 : i == 1 ? 2 : i == 2 ? 4 : i == 3 ? 1 : 5;
}
__host__ __device__ constexpr int img_offset(int m) {
  int o = 0;
  for (int i = 0; i < 5; ++i) {
    if (cls(i) == m) return o;
    o += kDig * tc::piece_bytes(cls(i));
  }
  return o;
}
constexpr int kImgBytes = img_offset(6);           // staged in shared memory
constexpr int kImgFirst = img_offset(2);           // class 3: the first copy
constexpr int kStepBytes = kImgBytes + 128;        // with det V
static_assert(kImgBytes % 128 == 0, "images must stay 128-byte aligned");
// TMEM: the A digits at columns 0 .., the accumulators behind them
constexpr int kColD = kDig * 24;
static_assert(kColD + kSum * 48 <= 512, "class 3 tile must fit the TMEM");
// kind::f16, D f32, A and B f16, K-major both, n columns
__host__ __device__ constexpr uint32_t idesc(int n) {
  return (1u << 4) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(tc::kRows >> 4) << 24);
}

// --------------------------------------------------------- step images
struct StepMats {
  long long v[kMaxSteps][72];  // V of each step, row-major 6 x 6 complex, fixed point
};

// Per step, the compound matrices C_m(V)[S', S] = det V[S', S] by Laplace
// expansion along the first row of S', in fixed point (integer multiplies:
// the FP64 units are the slower ones, and the entries keep 62 bits), then
// the digits of their real forms [[Re, -Im], [Im, Re]] (rows = output reals,
// columns = input reals, re/im interleaved, zero padding), K-major core
// matrices (tc::b_offset).  Two blocks per step: class 3, and the others.
__global__ void __launch_bounds__(512) k_fx_images(const __grid_constant__ StepMats sm,
                                                   unsigned char* out) {
  __shared__ longlong2 M[7][400];  // [m]: ns x ns
  __shared__ uint8_t list[7][20], index[64];
  const int tid = threadIdx.x, part = blockIdx.y;
  unsigned char* img = out + (size_t)blockIdx.x * kStepBytes;
  if (tid < 64) {
    const int m = __popc(tid);
    int k = 0;
    for (int x = 0; x < tid; ++x) k += __popc(x) == m;
    list[m][k] = (uint8_t)tid;
    index[tid] = (uint8_t)k;
  }
  if (tid < 36)
    M[1][tid] = make_longlong2(sm.v[blockIdx.x][2 * tid], sm.v[blockIdx.x][2 * tid + 1]);
  __syncthreads();
  for (int m = 2; m <= (part == 0 ? 3 : 6); ++m) {
    const int ns = tc::binom6(m), n1 = tc::binom6(m - 1);
    for (int e = tid; e < ns * ns; e += blockDim.x) {
      const int R = list[m][e / ns], S = list[m][e % ns];
      const int r0 = __ffs(R) - 1, R1 = index[R & (R - 1)];
      longlong2 a = make_longlong2(0, 0);
      bool neg = false;
      for (int c = S; c; c &= c - 1, neg = !neg) {
        const int j = __ffs(c) - 1;
        const longlong2 z = cmul_fx(M[1][r0 * 6 + j], M[m - 1][R1 * n1 + index[S ^ (1 << j)]]);
        a.x += neg ? -z.x : z.x;
        a.y += neg ? -z.y : z.y;
      }
      M[m][e] = a;
    }
    __syncthreads();
  }
  for (int ci = part; ci < (part == 0 ? 1 : 5); ++ci) {
    const int m = cls(ci), ns = tc::binom6(m), kpad = tc::kp(m), nh = tc::np(m) / 2;
    unsigned char* o = img + img_offset(m);
    for (int e = tid; e < nh * nh; e += blockDim.x) {
      const int r = e / nh, c = e - r * nh;
      longlong2 z = make_longlong2(0, 0);
      if (r < ns && c < ns) z = M[m][r * ns + c];
      uint32_t w0[kDig], w1[kDig];
      digits2(z.x, -z.y, w0);  // row 2r:     columns 2c, 2c + 1
      digits2(z.y, z.x, w1);   // row 2r + 1
      const int o0 = tc::b_offset(2 * r, 2 * c, kpad), o1 = tc::b_offset(2 * r + 1, 2 * c, kpad);
      for (int j = 0; j < kDig; ++j) {
        *reinterpret_cast<uint32_t*>(o + j * tc::piece_bytes(m) + o0) = w0[j];
        *reinterpret_cast<uint32_t*>(o + j * tc::piece_bytes(m) + o1) = w1[j];
      }
    }
  }
  if (part == 1 && tid == 0) *reinterpret_cast<longlong2*>(img + kImgBytes) = M[6][0];
}

// ------------------------------------------------------------ the sweep
__device__ __forceinline__ void timeout(int* status) {
  if (status) atomicCAS(status, 0, (int)FS_ERR_TIMEOUT);
}

// The strings of class m that column group g of a tile handles (20: 4g ..
// 4g + 3 and 16 + g; 15: 4g .. 4g + 3; 6: 2g, 2g + 1) and the entries of its
// row of gather addresses (padded to a power of two).
__host__ __device__ constexpr int grp_pad(int m) { return m == 3 ? 8 : (m == 2 || m == 4) ? 4 : 2; }
__host__ __device__ constexpr int grp_string(int m, int g, int j) {
  if (m == 3) return j < 4 ? 4 * g + j : j == 4 ? 16 + g : -1;
  const int k = (m == 2 || m == 4) ? 4 * g + j : 2 * g + j;
  return k < tc::binom6(m) ? k : -1;
}

// Per-thread state of the tile pipeline.
struct Thread {
  uint32_t lane0;  // TMEM base with this warp's lane offset
  int wg, row;     // column group; row within a tile
};
// The strings of one tile row that a thread owns (offset in the slab, -1:
// none), their digits, and the raw accumulators of their products.
struct Item {
  uint32_t p[3];  // 16-bit slab cells (a slab has fewer than 2^14), 0xFFFF: none
  __device__ __forceinline__ uint32_t off(int j) const { return (p[j >> 1] >> (16 * (j & 1))) & 0xFFFFu; }
};

// Gather and digits of one tile row of class shape M (3, 2 for 2 and 4, 1
// for 1 and 5): rows = count x vectors, row = vector * count + orbit.  Rows
// past the end and strings past the class's last carry zeros.
template <int M>
__device__ __forceinline__ void gather(const Thread& t, const longlong2* slab, int d,
                                       const uint16_t* ix, int count, int rows, int row0,
                                       Item& it, uint32_t (&w)[5][kDig]) {
  constexpr int P = grp_pad(M), G = M == 3 ? 5 : P;
  const int row = row0 + t.row;
  uint32_t q[3] = {0xFFFFFFFFu, 0xFFFFFFFFu, 0xFFFFFFFFu};
  if (row < rows) {
    const int kv = (int)(((float)row + 0.5f) * (1.f / (float)count)), o = row - kv * count;
    const uint16_t* src = ix + (t.wg * count + o) * P;
    if constexpr (P == 8) {
      const uint4 u = *reinterpret_cast<const uint4*>(src);
      q[0] = u.x;
      q[1] = u.y;
      q[2] = u.z;
    } else if constexpr (P == 4) {
      const uint2 u = *reinterpret_cast<const uint2*>(src);
      q[0] = u.x;
      q[1] = u.y;
    } else {
      q[0] = *reinterpret_cast<const uint32_t*>(src);
    }
    // the vector's first cell added to both halves (no carry between them:
    // cells stay below 2^14), except where there is no string
    const uint32_t b = (uint32_t)(kv * d), bb = b | (b << 16);
    if (P == 4 && t.wg == 3) {
      q[0] += bb;
      q[1] = ((q[1] + b) & 0xFFFFu) | 0xFFFF0000u;
    } else {
#pragma unroll
      for (int k = 0; k < (G + 1) / 2; ++k) q[k] += bb;
    }
  }
#pragma unroll
  for (int k = 0; k < 3; ++k) it.p[k] = q[k];
#pragma unroll
  for (int j = 0; j < G; ++j) {
    longlong2 x = make_longlong2(0, 0);
    if (it.off(j) != 0xFFFFu) x = slab[it.off(j)];
    digits2(x.x, x.y, w[j]);
  }
}
template <int M>
__device__ __forceinline__ void put_digits(const Thread& t, const uint32_t (&w)[5][kDig]) {
  constexpr int AC = tc::a_cols(M);
#pragma unroll
  for (int i = 0; i < kDig; ++i) {
    if constexpr (M == 1) {
      if (t.wg < 3) tc::tmem_st2(t.lane0 + i * AC + 2 * t.wg, w[0][i], w[1][i]);
    } else {
      const uint32_t q[4] = {w[0][i], w[1][i], w[2][i], w[3][i]};
      tc::tmem_st4(t.lane0 + i * AC + 4 * t.wg, q);
      if constexpr (M == 3) tc::tmem_st1(t.lane0 + i * AC + 16 + t.wg, w[4][i]);
    }
  }
}
// Digit i of A meets digits 1 .. 8 - i of B, which lie one after another as
// further rows, as their accumulators do: one product of up to 256 columns.
// (A product of 16 .. 48 columns takes 51 clocks: one per digit pair made a
// class 3 tile wait 4300 clocks for its products, this form 2250, near the
// 4096 multiply-adds per clock and SM.)
template <int M>
__device__ __forceinline__ void issue(uint32_t tbase, uint32_t b0, uint32_t bar) {
  constexpr int KP = tc::kp(M), AC = tc::a_cols(M), NP = tc::np(M), MAXJ = 256 / NP;
#pragma unroll
  for (int ks = 0; ks < KP / 16; ++ks)
#pragma unroll
    for (int i = 1; i <= kDig; ++i)
#pragma unroll
      for (int j = 1; j <= 8 - i; j += MAXJ) {
        const int nj = 8 - i - j + 1 < MAXJ ? 8 - i - j + 1 : MAXJ;
        const uint64_t bd =
            tc::sdesc(b0 + (j - 1) * tc::piece_bytes(M) + ks * 256, 128, (KP / 8) * 128);
        tc::mma_bf16(tbase + kColD + (i + j - 2) * NP, tbase + (i - 1) * AC + 8 * ks, bd,
                     idesc(nj * NP), ks == 0 && i == 1 ? 0u : 1u);
      }
  tc::mma_commit(bar);
}
// The raw accumulators of a thread's strings h and h + 1 (of the first four).
template <int M>
__device__ __forceinline__ void take(const Thread& t, int h, uint32_t (&f)[kSum][4]) {
  constexpr int NP = tc::np(M);
  const uint32_t dl = t.lane0 + kColD + (M == 1 ? 4 : 8) * t.wg + 2 * h;
#pragma unroll
  for (int s = 0; s < kSum; ++s) tc::tmem_ld4(dl + s * NP, f[s]);
  tc::wait_ld();
}
// The fifth string of a class 3 row, from its accumulators to the slab.
__device__ __forceinline__ void finish_fifth(const Thread& t, longlong2* slab, const Item& it) {
  const uint32_t dl = t.lane0 + kColD + 32 + 2 * t.wg;
  uint32_t h[kSum][2];
#pragma unroll
  for (int s = 0; s < kSum; ++s) tc::tmem_ld2(dl + s * tc::np(3), h[s]);
  tc::wait_ld();
  float re[kSum], im[kSum];
#pragma unroll
  for (int s = 0; s < kSum; ++s) {
    re[s] = __uint_as_float(h[s][0]);
    im[s] = __uint_as_float(h[s][1]);
  }
  if (it.off(4) != 0xFFFFu) slab[it.off(4)] = make_longlong2(join(re), join(im));
}
__device__ __forceinline__ void scatter(longlong2* slab, const Item& it, int h,
                                        const uint32_t (&f)[kSum][4]) {
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    float re[kSum], im[kSum];
#pragma unroll
    for (int s = 0; s < kSum; ++s) {
      re[s] = __uint_as_float(f[s][2 * j]);
      im[s] = __uint_as_float(f[s][2 * j + 1]);
    }
    const uint32_t o = it.off(h + j);
    if (o != 0xFFFFu) slab[o] = make_longlong2(join(re), join(im));
  }
}

// What decides how a vector is rotated: its range, wide when a nonzero
// amplitude lies below 2^-kTinyBits of its 2-norm (by the exponent of its larger
// part), or a sixteenth of them below 2^-kSmallBits or 2^-kApartBits.
//   A program that leaves blocks of orbitals apart keeps each block of a vector
// to its own accuracy in FP64, so that a vector whose range is wide when it is
// loaded goes to FP64 (kApartBits: below 2^-9 of the norm the digits' 62 bits are
// fewer than FP64's 53, at 2^-12 three fewer; a random vector of 3432 strings
// has 2^-6 on average and one amplitude in 2^10 there).
//   A program that joins all orbitals brings the rounding of the large
// amplitudes into the small ones in FP64 too.  There a wide range has to come
// out of the rotation as well, and the line (kSmallBits) lies below what the
// ansatz states near a determinant hold (12 orbitals, generators of 0.1: the last
// sixteenth of a vector at 2^-15 to 2^-20), whose sweeps would take 5 to 8 times
// as long.
//   A vector that starts with zeros is decided by its result under both, since
// what comes into them may be small (a determinant under a weak rotation); under
// a program with a rotation weaker than 2^-kWeakBits, where amplitudes could
// vanish altogether in between, it goes to FP64.
constexpr int kTinyBits = 30, kSmallBits = 22, kApartBits = 12, kWeakBits = 12;
// Orbitals are joined when the product of the rotations' moduli connects each
// to each by at least 2^-kJoinBits (random unitaries 2^-5 to 2^-8, generators
// with entries of 0.1 2^-6 to 2^-11, of 0.001 2^-12 to 2^-17).
constexpr int kJoinBits = 12;
struct Range {  // per vector: nonzero amplitudes << 16 | small ones (both below 2^14)
  uint32_t in[kMaxVec], out[kMaxVec];
  uint32_t tiny_in, tiny_out;  // bit per vector
};

struct Args {
  double2* st[2];  // blockIdx.y chooses: psi and the cotangent share a program
  int64_t d_b;
  int dir, d, nvec, KV, nsteps, norb, nchunk, has_x;
  const Seg* seg;        // per window position
  const uint16_t* idx;
  int cap_first, cap_rest;  // bytes of the staged addresses: class 3; the others
  const unsigned char* img;
  const uint32_t *masks_this, *masks_other;
  const double2 *ea_this, *ea_other;  // phases
  int* status;
  int* scale;  // null, or [2][nvec]: see launch_sweep_fx
  uint8_t a[kMaxSteps];     // window position of each step
  uint8_t full[kMaxSteps];  // class 6 moves in this step (det V != 1)
  // the program rotation by rotation, for vectors that take FP64
  const uint32_t* pairs;  // adjacent pair lists
  int npp, m, weak, joined;
  long long phase[2 * kMaxOrb];  // the diagonal layer, fixed point
  double c[kMaxGivens], sr[kMaxGivens], si[kMaxGivens];
  int8_t p[kMaxGivens];
};

__device__ __forceinline__ bool not_zero(double2 x) {
  return ((__double2hiint(x.x) | __double2hiint(x.y)) & 0x7FFFFFFF) | __double2loint(x.x) |
         __double2loint(x.y);
}

// A barrier of the sixteen data warps.
__device__ __forceinline__ void sync_data() {
  asm volatile("bar.sync 1, %0;" ::"n"(kThreads) : "memory");
}

// The vectors of `wide` (bit per vector of the slab) in FP64, by all data
// threads: from the state into their cells, rotation by rotation over the pairs
// of all of them (a pair list entry is read while the one before it is used),
// with the phases back to the state.  dtab: where the images were, for the
// diagonal layer (8 orbitals an entry); tab: the cross tables (null: none), bad_x the orbitals without an
// angle there; at: scratch for the first cells of the vectors.
static_assert((kMaxOrb + 7) / 8 * 256 * 16 <= kImgBytes, "");
__device__ __noinline__ void rotate_fp64(const Args& g, uint32_t wide, double2* slab,
                                         double2* state, longlong2* dtab, const longlong2* tab,
                                         const uint32_t* bad_x, int* at, int v0, int nv, int tid) {
  const int nw = __popc(wide), d = g.d, npp = g.npp, m = g.m, items = npp * nw;
  auto each = [&](auto&& f) {  // (vector, element, its place in the state)
    if (g.dir == 1) {
      for (uint32_t w = wide; w; w &= w - 1) {
        const int kv = __ffs(w) - 1;
        for (int e = tid; e < d; e += kThreads) f(kv, e, (int64_t)(v0 + kv) * g.d_b + e);
      }
    } else {
      for (int i = tid; i < d * nv; i += kThreads) {
        const int e = i / nv, kv = i - e * nv;
        if ((wide >> kv) & 1) f(kv, e, (int64_t)e * g.d_b + v0 + kv);
      }
    }
  };
  each([&](int kv, int e, int64_t s) { slab[(size_t)kv * d + e] = state[s]; });
  if (tid < nv && ((wide >> tid) & 1)) at[__popc(wide & ((1u << tid) - 1))] = tid * d;
  for (int i = tid; i < g.nchunk * 256; i += kThreads) {
    const uint64_t mask = (uint64_t)(i & 255) << (i / 256 * 8) & ((1ull << g.norb) - 1);
    longlong2 z = make_longlong2(1ll << 62, 0);
    for (uint32_t b = (uint32_t)mask; b; b &= b - 1) {
      const int p = __ffs(b) - 1;
      z = phase_mul(z, make_longlong2(g.phase[2 * p], g.phase[2 * p + 1]));
    }
    dtab[i] = z;
  }
  sync_data();
  const int first = tid % npp;
  uint32_t next = tid < items ? __ldg(g.pairs + (int64_t)g.p[0] * npp + first) : 0u;
  for (int k = 0; k < m; ++k) {
    const uint32_t* l = g.pairs + (int64_t)g.p[k] * npp;
    const double c = g.c[k], sr = g.sr[k], si = g.si[k];
    int w = tid / npp;
    for (int i = tid; i < items;) {
      const uint32_t pr = next;
      double2* x = slab + at[w];
      i += kThreads;
      if (i < items) {
        w = i / npp;
        next = __ldg(l + (i - w * npp));
      } else if (k + 1 < m) {
        next = __ldg(g.pairs + (int64_t)g.p[k + 1] * npp + first);
      }
      double2 a = x[pr & 0xFFFFu], b = x[pr >> 16];
      givens2<double>(a, b, c, sr, si);
      x[pr & 0xFFFFu] = a;
      x[pr >> 16] = b;
    }
    sync_data();
  }
  each([&](int kv, int e, int64_t s) {
    const uint32_t bits = __ldg(g.masks_this + e);
    const longlong2* t = tab ? tab + kv * g.nchunk * 256 : nullptr;
    longlong2 f = make_longlong2(1ll << 62, 0);
    for (int k = 0; k < g.nchunk; ++k) {
      const int v = k * 256 + ((bits >> (8 * k)) & 255);
      f = k ? phase_mul(f, dtab[v]) : dtab[v];
      if (t) f = phase_mul(f, t[v]);
    }
    double2 z = phase_to(f);
    if (g.ea_this) z = cmul<double>(z, __ldg(g.ea_this + e));
    if (g.ea_other) z = cmul<double>(z, __ldg(g.ea_other + v0 + kv));
    state[s] = t && (bits & bad_x[kv]) ? nan2() : cmul<double>(z, slab[(size_t)kv * d + e]);
  });
}

// Walks the tiles of a step: class cls(ci), rows row0 ..; ci = 5 past the
// last.  on_rest runs when the walk leaves class 3.
struct Walk {
  int ci = 0, row0 = 0;
  template <typename F>
  __device__ __forceinline__ void settle(const Seg& sg, int nv, F&& on_rest) {
    while (ci < 5 && row0 >= sg.cnt[ci] * nv) {
      if (ci == 0) on_rest();
      ++ci;
      row0 = 0;
    }
  }
};

// One CTA per slab, one CTA per SM (all of its TMEM): sixteen data warps and
// one that stages the images and issues the products.  (An issue blocks while
// the tensor cores are busy, and a data warp that issued a tile kept the
// other fifteen waiting.)  With 17 warps a thread has 96 registers, so the
// accumulators are taken two strings at a time.
__global__ void __launch_bounds__(kCta, 1)
    k_sweep_fx(const __grid_constant__ Args g, const __grid_constant__ Mat X) {
  extern __shared__ __align__(128) unsigned char smraw[];
  __shared__ __align__(8) uint64_t s_mbar[4];
  __shared__ uint32_t s_tmem;
  __shared__ uint32_t s_max[kMaxVec][kWarps];
  __shared__ float s_sum[kMaxVec][kWarps];
  __shared__ Seg s_seg[kMaxSteps];
  __shared__ int s_eb[kMaxVec];  // biased exponent of the scale, -1: not finite
  __shared__ Range s_range;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  double2* const state = g.st[blockIdx.y];
  const int d = g.d, v0 = blockIdx.x * g.KV, nv = min(g.KV, g.nvec - v0);
  unsigned char* simg = smraw;
  uint16_t* ix_first = reinterpret_cast<uint16_t*>(smraw + kImgBytes);
  uint16_t* ix_rest = reinterpret_cast<uint16_t*>(smraw + kImgBytes + g.cap_first);
  longlong2* slab = reinterpret_cast<longlong2*>(smraw + kImgBytes + g.cap_first + g.cap_rest);
  const uint32_t bar_first = tc::smem_u32(&s_mbar[0]), bar_rest = tc::smem_u32(&s_mbar[1]);
  const uint32_t bar_mma = tc::smem_u32(&s_mbar[2]), bar_ready = tc::smem_u32(&s_mbar[3]);
  if (tid == 0) {
    for (int i = 0; i < 3; ++i) tc::mbar_init(tc::smem_u32(&s_mbar[i]), 1);
    tc::mbar_init(bar_ready, kWarps);
    tc::mbar_fence_init();
  }
  if (warp == 0) tc::tmem_alloc(tc::smem_u32(&s_tmem), 512);
  for (int i = tid; i < g.nsteps; i += kCta) s_seg[i] = g.seg[g.a[i]];
  if (tid < kMaxVec) s_range.in[tid] = s_range.out[tid] = 0;
  if (tid == 0) s_range.tiny_in = s_range.tiny_out = 0;
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  // bits per vector, the same in all threads: the vectors of a wide range as
  // counted, of zeros throughout, and (the first, before any rotation) those
  // that go to FP64 at once and those that their result decides on
  const uint32_t small_bits = g.joined ? kSmallBits : kApartBits;
  auto wide_range = [&](const uint32_t (&count)[kMaxVec], uint32_t tiny) {
    return tiny | __ballot_sync(0xFFFFFFFFu,
                                lane < nv && (count[lane] & 0xFFFFu) * 16 > (uint32_t)d);
  };
  auto decide = [&](uint32_t& zero, uint32_t& later) {
    const uint32_t nz = lane < nv ? s_range.in[lane] >> 16 : 0;
    const bool fin = lane < nv && s_eb[lane] >= 0;
    zero = __ballot_sync(0xFFFFFFFFu, fin && nz == 0);
    const uint32_t some = __ballot_sync(0xFFFFFFFFu, fin && nz > 0 && nz < (uint32_t)d);
    const uint32_t range = wide_range(s_range.in, s_range.tiny_in) & ~zero;
    const uint32_t now = __ballot_sync(0xFFFFFFFFu, lane < nv && !fin) |
                         (g.weak ? some : 0) | (g.joined ? 0 : range);
    later = (some | range) & ~now;
    return now;
  };
  const uint32_t all = nv == 32 ? 0xFFFFFFFFu : (1u << nv) - 1;
  if (warp == kWarps) {
    // a step's images and gather addresses: class 3, then the other
    // classes, each copy issued once the step before has used its half
    auto stage_first = [&](int st) {
      const Seg& q = s_seg[st];
      const uint32_t len = 2u * (uint32_t)(q.start[1] - q.start[0]);
      tc::mbar_expect_tx(bar_first, kImgFirst + len);
      tc::bulk_g2s(tc::smem_u32(simg), g.img + (size_t)st * kStepBytes, kImgFirst, bar_first);
      if (len) tc::bulk_g2s(tc::smem_u32(ix_first), g.idx + q.start[0], len, bar_first);
    };
    auto stage_rest = [&](int st) {
      const Seg& q = s_seg[st];
      const uint32_t len = 2u * (uint32_t)(q.start[5] - q.start[1]);
      tc::mbar_expect_tx(bar_rest, kImgBytes - kImgFirst + len);
      tc::bulk_g2s(tc::smem_u32(simg) + kImgFirst, g.img + (size_t)st * kStepBytes + kImgFirst,
                   kImgBytes - kImgFirst, bar_rest);
      if (len) tc::bulk_g2s(tc::smem_u32(ix_rest), g.idx + q.start[1], len, bar_rest);
    };
    if (lane == 0) {
      stage_first(0);
      stage_rest(0);
    }
    __syncthreads();  // the vectors are loaded
    uint32_t zero, later;
    const bool skip = (decide(zero, later) | zero) == all;
    if (lane == 0 && skip) {  // no tiles: the copies have to land all the same
      if (!tc::mbar_wait(bar_first, 0)) timeout(g.status);
      if (!tc::mbar_wait(bar_rest, 0)) timeout(g.status);
    } else if (lane == 0) {
      const uint32_t tbase = s_tmem, bimg = tc::smem_u32(simg);
      uint32_t ph = 0, phr = 0;  // phases of the products and of the data warps
      for (int st = 0; st < g.nsteps; ++st) {
        const Seg& sg = s_seg[st];
        const uint32_t phs = (uint32_t)st & 1u;
        const bool more = st + 1 < g.nsteps;
        bool ahead = false;  // the next step's class 3 copy is under way
        if (!tc::mbar_wait(bar_first, phs)) timeout(g.status);
        Walk wk;
        // leaving class 3: its products are done and its addresses read (a
        // step without any has not been seen by every data warp yet)
        auto leave3 = [&]() {
          ahead = more && sg.cnt[0] > 0;
          if (ahead) stage_first(st + 1);
          if (!tc::mbar_wait(bar_rest, phs)) timeout(g.status);
        };
        wk.settle(sg, nv, leave3);
        while (wk.ci < 5) {
          if (!tc::mbar_wait(bar_ready, phr)) timeout(g.status);
          phr ^= 1u;
          tc::fence_after();
          const uint32_t b0 = bimg + img_offset(cls(wk.ci));
          if (wk.ci == 0) issue<3>(tbase, b0, bar_mma);
          else if (wk.ci < 3) issue<2>(tbase, b0, bar_mma);
          else issue<1>(tbase, b0, bar_mma);
          if (!tc::mbar_wait(bar_mma, ph)) timeout(g.status);
          ph ^= 1u;
          wk.row0 += tc::kRows;
          wk.settle(sg, nv, leave3);
        }
        // the data warps have ended the step
        if (!tc::mbar_wait(bar_ready, phr)) timeout(g.status);
        phr ^= 1u;
        if (more && !ahead) stage_first(st + 1);
        if (more) stage_rest(st + 1);
      }
    }
    return;
  }
  // ---- load
  double2* raw = reinterpret_cast<double2*>(slab);
  auto cp16 = [&](double2* dst, const double2* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(tc::smem_u32(dst)), "l"(src)
                 : "memory");
  };
  if (g.dir == 1) {
    for (int kv = 0; kv < nv; ++kv) {
      const double2* src = state + (int64_t)(v0 + kv) * g.d_b;
      for (int e = tid; e < d; e += kThreads) cp16(raw + (size_t)kv * d + e, src + e);
    }
  } else {
    for (int i = tid; i < d * nv; i += kThreads) {
      const int e = i / nv, kv = i - e * nv;
      cp16(raw + (size_t)kv * d + e, state + (int64_t)e * g.d_b + v0 + kv);
    }
  }
  // zeros in the A columns no tile writes (their B rows are zero, but a NaN
  // left in TMEM would not be)
  {
    const uint32_t z[4] = {0, 0, 0, 0};
    const uint32_t l0 = s_tmem + ((uint32_t)((warp & 3) * 32) << 16);
    for (int c = 4 * (warp >> 2); c < kColD; c += 16) tc::tmem_st4(l0 + c, z);
    tc::wait_st();
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
  sync_data();
  // ---- scale of each vector: the exponent of its largest part, then its
  // 2-norm in FP32 relative to that; `per` warps share a vector
  const int per = nv >= kWarps ? 1 : kWarps / nv, ngrp = kWarps / per;
  const int kv1 = warp / per, sub = warp - kv1 * per;
  if (kv1 < ngrp)
    for (int kv = kv1; kv < nv; kv += ngrp) {
      uint32_t mx = 0;
#pragma unroll 4
    for (int e = sub * 32 + lane; e < d; e += 32 * per) {
        const double2 x = raw[(size_t)kv * d + e];
        mx = max(mx, (uint32_t)exp_field(x.x));
        mx = max(mx, (uint32_t)exp_field(x.y));
      }
      mx = __reduce_max_sync(0xFFFFFFFFu, mx);
      if (lane == 0) s_max[kv][sub] = mx;
    }
  sync_data();
  if (kv1 < ngrp)
    for (int kv = kv1; kv < nv; kv += ngrp) {
      uint32_t f = 1;
      for (int i = 0; i < per; ++i) f = max(f, s_max[kv][i]);
      float s = 0.f;
#pragma unroll 4
    for (int e = sub * 32 + lane; e < d; e += 32 * per) {
        const double2 x = raw[(size_t)kv * d + e];
        const float a = rel_abs(x.x, (int)f), b = rel_abs(x.y, (int)f);
        s = fmaf(a, a, fmaf(b, b, s));
      }
#pragma unroll
      for (int k = 16; k > 0; k >>= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, k);
      if (lane == 0) s_sum[kv][sub] = s;
    }
  sync_data();
  if (kv1 < ngrp)
    for (int kv = kv1; kv < nv; kv += ngrp) {
      uint32_t f = 1;
      float s = 0.f;
      for (int i = 0; i < per; ++i) {
        f = max(f, s_max[kv][i]);
        s += s_sum[kv][i];
      }
      const bool finite = f < 0x7FF;
      const int eb = norm_exponent((int)f, s);
      if (sub == 0 && lane == 0) s_eb[kv] = finite ? eb : -1;
      uint32_t count = 0, tiny = 0;
#pragma unroll 4
    for (int e = sub * 32 + lane; e < d; e += 32 * per) {
        const double2 x = raw[(size_t)kv * d + e];
        slab[(size_t)kv * d + e] = finite ? make_longlong2(from_double(x.x, eb), from_double(x.y, eb))
                                          : make_longlong2(0, 0);
        const int q = max(exp_field(x.x), exp_field(x.y));
        const bool nz = q || not_zero(x);
        count += nz ? 0x10000u + (q < eb - (int)small_bits) : 0u;
        tiny |= nz && q < eb - kTinyBits;
      }
      count = __reduce_add_sync(0xFFFFFFFFu, count);
      tiny = __reduce_or_sync(0xFFFFFFFFu, tiny);
      if (lane == 0) {
        atomicAdd(&s_range.in[kv], count);
        if (tiny) atomicOr(&s_range.tiny_in, 1u << kv);
      }
    }
  Thread t;
  t.wg = warp >> 2;
  t.row = (warp & 3) * 32 + lane;
  t.lane0 = s_tmem + ((uint32_t)((warp & 3) * 32) << 16);
  uint32_t ph_mma = 0;
  __syncthreads();  // with the issuing warp
  uint32_t zero, later;
  uint32_t wide = decide(zero, later);
  const bool skip = (wide | zero) == all;
  if (skip) {  // the tables below go where the copies land
    if (!tc::mbar_wait(bar_first, 0)) timeout(g.status);
    if (!tc::mbar_wait(bar_rest, 0)) timeout(g.status);
  }
  // ---- window steps.  The tiles of a step touch different strings, so
  // they run as a pipeline: while the products of one tile run, the warps
  // join and scatter the tile before it and gather the tile after it.
  for (int st = 0; st < g.nsteps && !skip; ++st) {
    const Seg& sg = s_seg[st];
    const uint32_t ph = (uint32_t)st & 1u;
    Walk wk;
    auto leave3 = [&]() {
      if (!tc::mbar_wait(bar_rest, ph)) timeout(g.status);
    };
    Item cur, nxt;
    uint32_t w[5][kDig];
    // a warp whose 32 rows lie past the class's last, or that owns no
    // string of the class, leaves the tile alone
    auto active = [&]() {
      return wk.ci < 5 && wk.row0 + (warp & 3) * 32 < sg.cnt[wk.ci] * nv &&
             (wk.ci < 3 || t.wg < 3);
    };
    auto load = [&](Item& it) {  // gathers the next tile
      const int ci = wk.ci, cnt = sg.cnt[ci], rows = cnt * nv;
      const uint16_t* ix = ci == 0 ? ix_first : ix_rest + (sg.start[ci] - sg.start[1]);
      if (ci == 0) gather<3>(t, slab, d, ix, cnt, rows, wk.row0, it, w);
      else if (ci < 3) gather<2>(t, slab, d, ix, cnt, rows, wk.row0, it, w);
      else gather<1>(t, slab, d, ix, cnt, rows, wk.row0, it, w);
    };
    auto put = [&](int c) {
      if (c == 0) put_digits<3>(t, w);
      else if (c < 3) put_digits<2>(t, w);
      else put_digits<1>(t, w);
    };
    auto ready = [&]() {
      tc::wait_st();
      tc::fence_before();
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(bar_ready);
    };
    if (!tc::mbar_wait(bar_first, ph)) timeout(g.status);
    wk.settle(sg, nv, leave3);
    int cc = wk.ci;  // class of the tile whose products run
    bool ac = active();
    if (cc < 5) {
      if (ac) {
        load(cur);
        put(cc);
      }
      ready();
    }
    while (cc < 5) {
      wk.row0 += tc::kRows;
      wk.settle(sg, nv, leave3);
      const int cn = wk.ci;
      const bool an = active();
      if (an) load(nxt);
      if (!tc::mbar_wait(bar_mma, ph_mma)) timeout(g.status);
      ph_mma ^= 1u;
      tc::fence_after();
      if (an) put(cn);
      uint32_t f[kSum][4];
      if (ac) {
        if (cc == 0) finish_fifth(t, slab, cur);
        if (cc == 0) take<3>(t, 0, f);
        else if (cc < 3) take<2>(t, 0, f);
        else take<1>(t, 0, f);
        if (cc < 3) {
          scatter(slab, cur, 0, f);
          if (cc == 0) take<3>(t, 2, f);
          else take<2>(t, 2, f);
        }
      }
      if (cn < 5) ready();
      if (ac) scatter(slab, cur, cc < 3 ? 2 : 0, f);
      cur = nxt;
      cc = cn;
      ac = an;
    }
    ready();
    if (g.full[st]) {
      const longlong2 z = __ldg(reinterpret_cast<const longlong2*>(
          g.img + (size_t)st * kStepBytes + kImgBytes));
      const int cnt = sg.cnt[5];
      for (int i = tid; i < cnt * nv; i += kThreads) {
        const int kv = i / cnt, o = i - kv * cnt;
        longlong2* c = slab + (size_t)kv * d + __ldg(g.idx + sg.start[5] + o);
        const longlong2 x = *c;
        *c = cmul_fx(x, z);
      }
    }
    sync_data();
  }
  if (warp == 0) {
    tc::fence_after();
    tc::tmem_dealloc(s_tmem, 512);
  }
  // ---- the range now of the vectors that it decides on
  if (later) {
    for (int kv = 0; kv < nv; ++kv) {
      if (!((later >> kv) & 1)) continue;
      uint32_t count = 0, tiny = 0;
      for (int e = tid; e < d; e += kThreads) {
        const longlong2 x = slab[(size_t)kv * d + e];
        const unsigned long long u =
            (unsigned long long)(x.x < 0 ? -x.x : x.x) | (unsigned long long)(x.y < 0 ? -x.y : x.y);
        count += u && u < 1ull << (kFrac - small_bits);
        tiny |= u && u < 1ull << (kFrac - kTinyBits);
      }
      count = __reduce_add_sync(0xFFFFFFFFu, count);
      tiny = __reduce_or_sync(0xFFFFFFFFu, tiny);
      if (lane == 0 && count) atomicAdd(&s_range.out[kv], count);
      if (lane == 0 && tiny) atomicOr(&s_range.tiny_out, 1u << kv);
    }
    sync_data();
    wide |= later & wide_range(s_range.out, s_range.tiny_out);
  }
  if (g.scale && tid < nv)
    g.scale[(int64_t)blockIdx.y * g.nvec + v0 + tid] = (wide >> tid) & 1 ? -1 : s_eb[tid];
  // ---- phases, store.  The cross tables go where the images were (every
  // copy has landed and been read).
  const int tper = g.nchunk * 256;
  longlong2* tab = slab + (size_t)g.KV * d;
  if (g.has_x)
    cross_tables(g.masks_other, g.dir, g.norb, g.nchunk, X, v0, nv, tab,
                 reinterpret_cast<longlong2*>(simg), &s_max[0][0], tid, kThreads, [] { sync_data(); });
  auto finish = [&](int kv, int e) {
    const int eb = s_eb[kv];
    longlong2 c = slab[(size_t)kv * d + e];
    bool bad = false;
    if (g.has_x || g.ea_this || g.ea_other) {
      longlong2 f = make_longlong2(1ll << 62, 0);
      auto factor = [&](double2 z) {
        bad = bad || not_finite(z);
        f = phase_mul(f, phase_from(z));
      };
      if (g.ea_this) factor(__ldg(g.ea_this + e));
      if (g.ea_other) factor(__ldg(g.ea_other + v0 + kv));
      if (g.has_x) {
        const uint32_t m = __ldg(g.masks_this + e);
        bad = bad || (m & (&s_max[0][0])[kv]);
        for (int k = 0; k < g.nchunk; ++k)
          f = phase_mul(f, tab[kv * tper + k * 256 + ((m >> (8 * k)) & 255)]);
      }
      c = cmul_fx(c, f);
    }
    double2 v = make_double2(to_double(c.x, eb), to_double(c.y, eb));
    return bad ? nan2() : v;
  };
  if (g.dir == 1) {
    for (int kv = 0; kv < nv; ++kv)
      if (!((wide >> kv) & 1))
        for (int e = tid; e < d; e += kThreads)
          state[(int64_t)(v0 + kv) * g.d_b + e] = finish(kv, e);
  } else {
    for (int i = tid; i < d * nv; i += kThreads) {
      const int e = i / nv, kv = i - e * nv;
      if (!((wide >> kv) & 1)) state[(int64_t)e * g.d_b + v0 + kv] = finish(kv, e);
    }
  }
  // ---- the others, still as they were in the state, in FP64
  if (wide) {
    sync_data();  // the tables are read
    rotate_fp64(g, wide, raw, state, reinterpret_cast<longlong2*>(simg),
                g.has_x ? tab : nullptr, &s_max[0][0], reinterpret_cast<int*>(&s_sum[0][0]), v0,
                nv, tid);
  }
}

// ------------------------------------------------------------------ host
// Bytes of the staged gather addresses, of class 3 and of the classes 2, 4, 1
// and 5 together: the orbits of class m are the (n - m)-subsets of the N - 6
// orbitals outside, at every window position.
static void caps(int N, int n, int (&out)[2]) {
  out[0] = out[1] = 0;
  for (int i = 0; i < 5; ++i) {
    const int m = cls(i), k = n - m;
    int64_t c = k < 0 || k > N - tc::kW ? 0 : 1;
    for (int j = 1; c && j <= k; ++j) c = c * (N - tc::kW - k + j) / j;
    const int64_t b = (c * 4 * grp_pad(m) * 2 + 15) / 16 * 16;
    out[i > 0] += (int)std::min<int64_t>(b, 1 << 24);
  }
  for (int& x : out) x = (x + 127) / 128 * 128;
}

// Gather addresses of the steps, per window position: the classes 3, 2, 4,
// 1, 5 and 6, each as its four column groups of `count` orbit rows (class 6:
// one address per orbit); the orbits of a class in window_tables_host's
// order, whose aligned groups of eight read distinct banks.
static void build_index(Space* sp) {
  if (sp->fx_seg) return;
  const int N = sp->norb, n = sp->nocc, npos = N - tc::kW + 1;
  std::vector<uint32_t> orbits;
  std::vector<int> off;
  std::vector<uint16_t> offs;
  std::vector<uint8_t> okey;
  window_tables_host(N, n, tc::kW, orbits, off, offs, okey);
  std::vector<uint8_t> list[7];
  for (int x = 0; x < 64; ++x) list[__builtin_popcount(x)].push_back((uint8_t)x);
  std::vector<Seg> seg(npos);
  std::vector<uint16_t> idx;
  for (int a = 0; a < npos; ++a) {
    for (int ci = 0; ci < 5; ++ci) {
      const int m = cls(ci), P = grp_pad(m);
      std::vector<uint32_t> os;
      for (int k = off[a]; k < off[a + 1]; ++k)
        if ((int)(orbits[k] >> 24) == m) os.push_back(orbits[k]);
      while (idx.size() % 8) idx.push_back(0);
      seg[a].start[ci] = (int)idx.size();
      seg[a].cnt[ci] = (int)os.size();
      for (int g = 0; g < 4; ++g)
        for (uint32_t o : os) {
          const uint16_t* F = offs.data() + (((size_t)a * (n + 1) + ((o >> 16) & 0xFF)) << tc::kW);
          for (int j = 0; j < P; ++j) {
            const int s = grp_string(m, g, j);
            idx.push_back(s < 0 ? (uint16_t)0xFFFF : (uint16_t)((o & 0xFFFF) + F[list[m][s]]));
          }
        }
    }
    // class 6: the strings that fill the window
    while (idx.size() % 8) idx.push_back(0);
    seg[a].start[5] = (int)idx.size();
    int cnt = 0;
    const uint32_t win = 63u << a;
    int64_t r = 0;
    if (n >= 6) {  // strings in ascending order, as addresses are
      uint64_t x = (1ull << n) - 1;
      for (; !(x >> N); ++r) {
        if (((uint32_t)x & win) == win) {
          idx.push_back((uint16_t)r);
          ++cnt;
        }
        const uint64_t c = x & (~x + 1), y = x + c;
        x = (((y ^ x) >> 2) / c) | y;
      }
    }
    seg[a].cnt[5] = cnt;
  }
  while (idx.size() % 8) idx.push_back(0);
  if (sp->fx_idx) FS_CUDA(cudaFree(sp->fx_idx));  // of an attempt without room for the rest
  sp->fx_idx = nullptr;
  FS_CUDA(cudaMalloc(&sp->fx_idx, std::max<size_t>(idx.size(), 8) * sizeof(uint16_t)));
  FS_CUDA(cudaMemcpy(sp->fx_idx, idx.data(), idx.size() * sizeof(uint16_t),
                     cudaMemcpyHostToDevice));
  sp->fx_seg_h = seg;
  Seg* ds = nullptr;
  FS_CUDA(cudaMalloc(&ds, seg.size() * sizeof(Seg)));
  const cudaError_t e =
      cudaMemcpy(ds, seg.data(), seg.size() * sizeof(Seg), cudaMemcpyHostToDevice);
  if (e != cudaSuccess) cudaFree(ds);
  FS_CUDA(e);
  sp->fx_seg = ds;
}

}  // namespace fx

// Host fixed point with 62 fraction bits.
static inline int64_t hmul(int64_t a, int64_t b) {
  return (int64_t)(((__int128)a * b + ((__int128)1 << 61)) >> 62);
}
static inline int64_t hfix(double x) { return (int64_t)std::llrint(std::ldexp(x, 62)); }
// Scales x (n reals in fixed point, 2-norm 1 up to FP64 rounding) to 2-norm 1.
static void hunit(int64_t* x, int n) {
  __int128 s = (__int128)1 << 124;
  for (int i = 0; i < n; ++i) s -= (__int128)x[i] * x[i];
  const int64_t h = (int64_t)(s >> 63);  // (1 - norm^2) / 2
  for (int i = 0; i < n; ++i) x[i] += hmul(x[i], h);
}

static void unit_phase(zd d, int64_t* z) {
  z[0] = hfix(d.real());
  z[1] = hfix(d.imag());
  hunit(z, 2);
}

// The steps of a program (into plan and, as unitaries V, row-major 6 x 6
// complex fixed point, into V: products of FP64 matrices would put an error
// of some 2^-52 into each entry, the same for every amplitude), the diagonal
// layer multiplied into the last step that covers each orbital.  False when
// the program does not suit the sweep: a phase falls outside every window, or
// it has too many steps, or too few rotations a step, or an entry that no
// integer stands for (infinite, or not a number).
static bool fx_steps(Ctx* ctx, const RotProgram& rp, int N, FxPlan& plan,
                     std::vector<std::array<int64_t, 72>>& V) {
  const std::vector<WinStep>& steps = window_schedule(ctx, rp, N, tc::kW);
  if (steps.empty() || (int)steps.size() > fx::kMaxSteps ||
      rp.g.size() < fx::kMinGivensPerStep * steps.size() || !rp.finite())
    return false;
  std::vector<int> last(N, -1);
  for (size_t s = 0; s < steps.size(); ++s)
    for (int p = steps[s].a; p < steps[s].a + tc::kW; ++p) last[p] = (int)s;
  for (int p = 0; p < N; ++p)
    if (last[p] < 0 && rp.phase[p] != zd(1.0)) return false;
  // what the moduli of the rotations join (see Range)
  std::vector<double> join((size_t)N * N, 0.0);
  for (int p = 0; p < N; ++p) join[(size_t)p * N + p] = 1.0;
  plan.weak = false;
  for (const Givens& G : rp.g) {
    const double c = std::abs(G.c), s = std::abs(G.s), weaker = std::min(c, s);
    plan.weak = plan.weak || (weaker > 0 && weaker < std::ldexp(1.0, -fx::kWeakBits));
    double* x = join.data() + (size_t)G.p * N;
    for (int j = 0; j < N; ++j) {
      const double u = x[j], v = x[N + j];
      x[j] = c * u + s * v;
      x[N + j] = s * u + c * v;
    }
  }
  plan.joined =
      *std::min_element(join.begin(), join.end()) >= std::ldexp(1.0, -fx::kJoinBits);
  plan.nsteps = (int)steps.size();
  V.resize(steps.size());
  for (size_t s = 0; s < steps.size(); ++s) {
    const int a = steps[s].a;
    plan.a[s] = (uint8_t)a;
    auto& M = V[s];
    M.fill(0);
    for (int i = 0; i < 6; ++i) M[14 * i] = (int64_t)1 << 62;
    for (int k : steps[s].givens) {
      const Givens& G = rp.g[k];
      int64_t g[3] = {hfix(G.c), hfix(G.s.real()), hfix(G.s.imag())};
      hunit(g, 3);
      int64_t* x = M.data() + 12 * (G.p - a);
      for (int j = 0; j < 6; ++j) {
        const int64_t ur = x[2 * j], ui = x[2 * j + 1], vr = x[12 + 2 * j], vi = x[13 + 2 * j];
        x[2 * j] = hmul(g[0], ur) + hmul(g[1], vr) - hmul(g[2], vi);
        x[2 * j + 1] = hmul(g[0], ui) + hmul(g[1], vi) + hmul(g[2], vr);
        x[12 + 2 * j] = hmul(g[0], vr) - hmul(g[1], ur) - hmul(g[2], ui);
        x[13 + 2 * j] = hmul(g[0], vi) - hmul(g[1], ui) + hmul(g[2], ur);
      }
    }
    plan.full[s] = 0;
    for (int p = a; p < a + tc::kW; ++p) {
      if (last[p] != (int)s || rp.phase[p] == zd(1.0)) continue;
      int64_t z[2];
      unit_phase(rp.phase[p], z);
      int64_t* x = M.data() + 12 * (p - a);
      for (int j = 0; j < 6; ++j) {
        const int64_t re = hmul(x[2 * j], z[0]) - hmul(x[2 * j + 1], z[1]);
        x[2 * j + 1] = hmul(x[2 * j], z[1]) + hmul(x[2 * j + 1], z[0]);
        x[2 * j] = re;
      }
      plan.full[s] = 1;
    }
  }
  return true;
}

// Sectors the sweep takes: a window of orbitals, a vector and its step's
// images in one SM's shared memory, and enough amplitudes.
static bool fx_sector(const Ctx* ctx, const Space* sthis, const Space* sother) {
  if (sthis->norb < tc::kW || sthis->dim < 2 || sthis->dim * sother->dim < fx::kMinAmps)
    return false;
  int caps[2];
  fx::caps(sthis->norb, sthis->nocc, caps);
  const size_t tab = (size_t)((sthis->norb + 7) / 8) * 256 * 16;
  return fx::kImgBytes + (size_t)caps[0] + caps[1] + (size_t)sthis->dim * 16 + tab <=
         (size_t)ctx->prop.sharedMemPerBlockOptin - fx::kStaticBytes;
}

// Whether the forward sweep of a program is faster in digits (engine AUTO).  On
// few vectors both sweeps are chains of latencies.  Measured for one spin, up
// to one vector an SM, the FP64 sweep takes some 18 us and 1.25 us a rotation up
// to 300 strings, 1.65 at 924 (N = 12, n = 6), 3.4 at 3432; the digits 38 us
// and 5 us a step at 120 strings, 8 to 11 from 300 on.  N = 12 (12,6): 134
// against 95 us for a dense rotation (66 rotations, 6 steps), but 44 against 47
// for one of six orbitals (15, 1), and 67 against 86 for a Givens gate between
// the outer orbitals (21, 5).
static bool fx_pays(Ctx* ctx, const Space* sthis, const Space* sother, const RotProgram& rp) {
  const double d = (double)sthis->dim;
  const int64_t sms = ctx->prop.multiProcessorCount;
  const double waves = (double)((sother->dim + sms - 1) / sms);
  const double steps = (double)window_schedule(ctx, rp, sthis->norb, tc::kW).size();
  return (double)rp.g.size() * std::max(1.25, 1.0 + 7e-4 * d) * waves >=
         20.0 + steps * std::min(2.5 + 0.02 * d, 8.2 + 7e-4 * d);
}

FxPair fx_prepare(Ctx* ctx, const Space* sa, const Space* sb, int dtype, const RotProgram& pa,
                  const RotProgram& pb, bool forward, cudaStream_t st) {
  FxPair r;
  if (dtype != FS_C128 || ctx->sweep_engine == FS_SWEEP_CUDA_CORE || ctx->prop.major < 10)
    return r;
  const RotProgram* rp[2] = {&pa, &pb};
  bool sect[2] = {fx_sector(ctx, sa, sb), fx_sector(ctx, sb, sa)};
  unsigned char* img = nullptr;
  for (int s = 0; s < 2; ++s) {
    Space* sp = const_cast<Space*>(s ? sb : sa);
    if (forward) build_forward_tables_f64(sp);
    if (!sect[s]) continue;
    // (images of the longest programs, of both spins)
    constexpr size_t bytes = (size_t)2 * fx::kMaxSteps * fx::kStepBytes;
    if (!(sp->fx_seg && scratch_fits(ctx, "fx_images", bytes)) && capturing(st)) {
      sect[s] = false;
      continue;
    }
    try {
      fx::build_index(sp);
      img = (unsigned char*)scratch(ctx, "fx_images", bytes);
    } catch (const Fail&) {  // no room: the FP64 sweep needs neither
      sect[s] = false;
    }
  }
  for (int s = 0; forward && s < 2; ++s) {
    const Space *a = s ? sb : sa, *b = s ? sa : sb;
    sect[s] = sect[s] && !pairs_supported(ctx, a, b, dtype, *rp[s]) &&
              (ctx->sweep_engine != FS_SWEEP_AUTO || fx_pays(ctx, a, b, *rp[s]));
  }
  const bool shared = &pa == &pb;  // one program for both spins
  bool ok[2] = {false, false};
  std::vector<std::array<int64_t, 72>> V[2];
  for (int s = 0; s < 2; ++s) {
    if (shared ? s == 0 && (sect[0] || sect[1]) : sect[s])
      ok[s] = fx_steps(ctx, *rp[s], sa->norb, r.plan[s], V[s]);
  }
  const int n0 = ok[0] ? r.plan[0].nsteps : 0, n1 = ok[1] ? r.plan[1].nsteps : 0;
  if (n0 + n1 == 0) return r;
  r.plan[0].img = img;
  r.plan[1].img = img + (size_t)n0 * fx::kStepBytes;
  {
    ProfScope ps("fx_images", st, n0 + n1 > fx::kMaxSteps ? 2 : 1);
    fx::StepMats sm;
    int k = 0, at = 0;
    auto flush = [&]() {
      if (k == 0) return;
      fx::k_fx_images<<<dim3(k, 2), 512, 0, st>>>(sm, img + (size_t)at * fx::kStepBytes);
      FS_CUDA(cudaGetLastError());
      at += k;
      k = 0;
    };
    for (int s = 0; s < 2; ++s) {
      if (!ok[s]) continue;
      if (k + r.plan[s].nsteps > fx::kMaxSteps) flush();
      for (int q = 0; q < r.plan[s].nsteps; ++q, ++k) std::copy(V[s][q].begin(), V[s][q].end(), sm.v[k]);
    }
    flush();
  }
  if (shared) {
    for (int s = 0; s < 2; ++s)
      if (ok[0] && sect[s]) r.use[s] = 0;
  } else {
    for (int s = 0; s < 2; ++s)
      if (ok[s]) r.use[s] = s;
  }
  return r;
}

void launch_sweep_fx(Ctx* ctx, const Space* sa, const Space* sb, int dir, void* st0, void* st1,
                     const FxPlan& plan, const RotProgram& rp, const PhaseDev& ph,
                     cudaStream_t st, int* scale) {
  const Space* sthis = dir == 0 ? sa : sb;
  const Space* sother = dir == 0 ? sb : sa;
  fx::Args g{};
  g.st[0] = (double2*)st0;
  g.st[1] = (double2*)st1;
  const int nst = st1 ? 2 : 1;
  g.d_b = sb->dim;
  g.dir = dir;
  g.d = (int)sthis->dim;
  g.nvec = (int)sother->dim;
  g.nsteps = plan.nsteps;
  std::copy(plan.a, plan.a + plan.nsteps, g.a);
  std::copy(plan.full, plan.full + plan.nsteps, g.full);
  g.img = plan.img;
  g.scale = scale;
  g.pairs = sthis->pairs;
  g.npp = sthis->npp;
  g.m = (int)rp.g.size();
  FS_REQUIRE(g.m <= kMaxGivens, FS_ERR_ARG, "too many Givens rotations");
  for (int k = 0; k < g.m; ++k) {
    const Givens& G = rp.g[k];
    g.p[k] = (int8_t)G.p;
    g.c[k] = G.c;
    g.sr[k] = G.s.real();
    g.si[k] = G.s.imag();
  }
  g.weak = plan.weak;
  g.joined = plan.joined;
  for (int p = 0; p < sthis->norb; ++p) {
    int64_t z[2];
    unit_phase(rp.phase[p], z);
    g.phase[2 * p] = z[0];
    g.phase[2 * p + 1] = z[1];
  }
  g.norb = sthis->norb;
  g.nchunk = (sthis->norb + 7) / 8;
  g.has_x = ph.has_x;
  g.seg = (const fx::Seg*)sthis->fx_seg;
  g.idx = sthis->fx_idx;
  g.masks_this = sthis->masks;
  g.masks_other = sother->masks;
  g.ea_this = (const double2*)(dir == 0 ? ph.ea_a : ph.ea_b);
  g.ea_other = (const double2*)(dir == 0 ? ph.ea_b : ph.ea_a);
  g.status = ctx->d_status;
  // vectors per slab: the width with the least modelled time, a wave of slabs
  // costing its tiles (weights of the classes' accumulator columns, 48, 32 and
  // 16, and what they do not share) and, worth a thousandth of a class 3 tile
  // each, its amplitudes' load and store.  Measured, one spin: N = 12 (6,6) 7
  // vectors 98 us (chosen), 4 147, 2 270, 10 125; N = 11 (6,5) 4 73 (chosen), 2
  // 135, 8 77, 16 110; N = 13 (5,7) alpha 6 272 (chosen), 4 387, 7 321; N = 16
  // (3,3) 4 114 (chosen), 2 187, 8 133, 16 214.
  const size_t tab = ph.has_x ? (size_t)g.nchunk * 256 * 16 : 0;
  int caps[2];
  fx::caps(sthis->norb, sthis->nocc, caps);
  g.cap_first = caps[0];
  g.cap_rest = caps[1];
  const size_t fixed = fx::kImgBytes + (size_t)caps[0] + caps[1];
  const size_t avail = (size_t)ctx->prop.sharedMemPerBlockOptin - fx::kStaticBytes - fixed;
  const int kvmax =
      std::max(1, std::min<int>(fx::kMaxVec, (int)(avail / ((size_t)g.d * 16 + tab))));
  const int sms = ctx->prop.multiProcessorCount;
  double best = 0;
  for (int kv = 1; kv <= kvmax; ++kv) {
    static const double w[5] = {1.0, 0.75, 0.75, 0.4, 0.4};
    double c = 0;
    for (int s = 0; s < g.nsteps; ++s) {
      const fx::Seg& sg = sthis->fx_seg_h[g.a[s]];
      for (int i = 0; i < 5; ++i) c += w[i] * ((sg.cnt[i] * kv + tc::kRows - 1) / tc::kRows);
    }
    c += 4.0 + 1e-3 * g.d * kv;
    const int slabs = nst * ((g.nvec + kv - 1) / kv);
    c *= (slabs + sms - 1) / sms;
    if (kv == 1 || c < best) {
      best = c;
      g.KV = kv;
    }
  }
  // more than half an SM's shared memory: the CTA owns all TMEM of its SM
  const size_t smem = std::max(fixed + (size_t)g.KV * ((size_t)g.d * 16 + tab),
                               (size_t)ctx->prop.sharedMemPerMultiprocessor / 2 + 1024);
  allow_shared_memory(fx::k_sweep_fx);
  ProfScope ps(dir == 0 ? "sweep_alpha_fx" : "sweep_beta_fx", st);
  fx::k_sweep_fx<<<dim3((g.nvec + g.KV - 1) / g.KV, nst), fx::kCta, smem, st>>>(g, ph.X);
  FS_CUDA(cudaGetLastError());
}

}  // namespace fs
