// Gradient of Radic's determinant with respect to the matrix entries.
//
// d det_R / d A[:, J] = sign(J) * adj(A[:, J])^T, the cofactor matrix of each
// minor, so the gradient of det_R(A) scatter-adds every minor's signed
// cofactors into the columns J of the gradient.  Per minor (one thread, in
// registers): partial-pivot LU P M = L U with the row order tracked in
// idx[], B = U^{-1} L^{-1} = M^{-1} P^T, and cofactor(idx[s], j) =
// det(M) * B[j][s].  A block owns one run of dictionary ranks of one matrix
// and adds its cofactors into a shared-memory copy of that matrix's gradient
// (shared-memory atomics); blocks write their tiles to per-block slots and a
// second kernel adds a matrix's slots in block order and scales by the
// incoming gradient.  Binary64 throughout.  A minor with an exactly zero
// pivot (singular) takes a slow path that forms its cofactors from
// (m-1) x (m-1) determinants.
//
// For 3 <= m the default kernel shares the work per head, the first H = m-G
// columns (G = 2..4), as the forward prefix kernels do, in binary64 or in
// pairs of binary32.  With the head's rows T (pivot order) and B (the other G),
// A = A_TT, W = -A_BT A^{-1}, every later column x has the Schur complement
// z(x) = x_B + W x_T, and the subtree of the head adds up to alpha L, alpha the
// signed product of the pivots and L the sum of det[z(x_1) ... z(x_G)] over
// x_1 < ... < x_G.  L is a polynomial of the z(x), linear in each: with P[S]
// and R[S] the sums of the determinants of the rows S over all ascending
// sequences of |S| columns before, and after, column q (column parities folded
// into z),
//   g_q,i = dL / dz_i(x_q) = sum over T not holding i of +- P[T] R[rest],
// the sign that of bringing the rows (T, i, rest) into order.  P and R follow
// from column to column by one exterior product with z, G 2^(G-1) multiply-adds
// each: P from the first column on, R from the last column back.  Both only
// ever take columns in.  (R could also follow P forwards, taking z(x_q) out
// again, but what is left keeps the rounding of the sums that held it: with one
// column r times the others the gradient's error grew like r^2 2^-53.)  The two
// run in opposite directions, so R is kept once per segment of columns on the
// way back, and each segment is built again from there, every column's R
// stored, when P comes to it.  Then column q receives
// alpha (-1)^q [W^T; I] g_q, and the head's own columns
// alpha [L A^{-1} - A^{-1} Q W | -A^{-1} Q]^T with Q = sum_q (-1)^q x_T(q) g_q^T.
// A head thus costs O(k G (2^G + m)) operations for its k later columns,
// whatever the number C(k, G) of its minors.
//
// What bounds it: the binary64 pipe (a warp instruction takes 16 cycles of an
// SM, whether or not all its lanes are used) or, in pairs, dependent binary32
// chains at 8 warps per SM.  G trades the number of heads, C(n-G, m-G),
// against the cost of a column (bwd_plan).  256 matrices of 6 x 28, binary64:
// 0.58 ms with G = 4 (6.0 ms with G = 2 and lanes grouped by equal v, the pipe
// 83% busy; 0.57 ms with R taken forwards, see above).
//
// Lanes take heads in colexicographic order (by last column v, then in
// dictionary order), so that a warp is full whatever the sizes of the groups
// of equal v, and step through the columns together from the smallest v on;
// a lane joins in after its own v.
//
// Gathering the gradient: each warp adds into its own tile in shared memory
// (binary64 or pairs, as the kernel computes), without atomics, and the block
// adds its warps' tiles in warp order at the end.  Later columns are summed
// over the warp in registers (a reduce-scatter of the m rows, one lane per
// entry); a head column is added once per distinct column in the warp, or lane
// by lane where many lanes have columns of their own.  (Atomic binary64
// additions to shared memory retry under contention; adding every entry that
// way, with 32 lanes on one column, made them the bulk of the kernel.)
//
// A head with an exactly zero pivot has no A^{-1}; its warp sums its subtree
// without elimination, by the same exterior products over all m rows starting
// from the determinants of the head's own columns (singular_head), 2^m sums
// spread over the lanes.
//
#include <algorithm>
#include <cmath>
#include <cstring>
#include <type_traits>

#include "radic_prefix.cuh"

namespace radic {
namespace {

constexpr int kBwdThreads = 128;
constexpr int kBwdMaxM = 8;

struct BwdArgs {
  const double* A;
  long long lda, stride;  // row stride, matrix stride (elements)
  int batch, m, n;
  int chunks;             // blocks per matrix
  int seg;                // columns per segment of the suffix sums (head kernel; even)
  unsigned long long total;
  double* slots;          // batch x chunks x m x n (chunks > 1)
  const double* grad_out;
  double* grad;           // written directly when chunks == 1
};

// Full partial-pivot LU with multipliers stored below the diagonal; idx[s] is
// the original row in slot s.  Returns det(M) and whether a pivot was zero.
template <int M>
__device__ __forceinline__ double lu_full(double (&a)[M][M], int (&idx)[M], bool& zero_pivot) {
  double det = 1.0;
  bool neg = false;
  zero_pivot = false;
#pragma unroll
  for (int i = 0; i < M; ++i) idx[i] = i;
#pragma unroll
  for (int k = 0; k < M; ++k) {
#pragma unroll
    for (int i = k + 1; i < M; ++i) {
      const bool sw = mag_key(a[i][k]) > mag_key(a[k][k]);
#pragma unroll
      for (int j = 0; j < M; ++j) {
        const double x = a[k][j], y = a[i][j];
        a[k][j] = sw ? y : x;
        a[i][j] = sw ? x : y;
      }
      const int ik = idx[k], ii = idx[i];
      idx[k] = sw ? ii : ik;
      idx[i] = sw ? ik : ii;
      neg ^= sw;
    }
    const double piv = a[k][k];
    zero_pivot |= (piv == 0.0);
    det *= piv;
    const double r = rcp_f64(piv);
#pragma unroll
    for (int i = k + 1; i < M; ++i) {
      const double l = a[i][k] * r;
      a[i][k] = l;
#pragma unroll
      for (int j = k + 1; j < M; ++j) a[i][j] = fma(-l, a[k][j], a[i][j]);
    }
  }
  return neg ? -det : det;
}

// X = U^{-1} L^{-1} from the packed factors in a (L unit lower, U upper):
// first X = L^{-1} column by column (forward substitution), then, in place,
// X = U^{-1} X (back substitution).
template <int M, typename T = double>
__device__ __forceinline__ void inverse_factors(const T (&a)[M][M], T (&X)[M][M]) {
#pragma unroll
  for (int j = 0; j < M; ++j) {
#pragma unroll
    for (int i = 0; i < M; ++i) {
      if (i < j) X[i][j] = T(0);
      else if (i == j) X[i][j] = T(1);
      else {
        T s = -a[i][j];
#pragma unroll
        for (int k = j + 1; k < i; ++k) s = fma(-a[i][k], X[k][j], s);
        X[i][j] = s;
      }
    }
  }
  T rinv[M];
#pragma unroll
  for (int i = 0; i < M; ++i) rinv[i] = rcp_t(a[i][i]);
#pragma unroll
  for (int j = 0; j < M; ++j) {
#pragma unroll
    for (int i = M - 1; i >= 0; --i) {
      T s = X[i][j];
#pragma unroll
      for (int k = i + 1; k < M; ++k) s = fma(-a[i][k], X[k][j], s);
      X[i][j] = s * rinv[i];
    }
  }
}

// Slow path for a singular minor: cofactor(i, j) = (-1)^(i+j) det of M
// without row i and column j, by LU of each (m-1) x (m-1) submatrix.
template <int M>
__device__ __noinline__ void cofactors_slow(const double* As, int cs, const int (&c)[M], double (&cof)[M][M]) {
  for (int i = 0; i < M; ++i) {
    for (int j = 0; j < M; ++j) {
      double sub[M > 1 ? M - 1 : 1][M > 1 ? M - 1 : 1];
      int rr = 0;
      for (int r = 0; r < M; ++r) {
        if (r == i) continue;
        int cc = 0;
        for (int q = 0; q < M; ++q) {
          if (q == j) continue;
          sub[rr][cc++] = As[c[q] * cs + r];
        }
        ++rr;
      }
      double det = 1.0;
      bool neg = false;
      const int S = M - 1;
      for (int k = 0; k < S; ++k) {
        int p = k;
        for (int r = k + 1; r < S; ++r)
          if (fabs(sub[r][k]) > fabs(sub[p][k])) p = r;
        if (p != k) {
          for (int q = 0; q < S; ++q) {
            const double t = sub[k][q];
            sub[k][q] = sub[p][q];
            sub[p][q] = t;
          }
          neg = !neg;
        }
        const double piv = sub[k][k];
        det *= piv;
        if (piv == 0.0) break;
        for (int r = k + 1; r < S; ++r) {
          const double l = sub[r][k] / piv;
          for (int q = k + 1; q < S; ++q) sub[r][q] -= l * sub[k][q];
        }
      }
      if (neg) det = -det;
      cof[i][j] = ((i + j) & 1) ? -det : det;
    }
  }
}

template <int M>
__global__ void __launch_bounds__(kBwdThreads) k_backward(BwdArgs a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  constexpr int CS = ColStride<double, M>::value;
  const int n = a.n;
  const int b = blockIdx.y;
  const int chunk = blockIdx.x;
  uint64_t* binom = reinterpret_cast<uint64_t*>(smem_raw);
  size_t off = ((size_t)(n + 1) * (M + 1) * 8 + 15) / 16 * 16;
  double* As = reinterpret_cast<double*>(smem_raw + off);
  off += ((size_t)n * CS * 8 + 15) / 16 * 16;
  double* G = reinterpret_cast<double*>(smem_raw + off);  // M x n gradient tile
  build_binom(binom, n, M);
  const double* Ab = a.A + (long long)b * a.stride;
  for (int idx = threadIdx.x; idx < n * CS; idx += blockDim.x) {
    const int j = idx / CS, i = idx - j * CS;
    As[idx] = (i < M) ? Ab[(long long)i * a.lda + j] : 0.0;
  }
  for (int idx = threadIdx.x; idx < M * n; idx += blockDim.x) G[idx] = 0.0;
  __syncthreads();

  // this block's run of ranks, split evenly over its threads
  const unsigned long long per_chunk = (a.total + a.chunks - 1) / a.chunks;
  const unsigned long long c0 = (unsigned long long)chunk * per_chunk;
  const unsigned long long c1 = min(c0 + per_chunk, a.total);
  if (c0 < c1) {
    const unsigned long long per_thread = (c1 - c0 + blockDim.x - 1) / blockDim.x;
    const unsigned long long q0 = c0 + threadIdx.x * per_thread;
    const unsigned long long q1 = min(q0 + per_thread, c1);
    if (q0 < q1) {
      int c[M];
      unrank<M>(q0, n, binom, M + 1, c);
      for (unsigned long long q = q0; q < q1; ++q) {
        double mm[M][M];
        gather<double, M, CS>(As, c, mm);
        int idx[M];
        bool zp;
        const double det = lu_full<M>(mm, idx, zp);
        const double sgn = sign_negative<M>(c) ? -1.0 : 1.0;
        if (!zp) {
          double B[M][M];
          inverse_factors<M>(mm, B);
          const double s = sgn * det;
#pragma unroll
          for (int sl = 0; sl < M; ++sl) {
            double* grow = G + idx[sl] * n;
#pragma unroll
            for (int j = 0; j < M; ++j) atomicAdd(grow + c[j], s * B[j][sl]);
          }
        } else {
          double cof[M][M];
          cofactors_slow<M>(As, CS, c, cof);
          for (int i = 0; i < M; ++i)
            for (int j = 0; j < M; ++j) atomicAdd(G + i * n + c[j], sgn * cof[i][j]);
        }
        if (q + 1 < q1) successor<M>(c, n);
      }
    }
  }
  __syncthreads();
  double* slot = a.slots + ((size_t)b * a.chunks + chunk) * (size_t)M * n;
  for (int idx = threadIdx.x; idx < M * n; idx += blockDim.x) slot[idx] = G[idx];
}

__device__ __forceinline__ bool pivot_greater(double x, double y) { return mag_key(x) > mag_key(y); }
__device__ __forceinline__ bool pivot_greater(ff x, ff y) { return fabsf(x.hi) > fabsf(y.hi); }
__device__ __forceinline__ bool is_zero(double x) { return x == 0.0; }
__device__ __forceinline__ bool is_zero(ff x) { return x.hi == 0.0f; }
__device__ __forceinline__ double to_double(double x) { return x; }
__device__ __forceinline__ double to_double(ff x) { return static_cast<double>(x); }

__device__ __forceinline__ double shfl_x(double x, int off) { return __shfl_xor_sync(kFull, x, off); }
__device__ __forceinline__ ff shfl_x(ff x, int off) {
  return ff(__shfl_xor_sync(kFull, x.hi, off), __shfl_xor_sync(kFull, x.lo, off));
}

// Adds the sum over the warp's 32 lanes of v[0..M-1] (one value per row of
// the matrix) to column `tcol` of the warp's gradient tile.  Three exchange
// steps on lane bits 4, 3 and 2 halve the vector each time (a
// reduce-scatter), so each group of four lanes ends with one row summed over
// eight lanes; two butterfly steps on bits 1 and 0 finish the sum, and the
// group's first lane adds it in: one lane per entry, so no atomics.  Nine
// additions and nine exchanges per lane.  Every lane of the warp must call it.
template <typename T, int M>
__device__ __forceinline__ void warp_add_column(const T (&v)[M], T* tcol, int n, int lane) {
  static_assert(M <= 8, "rows are spread over lane bits 4..2");
  T p[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) p[j] = T(0);
#pragma unroll
  for (int j = 0; j < M; ++j) p[j] = v[j];
  const bool b4 = (lane & 16) != 0, b3 = (lane & 8) != 0, b2 = (lane & 4) != 0;
  T w4[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const T keep = b4 ? p[j + 4] : p[j], send = b4 ? p[j] : p[j + 4];
    w4[j] = keep + shfl_x(send, 16);
  }
  T w2[2];
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    const T keep = b3 ? w4[j + 2] : w4[j], send = b3 ? w4[j] : w4[j + 2];
    w2[j] = keep + shfl_x(send, 8);
  }
  T w = (b2 ? w2[1] : w2[0]) + shfl_x(b2 ? w2[0] : w2[1], 4);
  w = w + shfl_x(w, 2);
  w = w + shfl_x(w, 1);
  const int row = (b4 ? 4 : 0) + (b3 ? 2 : 0) + (b2 ? 1 : 0);
  if ((lane & 3) == 0 && row < M) tcol[row * n] += w;
  __syncwarp();
}

// The same for two adjacent columns at once: lane bit 4 picks the column and
// bits 3..1 the row, so the five exchange steps serve both columns (at most
// fourteen additions per lane for m <= 8) and lanes with bit 0 clear add the
// sums.  `second` (the same on every lane) says whether column tcol + 1 exists.
template <typename T, int M>
__device__ __forceinline__ void warp_add_columns2(const T (&va)[M], const T (&vb)[M], T* tcol, int n, int lane,
                                                  bool second) {
  static_assert(M <= 8, "rows are spread over lane bits 3..1");
  const bool b4 = (lane & 16) != 0, b3 = (lane & 8) != 0, b2 = (lane & 4) != 0, b1 = (lane & 2) != 0;
  T w8[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) w8[j] = T(0);
#pragma unroll
  for (int j = 0; j < M; ++j) {
    const T keep = b4 ? vb[j] : va[j], send = b4 ? va[j] : vb[j];
    w8[j] = keep + shfl_x(send, 16);
  }
  T w4[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const T keep = b3 ? w8[j + 4] : w8[j], send = b3 ? w8[j] : w8[j + 4];
    w4[j] = keep + shfl_x(send, 8);
  }
  T w2[2];
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    const T keep = b2 ? w4[j + 2] : w4[j], send = b2 ? w4[j] : w4[j + 2];
    w2[j] = keep + shfl_x(send, 4);
  }
  T w = (b1 ? w2[1] : w2[0]) + shfl_x(b1 ? w2[0] : w2[1], 2);
  w = w + shfl_x(w, 1);
  const int row = (b3 ? 4 : 0) + (b2 ? 2 : 0) + (b1 ? 1 : 0);
  if ((lane & 1) == 0 && row < M && (!b4 || second)) tcol[(b4 ? 1 : 0) + row * n] += w;
  __syncwarp();
}

// Adds u[0..M-1] to rows 0..M-1 of column `key` of the warp's tile for the
// lanes with key >= 0.  Lanes with the same column take turns, in lane order,
// one round per lane of the largest such group, so no two lanes write one
// entry in the same round.  Every lane of the warp must call it.
template <typename T, int M>
__device__ __forceinline__ void warp_tile_add(T* tile, int n, int key, const T (&u)[M], int lane) {
  const unsigned grp = __match_any_sync(kFull, key);
  const unsigned rank = __popc(grp & ((1u << lane) - 1u));
  const unsigned rounds = __reduce_max_sync(kFull, key >= 0 ? (unsigned)__popc(grp) : 0u);
  for (unsigned it = 0; it < rounds; ++it) {
    if (key >= 0 && rank == it) {
#pragma unroll
      for (int i = 0; i < M; ++i) tile[i * n + key] += u[i];
    }
    __syncwarp();
  }
}

// u[rho] = x[r] for the slot r with idx[r] == rho: values in pivot order back
// to the matrix's row order (selects only, no indexed registers).
template <typename T, int M>
__device__ __forceinline__ void unpermute(const T (&x)[M], const int (&idx)[M], T (&u)[M]) {
#pragma unroll
  for (int rho = 0; rho < M; ++rho) {
    T s = T(0);
#pragma unroll
    for (int r = 0; r < M; ++r) s = (idx[r] == rho) ? x[r] : s;
    u[rho] = s;
  }
}

// Adds u[0..M-1] to column `key` of the warp's tile for the lanes with key >=
// 0: one warp sum per distinct column where they are few, turns otherwise (a
// warp sum takes about three times as long as a turn).
template <typename T, int M>
__device__ __forceinline__ void warp_add_head_column(T* tile, int n, int key, const T (&u)[M], int lane) {
  const unsigned grp = __match_any_sync(kFull, key);
  const unsigned first = __ballot_sync(kFull, key >= 0 && lane == __ffs(grp) - 1);
  const unsigned rounds = __reduce_max_sync(kFull, key >= 0 ? (unsigned)__popc(grp) : 0u);
  if (3u * __popc(first) > rounds) {
    warp_tile_add<T, M>(tile, n, key, u, lane);
    return;
  }
  for (unsigned todo = first; todo; todo &= todo - 1) {
    const int col = __shfl_sync(kFull, key, __ffs(todo) - 1);
    T w[M];
#pragma unroll
    for (int i = 0; i < M; ++i) w[i] = key == col ? u[i] : T(0);
    warp_add_column<T, M>(w, tile + col, n, lane);
  }
}

// ---------------------------------------------------------------------------
// Exterior sums over sets of G rows (see the head of this file), unrolled at
// compile time.  Entry S of an array belongs to the rows in the bit set S;
// entry 0 (the empty set, 1) is never stored.
// ---------------------------------------------------------------------------
__host__ __device__ constexpr int bits_of(unsigned x) { return x ? static_cast<int>(x & 1u) + bits_of(x >> 1) : 0; }
// Parity of the order (T, i, U): pairs out of order.
__host__ __device__ constexpr bool odd_order(unsigned T, int i, unsigned U) {
  int inv = bits_of(T >> (i + 1)) + bits_of(U & ((1u << i) - 1u));
  for (unsigned r = U; r; r &= r - 1) {
    int u = 0;
    while (!((r >> u) & 1u)) ++u;
    inv += bits_of(T >> (u + 1));
  }
  return inv & 1;
}

template <typename T>
__device__ __forceinline__ T signed_of(bool neg, T x) {
  return neg ? -x : x;
}

// P[S] += sum over i in S of +- z_i P[S without i], z appended as the last
// column, for the sets of at most MAXS rows from SET down to 1.
template <typename T, int G, int MAXS, int SET>
__device__ __forceinline__ void append_column(T (&P)[1 << G], const T (&z)[G]) {
  if constexpr (SET >= 1) {
    constexpr int size = bits_of(SET);
    if constexpr (size <= MAXS) {
#pragma unroll
      for (int i = 0; i < G; ++i) {
        if ((SET >> i) & 1) {
          const bool neg = (size - 1 - bits_of(SET & ((1 << i) - 1))) & 1;
          if constexpr (size == 1) P[SET] = P[SET] + z[i];
          else P[SET] = fma(signed_of(neg, z[i]), P[SET ^ (1 << i)], P[SET]);
        }
      }
    }
    append_column<T, G, MAXS, SET - 1>(P, z);
  }
}

// R <- (1 + z) ^ R: z becomes the first column of R's sequences.
template <typename T, int G, int MAXS, int SET>
__device__ __forceinline__ void first_column(T (&R)[1 << G], const T (&z)[G]) {
  if constexpr (SET >= 1) {
    constexpr int size = bits_of(SET);
    if constexpr (size <= MAXS) {
#pragma unroll
      for (int i = 0; i < G; ++i) {
        if ((SET >> i) & 1) {
          const bool neg = bits_of(SET & ((1 << i) - 1)) & 1;
          if constexpr (size == 1) R[SET] = R[SET] + signed_of(neg, z[i]);
          else R[SET] = fma(signed_of(neg, z[i]), R[SET ^ (1 << i)], R[SET]);
        }
      }
    }
    first_column<T, G, MAXS, SET - 1>(R, z);
  }
}

// g_I: sum over the sets SET not holding I of +- P[SET] R[the other rows].
template <typename T, int G, int I, int SET>
__device__ __forceinline__ void contract_row(const T (&P)[1 << G], const T (&R)[1 << G], T& g) {
  if constexpr (SET < (1 << G)) {
    if constexpr (!((SET >> I) & 1)) {
      constexpr int rest = ((1 << G) - 1) ^ SET ^ (1 << I);
      constexpr bool neg = odd_order(SET, I, rest);
      if constexpr (SET == 0) g = signed_of(neg, R[rest]);
      else if constexpr (rest == 0) g = g + signed_of(neg, P[SET]);
      else g = fma(signed_of(neg, P[SET]), R[rest], g);
    }
    contract_row<T, G, I, SET + 1>(P, R, g);
  }
}
template <typename T, int G, int I = 0>
__device__ __forceinline__ void contract(const T (&P)[1 << G], const T (&R)[1 << G], T (&g)[G]) {
  if constexpr (I < G) {
    contract_row<T, G, I, 0>(P, R, g[I]);
    contract<T, G, I + 1>(P, R, g);
  }
}

// Gradient of a head's subtree without elimination, by the whole warp, in
// binary64 from the matrix in global memory: the same sums over sets of all M
// rows, a prefix sum V that starts from the determinants of the head's columns
// instead of 1, and suffix sums R over the later columns, both taking columns
// in only.  R is built from the last column back for as many columns at a time
// as the working memory holds.  Serves heads with an exactly zero pivot.  work:
// `arrays` (at least 4) arrays of 2^M words of shared memory; G: the block's
// gradient tile (shared-memory atomics).
template <int M, int GD>
__device__ __noinline__ void singular_head(const double* Ab, long long lda, const int (&c)[M - GD], int n,
                                           double* work, int arrays, double* G, int lane) {
  constexpr int H = M - GD, NS = 1 << M;
  // to <- E + E ^ x, the column appended (front: E + x ^ E), for the sets of
  // lo..hi rows; the others are copied.  Column parity of Eq. (1) folded in.
  auto wedge = [&](const double* E, double* to, int col, int lo, int hi, bool front) {
    double x[M];
#pragma unroll
    for (int i = 0; i < M; ++i) {
      const double e = Ab[(long long)i * lda + col];
      x[i] = (col & 1) ? -e : e;
    }
    for (int S = lane; S < NS; S += 32) {
      const int size = __popc(S);
      double acc = E[S];
      if (size >= lo && size <= hi) {
#pragma unroll
        for (int i = 0; i < M; ++i) {
          if ((S >> i) & 1) {
            const int below = __popc(S & ((1 << i) - 1));
            const bool neg = ((front ? below : size - 1 - below) & 1) != 0;
            acc = fma(neg ? -x[i] : x[i], E[S ^ (1 << i)], acc);
          }
        }
      }
      to[S] = acc;
    }
    __syncwarp();
  };
  auto unit = [&](double* E) {
    for (int S = lane; S < NS; S += 32) E[S] = S == 0 ? 1.0 : 0.0;
    __syncwarp();
  };
  // R over the columns from `col` on, into `to` (spare: another array)
  auto suffix = [&](int col, double* to, double* spare) {
    double *from = ((n - col) & 1) ? spare : to, *into = ((n - col) & 1) ? to : spare;
    unit(from);
    for (int q = n - 1; q >= col; --q) {
      wedge(from, into, q, 1, GD, true);
      double* t = from;
      from = into;
      into = t;
    }
  };
  // sum over the sets T of `lo` rows or more, without row i, of +- V[T] R[rest],
  // for every row i, into column `col` of the tile.  The sign is that of (T, i,
  // rest): T before the other rows (its row numbers less 0, 1, ...), then i
  // before those of `rest` below it.
  auto scatter = [&](const double* V, const double* R, int lo, int hi, int col, bool neg) {
    double s[M];
#pragma unroll
    for (int i = 0; i < M; ++i) s[i] = 0.0;
    for (int T = lane; T < NS; T += 32) {
      const int size = __popc(T);
      if (size < lo || size > hi) continue;
      const double vt = V[T];
      const int moved = __popc(T & 0xaa) + size * (size - 1) / 2;
#pragma unroll
      for (int i = 0; i < M; ++i) {
        if (!((T >> i) & 1)) {
          const int rest = (NS - 1) ^ T ^ (1 << i);
          const bool odd = ((moved + __popc(rest & ((1 << i) - 1))) & 1) != 0;
          s[i] = fma(odd ? -vt : vt, R[rest], s[i]);
        }
      }
    }
#pragma unroll
    for (int i = 0; i < M; ++i) {
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) s[i] += __shfl_xor_sync(kFull, s[i], off);
      if (lane == 0) atomicAdd(G + i * n + col, neg ? -s[i] : s[i]);
    }
    __syncwarp();
  };
  const bool common = (M * (M + 1) / 2 + M) & 1;  // (-1)^(r+s) without the column parities
  double *V = work, *next = work + NS, *R = work + 2 * NS;
  auto append = [&](int col, int lo, int hi) {
    wedge(V, next, col, lo, hi, false);
    double* t = V;
    V = next;
    next = t;
  };
  // head column j: the determinants of the other head columns (sets of H-1
  // rows) against the sums over GD columns; column j moves past H-1-j columns
  suffix(c[H - 1] + 1, R, R + NS);
  for (int j = 0; j < H; ++j) {
    unit(V);
    int size = 0;
    for (int t = 0; t < H; ++t) {
      if (t == j) continue;
      ++size;
      append(c[t], 1, size);
    }
    scatter(V, R, H - 1, H - 1, c[j], common ^ ((c[j] & 1) != 0) ^ (((H - 1 - j) & 1) != 0));
  }
  // later columns: V starts from the head's own determinants
  unit(V);
  for (int t = 0; t < H; ++t) append(c[t], 1, t + 1);
  for (int a0 = c[H - 1] + 1; a0 < n; a0 += arrays - 2) {
    const int a1 = min(n, a0 + arrays - 2);
    suffix(a1, R + (a1 - 1 - a0) * NS, next);  // R after column a1-1, then after each one before
    for (int col = a1 - 1; col > a0; --col) wedge(R + (col - a0) * NS, R + (col - 1 - a0) * NS, col, 1, GD, true);
    for (int col = a0; col < a1; ++col) {
      scatter(V, R + (col - a0) * NS, H, M - 1, col, common ^ ((col & 1) != 0));
      append(col, H + 1, M - 1);
    }
  }
}

// Blocks per SM that the head kernel's registers allow (its launch bound).
__host__ __device__ constexpr int bwd_resident(int m) { return m == 3 ? 4 : m == 4 ? 3 : 2; }
// Words a lane stores per column of a segment: R without its full set, and z.
__host__ __device__ constexpr int bwd_store_words(int G) { return (1 << G) - 2 + G; }
// Fewest columns per segment: what fits bwd_resident blocks at n = 64.
__host__ __device__ constexpr int bwd_min_segment(int G) { return G == 4 ? 4 : G == 3 ? 6 : 10; }
// A warp's working memory: a segment's columns, or a singular head's arrays of
// 2^m words.
__host__ __device__ inline size_t bwd_work_bytes(int m, int G, int seg) {
  const size_t cols = (size_t)seg * bwd_store_words(G) * 32 * 8, sing = (size_t)4 * 8 << m;
  return cols > sing ? cols : sing;
}

// Shared-memory layout of the head kernel.
template <typename T>
struct BwdSmem {
  uint64_t* binom;
  T* As;
  double* tile0;    // tile of the singular heads
  T* tiles;         // one m x n tile per warp
  unsigned char* work;  // bwd_work_bytes per warp
  size_t bytes;
  __host__ __device__ BwdSmem(unsigned char* base, int n, int m, int G, int seg, int warps) {
    size_t off = 0;
    auto take = [&](size_t b) {
      const size_t o = off;
      off += (b + 15) / 16 * 16;
      return o;
    };
    binom = reinterpret_cast<uint64_t*>(base + take((size_t)(n + 1) * (m + 1) * 8));
    As = reinterpret_cast<T*>(base + take((size_t)n * ((m + 1) / 2 * 2) * 8));
    tile0 = reinterpret_cast<double*>(base + take((size_t)m * n * 8));
    tiles = reinterpret_cast<T*>(base + take((size_t)warps * m * n * 8));
    work = base + take((size_t)warps * bwd_work_bytes(m, G, seg));
    bytes = off;
  }
};

template <typename T, int M, int G>
__global__ void __launch_bounds__(kBwdThreads, bwd_resident(M)) k_backward_heads(BwdArgs a) {
  constexpr int H = M - G, FULL = (1 << G) - 1, kWords = bwd_store_words(G);
  constexpr int CS = ColStride<T, M>::value;
  static_assert(sizeof(T) == 8 && CS == (M + 1) / 2 * 2, "layout of BwdSmem");
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int n = a.n, bs = M + 1;
  const int b = blockIdx.y, chunk = blockIdx.x;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, wpb = blockDim.x >> 5;
  const BwdSmem<T> sm(smem_raw, n, M, G, a.seg, wpb);
  unsigned char* const work = sm.work + (size_t)warp * bwd_work_bytes(M, G, a.seg);
  build_binom(sm.binom, n, M);
  const double* Ab = a.A + (long long)b * a.stride;
  for (int idx = threadIdx.x; idx < n * CS; idx += blockDim.x) {
    const int i = idx / n, j = idx - i * n;  // rows of A are contiguous
    sm.As[j * CS + i] = (i < M) ? to_elem<T>(Ab[(long long)i * a.lda + j]) : T(0);
  }
  for (int idx = threadIdx.x; idx < M * n; idx += blockDim.x) sm.tile0[idx] = 0.0;
  for (int idx = threadIdx.x; idx < wpb * M * n; idx += blockDim.x) sm.tiles[idx] = T(0);
  __syncthreads();
  const T* As = sm.As;
  T* Gw = sm.tiles + (size_t)warp * M * n;

  // heads in colexicographic order: those with last column v are the ranks
  // C(v, H) .. C(v+1, H) - 1
  const unsigned long long heads = sm.binom[(n - G) * bs + H];
  const unsigned long long tasks = (heads + 31) / 32;
  for (unsigned long long t = (unsigned long long)chunk * wpb + warp; t < tasks;
       t += (unsigned long long)a.chunks * wpb) {
    const bool live = t * 32 + lane < heads;
    const unsigned long long r = live ? t * 32 + lane : heads - 1;
    int v = H - 1, hi = n - G;  // C(v, H) <= r < C(hi, H)
    while (hi - v > 1) {
      const int mid = (v + hi) / 2;
      if (sm.binom[mid * bs + H] <= r) v = mid;
      else hi = mid;
    }
    int c[H];
    c[H - 1] = v;
    if constexpr (H > 1) {
      int head[H - 1];
      unrank<H - 1>(r - sm.binom[v * bs + H], v, sm.binom, bs, head);
#pragma unroll
      for (int j = 0; j < H - 1; ++j) c[j] = head[j];
    }
    const int col0 = __shfl_sync(kFull, v, 0) + 1;  // the smallest v is lane 0's
    // factor the M x H head: partial pivoting, L \ U packed in fa
    T fa[M][H];
#pragma unroll
    for (int j = 0; j < H; ++j)
#pragma unroll
      for (int i = 0; i < M; ++i) fa[i][j] = As[c[j] * CS + i];
    int idx[M];
#pragma unroll
    for (int i = 0; i < M; ++i) idx[i] = i;
    bool neg = false, zp = false;
    T prod = T(1);
#pragma unroll
    for (int kk = 0; kk < H; ++kk) {
#pragma unroll
      for (int i = kk + 1; i < M; ++i) {
        const bool sw = pivot_greater(fa[i][kk], fa[kk][kk]);
#pragma unroll
        for (int j = 0; j < H; ++j) {
          const T x = fa[kk][j], y = fa[i][j];
          fa[kk][j] = sw ? y : x;
          fa[i][j] = sw ? x : y;
        }
        const int ik = idx[kk], ii = idx[i];
        idx[kk] = sw ? ii : ik;
        idx[i] = sw ? ik : ii;
        neg ^= sw;
      }
      const T piv = fa[kk][kk];
      zp |= is_zero(piv);
      prod *= piv;
      const T rr = rcp_t(piv);
#pragma unroll
      for (int i = kk + 1; i < M; ++i) {
        const T l = fa[i][kk] * rr;
        fa[i][kk] = l;
#pragma unroll
        for (int j = kk + 1; j < H; ++j) fa[i][j] = fma(-l, fa[kk][j], fa[i][j]);
      }
    }
    for (unsigned sing = __ballot_sync(kFull, live && zp); sing; sing &= sing - 1) {
      int cs[H];
#pragma unroll
      for (int j = 0; j < H; ++j) cs[j] = __shfl_sync(kFull, c[j], __ffs(sing) - 1);
      singular_head<M, G>(Ab, a.lda, cs, n, reinterpret_cast<double*>(work),
                          (int)(bwd_work_bytes(M, G, a.seg) / (8u << M)), sm.tile0, lane);
    }
    // below, a singular or repeated head runs with non-finite or unwanted
    // values that `use` replaces by zeros
    const bool use = live && !zp;
    // W = -L21 L11^{-1} (G x H) and Ainv = U11^{-1} L11^{-1} (H x H)
    T W[G][H], Ai[H][H];
#pragma unroll
    for (int d = 0; d < G; ++d) {
#pragma unroll
      for (int j = H - 1; j >= 0; --j) {
        T sum = -fa[H + d][j];
#pragma unroll
        for (int i = j + 1; i < H; ++i) sum = fma(-W[d][i], fa[i][j], sum);
        W[d][j] = sum;
      }
    }
    {
      T top[H][H];
#pragma unroll
      for (int i = 0; i < H; ++i)
#pragma unroll
        for (int j = 0; j < H; ++j) top[i][j] = fa[i][j];
      inverse_factors<H, T>(top, Ai);
    }
    int sp = M * (M + 1) / 2 + G;
#pragma unroll
    for (int j = 0; j < H; ++j) sp += c[j] + 1;
    const T alpha = ((sp & 1) != neg) ? -prod : prod;
    auto schur = [&](int col, T (&z)[G]) {
      prefix_column<T, M, G>(As + col * CS, W, idx, z);
      if (col & 1) {
#pragma unroll
        for (int d = 0; d < G; ++d) z[d] = -z[d];
      }
    };
    // Segments of the later columns, last to first (step < 0, then 0): R[FULL] =
    // L in the end.  Then first to last: each segment's R built again from its
    // kept start (the first one's are still there), then the gradients of its
    // columns (summed over the warp) and Q.
    T R[1 << G], P[1 << G], L = T(0);
#pragma unroll
    for (int S = 0; S <= FULL; ++S) R[S] = P[S] = T(0);
    T Q[H][G];
#pragma unroll
    for (int i = 0; i < H; ++i)
#pragma unroll
      for (int d = 0; d < G; ++d) Q[i][d] = T(0);
    // local memory, written and read once per segment
    T kept[(kMaxN + bwd_min_segment(G) - 1) / bwd_min_segment(G)][FULL - 1];
    T* store = reinterpret_cast<T*>(work) + lane;
    auto column = [&](int col, int at, T (&val)[M]) {  // at: place in its segment
#pragma unroll
      for (int i = 0; i < M; ++i) val[i] = T(0);
      if (col > v) {
        T z[G], g[G];
#pragma unroll
        for (int S = 1; S < FULL; ++S) R[S] = store[(at * kWords + S - 1) * 32];
#pragma unroll
        for (int d = 0; d < G; ++d) z[d] = store[(at * kWords + FULL - 1 + d) * 32];
        contract<T, G>(P, R, g);
        append_column<T, G, G - 1, FULL>(P, z);
        const T* xc = As + col * CS;
#pragma unroll
        for (int i = 0; i < H; ++i) {
          const T xt = (col & 1) ? -xc[idx[i]] : xc[idx[i]];
#pragma unroll
          for (int d = 0; d < G; ++d) Q[i][d] = fma(xt, g[d], Q[i][d]);
        }
        const T sc = (col & 1) ? -alpha : alpha;
        T w[M];
#pragma unroll
        for (int d = 0; d < G; ++d) {
          g[d] = use ? sc * g[d] : T(0);
          w[H + d] = g[d];
        }
#pragma unroll
        for (int i = 0; i < H; ++i) {
          T s = use ? W[0][i] * g[0] : T(0);
#pragma unroll
          for (int d = 1; d < G; ++d) s = use ? fma(W[d][i], g[d], s) : T(0);
          w[i] = s;
        }
        unpermute<T, M>(w, idx, val);
      }
    };
    const int last = (n - 1 - col0) / a.seg;
#pragma unroll 1
    for (int step = -last; step <= last; ++step) {
      const int sg = step < 0 ? -step : step, a0 = col0 + sg * a.seg, a1 = min(n, a0 + a.seg);
      if (step <= 0) {
#pragma unroll
        for (int S = 1; S < FULL; ++S) kept[sg][S - 1] = R[S];
      } else {
#pragma unroll
        for (int S = 1; S < FULL; ++S) R[S] = kept[sg][S - 1];
      }
#pragma unroll 1
      for (int col = a1 - 1; col >= a0; --col) {
        if (col <= v) continue;
        T z[G];
        schur(col, z);
        if (step >= 0) {
          T* at = store + (col - a0) * kWords * 32;
#pragma unroll
          for (int S = 1; S < FULL; ++S) at[(S - 1) * 32] = R[S];
#pragma unroll
          for (int d = 0; d < G; ++d) at[(FULL - 1 + d) * 32] = z[d];
          if (step > 0 && col == a0) break;  // R before the segment was kept on the way back
        }
        first_column<T, G, G, FULL>(R, z);
      }
      if (step < 0) continue;
      if (step == 0) L = R[FULL];
      if constexpr (std::is_same<T, ff>::value) {
        // pairs: one column per warp sum (the column body is long; inlining it
        // twice measured slower, with instruction-fetch stalls)
        for (int col = a0; col < a1; ++col) {
          T va[M];
          column(col, col - a0, va);
          warp_add_column<T, M>(va, Gw + col, n, lane);
        }
      } else {
        for (int col = a0; col < a1; col += 2) {  // binary64: two columns per warp sum
          const bool two = col + 1 < a1;
          T va[M], vb[M];
          column(col, col - a0, va);
          if (two) {
            column(col + 1, col + 1 - a0, vb);
          } else {
#pragma unroll
            for (int i = 0; i < M; ++i) vb[i] = T(0);
          }
          warp_add_columns2<T, M>(va, vb, Gw + col, n, lane, two);
        }
      }
    }
    // head columns: alpha [L Ainv - Ainv Q W | -Ainv Q]^T, in pivot order row
    // r of column c[tt]: alpha (L Ainv[tt][r] - (Ainv Q)[tt] . W[.][r]), and
    // -alpha (Ainv Q)[tt][d] for the rows H + d
#pragma unroll
    for (int tt = 0; tt < H; ++tt) {
      T q[G];
#pragma unroll
      for (int d = 0; d < G; ++d) {
        q[d] = Ai[tt][0] * Q[0][d];
#pragma unroll
        for (int u = 1; u < H; ++u) q[d] = fma(Ai[tt][u], Q[u][d], q[d]);
      }
      T w[M], u[M];
#pragma unroll
      for (int r2 = 0; r2 < H; ++r2) {
        T s = L * Ai[tt][r2];
#pragma unroll
        for (int d = 0; d < G; ++d) s = fma(-q[d], W[d][r2], s);
        w[r2] = use ? alpha * s : T(0);
      }
#pragma unroll
      for (int d = 0; d < G; ++d) w[H + d] = use ? -(alpha * q[d]) : T(0);
      unpermute<T, M>(w, idx, u);
      warp_add_head_column<T, M>(Gw, n, use ? c[tt] : -1, u, lane);
    }
  }
  __syncthreads();
  // the block's tile: the singular heads' entries plus the warps' tiles in
  // warp order
  for (int idx = threadIdx.x; idx < M * n; idx += blockDim.x) {
    double sum = sm.tile0[idx];
    for (int w = 0; w < wpb; ++w) sum += to_double(sm.tiles[(size_t)w * M * n + idx]);
    if (a.chunks == 1) {
      const int i = idx / n, j = idx - i * n;
      a.grad[(long long)b * a.stride + (long long)i * a.lda + j] = sum * a.grad_out[b];
    } else {
      a.slots[((size_t)b * a.chunks + chunk) * (size_t)M * n + idx] = sum;
    }
  }
}

// grad_A[b] = grad_out[b] * sum over chunks (in order) of the tiles.
__global__ void k_backward_reduce(const double* slots, int batch, int m, int n, int chunks, const double* grad_out,
                                  double* grad, long long lda, long long stride) {
  const long long total = (long long)batch * m * n;
  for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < total;
       t += (long long)gridDim.x * blockDim.x) {
    const int b = (int)(t / (m * n));
    const int e = (int)(t - (long long)b * m * n);
    const int i = e / n, j = e - i * n;
    double s = 0.0;
    for (int k = 0; k < chunks; ++k) s += slots[((size_t)b * chunks + k) * (size_t)m * n + e];
    grad[(long long)b * stride + (long long)i * lda + j] = s * grad_out[b];
  }
}

const void* bwd_kernel(int m) {
  return m == 1   ? reinterpret_cast<const void*>(&k_backward<1>)
         : m == 2 ? reinterpret_cast<const void*>(&k_backward<2>)
                  : nullptr;
}

// Head kernel of m rows and subtrees of G columns (G = 2 up to m = 4, 3 and 4
// from m = 4 and 5 on).
template <typename T, int M>
const void* bwd_heads_kernel_m(int G) {
  if constexpr (M <= 4)
    if (G == 2) return reinterpret_cast<const void*>(&k_backward_heads<T, M, 2>);
  if constexpr (M >= 4)
    if (G == 3) return reinterpret_cast<const void*>(&k_backward_heads<T, M, 3>);
  if constexpr (M >= 5)
    if (G == 4) return reinterpret_cast<const void*>(&k_backward_heads<T, M, 4>);
  return nullptr;
}

template <typename T>
const void* bwd_heads_kernel(int m, int G) {
  switch (m) {
    case 3: return bwd_heads_kernel_m<T, 3>(G);
    case 4: return bwd_heads_kernel_m<T, 4>(G);
    case 5: return bwd_heads_kernel_m<T, 5>(G);
    case 6: return bwd_heads_kernel_m<T, 6>(G);
    case 7: return bwd_heads_kernel_m<T, 7>(G);
    case 8: return bwd_heads_kernel_m<T, 8>(G);
    default: return nullptr;
  }
}

struct BwdPlan {
  int G = 0, chunks = 1;
};

// Subtree depth and blocks per matrix of the head kernel.  Estimate for every
// available G, in binary64 warp instructions: a head's elimination, inverse and
// prefix columns, per later column the three exterior products, the
// contraction, Q and the m gradient entries with their warp sum.  An SM takes
// one such instruction in 16 cycles from all its warps together, one warp of
// its own every 64: the work spread over the SMs plus the longest task alone.
// A block's four warps share a matrix; a matrix is split over several blocks
// only as far as its tasks go, and until the batch gives every SM a few.
BwdPlan bwd_plan(int batch, int m, int n, int sms) {
  BwdPlan best;
  double best_time = 0.0;
  if (sms < 1) sms = 1;
  for (int G = m <= 4 ? 2 : 3; G <= 4 && G < m; ++G) {
    const int H = m - G;
    const double ext = G * (double)(1 << (G - 1)) - G;
    const double head = m * (double)H * H + 2.0 * H * H * H + H * (G * (double)H + (double)G * H + 3.0 * m) + 40.0;
    const double col = 3.0 * G * H + 3.0 * ext + G * (double)(1 << (G - 1)) + 2.0 * G * H + G + 10.0;
    double cols = 0.0, heads = 0.0;
    for (int v = H - 1; v <= n - 1 - G; ++v) {
      const double cnt = (double)binom_host(v, H - 1);
      heads += cnt;
      cols += cnt * (n - 1 - v);
    }
    const double tasks = std::ceil(heads / 32.0);
    const double work = (double)batch * (tasks * head + std::max(cols / 32.0, cols / heads * tasks) * col);
    const double longest = head + (n - H) * col;
    const double time = 16.0 * work / sms + 64.0 * longest;
    if (best.G == 0 || time < best_time) {
      best.G = G;
      best_time = time;
      const long long by_work = ((long long)tasks + kBwdThreads / 32 - 1) / (kBwdThreads / 32);
      const long long want = ((long long)sms * 8 + batch - 1) / batch;
      best.chunks = (int)std::max(1ll, std::min(std::min(by_work, want), 65535ll));
    }
  }
  return best;
}

// Columns per segment of the suffix sums: as many as the shared memory of the
// blocks that run together on an SM allows, because a segment's columns are
// computed twice, but for the first's.  (5000 matrices of 3 x 30, 16 columns and
// three blocks per SM 507 us, 12 and four 449; 64 of them, one block per SM, 12
// columns 51 us, 24 45.)
int bwd_segment(long long blocks, int m, int n, int G, int sms) {
  const int resident = (int)std::max(1ll, std::min<long long>((blocks + sms - 1) / sms, bwd_resident(m)));
  const size_t room = std::min<size_t>(228 * 1024 / resident - 1024, 227 * 1024);
  const size_t warps = kBwdThreads / 32, col = warps * bwd_store_words(G) * 32 * 8;
  const size_t fixed = BwdSmem<double>(nullptr, n, m, G, 0, (int)warps).bytes - warps * bwd_work_bytes(m, G, 0);
  const int fit = (int)((room - fixed) / col) & ~1, all = (n - (m - G) + 1) & ~1;
  return std::max(bwd_min_segment(G), std::min(fit, all));
}

int bwd_chunks(int batch, unsigned long long total) {
  const int sms = device_sm_count();
  const long long want = (long long)(sms > 0 ? sms : 1) * 16;  // about 16 blocks per SM in all
  long long ch = (want + batch - 1) / batch;
  const long long by_work = (long long)((total + 4095) / 4096);  // at least ~32 minors per thread
  if (ch > by_work) ch = by_work;
  if (ch < 1) ch = 1;
  if (ch > 65535) ch = 65535;
  return (int)ch;
}

size_t bwd_smem(int m, int n) {
  const int cs = ((m + 1) / 2) * 2;
  size_t off = ((size_t)(n + 1) * (m + 1) * 8 + 15) / 16 * 16;
  off += ((size_t)n * cs * 8 + 15) / 16 * 16;
  off += (size_t)m * n * 8;
  return off;
}

}  // namespace
}  // namespace radic

using namespace radic;

extern "C" {

size_t radic_backward_workspace_bytes(int batch, int m, int n) {
  if (batch < 1 || m < 1 || m > kBwdMaxM || n < 1 || n > kMaxN) return 0;
  const unsigned long long total = (m <= n) ? binom_host(n, m) : 0ull;
  int chunks = bwd_chunks(batch, total);
  if (m >= 3 && m <= n) chunks = bwd_plan(batch, m, n, device_sm_count()).chunks;
  return align_up((size_t)batch * chunks * m * n * sizeof(double), 256) + 256;
}

int radic_det_backward(const double* A, int batch, int m, int n, int64_t lda, int64_t stride, const double* grad_out,
                       double* grad_A, void* workspace, size_t workspace_bytes, void* stream) {
  return radic_det_backward_mode(A, batch, m, n, lda, stride, grad_out, grad_A, workspace, workspace_bytes,
                                 RADIC_MODE_FP64, stream);
}

int radic_det_backward_mode(const double* A, int batch, int m, int n, int64_t lda, int64_t stride,
                            const double* grad_out, double* grad_A, void* workspace, size_t workspace_bytes, int mode,
                            void* stream) {
  if (!A || !grad_out || !grad_A || batch < 1 || m < 1 || n < 1 || n > kMaxN || lda < n || stride < (int64_t)m * lda)
    return RADIC_EINVAL;
  if (mode != RADIC_MODE_FP64 && mode != RADIC_MODE_PAIR) return RADIC_EINVAL;
  if (m > kBwdMaxM) return RADIC_EUNSUPPORTED;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if (m > n) {  // det_R is identically zero: zero gradient
    for (int b = 0; b < batch; ++b)
      if (cudaMemset2DAsync(grad_A + (long long)b * stride, lda * sizeof(double), 0, n * sizeof(double), m, s) !=
          cudaSuccess)
        return RADIC_ECUDA;
    return RADIC_OK;
  }
  const size_t need = radic_backward_workspace_bytes(batch, m, n);
  if (!workspace || (reinterpret_cast<uintptr_t>(workspace) & 255u) || workspace_bytes < need) return RADIC_EWORKSPACE;
  BwdArgs a;
  a.A = A;
  a.lda = lda;
  a.stride = stride;
  a.batch = batch;
  a.m = m;
  a.n = n;
  a.total = binom_host(n, m);
  a.seg = 0;
  a.chunks = bwd_chunks(batch, a.total);
  a.slots = static_cast<double*>(workspace);
  a.grad_out = grad_out;
  a.grad = grad_A;
  const void* k;
  size_t smem;
  if (m >= 3) {  // shared per head
    const int sms = std::max(1, device_sm_count());
    const BwdPlan p = bwd_plan(batch, m, n, sms);
    a.chunks = p.chunks;
    a.seg = bwd_segment((long long)batch * p.chunks, m, n, p.G, sms);
    k = (mode == RADIC_MODE_PAIR) ? bwd_heads_kernel<ff>(m, p.G) : bwd_heads_kernel<double>(m, p.G);
    smem = BwdSmem<double>(nullptr, n, m, p.G, a.seg, kBwdThreads / 32).bytes;
  } else {
    k = bwd_kernel(m);
    smem = bwd_smem(m, n);
  }
  if (!k || !allow_smem(k, smem)) return RADIC_EUNSUPPORTED;
  void* params[] = {&a};
  if (cudaLaunchKernel(k, dim3(a.chunks, batch), dim3(kBwdThreads), params, smem, s) != cudaSuccess)
    return RADIC_ECUDA;
  if (m >= 3 && a.chunks == 1) return RADIC_OK;  // written by the kernel itself
  const long long total = (long long)batch * m * n;
  const unsigned blocks = (unsigned)std::min<long long>((total + 255) / 256, 65535);
  const double* slots = a.slots;
  int bb = batch, mm = m, nn = n, ch = a.chunks;
  long long l = lda, st = stride;
  void* rparams[] = {&slots, &bb, &mm, &nn, &ch, &grad_out, &grad_A, &l, &st};
  if (cudaLaunchKernel(reinterpret_cast<const void*>(&k_backward_reduce), dim3(blocks), dim3(256), rparams, 0, s) !=
      cudaSuccess)
    return RADIC_ECUDA;
  return RADIC_OK;
}

}  // extern "C"
