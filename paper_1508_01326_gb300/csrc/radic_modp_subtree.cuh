// Exact determinant, prefix mapping: sums of whole subtrees modulo a prime.
//
// A head is an ascending sequence of the first H = m-G columns; the minors
// that begin with it are its subtree, one for every G later columns.  One lane
// takes one head (unranked from its number, Section 4), eliminates it, and
// adds up its subtree without forming the minors one by one: with z(x) the
// G-entry Schur complement of a later column x, a minor is
//   det = +- prod(pivots) det[z(x_1) ... z(x_G)],
// and since a determinant is linear in its last column, the sums
//   E[S] = sum over x_1 < ... < x_k of det of the rows S of [z(x_1) ... z(x_k)],
// one for every set S of k of the G rows, follow from one another: taking the
// columns in order,
//   E[S] += sum over i in S of (-1)^(k-1-pos_S(i)) z_i E[S without i].
// A column costs G 2^(G-1) multiply-adds however many minors it closes, so a
// head with k later columns costs O(k) instead of its C(k, G) leaves.  The
// exact result needs only the signed sum (the floating modes also report the
// sum of magnitudes, which is not linear and needs every leaf).
//
// What bounds it: the integer multiply-add pipe (half rate: a 32x32->64
// multiply-add every two cycles per scheduler) and about as many ALU
// operations for the modular corrections.  Deeper subtrees divide the number
// of heads by (n-G)/(m-G) per step and double the cost of a column, and their
// E[] (2^G - 1 words) must stay in registers: G <= 6.  The host chooses G by
// that trade and by the longest lane (plan_subtree).
//
// Each grid row works one prime, so one launch serves every prime of the
// result; a block stages T A modulo its own prime only.  Column parities of
// Eq. (1) are folded into the staged copy.  Lanes of a warp hold heads with
// the same last column, so all lanes take the same later columns and read
// them from shared memory as broadcasts.
//
// Measured (GB300, one call, against one leaf product per minor): 12 x 40
// int8 (three primes) 2.63 ms against 233 ms, integer multiply pipe 52% and
// ALU 41% busy at 11 warps per SM; 10 x 24 int8 27 against 297 us; 8 x 32
// binary64 (15 primes, with the reconstruction) 39.5 us against 2.04 ms, the
// longest head alone 23 us of it; 3 x 12 12.4 against 30.6 us.
#pragma once

#include "radic_modp.cuh"

namespace radic {

namespace {

__host__ __device__ constexpr int popc_c(unsigned x) { return x ? static_cast<int>(x & 1u) + popc_c(x >> 1) : 0; }

// a[0] b[0] + ... accumulated without reduction: terms are below 2^62, so two
// may follow a value below 2^63; a value that reached 2^63 drops 2 p^2 (p^2
// just below 2^62) first.
struct LazySum {
  uint64_t acc = 0;
  template <int I>
  __device__ __forceinline__ void add(uint32_t a, uint32_t b, const Mont& mp) {
    if constexpr (I >= 4 && I % 2 == 0) acc -= (acc >> 63) ? 2 * mp.p2 : 0ull;
    acc += static_cast<uint64_t>(a) * b;
  }
  // Montgomery reduction of a sum of N terms, in [0, p).  The high word of
  // the sum is below p for one or two terms and below 2p for more (after the
  // fold above: 2^63 + 2 (p-1)^2 < 2p 2^32); subtracting the high word of
  // q p, q = sum / p modulo 2^32, leaves a value in (-p, p).
  template <int N>
  __device__ __forceinline__ uint32_t reduce(const Mont& mp) const {
    uint32_t h = static_cast<uint32_t>(acc >> 32);
    if constexpr (N > 2) h = min(h, h - mp.p);
    const uint32_t q = static_cast<uint32_t>(acc) * (0u - mp.pinv);
    const uint32_t d = h - __umulhi(q, mp.p);
    return min(d, d + mp.p);
  }
};

// One column into the subtree sums: E[S] for the sets S from SET down to 1
// (E[S without i] still holds the columns before this one).
template <int G, int SET, int I, int K>
__device__ __forceinline__ void set_terms(const uint32_t (&E)[1 << G], const uint32_t (&z)[G], const uint32_t (&nz)[G],
                                          const Mont& mp, LazySum& s) {
  if constexpr (I < G) {
    if constexpr ((SET >> I) & 1) {
      constexpr int size = popc_c(SET), pos = popc_c(SET & ((1 << I) - 1));
      s.template add<K>((size - 1 - pos) & 1 ? nz[I] : z[I], E[SET ^ (1 << I)], mp);
      set_terms<G, SET, I + 1, K + 1>(E, z, nz, mp, s);
    } else {
      set_terms<G, SET, I + 1, K>(E, z, nz, mp, s);
    }
  }
}
template <int G, int SET>
__device__ __forceinline__ void subtree_column(uint32_t (&E)[1 << G], const uint32_t (&z)[G], const uint32_t (&nz)[G],
                                               const Mont& mp) {
  if constexpr (SET >= 1) {
    constexpr int size = popc_c(SET);
    if constexpr (size == 1) {
      constexpr int i = popc_c(SET - 1);
      E[SET] = add_mod(E[SET], z[i], mp.p);
    } else {
      LazySum s;
      set_terms<G, SET, 0, 0>(E, z, nz, mp, s);
      E[SET] = add_mod(E[SET], s.reduce<size>(mp), mp.p);
    }
    subtree_column<G, SET - 1>(E, z, nz, mp);
  }
}

// Subtree sum of a column range from those of its two halves: E[all rows] =
// sum over S of +- E_first[S] E_second[rest], the sign that of moving the rows
// of S before the others (one per pair a in S, b not in S, a > b).
// The second half's sums come from the lane next door, one at a time.
template <int G, int SET>
__device__ __forceinline__ void join_terms(const uint32_t (&E)[1 << G], const Mont& mp, LazySum& s) {
  if constexpr (SET < (1 << G)) {
    constexpr int rest = ((1 << G) - 1) ^ SET;
    int inv = 0;
#pragma unroll
    for (int b = 0; b < G; ++b)
      if ((rest >> b) & 1) inv += popc_c(SET >> (b + 1));
    const uint32_t f = __shfl_xor_sync(kFull, E[rest], 1);
    s.template add<SET>((inv & 1) ? mp.p - E[SET] : E[SET], f, mp);
    join_terms<G, SET + 1>(E, mp, s);
  }
}

// c x + sum_t W[t] v[t] over N coefficients, in [0, p).
template <int N, int T = 0>
__device__ __forceinline__ void dot_terms(const uint32_t* W, const uint32_t* v, const Mont& mp, LazySum& s) {
  if constexpr (T < N) {
    s.template add<T + 1>(W[T], v[T], mp);
    dot_terms<N, T + 1>(W, v, mp, s);
  }
}
template <int N>
__device__ __forceinline__ uint32_t affine_dot(uint32_t c, uint32_t x, const uint32_t* W, const uint32_t* v,
                                               const Mont& mp) {
  LazySum s;
  s.template add<0>(c, x, mp);
  dot_terms<N>(W, v, mp, s);
  return s.reduce<N + 1>(mp);
}

template <int M>
__device__ __forceinline__ void load_column(const uint32_t* __restrict__ col, uint32_t (&x)[M]) {
#pragma unroll
  for (int i = 0; i < M; i += 4) {
    const uint4 v = *reinterpret_cast<const uint4*>(col + i);
    x[i] = v.x;
    if (i + 1 < M) x[i + 1] = v.y;
    if (i + 2 < M) x[i + 2] = v.z;
    if (i + 3 < M) x[i + 3] = v.w;
  }
}

// Elimination of the head c[0..J] one column at a time, without division:
// after J columns, c_J z(x)_i = cs x_i + sum_t W[i][t] x_t for the rows i >= J
// left.  Column c_J gives s_i = c_J z_i; its pivot is row J, and
//   W[i][t] <- s_J W[i][t] - s_i W[J][t],  W[i][J] = -s_i cs,  cs <- s_J cs.
// With c_{j+1} = s_j c_j the pivots' product is c_H / (c_1 ... c_{H-1}); q
// collects c_1 ... c_{H-1}.  A zero pivot (one residue in 2^31) leaves cs = 0.
template <int M, int G, int J>
__device__ __forceinline__ void head_step(const uint32_t* __restrict__ As, const int* c, uint32_t (&W)[M][M - G],
                                          uint32_t& cs, uint32_t& q, const Mont& mp) {
  constexpr int H = M - G, CS = ((M + 3) / 4) * 4;
  if constexpr (J < H) {
    uint32_t x[M];
    load_column<M>(As + c[J] * CS, x);
    uint32_t s[M];
#pragma unroll
    for (int i = J; i < M; ++i) s[i] = J == 0 ? x[i] : affine_dot<J>(cs, x[i], W[i], x, mp);
#pragma unroll
    for (int i = J + 1; i < M; ++i) {
      if constexpr (J > 0) {
#pragma unroll
        for (int t = 0; t < J; ++t) W[i][t] = ff_update(s[J], W[i][t], s[i], W[J][t], mp);
        W[i][J] = neg_mod(mmul(s[i], cs, mp), mp.p);
      } else {
        W[i][0] = neg_mod(s[i], mp.p);
      }
    }
    if constexpr (J > 0) {
      q = mmul(q, cs, mp);
      cs = mmul(s[J], cs, mp);
    } else {
      cs = s[0];
    }
    head_step<M, G, J + 1>(As, c, W, cs, q, mp);
  }
}

// The same sum with row exchanges, for a head whose leading pivots met a
// zero: num / den, num = 0 when the head is singular modulo p.
template <int M, int G>
__device__ __noinline__ void subtree_pivoting(const uint32_t* __restrict__ As, const int (&c)[M - G], int v, int n,
                                              Mont mp, uint32_t& num, uint32_t& den) {
  constexpr int H = M - G, CS = ((M + 3) / 4) * 4;
  uint32_t W[M][H], s[M];
  int idx[M];
  for (int i = 0; i < M; ++i) idx[i] = i;
  uint32_t cs = mp.one, q = mp.one;
  bool neg = false;
  num = 0u;
  den = mp.one;
  for (int J = 0; J < H; ++J) {
    const uint32_t* x = As + c[J] * CS;
    for (int i = J; i < M; ++i) {
      uint32_t t = mmul(cs, x[idx[i]], mp);
      for (int k = 0; k < J; ++k) t = add_mod(t, mmul(W[i][k], x[idx[k]], mp), mp.p);
      s[i] = t;
    }
    int r = J;
    while (r < M && s[r] == 0u) ++r;
    if (r == M) return;
    if (r != J) {
      for (int k = 0; k < J; ++k) {
        const uint32_t t = W[J][k];
        W[J][k] = W[r][k];
        W[r][k] = t;
      }
      const int ti = idx[J];
      idx[J] = idx[r];
      idx[r] = ti;
      const uint32_t t = s[J];
      s[J] = s[r];
      s[r] = t;
      neg = !neg;
    }
    for (int i = J + 1; i < M; ++i) {
      for (int k = 0; k < J; ++k) W[i][k] = ff_update(s[J], W[i][k], s[i], W[J][k], mp);
      W[i][J] = neg_mod(mmul(s[i], cs, mp), mp.p);
    }
    if (J > 0) q = mmul(q, cs, mp);
    cs = mmul(s[J], cs, mp);
  }
  uint32_t E[1 << G];
  for (int S = 0; S < (1 << G); ++S) E[S] = 0u;
  E[0] = mp.one;
  for (int col = v + 1; col < n; ++col) {
    const uint32_t* x = As + col * CS;
    uint32_t z[G];
    for (int d = 0; d < G; ++d) {
      uint32_t t = mmul(cs, x[idx[H + d]], mp);
      for (int k = 0; k < H; ++k) t = add_mod(t, mmul(W[H + d][k], x[idx[k]], mp), mp.p);
      z[d] = t;
    }
    for (int S = (1 << G) - 1; S >= 1; --S) {
      int rest = __popc(S) - 1;  // rows of S after row i
      for (int i = 0; i < G; ++i) {
        if (!((S >> i) & 1)) continue;
        const uint32_t t = mmul(z[i], E[S ^ (1 << i)], mp);
        E[S] = add_mod(E[S], (rest & 1) ? neg_mod(t, mp.p) : t, mp.p);
        --rest;
      }
    }
  }
  num = neg ? neg_mod(E[(1 << G) - 1], mp.p) : E[(1 << G) - 1];
  den = q;
  for (int d = 1; d < G; ++d) den = mmul(den, cs, mp);
}

// Shared-memory layout: binom | n x CS residues | 2 x (m x n) scratch rows |
// m x m triangular factors | row statistics | last-block flag | block sum.
struct SubtreeSmem {
  uint64_t* binom;
  uint32_t* As;
  uint32_t* rows;
  uint32_t* tri;
  RowStats* stats;
  int* last;
  unsigned long long* sum;  // the block's residue sum
  size_t bytes;
  __host__ __device__ SubtreeSmem(unsigned char* base, int n, int m) {
    size_t off = 0;
    auto take = [&](size_t b) {
      const size_t o = off;
      off += (b + 15) / 16 * 16;
      return o;
    };
    binom = reinterpret_cast<uint64_t*>(base + take((size_t)(n + 1) * (m + 1) * 8));
    As = reinterpret_cast<uint32_t*>(base + take((size_t)n * ((m + 3) / 4 * 4) * 4));
    rows = reinterpret_cast<uint32_t*>(base + take(2 * (size_t)m * n * 4));
    tri = reinterpret_cast<uint32_t*>(base + take((size_t)m * m * 4));
    stats = reinterpret_cast<RowStats*>(base + take(sizeof(RowStats)));
    last = reinterpret_cast<int*>(base + take(16));
    sum = reinterpret_cast<unsigned long long*>(base + take(16));
    bytes = off;
  }
};

template <int M, int G>
__global__ void __launch_bounds__(kMaxThreadsModp, G == 6 ? 3 : 4) k_modp_subtree(SingleArgs a, PrefixTable tab) {
  constexpr int H = M - G, CS = ((M + 3) / 4) * 4;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int n = a.n, bs = M + 1;
  const SubtreeSmem sm(smem_raw, n, M);
  const int kp = blockIdx.y;
  if (threadIdx.x == 0) *sm.sum = 0ull;
  build_binom(sm.binom, n, M);
  KeptEntries keep;
  row_stats(a, M, *sm.stats, keep);
  count_primes(a, M, static_cast<double>(sm.binom[n * bs + M]), *sm.stats);
  const int needed = sm.stats->needed, K = min(needed, (int)gridDim.y);
  if (kp >= K) return;  // a prime the bound does not need
  const Mont mp = make_mont(kp);
  stage_prime(a, M, CS, kp, mp, *sm.stats, keep, sm.tri, sm.rows, sm.As, true);

  const int lane = threadIdx.x & 31;
  const unsigned long long wpb = blockDim.x / 32;
  const unsigned long long nwarps = gridDim.x * wpb;
  uint32_t N = 0u, Dn = mp.one;  // the lane's sum as one fraction
  // tasks are numbered heaviest group (most later columns) first
  int v = tab.v_lo;
  for (unsigned long long t = blockIdx.x * wpb + (threadIdx.x >> 5); t < tab.total_tasks; t += nwarps) {
    while (v < tab.v_hi && t >= tab.task_start[v + 1]) ++v;
    const unsigned long long runlen = tab.run[v], cnt = tab.count[v];
    // two lanes share a head in the longest groups, each taking half of its
    // later columns
    const int lp = tab.lanes[v], sub = lane & (lp - 1);
    const int half = (n - 1 - v + lp - 1) / lp, col0 = v + 1 + sub * half, col1 = min(col0 + half, n);
    const unsigned long long groups = 32 / lp;
    const unsigned long long r0 =
        (t - tab.task_start[v]) * groups * runlen + (unsigned long long)(lane / lp) * runlen;
    const unsigned long long r1 = min(r0 + runlen, cnt);
    int c[H];
    constexpr int HH = H > 1 ? H - 1 : 1;
    int head[HH];
    if constexpr (H > 1) unrank<H - 1>(r0 < cnt ? r0 : 0ull, v, sm.binom, bs, head);
    for (unsigned long long it = 0; it < runlen; ++it) {
      if constexpr (H > 1) {
#pragma unroll
        for (int j = 0; j < H - 1; ++j) c[j] = head[j];
      }
      c[H - 1] = v;
      uint32_t W[M][H], cs = mp.one, q = mp.one;
      head_step<M, G, 0>(sm.As, c, W, cs, q, mp);
      uint32_t E[1 << G];
      E[0] = mp.one;
#pragma unroll
      for (int S = 1; S < (1 << G); ++S) E[S] = 0u;
#pragma unroll 1
      for (int col = col0; col < col1; ++col) {
        uint32_t x[M], z[G], nz[G];
        load_column<M>(sm.As + col * CS, x);
#pragma unroll
        for (int d = 0; d < G; ++d) {
          z[d] = affine_dot<H>(cs, x[H + d], W[H + d], x, mp);
          nz[d] = mp.p - z[d];
        }
        subtree_column<G, (1 << G) - 1>(E, z, nz, mp);
      }
      if (lp > 1) {
        LazySum s;
        join_terms<G, 0>(E, mp, s);
        E[(1 << G) - 1] = s.reduce<(1 << G)>(mp);  // the first lane's is the head's sum
      }
      if (r0 + it < r1 && sub == 0) {
        uint32_t num = E[(1 << G) - 1], den = q;
        if (cs == 0u) {
          subtree_pivoting<M, G>(sm.As, c, v, n, mp, num, den);
        } else {
#pragma unroll
          for (int d = 1; d < G; ++d) den = mmul(den, cs, mp);
        }
        N = add_mod(mmul(N, den, mp), mmul(num, Dn, mp), mp.p);
        Dn = mmul(Dn, den, mp);
      }
      if constexpr (H > 1) {
        if (r0 + it + 1 < r1) successor<H - 1>(head, v);
      }
    }
  }
  // lane sums in normal form, added as integers (order-independent)
  unsigned long long r = 0ull;
  if (N != 0u) r = redc(mmul(N, minv(Dn, mp), mp), mp.p, mp.pinv);
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) r += __shfl_xor_sync(kFull, r, off);
  if (lane == 0 && r != 0ull) atomicAdd(sm.sum, r);
  __syncthreads();
  if (threadIdx.x == 0) {
    if (*sm.sum) atomicAdd(&a.residue_sums[kp], *sm.sum);
    __threadfence();
    *sm.last = atomicAdd(&a.hdr->ticket[0], 1u) == gridDim.x * (unsigned)K - 1u;
  }
  __syncthreads();
  if (!*sm.last) return;
  // the last block: residues of det_R (the common sign (-1)^(r + m) of Eq. (1)
  // that the folded column parities leave), then the reconstruction
  if (threadIdx.x < 32) {
    __threadfence();
    uint32_t res = 0u;
    if (lane < K) {
      const uint32_t p = prime_at(lane);
      res = static_cast<uint32_t>(__ldcg(&a.residue_sums[lane]) % p);
      if ((M * (M + 1) / 2 + M) & 1) res = neg_mod(res, p);
    }
    const int status = __ldcg(&a.hdr->status);
    if (a.wide_out) {
      wide_crt_warp(res, K, needed, sm.stats->esum, status, a.total, a.wide_out);
    } else {
      uint32_t all[kMaxPrimes];
#pragma unroll
      for (int k = 0; k < kMaxPrimes; ++k) all[k] = __shfl_sync(kFull, res, k);
      if (lane == 0) crt_write(a.out, all, K, needed, status, a.total, sm.stats->esum);
    }
  }
}

template <int M, int G>
const void* kernel_mg() {
  if constexpr (M - G >= 1) return reinterpret_cast<const void*>(&k_modp_subtree<M, G>);
  else return nullptr;
}
template <int M>
const void* kernel_m(int G) {
  switch (G) {
    case 2: return kernel_mg<M, 2>();
    case 3: return kernel_mg<M, 3>();
    case 4: return kernel_mg<M, 4>();
    case 5: return kernel_mg<M, 5>();
    case 6: return kernel_mg<M, 6>();
    default: return nullptr;
  }
}

}  // namespace

}  // namespace radic
