// Shared parts of the exact (multi-modular) path: Montgomery arithmetic,
// staging of T A mod p, fraction sums, block reduction and the CRT epilogue.
// Included by the per-minor kernels (radic_modp.cu) and the prefix kernels
// (radic_modp_prefix.cu); everything here has internal linkage per file.
#pragma once

#include "radic_prefix.cuh"

namespace radic {

namespace {

constexpr int kMaxThreadsModp = 128;

// Constants of the primes, formed at compile time: the Montgomery constants
// (inverse of p modulo 2^32, R and R^2 modulo p, R = 2^32), and for Garner's
// mixed-radix form the partial products P_l = p_0 ... p_{l-1}: P_l and 1 / P_i
// modulo p_i (times R, so that one Montgomery product applies them), and P_l
// in base-2^32 limbs.
struct PrimeConst {
  uint32_t p, ninv, pinv, one, r2;  // ninv = -1/p, pinv = 1/p modulo 2^32
};
struct PrimeTables {
  PrimeConst c[kWidePrimes];
  uint32_t prod_mod[kWidePrimes][kWidePrimes];           // [l][i]: P_l R mod p_i
  uint32_t prod_inv[kWidePrimes];                        // R / P_i mod p_i
  uint32_t limbs[kWidePrimes + 1][RADIC_WIDE_LIMBS + 1];  // [l]: P_l
};

constexpr PrimeTables make_prime_tables() {
  PrimeTables t{};
  for (int i = 0; i < kWidePrimes; ++i) {
    const uint64_t p = kPrimeTable[i];
    uint32_t x = static_cast<uint32_t>(p);  // Newton iteration x <- x (2 - p x) for 1/p modulo 2^32
    for (int k = 0; k < 5; ++k) x *= 2u - static_cast<uint32_t>(p) * x;
    const uint64_t r1 = (1ull << 32) % p;
    t.c[i].p = static_cast<uint32_t>(p);
    t.c[i].pinv = x;
    t.c[i].ninv = 0u - x;
    t.c[i].one = static_cast<uint32_t>(r1);
    t.c[i].r2 = static_cast<uint32_t>(r1 * r1 % p);
    uint64_t prod = 1;
    for (int l = 0; l < kWidePrimes; ++l) {
      t.prod_mod[l][i] = static_cast<uint32_t>(prod * r1 % p);
      if (l == i) {  // prod = P_i: its inverse is P_i^(p-2)
        uint64_t r = 1, b = prod, e = p - 2;
        while (e) {
          if (e & 1) r = r * b % p;
          b = b * b % p;
          e >>= 1;
        }
        t.prod_inv[i] = static_cast<uint32_t>(r * r1 % p);
      }
      prod = prod * (kPrimeTable[l] % p) % p;
    }
  }
  t.limbs[0][0] = 1u;
  for (int l = 0; l < kWidePrimes; ++l) {
    uint64_t carry = 0;
    for (int j = 0; j <= RADIC_WIDE_LIMBS; ++j) {
      const uint64_t v = static_cast<uint64_t>(t.limbs[l][j]) * kPrimeTable[l] + carry;
      t.limbs[l + 1][j] = static_cast<uint32_t>(v);
      carry = v >> 32;
    }
  }
  return t;
}

// read-only global memory: lanes read different entries
static __device__ const PrimeTables c_primes = make_prime_tables();

__device__ __forceinline__ uint32_t prime_at(int k) { return __ldg(&c_primes.c[k].p); }

struct Mont {
  uint32_t p, pinv, one, r2;  // pinv = -1/p modulo 2^32
  uint64_t p2;
};

__device__ __forceinline__ uint32_t redc(uint64_t t, uint32_t p, uint32_t pinv) {
  const uint32_t mq = static_cast<uint32_t>(t) * pinv;
  const uint32_t u = static_cast<uint32_t>((t + static_cast<uint64_t>(mq) * p) >> 32);
  return u >= p ? u - p : u;
}
__device__ __forceinline__ uint32_t mmul(uint32_t a, uint32_t b, const Mont& mp) {
  return redc(static_cast<uint64_t>(a) * b, mp.p, mp.pinv);
}
// Montgomery form of (akk * aij - aik * akj) from Montgomery-form inputs.
__device__ __forceinline__ uint32_t ff_update(uint32_t akk, uint32_t aij, uint32_t aik, uint32_t akj,
                                              const Mont& mp) {
  const uint64_t t = static_cast<uint64_t>(akk) * aij + mp.p2 - static_cast<uint64_t>(aik) * akj;
  return redc(t, mp.p, mp.pinv);
}
__device__ __forceinline__ uint32_t add_mod(uint32_t a, uint32_t b, uint32_t p) {
  const uint32_t s = a + b;
  return s >= p ? s - p : s;
}
__device__ __forceinline__ uint32_t neg_mod(uint32_t a, uint32_t p) { return a ? p - a : 0u; }

__device__ __forceinline__ Mont make_mont(int k) {
  const PrimeConst c = c_primes.c[k];
  Mont mp;
  mp.p = c.p;
  mp.pinv = c.ninv;
  mp.one = c.one;
  mp.r2 = c.r2;
  mp.p2 = static_cast<uint64_t>(c.p) * c.p;
  return mp;
}

// x^e in Montgomery form.
__device__ inline uint32_t mpow(uint32_t x, uint32_t e, const Mont& mp) {
  uint32_t r = mp.one;
  while (e) {
    if (e & 1u) r = mmul(r, x, mp);
    x = mmul(x, x, mp);
    e >>= 1;
  }
  return r;
}
// x^(p-2) = 1/x (0 for 0) in Montgomery form.  p = 2^31 - d with d < 2^10, so
// the exponent 2^31 - (d + 2) is 21 ones followed by ten bits: the ones by
// doubling (x^(2^k - 1) for k = 1, 2, 4, 5, 10, 20, 21), the bits one at a
// time; about 42 dependent products instead of 60.
static_assert(kPrimeTable[kWidePrimes - 1] > (1u << 31) - (1u << 10) + 2u, "leading ones of p - 2");
__device__ inline uint32_t minv(uint32_t x, const Mont& mp) {
  auto sq = [&](uint32_t a, int k) {
    for (int i = 0; i < k; ++i) a = mmul(a, a, mp);
    return a;
  };
  const uint32_t a2 = mmul(sq(x, 1), x, mp), a4 = mmul(sq(a2, 2), a2, mp), a5 = mmul(sq(a4, 1), x, mp);
  const uint32_t a10 = mmul(sq(a5, 5), a5, mp), a20 = mmul(sq(a10, 10), a10, mp);
  uint32_t r = mmul(sq(a20, 1), x, mp);
  const uint32_t e = mp.p - 2u;
#pragma unroll 1
  for (int b = 9; b >= 0; --b) {
    r = mmul(r, r, mp);
    if ((e >> b) & 1u) r = mmul(r, x, mp);
  }
  return r;
}

__device__ inline uint64_t mix64(uint64_t z) {  // SplitMix64 finaliser
  z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
  z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
  return z ^ (z >> 31);
}

// Floating-point rows: e_i, the exponent of the lowest set bit among row i's
// nonzero entries, and the width w_i = top_i + 1 - e_i, top_i the exponent of
// the highest set bit: the integer row M_i = 2^-e_i A_i has |entry| < 2^w_i, so
// ||M_i|| < sqrt(n) 2^w_i.  A zero row has e_i = 0 and no bits (all its
// minors are zero).  Integer rows: the squared norm in binary32.
struct RowStats {
  int lo[kMaxM], hi[kMaxM];  // floating point: lowest and highest set bit
  float sq[kMaxM];           // integers
  float bits[kMaxM + 1];     // bits of the row's norm bound; [m]: log2 C(n,m)
  double bits64[kMaxM + 1];
  int nonfinite, needed, esum;
  __device__ __forceinline__ bool zero(int i) const { return hi[i] == -0x7fffffff; }
  __device__ __forceinline__ int exponent(int i) const { return zero(i) ? 0 : lo[i]; }
  __device__ __forceinline__ int width(int i) const { return zero(i) ? 0 : hi[i] + 1 - lo[i]; }
};

// Shared-memory layout: binom | K x (n x cs) residues (column-major, Montgomery
// form) | 2 x (m x n) scratch rows | m x m triangular factors | scratch words
// for reductions | Montgomery constants | row statistics.
__host__ __device__ inline size_t modp_smem_bytes(int n, int m, int cs, int threads) {
  size_t off = ((size_t)(n + 1) * (m + 1) * 8 + 15) / 16 * 16;
  off += (size_t)kMaxPrimes * n * cs * 4;
  off += (2 * (size_t)m * n * 4 + 15) / 16 * 16;
  off += ((size_t)m * m * 4 + 15) / 16 * 16;
  off += (size_t)(threads / 32) * kMaxPrimes * 4;
  off = (off + 15) / 16 * 16;
  off += kMaxPrimes * sizeof(Mont);
  off = (off + 15) / 16 * 16;
  return off + (sizeof(RowStats) + 15) / 16 * 16;
}

struct ModpSmem {
  uint64_t* binom;
  uint32_t* As;  // prime k at As + k * n * cs
  uint32_t* rows;
  uint32_t* tri;
  uint32_t* scratch;
  Mont* mont;
  RowStats* stats;
  __device__ ModpSmem(unsigned char* base, int n, int m, int cs, int threads) {
    size_t off = ((size_t)(n + 1) * (m + 1) * 8 + 15) / 16 * 16;
    binom = reinterpret_cast<uint64_t*>(base);
    As = reinterpret_cast<uint32_t*>(base + off);
    off += (size_t)kMaxPrimes * n * cs * 4;
    rows = reinterpret_cast<uint32_t*>(base + off);
    off += (2 * (size_t)m * n * 4 + 15) / 16 * 16;
    tri = reinterpret_cast<uint32_t*>(base + off);
    off += ((size_t)m * m * 4 + 15) / 16 * 16;
    scratch = reinterpret_cast<uint32_t*>(base + off);
    off += (size_t)(threads / 32) * kMaxPrimes * 4;
    off = (off + 15) / 16 * 16;
    mont = reinterpret_cast<Mont*>(base + off);
    off += kMaxPrimes * sizeof(Mont);
    off = (off + 15) / 16 * 16;
    stats = reinterpret_cast<RowStats*>(base + off);
  }
};

__device__ __forceinline__ long long load_int(const void* A, int dtype, long long idx) {
  return dtype == kI8 ? static_cast<long long>(static_cast<const int8_t*>(A)[idx])
                      : static_cast<long long>(static_cast<const int32_t*>(A)[idx]);
}

// ---------------------------------------------------------------------------
// Floating-point inputs.  A binary64 number (binary32 widens to it exactly)
// is +-mant * 2^t with an integer mant < 2^53, so every entry is a dyadic
// rational.  Row i times 2^-e_i, with e_i the exponent of the lowest set bit
// over the row's nonzero entries, is an integer row; every minor is linear
// in each row, so det_R(A) = 2^(sum_i e_i) det_R(M) with M that integer
// matrix, and det_R(M) is found exactly by the modular path.
// ---------------------------------------------------------------------------
struct FpBits {
  uint64_t mant;
  int t;
  bool neg, finite;
};
__device__ __forceinline__ FpBits fp_bits(double x) {
  const uint64_t b = static_cast<uint64_t>(__double_as_longlong(x));
  const int E = static_cast<int>((b >> 52) & 0x7ffu);
  const uint64_t f = b & ((1ull << 52) - 1ull);
  FpBits r;
  r.neg = (b >> 63) != 0;
  r.finite = E != 0x7ff;
  r.mant = E ? (f | (1ull << 52)) : f;
  r.t = E ? E - 1075 : -1074;
  return r;
}
__device__ __forceinline__ double load_fp(const void* A, int dtype, long long idx) {
  return dtype == kF32 ? static_cast<double>(static_cast<const float*>(A)[idx]) : static_cast<const double*>(A)[idx];
}
__device__ __forceinline__ bool is_fp_dtype(int dtype) { return dtype == kF32 || dtype == kF64; }

// Montgomery form of a 64-bit integer: hi 2^32 + lo, 2^32 = R.
__device__ __forceinline__ uint32_t to_mont64(uint64_t x, const Mont& mp) {
  const uint32_t hi = mmul(static_cast<uint32_t>(x >> 32), mp.r2, mp), lo = mmul(static_cast<uint32_t>(x), mp.r2, mp);
  return add_mod(mmul(hi, mp.r2, mp), lo, mp.p);
}

// Residue (normal form) of the integer x * 2^-e modulo p (e at most the
// exponent of x's lowest set bit, so that the shift below drops only zeros).
__device__ inline uint32_t fp_residue(double x, int e, const Mont& mp) {
  const FpBits f = fp_bits(x);
  if (f.mant == 0) return 0u;
  uint32_t r;
  if (f.t >= e) {
    const uint32_t two = add_mod(mp.one, mp.one, mp.p);
    r = mmul(to_mont64(f.mant, mp), mpow(two, static_cast<uint32_t>(f.t - e), mp), mp);
  } else {
    r = to_mont64(f.mant >> (e - f.t), mp);
  }
  r = redc(r, mp.p, mp.pinv);
  return f.neg ? neg_mod(r, mp.p) : r;
}

// Residue (normal form) of a 32-bit integer.
__device__ __forceinline__ uint32_t int_residue(long long v, uint32_t p) {
  if (v < 0) v += p;
  if (v < 0) v += p;  // -2^31 needs p twice for the primes below 2^31
  return static_cast<uint32_t>(v >= (long long)p ? v - p : v);
}

// ---------------------------------------------------------------------------
// Staging.  One pass loads the matrix, each thread keeping its first kKeep
// entries in registers, and forms the row statistics in shared memory; the
// residues, U A and L (U A) are one pass of the block each.  (Row by row, a
// warp per row and a binary64 sum and logarithm per row, this took 2.5 us of
// a 3 x 12 call and 6 us of 10 x 24.)
// ---------------------------------------------------------------------------
constexpr int kKeepModp = 4;
struct KeptEntries {
  double f[kKeepModp];
  int v[kKeepModp];
};

// Statistics of every row, the first kKeepModp entries of every thread kept.
// Ends with a barrier.
__device__ inline void row_stats(const SingleArgs& a, int m, RowStats& st, KeptEntries& keep) {
  const int n = a.n, mn = m * n;
  const bool fp = is_fp_dtype(a.dtype);
  for (int i = threadIdx.x; i < m; i += blockDim.x) {
    st.lo[i] = 0x7fffffff;
    st.hi[i] = -0x7fffffff;
  }
  if (threadIdx.x == 0) st.nonfinite = 0;
  __syncthreads();
  auto bits_of = [&](int i, double f) {
    const FpBits x = fp_bits(f);
    if (!x.finite) {
      st.nonfinite = 1;
    } else if (x.mant) {
      atomicMin(&st.lo[i], x.t + __ffsll(static_cast<long long>(x.mant)) - 1);
      atomicMax(&st.hi[i], x.t + 63 - __clzll(static_cast<long long>(x.mant)));
    }
  };
#pragma unroll
  for (int k = 0; k < kKeepModp; ++k) {
    const int idx = threadIdx.x + k * blockDim.x;
    if (idx < mn) {
      const int i = idx / n;
      const long long at = (long long)i * a.lda + (idx - i * n);
      if (fp) keep.f[k] = load_fp(a.A, a.dtype, at);
      else keep.v[k] = static_cast<int>(load_int(a.A, a.dtype, at));
    }
  }
  if (fp) {
#pragma unroll
    for (int k = 0; k < kKeepModp; ++k) {
      const int idx = threadIdx.x + k * blockDim.x;
      if (idx < mn) bits_of(idx / n, keep.f[k]);
    }
    for (int idx = threadIdx.x + kKeepModp * blockDim.x; idx < mn; idx += blockDim.x) {
      const int i = idx / n;
      bits_of(i, load_fp(a.A, a.dtype, (long long)i * a.lda + (idx - i * n)));
    }
  } else {
    // squared norms, a warp per row, four rows at a time (one round trip to
    // memory for all of them; float atomics on one word take turns)
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    for (int i0 = warp; i0 < m; i0 += 4 * nw) {
      float s[4];
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const int i = i0 + r * nw;
        s[r] = 0.0f;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int j = lane + 32 * h;
          const float v = (i < m && j < n) ? static_cast<float>(load_int(a.A, a.dtype, (long long)i * a.lda + j)) : 0.0f;
          s[r] += v * v;
        }
      }
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) {
#pragma unroll
        for (int r = 0; r < 4; ++r) s[r] += __shfl_xor_sync(kFull, s[r], off);
      }
#pragma unroll
      for (int r = 0; r < 4; ++r)
        if (lane == 0 && i0 + r * nw < m) st.sq[i0 + r * nw] = s[r];
    }
  }
  __syncthreads();
}

// Number of primes for |det_R(A)| <= C(n,m) prod_i ||row_i||_2 (Hadamard's
// inequality for every minor), plus a sign bit and a margin, into st.needed,
// and the total row exponent into st.esum.  The count is defined in binary64,
// whose logarithms and sums are long chains on a slow pipe: the block forms it
// in binary32, whose error is below kNear of a prime (at most 33 sums of at
// most 1100 bits for up to 32 primes: 2e-3 bits, 7e-5 primes, plus the norms'
// 1e-5), and in binary64 only when a count boundary is that close.  Ends with
// a barrier.
__device__ inline void count_primes(const SingleArgs& a, int m, double count, RowStats& st) {
  constexpr float kNear = 1e-3f;
  const bool fp = is_fp_dtype(a.dtype);
  for (int i = threadIdx.x; i <= m; i += blockDim.x) {
    if (i == m) st.bits[m] = log2f(fmaxf(static_cast<float>(count), 1.0f));
    else if (fp) st.bits[i] = st.zero(i) ? 0.0f : static_cast<float>(st.width(i)) + 0.5f * log2f((float)a.n);
    else st.bits[i] = 0.5f * log2f(fmaxf(st.sq[i], 1.0f));
  }
  __syncthreads();
  float est = 0.0f;
  for (int i = 0; i <= m; ++i) est += st.bits[i];
  const float q = (est + 2.0f) * (1.0f / 30.99f);
  int k = static_cast<int>(ceilf(q));
  if (fabsf(q - rintf(q)) <= kNear || !(q < 1e6f)) {  // the same in every thread
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    if (fp) {
      for (int i = threadIdx.x; i < m; i += blockDim.x)
        st.bits64[i] = st.zero(i) ? 0.0 : static_cast<double>(st.width(i)) + 0.5 * log2(static_cast<double>(a.n));
    } else {
      for (int i = warp; i < m; i += nw) {
        double s = 0.0;
        for (int j = lane; j < a.n; j += 32) {
          const double v = static_cast<double>(load_int(a.A, a.dtype, (long long)i * a.lda + j));
          s += v * v;
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(kFull, s, off);
        if (lane == 0) st.bits64[i] = 0.5 * log2(fmax(s, 1.0));
      }
    }
    if (threadIdx.x == 0) st.bits64[m] = log2(fmax(count, 1.0));
    __syncthreads();
    double bits = st.bits64[m];
    for (int i = 0; i < m; ++i) bits += st.bits64[i];
    k = static_cast<int>(ceil((bits + 2.0) / 30.99));
  }
  if (threadIdx.x == 0) {
    int es = 0;
    if (fp)
      for (int i = 0; i < m; ++i) es += st.exponent(i);
    st.needed = k < 1 ? 1 : k;
    st.esum = es;
    if (st.nonfinite) atomicExch(&a.hdr->status, RADIC_EINVAL);  // an entry is not finite
  }
  __syncthreads();
}

// (T A mod p) in Montgomery form into As (column-major, column stride cs,
// padding rows zero) for the prime mp: T = L U with L unit lower and U unit
// upper triangular, entries from a hash of (slot, row, column).  With
// alt_sign, odd columns are negated (the column parities of Eq. (1)).  tri:
// m x m words, rows: 2 m n words of shared scratch.
__device__ inline void stage_prime(const SingleArgs& a, int m, int cs, int slot, const Mont& mp, const RowStats& st,
                                   const KeptEntries& keep, uint32_t* tri, uint32_t* rows, uint32_t* As,
                                   bool alt_sign) {
  const int n = a.n, mn = m * n;
  const bool fp = is_fp_dtype(a.dtype);
  uint32_t* ua = rows + mn;
  for (int idx = threadIdx.x; idx < m * m; idx += blockDim.x) {
    const int i = idx / m, l = idx - i * m;
    const uint64_t h = l > i ? mix64(0x9e3779b97f4a7c15ull * (uint64_t)(slot * 4096 + i * 64 + l) + 1ull)
                             : mix64(0xd1b54a32d192ed03ull * (uint64_t)(slot * 4096 + i * 64 + l) + 7ull);
    const uint32_t r = static_cast<uint32_t>(h >> 33);  // 31 bits
    tri[idx] = r >= mp.p ? r - mp.p : r;
  }
#pragma unroll
  for (int k = 0; k < kKeepModp; ++k) {
    const int idx = threadIdx.x + k * blockDim.x;
    if (idx < mn) rows[idx] = fp ? fp_residue(keep.f[k], st.exponent(idx / n), mp) : int_residue(keep.v[k], mp.p);
  }
  for (int idx = threadIdx.x + kKeepModp * blockDim.x; idx < mn; idx += blockDim.x) {
    const int i = idx / n, j = idx - i * n;
    const long long at = (long long)i * a.lda + j;
    rows[idx] = fp ? fp_residue(load_fp(a.A, a.dtype, at), st.exponent(i), mp)
                   : int_residue(load_int(a.A, a.dtype, at), mp.p);
  }
  __syncthreads();
  // x + sum of u_l v_l over [l0, l1): two products per reduction
  auto dot = [&](uint32_t x, const uint32_t* u, const uint32_t* v, int l0, int l1) {
    int l = l0;
    for (; l + 1 < l1; l += 2) {
      const uint64_t t = static_cast<uint64_t>(u[l]) * v[l * n] + static_cast<uint64_t>(u[l + 1]) * v[(l + 1) * n];
      x = add_mod(x, redc(t, mp.p, mp.pinv), mp.p);
    }
    if (l < l1) x = add_mod(x, mmul(u[l], v[l * n], mp), mp.p);
    return x;
  };
  for (int idx = threadIdx.x; idx < mn; idx += blockDim.x) {
    const int i = idx / n, j = idx - i * n;
    ua[idx] = dot(rows[idx], tri + i * m, rows + j, i + 1, m);
  }
  __syncthreads();
  for (int idx = threadIdx.x; idx < n * cs; idx += blockDim.x) {
    const int j = idx / cs, i = idx - j * cs;
    uint32_t v = 0u;
    if (i < m) {
      v = mmul(dot(ua[i * n + j], tri + i * m, ua + j, 0, i), mp.r2, mp);
      if (alt_sign && (j & 1)) v = neg_mod(v, mp.p);
    }
    As[idx] = v;
  }
  __syncthreads();
}

// Stage binom and, for each prime of the pass, (T A mod p) in Montgomery
// form.  Slot k holds prime a.prime_base + k.  Returns K (primes this pass
// uses; 0 when the bound needs none of them) in every thread; sets *needed
// to the primes the bound asks for.
__device__ inline int stage_modp(const SingleArgs& a, const ModpSmem& sm, int m, int cs, int* needed) {
  const int n = a.n;
  const int base = a.prime_base;
  build_binom(sm.binom, n, m);
  if (threadIdx.x < kMaxPrimes && base + (int)threadIdx.x < kWidePrimes)
    sm.mont[threadIdx.x] = make_mont(base + threadIdx.x);
  KeptEntries keep;
  row_stats(a, m, *sm.stats, keep);
  count_primes(a, m, static_cast<double>(sm.binom[n * (m + 1) + m]), *sm.stats);
  *needed = sm.stats->needed;
  const int K = max(0, min(min(*needed, kWidePrimes) - base, kMaxPrimes));
  for (int k = 0; k < K; ++k)
    stage_prime(a, m, cs, k, sm.mont[k], *sm.stats, keep, sm.tri, sm.rows, sm.As + (size_t)k * n * cs, false);
  return K;
}

// Slow path: determinant (Montgomery form) with row exchanges and inverses.
template <int MC>
__device__ __noinline__ uint32_t det_pivoting(const uint32_t* As, int cs, const int* c, int m, Mont mp) {
  uint32_t x[MC * MC];
  for (int i = 0; i < m; ++i)
    for (int j = 0; j < m; ++j) x[i * MC + j] = As[c[j] * cs + i];
  uint32_t det = mp.one;
  for (int k = 0; k < m; ++k) {
    int p = -1;
    for (int i = k; i < m; ++i)
      if (x[i * MC + k] != 0u) {
        p = i;
        break;
      }
    if (p < 0) return 0u;
    if (p != k) {
      for (int j = 0; j < m; ++j) {
        const uint32_t t = x[k * MC + j];
        x[k * MC + j] = x[p * MC + j];
        x[p * MC + j] = t;
      }
      det = neg_mod(det, mp.p);
    }
    det = mmul(det, x[k * MC + k], mp);
    const uint32_t inv = minv(x[k * MC + k], mp);
    for (int i = k + 1; i < m; ++i) {
      const uint32_t l = mmul(x[i * MC + k], inv, mp);
      for (int j = k + 1; j < m; ++j)
        x[i * MC + j] = add_mod(x[i * MC + j], neg_mod(mmul(l, x[k * MC + j], mp), mp.p), mp.p);
    }
  }
  return det;
}

template <int M, int CS>
__device__ __forceinline__ void gather_u32(const uint32_t* __restrict__ As, const int (&c)[M],
                                           uint32_t (&x)[M][M]) {
#pragma unroll
  for (int j = 0; j < M; ++j) {
    const uint32_t* col = As + c[j] * CS;
#pragma unroll
    for (int i = 0; i < M; i += 4) {
      const uint4 v = *reinterpret_cast<const uint4*>(col + i);
      x[i][j] = v.x;
      if (i + 1 < M) x[i + 1][j] = v.y;
      if (i + 2 < M) x[i + 2][j] = v.z;
      if (i + 3 < M) x[i + 3][j] = v.w;
    }
  }
}

// Fraction-free elimination of one minor: det = num / den (Montgomery form).
template <int M>
__device__ __forceinline__ bool ff_det(uint32_t (&x)[M][M], const Mont& mp, uint32_t& num, uint32_t& den) {
  uint32_t P = mp.one, D = mp.one;
  bool zero_pivot = false;
#pragma unroll
  for (int k = 0; k < M - 1; ++k) {
    const uint32_t piv = x[k][k];
    zero_pivot |= (piv == 0u);
    if (k <= M - 3) {
      P = mmul(P, piv, mp);
      D = mmul(D, P, mp);
    }
#pragma unroll
    for (int i = k + 1; i < M; ++i)
#pragma unroll
      for (int j = k + 1; j < M; ++j) x[i][j] = ff_update(piv, x[i][j], x[i][k], x[k][j], mp);
  }
  num = x[M - 1][M - 1];
  den = D;
  return zero_pivot;
}

// Block sum modulo each prime; result in thread 0's r[].
__device__ inline void block_reduce_modp(uint32_t (&r)[kMaxPrimes], int K, uint32_t* scratch, const Mont* mont) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
  for (int k = 0; k < kMaxPrimes; ++k) {
    if (k < K) {
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) r[k] = add_mod(r[k], __shfl_xor_sync(kFull, r[k], off), mont[k].p);
    }
  }
  __syncthreads();
  if (lane == 0)
    for (int k = 0; k < K; ++k) scratch[warp * kMaxPrimes + k] = r[k];
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int k = 0; k < K; ++k) {
      uint32_t s = 0;
      for (int w = 0; w < nw; ++w) s = add_mod(s, scratch[w * kMaxPrimes + k], mont[k].p);
      r[k] = s;
    }
  }
}

// Garner reconstruction of the signed value in (-P/2, P/2].
__device__ inline void crt_write(radic_result* out, const uint32_t* res, int K, int needed, int status,
                                 unsigned long long total, int escale) {
  uint32_t v[kMaxPrimes];
#pragma unroll
  for (int i = 0; i < kMaxPrimes; ++i) {
    if (i >= K) break;
    const Mont mp = make_mont(i);
    uint32_t acc = 0u;  // value of the digits so far modulo p
#pragma unroll
    for (int l = 0; l < i; ++l) acc = add_mod(acc, mmul(v[l], c_primes.prod_mod[l][i], mp), mp.p);
    v[i] = mmul(add_mod(res[i], neg_mod(acc, mp.p), mp.p), c_primes.prod_inv[i], mp);
  }
  unsigned __int128 x = 0, big = 1;
#pragma unroll
  for (int i = 0; i < kMaxPrimes; ++i) {
    if (i < K) {
      x += static_cast<unsigned __int128>(v[i]) * big;
      big *= prime_at(i);
    }
  }
  __int128 sx = static_cast<__int128>(x);
  if (x > big / 2) sx = static_cast<__int128>(x) - static_cast<__int128>(big);
  const unsigned __int128 ux = static_cast<unsigned __int128>(sx);
  out->exact_lo = static_cast<long long>(static_cast<uint64_t>(ux));
  out->exact_hi = static_cast<long long>(static_cast<uint64_t>(ux >> 64));
  const bool negv = sx < 0;
  const unsigned __int128 mag = negv ? static_cast<unsigned __int128>(-sx) : static_cast<unsigned __int128>(sx);
  const double val = ldexp(static_cast<double>(static_cast<uint64_t>(mag >> 64)), 64) +
                     static_cast<double>(static_cast<uint64_t>(mag));
  out->value = ldexp(negv ? -val : val, escale);
  out->abs_sum = 0.0;
  out->err_bound = 0.0;
  out->minors = static_cast<long long>(total);
  out->flagged = 0;
  out->status = (needed > kMaxPrimes) ? RADIC_EOVERFLOW : status;
  out->n_primes = K;
  out->tier = kModeExact;
  out->exact_exp = escale;
  for (int i = 0; i < 5; ++i) out->reserved[i] = 0;
}

// Wide exact result from the residues modulo the first K primes (lane i
// holds residue i; K <= 32), by one whole warp.  Mixed-radix digits v_l
// (Garner): step l fixes v_l in lane l, and the later lanes add v_l P_l to
// their value modulo their own prime.  The integer is sum_l v_l P_l: lane j
// adds limb j of every term (the P_l are compile-time constants), then the
// warp resolves the carries.  The symmetric range (-M/2, M/2), M the product
// of the primes, gives the sign.  (Written serially, with an exponentiation
// per digit and a limb-by-limb Horner rule, this took 245 us for 15 primes;
// by a warp but with 64-bit divisions still 44 us.)
static_assert(kMaxN <= 64, "two entries of a row per lane");
static_assert(RADIC_WIDE_LIMBS == 32 && kWidePrimes == 32, "one lane per limb and prime; kAhead divides it");

// x + carry-in from the lane below until no lane carries; lane 31's carry is lost.
__device__ inline uint32_t warp_resolve_carry(uint64_t x, int lane) {
  for (;;) {
    const uint32_t c = static_cast<uint32_t>(x >> 32);
    if (!__any_sync(kFull, c != 0u)) return static_cast<uint32_t>(x);
    const uint32_t in = __shfl_up_sync(kFull, c, 1);
    x = (x & 0xffffffffull) + (lane > 0 ? in : 0u);
  }
}
// Limbs of a - b (a >= b), lane j holding limb j.
__device__ inline uint32_t warp_limbs_sub(uint32_t a, uint32_t b, int lane) {
  long long t = static_cast<long long>(a) - b;
  for (;;) {
    const int borrow = t < 0;
    if (!__any_sync(kFull, borrow)) return static_cast<uint32_t>(t);
    if (borrow) t += 1ll << 32;
    const int in = __shfl_up_sync(kFull, borrow, 1);
    if (lane > 0) t -= in;
  }
}

__device__ inline void wide_crt_warp(uint32_t res, int K, int needed, int escale, int status, unsigned long long total,
                                     radic_wide_result* out) {
  const int lane = threadIdx.x & 31;
  const Mont mp = make_mont(lane);
  const uint32_t inv = c_primes.prod_inv[lane];
  uint32_t acc = 0u;
  uint64_t lo = 0;   // limb j of the sum, 96 bits
  uint32_t hi = 0u;
  // constants are fetched kAhead steps at a time, ahead of the digit chain
  constexpr int kAhead = 8;
  for (int l0 = 0; l0 < K; l0 += kAhead) {
    uint32_t pm[kAhead], lm[kAhead];
#pragma unroll
    for (int u = 0; u < kAhead; ++u) {
      pm[u] = __ldg(&c_primes.prod_mod[l0 + u][lane]);
      lm[u] = __ldg(&c_primes.limbs[l0 + u][lane]);
    }
#pragma unroll
    for (int u = 0; u < kAhead; ++u) {
      if (l0 + u < K) {
        const uint32_t d = mmul(add_mod(res, neg_mod(acc, mp.p), mp.p), inv, mp);
        const uint32_t v = __shfl_sync(kFull, d, l0 + u);
        if (lane > l0 + u) acc = add_mod(acc, mmul(v, pm[u], mp), mp.p);
        const uint64_t t = static_cast<uint64_t>(v) * lm[u];
        lo += t;
        hi += lo < t ? 1u : 0u;
      }
    }
  }
  // x = sum over lanes of (hi 2^64 + lo) 2^(32 lane)
  const uint32_t mid = __shfl_up_sync(kFull, static_cast<uint32_t>(lo >> 32), 1);
  const uint32_t top = __shfl_up_sync(kFull, hi, 2);
  const uint32_t x = warp_resolve_carry((lo & 0xffffffffull) + (lane > 0 ? mid : 0u) + (lane > 1 ? top : 0u), lane);
  // d = M - x; the value is x when x < d (that is x < M/2), else -(M - x).
  // M < 2^(31 * 32) fits the 32 limbs.
  const uint32_t d = warp_limbs_sub(c_primes.limbs[K][lane], x, lane);
  const unsigned lt = __ballot_sync(kFull, x < d), gt = __ballot_sync(kFull, x > d);
  const bool x_less = lt > gt;  // the highest limb that differs decides
  const uint32_t mag = x_less ? x : d;
  const unsigned used = __ballot_sync(kFull, mag != 0u);
  const int nl = 32 - __clz(static_cast<int>(used));
  out->limbs[lane] = mag;
  double val = 0.0;
  const int low = nl > 3 ? nl - 3 : 0;
  for (int i = nl - 1; i >= low; --i) val = val * 4294967296.0 + static_cast<double>(__shfl_sync(kFull, mag, i));
  if (lane == 0) {
    const int sgn = nl == 0 ? 0 : (x_less ? 1 : -1);
    out->value = sgn < 0 ? -ldexp(val, 32 * low + escale) : ldexp(val, 32 * low + escale);
    out->status = (needed > kWidePrimes) ? RADIC_EOVERFLOW : status;
    out->n_primes = K;
    out->exact_exp = escale;
    out->sign = sgn;
    out->n_limbs = nl;
    out->minors = static_cast<long long>(total);
    out->reserved = 0;
  }
}

// Last-block epilogue shared by both mappings.
// Wide passes write the pass's residues into a.wide[prime index] instead;
// the pass with the first primes also writes needed, the exponent and the
// status after the kWidePrimes residue slots.
__device__ inline void finish_modp(const SingleArgs& a, const ModpSmem& sm, uint32_t (&r)[kMaxPrimes], int K,
                                   int needed) {
  block_reduce_modp(r, K, sm.scratch, sm.mont);
  if (threadIdx.x == 0)
    for (int k = 0; k < kMaxPrimes; ++k) a.modp_partials[blockIdx.x * kMaxPrimes + k] = (k < K) ? r[k] : 0u;
  if (last_block(&a.hdr->ticket[0])) {
    uint32_t t[kMaxPrimes] = {0, 0, 0, 0};
    for (int b = threadIdx.x; b < (int)gridDim.x; b += blockDim.x)
      for (int k = 0; k < K; ++k) t[k] = add_mod(t[k], __ldcg(&a.modp_partials[b * kMaxPrimes + k]), sm.mont[k].p);
    block_reduce_modp(t, K, sm.scratch, sm.mont);
    if (threadIdx.x == 0) {
      if (a.wide) {
        for (int k = 0; k < K; ++k) a.wide[a.prime_base + k] = t[k];
        if (a.prime_base == 0) {
          a.wide[kWidePrimes] = static_cast<uint32_t>(needed);
          a.wide[kWidePrimes + 1] = static_cast<uint32_t>(sm.stats->esum);
          a.wide[kWidePrimes + 2] = static_cast<uint32_t>(__ldcg(&a.hdr->status));
        }
      } else {
        crt_write(a.out, t, K, needed, __ldcg(&a.hdr->status), a.total, sm.stats->esum);
      }
    }
  }
}

// Adds the signed term num/den of one minor to the running fraction N/Dn of
// prime slot `k` (fraction form: N/Dn + s*num/den = (N*den + s*num*Dn)/(Dn*den)).
__device__ __forceinline__ void acc_fraction(uint32_t (&N)[kMaxPrimes], uint32_t (&Dn)[kMaxPrimes], int k,
                                             uint32_t num, uint32_t den, bool neg, const Mont& mp) {
#pragma unroll
  for (int kk = 0; kk < kMaxPrimes; ++kk) {
    if (kk == k) {
      uint32_t t = mmul(num, Dn[kk], mp);
      if (neg) t = neg_mod(t, mp.p);
      N[kk] = add_mod(mmul(N[kk], den, mp), t, mp.p);
      Dn[kk] = mmul(Dn[kk], den, mp);
    }
  }
}

// Residue N/Dn in normal form for every used prime.
__device__ inline void close_fractions(const uint32_t (&N)[kMaxPrimes], const uint32_t (&Dn)[kMaxPrimes], int K,
                                       const Mont* mont, uint32_t (&r)[kMaxPrimes]) {
#pragma unroll
  for (int k = 0; k < kMaxPrimes; ++k) {
    r[k] = 0u;
    if (k < K) {
      const Mont mp = mont[k];
      r[k] = redc(mmul(N[k], minv(Dn[k], mp), mp), mp.p, mp.pinv);
    }
  }
}

}  // namespace

}  // namespace radic
