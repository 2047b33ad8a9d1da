// C-ABI entry points of the single-matrix path: argument validation, launch
// planning (mapping, grid, workspace layout) and launches.  Validation happens
// entirely on the host before anything is enqueued.
#include <algorithm>
#include <cstring>
#include <mutex>
#include <new>
#include <string>
#include <unordered_map>

#include "radic_device.cuh"

namespace radic {

namespace {
constexpr BinomConst kBinomHost = make_binom_const();
}

unsigned long long binom_host(int n, int k) {
  if (k < 0 || k > n) return 0ull;
  return kBinomHost.v[n][k];
}

int device_sm_count() {
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 0;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
  return sms;
}

namespace {

bool valid_dtype(int d) { return d == kI8 || d == kI32 || d == kF32 || d == kF64; }
bool valid_mode(int md) { return md == kModeFp64 || md == kModeMixed || md == kModeExact || md == kModePair; }

int thread_limit(int mode) {
  if (mode == kModePair) return 0;  // prefix mapping only
  return mode == kModeFp64 ? kThreadMaxMFp64 : (mode == kModeMixed ? kThreadMaxMFp32 : kThreadMaxMModp);
}

int blocks_per_sm(const SinglePlan& p) {
  switch (p.mode) {
    case kModeFp64: return blocks_per_sm_fp64(p);
    case kModeMixed: return blocks_per_sm_mixed(p);
    case kModePair: return blocks_per_sm_pair(p);
    default: return blocks_per_sm_modp(p, p.mapping == RADIC_MAP_PREFIX ? kModpTerms : kModpDet);
  }
}

size_t smem_of(const SinglePlan& p) {
  switch (p.mode) {
    case kModeFp64: return smem_fp64(p);
    case kModeMixed: return smem_mixed(p);
    case kModePair: return smem_pair(p);
    default: return smem_modp(p, p.mapping == RADIC_MAP_PREFIX ? kModpTerms : kModpDet);
  }
}

void layout_workspace(SinglePlan& pl);

// Cost of one head of H = m - G columns with k later columns in the subtree
// kernel, in issued instructions: a dot product of N residues takes about
// 1.4 N + 8 (multiply-adds at half rate, folds, reduction and correction).
double subtree_cost(int m, int G, int k) {
  const int H = m - G;
  double head = 60.0, col = 0.0;
  for (int j = 0; j < H; ++j) head += (m - j) * (1.4 * (j + 1) + 8.0) + (m - j - 1) * (11.0 * j + 6.0);
  col += G * (1.4 * (H + 1) + 10.0);
  for (int s = 1; s <= G; ++s) col += (double)binom_host(G, s) * (s == 1 ? 3.0 : 1.4 * s + 10.0);
  return head + k * col;
}

// Subtree table of the EXACT determinant for heads of m - G columns: group v
// (last head column) holds C(v, H-1) heads, one head per lane and task (or
// ranks_per_task consecutive ones).  Heads with split_from or more later
// columns take two lanes, each half of the columns.
PrefixTable subtree_table(int m, int n, int G, int run_given, int split_from) {
  const int H = m - G;
  PrefixTable t{};
  t.v_lo = H - 1;
  t.v_hi = n - 1 - G;
  unsigned long long start = 0;
  for (int v = t.v_lo; v <= t.v_hi; ++v) {
    t.count[v] = binom_host(v, H - 1);
    t.lanes[v] = n - 1 - v >= split_from ? 2 : 1;
    const unsigned long long groups = 32 / t.lanes[v];
    t.run[v] = std::min<unsigned long long>(run_given > 0 ? run_given : 1, (t.count[v] + groups - 1) / groups);
    t.task_start[v] = start;
    start += (t.count[v] + groups * t.run[v] - 1) / (groups * t.run[v]);
  }
  if (t.v_hi + 1 < kMaxN) t.task_start[t.v_hi + 1] = start;
  t.total_tasks = start;
  return t;
}

// Depth G of the summed subtrees and from how many columns on a head takes two
// lanes: an explicit prefix depth is taken as it is; otherwise the choice whose
// estimated time is least.  Warps that share a scheduler issue about one of
// these instructions in two cycles, a warp on its own one in six (measured on
// the longest heads of 8 x 32): the estimate adds the work of the expected
// primes spread over the chip's schedulers and the longest task alone.  Small
// matrices thus take shallow subtrees (more, shorter lanes), large ones deep
// subtrees; splitting the columns of the longest heads, whose groups are too
// small to fill their warps anyway, nearly halves the longest task.  Every
// block stages the matrix for its prime (5 to 9 us), so the blocks of the
// expected primes together fill the chip once; large matrices take more
// blocks, of at least eight tasks a warp, because the number of primes is only
// known on the device and a last wave that is partly empty costs more.
void plan_subtree(SinglePlan& pl, const radic_options& d, int sms) {
  const int m = pl.m, n = pl.n;
  for (int w = 0; w < 2; ++w) {
    const double primes = w ? 12.0 : 2.0;  // typical counts: random binary64 rows; small integers
    int best = 0;
    double best_time = 0.0;
    for (int G = 2; G <= kSubtreeMax && G < m; ++G) {
      if (d.prefix_depth != 0 && G != d.prefix_depth) continue;
      const int kmax = n - m + G;  // later columns of the longest head
      for (const int split : {kMaxN + 1, (3 * kmax + 3) / 4, (kmax + 1) / 2}) {
        const PrefixTable t = subtree_table(m, n, G, d.ranks_per_task, split);
        double work = 0.0, longest = 0.0;
        for (int v = t.v_lo; v <= t.v_hi; ++v) {
          const int k = n - 1 - v;
          const double c = (double)t.run[v] * (t.lanes[v] == 2 ? subtree_cost(m, G, (k + 1) / 2) + 4.0 * (1 << G)
                                                                : subtree_cost(m, G, k));
          const unsigned long long next = v < t.v_hi ? t.task_start[v + 1] : t.total_tasks;
          work += c * (double)(next - t.task_start[v]);
          longest = std::max(longest, c);
        }
        const double time = 2.0 * primes * work / (4.0 * sms) + 6.0 * longest;
        if (best == 0 || time < best_time) {
          best = G;
          best_time = time;
          pl.stab[w] = t;
        }
      }
    }
    pl.subtree[w] = best;
    const int warps = pl.threads / 32;
    const unsigned long long need = (pl.stab[w].total_tasks + warps - 1) / warps;
    const int per_sm = std::max(1, blocks_per_sm_modp(pl, w ? kModpWide : kModpDet));
    const unsigned long long fill = (unsigned long long)(sms * per_sm / primes) + 1;
    const unsigned long long cap = std::max(fill, std::min(need / 8, 4ull * sms * per_sm));
    pl.sub_blocks[w] = d.blocks > 0 ? d.blocks : (int)std::max(1ull, std::min(need, cap));
  }
}

// `launch`: the plan is for this device, not for a host-only query.
int plan_prefix(SinglePlan pl, const radic_options& d, int sms, int per_sm, unsigned long long units, bool launch,
                SinglePlan* out) {
  const int m = pl.m, n = pl.n, D = pl.depth, P = m - D;
  PrefixTable& t = pl.ptab;
  t.v_lo = P - 1;
  t.v_hi = n - 1 - D;
  t.dynamic = d.deterministic ? 0 : 1;
  double total_cost = 0.0;
  double cost[kMaxN] = {0};
  for (int v = t.v_lo; v <= t.v_hi; ++v) {
    t.count[v] = binom_host(v, P - 1);
    cost[v] = prefix_cost(m, D, n - 1 - v);
    total_cost += cost[v] * (double)t.count[v];
  }
  const unsigned long long lanes = (unsigned long long)sms * per_sm * pl.threads;
  const double per_lane = total_cost / (double)lanes / 4.0;  // about four tasks per warp
  const double red = (double)m * P * P;  // elimination, repeated by every lane that shares a prefix
  // Smallest power of two of lanes that brings a lane's cost down to `target`.
  auto lanes_for = [&](int v, double target) {
    int lp = 1;
    while (lp < 32 && red + (cost[v] - red) / lp > target) lp *= 2;
    return lp;
  };
  auto run_for = [&](int v, int lp) {
    const unsigned long long groups = 32 / lp;  // lane groups per warp
    const double r = per_lane * lp / cost[v];
    unsigned long long run = r < 1.0 ? 1ull : (unsigned long long)r;
    if (d.ranks_per_task > 0) run = (unsigned long long)d.ranks_per_task;
    const unsigned long long maxrun = (t.count[v] + groups - 1) / groups;
    if (run > maxrun) run = maxrun > 0 ? maxrun : 1;
    return run;
  };
  // Lanes per prefix: a prefix with many candidate columns costs far more
  // than a lane's share of the launch (the leaves grow like C(k, D)), so
  // its column reductions and leaves are split over several lanes of the
  // warp, each of which repeats the factorisation.
  const bool seq = pl.mode == kModeFp64 && D == 2 && m >= 4;
  double target = 0.0;
  if (D == 3) {
    // Near the mean per-lane work.  With binary32 elimination: 1.4
    // times the mean lane work when that is large, three times when the
    // launch is small and the repeated factorisations would dominate.
    // Binary64 and pair leaves keep their pipes busy, so there the balance
    // of the warps' shares matters more than the repeated work: the mean
    // itself.  (Measured on the shapes of prefix_auto_depth, warps drawing
    // tasks from the shared counter.)
    const double mean = 4.0 * per_lane;
    target = (pl.mode == kModeMixed ? (mean >= 1000.0 ? 1.4 : 3.0) : 1.0) * mean;
  } else if (seq) {
    // Binary64 depth 2, whose small launches otherwise leave most SMs idle
    // behind one lane's chain of binary64 operations (5 x 16: 5 blocks on 152
    // SMs).  In the other modes splitting depth-2 prefixes measured slower.
    // The mean over one warp per scheduler, which is what keeps the binary64
    // pipe busy, as long as the tasks fit one wave of warps.
    target = total_cost / ((double)sms * 128.0);
    double work, longest, most = 0.0;  // of the plan with target tau, in cost units
    auto tasks_for = [&](double tau) {
      unsigned long long tasks = 0;
      work = longest = 0.0;
      for (int v = t.v_lo; v <= t.v_hi; ++v) {
        const int lp = lanes_for(v, tau);
        const unsigned long long run = run_for(v, lp), chunk = 32ull / lp * run, k = (t.count[v] + chunk - 1) / chunk;
        const double c = (double)run * (red + (cost[v] - red) / lp);
        tasks += k;
        work += (double)k * c;
        longest = std::max(longest, c);
        most = std::max(most, cost[v]);
      }
      return tasks;
    };
    if (tasks_for(target) > (unsigned long long)sms * per_sm * (pl.threads / 32) && target < 4.0 * red) {
      // A mean near or below the elimination itself splits every prefix as far
      // as it goes and repeats the elimination for nothing: the target with
      // the least estimate instead.  A cost unit takes an SM 10 ns and a lone
      // warp 30, a task as much as 95 units (fitted to 250 plans of m = 4..6,
      // n = 6..63).  6 x 23 on 32 lanes throughout 99 us, one lane each 71,
      // now 33; 5 x 26 41, 82, 27.
      double best = 0.0;
      for (double tau = std::max(target, 1.05 * red);; tau *= 1.15) {
        const double tasks = (double)tasks_for(tau), time = 10.0 * (work + 95.0 * tasks) / sms + 30.0 * longest;
        if (best == 0.0 || time < best) {
          best = time;
          target = tau;
        }
        if (tau >= most) break;
      }
    }
  }
  unsigned long long start = 0;
  for (int v = t.v_lo; v <= t.v_hi; ++v) {
    const int lp = d.lanes_per_prefix > 0 ? d.lanes_per_prefix : D == 3 || seq ? lanes_for(v, target) : 1;
    t.lanes[v] = lp;
    t.run[v] = run_for(v, lp);
    const unsigned long long chunk = 32ull / lp * t.run[v];
    start += (t.count[v] + chunk - 1) / chunk;
  }
  // Binary64 depth 3: the lanes of a group can factor a prefix each and then
  // share the leaves of one after the other (prefix_group), so that runs of up
  // to lp prefixes cost one elimination where every lane used to repeat the
  // prefix's own.  Runs grow to one task per resident warp by the cost of a
  // shared prefix's leaves (a lane's share, and per column what the group does
  // together).  Taken if it halves the tasks at least: 10 x 20 850 -> 341 us,
  // 9 x 20 432 -> 226, 8 x 20 178 -> 131.  (Grown by number alone, whatever
  // the leaves cost, 7 x 20 and 8 x 20 were 1.35 times slower than before.)
  if (pl.mode == kModeFp64 && D == 3 && m >= 7 && d.ranks_per_task == 0) {
    double total = 0.0;
    auto leaves = [&](int v) { return (cost[v] - red) / t.lanes[v] + 30.0 * (n - 1 - v); };
    for (int v = t.v_lo; v <= t.v_hi; ++v) total += (double)t.count[v] * (red + t.lanes[v] * leaves(v));
    const double share = total / (double)lanes;
    unsigned long long runs[kMaxN], tasks = 0;
    for (int v = t.v_lo; v <= t.v_hi; ++v) {
      const unsigned long long lp = t.lanes[v], groups = 32 / lp, maxrun = (t.count[v] + groups - 1) / groups;
      const unsigned long long fit = share > red ? (unsigned long long)((share - red) / leaves(v)) : 0ull;
      runs[v] = std::max(t.run[v], std::min({lp, fit, maxrun}));
      tasks += (t.count[v] + groups * runs[v] - 1) / (groups * runs[v]);
    }
    if (2 * tasks <= start) {
      t.share = 1;
      std::copy(runs + t.v_lo, runs + t.v_hi + 1, t.run + t.v_lo);
    }
  }
  start = 0;
  for (int v = t.v_lo; v <= t.v_hi; ++v) {
    const unsigned long long chunk = 32ull / t.lanes[v] * t.run[v];
    t.task_start[v] = start;
    start += (t.count[v] + chunk - 1) / chunk;
  }
  if (t.v_hi + 1 < kMaxN) t.task_start[t.v_hi + 1] = start;
  if (t.v_hi < t.v_lo) start = 0;
  t.total_tasks = start;
  const unsigned long long warps_per_block = pl.threads / 32;
  const unsigned long long need = (start + warps_per_block - 1) / warps_per_block;
  const unsigned long long cap = (unsigned long long)sms * per_sm;
  unsigned long long blocks = need < cap ? need : cap;
  if (d.blocks > 0) blocks = (unsigned long long)d.blocks;
  if (blocks < 1) blocks = 1;
  if (blocks > (1ull << 20)) return RADIC_EINVAL;
  pl.blocks = (int)blocks;
  pl.blocks2 = sms;
  // per-minor split used by the binary64 fall-back pass of the mixed mode
  const unsigned long long procs = (unsigned long long)pl.blocks2 * 128;
  pl.ranks_per_task = (units + procs - 1) / procs;
  if (pl.ranks_per_task < 1) pl.ranks_per_task = 1;
  pl.tasks = (units + pl.ranks_per_task - 1) / pl.ranks_per_task;
  if (pl.mode == kModeExact && launch) plan_subtree(pl, d, sms);  // asks the device for its occupancy
  layout_workspace(pl);
  *out = pl;
  return RADIC_OK;
}

// Plans a launch over `units` ranks (C(n,m) for radic_det, `count` for
// radic_terms).  Returns a RADIC_* code.
int make_plan_uncached(int m, int n, int mode, const radic_options* o, unsigned long long units, SinglePlan* p,
                       int sms_given = 0, int per_sm_given = 0);

// Plans are pure functions of (device, shape, mode, options, units); repeated
// calls on one shape (the common case when serving) reuse the plan instead of
// repeating the occupancy queries.  The kernel_events pointer is not part of
// the plan and is filled in per call.
int make_plan(int m, int n, int mode, const radic_options* o, unsigned long long units, SinglePlan* p) {
  int dev = 0;
  // without a device the uncached planner still reports argument errors first
  if (cudaGetDevice(&dev) != cudaSuccess) return make_plan_uncached(m, n, mode, o, units, p);
  radic_options key_opts;
  std::memset(&key_opts, 0, sizeof(key_opts));
  if (o) key_opts = *o;
  key_opts.kernel_events = nullptr;
  const int head[4] = {dev, m, n, mode};
  std::string key(reinterpret_cast<const char*>(head), sizeof(head));
  key.append(reinterpret_cast<const char*>(&units), sizeof(units));
  key.append(reinterpret_cast<const char*>(&key_opts), sizeof(key_opts));
  static std::mutex mu;
  static std::unordered_map<std::string, SinglePlan> cache;
  {
    std::lock_guard<std::mutex> lock(mu);
    auto it = cache.find(key);
    if (it != cache.end()) {
      *p = it->second;
      p->events = o ? o->kernel_events : nullptr;
      return RADIC_OK;
    }
  }
  const int rc = make_plan_uncached(m, n, mode, o, units, p);
  if (rc == RADIC_OK) {
    std::lock_guard<std::mutex> lock(mu);
    if (cache.size() >= 4096) cache.clear();
    cache.emplace(key, *p);
  }
  return rc;
}

// sms_given / per_sm_given > 0 replace the device's SM count and the
// occupancy query (host-only planning).
int make_plan_uncached(int m, int n, int mode, const radic_options* o, unsigned long long units, SinglePlan* p,
                       int sms_given, int per_sm_given) {
  if (m < 1 || m > kMaxM || n < 1 || n > kMaxN || !valid_mode(mode)) return RADIC_EINVAL;
  radic_options d;
  std::memset(&d, 0, sizeof(d));
  if (o) d = *o;
  SinglePlan pl;
  pl.mode = mode;
  pl.m = m;
  pl.n = n;
  pl.total = (m <= n) ? binom_host(n, m) : 0ull;
  const int auto_limit = (mode == kModeExact) ? kThreadMaxMModp : 8;
  const int prefix_limit = (mode == kModeFp64)    ? kPrefixMaxMFp64
                           : (mode == kModeMixed) ? kPrefixMaxMFp32
                           : (mode == kModePair)  ? kPrefixMaxMPair
                                                  : kPrefixMaxMModp;
  int mapping = d.mapping;
  if (mapping == RADIC_MAP_AUTO) {
    if (m >= 3 && m <= prefix_limit && m <= n) mapping = RADIC_MAP_PREFIX;
    else mapping = (m <= auto_limit ? RADIC_MAP_THREAD : RADIC_MAP_GROUP);
  }
  if (mapping != RADIC_MAP_THREAD && mapping != RADIC_MAP_GROUP && mapping != RADIC_MAP_PREFIX) return RADIC_EINVAL;
  if (mode == kModePair && mapping != RADIC_MAP_PREFIX) return RADIC_EUNSUPPORTED;
  if (mapping == RADIC_MAP_THREAD && m > thread_limit(mode)) return RADIC_EUNSUPPORTED;
  if (mapping == RADIC_MAP_PREFIX && (m < 3 || m > prefix_limit || m > n)) return RADIC_EUNSUPPORTED;
  pl.mapping = mapping;
  if (mapping == RADIC_MAP_PREFIX) {
    if (d.prefix_depth != 0 && d.prefix_depth != 2 && d.prefix_depth != 3) return RADIC_EINVAL;
    const int lp = d.lanes_per_prefix;
    if (lp < 0 || lp > 32 || (lp & (lp - 1)) != 0) return RADIC_EINVAL;
    if (d.prefix_depth == 3 && m < 4) return RADIC_EUNSUPPORTED;
    pl.depth = d.prefix_depth ? d.prefix_depth : prefix_auto_depth(m, n, false);
  }
  if (mapping == RADIC_MAP_GROUP) {
    const int gw = d.group_width ? d.group_width : (m <= 16 ? 16 : 32);
    if ((gw != 16 && gw != 32) || gw < m) return RADIC_EINVAL;
    pl.group = gw;
  }
  const int max_threads = (mode == kModeExact || mapping == RADIC_MAP_PREFIX) ? 128 : 256;
  pl.threads = d.threads_per_block ? d.threads_per_block : 128;
  if (pl.threads < 32 || pl.threads > max_threads || pl.threads % 32) return RADIC_EINVAL;
  if (d.ranks_per_task < 0 || d.ranks_per_task > (1 << 30)) return RADIC_EINVAL;
  pl.flag_cap = d.flag_capacity ? d.flag_capacity : 32;
  if (pl.flag_cap < 1 || pl.flag_cap > (1 << 16)) return RADIC_EINVAL;
  pl.growth = d.growth_threshold > 0.0 ? d.growth_threshold : 64.0;
  pl.events = d.kernel_events;
  pl.smem = smem_of(pl);

  const int sms = sms_given > 0 ? sms_given : device_sm_count();
  const int per_sm = per_sm_given > 0 ? per_sm_given : blocks_per_sm(pl);
  if (sms <= 0) return RADIC_ECUDA;
  if (per_sm <= 0) return RADIC_EUNSUPPORTED;
  // Work split of Section 5: K processors (threads, or lane groups) each take
  // one contiguous run of about C(n,m)/K ranks.  K is the number of resident
  // processors of a full-occupancy grid, so every processor gets one task and
  // no SM waits on a tail; an explicit ranks_per_task overrides the run length.
  if (mapping == RADIC_MAP_PREFIX) return plan_prefix(pl, d, sms, per_sm, units, per_sm_given <= 0, p);
  // Floating-point groups: the split into runs is that of 512 threads per SM
  // whatever the kernel's registers leave resident (at 128 threads a block:
  // four blocks for groups of 16, three for groups of 32), because the binary32
  // sums of bounds round per run; the blocks beyond those resident even out the
  // tail (17 x 22: 485 us against 508 with runs for the resident blocks).
  const unsigned long long cap =
      (unsigned long long)sms * (mapping == RADIC_MAP_GROUP && mode != kModeExact ? 512 / pl.threads : per_sm);
  const unsigned long long per_block =
      (mapping == RADIC_MAP_THREAD) ? (unsigned long long)pl.threads : (unsigned long long)(pl.threads / pl.group);
  unsigned long long L = (unsigned long long)d.ranks_per_task;
  if (L == 0) {
    const unsigned long long procs = cap * per_block;
    L = (units + procs - 1) / procs;
    if (L < 1) L = 1;
  }
  pl.ranks_per_task = L;
  pl.tasks = (units + L - 1) / L;
  const unsigned long long need = (pl.tasks + per_block - 1) / per_block;
  unsigned long long blocks = need < cap ? need : cap;
  // Runs of single minors: a second wave of blocks would start every
  // elimination afresh; the resident groups take consecutive minors instead,
  // which resume it (22 x 25: 149 us in two waves, 117 now, 113 by a kernel
  // that left four blocks resident).  With runs of two and three minors the
  // second wave is the better one (26 x 29 199 us against 267).
  const unsigned long long resident = (unsigned long long)sms * per_sm;
  if (mapping == RADIC_MAP_GROUP && blocks > resident && L == 1) {
    const unsigned long long per = (blocks + resident - 1) / resident;
    blocks = (need + per - 1) / per;
  }
  if (d.blocks > 0) blocks = (unsigned long long)d.blocks;
  if (blocks < 1) blocks = 1;
  if (blocks > (1ull << 20)) return RADIC_EINVAL;
  pl.blocks = (int)blocks;
  pl.blocks2 = sms;
  layout_workspace(pl);
  *p = pl;
  return RADIC_OK;
}

void layout_workspace(SinglePlan& pl) {
  const int mode = pl.mode;
  const int n_warps = pl.blocks * pl.threads / 32;
  size_t off = mode == kModeExact ? kExactHeaderBytes : kHeaderBytes;
  pl.off_partials = off;
  off = align_up(off + (size_t)pl.blocks * sizeof(FpPartial), 256);
  if (mode == kModeMixed || mode == kModePair) {
    pl.off_partials2 = off;
    off = align_up(off + (size_t)pl.blocks2 * sizeof(FpPartial), 256);
    pl.off_flag_count = off;
    off = align_up(off + (size_t)n_warps * sizeof(int), 256);
    pl.off_flag_ranks = off;
    off = align_up(off + (size_t)n_warps * pl.flag_cap * sizeof(unsigned long long), 256);
  }
  if (mode == kModeExact) {
    pl.off_modp = off;
    off = align_up(off + (size_t)pl.blocks * kMaxPrimes * sizeof(uint32_t), 256);
  }
  pl.ws_bytes = off;
}

__global__ void k_zero_result(radic_result* out, int tier) {
  out->value = 0.0;
  out->abs_sum = 0.0;
  out->err_bound = 0.0;
  out->exact_lo = 0;
  out->exact_hi = 0;
  out->minors = 0;
  out->flagged = 0;
  out->status = RADIC_OK;
  out->n_primes = (tier == kModeExact) ? 1 : 0;
  out->tier = tier;
  out->exact_exp = 0;
  for (int i = 0; i < 5; ++i) out->reserved[i] = 0;
}

template <int M>
__global__ void k_unrank(int n, unsigned long long q0, unsigned long long count, int L, uint8_t* cols) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  uint64_t* binom = reinterpret_cast<uint64_t*>(smem_raw);
  build_binom(binom, n, M);
  const unsigned long long tasks = (count + L - 1) / L;
  const unsigned long long nthreads = (unsigned long long)gridDim.x * blockDim.x;
  for (unsigned long long t = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; t < tasks; t += nthreads) {
    unsigned long long q = q0 + t * L;
    const unsigned long long q1 = min(q + L, q0 + count);
    int c[M];
    unrank<M>(q, n, binom, M + 1, c);
    for (; q < q1; ++q) {
#pragma unroll
      for (int i = 0; i < M; ++i) cols[(q - q0) * M + i] = static_cast<uint8_t>(c[i]);
      if (q + 1 < q1) successor<M>(c, n);
    }
  }
}

template <int G>
__global__ void k_unrank_dyn(int n, int m, unsigned long long q0, unsigned long long count, int L, uint8_t* cols) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  uint64_t* binom = reinterpret_cast<uint64_t*>(smem_raw);
  build_binom(binom, n, m);
  const unsigned long long tasks = (count + L - 1) / L;
  const unsigned long long nthreads = (unsigned long long)gridDim.x * blockDim.x;
  for (unsigned long long t = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; t < tasks; t += nthreads) {
    unsigned long long q = q0 + t * L;
    const unsigned long long q1 = min(q + L, q0 + count);
    int c[G];
    unrank_dyn<G>(q, n, m, binom, m + 1, c);
    for (; q < q1; ++q) {
#pragma unroll
      for (int i = 0; i < G; ++i)
        if (i < m) cols[(q - q0) * m + i] = static_cast<uint8_t>(c[i]);
      if (q + 1 < q1) successor_dyn<G>(c, n, m);
    }
  }
}

const void* unrank_kernel(int m) {
  switch (m) {
    case 1: return reinterpret_cast<const void*>(&k_unrank<1>);
    case 2: return reinterpret_cast<const void*>(&k_unrank<2>);
    case 3: return reinterpret_cast<const void*>(&k_unrank<3>);
    case 4: return reinterpret_cast<const void*>(&k_unrank<4>);
    case 5: return reinterpret_cast<const void*>(&k_unrank<5>);
    case 6: return reinterpret_cast<const void*>(&k_unrank<6>);
    case 7: return reinterpret_cast<const void*>(&k_unrank<7>);
    case 8: return reinterpret_cast<const void*>(&k_unrank<8>);
    case 9: return reinterpret_cast<const void*>(&k_unrank<9>);
    case 10: return reinterpret_cast<const void*>(&k_unrank<10>);
    case 11: return reinterpret_cast<const void*>(&k_unrank<11>);
    case 12: return reinterpret_cast<const void*>(&k_unrank<12>);
    default: return nullptr;
  }
}

}  // namespace

int launch_unrank(int n, int m, unsigned long long q0, unsigned long long count, uint8_t* cols, int L,
                  cudaStream_t s) {
  const int sms = device_sm_count();
  if (sms <= 0) return RADIC_ECUDA;
  const unsigned long long tasks = (count + L - 1) / L;
  unsigned long long blocks = (tasks + 127) / 128;
  if (blocks > (unsigned long long)sms * 8) blocks = (unsigned long long)sms * 8;
  if (blocks < 1) blocks = 1;
  const size_t smem = (size_t)(n + 1) * (m + 1) * 8;
  unsigned long long qq = q0, cc = count;
  int nn = n, mm = m, ll = L;
  cudaError_t e;
  if (const void* k = unrank_kernel(m)) {
    void* params[] = {&nn, &qq, &cc, &ll, &cols};
    e = cudaLaunchKernel(k, dim3((unsigned)blocks), dim3(128), params, smem, s);
  } else {
    void* params[] = {&nn, &mm, &qq, &cc, &ll, &cols};
    const void* k2 = (m <= 16) ? reinterpret_cast<const void*>(&k_unrank_dyn<16>)
                               : reinterpret_cast<const void*>(&k_unrank_dyn<32>);
    e = cudaLaunchKernel(k2, dim3((unsigned)blocks), dim3(128), params, smem, s);
  }
  return e == cudaSuccess ? RADIC_OK : RADIC_ECUDA;
}

}  // namespace radic

using namespace radic;

extern "C" {

const char* radic_status_string(int status) {
  switch (status) {
    case RADIC_OK: return "ok";
    case RADIC_EINVAL: return "invalid argument";
    case RADIC_EOVERFLOW: return "exact value may exceed the prime budget";
    case RADIC_ECUDA: return "CUDA runtime error";
    case RADIC_ETIMEOUT: return "device-side wait timed out";
    case RADIC_EWORKSPACE: return "workspace missing, misaligned or too small";
    case RADIC_EUNSUPPORTED: return "unsupported combination of arguments";
    default: return "unknown status";
  }
}

int radic_version(void) { return 10000; }

int radic_primes(uint32_t* primes, int max_count) {
  if (!primes || max_count <= 0) return 0;
  const int k = max_count < kMaxPrimes ? max_count : kMaxPrimes;
  for (int i = 0; i < k; ++i) primes[i] = kPrimes[i];
  return k;
}

size_t radic_workspace_bytes(int m, int n, int mode, const radic_options* opts) {
  SinglePlan p;
  if (make_plan(m, n, mode, opts, (m <= n && n <= kMaxN && m >= 1) ? binom_host(n, m) : 0ull, &p) != RADIC_OK)
    return 0;
  return p.ws_bytes;
}

int radic_plan_info(int m, int n, int mode, const radic_options* opts, int64_t* info, int count) {
  if ((!info && count > 0) || count < 0 || count > RADIC_PLAN_INFO_COUNT) return RADIC_EINVAL;
  SinglePlan p;
  const int rc =
      make_plan(m, n, mode, opts, (m <= n && n <= kMaxN && m >= 1 && n >= 1) ? binom_host(n, m) : 0ull, &p);
  if (rc != RADIC_OK) return rc;
  int64_t v[RADIC_PLAN_INFO_COUNT];
  v[0] = p.mapping;
  v[1] = (p.mapping == RADIC_MAP_PREFIX) ? p.depth : 0;
  v[2] = (p.mapping == RADIC_MAP_GROUP) ? p.group : 0;
  v[3] = p.threads;
  const bool subtree = p.mapping == RADIC_MAP_PREFIX && mode == kModeExact;
  v[4] = subtree ? p.sub_blocks[0] : p.blocks;
  v[5] = subtree                             ? (int64_t)p.stab[0].total_tasks
         : (p.mapping == RADIC_MAP_PREFIX) ? (int64_t)p.ptab.total_tasks
                                             : (int64_t)p.ranks_per_task;
  v[6] = subtree ? (int64_t)smem_modp(p, kModpDet) : (int64_t)p.smem;
  v[7] = (int64_t)p.ws_bytes;
  v[8] = subtree ? p.subtree[0] : 0;
  for (int i = 0; i < count; ++i) info[i] = v[i];
  return RADIC_OK;
}

int radic_prefix_plan_host(int m, int n, int mode, const radic_options* opts, int sms, int blocks_per_sm,
                           int64_t* info, int count) {
  if (!info || sms < 1 || blocks_per_sm < 1 || count < 8 + 4 * n) return RADIC_EINVAL;
  if (m < 1 || n < 1 || n > kMaxN || m > n) return RADIC_EINVAL;
  radic_options d;
  std::memset(&d, 0, sizeof(d));
  if (opts) d = *opts;
  d.mapping = RADIC_MAP_PREFIX;
  SinglePlan p;
  const int rc = make_plan_uncached(m, n, mode, &d, binom_host(n, m), &p, sms, blocks_per_sm);
  if (rc != RADIC_OK) return rc;
  const PrefixTable& t = p.ptab;
  for (int i = 0; i < count; ++i) info[i] = 0;
  info[0] = p.depth;
  info[1] = static_cast<int64_t>(t.total_tasks);
  info[2] = p.blocks;
  info[3] = t.v_lo;
  info[4] = t.v_hi;
  info[5] = t.dynamic;
  for (int v = t.v_lo; v <= t.v_hi; ++v) {
    info[8 + 4 * v + 0] = static_cast<int64_t>(t.count[v]);
    info[8 + 4 * v + 1] = static_cast<int64_t>(t.run[v]);
    info[8 + 4 * v + 2] = t.lanes[v];
    info[8 + 4 * v + 3] = static_cast<int64_t>(t.task_start[v]);
  }
  return RADIC_OK;
}

int radic_det(const void* A, int m, int n, int64_t lda, int dtype, int mode, const radic_options* opts,
              radic_result* out, void* workspace, size_t workspace_bytes, void* stream) {
  if (!A || !out || lda < n || !valid_dtype(dtype)) return RADIC_EINVAL;
  SinglePlan p;
  const unsigned long long total = (m >= 1 && n >= 1 && m <= n && n <= kMaxN) ? binom_host(n, m) : 0ull;
  const int rc = make_plan(m, n, mode, opts, total, &p);
  if (rc != RADIC_OK) return rc;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if (p.total == 0) {
    k_zero_result<<<1, 1, 0, s>>>(out, mode);
    return cudaGetLastError() == cudaSuccess ? RADIC_OK : RADIC_ECUDA;
  }
  if (!workspace || (reinterpret_cast<uintptr_t>(workspace) & 255u) || workspace_bytes < p.ws_bytes)
    return RADIC_EWORKSPACE;
  unsigned char* ws = static_cast<unsigned char*>(workspace);
  if (cudaMemsetAsync(ws, 0, mode == kModeExact ? kExactHeaderBytes : kHeaderBytes, s) != cudaSuccess)
    return RADIC_ECUDA;
  SingleArgs a;
  std::memset(&a, 0, sizeof(a));
  a.A = A;
  a.lda = lda;
  a.dtype = dtype;
  a.m = m;
  a.n = n;
  a.ranks_per_task = p.ranks_per_task;
  a.total = p.total;
  a.tasks = p.tasks;
  a.growth = p.growth;
  a.flag_cap = p.flag_cap;
  a.flag_prefix = (p.mapping == RADIC_MAP_PREFIX) ? m - p.depth : 0;
  a.n_warps = p.blocks * p.threads / 32;
  a.hdr = reinterpret_cast<WsHeader*>(ws);
  a.partials = reinterpret_cast<FpPartial*>(ws + p.off_partials);
  a.partials2 = reinterpret_cast<FpPartial*>(ws + p.off_partials2);
  a.flag_count = reinterpret_cast<int*>(ws + p.off_flag_count);
  a.flag_ranks = reinterpret_cast<unsigned long long*>(ws + p.off_flag_ranks);
  a.modp_partials = reinterpret_cast<uint32_t*>(ws + p.off_modp);
  a.residue_sums = reinterpret_cast<unsigned long long*>(ws + kHeaderBytes);
  a.out = out;
  int r;
  switch (mode) {
    case kModeFp64: r = launch_fp64(p, a, s); break;
    case kModeMixed: r = launch_mixed(p, a, s); break;
    case kModePair: r = launch_pair(p, a, s); break;
    default: r = launch_modp(p, a, s); break;
  }
  return r;
}

size_t radic_wide_workspace_bytes(int m, int n, const radic_options* opts) {
  SinglePlan p;
  const unsigned long long total = (m >= 1 && n >= 1 && m <= n && n <= kMaxN) ? binom_host(n, m) : 0ull;
  if (make_plan(m, n, kModeExact, opts, total, &p) != RADIC_OK) return 0;
  // the EXACT workspace, then the residues of every pass (kWidePrimes words,
  // then needed, exponent and status)
  return align_up(p.ws_bytes, 256) + 256;
}

int radic_det_exact_wide(const void* A, int m, int n, int64_t lda, int dtype, const radic_options* opts,
                         radic_wide_result* out, void* workspace, size_t workspace_bytes, void* stream) {
  if (!A || !out || lda < n || !valid_dtype(dtype)) return RADIC_EINVAL;
  SinglePlan p;
  const unsigned long long total = (m >= 1 && n >= 1 && m <= n && n <= kMaxN) ? binom_host(n, m) : 0ull;
  const int rc = make_plan(m, n, kModeExact, opts, total, &p);
  if (rc != RADIC_OK) return rc;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if (p.total == 0) return launch_wide_crt(nullptr, out, 0ull, s);
  const size_t off_wide = align_up(p.ws_bytes, 256);
  if (!workspace || (reinterpret_cast<uintptr_t>(workspace) & 255u) || workspace_bytes < off_wide + 256)
    return RADIC_EWORKSPACE;
  unsigned char* ws = static_cast<unsigned char*>(workspace);
  uint32_t* wide = reinterpret_cast<uint32_t*>(ws + off_wide);
  // the prefix mapping takes every prime in one launch and reconstructs in its
  // last block; the per-minor mappings take RADIC_MAX_PRIMES per pass
  const bool subtree = p.mapping == RADIC_MAP_PREFIX;
  for (int base = 0; base < kWidePrimes; base += subtree ? kWidePrimes : kMaxPrimes) {
    if (cudaMemsetAsync(ws, 0, kExactHeaderBytes, s) != cudaSuccess) return RADIC_ECUDA;
    SingleArgs a;
    std::memset(&a, 0, sizeof(a));
    a.A = A;
    a.lda = lda;
    a.dtype = dtype;
    a.m = m;
    a.n = n;
    a.ranks_per_task = p.ranks_per_task;
    a.total = p.total;
    a.tasks = p.tasks;
    a.growth = p.growth;
    a.n_warps = p.blocks * p.threads / 32;
    a.hdr = reinterpret_cast<WsHeader*>(ws);
    a.modp_partials = reinterpret_cast<uint32_t*>(ws + p.off_modp);
    a.prime_base = base;
    a.wide = wide;
    a.residue_sums = reinterpret_cast<unsigned long long*>(ws + kHeaderBytes);
    if (subtree) a.wide_out = out;
    const int r = launch_modp(p, a, s);
    if (r != RADIC_OK) return r;
  }
  if (subtree) return RADIC_OK;
  return launch_wide_crt(wide, out, p.total, s);
}

int radic_terms(const void* A, int m, int n, int64_t lda, int dtype, int mode, const radic_options* opts,
                uint64_t q0, uint64_t count, void* terms, void* stream) {
  if (!A || !terms || lda < n || !valid_dtype(dtype)) return RADIC_EINVAL;
  if (mode == kModeExact && (dtype == kF32 || dtype == kF64)) return RADIC_EINVAL;
  if (m < 1 || n < 1 || m > n || n > kMaxN || m > kMaxM) return RADIC_EINVAL;
  const unsigned long long total = binom_host(n, m);
  if (q0 >= total || count > total - q0) return RADIC_EINVAL;
  if (count == 0) return RADIC_OK;
  SinglePlan p;
  const int rc = make_plan(m, n, mode, opts, count, &p);
  if (rc != RADIC_OK) return rc;
  SingleArgs a;
  std::memset(&a, 0, sizeof(a));
  a.A = A;
  a.lda = lda;
  a.dtype = dtype;
  a.m = m;
  a.n = n;
  a.ranks_per_task = p.ranks_per_task;
  a.total = total;
  a.tasks = p.tasks;
  a.growth = p.growth;
  a.flag_cap = p.flag_cap;
  a.q0 = q0;
  a.count = count;
  a.terms = terms;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  switch (mode) {
    case kModeFp64: return launch_fp64(p, a, s);
    case kModeMixed: return launch_mixed(p, a, s);
    case kModePair: return launch_pair(p, a, s);
    default: return launch_modp(p, a, s);
  }
}

int radic_unrank(int n, int m, uint64_t q0, uint64_t count, uint8_t* cols, const radic_options* opts,
                 void* stream) {
  if (!cols || m < 1 || n < 1 || m > n || n > kMaxN || m > kMaxM) return RADIC_EINVAL;
  const unsigned long long total = binom_host(n, m);
  if (q0 >= total || count > total - q0) return RADIC_EINVAL;
  if (count == 0) return RADIC_OK;
  const int L = (opts && opts->ranks_per_task > 0) ? opts->ranks_per_task : 64;
  return launch_unrank(n, m, q0, count, cols, L, static_cast<cudaStream_t>(stream));
}

struct radic_graph {
  cudaGraph_t graph = nullptr;
  cudaGraphExec_t exec = nullptr;
};

int radic_graph_create(const void* A, int m, int n, int64_t lda, int dtype, int mode, const radic_options* opts,
                       radic_result* out, void* workspace, size_t workspace_bytes, radic_graph** graph) {
  if (!graph) return RADIC_EINVAL;
  *graph = nullptr;
  cudaStream_t cs;
  if (cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking) != cudaSuccess) return RADIC_ECUDA;
  radic_graph* g = new (std::nothrow) radic_graph;
  int rc = g ? RADIC_OK : RADIC_EINVAL;
  if (rc == RADIC_OK && cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal) != cudaSuccess) rc = RADIC_ECUDA;
  if (rc == RADIC_OK) {
    const int r = radic_det(A, m, n, lda, dtype, mode, opts, out, workspace, workspace_bytes, cs);
    const cudaError_t e = cudaStreamEndCapture(cs, &g->graph);
    if (r != RADIC_OK) rc = r;
    else if (e != cudaSuccess) rc = RADIC_ECUDA;
  }
  if (rc == RADIC_OK && cudaGraphInstantiate(&g->exec, g->graph, 0) != cudaSuccess) rc = RADIC_ECUDA;
  cudaStreamDestroy(cs);
  if (rc != RADIC_OK) {
    if (g) {
      if (g->exec) cudaGraphExecDestroy(g->exec);
      if (g->graph) cudaGraphDestroy(g->graph);
      delete g;
    }
    return rc;
  }
  *graph = g;
  return RADIC_OK;
}

int radic_graph_launch(radic_graph* graph, void* stream) {
  if (!graph || !graph->exec) return RADIC_EINVAL;
  return cudaGraphLaunch(graph->exec, static_cast<cudaStream_t>(stream)) == cudaSuccess ? RADIC_OK : RADIC_ECUDA;
}

int radic_graph_destroy(radic_graph* graph) {
  if (!graph) return RADIC_OK;
  if (graph->exec) cudaGraphExecDestroy(graph->exec);
  if (graph->graph) cudaGraphDestroy(graph->graph);
  delete graph;
  return RADIC_OK;
}

}  // extern "C"
