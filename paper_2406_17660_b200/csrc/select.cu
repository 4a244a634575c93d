// grass_select: compute_P of the GRASS paper (Section 3.2) -- Top-r; sampling
// with replacement from q ~ norm, norm^2 or uniform with rho_j = 1/sqrt(r q_sigma_j);
// and the same three distributions without replacement with rho = 1.
//
// m is at most a few tens of thousands and r at most a few thousand, so these are
// latency-bound kernels of 1024 threads a CTA; everything they need to agree on is
// agreed on through shared memory and scans, and the output order (ascending row) is
// produced by scans in row order, so the result does not depend on thread scheduling.
//
// Ranking (Top-r and without replacement) costs every row a score and six looks, so it runs on a
// cluster of eight CTAs, about two rows a thread, that exchange histograms and counts through
// distributed shared memory: 13824 rows without replacement took 37 us on one CTA, 14 on eight; up to
// 4096 rows one CTA is as fast for Top-r (10 us at 4096, 12 on a cluster: six cluster barriers).  A score costs a Philox
// block and an fp64 logarithm, so without replacement the cluster pays from 2049 rows (us on one CTA and on the cluster, r = m/64
// to m/2: 1025 rows 7.6 to 8.0 and 8.7 to 8.9, 1900 8.6 to 9.2 and 8.8 to 9.0, 2049 9.4 to 10.3 and 8.9 to 9.1, 4096 12.4 to 13.8 and
// 9.1 to 9.2).
// Sampling with replacement is a serial chain (running sum, search, expansion) and stays on one.
//
//   Top-r: the fp32 bit pattern of a non-negative float orders like the float,
//   so the r-th largest norm is found by a 4-pass, 8-bit-digit radix select.
//   Rows above the threshold are taken; rows equal to it are taken lowest row
//   first until r are chosen.
//
//   Without replacement: every row gets an exponential-race score (one Philox
//   word per row), and the Top-r machinery ranks the fp32 scores.
//
//   With replacement: fp64 inclusive running sum of the weights (block scan in
//   row order), then one thread per draw: Philox4x32-10 word -> u -> binary
//   search for min{k : c_k > u S}; hits are counted per row with integer
//   atomics (order-independent), and a last scan over the counts writes the
//   rows in ascending order with their rho.
#include "common.cuh"
#include "sm100_ptx.cuh"

namespace grass {
namespace {

constexpr int kThreads = 1024;
constexpr int kWarps = kThreads / 32;
constexpr uint32_t kStreamTag = 0x47524153u;

// ---- Philox4x32-10 (Salmon et al., SC'11) ----
__device__ __forceinline__ uint4 philox4x32_10(uint4 c, uint2 k) {
#pragma unroll
  for (int round = 0; round < 10; ++round) {
    const uint32_t hi0 = __umulhi(0xD2511F53u, c.x), lo0 = 0xD2511F53u * c.x;
    const uint32_t hi1 = __umulhi(0xCD9E8D57u, c.z), lo1 = 0xCD9E8D57u * c.z;
    c = make_uint4(hi1 ^ c.y ^ k.x, lo1, hi0 ^ c.w ^ k.y, lo0);
    k.x += 0x9E3779B9u;
    k.y += 0xBB67AE85u;
  }
  return c;
}

__device__ __forceinline__ uint32_t norm_key(float v) {
  return v == 0.f ? 0u : __float_as_uint(v);  // folds -0 into +0
}

__host__ __device__ __forceinline__ bool is_nr(int method) {
  return method == GRASS_SEL_MULTINOMIAL_NORM_NR || method == GRASS_SEL_MULTINOMIAL_NORM2_NR ||
         method == GRASS_SEL_UNIFORM_NR;
}
// Unnormalised q of the three sampling distributions (Section 3.2 A), in fp64.
__device__ __forceinline__ double sampling_weight(int method, float lambda) {
  const double l = static_cast<double>(lambda);
  if (method == GRASS_SEL_MULTINOMIAL_NORM2 || method == GRASS_SEL_MULTINOMIAL_NORM2_NR) return l * l;
  if (method == GRASS_SEL_UNIFORM || method == GRASS_SEL_UNIFORM_NR) return 1.0;
  return l;
}

struct SelectArgs {
  const float* norms;
  int m, r, method;
  uint32_t seed_lo, seed_hi, layer_id, epoch;
  int32_t* idx;
  float* rho;
  double* cdf;    // [m]   (sampling methods)
  int* counts;    // [m]   (sampling methods)
  int* status;
  int stage_norms;   // dynamic shared memory holds a copy of the norms (m floats) ...
  int stage_counts;  // ... followed by the hit counters (m ints)
  int stage_cdf;     // ... followed by the running sum (m doubles)
};

__device__ __forceinline__ uint32_t peer_smem(const void* p, int rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(ptx::smem_u32(p)), "r"(rank));
  return r;
}
__device__ __forceinline__ int ld_peer(uint32_t addr) {
  int v;
  asm volatile("ld.shared::cluster.s32 %0, [%1];" : "=r"(v) : "r"(addr));
  return v;
}

// Top-r and the -NR methods: the r largest keys, emitted in ascending row order.  The grid is one
// cluster; CTA c owns rows [c * rows_per_cta, ..).  Keys live in shared memory (stage_norms) or are read
// again from the norms / the scores in the workspace.
__global__ void __launch_bounds__(kThreads) select_rank_kernel(SelectArgs a, int rows_per_cta) {
  extern __shared__ __align__(16) float s_dyn[];
  __shared__ int s_hist[4][256], s_sum[256];
  __shared__ int s_bad, s_positive;                 // read by the whole cluster
  __shared__ int s_totals[2];                       // this CTA's rows equal to / above the threshold
  __shared__ uint32_t s_prefix;
  __shared__ int s_need, s_ok;
  __shared__ int s_eq_base[kWarps], s_out_base[kWarps];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int rank = blockIdx.x, ctas = gridDim.x;
  const int row0 = rank * rows_per_cta;
  const int rows = a.m - row0 < rows_per_cta ? (a.m - row0 > 0 ? a.m - row0 : 0) : rows_per_cta;
  const bool nr = is_nr(a.method);
  grid_dep_wait();
  if (tid < 256) {
#pragma unroll
    for (int p = 0; p < 4; ++p) s_hist[p][tid] = 0;
  }
  if (tid == 0) { s_bad = 0; s_positive = 0; s_prefix = 0u; s_need = a.r; }
  __syncthreads();

  // ---- every norm finite and >= 0; keys: the norms, or (without replacement) an exponential race
  // (Efraimidis & Spirakis): row k scores w_k / (-log u_k), u_k = (word_k + 1/2) 2^-32; the r
  // largest scores are distributed as r successive draws without replacement.  Scores are rounded to
  // fp32 and ranked as such. ----
  float* scores = a.stage_norms ? s_dyn : reinterpret_cast<float*>(a.cdf) + row0;
  const float* keys = a.stage_norms ? s_dyn : (nr ? scores : a.norms + row0);
  int bad = 0, positive = 0;
  for (int i0 = tid; i0 < rows; i0 += 4 * kThreads) {
    float v[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) v[u] = i0 + u * kThreads < rows ? a.norms[row0 + i0 + u * kThreads] : 0.f;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int i = i0 + u * kThreads;
      if (i >= rows) continue;
      const int k = row0 + i;
      if (!(v[u] >= 0.f) || isinf(v[u])) bad = k + 1;
      if (nr) {
        const uint4 blk = philox4x32_10(make_uint4(static_cast<uint32_t>(k >> 2), a.layer_id, a.epoch,
                                                   kStreamTag),
                                        make_uint2(a.seed_lo, a.seed_hi));
        const uint32_t sel = k & 3;
        const uint32_t word = sel == 0 ? blk.x : sel == 1 ? blk.y : sel == 2 ? blk.z : blk.w;
        const double uk = (static_cast<double>(word) + 0.5) * 0x1p-32;
        const double w = sampling_weight(a.method, v[u]);
        scores[i] = static_cast<float>(w / -log(uk));
        positive += w > 0.0;
      } else if (a.stage_norms) {
        s_dyn[i] = v[u];
      }
    }
  }
  if (bad) atomicMax(&s_bad, bad);
  if (nr) {
    positive = __reduce_add_sync(0xffffffffu, positive);
    if (lane == 0) atomicAdd(&s_positive, positive);
  }
  __syncthreads();

  // ---- radix select of the r-th largest key, 8 bits a pass ----
  bool ok = true;
  for (int pass = 3; pass >= 0; --pass) {
    const int shift = pass * 8;
    const uint32_t prefix = s_prefix;
    const uint32_t himask = pass == 3 ? 0u : (0xffffffffu << (shift + 8));
    int* hist = s_hist[pass];
    for (int i = tid; i < rows; i += kThreads) {
      const uint32_t key = norm_key(keys[i]);
      // norms share their leading bytes, so most of a warp lands in one bin: one atomic per
      // distinct bin per warp instead of one per row
      const bool in = (key & himask) == prefix;
      const uint32_t voters = __ballot_sync(__activemask(), in);
      if (in) {
        const uint32_t bin = (key >> shift) & 0xff;
        const uint32_t peers = __match_any_sync(voters, bin);
        if (lane == __ffs(peers) - 1) atomicAdd(&hist[bin], __popc(peers));
      }
    }
    // the cluster's histogram: thread t sums bin t over the CTAs, all loads in flight
    if (ctas > 1) {
      __syncwarp();
      ptx::cluster_sync_all();             // every CTA's histogram (and flags) of this pass
      if (tid < 256) {
        int v[8];
#pragma unroll
        for (int c = 0; c < 8; ++c) v[c] = c < ctas ? ld_peer(peer_smem(hist + tid, c)) : 0;
        s_sum[tid] = ((v[0] + v[1]) + (v[2] + v[3])) + ((v[4] + v[5]) + (v[6] + v[7]));
      }
      __syncthreads();
      hist = s_sum;
    } else {
      __syncthreads();
    }
    if (warp == 0) {
      // digit d with (keys above d) < need <= (keys at or above d), found by one warp in every CTA:
      // lane l owns bins 8l..8l+7 of the cluster's sum; a suffix scan over the lanes, then a look
      // inside one lane's bins
      int h[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) h[i] = hist[8 * lane + i];
      int mine = 0;
#pragma unroll
      for (int i = 0; i < 8; ++i) mine += h[i];
      int incl = mine;                     // keys in this lane's bins and all higher lanes'
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int dn = __shfl_down_sync(0xffffffffu, incl, o);
        if (lane + o < 32) incl += dn;
      }
      const int need = s_need;
      const int above = incl - mine;       // keys in higher lanes' bins
      const bool here = above < need && need <= incl;   // true in exactly one lane
      if (here) {
        int rem = need - above, d = 7;
        for (; d > 0; --d) {
          if (h[d] >= rem) break;
          rem -= h[d];
        }
        s_need = rem;                      // how many to take among keys with this digit
        s_prefix = prefix | (static_cast<uint32_t>(8 * lane + d) << shift);
      }
      if (pass == 3) {
        int worst = lane < ctas ? ld_peer(peer_smem(&s_bad, lane)) : 0;
        int pos = lane < ctas ? ld_peer(peer_smem(&s_positive, lane)) : 0;
        worst = __reduce_max_sync(0xffffffffu, worst);
        pos = __reduce_add_sync(0xffffffffu, pos);
        if (lane == 0) {
          s_ok = worst == 0 && (!nr || pos >= a.r);
          if (!s_ok && rank == 0) record_status(a.status, GRASS_ERR_DEGENERATE, worst != 0 ? worst - 1 : pos);
        }
      }
    }
    __syncthreads();
    if (pass == 3) ok = s_ok != 0;
    if (!ok) break;                        // the same decision in every CTA
  }
  grid_dep_launch();
  if (ok) {
    const uint32_t tau = s_prefix;         // key of the r-th largest norm
    const int need_eq = s_need;            // rows equal to tau to take, lowest row first
    // ---- emit in ascending row order.  Each warp owns a contiguous segment of the CTA's rows; one
    // counting pass, a scan over the warps' totals and the CTAs', one writing pass. ----
    const int seg = ((rows_per_cta + kWarps - 1) / kWarps + 31) & ~31;   // rows per warp, multiple of 32
    const int i_begin = warp * seg < rows ? warp * seg : rows, i_end = i_begin + seg < rows ? i_begin + seg : rows;
    int n_eq = 0, n_gt = 0;
    for (int i0 = i_begin; i0 < i_end; i0 += 32) {
      const int i = i0 + lane;
      const uint32_t key = i < i_end ? norm_key(keys[i]) : 0u;
      n_eq += __popc(__ballot_sync(0xffffffffu, i < i_end && key == tau));
      n_gt += __popc(__ballot_sync(0xffffffffu, i < i_end && key > tau));
    }
    if (lane == 0) { s_eq_base[warp] = n_eq; s_out_base[warp] = n_gt; }
    __syncthreads();
    if (warp == 0) {
      const int eq = __reduce_add_sync(0xffffffffu, s_eq_base[lane]);
      const int gt = __reduce_add_sync(0xffffffffu, s_out_base[lane]);
      if (lane == 0) { s_totals[0] = eq; s_totals[1] = gt; }
    }
    __syncwarp();
    if (ctas > 1) ptx::cluster_sync_all();               // every CTA's totals
    if (warp == 0) {
      // rows selected in the CTAs before this one: theirs above tau, and their share of the equal ones
      const int eq_c = lane < rank ? ld_peer(peer_smem(&s_totals[0], lane)) : 0;
      const int gt_c = lane < rank ? ld_peer(peer_smem(&s_totals[1], lane)) : 0;
      const int eq_before = __reduce_add_sync(0xffffffffu, eq_c);
      const int gt_before = __reduce_add_sync(0xffffffffu, gt_c);
      const int out_before = gt_before + (eq_before < need_eq ? eq_before : need_eq);
      // exclusive prefix of the eq counts, then of the selected counts, over the 32 warps
      const int eq = s_eq_base[lane], gt = s_out_base[lane];
      int eq_incl = eq;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int up = __shfl_up_sync(0xffffffffu, eq_incl, o);
        if (lane >= o) eq_incl += up;
      }
      const int eq_excl = eq_before + eq_incl - eq;
      int take = need_eq - eq_excl;                    // equal rows this warp may still take
      take = take < 0 ? 0 : (take > eq ? eq : take);
      const int sel = gt + take;
      int sel_incl = sel;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int up = __shfl_up_sync(0xffffffffu, sel_incl, o);
        if (lane >= o) sel_incl += up;
      }
      s_eq_base[lane] = eq_excl;
      s_out_base[lane] = out_before + sel_incl - sel;
    }
    __syncthreads();
    int eq_base = s_eq_base[warp], out_base = s_out_base[warp];
    const uint32_t lt_mask = (1u << lane) - 1u;
    for (int i0 = i_begin; i0 < i_end; i0 += 32) {
      const int i = i0 + lane;
      const uint32_t key = i < i_end ? norm_key(keys[i]) : 0u;
      const bool is_eq = i < i_end && key == tau, is_gt = i < i_end && key > tau;
      const uint32_t eq_bits = __ballot_sync(0xffffffffu, is_eq);
      const bool sel = is_gt || (is_eq && eq_base + __popc(eq_bits & lt_mask) < need_eq);
      const uint32_t sel_bits = __ballot_sync(0xffffffffu, sel);
      if (sel) {
        const int pos = out_base + __popc(sel_bits & lt_mask);
        a.idx[pos] = row0 + i;
        a.rho[pos] = 1.f;
      }
      eq_base += __popc(eq_bits);
      out_base += __popc(sel_bits);
    }
  }
  __syncwarp();
  if (ctas > 1) ptx::cluster_sync_all();   // no CTA leaves while another may read its shared memory
}

// With replacement.
__global__ void __launch_bounds__(kThreads) select_kernel(SelectArgs a) {
  extern __shared__ __align__(16) float s_dyn[];   // staged norms / scores, then hit counters
  __shared__ int s_flag;
  const int tid = threadIdx.x;
  const int m = a.m, r = a.r;
  grid_dep_wait();

  // ---- validate: every norm finite and >= 0 ----
  if (tid == 0) s_flag = 0;
  __syncthreads();
  {
    // the one pass that reads global memory: 8 loads in flight per thread, not one at a time
    int bad = 0;
    for (int k0 = tid; k0 < m; k0 += 8 * kThreads) {
      float v[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int k = k0 + u * kThreads;
        v[u] = k < m ? a.norms[k] : 0.f;
      }
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int k = k0 + u * kThreads;
        if (k < m) {
          if (a.stage_norms) s_dyn[k] = v[u];   // every later pass reads shared memory, not L2
          if (!(v[u] >= 0.f) || isinf(v[u])) bad = k + 1;
        }
      }
    }
    if (bad) atomicMax(&s_flag, bad);
  }
  __syncthreads();
  if (s_flag != 0) {
    if (tid == 0) record_status(a.status, GRASS_ERR_DEGENERATE, s_flag - 1);
    return;
  }

  const float* nrm = a.stage_norms ? s_dyn : a.norms;
  int* counts = a.stage_counts ? reinterpret_cast<int*>(s_dyn + ((m + 3) & ~3)) : a.counts;
  double* cdf = a.stage_cdf ? reinterpret_cast<double*>(s_dyn + 2 * ((m + 3) & ~3)) : a.cdf;

  // ---- with replacement: inverse CDF of the sampling weights.  A two-pass
  // scheme: a warp owns a contiguous segment of rows, sums it, one scan over the 32 warp
  // totals gives every segment its base, and a second pass writes the running sum. ----
  const int lane = tid & 31, warp = tid >> 5;
  const int seg = ((m + kWarps - 1) / kWarps + 31) & ~31;
  const int k_begin = warp * seg, k_end = k_begin + seg < m ? k_begin + seg : m;
  __shared__ double s_wbase[kWarps];
  __shared__ double s_total;
  __shared__ int s_cbase[kWarps];
  // local[k] = running sum inside the segment (warp scan per 32 rows, carried across the
  // segment); cdf[k] = base[warp] + local[k] with base[w + 1] = base[w] + local total of w added
  // by one thread in order.  A shuffle scan adds the same terms in a different order in every
  // lane, so neighbouring entries can disagree in the last bit; what a draw must never do is
  // land on a row of zero weight (rho would be infinite).  Therefore a zero-weight row takes
  // the entry of the nearest row of positive weight before it, bit for bit (0 if the slice has
  // none, which makes it equal to the previous slice's last entry): cdf[k] > target can then
  // first become true only at a row of positive weight.
  auto slice_scan = [&](int k0) {
    const int k = k0 + lane;
    const double w = k < k_end ? sampling_weight(a.method, nrm[k]) : 0.0;
    double v = w;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const double up = __shfl_up_sync(0xffffffffu, v, o);
      if (lane >= o) v += up;
    }
    const uint32_t positive = __ballot_sync(0xffffffffu, w > 0.0);
    const uint32_t at_or_before = positive & (0xffffffffu >> (31 - lane));
    const int src = at_or_before != 0u ? 31 - __clz(at_or_before) : 0;
    const double taken = __shfl_sync(0xffffffffu, v, src);
    return at_or_before != 0u ? taken : 0.0;
  };
  {
    double run = 0.0;
    for (int k0 = k_begin; k0 < k_end; k0 += 32)
      run = run + __shfl_sync(0xffffffffu, slice_scan(k0), 31);
    if (lane == 0) s_wbase[warp] = run;
  }
  __syncthreads();
  if (tid == 0) {
    double base = 0.0;
    for (int w = 0; w < kWarps; ++w) {
      const double t = s_wbase[w];
      s_wbase[w] = base;
      base = base + t;
    }
    s_total = base;
  }
  __syncthreads();
  const double S = s_total;
  if (!(S > 0.0)) {
    if (tid == 0) record_status(a.status, GRASS_ERR_DEGENERATE, -1);
    return;
  }
  {
    const double base = s_wbase[warp];
    double run = 0.0;
    for (int k0 = k_begin; k0 < k_end; k0 += 32) {
      const int k = k0 + lane;
      const double v = slice_scan(k0);
      if (k < k_end) {
        cdf[k] = base + (run + v);
        counts[k] = 0;
      }
      run = run + __shfl_sync(0xffffffffu, v, 31);
    }
  }
  __syncthreads();  // cdf and counts visible block-wide (same CTA: global writes + barrier)
  for (int j = tid; j < r; j += kThreads) {
    const uint4 blk = philox4x32_10(make_uint4(static_cast<uint32_t>(j >> 2), a.layer_id, a.epoch,
                                               kStreamTag),
                                    make_uint2(a.seed_lo, a.seed_hi));
    const uint32_t sel = j & 3;
    const uint32_t word = sel == 0 ? blk.x : sel == 1 ? blk.y : sel == 2 ? blk.z : blk.w;
    const double target = (static_cast<double>(word) * 0x1p-32) * S;
    int lo = 0, hi = m - 1;                  // first k with cdf[k] > target
    while (lo < hi) {
      const int mid = (lo + hi) >> 1;
      if (cdf[mid] > target) hi = mid; else lo = mid + 1;
    }
    // (the entries of zero-weight rows repeat their predecessor's, so lo has positive weight;
    // the loop below only guards the very last rows when the target rounds up to the total)
    while (lo > 0 && !(sampling_weight(a.method, nrm[lo]) > 0.0)) --lo;
    atomicAdd(&counts[lo], 1);
  }
  __syncthreads();
  grid_dep_launch();
  // expand the hit counts in row order: per-warp totals, one scan, one writing pass
  {
    int run = 0;
    for (int k0 = k_begin; k0 < k_end; k0 += 32) {
      const int k = k0 + lane;
      int c = k < k_end ? counts[k] : 0;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
      run += c;
    }
    if (lane == 0) s_cbase[warp] = run;
  }
  __syncthreads();
  if (warp == 0) {
    const int mine = s_cbase[lane];
    int incl = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int up = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += up;
    }
    s_cbase[lane] = incl - mine;
  }
  __syncthreads();
  int out_base = s_cbase[warp];
  for (int k0 = k_begin; k0 < k_end; k0 += 32) {
    const int k = k0 + lane;
    const int cnt = k < k_end ? counts[k] : 0;
    int incl = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int up = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += up;
    }
    if (cnt > 0) {
      const double q = sampling_weight(a.method, nrm[k]) / S;
      const float rho = static_cast<float>(1.0 / sqrt(static_cast<double>(r) * q));
      const int pos = out_base + incl - cnt;
      for (int i = 0; i < cnt; ++i) {
        a.idx[pos + i] = k;
        a.rho[pos + i] = rho;
      }
    }
    out_base += __shfl_sync(0xffffffffu, incl, 31);
  }
}

constexpr size_t kSelectBudget = 200 * 1024;     // dynamic shared memory

template <typename K>
int allow_smem(K kernel, bool (&done)[64]) {
  int dev = 0;
  GRASS_CUDA_TRY(cudaGetDevice(&dev));
  if (dev >= 0 && dev < 64 && !done[dev]) {
    GRASS_CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                        static_cast<int>(kSelectBudget)));
    done[dev] = true;
  }
  return GRASS_OK;
}

// Ranking: eight CTAs (the portable cluster size) from 4097 rows up, 2049 where rows are scored, else one.
int launch_rank(SelectArgs& a, cudaStream_t s) {
  const int ctas = a.m > (is_nr(a.method) ? 2 : 4) * kThreads ? 8 : 1;
  const int rows = static_cast<int>(round_up((static_cast<size_t>(a.m) + ctas - 1) / ctas, 32));
  a.stage_norms = rows * sizeof(float) <= kSelectBudget;
  static bool attr_set[64] = {false};
  const int rc = allow_smem(select_rank_kernel, attr_set);
  if (rc != GRASS_OK) return rc;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>(ctas));
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = a.stage_norms ? rows * sizeof(float) : 0;
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = static_cast<unsigned>(ctas);
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  attr[1] = dependent_launch_attr();
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  ProfileScope prof(GRASS_K_SELECT, s);
  GRASS_CUDA_TRY(cudaLaunchKernelEx(&cfg, select_rank_kernel, a, rows));
  return GRASS_OK;
}

// Stage the norms (and, if they still fit, the hit counters and the running sum) in shared memory: the
// with-replacement kernel is a chain of short passes over m values, each of which would otherwise wait
// on an L2 round trip.
int launch_select(SelectArgs& a, cudaStream_t s) {
  if (a.method == GRASS_SEL_TOPR || is_nr(a.method)) return launch_rank(a, s);
  const size_t m4 = (static_cast<size_t>(a.m) + 3) / 4 * 4 * sizeof(float);
  a.stage_norms = m4 <= kSelectBudget;
  a.stage_counts = a.stage_norms && 2 * m4 <= kSelectBudget;
  a.stage_cdf = a.stage_counts && 4 * m4 <= kSelectBudget;
  const size_t smem = a.stage_norms ? (a.stage_cdf ? 4 * m4 : a.stage_counts ? 2 * m4 : m4) : 0;
  static bool attr_set[64] = {false};
  const int rc = allow_smem(select_kernel, attr_set);
  if (rc != GRASS_OK) return rc;
  ProfileScope prof(GRASS_K_SELECT, s);
  GRASS_CUDA_TRY(launch_kernel(select_kernel, 1, kThreads, smem, s, a));
  return GRASS_OK;
}

size_t cdf_bytes(int64_t m) { return round_up(static_cast<size_t>(m) * sizeof(double), 256); }

}  // namespace
}  // namespace grass

extern "C" size_t grass_select_workspace_bytes(int64_t m, int32_t r, int method) {
  (void)r;
  if (m < 1) return 0;
  if (method == GRASS_SEL_TOPR) return 256;  // unused, but never zero so callers can allocate
  return grass::cdf_bytes(m) + grass::round_up(static_cast<size_t>(m) * sizeof(int), 256);
}

int grass::select_rows(const float* norms, int64_t m, int32_t r, int method, uint64_t seed,
                       uint32_t layer_id, uint32_t epoch, int32_t* idx, float* rho, void* ws,
                       size_t ws_bytes, cudaStream_t s) {
  if (norms == nullptr || idx == nullptr || rho == nullptr || m < 1 || m > 0x7fffffffLL ||
      r < 1 || r > m)
    return GRASS_ERR_INVALID_ARG;
  if (method < GRASS_SEL_TOPR || method > GRASS_SEL_UNIFORM_NR) return GRASS_ERR_UNSUPPORTED;
  SelectArgs a;
  a.cdf = nullptr;
  a.counts = nullptr;
  if (method != GRASS_SEL_TOPR) {
    if (ws == nullptr || !aligned_to(ws, 256) ||
        ws_bytes < grass_select_workspace_bytes(m, r, method))
      return GRASS_ERR_WORKSPACE;
    a.cdf = static_cast<double*>(ws);
    a.counts = reinterpret_cast<int*>(static_cast<char*>(ws) + cdf_bytes(m));
  }
  cudaError_t err;
  a.status = status_word(&err);
  if (a.status == nullptr) GRASS_CUDA_TRY(err);
  a.norms = norms;
  a.m = static_cast<int>(m);
  a.r = r;
  a.method = method;
  a.seed_lo = static_cast<uint32_t>(seed & 0xffffffffu);
  a.seed_hi = static_cast<uint32_t>(seed >> 32);
  a.layer_id = layer_id;
  a.epoch = epoch;
  a.idx = idx;
  a.rho = rho;
  return launch_select(a, s);
}

extern "C" int grass_select(const float* norms, int64_t m, int32_t r, int method, uint64_t seed,
                            uint32_t layer_id, uint32_t epoch, int32_t* idx, float* rho, void* ws,
                            size_t ws_bytes, void* stream) {
  return grass::select_rows(norms, m, r, method, seed, layer_id, epoch, idx, rho, ws, ws_bytes,
                            static_cast<cudaStream_t>(stream));
}

// ---------------------------------------------------------------------------
// grass_select_static: the same selection with its scratch in a fixed device
// array that is part of the library image, for callers that cannot allocate.
// ---------------------------------------------------------------------------
namespace grass {
namespace {

constexpr int kStaticMaxM = GRASS_SELECT_STATIC_MAX_M;

// Running sum (fp64) followed by the per-row hit counts (int32) for up to
// kStaticMaxM rows: 192 KiB, resident on every GPU that loads the library.
static __device__ __align__(256) unsigned char g_select_scratch[kStaticMaxM * (sizeof(double) + sizeof(int))];

// Device address of g_select_scratch on the current device, resolved once per
// device.  In host code the symbol name is only a handle; a kernel must be
// given the address the runtime reports for it.
int static_scratch(unsigned char** out) {
  static unsigned char* cached[64] = {nullptr};
  int dev = 0;
  GRASS_CUDA_TRY(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64) return GRASS_ERR_INVALID_ARG;
  if (cached[dev] == nullptr) {
    unsigned char* p = nullptr;
    GRASS_CUDA_TRY(cudaGetSymbolAddress(reinterpret_cast<void**>(&p), g_select_scratch));
    cached[dev] = p;
  }
  *out = cached[dev];
  return GRASS_OK;
}

}  // namespace
}  // namespace grass

extern "C" int grass_select_static(const float* norms, int64_t m, int32_t r, int method,
                                   uint64_t seed, uint32_t layer_id, uint32_t epoch, int32_t* idx,
                                   float* rho, void* stream) {
  using namespace grass;
  if (norms == nullptr || idx == nullptr || rho == nullptr || m < 1 || r < 1 || r > m)
    return GRASS_ERR_INVALID_ARG;
  if (m > kStaticMaxM) {
    fprintf(stderr, "grass_select_static: m = %lld exceeds the built-in scratch (%d rows); "
                    "use grass_select with a caller-provided workspace\n",
            static_cast<long long>(m), kStaticMaxM);
    return GRASS_ERR_WORKSPACE;
  }
  if (method < GRASS_SEL_TOPR || method > GRASS_SEL_UNIFORM_NR) return GRASS_ERR_UNSUPPORTED;
  unsigned char* scratch = nullptr;
  const int rc = static_scratch(&scratch);
  if (rc != GRASS_OK) return rc;
  cudaError_t err;
  SelectArgs a;
  a.status = status_word(&err);
  if (a.status == nullptr) GRASS_CUDA_TRY(err);
  a.cdf = reinterpret_cast<double*>(scratch);
  a.counts = reinterpret_cast<int*>(scratch + static_cast<size_t>(kStaticMaxM) * sizeof(double));
  a.norms = norms;
  a.m = static_cast<int>(m);
  a.r = r;
  a.method = method;
  a.seed_lo = static_cast<uint32_t>(seed & 0xffffffffu);
  a.seed_hi = static_cast<uint32_t>(seed >> 32);
  a.layer_id = layer_id;
  a.epoch = epoch;
  a.idx = idx;
  a.rho = rho;
  // Of the array the kernel can reach only the running sum, and only for m > 12800 with a
  // with-replacement method (everything else is staged in shared memory); it writes every
  // running-sum entry before reading it, so whatever an earlier call left there is never
  // observed.
  return launch_select(a, static_cast<cudaStream_t>(stream));
}
