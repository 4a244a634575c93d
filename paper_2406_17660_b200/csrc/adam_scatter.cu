// grass_adam_scatter: adam.update on the subspace state (Appendix A of the GRASS
// paper) and the row-sparse apply W <- W + alpha P U (Algorithm 1) in one pass;
// inside grass_layer_step also the split-K sum of the projected gradient.
//
// The steps are row-local: state row j and update row j feed only row idx[j] of W.
// Running them back to back in one kernel keeps G_C and U in registers: U is written
// only if the caller wants it, G_C is written once and never re-read.  Bytes per
// element: M and V 4 in + 4 out each, W in + out, and G_C 4 in (finished gradient) or
// 4 in per partial + 4 out.  The arithmetic is that of the separate kernels, operation
// for operation, so the results are bit-identical to calling them in turn.
//
// Bound by HBM where r n is large and by load latency where it is small; one kernel for each.
// Every load that does not depend on another is issued first.  Rows whose length or pitch rules
// 128-bit access out (n = 5461) keep a lane's columns 32 apart, so that every warp access is still
// one contiguous run of 128 bytes: the r = 512, n = 5461 update takes 20 us cold; eight consecutive
// scalars a thread took 49.
//
// idx is ascending, so repeated rows are adjacent (a "run"; sampling with replacement gives runs of
// two to hundreds).  The W row is rounded once, after the terms of its run are added in order of
// j.  A run costs a few memory latencies a row when one warp walks it, so longer runs are taken by
// several warps, a row each, that exchange the updates through shared memory.
#include "update_common.cuh"

namespace grass {
namespace {

constexpr int kRows = 8;                 // rows (warps) of a block of the narrow kernel
constexpr int kThreads = 256;
constexpr int kWalk = 4;                 // longest run one block of the wide kernel walks

// A lane's E columns of a row: with VEC groups of four (c .. c + 3, then 128 further on), else c,
// c + 32, ..; those at or past n are left alone.
template <int E, bool VEC>
__device__ __forceinline__ void load_e(const float* p, int64_t c, int64_t n, float (&v)[E]) {
  if constexpr (VEC) {
#pragma unroll
    for (int q = 0; q < E / 4; ++q)
      if (c + 128 * q < n) {
        const float4 t = *reinterpret_cast<const float4*>(p + c + 128 * q);
        v[4 * q] = t.x; v[4 * q + 1] = t.y; v[4 * q + 2] = t.z; v[4 * q + 3] = t.w;
      }
  } else {
#pragma unroll
    for (int i = 0; i < E; ++i)
      if (c + 32 * i < n) v[i] = p[c + 32 * i];
  }
}
template <int E, bool VEC>
__device__ __forceinline__ void store_e(float* p, int64_t c, int64_t n, const float (&v)[E]) {
  if constexpr (VEC) {
#pragma unroll
    for (int q = 0; q < E / 4; ++q)
      if (c + 128 * q < n)
        *reinterpret_cast<float4*>(p + c + 128 * q) =
            make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
  } else {
#pragma unroll
    for (int i = 0; i < E; ++i)
      if (c + 32 * i < n) p[c + 32 * i] = v[i];
  }
}
template <typename T, int E, bool VEC>
__device__ __forceinline__ void load_w(const T* p, int64_t c, int64_t n, T (&v)[E]) {
  if constexpr (VEC) {
    using V4 = typename WTraits<T>::vec4;
#pragma unroll
    for (int q = 0; q < E / 4; ++q)
      if (c + 128 * q < n)
        *reinterpret_cast<V4*>(v + 4 * q) = *reinterpret_cast<const V4*>(p + c + 128 * q);
  } else {
#pragma unroll
    for (int i = 0; i < E; ++i)
      if (c + 32 * i < n) v[i] = p[c + 32 * i];
  }
}
template <typename T, int E, bool VEC>
__device__ __forceinline__ void store_w(T* p, int64_t c, int64_t n, const T (&v)[E]) {
  if constexpr (VEC) {
    using V4 = typename WTraits<T>::vec4;
#pragma unroll
    for (int q = 0; q < E / 4; ++q)
      if (c + 128 * q < n)
        *reinterpret_cast<V4*>(p + c + 128 * q) = *reinterpret_cast<const V4*>(v + 4 * q);
  } else {
#pragma unroll
    for (int i = 0; i < E; ++i)
      if (c + 32 * i < n) p[c + 32 * i] = v[i];
  }
}

struct RowArgs {
  const float* part;
  float *Gc, *M, *V, *U;
  const float* rho;
  int64_t ldgc, ldstate, n;
  long long ld_part, split_stride;
  int split_k;
  bool part_by_row, reset;
};

// Gradient (the partials' sum, or Gc itself) and Adam of row j at this lane's columns; `row` is
// idx[j], or -1 where that is outside W (its gradient is zero if it would come from there).
template <int E, bool VEC, bool SPLIT>
__device__ __forceinline__ void update_row(const RowArgs& p, const AdamScalars& a, int j, int row,
                                           int64_t c, float rho, float (&u)[E]) {
  // partials in flight; more than two at four columns cost registers that more blocks use better
  constexpr int FLIGHT = E == 1 ? 16 : 2;
  float* mrow = p.M + static_cast<int64_t>(j) * p.ldstate;
  float* vrow = p.V + static_cast<int64_t>(j) * p.ldstate;
  float g[E] = {}, mv[E] = {}, vv[E] = {};
  if (!p.reset) {
    load_e<E, VEC>(mrow, c, p.n, mv);
    load_e<E, VEC>(vrow, c, p.n, vv);
  }
  if (SPLIT) {
    const int pr = p.part_by_row ? row : j;
    if (pr < 0) rho = 0.f;
    const float* part = p.part + (pr < 0 ? 0 : pr) * p.ld_part;
    load_e<E, VEC>(part, c, p.n, g);
    part += p.split_stride;
    for (int s = 1; s < p.split_k; s += FLIGHT) {     // the order of the adds is fixed
      float t[FLIGHT][E];
#pragma unroll
      for (int k = 0; k < FLIGHT; ++k) {
#pragma unroll
        for (int i = 0; i < E; ++i) t[k][i] = 0.f;
        if (s + k < p.split_k) load_e<E, VEC>(part + k * p.split_stride, c, p.n, t[k]);
      }
      part += FLIGHT * p.split_stride;
#pragma unroll
      for (int k = 0; k < FLIGHT; ++k)
        if (s + k < p.split_k)
#pragma unroll
          for (int i = 0; i < E; ++i) g[i] += t[k][i];
    }
#pragma unroll
    for (int i = 0; i < E; ++i) g[i] *= rho;
    store_e<E, VEC>(p.Gc + j * p.ldgc, c, p.n, g);
  } else {
    load_e<E, VEC>(p.Gc + j * p.ldgc, c, p.n, g);
  }
#pragma unroll
  for (int i = 0; i < E; ++i) adam_elem(g[i], mv[i], vv[i], u[i], a);
  store_e<E, VEC>(mrow, c, p.n, mv);
  store_e<E, VEC>(vrow, c, p.n, vv);
  if (p.U != nullptr) store_e<E, VEC>(p.U + static_cast<int64_t>(j) * p.ldstate, c, p.n, u);
}

// Small outputs: a warp is one selected row by 32 columns, a block kRows consecutive rows: as many
// warps as there are, and 16 partials of a column in flight.  The block that holds the first j of a
// run owns it, also where the run reaches past the block.
template <typename T, bool SPLIT>
__global__ void __launch_bounds__(kThreads, SPLIT ? 4 : 6)
adam_apply_narrow_kernel(const __grid_constant__ UpdateGroup grp, int64_t ldgc, int64_t ldstate,
                         int64_t m, int64_t n, int64_t ldw, int r, long long ld_part,
                         long long split_stride, int split_k, bool part_by_row, bool reset,
                         float alpha, AdamScalars a, int* status) {
  __shared__ float s_u[kRows][32];
  __shared__ float s_scale[kRows];
  grid_dep_wait();
  const int lay = blockIdx.z;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int32_t* idx = grp.idx[lay];
  const RowArgs p = {grp.part[lay], grp.Gc[lay], grp.M[lay], grp.V[lay], grp.U[lay], grp.rho[lay],
                     ldgc, ldstate, n, ld_part, split_stride, split_k, part_by_row, reset};
  const int64_t c = static_cast<int64_t>(blockIdx.x) * 32 + lane;
  const int ja = blockIdx.y * kRows, j = ja + warp;
  const int last = ja + kRows < r ? ja + kRows : r;       // rows of this block: [ja, last)
  const bool in = j < r;
  // every warp reads the block's rows and one more on either side (lane l: row ja - 1 + l) and
  // sees for itself where neighbours are equal: a block without repeats needs no barrier
  const int jl = ja - 1 + lane;
  const int idl = jl >= 0 && jl < r && lane < kRows + 2 ? idx[jl] : 0;
  const int idp = __shfl_up_sync(0xffffffffu, idl, 1);
  const uint32_t same =
      __ballot_sync(0xffffffffu, lane >= 1 && lane < kRows + 2 && jl >= 1 && jl < r && idl == idp);
  const int row = __shfl_sync(0xffffffffu, idl, warp + 1);
  const int before = __shfl_sync(0xffffffffu, idl, 0);    // row of the last j of the previous block
  const bool prev = in && (same >> (warp + 1) & 1u) != 0;
  // a run that began before this block is its owner's business
  const bool mine = in && (ja == 0 || before != row);
  const bool valid = row >= 0 && row < m;
  if (mine && !prev && !valid && lane == 0 && blockIdx.x == 0)
    record_status(status, GRASS_ERR_INVALID_ARG, row);
  T* w = static_cast<T*>(grp.W[lay]) + static_cast<int64_t>(valid ? row : 0) * ldw;
  const bool writer = mine && !prev && valid;             // first j of its run: adds to the W row
  T wv[1];
  if (writer) load_w<T, 1, false>(w, c, n, wv);
  const float rj = in && p.rho != nullptr ? p.rho[j] : 1.f;
  float u[1] = {}, acc = 0.f;
  if (mine) {
    update_row<1, false, SPLIT>(p, a, j, valid ? row : -1, c, rj, u);
    acc = apply_acc(0.f, alpha * rj, u[0]);
  }
  if (same != 0) {
    s_u[warp][lane] = u[0];
    if (lane == 0) s_scale[warp] = alpha * rj;
    __syncthreads();
    if (writer)
      for (int k = j + 1; k < last && idx[k] == row; ++k)
        acc = apply_acc(acc, s_scale[k - ja], s_u[k - ja][lane]);
    // the block's last run, where it reaches past the block and began in it
    const int tail = __shfl_sync(0xffffffffu, idl, last - ja);
    if (ja == 0 || before != tail) {
      for (int base = last; base < r && idx[base] == tail; base += kRows) {
        __syncthreads();                                  // s_u has been read
        const int k = base + warp;
        if (k < r && idx[k] == tail) {
          const float rk = p.rho != nullptr ? p.rho[k] : 1.f;
          update_row<1, false, SPLIT>(p, a, k, tail >= 0 && tail < m ? tail : -1, c, rk, u);
          s_u[warp][lane] = u[0];
          if (lane == 0) s_scale[warp] = alpha * rk;
        }
        __syncthreads();
        if (writer && row == tail)
          for (int q = 0; q < kRows && base + q < r && idx[base + q] == tail; ++q)
            acc = apply_acc(acc, s_scale[q], s_u[q][lane]);
      }
    }
  }
  if (writer) {
    wv[0] = WTraits<T>::add1(wv[0], acc);
    store_w<T, 1, false>(w, c, n, wv);
  }
}

// Long runs of the wide kernel: the blocks of the run deal out chunks of 128 columns of this block's
// columns [c0, c_end); the warps of a block take a row each, then warps 0..3 add their 32 columns'
// updates in order of j.
template <typename T, bool SPLIT>
__device__ __forceinline__ void apply_run(const RowArgs& p, const AdamScalars& a, int first, int run,
                                          int row, int mine, int64_t c0, int64_t c_end, T* w, bool valid,
                                          float alpha, float (*s_u)[128], float* s_scale) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
  for (int64_t cc = c0 + 128 * static_cast<int64_t>(mine); cc < c_end; cc += 128 * static_cast<int64_t>(run)) {
    float acc = 0.f;
    for (int base = 0; base < run; base += nwarps) {
      const int j = first + base + warp;
      if (base + warp < run) {
        const float rj = p.rho != nullptr ? p.rho[j] : 1.f;
        float u[4] = {};
        update_row<4, false, SPLIT>(p, a, j, row, cc + lane, rj, u);
#pragma unroll
        for (int i = 0; i < 4; ++i) s_u[warp][32 * i + lane] = u[i];
        if (lane == 0) s_scale[warp] = alpha * rj;
      }
      __syncthreads();
      const int here = run - base < nwarps ? run - base : nwarps;
      if (warp < 4)
        for (int q = 0; q < here; ++q) acc = apply_acc(acc, s_scale[q], s_u[q][32 * warp + lane]);
      __syncthreads();
    }
    const int64_t c = cc + 32 * warp + lane;
    if (warp < 4 && c < p.n && valid) w[c] = WTraits<T>::add1(w[c], acc);
  }
}

// Large outputs: a block is one selected row by E columns a thread: few, long contiguous
// stretches of M, V, G_C and W per SM at a time.  (Eight rows by 128 or 256 columns a block, the
// narrow kernel's shape, took 79 us cold for the 403 MB of 7B q,k,v,o, r = 1024; this takes 72.)
// Registers for four blocks an SM: at three the same update took 80 us, at five with E = 4 as well;
// with partials (r = 1024, n = 11008, 3 of them): 86 us at three blocks and four partials in flight,
// 76 as it is, against 81 for a separate reduction followed by the update.
template <typename T, int E, bool VEC, bool SPLIT>
__global__ void __launch_bounds__(kThreads, 4)
adam_apply_wide_kernel(const __grid_constant__ UpdateGroup grp, int64_t ldgc, int64_t ldstate, int64_t m,
                       int64_t n, int64_t ldw, int r, long long ld_part, long long split_stride,
                       int split_k, bool part_by_row, bool reset, float alpha, AdamScalars a, int* status) {
  __shared__ float s_u[kThreads / 32][128];               // long runs only
  __shared__ float s_scale[kThreads / 32];
  grid_dep_wait();
  const int lay = blockIdx.z, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int32_t* idx = grp.idx[lay];
  const RowArgs p = {grp.part[lay], grp.Gc[lay], grp.M[lay], grp.V[lay], grp.U[lay], grp.rho[lay],
                     ldgc, ldstate, n, ld_part, split_stride, split_k, part_by_row, reset};
  const int j0 = blockIdx.y;
  const int row = idx[j0];
  const bool prev = j0 > 0 && idx[j0 - 1] == row, next = j0 + 1 < r && idx[j0 + 1] == row;
  const bool valid = row >= 0 && row < m;
  if (!valid && !prev && threadIdx.x == 0 && blockIdx.x == 0)
    record_status(status, GRASS_ERR_INVALID_ARG, row);
  const int64_t width = static_cast<int64_t>(blockDim.x) * E, c0 = blockIdx.x * width;
  T* w = static_cast<T*>(grp.W[lay]) + static_cast<int64_t>(valid ? row : 0) * ldw;
  int run = 1;
  if (prev || next) {
    // contiguous equal entries before and after
    const int nthr = blockDim.x;
    int before = 0, after = 0, hit;
    for (int k = j0 - 1 - static_cast<int>(threadIdx.x);; k -= nthr) {
      before += hit = __syncthreads_count(k >= 0 && idx[k] == row);
      if (hit < nthr) break;
    }
    for (int k = j0 + 1 + static_cast<int>(threadIdx.x);; k += nthr) {
      after += hit = __syncthreads_count(k < r && idx[k] == row);
      if (hit < nthr) break;
    }
    run = before + 1 + after;
    if (run > kWalk) {
      apply_run<T, SPLIT>(p, a, j0 - before, run, valid ? row : -1, before, c0, c0 + width < n ? c0 + width : n, w, valid,
                          alpha, s_u, s_scale);
      return;
    }
    if (before > 0) return;                               // the first j walks a short run
  }
  const int64_t c = c0 + warp * (32 * E) + (VEC ? 4 * lane : lane);
  alignas(16) T wv[E];
  if (valid) load_w<T, E, VEC>(w, c, n, wv);
  float acc[E] = {};
  for (int j = j0; j < j0 + run; ++j) {
    const float rj = p.rho != nullptr ? p.rho[j] : 1.f;
    float u[E] = {};
    update_row<E, VEC, SPLIT>(p, a, j, valid ? row : -1, c, rj, u);
#pragma unroll
    for (int i = 0; i < E; ++i) acc[i] = apply_acc(acc[i], alpha * rj, u[i]);
  }
  if (valid) {
#pragma unroll
    for (int i = 0; i < E; ++i) wv[i] = WTraits<T>::add1(wv[i], acc[i]);
    store_w<T, E, VEC>(w, c, n, wv);
  }
}

// Column form: the state is r x n as before, but row j feeds column idx[j] of W (n x m).  A block is
// 32 state rows by 32 columns c: the updates are computed with c along the lanes (a warp four rows, all
// their loads in flight), scaled, turned in shared memory, and added with j along the lanes, so that
// the 32 lanes touch 32 ascending columns of one W row.  The W elements are fetched first: they depend on
// nothing but idx.  Bound by HBM: a W row is read and written nearly whole from r/m = 1/16 up.  The
// block that holds the first j of a run owns it.  7B gate (r = 512 of 4096 columns, n = 11008, three partials):
// separate reduction, Adam and scatter took 87 us, this takes 66 (82 at three
// blocks an SM).
template <typename T, bool SPLIT>
__global__ void __launch_bounds__(kThreads, 4)
adam_apply_cols_kernel(const __grid_constant__ UpdateGroup grp, int64_t ldgc, int64_t ldstate, int64_t m,
                       int64_t n, int64_t ldw, int r, long long ld_part, long long split_stride,
                       int split_k, bool part_by_row, bool reset, float alpha, AdamScalars a, int* status) {
  constexpr int J = 32, Q = 4;                            // state rows of a block, of a warp
  __shared__ float s_u[J][33];
  grid_dep_wait();
  const int lay = blockIdx.z, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int32_t* idx = grp.idx[lay];
  const float* rho = grp.rho[lay];
  const float* part = grp.part[lay];
  float *Gc = grp.Gc[lay], *M = grp.M[lay], *V = grp.V[lay], *U = grp.U[lay];
  // blocks run along j first: those of one moment cover whole rows of W (512-byte pieces of every row
  // otherwise: 74 us instead of 66)
  const unsigned jblocks = (r + J - 1) / J;
  const int ja = static_cast<int>(blockIdx.x % jblocks) * J, last = ja + J < r ? ja + J : r;
  const int64_t c0 = static_cast<int64_t>(blockIdx.x / jblocks) * 32;
  // the lane's column of W
  const int jl = ja + lane;
  const int col = jl < r ? idx[jl] : -1;
  const int before = ja > 0 ? idx[ja - 1] : -1;
  const int colp = __shfl_up_sync(0xffffffffu, col, 1);
  const bool foreign = jl < r && ja > 0 && col == before; // of a run that an earlier block owns
  const bool head = jl < r && !foreign && (lane == 0 || col != colp);
  const bool ok = head && col >= 0 && col < m;
  if (head && !ok && c0 == 0 && warp == 0) record_status(status, GRASS_ERR_INVALID_ARG, col);
  const uint32_t skip = __ballot_sync(0xffffffffu, foreign);
  T* w = static_cast<T*>(grp.W[lay]) + (ok ? col : 0);
  T wv[Q];
  if (ok) {
#pragma unroll
    for (int k = 0; k < Q; ++k)
      if (c0 + warp + 8 * k < n) wv[k] = w[(c0 + warp + 8 * k) * ldw];
  }
  // rows base + 4 warp .. + 3 of the chunk [base, stop): gradient, Adam, scaled update to s_u
  const int64_t c = c0 + lane;
  auto chunk = [&](int base, int stop, uint32_t off_rows) {
    float g[Q] = {}, mv[Q] = {}, vv[Q] = {}, s[Q], rj[Q];
    bool on[Q];
    const float* p[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) {
      const int jj = Q * warp + q, j = base + jj;
      on[q] = j < stop && c < n && (off_rows >> jj & 1u) == 0;
      const int js = on[q] ? j : base;
      rj[q] = rho != nullptr ? rho[js] : 1.f;
      s[q] = alpha * rj[q];
      if (SPLIT) {
        int pr = js;
        if (part_by_row) {
          pr = idx[js];
          if (pr < 0 || pr >= m) { pr = 0; rj[q] = 0.f; }
        }
        p[q] = part + pr * ld_part + (on[q] ? c : 0);
        g[q] = *p[q];
      } else if (on[q]) {
        g[q] = Gc[j * ldgc + c];
      }
      if (on[q] && !reset) {
        mv[q] = M[static_cast<int64_t>(j) * ldstate + c];
        vv[q] = V[static_cast<int64_t>(j) * ldstate + c];
      }
    }
    if (SPLIT) {
      for (int z = 1; z < split_k; z += 4) {
        float t[4][Q];
#pragma unroll
        for (int k = 0; k < 4; ++k)
#pragma unroll
          for (int q = 0; q < Q; ++q) t[k][q] = z + k < split_k ? p[q][(z + k) * split_stride] : 0.f;
#pragma unroll
        for (int k = 0; k < 4; ++k)
          if (z + k < split_k)
#pragma unroll
            for (int q = 0; q < Q; ++q) g[q] += t[k][q];
      }
    }
#pragma unroll
    for (int q = 0; q < Q; ++q) {
      if (!on[q]) continue;
      const int64_t so = static_cast<int64_t>(base + Q * warp + q) * ldstate + c;
      float u;
      if (SPLIT) {
        g[q] *= rj[q];
        Gc[(base + Q * warp + q) * ldgc + c] = g[q];
      }
      adam_elem(g[q], mv[q], vv[q], u, a);
      M[so] = mv[q];
      V[so] = vv[q];
      if (U != nullptr) U[so] = u;
      s_u[Q * warp + q][lane] = __fmul_rn(s[q], u);
    }
  };
  chunk(ja, last, skip);
  __syncthreads();
  float acc[Q] = {};
  if (ok)
    for (int i = lane; i < last - ja && (i == lane || idx[ja + i] == col); ++i)
#pragma unroll
      for (int k = 0; k < Q; ++k) acc[k] = __fadd_rn(acc[k], s_u[i][warp + 8 * k]);
  // the block's last run, where it reaches past the block and began in it
  const int tail = __shfl_sync(0xffffffffu, col, last - 1 - ja);
  if (ja == 0 || before != tail) {
    for (int base = last; base < r && idx[base] == tail; base += J) {
      int stop = base + 1;
      while (stop < r && stop < base + J && idx[stop] == tail) ++stop;
      __syncthreads();                                    // s_u has been read
      chunk(base, stop, 0u);
      __syncthreads();
      if (ok && col == tail)
        for (int i = 0; i < stop - base; ++i)
#pragma unroll
          for (int k = 0; k < Q; ++k) acc[k] = __fadd_rn(acc[k], s_u[i][warp + 8 * k]);
    }
  }
  if (ok) {
#pragma unroll
    for (int k = 0; k < Q; ++k)
      if (c0 + warp + 8 * k < n) w[(c0 + warp + 8 * k) * ldw] = WTraits<T>::add1(wv[k], acc[k]);
  }
}

template <typename T>
int launch_cols(const UpdateCall& u, cudaStream_t s) {
  cudaError_t err;
  int* status = status_word(&err);
  if (status == nullptr) GRASS_CUDA_TRY(err);
  const int64_t blocks = ((u.n + 31) / 32) * ((u.r + 31) / 32);
  if (blocks > 0x7fffffffLL) return GRASS_ERR_INVALID_ARG;
  dim3 grid(static_cast<unsigned>(blocks), 1, static_cast<unsigned>(u.count));
  ProfileScope prof(GRASS_K_ADAM_SCATTER, s);
  GRASS_CUDA_TRY(launch_kernel(u.split_k > 0 ? adam_apply_cols_kernel<T, true> : adam_apply_cols_kernel<T, false>,
                               grid, kThreads, 0, s, u.grp, u.ldgc, u.ldstate, u.m, u.n, u.ldw,
                               u.r, u.ld_part, u.split_stride, u.split_k, u.part_by_row, u.reset, u.alpha,
                               u.a, status));
  return GRASS_OK;
}

template <typename T, bool SPLIT>
int launch_narrow(const UpdateCall& u, int* status, cudaStream_t s) {
  dim3 grid(static_cast<unsigned>((u.n + 31) / 32), static_cast<unsigned>((u.r + kRows - 1) / kRows),
            static_cast<unsigned>(u.count));
  {
    ProfileScope prof(GRASS_K_ADAM_SCATTER, s);
    GRASS_CUDA_TRY(launch_kernel(adam_apply_narrow_kernel<T, SPLIT>, grid, kThreads, 0, s,
        u.grp, u.ldgc, u.ldstate, u.m, u.n, u.ldw, u.r, u.ld_part, u.split_stride, u.split_k, u.part_by_row,
        u.reset, u.alpha, u.a, status));
  }
  return GRASS_OK;
}

template <typename T, int E, bool SPLIT>
int launch_wide(const UpdateCall& u, int* status, cudaStream_t s) {
  bool vec = u.n % 4 == 0 && u.ldw % 4 == 0 && u.ldgc % 4 == 0 && u.ldstate % 4 == 0;
  for (int g = 0; g < u.count; ++g)
    vec = vec && aligned_to(u.grp.W[g], 4 * sizeof(T)) && aligned_to(u.grp.Gc[g], 16) &&
          aligned_to(u.grp.M[g], 16) && aligned_to(u.grp.V[g], 16) &&
          (u.grp.U[g] == nullptr || aligned_to(u.grp.U[g], 16));
  // short rows: no more warps than columns for them, and at least the four that apply_run needs
  int threads = kThreads;
  while (threads > 128 && static_cast<int64_t>(threads / 2) * E >= u.n) threads /= 2;
  const int64_t width = static_cast<int64_t>(threads) * E;
  dim3 grid(static_cast<unsigned>((u.n + width - 1) / width), static_cast<unsigned>(u.r),
            static_cast<unsigned>(u.count));
  {
    ProfileScope prof(GRASS_K_ADAM_SCATTER, s);
    GRASS_CUDA_TRY(launch_kernel(
        vec ? adam_apply_wide_kernel<T, E, true, SPLIT> : adam_apply_wide_kernel<T, E, false, SPLIT>, grid,
        threads, 0, s, u.grp, u.ldgc, u.ldstate, u.m, u.n, u.ldw, u.r, u.ld_part,
        u.split_stride, u.split_k, u.part_by_row, u.reset, u.alpha, u.a, status));
  }
  return GRASS_OK;
}

template <typename T>
int launch(const UpdateCall& u, cudaStream_t s) {
  cudaError_t err;
  int* status = status_word(&err);
  if (status == nullptr) GRASS_CUDA_TRY(err);
  // The wide kernel fills the GPU (148 SMs x 1024 threads x 4 columns) from about 600 k elements up.
  // A finished gradient gives a thread only 56 bytes of loads at four columns; eight keep enough in
  // flight for HBM.  With partials to sum, four columns already have 88 bytes in flight.
  const bool small = static_cast<double>(u.count) * u.r * u.n < 6e5;
  if (u.split_k > 0) return small ? launch_narrow<T, true>(u, status, s) : launch_wide<T, 4, true>(u, status, s);
  return small ? launch_narrow<T, false>(u, status, s) : launch_wide<T, 8, false>(u, status, s);
}

}  // namespace

int check_update(UpdateCall& u, double lr, double beta1, double beta2, double eps, int step,
                 double alpha) {
  if (u.m < 1 || u.n < 1 || u.r < 1 || u.r > (u.cols ? 65535 * 32 : 65535) || u.ldgc < u.n ||
      u.ldstate < u.n || u.ldw < (u.cols ? u.m : u.n) || u.m > 0x7fffffffLL)
    return GRASS_ERR_INVALID_ARG;
  for (int g = 0; g < u.count; ++g)
    if (u.grp.Gc[g] == nullptr || u.grp.M[g] == nullptr || u.grp.V[g] == nullptr ||
        u.grp.W[g] == nullptr || u.grp.idx[g] == nullptr)
      return GRASS_ERR_INVALID_ARG;
  if (!adam_args_ok(lr, beta1, beta2, eps, step)) return GRASS_ERR_INVALID_ARG;
  if (u.wdt != GRASS_F32 && u.wdt != GRASS_BF16) return GRASS_ERR_UNSUPPORTED;
  u.a = make_adam_scalars(lr, beta1, beta2, eps, step);
  u.alpha = static_cast<float>(alpha);
  return GRASS_OK;
}

int launch_update(const UpdateCall& u, cudaStream_t s) {
  if (u.cols) return u.wdt == GRASS_F32 ? launch_cols<float>(u, s) : launch_cols<__nv_bfloat16>(u, s);
  return u.wdt == GRASS_F32 ? launch<float>(u, s) : launch<__nv_bfloat16>(u, s);
}

}  // namespace grass

extern "C" int grass_adam_scatter_batched(int32_t count, const float* const* Gc, int64_t ldgc,
                                          float* const* M, float* const* V, float* const* U,
                                          int64_t ldstate, void* const* W, int wdt, int64_t m,
                                          int64_t n, int64_t ldw, const int32_t* const* idx,
                                          const float* const* rho, int32_t r, double lr,
                                          double beta1, double beta2, double eps, int32_t step,
                                          double alpha, void* stream) {
  using namespace grass;
  if (count < 1 || count > kMaxUpdateGroup || Gc == nullptr || M == nullptr || V == nullptr ||
      W == nullptr || idx == nullptr)
    return GRASS_ERR_INVALID_ARG;
  UpdateCall u = {};
  for (int g = 0; g < count; ++g) {
    u.grp.Gc[g] = const_cast<float*>(Gc[g]);    // split_k == 0: read only
    u.grp.M[g] = M[g]; u.grp.V[g] = V[g];
    u.grp.U[g] = U != nullptr ? U[g] : nullptr;
    u.grp.W[g] = W[g]; u.grp.idx[g] = idx[g];
    u.grp.rho[g] = rho != nullptr ? rho[g] : nullptr;
  }
  u.count = count; u.wdt = wdt; u.r = r;
  u.m = m; u.n = n; u.ldgc = ldgc; u.ldstate = ldstate; u.ldw = ldw;
  const int rc = check_update(u, lr, beta1, beta2, eps, step, alpha);
  return rc != GRASS_OK ? rc : launch_update(u, static_cast<cudaStream_t>(stream));
}

extern "C" int grass_adam_scatter(const float* Gc, int64_t ldgc, float* M, float* V, float* U,
                                  int64_t ldstate, void* W, int wdt, int64_t m, int64_t n,
                                  int64_t ldw, const int32_t* idx, const float* rho, int32_t r,
                                  double lr, double beta1, double beta2, double eps, int32_t step,
                                  double alpha, void* stream) {
  return grass_adam_scatter_batched(1, &Gc, ldgc, &M, &V, &U, ldstate, &W, wdt, m, n, ldw, &idx, &rho, r,
                                    lr, beta1, beta2, eps, step, alpha, stream);
}
