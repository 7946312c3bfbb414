// Cubic B-spline coefficients of f_ini (Sec. 2.2.2): for every x row a
// tridiagonal system along v, then for every v column one along x.  The
// systems share one constant matrix (rows (1, 4, 1)/6 with the zero-slope
// ghosts eta_{-1} = eta_1, eta_n = eta_{n-2}), so its LU factors c'_i and
// 1/den_i are computed once on the host and each system is one forward and
// one backward sweep.
//
// Row systems are contiguous in memory: a warp per row scans groups of 32
// entries.  Column systems are strided by nv: a lane per column, so a warp's
// loads at a given step are 32 consecutive values, and warps split the rows into
// chunks joined by their carries.  Larger grids take a third way, chunks that
// warm up (below).
#include <algorithm>

#include "common.cuh"

namespace vm {
namespace {

// Row systems, one warp per row: both sweeps are linear recurrences,
// d_j = a_j d_{j-1} + b_j (forward: a_j = -sub_j / den_j, b_j = 6 f_j / den_j)
// and eta_j = -c'_j eta_{j+1} + d_j (backward).  A recurrence over a group of
// 32 consecutive entries is an inclusive scan of affine maps (a, b), composed
// as (a2, b2) o (a1, b1) = (a2 a1, a2 b1 + b2), in five shuffle steps; the
// group then continues from the previous group's last value.  Loads and
// stores are coalesced (32 consecutive entries per warp instruction).
template <typename R, typename C>
__device__ __forceinline__ void rows_scan_body(const Grid& g, const R* __restrict__ src, R* __restrict__ dst,
                                               const C* __restrict__ th, int vb) {
  const int lane = threadIdx.x & 31;
  const int row = vb * 4 + (threadIdx.x >> 5);
  if (row >= g.nx) return;
  const int nv = g.nv;
  const C* cp = th;
  const C* inv = th + nv;
  const R* f = src + (size_t)row * nv;
  R* d = dst + (size_t)row * nv;
  // forward
  R carry = R(0);
  for (int j0 = 0; j0 < nv; j0 += 32) {
    const int j = j0 + lane;
    R a = R(1), b = R(0);  // identity for lanes past the end
    if (j < nv) {
      const R sub = (j == 0) ? R(0) : ((j == nv - 1) ? R(2) : R(1));
      const R iv = (R)inv[j];
      a = -sub * iv;
      b = R(6) * f[j] * iv;
    }
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const R ap = __shfl_up_sync(0xffffffffu, a, o), bp = __shfl_up_sync(0xffffffffu, b, o);
      if (lane >= o) {
        b = a * bp + b;
        a = a * ap;
      }
    }
    const R v = a * carry + b;
    if (j < nv) d[j] = v;
    carry = __shfl_sync(0xffffffffu, v, 31);
  }
  __syncwarp();
  // backward: eta_{nv-1} = d_{nv-1}; groups from the end, scanned towards lower j
  carry = R(0);
  const int last0 = ((nv - 1) / 32) * 32;
  for (int j0 = last0; j0 >= 0; j0 -= 32) {
    const int j = j0 + lane;
    R a = R(1), b = R(0);
    if (j < nv) {
      a = (j == nv - 1) ? R(0) : -(R)cp[j];
      b = d[j];
    }
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const R an = __shfl_down_sync(0xffffffffu, a, o), bn = __shfl_down_sync(0xffffffffu, b, o);
      if (lane + o < 32) {
        b = a * bn + b;
        a = a * an;
      }
    }
    const R v = a * carry + b;
    if (j < nv) d[j] = v;
    carry = __shfl_sync(0xffffffffu, v, 0);
  }
}

template <typename R, typename C>
__global__ void __launch_bounds__(128) k_rows_scan(Grid g, const R* __restrict__ src, R* __restrict__ dst,
                                                   const C* __restrict__ th) {
  if (gate_shut(g)) return;
  rows_scan_body(g, src, dst, th, blockIdx.x);
}

// Column systems: a block per 32 consecutive columns (lane = column, so
// every load and store is coalesced) and CW warps, warp w owning a chunk of
// consecutive rows.  Both sweeps are affine recurrences in the row,
//   forward  d_i = (6 f_i - sub_i d_{i-1}) / den_i = a_i d_{i-1} + (6 f_i / den_i),  a_i = -sub_i / den_i,
//   backward e_i = d_i - c'_i e_{i+1},
// so each warp first runs its chunk from a zero carry, keeping the chunk's
// composition (the product of its factors A, and its last value B); warp 0
// then chains the chunks' carries in order (CW steps per column); and each
// warp adds to every row the product of the chunk's factors up to that row
// times the carry that enters the chunk.  The whole column takes about
// 3 nx / CW dependent steps instead of 2 nx.
constexpr int CW = 32;  // warps per column block

template <typename R, typename C>
__device__ __forceinline__ void cols_body(const Grid& g, R* __restrict__ x, const C* __restrict__ th, int vb) {
  __shared__ R cB[CW][32];  // per chunk and column: the chunk's last value from a zero carry
  __shared__ R cC[CW][32];  // ... then the carry entering the chunk
  __shared__ C cA[CW];      // per chunk: the product of its factors (the same for every column)
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int nx = g.nx, nv = g.nv;
  const int j = vb * 32 + lane;
  const bool col = j < nv;
  const C* cp = th;
  const C* inv = th + nx;
  const int L = (nx + CW - 1) / CW;
  const int i0 = min(w * L, nx), i1 = min(i0 + L, nx);  // this warp's rows [i0, i1)
  R* xc = x + (col ? j : 0);
  // forward, each chunk from a zero carry
  {
    R d = R(0);
    C A = C(1);
#pragma unroll 8
    for (int i = i0; i < i1; i++) {
      const C sub = (i == 0) ? C(0) : ((i == nx - 1) ? C(2) : C(1));
      const R f = col ? xc[(size_t)i * nv] : R(0);
      d = (R(6) * f - (R)sub * d) * (R)inv[i];
      A *= -sub * inv[i];
      if (col) xc[(size_t)i * nv] = d;
    }
    cB[w][lane] = d;
    if (lane == 0) cA[w] = A;
  }
  __syncthreads();
  if (w == 0) {
    R c = R(0);
    for (int q = 0; q < CW; q++) {
      cC[q][lane] = c;
      c = (R)cA[q] * c + cB[q][lane];
    }
  }
  __syncthreads();
  // forward completed (d_i += P_i carry), then the backward sweep of the
  // chunk from a zero carry: e_i = d_i - c'_i e_{i+1}, e at i1 taken as 0
  {
    const R cin = cC[w][lane];
    C P = C(1);
#pragma unroll 8
    for (int i = i0; i < i1; i++) {
      const C sub = (i == 0) ? C(0) : ((i == nx - 1) ? C(2) : C(1));
      P *= -sub * inv[i];
      if (col) xc[(size_t)i * nv] += (R)P * cin;
    }
    R e = R(0);
    C Q = C(1);
#pragma unroll 8
    for (int i = i1 - 1; i >= i0; i--) {
      const C c = (i == nx - 1) ? C(0) : cp[i];
      const R d = col ? xc[(size_t)i * nv] : R(0);
      e = d - (R)c * e;
      Q *= -c;
      if (col) xc[(size_t)i * nv] = e;
    }
    __syncthreads();  // every warp has read its cC entry
    cB[w][lane] = e;
    if (lane == 0) cA[w] = Q;
  }
  __syncthreads();
  if (w == 0) {
    R c = R(0);
    for (int q = CW - 1; q >= 0; q--) {
      cC[q][lane] = c;
      c = (R)cA[q] * c + cB[q][lane];
    }
  }
  __syncthreads();
  {
    const R cin = cC[w][lane];
    C Q = C(1);
#pragma unroll 8
    for (int i = i1 - 1; i >= i0; i--) {
      const C c = (i == nx - 1) ? C(0) : cp[i];
      Q *= -c;
      if (col) xc[(size_t)i * nv] += (R)Q * cin;
    }
  }
}

template <typename R, typename C>
__global__ void __launch_bounds__(32 * CW) k_cols(Grid g, R* __restrict__ x, const C* __restrict__ th) {
  if (gate_shut(g)) return;
  cols_body(g, x, th, blockIdx.x);
}

// ---- larger grids: recursive filters that warm up ----
//
// The zero-slope ghosts make the system that of the data mirrored at its ends,
// on an infinite line, and its matrix (1, 4, 1) / 6 the product of a causal and
// an anticausal one-pole filter with the pole z = sqrt(3) - 2 (Unser, Aldroubi
// and Eden 1993):
//   c_k = f_k + z c_{k-1},  e_k = c_k + z e_{k+1},  eta_k = -6 z e_k,
// with the same coefficients everywhere.  A filter forgets its start by z per
// step, so a chunk swept from WARM = 32 entries before its own (of the mirrored
// data at an end) has the carry to 5e-19 of the carry there: a thousandth of a
// rounding of the largest coefficient around, though not of its own size where f
// falls by more than that within the warm-up (behind a cut edge).  No carries are
// chained and no chunk is corrected.  An entry that is not finite spreads to the
// chunks whose sweep or warm-up holds it (the LU sweeps spread it over its whole
// line).  An entry takes two FP64
// operations, times 1 + WARM / chunk, where the scan of a row takes 28 and the
// chained column sweeps 12 (this GPU has two FP64 lanes per SM); the factors of
// both axes are applied at the end.  One pass over memory per axis, where the
// column sweeps took four; rows go to a scratch array, since a block of columns
// reads rows around its own.  Bound by that pass and by FP64 issue: 4096 x 4096
// FP64 rows 0.89 -> 0.15 ms, columns 0.46 -> 0.16 ms; FP32 0.114 -> 0.042 and
// 0.109 -> 0.034 ms.  Error of FP32 coefficients against 64 bits 6e-8 to 1e-7
// (2-norm), of the sweeps 1e-7 to 2.2e-7.
constexpr int WARM = 32;
constexpr double POLE = -0.26794919243112270647;  // sqrt(3) - 2

template <typename R>
__device__ __forceinline__ void copy_async(R* to, const R* from) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"((unsigned)__cvta_generic_to_shared(to)), "l"(from),
               "n"(sizeof(R))
               : "memory");
}
__device__ __forceinline__ void copy_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// Entry j of n, or its mirror image (|j| and n - 1 - j above -(n - 1)).
__device__ __forceinline__ int mirrored(int j, int n) { return j < 0 ? -j : (j >= n ? 2 * (n - 1) - j : j); }

constexpr int ROW_L = 128;  // longest chunk of a row sweep: a warp takes up to 32 of them

// Segments of a row of nv entries (of at most 32 chunks), and the chunk length.
__host__ __device__ __forceinline__ int row_segments(int nv) { return (nv + 32 * ROW_L - 1) / (32 * ROW_L); }
__host__ __device__ __forceinline__ int row_chunk(int nv) {
  const int ns = row_segments(nv);
  return ((nv + ns - 1) / ns + 31) / 32;
}

// A warp per row segment, a lane per chunk, staged in shared memory with WARM
// entries more on each side (chunks an odd number of words apart).
template <typename R>
__device__ __forceinline__ void rows_filter_body(int nv, const R* __restrict__ src, R* __restrict__ dst, int row,
                                                 int seg, R* row_sh) {
  constexpr R z = (R)POLE;
  const int L = row_chunk(nv), P = L | 1, lane = threadIdx.x & 31;
  const int s0 = seg * 32 * L;
  if (s0 >= nv) return;
  const int n = min(32 * L, nv - s0);  // entries of the segment
  const R* f = src + (size_t)row * nv;
  R* head = row_sh + 32 * P;  // the WARM entries before the segment
  R* tail = head + WARM;      // and after it
  const int q0 = lane / L, dq = 32 / L, dr = 32 - dq * L;
  {
    int q = q0, r = lane - q0 * L;
#pragma unroll 4
    for (int e = lane; e < n; e += 32) {
      copy_async(row_sh + q * P + r, f + s0 + e);
      q += dq;
      r += dr;
      if (r >= L) {
        r -= L;
        q++;
      }
    }
    copy_async(head + lane, f + mirrored(s0 - WARM + lane, nv));
    copy_async(tail + lane, f + mirrored(s0 + n + lane, nv));
  }
  copy_wait();
  __syncwarp();
  const int a = lane * L, b = min(a + L, n);  // the lane's entries of the segment
  R* own = row_sh + lane * P;
  // forward over the entries before the chunk, then its own (every lane has read
  // its neighbours' entries before any is overwritten); the chunk that ends the
  // segment goes on over the entries after it
  R c = R(0);
  {
    int e = a - WARM, q = e < 0 ? 0 : e / L, r = e < 0 ? 0 : e - q * L;
    const R* at = row_sh + q * P + r;
    for (int k = 0; k < WARM; k++, e++) {
      c = fma(z, c, e < 0 ? head[WARM + e] : *at);
      if (e >= 0) {
        at++;
        if (++r == L) {
          r = 0;
          at += P - L;
        }
      }
    }
  }
  __syncwarp();
#pragma unroll 4
  for (int k = 0; k < b - a; k++) own[k] = c = fma(z, c, own[k]);
  if (a < n && b == n)
    for (int k = 0; k < WARM; k++) tail[k] = c = fma(z, c, tail[k]);
  __syncwarp();
  // backward over the entries after the chunk, then its own
  R x = R(0);
  if (a < n) {
    int e = b + WARM - 1, q = (e < n ? e : n - 1) / L, r = (e < n ? e : n - 1) - q * L;
    const R* at = row_sh + q * P + r;
    for (int k = 0; k < WARM; k++, e--) {
      x = fma(z, x, e >= n ? tail[e - n] : *at);
      if (e < n) {
        at--;
        if (--r < 0) {
          r = L - 1;
          at -= P - L;
        }
      }
    }
  }
  __syncwarp();
#pragma unroll 4
  for (int k = b - a - 1; k >= 0; k--) own[k] = x = fma(z, x, own[k]);
  __syncwarp();
  R* o = dst + (size_t)row * nv + s0;
  int q = q0, r = lane - q0 * L;
#pragma unroll 4
  for (int e = lane; e < n; e += 32) {
    o[e] = row_sh[q * P + r];
    q += dq;
    r += dr;
    if (r >= L) {
      r -= L;
      q++;
    }
  }
}

template <typename R>
__global__ void __launch_bounds__(32) k_rows_filter(Grid g, const R* __restrict__ src, R* __restrict__ dst) {
  extern __shared__ double spline_sh[];
  if (gate_shut(g)) return;
  const int ns = row_segments(g.nv), row = blockIdx.x / ns;
  rows_filter_body(g.nv, src, dst, row, blockIdx.x - row * ns, reinterpret_cast<R*>(spline_sh));
}

constexpr int COL_ROWS = 320;                   // rows that a column block writes
constexpr int COL_W = 5;                        // its warps (each a chunk of the rows),
constexpr int COL_W_FEW = 20;                   // and where there are fewer blocks than the chip takes

// A block per 32 columns and COL_ROWS rows, in shared memory with WARM rows more
// on each side; a warp sweeps L of them.
template <typename R>
__device__ __forceinline__ void cols_filter_body(const Grid& g, const R* __restrict__ src, R* __restrict__ dst, int bx,
                                                 int by, int L, int nw, R* col_sh) {
  constexpr R z = (R)POLE, scale = (R)(36.0 * POLE * POLE);
  const int nx = g.nx, nv = g.nv, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int j = bx * 32 + lane;
  const int r0 = by * COL_ROWS, n = min(COL_ROWS, nx - r0);  // rows [r0, r0 + n)
  const bool col = j < nv;
  R* T = col_sh + 32 * WARM + lane;  // T[32 r]: row r0 + r
  const R* f = src + (col ? j : 0);
#pragma unroll 4
  for (int r = w - WARM; r < n + WARM; r += nw) copy_async(T + 32 * r, f + (size_t)mirrored(r0 + r, nx) * nv);
  copy_wait();
  __syncthreads();
  const int a = w * L, b = min(a + L, n);
  R c = R(0);
  if (a < n) {
#pragma unroll 8
    for (int k = 0; k < WARM; k++) c = fma(z, c, T[32 * (a - WARM + k)]);
  }
  __syncthreads();
#pragma unroll 4
  for (int r = a; r < b; r++) T[32 * r] = c = fma(z, c, T[32 * r]);
  if (a < n && b == n)
    for (int k = 0; k < WARM; k++) T[32 * (n + k)] = c = fma(z, c, T[32 * (n + k)]);
  __syncthreads();
  R x = R(0);
  if (a < n) {
#pragma unroll 8
    for (int k = WARM - 1; k >= 0; k--) x = fma(z, x, T[32 * (b + k)]);
  }
  __syncthreads();
#pragma unroll 4
  for (int r = b - 1; r >= a; r--) {
    x = fma(z, x, T[32 * r]);
    if (col) dst[(size_t)(r0 + r) * nv + j] = x * scale;
  }
}

template <typename R, int NW>
__global__ void __launch_bounds__(32 * NW) k_cols_filter(Grid g, const R* __restrict__ src, R* __restrict__ dst) {
  extern __shared__ double spline_sh[];
  if (gate_shut(g)) return;
  cols_filter_body(g, src, dst, blockIdx.x, blockIdx.y, COL_ROWS / NW, NW, reinterpret_cast<R*>(spline_sh));
}

// Grids whose coefficients take the filters: the mirrored data of a warm-up lie
// on the grid, and FP64 solves below fixed_on keep the sweeps' rounding along
// with that of their values (5 to 15 us a solve).  FP32 solves have the same line
// only to have one.
__host__ __device__ __forceinline__ bool filters_on(const Grid& g) {
  return g.nx > WARM && g.nv > WARM && (long long)g.nx * g.nv >= kFixedSites;
}

// Column blocks of a grid, and the warps of each.
__host__ __device__ __forceinline__ int col_windows(const Grid& g) { return (g.nx + COL_ROWS - 1) / COL_ROWS; }
__host__ __device__ __forceinline__ int col_warps(const Grid& g) {
  return (long long)((g.nv + 31) / 32) * col_windows(g) >= 152 * 2 ? COL_W : COL_W_FEW;
}

size_t row_smem(int nv, size_t word) { return (32 * (size_t)(row_chunk(nv) | 1) + 2 * WARM) * word; }
size_t col_smem(int nx, size_t word) { return 32 * (size_t)(std::min(nx, COL_ROWS) + 2 * WARM) * word; }

// ---- group launches: f_ini -> eta of every solve ----
template <typename R>
__global__ void __launch_bounds__(128) k_rows_group(const SolveDesc* __restrict__ D, const int* __restrict__ off,
                                                  int ns, int total) {
  extern __shared__ double spline_sh[];
  GROUP_LOOP(off, ns, total)
  const int row = vb * 4 + (int)(threadIdx.x >> 5);
  if (filters_on(gsh)) {
    R* sh = reinterpret_cast<R*>(spline_sh) + (threadIdx.x >> 5) * (32 * (row_chunk(gsh.nv) | 1) + 2 * WARM);
    for (int q = 0; row < gsh.nx && q < row_segments(gsh.nv); q++) {
      rows_filter_body(gsh.nv, (const R*)d.fini, (R*)d.tmp, row, q, sh);
      __syncwarp();
    }
  } else if constexpr (sizeof(R) == 4)
    rows_scan_body<float, float>(gsh, (const float*)d.fini, (float*)d.eta, d.thvf, vb);
  else
    rows_scan_body<double, double>(gsh, (const double*)d.fini, (double*)d.eta, d.thv, vb);
  GROUP_END
}

template <typename R>
__global__ void __launch_bounds__(32 * CW) k_cols_group(const SolveDesc* __restrict__ D, const int* __restrict__ off,
                                                      int ns, int total) {
  extern __shared__ double spline_sh[];
  GROUP_LOOP(off, ns, total)
  if (filters_on(gsh)) {
    for (int q = 0; q < col_windows(gsh); q++) {
      cols_filter_body(gsh, (const R*)d.tmp, (R*)d.eta, vb, q, COL_ROWS / col_warps(gsh), CW,
                       reinterpret_cast<R*>(spline_sh));
      __syncthreads();
    }
  } else if constexpr (sizeof(R) == 4)
    cols_body<float, float>(gsh, (float*)d.eta, d.thxf, vb);
  else
    cols_body<double, double>(gsh, (double*)d.eta, d.thx, vb);
  GROUP_END
}

template <typename R>
void filter_rows(vm_solver* s, const void* src) {
  k_rows_filter<R><<<(unsigned)(s->g.nx * row_segments(s->g.nv)), 32, row_smem(s->g.nv, sizeof(R)), s->stream>>>(
      s->g, (const R*)src, (R*)s->tmp);
}

template <typename R>
void filter_cols(vm_solver* s, void* dst) {
  const dim3 blocks((unsigned)((s->g.nv + 31) / 32), (unsigned)col_windows(s->g));
  const size_t smem = col_smem(s->g.nx, sizeof(R));
  if (col_warps(s->g) == COL_W)
    k_cols_filter<R, COL_W><<<blocks, 32 * COL_W, smem, s->stream>>>(s->g, (const R*)s->tmp, (R*)dst);
  else
    k_cols_filter<R, COL_W_FEW><<<blocks, 32 * COL_W_FEW, smem, s->stream>>>(s->g, (const R*)s->tmp, (R*)dst);
}

template <typename K>
bool cols_prepare(K kernel, size_t word) {
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)col_smem(COL_ROWS, word)) ==
         cudaSuccess;
}
template <typename K>
bool rows_prepare(K kernel, size_t word) {
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)(4 * row_smem(32 * ROW_L, word))) == cudaSuccess;
}

}  // namespace

// src -> dst; the filters go through s->tmp, which holds nothing from one call to
// the next.
void launch_spline_solve(vm_solver* s, const void* src, void* dst) {
  const unsigned cb = (unsigned)((s->g.nv + 31) / 32);
  const unsigned sb = (unsigned)((s->g.nx + 3) / 4);
  const bool filter = filters_on(s->g);
  int ps = prof_begin(s, KID_SPLINE_ROWS);
  if (s->fp32) {
    if (filter)
      filter_rows<float>(s, src);
    else
      k_rows_scan<float, float><<<sb, 128, 0, s->stream>>>(s->g, (const float*)src, (float*)dst, s->thomas_vf);
  } else if (filter) {
    filter_rows<double>(s, src);
  } else {
    k_rows_scan<double, double><<<sb, 128, 0, s->stream>>>(s->g, (const double*)src, (double*)dst, s->thomas_v);
  }
  prof_end(s, ps);
  ps = prof_begin(s, KID_SPLINE_COLS);
  if (s->fp32) {
    if (filter)
      filter_cols<float>(s, dst);
    else
      k_cols<float, float><<<cb, 32 * CW, 0, s->stream>>>(s->g, (float*)dst, s->thomas_xf);
  } else if (filter) {
    filter_cols<double>(s, dst);
  } else {
    k_cols<double, double><<<cb, 32 * CW, 0, s->stream>>>(s->g, (double*)dst, s->thomas_x);
  }
  prof_end(s, ps);
  s->launches += 2;
}

// Opt the filters in to shared memory (up to the largest they ask for): a
// solver's, and a group's.
bool spline_prepare(const vm_solver* s) {
  if (!filters_on(s->g)) return true;
  const bool few = col_warps(s->g) == COL_W_FEW;
  if (s->fp32)
    return few ? cols_prepare(k_cols_filter<float, COL_W_FEW>, 4) : cols_prepare(k_cols_filter<float, COL_W>, 4);
  return few ? cols_prepare(k_cols_filter<double, COL_W_FEW>, 8) : cols_prepare(k_cols_filter<double, COL_W>, 8);
}
bool group_spline_prepare() {
  return cols_prepare(k_cols_group<double>, 8) && cols_prepare(k_cols_group<float>, 4) &&
         rows_prepare(k_rows_group<double>, 8) && rows_prepare(k_rows_group<float>, 4);
}

// Shared memory of the group's sweeps for grid g (4 rows a block).
void group_spline_smem(const Grid& g, bool fp32, size_t& rows, size_t& cols) {
  const size_t word = fp32 ? 4 : 8;
  rows = filters_on(g) ? 4 * row_smem(g.nv, word) : 0;
  cols = filters_on(g) ? col_smem(g.nx, word) : 0;
}

void group_spline(const GroupPlan& G) {
  const unsigned rb = group_grid(G, GP_ROWS, G.tot_rows4), cb = group_grid(G, GP_COLS, G.tot_cols);
  if (G.fp32) {
    k_rows_group<float><<<rb, 128, G.row_smem, G.stream>>>(G.D, G.off_rows4, G.ns, G.tot_rows4);
    k_cols_group<float><<<cb, 32 * CW, G.col_smem, G.stream>>>(G.D, G.off_cols, G.ns, G.tot_cols);
  } else {
    k_rows_group<double><<<rb, 128, G.row_smem, G.stream>>>(G.D, G.off_rows4, G.ns, G.tot_rows4);
    k_cols_group<double><<<cb, 32 * CW, G.col_smem, G.stream>>>(G.D, G.off_cols, G.ns, G.tot_cols);
  }
}

}  // namespace vm
