// kernels_nbr.cu -- table set-up, neighbour lists, electron density and
// total energy (EAM, Daw-Baskes form; the short-range many-body potential of
// Sec. III A of Sadigh et al.).
#include "common.cuh"
#include "kernels.h"
#include "multi.cuh"

namespace vcsgc {

// ------------------------------------------------------------ splines
// Hermite data (y_j, m_j) on [x_j, x_j + h] -> power-form cubic in t:
//   c0 = y0, c1 = h m0, c2 = 3 (y1 - y0) - h (2 m0 + m1), c3 = 2 (y0 - y1) + h (m0 + m1).
// Missing derivatives: central differences, one-sided at the ends.
__global__ void k_spline_coeffs(const double* y, const double* m, int n, double h, Cubic* out) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= n - 1) return;
  auto slope = [&](int q) -> double {
    if (m) return m[q];
    if (q == 0) return (y[1] - y[0]) / h;
    if (q == n - 1) return (y[n - 1] - y[n - 2]) / h;
    return (y[q + 1] - y[q - 1]) / (2.0 * h);
  };
  const double y0 = y[j], y1 = y[j + 1];
  const double m0 = h * slope(j), m1 = h * slope(j + 1);
  out[j] = Cubic{y0, m0, 3.0 * (y1 - y0) - 2.0 * m0 - m1, 2.0 * (y0 - y1) + m0 + m1};
}

void launch_spline_coeffs(const double* y, const double* m, int n, double h, Cubic* out,
                          cudaStream_t st) {
  k_spline_coeffs<<<(n + 255) / 256, 256, 0, st>>>(y, m, n, h, out);
}

__global__ void k_spline_derivs(const Cubic* c, int n_int, double inv_h, Cubic* out) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= n_int) return;
  const Cubic q = c[j];
  out[j] = Cubic{q.y * inv_h, 2.0 * q.z * inv_h, 3.0 * q.w * inv_h, 0.0};
}

void launch_spline_derivs(const Cubic* c, int n_int, double h, Cubic* out, cudaStream_t st) {
  k_spline_derivs<<<(n_int + 255) / 256, 256, 0, st>>>(c, n_int, 1.0 / h, out);
}

__global__ void k_to_cubic32(const Cubic* c, int n_int, Cubic32* out) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= n_int) return;
  const Cubic q = c[j];
  out[j] = Cubic32{(float)q.x, (float)q.y, (float)q.z, (float)q.w};
}

void launch_to_cubic32(const Cubic* c, int n_int, Cubic32* out, cudaStream_t st) {
  k_to_cubic32<<<(n_int + 255) / 256, 256, 0, st>>>(c, n_int, out);
}

// ------------------------------------------------------- shell tables
// Rigid lattice: the pair part of dE(A->B) is
//   sum_s [ (z_s - b_s) (phi_BA - phi_AA)(r_s) + b_s (phi_BB - phi_AB)(r_s) ]
//   = C_A + sum_s b_s G_A[s],
// C_A = sum_s z_s (phi_AB - phi_AA)(r_s), G_A[s] = (phi_BB - 2 phi_AB + phi_AA)(r_s).
// value of table q at r: FP64, or FP32 interpolation widened (mixed form)
__device__ __forceinline__ double tab_val(const Tables& tab, const Tables32* t32, int q, double r,
                                          unsigned* err) {
  if (t32) {
    float t;
    const int j = spline32_locate(t32->sp[q], (float)r, t, err);
    return (double)spline32_val_at(t32->sp[q], j, t);
  }
  return spline_val(tab.sp[q], r, err);
}

__global__ void k_shell_tables(Tables tab, Tables32 tab32, int mixed, const int* h2, const int* z,
                               int S, double a, double* out, unsigned* err) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  const Tables32* t32 = mixed ? &tab32 : nullptr;
  double C = 0.0;
  for (int s = 0; s < S; ++s) {
    const double r = 0.5 * a * sqrt((double)h2[s]);
    const double pAA = tab_val(tab, t32, 0, r, err);
    const double pAB = tab_val(tab, t32, 1, r, err);
    const double pBB = tab_val(tab, t32, 2, r, err);
    C += (double)z[s] * (pAB - pAA);
    out[1 + s] = (pBB - pAB) - (pAB - pAA);
    out[1 + S + s] = tab_val(tab, t32, 4, r, err) - tab_val(tab, t32, 3, r, err);
    out[1 + 2 * S + s] = r;
  }
  out[0] = C;
}

// Energy table of the rigid lattice with one density function (uniform
// rho0): etab[s], etab[S + s], etab[2S + s] = phi_AA, phi_AB, phi_BB at r_s
// (r_s = shell_tab[1 + 2S + s]), etab[3S] = F_A(rho0), etab[3S + 1] =
// F_B(rho0), etab[3S + 2 + s] = z_s.  Site energy: F_t(rho0) + 1/2 sum_s
// [(z_s - b_s) phi_{tA}(r_s) + b_s phi_{tB}(r_s)].
__global__ void k_lattice_energy_table(Tables tab, Tables32 tab32, int mixed, const double* shell_tab, int S,
                                       LatZ z, const double* rho, double* etab, unsigned* err) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  const Tables32* t32 = mixed ? &tab32 : nullptr;
  for (int s = 0; s < S; ++s) {
    const double r = shell_tab[1 + 2 * S + s];
    etab[s] = tab_val(tab, t32, 0, r, err);
    etab[S + s] = tab_val(tab, t32, 1, r, err);
    etab[2 * S + s] = tab_val(tab, t32, 2, r, err);
    etab[3 * S + 2 + s] = (double)z.z[s];
  }
  etab[3 * S] = tab_val(tab, t32, 5, rho[0], err);
  etab[3 * S + 1] = tab_val(tab, t32, 6, rho[0], err);
}

void launch_lattice_energy_table(Tables tab, const Tables32* tab32, const double* shell_tab, int S, LatZ z,
                                 const double* rho, double* etab, unsigned* err, cudaStream_t st) {
  Tables32 t{};
  if (tab32) t = *tab32;
  k_lattice_energy_table<<<1, 32, 0, st>>>(tab, t, tab32 ? 1 : 0, shell_tab, S, z, rho, etab, err);
}

void launch_shell_tables(Tables tab, const int* h2, const int* z, int S, double a, double* out,
                         unsigned* err, cudaStream_t st, const Tables32* tab32) {
  Tables32 t{};
  if (tab32) t = *tab32;
  k_shell_tables<<<1, 32, 0, st>>>(tab, t, tab32 ? 1 : 0, h2, z, S, a, out, err);
}

// --------------------------------------------------- lattice neighbours
// Site (cx, cy, cz, b) has half-lattice coordinates H = 2 c + b; the
// neighbour at offset h has coordinates H + h (periodic in 2 n), basis
// (H + h) mod 2 and cell (H + h) / 2.
__global__ void k_lattice_nbr(int nx, int ny, int nz, const int3* hoff, int K, int* nbr, int* cnt) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const long long N = 2LL * nx * ny * nz;
  if (i >= N) return;
  const int b = (int)(i & 1);
  const long long cell = i >> 1;
  const int cx = (int)(cell % nx), cy = (int)((cell / nx) % ny), cz = (int)(cell / ((long long)nx * ny));
  const int X = 2 * cx + b, Y = 2 * cy + b, Z = 2 * cz + b;
  for (int k = 0; k < K; ++k) {
    const int3 h = hoff[k];
    int hx = (X + h.x) % (2 * nx); if (hx < 0) hx += 2 * nx;
    int hy = (Y + h.y) % (2 * ny); if (hy < 0) hy += 2 * ny;
    int hz = (Z + h.z) % (2 * nz); if (hz < 0) hz += 2 * nz;
    const int bb = hx & 1;
    const long long j = (((long long)(hz >> 1) * ny + (hy >> 1)) * nx + (hx >> 1)) * 2 + bb;
    nbr[i * K + k] = (int)j;
  }
  cnt[i] = K;
}

void launch_lattice_neighbours(int nx, int ny, int nz, const int3* hoff, int K, int* nbr, int* cnt,
                               cudaStream_t st) {
  const long long N = 2LL * nx * ny * nz;
  k_lattice_nbr<<<(unsigned)((N + 127) / 128), 128, 0, st>>>(nx, ny, nz, hoff, K, nbr, cnt);
}

// ------------------------------------------------------ cell neighbours
// periodic image of v in [0, L): positions outside the box (a caller's, or
// one rounding step past an edge) are binned where their image lies
__device__ __forceinline__ double wrap_into(double v, double L) {
  const double w = v - L * floor(v / L);
  return w < L ? w : 0.0;  // v a hair below a multiple of L rounds up to L
}

// (int)(w / L * n), clamped; the product with 1 / L decides unless it lies so
// near a whole number that the division could round to the other side
__device__ __forceinline__ int cell_index(double w, double L, double n_over_L, int n) {
  const double u = w * n_over_L, fl = floor(u), t = u - fl;
  const int c = t > 1e-6 && t < 1.0 - 1e-6 ? (int)fl : (int)(w / L * n);
  return c < n ? c : n - 1;
}

// wrapped coordinate; the division (a dozen FP64 instructions) only outside
__device__ __forceinline__ double wrap_cell(double v, double L) { return v >= 0.0 && v < L ? v : wrap_into(v, L); }

__global__ void __launch_bounds__(128) k_cell_assign(long long N, const double* x, const double* y, const double* z,
                                                     double bx, double by, double bz, double nbx, double nby,
                                                     double nbz, int nx, int ny, int nz, int* cell_of, int* count) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= N) return;
  const int cx = cell_index(wrap_cell(x[i], bx), bx, nbx, nx);
  const int cy = cell_index(wrap_cell(y[i], by), by, nby, ny);
  const int cz = cell_index(wrap_cell(z[i], bz), bz, nbz, nz);
  const int c = (cz * ny + cy) * nx + cx;
  cell_of[i] = c;
  atomicAdd(&count[c], 1);
}

// exclusive scan of count[0..n) into start[0..n], one block, SCAN_ITEMS
// consecutive counts per thread (a chain of n / 8192 block scans); count and
// start are 16-byte aligned
constexpr int SCAN_ITEMS = 8;
__global__ void __launch_bounds__(1024) k_scan(const int* count, int n, int* start) {
  __shared__ int warp_sum[32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  int carry = 0;
  for (int base = 0; base < n; base += 1024 * SCAN_ITEMS) {
    const int i0 = base + threadIdx.x * SCAN_ITEMS;
    __align__(16) int v[SCAN_ITEMS];
    int own = 0;
    const bool full = i0 + SCAN_ITEMS <= n;
    if (full) {
      *reinterpret_cast<int4*>(v) = *reinterpret_cast<const int4*>(count + i0);
      *reinterpret_cast<int4*>(v + 4) = *reinterpret_cast<const int4*>(count + i0 + 4);
    } else {
#pragma unroll
      for (int q = 0; q < SCAN_ITEMS; ++q) v[q] = i0 + q < n ? count[i0 + q] : 0;
    }
#pragma unroll
    for (int q = 0; q < SCAN_ITEMS; ++q) own += v[q];
    int s = own;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int q = __shfl_up_sync(0xffffffffu, s, o);
      if (lane >= o) s += q;
    }
    __syncthreads();  // warp_sum is read by the round before
    if (lane == 31) warp_sum[w] = s;
    __syncthreads();
    int ws = warp_sum[lane];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int q = __shfl_up_sync(0xffffffffu, ws, o);
      if (lane >= o) ws += q;
    }
    int at = carry + s - own + (w ? __shfl_sync(0xffffffffu, ws, w - 1) : 0);
#pragma unroll
    for (int q = 0; q < SCAN_ITEMS; ++q) {
      const int own_start = at;
      at += v[q];
      v[q] = own_start;
    }
    if (full) {
      *reinterpret_cast<int4*>(start + i0) = *reinterpret_cast<int4*>(v);
      *reinterpret_cast<int4*>(start + i0 + 4) = *reinterpret_cast<int4*>(v + 4);
    } else {
#pragma unroll
      for (int q = 0; q < SCAN_ITEMS; ++q)
        if (i0 + q < n) start[i0 + q] = v[q];
    }
    carry += __shfl_sync(0xffffffffu, ws, 31);
  }
  if (threadIdx.x == 0) start[n] = carry;
}

__global__ void k_cell_scatter(long long N, const int* cell_of, const int* start, int* cursor, int* sorted) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= N) return;
  const int c = cell_of[i];
  sorted[start[c] + atomicAdd(&cursor[c], 1)] = (int)i;
}

// Order each bin's members by index in place (the tables are the same whatever
// order the scatter's atomics took): a block per bin ranks them in shared
// memory; 512 domains of 170 atoms took 700 us with a thread per bin.
// Larger bins are sorted by one thread as they lie.
constexpr int SORT_CAP = 4096;
__global__ void __launch_bounds__(256) k_sort_bins(const int* start, int* sorted) {
  __shared__ int s_v[SORT_CAP];
  const int b = start[blockIdx.x], n = start[blockIdx.x + 1] - b;
  int* v = sorted + b;
  if (n > SORT_CAP) {
    if (threadIdx.x == 0)
      for (int p = 1; p < n; ++p) {
        const int e = v[p];
        int q = p - 1;
        while (q >= 0 && v[q] > e) {
          v[q + 1] = v[q];
          --q;
        }
        v[q + 1] = e;
      }
    return;
  }
  for (int p = threadIdx.x; p < n; p += 256) s_v[p] = v[p];
  __syncthreads();
  for (int p = threadIdx.x; p < n; p += 256) {
    const int e = s_v[p];
    int rank = 0;
    for (int q = 0; q < n; ++q) rank += s_v[q] < e;
    v[rank] = e;
  }
}

// Cell-sorted atoms: (x, y, z, index) of each cell's members in ascending
// index, from their scattered order; a warp per cell ranks them.
__global__ void __launch_bounds__(128) k_cell_pack(int ncell, const int* start, const int* scattered, const double* x,
                                                   const double* y, const double* z, double bx, double by, double bz,
                                                   float4* p4) {
  const int c = (int)(((long long)blockIdx.x * 128 + threadIdx.x) >> 5), lane = threadIdx.x & 31;
  if (c >= ncell) return;
  const int b = start[c], n = start[c + 1] - b;
  for (int p = lane; p < n; p += 32) {
    const int i = scattered[b + p];
    int rank = 0;
    for (int q = 0; q < n; ++q) rank += scattered[b + q] < i;
    p4[b + rank] = make_float4((float)wrap_cell(x[i], bx), (float)wrap_cell(y[i], by), (float)wrap_cell(z[i], bz),
                               __int_as_float(i));
  }
}

// Candidates are tested in FP32 against (rl + m)^2, m = 0.01 A + 1e-6 L_max:
// the wrapped coordinates lie in [0, L), so the FP32 minimum-image distance
// is within about 7 L 2^-24 < 1e-6 L of the exact one, and every pair within
// rl is listed; the few extra pairs in [rl, rl + m) are skipped where the
// list is used (r >= r_c).
//
// A block per cell stages the 27 cells' atoms in shared memory (a thread per
// atom read them by index, 27 times each) and each of its warps tests them,
// 32 at a time, against NB_ATOMS of the cell's own atoms; the ballot places
// the neighbours in candidate order, so rows are written coalesced and come
// out by cell, then by index.  The half list (j > i, null: not wanted) is
// taken from the finished rows.  Bound by instruction issue (77 %), 15 per
// candidate and atom.  1.36 M atoms, both lists: 0.95 ms, 2.29 ms with a
// thread per atom and a pass of its own for the half list; the whole rebuild
// 2.6 -> 1.2 ms, of 86 k atoms 0.48 -> 0.11 ms.
constexpr int NB_CAP = 1024;  // candidates staged at a time (the usual 27 cells hold 400 to 600)
constexpr int NB_ATOMS = 4;
constexpr int NB_WARPS = 4;

// candidates s_c[0, nc), padded to a multiple of 32 with NaN, which no test
// passes (as no atom at NaN does: own[q] of a missing atom)
// NA: how many of own[] the warp has
template <bool WRAP, int NA>
__device__ __forceinline__ void cell_rows(const float4* s_c, int nc, const float4 (&own)[NB_ATOMS], int (&m)[NB_ATOMS],
                                          float bx, float by, float bz, float rl2, int K, int* nbr, int lane) {
  const float ibx = 1.0f / bx, iby = 1.0f / by, ibz = 1.0f / bz;
  const unsigned below = (1u << lane) - 1u;
  int* row[NA];
#pragma unroll
  for (int q = 0; q < NA; ++q) row[q] = nbr + (long long)__float_as_int(own[q].w) * K;
  for (int k0 = 0; k0 < nc; k0 += 32) {
    const float4 c = s_c[k0 + lane];
    const int j = __float_as_int(c.w);
#pragma unroll
    for (int q = 0; q < NA; ++q) {
      float dx = c.x - own[q].x, dy = c.y - own[q].y, dz = c.z - own[q].z;
      if (WRAP) {
        dx -= bx * rintf(dx * ibx);
        dy -= by * rintf(dy * iby);
        dz -= bz * rintf(dz * ibz);
      }
      const bool in = (dx * dx + dy * dy + dz * dz < rl2) & (j != __float_as_int(own[q].w));
      const unsigned bal = __ballot_sync(0xffffffffu, in);
      const int at = m[q] + __popc(bal & below);
      if (in & (at < K)) row[q][at] = j;
      m[q] += __popc(bal);
    }
  }
}

template <bool WRAP>
__device__ __forceinline__ void cell_rows_n(int na, const float4* s_c, int nc, const float4 (&own)[NB_ATOMS],
                                            int (&m)[NB_ATOMS], float bx, float by, float bz, float rl2, int K,
                                            int* nbr, int lane) {
  if (na >= 4) cell_rows<WRAP, 4>(s_c, nc, own, m, bx, by, bz, rl2, K, nbr, lane);
  else if (na == 3) cell_rows<WRAP, 3>(s_c, nc, own, m, bx, by, bz, rl2, K, nbr, lane);
  else if (na == 2) cell_rows<WRAP, 2>(s_c, nc, own, m, bx, by, bz, rl2, K, nbr, lane);
  else if (na == 1) cell_rows<WRAP, 1>(s_c, nc, own, m, bx, by, bz, rl2, K, nbr, lane);
}

__global__ void __launch_bounds__(32 * NB_WARPS) k_cell_nbr(const float4* p4, const int* start, float bx, float by,
                                                            float bz, int nx, int ny, int nz, float rl2, int K,
                                                            int* nbr, int* cnt, int* nbr_h, int* cnt_h,
                                                            unsigned* err) {
  __shared__ float4 s_c[NB_CAP];
  __shared__ int s_b[27], s_at[28];
  const int c = blockIdx.x, h0 = start[c], nh = start[c + 1] - h0;
  if (nh == 0) return;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int cx = c % nx, cy = (c / nx) % ny, cz = c / (nx * ny);
  if (w == 0) {
    int n = 0;
    if (lane < 27) {
      const int ox = lane % 3 - 1, oy = (lane / 3) % 3 - 1, oz = lane / 9 - 1;
      const int qx = (cx + ox + nx) % nx, qy = (cy + oy + ny) % ny, qz = (cz + oz + nz) % nz;
      const int q = (qz * ny + qy) * nx + qx;
      s_b[lane] = start[q];
      n = start[q + 1] - start[q];
    }
    int s = n;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int q = __shfl_up_sync(0xffffffffu, s, o);
      if (lane >= o) s += q;
    }
    if (lane < 28) s_at[lane] = s - n;
  }
  __syncthreads();
  const int total = s_at[27];
  // away from the faces no difference reaches half the box (five cells and
  // more), where the nearest image is the difference itself
  const bool inside = nx > 4 && ny > 4 && nz > 4 && cx > 0 && cx < nx - 1 && cy > 0 && cy < ny - 1 && cz > 0 &&
                      cz < nz - 1;
  for (int a0 = 0; a0 < nh; a0 += NB_WARPS * NB_ATOMS) {
    float4 own[NB_ATOMS];
    int m[NB_ATOMS];
#pragma unroll
    for (int q = 0; q < NB_ATOMS; ++q) {
      const int a = a0 + q * NB_WARPS + w;
      own[q] = a < nh ? p4[h0 + a] : make_float4(NAN, NAN, NAN, __int_as_float(-1));
      m[q] = 0;
    }
    for (int lo = 0; lo < total; lo += NB_CAP) {
      const int nc = total - lo < NB_CAP ? total - lo : NB_CAP, nc32 = (nc + 31) & ~31;
      if (a0 == 0 || total > NB_CAP) {
        __syncthreads();
        // candidate p is in the last cell that starts at or before it
        for (int p = lo + threadIdx.x; p < lo + nc32; p += 32 * NB_WARPS) {
          int q = 0;
#pragma unroll
          for (int o = 16; o > 0; o >>= 1)
            if (q + o < 27 && s_at[q + o] <= p) q += o;
          s_c[p - lo] = p < total ? p4[s_b[q] + p - s_at[q]] : make_float4(NAN, NAN, NAN, __int_as_float(-1));
        }
        __syncthreads();
      }
      const int na = (nh - a0 - w + NB_WARPS - 1) / NB_WARPS;
      if (inside) cell_rows_n<false>(na, s_c, nc, own, m, bx, by, bz, rl2, K, nbr, lane);
      else cell_rows_n<true>(na, s_c, nc, own, m, bx, by, bz, rl2, K, nbr, lane);
    }
#pragma unroll
    for (int q = 0; q < NB_ATOMS; ++q) {
      const int i = __float_as_int(own[q].w);
      if (i < 0) continue;
      const int mm = m[q] < K ? m[q] : K;
      int* row = nbr + (long long)i * K;
      for (int k = mm + lane; k < K; k += 32) row[k] = -1;
      if (lane == 0) {
        if (m[q] > K) atomicOr(err, ERRF_OVERFLOW);
        cnt[i] = mm;
      }
    }
    if (nbr_h) {
      __syncwarp();  // the rows are read back by other lanes than wrote them
#pragma unroll
      for (int q = 0; q < NB_ATOMS; ++q) {
        const int i = __float_as_int(own[q].w);
        if (i < 0) continue;
        const int mm = m[q] < K ? m[q] : K;
        const int* row = nbr + (long long)i * K;
        int* half = nbr_h + (long long)i * K;
        int mh = 0;
        for (int k0 = 0; k0 < mm; k0 += 32) {
          const int j = k0 + lane < mm ? row[k0 + lane] : -1;
          const unsigned bal = __ballot_sync(0xffffffffu, j > i);
          if (j > i) half[mh + __popc(bal & ((1u << lane) - 1u))] = j;
          mh += __popc(bal);
        }
        if (lane == 0) cnt_h[i] = mh;
      }
    }
  }
}

void launch_cell_neighbours(long long N, const double* x, const double* y, const double* z,
                            const double box[3], double rl, CellList cl, int K, int* nbr, int* cnt,
                            int* nbr_h, int* cnt_h, unsigned* err, cudaStream_t st) {
  const int ncell = cl.nc[0] * cl.nc[1] * cl.nc[2];
  const unsigned g = (unsigned)((N + 127) / 128);
  cudaMemsetAsync(cl.cell_count, 0, sizeof(int) * ncell, st);
  cudaMemsetAsync(cl.cell_cursor, 0, sizeof(int) * ncell, st);
  k_cell_assign<<<g, 128, 0, st>>>(N, x, y, z, box[0], box[1], box[2], cl.nc[0] / box[0], cl.nc[1] / box[1],
                                   cl.nc[2] / box[2], cl.nc[0], cl.nc[1], cl.nc[2], cl.cell_of, cl.cell_count);
  k_scan<<<1, 1024, 0, st>>>(cl.cell_count, ncell, cl.cell_start);
  // the rows (at least N integers) hold the scattered order until they are written
  k_cell_scatter<<<g, 128, 0, st>>>(N, cl.cell_of, cl.cell_start, cl.cell_cursor, nbr);
  k_cell_pack<<<(unsigned)(((long long)ncell * 32 + 127) / 128), 128, 0, st>>>(ncell, cl.cell_start, nbr, x, y, z, box[0],
                                                                              box[1], box[2], cl.p4);
  const float rlm = (float)(rl + cell_list_margin(box));
  k_cell_nbr<<<ncell, 32 * NB_WARPS, 0, st>>>(cl.p4, cl.cell_start, (float)box[0], (float)box[1], (float)box[2],
                                              cl.nc[0], cl.nc[1], cl.nc[2], rlm * rlm, K, nbr, cnt, nbr_h, cnt_h, err);
}

// ------------------------------------------------- spatial colour schedule
// Domain of every atom for the SPATIAL schedule (boxes of the periodic cell,
// Sec. III A): box index from floor(v / L * n) clamped to the grid -- the
// host's rule, so the tables are the same -- mapped to its domain rank
// (colour-major, then box index) by dom_of_block.
__device__ __forceinline__ int spatial_box(double v, double L, int n) {
  const int q = (int)floor(v / L * n);
  return q < 0 ? 0 : (q >= n ? n - 1 : q);
}

__global__ void k_spatial_assign(long long N, const double* x, const double* y, const double* z, double bx,
                                 double by, double bz, int nbx, int nby, int nbz, const int* dom_of_block,
                                 int* dom_of, int* count) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= N) return;
  const int b = (spatial_box(z[i], bz, nbz) * nby + spatial_box(y[i], by, nby)) * nbx + spatial_box(x[i], bx, nbx);
  const int d = dom_of_block[b];
  dom_of[i] = d;
  atomicAdd(&count[d], 1);
}

void launch_spatial_schedule(long long N, const double* x, const double* y, const double* z, const double box[3],
                             const int nb[3], const int* dom_of_block, int ndom, int* dom_of, int* count,
                             int* cursor, int* dom_start, int* dom_sites, cudaStream_t st) {
  const unsigned g = (unsigned)((N + 127) / 128);
  cudaMemsetAsync(count, 0, sizeof(int) * ndom, st);
  cudaMemsetAsync(cursor, 0, sizeof(int) * ndom, st);
  k_spatial_assign<<<g, 128, 0, st>>>(N, x, y, z, box[0], box[1], box[2], nb[0], nb[1], nb[2], dom_of_block, dom_of,
                                      count);
  // counting sort by domain, ascending atom index within a domain (the
  // cell-list kernels with domains as bins)
  k_scan<<<1, 1024, 0, st>>>(count, ndom, dom_start);
  k_cell_scatter<<<g, 128, 0, st>>>(N, dom_of, dom_start, cursor, dom_sites);
  k_sort_bins<<<ndom, 256, 0, st>>>(dom_start, dom_sites);
}

// ------------------------------------------------------ density, energy
__device__ __forceinline__ double pair_r(const McArgs& a, bool shell, int i, int k, int j, int s) {
  if (shell) return a.shell_tab[1 + 2 * a.n_shells + s];
  double dx = a.x[j] - a.x[i], dy = a.y[j] - a.y[i], dz = a.z[j] - a.z[i];
  dx -= a.box[0] * rint(dx / a.box[0]);
  dy -= a.box[1] * rint(dy / a.box[1]);
  dz -= a.box[2] * rint(dz / a.box[2]);
  const double r2 = dx * dx + dy * dy + dz * dz;
  return r2 * rsqrt_nr(r2);
}

// FP32 distance of pair (i, j) for the mixed form (r_s on the rigid lattice)
__device__ __forceinline__ float pair_r32(const McArgs& a, bool shell, int i, int j, int s) {
  if (shell) return (float)a.shell_tab[1 + 2 * a.n_shells + s];
  const float dx = fix_diff(a.ux[j], a.ux[i], a.ul[0]);
  const float dy = fix_diff(a.uy[j], a.uy[i], a.ul[1]);
  const float dz = fix_diff(a.uz[j], a.uz[i], a.ul[2]);
  return sqrtf(dx * dx + dy * dy + dz * dz);
}

// table q at the pair distance: FP64, or FP32 widened to FP64 (mixed)
template <bool MIXED>
__device__ __forceinline__ double pair_tab(const McArgs& a, int q, double r64, float r32) {
  if constexpr (MIXED) {
    float t;
    const int j = spline32_locate(a.tab32.sp[q], r32, t, a.err);
    return (double)spline32_val_at(a.tab32.sp[q], j, t);
  } else {
    return spline_val(a.tab.sp[q], r64, a.err);
  }
}

// rho_i = sum_k f_{t_k}(r_ik) (FP64 sum); dF_i = F_B(rho_i) - F_A(rho_i) (FP64)
template <bool SHELL, bool MIXED>
__global__ void k_rho(McArgs a, int r, double* dF) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= a.N) return;
  const uint8_t* ty = a.types + (long long)r * a.N;
  const int* row = a.nbr + i * a.K;
  const int cnt = a.nbr_cnt[i];
  double rho = 0.0;
  int s = 0;
  for (int k = 0; k < cnt; ++k) {
    if (SHELL) while (k >= a.shell_end[s]) ++s;
    const int j = row[k];
    double rr = 0.0;
    float rf = 0.0f;
    if (MIXED) {
      rf = pair_r32(a, SHELL, (int)i, j, s);
      if (rf >= (float)a.rc) continue;
    } else {
      rr = pair_r(a, SHELL, (int)i, k, j, s);
      if (rr >= a.rc) continue;
    }
    rho += pair_tab<MIXED>(a, 3 + ty[j], rr, rf);
  }
  double* out = a.rho + (a.rho_per_rep ? (long long)r * a.N : 0);
  out[i] = rho;
  if (dF) dF[i] = spline_val(a.tab.sp[6], rho, a.err) - spline_val(a.tab.sp[5], rho, a.err);
}

void launch_rho(const McArgs& a, bool shell, int r, cudaStream_t st) {
  const unsigned g = (unsigned)((a.N + 127) / 128);
  double* dF = const_cast<double*>(a.dF);
  if (a.mixed && !shell) launch_fix_positions(a.N, a.x, a.y, a.z, a.box, a.ux, a.uy, a.uz, st);
  if (a.mixed) {
    if (shell) k_rho<true, true><<<g, 128, 0, st>>>(a, r, dF);
    else k_rho<false, true><<<g, 128, 0, st>>>(a, r, dF);
  } else {
    if (shell) k_rho<true, false><<<g, 128, 0, st>>>(a, r, dF);
    else k_rho<false, false><<<g, 128, 0, st>>>(a, r, dF);
  }
}

constexpr int E_BLOCK = 256;
int energy_blocks(long long N) { return (int)((N + E_BLOCK - 1) / E_BLOCK); }

// e_i = 1/2 sum_k phi_{t_i t_k}(r_ik) + F_{t_i}(rho_i), block partial sums
template <bool SHELL, bool MIXED>
__global__ void __launch_bounds__(E_BLOCK) k_energy(McArgs a, int r, double* part) {
  const long long i = (long long)blockIdx.x * E_BLOCK + threadIdx.x;
  double e = 0.0;
  if (i < a.N) {
    const uint8_t* ty = a.types + (long long)r * a.N;
    const int* row = a.nbr + i * a.K;
    const int cnt = a.nbr_cnt[i];
    const int ti = ty[i];
    double rho = 0.0, ph = 0.0;
    int s = 0;
    const PairBox box = pair_box(a.box);
    const double xi = a.x[i], yi = a.y[i], zi = a.z[i], rc2 = a.rc * a.rc;
    for (int k = 0; k < cnt; ++k) {
      if (SHELL) while (k >= a.shell_end[s]) ++s;
      const int j = row[k];
      double rr = 0.0;
      float rf = 0.0f;
      if (!SHELL && !MIXED) {
        // explicit positions in FP64: one distance (pair_r2, sqrt3) and one
        // interval for both tables, 18 FP64 operations per pair where three
        // divisions and two table lookups took 80; 86 k atoms 898 -> 318 us
        double dx = a.x[j] - xi, dy = a.y[j] - yi, dz = a.z[j] - zi, ir, t;
        const double r2 = pair_r2(box, dx, dy, dz);
        if (outside(r2, rc2)) continue;
        rr = sqrt3(r2, ir);
        if (!not_finite(rr)) {
          const int tj = ty[j], q = locate_in(a.tab.sp[0], rr, t);
          ph += spline_val_at(a.tab.sp[ti + tj], q, t);
          rho += spline_val_at(a.tab.sp[3 + tj], q, t);
          continue;
        }
      } else if (MIXED) {
        rf = pair_r32(a, SHELL, (int)i, j, s);
        if (rf >= (float)a.rc) continue;
      } else {
        rr = pair_r(a, SHELL, (int)i, k, j, s);
        if (rr >= a.rc) continue;
      }
      const int tj = ty[j];
      ph += pair_tab<MIXED>(a, ti + tj, rr, rf);
      rho += pair_tab<MIXED>(a, 3 + tj, rr, rf);
    }
    e = 0.5 * ph + spline_val(a.tab.sp[5 + ti], rho, a.err);
  }
  __shared__ double sh[E_BLOCK / 32];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) e += __shfl_xor_sync(0xffffffffu, e, o);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = e;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < E_BLOCK / 32; ++w) t += sh[w];
    part[blockIdx.x] = t;
  }
}

void launch_energy(const McArgs& a, bool shell, int r, double* part, cudaStream_t st) {
  const int g = energy_blocks(a.N);
  if (a.mixed && !shell) launch_fix_positions(a.N, a.x, a.y, a.z, a.box, a.ux, a.uy, a.uz, st);
  if (a.mixed) {
    if (shell) k_energy<true, true><<<g, E_BLOCK, 0, st>>>(a, r, part);
    else k_energy<false, true><<<g, E_BLOCK, 0, st>>>(a, r, part);
  } else {
    if (shell) k_energy<true, false><<<g, E_BLOCK, 0, st>>>(a, r, part);
    else k_energy<false, false><<<g, E_BLOCK, 0, st>>>(a, r, part);
  }
}

// ---------------------------------- densities and energy, five-shell lattice
// A site's neighbours lie on five shells, so its density and its pair energy
// depend on the B counts b_s of the shells alone:
//   rho_i = sum_s [(z_s - b_s) f_A(r_s) + b_s f_B(r_s)]: five table entries;
//   sum of pairs = 1/2 sum_s {z_s [N phi_AA + 2 n_B (phi_AB - phi_AA)] + (phi_BB -
//   2 phi_AB + phi_AA) P_s}(r_s), P_s = sum over B sites of b_s: whole numbers.
// Per site that leaves the embedding cubic and five additions in FP64 (GB300
// has 2 FP64 lanes per SM and clock), against two table cubics for each of 58
// neighbours: 80^3 x 8 replicas, densities and energies 28.5 -> 0.4 ms.  Every
// replica in one launch.  shell: f_A, f_B, phi_AA, phi_AB, phi_BB at the five
// radii.  part[r][blocks]: sums of F over a block's sites; tot[r][6]: P_s, n_B.
constexpr int SS_BLOCK = 256, SS_SITES = 4;

__global__ void k_shell_values(Tables tab, Tables32 tab32, int mixed, const double* shell_tab, double* out,
                               unsigned* err) {
  const int s = threadIdx.x;
  if (s >= 5) return;
  const Tables32* t32 = mixed ? &tab32 : nullptr;
  const double r = shell_tab[11 + s];
  const int q[5] = {3, 4, 0, 1, 2};
  for (int k = 0; k < 5; ++k) out[5 * k + s] = tab_val(tab, t32, q[k], r, err);
}

void launch_shell_values(const McArgs& a, double* out, cudaStream_t st) {
  k_shell_values<<<1, 32, 0, st>>>(a.tab, a.tab32, a.mixed, a.shell_tab, out, a.err);
}

template <int B>
__device__ __forceinline__ void shell_counts(const uint8_t* ty, int nx, int ny, int nz, int cx, int cy, int cz,
                                             int (&b)[5]) {
  int xo[5], yo[5], zo[5];
#pragma unroll
  for (int d = -2; d <= 2; ++d) {
    const int X = cx + d, Y = cy + d, Z = cz + d;
    xo[d + 2] = 2 * (X < 0 ? X + nx : (X >= nx ? X - nx : X));
    yo[d + 2] = 2 * nx * (Y < 0 ? Y + ny : (Y >= ny ? Y - ny : Y));
    zo[d + 2] = 2 * nx * ny * (Z < 0 ? Z + nz : (Z >= nz ? Z - nz : Z));
  }
#pragma unroll
  for (int s = 0; s < 5; ++s) b[s] = 0;
#pragma unroll
  for (int k = 0; k < MK_BCC5_N; ++k) {
    const int code = mk_bcc5_code(k);
    const int hx = (code & 15) - 4, hy = ((code >> 4) & 15) - 4, hz = ((code >> 8) & 15) - 4;
    const int bb = B ^ (hx & 1);
    b[code >> 12] += ty[zo[((B + hz - bb) >> 1) + 2] + yo[((B + hy - bb) >> 1) + 2] + xo[((B + hx - bb) >> 1) + 2] + bb];
  }
}

__global__ void __launch_bounds__(SS_BLOCK)
    k_shell_state(McArgs a, int nx, int ny, int nz, const double* shell, int r0, double* rho, double* part,
                  unsigned long long* tot) {
  const int r = r0 + blockIdx.y;
  __shared__ double s_t[5][25];  // (z - b) f_A + b f_B
  __shared__ double s_e[SS_BLOCK / 32];
  for (int q = threadIdx.x; q < 125; q += SS_BLOCK) {
    constexpr int z[5] = {8, 6, 12, 24, 8};
    const int s = q / 25, b = q - 25 * s;
    s_t[s][b] = b <= z[s] ? (double)(z[s] - b) * shell[s] + (double)b * shell[5 + s] : 0.0;
  }
  __syncthreads();
  const uint8_t* ty = a.types + (long long)r * a.N;
  // a warp takes sites of one basis (its lanes run one of the two unrolled
  // neighbour tables): site 2 cell + basis
  double e = 0.0;
  int P[6] = {0, 0, 0, 0, 0, 0};
  const long long half = a.N >> 1;
#pragma unroll 1
  for (int u = 0; u < SS_SITES; ++u) {
    const long long cell = ((long long)blockIdx.x * (SS_SITES / 2) + (u >> 1)) * SS_BLOCK + threadIdx.x;
    const int basis = u & 1;
    if (cell >= half) continue;
    const int cx = (int)(cell % nx), cyz = (int)(cell / nx);
    const int cy = cyz % ny, cz = cyz / ny;
    int b[5];
    if (basis) shell_counts<1>(ty, nx, ny, nz, cx, cy, cz, b);
    else shell_counts<0>(ty, nx, ny, nz, cx, cy, cz, b);
    double d = s_t[0][b[0]];
#pragma unroll
    for (int s = 1; s < 5; ++s) d += s_t[s][b[s]];
    const long long i = 2 * cell + basis;
    if (rho) rho[(long long)r * a.N + i] = d;
    const int t = ty[i];
    e += spline_val(a.tab.sp[5 + t], d, a.err);
    if (t) {
#pragma unroll
      for (int s = 0; s < 5; ++s) P[s] += b[s];
      P[5] += 1;
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) e += __shfl_xor_sync(0xffffffffu, e, o);
  if ((threadIdx.x & 31) == 0) s_e[threadIdx.x >> 5] = e;
#pragma unroll
  for (int s = 0; s < 6; ++s) {
    const int v = __reduce_add_sync(0xffffffffu, P[s]);
    if ((threadIdx.x & 31) == 0 && v) atomicAdd(tot + 6 * blockIdx.y + s, (unsigned long long)v);
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double v = 0.0;
    for (int w = 0; w < SS_BLOCK / 32; ++w) v += s_e[w];
    part[(long long)blockIdx.y * gridDim.x + blockIdx.x] = v;
  }
}

int shell_state_blocks(long long N) {
  const long long per = (long long)SS_BLOCK * (SS_SITES / 2);
  return (int)((N / 2 + per - 1) / per);
}

void launch_shell_state(const McArgs& a, const int n3[3], const double* shell, int r0, int nrep, double* rho,
                        double* part, unsigned long long* tot, cudaStream_t st) {
  cudaMemsetAsync(tot, 0, sizeof(unsigned long long) * 6 * nrep, st);
  k_shell_state<<<dim3((unsigned)shell_state_blocks(a.N), (unsigned)nrep), SS_BLOCK, 0, st>>>(
      a, n3[0], n3[1], n3[2], shell, r0, rho, part, tot);
}

}  // namespace vcsgc
