// kernels_md.cu -- EAM forces and BAOAB Langevin velocity Verlet, the MD half
// of the hybrid MC/MD scheme (Sec. IV A of Sadigh et al.).
//   rho pass:   rho_i = sum_j f_{t_j}(r_ij), F'(rho_i), F_B(rho_i) - F_A(rho_i)
//   force pass: F_i = sum_j [phi'_{t_i t_j} + F'_i f'_{t_j} + F'_j f'_{t_i}](r_ij) (x_j - x_i)/r_ij
//   B A O A B:  half kick, half drift, Ornstein-Uhlenbeck velocity update with
//               Philox normals, half drift, (forces), half kick.
#include "common.cuh"
#include "kernels.h"

namespace vcsgc {

__device__ __forceinline__ double mimg(double d, double L, double iL) { return d - L * rint(d * iL); }

template <bool MIXED>
__global__ void k_md_rho(MdArgs m) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= m.N) return;
  const int* row = m.nbr + i * m.K;
  const int cnt = m.nbr_cnt[i];
  const double xi = m.x[i], yi = m.y[i], zi = m.z[i];
  const uint32_t uxi = MIXED ? m.ux[i] : 0u, uyi = MIXED ? m.uy[i] : 0u, uzi = MIXED ? m.uz[i] : 0u;
  const double ix = 1.0 / m.box[0], iy = 1.0 / m.box[1], iz = 1.0 / m.box[2];
  const double rc2 = m.rc * m.rc;
  double rho = 0.0;
  for (int k = 0; k < cnt; ++k) {
    const int j = row[k];
    if constexpr (MIXED) {
      const float dx = fix_diff(m.ux[j], uxi, m.ul[0]);
      const float dy = fix_diff(m.uy[j], uyi, m.ul[1]);
      const float dz = fix_diff(m.uz[j], uzi, m.ul[2]);
      const float r2 = dx * dx + dy * dy + dz * dz;
      if (r2 >= (float)rc2) continue;
      float t;
      const Spline32& sp = m.tab32.sp[3 + m.types[j]];
      const int q = spline32_locate(sp, sqrtf(r2), t, m.err);
      rho += (double)spline32_val_at(sp, q, t);
    } else {
      const double dx = mimg(m.x[j] - xi, m.box[0], ix);
      const double dy = mimg(m.y[j] - yi, m.box[1], iy);
      const double dz = mimg(m.z[j] - zi, m.box[2], iz);
      const double r2 = dx * dx + dy * dy + dz * dz;
      if (r2 >= rc2) continue;
      rho += spline_val(m.tab.sp[3 + m.types[j]], r2 * rsqrt_nr(r2), m.err);
    }
  }
  m.rho[i] = rho;
  double t;
  const int ti = m.types[i];
  const int q = spline_locate(m.tab.sp[5 + ti], rho, t, m.err);
  m.dFp[i] = spline_der_at(m.tab.sp[5 + ti], q, t);
  if (MIXED) m.dFp32[i] = (float)m.dFp[i];
  m.dF[i] = spline_val_at(m.tab.sp[6], q, t) - spline_val_at(m.tab.sp[5], q, t);
}
// Position and species of every atom in one 32-byte record (FP64 passes) or
// one 16-byte one (mixed): a neighbour is one sector instead of four.
__global__ void k_md_records(MdArgs m) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= m.N) return;
  if (m.mixed) m.u4[i] = make_uint4(m.ux[i], m.uy[i], m.uz[i], (uint32_t)m.types[i]);
  else {
    const Cubic p{m.x[i], m.y[i], m.z[i], __hiloint2double(0, (int)m.types[i])};
    m.p4[i] = p;
    if (m.pair_ui) m.f4[i] = make_float4((float)p.x, (float)p.y, (float)p.z, 0.0f);
  }
}
__device__ __forceinline__ int record_type(const Cubic& p) { return __double2loint(p.w); }

// sum of v over the LPA lanes of an atom (every lane of the warp takes part)
template <int LPA>
__device__ __forceinline__ double lane_sum(double v) {
#pragma unroll
  for (int o = LPA / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// The passes on the half list (each pair once, j > i) give LPA lanes to an
// atom: they share its row, so a warp's rows differ less in length (8 atoms
// instead of 32) and a row of 30 is a chain of 8 pairs instead of 30.
//
// FP64: bound by the FP64 pipe (86 % active), 16 instructions per pair for the
// density and 26 for the force where the straightforward form took 31 and 46.
// 1.36 M atoms, 39 M pairs within the cutoff: density 1.80 ms, force 2.97 ms, a
// whole step 10.2 -> 5.8 ms; mixed 2.81 -> 2.06 ms.  They serve single forces
// and what has no memory for pair blocks (below).
// rho_i and rho_j both receive the pair's density (atomic adds into rho, zeroed
// before); with one density function (SAME) one table value serves both ends.
template <int LPA, bool SAME>
__global__ void __launch_bounds__(128) k_md_rho_half(MdArgs m) {
  const long long g = (long long)blockIdx.x * 128 + threadIdx.x;
  const long long i = g / LPA;
  const int sub = (int)(g % LPA);
  const bool live = i < m.N;
  const int* row = m.nbr_h + (live ? i : 0) * m.K;
  const int cnt = live ? m.cnt_h[i] : 0;
  const Cubic pi = m.p4[live ? i : 0];
  const PairBox box = pair_box(m.box);
  const double rc2 = m.rc * m.rc;
  const int ti = record_type(pi);
  double rho = 0.0;
  for (int k = sub; k < cnt; k += LPA) {
    const int j = row[k];
    const Cubic pj = m.p4[j];
    double dx = pj.x - pi.x, dy = pj.y - pi.y, dz = pj.z - pi.z;
    const double r2 = pair_r2(box, dx, dy, dz);
    if (outside(r2, rc2)) continue;
    double ir, t;
    const double r = sqrt3(r2, ir);
    const int q = locate_in(m.tab.sp[3], r, t);
    const double fj = spline_val_at(m.tab.sp[SAME ? 3 : 3 + record_type(pj)], q, t);  // density of j at i
    const double fi = SAME ? fj : spline_val_at(m.tab.sp[3 + ti], q, t);
    rho += fj;
    atomicAdd(m.rho + j, fi);
  }
  rho = lane_sum<LPA>(rho);
  if (live && sub == 0) atomicAdd(m.rho + i, rho);
}

// warp sum of the per-thread virial terms, one atomic per warp (every lane
// of the warp reaches this point)
__device__ __forceinline__ void add_virial(const MdArgs& m, double vir) {
  if (!m.vir) return;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) vir += __shfl_xor_sync(0xffffffffu, vir, o);
  if ((threadIdx.x & 31) == 0 && vir != 0.0) atomicAdd(m.vir, vir);
}

// The same passes with pair blocks (MD proper).  Rows differ in length (29 on
// average, deviation 9 near a crystal's faces) and hold pairs beyond r_c, so
// that a warp's FP64 lanes were 65 % full, and the force pass formed every r
// and 1 / r again.  Here a warp takes the rows of GROUP atoms:
//  1. it screens them in FP32, a row at a time (a margin keeps every pair within
//     r_c; the FP32 pipe is 30 times as wide), into one list in shared memory;
//  2. each lane takes an equal stretch of that list, so all lanes are busy but
//     in the last row, sums an atom's density over its stretch and adds it when
//     the stretch passes on to the next atom;
//  3. r (in table intervals) and 1 / r stay in the pair block, stored lane by
//     lane as the force pass reads them, which then needs 17 FP64 operations
//     per pair instead of 26, for 40 bytes of memory traffic.
// Both are bound by the FP64 pipe.  1.36 M atoms: density 1.80 -> 1.42 ms, force
// 2.97 -> 1.41, a whole step 5.6 -> 3.6 ms.
constexpr int PAIR_LIST = 544;  // longest list; taken when more than PAIR_LIST - 32 are in it
constexpr double PAIR_NONE = -1.0;
constexpr uint32_t PAIR_ATOM = (1u << 28) - 1u;

template <int GROUP, bool SAME>
__global__ void __launch_bounds__(128) k_md_rho_pairs(MdArgs m) {
  __shared__ uint32_t s_list[4][PAIR_LIST];
  __shared__ Cubic s_p[4][GROUP];
  __shared__ float4 s_f[4][GROUP];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const long long grp = (long long)blockIdx.x * 4 + w, i0 = grp * GROUP;
  if (i0 >= m.N) return;
  const int na = m.N - i0 < GROUP ? (int)(m.N - i0) : GROUP;
  int cnt = 0;
  if (lane < na) {
    cnt = m.cnt_h[i0 + lane];
    s_p[w][lane] = m.p4[i0 + lane];
    s_f[w][lane] = m.f4[i0 + lane];
  }
  __syncwarp();
  const PairBox box = pair_box(m.box);
  const double rc2 = m.rc * m.rc;
  const float bx = (float)m.box[0], by = (float)m.box[1], bz = (float)m.box[2];
  const float bm = bx > by ? (bx > bz ? bx : bz) : (by > bz ? by : bz);
  const float rm = (float)m.rc + 0.01f + 1e-6f * bm, rm2 = rm * rm;
  const unsigned below = (1u << lane) - 1u;
  uint32_t* list = s_list[w];
  const long long p0 = 32ll * m.pair_off[grp];
  int rows = 0, T = 0;

  const auto take = [&]() {
    __syncwarp();
    const int per = (T + 31) >> 5, e0 = lane * per;
    int cur = -1;
    double rho = 0.0;
    Cubic pi{};
    for (int it = 0; it < per; ++it) {
      const int e = e0 + it;
      const long long at = p0 + 32ll * (rows + it) + lane;
      double2 keep = make_double2(PAIR_NONE, 0.0);
      if (e < T) {
        const uint32_t v = list[e];
        const int a = (int)(v >> 28), j = (int)(v & PAIR_ATOM);
        if (a != cur) {
          if (cur >= 0) atomicAdd(m.rho + i0 + cur, rho);
          cur = a;
          rho = 0.0;
          pi = s_p[w][a];
        }
        const Cubic pj = m.p4[j];
        double dx = pj.x - pi.x, dy = pj.y - pi.y, dz = pj.z - pi.z;
        const double r2 = pair_r2(box, dx, dy, dz);
        m.pair_j[at] = v;
        if (!outside(r2, rc2)) {
          double ir, t;
          const double u = sqrt3(r2, ir) * m.tab.sp[3].inv_h;
          const int q = locate_u(m.tab.sp[3], u, t);
          keep = make_double2(u, ir);
          const double fj = spline_val_at(m.tab.sp[SAME ? 3 : 3 + record_type(pj)], q, t);  // density of j at i
          const double fi = SAME ? fj : spline_val_at(m.tab.sp[3 + record_type(pi)], q, t);
          rho += fj;
          atomicAdd(m.rho + j, fi);
        }
      }
      m.pair_ui[at] = keep;
    }
    if (cur >= 0) atomicAdd(m.rho + i0 + cur, rho);
    rows += per;
    T = 0;
    __syncwarp();
  };

#pragma unroll 2
  for (int a = 0; a < na; ++a) {
    const int n = __shfl_sync(0xffffffffu, cnt, a);
    const int* row = m.nbr_h + (i0 + a) * m.K;
    const float4 fi = s_f[w][a];
    for (int k0 = 0; k0 < n; k0 += 32) {
      int j = 0;
      bool near = false;
      if (k0 + lane < n) {
        j = row[k0 + lane];
        const float4 f = m.f4[j];
        float dx = fabsf(f.x - fi.x), dy = fabsf(f.y - fi.y), dz = fabsf(f.z - fi.z);
        dx = dx > 0.5f * bx ? bx - dx : dx;
        dy = dy > 0.5f * by ? by - dy : dy;
        dz = dz > 0.5f * bz ? bz - dz : dz;
        near = !(dx * dx + dy * dy + dz * dz >= rm2);  // NaN goes on to the FP64 test
      }
      const unsigned bal = __ballot_sync(0xffffffffu, near);
      if (near) list[T + __popc(bal & below)] = (uint32_t)j | (uint32_t)a << 28;
      T += __popc(bal);
      if (T > PAIR_LIST - 32) take();
    }
  }
  if (T > 0) take();
  if (lane == 0) m.pair_rows[grp] = rows;
}

template <int GROUP, bool SAME, bool VIR>
__global__ void __launch_bounds__(128) k_md_force_pairs(MdArgs m) {
  __shared__ Cubic s_p[4][GROUP];
  __shared__ double s_F[4][GROUP];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const long long grp = (long long)blockIdx.x * 4 + w, i0 = grp * GROUP;
  if (i0 >= m.N) return;
  if (lane < GROUP && i0 + lane < m.N) {
    s_p[w][lane] = m.p4[i0 + lane];
    s_F[w][lane] = m.dFp[i0 + lane];
  }
  __syncwarp();
  const int rows = m.pair_rows[grp];
  const long long p0 = 32ll * m.pair_off[grp] + lane;
  const PairBox box = pair_box(m.box);
  double fx = 0.0, fy = 0.0, fz = 0.0, vir = 0.0, Fi = 0.0;
  Cubic pi{};
  int cur = -1;
  bool bad = false;
  const auto flush = [&]() {
    bad |= not_finite(fx) | not_finite(fy) | not_finite(fz);
    atomicAdd(m.fx + i0 + cur, fx);
    atomicAdd(m.fy + i0 + cur, fy);
    atomicAdd(m.fz + i0 + cur, fz);
  };
  for (int it = 0; it < rows; ++it) {
    const double2 ui = m.pair_ui[p0 + 32ll * it];
    if (__double2hiint(ui.x) == __double2hiint(PAIR_NONE)) continue;
    const uint32_t v = m.pair_j[p0 + 32ll * it];
    const int a = (int)(v >> 28), j = (int)(v & PAIR_ATOM);
    const Cubic pj = m.p4[j];
    const double Fj = m.dFp[j];
    if (a != cur) {
      if (cur >= 0) flush();
      cur = a;
      fx = fy = fz = 0.0;
      pi = s_p[w][a];
      Fi = s_F[w][a];
    }
    double dx = pj.x - pi.x, dy = pj.y - pi.y, dz = pj.z - pi.z;
    pair_image(box, dx, dy, dz);
    double t;
    const int q = locate_u(m.tab.sp[0], ui.x, t);
    const int ti = record_type(pi), tj = record_type(pj);
    double gg;
    if (SAME) {
      gg = fma(Fi + Fj, spline_dval_at(m.tab.dsp[3], q, t), spline_dval_at(m.tab.dsp[ti + tj], q, t));
    } else {
      gg = fma(Fj, spline_dval_at(m.tab.dsp[3 + ti], q, t),
               fma(Fi, spline_dval_at(m.tab.dsp[3 + tj], q, t), spline_dval_at(m.tab.dsp[ti + tj], q, t)));
    }
    const double gr = -gg * ui.y;  // the force on j
    const double gx = gr * dx, gy = gr * dy, gz = gr * dz;
    fx -= gx;
    fy -= gy;
    fz -= gz;
    if (VIR) vir = fma(gr, fma(dz, dz, fma(dy, dy, dx * dx)), vir);
    atomicAdd(m.fx + j, gx);
    atomicAdd(m.fy + j, gy);
    atomicAdd(m.fz + j, gz);
  }
  if (cur >= 0) flush();
  if (bad) atomicOr(m.err, ERRF_NONFINITE);
  if (VIR) add_virial(m, vir);
}

// rows of 32 entries that a group's pairs can need: all of its half rows, and
// what the lists of PAIR_LIST - 31 entries and more leave of their last row
__global__ void k_md_pair_offsets(long long N, int group, const int* cnt_h, uint32_t* off, unsigned* total) {
  const long long g = (long long)blockIdx.x * 128 + threadIdx.x;
  const int lane = threadIdx.x & 31;
  unsigned need = 0u;
  if (g * group < N) {
    int sum = 0;
    for (int a = 0; a < group && g * group + a < N; ++a) sum += cnt_h[g * group + a];
    need = (unsigned)(sum / 32 + sum / 448 + 2);
  }
  unsigned at = need;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned q = __shfl_up_sync(0xffffffffu, at, o);
    if (lane >= o) at += q;
  }
  unsigned first = 0u;
  if (lane == 31) first = atomicAdd(total, at);
  first = __shfl_sync(0xffffffffu, first, 31);
  if (g * group < N) off[g] = first + at - need;
}

// mixed form on the half list: FP32 geometry and tables, FP64 sums
template <int LPA>
__global__ void __launch_bounds__(128) k_md_rho_half32(MdArgs m) {
  const long long g = (long long)blockIdx.x * 128 + threadIdx.x;
  const long long i = g / LPA;
  const int sub = (int)(g % LPA);
  const bool live = i < m.N;
  const int* row = m.nbr_h + (live ? i : 0) * m.K;
  const int cnt = live ? m.cnt_h[i] : 0;
  const uint4 ui = m.u4[live ? i : 0];
  const float rc2 = (float)(m.rc * m.rc);
  const int ti = (int)ui.w;
  double rho = 0.0;
  for (int k = sub; k < cnt; k += LPA) {
    const int j = row[k];
    const uint4 uj = m.u4[j];
    const float dx = fix_diff(uj.x, ui.x, m.ul[0]);
    const float dy = fix_diff(uj.y, ui.y, m.ul[1]);
    const float dz = fix_diff(uj.z, ui.z, m.ul[2]);
    const float r2 = dx * dx + dy * dy + dz * dz;
    if (r2 >= rc2) continue;
    const int tj = (int)uj.w;
    float t;
    const int q = spline32_locate(m.tab32.sp[3], sqrtf(r2), t, m.err);
    const float fj = spline32_val_at(m.tab32.sp[3 + tj], q, t);
    const float fi = m.same_dens ? fj : spline32_val_at(m.tab32.sp[3 + ti], q, t);
    rho += widen(fj);
    atomicAdd(m.rho + j, widen(fi));
  }
  rho = lane_sum<LPA>(rho);
  if (live && sub == 0) atomicAdd(m.rho + i, rho);
}

template <int LPA>
__global__ void __launch_bounds__(128) k_md_force_half32(MdArgs m) {
  const long long g = (long long)blockIdx.x * 128 + threadIdx.x;
  const long long i = g / LPA;
  const int sub = (int)(g % LPA);
  const bool live = i < m.N;
  const int* row = m.nbr_h + (live ? i : 0) * m.K;
  const int cnt = live ? m.cnt_h[i] : 0;
  const uint4 ui = m.u4[live ? i : 0];
  const int ti = (int)ui.w;
  const float Fi = m.dFp32[live ? i : 0];
  const float rc2 = (float)(m.rc * m.rc);
  double fx = 0.0, fy = 0.0, fz = 0.0;
  for (int k = sub; k < cnt; k += LPA) {
    const int j = row[k];
    const uint4 uj = m.u4[j];
    const float dx = fix_diff(uj.x, ui.x, m.ul[0]);
    const float dy = fix_diff(uj.y, ui.y, m.ul[1]);
    const float dz = fix_diff(uj.z, ui.z, m.ul[2]);
    const float r2 = dx * dx + dy * dy + dz * dz;
    if (r2 >= rc2) continue;
    const float ir = rsqrtf(r2);
    const int tj = (int)uj.w;
    float t;
    const int q = spline32_locate(m.tab32.sp[0], r2 * ir, t, m.err);
    const float Fj = m.dFp32[j];
    float gg;
    if (m.same_dens) {
      gg = fmaf(Fi + Fj, spline32_dval_at(m.tab32.dsp[3], q, t), spline32_dval_at(m.tab32.dsp[ti + tj], q, t));
    } else {
      gg = fmaf(Fj, spline32_dval_at(m.tab32.dsp[3 + ti], q, t),
                fmaf(Fi, spline32_dval_at(m.tab32.dsp[3 + tj], q, t), spline32_dval_at(m.tab32.dsp[ti + tj], q, t)));
    }
    const float gr = gg * ir;
    const double gx = widen(gr * dx), gy = widen(gr * dy), gz = widen(gr * dz);
    fx += gx;
    fy += gy;
    fz += gz;
    atomicAdd(m.fx + j, -gx);
    atomicAdd(m.fy + j, -gy);
    atomicAdd(m.fz + j, -gz);
  }
  if (not_finite(fx) | not_finite(fy) | not_finite(fz)) atomicOr(m.err, ERRF_NONFINITE);
  fx = lane_sum<LPA>(fx);
  fy = lane_sum<LPA>(fy);
  fz = lane_sum<LPA>(fz);
  if (live && sub == 0) {
    atomicAdd(m.fx + i, fx);
    atomicAdd(m.fy + i, fy);
    atomicAdd(m.fz + i, fz);
  }
}

// F'(rho_i) and F_B(rho_i) - F_A(rho_i) once rho is complete
__global__ void k_md_embed(MdArgs m) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= m.N) return;
  const double rho = m.rho[i];
  double t;
  const int ti = m.types[i];
  const int q = spline_locate(m.tab.sp[5 + ti], rho, t, m.err);
  m.dFp[i] = spline_der_at(m.tab.sp[5 + ti], q, t);
  m.dF[i] = spline_val_at(m.tab.sp[6], q, t) - spline_val_at(m.tab.sp[5], q, t);
  if (m.mixed) m.dFp32[i] = (float)m.dFp[i];
}

// FP64 forces on the half list: F_i += g (x_j - x_i) / r, F_j -= the same,
// g = phi'_{ti tj} + F'_i f'_{tj} + F'_j f'_{ti} (one density derivative
// when same_dens); force arrays zeroed before.  The virial term of the
// pair, r_ij . F_ij = -g r, goes to *m.vir when it is set.
template <int LPA, bool SAME, bool VIR>
__global__ void __launch_bounds__(128) k_md_force_half(MdArgs m) {
  const long long g = (long long)blockIdx.x * 128 + threadIdx.x;
  const long long i = g / LPA;
  const int sub = (int)(g % LPA);
  const bool live = i < m.N;
  const int* row = m.nbr_h + (live ? i : 0) * m.K;
  const int cnt = live ? m.cnt_h[i] : 0;
  const Cubic pi = m.p4[live ? i : 0];
  const int ti = record_type(pi);
  const double Fi = m.dFp[live ? i : 0];
  const PairBox box = pair_box(m.box);
  const double rc2 = m.rc * m.rc;
  double fx = 0.0, fy = 0.0, fz = 0.0, vir = 0.0;
  for (int k = sub; k < cnt; k += LPA) {
    const int j = row[k];
    const Cubic pj = m.p4[j];
    const double Fj = m.dFp[j];
    double dx = pj.x - pi.x, dy = pj.y - pi.y, dz = pj.z - pi.z;
    const double r2 = pair_r2(box, dx, dy, dz);
    if (outside(r2, rc2)) continue;
    double ir, t;
    const double r = sqrt3(r2, ir);
    const int tj = record_type(pj);
    const int q = locate_in(m.tab.sp[0], r, t);
    double gg;
    if (SAME) {
      gg = fma(Fi + Fj, spline_dval_at(m.tab.dsp[3], q, t), spline_dval_at(m.tab.dsp[ti + tj], q, t));
    } else {
      gg = fma(Fj, spline_dval_at(m.tab.dsp[3 + ti], q, t),
               fma(Fi, spline_dval_at(m.tab.dsp[3 + tj], q, t), spline_dval_at(m.tab.dsp[ti + tj], q, t)));
    }
    const double gr = -gg * ir;  // the force on j: a negated operand costs nothing, a negated result a pass
    const double gx = gr * dx, gy = gr * dy, gz = gr * dz;
    fx -= gx;
    fy -= gy;
    fz -= gz;
    if (VIR) vir = fma(gr, r2, vir);
    atomicAdd(m.fx + j, gx);
    atomicAdd(m.fy + j, gy);
    atomicAdd(m.fz + j, gz);
  }
  if (not_finite(fx) | not_finite(fy) | not_finite(fz)) atomicOr(m.err, ERRF_NONFINITE);
  fx = lane_sum<LPA>(fx);
  fy = lane_sum<LPA>(fy);
  fz = lane_sum<LPA>(fz);
  if (live && sub == 0) {
    atomicAdd(m.fx + i, fx);
    atomicAdd(m.fy + i, fy);
    atomicAdd(m.fz + i, fz);
  }
  if (VIR) add_virial(m, vir);
}

template <bool MIXED>
__device__ __forceinline__ void force_row(const MdArgs& m, long long i, double& vir) {
  const int* row = m.nbr + i * m.K;
  const int cnt = m.nbr_cnt[i];
  const double xi = m.x[i], yi = m.y[i], zi = m.z[i];
  const int ti = m.types[i];
  const double Fi = m.dFp[i];
  const double ix = 1.0 / m.box[0], iy = 1.0 / m.box[1], iz = 1.0 / m.box[2];
  const double rc2 = m.rc * m.rc;
  double fx = 0.0, fy = 0.0, fz = 0.0;
  const float Fi32 = (float)Fi;
  const uint32_t uxi = MIXED ? m.ux[i] : 0u, uyi = MIXED ? m.uy[i] : 0u, uzi = MIXED ? m.uz[i] : 0u;
  for (int k = 0; k < cnt; ++k) {
    const int j = row[k];
    if constexpr (MIXED) {
      // FP32 geometry and table derivatives, FP64 force sums
      const float dx = fix_diff(m.ux[j], uxi, m.ul[0]);
      const float dy = fix_diff(m.uy[j], uyi, m.ul[1]);
      const float dz = fix_diff(m.uz[j], uzi, m.ul[2]);
      const float r2 = dx * dx + dy * dy + dz * dz;
      if (r2 >= (float)rc2) continue;
      const float ir = rsqrtf(r2);
      const int tj = m.types[j];
      float t;
      const int q = spline32_locate(m.tab32.sp[0], r2 * ir, t, m.err);
      const float g = fmaf(m.dFp32[j], spline32_dval_at(m.tab32.dsp[3 + ti], q, t),
                           fmaf(Fi32, spline32_dval_at(m.tab32.dsp[3 + tj], q, t),
                                spline32_dval_at(m.tab32.dsp[ti + tj], q, t)));
      const float gr = g * ir;
      fx += (double)(gr * dx);
      fy += (double)(gr * dy);
      fz += (double)(gr * dz);
      continue;
    }
    const double dx = mimg(m.x[j] - xi, m.box[0], ix);
    const double dy = mimg(m.y[j] - yi, m.box[1], iy);
    const double dz = mimg(m.z[j] - zi, m.box[2], iz);
    const double r2 = dx * dx + dy * dy + dz * dz;
    if (r2 >= rc2) continue;
    const double ir = rsqrt_nr(r2);
    const int tj = m.types[j];
    double t;
    const int q = spline_locate(m.tab.sp[0], r2 * ir, t, m.err);
    const double g = fma(m.dFp[j], spline_dval_at(m.tab.dsp[3 + ti], q, t),
                         fma(Fi, spline_dval_at(m.tab.dsp[3 + tj], q, t),
                             spline_dval_at(m.tab.dsp[ti + tj], q, t)));
    const double gr = g * ir;
    fx = fma(gr, dx, fx);
    fy = fma(gr, dy, fy);
    fz = fma(gr, dz, fz);
    vir -= 0.5 * gr * r2;  // each pair is seen from both ends
  }
  if (!isfinite(fx) || !isfinite(fy) || !isfinite(fz)) atomicOr(m.err, ERRF_NONFINITE);
  m.fx[i] = fx;
  m.fy[i] = fy;
  m.fz[i] = fz;
}

template <bool MIXED>
__global__ void k_md_force(MdArgs m) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  double vir = 0.0;
  if (i < m.N) force_row<MIXED>(m, i, vir);
  if (!MIXED) add_virial(m, vir);
}

// v - L floor(v / L): a drift leaves the box by less than its length but for
// runaway atoms, so the division (a dozen FP64 instructions) is the exception
__device__ __forceinline__ double wrap_box(double v, double L) {
  double w = v;
  if (v < 0.0) w = v + L;
  else if (v >= L) w = v - L;
  if (!(w >= 0.0 && w <= L)) w = v - L * floor(v / L);
  if (w >= L) w -= L;
  if (w < 0.0) w = 0.0;
  return w;
}
// minimum image of a difference of two positions in [0, L)
__device__ __forceinline__ double mimg_box(double d, double L) {
  return d > 0.5 * L ? d - L : (d < -0.5 * L ? d + L : d);
}
// largest squared displacement: block maximum, then one atomic per block (one
// per atom on a single address took most of a drift kernel's time).
// Non-negative doubles order like their bit patterns.
__device__ __forceinline__ void max_displacement(const MdArgs& m, double d2) {
  unsigned long long b = (unsigned long long)__double_as_longlong(d2);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long q = __shfl_xor_sync(0xffffffffu, b, o);
    b = q > b ? q : b;
  }
  __shared__ unsigned long long s_max[4];
  if ((threadIdx.x & 31) == 0) s_max[threadIdx.x >> 5] = b;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < 4; ++w) b = s_max[w] > b ? s_max[w] : b;
    atomicMax(m.max_disp2_bits, b);
  }
}

// Box-Muller: two standard normals from two uniforms
__device__ __forceinline__ void normals(uint4 w, double& z0, double& z1) {
  const double u1 = (double)top53(w.x, w.y) * 0x1p-53;
  const double u2 = (double)top53(w.z, w.w) * 0x1p-53;
  const double rr = sqrt(-2.0 * log(1.0 - u1));
  double s, c;
  sincospi(2.0 * u2, &s, &c);
  z0 = rr * c;
  z1 = rr * s;
}

// the first of the two only
__device__ __forceinline__ double normal(uint4 w) {
  const double u1 = (double)top53(w.x, w.y) * 0x1p-53;
  const double u2 = (double)top53(w.z, w.w) * 0x1p-53;
  return sqrt(-2.0 * log(1.0 - u1)) * cospi(2.0 * u2);
}

__global__ void __launch_bounds__(128) k_md_first_half(MdArgs m, long long step) {
  const long long i = (long long)blockIdx.x * 128 + threadIdx.x;
  double d2 = 0.0;
  if (i < m.N) {
    const int ti = m.types[i];
    const double im = m.im[ti];
    const double h = 0.5 * m.dt;
    double vx = m.vx[i] + h * m.fx[i] * im;
    double vy = m.vy[i] + h * m.fy[i] * im;
    double vz = m.vz[i] + h * m.fz[i] * im;
    double x = m.x[i] + h * vx, y = m.y[i] + h * vy, z = m.z[i] + h * vz;
    if (m.c2 > 0.0) {
      const double sig = m.sig[ti];  // c2 sqrt(kT / mass)
      const uint4 c0 = make_uint4((uint32_t)step, (uint32_t)((uint64_t)step >> 32), (uint32_t)i, TAG_NOISE0);
      const uint4 c1 = make_uint4((uint32_t)step, (uint32_t)((uint64_t)step >> 32), (uint32_t)i, TAG_NOISE1);
      double z0, z1;
      normals(philox4x32_10(c0, m.key), z0, z1);
      const double z2 = normal(philox4x32_10(c1, m.key));
      vx = m.c1 * vx + sig * z0;
      vy = m.c1 * vy + sig * z1;
      vz = m.c1 * vz + sig * z2;
    }
    x = wrap_box(x + h * vx, m.box[0]);
    y = wrap_box(y + h * vy, m.box[1]);
    z = wrap_box(z + h * vz, m.box[2]);
    m.vx[i] = vx;
    m.vy[i] = vy;
    m.vz[i] = vz;
    m.x[i] = x;
    m.y[i] = y;
    m.z[i] = z;
    const double dx = mimg_box(x - m.x0[i], m.box[0]);
    const double dy = mimg_box(y - m.y0[i], m.box[1]);
    const double dz = mimg_box(z - m.z0[i], m.box[2]);
    d2 = dx * dx + dy * dy + dz * dz;
  }
  max_displacement(m, d2);
}

__global__ void k_md_second_half(MdArgs m) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= m.N) return;
  const double im = m.im[m.types[i]];
  const double h = 0.5 * m.dt;
  m.vx[i] += h * m.fx[i] * im;
  m.vy[i] += h * m.fy[i] * im;
  m.vz[i] += h * m.fz[i] * im;
}

__global__ void k_md_snapshot(MdArgs m) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i == 0) *m.max_disp2_bits = 0ull;
  if (i >= m.N) return;
  m.x0[i] = m.x[i];
  m.y0[i] = m.y[i];
  m.z0[i] = m.z[i];
}

// Nose-Hoover / MTK sub-flows (the step's scalars are integrated on the
// host): v <- v s e1 + (F/m) he2, and r <- wrap(r e1 + v e2dt) in the
// current box with the displacement from the last neighbour build measured
// against the snapshot scaled by lam = L / L_build.
__global__ void k_nh_kick(MdArgs m, double s, double e1, double he2) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= m.N) return;
  const double im = m.im[m.types[i]];
  const double se = s * e1, ke = he2 * im;
  m.vx[i] = fma(m.vx[i], se, m.fx[i] * ke);
  m.vy[i] = fma(m.vy[i], se, m.fy[i] * ke);
  m.vz[i] = fma(m.vz[i], se, m.fz[i] * ke);
}

__global__ void __launch_bounds__(128) k_nh_drift(MdArgs m, double e1, double e2dt) {
  const long long i = (long long)blockIdx.x * 128 + threadIdx.x;
  double d2 = 0.0;
  if (i < m.N) {
    const double x = wrap_box(fma(m.x[i], e1, m.vx[i] * e2dt), m.box[0]);
    const double y = wrap_box(fma(m.y[i], e1, m.vy[i] * e2dt), m.box[1]);
    const double z = wrap_box(fma(m.z[i], e1, m.vz[i] * e2dt), m.box[2]);
    m.x[i] = x;
    m.y[i] = y;
    m.z[i] = z;
    const double dx = mimg(x - m.x0[i] * m.lam, m.box[0], 1.0 / m.box[0]);
    const double dy = mimg(y - m.y0[i] * m.lam, m.box[1], 1.0 / m.box[1]);
    const double dz = mimg(z - m.z0[i] * m.lam, m.box[2], 1.0 / m.box[2]);
    d2 = dx * dx + dy * dy + dz * dz;
  }
  max_displacement(m, d2);
}

// positions x0 + alpha d (conjugate-gradient line search), wrapped, with the
// displacement check of the MD step
__global__ void __launch_bounds__(128) k_cg_place(MdArgs m, const double* x0, const double* d, double alpha) {
  const long long i = (long long)blockIdx.x * 128 + threadIdx.x;
  double d2 = 0.0;
  if (i < m.N) {
    const long long N = m.N;
    const double x = wrap_box(fma(alpha, d[i], x0[i]), m.box[0]);
    const double y = wrap_box(fma(alpha, d[N + i], x0[N + i]), m.box[1]);
    const double z = wrap_box(fma(alpha, d[2 * N + i], x0[2 * N + i]), m.box[2]);
    m.x[i] = x;
    m.y[i] = y;
    m.z[i] = z;
    const double dx = mimg_box(x - m.x0[i], m.box[0]);
    const double dy = mimg_box(y - m.y0[i], m.box[1]);
    const double dz = mimg_box(z - m.z0[i], m.box[2]);
    d2 = dx * dx + dy * dy + dz * dz;
  }
  max_displacement(m, d2);
}

constexpr int DOT_BLOCK = 256;
int dot_blocks(long long n) { return (int)((n + DOT_BLOCK - 1) / DOT_BLOCK); }

// block partials of sum_k a[k] b[k], k < n
__global__ void __launch_bounds__(DOT_BLOCK) k_dot(const double* a, const double* b, long long n, double* part) {
  const long long k = (long long)blockIdx.x * DOT_BLOCK + threadIdx.x;
  double v = k < n ? a[k] * b[k] : 0.0;
  __shared__ double sh[DOT_BLOCK / 32];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < DOT_BLOCK / 32; ++w) t += sh[w];
    part[blockIdx.x] = t;
  }
}

// max over atoms of |v_i|^2 for a 3N SoA vector, as double bits
__global__ void k_max_norm2(const double* a, long long N, unsigned long long* out) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= N) return;
  const double v = a[i] * a[i] + a[N + i] * a[N + i] + a[2 * N + i] * a[2 * N + i];
  atomicMax(out, (unsigned long long)__double_as_longlong(v));
}

constexpr int KE_BLOCK = 256;
int kinetic_blocks(long long N) { return (int)((N + KE_BLOCK - 1) / KE_BLOCK); }

__global__ void __launch_bounds__(KE_BLOCK) k_kinetic(MdArgs m, double* part) {
  const long long i = (long long)blockIdx.x * KE_BLOCK + threadIdx.x;
  double e = 0.0;
  if (i < m.N) {
    const double v2 = m.vx[i] * m.vx[i] + m.vy[i] * m.vy[i] + m.vz[i] * m.vz[i];
    e = 0.5 * m.mass[m.types[i]] / FTM * v2;
  }
  __shared__ double sh[KE_BLOCK / 32];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) e += __shfl_xor_sync(0xffffffffu, e, o);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = e;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < KE_BLOCK / 32; ++w) t += sh[w];
    part[blockIdx.x] = t;
  }
}

static unsigned grid_of(long long N) { return (unsigned)((N + 127) / 128); }

__global__ void k_fix_positions(long long N, const double* x, const double* y, const double* z, double sx, double sy,
                                double sz, uint32_t* ux, uint32_t* uy, uint32_t* uz) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= N) return;
  // x 2^32 / L rounded to an integer, reduced mod 2^32 (two's complement
  // wrap of a negative or >= 2^32 value is the periodic reduction)
  ux[i] = (uint32_t)(unsigned long long)llrint(x[i] * sx);
  uy[i] = (uint32_t)(unsigned long long)llrint(y[i] * sy);
  uz[i] = (uint32_t)(unsigned long long)llrint(z[i] * sz);
}

void launch_fix_positions(long long N, const double* x, const double* y, const double* z, const double box[3],
                          uint32_t* ux, uint32_t* uy, uint32_t* uz, cudaStream_t st) {
  if (N < 1 || !ux || !uy || !uz) return;
  const double two32 = 4294967296.0;
  k_fix_positions<<<grid_of(N), 128, 0, st>>>(N, x, y, z, two32 / box[0], two32 / box[1], two32 / box[2], ux, uy,
                                              uz);
}

// lanes per atom of the half-list passes: 4, or 16 while 4 leave the GPU short
// of warps (a row is then a chain of two pairs).  Below 20000 atoms 4 lanes are
// under 2500 warps, 16 per SM.  A step of 3456 atoms took 294 us with a thread
// per atom and 97 with 16 lanes.
constexpr long long MD_FEW = 20000;

// atoms of a pair block.  16 fill 14.5 rows of 32 lanes with their 464 pairs;
// fewer leave more lanes idle in the last row but give the GPU more warps.  A
// step with 2 / 4 / 16: 5488 atoms 90 / 101 / 178 us, 86 k (nanocrystal) 321 /
// 327 / 380, 351 k 1110 / 1073 / 1086, 1.36 M 3932 / 3791 / 3645.
int md_pair_group(long long N) { return N < 100000 ? 2 : N < 500000 ? 4 : 16; }

void launch_md_pair_offsets(long long N, const int* cnt_h, uint32_t* pair_off, unsigned* total, cudaStream_t st) {
  const int group = md_pair_group(N);
  k_md_pair_offsets<<<grid_of((N + group - 1) / group), 128, 0, st>>>(N, group, cnt_h, pair_off, total);
}

template <int GROUP>
static void rho_pairs(const MdArgs& m, cudaStream_t st) {
  const unsigned g = grid_of((m.N + GROUP - 1) / GROUP * 32);
  if (m.same_dens) k_md_rho_pairs<GROUP, true><<<g, 128, 0, st>>>(m);
  else k_md_rho_pairs<GROUP, false><<<g, 128, 0, st>>>(m);
}

template <int GROUP>
static void force_pairs(const MdArgs& m, cudaStream_t st) {
  const unsigned g = grid_of((m.N + GROUP - 1) / GROUP * 32);
  if (m.vir && m.same_dens) k_md_force_pairs<GROUP, true, true><<<g, 128, 0, st>>>(m);
  else if (m.vir) k_md_force_pairs<GROUP, false, true><<<g, 128, 0, st>>>(m);
  else if (m.same_dens) k_md_force_pairs<GROUP, true, false><<<g, 128, 0, st>>>(m);
  else k_md_force_pairs<GROUP, false, false><<<g, 128, 0, st>>>(m);
}

template <int LPA>
static void rho_half(const MdArgs& m, cudaStream_t st) {
  const unsigned g = grid_of(m.N * LPA);
  if (m.mixed) k_md_rho_half32<LPA><<<g, 128, 0, st>>>(m);
  else if (m.same_dens) k_md_rho_half<LPA, true><<<g, 128, 0, st>>>(m);
  else k_md_rho_half<LPA, false><<<g, 128, 0, st>>>(m);
}

template <int LPA>
static void force_half(const MdArgs& m, cudaStream_t st) {
  const unsigned g = grid_of(m.N * LPA);
  if (m.mixed) k_md_force_half32<LPA><<<g, 128, 0, st>>>(m);
  else if (m.vir && m.same_dens) k_md_force_half<LPA, true, true><<<g, 128, 0, st>>>(m);
  else if (m.vir) k_md_force_half<LPA, false, true><<<g, 128, 0, st>>>(m);
  else if (m.same_dens) k_md_force_half<LPA, true, false><<<g, 128, 0, st>>>(m);
  else k_md_force_half<LPA, false, false><<<g, 128, 0, st>>>(m);
}

void launch_md_rho(const MdArgs& m, cudaStream_t st) {
  if (m.mixed) launch_fix_positions(m.N, m.x, m.y, m.z, m.box, m.ux, m.uy, m.uz, st);
  if (m.nbr_h) {
    k_md_records<<<grid_of(m.N), 128, 0, st>>>(m);
    cudaMemsetAsync(m.rho, 0, sizeof(double) * m.N, st);
    if (m.pair_ui && md_pair_group(m.N) == 2) rho_pairs<2>(m, st);
    else if (m.pair_ui && md_pair_group(m.N) == 4) rho_pairs<4>(m, st);
    else if (m.pair_ui) rho_pairs<16>(m, st);
    else if (m.N < MD_FEW) rho_half<16>(m, st);
    else rho_half<4>(m, st);
    k_md_embed<<<grid_of(m.N), 128, 0, st>>>(m);
  } else if (m.mixed) {
    k_md_rho<true><<<grid_of(m.N), 128, 0, st>>>(m);
  } else {
    k_md_rho<false><<<grid_of(m.N), 128, 0, st>>>(m);
  }
}
void launch_md_force(const MdArgs& m, cudaStream_t st) {
  if (m.nbr_h) {
    cudaMemsetAsync(m.fx, 0, sizeof(double) * 3 * m.N, st);
    if (m.pair_ui && md_pair_group(m.N) == 2) force_pairs<2>(m, st);
    else if (m.pair_ui && md_pair_group(m.N) == 4) force_pairs<4>(m, st);
    else if (m.pair_ui) force_pairs<16>(m, st);
    else if (m.N < MD_FEW) force_half<16>(m, st);
    else force_half<4>(m, st);
  } else if (m.mixed) {
    k_md_force<true><<<grid_of(m.N), 128, 0, st>>>(m);
  } else {
    k_md_force<false><<<grid_of(m.N), 128, 0, st>>>(m);
  }
}
void launch_md_first_half(const MdArgs& m, long long step, cudaStream_t st) {
  k_md_first_half<<<grid_of(m.N), 128, 0, st>>>(m, step);
}
void launch_md_second_half(const MdArgs& m, cudaStream_t st) {
  k_md_second_half<<<grid_of(m.N), 128, 0, st>>>(m);
}
void launch_md_snapshot(const MdArgs& m, cudaStream_t st) { k_md_snapshot<<<grid_of(m.N), 128, 0, st>>>(m); }
void launch_nh_kick(const MdArgs& m, double s, double e1, double he2, cudaStream_t st) {
  k_nh_kick<<<grid_of(m.N), 128, 0, st>>>(m, s, e1, he2);
}
void launch_nh_drift(const MdArgs& m, double e1, double e2dt, cudaStream_t st) {
  k_nh_drift<<<grid_of(m.N), 128, 0, st>>>(m, e1, e2dt);
}
void launch_cg_place(const MdArgs& m, const double* x0, const double* d, double alpha, cudaStream_t st) {
  k_cg_place<<<grid_of(m.N), 128, 0, st>>>(m, x0, d, alpha);
}
void launch_dot(const double* a, const double* b, long long n, double* part, cudaStream_t st) {
  k_dot<<<dot_blocks(n), DOT_BLOCK, 0, st>>>(a, b, n, part);
}
void launch_max_norm2(const double* a, long long N, unsigned long long* out, cudaStream_t st) {
  k_max_norm2<<<grid_of(N), 128, 0, st>>>(a, N, out);
}
__global__ void k_axpby(double* d, const double* g, double beta, long long n) {
  const long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (k < n) d[k] = fma(beta, d[k], g[k]);
}
void launch_axpby(double* d, const double* g, double beta, long long n, cudaStream_t st) {
  k_axpby<<<grid_of(n), 128, 0, st>>>(d, g, beta, n);
}
void launch_kinetic(const MdArgs& m, double* part, cudaStream_t st) {
  k_kinetic<<<kinetic_blocks(m.N), KE_BLOCK, 0, st>>>(m, part);
}

}  // namespace vcsgc
