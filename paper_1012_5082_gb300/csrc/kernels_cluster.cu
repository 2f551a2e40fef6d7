// kernels_cluster.cu -- the fused colour step of the rigid BCC lattice with
// one density function as one persistent launch: a replica's species stay in
// shared memory while many colour steps (composite moves of Sec. III B 2) run
// back to back, so a step costs barriers instead of a launch and its L2
// round trips.  Two kernels:
//
// k_cluster_steps (SUBLATTICE schedule): one thread-block cluster per
//   replica.  The bit-packed species rows (kernels_lattice.cu's layout
//   without the pending half: 32 species bits per 32-bit word, four halo
//   bits at each row end) are tiled over the cluster's CTAs in (y, z): CTA
//   (ty, tz) of a TY x TZ grid owns rows [ty Ty, (ty + 1) Ty) x [tz Tz,
//   (tz + 1) Tz) and keeps them with a halo of two rows on each side, so a
//   trial's dE reads only its own shared memory.
// k_pick_steps (BLOCKS and OVERLAP schedules, up to a few thousand trials per
//   step): one CTA per replica with the whole lattice in shared memory.
//
// Random numbers, site picks and the logarithms of the uniforms depend on no
// state, so a first launch (k_chain_draws) makes those of a chunk of steps on
// every SM, and the chain reads them a step ahead: -ln u per trial (the test u
// < exp(-X) becomes X < -ln u, no exponential), the colour and -ln u of the
// global stage per step.  (0.1 us per step of 64,000 trials; inside the chain
// the ten Philox rounds of a group's four trials were a third of its
// instructions.)
//
// Colour step k of k_cluster_steps, every CTA:
//   1. proposes step k on the species as they stand, while the barrier of step
//      k-1 completes: right if step k-1 is rejected, which is the usual case;
//   2. after the barrier sums the CTAs' partials of step k-1 (each CTA pushed
//      its own into every CTA's shared memory before it arrived) and takes
//      the global decision G_{k-1} (Eq. trans_vcsgc_par2) -- every thread the
//      same;
//   3. only if G_{k-1}: every thread flips the trials it accepted in step k-1,
//      one more barrier (with the changed words stored into the halo copies of
//      the other CTAs) follows, and step k is proposed again.  A rejected step
//      changes nothing, so it costs one barrier, hidden behind the proposal;
//   4. reduces dn, accepts, ties and per-shell sums of step k, pushes the
//      partials and arrives at the barrier.
// An extra warp keeps the replica's counters and sums off the trial warps'
// path and decodes the colour two steps ahead.
//
// Words of the halo copies are stored with plain st.shared::cluster: all
// stores of one word in one step carry the same value, so their order is
// free.  (Distributed-shared XORs lost updates when two met in one word.)
//
// Measured, 80^3 x 8 replicas (64,000 trials per step): 2.3 us per step against
// 4.2 for the per-step launch; what sizes it serves, and both sides there:
// resident_shape in vcsgc_capi.cu.  Bound: the latency of one step's chain of
// about 700 instructions per warp at two warps per scheduler (issue 40 %
// active), not a pipe.
//
// Every CTA of a cluster runs the same number of cluster barriers (the
// global decision is the same in each; a last barrier before any CTA exits);
// clusters of different replicas never wait on each other.
#include "common.cuh"
#include "kernels.h"
#include "lattice.cuh"

#include <type_traits>

namespace vcsgc {

namespace {

__device__ __forceinline__ uint32_t cl_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ uint32_t cl_nctas() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ uint32_t cl_id() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%clusterid.x;" : "=r"(r));
  return r;
}
__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
// shared::cluster address of the same variable in CTA `rank` of the cluster
__device__ __forceinline__ uint32_t cl_map(uint32_t a, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
  return r;
}
__device__ __forceinline__ void cl_st_u32(uint32_t a, uint32_t v) {
  asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ void cl_st_u64(uint32_t a, unsigned long long v) {
  asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(a), "l"(v) : "memory");
}
// cluster barrier, split: arrive (release: this thread's earlier shared and
// distributed-shared writes become visible; it waits for the thread's loads
// in flight too) or relaxed (for threads that stored nothing the other CTAs
// read) and wait (acquire); a cluster of one CTA takes the block barrier at
// the wait
__device__ __forceinline__ void cl_arrive(bool solo) {
  if (solo) return;
  __syncwarp();
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cl_arrive_relaxed(bool solo) {
  if (solo) return;
  __syncwarp();
  asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
}
__device__ __forceinline__ void cl_wait(bool solo) {
  if (solo) {
    __syncthreads();
    return;
  }
  __syncwarp();
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// loads of the chain's draws, a step ahead of their use: volatile, so that the
// compiler leaves them where they stand instead of next to the use
__device__ __forceinline__ int2 ld_ahead(const int2* p) {
  int2 v;
  asm volatile("ld.global.nc.v2.s32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "l"(p));
  return v;
}
template <int N>
struct alignas(4 * N) Draw {  // -ln u of a group's trials
  float l[N];
};
__device__ __forceinline__ Draw<4> ld_draw(const Draw<4>* p) {
  Draw<4> v;
  asm volatile("ld.global.nc.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(v.l[0]), "=f"(v.l[1]), "=f"(v.l[2]), "=f"(v.l[3])
               : "l"(p));
  return v;
}
__device__ __forceinline__ Draw<1> ld_draw(const Draw<1>* p) {
  Draw<1> v;
  asm volatile("ld.global.nc.f32 %0, [%1];" : "=f"(v.l[0]) : "l"(p));
  return v;
}

// ---- counts of four trial sites at once
// The trial sites of one row and colour lie 8 bits apart (period 4 along x,
// two half-lattice units per cell), so after a funnel shift by q0 a 32-bit
// word of a neighbour row holds the 7-bit windows (x offsets -3..3 at bits
// 0..6) of four trials in its four bytes.  The B neighbours are summed in
// fields inside each byte: a masked word is added in place, its bit fields
// spaced so that the sums (at most 8 rows) do not meet; one mask and one add
// serve four trials.  By parity of the neighbour's y, z offset (h = half-
// lattice units, rows of odd h hold odd x offsets):
//   (1,1)  4 rows: x +-1 shell 1, +-3 shell 4     (1,3),(3,1) 8 rows: x +-1 shell 4
//   (0,0)  1 row:  x +-2 shell 2                  (0,2),(2,0) 4 rows: x 0 shell 2, +-2 shell 3
//   (2,2)  4 rows: x 0 shell 3, +-2 shell 5
// About 110 integer operations and 26 loads for four trials, against 33
// popc (a sixth of the ALU rate) and masks for each.  NSH = 2: the first
// two shells only.  c[s]: counts per byte; the return value: own species.
__host__ __device__ constexpr int half_class(int B, int d) {  // |h| of the odd offset of row d, 0: none
  const int h = 2 * d + (B ? -1 : 1);
  return (h == 1 || h == -1) ? 1 : ((h == 3 || h == -3) ? 3 : 0);
}

// row(dy, dz): the first of the two words of the window in row (dy, dz).
template <int B, int NSH, typename Row>
__device__ __forceinline__ uint32_t swar_counts(Row row, int q0, uint32_t (&c)[NSH]) {
  constexpr uint32_t K = 0x01010101u;
  uint32_t A = 0u, Bq = 0u, C = 0u, D = 0u, E1 = 0u, E2 = 0u, F1 = 0u, F2 = 0u, H1 = 0u, own = 0u;
#pragma unroll
  for (int dz = -2; dz <= 2; ++dz) {
#pragma unroll
    for (int dy = -2; dy <= 2; ++dy) {
      const int oy = half_class(B, dy), oz = half_class(B, dz);
      const bool near = oy == 1 && oz == 1;
      const bool far = NSH == 5 && ((oy == 1 && oz == 3) || (oy == 3 && oz == 1));
      const int ay = dy < 0 ? -dy : dy, az = dz < 0 ? -dz : dz;
      const bool centre = ay + az == 0, cross = ay + az == 1, corner = NSH == 5 && ay == 1 && az == 1;
      if (!(near || far || centre || cross || corner)) continue;
      const uint32_t* p = row(dy, dz);
      const uint32_t v = __funnelshift_r(p[0], p[1], q0);
      if (near) {
        if (NSH == 5) {
          A += v & (0x11u * K);
          Bq += (v >> 2) & (0x11u * K);
        } else {
          C += v & (0x04u * K);
          D += v & (0x10u * K);
        }
      }
      if (far) {
        C += v & (0x04u * K);
        D += v & (0x10u * K);
      }
      if (centre) {
        H1 = v;
        own = (v >> 3) & K;
      }
      if (cross) {
        E2 += v & (0x08u * K);
        if (NSH == 5) E1 += v & (0x22u * K);
      }
      if (corner) {
        F2 += v & (0x08u * K);
        F1 += v & (0x22u * K);
      }
    }
  }
  const uint32_t m4 = 0x0Fu * K, m3 = 0x07u * K;
  c[1] = ((E2 >> 3) & m3) + ((H1 >> 1) & K) + ((H1 >> 5) & K);
  if constexpr (NSH == 5) {
    c[0] = ((A >> 4) & m4) + (Bq & m4);
    c[2] = ((E1 >> 1) & m3) + ((E1 >> 5) & m3) + ((F2 >> 3) & m3);
    c[3] = (A & m4) + ((Bq >> 4) & m4) + ((C >> 2) & m4) + ((D >> 4) & m4);
    c[4] = ((F1 >> 1) & m3) + ((F1 >> 5) & m3);
  } else {
    c[0] = ((C >> 2) & m3) + ((D >> 4) & m3);
  }
  return own;
}

// the same counts of one trial site (byte 0) by popc on the compile-time
// five-shell rows, for periods other than 4 along x
template <int B>
__device__ __forceinline__ uint32_t popc_counts(const uint32_t* base, int rstride, int zstride, int q0,
                                                uint32_t (&c)[5]) {
#pragma unroll
  for (int s = 0; s < 5; ++s) c[s] = 0u;
  const uint32_t* p0 = base + (q0 >> 5);
  const int sh = q0 & 31;
  uint32_t own = 0u;
#pragma unroll
  for (int q = 0; q < 13; ++q) {
    const unsigned long long code = bcc5_row(B, q);
    const int dy = (int)((code >> 40) & 15) - 2, dz = (int)((code >> 44) & 15) - 2;
    const uint32_t* p = p0 + dz * zstride + dy * rstride;
    const uint32_t win = __funnelshift_r(p[0], p[1], sh);
    if (dy == 0 && dz == 0) own = (win >> 3) & 1u;
#pragma unroll
    for (int s = 0; s < 5; ++s) {
      const uint32_t m = (uint32_t)(code >> (7 * s)) & 0x7Fu;
      if (m) c[s] += __popc(win & m);
    }
  }
  return own;
}

// Screen of u < exp(-X) in the logarithm, X < l with l = -ln u: 1 accept, 0
// reject, -1 open (decided in FP64).  x32 is within dx of X.  l carries the
// rounding of u to float (2^-23 relative, so absolute in l) and the error of
// the logarithm; (|x32| + l + 1) 2^-20 covers these, the sums' rounding and the 2^-21 |x32|
// of lattice_accept with room, so a decision is the FP64 one.  l is NaN for u
// = 0 (open).  l comes from __logf (documented: 2^-21.4 absolute on [0.5, 2],
// 3 ulp elsewhere).
__device__ __forceinline__ int log_screen(float x32, float dx, float l) {
  const float e = fmaf(fabsf(x32) + l, 9.5367431640625e-07f, dx + 9.5367431640625e-07f);
  return x32 + e < l ? 1 : (x32 - e > l ? 0 : -1);
}
__device__ __forceinline__ float neg_log_u(uint64_t u53) {
  return u53 ? -__logf(u53_float(u53) * 1.1102230246251565e-16f) : __int_as_float(0x7FFFFFFF);
}

// the two signed 16-bit sums of a packed word
__device__ __forceinline__ int sum_lo(int w) { return (int)(short)(w & 0xFFFF); }
__device__ __forceinline__ int sum_hi(int w) { return (w - sum_lo(w)) >> 16; }

// Running sums of a launch's steps, kept by one thread and folded into the
// replica's state once at the end: integers, but for the sums of c and c^2,
// which grow a step at a time as in the per-step launch (an FP64 addition
// each; c changes only with an accepted step, and its quotient is taken by the
// reciprocal and one residual correction, q + (x - q N) / N, instead of a division).
struct StepSums {
  long long trials = 0, local_acc = 0, flips = 0, dn = 0;
  int near_ties = 0, global_trials = 0, global_acc = 0;
  double sum_c, sum_c2, c, c2, N, rN;

  __device__ __forceinline__ void begin(const RepState& S, const LatGeom& g, int n_now) {
    N = (double)g.n_sites;
    rN = 1.0 / N;
    sum_c = S.sum_c;
    sum_c2 = S.sum_c2;
    set_n(n_now);
  }
  __device__ __forceinline__ void set_n(int n_now) {
    const double x = (double)n_now, q = x * rN;
    c = fma(fma(-q, N, x), rN, q);  // x / N
    c2 = c * c;
  }

  // one decided step; n_now: B count after it
  __device__ __forceinline__ void step(int D, int dn_, int nacc, int gtie, int G, int n_now) {
    trials += D;
    local_acc += nacc;
    near_ties += gtie;
    global_trials += nacc > 0 ? 1 : 0;
    if (G) {
      global_acc += 1;
      flips += nacc;
      dn += dn_;
      set_n(n_now);
    }
    sum_c += c;
    sum_c2 += c2;
  }

  // sb: sum over the accepted moves of s_i b_s (per shell)
  __device__ __forceinline__ void fold(RepState& S, const LatArgs& a, const long long* sb, int n_sh,
                                       long long ties, int n, int n_now, long long k_next) const {
    S.trials += trials;
    S.local_acc += local_acc;
    S.near_ties += near_ties + ties;
    S.global_trials += global_trials;
    S.global_acc += global_acc;
    S.flips += flips;
    // sum over the accepted moves of s_i (C + sum_s b_s G_s + dF0)
    double e = a.C * (double)dn;
    for (int q = 0; q < n_sh; ++q) e = fma((double)sb[q], a.G[q], e);
    S.energy += e + a.dF0 * (double)dn;
    S.n = n_now;
    S.sum_c = sum_c;
    S.sum_c2 = sum_c2;
    S.steps += n;
    S.step = k_next;
    S.fin_step = k_next - 1;
  }
};

// what the per-step launch expects before step kn: nothing pending, step kn - 1
// finalised, zero accumulators, and (with the colour table, lat_colours_ahead)
// the step base.  It is written here and not by a launch of its own, or by the
// host when a per-step launch comes: the chain's position is then the device's
// alone, whatever the caller captures and replays.
__device__ __forceinline__ void hand_over(const LatArgs& a, int r, const RepState& S, long long kn) {
  a.rs[r] = S;
  if (r == 0) a.ctl->base_step = kn;
  a.n_start[r * 2 + (int)(kn & 1)] = S.n;
  StepAcc* A = a.acc + r * 3;
  for (int q = 0; q < 3; ++q) {
    A[q].dn = 0;
    A[q].nacc = 0;
    A[q].sum_de = 0.0;
    A[q].ties = 0;
    A[q].s1 = 0;
    for (int f = 0; f < 8; ++f) A[q].sb[f] = 0;
  }
}

// the CTA's tile of one replica
struct TileView {
  int ty, tz;  // tile indices
  int RY;      // rows per plane in shared memory (Ty + 4)
  int Y0, Z0;  // first owned row, plane
};

// Flip the accepted sites of one group: acc holds a byte flag per site, site i
// at half coordinate H + 8 i (one site: flag 0).  XORs the words of the row
// `row` (its x-halo bits at the far end included) and returns the words that
// changed as f(word) for every one of them.
struct GroupWords {
  uint32_t lo, hi;    // masks of words w, w + 1
  int w;              // first word
  int hw;             // x-halo word (-1: none)
  uint32_t hm;        // its mask
};
__device__ __forceinline__ GroupWords group_words(int nx, int H, uint32_t acc) {
  GroupWords q;
  const int p = LAT_HALO + H;
  const unsigned long long m = (unsigned long long)acc << (p & 31);
  q.lo = (uint32_t)m;
  q.hi = (uint32_t)(m >> 32);
  q.w = p >> 5;
  q.hw = -1;
  q.hm = 0u;
  // a row's first (H < 4) and last (H >= 2 nx - 4) sites have a copy beyond
  // the other end (nx >= 8 sites of one colour never need both)
  if (H < LAT_HALO && (acc & 1u)) {
    q.hw = (p + 2 * nx) >> 5;
    q.hm = 1u << ((p + 2 * nx) & 31);
  }
  const int last = (31 - __clz((int)(acc | 1u))) >> 3;  // the group's last accepted site
  const int pl = p + 8 * last - 2 * nx;
  if (pl >= 0 && (acc >> (8 * last) & 1u)) {
    q.hw = 0;  // pl < 4
    q.hm |= 1u << pl;
  }
  return q;
}

// Store the current words of those sites' row (owned by this CTA, at oy, oz in
// the tile) into every other copy of the row in the cluster: the tile's own
// halo and the halos of the tiles at offsets -1 and 1 in y and z (tiles of two
// rows or more, so no tile holds more).
__device__ __forceinline__ void push_copies(uint32_t* rows, uint32_t rows_addr, const ClTile& T, const TileView& v,
                                            int W, int oy, int oz, const GroupWords& q) {
  const uint32_t* own = rows + ((oz + 2) * v.RY + (oy + 2)) * W;
  const uint32_t v0 = own[q.w], v1 = own[q.w + 1], vh = q.hw >= 0 ? own[q.hw] : 0u;
#pragma unroll
  for (int b = -1; b <= 1; ++b) {
    if ((b < 0 && oz >= 2) || (b > 0 && oz < T.Tz - 2)) continue;
    int tz = v.tz + b;
    tz = tz < 0 ? tz + T.TZ : (tz >= T.TZ ? tz - T.TZ : tz);
    const int lz = oz + 2 - b * T.Tz;
#pragma unroll
    for (int a = -1; a <= 1; ++a) {
      if ((a == 0 && b == 0) || (a < 0 && oy >= 2) || (a > 0 && oy < T.Ty - 2)) continue;
      int ty = v.ty + a;
      ty = ty < 0 ? ty + T.TY : (ty >= T.TY ? ty - T.TY : ty);
      const int ly = oy + 2 - a * T.Ty;
      const uint32_t la = cl_map(rows_addr + (uint32_t)((lz * v.RY + ly) * W) * 4u, (uint32_t)(tz * T.TY + ty));
      cl_st_u32(la + 4u * q.w, v0);
      if (q.hi) cl_st_u32(la + 4u * (q.w + 1), v1);
      if (q.hw >= 0) cl_st_u32(la + 4u * q.hw, vh);
    }
  }
}

// global decision of step k from its sums, identical in every thread; lg = -ln
// of its uniform (screen of global_accept's Y32 and bound, else global_accept)
__device__ __forceinline__ int decide(const LatArgs& a, const LatRep& lr, const RepParams& p, int dn, int nacc,
                                      int n_prev, float lg, long long k, int* tie) {
  if (nacc == 0) return 0;
  const float fdn = (float)dn, fn = (float)n_prev, diff = fn - lr.n0_32;
  const float y32 = lr.bk32 * fdn * fmaf(2.0f, diff, fdn);
  const float dy = fabsf(lr.bk32 * fdn) * (fabsf(fdn) + 2.0f * (fn + lr.n0_32)) * 4.76837158203125e-07f;
  const int dec = log_screen(y32, dy, lg);
  if (dec >= 0) return dec;
  uint64_t ug;
  lat_colour(a, p.key, k, &ug);
  return global_accept(lr, p, dn, n_prev, ug, tie) ? 1 : 0;
}

}  // namespace

// Draws of the next m steps from the control block's base: step j's of replica r at lu + j P + off[r]
// (SUBLATTICE: -ln u of the trials, rows of the colour padded to whole groups
// of GS) or su (else: site, -1 past the colour's domains, and -ln u of domain
// d), and the step's colour (SUBLATTICE) or number of domains and -ln of its
// global uniform at cg[j R + r].  blockIdx = (trials / 256, j, r).
template <int GS>
__global__ void __launch_bounds__(256) k_chain_draws(LatArgs a, ChainDraws cd) {
  const int r = blockIdx.z, j = blockIdx.y;
  const long long base = a.ctl->base_step;
  const LatGeom g = a.geom[r];
  const uint2 key = a.rp[r].key;
  const long long k = base + j;
  const int t = blockIdx.x * 256 + threadIdx.x;
  uint64_t ug;
  int c = 0;
  if (r + j + t == 0) *cd.base = base;  // the chain moves the control block's while its last CTAs may not have started
  if (GS == 0 || t == 0) c = lat_colour(a, key, k, &ug);
  if (t == 0)
    cd.cg[(size_t)j * a.R + r] =
        make_int2(GS > 0 ? c : a.col_start[c + 1] - a.col_start[c], __float_as_int(neg_log_u(ug)));
  if constexpr (GS > 0) {
    const int pitch = (g.nxq + GS - 1) / GS * GS;
    const int row = fdiv(t, pitch, __frcp_rn((float)pitch)), x = t - row * pitch;
    if ((long long)row * g.nxq >= g.d || x >= g.nxq) return;
    const uint4 w = philox4x32_10(make_uint4((uint32_t)k, (uint32_t)((uint64_t)k >> 32),
                                             (uint32_t)(row * g.nxq + x), TAG_TRIAL), key);
    cd.lu[(size_t)j * cd.P + cd.off[r] + t] = neg_log_u(top53(w.z, w.w));
  } else {
    if (t >= g.dmax) return;
    const int c0 = a.col_start[c];
    int2* out = cd.su + (size_t)j * cd.P + cd.off[r] + t;
    if (t >= a.col_start[c + 1] - c0) {
      *out = make_int2(-1, 0);
      return;
    }
    const uint4 w = philox4x32_10(make_uint4((uint32_t)k, (uint32_t)((uint64_t)k >> 32), (uint32_t)t, TAG_TRIAL), key);
    const int db = a.dom_start[c0 + t], size = a.dom_start[c0 + t + 1] - db;
    const int site = a.dom_sites[db + pick_index(a.pick, w.x, w.y, size)];
    *out = make_int2(site, __float_as_int(neg_log_u(top53(w.z, w.w))));
  }
}

// One cluster per replica (replica = cluster index).  A worker thread takes a
// group of GS = 4 trials of one row word (SWAR) or one trial; block = BS
// workers and one bookkeeping warp.  Dynamic shared memory: the tile's rows
// with halo, two pad words, two bytes per group (its accepted trials of the
// last two steps).
struct StepGeo {  // a step's colour on this tile
  int px, py, pz, b;
  int kyb, kzb, cy, cz;  // first row and plane of the colour in the tile, and their numbers
};

template <int NSH, bool SWAR, int BS>
__global__ void __launch_bounds__(BS + 32, 1)
    k_cluster_steps(LatArgs a, const ClTile* tiles, ChainDraws cd, int n) {
  extern __shared__ __align__(16) uint32_t cl_smem[];
  __shared__ int s_part[2][16];               // every CTA's dn and nacc (16 bits each), by step parity
  __shared__ int s_acc[2];                    // this CTA's
  __shared__ int s_sb[NSH];                   // this CTA's per-shell sums of an accepted step
  __shared__ __align__(16) StepGeo s_geo[4];  // step j at j mod 4
  __shared__ float s_lg[4];
  __shared__ unsigned long long s_fin[16][NSH + 1];  // leader: every CTA's sb and ties of the launch
  constexpr int GS = SWAR ? 4 : 1;

  const int r = (int)cl_id();
  const uint32_t rank = cl_rank();
  const long long base = *cd.base;
  const int nctas = (int)cl_nctas();
  const bool solo = nctas == 1;
  const ClTile T = tiles[r];
  const LatGeom g = a.geom[r];
  const RepParams p = a.rp[r];
  const LatRep lr = a.lrep[r];
  TileView v;
  v.ty = (int)rank % T.TY;
  v.tz = (int)rank / T.TY;
  v.RY = T.Ty + 4;
  v.Y0 = v.ty * T.Ty;
  v.Z0 = v.tz * T.Tz;
  const int W = g.W, RZ = T.Tz + 4, zstride = v.RY * W;
  uint32_t* rows = cl_smem;
  const int nwords = RZ * v.RY * W;
  uint8_t* s_mask = reinterpret_cast<uint8_t*>(cl_smem + nwords + 2);
  const int mcap = (T.lcap + 15) / 16 * 16;
  const uint32_t rows_addr = smem_addr(rows);
  const int lane = threadIdx.x & 31, wi = threadIdx.x >> 5;
  const bool worker = wi < BS / 32;

  // ---- load the tile with halo (pending bits are clear: the host applied
  //      any pending commit before this launch)
  {
    const unsigned long long* src = a.bits + g.bits_off;
    for (int q = threadIdx.x; q < nwords; q += BS + 32) {
      const int w = q % W;
      const int rr = q / W;
      const int ly = rr % v.RY, lz = rr / v.RY;
      int Y = (v.Y0 - 2 + ly) % g.ny;
      Y = Y < 0 ? Y + g.ny : Y;
      int Z = (v.Z0 - 2 + lz) % g.nz;
      Z = Z < 0 ? Z + g.nz : Z;
      rows[q] = (uint32_t)__ldcg(src + ((long long)Z * g.ny + Y) * W + w);
    }
    if (threadIdx.x < 2) rows[nwords + threadIdx.x] = 0u;
  }
  if (threadIdx.x < 2) s_acc[threadIdx.x] = 0;
  if (threadIdx.x < NSH) s_sb[threadIdx.x] = 0;
  StepSums sums;
  long long sb_sum = 0;  // bookkeeping lane q < NSH: this CTA's shell-q sum over accepted steps
  int ties = 0;          // this thread's near ties
  // whole sublattice periods per tile: the rows of every colour are at the
  // same places in it
  const bool whole = T.Ty % a.qy == 0 && T.Tz % a.qz == 0;
  StepGeo s0{0, 0, 0, 0, v.Y0 / a.qy, v.Z0 / a.qz, T.Ty / a.qy, T.Tz / a.qz};
  // draws of step j, and its colour on this tile from them (one thread, which
  // loads a step ahead: this chain must not be longer than a step)
  auto draw = [&](int j) { return j < n ? ld_ahead(cd.cg + (size_t)j * a.R + r) : make_int2(0, 0); };
  auto geo = [&](int j, int2 cg) {
    StepGeo s = s0;
    s.b = cg.x & 1;
    const int pc = cg.x >> 1, pq = fdiv(pc, a.qx, a.rcp_qx);
    s.px = pc - pq * a.qx;
    s.pz = fdiv(pq, a.qy, a.rcp_qy);
    s.py = pq - s.pz * a.qy;
    if (!whole) {
      s.kyb = (v.Y0 - s.py + a.qy - 1) / a.qy;
      s.kzb = (v.Z0 - s.pz + a.qz - 1) / a.qz;
      s.cy = (v.Y0 + T.Ty - s.py + a.qy - 1) / a.qy - s.kyb;
      s.cz = (v.Z0 + T.Tz - s.pz + a.qz - 1) / a.qz - s.kzb;
    }
    s_geo[j & 3] = s;
    s_lg[j & 3] = __int_as_float(cg.y);
  };
  int2 cg_next = make_int2(0, 0);  // of step j + 2
  if (!worker && lane == 0) {
    geo(0, draw(0));
    geo(1, draw(1));
    cg_next = draw(2);
  }
  int n_prev = (int)__ldcg(&a.rs[r].n);  // B count at the start of the previous step
  if (!worker) sums.begin(a.rs[r], g, n_prev);
  float bG[NSH];                         // beta G_s
#pragma unroll
  for (int s = 0; s < NSH; ++s) bG[s] = lr.beta32 * a.G32[s];
  const float bC = lr.beta32 * lr.cpd32;
  __syncthreads();
  cl_arrive(solo);
  cl_wait(solo);

  const int nwq = SWAR ? (g.nxq + 3) / 4 : g.nxq;  // groups per row
  const float rcp_nwq = 1.0f / (float)nwq;
  struct Group {
    int ky, kz, jw;
  };
  auto decode = [&](const StepGeo& s, int t) {
    const int tq = fdiv(t, nwq, rcp_nwq);
    Group q;
    q.jw = t - tq * nwq;
    const int kzl = fdiv(tq, s.cy, __frcp_rn((float)s.cy));
    q.ky = s.kyb + tq - kzl * s.cy;
    q.kz = s.kzb + kzl;
    return q;
  };
  Group mine{0, 0, 0};  // whole tiles: this thread's first group, of every step
  if (whole && worker) mine = decode(s_geo[0], threadIdx.x);
  const float* lu = cd.lu + cd.off[r];
  auto load = [&](int j, const Group& q) {
    return ld_draw(reinterpret_cast<const Draw<GS>*>(lu + (size_t)j * cd.P + ((q.kz * g.nyq + q.ky) * nwq + q.jw) * GS));
  };

  // propose step j (colour s); cur: the first group's draws.  P: two 16-bit
  // sums each -- dn nacc, sb0 sb1, sb2 sb3, sb4; returns the near ties
  auto propose = [&](int j, const StepGeo& s, int ng, Draw<GS> cur, int (&P)[4]) {
    int tie = 0;
    const long long k = base + j;
    uint8_t* mask = s_mask + (j & 1) * mcap;
    P[0] = P[1] = P[2] = P[3] = 0;
    const int q0 = LAT_HALO + 2 * s.px + s.b - 3;
#pragma unroll 1
    for (int t = threadIdx.x; t < ng; t += BS) {
      const Group q = whole && t < BS ? mine : decode(s, t);
      const Draw<GS> dr = cur;
      if (t + BS < ng) cur = load(j, decode(s, t + BS));  // one group ahead
      const int ly = s.py + a.qy * q.ky - v.Y0 + 2, lz = s.pz + a.qz * q.kz - v.Z0 + 2;
      const uint32_t* row = rows + lz * zstride + ly * W;
      uint32_t cw[NSH], own;
      if constexpr (SWAR) {
        auto at = [&](int dy, int dz) { return row + q.jw + dz * zstride + dy * W; };
        own = s.b ? swar_counts<1, NSH>(at, q0, cw) : swar_counts<0, NSH>(at, q0, cw);
      } else {
        own = s.b ? popc_counts<1>(row, W, zstride, q0 + 2 * a.qx * q.jw, cw)
                  : popc_counts<0>(row, W, zstride, q0 + 2 * a.qx * q.jw, cw);
      }
      uint32_t acc = 0u, open = 0u;  // accepted and open trials: byte flags
#pragma unroll
      for (int i = 0; i < GS; ++i) {
        float x = bC;
#pragma unroll
        for (int s2 = 0; s2 < NSH; ++s2)
          x = fmaf(__uint_as_float(__byte_perm(cw[s2], 0x4B000000u, 0x7440 + i)) - 8388608.0f, bG[s2], x);
        x = __uint_as_float(__float_as_uint(x) ^ ((own << (31 - 8 * i)) & 0x80000000u));
        const int dec = log_screen(x, lr.dx, dr.l[i]);
        acc |= dec > 0 ? 1u << (8 * i) : 0u;
        open |= dec < 0 ? 1u << (8 * i) : 0u;
      }
      if constexpr (SWAR) {
        const int live = g.nxq - 4 * q.jw;  // trials of the row's last word
        const uint32_t lm = live >= 4 ? 0x01010101u : 0x01010101u >> (8 * (4 - live));
        acc &= lm;
        open &= lm;
      }
      while (open) {  // undecided by the screen: FP64
        const int i = (__ffs(open) - 1) >> 3;
        open &= open - 1u;
        int cnt[NSH];
#pragma unroll
        for (int s2 = 0; s2 < NSH; ++s2) cnt[s2] = (int)((cw[s2] >> (8 * i)) & 255u);
        const uint32_t d = (uint32_t)((q.kz * g.nyq + q.ky) * g.nxq + GS * q.jw + i);
        const uint4 w = philox4x32_10(make_uint4((uint32_t)k, (uint32_t)((uint64_t)k >> 32), d, TAG_TRIAL), p.key);
        int tie1 = 0;
        if (lattice_accept<NSH>(a, lr, p, cnt, 0, (own >> (8 * i)) & 1, top53(w.z, w.w), &tie1)) acc |= 1u << (8 * i);
        tie += tie1;
      }
      // byte flags -> bits 0..3
      mask[t] = (uint8_t)(SWAR ? (acc * 0x10204080u) >> 28 : acc);
      // signed sums over the group: +1 for A -> B, -1 for B -> A
      const int sg = (int)(acc ^ ((acc & own) * 0xFEu));
      P[0] += __dp4a(0x01010101, sg, 0) + (__popc(acc) << 16);
      P[1] += __dp4a((int)cw[0], sg, 0) + (__dp4a((int)cw[1], sg, 0) << 16);
      if constexpr (NSH == 5) {
        P[2] += __dp4a((int)cw[2], sg, 0) + (__dp4a((int)cw[3], sg, 0) << 16);
        P[3] += __dp4a((int)cw[4], sg, 0);
      }
    }
    return tie;
  };

  Draw<GS> d_cur{}, d_next{};
  {
    const StepGeo s = s_geo[0];
    if (worker && n > 0 && threadIdx.x < s.cy * s.cz * nwq) d_cur = load(0, whole ? mine : decode(s, threadIdx.x));
  }
  int Pp[3] = {0, 0, 0};  // the previous step's per-shell sums of this thread
  for (int j = 0; j <= n; ++j) {
    const int par = j & 1;
    const bool more = j < n;
    const StepGeo s = s_geo[j & 3];
    const int ng = more ? s.cy * s.cz * nwq : 0;
    int P[4], tie = 0;
    if (worker) {
      // the next step's first draws
      if (j + 1 < n) {
        const StepGeo sn = s_geo[(j + 1) & 3];
        if (threadIdx.x < sn.cy * sn.cz * nwq) d_next = load(j + 1, whole ? mine : decode(sn, threadIdx.x));
      }
    } else if (lane == 0) {
      geo(j + 2, cg_next);  // read from step j + 1 on
      cg_next = draw(j + 3);
    }
    for (bool again = false;;) {
      // ---- 1. propose step j on the species as they stand.  While other CTAs
      //      have passed the barrier of step j - 1 they may already be storing
      //      its flips into this CTA's halo: then it was accepted, and what is
      //      proposed here is thrown away below.
      if (worker) tie = propose(j, s, ng, d_cur, P);
      if (again || j == 0) break;
      cl_wait(solo);  // barrier of step j - 1
      // ---- 2. global decision of step j - 1, every thread alike
      const int w = lane < nctas ? s_part[par ^ 1][lane] : 0;
      const int dn = __reduce_add_sync(0xffffffffu, sum_lo(w));
      const int nacc = __reduce_add_sync(0xffffffffu, sum_hi(w));
      int gtie = 0;
      const int G = decide(a, lr, p, dn, nacc, n_prev, s_lg[(j - 1) & 3], base + j - 1, &gtie);
      if (G) n_prev += dn;
      if (!worker) sums.step(g.d, dn, nacc, gtie, G, n_prev);
      if (!G) break;
      // ---- 3. an accepted step: flip this thread's accepted trials, then the
      //      halo copies of the other CTAs, and propose step j again
      const StepGeo sp = s_geo[(j - 1) & 3];
      const int pg = sp.cy * sp.cz * nwq;
      const uint8_t* mask = s_mask + (par ^ 1) * mcap;
      auto each = [&](auto f) {
        for (int t = threadIdx.x; t < pg; t += BS) {
          const uint32_t m4 = mask[t];
          if (!m4) continue;
          const Group q = whole && t < BS ? mine : decode(sp, t);
          f(sp.py + a.qy * q.ky - v.Y0, sp.pz + a.qz * q.kz - v.Z0,
            group_words(g.nx, 2 * (sp.px + a.qx * GS * q.jw) + sp.b, (m4 * 0x00204081u) & 0x01010101u));
        }
      };
      __syncthreads();  // every warp of this CTA is done with its rows
      if (worker) {
        each([&](int oy, int oz, const GroupWords& q) {
          uint32_t* own = rows + ((oz + 2) * v.RY + (oy + 2)) * W;
          if (q.lo) atomicXor(own + q.w, q.lo);
          if (q.hi) atomicXor(own + q.w + 1, q.hi);
          if (q.hw >= 0) atomicXor(own + q.hw, q.hm);
        });
        if (__ballot_sync(0xffffffffu, (Pp[0] | Pp[1] | Pp[2]) != 0)) {
#pragma unroll
          for (int q = 0; q < 3; ++q) Pp[q] = __reduce_add_sync(0xffffffffu, Pp[q]);
          if (lane < NSH) {
            const int u = lane < 2 ? Pp[0] : (lane < 4 ? Pp[1] : Pp[2]);
            atomicAdd(&s_sb[lane], (lane & 1) ? sum_hi(u) : sum_lo(u));
          }
        }
      }
      __syncthreads();
      if (!worker && lane < NSH) {
        sb_sum += s_sb[lane];
        s_sb[lane] = 0;  // the next adds follow a block barrier
      }
      if (worker)
        each([&](int oy, int oz, const GroupWords& q) {
          // rows two or more from the tile's edges have no other copy
          if (oy < 2 || oy >= T.Ty - 2 || oz < 2 || oz >= T.Tz - 2) push_copies(rows, rows_addr, T, v, W, oy, oz, q);
        });
      cl_arrive(solo);
      cl_wait(solo);
      again = true;
    }
    if (!more) break;
    d_cur = d_next;

    // ---- 4. this CTA's sums of step j
    if (worker) {
      ties += tie;
#pragma unroll
      for (int q = 0; q < 3; ++q) Pp[q] = P[1 + q];
      if (__ballot_sync(0xffffffffu, P[0] != 0)) {
        const int w = __reduce_add_sync(0xffffffffu, P[0]);
        if (lane == 0) atomicAdd(&s_acc[par], w);
      }
    } else if (lane == 0) {
      s_acc[par ^ 1] = 0;  // step j - 1's sums, pushed before the last barrier
    }
    __syncthreads();
    // every CTA's copy of this CTA's sums of step j: by the bookkeeping warp,
    // so that no worker waits here for the draws it is loading (a release by
    // every warp took 1.1 us of a 2.6 us step)
    if (worker) {
      cl_arrive_relaxed(solo);
    } else {
      if (lane < nctas) {
        const int w = s_acc[par];
        if (solo) s_part[par][0] = w;
        else cl_st_u32(cl_map(smem_addr(&s_part[par][rank]), (uint32_t)lane), (uint32_t)w);
      }
      cl_arrive(solo);
    }
  }

  // the launch's per-shell sums and near ties of this CTA, to the leader
  if (threadIdx.x == 0) s_acc[0] = 0;
  __syncthreads();
  ties = __reduce_add_sync(0xffffffffu, ties);
  if (lane == 0 && ties) atomicAdd(&s_acc[0], ties);
  __syncthreads();
  if (!worker && lane <= NSH) {
    const unsigned long long u = lane < NSH ? (unsigned long long)sb_sum : (unsigned long long)s_acc[0];
    cl_st_u64(cl_map(smem_addr(&s_fin[rank][lane]), 0u), u);
  }
  // ---- write back the owned rows, then a last cluster barrier: no CTA
  //      leaves while another may still store into its shared memory
  {
    unsigned long long* dst = a.bits + g.bits_off;
    const int nw = T.Tz * T.Ty * W;
    for (int q = threadIdx.x; q < nw; q += BS + 32) {
      const int w = q % W;
      const int rr = q / W;
      const int oy = rr % T.Ty, oz = rr / T.Ty;
      dst[((long long)(v.Z0 + oz) * g.ny + v.Y0 + oy) * W + w] =
          (unsigned long long)rows[((oz + 2) * v.RY + (oy + 2)) * W + w];
    }
  }
  cl_arrive(solo);
  cl_wait(solo);
  if (rank == 0 && !worker && lane == 0) {
    long long sb[NSH + 1];
    for (int q = 0; q <= NSH; ++q) {
      sb[q] = 0;
      for (int c = 0; c < nctas; ++c) sb[q] += (long long)s_fin[c][q];
    }
    RepState S = a.rs[r];
    sums.fold(S, a, sb, NSH, sb[NSH], n, n_prev, base + n);
    hand_over(a, r, S, base + n);
  }
  if (rank == 0) lat_colours_ahead(a, r, p.key, base + n, threadIdx.x, BS + 32);
}

// ------------------------------------------------ one CTA per replica, picks
// BLOCKS and OVERLAP schedules: domain d of the colour picks one of its sites
// (k_chain_draws).  The whole replica's rows are in shared memory (no halo
// rows; y and z wrap), one trial per thread and round.  With one warp the
// step needs no block barrier at all.  NSH = 5 or 2: the compile-time BCC
// shells, 0: the runtime row table.
struct PickRow {
  int dy, dz;
  uint32_t mask[LAT_MAX_SH];
};

template <int NSH, int MAXB>
__global__ void __launch_bounds__(MAXB, 1) k_pick_steps(LatArgs a, ChainDraws cd, int n) {
  extern __shared__ __align__(16) uint32_t cl_smem[];
  constexpr int NS = NSH > 0 ? NSH : LAT_MAX_SH;
  constexpr int NP = (NS + 1) / 2;  // words of two 16-bit per-shell sums
  __shared__ PickRow s_row[NSH > 0 ? 1 : 2 * LAT_MAX_ROWS];
  __shared__ int s_acc[3];  // dn and nacc (16 bits each); step j at j mod 3
  __shared__ int s_sb[NS + 1];

  const int r = blockIdx.x;
  const int BS = (int)blockDim.x;
  const long long base = *cd.base;
  const bool one = BS == 32;
  const LatGeom g = a.geom[r];
  const RepParams p = a.rp[r];
  const LatRep lr = a.lrep[r];
  const int W = g.W, nwords = g.ny * g.nz * W;
  uint32_t* rows = cl_smem;
  const int lane = threadIdx.x & 31;

  for (int q = threadIdx.x; q < nwords + 2; q += BS) rows[q] = q < nwords ? (uint32_t)__ldcg(a.bits + g.bits_off + q) : 0u;
  if (NSH == 0)
    for (int q = threadIdx.x; q < 2 * LAT_MAX_ROWS; q += BS) {
      const LatRow& src = a.rows[q / LAT_MAX_ROWS][q % LAT_MAX_ROWS];
      s_row[q].dy = src.dy;
      s_row[q].dz = src.dz;
      for (int s = 0; s < LAT_MAX_SH; ++s) s_row[q].mask[s] = src.mask[s];
    }
  if (threadIdx.x < 3) s_acc[threadIdx.x] = 0;
  if (threadIdx.x <= NS) s_sb[threadIdx.x] = 0;
  StepSums sums;         // thread 0
  long long sb_sum[NS];  // thread 0: per-shell sums over accepted steps
#pragma unroll
  for (int s = 0; s < NS; ++s) sb_sum[s] = 0;
  int ties = 0;
  int n_prev = (int)__ldcg(&a.rs[r].n);
  sums.begin(a.rs[r], g, n_prev);
  float bG[NS];
#pragma unroll
  for (int s = 0; s < NS; ++s) bG[s] = lr.beta32 * a.G32[s];
  const float bC = lr.beta32 * lr.cpd32;
  __syncthreads();

  // site and -ln u of this thread's trial d of step j
  const int2* su = cd.su + cd.off[r];
  const int dmax = g.dmax;
  auto load = [&](int j, int d) {
    return j < n && d < dmax ? ld_ahead(su + (size_t)j * cd.P + d) : make_int2(-1, 0);
  };
  int2 nx = load(0, threadIdx.x);
  int2 cg = n > 0 ? __ldg(cd.cg + r) : make_int2(0, 0);

  int par = 0;
#pragma unroll 1
  for (int j = 0; j < n; ++j, par = par == 2 ? 0 : par + 1) {
    int2 cur = nx;
    const int2 cgj = cg;
    nx = load(j + 1, threadIdx.x);
    if (j + 1 < n) cg = ld_ahead(cd.cg + (size_t)(j + 1) * a.R + r);
    unsigned amask = 0u;  // accepted rounds
    const int first = cur.x;
    int P0 = 0, P[NP];
#pragma unroll
    for (int q = 0; q < NP; ++q) P[q] = 0;
    int rd = 0;
#pragma unroll 1
    for (int d = threadIdx.x; d < dmax; d += BS, ++rd) {
      const int site = cur.x;
      const float l = __int_as_float(cur.y);
      if (d + BS < dmax) cur = load(j, d + BS);
      if (site < 0) continue;
      const int cell = site >> 1, b = site & 1;
      const int q = fdiv(cell, g.nx, g.rcp_nx);
      const int X = cell - q * g.nx, Z = fdiv(q, g.ny, g.rcp_ny), Y = q - Z * g.ny;
      const int H = 2 * X + b;
      uint32_t cw[NS];
      uint32_t own;
      if constexpr (NSH > 0) {
        const int q0 = LAT_HALO + H - 3, sh = q0 & 31;
        const uint32_t* b0 = rows + (q0 >> 5);
        int yo[5], zo[5];
#pragma unroll
        for (int e = -2; e <= 2; ++e) {
          yo[e + 2] = wrap_add(Y, e, g.ny) * W;
          zo[e + 2] = wrap_add(Z, e, g.nz) * g.ny * W;
        }
        auto at = [&](int dy, int dz) { return b0 + zo[dz + 2] + yo[dy + 2]; };
        own = b ? swar_counts<1, NSH>(at, sh, cw) : swar_counts<0, NSH>(at, sh, cw);
        own &= 1u;
#pragma unroll
        for (int s = 0; s < NS; ++s) cw[s] &= 255u;
      } else {
        const int q0 = LAT_HALO + H - a.hmax, sh = q0 & 31;
        const int nr = a.n_rows[b];
        const PickRow* tab = s_row + b * LAT_MAX_ROWS;
#pragma unroll
        for (int s = 0; s < NS; ++s) cw[s] = 0u;
        for (int e = 0; e < nr; ++e) {
          const int yy = wrap_add(Y, tab[e].dy, g.ny), zz = wrap_add(Z, tab[e].dz, g.nz);
          const uint32_t* pr = rows + (zz * g.ny + yy) * W + (q0 >> 5);
          const uint32_t win = __funnelshift_r(pr[0], pr[1], sh);
#pragma unroll
          for (int s = 0; s < NS; ++s) cw[s] += __popc(win & tab[e].mask[s]);
        }
        const int pp = LAT_HALO + H;
        own = (rows[q * W + (pp >> 5)] >> (pp & 31)) & 1u;
      }
      float x = bC;
#pragma unroll
      for (int s = 0; s < NS; ++s) x = fmaf(__uint_as_float(cw[s] | 0x4B000000u) - 8388608.0f, bG[s], x);
      x = own ? -x : x;
      int dec = log_screen(x, lr.dx, l);
      if (dec < 0) {  // undecided by the screen: FP64
        int cnt[NS], tie1 = 0;
#pragma unroll
        for (int s = 0; s < NS; ++s) cnt[s] = (int)cw[s];
        const long long k = base + j;
        const uint4 w =
            philox4x32_10(make_uint4((uint32_t)k, (uint32_t)((uint64_t)k >> 32), (uint32_t)d, TAG_TRIAL), p.key);
        dec = lattice_accept<NS>(a, lr, p, cnt, 0, (int)own, top53(w.z, w.w), &tie1) ? 1 : 0;
        ties += tie1;
      }
      if (dec > 0) {
        amask |= 1u << rd;
        P0 += (own ? -1 : 1) + (1 << 16);
#pragma unroll
        for (int s = 0; s < NS; ++s) {
          const int v = own ? -(int)cw[s] : (int)cw[s];
          P[s / 2] += (s & 1) ? v << 16 : v;
        }
      }
    }
    // dn and nacc of the step, in every thread
    int w = 0;
    if (__ballot_sync(0xffffffffu, P0 != 0)) {
      w = __reduce_add_sync(0xffffffffu, P0);
      if (!one && lane == 0) atomicAdd(&s_acc[par], w);
    }
    if (!one) {
      // step j - 2's sums, last read before the barrier of step j - 1, are
      // cleared for step j + 1
      if (threadIdx.x == 0) s_acc[par == 2 ? 0 : par + 1] = 0;
      __syncthreads();
      w = s_acc[par];
    }
    const int dn = sum_lo(w), nacc = sum_hi(w);
    int gtie = 0;
    const int G = decide(a, lr, p, dn, nacc, n_prev, __int_as_float(cgj.y), base + j, &gtie);
    if (G) {
      n_prev += dn;
      if (amask) {
        int rq = 0;
        for (int d = threadIdx.x; d < dmax; d += BS, ++rq) {
          if (!(amask >> rq & 1u)) continue;
          const int st = rq == 0 ? first : __ldg(su + (size_t)j * cd.P + d).x;
          const int cell = st >> 1;
          const int q = fdiv(cell, g.nx, g.rcp_nx);
          const GroupWords gw = group_words(g.nx, 2 * (cell - q * g.nx) + (st & 1), 1u);
          atomicXor(rows + q * W + gw.w, gw.lo);
          if (gw.hw >= 0) atomicXor(rows + q * W + gw.hw, gw.hm);
        }
      }
      // per-shell sums: warp, then block
      if (__ballot_sync(0xffffffffu, amask != 0u)) {
#pragma unroll
        for (int q = 0; q < NP; ++q) {
          const int u = __reduce_add_sync(0xffffffffu, P[q]);
          if (lane == 0) {
            atomicAdd(&s_sb[2 * q], sum_lo(u));
            if (2 * q + 1 < NS) atomicAdd(&s_sb[2 * q + 1], sum_hi(u));
          }
        }
      }
      __syncthreads();  // flips and sums are in
      if (threadIdx.x == 0) {
#pragma unroll
        for (int s = 0; s < NS; ++s) {
          sb_sum[s] += s_sb[s];
          s_sb[s] = 0;  // the next adds of other warps follow a block barrier
        }
      }
    }
    if (threadIdx.x == 0) sums.step(cgj.x, dn, nacc, gtie, G, n_prev);
  }

  __syncthreads();
  ties = __reduce_add_sync(0xffffffffu, ties);
  if (lane == 0 && ties) atomicAdd(&s_sb[NS], ties);
  __syncthreads();
  for (int q = threadIdx.x; q < nwords; q += BS) a.bits[g.bits_off + q] = (unsigned long long)rows[q];
  if (threadIdx.x == 0) {
    RepState S = a.rs[r];
    sums.fold(S, a, sb_sum, NS, s_sb[NS], n, n_prev, base + n);
    hand_over(a, r, S, base + n);
  }
  lat_colours_ahead(a, r, p.key, base + n, threadIdx.x, BS);
}

namespace {

using ClusterKernel = void (*)(LatArgs, const ClTile*, ChainDraws, int);

template <int BS>
ClusterKernel cluster_kernel_bs(const LatArgs& a) {
  if (a.bcc2) return k_cluster_steps<2, true, BS>;
  return a.qx == 4 ? k_cluster_steps<5, true, BS> : k_cluster_steps<5, false, BS>;
}
ClusterKernel cluster_kernel(const LatArgs& a, int block) {
  return block == 256 ? cluster_kernel_bs<256>(a) : cluster_kernel_bs<512>(a);
}

using PickKernel = void (*)(LatArgs, ChainDraws, int);

PickKernel pick_kernel(const LatArgs& a, int block) {
  if (block <= 64) return a.bcc5 ? k_pick_steps<5, 64> : (a.bcc2 ? k_pick_steps<2, 64> : k_pick_steps<0, 64>);
  return a.bcc5 ? k_pick_steps<5, 512> : (a.bcc2 ? k_pick_steps<2, 512> : k_pick_steps<0, 512>);
}

void cluster_config(cudaLaunchConfig_t& cfg, cudaLaunchAttribute& attr, int blocks, int csize, int block, size_t smem) {
  cfg.gridDim = dim3((unsigned)blocks);
  cfg.blockDim = dim3((unsigned)(block + 32));
  cfg.dynamicSmemBytes = smem;
  attr.id = cudaLaunchAttributeClusterDimension;
  attr.val.clusterDim.x = (unsigned)csize;
  attr.val.clusterDim.y = 1;
  attr.val.clusterDim.z = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
}

}  // namespace

cudaError_t launch_chain_draws(const LatArgs& a, const ChainDraws& cd, int m, cudaStream_t st) {
  const dim3 grid((unsigned)((cd.pmax + 255) / 256), (unsigned)m, (unsigned)a.R);
  if (!a.sublattice) k_chain_draws<0><<<grid, 256, 0, st>>>(a, cd);
  else if (a.qx == 4) k_chain_draws<4><<<grid, 256, 0, st>>>(a, cd);
  else k_chain_draws<1><<<grid, 256, 0, st>>>(a, cd);
  return cudaGetLastError();
}

// Attributes belong to a kernel, not to a context: every context sets the same
// largest size, so that none lowers it under another thread's launch.
cudaError_t resident_attributes(const LatArgs& a) {
  cudaError_t e = cudaSuccess;
  for (int block : {256, 512}) {
    if (a.sublattice) {
      const ClusterKernel k = cluster_kernel(a, block);
      if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
      if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)CL_SMEM_MAX);
    } else if (e == cudaSuccess) {
      e = cudaFuncSetAttribute(pick_kernel(a, block == 256 ? 64 : 512), cudaFuncAttributeMaxDynamicSharedMemorySize,
                               (int)PICK_SMEM_MAX);
    }
  }
  return e;
}

cudaError_t launch_cluster_steps(const LatArgs& a, const ClTile* d_tiles, const ChainDraws& cd, size_t smem, int csize,
                                 int block, int n, cudaStream_t st) {
  const ClusterKernel k = cluster_kernel(a, block);
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  cluster_config(cfg, attr[0], a.R * csize, csize, block, smem);
  cfg.stream = st;
  return cudaLaunchKernelEx(&cfg, k, a, d_tiles, cd, n);
}

int cluster_capacity(const LatArgs& a, int csize, int block, size_t smem) {
  const ClusterKernel k = cluster_kernel(a, block);
  int n = 0;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  cluster_config(cfg, attr[0], csize, csize, block, smem);
  if (cudaOccupancyMaxActiveClusters(&n, k, &cfg) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return n;
}

int pick_capacity(const LatArgs& a, int block, size_t smem) {
  int n = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, pick_kernel(a, block), block, smem) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return n;
}

cudaError_t launch_pick_steps(const LatArgs& a, const ChainDraws& cd, size_t smem, int block, int n, cudaStream_t st) {
  pick_kernel(a, block)<<<a.R, block, smem, st>>>(a, cd, n);
  return cudaGetLastError();
}

}  // namespace vcsgc
