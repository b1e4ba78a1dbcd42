// Individual power-of-two time steps on a static mesh (Sec. 7.2) with the
// signal-speed criterion of eq. (EqnTiStepIndividual), templated on the bulk
// arithmetic type like hydro.cuh (instantiated in hydro_f64.cu and
// hydro_f32.cu).
//
// A cycle of length dt_max runs in integer ticks of dt_max / 2^D (D =
// max_depth); cell i steps by 2^(D - bin_i) ticks and is active at a tick
// its step divides.  Per tick with active cells the host enqueues:
//
//  k_ind_activate  active cells: W from Q (cw), their walk record, the
//                  active-cell list                          (Sec. 7.2)
//  k_ind_leaf / k_ind_up   per bucket of a uniform-grid pyramid over the
//                  box: the largest c + |v| of its cells and that cell
//  k_ind_cells     active cells: limited gradients (eq. eqngrad2), the
//                  neighbours entering with their stored W, by every other
//                  CTA (ind_grad)                            (Sec. 3.1);
//                  dt_i = C min(tau_i, R_i/(c_i+|v_i|)) by a pruned walk of
//                  the pyramid, the new bin (a shorter step freely, a longer
//                  one at most twice the current step and only where that
//                  step starts now) and the bin histogram, by the others
//                  (ind_bins)                                (Sec. 7.1, 7.2)
//  k_ind_faces     faces with an active cell: the active-face list, their
//                  step (the smaller of the two cells') and stamps
//  k_ind_flux      active faces: extrapolation, each side predicted from its
//                  own last activation to the middle of the face's step,
//                  Riemann solve, flux (Sec. 3.3); in the FP64 form one
//                  launch for few faces and one for many, of which the
//                  other leaves at once
//  k_ind_update    touched cells: Q -= sum over active faces of
//                  +-dt_f A F (pairwise, conservative; no atomics)
//
// and reads back the bin histogram (64 counters) to find the next tick.
// Lists are built with warp-aggregated atomics; their order is not
// deterministic, but every list item is computed independently and every
// per-cell sum runs in the cell's fixed incidence order, so the results are.
#pragma once

#include "hydro.cuh"

namespace amm {

__device__ __forceinline__ int warp_append(int* counter, bool pred) {
  const unsigned lane = threadIdx.x & 31u;
  const unsigned mask = __ballot_sync(0xffffffffu, pred);
  if (mask == 0u) return -1;
  const int leader = __ffs(mask) - 1;
  int base = 0;
  if ((int)lane == leader) base = atomicAdd(counter, __popc(mask));
  base = __shfl_sync(0xffffffffu, base, leader);
  return pred ? base + __popc(mask & ((1u << lane) - 1u)) : -1;
}

__device__ __forceinline__ long long step_ticks(int depth, int b) { return 1ll << (depth - b); }

// ------------------------------------------------------------- activation
template <typename real>
__global__ void k_ind_activate(HydroView<real> v, IndView d) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const bool in = i < d.n;
  const long long tick = d.loop->tick;
  bool active = false;
  if (in) active = (tick & (step_ticks(d.depth, d.bin[i]) - 1)) == 0;
  const int at = warp_append(d.count, active);
  if (!in) return;
  d.act[i] = active ? 1 : 0;
  if (!active) return;
  d.list[at] = i;
  const size_t n = (size_t)v.n;
  const double m = v.Q[i], px = v.Q[n + i], py = v.Q[2 * n + i], pz = v.Q[3 * n + i], E = v.Q[4 * n + i];
  const real P = prims_from_Q(v, i, m, px, py, pz, E);
  if (!(m > 0.0) || !(P > (real)0)) {
    atomicAdd(&v.stats->nonpos, 1ull);
    atomicOr(&v.stats->status, (unsigned)ST_NONPOS);
    atomicOr(v.box_status, (unsigned)ST_NONPOS);
  }
  if (d.signal) {
    // the walk record: position, sound speed, velocity and speed in FP64
    const R4<real> w = v.cw[2 * (size_t)i];
    const double rho = (double)w.x, Pd = (double)P;
    const double vx = (double)w.y, vy = (double)w.z, vz = (double)w.w;
    const double* g = d.gen + 3 * (size_t)i;
    double4 a, b;
    a.x = g[0]; a.y = g[1]; a.z = g[2];
    a.w = sqrt(d.gamma * Pd / rho);
    b.x = vx; b.y = vy; b.z = vz;
    b.w = sqrt(vx * vx + vy * vy + vz * vz);
    const int s = d.cell_slot[i];
    d.rec[2 * (size_t)s] = a;
    d.rec[2 * (size_t)s + 1] = b;
    d.rec32[2 * (size_t)s] = make_float4((float)a.x, (float)a.y, (float)a.z, (float)a.w);
    d.rec32[2 * (size_t)s + 1] = make_float4((float)b.x, (float)b.y, (float)b.z, (float)b.w);
  }
}

// ------------------------------------------------------------ the pyramid
// coordinates of bucket b of a level
__device__ __forceinline__ void bucket_coords(int dim, int l, int b, int& ix, int& iy, int& iz) {
  const int m = (1 << l) - 1;
  if (dim == 3) {
    ix = b >> (2 * l); iy = (b >> l) & m; iz = b & m;
  } else {
    ix = b >> l; iy = b & m; iz = 0;
  }
}

// The two finest levels: a warp per bucket of the second finest, its lanes shared
// out among the 2^dim leaf buckets in it, so that the records of a leaf are read at
// once instead of one behind the other (a thread per leaf took 20 us a tick,
// 4.5 now).
static __global__ void __launch_bounds__(256) k_ind_leaf(IndView d) {
  const int l = d.levels - 2, side = 1 << l, cs = 2 * side;
  const int per = 1 << (d.dim * l);
  const int b = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (b >= per) return;
  const int lanes = 32 >> d.dim, q = lane / lanes;
  int ix, iy, iz;
  bucket_coords(d.dim, l, b, ix, iy, iz);
  const int jx = 2 * ix + (q & 1), jy = 2 * iy + ((q >> 1) & 1), jz = 2 * iz + ((q >> 2) & 1);
  const int leaf = (d.dim == 3) ? (jx * cs + jy) * cs + jz : jx * cs + jy;
  // FP32 records, the maximum raised by 1e-5 to cover their rounding (the
  // bounds are used in FP32 only); an empty bucket keeps -1 and a valid slot
  float m = -1.0f;
  const int s0 = d.leaf_off[leaf], s1 = d.leaf_off[leaf + 1];
  int arg = min(s0, d.n - 1);
  for (int s = s0 + lane % lanes; s < s1; s += lanes) {
    const float4 a = d.rec32[2 * (size_t)s], c = d.rec32[2 * (size_t)s + 1];
    if (a.w + c.w > m) {
      m = a.w + c.w;
      arg = s;
    }
  }
  if (m >= 0.0f) m *= 1.0f + 1e-5f;
  for (int o = 1; o < 32; o <<= 1) {
    if (o == lanes && lane % lanes == 0) d.node[d.level_off[l + 1] + leaf] = make_float2(m, __int_as_float(arg));
    const float mo = __shfl_xor_sync(0xffffffffu, m, o);
    const int ao = __shfl_xor_sync(0xffffffffu, arg, o);
    if (mo > m || (mo == m && ao < arg)) {
      m = mo;
      arg = ao;
    }
  }
  if (lane == 0) d.node[d.level_off[l] + b] = make_float2(m, __int_as_float(arg));
}

// all coarser levels by one CTA, finest first
static __global__ void __launch_bounds__(1024) k_ind_up(IndView d) {
  const int ch = (d.dim == 3) ? 8 : 4;
  for (int l = d.levels - 3; l >= 0; l--) {
    const int per = 1 << (d.dim * l), side = 1 << l;
    for (int b = threadIdx.x; b < per; b += blockDim.x) {
      int ix, iy, iz;
      bucket_coords(d.dim, l, b, ix, iy, iz);
      const int cs = side * 2;
      float2 m = make_float2(-2.0f, 0.0f);
      for (int q = 0; q < ch; q++) {
        const int jx = 2 * ix + (q & 1), jy = 2 * iy + ((q >> 1) & 1), jz = 2 * iz + ((q >> 2) & 1);
        const int cb = (d.dim == 3) ? (jx * cs + jy) * cs + jz : jx * cs + jy;
        const float2 c = d.node[d.level_off[l + 1] + cb];
        if (c.x > m.x) m = c;
      }
      d.node[d.level_off[l] + b] = m;
    }
    __syncthreads();
  }
}

// ---------------------------------------------------- gradients of active cells
// The active cells' gradients by CTAs of BINS_WARPS warps, G lanes per cell.  The
// warps of a round are numbered across the CTAs first, so that few cells spread
// over all SMs' FP64 pipes.
constexpr int BINS_WARPS = 4;
template <typename real, int G>
__device__ __forceinline__ void ind_grad(const HydroView<real>& v, const IndView& d, int cta, int ctas) {
  constexpr int CELLS = 32 / G;
  const int count = d.count[0];
  const int lane = (int)threadIdx.x % G;
  for (int w = ((int)threadIdx.x >> 5) * ctas + cta; w * CELLS < count; w += ctas * BINS_WARPS) {
    const int idx = w * CELLS + ((int)threadIdx.x & 31) / G;
    const bool valid = idx < count;
    const int i = d.list[valid ? idx : 0];
    R4<real> Wi, cg;
    real Pi;
    grad_cell<real, G, false>(v, i, i, valid, lane, Wi, Pi, cg);
  }
}

// ------------------------------------------------------ bins of active cells
// Periodic distance from x to the interval [lo, lo + h] on a circle of length L.
__device__ __forceinline__ float interval_gap(float x, float lo, float h, float L) {
  const float hi = lo + h;
  if (x >= lo && x <= hi) return 0.0f;
  const float a = (x < lo) ? lo - x : x - hi;       // direct
  const float b = (x < lo) ? x + L - hi : lo + L - x;  // through the periodic boundary
  return a < b ? a : b;
}

// r_ij / (c_i + c_j - v_ij . r_ij / r_ij) for the cell in walk slot s, to the
// nearest periodic image; +inf where the signal speed is not positive
__device__ __forceinline__ double pair_tau(const IndView& d, int s, double xi, double yi, double zi, double ci,
                                          double vx, double vy, double vz) {
  const double4 a = d.rec[2 * (size_t)s], c = d.rec[2 * (size_t)s + 1];
  double dx = xi - a.x, dy = yi - a.y, dz = zi - a.z;
  if (dx > 0.5 * d.box[0]) dx -= d.box[0]; else if (dx < -0.5 * d.box[0]) dx += d.box[0];
  if (dy > 0.5 * d.box[1]) dy -= d.box[1]; else if (dy < -0.5 * d.box[1]) dy += d.box[1];
  if (d.dim == 3) {
    if (dz > 0.5 * d.box[2]) dz -= d.box[2]; else if (dz < -0.5 * d.box[2]) dz += d.box[2];
  } else {
    dz = 0.0;
  }
  const double r = sqrt(dx * dx + dy * dy + dz * dz);
  const double vr = (vx - c.x) * dx + (vy - c.y) * dy + (vz - c.z) * dz;
  const double sig = ci + a.w - vr / r;
  return sig > 0.0 ? r / sig : INFINITY;
}

// the warp's minimum of non-negative values (which order like their bits: no
// FP64 comparisons)
__device__ __forceinline__ double warp_min_d(double x) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const unsigned h = __reduce_min_sync(0xffffffffu, hi);
  const unsigned l = __reduce_min_sync(0xffffffffu, hi == h ? lo : 0xffffffffu);
  return __hiloint2double((int)h, (int)l);
}

// FP32 bounds of a pair's value r / sig, from the FP32 records, with margins
// well above the FP32 rounding of the positions (eps, absolute), of the
// speeds (relative 1e-5) and of the direction of r_ij (|v_ij| eps / r):
// lo <= the FP64 value <= hi; lo = 0 where the pair is too close to bound,
// lo = hi = +inf where the signal speed cannot be positive.
__device__ __forceinline__ void pair_tau_bounds(const IndView& d, int s, float xi, float yi, float zi, float ci,
                                                float vx, float vy, float vz, float eps, float& lo, float& hi) {
  const float4 a = d.rec32[2 * (size_t)s], c = d.rec32[2 * (size_t)s + 1];
  float dx = xi - a.x, dy = yi - a.y, dz = zi - a.z;
  const float bx = (float)d.box[0], by = (float)d.box[1], bz = (float)d.box[2];
  if (dx > 0.5f * bx) dx -= bx; else if (dx < -0.5f * bx) dx += bx;
  if (dy > 0.5f * by) dy -= by; else if (dy < -0.5f * by) dy += by;
  if (d.dim == 3) {
    if (dz > 0.5f * bz) dz -= bz; else if (dz < -0.5f * bz) dz += bz;
  } else {
    dz = 0.0f;
  }
  const float r = sqrtf(dx * dx + dy * dy + dz * dz);
  const float rlo = r - 4.0f * eps, rhi = r + 4.0f * eps;
  lo = 0.0f;
  hi = INFINITY;
  if (!(rlo > 0.0f)) return;
  const float ux = vx - c.x, uy = vy - c.y, uz = vz - c.z;
  const float du = sqrtf(ux * ux + uy * uy + uz * uz);
  const float sig = ci + a.w - (ux * dx + uy * dy + uz * dz) / r;
  const float m = 1e-5f * (ci + a.w + du) + 2.0f * du * (4.0f * eps) / rlo;
  const float sig_hi = sig + m, sig_lo = sig - m;
  if (!(sig_hi > 0.0f)) {
    lo = INFINITY;
    return;
  }
  lo = rlo / sig_hi * (1.0f - 1e-5f);
  if (sig_lo > 0.0f) hi = rhi / sig_lo * (1.0f + 1e-5f);
}

// One warp per active cell: dt_i = C min(tau_i, R_i / (c_i + |v_i|)) of
// eq. (EqnTiStepIndividual), then the cell's bin.
//
// tau_i = min_j r_ij / (c_i + c_j - v_ij . r_ij / r_ij) by a walk of the
// pyramid.  A bucket cannot hold a pair below gap / (c_i + |v_i| + max_j
// (c_j + |v_j|)) (r >= gap, signal speed <= c_i + c_j + |v_i - v_j|); the walk
// skips buckets whose bound is not below the current one and opens the others.
// The bounds and a first screen of the pairs run in FP32 with conservative
// margins; every pair that passes the screen is evaluated exactly in FP64, so
// the minimum is the FP64 minimum over all pairs, in whatever order it is
// found.  It starts from the pairs with the fastest cell of every bucket of a
// coarse level (any pair value bounds the minimum) and the cells of the 3^dim
// buckets around the cell.
//
// What bounds it is the latency of one warp's chain, for most ticks start few
// cells: so a step of the walk opens as many buckets as their children fill the
// lanes (32 / 2^dim), from the top of a stack; the buckets to scan are gathered
// and their cells spread over the lanes; and the pairs that pass the screen are
// listed and evaluated together at the end.  (With one bucket opened per step,
// a lane per bucket scanned, FP64 pairs at once and 64 cells a bucket: 92 us for a few
// cells, 1.5 ms for 32768; 25 us and 0.34 ms now.)
constexpr int WALK_STACK = 256;   // a step pops 32 / 2^dim buckets and pushes at most 32, over at most 9 levels
constexpr int WALK_PENDING = 64;

struct WalkShared {
  unsigned node[WALK_STACK];
  float lb[WALK_STACK];
  int base[33], off[33];          // a scan's runs of slots
  int leaf[32];                   // buckets to scan
  int pending[WALK_PENDING];      // pairs to evaluate exactly
};

// the cell the walk is for, and its bounds
struct WalkCell {
  int self;                       // its slot
  double xi, yi, zi, ci, vx, vy, vz;
  float xf, yf, zf, cf, vxf, vyf, vzf, eps;
  double cur;                     // the minimum so far, exact
  float curf;                     // an upper bound of the minimum
  int npend;
};

__device__ __forceinline__ void walk_flush(const IndView& d, WalkShared& S, WalkCell& C, int lane) {
  __syncwarp();
  double t = INFINITY;
  for (int q = lane; q < C.npend; q += 32) {
    const double ts = pair_tau(d, S.pending[q], C.xi, C.yi, C.zi, C.ci, C.vx, C.vy, C.vz);
    t = ts < t ? ts : t;
  }
  t = warp_min_d(t);
  C.npend = 0;
  if (t < C.cur) {
    C.cur = t;
    C.curf = fminf(C.curf, (float)t * (1.0f + 1e-5f));
  }
  __syncwarp();
}

// The cells of the lanes' runs [s0, s1) of slots, SCAN_PER a lane at a time: their
// upper bounds tighten curf, then those whose lower bound stays below it are listed.
constexpr int SCAN_PER = 8;
__device__ __forceinline__ void walk_scan(const IndView& d, WalkShared& S, WalkCell& C, int lane, int s0, int s1) {
  const int cnt = s1 - s0;
  int pre = cnt;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, pre, o);
    if (lane >= o) pre += y;
  }
  __syncwarp();
  S.base[lane] = s0;
  S.off[lane] = pre - cnt;
  const int total = __shfl_sync(0xffffffffu, pre, 31);
  __syncwarp();
  for (int q0 = 0; q0 < total; q0 += 32 * SCAN_PER) {
    float lo[SCAN_PER], hmin = INFINITY;
    int slot[SCAN_PER];
#pragma unroll
    for (int u = 0; u < SCAN_PER; u++) {
      const int q = q0 + 32 * u + lane;
      int r = 0;   // the last run that starts at or before q
#pragma unroll
      for (int o = 16; o > 0; o >>= 1)
        if (S.off[r + o] <= q) r += o;
      const int s = q < total ? S.base[r] + (q - S.off[r]) : C.self;
      float hi;
      pair_tau_bounds(d, s, C.xf, C.yf, C.zf, C.cf, C.vxf, C.vyf, C.vzf, C.eps, lo[u], hi);
      if (s == C.self) lo[u] = hi = INFINITY;
      hmin = fminf(hmin, hi);
      slot[u] = s;
    }
    C.curf = fminf(C.curf, __uint_as_float(__reduce_min_sync(0xffffffffu, __float_as_uint(hmin))));
#pragma unroll
    for (int u = 0; u < SCAN_PER; u++) {
      const bool need = lo[u] < C.curf;
      const unsigned m = __ballot_sync(0xffffffffu, need);
      if (m == 0u) continue;
      if (C.npend + __popc(m) > WALK_PENDING) walk_flush(d, S, C, lane);
      if (need) S.pending[C.npend + __popc(m & ((1u << lane) - 1u))] = slot[u];
      C.npend += __popc(m);
    }
  }
}

// first node of a pyramid level
__device__ __forceinline__ int level_start(int l, int dim) { return dim == 3 ? ((1 << (3 * l)) - 1) / 7 : ((1 << (2 * l)) - 1) / 3; }

template <typename real>
__device__ __forceinline__ void ind_bins(const HydroView<real>& v, const IndView& d, int cta, int ctas) {
  __shared__ WalkShared shared[BINS_WARPS];
  const unsigned full = 0xffffffffu;
  const int lane = (int)threadIdx.x & 31, w = (int)threadIdx.x >> 5;
  WalkShared& S = shared[w];
  const int count = d.count[0];
  const long long tick = d.loop->tick;
  const float bx = (float)d.box[0], by = (float)d.box[1], bz = (float)d.box[2];
  for (int idx = w * ctas + cta; idx < count; idx += ctas * BINS_WARPS) {
    const int i = d.list[idx];
    // the cell's position, sound speed, velocity and speed in FP64: the walk
    // record the activation kernel wrote (one thread per cell), rather than
    // every lane of this warp repeating the FP64 square roots on the narrow
    // FP64 pipe
    WalkCell C;
    double si;
    if (d.signal) {
      const int slot = d.cell_slot[i];
      C.self = slot;
      const double4 ra = d.rec[2 * (size_t)slot], rb = d.rec[2 * (size_t)slot + 1];
      C.xi = ra.x; C.yi = ra.y; C.zi = ra.z; C.ci = ra.w;
      C.vx = rb.x; C.vy = rb.y; C.vz = rb.z; si = rb.w;
    } else {
      const R4<real> wi = v.cw[2 * (size_t)i];
      const double rho = (double)wi.x, P = (double)v.cw[2 * (size_t)i + 1].x;
      C.vx = (double)wi.y; C.vy = (double)wi.z; C.vz = (double)wi.w;
      C.xi = C.yi = C.zi = 0.0;
      C.ci = sqrt(d.gamma * P / rho);
      si = sqrt(C.vx * C.vx + C.vy * C.vy + C.vz * C.vz);
    }
    double cur = (double)v.crad[i] / (C.ci + si);           // R_i / (c_i + |v_i|)
    if (d.signal) {
      C.cur = cur;
      C.npend = 0;
      C.xf = (float)C.xi; C.yf = (float)C.yi; C.zf = (float)C.zi;
      C.cf = (float)C.ci; C.vxf = (float)C.vx; C.vyf = (float)C.vy; C.vzf = (float)C.vz;
      C.eps = 1e-6f * fmaxf(bx, fmaxf(by, bz));
      const float minef = (float)(C.ci + si);
      // the pruning bound curf >= the FP64 minimum: the local term, and upper
      // bounds of the pairs with the fastest cell of each coarse bucket
      C.curf = (float)cur * (1.0f + 1e-5f);
      const int leaf = d.levels - 1;
      const int ls = leaf < 2 ? leaf : 2;
      {
        const int n0 = level_start(ls, d.dim), n1 = level_start(ls + 1, d.dim);
        float t = INFINITY;
        for (int b = n0 + lane; b < n1; b += 32) {
          const int s = __float_as_int(d.node[b].y);
          if (s != C.self) {
            float lo, hi;
            pair_tau_bounds(d, s, C.xf, C.yf, C.zf, C.cf, C.vxf, C.vyf, C.vzf, C.eps, lo, hi);
            t = hi < t ? hi : t;
          }
        }
        C.curf = fminf(C.curf, __uint_as_float(__reduce_min_sync(full, __float_as_uint(t))));
      }
      const int lnch = d.dim;                    // log2 of the children per bucket
      const int nch = 1 << lnch;
      // the cell's own leaf bucket and its 3^dim - 1 neighbours first (lane q
      // takes neighbour q), so the walk below starts from a tight bound and
      // skips them
      const int lside = 1 << leaf;
      const int lx = min(lside - 1, max(0, (int)floorf(C.xf / bx * (float)lside)));
      const int ly = min(lside - 1, max(0, (int)floorf(C.yf / by * (float)lside)));
      const int lz = (d.dim == 3) ? min(lside - 1, max(0, (int)floorf(C.zf / bz * (float)lside))) : 0;
      {
        const int nnb = (d.dim == 3) ? 27 : 9;
        int s0 = 0, s1 = 0;
        if (lane < nnb) {
          const int qx = lane % 3 - 1, qy = (lane / 3) % 3 - 1, qz = (d.dim == 3) ? lane / 9 - 1 : 0;
          const int jx = (lx + qx + lside) & (lside - 1), jy = (ly + qy + lside) & (lside - 1),
                    jz = (lz + qz + lside) & (lside - 1);
          const int b = (d.dim == 3) ? (jx * lside + jy) * lside + jz : jx * lside + jy;
          s0 = d.leaf_off[b];
          s1 = d.leaf_off[b + 1];
        }
        walk_scan(d, S, C, lane, s0, s1);
      }
      // the walk from the root; leaves to scan are gathered until 32 are there
      // or the stack is empty
      int sp = 1, nleaf = 0;
      if (lane == 0) {
        S.node[0] = 0u;                          // level 0, bucket 0
        S.lb[0] = 0.0f;
      }
      __syncwarp();
      while (sp > 0 || nleaf > 0) {
        if (sp == 0 || nleaf > 32 - nch) {
          int s0 = 0, s1 = 0;
          if (lane < nleaf) {
            s0 = d.leaf_off[S.leaf[lane]];
            s1 = d.leaf_off[S.leaf[lane] + 1];
          }
          nleaf = 0;
          walk_scan(d, S, C, lane, s0, s1);
          continue;
        }
        // open up to 32 / nch buckets from the top (as many as leave room for
        // their leaves); lane q takes child q % nch of the q / nch-th
        const int take = min(sp, min(32, 32 - nleaf) >> lnch);
        sp -= take;
        const int par = lane >> lnch, ch = lane & (nch - 1);
        bool ok = false, isleaf = false;
        float lb = 0.0f;
        unsigned ce = 0u;
        int cb = 0;
        if (par < take && S.lb[sp + par] < C.curf) {
          const unsigned e = S.node[sp + par];
          const int l = (int)(e >> 27) + 1;      // the children's level
          const unsigned jx = 2u * ((e >> 18) & 511u) + (ch & 1), jy = 2u * ((e >> 9) & 511u) + ((ch >> 1) & 1),
                         jz = 2u * (e & 511u) + ((ch >> 2) & 1);
          const int cside = 1 << l;
          cb = (d.dim == 3) ? ((int)jx * cside + (int)jy) * cside + (int)jz : (int)jx * cside + (int)jy;
          const float fast = d.node[level_start(l, d.dim) + cb].x;
          isleaf = l == leaf;
          bool near = false;
          if (isleaf) {
            // a leaf of the neighbourhood scanned above (periodic distance <= 1)
            const int ax = abs((int)jx - lx), ay = abs((int)jy - ly), az = abs((int)jz - lz);
            near = min(ax, lside - ax) <= 1 && min(ay, lside - ay) <= 1 && min(az, lside - az) <= 1;
          }
          if (fast >= 0.0f && !near) {
            const float inv = __int_as_float((127 - l) << 23);   // 1 / cside
            const float hx = bx * inv, hy = by * inv, hz = bz * inv;
            const float gx = interval_gap(C.xf, (float)jx * hx, hx, bx);
            const float gy = interval_gap(C.yf, (float)jy * hy, hy, by);
            const float gz = (d.dim == 3) ? interval_gap(C.zf, (float)jz * hz, hz, bz) : 0.0f;
            const float gap = fmaxf(sqrtf(gx * gx + gy * gy + gz * gz) - C.eps, 0.0f);
            lb = gap / ((minef + fast) * (1.0f + 1e-5f));
            ok = lb < C.curf;
            ce = ((unsigned)l << 27) | (jx << 18) | (jy << 9) | jz;
          }
        }
        __syncwarp();                            // (the popped entries are read)
        const unsigned lm = __ballot_sync(full, ok && isleaf), nm = __ballot_sync(full, ok && !isleaf);
        const unsigned below = (1u << lane) - 1u;
        if (ok && isleaf) S.leaf[nleaf + __popc(lm & below)] = cb;
        if (ok && !isleaf) {
          S.node[sp + __popc(nm & below)] = ce;
          S.lb[sp + __popc(nm & below)] = lb;
        }
        nleaf += __popc(lm);
        sp += __popc(nm);
        __syncwarp();
      }
      walk_flush(d, S, C, lane);
      cur = C.cur;
    }
    if (lane == 0) {
      const double dti = d.cfl * cur;
      // the largest step dt_max 2^-b not above dt_i, from the exponents and
      // significands (dt_max 2^-b is exact): with dt_max = m1 2^e1 and
      // dt_i = m2 2^e2, b = e1 - e2, plus one if m1 > m2
      const double dtm = d.dtick * (double)(1ll << d.depth);
      int b = 0;
      if (dti < dtm) {
        const long long u1 = __double_as_longlong(dtm), u2 = __double_as_longlong(dti);
        const int e1 = (int)((u1 >> 52) & 0x7ff), e2 = (int)((u2 >> 52) & 0x7ff);
        const long long m1 = u1 & 0xfffffffffffffll, m2 = u2 & 0xfffffffffffffll;
        b = (e2 == 0) ? d.depth + 1 : e1 - e2 + (m1 > m2 ? 1 : 0);   // zero or subnormal: below every bin
      }
      if (b > d.depth) {
        atomicOr(&v.stats->status, (unsigned)ST_DEPTH);
        b = d.depth;
      }
      const int old = d.bin[i];
      int nb = b;
      if (tick != 0 && b < old)   // at most twice the step, where that step starts now
        nb = ((tick & (step_ticks(d.depth, old - 1) - 1)) == 0) ? old - 1 : old;
      if (nb != old) {
        atomicSub(d.hist + old, 1u);
        atomicAdd(d.hist + nb, 1u);
        d.bin[i] = (signed char)nb;
      }
    }
    __syncwarp();
  }
}

// ------------------------------------------------------------ active faces
template <typename real>
__global__ void k_ind_faces(HydroView<real> v, IndView d) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  const bool in = k < d.nf;
  int2 e = make_int2(0, 0);
  bool active = false;
  if (in) {
    e = v.lr[k];
    active = d.act[e.x] || d.act[e.y];
  }
  const int at = warp_append(d.count + 1, active);
  if (!active) return;
  const int stamp = d.loop->stamp;
  d.flist[at] = k;
  d.fstamp[k] = stamp;
  d.cstamp[e.x] = stamp;   // both writers store the same value
  d.cstamp[e.y] = stamp;
  const long long sL = step_ticks(d.depth, d.bin[e.x]), sR = step_ticks(d.depth, d.bin[e.y]);
  d.fdt[k] = (double)(sL < sR ? sL : sR) * d.dtick;
}

// ---------------------------------------------------- fluxes of active faces
// Gradients and bins of the active cells need nothing of one another: odd CTAs take
// the ones, even CTAs the others, so that the two chains of a tick with few cells
// overlap.  Few cells get 16 lanes each for their gradients, about an incidence a
// lane; many get 4.  (Two kernels, the gradients with 4 lanes in CTAs of 256: 25 + 92 us
// a tick for some 70 cells, 24 now, and 1.6 -> 0.52 ms for 32768 cells.)
template <typename real>
__global__ void __launch_bounds__(32 * BINS_WARPS, 4) k_ind_cells(HydroView<real> v, IndView d, int few) {
  const int cta = (int)blockIdx.x >> 1, ctas = (int)gridDim.x >> 1;
  if ((blockIdx.x & 1) == 0)
    ind_bins(v, d, cta, ctas);
  else if (d.count[0] <= few)
    ind_grad<real, 16>(v, d, cta, ctas);
  else
    ind_grad<real, 4>(v, d, cta, ctas);
}

// Runs for more than `above` active faces and at most `most`.  FP64 form: what
// bounds the few faces of most ticks is the chain of one warp's FP64 instructions,
// which cost the same however few lanes are on; so warps (B = 32) take few faces each,
// down to one, with a lane for each side of a face, and the pipes of all SMs are used (70 us a tick
// with CTAs of 128 for some 340 faces, 47 so, 22 with fixed64.cuh).  Many faces go to CTAs of 128, which group their solves.
template <typename real, int B>
__global__ void __launch_bounds__(B) k_ind_flux(HydroView<real> v, IndView d, int above, int most) {
  const int count = d.count[1];
  if (count <= above || count > most) return;
  const long long tick = d.loop->tick;
  int per = B;                                            // faces per CTA; a lane per side for B = 32
  if (B == 32) {
    per = 16;
    while (per > 1 && (per >> 1) * (int)gridDim.x >= count) per >>= 1;
  }
  const int t = (int)threadIdx.x & (per - 1);             // (the lanes beyond per repeat the first ones' faces)
  for (int blk = blockIdx.x; blk * per < count; blk += gridDim.x) {
    const int idx = blk * per + t;
    const bool valid = idx < count && t == (int)threadIdx.x;
    const int k = d.flist[idx < count ? idx : count - 1];
    const int2 e = v.lr[k];
    const long long sL = step_ticks(d.depth, d.bin[e.x]), sR = step_ticks(d.depth, d.bin[e.y]);
    const long long sf = sL < sR ? sL : sR;
    const long long t2 = 2 * tick + sf;                   // twice the middle of the face's step
    const double hL = (double)(t2 - 2 * (tick - (tick & (sL - 1)))) * (0.5 * d.dtick);
    const double hR = (double)(t2 - 2 * (tick - (tick & (sR - 1)))) * (0.5 * d.dtick);
    FaceWork<real> f;
    face_prepare<real, false>(v, k, valid, (real)hL, (real)hR, f);
    face_finish<real, B, false>(v, f, 0, min(per, count - blk * per), false, (real)0);
    if (B > 32) __syncthreads();
  }
}

// --------------------------------------------------- the pairwise exchange
// Four lanes per cell, each with every fourth incidence, its face's stamp, step
// and flux loaded whether or not the face is active (a thread per cell waited for
// each in turn: 31 us a tick, 13 now, 32768 cells with few touched).
template <typename real>
__global__ void __launch_bounds__(256) k_ind_update(HydroView<real> v, IndView d) {
  constexpr int G = 4;
  const int i = (int)((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) / G), lane = threadIdx.x % G;
  const int stamp = d.loop->stamp;
  const bool touched = i < d.n && d.cstamp[i] == stamp;
  if (!__any_sync(0xffffffffu, touched)) return;
  double s[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
  if (touched) {
    const int q1 = v.csr_off[i + 1];
#pragma unroll 4
    for (int q = v.csr_off[i] + lane; q < q1; q += G) {
      const int2 e = v.csr[q];
      const int k = e.x >> 1;
      const R4<real> f = v.flux[k];
      const real fE = v.fluxE[k];
      const double dt = d.fdt[k];
      if (d.fstamp[k] != stamp) continue;
      const double w = (e.x & 1) ? -dt : dt;
      s[0] += w * (double)f.x;
      s[1] += w * (double)f.y;
      s[2] += w * (double)f.z;
      s[3] += w * (double)f.w;
      s[4] += w * (double)fE;
    }
  }
#pragma unroll
  for (int a = 0; a < 5; a++) s[a] = group_sum<G>(s[a]);
  if (!touched) return;
  const size_t n = (size_t)d.n;
  // (lane a writes component a, lane 0 also the last)
  v.Q[lane * n + i] -= lane == 0 ? s[0] : (lane == 1 ? s[1] : (lane == 2 ? s[2] : s[3]));
  if (lane == 0) v.Q[4 * n + i] -= s[4];
}

// ----------------------------------------------------------- the next tick
// One warp: the deepest bin in use (from the histogram), the counters, the
// next tick (the next multiple of the shortest step), a fresh stamp and
// cleared list counters; the cycle's while condition stays set while ticks
// remain, no cell has failed and the sub-step cap is not reached.
static __global__ void k_ind_next(IndView d) {
  const int lane = (int)threadIdx.x;
  const unsigned h0 = lane <= d.depth ? d.hist[lane] : 0u;
  const unsigned h1 = lane + 32 <= d.depth ? d.hist[lane + 32] : 0u;
  const unsigned m0 = __ballot_sync(0xffffffffu, h0 != 0u), m1 = __ballot_sync(0xffffffffu, h1 != 0u);
  if (lane != 0) return;
  const int deepest = m1 ? 32 + 31 - __clz(m1) : (m0 ? 31 - __clz(m0) : 0);
  IndLoop* L = d.loop;
  L->substeps++;
  L->activations += (unsigned long long)d.count[0];
  L->face_fluxes += (unsigned long long)d.count[1];
  L->deepest = deepest > L->deepest ? deepest : L->deepest;
  const long long smin = 1ll << (d.depth - deepest);
  L->tick = (L->tick / smin + 1) * smin;
  L->stamp++;
  d.count[0] = 0;
  d.count[1] = 0;
  const DeviceStats* S = d.stats;
  const bool failed = (S->status & (ST_NEWTON_CAP | ST_NONPOS | ST_DEPTH)) != 0u;
  const bool capped = L->substeps >= L->max_substeps;
  if (capped && L->tick < L->T) atomicOr(&d.stats->status, (unsigned)ST_SUBSTEPS);
  L->go = (L->tick < L->T && !failed && !capped) ? 1 : 0;
  if (d.in_graph) cudaGraphSetConditional(d.handle, (unsigned)L->go);
}

// ---------------------------------------------------------------- launchers
template <typename real>
cudaError_t launch_individual_tick(amm_ctx* c, const IndView& d) {
  HydroView<real> v = make_view<real>(c, 0.0);
  v.fixed_acc = 0;                 // per-face steps: the FP64 gather below
  const int grid_c = nblk(c->n, 256);
  k_ind_activate<real><<<grid_c, 256, 0, c->stream>>>(v, d);
  if (d.signal) {
    const int parents = 1 << (d.dim * (d.levels - 2));
    k_ind_leaf<<<nblk((int64_t)parents * 32, 256), 256, 0, c->stream>>>(d);
    k_ind_up<<<1, 1024, 0, c->stream>>>(d);
  }
  // list kernels: a fixed grid strides over the list, whose length only the
  // device knows
  constexpr int sms = 152;
  const int g_cells = nblk(c->n, BINS_WARPS), g_flux = nblk(c->nf, 128);
  k_ind_cells<real><<<2 * (g_cells < sms * 8 ? g_cells : sms * 8), 32 * BINS_WARPS, 0, c->stream>>>(v, d, sms * 4);
  k_ind_faces<real><<<nblk(c->nf, 256), 256, 0, c->stream>>>(v, d);
  constexpr int few = sizeof(real) == 8 ? sms * 32 * 2 : 0;
  if constexpr (few > 0) k_ind_flux<real, 32><<<sms * 4, 32, 0, c->stream>>>(v, d, 0, few);
  k_ind_flux<real, 128><<<g_flux < sms * 8 ? g_flux : sms * 8, 128, 0, c->stream>>>(v, d, few, 0x7fffffff);
  k_ind_update<real><<<nblk(c->n * 4, 256), 256, 0, c->stream>>>(v, d);
  return cudaGetLastError();
}

#define AMM_INSTANTIATE_INDIVIDUAL(real) \
  template cudaError_t launch_individual_tick<real>(amm_ctx*, const IndView&);

}  // namespace amm
