// Reverse mode of one kick-drift-kick step and of the grid-density loss.
//
// The paper has no adjoint; these kernels differentiate the forward path of
// this library (Sec. II-A time integration with the density loop, the
// smoothing-length solve and the force loop of Sec. III) with respect to the
// state before the step, for a loss on a later state.  The discrete parts
// (active set, time bins, integer times, which pairs are neighbours) are
// piecewise constant and are taken from the forward run.
//
// One step backwards (sph_step_bwd): the caller hands in the state before
// and after the step (in the caller's particle order) and the adjoint of the
// state after it; the adjoint is replaced by the adjoint of the state before.
//   1. prepare (caller order): positions at the step's tick, predicted v and
//      A, P and c inputs, h / rho / f as the force loop saw them; the adjoint
//      of both half-kicks of the active particles;
//   2. a cell build of these internal copies (its own sort) and the active
//      work groups;
//   3. force adjoint: for every active i and neighbour j, the derivative of
//      a_i and Adot_i with respect to positions, predicted velocities, H,
//      f P / rho^2, c and rho of both particles (j's share by FP64 atomics);
//   4. equation-of-state adjoint: f P / rho^2 and c back to f, P, rho, then
//      P = A_pred rho^gamma back to A_pred and rho (on the first step
//      A = (gamma - 1) u / rho^(gamma - 1) back to u and rho);
//   5. density adjoint in two passes over the same pairs: the sums that fix
//      the derivatives of rho, f and of the smoothing-length equation
//      F(h, x) = h^3 n(h) - eta^3 (implicit h: dh/dx = -F_x / F_h), then the
//      position derivatives of every pair;
//   6. scatter back to caller order with the prediction (v_pred = v + a dtp,
//      A_pred = A + Adot dtp) and drift (x += v dt) adjoints.
// Pair arithmetic is FP32 as in the forward loops; every adjoint accumulator
// is FP64.
#include <algorithm>
#include <cstddef>
#include <cstring>

#include "sph_pairloop.cuh"

namespace sph {
namespace {

constexpr double KN_D = 2.5464790894703255;  // 8 / pi

__device__ __forceinline__ double wrap_box(double x, double box) {
  if (x < 0.0) x += box;
  if (x >= box) x -= box;
  return x;
}

__device__ __forceinline__ double min_img(double d, double box) {
  if (d > 0.5 * box) d -= box;
  else if (d < -0.5 * box) d += box;
  return d;
}

// ---------------------------------------------------------------------------
// 1. prepare, in caller order
// ---------------------------------------------------------------------------
__global__ void k_adj_prepare(sph_particles pre, sph_particles post, sph_particles W,
                              sph_adjoint adj, long long ti, int first, double dt_min, double box,
                              double gamma) {
  const long long n = pre.n;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x) {
    // (here and in the gather and the scatter every load stands before the first
    // store: the compiler keeps a load behind a store that might write what it
    // reads.  32,768 particles: 7.5 -> 5.1 us, the scatter 9.4 -> 5.4.)
    const long long te = pre.ti_end[i], tb = pre.ti_begin[i];
    const bool act = te == ti;
    const sph_particles &now = act ? post : pre;
    const float h = now.h[i], rho = now.rho[i], f = now.f[i];
    const float Adot_now = act ? post.Adot[i] : 0.0f;
    const long long ptb = act ? post.ti_begin[i] : 0, pte = act ? post.ti_end[i] : 0;
    const double avx = act ? adj.vx[i] : 0.0, avy = act ? adj.vy[i] : 0.0,
                 avz = act ? adj.vz[i] : 0.0, aA = act ? adj.A[i] : 0.0;
    const double aax = act ? adj.ax[i] : 0.0, aay = act ? adj.ay[i] : 0.0,
                 aaz = act ? adj.az[i] : 0.0, aAdot = act ? adj.Adot[i] : 0.0;
    const float vx = pre.vx[i], vy = pre.vy[i], vz = pre.vz[i];
    const float ax = pre.ax[i], ay = pre.ay[i], az = pre.az[i];
    const float A = pre.A[i], Adot = pre.Adot[i], m = pre.m[i];
    const int bi = pre.bin[i] & (MAX_BINS - 1);
    // positions at the step's tick (the forward drift, applied to every particle)
    const double dtd = (double)(ti - pre.ti_drift[i]) * dt_min;
    double x = pre.x[i], y = pre.y[i], z = pre.z[i];
    if (dtd != 0.0) {
      x = wrap_box(x + (double)vx * dtd, box);
      y = wrap_box(y + (double)vy * dtd, box);
      z = wrap_box(z + (double)vz * dtd, box);
    }
    W.x[i] = x;
    W.y[i] = y;
    W.z[i] = z;
    // prediction at the tick
    const double dtp = ((double)(ti - tb) - 0.5 * (double)(1ll << bi)) * dt_min;
    const float fdtp = (float)dtp;
    W.vx[i] = vx + ax * fdtp;
    W.vy[i] = vy + ay * fdtp;
    W.vz[i] = vz + az * fdtp;
    float Ap;
    if (first) Ap = (float)(gamma - 1.0) * A / powf(rho, (float)gamma - 1.0f);  // A holds u
    else Ap = (float)((double)A + (double)Adot * dtp);
    W.A[i] = Ap;
    W.h[i] = h;
    W.rho[i] = rho;
    W.f[i] = f;
    W.m[i] = m;
    // the cell build's refresh predicts with a and Adot: zero, so the records
    // carry exactly v_pred and A_pred; vsig carries the forward Adot of the
    // active particles (the force adjoint needs it)
    W.ax[i] = 0.0f;
    W.ay[i] = 0.0f;
    W.az[i] = 0.0f;
    W.Adot[i] = 0.0f;
    W.vsig[i] = Adot_now;
    W.P[i] = 0.0f;
    W.c[i] = 0.0f;
    W.bin[i] = act ? 0 : 1;  // the backward marks bin 0 active
    W.ti_begin[i] = ti;
    W.ti_end[i] = ti + 1;
    W.ti_drift[i] = ti;
    W.active[i] = 0;
    // adjoint of the two half-kicks of an active particle:
    // v += a dt_old / 2 and v += a dt_new / 2 (likewise A with Adot)
    if (act) {
      const double half = 0.5 * (double)(te - tb) * dt_min + 0.5 * (double)(pte - ptb) * dt_min;
      adj.ax[i] = aax + avx * half;
      adj.ay[i] = aay + avy * half;
      adj.az[i] = aaz + avz * half;
      adj.Adot[i] = aAdot + aA * half;
    }
  }
}

// ---------------------------------------------------------------------------
// 2b. gather the adjoint state into the backward build's order
// ---------------------------------------------------------------------------
__global__ void k_adj_gather(View v, AdjWork w, sph_adjoint adj, double gamma) {
  const long long n = v.n;
  for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < n;
       k += (long long)gridDim.x * blockDim.x) {
    const int o = w.perm[k];
    const bool act = v.bin[k] == 0;
    const double xb = adj.x[o], yb = adj.y[o], zb = adj.z[o], hb = adj.h[o], rb = adj.rho[o],
                 fb = adj.f[o];
    const double axb = act ? adj.ax[o] : 0.0, ayb = act ? adj.ay[o] : 0.0,
                 azb = act ? adj.az[o] : 0.0, Adb = act ? adj.Adot[o] : 0.0;
    const float sum = act ? v.vsig[k] : 0.0f, rho = act ? v.rho[k] : 1.0f;
    w.xb[k] = xb;
    w.yb[k] = yb;
    w.zb[k] = zb;
    w.hb[k] = hb;
    w.fb[k] = fb;
    w.vpxb[k] = 0.0;
    w.vpyb[k] = 0.0;
    w.vpzb[k] = 0.0;
    w.Qb[k] = 0.0;
    w.cb[k] = 0.0;
    if (act) {
      // this step computed a and Adot of the active particles: their adjoints
      // are consumed here (what remains for the old values comes from the
      // prediction, added in the scatter)
      w.axb[k] = axb;
      w.ayb[k] = ayb;
      w.azb[k] = azb;
      w.Adotb[k] = Adb;
      adj.ax[o] = 0.0;
      adj.ay[o] = 0.0;
      adj.az[o] = 0.0;
      adj.Adot[o] = 0.0;
      // Adot = (gamma - 1)/2 rho^(1 - gamma) sum(...): its rho-dependence
      w.rhob[k] = rb + Adb * (double)sum * (1.0 - gamma) / (double)rho;
    } else {
      w.rhob[k] = rb;
      w.axb[k] = w.ayb[k] = w.azb[k] = w.Adotb[k] = 0.0;
    }
  }
}

// ---------------------------------------------------------------------------
// 3. force adjoint: one warp per active work group, one lane per particle;
//    with COOP the 8 warps of a block share a group (each takes the neighbour
//    chunks with its index modulo 8) and combine the particle's own sums in
//    warp order through the start of their staging buffers
// ---------------------------------------------------------------------------
// The adjoint loops run the forward loops' scheme: a batch's accept masks
// first, the records across the lanes, then each lane its own pairs; the FP32
// values become FP64 by integer instructions (widen).  One step's gradient of
// 32,768 particles has about as many groups as the chip has warps, so what
// counts is the longest warp's chain of pairs and their 10 (density: 3) FP64
// atomics each: 128 records' masks by every lane on its own and conversions at
// the FP64 rate took 1304 us, now 998 (density passes 325 -> 194 and 507 ->
// 359).  Two blocks an SM (128 registers) give 1183: their spread of the work
// is no better and the loop body stalls on its spilled operands.
constexpr int S_ADJ = 160, S_ADJ_DENS = 256;  // staged records of three arrays, of one
using StageA = Stage<S_ADJ, 3, 208, true, true>;
using StageB = Stage<S_ADJ_DENS, 1, 320, true, true>;

template <class St = StageA>
__device__ __forceinline__ double *adj_red_area(int warp) {
  extern __shared__ __align__(16) char smem_dyn[];
  static_assert(S_ADJ * 3 * 16 >= 11 * 32 * 8 && S_ADJ_DENS * 16 >= 5 * 32 * 8,
                "the reduction areas fit the start of a staging buffer");
  return reinterpret_cast<double *>(smem_dyn + (size_t)warp * St::bytes());
}

// The COOP reduction: the 8 warps' per-lane partial sums part[0..N) added in
// warp order, the result in every warp; a failure in any warp becomes every
// warp's (so that all take the same branches).
template <class St, int N>
__device__ __forceinline__ void coop_reduce(double (&part)[N], bool &failed) {
  const int lane = lane_id(), warp = threadIdx.x >> 5;
  double *mine = adj_red_area<St>(warp);
#pragma unroll
  for (int k = 0; k < N; k++) mine[k * 32 + lane] = part[k];
  mine[N * 32 + lane] = failed ? 1.0 : 0.0;
  __syncthreads();
  bool any = false;
#pragma unroll
  for (int k = 0; k < N; k++) part[k] = 0.0;
  for (int q = 0; q < WARPS_PER_BLOCK; q++) {
    const double *rw = adj_red_area<St>(q);
#pragma unroll
    for (int k = 0; k < N; k++) part[k] += rw[k * 32 + lane];
    any = any || rw[N * 32 + lane] != 0.0;
  }
  __syncthreads();
  fence_proxy_async();  // the staging buffers take bulk copies again
  failed = __any_sync(FULL, any);
}

template <bool COOP>
__device__ void force_adj_group(const View &v, const AdjWork &w, int wg, const CellFrame &F,
                                StageA &st, WarpCounters &wc) {
  const int lane = lane_id();
  const int warp = threadIdx.x >> 5;
  const Group Wg = group_of(v, wg, F);
  const int a = Wg.a, b = Wg.b;
  const int nact = leaf_actives(v, a, b, 0, -1, st.act);
  if (nact == 0) return;
  const float qox = F.kx * F.wq, qoy = F.ky * F.wq, qoz = F.kz * F.wq;
  const float clx = Wg.lx + qox, cly = Wg.ly + qoy, clz = Wg.lz + qoz;
  const float chx = Wg.hx + qox, chy = Wg.hy + qoy, chz = Wg.hz + qoz;
  const float ceps = 1e-5f * F.wf;
  const float alpha = (float)v.alpha;
  const float4 *srcs[3] = {v.rec_xH, v.rec_v, v.rec_h};
  const float4 *sx_rec = st.rec, *sv_rec = st.rec + S_ADJ, *sh_rec = st.rec + 2 * S_ADJ;
  // one round: a work group holds at most 32 particles
  const bool valid = lane < nact;
  const int i = valid ? st.act[lane] : a;
  const float4 xl = v.rec_xH[i];
  const float3 lo3 = leaf_offset(v, i, F);
  const float4 xi = make_float4(xl.x + lo3.x, xl.y + lo3.y, xl.z + lo3.z, xl.w);
  const float4 vi = v.rec_v[i];
  const float4 hi4 = v.rec_h[i];  // rho, Q = f P / rho^2, c, 1 / H
  const float Hi2 = xi.w * xi.w;
  const float Hinv2 = hi4.w * hi4.w;
  const float nHi4 = KERNEL_NORM * Hinv2 * Hinv2;
  const float Hs = warp_max(valid ? xi.w : 0.0f);
  // adjoints of the outputs a_i and Adot_i
  const float abx = valid ? (float)w.axb[i] : 0.0f, aby = valid ? (float)w.ayb[i] : 0.0f,
              abz = valid ? (float)w.azb[i] : 0.0f;
  const float Bi = valid ? (float)(0.5 * (v.gamma - 1.0) * pow((double)hi4.x, 1.0 - v.gamma) *
                                   w.Adotb[i])
                         : 0.0f;
  const bool live = valid && (abx != 0.0f || aby != 0.0f || abz != 0.0f || Bi != 0.0f);
  const int nsph = compact_spheres(st.sph, live, make_float4(xi.x, xi.y, xi.z, xi.w));
  const TestSet ts = test_set(st.tst, live, xi.x, xi.y, xi.z, Hi2);
  // the particle's own adjoint sums: FP32 partial sums per neighbour cell,
  // folded into FP64 where the cell changes (FP64 arithmetic is scarce)
  double dxi = 0.0, dyi = 0.0, dzi = 0.0, dvxi = 0.0, dvyi = 0.0, dvzi = 0.0;
  double Hbi = 0.0, Qbi = 0.0, cbi = 0.0, rbi = 0.0;
  float pdx = 0.f, pdy = 0.f, pdz = 0.f, pvx = 0.f, pvy = 0.f, pvz = 0.f;
  float pH = 0.f, pQ = 0.f, pc = 0.f, pr = 0.f;
  int cur = -1;
  auto fold_cell = [&]() {
    dxi += widen(pdx); dyi += widen(pdy); dzi += widen(pdz);
    dvxi += widen(pvx); dvyi += widen(pvy); dvzi += widen(pvz);
    Hbi += widen(pH); Qbi += widen(pQ); cbi += widen(pc); rbi += widen(pr);
    pdx = pdy = pdz = pvx = pvy = pvz = pH = pQ = pc = pr = 0.f;
  };
  auto leaf_ok = [&](int l, float sx, float sy, float sz, LeafBox &lb) {
    const float4 loj = v.leaf_lo[l], hij = v.leaf_hi[l];
    const float R = fmaxf(Hs, loj.w);
    lb = leaf_box(loj, hij, sx, sy, sz, loj.w);
    return box_gap2(Wg.lx, Wg.ly, Wg.lz, Wg.hx, Wg.hy, Wg.hz, loj, hij, sx, sy, sz) <
           R * R * 1.0002f;
  };
  auto chunk_ok = [&](int gg, float sx, float sy, float sz) {
    const float4 loc = v.chunk_lo[gg];
    const float R = fmaxf(Hs, loc.w) + ceps;
    return box_gap2(clx, cly, clz, chx, chy, chz, loc, v.chunk_hi[gg], sx, sy, sz) < R * R;
  };
  auto consume = [&](int base, int total) {
    // accept masks of the whole batch (as the forward force loop)
    const int wend = (total + 31) >> 5;
#pragma unroll 1
    for (int q = 0; q < wend; q++)
      test_masks<true>(st.tst, ts.n, sx_rec[min(base + 32 * q + lane, S_ADJ - 1)],
                       32 * q + lane < total, st.mask + 32 * q);
    __syncwarp();
    int left = 0, k0 = base - 1, word = 0;
    if (live)
      for (int q = 0; q < wend; q++) left += __popc(st.mask[32 * q + ts.rank]);
    unsigned mask = st.mask[ts.rank];
    for (; left > 0; left--) {
      while (mask == 0u) {
        word++;
        k0 += 32;
        mask = st.mask[32 * word + ts.rank];
      }
      const int k = k0 + __ffs(mask);
      mask &= mask - 1;
      const int j = st.recj[k];
      if (j == i) continue;
      const int ci = st.recc[k];
      if (ci != cur) {
        fold_cell();
        cur = ci;
      }
      const float4 pj = sx_rec[k];
      const float4 vj = sv_rec[k];
      const float4 hj = sh_rec[k];
      const float dx = xi.x - pj.x, dy = xi.y - pj.y, dz = xi.z - pj.z;
      const float r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
      if (!(r2 > 0.0f)) continue;  // coincident: no direction, no gradient
      const float rinv = rsqrtf(r2);
      const float r = r2 * rinv;
      const float qi = r * hi4.w, qj = r * hj.w;
      const float hj2 = hj.w * hj.w;
      const float nHj4 = KERNEL_NORM * hj2 * hj2;
      const float wpi = qi < 1.0f ? kernel_dw(qi) : 0.0f;
      const float wpj = qj < 1.0f ? kernel_dw(qj) : 0.0f;
      const float wppi = qi < 1.0f ? kernel_d2w(qi) : 0.0f;
      const float wppj = qj < 1.0f ? kernel_d2w(qj) : 0.0f;
      const float dWi = wpi * nHi4, dWj = wpj * nHj4;
      const float dvx = vi.x - vj.x, dvy = vi.y - vj.y, dvz = vi.z - vj.z;
      const float dvdr = fmaf(dvx, dx, fmaf(dvy, dy, dvz * dz));
      const float uu = dvdr * rinv;
      const float wij = fminf(0.0f, uu);
      const float vsij = hi4.z + hj.z - 3.0f * wij;
      const float rs = hi4.x + hj.x;
      const float Pi = -alpha * vsij * wij / rs;
      const float Wb = 0.5f * (dWi + dWj);
      const float K = fmaf(hi4.y, dWi, fmaf(hj.y, dWj, Pi * Wb));
      const float mj = vj.w;
      const float gdot = fmaf(abx, dx, fmaf(aby, dy, abz * dz));
      // the pair's share of the loss: -m_j K / r (abar . d) + B m_j Pi Wb u
      const float Kb = -mj * rinv * gdot;
      const float Pib = fmaf(Kb, Wb, Bi * mj * Wb * uu);
      const float Wbb = fmaf(Kb, Pi, Bi * mj * Pi * uu);
      float ub = Bi * mj * Pi * Wb;
      const float dWib = fmaf(Kb, hi4.y, 0.5f * Wbb);
      const float dWjb = fmaf(Kb, hj.y, 0.5f * Wbb);
      const float cpart = Pib * (-alpha * wij / rs);
      const float rpart = Pib * (-Pi / rs);
      if (uu < 0.0f) ub = fmaf(Pib, -alpha * (vsij - 3.0f * wij) / rs, ub);
      const float rinvb = fmaf(-mj * K, gdot, ub * dvdr);
      // dW/dr and dW/dH of each smoothing length (q w'' + 4 w' over H^5)
      const float rb = fmaf(dWib, wppi * nHi4 * hi4.w,
                            fmaf(dWjb, wppj * nHj4 * hj.w, -rinvb * rinv * rinv));
      const float Hib = -dWib * fmaf(qi, wppi, 4.0f * wpi) * nHi4 * hi4.w;
      const float Hjb = -dWjb * fmaf(qj, wppj, 4.0f * wpj) * nHj4 * hj.w;
      const float gK = -mj * K * rinv;
      const float ex = dx * rinv, ey = dy * rinv, ez = dz * rinv;
      const float bx = fmaf(gK, abx, fmaf(ub * rinv, dvx, rb * ex));
      const float by = fmaf(gK, aby, fmaf(ub * rinv, dvy, rb * ey));
      const float bz = fmaf(gK, abz, fmaf(ub * rinv, dvz, rb * ez));
      const float vbx = ub * ex, vby = ub * ey, vbz = ub * ez;
      pdx += bx; pdy += by; pdz += bz;
      pvx += vbx; pvy += vby; pvz += vbz;
      pH += Hib;
      pQ += Kb * dWi;
      pc += cpart;
      pr += rpart;
      atomicAdd(&w.xb[j], -widen(bx));
      atomicAdd(&w.yb[j], -widen(by));
      atomicAdd(&w.zb[j], -widen(bz));
      atomicAdd(&w.vpxb[j], -widen(vbx));
      atomicAdd(&w.vpyb[j], -widen(vby));
      atomicAdd(&w.vpzb[j], -widen(vbz));
      atomicAdd(&w.hb[j], (double)GAMMA_K * widen(Hjb));
      atomicAdd(&w.Qb[j], widen(Kb * dWj));
      atomicAdd(&w.cb[j], widen(cpart));
      atomicAdd(&w.rhob[j], widen(rpart));
    }
  };
  const Reach reach = {clx, cly, clz, chx, chy, chz,
                       fmaxf(Hs, __uint_as_float(v.ds->Hmax_bits)) + ceps,
                       __uint_as_float(v.ds->excursion_bits), st.sph, nsph};
  int skip = 0, nlist = 0;
  bool more = false;
  do {
    if (more) compact_spheres(st.sph, live, make_float4(xi.x, xi.y, xi.z, xi.w));  // (the staging took their room)
    nlist = search(v, F, reach, st, leaf_ok, chunk_ok, skip, more, COOP ? warp : -1);
    stage_list(srcs, st, nlist, consume, wc);
    skip += nlist;
  } while (more && !st.failed);
  fold_cell();
  if constexpr (COOP) {
    double sum[10] = {dxi, dyi, dzi, dvxi, dvyi, dvzi, Hbi, Qbi, cbi, rbi};
    bool failed = st.failed;
    coop_reduce<StageA, 10>(sum, failed);
    st.failed = failed;  // the same in every warp
    dxi = sum[0]; dyi = sum[1]; dzi = sum[2];
    dvxi = sum[3]; dvyi = sum[4]; dvzi = sum[5];
    Hbi = sum[6]; Qbi = sum[7]; cbi = sum[8]; rbi = sum[9];
  }
  if (live && (!COOP || warp == 0)) {
    atomicAdd(&w.xb[i], dxi);
    atomicAdd(&w.yb[i], dyi);
    atomicAdd(&w.zb[i], dzi);
    atomicAdd(&w.vpxb[i], dvxi);
    atomicAdd(&w.vpyb[i], dvyi);
    atomicAdd(&w.vpzb[i], dvzi);
    atomicAdd(&w.hb[i], (double)GAMMA_K * Hbi);
    atomicAdd(&w.Qb[i], Qbi);
    atomicAdd(&w.cb[i], cbi);
    atomicAdd(&w.rhob[i], rbi);
  }
  __syncwarp();
}

// A step with at most two groups per block gives each group a whole block
// (its time is otherwise the latency of single warps on the largest groups).
__global__ void __launch_bounds__(PT, 1) k_adj_force(View v, AdjWork w) {
  DevState *ds = v.ds;
  __shared__ int s_go, s_nq, s_item;
  if (threadIdx.x == 0) {
    s_go = ds->halt ? 0 : 1;
    s_nq = ds->n_active_groups + ds->n_heavy_groups;
  }
  __syncthreads();
  if (!s_go) return;  // the whole block
  StageA st;
  stage_init(st);
  const int lane = lane_id();
  const int nq = s_nq;
  WarpCounters wc = {0, 0, 0, 0, 0, 0};
  if (nq <= 2 * (int)gridDim.x) {
    for (;;) {
      if (threadIdx.x == 0) s_item = atomicAdd(&ds->head_force, 1);
      __syncthreads();
      const int item = s_item;
      __syncthreads();
      if (item >= nq || st.failed) break;  // (st.failed is the same in every warp)
      const int wg = active_group(v, ds, item);
      if (!SPH_IN(ds, wg, ds->n_groups, SPH_CHECK_GROUP)) break;
      force_adj_group<true>(v, w, wg, frame_of(v, ds, wg), st, wc);
    }
  } else {
    for (;;) {
      int item = 0;
      if (lane == 0) item = atomicAdd(&ds->head_force, 1);
      item = __shfl_sync(FULL, item, 0);
      if (item >= nq || st.failed) break;
      const int wg = active_group(v, ds, item);
      if (!SPH_IN(ds, wg, ds->n_groups, SPH_CHECK_GROUP)) break;
      force_adj_group<false>(v, w, wg, frame_of(v, ds, wg), st, wc);
    }
  }
  if (lane == 0 && wc.timeout) record_error(ds, SPH_ERR_TIMEOUT, wc.timeout, true);
}

// ---------------------------------------------------------------------------
// 4. equation-of-state adjoint (backward-build order)
// ---------------------------------------------------------------------------
// Q = f P / rho^2, c = sqrt(gamma P / rho), P = A_pred rho^gamma.  Leaves
// d loss / d A_pred in Qb and, on the first step (A_pred = (gamma - 1) u /
// rho^(gamma - 1)), d loss / d u in cb.
__global__ void k_adj_eos(View v, AdjWork w, sph_adjoint adj, int first) {
  const long long n = v.n;
  const double g = v.gamma;
  for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < n;
       k += (long long)gridDim.x * blockDim.x) {
    const double rho = v.rho[k];
    if (!(rho > 0.0)) {
      w.Qb[k] = 0.0;
      w.cb[k] = 0.0;
      continue;
    }
    const double Qb = w.Qb[k], cbar = w.cb[k];
    // nothing came back to this particle's pressure and sound speed: every term
    // below is a zero (in a sparse step nearly everywhere; the power and the
    // divisions run at the FP64 rate: 32,768 particles, 18.7 -> 4 us in such a step)
    if (!first && Qb == 0.0 && cbar == 0.0 && (v.f[k] + v.P[k] + v.c[k]) * 0.0f == 0.0f) {
      w.cb[k] = 0.0;
      w.Qb[k] = 0.0;
      continue;
    }
    const double f = v.f[k], P = v.P[k], c = v.c[k], Ap = v.A[k];
    double rb = w.rhob[k];
    w.fb[k] += Qb * P / (rho * rho);
    double Pb = Qb * f / (rho * rho);
    rb += -2.0 * Qb * (f * P / (rho * rho)) / rho;
    if (P > 0.0) Pb += cbar * c / (2.0 * P);
    rb += -cbar * c / (2.0 * rho);
    const double Apb = Pb * pow(rho, g);
    rb += Pb * g * P / rho;
    if (first) {
      // the entropy of the first step: A = (gamma - 1) u / rho^(gamma - 1);
      // the state's A adjoint (after the kicks) and A_pred's both land on it
      const double Ab = adj.A[w.perm[k]] + Apb;
      w.cb[k] = Ab * (g - 1.0) / pow(rho, g - 1.0);  // d loss / d u
      rb += Ab * Ap * (1.0 - g) / rho;
    } else {
      w.cb[k] = 0.0;
    }
    w.Qb[k] = Apb;
    w.rhob[k] = rb;
  }
}

// ---------------------------------------------------------------------------
// 5. density adjoint (two passes over the pairs r < H_i of the active i)
// ---------------------------------------------------------------------------
// Pass 1 sums, per active i (q = r / H, w and derivatives over 8/pi, self
// included where it contributes):
//   sr = sum m w,  srt = sum m (3 w + q w'),  s1 = sum q w',
//   s2 = sum m q (4 w' + q w'')
// rho = (8/pi) sr / H^3, f = 3 sr / (3 sr - srt), F = (8/pi)/GAMMA_K^3 sum w - eta^3.
// With h_bar the adjoint of h as an output, the total h adjoint is
//   hbt = h_bar + rho_bar d rho/dh + f_bar d f/dh   (explicit h-dependence)
// and the implicit solve turns it into lambda = -hbt / F_h, F_h = -(8/pi)/GAMMA_K^3 s1 / h.
// Pass 2: every pair's r-derivative r_bar = (ka m_j w' + kb m_j (4 w' + q w'') + km w') / H.
template <int PASS, bool COOP>
__device__ void density_adj_group(const View &v, const AdjWork &w, int wg, const CellFrame &F,
                                  StageB &st, WarpCounters &wc) {
  const int lane = lane_id();
  const int warp = threadIdx.x >> 5;
  const Group Wg = group_of(v, wg, F);
  const int a = Wg.a, b = Wg.b;
  const int nact = leaf_actives(v, a, b, 0, -1, st.act);
  if (nact == 0) return;
  const float qox = F.kx * F.wq, qoy = F.ky * F.wq, qoz = F.kz * F.wq;
  const float clx = Wg.lx + qox, cly = Wg.ly + qoy, clz = Wg.lz + qoz;
  const float chx = Wg.hx + qox, chy = Wg.hy + qoy, chz = Wg.hz + qoz;
  const float ceps = 1e-5f * F.wf;
  const float4 *srcs[1] = {v.rec_xm};
  const bool valid = lane < nact;
  const int i = valid ? st.act[lane] : a;
  const float4 xl = v.rec_xm[i];
  const float3 lo3 = leaf_offset(v, i, F);
  const float4 xi = make_float4(xl.x + lo3.x, xl.y + lo3.y, xl.z + lo3.z, xl.w);
  const float H = GAMMA_K * v.h[i];
  const float Hinv = 1.0f / H;
  const float H2 = H * H;
  float ka = 0.0f, kb = 0.0f, km = 0.0f;
  bool live;
  if (PASS == 1) {
    live = valid && (w.hb[i] != 0.0 || w.rhob[i] != 0.0 || w.fb[i] != 0.0);
  } else {
    if (valid) {
      ka = (float)w.ka[i];
      kb = (float)w.kb[i];
      km = (float)w.km[i];
    }
    live = valid && (ka != 0.0f || kb != 0.0f || km != 0.0f);
  }
  const float Hs = warp_max(live ? H : 0.0f);
  const int nsph = compact_spheres(st.sph, live, make_float4(xi.x, xi.y, xi.z, H));
  const TestSet ts = test_set(st.tst, live, xi.x, xi.y, xi.z, H2);
  // FP32 partial sums per neighbour cell, folded into FP64 where the cell changes
  double sr = 0.0, srt = 0.0, s1 = 0.0, s2 = 0.0;
  double dxi = 0.0, dyi = 0.0, dzi = 0.0;
  float p0 = 0.f, p1 = 0.f, p2 = 0.f, p3 = 0.f;
  int cur = -1;
  auto fold_cell = [&]() {
    if (PASS == 1) {
      sr += widen(p0); srt += widen(p1); s1 += widen(p2); s2 += widen(p3);
    } else {
      dxi += widen(p0); dyi += widen(p1); dzi += widen(p2);
    }
    p0 = p1 = p2 = p3 = 0.f;
  };
  const float R2 = Hs * Hs * 1.0002f, Rc = Hs + ceps;
  auto leaf_ok = [&](int l, float sx, float sy, float sz, LeafBox &lb) {
    const float4 lo = v.leaf_lo[l], hi = v.leaf_hi[l];
    lb = leaf_box(lo, hi, sx, sy, sz, 0.0f);
    return box_gap2(Wg.lx, Wg.ly, Wg.lz, Wg.hx, Wg.hy, Wg.hz, lo, hi, sx, sy, sz) < R2;
  };
  auto chunk_ok = [&](int gg, float sx, float sy, float sz) {
    return box_gap2(clx, cly, clz, chx, chy, chz, v.chunk_lo[gg], v.chunk_hi[gg], sx, sy, sz) <
           Rc * Rc;
  };
  auto consume = [&](int base, int total) {
    // accept masks of the whole batch (as the forward force loop)
    const int wend = (total + 31) >> 5;
#pragma unroll 1
    for (int q = 0; q < wend; q++)
      test_masks<false>(st.tst, ts.n, st.rec[min(base + 32 * q + lane, S_ADJ_DENS - 1)],
                       32 * q + lane < total, st.mask + 32 * q);
    __syncwarp();
    int left = 0, k0 = base - 1, word = 0;
    if (live)
      for (int q = 0; q < wend; q++) left += __popc(st.mask[32 * q + ts.rank]);
    unsigned mask = st.mask[ts.rank];
    for (; left > 0; left--) {
      while (mask == 0u) {
        word++;
        k0 += 32;
        mask = st.mask[32 * word + ts.rank];
      }
      const int k = k0 + __ffs(mask);
      mask &= mask - 1;
      const int j = st.recj[k];
      const int ci = st.recc[k];
      if (ci != cur) {
        fold_cell();
        cur = ci;
      }
      const float4 pj = st.rec[k];
      const float dx = xi.x - pj.x, dy = xi.y - pj.y, dz = xi.z - pj.z;
      const float r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
      const float rr = r2 * rsqrtf(fmaxf(r2, 1e-30f));
      const float q = rr * Hinv;
      float wq, dwq;
      kernel_wd(q, wq, dwq);
      const float d2 = kernel_d2w(q);
      if (PASS == 1) {
        p0 += pj.w * wq;
        p1 += pj.w * fmaf(q, dwq, 3.0f * wq);
        p2 += q * dwq;
        p3 += pj.w * q * fmaf(q, d2, 4.0f * dwq);
      } else {
        if (j == i || !(r2 > 0.0f)) continue;
        const float rbar = (ka * pj.w * dwq + kb * pj.w * fmaf(q, d2, 4.0f * dwq) + km * dwq) * Hinv;
        const float rinv = rsqrtf(r2);
        const float bx = rbar * dx * rinv, by = rbar * dy * rinv, bz = rbar * dz * rinv;
        p0 += bx; p1 += by; p2 += bz;
        atomicAdd(&w.xb[j], -widen(bx));
        atomicAdd(&w.yb[j], -widen(by));
        atomicAdd(&w.zb[j], -widen(bz));
      }
    }
  };
  int skip = 0, nlist = 0;
  bool more = false;
  const Reach reach = {clx, cly, clz, chx, chy, chz, Rc, __uint_as_float(v.ds->excursion_bits),
                       st.sph, nsph};
  if (Hs > 0.0f) {
    do {
      if (more) compact_spheres(st.sph, live, make_float4(xi.x, xi.y, xi.z, H));  // (the staging took their room)
      nlist = search(v, F, reach, st, leaf_ok, chunk_ok, skip, more, COOP ? warp : -1);
      stage_list(srcs, st, nlist, consume, wc);
      skip += nlist;
    } while (more && !st.failed);
  }
  fold_cell();
  if constexpr (COOP) {
    double sum[4] = {PASS == 1 ? sr : dxi, PASS == 1 ? srt : dyi, PASS == 1 ? s1 : dzi, s2};
    bool failed = st.failed;
    coop_reduce<StageB, 4>(sum, failed);
    st.failed = failed;  // the same in every warp
    if (PASS == 1) {
      sr = sum[0]; srt = sum[1]; s1 = sum[2]; s2 = sum[3];
    } else {
      dxi = sum[0]; dyi = sum[1]; dzi = sum[2];
    }
    if (warp != 0) return;  // the first warp writes the results
  }
  if (PASS == 1 && valid && !live) {
    // nothing flows back through this particle's density
    w.ka[i] = 0.0;
    w.kb[i] = 0.0;
    w.km[i] = 0.0;
  } else if (PASS == 1 && live) {
    // (the self pair r = 0 was among the records: w(0) = 1, w'(0) = 0)
    const double h = (double)v.h[i];
    const double Hd = (double)GAMMA_K * h;
    const double H3 = Hd * Hd * Hd;
    const double D = 3.0 * sr - srt;
    const double dfdsr = -3.0 * srt / (D * D), dfdsrt = 3.0 * sr / (D * D);
    const double drho_dh = -KN_D * srt / (H3 * h);
    const double S1 = srt - 3.0 * sr;  // sum m q w'
    const double df_dh = dfdsr * (-S1 / h) + dfdsrt * (-s2 / h);
    const double g3 = (double)GAMMA_K * (double)GAMMA_K * (double)GAMMA_K;
    const double Fh = -(KN_D / g3) * s1 / h;
    const double rb = w.rhob[i], fbar = w.fb[i];
    const double hbt = w.hb[i] + rb * drho_dh + fbar * df_dh;
    const double lam = Fh != 0.0 ? -hbt / Fh : 0.0;
    w.ka[i] = rb * KN_D / H3 + fbar * dfdsr;
    w.kb[i] = fbar * dfdsrt;
    w.km[i] = lam * KN_D / g3;
    // consumed: this step computed h, rho and f of i
    w.hb[i] = 0.0;
    w.rhob[i] = 0.0;
    w.fb[i] = 0.0;
  } else if (PASS == 2 && live) {
    atomicAdd(&w.xb[i], dxi);
    atomicAdd(&w.yb[i], dyi);
    atomicAdd(&w.zb[i], dzi);
  }
  __syncwarp();
}

// (as k_adj_force: a whole block per group in steps with few groups)
template <int PASS>
__global__ void __launch_bounds__(PT, 1) k_adj_density(View v, AdjWork w) {
  DevState *ds = v.ds;
  __shared__ int s_go, s_nq, s_item;
  if (threadIdx.x == 0) {
    s_go = ds->halt ? 0 : 1;
    s_nq = ds->n_active_groups + ds->n_heavy_groups;
  }
  __syncthreads();
  if (!s_go) return;  // the whole block
  StageB st;
  stage_init(st);
  const int lane = lane_id();
  const int nq = s_nq;
  int *head = PASS == 1 ? &ds->head_density : &ds->head_misc;
  WarpCounters wc = {0, 0, 0, 0, 0, 0};
  if (nq <= 2 * (int)gridDim.x) {
    for (;;) {
      if (threadIdx.x == 0) s_item = atomicAdd(head, 1);
      __syncthreads();
      const int item = s_item;
      __syncthreads();
      if (item >= nq || st.failed) break;  // (st.failed is the same in every warp)
      const int wg = active_group(v, ds, item);
      if (!SPH_IN(ds, wg, ds->n_groups, SPH_CHECK_GROUP)) break;
      density_adj_group<PASS, true>(v, w, wg, frame_of(v, ds, wg), st, wc);
    }
  } else {
    for (;;) {
      int item = 0;
      if (lane == 0) item = atomicAdd(head, 1);
      item = __shfl_sync(FULL, item, 0);
      if (item >= nq || st.failed) break;
      const int wg = active_group(v, ds, item);
      if (!SPH_IN(ds, wg, ds->n_groups, SPH_CHECK_GROUP)) break;
      density_adj_group<PASS, false>(v, w, wg, frame_of(v, ds, wg), st, wc);
    }
  }
  if (lane == 0 && wc.timeout) record_error(ds, SPH_ERR_TIMEOUT, wc.timeout, true);
}

// ---------------------------------------------------------------------------
// 6. back to caller order: prediction and drift adjoints
// ---------------------------------------------------------------------------
__global__ void k_adj_scatter(View v, AdjWork w, sph_particles pre, sph_particles post,
                              sph_adjoint adj, long long ti, int first, double dt_min) {
  const long long n = v.n;
  for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < n;
       k += (long long)gridDim.x * blockDim.x) {
    const int o = w.perm[k];
    const double xb = w.xb[k], yb = w.yb[k], zb = w.zb[k];
    const double avx = adj.vx[o], avy = adj.vy[o], avz = adj.vz[o];
    const double aax = adj.ax[o], aay = adj.ay[o], aaz = adj.az[o];
    const double aA = adj.A[o], aAdot = adj.Adot[o];
    const double cb = w.cb[k], Qb = w.Qb[k], hb = w.hb[k], rb = w.rhob[k], fb = w.fb[k];
    // drift of this step: x(ti) = x + v (ti - ti_drift) dt_min, for the
    // particles the forward drifted (those whose ti_drift moved)
    const double dtd = (double)(post.ti_drift[o] - pre.ti_drift[o]) * dt_min;
    // prediction: v_pred = v + a dtp, A_pred = A + Adot dtp
    const int bi = pre.bin[o] & (MAX_BINS - 1);
    const double dtp = ((double)(ti - pre.ti_begin[o]) - 0.5 * (double)(1ll << bi)) * dt_min;
    const double vpx = w.vpxb[k], vpy = w.vpyb[k], vpz = w.vpzb[k];
    adj.x[o] = xb;
    adj.y[o] = yb;
    adj.z[o] = zb;
    adj.vx[o] = avx + (vpx + xb * dtd);
    adj.vy[o] = avy + (vpy + yb * dtd);
    adj.vz[o] = avz + (vpz + zb * dtd);
    adj.ax[o] = aax + vpx * dtp;
    adj.ay[o] = aay + vpy * dtp;
    adj.az[o] = aaz + vpz * dtp;
    if (first) {
      adj.A[o] = cb;  // A held u before the first step
    } else {
      adj.A[o] = aA + Qb;
      adj.Adot[o] = aAdot + Qb * dtp;
    }
    adj.h[o] = hb;
    adj.rho[o] = rb;
    adj.f[o] = fb;
  }
}

// ---------------------------------------------------------------------------
// grid-density loss
// ---------------------------------------------------------------------------
// Range of grid indices (unwrapped) whose point centres (a + 1/2) s lie within
// H of x along one axis; at most n_grid of them.
__device__ __forceinline__ void grid_range(double x, double H, double s, int ng, int &a0, int &cnt) {
  a0 = (int)ceil((x - H) / s - 0.5);
  const int a1 = (int)floor((x + H) / s - 0.5);
  cnt = min(a1 - a0 + 1, ng);
}

__device__ __forceinline__ double shfl_d(double x, int src) {
  return __shfl_sync(FULL, x, src);
}

// The kernel of one particle (c = m (8/pi) / H^3, hi = 1 / H) at a grid point:
// offsets in units of H, q2 their square sum, f about the same in FP32.
// Forward: adds m W to the point.  BWD: adds to acc the point's d loss / d x,
// y, z and, unscaled, d h.
template <bool BWD>
struct GridKernel {
  double c, T, c_in, c_out;  // dW/dr = T w'(q); scales of the two pieces
  __device__ GridKernel(double c_, double hi)
      : c(c_), T(c_ * hi), c_in(BWD ? T : -6.0 * c_), c_out(BWD ? -6.0 * T : 2.0 * c_) {}
  __device__ __forceinline__ void point(double dx, double dy, double dz, double q2, float f,
                                        long long gidx, double *rho_g, const double *rho_bar,
                                        double (&acc)[4]) const {
    const double y0 = f > 1e-30f ? widen(rsqrtf(f)) : 0.0;
    const double t = q2 * y0;
    const double e = fma(-t, y0, 1.0);
    const double pe = fma(0.375, e, 0.5) * e;
    const double q = fma(t, pe, t);
    const double u = 1.0 - q;
    const bool inner = __double2hiint(q) < 0x3fe00000;  // q < 1/2
    const bool in = __double2hiint(u) >= 0;             // q <= 1
    const double sq = inner ? q : u;
    const double s2 = sq * sq;
    if (!BWD) {
      // 1 - 6 q^2 (1 - q), 2 (1 - q)^3
      const double w = fma(s2 * u, inner ? c_in : c_out, inner ? c : 0.0);
      if (in) atomicAdd(&rho_g[gidx], w);
    } else {
      const double gb = in ? rho_bar[gidx] : 0.0;
      // w' / q: -12 + 18 q, -6 (1 - q)^2 / q
      const double yq = fma(y0, pe, y0);
      const double v = inner ? fma(18.0, q, -12.0) : s2 * yq;
      const double g = (gb * (inner ? c_in : c_out)) * v;
      acc[0] = fma(g, dx, acc[0]);
      acc[1] = fma(g, dy, acc[1]);
      acc[2] = fma(g, dz, acc[2]);
      // 3 w + q w': 3 + q^2 (36 q - 30), (1 - q)^2 (6 - 12 q)
      const double wh =
          fma(s2, fma(inner ? 36.0 : -12.0, q, inner ? -30.0 : 6.0), inner ? 3.0 : 0.0);
      acc[3] = fma(gb, wh, acc[3]);
    }
  }
};

// Adds m W(|x_g - x|, h) of every particle to the grid points within its
// support (FP64 atomics); with BWD, reads d loss / d rho_g instead and
// accumulates d loss / d x, d h (and d v through the drift to the tick).
//
// Everything is FP64, and FP64 bounds it: a warp's FP64 instruction occupies
// an SM for 16 cycles, 64 issue slots, so the layout spends integer and FP32
// work to save FP64.  A warp takes up to 32 particles, each lane setting one
// up (its divisions and grid range once, not in every lane); then the warp
// works on one particle at a time, in units of its support (q = r / H).  Per
// axis a table of the offsets in the box of grid points around it (up to 32
// per axis at a time); an FP32 test of every point of the box (half of them lie
// outside the support), the ones it cannot exclude queued and evaluated 32 at
// a time, with 11 FP64 instructions per point (21 with BWD): q by a
// third-order step from an FP32 reciprocal square root (its error 4e-7 cubed
// is below FP64's), one polynomial for both pieces of the kernel with
// selected coefficients, its scale folded into them.  One thread per particle
// computed the offsets of each point anew, with FP64 square roots and
// divisions, 45 and more FP64 instructions per point of the whole box.
// 110,592 particles on a 64^3 grid (113 points in a support): 1885 -> 463 us,
// backward 3385 -> 787 us; 262,144 on 32^3 514 -> 421 us and 894 -> 530 us;
// 2,744 on 128^3 (supports of 40,000 points) 153 -> 2.5 ms and 182 -> 4.3 ms.
// Against extended precision a point's W is off by 4.0e-17 rms (before 4.5e-17),
// its d/dh by 1.1e-16 (1.5e-16).  Against 64-bit sums of the textbook form
// (r / H, then the two cubics), whose roundings the form before shared, the
// distance grew: densities and adjoints of a clumpy set 2.9e-16 -> 5.3e-16.
// Where at least GD_LANES of a warp's particles have boxes of at most GD_FEW
// points, those are one lane's work each, all at once: a warp per particle costs
// some 20 FP64 instructions before its first point (27,000 particles on a 16^3
// grid: 114 us, a lane per particle 75 us; here 72 us).  With fewer such particles
// a point of a lane's own costs about as much as a particle of the warp's, and
// the longest lane counts: lanes only for twice as many particles as points (a
// support that misses most points, 1,000,000 particles on 16^3: 553 -> 285 us,
// backward 836 -> 323).  They come after the warp's own particles: first, every
// warp sends them at once, and the points of a clump, or of a coarse grid, take
// many additions each (a clumpy 111k on 64^3 460 -> 538 us where one clump meets a
// point; 262,144 on 32^3 521 us first, 421 last).
constexpr int GD_WARPS = 4, GD_SIDE = 32, GD_FEW = 27, GD_LANES = 16;
struct GridWarp {
  double d[3][GD_SIDE];   // (x - x_g) / H along each axis
  double d2x[GD_SIDE];    // its square, first axis
  float f2[3][GD_SIDE];   // FP32 squares
  int ix[3][GD_SIDE];     // grid index in the periodic box
  unsigned short q[64];   // queued points: index x | y << 5 | z << 10
};

template <bool BWD>
__global__ void __launch_bounds__(GD_WARPS * 32, 6)
    k_grid_density(sph_particles p, int ng, long long ti, double dt_min, double box,
                   double *rho_g, const double *rho_bar, sph_adjoint adj, int per_warp) {
  __shared__ GridWarp s_w[GD_WARPS];
  GridWarp &S = s_w[threadIdx.x >> 5];
  const int lane = lane_id();
  const unsigned below = (1u << lane) - 1u;
  const long long n = p.n;
  const double s = box / ng;
  const long long stride = (long long)gridDim.x * GD_WARPS * per_warp;
  for (long long j0 = ((long long)blockIdx.x * GD_WARPS + (threadIdx.x >> 5)) * per_warp; j0 < n;
       j0 += stride) {
    // one particle per lane
    const int cnt = (int)(n - j0 < per_warp ? n - j0 : per_warp);
    const long long j = j0 + lane;
    double X[3] = {0.0, 0.0, 0.0}, dtd = 0.0, Hinv = 0.0, C = 0.0;
    int a0[3] = {0, 0, 0}, na[3] = {0, 0, 0};
    if (lane < cnt) {
      dtd = (double)(ti - p.ti_drift[j]) * dt_min;
      X[0] = wrap_box(p.x[j] + (double)p.vx[j] * dtd, box);
      X[1] = wrap_box(p.y[j] + (double)p.vy[j] * dtd, box);
      X[2] = wrap_box(p.z[j] + (double)p.vz[j] * dtd, box);
      const double H = GAMMA_K_D * (double)p.h[j];
      Hinv = 1.0 / H;
      C = (double)p.m[j] * KN_D * (Hinv * Hinv * Hinv);
#pragma unroll
      for (int k = 0; k < 3; k++) grid_range(X[k], H, s, ng, a0[k], na[k]);
    }
    double o[4] = {0.0, 0.0, 0.0, 0.0};  // BWD: this lane's particle
    // boxes of a few points: one lane per particle, all at once (below)
    const int box3 = na[0] > 0 && na[1] > 0 && na[2] > 0 && na[0] <= GD_FEW && na[1] <= GD_FEW &&
                             na[2] <= GD_FEW
                         ? na[0] * na[1] * na[2]
                         : 0;
    bool few = box3 > 0 && box3 <= GD_FEW;
    const int lanes = __popc(__ballot_sync(FULL, few));
    if (lanes < GD_LANES && 2 * __reduce_max_sync(FULL, few ? box3 : 0) > lanes) few = false;
    for (unsigned todo = __ballot_sync(FULL, !few && na[0] > 0 && na[1] > 0 && na[2] > 0); todo;
         todo &= todo - 1u) {
      const int k = __ffs(todo) - 1;
      const double hi = shfl_d(Hinv, k), c = shfl_d(C, k);
      const double xk[3] = {shfl_d(X[0], k), shfl_d(X[1], k), shfl_d(X[2], k)};
      int ak[3], nk[3];
#pragma unroll
      for (int q = 0; q < 3; q++) {
        ak[q] = __shfl_sync(FULL, a0[q], k);
        nk[q] = __shfl_sync(FULL, na[q], k);
      }
      const GridKernel<BWD> K(c, hi);
      double acc[4] = {0.0, 0.0, 0.0, 0.0};
      auto point = [&](unsigned int id) {
        const int ix = id & 31, iy = (id >> 5) & 31, iz = id >> 10;
        const double dx = BWD ? S.d[0][ix] : 0.0, dy = S.d[1][iy], dz = S.d[2][iz];
        const long long gidx = S.ix[0][ix] + (long long)ng * (S.ix[1][iy] + (long long)ng * S.ix[2][iz]);
        K.point(dx, dy, dz, fma(dz, dz, fma(dy, dy, S.d2x[ix])),
                S.f2[0][ix] + S.f2[1][iy] + S.f2[2][iz], gidx, rho_g, rho_bar, acc);
      };
      for (int z0 = 0; z0 < nk[2]; z0 += GD_SIDE)
        for (int y0 = 0; y0 < nk[1]; y0 += GD_SIDE)
          for (int x0 = 0; x0 < nk[0]; x0 += GD_SIDE) {
            const int b0[3] = {x0, y0, z0};
            int side[3];
#pragma unroll
            for (int q = 0; q < 3; q++) side[q] = min(GD_SIDE, nk[q] - b0[q]);
            // the three tables, the axes one after the other in the lanes
            __syncwarp();
            for (int e = lane; e < side[0] + side[1] + side[2]; e += 32) {
              const int ax = e < side[0] ? 0 : (e < side[0] + side[1] ? 1 : 2);
              const int i = e - (ax > 0 ? side[0] : 0) - (ax > 1 ? side[1] : 0);
              const int at = ((ax == 0 ? ak[0] + x0 : ax == 1 ? ak[1] + y0 : ak[2] + z0) + i);
              const int w = (at % ng + ng) % ng;
              const double xa = ax == 0 ? xk[0] : ax == 1 ? xk[1] : xk[2];
              const double d = min_img(xa - (w + 0.5) * s, box) * hi;
              S.d[ax][i] = d;
              const double d2 = d * d;
              if (ax == 0) S.d2x[i] = d2;
              S.f2[ax][i] = (float)d2;
              S.ix[ax][i] = w;
            }
            __syncwarp();
            const int total = side[0] * side[1] * side[2];  // at most 2^15: exact in FP32
            const float rx = 1.0f / (float)side[0], ry = 1.0f / (float)side[1];
            int nq = 0;
            for (int t0 = 0;; t0 += 32) {
              const bool last = t0 >= total;  // the rest of the queue
              if (!last) {
                const int t = t0 + lane;
                const int tyz = (int)(((float)t + 0.5f) * rx);
                const int iz = (int)(((float)tyz + 0.5f) * ry);
                const int ix = t - tyz * side[0], iy = tyz - iz * side[1];
                // (three roundings of 6e-8 each: nothing within the support is lost)
                const bool near = t < total && S.f2[0][ix] + S.f2[1][iy] + S.f2[2][iz] < 1.000001f;
                const unsigned m = __ballot_sync(FULL, near);
                if (near) S.q[nq + __popc(m & below)] = (unsigned short)(ix | (iy << 5) | (iz << 10));
                nq += __popc(m);
                __syncwarp();
              }
              if (nq >= 32 || last) {
                if (lane < nq) point(S.q[lane]);
                const unsigned short rest = S.q[32 + lane];
                __syncwarp();
                S.q[lane] = rest;
                nq -= 32;
                __syncwarp();
              }
              if (last) break;
            }
          }
      if (BWD) {
        // the four sums over the warp, half the values dropped at each of the
        // first two exchanges (6 additions instead of 20)
        const bool up = lane & 16, up2 = lane & 8;
        double v0 = up ? acc[2] : acc[0], v1 = up ? acc[3] : acc[1];
        v0 += __shfl_xor_sync(FULL, up ? acc[0] : acc[2], 16);
        v1 += __shfl_xor_sync(FULL, up ? acc[1] : acc[3], 16);
        double r = up2 ? v1 : v0;
        r += __shfl_xor_sync(FULL, up2 ? v0 : v1, 8);
#pragma unroll
        for (int o = 4; o; o >>= 1) r += __shfl_xor_sync(FULL, r, o);
        const double r0 = shfl_d(r, 0), r1 = shfl_d(r, 8), r2 = shfl_d(r, 16), r3 = shfl_d(r, 24);
        if (lane == k) {
          o[0] = r0;
          o[1] = r1;
          o[2] = r2;
          o[3] = r3;
        }
      }
    }
    if (few) {
      const GridKernel<BWD> K(C, Hinv);
      for (int c = 0; c < na[2]; c++) {
        const int iz = ((a0[2] + c) % ng + ng) % ng;
        const double dz = min_img(X[2] - (iz + 0.5) * s, box) * Hinv;
        for (int b = 0; b < na[1]; b++) {
          const int iy = ((a0[1] + b) % ng + ng) % ng;
          const double dy = min_img(X[1] - (iy + 0.5) * s, box) * Hinv;
          for (int a = 0; a < na[0]; a++) {
            const int ix = ((a0[0] + a) % ng + ng) % ng;
            const double dx = min_img(X[0] - (ix + 0.5) * s, box) * Hinv;
            const double q2 = fma(dz, dz, fma(dy, dy, dx * dx));
            if (q2 < 1.0)
              K.point(dx, dy, dz, q2, (float)q2, ix + (long long)ng * (iy + (long long)ng * iz), rho_g,
                      rho_bar, o);
          }
        }
      }
    }
    if (BWD && lane < cnt) {
      adj.x[j] += o[0];
      adj.y[j] += o[1];
      adj.z[j] += o[2];
      adj.vx[j] += o[0] * dtd;
      adj.vy[j] += o[1] * dtd;
      adj.vz[j] += o[2] * dtd;
      // dW/dh = -GAMMA_K (8/pi) H^-4 (3 w + q w'); a support without a point
      // (of h = 0, whose 1 / H is infinite, among them) adds nothing
      if (o[3] != 0.0) adj.h[j] += -GAMMA_K_D * (C * Hinv) * o[3];
    }
  }
}

// ---------------------------------------------------------------------------
// state copy (optionally into the caller's order)
// ---------------------------------------------------------------------------
// Every load of a particle's ~25 arrays is issued before the first store (src
// and dst could overlap as far as the compiler knows, and one array after the
// other kept one load in flight per thread: 2.1M particles 130 -> 67 us,
// 6.9 TB/s).  With a permutation the scattered stores bound it, and of states far
// larger than L2 they are slower out of one batch per thread: one array after the
// other then (2.1M particles 1628 -> 1504 us, 1575 array by array in the
// structure's order; at 600,000 the batch is ahead, 91 against 104 us).
struct CopyFields {
  const unsigned long long *s8[6];
  unsigned long long *d8[6];
  const unsigned int *s4[19];
  unsigned int *d4[19];
  const uint8_t *s1[2];
  uint8_t *d1[2];
};

template <bool BATCH>
__global__ void __launch_bounds__(256)
    k_state_copy(CopyFields f, long long n, const int32_t *__restrict__ perm) {
  for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < n;
       k += (long long)gridDim.x * blockDim.x) {
    const long long d = perm ? (long long)perm[k] : k;
    if constexpr (BATCH) {
      unsigned long long a[6];
      unsigned int b[19];
      uint8_t c[2];
#pragma unroll
      for (int q = 0; q < 6; q++) a[q] = f.s8[q][k];
#pragma unroll
      for (int q = 0; q < 19; q++) b[q] = f.d4[q] ? f.s4[q][k] : 0u;
#pragma unroll
      for (int q = 0; q < 2; q++) c[q] = f.s1[q][k];
#pragma unroll
      for (int q = 0; q < 6; q++) f.d8[q][d] = a[q];
#pragma unroll
      for (int q = 0; q < 19; q++)
        if (f.d4[q]) f.d4[q][d] = b[q];
#pragma unroll
      for (int q = 0; q < 2; q++) f.d1[q][d] = c[q];
    } else {
#pragma unroll
      for (int q = 0; q < 6; q++) f.d8[q][d] = f.s8[q][k];
#pragma unroll
      for (int q = 0; q < 19; q++)
        if (f.d4[q]) f.d4[q][d] = f.s4[q][k];
#pragma unroll
      for (int q = 0; q < 2; q++) f.d1[q][d] = f.s1[q][k];
    }
  }
}

constexpr size_t ADJ_DENS_SMEM = StageB::bytes() * WARPS_PER_BLOCK;
constexpr size_t ADJ_FORCE_SMEM = StageA::bytes() * WARPS_PER_BLOCK;

int grid_for(long long n) {
  long long g = (n + 255) / 256;
  if (g < 1) g = 1;
  if (g > 4096) g = 4096;
  return (int)g;
}

}  // namespace

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------
cudaError_t launch_adj_prepare(const sph_particles &pre, const sph_particles &post,
                               const sph_particles &W, const sph_adjoint &adj, long long ti,
                               int first, double dt_min, double box, double gamma,
                               cudaStream_t st) {
  if (pre.n == 0) return cudaSuccess;
  note_launches(1);
  k_adj_prepare<<<grid_for(pre.n), 256, 0, st>>>(pre, post, W, adj, ti, first, dt_min, box, gamma);
  return cudaGetLastError();
}

cudaError_t launch_adj_step(const View &v, const AdjWork &w, const sph_particles &pre,
                            const sph_particles &post, const sph_adjoint &adj, long long ti,
                            int first, int grid_pairs, cudaStream_t st) {
  if (v.n == 0) return cudaSuccess;
  // (the pair kernels' shared memory is set by adj_blocks_per_sm)
  const int g = grid_for(v.n);
  note_launches(6);
  k_adj_gather<<<g, 256, 0, st>>>(v, w, adj, v.gamma);
  k_adj_force<<<grid_pairs, PT, ADJ_FORCE_SMEM, st>>>(v, w);
  k_adj_eos<<<g, 256, 0, st>>>(v, w, adj, first);
  k_adj_density<1><<<grid_pairs, PT, ADJ_DENS_SMEM, st>>>(v, w);
  k_adj_density<2><<<grid_pairs, PT, ADJ_DENS_SMEM, st>>>(v, w);
  k_adj_scatter<<<g, 256, 0, st>>>(v, w, pre, post, adj, ti, first, v.dt_min);
  return cudaGetLastError();
}

cudaError_t launch_grid_density(const sph_particles &p, int n_grid, long long ti, double dt_min,
                                double box, double *rho_g, const double *rho_bar,
                                const sph_adjoint *adj, int num_sms, cudaStream_t st) {
  if (p.n == 0) return cudaSuccess;
  note_launches(1);
  // particles per warp: up to 32 share a set-up, fewer where there would be
  // less than 16 warps per SM (110,592 particles, where this gives 32 and 23
  // warps per SM: 422 us; 22 particles per warp, 33 warps per SM: 477 us, both
  // before the lanes' own way)
  const long long slots = 16ll * num_sms;
  int per_warp = (int)std::max<long long>(1, std::min<long long>(32, p.n / slots));
  // (few points per particle, 48 n_grid^3 / n on average: the lanes work on a
  // particle each, and every lane should have one)
  if (48.0 * n_grid * n_grid * n_grid <= 12.0 * (double)p.n) per_warp = 32;
  const long long warps = (p.n + per_warp - 1) / per_warp;
  const int grid = (int)std::min<long long>((warps + GD_WARPS - 1) / GD_WARPS, 64ll * num_sms);
  sph_adjoint none;
  memset(&none, 0, sizeof(none));
  if (adj)
    k_grid_density<true><<<grid, GD_WARPS * 32, 0, st>>>(p, n_grid, ti, dt_min, box, nullptr, rho_bar,
                                                         *adj, per_warp);
  else
    k_grid_density<false><<<grid, GD_WARPS * 32, 0, st>>>(p, n_grid, ti, dt_min, box, rho_g, nullptr,
                                                          none, per_warp);
  return cudaGetLastError();
}

// Resident blocks per SM of the adjoint pair kernels (the smallest over the
// three; 0 when they cannot run).
int adj_blocks_per_sm() {
  struct K {
    const void *fn;
    size_t smem;
  } ks[3] = {{(const void *)k_adj_force, ADJ_FORCE_SMEM},
             {(const void *)k_adj_density<1>, ADJ_DENS_SMEM},
             {(const void *)k_adj_density<2>, ADJ_DENS_SMEM}};
  int best = 1 << 30;
  for (const K &k : ks) {
    if (cudaFuncSetAttribute(k.fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)k.smem) !=
        cudaSuccess) {
      cudaGetLastError();
      return 0;
    }
    int nb = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k.fn, PT, k.smem) != cudaSuccess) {
      cudaGetLastError();
      return 0;
    }
    best = nb < best ? nb : best;
  }
  return best;
}

cudaError_t launch_state_copy(const sph_particles &src, const sph_particles &dst,
                              const int32_t *perm, cudaStream_t st) {
  if (src.n == 0) return cudaSuccess;
  note_launches(1);
  CopyFields f;
  const void *s8[6] = {src.x, src.y, src.z, src.ti_begin, src.ti_end, src.ti_drift};
  void *d8[6] = {dst.x, dst.y, dst.z, dst.ti_begin, dst.ti_end, dst.ti_drift};
  const void *s4[19] = {src.vx, src.vy, src.vz, src.ax, src.ay, src.az, src.A, src.Adot, src.h,
                        src.rho, src.f, src.P, src.c, src.vsig, src.m, src.ngb_density,
                        src.ngb_force, src.div_v, src.curl_v};
  void *d4[19] = {dst.vx, dst.vy, dst.vz, dst.ax, dst.ay, dst.az, dst.A, dst.Adot, dst.h,
                  dst.rho, dst.f, dst.P, dst.c, dst.vsig, dst.m, dst.ngb_density,
                  dst.ngb_force, dst.div_v, dst.curl_v};
  for (int q = 0; q < 6; q++) {
    f.s8[q] = (const unsigned long long *)s8[q];
    f.d8[q] = (unsigned long long *)d8[q];
  }
  for (int q = 0; q < 19; q++) {  // (an optional array that either state lacks is skipped)
    f.s4[q] = (const unsigned int *)s4[q];
    f.d4[q] = s4[q] ? (unsigned int *)d4[q] : nullptr;
  }
  f.s1[0] = (const uint8_t *)src.bin;
  f.s1[1] = src.active;
  f.d1[0] = (uint8_t *)dst.bin;
  f.d1[1] = dst.active;
  // (126 bytes a particle and state: one of 2^20 fills the 129 MB of L2; 1,000,003
  // particles 407 us in batches, 391 array by array, without the optional arrays 254, 261)
  if (perm && src.n > 1ll << 20)
    k_state_copy<false><<<grid_for(src.n), 256, 0, st>>>(f, src.n, perm);
  else
    k_state_copy<true><<<grid_for(src.n), 256, 0, st>>>(f, src.n, perm);
  return cudaGetLastError();
}

}  // namespace sph
