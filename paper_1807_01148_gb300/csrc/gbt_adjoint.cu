// Calibration adjoint of the step (not in the paper; the calibration workload of this
// library).  Loss L = sum over observations k and trips v of (p_v(t_k) - target)^2,
// p_v = route progress (completed link lengths + x; 0 before departure; the route's
// length after arrival).  The gradient with respect to every class's IDM parameters
// (v0, T, a, b, s0) holds the discrete decisions of the run fixed: the forward pass
// tapes, per vehicle-step, which form of Eq. 7 gave the acceleration (leader on the
// link, leader across the link end, free road, closed stop line), the gap and speeds
// that entered it, and how the ballistic move ended (normal, stopped within the step,
// clamped at the stop line, arrived).  The reverse sweep runs in binary64.
#include "gbt_observe.cuh"

namespace gbt {

#define GS(i, n) for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < (n); i += gridDim.x * blockDim.x)

// Route progress of every trip at the current state (buffer A).  With target: the
// residual of the active trips goes to res (0 for the others, whose progress is
// constant) and the squared residuals of all trips are added to ctl->loss; with p_out:
// the progress itself.
__global__ void k_observe(Dev d, const double* target, double* res, double* p_out) {
  const int nA = d.ctl->nA;
  const int total = nA + d.n_trips;
  double acc = 0.0;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < total; i += gridDim.x * blockDim.x) {
    int vid;
    double p;
    bool active;
    if (i < nA) {
      if (d.A.link[i] < 0) continue;
      vid = d.A.vid[i];
      p = prefix_len(d, vid, d.A.cur[i]) + (double)d.A.x[i];
      active = true;
    } else {
      vid = i - nA;
      const uint8_t st = d.status[vid];
      if (st == kActive) continue;
      p = st == kArrived ? prefix_len(d, vid, d.rlen[vid]) : 0.0;
      active = false;
    }
    if (p_out) p_out[vid] = p;
    if (target) {
      const double r = p - target[vid];
      acc += r * r;
      res[vid] = active ? r : 0.0;
    }
  }
  if (target) {
    const double b = block_sum(acc);
    if (threadIdx.x == 0) atomicAdd(&d.ctl->loss, b);
  }
}

void launch_observe(const Dev& d, int grid, cudaStream_t s, const double* target, double* res, double* p_out) {
  k_observe<<<grid, 256, 0, s>>>(d, target, res, p_out);
}

__global__ void k_tape_begin(Dev d) { d.ctl->tape_t0 = d.ctl->t; }

void launch_tape_begin(const Dev& d, cudaStream_t s) { k_tape_begin<<<1, 1, 0, s>>>(d); }

// Reverse of step t.  lx, lv: adjoint of the state after the step (by trip id), plus
// 2 * residual when that state was observed; nx, nv (zero): adjoint of the state before it;
// zx, zv (or null): zeroed for the step before that.  What bounds it is the binary64 rate of an
// SM (a warp's operation takes it some 16 cycles, however few threads are active), and most
// trips are not on the road: a block first lists its tile's vehicles, so that full warps work
// on them and the others on nothing; the class's roots and quotients are taken once per
// block, the vehicle's divisors inverted once.  Parameter gradients are summed per warp and
// class with shuffles, then per block in shared memory.
constexpr int kAdjThreads = 64, kAdjTile = 256;

__global__ void __launch_bounds__(kAdjThreads) k_adj_step(Dev d, const TapeRec* slab, const double* lx, const double* lv,
                                                  const double* res, double* nx, double* nv, double* zx, double* zv,
                                                  double* grad, int n_class) {
  extern __shared__ double sg[];              // gradient [n_class][5], then per class cc, cc / 2a, cc / 2b
  double* sc = sg + n_class * 5;
  for (int q = threadIdx.x; q < n_class * 5; q += blockDim.x) sg[q] = 0.0;
  for (int c = threadIdx.x; c < n_class; c += blockDim.x) {
    const double A = d.cls[c].a, Bb = d.cls_b[c];
    const double cc = 1.0 / (2.0 * sqrt(A * Bb));
    sc[c * 3] = cc;
    sc[c * 3 + 1] = cc / (2.0 * A);
    sc[c * 3 + 2] = cc / (2.0 * Bb);
  }
  __syncthreads();
  const double dt = d.dt, h = 0.5 * dt * dt;
  const int wl = threadIdx.x & 31;
  __shared__ int s_n;
  __shared__ int s_list[kAdjTile];
  for (int base = blockIdx.x * kAdjTile; base < d.n_trips; base += gridDim.x * kAdjTile) {
    if (threadIdx.x == 0) s_n = 0;
    __syncthreads();
    for (int i = base + threadIdx.x; i < base + kAdjTile && i < d.n_trips; i += kAdjThreads) {
      if (slab[i].valid) s_list[atomicAdd(&s_n, 1)] = i;
      if (zx) {
        zx[i] = 0.0;
        zv[i] = 0.0;
      }
    }
    __syncthreads();
    const int n = s_n;
    for (int k0 = threadIdx.x & ~31; k0 < n; k0 += kAdjThreads) {
      const int i = k0 + wl < n ? s_list[k0 + wl] : -1;
      double mu = 0.0;
      TapeRec r;
      r.valid = 0;
      if (i >= 0) r = slab[i];
      if (r.valid) {
        const double lxp = lx[i] + (res ? 2.0 * res[i] : 0.0);
        const double lvp = lv[i];
        if (r.branch == kBrNormal) {
          mu = lxp * h + lvp * dt;
          atomicAdd(&nx[i], lxp);
          atomicAdd(&nv[i], lxp * dt + lvp);
        } else if (r.branch == kBrStop) {
          const double va = (double)r.v / (double)r.a;
          mu = lxp * va * va * 0.5;
          atomicAdd(&nx[i], lxp);
          atomicAdd(&nv[i], -lxp * va);
        }
      }
      const bool has = mu != 0.0 && r.kind != kFormNone;
      int c = 0;
      double g0 = 0.0, gT = 0.0, gA = 0.0, gB = 0.0, gs = 0.0;
      if (has) {
        const LinkRec L = d.links[r.link];
        c = L.cls;
        const ClassPar P = d.cls[c];
        const double A = P.a, T = P.T, v = r.v, iv0 = 1.0 / (double)L.v0;
        const double rr = v * iv0, r3 = rr * rr * rr, r4 = r3 * rr;
        double dA = 1.0 - r4, dv = -4.0 * A * r3 * iv0;
        if (d.cls_v0_param[c]) g0 = mu * (4.0 * A * r4 * iv0);
        if (r.kind != kFormFree) {
          // the floors of Eq. 7, decided in binary32 exactly as the forward pass did
          const float dv32 = r.v - r.vl;
          const float t1 = r.v * P.T;
          const float t2 = (r.v * dv32) / P.sab2;
          const bool dyn_on = (t1 + t2) > 0.0f;
          const bool floored = !(r.s >= d.s_min) || r.s == d.s_min;
          const double cc = sc[c * 3];
          const double dvv = v - (double)r.vl;
          const double ss = (double)P.s0 + (dyn_on ? v * T + v * dvv * cc : 0.0);
          const double ise = 1.0 / (floored ? (double)d.s_min : (double)r.s);
          const double q = ss * ise;
          const double k2 = -2.0 * A * q * ise;
          double dvl = 0.0;
          dA += -q * q;
          gs = mu * k2;
          if (dyn_on) {
            gT = mu * (k2 * v);
            dA -= k2 * v * dvv * sc[c * 3 + 1];
            gB = -mu * (k2 * v * dvv * sc[c * 3 + 2]);
            dv += k2 * (T + (dvv + v) * cc);
            dvl = k2 * (-v * cc);
          }
          const double ds = floored ? 0.0 : 2.0 * A * q * q * ise;
          atomicAdd(&nx[i], -mu * ds);
          if (r.kind == kFormLead || r.kind == kFormNext) {
            atomicAdd(&nx[r.lead], mu * ds);
            atomicAdd(&nv[r.lead], mu * dvl);
          }
        }
        atomicAdd(&nv[i], mu * dv);
        gA = mu * dA;
      }
      // sums per class over the warp
      unsigned left = __ballot_sync(0xffffffffu, has);
      while (left) {
        const int lead = __ffs(left) - 1;
        const int cl = __shfl_sync(0xffffffffu, c, lead);
        const bool in = has && c == cl;
        double q0 = in ? g0 : 0.0, q1 = in ? gT : 0.0, q2 = in ? gA : 0.0, q3 = in ? gB : 0.0, q4 = in ? gs : 0.0;
  #pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
          q0 += __shfl_xor_sync(0xffffffffu, q0, o);
          q1 += __shfl_xor_sync(0xffffffffu, q1, o);
          q2 += __shfl_xor_sync(0xffffffffu, q2, o);
          q3 += __shfl_xor_sync(0xffffffffu, q3, o);
          q4 += __shfl_xor_sync(0xffffffffu, q4, o);
        }
        // five threads, one parameter each
        const double q = wl == 0 ? q0 : wl == 1 ? q1 : wl == 2 ? q2 : wl == 3 ? q3 : q4;
        if (wl < 5 && q != 0.0) atomicAdd(&sg[cl * 5 + wl], q);
        left &= ~__ballot_sync(0xffffffffu, in);
      }
    }
    __syncthreads();
  }
  __syncthreads();
  for (int q = threadIdx.x; q < n_class * 5; q += blockDim.x)
    if (sg[q] != 0.0) atomicAdd(&grad[q], sg[q]);
}

void launch_adj_step(const Dev& d, int grid, cudaStream_t s, const TapeRec* slab, const double* lx,
                     const double* lv, const double* res, double* nx, double* nv, double* zx, double* zv, double* grad,
                     int n_class) {
  const int need = (d.n_trips + kAdjTile - 1) / kAdjTile;
  const int blocks = need < 1 ? 1 : need < grid ? need : grid;
  k_adj_step<<<blocks, kAdjThreads, (size_t)n_class * 8 * sizeof(double), s>>>(d, slab, lx, lv, res, nx, nv, zx, zv, grad,
                                                                       n_class);
}

}  // namespace gbt
