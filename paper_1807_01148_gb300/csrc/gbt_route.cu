// Trip planning on the GPU (Waddell et al., Sec. 6.3.1 and Sec. 6 "Simulation scale"):
// one shortest-path tree per distinct origin, shared by all trips from that origin
// (the paper replaces per-agent Dijkstra by per-source trees for a two-orders-of-
// magnitude speed-up), on integer decisecond link costs.
//
// Each CTA of a persistent grid takes origins from an atomic work counter and runs a
// near-far variant of delta-stepping (Meyer & Sanders 2003): nodes whose tentative
// distance is below the current threshold T are relaxed in synchronous rounds from a
// deduplicated near queue; farther improvements go to a deduplicated far pile, which
// is split when the near queue empties (T = smallest live far distance + delta).
// Distances are 64-bit words tagged with a per-CTA epoch, so no per-origin reset of
// the node records is needed.  Once the near queue is empty every distance below T is
// final: the tree ends there when all destinations of its trips lie below T (the walks
// back from them only see nodes nearer than they are).  The tree is then read back for
// every trip of the origin by walking from the destination: at node v take the lowest-id
// in-link u -> v with dist[u] + c = dist[v] (a unique, canonical shortest path).  In the
// all-or-nothing mode (R.flow set) that walk adds one trip to every link of the path
// instead of storing it: the direction finding of Frank-Wolfe (Sec. 5.2).
//
// A round is a chain of dependent memory accesses, so its length is what counts: four
// threads share a node's out-links, (head, cost) pairs lie together, a node's distance and
// queue tags are one 16-byte record, the near queue is in shared memory (its overflow in
// global memory), and one barrier ends a round.  A trip's walk is made by eight threads,
// which test as many in-links at once and fetch the in-links of the candidates beforehand.
// Measured, 12,000 trips on the metro (225,000 nodes, 11,700 trees): 343 -> 43 ms a call; 60,000
// trips on 12,000 nodes, an assignment of all trees: 27.3 -> 5.9 ms.
#include <climits>

#include "gbt_internal.cuh"

namespace gbt {

constexpr int kRouteThreads = 256, kNearCap = 2048;   // near-queue entries in shared memory
constexpr int kWalkLanes = 8;

__device__ __forceinline__ unsigned long long dkey(unsigned hi, int d) {
  return ((unsigned long long)hi << 32) | (unsigned)d;
}
__device__ __forceinline__ int dval_of(unsigned long long k, unsigned hi) {
  return (unsigned)(k >> 32) == hi ? (int)(unsigned)k : INT_MAX;
}
__device__ __forceinline__ int dval(const RouteNode* node, int v, unsigned hi) { return dval_of(node[v].key, hi); }

// Walk from v (distance dv) back to o by the eight threads of a group.  Returns the number
// of links, -1 when no tight in-link is found; sink(j, link) is called by one of the threads
// for the j-th link from the end.
template <bool PACKED, typename Sink>
__device__ __forceinline__ int walk_back(const RouteDev& R, const RouteNode* node, unsigned hi, int o, int v, int dv,
                                         Sink sink) {
  const int lane = threadIdx.x & 31, gl = lane & (kWalkLanes - 1), g0 = lane - gl;
  const unsigned gm = ((1u << kWalkLanes) - 1u) << g0;
  int s = R.in_start[v], e = R.in_start[v + 1], n = 0;
  while (v != o) {
    unsigned hit = 0;
    int u = 0, du = 0, us = 0, ue = 0, p = 0;
    for (int p0 = s; p0 < e && !hit; p0 += kWalkLanes) {
      p = p0 + gl;
      bool ok = false;
      if (p < e) {
        int2 x;
        if (PACKED) {
          x = R.in_edge[p];
        } else {
          const int l = R.in_link[p];
          x = make_int2(R.lfrom[l], R.cost[l]);
        }
        u = x.x;
        du = dval(node, u, hi);
        us = R.in_start[u];
        ue = R.in_start[u + 1];
        ok = du != INT_MAX && du + x.y == dv;
      }
      hit = __ballot_sync(gm, ok) & gm;
    }
    if (!hit || n >= R.nn) return -1;
    const int src = __ffs(hit) - 1;   // ascending link ids: the first one
    if (lane == src) sink(n, R.in_link[p]);
    n++;
    v = __shfl_sync(gm, u, src);
    dv = __shfl_sync(gm, du, src);
    s = __shfl_sync(gm, us, src);
    e = __shfl_sync(gm, ue, src);
  }
  return n;
}

// PACKED: the links of a node as (node, cost) pairs; otherwise by id, through arrays per link
// (sim_sssp_static, which has no memory to pack them in, and planning under a memory cap).
template <bool PACKED>
__global__ void __launch_bounds__(kRouteThreads) k_sssp_route(RouteDev R) {
  __shared__ int sh_oi, sh_nf, sh_nf2, sh_min;
  __shared__ int sh_nq[3];
  __shared__ unsigned sh_epoch;
  __shared__ int sh_q[2][kNearCap];
  const int tid = threadIdx.x, bd = kRouteThreads;
  const size_t base = (size_t)blockIdx.x * (size_t)R.nn;
  RouteNode* node = R.node + base;
  int* Q[2] = {R.qa + base, R.qb + base};
  int* F = R.fa + base;
  int* Fn = R.fb + base;
  int round = R.cta_round[blockIdx.x];   // tags near-queue membership; never repeats within this CTA
  for (;;) {
    __syncthreads();
    if (tid == 0) {
      sh_oi = atomicAdd(R.work, 1);
      sh_epoch = ++R.cta_epoch[blockIdx.x];
    }
    __syncthreads();
    const int oi = sh_oi;
    if (oi >= R.n_origins) break;
    const unsigned ep = sh_epoch;
    const unsigned hi = 0xFFFFFFFFu - ep;
    const int o = R.origins[oi];
    const int t0 = R.otrip_start[o], t1 = R.otrip_start[o + 1];
    round++;
    int cur = 0;   // counter of the current near queue; the queues alternate with it
    if (tid == 0) {
      node[o].key = dkey(hi, 0);
      node[o].q = round;
      sh_q[0][0] = o;
      sh_nq[0] = 1;
      sh_nq[1] = sh_nq[2] = 0;
      sh_nf = 0;
    }
    int b = 0;
    __syncthreads();
    int T = R.delta;
    for (;;) {
      // ---- relax the near bucket in rounds until it is empty
      for (;;) {
        const int nq = sh_nq[cur];
        if (nq == 0) break;
        const int nxt = cur == 2 ? 0 : cur + 1, old = nxt == 2 ? 0 : nxt + 1;
        if (tid == 0) sh_nq[old] = 0;   // the previous round's counter is the one after the next's
        round++;
        const int* qs = sh_q[b];
        const int* qg = Q[b];
        int* ns = sh_q[b ^ 1];
        int* ng = Q[b ^ 1];
        for (int k = tid; k < 4 * nq; k += bd) {
          const int i = k >> 2;
          const int u = i < kNearCap ? qs[i] : qg[i];
          const int s = R.out_start[u], e = R.out_start[u + 1];
          const int du = dval(node, u, hi);
          for (int q = s + (k & 3); q < e; q += 4) {
            int2 x;
            if (PACKED) {
              x = R.out_edge[q];
            } else {
              const int l = R.out_link[q];
              x = make_int2(R.lto[l], R.cost[l]);
            }
            const int v = x.x, nd = du + x.y;
            const unsigned long long nk = dkey(hi, nd);
            if (nk < atomicMin(&node[v].key, nk)) {
              if (nd < T) {
                if (atomicExch(&node[v].q, round) != round) {
                  const int at = atomicAdd(&sh_nq[nxt], 1);
                  if (at < kNearCap) ns[at] = v;
                  else ng[at] = v;
                }
              } else if (atomicExch(&node[v].f, (int)ep) != (int)ep) {
                F[atomicAdd(&sh_nf, 1)] = v;
              }
            }
          }
        }
        __syncthreads();
        cur = nxt;
        b ^= 1;
      }
      // ---- every distance below T is final: done when all destinations are (without trips
      // the whole tree is asked for)
      bool open = t0 == t1;
      for (int k = t0 + tid; k < t1; k += bd) open = open || dval(node, R.dest[R.otrip_list[k]], hi) >= T;
      if (!__syncthreads_or(open)) break;
      // ---- split the far pile: smallest live distance opens the next bucket
      const int nf = sh_nf;
      if (nf == 0) break;
      if (tid == 0) {
        sh_min = INT_MAX;
        sh_nf2 = 0;
        sh_nq[0] = sh_nq[1] = sh_nq[2] = 0;
      }
      __syncthreads();
      int mine = INT_MAX;
      for (int k = tid; k < nf; k += bd) {
        const int dv = dval(node, F[k], hi);
        if (dv >= T && dv < mine) mine = dv;
      }
      mine = __reduce_min_sync(0xffffffffu, mine);
      if ((tid & 31) == 0 && mine != INT_MAX) atomicMin(&sh_min, mine);
      __syncthreads();
      const int mn = sh_min;
      if (mn == INT_MAX) break;
      const int Tprev = T;
      T = mn + R.delta;
      round++;
      cur = 0;
      b = 0;
      for (int k = tid; k < nf; k += bd) {
        const int v = F[k];
        const int dv = dval(node, v, hi);
        if (dv < Tprev) {
          node[v].f = 0;
        } else if (dv < T) {
          node[v].f = 0;
          node[v].q = round;
          const int at = atomicAdd(&sh_nq[0], 1);
          if (at < kNearCap) sh_q[0][at] = v;
          else Q[0][at] = v;
        } else {
          Fn[atomicAdd(&sh_nf2, 1)] = v;
        }
      }
      __syncthreads();
      if (tid == 0) sh_nf = sh_nf2;
      int* tf = F; F = Fn; Fn = tf;
      __syncthreads();
    }
    __syncthreads();
    // ---- canonical routes of the trips from o, a group of threads each; the path is noted
    // in the queue arrays (idle now) and copied, or walked again where it is longer than a
    // group's share of them
    const int grp = tid / kWalkLanes, gl = tid % kWalkLanes;
    const unsigned gm = ((1u << kWalkLanes) - 1u) << ((tid & 31) - gl);
    constexpr int kGroups = kRouteThreads / kWalkLanes;
    const int room = R.nn / (kGroups / 4);
    int* note = (grp & 2 ? (grp & 1 ? Fn : F) : Q[grp & 1]) + (size_t)(grp >> 2) * room;
    for (int k = t0 + grp; k < t1; k += kGroups) {
      const int i = R.otrip_list[k];
      const int d = R.dest[i];
      const int dd = dval(node, d, hi);
      int n = -1;
      if (dd != INT_MAX)
        n = walk_back<PACKED>(R, node, hi, o, d, dd, [&](int j, int link) {
          if (R.flow) atomicAdd(&R.flow[link], 1u);
          else if (j < room) note[j] = link;
        });
      if (n < 0) {
        if (gl == 0) {
          atomicOr(&R.ctl->err, dd == INT_MAX ? kErrUnreach : kErrRoute);
          atomicExch(&R.ctl->err_info, i);
          if (!R.flow) {
            R.roff[i] = 0;
            R.rlen[i] = 0;
          }
        }
        continue;
      }
      if (R.flow) continue;   // all-or-nothing: the path is counted, not stored
      unsigned long long off = 0;
      if (gl == 0) {
        off = atomicAdd(&R.ctl->route_cursor, (unsigned long long)n);
        R.rlen[i] = n;
        R.roff[i] = off + (unsigned long long)n > R.cap ? 0 : (int)off;
      }
      off = __shfl_sync(gm, off, (tid & 31) - gl);
      if (off + (unsigned long long)n > R.cap) continue;   // the host grows the store to route_cursor and reruns
      if (n <= room) {
        __syncwarp(gm);
        for (int j = gl; j < n; j += kWalkLanes) R.routes[off + (unsigned)(n - 1 - j)] = note[j];
        __syncwarp(gm);   // read before the next trip's walk writes
      } else {
        walk_back<PACKED>(R, node, hi, o, d, dd, [&](int j, int link) { R.routes[off + (unsigned)(n - 1 - j)] = link; });
      }
    }
  }
  if (tid == 0) R.cta_round[blockIdx.x] = round;
}

void launch_route(const RouteDev& R, int n_cta, cudaStream_t s) {
  if (R.out_edge) k_sssp_route<true><<<n_cta, kRouteThreads, 0, s>>>(R);
  else k_sssp_route<false><<<n_cta, kRouteThreads, 0, s>>>(R);
}

// first link of every trip's route (departure-queue keys)
__global__ void k_first_links(const int32_t* roff, const int32_t* routes, int n, int32_t* out) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) out[i] = routes[roff[i]];
}

void launch_first_links(const int32_t* roff, const int32_t* routes, int n, int32_t* out, cudaStream_t s) {
  int grid = (n + 255) / 256;
  if (grid > 4096) grid = 4096;
  if (grid < 1) grid = 1;
  k_first_links<<<grid, 256, 0, s>>>(roff, routes, n, out);
}

// route of every trip copied to its new offset (compaction of the route store)
__global__ void k_compact_routes(const int32_t* roff, const int32_t* rlen, const int32_t* src,
                                 const int32_t* new_off, int32_t* dst, int n) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const int32_t* a = src + roff[i];
    int32_t* b = dst + new_off[i];
    for (int k = 0; k < rlen[i]; k++) b[k] = a[k];
  }
}

void launch_compact_routes(const int32_t* roff, const int32_t* rlen, const int32_t* src, const int32_t* new_off,
                           int32_t* dst, int n, cudaStream_t s) {
  int grid = (n + 255) / 256;
  if (grid > 4096) grid = 4096;
  if (grid < 1) grid = 1;
  k_compact_routes<<<grid, 256, 0, s>>>(roff, rlen, src, new_off, dst, n);
}

}  // namespace gbt
