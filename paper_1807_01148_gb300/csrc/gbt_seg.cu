// Kernels of the link-segment step (gbt_seg.cuh), the conversion between the two forms of
// the state, the readers of this form and the host side of its layout.
//
// Sorted form: buffer A (unsorted next state, lane counts), sorted every step.  Segment
// form: records in per-link segments.  The segment form is laid out from the sorted one
// (count, scan, scatter, rank, place) whenever a state was loaded, and written back to
// buffer A for checkpoints and for whatever reads that.
#include <algorithm>
#include <vector>

#include "gbt_observe.cuh"
#include "gbt_seg.cuh"

namespace gbt {

// On a network of few groups the next kernel of the step is let in as soon as this one runs:
// the SMs have room for its blocks, which then wait for this kernel's end with their start-up
// behind them.  (On a large network they would take the room of running blocks.)
__device__ __forceinline__ void griddep_next(const SegDev& d) {
  if (!d.packed) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// Bound by the latency of its dependent loads (range and slot arrays, front record and link
// record, rear record of the next lane; a quarter of metro, 527,500 vehicles: 22.7 cycles per
// instruction on loads, DRAM at 24%): six blocks of 40 registers per SM.
template <bool TYPES, bool TAPE>
__global__ void __launch_bounds__(256, 6) k_seg_front(SegDev d) {
  griddep_wait();
  griddep_next(d);
  if (seg_stopped(d)) return;
  seg_front<TYPES, TAPE>(d, (int)d.ctl->t);
}

// The lists of the next kPackSteps steps.  Packed in the front phase of every step they cost as
// much as the idle lanes that they save (metro, 2.11M vehicles: 253 us per step against 247 in
// the sorted form); kept for 8 steps, 241.
__global__ void __launch_bounds__(256) k_seg_pack(SegDev d) {
  griddep_wait();
  if (seg_stopped(d)) return;
  __shared__ SegPack packs[8];
  seg_pack_all(d, packs, (int)d.ctl->t);
}

// Bound by instruction issue and latency together (a quarter of metro, 527,500 vehicles: 52 warp
// instructions per vehicle at 17.9 active threads, 41% of issue slots; per instruction 2.8 cycles of
// fixed latency, 2.5 at barriers, 2.4 on loads).  Three blocks of 80 registers measured better than
// four of 64, whose spills miss the little L1 that the staging areas leave: metro, 2.11M vehicles,
// 4 steps 1,110 -> 1,077 us; 64 grids, 10 steps 670 -> 645; two blocks: 1,269 and 743.
template <bool OUT, bool TYPES, bool TAPE>
__global__ void __launch_bounds__(kSegThreads, 3) k_seg_move(SegDev d) {
  griddep_wait();
  griddep_next(d);
  if (seg_stopped(d)) return;
  extern __shared__ __align__(16) unsigned char seg_smem[];
  seg_move<OUT, TYPES, TAPE>(d, seg_smem, (int)d.ctl->tm);
}

// Sec. 6.4 per-edge sample of the state at step t (see ph_edge_sample): one thread per link
// over its segment.  After the front phase, which may stop the step (Ctl::grow): a step that
// does not take place now is sampled when it does.
__device__ __forceinline__ void seg_edge_sample(const SegDev& d, long long t) {
  if (t % d.samp_every != 0) return;
  const long long k = t / d.samp_every;
  const long long w = k / d.samp_per;
  const bool closes = (k % d.samp_per) == d.samp_per - 1;
  const long long k0 = d.ctl->samp_k0;
  const long long from = w * d.samp_per > k0 ? w * d.samp_per : k0;
  const double taken = (double)(k - from + 1);
  GRID_STRIDE(e, d.n_links) {
    const LinkRec L = d.links[e];
    const int g = d.lslot[e];
    const uint32_t last = d.rng[g + L.lanes - 1];
    const int n = rng_start(last) + rng_count(last);
    const VehRec* r = d.rec + d.lane_seg[g].x;
    double vs = 0.0;
    for (int q = 0; q < n; q++) vs += (double)r[q].v;
    const double cap = ((double)L.len * (double)L.lanes) / ((double)d.vlen + (double)d.cls[L.cls].s0);
    const double u = d.acc_u[e] + (double)n / cap;
    const double sp = d.acc_s[e] + (n > 0 ? vs / (double)n : (double)L.v0);
    if (closes) {
      const size_t o = (size_t)w * (size_t)d.n_links + (size_t)e;
      d.out_u[o] = u / taken;
      d.out_s[o] = sp / taken;
      d.acc_u[e] = 0.0;
      d.acc_s[e] = 0.0;
    } else {
      d.acc_u[e] = u;
      d.acc_s[e] = sp;
    }
  }
  if (closes && blockIdx.x == 0 && threadIdx.x == 0) d.out_n[w] = (int32_t)(k - from + 1);
}

__global__ void k_seg_edge_sample(SegDev d) {
  griddep_wait();
  if (seg_stopped(d)) return;
  seg_edge_sample(d, d.ctl->t);
}

// ------------------------------------------------------------------ persistent step
// All steps in one cooperative launch: two grid barriers per step, and one more where the lists
// are packed or the links sampled.
template <bool OUT, bool TYPES>
__device__ __forceinline__ void seg_persistent(const SegDev& d, GridSync* gs, int n_steps, long long limit,
                                               unsigned char* smem) {
  int* err = &d.ctl->err;
  const int t0 = (int)*(volatile long long*)&d.ctl->t;
  for (int step = 0; step < n_steps; step++) {
    const int t = t0 + step;
    if (d.packed && step % kPackSteps == 0) {
      seg_pack_all(d, reinterpret_cast<SegPack*>(smem), t);
      if (!grid_barrier(gs, err, limit)) return;
    }
    seg_front<TYPES, false>(d, t);
    if (!grid_barrier(gs, err, limit)) return;
    // set before the barrier, the same for every block (one thread asks: see step_timed_out)
    if (__syncthreads_or(threadIdx.x == 0 && *(volatile int*)&d.ctl->grow)) return;
    if (d.acc_u && t % d.samp_every == 0) {   // the move phase changes what it reads
      seg_edge_sample(d, t);
      if (!grid_barrier(gs, err, limit)) return;
    }
    seg_move<OUT, TYPES, false>(d, smem, t);
    if (!grid_barrier(gs, err, limit)) return;
  }
}

__global__ void __launch_bounds__(1024, 1) k_seg_persistent(SegDev d, GridSync* gs, int n_steps, long long limit) {
  extern __shared__ __align__(16) unsigned char seg_smem[];
  if (*(volatile int*)&d.ctl->grow) return;
  const bool out = d.emis || d.tt_sum;
  if (d.vtype) {
    if (out) seg_persistent<true, true>(d, gs, n_steps, limit, seg_smem);
    else seg_persistent<false, true>(d, gs, n_steps, limit, seg_smem);
  } else {
    if (out) seg_persistent<true, false>(d, gs, n_steps, limit, seg_smem);
    else seg_persistent<false, false>(d, gs, n_steps, limit, seg_smem);
  }
}

static size_t seg_persistent_smem(int threads) {
  return std::max<size_t>(kSegSmemBytes, (size_t)(threads / 32) * kSegWarpBytes);
}

cudaError_t launch_seg_persistent(const SegDev& d, GridSync* gs, int blocks, int threads, int n_steps, long long limit,
                                  cudaStream_t s) {
  SegDev dd = d;
  void* args[] = {&dd, &gs, &n_steps, &limit};
  return cudaLaunchCooperativeKernel((const void*)k_seg_persistent, dim3(blocks), dim3(threads), args,
                                     seg_persistent_smem(threads), s);
}

// Whether `per_sm` blocks of the persistent kernel are co-resident on an SM.
bool seg_persistent_fits(int threads, int per_sm) {
  int nb = 0;
  const size_t smem = seg_persistent_smem(threads);
  if (cudaFuncSetAttribute(k_seg_persistent, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)seg_persistent_smem(1024)) != cudaSuccess ||
      cudaFuncSetAttribute(k_seg_persistent, cudaFuncAttributePreferredSharedMemoryCarveout,
                           cudaSharedmemCarveoutMaxShared) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_seg_persistent, threads, smem) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return nb >= per_sm;
}

// ------------------------------------------------------------------ between the forms
// Static lane records from the link records and class parameters (after creation, and
// whenever the class parameters change).
__global__ void k_seg_lane_stat(SegDev d, LaneStat* out, uint32_t* info_out, int32_t* to) {
  GRID_STRIDE(lg, d.n_lanes) {
    const int e = d.lane_link[lg];
    const LinkRec L = d.links[e];
    const ClassPar P = d.cls[L.cls];
    const int lane = lg - L.lane_base, g = d.lslot[e] + lane;
    const unsigned info = (unsigned)lane | (unsigned)(L.lanes - 1) << 3 | (unsigned)L.ctrl << 6 |
                          (unsigned)L.cls << 8 | (unsigned)L.in_index << 16 | (unsigned)L.n_in << 24;
    out[g] = LaneStat{L.len, L.v0, P.T, P.s0, P.a, P.sab2, info, e};
    info_out[g] = info;
    to[g] = L.to;
  }
}

void launch_seg_lane_stat(const SegDev& d, int grid, cudaStream_t s) {
  k_seg_lane_stat<<<grid, 256, 0, s>>>(d, const_cast<LaneStat*>(d.lstat), const_cast<uint32_t*>(d.sinfo),
                                      const_cast<int32_t*>(d.slot_to));
}

// the last lane change of a vehicle rides in the high bits of its movement class while the
// sorted form is laid out
__global__ void k_seg_mark(SegDev d) {
  const int nA = d.ctl->nA;
  GRID_STRIDE(s, nA) {
    const int c = d.adec[s];
    d.A.mv[s] = (uint8_t)((d.A.mv[s] & 3) | (c > 0 ? 1 : c < 0 ? 2 : 0) << 2);
  }
}

__global__ void k_seg_unmark(SegDev d) {
  const int nA = d.ctl->nA;
  GRID_STRIDE(s, nA) d.A.mv[s] &= 3;
}

// Place the sorted vehicles into the segments (the fit is checked first: a state that does
// not fit sets Ctl::grow and is laid out again in larger segments).
__global__ void k_seg_place_lanes(SegDev d) {
  GRID_STRIDE(g, d.n_slots) {
    const uint32_t info = d.sinfo[g];
    int next = INT_MAX;
    uint32_t r = 0;
    if ((info >> 6 & 3u) != (uint32_t)kCtrlPad) {
      const int e = d.lstat[g].link;
      const int lane = (int)(info & 7u), lanes = (int)(info >> 3 & 7u) + 1;
      const int lg0 = d.links[e].lane_base;
      const int start = d.lane_start[lg0 + lane] - d.lane_start[lg0];
      const int end = d.lane_start[lg0 + lane + 1] - d.lane_start[lg0];
      r = (uint32_t)(start & 0xffff) | (uint32_t)(end - start & 0x3fff) << 16;   // beyond these bits: grow is set
      if (lane == lanes - 1) {
        const int most = end + lanes;
        if (most > kSegBig) atomicMax(&d.ctl->grow, 2);
        else if (most > d.lane_seg[g].y) atomicMax(&d.ctl->grow, 1);
      }
      if (lane == 0) {
        const int hd = d.q_head[e];
        if (hd < d.q_end[e]) next = d.depart[d.q_items[hd]];
      }
    }
    d.rng[g] = r;
    d.qnext[g] = next;
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    const int t = (int)d.ctl->t;
    Ctl* c = d.ctl;
    for (int p = 0; p < 2; p++)
      c->n_bigl[p] = c->n_run[p] = c->add_run[p] = c->n_late[p] = 0;
    c->pk_run = c->pk_step = 0;
    c->pk_veh = c->nB;
    d.ctl->nact[(t + 1) & 1] = d.ctl->active_last;
  }
}

__global__ void k_seg_place(SegDev d) {
  if (d.ctl->grow) return;
  const int nB = d.ctl->nB;
  const int t = (int)d.ctl->t;
  GRID_STRIDE(p, nB) {
    const int lg = d.tg[p];   // lane id
    const int e = d.lane_link[lg];
    const LinkRec& L = d.links[e];
    const int lane = lg - L.lane_base, g = d.lslot[e] + lane;
    const int vid = d.B.vid[p], nxt = d.B.nxt[p], cur = d.B.cur[p];
    const float x = d.B.x[p], v = d.B.v[p];
    const unsigned rem = d.loop ? 0u : (unsigned)(d.rlen[vid] - 1 - cur);
    const VehRec r{x, v, vid, nxt, nxt >= 0 ? d.lnext[nxt].nlb : -1, d.roff[vid] + cur,
                   d.tau[mand_index(d.hseed[vid], cur)], (unsigned)lane | (unsigned)(d.B.mv[p] & 15) << 3 | rem << 7};
    seg_store(d.rec + d.lane_seg[g].x + (p - d.lane_start[L.lane_base]), r);
    if (p == d.lane_start[lg]) d.rear2[(size_t)(t & 1) * d.n_slots + g] = RearRec{x, v, vid, (unsigned)t + 1u};
    if (p + 1 == d.lane_start[lg + 1] && L.ctrl == kCtrlStop && nxt >= 0 && L.len - x <= d.stop_acq)
      atomicMin(&d.acq[L.to], epoch_key(t, rr_rank(L, t), lane));
  }
}

void launch_kernel(int k, const Dev& d, int grid, cudaStream_t s);
void launch_count(const Dev& d, int grid, cudaStream_t s);

// Buffer A -> segments.  The lane counts are made anew, so that it does not matter whether
// the counts of A are current.
cudaError_t launch_seg_import(const SegDev& d, int grid, cudaStream_t s) {
  cudaError_t e = cudaMemsetAsync(d.cnt, 0, (size_t)d.n_lanes * 4, s);
  if (e == cudaSuccess) e = cudaMemsetAsync(d.rear2, 0, (size_t)d.n_slots * 2 * sizeof(RearRec), s);
  if (e == cudaSuccess) e = cudaMemsetAsync(d.best2, 0xFF, (size_t)d.n_slots * 8, s);
  if (e == cudaSuccess) e = cudaMemsetAsync(d.listed, 0, (size_t)d.n_links * 4, s);
  if (e == cudaSuccess) e = cudaMemsetAsync(&d.ctl->grow, 0, sizeof(int), s);
  if (e != cudaSuccess) return e;
  k_seg_mark<<<grid, 256, 0, s>>>(d);
  launch_count(d, grid, s);
  for (int k = kKScanSum; k <= kKRank; k++) launch_kernel(k, d, grid, s);
  k_seg_place_lanes<<<grid, 256, 0, s>>>(d);
  k_seg_place<<<grid, 256, 0, s>>>(d);
  k_seg_unmark<<<grid, 256, 0, s>>>(d);
  return cudaGetLastError();
}

// Every vehicle of the segments, a group of lanes per warp: f(record, link).
template <typename F>
__device__ __forceinline__ void seg_for_each(const SegDev& d, F f) {
  const int wl = threadIdx.x & 31;
#pragma unroll 1
  GRID_STRIDE(g, d.n_slots) {
    const float4 B = reinterpret_cast<const float4*>(d.lstat + g)[1];
    const uint32_t rg = d.rng[g];
    const int e = __float_as_int(B.w);
    const int start = d.lane_seg[g].x + rng_start(rg), cnt = rng_count(rg);
    const int inc = warp_inclusive(cnt);
    const int pos = inc - cnt, n = __shfl_sync(0xffffffffu, inc, 31);
#pragma unroll 1
    for (int i0 = 0; i0 < n; i0 += 32) {
      const int i = i0 + wl;
      // lane of vehicle i: the number of lanes that end at or before it
      int j = 0;
#pragma unroll
      for (int b = 16; b > 0; b >>= 1) {
        const int q = __shfl_sync(0xffffffffu, inc, j + b - 1);
        if (q <= i) j += b;
      }
      const int s = __shfl_sync(0xffffffffu, start, j & 31), p = __shfl_sync(0xffffffffu, pos, j & 31);
      const int el = __shfl_sync(0xffffffffu, e, j & 31);
      if (i < n) f(seg_load(d.rec + s + (i - p)), el);
    }
  }
}

// Segments -> buffer A (slots in no particular order; its counts follow by k_count).
__global__ void k_seg_export(SegDev d) {
  if (blockIdx.x == 0 && threadIdx.x == 0) d.ctl->active_last = d.ctl->nact[((int)d.ctl->t + 1) & 1];
  seg_for_each(d, [&](const VehRec& r, int e) {
    const unsigned m = __activemask();
    const int wl = threadIdx.x & 31, lead = __ffs(m) - 1;
    int b = 0;
    if (wl == lead) b = atomicAdd(&d.ctl->nA, __popc(m));
    const int s = __shfl_sync(m, b, lead) + __popc(m & ((1u << wl) - 1u));
    d.A.x[s] = r.x;
    d.A.v[s] = r.v;
    d.A.vid[s] = r.vid;
    d.A.link[s] = e;
    d.A.nxt[s] = r.nxt;
    d.A.cur[s] = r.ri - d.roff[r.vid];
    d.A.lane[s] = (int)(r.meta & 7u);
    d.A.mv[s] = (uint8_t)(r.meta >> 3 & 3u);
    const unsigned c = r.meta >> 5 & 3u;
    d.adec[s] = (int8_t)(c == 1 ? 1 : c == 2 ? -1 : 0);
  });
}

cudaError_t launch_seg_export(const SegDev& d, int grid, cudaStream_t s) {
  cudaError_t e = cudaMemsetAsync(&d.ctl->nA, 0, sizeof(int), s);
  if (e == cudaSuccess) e = cudaMemsetAsync(d.cnt, 0, (size_t)d.n_lanes * 4, s);
  if (e != cudaSuccess) return e;
  k_seg_export<<<grid, 256, 0, s>>>(d);
  launch_count(d, grid, s);
  return cudaGetLastError();
}

// ------------------------------------------------------------------ readers
__global__ void k_seg_state_out(SegDev d, int32_t* link, int32_t* lane, int32_t* cursor, float* x, float* v,
                                int8_t* dec) {
  seg_for_each(d, [&](const VehRec& r, int e) {
    const int i = r.vid;
    if (link) link[i] = e;
    if (lane) lane[i] = (int)(r.meta & 7u);
    if (cursor) cursor[i] = r.ri - d.roff[i];
    if (x) x[i] = r.x;
    if (v) v[i] = r.v;
    const unsigned c = r.meta >> 5 & 3u;
    if (dec) dec[i] = (int8_t)(c == 1 ? 1 : c == 2 ? -1 : 0);
  });
}

void launch_seg_state_out(const SegDev& d, int grid, cudaStream_t s, int32_t* link, int32_t* lane, int32_t* cursor,
                          float* x, float* v, int8_t* dec) {
  k_seg_state_out<<<grid, 256, 0, s>>>(d, link, lane, cursor, x, v, dec);
}

// k_observe on the segments.
__global__ void k_seg_observe(SegDev d, const double* target, double* res, double* p_out) {
  double acc = 0.0;
  seg_for_each(d, [&](const VehRec& r, int) {
    const double p = prefix_len(d, r.vid, r.ri - d.roff[r.vid]) + (double)r.x;
    if (p_out) p_out[r.vid] = p;
    if (target) {
      const double q = p - target[r.vid];
      acc += q * q;
      res[r.vid] = q;
    }
  });
  GRID_STRIDE(vid, d.n_trips) {
    const uint8_t st = d.status[vid];
    if (st == kActive) continue;
    const double p = st == kArrived ? prefix_len(d, vid, d.rlen[vid]) : 0.0;
    if (p_out) p_out[vid] = p;
    if (target) {
      const double q = p - target[vid];
      acc += q * q;
      res[vid] = 0.0;
    }
  }
  if (target) {
    const double b = block_sum(acc);
    if (threadIdx.x == 0) atomicAdd(&d.ctl->loss, b);
  }
}

void launch_seg_observe(const SegDev& d, int grid, cudaStream_t s, const double* target, double* res, double* p_out) {
  k_seg_observe<<<grid, 256, 0, s>>>(d, target, res, p_out);
}

// ------------------------------------------------------------------ launch
template <typename... KArgs, typename... Args>
static void launch_pdl3(void (*kern)(KArgs...), int grid, int block, size_t smem, cudaStream_t s, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3((unsigned)block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, kern, args...);
}

template <typename K>
static int seg_move_blocks(K kern) {
  int nb = 0;
  if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSegSmemBytes) != cudaSuccess ||
      cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared) !=
          cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kern, kSegThreads, kSegSmemBytes) != cudaSuccess)
    return 0;
  return nb;
}

// Grids: one resident wave, or what the lanes and groups need.  Where the groups outnumber the
// warps of a resident move phase, their runs are packed (Dev::packed = those warps).
void seg_grids(SegDev& d, int sm_count) {
  int f[4] = {};
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&f[0], k_seg_front<false, false>, 256, 0);
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&f[1], k_seg_front<true, false>, 256, 0);
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&f[2], k_seg_front<false, true>, 256, 0);
  const int fneed = (d.n_slots + 255) / 256;
  for (int v = 0; v < 3; v++) d.seg_front_grid[v] = std::max(1, std::min(fneed, std::max(1, f[v]) * sm_count));
  const int m[5] = {seg_move_blocks(k_seg_move<false, false, false>), seg_move_blocks(k_seg_move<true, false, false>),
                    seg_move_blocks(k_seg_move<false, true, false>), seg_move_blocks(k_seg_move<true, true, false>),
                    seg_move_blocks(k_seg_move<false, false, true>)};
  const int warps = std::max(1, m[0]) * sm_count * kSegWarps;
  d.packed = d.n_slots / 32 > warps ? warps : 0;
  d.parts = std::max(1, std::min(8, warps / std::max(1, d.n_slots / 32)));
  for (int v = 0; v < 5; v++) d.seg_move_grid[v] = std::max(1, std::min(d.n_slots / 32 * d.parts, std::max(1, m[v]) * sm_count));
}

void launch_seg_front(const SegDev& d, cudaStream_t s) {
  if (d.tape) launch_pdl3(k_seg_front<false, true>, d.seg_front_grid[2], 256, 0, s, d);
  else if (d.vtype) launch_pdl3(k_seg_front<true, false>, d.seg_front_grid[1], 256, 0, s, d);
  else launch_pdl3(k_seg_front<false, false>, d.seg_front_grid[0], 256, 0, s, d);
}

void launch_seg_move(const SegDev& d, cudaStream_t s) {
  const bool out = d.emis || d.tt_sum;
  const int v = d.tape ? 4 : (out ? 1 : 0) + (d.vtype ? 2 : 0);
  const int grid = d.seg_move_grid[v];
  switch (v) {
    case 0: launch_pdl3(k_seg_move<false, false, false>, grid, kSegThreads, kSegSmemBytes, s, d); break;
    case 1: launch_pdl3(k_seg_move<true, false, false>, grid, kSegThreads, kSegSmemBytes, s, d); break;
    case 2: launch_pdl3(k_seg_move<false, true, false>, grid, kSegThreads, kSegSmemBytes, s, d); break;
    case 3: launch_pdl3(k_seg_move<true, true, false>, grid, kSegThreads, kSegSmemBytes, s, d); break;
    default: launch_pdl3(k_seg_move<false, false, true>, grid, kSegThreads, kSegSmemBytes, s, d); break;
  }
}

// Networks with packed runs: before the first step after the state was laid out, and at least
// every kPackSteps steps.
void launch_seg_pack(const SegDev& d, cudaStream_t s) {
  const int tile = 8 * kPackSlots;
  launch_pdl3(k_seg_pack, std::max(1, (d.n_slots + tile - 1) / tile), 256, 0, s, d);
}

void launch_seg_step(const SegDev& d, int grid, cudaStream_t s) {
  launch_seg_front(d, s);
  if (d.acc_u) launch_pdl3(k_seg_edge_sample, grid, 256, 0, s, d);
  launch_seg_move(d, s);
}

// The same step with an event after either phase; ms[0] front (with the packing and the edge sample), ms[1] move.
cudaError_t launch_seg_steps_timed(const SegDev& d, int grid, cudaStream_t s, int n, float* ms) {
  cudaEvent_t ev[3];
  for (int k = 0; k < 3; k++) {
    cudaError_t e = cudaEventCreate(&ev[k]);
    if (e != cudaSuccess) return e;
  }
  cudaError_t err = cudaSuccess;
  for (int it = 0; it < n && err == cudaSuccess; it++) {
    cudaEventRecord(ev[0], s);
    if (d.packed && it % kPackSteps == 0) launch_seg_pack(d, s);
    launch_seg_front(d, s);
    if (d.acc_u) launch_pdl3(k_seg_edge_sample, grid, 256, 0, s, d);
    cudaEventRecord(ev[1], s);
    launch_seg_move(d, s);
    cudaEventRecord(ev[2], s);
    err = cudaEventSynchronize(ev[2]);
    for (int k = 0; k < 2 && err == cudaSuccess; k++) {
      float q = 0.0f;
      err = cudaEventElapsedTime(&q, ev[k], ev[k + 1]);
      ms[k] += q;
    }
  }
  for (int k = 0; k < 3; k++) cudaEventDestroy(ev[k]);
  return err;
}

// Segment capacities: what a link's lanes hold bumper to bumper with the shortest vehicle,
// plus two vehicles per lane (the one a step may bring, and one of slack), and no more than
// all trips.  A state denser than that (overlapping vehicles) is laid out again in larger
// segments: at least twice the link's vehicles.
void seg_capacities(int n_links, const float* len, const uint8_t* lanes, int n_trips, float vlen_min,
                    const int32_t* now, std::vector<int32_t>& cap) {
  cap.resize((size_t)n_links);
  for (int e = 0; e < n_links; e++) {
    const double per = vlen_min > 0.0f ? (double)len[e] / (double)vlen_min : 1e9;
    double c = (std::min(per, 1e7) + 2.0) * lanes[e];
    c = std::min(c, (double)n_trips);
    if (now) c = std::max(c, 2.0 * now[e]);
    cap[e] = (int32_t)std::min(c, (double)kSegBig) + lanes[e];
  }
}

// Slots of the links' first lanes: whole consecutive links fill groups of kGroupLanes slots.
// Returns the number of slots.
int seg_slots(int n_links, const uint8_t* lanes, std::vector<int32_t>& lslot) {
  lslot.resize((size_t)n_links);
  int next = 0;
  for (int e = 0; e < n_links; e++) {
    if (next % kGroupLanes + lanes[e] > kGroupLanes) next = (next / kGroupLanes + 1) * kGroupLanes;
    lslot[e] = next;
    next += lanes[e];
  }
  return (next + kGroupLanes - 1) / kGroupLanes * kGroupLanes;
}

}  // namespace gbt
