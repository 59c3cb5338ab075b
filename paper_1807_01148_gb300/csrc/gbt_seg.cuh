// The step without a sort (link-segment form of the state).
//
// Every link owns a segment of 32-byte vehicle records and keeps its vehicles there in
// (lane, position, id) order.  A step is two phases:
//
// Lanes are numbered by slots: the lanes of whole consecutive links fill groups of 32, so
// that the lanes of a link are always threads of one warp.
//
//   front  one thread per lane: the lane's front vehicle, its acceleration behind the rearmost
//          vehicle of the next link's lane or the stop line, its admission bid and, for a
//          bidder, its record after crossing;
//   move   a warp per run (whole links, at most 32 lanes and about 90 vehicles: a part of a
//          group, or on large networks a list of links with something to do that is packed
//          anew every 8 steps): its vehicles staged in shared memory, own-lane Eq. 7,
//          lane-change decisions, conflicts, ballistic move; then the new order of the same
//          links is written in place.  Vehicles that won an admission are pulled by the
//          target lane (at most one per lane and step), departures are appended by the
//          first link's warp.
//
// The model admits at most one vehicle per lane and step, so a lane's new order is its
// stayers in their old order plus a few incoming vehicles (lane changers, one crossing or
// departing vehicle), each ranked by counting; a lane whose stayers are out of order
// (overlapping vehicles) is ranked by counting altogether.  Nothing else moves: no lane
// counts, scan, scatter or gather, and each vehicle is read and written once per step.
//
// Every decision reads the state at t only, so the result does not depend on the order in
// which warps run, and equals the sorted form's bit for bit.
#pragma once
#include <climits>

#include "gbt_rebuild.cuh"

namespace gbt {

// A warp stages up to kSegN vehicles; 8 warps of 6.8 KB let 4 blocks of 256 threads onto an SM
// (what a persistent launch may ask for; the kernel of its own takes 3).  A link with more vehicles is staged by a whole block
// (kSegBig of them in the same memory); one with still more stops the stepping in this form
// (Ctl::grow = 2) and the sorted form goes on.
constexpr int kSegN = 96, kSegBig = 1024;
constexpr int kSegThreads = 256, kSegWarps = kSegThreads / 32;
constexpr int kGroupLanes = 32;
// Links with something to do are packed into runs of at most 32 lanes and about this many
// vehicles (the rest of the staging area is for incoming ones).
constexpr int kRunVeh = 84;
constexpr int kCtrlPad = 3;   // control of an empty slot
constexpr int kSegFrontFl = 1, kSegHolder = 2, kSegCand = 4, kSegClosed = 8;   // kFlag* plus the signal's state
constexpr int kSegWon = 1 << 30;
constexpr uint8_t kGone = 255, kNew = 254;

template <int N_, int NL_, typename IDX>
struct SegSmemT {
  static constexpr int N = N_, NL = NL_;
  using Idx = IDX;
  float4 la[NL_], lb[NL_];   // len, v0, T, s0 | a, sab2, info, link
  float x[N_], v[N_], a[N_], om[N_], at[N_], tau[N_];
  int32_t vid[N_], nxt[N_], nlb[N_], ri[N_];
  uint32_t meta[N_];         // VehRec::meta >> 3, the lane change settled in this step in its bits 2-3
  int32_t pos[NL_ + 1];      // first staged index of the lane
  int32_t gs[NL_];           // its slot
  int32_t to[NL_];           // its link's head node (stop-controlled links)
  int32_t sg[NL_];           // its link's segment
  int32_t wb[NL_];           // record index minus staged index; later the first record of the new order
  int32_t cn[NL_];           // front's acceleration; later the new count
  int32_t ic[NL_];           // incoming vehicles
  int32_t in0[NL_];          // first of them in the list (chained in at[]), -1 without one
  int32_t ff[NL_];           // front's flags
  uint32_t stay[(N_ + 31) / 32];
  int32_t sb[(N_ + 31) / 32];
  int32_t n, m, n_list, n_in;
  uint32_t bad;
  IDX list[N_];
  uint8_t jo[N_], fl[N_], it[N_];
  uint8_t nz[NL_];
};
using SegSmem = SegSmemT<kSegN, kGroupLanes, uint8_t>;
using SegSmemBig = SegSmemT<kSegBig, 8, uint16_t>;
constexpr size_t kSegWarpBytes = (sizeof(SegSmem) + 15) / 16 * 16;
static_assert(sizeof(SegSmemBig) <= kSegWarps * kSegWarpBytes, "a block's staging areas hold a big link");
constexpr size_t kSegSmemBytes = kSegWarps * kSegWarpBytes;
static_assert(4 * (kSegSmemBytes + 1024) <= 228 * 1024, "four blocks per SM");

// A link whose vehicles (and one more per lane, and one departure) do not fit a warp's
// staging area.
__device__ __forceinline__ bool seg_big(int vehicles, int lanes) { return vehicles + lanes >= kSegN; }

// Fields of SegDev::rng.
__device__ __forceinline__ int rng_start(uint32_t r) { return (int)(r & 0xffffu); }
__device__ __forceinline__ int rng_count(uint32_t r) { return (int)(r >> 16 & 0x3fffu); }

__device__ __forceinline__ bool seg_stopped(const SegDev& d) {
  const int err = d.ctl->err, grow = d.ctl->grow;   // (cached: see step_timed_out)
  return (err & kErrTimeout) != 0 || grow != 0;
}

__device__ __forceinline__ VehRec seg_load(const VehRec* p) {
  const float4 a = reinterpret_cast<const float4*>(p)[0], b = reinterpret_cast<const float4*>(p)[1];
  return VehRec{a.x, a.y, __float_as_int(a.z), __float_as_int(a.w), __float_as_int(b.x), __float_as_int(b.y), b.z,
                __float_as_uint(b.w)};
}

__device__ __forceinline__ void seg_store(VehRec* p, const VehRec& r) {
  reinterpret_cast<float4*>(p)[0] = make_float4(r.x, r.v, __int_as_float(r.vid), __int_as_float(r.nxt));
  reinterpret_cast<float4*>(p)[1] =
      make_float4(__int_as_float(r.nlb), __int_as_float(r.ri), r.tau, __uint_as_float(r.meta));
}

// Admission key of step t: epoch, round-robin rank, lane; the in-link index tells the
// target lane where its winner comes from.
__device__ __forceinline__ unsigned long long seg_key(int t, int rr, int lane, int in_index) {
  return ((unsigned long long)(0xFFFFFFFEu - (unsigned)t) << 32) |
         (unsigned long long)((unsigned)rr << 16 | (unsigned)lane << 8 | (unsigned)in_index);
}

__device__ __forceinline__ int ctrl_of(unsigned info) { return (int)(info >> 6 & 3u); }

// Round-robin rank of a link at its head node in step t (rr_rank on the slot's info).
__device__ __forceinline__ int seg_rr(unsigned info, int t) {
  const int n = (int)(info >> 24);
  return ((int)(info >> 16 & 255u) + n - t % n) % n;
}

// Movement class from a link onto the next one (turn_class on their headings).
__device__ __forceinline__ int seg_turn(const LinkNext& a, const LinkNext& b) {
  return turn_class(0, 0, a.hx, a.hy, (long long)a.hx + b.hx, (long long)a.hy + b.hy);
}

// Eq. 7 parameters of trip vid on a lane (types: its vehicle's).
template <bool TYPES>
__device__ __forceinline__ void seg_par(const SegDev& d, const float4& A, const float4& B, int vid, ClassPar& P,
                                        float& v0) {
  if (TYPES) {
    const int ty = d.vtype[vid];
    P = d.cls_ty[(int)(__float_as_uint(B.z) >> 8 & 255u) * d.n_vty + ty];
    v0 = fminf(A.y, d.vty_vmax[ty]);
  } else {
    P = ClassPar{B.x, B.y, A.z, A.w};
    v0 = A.y;
  }
}

// acc_front on the records of this form: om is the vehicle's free-road term, nlb its next
// link's lanes, rin / tag the rear records of step t.
template <bool TYPES>
__device__ __forceinline__ float seg_acc_front(const SegDev& d, const RearRec* rin, unsigned tag, float len,
                                               const ClassPar& P, float om, int vid, int nlb, int lane, float x,
                                               float v, bool closed, TapeForm* f, int* gt = nullptr,
                                               bool* lead = nullptr, float* room = nullptr) {
  const float a_free = P.a * (om - 0.0f);
  if (nlb < 0) {
    if (f) *f = TapeForm{-1, 0.0f, 0.0f, kFormFree, 0, 0, 0};
    return a_free;
  }
  const int lm = nlb & 7;
  const int g = (nlb >> 3) + (lane < lm ? lane : lm);
  const RearRec r = rin[g];
  const bool has = r.tag == tag && r.vid != vid;
  if (gt) *gt = g;
  if (lead) *lead = has;
  float a1 = a_free;
  if (f) *f = TapeForm{-1, 0.0f, 0.0f, kFormFree, 0, 0, 0};
  if (has) {
    const float len_r = veh_len<TYPES>(d, r.vid);
    if (room) *room = r.x - len_r;
    const float s = ((len - x) + r.x) - len_r;
    a1 = idm_om(P, om, d.s_min, s, v, r.v);
    if (f) *f = TapeForm{r.vid, s, r.v, kFormNext, 0, 0, 0};
  }
  if (closed) {
    const float s2 = len - x;
    const float a2 = idm_om(P, om, d.s_min, s2, v, 0.0f);
    if (a2 < a1) {
      if (f) *f = TapeForm{-1, s2, 0.0f, kFormStop, 0, 0, 0};
      return a2;
    }
  }
  return a1;
}

__device__ __forceinline__ int warp_inclusive(int v) {
  const int wl = threadIdx.x & 31;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, v, o);
    if (wl >= o) v += y;
  }
  return v;
}

// End of the run of whole links that begins at lane ja of the warp's run: as many links as
// stay within `most`, at least one.  inc: inclusive sums over the lanes of what counts;
// lane, lanes: the thread's lane within its link; in: the thread holds a lane.
__device__ __forceinline__ int seg_run_end(int ja, int inc, int lane, int lanes, bool in, int most) {
  const int wl = threadIdx.x & 31;
  const int upto = __shfl_sync(0xffffffffu, inc, (wl + lanes - 1 - lane) & 31);   // with the whole link
  const int base = ja ? __shfl_sync(0xffffffffu, inc, ja - 1) : 0;
  const int fit = __popc(__ballot_sync(0xffffffffu, in && wl >= ja && upto - base <= most));
  const int one = __shfl_sync(0xffffffffu, lanes, ja);
  return ja + (fit > one ? fit : one);
}

// ------------------------------------------------------------------ front phase
// A block's staging of seg_pack: kPackSlots slots per warp.
constexpr int kPackSlots = 256;
struct SegPack {
  int32_t v[kPackSlots];            // vehicles up to and with the active lane
  int32_t slot[kPackSlots];
  uint16_t first[kPackSlots + 1];   // first active lane of each run
  uint8_t last[kPackSlots];         // the active lane is its link's last one
  int32_t n_run, run0;
};

// For one lane of every link with vehicles: lists it when it is left to a whole block, and
// stops the step where a segment may run full (the step brings a link at most one vehicle per
// lane; they must fit, or the move phase does not run).
__device__ __forceinline__ void seg_check_link(const SegDev& d, int g, int lanes, int total, int cap, int t) {
  if (total + lanes > kSegBig || total + lanes > cap)
    atomicMax(&d.ctl->grow, total + lanes > kSegBig ? 2 : 1);
  if (seg_big(total, lanes)) d.big_links[atomicAdd(&d.ctl->n_bigl[t & 1], 1)] = d.lstat[g].link;
}

// Packs the links that have something to do (vehicles, a departure due before the next
// packing) into runs of whole links, kPackSlots slots per warp of the block: the active lanes
// are compacted, then cut greedily into at most 32 lanes and `most` vehicles.  On a sparse
// network a run gathers the few busy links of many slots.  The lists hold for kPackSteps
// steps: links that empty stay in them, links that are entered in between are added by the
// move phase.  One allocation of runs per block: thousands of additions to one counter would
// outlast the rest.
constexpr int kPackHorizon = 2 * kPackSteps;

__device__ __forceinline__ void seg_pack(const SegDev& d, SegPack* packs, int base, int most, int t) {
  const int wl = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  SegPack& P = packs[warp];
  base += warp * kPackSlots;
  int n = 0, veh = 0;
#pragma unroll 2
  for (int b = base; b < base + kPackSlots && b < d.n_slots; b += 32) {
    const int g = b + wl;
    const uint32_t r = d.rng[g], info = d.sinfo[g];
    const int q = d.qnext[g];
    const int lane = (int)(info & 7u), lanes = (int)(info >> 3 & 7u) + 1;
    const bool lane_ok = (info >> 6 & 3u) != (unsigned)kCtrlPad;
    const int cnt = rng_count(r), end = rng_start(r) + cnt;
    const int total = __shfl_sync(0xffffffffu, end, (wl + lanes - 1 - lane) & 31);
    const bool due = __shfl_sync(0xffffffffu, q <= t + kPackHorizon ? 1 : 0, (wl - lane) & 31) != 0;
    const bool act = lane_ok && (total > 0 || due);
    if (act && lane == 0) d.listed[d.lstat[g].link] = t + 1;
    const unsigned m = __ballot_sync(0xffffffffu, act);
    const int inc = warp_inclusive(act ? cnt : 0);
    if (act) {
      const int i = n + __popc(m & ((1u << wl) - 1u));
      P.v[i] = veh + inc;
      P.slot[i] = g;
      P.last[i] = lane == lanes - 1 ? 1 : 0;
    }
    n += __popc(m);
    veh += __shfl_sync(0xffffffffu, inc, 31);
    if (r >> 30) d.rng[g] = r & 0x3fffffffu;   // a block's mark: the lists may leave the link out (see seg_move)
  }
  __syncwarp();
  // as many links as stay within the limits, at least one (a link has at most 8 lanes, so
  // one ends in the window of 32)
  int k = 0, before = 0;
#pragma unroll 1
  for (int s = 0; s < n; k++) {
    const int q = s + wl;
    const int v = q < n ? P.v[q] : 0;
    const bool end = q < n && P.last[q];
    const unsigned mf = __ballot_sync(0xffffffffu, end && v - before <= most);
    const unsigned ml = __ballot_sync(0xffffffffu, end);
    const int e = mf ? 31 - __clz(mf) : __ffs(ml) - 1;
    if (wl == 0) P.first[k] = (uint16_t)s;
    before = __shfl_sync(0xffffffffu, v, e);
    s += e + 1;
  }
  if (wl == 0) {
    P.first[k] = (uint16_t)n;
    P.n_run = k;
  }
  __syncthreads();
  if (warp == 0) {
    const int ki = wl < nw ? packs[wl].n_run : 0;
    const int kk = warp_inclusive(ki);
    int b = 0;
    if (wl == 31 && kk) b = atomicAdd(&d.ctl->pk_run, kk);
    const int run0 = __shfl_sync(0xffffffffu, b, 31);
    if (wl < nw) packs[wl].run0 = run0 + kk - ki;
  }
  __syncthreads();
#pragma unroll 1
  for (int q = 0; q < k; q++) {
    const int i = P.first[q] + wl;
    d.tl[(size_t)(P.run0 + q) * 32 + wl] = i < P.first[q + 1] ? P.slot[i] : -1;
  }
  __syncthreads();
}

// The whole packing of step t, by all blocks.
__device__ __forceinline__ void seg_pack_all(const SegDev& d, SegPack* packs, int t) {
  if (blockIdx.x == 0 && threadIdx.x == 0) d.ctl->pk_step = t + 1;
  // about one run per resident warp when there are few vehicles
  const int most = max(32, min(kRunVeh, max(d.ctl->nact[(t + 1) & 1], d.ctl->pk_veh) / d.packed));
  const int step = (int)(blockDim.x >> 5) * kPackSlots;
#pragma unroll 1
  for (int k = blockIdx.x; k * step < d.n_slots; k += gridDim.x) seg_pack(d, packs, k * step, most, t);
}

// One thread per lane (packed: of the listed links) settles the lane's front; level by level
// the loads are: slot arrays, front record and link record, rear record of the next lane.
template <bool TYPES, bool TAPE>
__device__ __forceinline__ void seg_front(const SegDev& d, int t) {
  const RearRec* rin = d.rear2 + (size_t)(t & 1) * d.n_slots;
  const unsigned tag = (unsigned)t + 1u;
  int n = d.n_slots, pk = 0;
  if (d.packed) {
    const int p = (t + 1) & 1;
    const Ctl* c = d.ctl;
    pk = c->pk_step;
    n = 32 * (pk == t + 1 ? c->pk_run : c->n_run[p] + c->add_run[p]);
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    const int q = t & 1, p = q ^ 1;
    Ctl* c = d.ctl;
    c->tm = t;
    c->nact[q] = 0;
    c->n_run[q] = n >> 5;
    c->add_run[q] = 0;
    c->n_bigl[p] = c->n_late[p] = 0;
  }
  const int wl = threadIdx.x & 31;
#pragma unroll 1
  GRID_STRIDE(k, n) {
    const int g = d.packed ? d.tl[k] : k;
    if (g < 0) continue;
    const uint32_t r = d.rng[g];
    const int cnt = rng_count(r), end = rng_start(r) + cnt;
    // (the slot's other arrays are loaded along with its range)
    const float4* ls = reinterpret_cast<const float4*>(d.lstat + g);
    const uint32_t info = d.sinfo[g];
    const int2 sg = d.lane_seg[g];
    const float4 B = ls[1], A = ls[0];
    const int lane = (int)(info & 7u), lanes = (int)(info >> 3 & 7u) + 1, ctrl = ctrl_of(info);
    if (d.packed) {
      if (lane == lanes - 1 && end > 0) seg_check_link(d, g, lanes, end, sg.y, t);
    } else {
      const int total = __shfl_sync(0xffffffffu, end, (wl + lanes - 1 - lane) & 31);
      if (lane == lanes - 1 && total > 0) seg_check_link(d, g, lanes, total, sg.y, t);
      const bool big = seg_big(total, lanes);
      // parts of about the same number of vehicles, 16 at least
      const int w = big ? 0 : cnt, all = __reduce_add_sync(0xffffffffu, w);
      unsigned long long cuts = ~0ull;
      if (all > 16 && d.parts > 1) {
        const int most = max(16, (all + d.parts - 1) / d.parts);
        const bool in = ctrl != kCtrlPad;
        const int inc = warp_inclusive(w);
        cuts = 0;
        int ja = 0;
#pragma unroll 1
        for (int p = 1; p < 8; p++) {
          if (ja < 32) ja = min(32, seg_run_end(ja, inc, lane, lanes, in, most));
          cuts |= (unsigned long long)(p < d.parts ? ja : 255) << (8 * p - 8);
        }
      }
      if (wl == 0) d.cuts[g >> 5] = cuts;
    }
    if (cnt == 0) continue;
    const VehRec f = seg_load(d.rec + sg.x + end - 1);
    const int e = __float_as_int(B.w);
    LinkRec L;
    if (ctrl != kCtrlNone) L = d.links[e];
    ClassPar P;
    float v0;
    seg_par<TYPES>(d, A, B, f.vid, P, v0);
    bool hold = false, red = false;
    if (ctrl == kCtrlStop) hold = is_holder(d, L, t, f.vid, lane, true);
    if (ctrl == kCtrlSignal) red = !signal_green(L, t * d.dt_ds);
    const bool closed = f.nxt >= 0 && (ctrl == kCtrlStop ? !hold : red);
    const float om = free_term(f.v, v0);
    int gt = 0;
    bool lead = false;
    float room = 0.0f;
    TapeForm tf;
    const float a = seg_acc_front<TYPES>(d, rin, tag, A.x, P, om, f.vid, f.nlb, lane, f.x, f.v, closed,
                                         TAPE ? &tf : nullptr, &gt, &lead, &room);
    if (TAPE) {
      TapeRec* r = tape_slot(d, t, f.vid);
      r->lead = tf.lead;
      r->kind = tf.kind;
      r->s = tf.s;
      r->vl = tf.vl;
    }
    float xo, vo;
    ballistic(f.x, f.v, a, d.dt, d.hdt2, xo, vo);
    int fl = (hold ? kSegHolder : 0) | (red ? kSegClosed : 0);
    if (f.nxt >= 0 && !closed && xo >= A.x && (!lead || (xo - A.x) <= room)) {
      fl |= kSegCand;
      atomicMin(&d.best2[gt], seg_key(t, seg_rr(info, t), lane, (int)(info >> 16 & 255u)));
      // an unlisted link is noted for the vehicle that may enter it
      if (d.packed && d.listed[f.nxt] != pk && atomicExch(&d.listed[f.nxt], pk) != pk)
        d.late[atomicAdd(&d.ctl->n_late[t & 1], 1)] = f.nxt;
      // the record after crossing, pulled by the target lane if this bid wins (a bidding
      // front never changes lanes: its own-lane move reaches the link end)
      const int off = d.roff[f.vid];
      int nri = f.ri + 1, nnxt = -1;
      unsigned rem = f.meta >> 7;
      if (d.loop) {
        const int len = d.rlen[f.vid];
        nri = off + (f.ri - off + 1) % len;
        nnxt = d.routes[off + (nri - off + 1) % len];
      } else if (--rem >= 1) {
        nnxt = d.routes[nri + 1];
      }
      const LinkNext X = d.lnext[f.nxt];
      const LinkNext X2 = nnxt >= 0 ? d.lnext[nnxt] : LinkNext{0, 0, -1, 0};
      const unsigned mc = (unsigned)(nnxt >= 0 ? seg_turn(X, X2) : kTurnEnd);
      const int lm = f.nlb & 7;
      const unsigned m = (unsigned)(lane < lm ? lane : lm);
      seg_store(d.cr2 + g, VehRec{xo - A.x, vo, f.vid, nnxt, X2.nlb, nri,
                                  d.tau[mand_index(d.hseed[f.vid], nri - off)], m | mc << 3 | rem << 7});
    }
    d.fres[g] = make_int2(__float_as_int(a), fl | gt << 4);
  }
}

// ------------------------------------------------------------------ move phase
// The lane of a thread (the first 32 threads of a team hold a lane each).
struct SegLane {
  bool on;               // part of the run
  bool ext;              // a crossing vehicle comes in (its record: cr2[src])
  bool due;              // first lane of a link whose departure queue is due
  bool done;             // a whole block has written the lane in this step
  int g, to, src, cnt, start, seg;
  int2 fr;
  float4 la, lb;
};

template <typename SM>
__device__ __forceinline__ int seg_stayers_before(const SM& S, int i) {
  return S.sb[i >> 5] + __popc(S.stay[i >> 5] & ((1u << (i & 31)) - 1u));
}

// First staged index q in [s0, s1) whose (x, vid) exceeds (x, vid).
template <typename SM>
__device__ __forceinline__ int seg_upper(const SM& S, int s0, int s1, float x, int vid) {
  int lo = s0, hi = s1;
#pragma unroll 1
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    const float xm = S.x[mid];
    if (xm > x || (xm == x && S.vid[mid] > vid)) hi = mid;
    else lo = mid + 1;
  }
  return lo;
}

// Lane-change decision of the vehicle at staged index i from the state at t: MOBIL
// incentive (Kesting, Treiber & Helbing 2007) for discretionary changes, mandatory changes
// toward the lanes of the next movement once within the drawn switch distance, gap
// acceptance = positive lead and lag gaps and both the changer's and the new follower's
// accelerations >= -b_safe.
template <typename SM, bool TYPES, bool TAPE>
__device__ __forceinline__ void seg_decide(const SegDev& d, SM& S, int i, const RearRec* rin, unsigned tag) {
  const int j = S.jo[i];
  const float4 A = S.la[j], B = S.lb[j];
  const unsigned info = __float_as_uint(B.z);
  const int lane = (int)(info & 7u), lanes = (int)(info >> 3 & 7u) + 1;
  const float x = S.x[i], v = S.v[i], om = S.om[i];
  const int vid = S.vid[i], nlb = S.nlb[i];
  ClassPar P;
  float v0;
  seg_par<TYPES>(d, A, B, vid, P, v0);
  const int M = lane_mask((int)(S.meta[i] & 3u), lanes);
  int dirs[2];
  int nd = 0;
  bool mand = false;
  if ((M >> lane) & 1) {
    if (lane + 1 < lanes && ((M >> (lane + 1)) & 1)) dirs[nd++] = 1;
    if (lane >= 1 && ((M >> (lane - 1)) & 1)) dirs[nd++] = -1;
  } else {
    const int ms = __ffs(M) - 1;
    const int dd = ms > lane ? 1 : -1;
    const int ncross = ms > lane ? ms - lane : lane - ms;
    const float thr = (d.lam * (float)ncross) * S.tau[i];
    mand = A.x - x <= thr;
    dirs[nd++] = dd;
  }
  const int flp = S.fl[i];
  const bool front = (flp & kSegFrontFl) != 0;
  const bool stop = (info >> 6 & 3u) == (unsigned)kCtrlStop;
  const bool red = (S.ff[j] & kSegClosed) != 0;
  const bool closed_self = nlb >= 0 && (stop ? !(flp & kSegHolder) : red);
  int chosen = 0;
  float chosen_inc = 0.0f, chosen_at = 0.0f;
  float dno = 0.0f;
  bool dno_known = false;
#pragma unroll 1
  for (int k = 0; k < nd; k++) {
    const int dd = dirs[k];
    const int s0 = S.pos[j + dd], s1 = S.pos[j + dd + 1];
    const int up = seg_upper(S, s0, s1, x, vid);
    const int Ln = up < s1 ? up : -1;
    const int Fn = up > s0 ? up - 1 : -1;
    float ac;
    TapeForm cf;
    if (Ln >= 0) {
      const float sl = (S.x[Ln] - x) - (TYPES ? veh_len<true>(d, S.vid[Ln]) : d.vlen);
      if (!(sl > 0.0f)) continue;
      ac = idm_om(P, om, d.s_min, sl, v, S.v[Ln]);
      if (TAPE) cf = TapeForm{S.vid[Ln], sl, S.v[Ln], kFormLead, 0, 0, 0};
    } else {
      ac = seg_acc_front<TYPES>(d, rin, tag, A.x, P, om, vid, nlb, lane + dd, x, v, closed_self,
                                TAPE ? &cf : nullptr);
    }
    if (!(ac >= -d.mbsafe)) continue;
    float an = 0.0f;
    if (Fn >= 0) {
      const float sg = (x - S.x[Fn]) - veh_len<TYPES>(d, vid);
      if (!(sg > 0.0f)) continue;
      ClassPar PF = P;
      float v0F = v0;
      if (TYPES) seg_par<true>(d, A, B, S.vid[Fn], PF, v0F);
      an = idm_om(PF, S.om[Fn], d.s_min, sg, S.v[Fn], v);
      if (!(an >= -d.mbsafe)) continue;
    }
    if (mand) {
      chosen = dd;
      chosen_at = ac;
      if (TAPE) d.tform[vid] = cf;
      break;
    }
    const float dc = ac - S.a[i];
    const float dn = Fn >= 0 ? an - S.a[Fn] : 0.0f;
    if (!dno_known) {   // the old follower's gain does not depend on the direction
      dno_known = true;
      if (i > S.pos[j]) {   // old follower F = i - 1
        const int F = i - 1;
        ClassPar PF = P;
        float v0F = v0;
        const int vF = S.vid[F];
        if (TYPES) seg_par<true>(d, A, B, vF, PF, v0F);
        float ao;
        if (!front) {
          const float sF = (S.x[i + 1] - S.x[F]) - (TYPES ? veh_len<true>(d, S.vid[i + 1]) : d.vlen);
          ao = idm_om(PF, S.om[F], d.s_min, sF, S.v[F], S.v[i + 1]);
        } else {
          const int nF = S.nlb[F];
          const bool holdF = (S.fl[F] & kSegHolder) != 0;
          const bool closedF = nF >= 0 && (stop ? !holdF : red);
          ao = seg_acc_front<TYPES>(d, rin, tag, A.x, PF, S.om[F], vF, nF, lane, S.x[F], S.v[F], closedF, nullptr);
        }
        dno = ao - S.a[F];
      }
    }
    float inc = dc + d.mp * (dn + dno);
    if (dd < 0) inc = inc + d.mbias;
    if (!(inc > d.mathr)) continue;
    if (chosen == 0 || inc > chosen_inc) {
      chosen = dd;
      chosen_inc = inc;
      chosen_at = ac;
      if (TAPE) d.tform[vid] = cf;
    }
  }
  S.it[i] = (uint8_t)(chosen > 0 ? 1 : chosen < 0 ? 2 : 0);
  S.at[i] = chosen_at;
}

// Whether the lane change of staged vehicle i to lane j2 is cancelled by a lower-id
// vehicle changing into the same lane less than (vehicle length + s0) away (the longer of
// the two lengths with vehicle types).  Such vehicles sit in the lanes next to j2; each
// lane is sorted, so the scan covers a window around x that holds every vehicle that can
// pass the test.
template <typename SM, bool TYPES>
__device__ __forceinline__ bool seg_cancelled(const SegDev& d, const SM& S, int i, int j, int j2, int first, int last) {
  const float s0c = S.la[j].w;
  const float x = S.x[i];
  const int vid = S.vid[i];
  const float len_self = TYPES ? veh_len<true>(d, vid) : d.vlen;
  const float thr = d.vlen + s0c;
  const float win = 2.0f * ((TYPES ? d.vlen_max : d.vlen) + s0c) + 1.0f;
#pragma unroll 1
  for (int side = -1; side <= 1; side += 2) {
    const int js = j2 + side;
    if (js < first || js > last) continue;
    const int s1 = S.pos[js + 1];
    int lo = S.pos[js], hi = s1;
#pragma unroll 1
    while (lo < hi) {
      const int mid = (lo + hi) >> 1;
      if (S.x[mid] < x - win) lo = mid + 1;
      else hi = mid;
    }
    const int code = side < 0 ? 1 : 2;   // a vehicle of lane j2 - 1 changing left, of j2 + 1 changing right
#pragma unroll 1
    for (int q = lo; q < s1 && S.x[q] <= x + win; q++) {
      if (S.it[q] != code || S.vid[q] >= vid) continue;
      const float thr_q = TYPES ? fmaxf(len_self, veh_len<true>(d, S.vid[q])) + s0c : thr;
      if (fabsf(S.x[q] - x) < thr_q) return true;
    }
  }
  return false;
}

// The head of a link's queue of due trips enters at x = 0, v = 0 in the allowed lane with
// the largest rear space (ties to the lowest lane) that received no vehicle from upstream
// in this step, if that space is at least s0 + vehicle length.  Called by the thread of the
// link's first lane j0.
template <typename SM, bool OUT, bool TYPES>
__device__ __noinline__ void seg_depart(const SegDev& d, SM& S, int n, int j0, int t, int* count) {
  const float4 B = S.lb[j0];
  const int e = __float_as_int(B.w);
  const int lanes = (int)(__float_as_uint(B.z) >> 3 & 7u) + 1;
  const int hd = d.q_head[e];
  const int h = d.q_items[hd];
  const int off = d.roff[h], len = d.rlen[h];
  const int e2 = len >= 2 ? d.routes[off + 1] : (d.loop ? d.routes[off] : -1);
  const LinkNext X2 = e2 >= 0 ? d.lnext[e2] : LinkNext{0, 0, -1, 0};
  const int mc = e2 >= 0 ? seg_turn(d.lnext[e], X2) : kTurnEnd;
  const int M = lane_mask(mc, lanes);
  int bl = -1;
  float brs = 0.0f;
#pragma unroll 1
  for (int l = 0; l < lanes; l++) {
    if (!((M >> l) & 1)) continue;
    if (S.ic[j0 + l]) continue;   // a crossing vehicle
    const int p = S.pos[j0 + l];
    const float rs = S.pos[j0 + l + 1] > p ? S.x[p] - veh_len<TYPES>(d, S.vid[p]) : INFINITY;
    if (bl < 0 || rs > brs) {
      bl = l;
      brs = rs;
    }
  }
  if (bl < 0) return;
  const float need = S.la[j0].w + veh_len<TYPES>(d, h);
  if (!(brs >= need)) return;
  const int i = n + atomicAdd(&S.m, 1);
  S.x[i] = 0.0f;
  S.v[i] = 0.0f;
  S.vid[i] = h;
  S.nxt[i] = e2;
  S.nlb[i] = X2.nlb;
  S.ri[i] = off;
  S.tau[i] = d.tau[mand_index(d.hseed[h], 0)];
  S.meta[i] = (unsigned)mc | (d.loop ? 0u : (unsigned)(len - 1) << 4);
  S.jo[i] = kNew;
  S.it[i] = (uint8_t)(j0 + bl);
  S.ic[j0 + bl] = 1;
  d.status[h] = kActive;
  d.ins_step[h] = t;
  if (OUT && d.enter) d.enter[h] = t;
  d.q_head[e] = hd + 1;
  d.qnext[S.gs[j0]] = hd + 1 < d.q_end[e] ? d.depart[d.q_items[hd + 1]] : INT_MAX;
  atomicAdd(&count[3], 1);
}

// One run: the vehicles of whole links (lanes with ln.on, one per thread), at most S.N of
// them with the incoming ones.  NT = 32: the team is a warp; 0: the whole block.  count:
// vehicles advanced, lane-change decisions, arrivals, departures (shared memory).  What a
// thread knows of its lane goes to shared memory at once: kept in registers over the whole
// run it spilled, and next to the staging areas the L1 is too small to hold the spills.
template <int NT, typename SM, bool OUT, bool TYPES, bool TAPE>
__device__ __forceinline__ void seg_run(const SegDev& d, SM& S, const SegLane& ln, int nl, int t,
                                        int* count) {
  const int tid = NT == 32 ? (int)(threadIdx.x & 31) : (int)threadIdx.x;
  const int nt = NT == 32 ? 32 : (int)blockDim.x;
  const int wl = threadIdx.x & 31;
  const unsigned lt = (1u << wl) - 1u;
  auto sync = [&]() {
    if (NT == 32) __syncwarp();
    else __syncthreads();
  };
  const RearRec* rin = d.rear2 + (size_t)(t & 1) * d.n_slots;
  const unsigned tag = (unsigned)t + 1u;
  auto stage = [&](int i, int j, const VehRec& r) {
    S.x[i] = r.x;
    S.v[i] = r.v;
    S.vid[i] = r.vid;
    S.nxt[i] = r.nxt;
    S.nlb[i] = r.nlb;
    S.ri[i] = r.ri;
    S.tau[i] = r.tau;
    S.meta[i] = r.meta >> 3 & ~12u;
    S.jo[i] = (uint8_t)j;
  };
  // ---- lane tables, crossing vehicles
  int n = 0, my_pos = 0;
  const bool on = ln.on, due = ln.on && ln.due;
  const int c = ln.on ? ln.cnt : 0;
  unsigned nzm = 0;
  if (NT == 32 || tid < 32) {
    const int inc = warp_inclusive(c);
    my_pos = inc - c;
    n = __shfl_sync(0xffffffffu, inc, 31);
    nzm = __ballot_sync(0xffffffffu, c > 0);
    const unsigned xm = __ballot_sync(0xffffffffu, ln.on && ln.ext);
    if (tid < nl) {
      S.pos[tid] = my_pos;
      S.gs[tid] = ln.g;
      S.to[tid] = ln.to;
      S.sg[tid] = ln.seg;
      S.wb[tid] = ln.seg + ln.start - my_pos;
      S.la[tid] = ln.la;
      S.lb[tid] = ln.lb;
      S.cn[tid] = ln.fr.x;
      S.ff[tid] = ln.fr.y;
      S.ic[tid] = ln.on && ln.ext ? 1 : 0;
      S.in0[tid] = -1;
      if (c > 0) S.nz[__popc(nzm & lt)] = (uint8_t)tid;
    }
    if (tid == 0) {
      S.pos[nl] = n;
      S.n = n;
      S.m = __popc(xm);
      S.n_list = 0;
      S.n_in = 0;
      S.bad = 0;
      atomicAdd(&count[0], n);
    }
    if (ln.on && ln.ext) {
      const int i = n + __popc(xm & lt);
      stage(i, kNew, seg_load(d.cr2 + ln.src));
      S.it[i] = (uint8_t)tid;
    }
  }
  sync();
  if (NT != 32) n = S.n;
  // ---- vehicles
  if (NT == 32) {
    // two windows of 32 vehicles at a time, so that their loads overlap
#pragma unroll 1
    for (int i0 = 0; i0 < n; i0 += 64) {
      VehRec r[2];
      int jj[2];
#pragma unroll
      for (int u = 0; u < 2; u++) {
        // lanes that begin inside this window, as a mask: the lane of vehicle i is the last
        // non-empty one that begins at or before it
        const int iu = i0 + 32 * u, i = iu + wl;
        const bool here = c > 0 && my_pos >= iu && my_pos < iu + 32;
        const unsigned hm = __reduce_or_sync(0xffffffffu, here ? 1u << (my_pos - iu) : 0u);
        const int hb = __popc(__ballot_sync(0xffffffffu, c > 0 && my_pos < iu));
        if (i < n) {
          jj[u] = S.nz[hb + __popc(hm & (lt | 1u << wl)) - 1];
          r[u] = seg_load(d.rec + S.wb[jj[u]] + i);
        }
      }
#pragma unroll
      for (int u = 0; u < 2; u++)
        if (i0 + 32 * u + wl < n) stage(i0 + 32 * u + wl, jj[u], r[u]);
    }
  } else {
#pragma unroll 1
    for (int i = tid; i < n; i += nt) {
      int j = 0;
#pragma unroll 1
      for (int k = 1; k < nl; k++) j += S.pos[k] <= i ? 1 : 0;
      stage(i, j, seg_load(d.rec + S.wb[j] + i));
    }
  }
  sync();
  // ---- own-lane step, lane-change candidates
#pragma unroll 1
  for (int i0 = tid & ~31; i0 < n; i0 += nt) {
    const int i = i0 + wl;
    bool el = false;
    if (i < n) {
      const int j = S.jo[i];
      const float4 A = S.la[j], B = S.lb[j];
      const unsigned info = __float_as_uint(B.z);
      const float x = S.x[i], v = S.v[i];
      const int vid = S.vid[i];
      ClassPar P;
      float v0;
      seg_par<TYPES>(d, A, B, vid, P, v0);
      const float om = free_term(v, v0);
      float a;
      int fl;
      if (i + 1 == S.pos[j + 1]) {   // the front: settled by the front phase
        a = __int_as_float(S.cn[j]);
        fl = (S.ff[j] & (kSegHolder | kSegCand)) | kSegFrontFl;
      } else {
        const int vl = S.vid[i + 1];
        const float sg = (S.x[i + 1] - x) - (TYPES ? veh_len<true>(d, vl) : d.vlen);
        a = idm_om(P, om, d.s_min, sg, v, S.v[i + 1]);
        // a stop-sign holder acquired the node within stop_acquire_m of the line and has
        // not moved back since: farther vehicles cannot hold it
        fl = 0;
        if ((info >> 6 & 3u) == (unsigned)kCtrlStop && A.x - x <= d.stop_acq &&
            d.holder[S.to[j]] == vid)
          fl = kSegHolder;
        if (TAPE) {
          TapeRec* r = tape_slot(d, t, vid);
          r->lead = vl;
          r->kind = kFormLead;
          r->s = sg;
          r->vl = S.v[i + 1];
        }
      }
      float xo, vo;
      ballistic(x, v, a, d.dt, d.hdt2, xo, vo);
      el = (info & 0x38u) != 0 && x >= d.zone && xo < A.x - d.zone;
      S.a[i] = a;
      S.om[i] = om;
      S.fl[i] = (uint8_t)fl;
      S.it[i] = 0;
    }
    const unsigned m = __ballot_sync(0xffffffffu, el);
    if (m) {
      int b = 0;
      if (wl == 0) b = atomicAdd(&S.n_list, __popc(m));
      b = __shfl_sync(0xffffffffu, b, 0);
      if (el) S.list[b + __popc(m & lt)] = (typename SM::Idx)i;
    }
  }
  if ((NT == 32 || tid < 32) && due) seg_depart<SM, OUT, TYPES>(d, S, n, tid, t, count);
  sync();
  // ---- lane-change decisions
  const int nc = S.n_list;
  if (tid == 0) atomicAdd(&count[1], nc);
#pragma unroll 1
  for (int q = tid; q < nc; q += nt) seg_decide<SM, TYPES, TAPE>(d, S, S.list[q], rin, tag);
  sync();
  // ---- simultaneous changes: the change that stands, in bits 4-5 of fl
#pragma unroll 1
  for (int q = tid; q < nc; q += nt) {
    const int i = S.list[q];
    const int code = S.it[i];
    if (code == 0) continue;
    const int j = S.jo[i], j2 = code == 1 ? j + 1 : j - 1;
    const unsigned info = __float_as_uint(S.lb[j].z);
    const int first = j - (int)(info & 7u), last = first + (int)(info >> 3 & 7u);
    if (!seg_cancelled<SM, TYPES>(d, S, i, j, j2, first, last)) S.fl[i] |= (uint8_t)(code << 4);
  }
  sync();
  // ---- final move; it[] becomes the new lane (kGone: left the link)
#pragma unroll 1
  for (int i = tid; i < n; i += nt) {
    const int j = S.jo[i];
    const int fl = S.fl[i], code = fl >> 4;
    const float len = S.la[j].x;
    const float x = S.x[i], v = S.v[i];
    const int vid = S.vid[i];
    const float acc = code ? S.at[i] : S.a[i];
    float nx, nv;
    ballistic(x, v, acc, d.dt, d.hdt2, nx, nv);
    if (OUT && d.emis) {
      // Eq. 8-9 at this step's speed and acceleration, over dt
      double2 q = d.emis[vid];
      q.x += (double)(fuel_rate(v, acc) * d.dt);
      q.y += (double)(co_rate(v) * d.dt);
      d.emis[vid] = q;
    }
    const int e = __float_as_int(S.lb[j].w);
    TapeRec* rec = nullptr;
    if (TAPE) {
      rec = tape_slot(d, t, vid);
      if (code) {
        const TapeForm cf = d.tform[vid];
        rec->lead = cf.lead;
        rec->kind = cf.kind;
        rec->s = cf.s;
        rec->vl = cf.vl;
      }
      rec->link = e;
      rec->v = v;
      rec->a = acc;
      rec->branch = (v + acc * d.dt >= 0.0f) ? kBrNormal : kBrStop;
      rec->crossed = 0;
      rec->valid = 1;
    }
    int nj = code == 0 ? j : code == 1 ? j + 1 : j - 1;
    bool crossed = false, arrived = false;
    if (nx >= len) {
      if (S.nxt[i] < 0) {
        arrived = true;
        nj = kGone;
        if (TAPE) rec->branch = kBrArrive;
        if (OUT && d.tt_sum) note_exit(d, vid, e, t);
        d.status[vid] = kArrived;
        d.arr_step[vid] = t;
        atomicAdd(&count[2], 1);
      } else if ((fl & kSegCand) && (S.ff[j] & kSegWon)) {
        crossed = true;
        nj = kGone;
        if (TAPE) rec->crossed = 1;
        if (OUT && d.tt_sum) {
          note_exit(d, vid, e, t);
          d.enter[vid] = t;
        }
      } else {
        nx = len;
        nv = 0.0f;
        if (TAPE) rec->branch = kBrClamp;
      }
    }
    if ((fl & kSegHolder) && !arrived) d.holder[S.to[j]] = crossed ? -1 : vid;
    S.x[i] = nx;
    S.v[i] = nv;
    S.it[i] = (uint8_t)nj;
    S.meta[i] |= (unsigned)code << 2;
  }
  sync();
  // ---- the new order: stayers as a bit mask, the incoming ones as a list
  const int ne = n + S.m;
#pragma unroll 1
  for (int i0 = tid & ~31; i0 < ne; i0 += nt) {
    const int i = i0 + wl;
    int nj = kGone;
    bool st = false, in = false;
    if (i < ne) {
      nj = S.it[i];
      st = nj == S.jo[i];
      in = nj != kGone && !st;
    }
    const unsigned ms = __ballot_sync(0xffffffffu, st), mi = __ballot_sync(0xffffffffu, in);
    if (wl == 0) S.stay[i0 >> 5] = ms;
    if (mi) {
      int b = 0;
      if (wl == 0) b = atomicAdd(&S.n_in, __popc(mi));
      b = __shfl_sync(0xffffffffu, b, 0);
      if (in) {
        const int k = b + __popc(mi & lt);
        S.list[k] = (typename SM::Idx)i;
        reinterpret_cast<int*>(S.at)[k] = atomicExch(&S.in0[nj], k);
        if (S.jo[i] != kNew) atomicAdd(&S.ic[nj], 1);   // the others were counted as they came
      }
    }
  }
  sync();
  const int nw = (ne + 31) >> 5;
  if (NT == 32 || tid < 32) {
    int before = 0;
#pragma unroll 1
    for (int w0 = 0; w0 < nw; w0 += 32) {
      const int w = w0 + wl;
      const int pc = w < nw ? __popc(S.stay[w]) : 0;
      int inc = pc;
#pragma unroll
      for (int o = 1; o < (NT == 32 ? 4 : 32); o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, inc, o);
        if (wl >= o) inc += y;
      }
      if (w < nw) S.sb[w] = before + inc - pc;
      before += __shfl_sync(0xffffffffu, inc, 31);
    }
  }
  sync();
  const int K = S.n_in;
  if (NT == 32 || tid < 32) {
    // new counts and starts of the lanes
    int cnt = 0, lane = 0;
    if (tid < nl && on) {
      const int p0 = S.pos[tid], p1 = S.pos[tid + 1];
      if (p1 > p0) {
        const int last = p1 - 1;
        cnt = seg_stayers_before(S, last) + (int)(S.stay[last >> 5] >> (last & 31) & 1u) - seg_stayers_before(S, p0);
      }
      cnt += S.ic[tid];
      lane = (int)(__float_as_uint(S.lb[tid].z) & 7u);
    }
    const int inc = warp_inclusive(cnt);
    const int first = __shfl_sync(0xffffffffu, inc - cnt, (wl - lane) & 31);
    if (tid < nl && on) {
      const int s = inc - cnt - first;
      S.wb[tid] = S.sg[tid] + s;
      S.cn[tid] = cnt;
      d.rng[S.gs[tid]] = (uint32_t)s | (uint32_t)cnt << 16 | (NT == 32 ? 0u : 2u + (unsigned)(t & 1)) << 30;
    }
  }
  // a stayer not below the next stayer of its lane: the whole lane is ranked by counting
#pragma unroll 1
  for (int i = tid; i < n; i += nt) {
    if (S.it[i] != S.jo[i]) continue;
    const int j = S.jo[i], p1 = S.pos[j + 1];
    int q = i + 1;
#pragma unroll 1
    while (q < p1 && S.it[q] != j) q++;
    if (q < p1 && !key_less(S.x[i], S.vid[i], S.x[q], S.vid[q])) atomicOr(&S.bad, 1u << j);
  }
  sync();
  // ranks, in om[]
  const unsigned bad = S.bad;
  int* rank = reinterpret_cast<int*>(S.om);
#pragma unroll 1
  for (int i0 = tid & ~31; i0 < n; i0 += nt) {
    const int i = i0 + wl;
    const bool st = i < n && S.it[i] == S.jo[i];
    int j = -1, vid = 0, below = 0;
    float x = 0.0f;
    if (st) {
      j = S.jo[i];
      x = S.x[i];
      vid = S.vid[i];
      if (bad >> j & 1u) {
#pragma unroll 1
        for (int q = S.pos[j]; q < S.pos[j + 1]; q++)
          below += S.it[q] == j && key_less(S.x[q], S.vid[q], x, vid) ? 1 : 0;
      } else {
        below = seg_stayers_before(S, i) - seg_stayers_before(S, S.pos[j]);
      }
    }
    if (st) {
#pragma unroll 1
      for (int k = S.in0[j]; k >= 0; k = reinterpret_cast<const int*>(S.at)[k]) {
        const int q = S.list[k];
        below += key_less(x, vid, S.x[q], S.vid[q]) ? 0 : 1;
      }
      rank[i] = below;
    }
  }
  // an incoming vehicle: a warp counts the stayers and the other incoming ones below it
#pragma unroll 1
  for (int k = tid >> 5; k < K; k += nt >> 5) {
    const int i = S.list[k], j = S.it[i];
    const float x = S.x[i];
    const int vid = S.vid[i];
    int r = 0;
#pragma unroll 1
    for (int q = S.pos[j] + wl; q - wl < S.pos[j + 1]; q += 32)
      r += __popc(__ballot_sync(0xffffffffu, q < S.pos[j + 1] && S.it[q] == j && key_less(S.x[q], S.vid[q], x, vid)));
#pragma unroll 1
    for (int k2 = S.in0[j]; k2 >= 0; k2 = reinterpret_cast<const int*>(S.at)[k2])
      r += key_less(S.x[S.list[k2]], S.vid[S.list[k2]], x, vid) ? 1 : 0;
    if (wl == 0) rank[i] = r;
  }
  sync();
  // the records of the new order, the lanes' rearmost vehicles and the bids for stop signs
  const unsigned tag_out = tag + 1u;
  RearRec* rout = d.rear2 + (size_t)((t + 1) & 1) * d.n_slots;
#pragma unroll 1
  for (int i = tid; i < ne; i += nt) {
    const int j = S.it[i];
    if (j == kGone) continue;
    const int r = rank[i];
    const unsigned info = __float_as_uint(S.lb[j].z);
    const VehRec o{S.x[i],   S.v[i],   S.vid[i], S.nxt[i],
                   S.nlb[i], S.ri[i],  S.tau[i], (info & 7u) | S.meta[i] << 3};
    seg_store(d.rec + S.wb[j] + r, o);
    if (r == 0) rout[S.gs[j]] = RearRec{o.x, o.v, o.vid, tag_out};
    if ((info >> 6 & 3u) == (unsigned)kCtrlStop && r == S.cn[j] - 1 && o.nxt >= 0 && S.la[j].x - o.x <= d.stop_acq) {
      // the new front bids for the node at its link's end for the next step (read only
      // while the node is free then)
      atomicMin(&d.acq[S.to[j]], epoch_key(t + 1, seg_rr(info, t + 1), (int)(info & 7u)));
    }
  }
  sync();   // the staging area is free
}

// What the thread of slot g needs (g < 0: none).
__device__ __forceinline__ SegLane seg_lane(const SegDev& d, int g, int t) {
  SegLane ln;
  ln.on = ln.ext = ln.due = ln.done = false;
  ln.g = g;
  ln.to = ln.src = ln.cnt = ln.start = ln.seg = 0;
  ln.fr = make_int2(0, 0);
  ln.la = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
  ln.lb = make_float4(0.0f, 0.0f, 0.0f, __int_as_float(-1));
  if (g < 0) return ln;
  ln.on = true;
  // one level of loads that depend on nothing
  const uint32_t r = d.rng[g];
  const unsigned long long bk = d.best2[g];
  const int q = d.qnext[g], tail = d.stail[g];
  const float4* ls = reinterpret_cast<const float4*>(d.lstat + g);
  ln.lb = ls[1];
  ln.la = ls[0];
  ln.seg = d.lane_seg[g].x;
  ln.to = d.slot_to[g];
  ln.fr = d.fres[g];
  ln.start = rng_start(r);
  ln.cnt = rng_count(r);
  ln.done = (r >> 30) == 2u + (unsigned)(t & 1);
  const unsigned info = __float_as_uint(ln.lb.z);
  if (ln.cnt == 0) ln.fr.y = 0;   // an empty lane's record is an older step's
  if (epoch_current(bk, t)) {
    ln.ext = true;
    ln.src = d.nin_slot[tail + (int)((unsigned)bk & 255u)] + (int)((unsigned)bk >> 8 & 255u);
  }
  if (ln.fr.y & kSegCand) {
    const unsigned long long k = d.best2[ln.fr.y >> 4];
    if (epoch_current(k, t) && ((unsigned)k & 0xFFFFu) == ((info & 7u) << 8 | (info >> 16 & 255u)))
      ln.fr.y |= kSegWon;
  }
  ln.fr.y &= kSegWon | 15;
  ln.due = q <= t;
  return ln;
}

// An unlisted link (no vehicles, no departures) that crossing vehicles may have entered, by
// one thread: at most one vehicle per lane, already in order.
__device__ __forceinline__ void seg_enter(const SegDev& d, int e, int t) {
  const int g0 = d.lslot[e];
  const int seg = d.lane_seg[g0].x, tail = d.stail[g0], to = d.slot_to[g0];
  const unsigned info = d.sinfo[g0];
  const int lanes = (int)(info >> 3 & 7u) + 1;
  RearRec* rout = d.rear2 + (size_t)((t + 1) & 1) * d.n_slots;
  int n = 0;
#pragma unroll 1
  for (int l = 0; l < lanes; l++) {
    const unsigned long long k = d.best2[g0 + l];
    const bool in = epoch_current(k, t);
    d.rng[g0 + l] = (uint32_t)n | (in ? 1u << 16 : 0u);
    if (!in) continue;
    const VehRec r = seg_load(d.cr2 + d.nin_slot[tail + (int)((unsigned)k & 255u)] + (int)((unsigned)k >> 8 & 255u));
    seg_store(d.rec + seg + n, r);
    rout[g0 + l] = RearRec{r.x, r.v, r.vid, (unsigned)t + 2u};
    n++;
    if ((info >> 6 & 3u) == (unsigned)kCtrlStop && r.nxt >= 0 && d.lstat[g0].len - r.x <= d.stop_acq)
      atomicMin(&d.acq[to], epoch_key(t + 1, seg_rr(info, t + 1), l));
  }
}

// The links noted in this step, 32 per warp: their vehicles, and their place in the lists of
// the steps until the next packing.
__device__ __forceinline__ void seg_late(const SegDev& d, int first, int t) {
  const int wl = threadIdx.x & 31, q = t & 1;
  const bool in = first + wl < d.ctl->n_late[q];
  int lanes = 0, g0 = 0;
  if (in) {
    const int e = d.late[first + wl];
    g0 = d.lslot[e];
    lanes = (int)(d.sinfo[g0] >> 3 & 7u) + 1;
    seg_enter(d, e, t);
  }
  const int inc = warp_inclusive(lanes);
  const int n = __popc(__ballot_sync(0xffffffffu, in));
#pragma unroll 1
  for (int s = 0, before = 0; s < n;) {
    const int e = s + __popc(__ballot_sync(0xffffffffu, in && wl >= s && inc - before <= 32)) - 1;
    const int to = __shfl_sync(0xffffffffu, inc, e);
    int run = 0;
    if (wl == 0) run = d.ctl->n_run[q] + atomicAdd(&d.ctl->add_run[q], 1);
    int32_t* row = d.tl + (size_t)__shfl_sync(0xffffffffu, run, 0) * 32;
    if (wl >= to - before) row[wl] = -1;
    if (wl >= s && wl <= e)
#pragma unroll 1
      for (int l = 0; l < lanes; l++) row[inc - lanes - before + l] = g0 + l;
    before = to;
    s = e + 1;
  }
}

// The move phase of step t.  First the links left to whole blocks, then the runs, one per
// warp (one whose incoming vehicles take it beyond the staging area in several passes), then
// the unlisted links that vehicles enter, 32 per warp.  Units of one run per warp are dealt to
// the blocks after the big links (a unit each); few runs spread over all blocks.
template <bool OUT, bool TYPES, bool TAPE>
__device__ __forceinline__ void seg_move(const SegDev& d, unsigned char* smem, int t) {
  const int warp = threadIdx.x >> 5, wl = threadIdx.x & 31;
  __shared__ int s_cn[4];
  if (threadIdx.x < 4) s_cn[threadIdx.x] = 0;
  __syncthreads();
  const int nbig = d.ctl->n_bigl[t & 1];
#pragma unroll 1
  for (int b = blockIdx.x; b < nbig; b += gridDim.x) {
    const int e = d.big_links[b];
    const int g0 = d.lslot[e], nl = d.links[e].lanes;
    const SegLane ln = seg_lane(d, (int)threadIdx.x < nl ? g0 + (int)threadIdx.x : -1, t);
    seg_run<0, SegSmemBig, OUT, TYPES, TAPE>(d, *reinterpret_cast<SegSmemBig*>(smem), ln, nl, t, s_cn);
  }
  SegSmem& S = *reinterpret_cast<SegSmem*>(smem + (size_t)warp * kSegWarpBytes);
  const int n_grp = d.n_slots >> 5;
  const int n_run = d.packed ? d.ctl->n_run[t & 1] : n_grp * d.parts;
  const int n_late = d.packed ? d.ctl->n_late[t & 1] : 0;
  const int n_all = n_run + (n_late + 31) / 32;
  const int per = min((int)(blockDim.x >> 5), (n_all + (int)gridDim.x - 1) / (int)gridDim.x);
  const int b0 = (int)((blockIdx.x + gridDim.x - (unsigned)nbig % gridDim.x) % gridDim.x);
#pragma unroll 1
  for (int k = b0 * per + warp; warp < per && k < n_all; k += gridDim.x * per) {
    if (k >= n_run) {
      seg_late(d, (k - n_run) * 32, t);
      continue;
    }
    int g, ja = 0, jend;
    if (d.packed) {
      g = d.tl[(size_t)k * 32 + wl];
      jend = __popc(__ballot_sync(0xffffffffu, g >= 0));
    } else {   // part p of group k - p n_grp
      const int p = k / n_grp, grp = k - p * n_grp;
      const unsigned long long cuts = d.cuts[grp];
      ja = p ? (int)(cuts >> (8 * p - 8) & 255u) : 0;
      jend = p < 7 ? min(32, (int)(cuts >> (8 * p) & 255u)) : 32;
      if (ja >= jend) continue;
      g = grp * 32 + wl;
    }
#pragma unroll 1
    do {
      SegLane ln = seg_lane(d, g, t);
      {   // not: empty slots, links left to whole blocks (one may have been through, and have
          // left fewer vehicles: its last lane's range, one word, tells either way)
        const unsigned info = __float_as_uint(ln.lb.z);
        const int lane = (int)(info & 7u), lanes = (int)(info >> 3 & 7u) + 1;
        const bool big = __shfl_sync(0xffffffffu, ln.done || seg_big(ln.start + ln.cnt, lanes) ? 1 : 0,
                                     (wl + lanes - 1 - lane) & 31) != 0;
        if (ctrl_of(info) == kCtrlPad || big) ln.on = false;
      }
      ln.on = ln.on && wl >= ja && wl < jend;
      const int w = ln.on ? ln.cnt + (ln.ext ? 1 : 0) + (ln.due ? 1 : 0) : 0;
      int jb = jend;
      if (__reduce_add_sync(0xffffffffu, w) > kSegN) {
        const unsigned info = __float_as_uint(ln.lb.z);
        jb = min(jb, seg_run_end(ja, warp_inclusive(w), (int)(info & 7u), (int)(info >> 3 & 7u) + 1, ln.on || wl < jend, kSegN));
        ln.on = ln.on && wl < jb;
      }
      if (__any_sync(0xffffffffu, ln.on && (ln.cnt || ln.ext || ln.due)))
        seg_run<32, SegSmem, OUT, TYPES, TAPE>(d, S, ln, 32, t, s_cn);
      else if (ln.on && d.rng[g])   // nothing here but the mark of a block that emptied the link in the
        d.rng[g] = 0;               // step before; in the next step it would pass for that step's
      ja = jb;
    } while (ja < jend);
  }
  __syncthreads();
  // counters: one set of additions per block
  if (threadIdx.x == 0) {
    Ctl* c = d.ctl;
    if (s_cn[0]) {
      atomicAdd(&c->nact[t & 1], s_cn[0]);
      atomicAdd(&c->veh_steps, (unsigned long long)s_cn[0]);
    }
    if (s_cn[1]) atomicAdd(&c->lc_evals, (unsigned long long)s_cn[1]);
    if (s_cn[2]) atomicAdd(&c->arrived, (unsigned long long)s_cn[2]);
    if (s_cn[3]) atomicAdd(&c->departed, (unsigned long long)s_cn[3]);
    if (blockIdx.x == 0) {
      c->t = (long long)t + 1;
      c->pk_run = c->pk_veh = 0;   // for the next packing
    }
  }
}

}  // namespace gbt
