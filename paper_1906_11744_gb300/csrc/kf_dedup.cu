// Duplicate handling (Sec. 4.2): seed cleaning before building and duplicate
// removal after it.
//
// Kinematic closeness of two tracks or seeds (the paper names pT, eta and phi
// as criteria of both steps): |d eta| < deta, |d phi0| < dphi (difference on
// the circle), ||k_A| - |k_B|| <= dpt max(|k_A|, |k_B|) with k = q/pT; a cut
// <= 0 is not applied.  eta = -ln tan(theta/2); phi0 is the direction of
// motion at the point of the helix closest to the z axis, which every state
// along the helix shares.
//
// Duplicate removal, definition (sequential): visit the tracks of an event by
// (more hits, lower chi2 sum, lower index); keep a track unless it shares more
// than frac * min(nA, nB) hits with a track already kept and (with the
// kinematic pre-cuts) is kinematically close to it.  A track without hits (a
// cleaned seed's) is never kept.
//
// Seed cleaning, definition (sequential): visit the seeds of an event by
// index; drop a seed when a seed already kept is kinematically close to it and
// shares at least min_shared of its three hits.  Parallel form: the same
// conflict lists and resolution rounds as below, the pairs found by scanning
// each seed's neighbours in the theta order of the event.
//
// Parallel form, identical result, over a whole batch or one event:
//   1. k_dd_build: one thread per hit of a track pushes its entry on the list
//      of its hit (head[hit] and next[entry], one atomic exchange each);
//   2. k_dd_conflicts: eight lanes per track walk the lists of its hits (for
//      most tracks one head and one next read per hit) and one of them counts
//      the shared hits per partner; a pair over the threshold is a conflict,
//      recorded at the lower-priority track; a track without conflicts is kept
//      at once;
//   3. k_dd_rounds, one block per event: an undecided track is removed as soon
//      as one of its higher-priority conflicts is kept, and kept as soon as
//      all of them are removed.  The decisions equal the sequential walk's,
//      because each one only depends on the final decisions of higher-priority
//      tracks; every round settles at least the highest-priority undecided
//      track.
// All three are bound by the latency and number of the scattered 4-byte
// accesses to the hit table; lists need one per entry, where a table of owner
// ranges (count, scan over all hits, fill) needed two and the scan.
// Measured on an 8,800-track event through the allocation-free entry: 640 us
// in one block over owner ranges, 32 us so (the walks 15 of them, the rounds 7).
// Scratch (the lists, the conflict lists and the decision states) lives in
// global memory owned by the caller.
#include <algorithm>
#include <mutex>

#include "kf_internal.h"

namespace kfg {

namespace {

constexpr int DEDUP_THREADS = 1024;
constexpr int DD_THREADS = 256;
constexpr int DD_LANES = 8;   // lanes per track when its hits are tested for other owners
constexpr int DD_OTHERS = 3;  // other owners of a hit that its lane holds
constexpr unsigned DD_NONE = 0xFFFFFFFFu;
// A single event of up to this many tracks is done by one block: 20 us against
// 29 at 110 tracks, 27 against 31 at 220, 57 against 30 at 440.
constexpr int DD_ONE_TRACKS = 256;
constexpr size_t DD_ONE_HEADS = 16384;

// (eta, phi0, |q/pT|) of a state.  phi0 = atan2(-v_x, v_y) with
// v = h c = (h x - sin phi, h y + cos phi), h times the centre c of the track
// circle: the closest point to the axis lies along c, where the direction of
// motion is sign(h) (c_y, -c_x)/|c|.  For h = 0, v = (-sin phi, cos phi) and
// phi0 = phi.  Accurate library functions: these values decide which tracks
// are kept.
struct Kin {
  float eta, phi0, ak;
};
__device__ __forceinline__ Kin kin_of(float x, float y, float kappa, float phi, float theta, float kb) {
  const float h = kb * kappa;
  float s, c;
  sincosf(phi, &s, &c);
  Kin k;
  k.eta = -logf(tanf(0.5f * theta));
  k.phi0 = atan2f(-fmaf(h, x, -s), fmaf(h, y, c));
  k.ak = fabsf(kappa);
  return k;
}
__device__ __forceinline__ bool kin_close(const Kin& a, const Kin& b, float deta, float dphi, float dpt) {
  if (deta > 0.f && !(fabsf(a.eta - b.eta) < deta)) return false;
  if (dphi > 0.f) {
    float d = fabsf(a.phi0 - b.phi0);
    if (d > PI_F) d = TWO_PI_F - d;
    if (!(d < dphi)) return false;
  }
  if (dpt > 0.f && !(fabsf(a.ak - b.ak) <= dpt * fmaxf(a.ak, b.ak))) return false;
  return true;
}
// Kinematics of track t from its state [6][ns].
__device__ __forceinline__ Kin track_kin(const DedupParams& P, int t) {
  const float* q = P.trk_p + t;
  const size_t n = (size_t)P.ns;
  return kin_of(q[0], q[n], q[3 * n], q[4 * n], q[5 * n], P.kb);
}

__device__ __forceinline__ bool prio_less(int na, float ca, int ia, int nb, float cb, int ib) {
  if (na != nb) return na > nb;
  if (ca != cb) return ca < cb;
  return ia < ib;
}

// Head of the owner list of hit 0 of track t's event (hit h's head at [h]).
__device__ __forceinline__ unsigned* dd_heads(const DedupParams& P, int t) {
  if (!P.seed_event) return P.head;  // a single event
  const int e = P.seed_event[t];
  return P.head + P.hit_off[e] + e;
}

// The list heads empty and (clear_status) the status word zero: one launch
// instead of two memsets where a call is bound by its launches.
__global__ void __launch_bounds__(DD_THREADS) k_dd_begin(unsigned* head, size_t n_heads, int* clear_status) {
  const size_t i = blockIdx.x * (size_t)DD_THREADS + threadIdx.x, nt = (size_t)gridDim.x * DD_THREADS;
  if (i == 0 && clear_status) *clear_status = ST_OK;
  for (size_t k = i; k < n_heads; k += nt) head[k] = DD_NONE;
}

// Entry id = t L + j for hit j of track t of [t_begin, t_end).
__global__ void __launch_bounds__(DD_THREADS) k_dd_build(const DedupParams P, int t_begin, int t_end) {
  const unsigned i = blockIdx.x * (unsigned)DD_THREADS + threadIdx.x;
  const unsigned r = i / (unsigned)P.L;
  if (r >= (unsigned)(t_end - t_begin)) return;
  const int t = t_begin + (int)r, j = (int)(i - r * (unsigned)P.L);
  if (j >= P.out_n[t]) return;
  const unsigned id = (unsigned)t * (unsigned)P.L + j;
  P.next[id] = atomicExch(dd_heads(P, t) + P.out_hits[id], id);
}

// Conflicts and first decision of track t (valid) by a group of DD_LANES
// lanes; the whole warp calls this.
__device__ __forceinline__ void dd_conflicts(const DedupParams& P, int t, bool valid) {
  const int lane = threadIdx.x & 31, gl = threadIdx.x & (DD_LANES - 1);
  const int L = P.L;
  const int n = valid ? min(P.out_n[t], L) : 0;
  const unsigned id0 = (unsigned)t * (unsigned)L;
  const unsigned* head = valid ? dd_heads(P, t) : P.head;
  int pid[DEDUP_PARTNER_CAP];  // the leading lane's: partners and shared hits
  int pcnt[DEDUP_PARTNER_CAP];
  int np = 0;
  bool overflow = false;
  auto partner = [&](int u) {
    int k = 0;
    while (k < np && pid[k] != u) ++k;
    if (k < np) {
      pcnt[k]++;
    } else if (np < DEDUP_PARTNER_CAP) {
      pid[np] = u;
      pcnt[np] = 1;
      ++np;
    } else {
      overflow = true;
    }
  };
  // Each lane walks the list of its hit and holds the first few other owners;
  // then the leading lane takes them over by shuffles.  A hit with more
  // owners than that is walked again by the leading lane alone.
  for (int b = 0; b < L; b += DD_LANES) {
    const int j = b + gl;
    int other[DD_OTHERS];
#pragma unroll
    for (int k = 0; k < DD_OTHERS; ++k) other[k] = -1;
    unsigned q = DD_NONE;  // the list's rest
    unsigned q0 = DD_NONE;
    if (j < n) {
      q = q0 = head[P.out_hits[id0 + j]];
#pragma unroll
      for (int k = 0; k < DD_OTHERS; ++k) {
        if (q != DD_NONE && q - id0 < (unsigned)L) q = P.next[q];  // its own entry
        if (q != DD_NONE && q - id0 >= (unsigned)L) {
          other[k] = (int)(q / (unsigned)L);
          q = P.next[q];
        }
      }
      if (q != DD_NONE && q - id0 < (unsigned)L) q = P.next[q];
    }
    const bool more = q != DD_NONE;
    if (!__any_sync(0xffffffffu, other[0] >= 0 || more)) continue;
#pragma unroll 1
    for (int i = 0; i < DD_LANES; ++i) {
      const int src = lane - gl + i;
      const bool m = __shfl_sync(0xffffffffu, (int)more, src) != 0;
      const unsigned first = __shfl_sync(0xffffffffu, q0, src);
      int o[DD_OTHERS];
#pragma unroll
      for (int k = 0; k < DD_OTHERS; ++k) o[k] = __shfl_sync(0xffffffffu, other[k], src);
      if (gl != 0) continue;
      if (!m) {
#pragma unroll
        for (int k = 0; k < DD_OTHERS; ++k)
          if (o[k] >= 0) partner(o[k]);
      } else {
        unsigned long long steps = (unsigned long long)P.ns * L;  // no list is longer
        for (unsigned e = first; e != DD_NONE && steps && !overflow; e = P.next[e], --steps)
          if (e - id0 >= (unsigned)L) partner((int)(e / (unsigned)L));
      }
    }
  }
  if (!valid || gl != 0) return;
  if (np == 0) {  // no track (a cleaned seed): removed; nothing shared: kept
    P.n_conf[t] = 0;
    P.state[t] = n == 0 ? 2 : 1;
    return;
  }
  const float c = P.out_chi2[t];
  if (overflow) atomicCAS(P.status, ST_OK, ST_DEDUP_PARTNERS);
  const bool kin = P.trk_p != nullptr;
  Kin kt;
  if (kin) kt = track_kin(P, t);
  int nc = 0;
  for (int k = 0; k < np; ++k) {
    const int u = pid[k];
    const int nu = P.out_n[u];
    if ((float)pcnt[k] > P.frac * (float)min(n, nu) && prio_less(nu, P.out_chi2[u], u, n, c, t) &&
        (!kin || kin_close(kt, track_kin(P, u), P.deta, P.dphi, P.dpt))) {
      if (nc < DEDUP_CONF_CAP) P.conf[(size_t)t * DEDUP_CONF_CAP + nc] = u;
      else atomicCAS(P.status, ST_OK, ST_DEDUP_CONFLICTS);
      ++nc;
    }
  }
  P.n_conf[t] = min(nc, DEDUP_CONF_CAP);
  P.state[t] = nc == 0 ? 1 : 0;
}
__global__ void __launch_bounds__(DD_THREADS) k_dd_conflicts(const DedupParams P, int t_begin, int t_end) {
  const int t = t_begin + (int)(blockIdx.x * (DD_THREADS / DD_LANES) + threadIdx.x / DD_LANES);
  dd_conflicts(P, t, t < t_end);
}

// Resolution rounds of items [s0, s1) (an event's tracks or seeds) by the
// whole block, then the keep flags.  Each item's conflicts are the
// higher-priority items that remove it if kept.
struct Rounds {
  const int* n_conf;
  const int* conf;
  unsigned char* state;
  unsigned char* keep;
  int* status;
  int err;         // status value when the rounds do not settle
  int max_rounds;  // rounds before giving up; 0: n + 4, which always settles
};
// One step of item t: removed as soon as one of its conflicts is kept, kept
// as soon as all of them are removed.  Returns false while undecided.
__device__ __forceinline__ bool dd_decide(const Rounds& P, int t) {
  if (P.state[t] != 0) return true;
  const int nc = min(P.n_conf[t], DEDUP_CONF_CAP);
  bool any_kept = false, all_removed = true;
  for (int k = 0; k < nc; ++k) {
    const unsigned char s = ((volatile unsigned char*)P.state)[P.conf[(size_t)t * DEDUP_CONF_CAP + k]];
    if (s == 1) any_kept = true;
    if (s != 2) all_removed = false;
  }
  if (any_kept) P.state[t] = 2;
  else if (all_removed) P.state[t] = 1;
  else return false;
  return true;
}
// Rounds by the whole block over items item(0..n) until every one is decided
// (at most n + 2 rounds: each settles the highest-priority undecided item),
// or, with a round cap, until the cap (the status then records the failure).
template <class Item>
__device__ void dd_rounds_over(const Rounds& P, int n, Item item) {
  __shared__ int sh_flag;
  const int tid = threadIdx.x, nt = blockDim.x;
  for (int round = 0;; ++round) {
    if (tid == 0) sh_flag = 0;
    __syncthreads();
    bool undecided = false;
    for (int i = tid; i < n; i += nt)
      if (!dd_decide(P, item(i))) undecided = true;
    if (undecided) sh_flag = 1;
    __syncthreads();
    const int more = sh_flag;
    __syncthreads();
    if (!more) break;
    if (round + 1 >= (P.max_rounds > 0 ? P.max_rounds : n + 4)) {
      if (tid == 0) atomicCAS(P.status, ST_OK, P.err);
      break;
    }
  }
}
// The same over the tracks [s0, s1) of an event, whose first decisions are
// taken: the states and the undecided tracks' list are held in shared memory
// (a round then costs a barrier and the conflict lists' reads, which stay in
// L1: 18 -> 7 us for 8,800 tracks), in global memory for a larger event.
constexpr int ROUNDS_STATES = 24576, ROUNDS_LIST = 5120;
__device__ void dd_rounds(const Rounds& P, int s0, int s1) {
  __shared__ __align__(16) unsigned char st[ROUNDS_STATES];
  __shared__ int list[ROUNDS_LIST];
  __shared__ int n_list, undecided_any;
  const int n = s1 - s0, tid = threadIdx.x, nt = blockDim.x;
  if (tid == 0) n_list = 0;
  __syncthreads();
  if (n <= ROUNDS_STATES)
    for (int i = tid; i < n; i += nt) {
      const unsigned char v = P.state[s0 + i];
      st[i] = v;
      if (v == 0) {
        const int k = atomicAdd(&n_list, 1);
        if (k < ROUNDS_LIST) list[k] = i;
      }
    }
  __syncthreads();
  if (n <= ROUNDS_STATES && n_list <= ROUNDS_LIST) {
    const int m = n_list;
    volatile unsigned char* const vst = st;
    for (int round = 0; m > 0; ++round) {
      if (tid == 0) undecided_any = 0;
      __syncthreads();
      bool undecided = false;
      for (int k = tid; k < m; k += nt) {
        const int i = list[k];
        if (vst[i] != 0) continue;
        const int* conf = P.conf + (size_t)(s0 + i) * DEDUP_CONF_CAP;
        const int nc = min(P.n_conf[s0 + i], DEDUP_CONF_CAP);
        bool any_kept = false, all_removed = true;
        for (int c = 0; c < nc; ++c) {
          const unsigned char v = vst[conf[c] - s0];
          any_kept = any_kept || v == 1;
          all_removed = all_removed && v == 2;
        }
        if (any_kept) vst[i] = 2;
        else if (all_removed) vst[i] = 1;
        else undecided = true;
      }
      if (undecided) undecided_any = 1;
      __syncthreads();
      const int more = undecided_any;
      __syncthreads();
      if (!more) break;
      if (round + 1 >= (P.max_rounds > 0 ? P.max_rounds : n + 4)) {
        if (tid == 0) atomicCAS(P.status, ST_OK, P.err);
        break;
      }
    }
    for (int i = tid; i < n; i += nt) P.keep[s0 + i] = vst[i] == 1 ? 1 : 0;
    return;
  }
  dd_rounds_over(P, s1 - s0, [&](int i) { return s0 + i; });
  for (int t = s0 + threadIdx.x; t < s1; t += blockDim.x) P.keep[t] = P.state[t] == 1 ? 1 : 0;
}

__global__ void __launch_bounds__(DEDUP_THREADS) k_dd_rounds(const DedupParams P, int e_begin) {
  const int e = e_begin + blockIdx.x;
  dd_rounds(Rounds{P.n_conf, P.conf, P.state, P.keep, P.status, ST_DEDUP_ROUNDS, P.max_rounds},
            P.seed_off ? P.seed_off[e] : 0, P.seed_off ? P.seed_off[e + 1] : P.ns);
}

// All three steps of one small event's tracks [s0, s1) in a block: at this
// size the launches cost more than one block's time.
__global__ void __launch_bounds__(DEDUP_THREADS) k_dd_one(const DedupParams P, int s0, int s1, size_t head_begin,
                                                          int n_heads, int* clear_status) {
  const int tid = threadIdx.x, L = P.L;
  if (tid == 0 && clear_status) *clear_status = ST_OK;
  for (int i = tid; i < n_heads; i += DEDUP_THREADS) P.head[head_begin + i] = DD_NONE;
  __syncthreads();
  const int warp = tid >> 5, lane = tid & 31;
  for (int t = s0 + warp; t < s1; t += DEDUP_THREADS / 32) {  // one warp per track
    const int n = min(P.out_n[t], L);
    unsigned* head = dd_heads(P, t);
    for (int j = lane; j < n; j += 32) {
      const unsigned id = (unsigned)t * (unsigned)L + j;
      P.next[id] = atomicExch(head + P.out_hits[id], id);
    }
  }
  __syncthreads();
  constexpr int PER = DEDUP_THREADS / DD_LANES;
  for (int t = s0; t < s1; t += PER) dd_conflicts(P, t + tid / DD_LANES, t + tid / DD_LANES < s1);
  __syncthreads();
  dd_rounds(Rounds{P.n_conf, P.conf, P.state, P.keep, P.status, ST_DEDUP_ROUNDS, P.max_rounds}, s0, s1);
}

// ------------------------------------------------------------ seed cleaning
// Kinematics and hits of the seed at each position of the theta order; its
// conflict count cleared and its state preset to kept (a seed without
// conflicts is kept); the event's list of seeds with conflicts emptied.
__global__ void k_sc_kin(const SeedCleanParams P, int pos_begin, int pos_end) {
  const int j = pos_begin + blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= pos_end) return;
  const int e = P.seed_event[j];
  if (j == P.seed_off[e]) P.list_cnt[e] = 0;
  const int s = P.order[j];
  const size_t n = (size_t)P.ns;
  const float th = P.sp[5 * n + s];
  const Kin k = kin_of(P.sp[s], P.sp[n + s], P.sp[3 * n + s], P.sp[4 * n + s], th, P.kb);
  P.kin[j] = make_float4(k.eta, k.phi0, k.ak, __int_as_float(seed_theta_bin(th)));
  P.kseed[j] = make_int4(s, P.sh[s], P.sh[n + s], P.sh[2 * n + s]);
  P.n_conf[j] = 0;
  P.state[j] = 1;
}

// Duplicate pairs, each tested once: the seed at position j against the
// later positions of its event within its theta-bin window.  A pair found is
// a conflict of its higher-index seed (conflict lists and decision states are
// kept by position, so that the resolution reads them in order); a seed's
// first conflict makes it undecided and enters it in its event's list (at
// most one entry per position of the event).  The theta
// order is sorted by theta bin, and every seed within deta in eta of seed j
// has theta below theta(eta_j - deta), theta(eta) = 2 atan(exp(-eta)): the
// scan stops past that bin (one bin more absorbs rounding).  A later position
// in the same or a later bin can also lie below eta_j; both halves of the
// window are covered because the lower member of every pair scans upward.
__global__ void k_sc_conflicts(const SeedCleanParams P, int pos_begin, int pos_end) {
  const int j = pos_begin + blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= pos_end) return;
  const int e = P.seed_event[j];  // positions and seed indices share the event ranges
  const int lo = P.seed_off[e], hi = P.seed_off[e + 1];
  const float4 a4 = P.kin[j];
  const Kin a{a4.x, a4.y, a4.z};
  const int b_hi = seed_theta_bin(2.f * atanf(expf(-(a.eta - P.deta)))) + 1;
  int4 me = make_int4(-1, 0, 0, 0);
  for (int q = j + 1; q < hi; ++q) {
    const float4 b4 = P.kin[q];
    if (__float_as_int(b4.w) > b_hi) break;
    if (!kin_close(a, Kin{b4.x, b4.y, b4.z}, P.deta, P.dphi, P.dpt)) continue;
    if (me.x < 0) me = P.kseed[j];
    const int4 o = P.kseed[q];
    const int shared = (me.y == o.y) + (me.y == o.z) + (me.y == o.w) + (me.z == o.y) + (me.z == o.z) +
                       (me.z == o.w) + (me.w == o.y) + (me.w == o.z) + (me.w == o.w);
    if (shared < P.min_shared) continue;
    const int t = o.x > me.x ? q : j, u = o.x > me.x ? j : q;  // t is removed by u if u is kept
    const int slot = atomicAdd(&P.n_conf[t], 1);
    if (slot < DEDUP_CONF_CAP) P.conf[(size_t)t * DEDUP_CONF_CAP + slot] = u;
    else atomicCAS(P.status, ST_OK, ST_SEED_CONFLICTS);
    if (slot == 0) {
      P.state[t] = 0;
      P.list[lo + atomicAdd(&P.list_cnt[e], 1)] = t;
    }
  }
}

// Per event (one block): the resolution rounds over the event's seeds with
// conflicts; then the new order of its positions: kept seeds first in theta
// order, the dropped ones from the end.  Tiles of positions are split one
// after the other, a ballot per warp and a scan over the warps each, so that
// states and orders are read and written coalesced.
__global__ void __launch_bounds__(DEDUP_THREADS) k_sc_resolve(const SeedCleanParams P, int e_begin) {
  constexpr int NW = DEDUP_THREADS / 32;
  __shared__ int s_warp[2][NW];
  const int e = e_begin + blockIdx.x;
  const int s0 = P.seed_off[e], s1 = P.seed_off[e + 1];
  if (s1 <= s0) {
    if (threadIdx.x == 0) P.kept_cnt[e] = 0;
    return;
  }
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int* list = P.list + s0;
  dd_rounds_over(Rounds{P.n_conf, P.conf, P.state, nullptr, P.status, ST_SEED_ROUNDS, P.max_rounds}, P.list_cnt[e],
                 [&](int i) { return list[i]; });
  __syncthreads();
  int kept = 0;  // kept positions before this tile
  for (int t0 = s0, buf = 0; t0 < s1; t0 += DEDUP_THREADS, buf ^= 1) {
    const int j = t0 + tid;
    const bool in = j < s1;
    const int seed = in ? P.order[j] : 0;
    const bool keep = in && P.state[j] == 1;
    const unsigned b = __ballot_sync(0xffffffffu, keep);
    if (lane == 0) s_warp[buf][warp] = __popc(b);
    __syncthreads();  // (the other buffer is rewritten only after the next one)
    const int w = lane < NW ? s_warp[buf][lane] : 0;
    int incl = w;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += v;
    }
    const int before = __shfl_sync(0xffffffffu, incl - w, warp) + __popc(b & ((1u << lane) - 1u));
    const int k = kept + before;  // kept positions before j
    if (keep) P.clean_order[s0 + k] = seed;
    else if (in) P.clean_order[s1 - 1 - (j - s0 - k)] = seed;
    kept += __shfl_sync(0xffffffffu, incl, 31);
  }
  if (tid == 0) P.kept_cnt[e] = kept;
}

// The empty outputs of the dropped seeds, one warp per DROP_POS positions of
// the new order (the dropped ones lie together at an event's end: 49 us for
// 2,200 of 160,000 seeds with 32 positions per warp), their scattered writes
// over the whole chip.
constexpr int DROP_POS = 4, DROP_THREADS = 256;
__global__ void __launch_bounds__(DROP_THREADS) k_sc_dropped(const SeedCleanParams P, int pos_begin, int pos_end) {
  const int lane = threadIdx.x & 31;
  const int j = pos_begin + (int)((blockIdx.x * DROP_THREADS + threadIdx.x) >> 5) * DROP_POS + lane;
  bool drop = false;
  int seed = 0;
  if (lane < DROP_POS && j < pos_end) {
    const int e = P.seed_event[j];  // positions and seed indices share the event ranges
    drop = j - P.seed_off[e] >= P.kept_cnt[e];
    seed = P.clean_order[j];
  }
  const size_t n = (size_t)P.ns;
  for (unsigned m = __ballot_sync(0xffffffffu, drop); m; m &= m - 1) {
    const int s = __shfl_sync(0xffffffffu, seed, __ffs(m) - 1);
    for (int l = lane; l < P.L; l += 32) P.out_hits[(size_t)s * P.L + l] = -1;
    if (lane < 21) P.out_C[lane * n + s] = P.sc[lane * n + s];
    if (lane < 6) P.out_p[lane * n + s] = P.sp[lane * n + s];
    if (lane == 0) {
      P.keep[s] = 0;
      P.out_n[s] = 0;
      P.out_chi2[s] = 0.f;
    }
  }
}

}  // namespace

cudaError_t launch_dedup(const DedupParams& P, int t_begin, int t_end, int e_begin, int n_events, size_t head_begin,
                         size_t n_heads, bool clear_status, cudaStream_t st) {
  if (n_events <= 0) return cudaSuccess;
  const int n = t_end - t_begin;
  if (n_events == 1 && n > 0 && n <= DD_ONE_TRACKS && n_heads <= DD_ONE_HEADS) {
    k_dd_one<<<1, DEDUP_THREADS, 0, st>>>(P, t_begin, t_end, head_begin, (int)n_heads,
                                          clear_status ? P.status : nullptr);
    return cudaGetLastError();
  }
  if (clear_status) {  // (with tracks: kf_remove_duplicates_noalloc)
    const size_t blocks = (n_heads + DD_THREADS - 1) / DD_THREADS;
    k_dd_begin<<<(unsigned)std::min<size_t>(std::max<size_t>(blocks, 1), 8 * CHIP_SMS), DD_THREADS, 0, st>>>(
        P.head + head_begin, n_heads, P.status);
  } else if (n > 0) {
    const cudaError_t e = cudaMemsetAsync(P.head + head_begin, 0xFF, sizeof(unsigned) * n_heads, st);
    if (e != cudaSuccess) return e;
  }
  if (n > 0) {
    const size_t entries = (size_t)n * P.L;
    k_dd_build<<<(unsigned)((entries + DD_THREADS - 1) / DD_THREADS), DD_THREADS, 0, st>>>(P, t_begin, t_end);
    constexpr int PER = DD_THREADS / DD_LANES;
    k_dd_conflicts<<<(n + PER - 1) / PER, DD_THREADS, 0, st>>>(P, t_begin, t_end);
  }
  k_dd_rounds<<<n_events, DEDUP_THREADS, 0, st>>>(P, e_begin);
  return cudaGetLastError();
}

cudaError_t launch_seed_clean(const SeedCleanParams& P, int pos_begin, int pos_end, int e_begin, int n_events,
                              cudaStream_t st) {
  if (n_events <= 0) return cudaSuccess;
  const int n = pos_end - pos_begin;
  if (n > 0) {
    const int threads = 256, blocks = (n + threads - 1) / threads;
    k_sc_kin<<<blocks, threads, 0, st>>>(P, pos_begin, pos_end);
    k_sc_conflicts<<<blocks, threads, 0, st>>>(P, pos_begin, pos_end);
  }
  k_sc_resolve<<<n_events, DEDUP_THREADS, 0, st>>>(P, e_begin);
  if (n > 0) {
    const int per = DROP_THREADS / 32 * DROP_POS;  // positions per block
    k_sc_dropped<<<(n + per - 1) / per, DROP_THREADS, 0, st>>>(P, pos_begin, pos_end);
  }
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Allocation-free duplicate removal (kf_remove_duplicates_noalloc).
//
// Some callers cannot allocate device memory at all: code that runs inside a
// host framework which owns every device allocation through its own pool, a
// trigger-style pipeline that forbids cudaMalloc/cudaFree on its hot path
// because they synchronize the device, or a plugin living within another
// library's fixed memory budget.  For them the duplicate-removal kernel also
// runs on a fixed scratch area in a file-scope device array, sized for one
// event of at most KF_NOALLOC_MAX_TRACKS tracks and KF_NOALLOC_MAX_HITS hits.
// The array exists once per device that loads the library and stays until the
// process exits.  Every call shares it: two calls whose kernels overlap on the
// GPU (different streams, or different host threads) race and give undefined
// results, so such calls must be ordered.
namespace {

constexpr size_t NA_HEAD_BYTES = ((size_t)(KF_NOALLOC_MAX_HITS) * 4 + 255) / 256 * 256;
constexpr size_t NA_NEXT_BYTES = (size_t)KF_NOALLOC_MAX_TRACKS * KF_MAX_LAYERS * 4;
constexpr size_t NA_CONF_BYTES = (size_t)KF_NOALLOC_MAX_TRACKS * DEDUP_CONF_CAP * 4;
constexpr size_t NA_NCONF_BYTES = (size_t)KF_NOALLOC_MAX_TRACKS * 4;
constexpr size_t NA_STATE_BYTES = ((size_t)KF_NOALLOC_MAX_TRACKS + 255) / 256 * 256;
constexpr size_t NA_MISC_BYTES = 256;  // the status word
constexpr size_t NA_BYTES =
    NA_HEAD_BYTES + NA_NEXT_BYTES + NA_CONF_BYTES + NA_NCONF_BYTES + NA_STATE_BYTES + NA_MISC_BYTES;

static __device__ __align__(256) unsigned char kf_noalloc_scratch[NA_BYTES];

// Device address of the scratch array per device, found once per device.
constexpr int NA_MAX_DEVICES = 64;
std::mutex na_mutex;
unsigned char* na_ptr[NA_MAX_DEVICES] = {};

}  // namespace

}  // namespace kfg

extern "C" int kf_remove_duplicates_noalloc(int n_tracks, int n_layers, int n_hits, const int* hits,
                                            const int* n_found, const float* chi2, float dup_shared_frac,
                                            unsigned char* keep, int* status, void* stream) {
  using namespace kfg;
  if (n_tracks < 0 || n_hits < 0 || n_layers < 1 || n_layers > KF_MAX_LAYERS || !(dup_shared_frac >= 0.f))
    return KF_ERR_ARG;
  if (n_tracks > KF_NOALLOC_MAX_TRACKS || n_hits > KF_NOALLOC_MAX_HITS) return KF_ERR_CAPACITY;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  if (n_tracks == 0) {  // nothing to remove; the status still reads "no error"
    if (status && cudaMemsetAsync(status, 0, sizeof(int), st) != cudaSuccess) return KF_ERR_CUDA;
    return KF_OK;
  }
  if (!hits || !n_found || !chi2 || !keep) return KF_ERR_ARG;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= NA_MAX_DEVICES) return KF_ERR_CUDA;
  unsigned char* base;
  {
    std::lock_guard<std::mutex> lock(na_mutex);
    if (!na_ptr[dev]) {
      void* p = nullptr;
      if (cudaGetSymbolAddress(&p, kf_noalloc_scratch) != cudaSuccess || !p) return KF_ERR_CUDA;
      na_ptr[dev] = static_cast<unsigned char*>(p);
    }
    base = na_ptr[dev];
  }
  DedupParams D;
  D.out_hits = hits;
  D.out_n = n_found;
  D.out_chi2 = chi2;
  D.seed_off = nullptr;  // one event of n_tracks tracks
  D.seed_event = nullptr;
  D.hit_off = nullptr;
  D.L = n_layers;
  D.ns = n_tracks;
  D.frac = dup_shared_frac;
  D.head = reinterpret_cast<unsigned*>(base);
  D.next = reinterpret_cast<unsigned*>(base + NA_HEAD_BYTES);
  D.conf = reinterpret_cast<int*>(base + NA_HEAD_BYTES + NA_NEXT_BYTES);
  D.n_conf = reinterpret_cast<int*>(base + NA_HEAD_BYTES + NA_NEXT_BYTES + NA_CONF_BYTES);
  D.state = base + NA_HEAD_BYTES + NA_NEXT_BYTES + NA_CONF_BYTES + NA_NCONF_BYTES;
  D.keep = keep;
  D.status = status ? status : reinterpret_cast<int*>(base + NA_BYTES - NA_MISC_BYTES);
  if (launch_dedup(D, 0, n_tracks, 0, 1, 0, (size_t)n_hits, true, st) != cudaSuccess) return KF_ERR_CUDA;
  return KF_OK;
}
