// Internal launch interface between the C ABI layer and the kernels.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "kf_common.cuh"

namespace kfg {

// Device-side status word values (sticky; read by kf_sync / kf_get_*).
enum : int {
  ST_OK = 0,
  ST_DEDUP_PARTNERS = 1,   // a track shares hits with more tracks than the partner table holds
  ST_DEDUP_CONFLICTS = 2,  // more higher-priority conflicts than the conflict table holds
  ST_DEDUP_ROUNDS = 3,     // the resolution loop hit its iteration bound
  ST_SEED_CONFLICTS = 4,   // seed cleaning: more lower-index duplicates than the conflict table holds
  ST_SEED_ROUNDS = 5,      // seed cleaning: the resolution loop hit its iteration bound
};

// SMs of the chip, for grids of kernels that are launched without a context.
constexpr int CHIP_SMS = 152;

// Seeds of an event are taken in order of their polar angle, counting-sorted
// into SEED_THETA_BINS equal bins of [0, pi] (the order within a bin is
// arbitrary).
constexpr int SEED_THETA_BINS = 1024;
__device__ __forceinline__ int seed_theta_bin(float theta) {
  return min(max((int)(theta * ((float)SEED_THETA_BINS / PI_F)), 0), SEED_THETA_BINS - 1);
}

struct FindParams {
  DevGeom g;
  const float* hx;
  const float* hy;
  const float* hz;
  const int* hlayer;
  const int* hit_off;        // [n_events + 1]
  const float4* hb;          // binned hits (x, y, z, event-local index as int bits)
  const unsigned* bin_off;   // [n_events * n_layers * n_bins + 1] global offsets into hb
  const float* eta_edges;    // [KF_MAX_LAYERS][MAX_ETA_BINS + 1] z edges of the eta bins
  const unsigned char* eta_lut;  // [KF_MAX_LAYERS][ETA_LUT] first guess of the eta bin
  const float* sp;           // seed params [6][ns]
  const float* sc;           // seed cov [21][ns]
  const int* sh;             // seed hits [3][ns]
  const int* seed_event;     // [ns]
  const Align4* align;       // [n_layers]
  int ns;                    // seed stride
  int s_begin, s_end;        // seed range of this launch
  const int* order;          // [ns] order of the seeds within each event (or null)
  const int* seed_off;       // [n_events + 1]
  const int* kept_cnt;       // [n_events] seeds left by seed cleaning (or null: every seed);
                             // with it, order lists each event's kept seeds first
  int* out_hits;             // [ns][n_layers]
  int* out_n;                // [ns]
  float* out_chi2;           // [ns]
  float* out_p;              // [6][ns]
  float* out_C;              // [21][ns]
  unsigned* queue;           // [3] work counters of the main and careful passes and the
                             // number of listed seeds (zeroed before the launch)
  int* tangent_list;         // [ns] seeds the main pass left to the careful pass
  unsigned* rec;             // [rec_cap][find_record_words()] what it left of their searches
  int rec_cap;
  float* sfit;               // [29][ns] seed kernel: the state the first layer's children come
                             // from (p, C), the seed's chi2 sum, the first layer's counts
  unsigned long long* skeys; // [max_cands][ns] seed kernel: the first layer's children (keys)
  unsigned char* sflag;      // [ns] seed kernel: bit 1 near-tangent crossing, bit 2 carried,
                             // bits 3-7 number of children
  unsigned long long* counters;  // [8], see kf_get_counters
  int persistent;
};

struct BinParams {
  DevGeom g;
  const float* hx;
  const float* hy;
  const float* hz;
  const int* hlayer;
  const int* hit_off;
  int n_events;
  int h_begin, h_end;     // hit range of this launch
  const float* eta_edges; // [KF_MAX_LAYERS][MAX_ETA_BINS + 1]
  const unsigned char* eta_lut;  // [KF_MAX_LAYERS][ETA_LUT]
  unsigned* cnt;          // [n_bins_total + 1] counts, then offsets
  unsigned* key;          // [n_hits]
  unsigned* rank;         // [n_hits]
  float4* hb;             // [n_hits]
  float4* grouped;        // [n_hits] hits grouped by (event, layer) (layer-grouped form)
  unsigned* gtab;         // bin_group_elems(): bucket counts, bases (+ total) of the (event,
                          // layer, chunk of eta rows) buckets
};

struct DedupParams {
  const int* out_hits;   // [ns][L]
  const int* out_n;
  const float* out_chi2;
  const int* hit_off;    // [n_events + 1]
  const int* seed_off;   // [n_events + 1]; null: one event of ns tracks
  const int* seed_event; // [ns]; null: one event
  int L;                 // at most 64
  int ns;
  float frac;
  unsigned* head;        // event e's hit h at [hit_off[e] + e + h]: the last entry of its owner list
  unsigned* next;        // [ns * L] the entry before
  int* conf;             // [ns * DEDUP_CONF_CAP]
  int* n_conf;           // [ns]
  unsigned char* state;  // [ns]
  unsigned char* keep;   // [ns]
  int* status;
  // Kinematic pre-cuts (null trk_p: none): a pair is a duplicate only if its
  // states trk_p [6][ns] are also close in eta, phi0 and pT (a cut <= 0 is off).
  const float* trk_p = nullptr;
  float kb = 0.f;        // h = kb * q/pT
  float deta = 0.f, dphi = 0.f, dpt = 0.f;
  int max_rounds = 0;    // resolution rounds before giving up (0: until settled)
};

struct SeedCleanParams {
  float kb;              // h = kb * q/pT
  const float* sp;       // seed params [6][ns]
  const float* sc;       // seed cov [21][ns]
  const int* sh;         // seed hits [3][ns]
  const int* seed_off;   // [n_events + 1]
  const int* seed_event; // [ns]
  const int* order;      // [ns] the theta order of each event's seeds
  int ns;
  int L;
  float deta, dphi, dpt; // cuts (deta > 0; dphi, dpt <= 0: not applied)
  int min_shared;        // seed hits shared, at least
  float4* kin;           // [ns] by position in order: (eta, phi0, |q/pT|, theta bin as int bits)
  int4* kseed;           // [ns] by position: (seed, its three hits)
  int* conf;             // [ns * DEDUP_CONF_CAP] by position: positions of the lower-index duplicates
  int* n_conf;           // [ns] by position
  unsigned char* state;  // [ns] by position
  int* list;             // [ns] per event (at its positions): the positions with conflicts
  int* list_cnt;         // [n_events]
  int* clean_order;      // [ns] per event: the kept seeds in theta order, then the dropped ones
  int* kept_cnt;         // [n_events]
  // outputs written for a dropped seed: an empty track, not kept
  int* out_hits;         // [ns][L]
  int* out_n;
  float* out_chi2;
  float* out_p;          // [6][ns]
  float* out_C;          // [21][ns]
  unsigned char* keep;   // [ns]
  int* status;
  int max_rounds = 0;    // resolution rounds before giving up (0: until settled)
};

// The adjoint redoes in double only the steps closer to tangent than this
// (its tolerance is looser than the fit's; the fit's threshold is 0.5).
constexpr float ADJOINT_CAREFUL_COS = 0.2f;
constexpr unsigned CAREFUL_DBL_BIT = 0x80000000u;  // careful_list entry: a crossing below ADJOINT_CAREFUL_COS

constexpr int DEDUP_PARTNER_CAP = 32;
constexpr int DEDUP_CONF_CAP = 16;

// Grid of a careful pass of the fit or its adjoint over a list whose length only
// the device knows: short lists are dealt evenly to the first `spread` blocks
// (a double-precision instruction takes its unit 64 clocks whatever its active
// lanes), longer ones go a block's threads at a time over the whole grid, and a
// block without a track ends at once.  The list can hold every track (a loose
// prior), so the grid has room for all of them, up to twelve blocks per SM (of
// one warp, 8 and 16 are slower): the fit and the gradient (ckpt_stride 1) of
// 800,000 such tracks took 8.2 and 7.0 ms in grids for the usual 64th of the
// tracks, 4.4 and 1.6 so; those of 80,000 1.14 and 1.10, 0.55 and 0.23 so.
inline int careful_blocks(int n_tracks, int threads, int spread, int num_sms) {
  const int packed = n_tracks / threads + 1, most = 12 * num_sms;
  const int few = n_tracks < spread ? n_tracks : spread;
  const int many = packed < most ? packed : most;
  return few > many ? few : many;
}

struct FitParams {
  DevGeom g;
  const float* hx;
  const float* hy;
  const float* hz;
  const int* hlayer;
  const int* hit_off;
  const float* sp;
  const float* sc;
  const int* seed_event;
  const Align4* align;
  int ns;
  const int* lists;       // [ns][max_len]
  const int* n_list;      // [ns]
  int max_len;
  const unsigned char* keep;  // may be null
  // false: the FP32 pass runs beside duplicate removal and fits every track
  // (keep is still being written); launch_fit_unkept clears the removed
  // tracks' outputs afterwards, and the careful pass reads keep as usual
  bool keep_in_main = true;
  float* fit_p;           // [6][ns]
  float* fit_C;           // [21][ns]
  float* fit_chi2;        // [ns]
  int* fit_status;        // [ns]
  int* careful_list;      // [ns] positions (in order) of the tracks refitted with double-precision steps;
                          // the careful pass adds CAREFUL_DBL_BIT where the adjoint needs double steps
  unsigned* careful_count;  // zeroed by launch_fit_main
  unsigned char* careful_flag;  // [ns] by track: for the tracks of careful_list 1 + the step the FP32
                                // pass stopped at (255 at most), else 0
  int* dbl_list;          // [ns] positions of the careful tracks with CAREFUL_DBL_BIT, packed
  unsigned* dbl_count;    // their number (zeroed by launch_fit_main)
  float* ckpt;            // [ckpt_slices][27][ns] by position: states before every ckpt_stride-th hit, or null
  int ckpt_stride;
  int ckpt_slices;        // checkpoints per track the buffer holds
  int num_sms;
  int careful_spread;     // blocks over which a short careful list is dealt (set at its launch)
  // Tracks of each window of 4,096 by decreasing hit count (duplicates
  // last): position i of the fit and of the adjoint takes track order[i], so
  // that a warp's tracks run about the same number of steps.
  int* order;             // [ns] written by launch_fit_main
};

constexpr int MAX_CKPT = KF_MAX_LAYERS;  // checkpoints per track at most
// Checkpoints per track for tracks of up to max_len hits.
inline int ckpt_slices_for(int max_len, int stride) {
  const int n = (max_len + stride - 1) / stride;
  return n < MAX_CKPT ? n : MAX_CKPT;
}
constexpr int DEFAULT_CKPT_STRIDE = 1;
constexpr int MAX_CKPT_STRIDE = 8;

struct AdjParams {
  DevGeom g;
  const float* hx;
  const float* hy;
  const float* hz;
  const int* hlayer;
  const int* hit_off;
  const float* sp;
  const float* sc;
  const int* seed_event;
  const Align4* align;
  int ns;
  int n_hits;
  const int* lists;
  const int* n_list;
  int max_len;
  const unsigned char* keep;   // may be null
  const int* fit_status;       // tracks with a status other than KF_FIT_OK are skipped
  int stride;                  // checkpoint stride
  float* g_hits;               // [n_hits][3] (required: the alignment gradient is summed from it)
  float* g_seed;               // [6][ns] or null
  float* g_align;              // [n_layers][2]
  double* g_align_acc;         // [2 * KF_MAX_LAYERS] accumulator
  const int* careful_list;     // positions of the tracks the fit flagged as near-tangent ...
  const unsigned* careful_count;
  const unsigned char* careful_flag;  // ... and their per-track flag
  const int* dbl_list;         // the careful tracks whose adjoint needs double steps, packed
  const unsigned* dbl_count;
  const float* ckpt;           // the fit's checkpoints [slices][27][ns] by position
  const int* order;            // the fit's track order (position -> track)
  int num_sms;
  bool after_fit;              // the fit's careful pass runs on the same branch before the careful passes
  int careful_spread;          // as FitParams'
};

// kf_copy.cu
// Up to seven copies of one launch.
struct CopyList {
  int n = 0;
  void* dst[7];
  const void* src[7];
  size_t bytes[7];
  void add(void* d, const void* s, size_t b) {
    if (!d || b == 0) return;
    dst[n] = d;
    src[n] = s;
    bytes[n++] = b;
  }
};
// Event offsets as a kernel argument (n = 0: they are copied instead).
constexpr int OFFSET_ARG = 128;
struct OffsetArg {
  int n = 0;
  int v[OFFSET_ARG];
};
// What a finding call starts from: counters and queue zero, keep flags set, and
// (batched form) the binning's bucket counts zero.
struct FindBegin {
  unsigned long long* counters;
  unsigned* queue;
  unsigned* table;
  unsigned char* keep;
  int n_counters, n_queue;
  size_t n_table;
  int n_keep;
};
cudaError_t launch_copy(const CopyList& c, int num_sms, cudaStream_t st);
// Copies, offsets and checks of kf_load_hits / kf_load_seeds; layer, sh: where
// the checked values are (the source or the copy); bad[2]: host memory, zeroed
// by the caller, read after a synchronization.
cudaError_t launch_load_hits(const CopyList& c, const int* layer, int n, int n_surf, const OffsetArg& o, int* hit_off,
                             int* bad, int num_sms, cudaStream_t st);
cudaError_t launch_load_seeds(const CopyList& c, const int* sh, int n, int n_events, const OffsetArg& o, int* seed_off,
                              const int* hit_off, const int* hlayer, int n_layers, int* seed_event,
                              unsigned char* keep, int* bad, int num_sms, cudaStream_t st);
cudaError_t launch_find_begin(const FindBegin& b, int num_sms, cudaStream_t st);
// kf_adjoint.cu
// Adjoint: zero the accumulators, the FP32 pass, the passes over the fit's
// careful list, without and with double-precision steps (independent: any
// order or concurrently), then the alignment gradient from its
// double-precision sums.
enum { ADJ_MAIN = 0, ADJ_LIST = 1, ADJ_DBL = 2 };
cudaError_t launch_adjoint_begin(const AdjParams& P, cudaStream_t st);
cudaError_t launch_adjoint_pass(const AdjParams& P, int pass, cudaStream_t st);
cudaError_t launch_adjoint_end(const AdjParams& P, cudaStream_t st);
bool adjoint_stride_ok(int stride, int max_len);
// kf_find.cu
// Finding: the main pass (gives up and lists seeds that meet a near-tangent
// crossing), then the careful pass over the listed seeds (persistent, any
// grid; the count is read on the device).
cudaError_t launch_find_main(const FindParams& P, int lanes, int regcap, int threads, int grid_cap,
                             cudaStream_t st);
cudaError_t launch_find_careful(const FindParams& P, int lanes, int grid, cudaStream_t st);
// Per event, the seeds sorted by theta (params row 5) into order[].
cudaError_t launch_seed_order(const float* theta, const int* seed_off, int n_events, int* order, cudaStream_t st);
size_t find_smem_bytes(int threads, int n_layers, int n_eta);
bool find_lanes_supported(int lanes);
size_t find_record_words(int n_plan, int max_cands);  // words of a seed's record (FindParams::rec)
// Sets the dynamic shared-memory limit of the kernel variant (must run
// outside stream capture) and reports resident blocks per SM.
cudaError_t find_prepare(int lanes, int regcap, int threads, const DevGeom& g, int* blocks_per_sm);
// The disk variants (kf_find_disk.cu), called by the entry points above for a
// detector with endcap disks.
cudaError_t find_prepare_disk(int lanes, int regcap, int threads, const DevGeom& g, int* blocks_per_sm);
cudaError_t launch_find_main_disk(const FindParams& P, int lanes, int regcap, int threads, int grid_cap,
                                  cudaStream_t st);
cudaError_t launch_find_careful_disk(const FindParams& P, int lanes, int grid, cudaStream_t st);
// kf_bin.cu
cudaError_t launch_bin(const BinParams& P, size_t bin_begin, size_t n_bins, unsigned first_pos, int max_event_hits,
                       unsigned* scan_tmp, size_t scan_tmp_elems, cudaStream_t st);
// Bucket counts (BinParams::gtab) that launch_bin expects zeroed; 0: none (the
// general form).
size_t bin_table_elems(const BinParams& P, int n_events);
size_t scan_tmp_elems(size_t n);
size_t bin_group_elems(int n_events, int n_layers, int n_eta, int n_phi);
// kf_dedup.cu
// Tracks [t_begin, t_end), those of events [e_begin, e_begin + n_events), whose
// list heads are head[head_begin, head_begin + n_heads).  clear_status: the
// status word is zeroed first.
cudaError_t launch_dedup(const DedupParams& P, int t_begin, int t_end, int e_begin, int n_events, size_t head_begin,
                         size_t n_heads, bool clear_status, cudaStream_t st);
// Seed cleaning of the seeds at positions [pos_begin, pos_end) of the theta
// order, which are those of events [e_begin, e_begin + n_events).
cudaError_t launch_seed_clean(const SeedCleanParams& P, int pos_begin, int pos_end, int e_begin, int n_events,
                              cudaStream_t st);
// kf_fit.cu: the FP32 pass (flags and lists near-tangent tracks) and the
// careful pass over the list; launch_fit runs both.
cudaError_t launch_fit_main(const FitParams& P, cudaStream_t st);
cudaError_t launch_fit_careful(const FitParams& P, cudaStream_t st);
cudaError_t launch_fit(const FitParams& P, cudaStream_t st);
// After a main pass with keep_in_main false: the removed tracks' outputs
// zeroed and their status KF_FIT_SKIPPED, as the main pass would have left them.
cudaError_t launch_fit_unkept(const FitParams& P, cudaStream_t st);

}  // namespace kfg
