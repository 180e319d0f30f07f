// Mixed-precision Monte Carlo packet transport (same method as
// mc_transport.cu, Kerzendorf & Sim 2014 Sects. 2.4-2.7, 2.9), for one model
// or for a batch of models in one persistent launch.
//
// Precision split.  Geometry (x mu, impact parameter, radius), path lengths,
// optical depths, the logarithm of the event draw, packet energies (relative
// to the injection energy) and the frame factors are binary32.  Binary64 is
// kept where the method needs it: the lab and comoving frequencies, the
// Sobolev-resonance comparison against the frequency-sorted line list
// (integer keys of binary64 values) and the frequency thresholds that the
// optical depth is accumulated into.  J, nu_bar and J_blue are summed exactly
// as 64-bit fixed point from binary32 contributions (order-independent).  The
// lab frequency after a re-emission is nu_c / D to binary64 accuracy (Newton
// step on the binary32 reciprocal), so the comoving frequency at the emission
// point is the emitting line's frequency.  Conversions between the two
// formats are done on the bit patterns with integer operations (on this GPU a
// conversion instruction takes the binary64 pipe).
//
// Batched launch.  Packets of all models are claimed from one queue (models
// laid out by a prefix sum of their packet counts, largest first so that the
// longest random walks start first); a lane that claims a packet of another
// model loads that model's context and first flushes its register
// accumulators to the previous model.
//
// It also has the binary64 kernel's lone walks and pool: a warp down to its
// last walks runs one with all 32 lanes (32-line windows scanned in one step
// through a binary32 filter against this kernel's own threshold chain, the
// emission record loaded as soon as the scan names the line, the walk's draws
// computed ahead by the warp).
#include <cstdint>

#include "mc_device.cuh"
#include "mc_internal.h"

namespace mcgpu {

namespace {

// single-model launches take 128 threads per block, batched ones 64, 128 or 256
constexpr int kMaxBlock = 256;
constexpr size_t kLoneWords = sizeof(PoolWalk) / sizeof(unsigned long long) + kWarpDraws;
// A lone walk tries its line-event loop within so many segments of its last line
// event: every try scans the window once more where it is not one.  50,000
// packets through 400 shells, one segment in eight a line event: 39.0 -> 33.3 ms;
// trapped walks as before.
constexpr int kLoopTries = 3;
constexpr int kLineEvent = 1, kElectronEvent = 2, kShellEvent = 3;

struct PacketM {
  double nu_lab;               // binary64
  float p, q;                  // x mu, x^2 - p^2
  float e_lab, inv_nu, inv_D;  // e_lab relative to the injection energy
  int32_t shell, next_line;
  uint32_t pid;
  bool have_inv_D;
  uint32_t cnt[kNCounters];
};

// What a lane needs of its packet's model.
struct MCtx {
  const float *xi2, *xo2, *kap, *ikap;
  const double *nu;
  const float *tau32;
  const unsigned long long *row_info;
  const int32_t *line_row;           // macro atom: upper level of each line
  const MaRow *ma_row;               // macro atom: level table
  const MaJump *ma_jump;             // macro atom: jump entries
  const DbrSlot *bucket;
  const DbrRec *rec;
  const float *inv_nu32;
  double *j_blue, *j_est, *nu_bar, *spectrum;
  unsigned long long *stats;
  unsigned long long *est_fix;  // [2 S] J, nu_bar in fixed point (this block's copy)
  unsigned long long *jb_fix;   // [S L] J_blue in fixed point (the j_blue buffer, converted after the launch)
  float inv_nu_ref, nu_ref;
  const double *planck;
  int32_t S, L, spec_bins;
  uint32_t key0, key1, iteration;
  double spec_lo, spec_dnu, e_cmf, nu_scale;
  uint64_t max_segments, first_packet;
  float x0, x0sq;
  int32_t *rec_status;
  double *rec_nu, *rec_e;
  unsigned long long *rec_cnt;
};

__device__ __forceinline__ void load_ctx(MCtx &c, const TransportParams &q, const float *shell) {
  c.S = q.S;
  c.L = q.L;
  c.xi2 = shell;
  c.xo2 = shell + q.S;
  c.kap = shell + 2 * q.S;
  c.ikap = shell + 3 * q.S;
  c.nu = q.nu;
  c.tau32 = q.tau32;
  c.row_info = q.row_info;
  c.line_row = q.line_row;
  c.ma_row = q.ma_row;
  c.ma_jump = q.ma_jump;
  c.bucket = q.dbr_bucket;
  c.rec = q.dbr_rec;
  c.inv_nu32 = q.inv_nu32;
  c.j_blue = q.j_blue;
  c.j_est = q.j_est;
  c.nu_bar = q.nu_bar;
  c.spectrum = q.spectrum;
  c.stats = q.stats;
  c.est_fix = q.est_fix + static_cast<size_t>(blockIdx.x % q.est_copies) * 2 * q.S;
  c.jb_fix = reinterpret_cast<unsigned long long *>(q.j_blue);
  c.inv_nu_ref = static_cast<float>(q.inv_nu_ref);
  c.nu_ref = static_cast<float>(q.nu_scale);
  c.planck = q.planck_cdf;
  c.spec_bins = q.spec_bins;
  c.key0 = q.key0;
  c.key1 = q.key1;
  c.iteration = q.iteration;
  c.spec_lo = q.spec_lo;
  c.spec_dnu = q.spec_dnu;
  c.e_cmf = q.e_cmf;
  c.nu_scale = q.nu_scale;
  c.max_segments = q.max_segments;
  c.first_packet = q.first_packet;
  c.x0 = static_cast<float>(q.x_in[0]);
  c.x0sq = shell[0];
  c.rec_status = q.rec_status;
  c.rec_nu = q.rec_nu;
  c.rec_e = q.rec_e;
  c.rec_cnt = q.rec_cnt;
}

__device__ __forceinline__ int32_t first_redward_m(const double *nu, int32_t L, double v) {
  const long long kv = __double_as_longlong(v);
  const long long *nb = reinterpret_cast<const long long *>(nu);
  int32_t lo = 0, hi = L;
  while (lo < hi) {
    const int32_t mid = (lo + hi) >> 1;
    if (__ldg(nb + mid) < kv) hi = mid; else lo = mid + 1;
  }
  return lo;
}

// binary32 value of a positive binary64 (given as its bit pattern) inside
// binary32's normal range, rounded toward zero, with integer operations only
// (the line frequencies are validated to lie in that range).
__device__ __forceinline__ float f32_of_positive_f64(long long bits) {
  const unsigned long long b = static_cast<unsigned long long>(bits);
  const uint32_t e = static_cast<uint32_t>(b >> 52) - 1023u + 127u;
  const uint32_t m = static_cast<uint32_t>(b >> 29) & 0x7fffffu;
  return __uint_as_float((e << 23) | m);
}

// Conversions between binary32 and binary64 with integer operations only
// (on this GPU a conversion through the binary64 pipe costs as much as a
// binary64 multiply).  Exact binary64 value of a finite binary32 (binary32
// subnormals, below 1.2e-38, are taken as zero):
__device__ __forceinline__ double f64_of_f32(float x) {
  const uint32_t b = __float_as_uint(x);
  const uint32_t e = (b >> 23) & 0xffu;
  const unsigned long long bits = (static_cast<unsigned long long>(b >> 31) << 63) |
                                  (static_cast<unsigned long long>(e + (1023u - 127u)) << 52) |
                                  (static_cast<unsigned long long>(b & 0x7fffffu) << 29);
  return e ? __longlong_as_double(static_cast<long long>(bits)) : 0.0;
}
// binary32 of max(d, 0) for a binary64 d below binary32's overflow, rounded
// toward zero; values below binary32's normal range give zero.
__device__ __forceinline__ float f32_of_f64_max0(double d) {
  const long long bits = __double_as_longlong(d);
  const int e = static_cast<int>((static_cast<unsigned long long>(bits) >> 52) & 0x7ffu) - (1023 - 127);
  const uint32_t m = static_cast<uint32_t>(static_cast<unsigned long long>(bits) >> 29) & 0x7fffffu;
  return (bits > 0 && e > 0) ? __uint_as_float((static_cast<uint32_t>(e) << 23) | m) : 0.0f;
}

__device__ __forceinline__ float max0f(float v) { return v > 0.0f ? v : 0.0f; }

// Macro atom (Sect. 2.5): the binary64 kernel's walk (integer thresholds, the
// same draws in the same order) on a lane's model context; returns the
// branching-row info of the level the atom deactivates from.
// In lone-walker mode (wd non-null) the draws come from the warp's buffer,
// and past its end each is computed on its own: the same values either way.
__device__ __forceinline__ unsigned long long ma_draw(DrawStream &ds, const WarpDraws *wd) {
  if (!wd) return ds.next_u53();
  if (ds.d - wd->base < kWarpDraws) return wd->take_u53(ds);
  ++ds.d;
  return u53_past_buffer(ds.k0, ds.k1, ds.packet, ds.iteration, ds.d - 1u);
}

struct LoneMaDraws {
  DrawStream *ds;
  const WarpDraws *wd;
  __device__ __forceinline__ unsigned long long next() const { return ma_draw(*ds, wd); }
};

__device__ __forceinline__ unsigned long long macroatom_walk_m(const MCtx &c, int32_t row, DrawStream &ds,
                                                               const WarpDraws *wd) {
  for (uint32_t n = 0; n < kMaMaxJumps; ++n) {
    const MaRow *mr = c.ma_row + row;
    const unsigned long long thr = __ldg(&mr->jump_thr);
    const uint2 jb = __ldg(reinterpret_cast<const uint2 *>(&mr->jump_begin));  // begin, length
    const unsigned long long za = ma_draw(ds, wd);
    if (!(za < thr)) {
      const uint2 db = __ldg(reinterpret_cast<const uint2 *>(&mr->dbr_begin));
      return static_cast<unsigned long long>(db.x) | (static_cast<unsigned long long>(db.y) << 32);
    }
    const unsigned long long zb = ma_draw(ds, wd);
    const MaJump *jp = c.ma_jump + jb.x;
    int32_t next = __ldg(&jp[jb.y - 1].target);
    for (uint32_t k = 0; k < jb.y; ++k) {
      if (zb < __ldg(&jp[k].thr)) { next = __ldg(&jp[k].target); break; }
    }
    row = next;
  }
  const uint2 db = __ldg(reinterpret_cast<const uint2 *>(&c.ma_row[row].dbr_begin));
  return static_cast<unsigned long long>(db.x) | (static_cast<unsigned long long>(db.y) << 32);
}

// x mu at the shell exit, +sqrt(x_out^2 - q) or -sqrt(x_in^2 - q).
__device__ __forceinline__ float shell_exit_f(float q, bool inner, float xi2, float xo2) {
  const float root = sqrtf(max0f((inner ? xi2 : xo2) - q));
  return inner ? -root : root;
}

// Does an event at path length l come before the shell exit?  x mu grows by
// l along the ray and x^2 = q + (x mu)^2: before an outward exit exactly when
// x^2 < x_out^2 there; before an inner exit exactly when x mu < 0 and
// x^2 > x_in^2 there.
__device__ __forceinline__ bool inside_shell_f(float pp, float q, float l, bool inner, float xi2,
                                               float xo2) {
  const float pl = pp + l;
  const float r2 = fmaf(pl, pl, q);
  return inner ? (pl < 0.0f && r2 > xi2) : r2 < xo2;
}

// uniform in (0, 1] with 24 random bits (a 32-bit conversion)
__device__ __forceinline__ float open0f(unsigned long long u53) {
  return static_cast<float>(static_cast<uint32_t>(u53 >> 29) + 1u) * 0x1.0p-24f;
}

struct Stats {
  unsigned long long v[kNStats];
};

__device__ __forceinline__ void flush_stats(Stats &st, unsigned long long *dst) {
#pragma unroll
  for (int i = 0; i < kNStats; ++i) {
    if (st.v[i]) atomicAdd(dst + i, st.v[i]);
    st.v[i] = 0ull;
  }
}

// What the pool keeps of a walk (and its model in a batch).
__device__ __forceinline__ PoolWalk pack_walk(const PacketM &pk, uint32_t d, int32_t model) {
  PoolWalk w;
  w.f[0] = pk.nu_lab;
  w.f[1] = static_cast<double>(model);
#pragma unroll
  for (int k = 2; k < 8; ++k) w.f[k] = 0.0;
  w.i[0] = static_cast<uint32_t>(pk.shell);
  w.i[1] = static_cast<uint32_t>(pk.next_line);
  w.i[2] = pk.pid;
  w.i[3] = d;
  w.i[4] = pk.have_inv_D ? 1u : 0u;
  w.i[5] = __float_as_uint(pk.p);
#pragma unroll
  for (int k = 0; k < kNCounters; ++k) w.i[6 + k] = pk.cnt[k];
  w.i[12] = __float_as_uint(pk.q);
  w.i[13] = __float_as_uint(pk.e_lab);
  w.i[14] = __float_as_uint(pk.inv_nu);
  w.i[15] = __float_as_uint(pk.inv_D);
  return w;
}

// One kernel source serves a single model (p.n_models == 0) and a batch, so a
// model's results do not depend on the company it is launched in.  It is
// compiled twice: MINB = 1 (blocks of 128 threads, three per SM at up to 168
// registers, with lone walks) for single models and for batches of 128
// threads a block, and MINB = 2 for batches of 64 or 256 threads or of many models,
// and for short line lists (128 registers: 16 resident warps per SM, without lone walks).  A batch of 12
// uneven models (2.9e6 packets): 330 ms a launch with the second (26 ms until
// the queue is empty, then the longest walks at 2.5 us a segment), 209 ms with
// the first (34 ms, and 1.3 us), 185 since the lone loop takes fewer
// instructions; of 40: 577 (156) and 430 (187), now 397.  The arithmetic
// is the same instruction for instruction, lone walks included; the batch
// tests check the bits.
template <int MODE, bool JB, bool REC, int MINB>
__global__ void __launch_bounds__(MINB == 1 ? 128 : kMaxBlock, MINB == 1 ? 3 : MINB)
    transport_mixed(const TransportParams p) {
  extern __shared__ unsigned long long smem_u64[];
  const unsigned lane = threadIdx.x & 31u;
  const unsigned lanemask_lt = (1u << lane) - 1u;
  const unsigned long long jb_pol = l2_evict_first_policy();
  MCtx c;
  int32_t cur_model = -1;
  unsigned long long *prefix = smem_u64;
  const bool batch = p.n_models > 0;
  constexpr bool kLoneBuild = MINB == 1;
  if (batch) {
    for (int i = threadIdx.x; i <= p.n_models; i += blockDim.x) prefix[i] = p.batch_prefix[i];
    __syncthreads();
  } else {
    float *shf = reinterpret_cast<float *>(smem_u64);
    for (int i = threadIdx.x; i < 4 * p.S; i += blockDim.x) shf[i] = p.shell32[i];
    __syncthreads();
    load_ctx(c, p, shf);
    cur_model = 0;
  }
  const unsigned long long t_start = global_ns();
  uint32_t polls = 0u;  // loop iterations between looks at the host's stop request
  if (lane == 0u) atomicCAS(p.flags + 3, 0ull, t_start);

  PacketM pk;
  DrawStream ds;
  // few packets are spread over all warps of the grid, so many to each (see the
  // binary64 kernel)
  const unsigned long long n_warps = static_cast<unsigned long long>(gridDim.x) * (blockDim.x >> 5);
  const unsigned quota = static_cast<unsigned>(min(32ull, (p.n_packets + n_warps - 1ull) / n_warps));
  bool alive = false, finished = lane >= quota;
  // Lone walks (kLoneBuild): once the packet queue is empty and few walks of a
  // warp are left, or a walk comes from the pool, every lane takes one walk's
  // state and runs its segments, as in the binary64 kernel: the lanes load the
  // line list 32 lines at a time in one coalesced load (line lwin_j0 + lane in
  // each lane), scan the window in one step, compute the walk's draws 64 at a
  // time into a per-warp shared buffer, and only lane 0 makes the walk's side
  // effects.
  WarpDraws wd;
  unsigned long long *warp_mem =
      smem_u64 + (batch ? static_cast<size_t>(p.n_models) + 1 : 2 * static_cast<size_t>(p.S)) +
      kLoneWords * (threadIdx.x >> 5);
  wd.init(!kLoneBuild ? nullptr : warp_mem + sizeof(PoolWalk) / sizeof(unsigned long long));
  bool drained = false;  // warp-uniform: the packet queue is empty
  bool lone = false;
  int tries = 0;
  int32_t lwin_j0 = 0, lwin_s = -1;
  long long lwin_b = 0;
  float lwin_t = 0.0f;
  unsigned long long lwin_r = 0ull;
  Stats st;
#pragma unroll
  for (int i = 0; i < kNStats; ++i) st.v[i] = 0ull;
  int32_t acc_s = -1;
  unsigned long long acc_j = 0ull, acc_nb = 0ull;  // fixed point, see kEstFixScale
  // the lane's current shell and its constants (reloaded on a shell or model change)
  int32_t cs = -1;
  float c_kap = 0.0f, c_ikap = 0.0f, c_xi2 = 0.0f, c_xo2 = 0.0f;
  // MINB == 1: lines next_line, next_line + 1 of the next segment,
  // loaded by the event that began it (see the binary64 kernel)
  bool lw_ok = false;
  long long lw_b0 = 0, lw_b1 = 0;
  float lw_t0 = 0.0f, lw_t1 = 0.0f;
  unsigned long long lw_r0 = 0ull, lw_r1 = 0ull;

  for (;;) {
    const bool need = !lone && !alive && !finished;
    const unsigned needmask = lone ? 0u : __ballot_sync(0xffffffffu, need);
    if (needmask) {
      const int leader = __ffs(needmask) - 1;
      unsigned long long base = 0ull;
      if (static_cast<int>(lane) == leader)
        base = atomicAdd(p.work_counter, static_cast<unsigned long long>(__popc(needmask)));
      base = __shfl_sync(0xffffffffu, base, leader);
      if (base + __popc(needmask) > p.n_packets) drained = true;
      if (need) {
        unsigned long long id = base + __popc(needmask & lanemask_lt);
        if (id < p.n_packets) {
          if (batch) {
            int lo = 0, hi = p.n_models;  // model m with prefix[m] <= id < prefix[m+1]
            while (hi - lo > 1) {
              const int mid = (lo + hi) >> 1;
              if (prefix[mid] <= id) lo = mid; else hi = mid;
            }
            if (lo != cur_model) {
              if (cur_model >= 0) {
                if (acc_s >= 0) {
                  atomicAdd(c.est_fix + acc_s, acc_j);
                  atomicAdd(c.est_fix + c.S + acc_s, acc_nb);
                }
                flush_stats(st, c.stats);
              }
              acc_s = -1; acc_j = 0ull; acc_nb = 0ull;
              load_ctx(c, p.batch[lo], p.batch[lo].shell32);
              cur_model = lo;
              cs = -1;
            }
            id -= prefix[lo];
          }
          // injection (Sect. 2.4), same draws as the binary64 kernel
          pk.pid = static_cast<uint32_t>(c.first_packet + id);
          ds.init(c.key0, c.key1, pk.pid, c.iteration);
          const double z0 = ds.closed0();
          const double z1 = ds.open0(), z2 = ds.open0(), z3 = ds.open0(), z4 = ds.open0();
          int l = 1;
          while (l < kPlanckLmax && c.planck[l] < z0) ++l;
          double xi = -log_pos(((z1 * z2) * z3) * z4);
          if (l > 1) xi = xi / static_cast<double>(l);
          const double nu_cmf = c.nu_scale * xi;
          const float mu = sqrtf(open0f(ds.next_u53()));
          const float pp = c.x0 * mu;
          const float D = 1.0f - pp;
          const float iD = 1.0f / D;
          pk.p = pp;
          pk.q = max0f(fmaf(-pp, pp, c.x0sq));
          pk.nu_lab = nu_cmf * static_cast<double>(iD);
          pk.e_lab = iD;  // E_lab / E_cmf(injection)
          pk.inv_nu = static_cast<float>(1.0 / nu_cmf) * D;
          pk.inv_D = iD;
          pk.have_inv_D = true;
          pk.shell = 0;
          pk.next_line = first_redward_m(c.nu, c.L, nu_cmf);
#pragma unroll
          for (int k = 0; k < kNCounters; ++k) pk.cnt[k] = 0u;
          alive = true;
          lw_ok = false;
        } else {
          finished = true;
          atomicCAS(p.flags + 1, 0ull, global_ns());
        }
      }
    }
    int from_pool = -1;
    if (!lone && __all_sync(0xffffffffu, finished && !alive)) {
      if (!kLoneBuild || !p.pool) break;
      if (lane == 0u) from_pool = pool_take(p);
      from_pool = __shfl_sync(0xffffffffu, from_pool, 0);
      if (from_pool < 0) break;
    }
    if (p.timeout_ns) {
      bool late = false;
      if (lane == 0u) late = (global_ns() - t_start) > p.timeout_ns;
      late = __shfl_sync(0xffffffffu, late, 0);
      if (late) {
        if (lane == 0u) atomicExch(p.flags, 1ull);
        break;
      }
    }
    if ((++polls & 255u) == 0u && p.cancel) {  // the host's stop request (mc_cancel)
      uint32_t stop = 0u;
      if (lane == 0u) stop = load_sys_u32(p.cancel);
      stop = __shfl_sync(0xffffffffu, stop, 0);
      if (stop) {
        if (lane == 0u) atomicExch(p.flags, 2ull);
        break;
      }
    }
    if (kLoneBuild) {
      if (lone) {
        wd.keep_u(ds, c.key0, c.key1, c.iteration, lane);
      } else {
        const unsigned live = __ballot_sync(0xffffffffu, alive);
        const unsigned n_live = __popc(live);
        bool go_lone = from_pool >= 0;
        if ((drained || quota == 1u) && n_live != 0u && n_live <= (p.pool ? kPoolLive : 1u))
          go_lone = n_live == 1u || __all_sync(0xffffffffu, !alive || pk.cnt[0] >= kPoolAge);
        if (go_lone) {
          // the lanes hand their estimator sums over; the warp keeps its oldest
          // walk, or takes one from the pool, and all lanes take its state
          const unsigned F = 0xffffffffu;
          if (acc_s >= 0) {
            atomicAdd(c.est_fix + acc_s, acc_j);
            atomicAdd(c.est_fix + c.S + acc_s, acc_nb);
          }
          acc_s = -1; acc_j = 0ull; acc_nb = 0ull;
          const PoolWalk *from = p.pool + from_pool;
          if (from_pool < 0) {
            const unsigned age = alive ? pk.cnt[0] + 1u : 0u;
            const unsigned oldest = __reduce_max_sync(F, age);
            const int owner = __ffs(__ballot_sync(F, age == oldest)) - 1;
            const PoolWalk w = pack_walk(pk, ds.d, cur_model);
            if (n_live > 1u) {
              const unsigned others = live & ~(1u << owner);
              unsigned long long place = 0ull;
              if (lane == 0u) place = atomicAdd(p.pool_ctl, static_cast<unsigned long long>(n_live - 1u));
              place = __shfl_sync(F, place, 0) + __popc(others & lanemask_lt);
              // (the pool holds what every warp can hand over once)
              if (((others >> lane) & 1u) && place < p.pool_cap) pool_put(p, static_cast<unsigned>(place), w);
            }
            if (static_cast<int>(lane) == owner) *reinterpret_cast<PoolWalk *>(warp_mem) = w;
            from = reinterpret_cast<const PoolWalk *>(warp_mem);
          }
          __syncwarp();
          {
            const volatile PoolWalk *w = from;  // (another SM may have written it: not through L1)
            pk.nu_lab = w->f[0];
            if (batch) {
              const int32_t model = static_cast<int32_t>(w->f[1]);
              if (model != cur_model) {
                if (cur_model >= 0) flush_stats(st, c.stats);
                load_ctx(c, p.batch[model], p.batch[model].shell32);
                cur_model = model;
              }
            }
            pk.shell = static_cast<int32_t>(w->i[0]);
            pk.next_line = static_cast<int32_t>(w->i[1]);
            pk.pid = w->i[2];
            ds.init(c.key0, c.key1, pk.pid, c.iteration);
            ds.d = w->i[3];
            pk.have_inv_D = w->i[4] != 0u;
            pk.p = __uint_as_float(w->i[5]);
#pragma unroll
            for (int k = 0; k < kNCounters; ++k) pk.cnt[k] = w->i[6 + k];
            pk.q = __uint_as_float(w->i[12]);
            pk.e_lab = __uint_as_float(w->i[13]);
            pk.inv_nu = __uint_as_float(w->i[14]);
            pk.inv_D = __uint_as_float(w->i[15]);
          }
          __syncwarp();
          cs = -1;
          lwin_s = -1;
          alive = true;
          lone = true;
          tries = kLoopTries;
          wd.pid = kNoPacket;
          wd.keep_u(ds, c.key0, c.key1, c.iteration, lane);
        }
      }
    }
    if (!alive) continue;
    const bool act = !lone || lane == 0u;  // makes the walk's side effects
    // the walk's next draw: from the warp's buffer in lone mode
    // (a macro atom's internal jumps can take more draws than the buffer holds)
    auto next_u = [&]() -> unsigned long long {
      if (!lone) return ds.next_u53();
      return MODE == 2 ? ma_draw(ds, &wd) : wd.take_u53(ds);
    };
    auto lone_reload = [&](int32_t s_, int32_t j0) {
      lwin_j0 = j0;
      lwin_s = s_;
      const int32_t jj = j0 + static_cast<int32_t>(lane);
      lwin_b = 0;
      lwin_t = 0.0f;
      lwin_r = 0ull;
      if (jj < c.L) {
        lwin_b = __ldg(reinterpret_cast<const long long *>(c.nu) + jj);
        lwin_t = __ldg(c.tau32 + static_cast<size_t>(s_) * static_cast<size_t>(c.L) + jj);
        if (MODE == 1) lwin_r = __ldg(c.row_info + jj);
      }
    };
    auto lone_fetch = [&](int32_t s_, int32_t jj, long long &b, float &t, unsigned long long &r) {
      int idx = jj - lwin_j0;
      if (lwin_s != s_ || idx < 0 || idx >= 32) {
        lone_reload(s_, jj);
        idx = 0;
      }
      b = __shfl_sync(0xffffffffu, lwin_b, idx);
      t = __shfl_sync(0xffffffffu, lwin_t, idx);
      r = __shfl_sync(0xffffffffu, lwin_r, idx);
    };

    if (kLoneBuild && MODE >= 1 && lone && tries > 0 && pk.next_line < c.L) {
      // Line event after line event of a lone walk, the bulk of a trapped walk,
      // in a loop of its own (the binary64 kernel's: loads stay in their
      // registers from where they are issued to where they are used).  The
      // absorbing line is the first one whose own depth absorbs, with the depths
      // before it as one integer reduction; the signs are taken in binary32 from
      // path lengths with a bound (ScanF's budget: this kernel's thresholds differ
      // from exact arithmetic by the roundings of c_e and of its products, a few
      // 2^-24 of either side) or, for the first line against the exit, exactly as
      // below.  It leaves, with nothing changed, at a segment that is anything
      // else or in doubt.  (Walk of 83,154 segments alone: 152 -> 91 ms, and 87 with
      // fewer instructions in the loop; 74 without J_blue.)
      const unsigned F = 0xffffffffu;
      const uint32_t cap = c.max_segments < 0xffffffffull ? static_cast<uint32_t>(c.max_segments) : 0xffffffffu;
      if (pk.shell != cs) {
        cs = pk.shell;
        c_kap = c.kap[cs];
        c_ikap = c.ikap[cs];
        c_xi2 = c.xi2[cs];
        c_xo2 = c.xo2[cs];
      }
      if (cs != acc_s) {
        if (acc_s >= 0 && act) {
          atomicAdd(c.est_fix + acc_s, acc_j);
          atomicAdd(c.est_fix + c.S + acc_s, acc_nb);
        }
        acc_s = cs; acc_j = 0ull; acc_nb = 0ull;
      }
      const long long *nub = reinterpret_cast<const long long *>(c.nu);
      const float *tau_s = c.tau32 + static_cast<size_t>(cs) * static_cast<size_t>(c.L);
      long long w_b;
      float w_t;
      unsigned long long w_r;
      int32_t w0 = pk.next_line;
      auto reload = [&]() {
        const int32_t jj = min(w0 + static_cast<int32_t>(lane), c.L - 1);
        w_b = static_cast<long long>(load_here(nub + jj));
        w_t = load_here_f(tau_s + jj);
        if (MODE == 1) w_r = load_here(c.row_info + jj);
        else w_r = load_here32(c.line_row + jj);
      };
      w_b = lwin_b;
      w_t = lwin_t;
      w_r = lwin_r;
      if (MODE == 2 || lwin_s != cs || lwin_j0 != w0) reload();
      double nu_c = pk.nu_lab * f64_of_f32(1.0f - pk.p), r1 = 0.0;
      float inv_c = 0.0f, g_w = 0.0f, g_b = 0.0f;
      uint32_t n_log = 0u;
      bool fresh = false;
      unsigned long long s_j = 0ull, s_nb = 0ull;  // this lane's sums of the logged segments
      auto sum_log = [&]() {
        s_j += __float2ull_rn(g_w);
        s_nb += __float2ull_rn(g_b);
        g_w = 0.0f;
        g_b = 0.0f;
        n_log = 0u;
      };
      // (The segments of the inner loop are counted out beforehand, as in the
      // binary64 kernel: to the next look at the clock and the stop word, the cap, 32
      // logged, three draws each.)
      bool certain = true;
      while (certain) {
        if (n_log == 32u) sum_log();
        wd.keep_u(ds, c.key0, c.key1, c.iteration, lane);
        uint32_t di = ds.d - wd.base, n_ev = 0u, n_line = 0u;
        uint32_t room = min(min(255u - (polls & 255u), cap - pk.cnt[0]), 32u - n_log);
        if (MODE != 2) room = min(room, (kWarpDraws - di) / 3u);
        if (room == 0u) break;
#pragma unroll 1
        do {
          const float tau0 = -__logf(open0f(wd.u[di]));
          unsigned long long u_em = wd.u[di + 1u], um = wd.u[di + 2u];
          const float pp = pk.p, q = pk.q, Df = 1.0f - pp;
          const bool inner = pp < 0.0f && q <= c_xi2;
          const float lx = Df - (1.0f - shell_exit_f(q, inner, c_xi2, c_xo2));
          ScanF f;
          f.tf = c_kap * Df;
          scan_frequency(f, nu_c, Df);
          // (each lane the record index of its own line, while the scan runs)
          const uint32_t my_slot = MODE == 1 ? bucket_index(w_r, u_em) : 0u;
          const bool there = w0 + static_cast<int32_t>(lane) < c.L;
          bool ok;
          const float l = scan_delta(f, w_b, ok) * f.lf;
          const float a = l * f.tf;
          const float own = there ? w_t : 0.0f;
          const float M = fmaf(0x1.0p-19f + 0x1.0p-18f, a + tau0, fmaf(f.tf, 0x1.0p-43f, 0x1.0p-100f));
          const float left = tau0 - a;
          const bool inside = lx - l > fmaf(0x1.0p-19f, l, 0x1.0p-43f);
          const unsigned thick = __ballot_sync(F, there && ok && left - own < -M);
          const int k = 31 - __clz(thick & (0u - thick));
          const long long hit = __shfl_sync(F, w_b, k);
          uint4 ra, rc;
          if (MODE == 1) load_slot_here64(c.bucket + __shfl_sync(F, my_slot, k), ra, rc);
          unsigned long long rinfo = __shfl_sync(F, w_r, k);
          const bool prior = static_cast<int>(lane) < k;
          const unsigned sum = __reduce_add_sync(
              F, prior ? __float2uint_rd(fminf(fmaxf(own, 0.0f), 63.0f) * 0x1.0p21f) : 0u);
          const float rk = left - static_cast<float>(sum) * 0x1.0p-21f;
          // (a line at or behind the packet, up to 2^-24 of the frequency after a
          // scattering or a crossing, has l = 0 here and a depth below 0 before it)
          const bool good = static_cast<int>(lane) == k
                                ? (f.ec > 0 && f.ec < 2047 && (inside || k == 0) && l > 0.0f &&
                                   rk > M + 0x1.0p-15f)
                                : !(prior && own < 0.0f);
          certain = __all_sync(F, good) && thick != 0u;
          if (!certain) break;
          if (fresh) {
            pk.nu_lab = nu_c * r1;
            pk.inv_nu = inv_c * Df;
            fresh = false;
          }
          const float inv_nu = pk.inv_nu;
          const double nu_cmf = pk.nu_lab * f64_of_f32(Df);
          const float lj = f32_of_f64_max0(nu_cmf - __longlong_as_double(hit)) * inv_nu;
          certain = k != 0 || inside_shell_f(pp, q, lj, inner, c_xi2, c_xo2);
          if (!certain) break;
          if (MODE == 2) {  // internal jumps, then the record of the level they end in
            ds.d = wd.base + di + 1u;
            const LoneMaDraws md{&ds, &wd};
            rinfo = macroatom_walk_lone(c.ma_row, c.ma_jump, static_cast<int32_t>(rinfo), md, lane);
            u_em = md.next();
            load_slot_here64(bucket_slot(c.bucket, rinfo, u_em), ra, rc);
            um = md.next();
            di = ds.d - wd.base;
          } else {
            di += 3u;
          }
          n_ev += 1u;
          n_line += static_cast<uint32_t>(k);
          if (JB && static_cast<int>(lane) <= k) {
            const float e_jb = ((pk.e_lab * inv_nu) * c.nu_ref) * kEstFixScaleF;
            red_add_evict_first(c.jb_fix + static_cast<size_t>(cs) * static_cast<size_t>(c.L) + w0 +
                                    static_cast<int32_t>(lane),
                                __float2ull_rn((f32_of_positive_f64(w_b) * inv_nu) * e_jb), jb_pol);
          }
          const float wgt = ((pk.e_lab * Df) * Df) * lj;
          if (lane == n_log) {
            g_w = wgt * kEstFixScaleF;
            g_b = (wgt * (f32_of_positive_f64(__double_as_longlong(nu_cmf)) * c.inv_nu_ref)) * kEstFixScaleF;
          }
          ++n_log;
          const float pl = pp + lj;
          const float r2n = fmaf(pl, pl, q);
          const float xn = sqrtf(r2n);
          const float e_c = pk.e_lab * (1.0f - pl);
          int32_t em = slot_line(ra, rc, u_em);
          if (em < 0) em = search_row_lone(c.rec, rinfo, rc.z, u_em, lane);
          w0 = em + 1;
          reload();
          nu_c = __longlong_as_double(static_cast<long long>(load_here(c.nu + em)));
          inv_c = load_here_f(c.inv_nu32 + em);
          // ... and while the window is on its way:
          const float mu2 = static_cast<float>(static_cast<int32_t>(um >> 29) - (1 << 23)) * 0x1.0p-23f;
          const float pn = xn * mu2;
          const float D2 = 1.0f - pn;
          const float iD2 = 1.0f / D2;
          const double r0 = f64_of_f32(iD2);
          r1 = fma(r0, fma(-f64_of_f32(D2), r0, 1.0), r0);
          pk.p = pn;
          pk.q = max0f(fmaf(-pn, pn, r2n));
          pk.e_lab = e_c * iD2;
          pk.inv_D = iD2;
          pk.have_inv_D = true;
          fresh = true;
        } while (n_ev != room && (MODE != 2 || di + 3u <= kWarpDraws));
        polls += n_ev;
        pk.cnt[0] += n_ev;
        pk.cnt[1] += n_line + n_ev;
        pk.cnt[2] += n_line + n_ev;
        pk.cnt[3] += n_ev;
        ds.d = wd.base + di;
      }
      if (fresh) {
        pk.nu_lab = nu_c * r1;
        pk.inv_nu = inv_c * (1.0f - pk.p);
      }
      sum_log();
      if (s_j) atomicAdd(c.est_fix + cs, s_j);
      if (s_nb) atomicAdd(c.est_fix + c.S + cs, s_nb);
      pk.next_line = w0;
      lwin_j0 = w0;
      lwin_s = cs;
      lwin_b = w_b;
      lwin_t = w_t;
      lwin_r = w_r;
      wd.keep_u(ds, c.key0, c.key1, c.iteration, lane);
    }
    int status = 0;
    if (pk.cnt[0] >= c.max_segments) {
      status = 3;
    } else {
      pk.cnt[0] += 1u;
      const int32_t s = pk.shell;
      const int32_t L = c.L;
      const float pp = pk.p, q = pk.q, inv_nu = pk.inv_nu;
      const double nu_lab = pk.nu_lab;
      const float Df = 1.0f - pp;
      const float inv_D = pk.have_inv_D ? pk.inv_D : 1.0f / Df;
      const double nu_cmf = nu_lab * f64_of_f32(Df);
      const float eD2 = (pk.e_lab * Df) * Df;
      if (s != cs) {
        cs = s;
        c_kap = c.kap[s];
        c_ikap = c.ikap[s];
        c_xi2 = c.xi2[s];
        c_xo2 = c.xo2[s];
      }
      const float kap = c_kap;
      const bool thomson = kap > 0.0f;
      const float tau0 = -__logf(open0f(next_u()));
      const float xi2 = c_xi2, xo2 = c_xo2;
      const bool inner = pp < 0.0f && q <= xi2;
      // shell exit threshold only once a line is passed or the exit wins
      // (see inside_shell_f)
      float p_exit = 0.0f;
      long long key_shell = kKeyNegInf;
      bool have_shell = false;
      float c_e = 0.0f, tau_rem = tau0;
      double thr_e = 0.0;
      long long key_e = kKeyNegInf;
      if (thomson) {
        c_e = (f32_of_positive_f64(__double_as_longlong(nu_lab)) * c_ikap) * inv_D;  // nu_lab / k
        thr_e = nu_cmf - f64_of_f32(tau0 * c_e);
        key_e = rawkey(thr_e);  // compared only with positive keys
      }
      long long key_thr = key_e;
      // J_blue contribution E_lab (nu_j / nu_lab)^2 / nu_j = (nu_j / nu_lab) E_lab / nu_lab,
      // in units of E / nu_ref and 2^-32 (fixed point, like J and nu_bar)
      const float e_jb = JB ? ((pk.e_lab * inv_nu) * c.nu_ref) * kEstFixScaleF : 0.0f;
      const size_t row = static_cast<size_t>(s) * static_cast<size_t>(L);
      const float *tau_s = c.tau32 + row;
      const long long *nub = reinterpret_cast<const long long *>(c.nu);
      int32_t j = pk.next_line;
      int kind = 0;
      float l = 0.0f;
      double nu_hit = 0.0;
      unsigned long long rinfo_hit = 0ull;
      long long bj = 0, bj_n = 0;
      float taul = 0.0f, tau_n = 0.0f;
      unsigned long long rinfo = 0ull, rinfo_n = 0ull;
      // An absorbing line (Sect. 2.6): with no line passed yet its Sobolev
      // point is also placed against the shell exit; if the exit comes first
      // the scan ends with no event (kind stays 0).
      auto absorb = [&](long long b_, unsigned long long r_) {
        const double nuj = __longlong_as_double(b_);
        const float lj = f32_of_f64_max0(nu_cmf - nuj) * inv_nu;
        if (!have_shell && !inside_shell_f(pp, q, lj, inner, xi2, xo2)) return;  // exit comes first
        pk.cnt[2] += 1u;
        if (JB && act)
          red_add_evict_first(c.jb_fix + row + j, __float2ull_rn((f32_of_positive_f64(b_) * inv_nu) * e_jb), jb_pol);
        kind = kLineEvent;
        l = lj;
        nu_hit = nuj;
        rinfo_hit = r_;
      };
      bool fast = false;  // the lone scan settled the segment's line event
      // downbranch: the absorbing line's emission record, loaded as soon as the
      // lone scan names the line (the emission draw is the next in the buffer)
      bool have_slot = false;
      uint4 slot_a = make_uint4(0u, 0u, 0u, 0u), slot_h = slot_a;
      if (lone) {
        int idx = j - lwin_j0;
        if (lwin_s != s || idx < 0 || idx >= 32) {
          lone_reload(s, j);
          idx = 0;
        }
        if (thomson) {
          // The scan of lines j0 + idx .. j0 + 31 of the window in one step (the
          // binary64 kernel's window scan in this kernel's arithmetic): in the
          // scan below the threshold after line k is T_k = thr_e + sum of the
          // binary32 products tau_i c_e (binary64 sums); it stops at line k when
          // nu_k <= T_{k-1} (beyond d_e), when nu_k lies beyond the shell exit
          // (exact key comparison), or when T_k > nu_k (absorbed).  Each lane
          // forms A = nu_k - T_{k-1} and B = nu_k - T_k in binary32 from the
          // binary64 difference nu_k - thr_e (truncated) and a prefix sum of the
          // same products, with a bound M on |error|: the truncation (2u) and
          // the five summation levels (5u), the final difference (u), the scan's
          // binary64 sums (at most 2^-48 (|thr_e| + C)) and products below the
          // binary32 normal range that the scan drops (32 2^-126):  M = 2^-20
          // (|d| + C) + 2^-44 |thr_e| + 2^-120.  Where every sign up to the first
          // line that stops the scan is certain and that line absorbs, the
          // result is the scan's; otherwise the scan below runs as usual.
          const float pe = shell_exit_f(q, inner, xi2, xo2);
          const long long ksh = rawkey(nu_lab * f64_of_f32(1.0f - pe));
          const int32_t jl = lwin_j0 + static_cast<int32_t>(lane);
          const bool cand = static_cast<int>(lane) >= idx;
          const bool valid = cand && jl < L;
          const float dk = f32_rz_any(__longlong_as_double(lwin_b) - thr_e);
          float P = valid ? lwin_t * c_e : 0.0f;
#pragma unroll
          for (int o = 1; o < 32; o <<= 1) {
            const float y = __shfl_up_sync(0xffffffffu, P, o);
            if (static_cast<int>(lane) >= o) P = __fadd_rn(P, y);
          }
          float Px = __shfl_up_sync(0xffffffffu, P, 1);
          if (lane == 0u) Px = 0.0f;
          const float A = __fsub_rn(dk, Px), B = __fsub_rn(dk, P);
          const float M = __fadd_rn(__fmul_rn(0x1.0p-20f, __fadd_rn(fabsf(dk), P)),
                                    __fadd_rn(__fmul_rn(0x1.0p-44f, fabsf(f32_rz_any(thr_e))), 0x1.0p-120f));
          const bool e_no = A > M;                      // certainly before d_e
          const bool a_yes = B < -M, a_no = B > M;      // certainly absorbed / passed
          const bool x_no = lwin_b > ksh;               // before the exit
          const bool pass = valid && e_no && a_no && x_no;
          const bool take = valid && e_no && a_yes && (static_cast<int>(lane) == idx || x_no);
          const unsigned stop = __ballot_sync(0xffffffffu, cand && !pass);
          const unsigned took = __ballot_sync(0xffffffffu, take);
          const int kstar = __ffs(stop) - 1;
          if (kstar >= 0 && ((took >> kstar) & 1u)) {
            fast = true;
            const int npass = kstar - idx;
            pk.cnt[1] += static_cast<uint32_t>(npass + 1);
            pk.cnt[2] += static_cast<uint32_t>(npass);
            if (JB && cand && static_cast<int>(lane) < kstar)  // the lines passed, one lane each
              red_add_evict_first(c.jb_fix + row + jl,
                                  __float2ull_rn((f32_of_positive_f64(lwin_b) * inv_nu) * e_jb), jb_pol);
            if (npass > 0) {  // as the scan leaves it after its first pass
              p_exit = pe;
              key_shell = ksh;
              have_shell = true;
            }
            j = lwin_j0 + kstar;
            bj = __shfl_sync(0xffffffffu, lwin_b, kstar);
            rinfo = __shfl_sync(0xffffffffu, lwin_r, kstar);
            if (MODE == 1) {
              load_slot(bucket_slot(c.bucket, rinfo, wd.peek_u53(ds)), slot_a, slot_h);
              have_slot = true;
            }
          }
        }
        if (!fast) {
          lone_fetch(s, j, bj, taul, rinfo);
          lone_fetch(s, j + 1, bj_n, tau_n, rinfo_n);
        }
      } else if (MINB == 1 && lw_ok) {
        bj = lw_b0; taul = lw_t0; rinfo = lw_r0;
        bj_n = lw_b1; tau_n = lw_t1; rinfo_n = lw_r1;
      } else {
        if (j < L) {
          bj = __ldg(nub + j);
          taul = __ldg(tau_s + j);
          if (MODE == 1) rinfo = __ldg(c.row_info + j);
        }
        if (j + 1 < L) {
          bj_n = __ldg(nub + j + 1);
          tau_n = __ldg(tau_s + j + 1);
          if (MODE == 1) rinfo_n = __ldg(c.row_info + j + 1);
        }
      }
      lw_ok = false;
      long long bj_nn = 0;
      float tau_nn = 0.0f;
      unsigned long long rinfo_nn = 0ull;
      if (fast) absorb(bj, rinfo);
      else while (j < L) {
        pk.cnt[1] += 1u;
        bj_nn = 0;
        tau_nn = 0.0f;
        rinfo_nn = 0ull;
        if (lone) {
          lone_fetch(s, j + 2, bj_nn, tau_nn, rinfo_nn);
        } else if (j + 2 < L) {
          bj_nn = __ldg(nub + j + 2);
          tau_nn = __ldg(tau_s + j + 2);
          if (MODE == 1) rinfo_nn = __ldg(c.row_info + j + 2);
        }
        if (bj <= key_thr) break;
        const double nuj = __longlong_as_double(bj);
        bool absorbed;
        double t = 0.0;
        if (thomson) {
          t = thr_e + f64_of_f32(taul * c_e);
          absorbed = rawkey(t) > bj;  // nu_j > 0
        } else {
          absorbed = taul > tau_rem;
        }
        if (!absorbed) {
          if (!have_shell) {  // a line is passed: the scan needs the exit threshold
            p_exit = shell_exit_f(q, inner, xi2, xo2);
            key_shell = rawkey(nu_lab * f64_of_f32(1.0f - p_exit));  // > 0
            have_shell = true;
            key_thr = key_shell > key_e ? key_shell : key_e;
            if (bj <= key_shell) break;  // this line lies beyond the exit
          }
          pk.cnt[2] += 1u;
          if (JB && act) red_add_evict_first(c.jb_fix + row + j, __float2ull_rn((f32_of_positive_f64(bj) * inv_nu) * e_jb), jb_pol);
          if (thomson) {
            thr_e = t;
            key_e = rawkey(t);
            key_thr = key_shell > key_e ? key_shell : key_e;
          } else {
            tau_rem -= taul;
          }
        } else {
          absorb(bj, rinfo);
          break;
        }
        ++j;
        bj = bj_n; taul = tau_n; rinfo = rinfo_n;
        bj_n = bj_nn; tau_n = tau_nn; rinfo_n = rinfo_nn;
      }
      if (kind == 0) {
        const float le = thomson ? f32_of_f64_max0(nu_cmf - thr_e) * inv_nu : 0.0f;
        const bool electron = have_shell ? key_e > key_shell
                                         : thomson && inside_shell_f(pp, q, le, inner, xi2, xo2);
        if (electron) {
          kind = kElectronEvent;
          l = le;
        } else {
          if (!have_shell) p_exit = shell_exit_f(q, inner, xi2, xo2);
          kind = kShellEvent;
          l = max0f(p_exit - pp);
        }
      }
      // estimators: binary32 contribution (units of E), summed in fixed point
      const float wgt = eD2 * l;
      if (s != acc_s) {
        if (acc_s >= 0 && act) {
          atomicAdd(c.est_fix + acc_s, acc_j);
          atomicAdd(c.est_fix + c.S + acc_s, acc_nb);
        }
        acc_s = s; acc_j = 0ull; acc_nb = 0ull;
      }
      // (x 2^32 is exact; the binary32 to integer conversions do not touch
      // the binary64 pipe)
      acc_j += __float2ull_rn(wgt * kEstFixScaleF);
      acc_nb += __float2ull_rn((wgt * (f32_of_positive_f64(__double_as_longlong(nu_cmf)) * c.inv_nu_ref)) *
                               kEstFixScaleF);
      pk.next_line = j;
      if (MODE >= 1) tries = kind == kLineEvent ? kLoopTries : tries - 1;
      if (kind == kShellEvent) {
        pk.cnt[5] += 1u;
        const int32_t ns = inner ? s - 1 : s + 1;
        pk.p = p_exit;
        pk.shell = ns;
        pk.have_inv_D = false;
        if (ns >= c.S) status = 1;
        else if (ns < 0) status = 2;
      } else {
        const float pl = pp + l;
        const float r2n = fmaf(pl, pl, q);
        const float xn = sqrtf(r2n);
        const float D1 = 1.0f - pl;
        const float e_c = pk.e_lab * D1;
        double nu_c;
        float inv_nu_c;
        if (kind == kLineEvent) {
          pk.cnt[3] += 1u;
          if (MODE >= 1) {
            // MODE 2: macro atom, internal jumps before the emission pick
            const unsigned long long rinfo_em =
                MODE == 2 ? macroatom_walk_m(c, __ldg(c.line_row + j), ds, lone ? &wd : nullptr) : rinfo_hit;
            const unsigned long long u_em = next_u();
            if (!have_slot) load_slot(bucket_slot(c.bucket, rinfo_em, u_em), slot_a, slot_h);
            int32_t emit = slot_line(slot_a, slot_h, u_em);
            if (emit < 0)
              emit = have_slot ? search_row_lone(c.rec, rinfo_em, slot_h.z, u_em, lane)
                               : search_row(c.rec, static_cast<uint32_t>(rinfo_em) + slot_h.z, u_em);
            nu_c = __ldg(c.nu + emit);
            inv_nu_c = __ldg(c.inv_nu32 + emit);
            pk.next_line = emit + 1;
            if (lone) {
              lone_reload(s, pk.next_line);
            } else if (MINB == 1) {  // the next segment's first lines, loaded now
              const int32_t nl = pk.next_line;
              lw_b0 = 0; lw_t0 = 0.0f; lw_r0 = 0ull; lw_b1 = 0; lw_t1 = 0.0f; lw_r1 = 0ull;
              if (nl < L) {
                lw_b0 = __ldg(nub + nl);
                lw_t0 = __ldg(tau_s + nl);
                if (MODE == 1) lw_r0 = __ldg(c.row_info + nl);
              }
              if (nl + 1 < L) {
                lw_b1 = __ldg(nub + nl + 1);
                lw_t1 = __ldg(tau_s + nl + 1);
                if (MODE == 1) lw_r1 = __ldg(c.row_info + nl + 1);
              }
              lw_ok = true;
            }
          } else {
            nu_c = nu_hit;
            inv_nu_c = 1.0f / f32_of_positive_f64(__double_as_longlong(nu_hit));
            pk.next_line = j + 1;
            if (MINB == 1) {  // lines j + 1, j + 2 are in the scan's registers
              lw_b0 = bj_n; lw_t0 = tau_n; lw_r0 = rinfo_n;
              lw_b1 = bj_nn; lw_t1 = tau_nn; lw_r1 = rinfo_nn;
              lw_ok = true;
            }
          }
        } else {
          pk.cnt[4] += 1u;
          nu_c = nu_lab * f64_of_f32(D1);
          inv_nu_c = inv_nu / D1;
          if (MINB == 1) {  // the next segment starts at line j again
            lw_b0 = bj; lw_t0 = taul; lw_r0 = rinfo;
            lw_b1 = bj_n; lw_t1 = tau_n; lw_r1 = rinfo_n;
            lw_ok = true;
          }
        }
        const unsigned long long um = next_u();
        const float mu2 = static_cast<float>(static_cast<int32_t>(um >> 29) - (1 << 23)) * 0x1.0p-23f;
        const float pn = xn * mu2;
        const float D2 = 1.0f - pn;
        const float iD2 = 1.0f / D2;
        // nu_lab = nu_c / D2 to binary64 accuracy: one Newton step on 1/D2
        const double D2d = f64_of_f32(D2), r0 = f64_of_f32(iD2);
        const double r1 = fma(r0, fma(-D2d, r0, 1.0), r0);
        pk.p = pn;
        pk.q = max0f(fmaf(-pn, pn, r2n));
        pk.nu_lab = nu_c * r1;
        pk.e_lab = e_c * iD2;
        pk.inv_nu = inv_nu_c * D2;
        pk.inv_D = iD2;
        pk.have_inv_D = true;
      }
    }
    if (status != 0 && !act) {  // a lone walk, not lane 0: drop it
      alive = false;
      lone = false;
      acc_s = -1;
      acc_j = 0ull;
      acc_nb = 0ull;
    } else if (status != 0) {
      lone = false;
      if (status == 1) st.v[kStEscaped] += 1ull;
      else if (status == 2) st.v[kStReabsorbed] += 1ull;
      else st.v[kStCapped] += 1ull;
      st.v[kStSegments] += pk.cnt[0];
      st.v[kStLineChecks] += pk.cnt[1];
      st.v[kStResonances] += pk.cnt[2];
      st.v[kStLineInteractions] += pk.cnt[3];
      st.v[kStEScatters] += pk.cnt[4];
      st.v[kStShellCrossings] += pk.cnt[5];
      const double e_lab = static_cast<double>(pk.e_lab) * c.e_cmf;
      if (status == 1) {
        int b;
        if (pk.nu_lab < c.spec_lo) b = c.spec_bins;
        else {
          const double t = (pk.nu_lab - c.spec_lo) / c.spec_dnu;
          b = (t >= 0.0 && t < static_cast<double>(c.spec_bins)) ? static_cast<int>(floor(t))
                                                                   : c.spec_bins + 1;
        }
        atomicAdd(c.spectrum + b, e_lab);
      }
      if (REC) {
        const uint64_t r = pk.pid - c.first_packet;
        c.rec_status[r] = status;
        c.rec_nu[r] = pk.nu_lab;
        c.rec_e[r] = e_lab;
#pragma unroll
        for (int k = 0; k < kNCounters; ++k) c.rec_cnt[r * kNCounters + k] = pk.cnt[k];
      }
      alive = false;
    }
  }
  if (cur_model >= 0) {
    if (acc_s >= 0 && (!lone || lane == 0u)) {  // (a launch stopped in lone mode)
      atomicAdd(c.est_fix + acc_s, acc_j);
      atomicAdd(c.est_fix + c.S + acc_s, acc_nb);
    }
    flush_stats(st, c.stats);
  }
  if (lane == 0u) atomicMax(p.flags + 2, global_ns());
}

template <int MODE, bool JB, bool REC, int MINB>
const void *kptr() {
  return reinterpret_cast<const void *>(&transport_mixed<MODE, JB, REC, MINB>);
}

template <int MINB>
const void *select_m(int line_mode, bool jb, bool rec) {
  if (line_mode == 0) {
    if (jb) return rec ? kptr<0, true, true, MINB>() : kptr<0, true, false, MINB>();
    return rec ? kptr<0, false, true, MINB>() : kptr<0, false, false, MINB>();
  }
  if (line_mode == 2) {
    if (jb) return rec ? kptr<2, true, true, MINB>() : kptr<2, true, false, MINB>();
    return rec ? kptr<2, false, true, MINB>() : kptr<2, false, false, MINB>();
  }
  if (jb) return rec ? kptr<1, true, true, MINB>() : kptr<1, true, false, MINB>();
  return rec ? kptr<1, false, true, MINB>() : kptr<1, false, false, MINB>();
}

const void *select_b(int line_mode, bool jb, bool rec) { return select_m<2>(line_mode, jb, rec); }

}  // namespace

// A single model's launches take the build with lone walks, except through
// downbranch or macro-atom lists below kLoneLinesSingle lines: 20 shells, 2000 lines,
// ms with it and without: 2000 packets 0.65 and 0.47, 2e4 0.87 and 0.69, 1e6 5.24 and 4.49;
// 5000 lines 1.31 and 1.13, 1.87 and 1.59, 8.43 and 7.44; 12 shells, 9000 lines 1.64 and
// 1.95, 2.92 and 3.04, 11.1 and 10.4; 15,000 lines 5.7 and 9.0, 6.8 and 9.9, 20.7 and 21.6.
// (Scattering lists: 2000 lines 1e6 packets 2.71 and 2.95, 12,347 lines 5.1 and 4.9.)
constexpr int kLoneLinesSingle = 6'000;
bool mixed_lone(int line_mode, int L) { return line_mode == 0 || L >= kLoneLinesSingle; }
const void *select_mixed_kernel(int line_mode, bool jb, bool rec, int L) {
  return mixed_lone(line_mode, L) ? select_m<1>(line_mode, jb, rec) : select_b(line_mode, jb, rec);
}

// single-model launches (128 threads): shell tables, then per warp a walk
// handed to all lanes and the lone walk's draw buffer
size_t mixed_smem_bytes(int S) {
  return 4 * static_cast<size_t>(S) * sizeof(float) + (128 / 32) * kLoneWords * sizeof(unsigned long long);
}

// Whether a batch's launches of 128 threads a block take the build with the lone
// walk.  Up to kLoneModels models:  Two batches on their own streams, model iterations/s
// with it and without: 2 x 8 models 78 and 45, 2 x 16 91 and 63, 2 x 32 133 and
// 111, 2 x 64 170 and 155, 2 x 128 188 and 189 (256 models, ten iterations with
// updates: 18.7 and 19.7 models/s): there one batch's queue fills the other's tail.
// And only where a model's line list is long, for walks to be trapped in: 8 models
// of 1e5 packets, ms with it and without: 3000 lines 4.90 and 4.01, 6000 7.67 and 6.59,
// 12,000 14.5 and 14.4, 25,000 31.0 and 37.8, 50,000 63 and 82; of 3000 packets 1.03 and 0.91,
// 2.10 and 1.74, 5.2 and 6.4, 11.9 and 19.4, 15.6 and 31.3.
constexpr int kLoneModels = 96, kLoneLines = 10'000;
bool batch_lone(int n_models, uint32_t most_lines) {
  return n_models <= kLoneModels && most_lines >= static_cast<uint32_t>(kLoneLines);
}

namespace {
const void *batch_kernel(int line_mode, bool jb, bool rec, bool lone, int block) {
  return lone && block == 128 ? select_m<1>(line_mode, jb, rec) : select_b(line_mode, jb, rec);
}
size_t batch_smem_bytes(int n_models, bool lone, int block) {
  return (static_cast<size_t>(n_models) + 1 + (lone && block == 128 ? 4 * kLoneWords : 0)) *
         sizeof(unsigned long long);
}
}  // namespace

cudaError_t batch_occupancy(int line_mode, bool j_blue, bool record, int n_models, bool lone, int block,
                            int *blocks_per_sm) {
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm,
                                                       batch_kernel(line_mode, j_blue, record, lone, block), block,
                                                       batch_smem_bytes(n_models, lone, block));
}

cudaError_t launch_transport_batch(const TransportParams &p, int line_mode, bool j_blue, bool record, bool lone,
                                   int grid, int block, cudaStream_t st) {
  void *args[] = {const_cast<TransportParams *>(&p)};
  return cudaLaunchKernel(batch_kernel(line_mode, j_blue, record, lone, block), dim3(grid), dim3(block), args,
                          batch_smem_bytes(p.n_models, lone, block), st);
}

}  // namespace mcgpu
