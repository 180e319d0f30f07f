// Monte Carlo packet transport through homologously expanding shells
// (Kerzendorf & Sim 2014, Sects. 2.4-2.7 and 2.9), one packet per thread in a
// persistent grid.
//
// GB300 notes.  A binary64 warp instruction occupies its SM sub-partition's
// pipe for 64 cycles, whatever the number of active lanes (a 64-bit integer
// high product takes 27, a binary32 operation 1), and a line-thick model is
// latency-bound by its longest random walks (the packet queue empties within a
// few percent of the kernel time), so the kernel minimises binary64
// instructions per flight segment:
//  * the packet carries p = x mu and q = x^2 - p^2 (conserved in free flight;
//    radii in units of c t_exp): D = 1 - p, x^2 = q + p^2, the shell exit is
//    at p = +-sqrt(x_b^2 - q) and a flight of length l is p += l;
//  * the line scan is decided in binary32 wherever an error bound allows, and
//    by a binary64 scan elsewhere (see ScanF);
//  * 1/nu_lab is carried and nu_lab taken only where it is needed, E/nu_lab is
//    carried instead of E_lab (the same in both frames);
//  * downbranch emission is an integer guide-table search, and the next
//    line's nu/tau loads are issued before the current line is resolved;
//  * lanes stay converged: a lane that finishes claims the next packet at the
//    loop head (warp-aggregated atomic); shell estimators accumulate in
//    registers and are flushed once per shell change;
//  * a warp down to its last live walk runs it with all 32 lanes (the lone
//    walk), and few packets are spread over all warps.
// Longest walk of the 500,000-line model (94,495 segments) alone, with J_blue: 212
// ms with a binary64 scan, 165 ms with the scan in binary32, 107 ms with the lone
// walk's line-event loop, 96 ms with reciprocal and square root on the integer
// pipe, 90 ms with fewer instructions in that loop (2.25 -> 0.95 us a segment,
// 0.81 without J_blue; bound by one warp's fixed latencies and its loads alike, see
// there); its 1e6-packet iteration 236 -> 104 to 119 ms (queue 9.9 -> 6.2 ms).
#pragma once

#include <cstdint>

#include "mc_device.cuh"
#include "mc_internal.h"

namespace mcgpu {

namespace {

constexpr int kBlock = 128;
// per warp: a walk handed to all lanes, then its draws
constexpr size_t kDrawBytes = kWarpDraws * (2 * sizeof(double) + sizeof(float));
constexpr size_t kLoneBytes = sizeof(PoolWalk) + kDrawBytes + 32 * 2 * sizeof(double2);
// doubles of the shell tables x_in^2, x_out^2, x_in, x_out, kappa (what follows is 16-byte aligned)
__host__ __device__ constexpr size_t shell_words(int S) { return (5 * static_cast<size_t>(S) + 1) & ~size_t{1}; }
constexpr int kLineEvent = 1, kElectronEvent = 2, kShellEvent = 3;

struct Packet {
  double p, q;  // x mu, x^2 - p^2
  // 1/nu_lab and E_lab / nu_lab = E_cmf / nu_cmf: the first-order Doppler
  // factor scales energy and frequency alike, so the ratio is the same in
  // both frames; it changes only when a line re-emits at another frequency
  // (Thomson and resonant scatterings keep both comoving values).
  double inv_nu, e_per_nu;
  // Frame quantities at the start of the next flight segment, carried from
  // the event that began it (have_cmf): D = 1 - p, the comoving frequency
  // and energy there; after a shell crossing they are taken from nu_lab.
  double D, nu_cmf, e_cmf;
  double nu_lab;  // have_lab: nu_cmf / D, taken where it is needed
  int32_t shell, next_line;
  uint32_t pid;
  bool have_cmf, have_lab;
  uint32_t cnt[kNCounters];
};

// First index j with nu[j] < v (nu strictly descending, positive): lower
// bound on the int64 images of the frequencies.
__device__ __forceinline__ int32_t first_redward(const double *nu, int32_t L, double v) {
  const long long kv = __double_as_longlong(v);
  const long long *nb = reinterpret_cast<const long long *>(nu);
  int32_t lo = 0, hi = L;
  while (lo < hi) {
    const int32_t mid = (lo + hi) >> 1;
    if (__ldg(nb + mid) < kv) hi = mid; else lo = mid + 1;
  }
  return lo;
}

// The emitted line of a downbranch row: through the bucket slots, or without
// them (caller-owned buffers) by bisection of the row's cdf.
template <bool SLOTS>
__device__ __forceinline__ int32_t downbranch_pick(const TransportParams &p, int32_t j,
                                                   unsigned long long rinfo, unsigned long long u) {
  if (SLOTS) {
    uint4 a, c;
    load_slot(bucket_slot(p.dbr_bucket, rinfo, u), a, c);
    const int32_t line = slot_line(a, c, u);
    return line >= 0 ? line : search_row(p.dbr_rec, static_cast<uint32_t>(rinfo) + c.z, u);
  }
  const int32_t row = __ldg(p.line_row + j);
  uint32_t lo = __ldg(p.dbr_offset + row), hi = __ldg(p.dbr_offset + row + 1) - 1u;
  const long long kz = __double_as_longlong(static_cast<double>(u) * 0x1.0p-53);
  const long long *cb = reinterpret_cast<const long long *>(p.dbr_cdf);
  while (lo < hi) {
    const uint32_t mid = (lo + hi) >> 1;
    if (kz < __ldg(cb + mid)) hi = mid; else lo = mid + 1u;
  }
  return static_cast<int32_t>(__ldg(p.dbr_line + lo));
}

// Macro atom (Sect. 2.5, mode macroatom): activated in level `row` (the
// absorbing line's upper level), the atom jumps -- decision draw u53 below
// the level's threshold, then a draw for the target -- until it deactivates;
// returns the branching-row info (begin | length << 32) of the level it
// deactivates from, for the emission pick.  After kMaMaxJumps jumps it
// deactivates without the decision draw.
template <class Draws>
__device__ __forceinline__ unsigned long long macroatom_walk(const TransportParams &p, int32_t row, const Draws &md) {
  for (uint32_t n = 0; n < kMaMaxJumps; ++n) {
    const MaRow *mr = p.ma_row + row;
    const unsigned long long thr = __ldg(&mr->jump_thr);
    const uint2 jb = __ldg(reinterpret_cast<const uint2 *>(&mr->jump_begin));  // begin, length
    const unsigned long long za = md.next();
    if (!(za < thr)) {
      const uint2 db = __ldg(reinterpret_cast<const uint2 *>(&mr->dbr_begin));
      return static_cast<unsigned long long>(db.x) | (static_cast<unsigned long long>(db.y) << 32);
    }
    const unsigned long long zb = md.next();
    const MaJump *jp = p.ma_jump + jb.x;
    int32_t next = __ldg(&jp[jb.y - 1].target);
    for (uint32_t k = 0; k < jb.y; ++k) {
      if (zb < __ldg(&jp[k].thr)) { next = __ldg(&jp[k].target); break; }
    }
    row = next;
  }
  const uint2 db = __ldg(reinterpret_cast<const uint2 *>(&p.ma_row[row].dbr_begin));
  return static_cast<unsigned long long>(db.x) | (static_cast<unsigned long long>(db.y) << 32);
}

// The emitted line of entries [lo, hi] of the caller's table by a whole warp: the
// first entry k with u 2^-53 < cdf[k] (the last's cdf is 1), 32 probes a round.
__device__ __forceinline__ int32_t search_cdf_lone(const TransportParams &p, uint32_t lo, uint32_t hi,
                                                   unsigned long long u, unsigned lane) {
  const long long kz = __double_as_longlong(static_cast<double>(u) * 0x1.0p-53);
  const long long *cb = reinterpret_cast<const long long *>(p.dbr_cdf);
  while (lo < hi) {
    const uint32_t n = hi - lo, step = (n + 31u) >> 5;
    const uint32_t i = lo + min((lane + 1u) * step, n) - 1u;
    const unsigned m = __ballot_sync(0xffffffffu, kz < __ldg(cb + i));
    if (m == 0u) {
      lo = hi;
    } else {
      const uint32_t k = static_cast<uint32_t>(__ffs(m)) - 1u;
      hi = lo + min((k + 1u) * step, n) - 1u;
      lo += k * step;
    }
  }
  return static_cast<int32_t>(__ldg(p.dbr_line + lo));
}

// max(v, 0) through the integer keys (no binary64 instruction).
__device__ __forceinline__ double max0(double v) { return rawkey(v) > 0 ? v : 0.0; }

// x mu at the shell exit: +sqrt(x_out^2 - q), or -sqrt(x_in^2 - q) when the
// ray meets the inner sphere.
__device__ __forceinline__ double shell_exit(double q, bool inner, double xi2, double xo2) {
  const double root = sqrt64((inner ? xi2 : xo2) - q);
  return inner ? -root : root;
}

// Injection at the inner boundary, Sect. 2.4: Planck-sampled comoving
// frequency (Carter & Cashwell series method), mu = sqrt(z), equal comoving
// energy (Eq. 10), lab-frame values by the first-order Doppler factor.
__device__ __forceinline__ double inject(const TransportParams &p, const double *planck, double x0,
                                         double x0sq, Packet &pk, DrawStream &ds) {
  const double z0 = ds.closed0();
  const double z1 = ds.open0(), z2 = ds.open0(), z3 = ds.open0(), z4 = ds.open0();
  int l = 1;
  while (l < kPlanckLmax && planck[l] < z0) ++l;
  double xi = -log_pos(((z1 * z2) * z3) * z4);
  if (l > 1) xi = xi / static_cast<double>(l);
  const double nu_cmf = p.nu_scale * xi;
  const double mu = sqrt(ds.open0());
  const double pp = x0 * mu;
  const double D = 1.0 - pp;
  pk.p = pp;
  pk.q = max0(fma(-pp, pp, x0sq));
  const double inv_nu_cmf = rcp64(nu_cmf);
  pk.e_per_nu = p.e_cmf * inv_nu_cmf;
  pk.inv_nu = inv_nu_cmf * D;
  pk.D = D;
  pk.nu_cmf = nu_cmf;
  pk.e_cmf = p.e_cmf;
  pk.have_cmf = true;
  pk.have_lab = false;
  pk.shell = 0;
#pragma unroll
  for (int c = 0; c < kNCounters; ++c) pk.cnt[c] = 0u;
  return nu_cmf;
}

// Spectrum bin of a lab frequency; below the range -> bins, above (or NaN)
// -> bins + 1 (Sect. 2.9 direct binning).
__device__ __forceinline__ int spectrum_bin(const TransportParams &p, double nu_lab) {
  if (nu_lab < p.spec_lo) return p.spec_bins;
  const double t = (nu_lab - p.spec_lo) / p.spec_dnu;
  return (t >= 0.0 && t < static_cast<double>(p.spec_bins)) ? static_cast<int>(floor(t)) : p.spec_bins + 1;
}

// ---- virtual packets (Sect. 2.9, Eqs. 19-21)
// Whenever an r-packet is about to start a trajectory (injection, or after an
// interaction), N_v v-packets leave its position with its comoving frequency
// and energy, in directions mu_v = mu_min + (1 - mu_min) z, z in (0, 1], with
// mu_min = -sqrt(1 - (x_in / x)^2) so that none meets the inner boundary.  A
// v-packet never interacts: it collects the Sobolev depths of the lines it
// passes and the electron-scattering depth kappa' D l of each segment (D at
// the segment start) on its way out, and adds exp(-tau_v) times its lab
// energy to the bin of its lab frequency.  Comoving energies: E (1 - mu_min)
// / (2 N_v) after an interaction (Eq. 19), E 2 mu_v / N_v at injection
// (Eq. 20).  Draws come from Philox stream 1 (counter word 3 = 1), the v-draw
// index counting on across the packet's launches, so the r-packet's own
// draws are untouched.

//
// A warp queues the launches of its r-packets in shared memory and, once there
// are 32, flies the v-packets of all of them with its 32 lanes, one v-packet
// each: a random walk then does not wait for its own v-packets on one lane (and
// a lone walk's 32 lanes have work of their own).  Each lane loads four lines
// ahead, and sums depths in fixed point (units of 2^-52), which takes no
// binary64 instruction for a line; a sum that reaches 512 moves to a binary64 one
// (a depth is not bounded, and negative ones may bring a sum back; the check of
// every line takes 1e5 packets of a 1e5-line model, three v-packets a launch and a
// cut of 30, from 65.2 to 68.0 ms; 416 when each lane flew its own launches).

struct VirtualLaunch {
  double x, r2, nu_cmf, e_cmf;  // radius (units of c t_exp), its square, comoving nu and E
  int32_t shell, next_line;     // shell: -1 at injection (in shell 0)
  uint32_t pid, first_draw;
};
constexpr int kVirtualQueue = 64;  // launches a warp holds: fewer than 32 left, and 32 more

__device__ __forceinline__ double vdraw_open0(const TransportParams &p, uint32_t pid, uint32_t d) {
  const uint4 o = philox4x32_10(make_uint4(d >> 1, pid, p.iteration, 1u), p.key0, p.key1);
  const unsigned long long u = (d & 1u) ? DrawStream::u53_of(o.z, o.w) : DrawStream::u53_of(o.x, o.y);
  return __ull2double_rn(u + 1ull) * 0x1.0p-53;
}

// A depth in units of 2^-52, rounded to nearest; 1024 (2^62) at most in magnitude.
__device__ __forceinline__ long long depth_fix(double t) {
  const unsigned long long b = static_cast<unsigned long long>(__double_as_longlong(t));
  const int e = static_cast<int>((b >> 52) & 0x7ffull) - 1023;
  const unsigned long long m = (b & 0x000fffffffffffffull) | 0x0010000000000000ull;
  unsigned long long v = e >= 10 ? 1ull << 62 : m << (e & 15);
  if (e < 0) v = e < -54 ? 0ull : (m + (1ull << (-e - 1))) >> -e;
  return b >> 63 ? -static_cast<long long>(v) : static_cast<long long>(v);
}

// Flies the v-packets of the queued launches.  Out of line: the transport loop
// keeps its registers.
__device__ __noinline__ void fly_virtual(const TransportParams &p, const double *sh, const VirtualLaunch *queue,
                                         unsigned count, unsigned lane) {
  const int32_t S = p.S, L = p.L;
  const unsigned nv = static_cast<unsigned>(p.n_virtual);
  const double *s_xi2 = sh, *s_xo2 = sh + S, *s_kap = sh + 4 * S;
  const long long *nub = reinterpret_cast<const long long *>(p.nu);
  const bool cut = rawkey(p.tau_v_max) > 0;
  auto cut_left = [&](double t) {
    const long long v = depth_fix(t);
    return cut && v < 1ll << 62 ? v : 0x7fffffffffffffffll;
  };
  auto in_range = [](long long v) { return static_cast<unsigned long long>(v + (1ll << 61)) < 1ull << 62; };
  __syncwarp();
  for (unsigned t = lane; t < count * nv; t += 32u) {
    const unsigned k = t / nv, i = t - k * nv;
    const VirtualLaunch v = queue[k];
    // x_in[0] / x with its remainder: 1 where x is x_in[0], and 1 - ri^2 loses nothing
    const double ix = rcp64(v.x), r0 = sh[2 * S] * ix, ri = fma(fma(-r0, v.x, sh[2 * S]), ix, r0);
    const double mu_min = -sqrt64(max0(fma(-ri, ri, 1.0)));
    const double mu_v = fma(1.0 - mu_min, vdraw_open0(p, v.pid, v.first_draw + i), mu_min);
    double pc = v.x * mu_v;
    const double D = 1.0 - pc, iD = rcp64(D);
    const double q = max0(fma(-pc, pc, v.r2));
    const double inv_nv = rcp64(static_cast<double>(p.n_virtual));
    const double e_v = (v.shell < 0 ? v.e_cmf * (2.0 * mu_v) : v.e_cmf * (0.5 * (1.0 - mu_min))) * inv_nv;
    const double nu_lab = v.nu_cmf * iD;
    // the depth so far: deep + tau 2^-52, |tau| < 2^61 (512) unless over the cut;
    // cap: what the cut leaves for tau (nothing exceeds the largest integer)
    long long tau = 0, cap = cut_left(p.tau_v_max);
    double deep = 0.0;
    auto add_deep = [&](double t) {
      deep += t + static_cast<double>(tau) * 0x1.0p-52;
      tau = 0;
      cap = cut_left(p.tau_v_max - deep);
    };
    int32_t s = v.shell < 0 ? 0 : v.shell, j = v.next_line;
    for (;;) {
      const double xi2 = s_xi2[s], xo2 = s_xo2[s];
      const bool inner = strictly_negative(pc) && rawkey(q) <= rawkey(xi2);
      const double p_exit = shell_exit(q, inner, xi2, xo2);
      // Sobolev points before the exit: nu_j > nu_lab (1 - p_exit)
      const long long key_exit = rawkey(nu_lab * (1.0 - p_exit));
      const double *tau_s = p.tau + static_cast<size_t>(s) * static_cast<size_t>(L);
      bool in = true;
      while (in) {
        long long b[4];
        double d[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const int32_t jj = min(j + c, L - 1);
          b[c] = __ldg(nub + jj);
          d[c] = __ldg(tau_s + jj);
        }
        bool wide = false;  // line j's depth leaves tau's range
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          in = in && j < L && b[c] > key_exit;
          if (in) {
            const long long sum = tau + depth_fix(d[c]);
            in = sum <= cap;
            wide = in && !in_range(sum);
            if (wide) {
              in = false;
            } else {
              tau = sum;
              ++j;
            }
          }
        }
        if (wide) {
          add_deep(__ldg(tau_s + j));
          ++j;
          in = tau <= cap;
        }
      }
      if (tau > cap) break;
      {
        const double t = (s_kap[s] * (1.0 - pc)) * max0(p_exit - pc);
        const long long sum = tau + depth_fix(t);
        if (sum <= cap && !in_range(sum)) add_deep(t);
        else tau = sum;
      }
      pc = p_exit;
      s += inner ? -1 : 1;
      // over the cut; out; or met the inner boundary (only by rounding)
      if (tau > cap || s >= S || s < 0) break;
    }
    if (s >= S && tau <= cap)
      atomicAdd(p.spectrum_v + spectrum_bin(p, nu_lab),
                (e_v * iD) * exp(-(deep + static_cast<double>(tau) * 0x1.0p-52)));
  }
  __syncwarp();
}

// ---- the line scan in binary32, with certainty
//
// The scan of Sect. 2.6 stops at the first line that lies beyond the
// electron-scattering point, beyond the shell exit, or absorbs the packet.
// Each of these is a sign, and nearly always one that binary32 settles: a
// line at path length l (units of c t_exp) is passed when
//   tau - C - kappa' D l > 0,   l < l_exit   and   tau - C - tau_k - kappa' D l > 0,
// C the depths of the lines passed before it.  Every quantity is formed in
// binary32 with a bound on its error that also covers the rounding of the
// binary64 scan below (exact_scan); where a sign lies within its bound, the
// segment is resolved by exact_scan, so that the events are the binary64
// scan's.  Binary64 warp instructions hold their SM sub-partition's pipe for 64
// cycles each; this takes the reciprocal 1/D, nu_lab, the thresholds and one
// fma per line off it, and the draw's binary64 logarithm (needed by exact_scan
// only): 40 -> 18 binary64 instructions for a line event.
//
// Error budget (u = 2^-24).  Frequency difference: the significands subtracted
// as integers in units of nu_cmf's last place (a line in a lower binade is
// truncated to it: at most one unit), converted in two halves (2u).  l: that
// difference (2u), D = 1 - p in binary32 (2u), 1/significand (truncated 2u, approximate
// reciprocal 2u) and two products (2u) -- below 2^-20 l.  kappa' D l: three
// more roundings -- below 2^-20 of it.  tau: its binary32 logarithm (8u); the
// depths: truncated (2u each), and n differences (u each of tau).  M = (2^-19 + n 2^-23) (kappa' D l + tau)
// + kappa' D (2^-44 + n 2^-51) + 2^-100 bounds these, the unit of the
// significands and the binary64 chain's n fmas (2^-53 nu each).
// Path length to the exit: x mu there is +-sqrt(x_b^2 - q) (P, in binary32 from
// the operands truncated, the difference's error e1 carried through the root).
// Near-tangent exits (x_b^2 - q within 4 e1) are not bounded.
__device__ __forceinline__ ScanF scan_setup(double nu_cmf, float pf, float qf, float kap, bool inner,
                                            float xi2, float xo2, float tau) {
  ScanF f;
  const float Df = 1.0f - pf;
  f.tf = kap * Df;
  f.tau = tau;
  const float xb2 = inner ? xi2 : xo2;
  const float dq = xb2 - qf;
  const float e1 = 0x1.0p-22f * (xb2 + dq);
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(dq));
  const float P = dq * r;
  f.lx = (inner ? -P : P) - pf;
  f.mx = dq >= 4.0f * e1 ? fmaf(0x1.0p-20f, P + fabsf(pf), fmaf(e1, r, 0x1.0p-44f)) : __int_as_float(0x7f800000);
  // (the frequency last: on a lone walk it is still on its way)
  scan_frequency(f, nu_cmf, Df);
  if (f.ec <= 0 || f.ec >= 2047) f.mx = __int_as_float(0x7f800000);
  return f;
}

// Draws of a lone walk, computed ahead by its warp: the walk's draws base ..
// base + 63 as u53, as the isotropic mu and as -ln of the open-interval draw
// (binary32).
struct LoneDraws {
  unsigned long long *u;
  double *m;
  float *t;
  uint32_t base;

  // All 32 lanes: refill when fewer than the three draws that a segment may
  // take are left (a macro atom's jumps past the end are computed one by one).
  __device__ __forceinline__ void keep(uint32_t d, uint32_t pid, uint32_t it, uint32_t k0, uint32_t k1,
                                       unsigned lane, bool first) {
    if (!first && d + 3u <= base + kWarpDraws) return;
    base = d & ~1u;
    const uint4 o = philox4x32_10(make_uint4((base >> 1) + lane, pid, it, 0u), k0, k1);
    __syncwarp();  // every lane has read the old contents
#pragma unroll 1
    for (int h = 0; h < 2; ++h) {
      const unsigned long long v = h ? DrawStream::u53_of(o.z, o.w) : DrawStream::u53_of(o.x, o.y);
      const int i = 2 * static_cast<int>(lane) + h;
      u[i] = v;
      t[i] = neg_log_u53_f(v + 1ull);
      m[i] = DrawStream::mu_from_u53(v);
    }
    __syncwarp();
  }
};

// A macro atom's draws: from the lane's own stream, or from a lone walk's
// buffer and past its end one by one.
struct MaDraws {
  DrawStream *ds;
  const LoneDraws *ld;  // nullptr: the lane's own stream
  uint32_t *d;
  uint32_t k0, k1, pid, it;
  __device__ __forceinline__ unsigned long long next() const {
    if (!ld) return ds->next_u53();
    const uint32_t i = (*d)++ - ld->base;
    return i < kWarpDraws ? ld->u[i] : u53_past_buffer(k0, k1, pid, it, *d - 1u);
  }
};

// LINES: what an absorbing line does -- 0 scatter, 1 downbranch, 2 macro atom,
// 3 downbranch from the caller's table alone (no bucket slots).
// VIRT: with virtual packets.
template <int LINES, bool JB, bool REC, bool VIRT>
__global__ void __launch_bounds__(kBlock, 3) transport_fp64(const TransportParams p) {
  constexpr int MODE = LINES == 3 ? 1 : LINES;
  constexpr bool kSlots = LINES == 1 || LINES == 2;  // the model's tables: bucket slots, row info
  extern __shared__ double sh[];
  const int32_t S = p.S, L = p.L;
  for (int i = threadIdx.x; i < S; i += blockDim.x) {
    const double xi = p.x_in[i], xo = p.x_out[i], kap = p.kappa[i];
    sh[i] = xi * xi;
    sh[S + i] = xo * xo;
    sh[2 * S + i] = xi;
    sh[3 * S + i] = xo;
    sh[4 * S + i] = kap;
  }
  __syncthreads();
  const double *s_xi2 = sh, *s_xo2 = sh + S, *s_kap = sh + 4 * S;
  const double x0 = sh[2 * S], x0sq = sh[0];

  const unsigned lane = threadIdx.x & 31u;
  const unsigned lanemask_lt = (1u << lane) - 1u;
  const unsigned long long jb_pol = l2_evict_first_policy();
  const unsigned long long t_start = global_ns();
  uint32_t polls = 0u;  // loop iterations between looks at the host's stop request
  if (lane == 0u) atomicCAS(p.flags + 3, 0ull, t_start);

  // Few packets are spread over all warps of the grid, so many to each: a warp
  // runs its lanes' events one kind after the other, and the binary64 pipe
  // serves a warp instruction for one lane or 32 in the same time.  (1000
  // packets of a 200-line scatter model: 126 -> 81 us with this and the scan.)
  const unsigned long long n_warps = static_cast<unsigned long long>(gridDim.x) * (kBlock / 32);
  const unsigned quota = static_cast<unsigned>(min(32ull, (p.n_packets + n_warps - 1ull) / n_warps));

  // this block's copy of the estimator sums
  double *j_sum = p.est_part ? p.est_part + static_cast<size_t>(blockIdx.x % p.est_copies) * 2 * S : p.j_est;
  double *nb_sum = p.est_part ? j_sum + S : p.nu_bar;

  Packet pk{};
  DrawStream ds;
  bool alive = false, finished = lane >= quota;
  bool drained = false;  // warp-uniform: the packet queue is empty
  uint32_t vdraws = 0u;  // v-packet draws used by this lane's packet
  // the warp's queued launches (VIRT)
  VirtualLaunch *vq = reinterpret_cast<VirtualLaunch *>(reinterpret_cast<char *>(sh + shell_words(S)) +
                                                        (kBlock / 32) * kLoneBytes) +
                      kVirtualQueue * (threadIdx.x >> 5);
  unsigned n_vq = 0u;
  // the lanes that have a launch queue it
  auto queue_virtual = [&](bool has, const VirtualLaunch &v) {
    const unsigned m = __ballot_sync(0xffffffffu, has);
    if (has) vq[n_vq + __popc(m & lanemask_lt)] = v;
    n_vq += __popc(m);
    if (n_vq >= kVirtualQueue / 2) {
      fly_virtual(p, sh, vq, n_vq, lane);
      n_vq = 0u;
    }
  };
  unsigned long long n_esc = 0, n_reab = 0, n_cap = 0, n_seg = 0, n_chk = 0, n_res = 0, n_lint = 0,
                     n_esca = 0, n_shell = 0;
  int32_t acc_s = -1;
  double acc_j = 0.0, acc_nb = 0.0;
  const long long *nub = reinterpret_cast<const long long *>(p.nu);
  // the lane's current shell and its constants (reloaded on a shell change)
  int32_t cs = -1;
  double c_xi2 = 0.0, c_xo2 = 0.0;
  float f_kap = 0.0f, f_xi2 = 0.0f, f_xo2 = 0.0f;
  auto enter_shell = [&](int32_t s_) {
    cs = s_;
    c_xi2 = s_xi2[s_];
    c_xo2 = s_xo2[s_];
    f_kap = f32_rz_any(s_kap[s_]);
    f_xi2 = f32_rz_any(c_xi2);
    f_xo2 = f32_rz_any(c_xo2);
  };
  // Lines next_line and next_line + 1 of the next segment (frequency bits,
  // Sobolev depth in the segment's shell, branching-row info), loaded by the
  // event that began it as soon as next_line is known, so that their latency
  // overlaps the event's arithmetic instead of opening the next scan.
  bool lw_ok = false;
  long long lw_b0 = 0, lw_b1 = 0;
  double lw_t0 = 0.0, lw_t1 = 0.0;
  unsigned long long lw_r0 = 0ull, lw_r1 = 0ull;
  auto load_window = [&](int32_t s_, int32_t j_) {
    const double *ts = p.tau + static_cast<size_t>(s_) * static_cast<size_t>(L);
    lw_b0 = 0; lw_t0 = 0.0; lw_r0 = 0ull; lw_b1 = 0; lw_t1 = 0.0; lw_r1 = 0ull;
    if (j_ < L) {
      lw_b0 = __ldg(nub + j_);
      lw_t0 = __ldg(ts + j_);
      if (LINES == 1) lw_r0 = __ldg(p.row_info + j_);
    }
    if (j_ + 1 < L) {
      lw_b1 = __ldg(nub + j_ + 1);
      lw_t1 = __ldg(ts + j_ + 1);
      if (LINES == 1) lw_r1 = __ldg(p.row_info + j_ + 1);
    }
    lw_ok = true;
  };

  // ---- steps of a segment, shared by a lane's own walk and the lone walk, so
  // that a packet's history does not depend on which of the two runs it
  // nu_lab, taken only where it is needed (a shell change, an electron
  // scattering, exact_scan, the end of the walk)
  auto need_lab = [&]() {
    if (!pk.have_lab) {
      pk.nu_lab = pk.nu_cmf * rcp64<true>(pk.D);
      pk.have_lab = true;
    }
  };
  // after a shell crossing: Doppler factor D = 1 - mu v/c at the boundary
  // point, comoving frequency and energy (Sect. 2.5)
  auto need_cmf = [&]() {
    if (!pk.have_cmf) {
      pk.D = 1.0 - pk.p;
      pk.nu_cmf = pk.nu_lab * pk.D;
      pk.e_cmf = pk.e_per_nu * pk.nu_cmf;
      pk.have_cmf = true;
    }
  };
  // The event of a segment that scanned lines [j0, j) without doubt, by
  // binary64 comparisons: frequency thresholds in place of path lengths (a
  // Sobolev point comes before d_e while nu_line > thr_e, and before the shell
  // exit while nu_line > nu_lab (1 - p_exit); a line of depth tau moves thr_e up by
  // tau nu_lab / k and absorbs exactly when thr_e then exceeds nu_line).
  // Updates j; nu_hit: the absorbing line's frequency bits; thr: thr_e.
  auto exact_scan = [&](unsigned long long u_tau, bool inner, int32_t j0, int32_t &j, bool act, double e_inv2, long long &nu_hit,
                        double &thr, double &p_exit) -> int {
    need_lab();
    const double tau = neg_log_u53(u_tau + 1ull);
    const double nu_lab = pk.nu_lab;
    const double *ts = p.tau + static_cast<size_t>(cs) * static_cast<size_t>(L);
    p_exit = shell_exit(pk.q, inner, c_xi2, c_xo2);
    const long long key_x = rawkey(nu_lab * (1.0 - p_exit));  // > 0
    const double kap = s_kap[cs];
    const bool thomson = rawkey(kap) > 0;
    double c_e = 0.0, rem = tau;
    long long key_e = kKeyNegInf;
    thr = 0.0;
    if (thomson) {
      c_e = (nu_lab * (p.inv_kappa ? __ldg(p.inv_kappa + cs) : 1.0 / kap)) * rcp64(pk.D);  // nu_lab / k, k = kappa' D
      thr = fma(-tau, c_e, pk.nu_cmf);
    }
    for (int32_t i = j0; i < j; ++i) {
      const double t = __ldg(ts + i);
      if (thomson) thr = fma(t, c_e, thr);
      else rem -= t;
    }
    if (thomson) key_e = rawkey(thr);
    for (; j < L; ++j) {
      const long long b = __ldg(nub + j);
      if (b <= key_e || b <= key_x) break;
      const double t = __ldg(ts + j);
      const double moved = fma(t, c_e, thr);
      if (thomson ? rawkey(moved) > b : rawkey(t) > rawkey(rem)) {
        nu_hit = b;
        return kLineEvent;
      }
      if (JB && act)
        red_add_evict_first(p.j_blue + static_cast<size_t>(cs) * static_cast<size_t>(L) + j, e_inv2, jb_pol);
      if (thomson) {
        thr = moved;
        key_e = rawkey(thr);
      } else {
        rem -= t;
      }
    }
    return (thomson && key_e > key_x) ? kElectronEvent : kShellEvent;
  };
  // Where an absorbing line's Sobolev point lies: nu_lab (1 - x mu) = nu_j (a
  // resonance that rounding puts behind the packet is taken where it is).
  auto line_point = [&](double nuj, double &l, double &r2) {
    l = max0(fma(-nuj, pk.inv_nu, pk.D));
    const double pl = rawkey(l) > 0 ? fma(-nuj, pk.inv_nu, 1.0) : pk.p;
    r2 = fma(pl, pl, pk.q);
  };
  // isotropic re-emission at radius^2 r2 with comoving frequency nu_c
  auto leave = [&](double r2, double mu, double nu_c, double inv_nu_c) -> double {
    const double xn = sqrt64(r2);
    const double pn = xn * mu;
    pk.D = fma(-xn, mu, 1.0);
    pk.p = pn;
    pk.q = max0(fma(-pn, pn, r2));
    pk.inv_nu = inv_nu_c * pk.D;
    pk.nu_cmf = nu_c;  // = nu_lab D
    pk.have_lab = false;
    return xn;
  };

  for (;;) {
    // ---- claim packets for idle lanes (one atomic per warp)
    const bool need = !alive && !finished;
    const unsigned needmask = __ballot_sync(0xffffffffu, need);
    if (needmask) {
      const int leader = __ffs(needmask) - 1;
      unsigned long long base = 0ull;
      if (static_cast<int>(lane) == leader)
        base = atomicAdd(p.work_counter, static_cast<unsigned long long>(__popc(needmask)));
      base = __shfl_sync(0xffffffffu, base, leader);
      if (base + __popc(needmask) > p.n_packets) drained = true;
      if (need) {
        const unsigned long long id = base + __popc(needmask & lanemask_lt);
        if (id < p.n_packets) {
          pk.pid = static_cast<uint32_t>(p.first_packet + id);
          ds.init(p.key0, p.key1, pk.pid, p.iteration);
          const double nu_cmf0 = inject(p, p.planck_cdf, x0, x0sq, pk, ds);
          if (quota != 1u) pk.next_line = first_redward(p.nu, L, nu_cmf0);
          alive = true;
          lw_ok = false;
          vdraws = 0u;
        } else {
          finished = true;
          atomicCAS(p.flags + 1, 0ull, global_ns());
        }
      }
    }
    const unsigned live = __ballot_sync(0xffffffffu, alive);
    if (quota == 1u && needmask && live) {  // the one packet just claimed
      const int32_t j = first_redward_warp(p.nu, L, __shfl_sync(0xffffffffu, pk.nu_cmf, 0), lane);
      pk.next_line = j;
    }
    if (VIRT && needmask) {  // the packets just injected (needmask: warp-uniform)
      const bool has = need && alive;
      queue_virtual(has, VirtualLaunch{x0, x0sq, pk.nu_cmf, p.e_cmf, -1, pk.next_line, pk.pid, 0u});
      if (has) vdraws = static_cast<uint32_t>(p.n_virtual);
    }
    int from_pool = -1;
    if (!live && __all_sync(0xffffffffu, finished)) {
      if (p.pool && lane == 0u) from_pool = pool_take(p);
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
    if (p.cancel && (++polls & 255u) == 0u) {  // the host's stop request (mc_cancel)
      uint32_t stop = 0u;
      if (lane == 0u) stop = load_sys_u32(p.cancel);
      stop = __shfl_sync(0xffffffffu, stop, 0);
      if (stop) {
        if (lane == 0u) atomicExch(p.flags, 2ull);
        break;
      }
    }
    const unsigned n_live = __popc(live);
    bool go_lone = from_pool >= 0;
    if ((drained || quota == 1u) && n_live != 0u && n_live <= (p.pool ? kPoolLive : 1u))
      go_lone = n_live == 1u || __all_sync(0xffffffffu, !alive || pk.cnt[0] >= kPoolAge);
    if (go_lone) {
      // ---- lone walk: the queue is empty and few walks of the warp are left (or
      // the launch has few packets for each warp).  The warp hands all but the
      // oldest to the pool -- walk lengths are heavy-tailed, so that the oldest is
      // expected to be the longest -- and runs that one with all 32 lanes to its
      // end, then takes others from the pool.  A walk that shares its warp
      // advances at 4 to 8 us a segment, a lone one at 0.8 to 0.95 (1.5 with all
      // warps of the SM in this mode).
      // All 32 lanes hold the walk's state; the line list comes 32 lines at a
      // time (line w0 + lane in each lane, one coalesced load), the scan of such a
      // window in one step, the draws computed ahead; lane 0 makes the walk's side
      // effects.  The loads of a line event are then two dependent ones (the
      // emission record, the window behind the emitted line); the event's binary64
      // arithmetic runs while they are in flight.
      const unsigned F = 0xffffffffu;
      if (acc_s >= 0) {
        atomicAdd(j_sum + acc_s, acc_j);
        atomicAdd(nb_sum + acc_s, acc_nb);
      }
      acc_s = -1;
      char *warp_mem = reinterpret_cast<char *>(sh + shell_words(S)) + kLoneBytes * (threadIdx.x >> 5);
      const PoolWalk *from = p.pool + from_pool;
      if (from_pool < 0) {
        const unsigned age = alive ? pk.cnt[0] + 1u : 0u;
        const unsigned oldest = __reduce_max_sync(F, age);
        const int owner = __ffs(__ballot_sync(F, age == oldest)) - 1;
        PoolWalk w;
        w.f[0] = pk.p; w.f[1] = pk.q; w.f[2] = pk.inv_nu; w.f[3] = pk.e_per_nu;
        w.f[4] = pk.D; w.f[5] = pk.nu_cmf; w.f[6] = pk.e_cmf; w.f[7] = pk.nu_lab;
        w.i[0] = static_cast<uint32_t>(pk.shell);
        w.i[1] = static_cast<uint32_t>(pk.next_line);
        w.i[2] = pk.pid;
        w.i[3] = ds.d;
        w.i[4] = (pk.have_cmf ? 1u : 0u) | (pk.have_lab ? 2u : 0u);
        w.i[5] = vdraws;
#pragma unroll
        for (int c = 0; c < kNCounters; ++c) w.i[6 + c] = pk.cnt[c];
#pragma unroll
        for (int c = 12; c < 16; ++c) w.i[c] = 0u;
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
      uint32_t d;
      {
        const volatile PoolWalk *w = from;  // (another SM may have written it: not through L1)
        pk.p = w->f[0]; pk.q = w->f[1]; pk.inv_nu = w->f[2]; pk.e_per_nu = w->f[3];
        pk.D = w->f[4]; pk.nu_cmf = w->f[5]; pk.e_cmf = w->f[6]; pk.nu_lab = w->f[7];
        pk.shell = static_cast<int32_t>(w->i[0]);
        pk.next_line = static_cast<int32_t>(w->i[1]);
        pk.pid = w->i[2];
        d = w->i[3];
        vdraws = w->i[5];
        pk.have_cmf = (w->i[4] & 1u) != 0u;
        pk.have_lab = (w->i[4] & 2u) != 0u;
#pragma unroll
        for (int c = 0; c < kNCounters; ++c) pk.cnt[c] = w->i[6 + c];
      }
      __syncwarp();
      LoneDraws ld;
      ld.u = reinterpret_cast<unsigned long long *>(warp_mem + sizeof(PoolWalk));
      ld.m = reinterpret_cast<double *>(ld.u + kWarpDraws);
      ld.t = reinterpret_cast<float *>(ld.m + kWarpDraws);
      ld.keep(d, pk.pid, p.iteration, p.key0, p.key1, lane, true);
      enter_shell(pk.shell);
      const uint32_t cap = p.max_segments < 0xffffffffull ? static_cast<uint32_t>(p.max_segments) : 0xffffffffu;
      int32_t w0 = 0;
      long long w_b = 0;
      double w_t = 0.0;
      unsigned long long w_r = 0ull;
      auto reload = [&](int32_t j_) {
        w0 = j_;
        // (lanes behind the list load its last line; the scan leaves them out)
        const int32_t jj = min(j_ + static_cast<int32_t>(lane), L - 1);
        w_b = static_cast<long long>(load_here(nub + jj));
        w_t = __longlong_as_double(static_cast<long long>(
            load_here(p.tau + static_cast<size_t>(cs) * static_cast<size_t>(L) + jj)));
        if (LINES == 1) w_r = load_here(p.row_info + jj);
        if (LINES >= 2) w_r = load_here32(p.line_row + jj);
      };
      reload(pk.next_line);
      // After a line's re-emission E/nu and 1/nu_lab are taken when the next event
      // needs them: the emitted line's frequency is in flight until then.  (Its
      // reciprocal from a table of 1/nu arrived later still: 4 MB touched at
      // random, mostly from DRAM.)
      bool fresh = false;
      auto settle = [&]() {
        if (fresh) {
          const double inv_c = rcp64<true>(pk.nu_cmf);
          pk.inv_nu = inv_c * pk.D;
          if (MODE >= 1) pk.e_per_nu = pk.e_cmf * inv_c;  // re-emitted at another frequency
          fresh = false;
        }
      };
      // The estimator terms of a segment (Eqs. 13-14) are logged in shared memory
      // (all lanes store the same values to one place) and evaluated for 32 segments
      // at once, a lane each.
      double2 *lg_x = reinterpret_cast<double2 *>(warp_mem + sizeof(PoolWalk) + kDrawBytes);
      uint32_t n_log = 0u;
      double a_j = 0.0, a_nb = 0.0;  // this lane's sums in shell cs
      auto sum_log = [&]() {
        __syncwarp();
        double wgt = 0.0, nu = 0.0;
        if (lane < n_log) {
          const double2 x = lg_x[2u * lane], y = lg_x[2u * lane + 1u];
          nu = y.y;
          wgt = ((x.x * nu) * (nu * x.y)) * y.x;  // E_cmf D l
        }
        __syncwarp();
        a_j += wgt;
        a_nb = fma(wgt, nu, a_nb);
        n_log = 0u;
      };
      auto put_log = [&](double l) {
        lg_x[2u * n_log] = make_double2(pk.e_per_nu, pk.inv_nu);
        lg_x[2u * n_log + 1u] = make_double2(l, pk.nu_cmf);  // path length, nu_cmf
        ++n_log;
      };
      auto log_segment = [&](double l, int32_t j, int32_t n) {
        if (n_log == 32u) sum_log();
        put_log(l);
        if (JB) {
          const double e_inv2 = pk.e_per_nu * pk.inv_nu;
          double *cell = p.j_blue + static_cast<size_t>(cs) * static_cast<size_t>(L) + j;
          for (int32_t i = static_cast<int32_t>(lane); __any_sync(F, i < n); i += 32)
            if (i < n) red_add_evict_first(cell + i, e_inv2, jb_pol);
        }
      };
      auto flush_shell = [&]() {
        sum_log();
        if (rawkey(a_j) > 0) {
          atomicAdd(j_sum + cs, a_j);
          atomicAdd(nb_sum + cs, a_nb);
        }
        a_j = 0.0;
        a_nb = 0.0;
      };
      int status = 0;
      bool stopped = false;
      need_cmf();
      while (status == 0) {
        if (LINES != 0) {
          // Line event after line event, the bulk of a trapped walk: a loop of its
          // own, so that the loads in flight stay in their registers from where
          // they are issued to where they are used (a copy of one where paths meet
          // would wait for it).  It leaves, with nothing changed, at a segment that
          // is anything else.
          // What bounded it was the number of its instructions (a lone warp issued
          // one in 5.9 cycles, 3.1 of them fixed latencies and 0.6 waits for loads; 416 a
          // segment).  So the segments it may take are counted out beforehand (to the
          // next look at the clock and the stop word, the cap, 32 logged, three draws
          // each), its counters are two, a segment's estimator terms are two shared
          // stores, and the J_blue terms of the lines passed one atomic of the lanes:
          // 361 a segment, and of the cycles between two 2.4 are fixed latencies, 1.1
          // shuffles, conversions and binary64, and 2.3 waits for the two dependent
          // loads, which the instructions no longer cover.  A walk of 94,495 segments
          // alone: 100.4 -> 76.0 ms, with J_blue (and its zeroing, which leaves the
          // caches cold) 96.0 -> 89.8; 5e4 lines, 1e5 packets: 32.6 -> 25.5 ms.
          bool certain = true;
          while (certain) {
            if (n_log == 32u) sum_log();
            ld.keep(d, pk.pid, p.iteration, p.key0, p.key1, lane, false);
            uint32_t di = d - ld.base, n_ev = 0u, n_line = 0u;
            uint32_t room = min(min(255u - (polls & 255u), cap - pk.cnt[0]), 32u - n_log);
            if (LINES != 2) room = min(room, (kWarpDraws - di) / 3u);
            if (room == 0u) break;
#pragma unroll 1
            do {
              unsigned long long u_em = ld.u[di + 1u];
              double mu = ld.m[di + 2u];
              const float pf = f32_rz_small(pk.p), qf = f32_rz_small(pk.q);
              // (truncation keeps the order, and at equality the exit is not bounded)
              const bool inner = pf < 0.0f && qf <= f_xi2;
              const ScanF f = scan_setup(pk.nu_cmf, pf, qf, f_kap, inner, f_xi2, f_xo2, ld.t[di]);
              // (each lane the record index of its own line, while the scan runs)
              const uint32_t my_slot = LINES == 1 ? bucket_index(w_r, u_em) : 0u;
              const bool there = w0 + static_cast<int32_t>(lane) < L;
              bool ok;
              const float l = scan_delta(f, w_b, ok) * f.lf;
              const float a = l * f.tf;
              const float own = there ? f32_rz_below_inf(w_t) : 0.0f;
              const float M = fmaf(0x1.0p-19f + 0x1.0p-18f, a + f.tau, fmaf(f.tf, 0x1.0p-43f, 0x1.0p-100f));
              const float left = f.tau - a;
              const bool inside = f.lx - l > fmaf(0x1.0p-19f, l, f.mx);
              // (a line of the caller's table that cannot absorb need not have a row)
              const unsigned thick = __ballot_sync(F, there && ok && left - own < -M && (LINES != 3 || own > 0.0f));
              const int k = 31 - __clz(thick & (0u - thick));
              const long long hit = __shfl_sync(F, w_b, k);
              uint4 ra, rc;
              uint32_t row_lo = 0u, row_hi = 0u;
              if (LINES == 1) load_slot_here(p.dbr_bucket + __shfl_sync(F, my_slot, k), ra, rc);
              unsigned long long rinfo = __shfl_sync(F, w_r, k);
              if (LINES == 3 && thick != 0u) {
                row_lo = load_here32(p.dbr_offset + rinfo);
                row_hi = load_here32(p.dbr_offset + rinfo + 1);
              }
              const bool prior = static_cast<int>(lane) < k;
              const unsigned sum = __reduce_add_sync(
                  F, prior ? __float2uint_rd(fminf(fmaxf(own, 0.0f), 63.0f) * 0x1.0p21f) : 0u);
              const float rk = left - static_cast<float>(sum) * 0x1.0p-21f;
              // (and the point lies ahead of the packet, beyond its rounding)
              const bool good = static_cast<int>(lane) == k ? (inside && rk > M + 0x1.0p-15f && l > 0x1.0p-40f)
                                                            : !(prior && own < 0.0f);
              certain = __all_sync(F, good) && thick != 0u;
              if (!certain) break;
              if (LINES == 2) {  // internal jumps, then the record of the level they end in
                d = ld.base + di + 1u;
                const MaDraws md{nullptr, &ld, &d, p.key0, p.key1, pk.pid, p.iteration};
                rinfo = macroatom_walk_lone(p.ma_row, p.ma_jump, static_cast<int32_t>(rinfo), md, lane);
                u_em = md.next();
                load_slot_here(bucket_slot(p.dbr_bucket, rinfo, u_em), ra, rc);
                mu = d - ld.base < kWarpDraws ? ld.m[d - ld.base] : DrawStream::mu_from_u53(u53_past_buffer(
                    p.key0, p.key1, pk.pid, p.iteration, d));
                di = d + 1u - ld.base;
              } else {
                di += 3u;
              }
              settle();
              n_ev += 1u;
              n_line += static_cast<uint32_t>(k);
              // line_point and sqrt64 without their special cases (a binary64
              // result takes 45 cycles longer to an integer compare than to the
              // next binary64 instruction)
              const double nuj = __longlong_as_double(hit);
              const double lp = fma(-nuj, pk.inv_nu, pk.D);
              const double pl = fma(-nuj, pk.inv_nu, 1.0);
              const double r2 = fma(pl, pl, pk.q);
              put_log(lp);
              if (JB) {
                const double e_inv2 = pk.e_per_nu * pk.inv_nu;
                if (static_cast<int>(lane) <= k)
                  red_add_evict_first(p.j_blue + static_cast<size_t>(cs) * static_cast<size_t>(L) + w0 +
                                          static_cast<int32_t>(lane), e_inv2, jb_pol);
              }
              int32_t em;
              if (kSlots) {
                // (not before r2 is there: scheduled earlier, it would wait for the
                // record with the event's arithmetic behind it)
                em = slot_line(ra, rc, u_em ^ (static_cast<unsigned long long>(
                                           static_cast<uint32_t>(__double2hiint(r2)) & p.zero) << 32));
                if (em < 0) em = search_row_lone(p.dbr_rec, rinfo, rc.z, u_em, lane);
              } else {
                em = search_cdf_lone(p, row_lo, row_hi - 1u, u_em, lane);
              }
              reload(em + 1);
              pk.next_line = em + 1;
              pk.nu_cmf = __longlong_as_double(static_cast<long long>(load_here(p.nu + em)));
              // ... and while the window is on its way:
              const double xn = sqrt64_pos(r2);
              pk.e_cmf = pk.e_per_nu * nuj;
              const double pn = xn * mu;
              pk.D = fma(-xn, mu, 1.0);
              pk.p = pn;
              pk.q = max0(fma(-pn, pn, r2));
              pk.have_lab = false;
              fresh = true;
              if (VIRT) {
                queue_virtual(lane == 0u, VirtualLaunch{xn, r2, pk.nu_cmf, pk.e_cmf, cs, em + 1, pk.pid, vdraws});
                vdraws += static_cast<uint32_t>(p.n_virtual);
              }
            } while (n_ev != room && (LINES != 2 || di + 3u <= kWarpDraws));
            polls += n_ev;
            pk.cnt[0] += n_ev;
            pk.cnt[1] += n_line + n_ev;
            pk.cnt[2] += n_line + n_ev;
            pk.cnt[3] += n_ev;
            d = ld.base + di;
          }
        }
        if (p.timeout_ns && __any_sync(F, (global_ns() - t_start) > p.timeout_ns)) {
          if (lane == 0u) atomicExch(p.flags, 1ull);
          stopped = true;
          break;
        }
        if ((++polls & 255u) == 0u && p.cancel && __any_sync(F, load_sys_u32(p.cancel) != 0u)) {
          if (lane == 0u) atomicExch(p.flags, 2ull);
          stopped = true;
          break;
        }
        if (pk.cnt[0] >= cap) {
          status = 3;
          break;
        }
        ld.keep(d, pk.pid, p.iteration, p.key0, p.key1, lane, false);
        pk.cnt[0] += 1u;
        const uint32_t di = d - ld.base;
        d += 1u;
        // the draws of a line event (the buffer holds three)
        const unsigned long long u_em = ld.u[di + 1u];
        const double mu_line = ld.m[di + (MODE == 1 ? 2u : 1u)];
        const bool inner = strictly_negative(pk.p) && rawkey(pk.q) <= rawkey(c_xi2);
        const ScanF f = scan_setup(pk.nu_cmf, f32_rz_small(pk.p), f32_rz_small(pk.q), f_kap, inner, f_xi2, f_xo2, ld.t[di]);
        const int32_t j0 = pk.next_line;
        int32_t j = j0, j_log = j0;  // the lines passed before j_log have their J_blue sums
        int kind = -1;               // -1 open, 0 in doubt
        long long hit = 0;
        unsigned long long rinfo = 0ull;
        uint4 ra = make_uint4(0u, 0u, 0u, 0u), rc = ra;
        float C = 0.0f;
        while (kind < 0) {  // one window at a time
          const int idx = j - w0;
          const bool cand = static_cast<int>(lane) >= idx;
          const bool there = w0 + static_cast<int32_t>(lane) < L;
          bool ok;
          const float l = scan_delta(f, w_b, ok) * f.lf;
          const float a = l * f.tf;
          const float own = (cand && there) ? f32_rz_any(w_t) : 0.0f;
          const float n = static_cast<float>(j - j0 + 32);
          const float m0 = fmaf(f.tf, fmaf(n, 0x1.0p-51f, 0x1.0p-44f), 0x1.0p-100f);
          const float m1 = fmaf(n, 0x1.0p-23f, 0x1.0p-19f);
          const float M = fmaf(m1, a + f.tau, m0);
          const float ra_ = (f.tau - C) - a;                 // before any line of the window
          const float xm = f.lx - l, xM = fmaf(0x1.0p-19f, l, f.mx);
          const bool inside = xm > xM;                       // certainly before the exit
          // First the line that absorbs by its own depth: the depths before it
          // only have to leave it in reach.  Their sum is one integer
          // reduction (units of 2^-21, at most 2^-16 too small), and then every
          // line before it is passed (path lengths and depths only grow); the
          // record of its emission is on its way meanwhile.
          const unsigned thick = __ballot_sync(F, cand && there && ok && ra_ - own < -M);
          int k = 31 - __clz(thick & (0u - thick));  // its lane, or -1: then lane 31 stands in, to no effect
          bool taken = false;
          hit = __shfl_sync(F, w_b, k);
          if (LINES == 1) {
            rinfo = __shfl_sync(F, w_r, k);
            load_slot_here(bucket_slot(p.dbr_bucket, rinfo, u_em), ra, rc);
          }
          {
            const bool prior = cand && static_cast<int>(lane) < k;
            const unsigned sum = __reduce_add_sync(
                F, prior ? __float2uint_rd(fminf(fmaxf(own, 0.0f), 63.0f) * 0x1.0p21f) : 0u);
            const float rk = ra_ - static_cast<float>(sum) * 0x1.0p-21f;
            const bool good = static_cast<int>(lane) == k ? (inside && rk > M + 0x1.0p-15f) : !(prior && own < 0.0f);
            taken = __all_sync(F, good) && thick != 0u;
          }
          unsigned stop = 1u, outs = 0u;
          float Px = 0.0f;
          if (!taken) {
            // the depths before each line (exclusive prefix, so that a thick
            // line's own depth does not round them away)
            Px = __shfl_up_sync(F, own, 1);
            if (lane == 0u) Px = C;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
              const float y = __shfl_up_sync(F, Px, o);
              if (static_cast<int>(lane) >= o) Px = __fadd_rn(Px, y);
            }
            const float r0 = (f.tau - Px) - a;                 // before this line
            const float r1 = r0 - own;                         // after it
            const bool before = there && ok && r0 > M;         // certainly before d_e
            const bool pass = before && inside && r1 > M && own >= 0.0f;
            const bool take = before && inside && r1 < -M;
            // the exit comes before this line and before d_e
            const float ax = f.lx * f.tf;
            const float rx = (f.tau - Px) - ax;
            const bool out = (!there || (ok && xm < -xM)) &&
                             rx > fmaf(m1, fabsf(ax) + f.tau, fmaf(f.tf, f.mx, m0));
            stop = __ballot_sync(F, cand && !pass);
            const unsigned took = __ballot_sync(F, take);
            outs = __ballot_sync(F, out);
            k = stop ? __ffs(stop) - 1 : 32;
            taken = stop && ((took >> k) & 1u);
            if (taken) {
              hit = __shfl_sync(F, w_b, k);
              if (LINES == 1) {
                rinfo = __shfl_sync(F, w_r, k);
                load_slot_here(bucket_slot(p.dbr_bucket, rinfo, u_em), ra, rc);
              }
            }
          }
          j = w0 + k;
          if (taken) {
            kind = kLineEvent;
          } else if (stop) {
            kind = ((outs >> k) & 1u) ? kShellEvent : 0;
          } else {
            if (JB) {  // a window passed whole: one lane a line, not left to the log
              settle();
              if (cand)
                red_add_evict_first(p.j_blue + static_cast<size_t>(cs) * static_cast<size_t>(L) + w0 +
                                        static_cast<int32_t>(lane), pk.e_per_nu * pk.inv_nu, jb_pol);
              j_log = j;
            }
            C = __shfl_sync(F, Px + own, 31);
            reload(j);
          }
        }
        settle();
        double thr = 0.0, p_exit = 0.0;
        if (kind == 0) {
          kind = exact_scan(ld.u[di], inner, j0, j, false, 0.0, hit, thr, p_exit);
          if (kind == kLineEvent) {
            if (LINES == 1) {
              rinfo = __ldg(p.row_info + j);
              load_slot_here(bucket_slot(p.dbr_bucket, rinfo, u_em), ra, rc);
            }
          }
        }
        const uint32_t npass = static_cast<uint32_t>(j - j0);
        pk.cnt[1] += npass + (j < L ? 1u : 0u);
        pk.cnt[2] += npass;
        pk.next_line = j;
        if (kind == kLineEvent) {
          pk.cnt[2] += 1u;
          pk.cnt[3] += 1u;
          const double nuj = __longlong_as_double(hit);
          double l, r2;
          line_point(nuj, l, r2);
          const double xn = sqrt64(r2);
          log_segment(l, j_log, j - j_log + 1);
          double mu = mu_line;
          int32_t em = 0;
          if (MODE == 2) {
            const MaDraws md{nullptr, &ld, &d, p.key0, p.key1, pk.pid, p.iteration};
            rinfo = macroatom_walk_lone(p.ma_row, p.ma_jump, __ldg(p.line_row + j), md, lane);
            em = downbranch_pick<true>(p, j, rinfo, md.next());
            mu = DrawStream::mu_from_u53(md.next());
          } else if (MODE == 1) {
            d += 2u;
            if (kSlots) {
              em = slot_line(ra, rc, u_em);
              if (em < 0) em = search_row_lone(p.dbr_rec, rinfo, rc.z, u_em, lane);
            } else {
              em = downbranch_pick<false>(p, j, rinfo, u_em);
            }
          } else {
            d += 1u;
          }
          if (MODE >= 1) {
            pk.next_line = em + 1;
            reload(em + 1);
            pk.nu_cmf = __longlong_as_double(static_cast<long long>(load_here(p.nu + em)));
          } else {
            pk.next_line = j + 1;
            pk.nu_cmf = nuj;
          }
          pk.e_cmf = pk.e_per_nu * nuj;
          const double pn = xn * mu;
          pk.D = fma(-xn, mu, 1.0);
          pk.p = pn;
          pk.q = max0(fma(-pn, pn, r2));
          pk.have_lab = false;
          fresh = true;
          if (VIRT) {
            queue_virtual(lane == 0u, VirtualLaunch{xn, r2, pk.nu_cmf, pk.e_cmf, cs, pk.next_line, pk.pid, vdraws});
            vdraws += static_cast<uint32_t>(p.n_virtual);
          }
        } else if (kind == kShellEvent) {
          pk.cnt[5] += 1u;
          p_exit = shell_exit(pk.q, inner, c_xi2, c_xo2);
          log_segment(max0(p_exit - pk.p), j_log, j - j_log);
          need_lab();
          flush_shell();
          const int32_t ns = inner ? cs - 1 : cs + 1;
          pk.p = p_exit;
          pk.have_cmf = false;
          if (ns >= S) status = 1;
          else if (ns < 0) status = 2;
          else {
            enter_shell(ns);
            reload(j);
          }
        } else {
          pk.cnt[4] += 1u;
          const double l = max0(fma(-thr, pk.inv_nu, pk.D));
          const double pl = pk.p + l;
          log_segment(l, j_log, j - j_log);
          const double D1 = 1.0 - pl;
          const double nu_c = pk.nu_lab * D1;
          pk.e_cmf = pk.e_per_nu * nu_c;
          const double r2 = fma(pl, pl, pk.q);
          const double xn = leave(r2, ld.m[d - ld.base], nu_c, pk.inv_nu * rcp64(D1));
          d += 1u;
          if (VIRT) {
            queue_virtual(lane == 0u, VirtualLaunch{xn, r2, nu_c, pk.e_cmf, cs, j, pk.pid, vdraws});
            vdraws += static_cast<uint32_t>(p.n_virtual);
          }
        }
        if (LINES != 0 ? pk.next_line != w0 : pk.next_line < w0 || pk.next_line - w0 >= 32)
          reload(pk.next_line);  // behind the window (or the loop above starts at its first lane)
        if (status == 0) need_cmf();
      }
      settle();
      need_lab();
      flush_shell();
      if (status != 0 && lane == 0u) {
        if (status == 1) ++n_esc;
        else if (status == 2) ++n_reab;
        else ++n_cap;
        n_seg += pk.cnt[0];
        n_chk += pk.cnt[1];
        n_res += pk.cnt[2];
        n_lint += pk.cnt[3];
        n_esca += pk.cnt[4];
        n_shell += pk.cnt[5];
        const double e_lab = pk.e_per_nu * pk.nu_lab;
        if (status == 1) atomicAdd(p.spectrum + spectrum_bin(p, pk.nu_lab), e_lab);
        if (REC) {
          const uint32_t r = static_cast<uint32_t>(pk.pid - p.first_packet);
          p.rec_status[r] = status;
          p.rec_nu[r] = pk.nu_lab;
          p.rec_e[r] = e_lab;
#pragma unroll
          for (int c = 0; c < kNCounters; ++c) p.rec_cnt[static_cast<size_t>(r) * kNCounters + c] = pk.cnt[c];
        }
      }
      if (stopped) break;
      alive = false;
      lw_ok = false;
      continue;
    }
    if (!VIRT && !alive) continue;

    // ---- one flight segment of every live lane (Sect. 2.6)
    int status = 0;
    bool left = false;  // the lane's packet interacted: v-packets leave with it
    double left_x = 0.0, left_r2 = 0.0;
    if (VIRT && !alive) {
    } else if (pk.cnt[0] >= p.max_segments) {
      status = 3;  // capped
      need_lab();
    } else {
      pk.cnt[0] += 1u;
      const int32_t s = pk.shell;
      if (s != cs) enter_shell(s);
      need_cmf();
      // optical depth to the next event, tau = -ln z
      const unsigned long long u_tau = ds.next_u53();
      const bool inner = strictly_negative(pk.p) && rawkey(pk.q) <= rawkey(c_xi2);  // q, x_in^2 >= 0
      const ScanF f = scan_setup(pk.nu_cmf, f32_rz_small(pk.p), f32_rz_small(pk.q), f_kap, inner, f_xi2, f_xo2,
                                 neg_log_u53_f(u_tau + 1ull));
      // J_blue weight of this segment, E_lab / nu_lab^2 (Eq. 17 without its
      // line factor nu_j, applied per cell after the launch)
      const double e_inv2 = JB ? pk.e_per_nu * pk.inv_nu : 0.0;
      const size_t row = static_cast<size_t>(s) * static_cast<size_t>(L);
      const double *tau_s = p.tau + row;
      const int32_t j0 = pk.next_line;
      int32_t j = j0;
      int kind = 0;
      if (!lw_ok) load_window(s, j);
      // two lines ahead are always in flight while line j is resolved
      long long bj = lw_b0, bj_n = lw_b1, bj_nn = 0;
      double taul = lw_t0, tau_n = lw_t1, tau_nn = 0.0;
      unsigned long long rinfo = lw_r0, rinfo_n = lw_r1, rinfo_nn = 0ull;
      lw_ok = false;
      float rem = f.tau, m1 = 0x1.0p-19f, m0 = fmaf(f.tf, 0x1.0p-44f, 0x1.0p-100f);
      const float m0_step = f.tf * 0x1.0p-51f;
      for (;;) {
        bool at_exit = j >= L;
        if (!at_exit) {
          bj_nn = 0;
          tau_nn = 0.0;
          rinfo_nn = 0ull;
          if (j + 2 < L) {
            bj_nn = __ldg(nub + j + 2);
            tau_nn = __ldg(tau_s + j + 2);
            if (LINES == 1) rinfo_nn = __ldg(p.row_info + j + 2);
          }
          bool ok;
          const float l = scan_delta(f, bj, ok) * f.lf;
          const float a = l * f.tf;
          const float M = fmaf(m1, a + f.tau, m0);
          const float r0 = rem - a;
          if (!ok || !(r0 > M)) break;  // beyond d_e, or in doubt
          const float xm = f.lx - l, xM = fmaf(0x1.0p-19f, l, f.mx);
          if (!(xm > xM)) {
            if (!(xm < -xM)) break;  // in doubt
            at_exit = true;
          } else {
            const float tf = f32_rz_any(taul);
            const float r1 = r0 - tf;
            if (r1 < -M) {
              kind = kLineEvent;
              break;
            }
            if (!(r1 > M) || tf < 0.0f) break;  // in doubt
            rem -= tf;
          }
        }
        if (at_exit) {  // no line before the exit; certainly before d_e?
          const float ax = f.lx * f.tf;
          if (rem - ax > fmaf(m1, fabsf(ax) + f.tau, fmaf(f.tf, f.mx, m0))) kind = kShellEvent;
          break;
        }
        m1 += 0x1.0p-23f;
        m0 += m0_step;
        if (JB) red_add_evict_first(p.j_blue + row + j, e_inv2, jb_pol);
        ++j;
        bj = bj_n; taul = tau_n; rinfo = rinfo_n;
        bj_n = bj_nn; tau_n = tau_nn; rinfo_n = rinfo_nn;
      }
      double thr = 0.0, p_exit = 0.0;
      long long hit = bj;
      bool exact = false;
      if (kind == 0) {
        exact = true;
        kind = exact_scan(u_tau, inner, j0, j, true, e_inv2, hit, thr, p_exit);
        if (LINES == 1 && kind == kLineEvent) rinfo = __ldg(p.row_info + j);
      } else if (kind == kShellEvent) {
        p_exit = shell_exit(pk.q, inner, c_xi2, c_xo2);
      }
      const uint32_t npass = static_cast<uint32_t>(j - j0);
      pk.cnt[1] += npass + (j < L ? 1u : 0u);
      pk.cnt[2] += npass + (kind == kLineEvent ? 1u : 0u);
      pk.next_line = j;
      double l, r2 = 0.0;
      const double nuj = __longlong_as_double(hit);
      if (kind == kLineEvent) {
        if (JB) red_add_evict_first(p.j_blue + row + j, e_inv2, jb_pol);
        line_point(nuj, l, r2);
      } else if (kind == kShellEvent) {
        l = max0(p_exit - pk.p);
      } else {
        l = max0(fma(-thr, pk.inv_nu, pk.D));
      }
      // estimators, Eqs. 13-14 (segment-start comoving values)
      const double wgt = (pk.e_cmf * pk.D) * l;
      if (s != acc_s) {
        if (acc_s >= 0) {
          atomicAdd(j_sum + acc_s, acc_j);
          atomicAdd(nb_sum + acc_s, acc_nb);
        }
        acc_s = s; acc_j = 0.0; acc_nb = 0.0;
      }
      acc_j += wgt;
      acc_nb = fma(wgt, pk.nu_cmf, acc_nb);
      if (kind == kShellEvent) {
        // move to the boundary; free flight keeps q, nu_lab and E_lab
        pk.cnt[5] += 1u;
        need_lab();
        const int32_t ns = inner ? s - 1 : s + 1;
        pk.p = p_exit;
        pk.shell = ns;
        pk.have_cmf = false;
        if (ns >= S) status = 1;
        else if (ns < 0) status = 2;
      } else {
        double nu_c, inv_c;
        if (kind == kLineEvent) {
          pk.cnt[3] += 1u;
          pk.e_cmf = pk.e_per_nu * nuj;  // E / nu times the line's own frequency
          if (MODE >= 1) {
            // MODE 2: macro atom, internal jumps before the emission pick
            unsigned long long rinfo_em = rinfo;
            if (MODE == 2) {
              const MaDraws md{&ds, nullptr, nullptr, 0u, 0u, 0u, 0u};
              rinfo_em = macroatom_walk(p, __ldg(p.line_row + j), md);
            }
            const int32_t em = downbranch_pick<kSlots>(p, j, rinfo_em, ds.next_u53());
            nu_c = __ldg(p.nu + em);
            inv_c = rcp64(nu_c);
            pk.next_line = em + 1;
            load_window(s, pk.next_line);
            pk.e_per_nu = pk.e_cmf * inv_c;  // re-emitted at another frequency
          } else {
            nu_c = nuj;
            inv_c = rcp64(nuj);
            pk.next_line = j + 1;
            if (!exact) {
              lw_ok = true;  // lines j + 1, j + 2 are in the scan's registers
              lw_b0 = bj_n; lw_t0 = tau_n; lw_r0 = rinfo_n;
              lw_b1 = bj_nn; lw_t1 = tau_nn; lw_r1 = rinfo_nn;
            }
          }
        } else {
          pk.cnt[4] += 1u;
          const double pl = pk.p + l;
          r2 = fma(pl, pl, pk.q);
          const double D1 = 1.0 - pl;
          nu_c = pk.nu_lab * D1;
          inv_c = pk.inv_nu * rcp64(D1);
          pk.e_cmf = pk.e_per_nu * nu_c;
        }
        left_x = leave(r2, DrawStream::mu_from_u53(ds.next_u53()), nu_c, inv_c);
        left_r2 = r2;
        left = true;
      }
    }
    if (status != 0) {
      if (status == 1) ++n_esc;
      else if (status == 2) ++n_reab;
      else ++n_cap;
      n_seg += pk.cnt[0];
      n_chk += pk.cnt[1];
      n_res += pk.cnt[2];
      n_lint += pk.cnt[3];
      n_esca += pk.cnt[4];
      n_shell += pk.cnt[5];
      const double e_lab = pk.e_per_nu * pk.nu_lab;
      if (status == 1) atomicAdd(p.spectrum + spectrum_bin(p, pk.nu_lab), e_lab);
      if (REC) {
        const uint32_t r = static_cast<uint32_t>(pk.pid - p.first_packet);
        p.rec_status[r] = status;
        p.rec_nu[r] = pk.nu_lab;
        p.rec_e[r] = e_lab;
#pragma unroll
        for (int c = 0; c < kNCounters; ++c) p.rec_cnt[static_cast<size_t>(r) * kNCounters + c] = pk.cnt[c];
      }
      alive = false;
    }
    if (VIRT) {
      __syncwarp();
      queue_virtual(left, VirtualLaunch{left_x, left_r2, pk.nu_cmf, pk.e_cmf, cs, pk.next_line, pk.pid, vdraws});
      if (left) vdraws += static_cast<uint32_t>(p.n_virtual);
    }
  }
  if (VIRT && n_vq) fly_virtual(p, sh, vq, n_vq, lane);
  if (acc_s >= 0) {
    atomicAdd(j_sum + acc_s, acc_j);
    atomicAdd(nb_sum + acc_s, acc_nb);
  }
  unsigned long long st[kNStats] = {n_esc, n_reab, n_cap, n_seg, n_chk, n_res, n_lint, n_esca, n_shell};
#pragma unroll
  for (int i = 0; i < kNStats; ++i) {
    unsigned long long v = st[i];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if (lane == 0u && v) atomicAdd(p.stats + i, v);
  }
  if (lane == 0u) atomicMax(p.flags + 2, global_ns());
}

template <int LINES, bool JB, bool REC, bool VIRT>
const void *kernel_ptr() {
  return reinterpret_cast<const void *>(&transport_fp64<LINES, JB, REC, VIRT>);
}

template <int LINES, bool VIRT>
const void *select_lines(bool jb, bool rec) {
  if (jb) return rec ? kernel_ptr<LINES, true, true, VIRT>() : kernel_ptr<LINES, true, false, VIRT>();
  return rec ? kernel_ptr<LINES, false, true, VIRT>() : kernel_ptr<LINES, false, false, VIRT>();
}

}  // namespace

}  // namespace mcgpu
