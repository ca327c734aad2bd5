// thor_shell.cu -- photon-packet loop through gridless spherical shells (THOR
// Sec. 3.3-3.4): emission, propagation with the velocity-gradient step limiter
// (Sec. 5.1), interaction channel choice, resonant / dust scattering, escape tally.
//
// Execution model: persistent warps.  Every loop iteration is one event (draw tau,
// propagate to the interaction or the boundary, interact) for every live lane;
// lanes whose packet finished are refilled from the photon work queue with one
// warp-aggregated atomic (ballot of the idle lanes), so a warp stays full until the
// queue drains (runs with fewer photons than lanes fill per_warp lanes of every warp).
// The packet state lives in registers; the time-sliced variant (serving) resumes its
// packets from a list spread over all warps and appends the survivors to the next one.
#include "thor_device.cuh"
#include "thor_internal.h"

namespace thor {
namespace {

constexpr unsigned kFull = 0xffffffffu;
// A flight of many sub-steps (thin gas: hundreds to thousands per event) is interrupted after
// kFlySteps of them, and the packet's next turn resumes it: a warp's iteration is one event
// per lane, and lanes with short events would wait for the longest flight of each (Mg II
// sphere, 8500 sub-steps per photon: 5.4 of 32 lanes were active).  Photon::fly: kFlyNone, or
// the distance along the segment, or kFlyBall inside the safety ball (the packet's own
// position then holds the progress).
constexpr int kFlySteps = 128;
constexpr float kFlyNone = -1.0f, kFlyBall = -2.0f;
constexpr float kSafePending = -1.0f;  // Photon::safe: not formed yet (power laws; the offset is zero)
constexpr uint32_t kLongLived = 1u << 14;  // served rounds: packets past this many events run one per warp
constexpr uint32_t kPriBudget = 16;        // served rounds: budget multiple of a priority warp (one packet)

struct Photon {
  double px, py, pz;  // FP64 anchor; the position is anchor + offset
  float ox, oy, oz;   // FP32 offset moved since the anchor (inside the safety ball)
  float3 k;
  float x;     // gas-frame frequency at p (in gas)
  float X;     // lab frequency (in the cavity, and at escape)
  float safe;  // lower bound on the distance from p to any shell boundary (0 = unknown)
  int region;  // 1 = inside the empty cavity
  uint32_t nscat, ndust, iters, steps;
  float fly, fly_tau;    // an event interrupted in flight (kFly*): where, and the depth left
  // power law: position in FP32, r, 1 / r, density and speed there (pl_ir = 0: not formed)
  float qx, qy, qz, pl_r, pl_ir, pl_nr, pl_v;
  float X0;              // emitted lab frequency
  float col_hi, col_lo;  // HI column traversed (power-law shells), two-level FP32 sum
  StreamKey key;  // key.event: last completed event
  int model;
  unsigned long long pid;
};

__device__ __forceinline__ int find_entry(const WorkQueue& q, unsigned long long g) {
  int lo = 0, hi = q.n_entries - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (q.prefix[mid] <= g) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// Emission (Sec. 3.4): central point source, isotropic, line profile in the source frame;
// with a continuum (Sec. 5.1) word 4 picks the line (probability p_line) or the flat
// continuum, whose position is word 5.
__device__ __forceinline__ void shell_emit(const ShellModel& m, Photon& ph) {
  Rng rng;
  rng.init(((uint64_t)m.seed_hi << 32) | m.seed_lo, ph.pid, m.cont_C > 0.0f ? 2u : 1u);
  ph.key = rng;
  ph.px = 0.0; ph.py = 0.0; ph.pz = 0.0;
  ph.ox = 0.0f; ph.oy = 0.0f; ph.oz = 0.0f;
  ph.k = iso_dir(rng.u(0), rng.u(1));
  float X = m.X0;
  if (m.cont_C > 0.0f && rng.u(4) > m.p_line) {
    X = __fmaf_rn(m.cont_C, __fmaf_rn(2.0f, rng.u(5), -1.0f), X);
  } else if (m.line == 1) {
    const float R1 = rng.u(2), R2 = rng.u(3);
    X = __fmaf_rn(m.sigma * sqrtf(-2.0f * __logf(R1)), cospif(2.0f * R2), X);
  }
  ph.X = X;
  ph.X0 = X;
  ph.col_hi = 0.0f; ph.col_lo = 0.0f;
  ph.x = X * m.inv_vth;  // gas at rest at the centre
  ph.region = (m.R_in > 0.0) ? 1 : 0;
  ph.safe = (float)m.R_out;
  ph.nscat = 0; ph.ndust = 0; ph.iters = 0; ph.steps = 0;
  ph.fly = kFlyNone; ph.fly_tau = 0.0f;
  ph.pl_ir = 0.0f;
}

// Move by s along k inside the safety ball: FP32 offset only.  The moves since the last
// anchor sum to at most the safety distance (< R_out - R_in), and the offset of a packet
// trapped in the core stays tiny, so FP32 keeps it far below the step size.
__device__ __forceinline__ void advance(Photon& ph, float s) {
  ph.ox = __fmaf_rn(s, ph.k.x, ph.ox);
  ph.oy = __fmaf_rn(s, ph.k.y, ph.oy);
  ph.oz = __fmaf_rn(s, ph.k.z, ph.oz);
}
// Fold the offset into the FP64 anchor (before any use of the absolute position).
__device__ __forceinline__ void anchor(Photon& ph) {
  if (ph.ox == 0.0f && ph.oy == 0.0f && ph.oz == 0.0f) return;  // already folded (FP64 runs at 1/64 of FP32)
  ph.px += (double)ph.ox; ph.py += (double)ph.oy; ph.pz += (double)ph.oz;
  ph.ox = 0.0f; ph.oy = 0.0f; ph.oz = 0.0f;
}

// FP64 sums of three products and r^2 - R^2 as the two event functions round them: which
// products are fused is part of a history's bits (kPower: the power-law event), so nothing
// here is left to the compiler.
template <bool kPower>
__device__ __forceinline__ double dot3(double ax, double ay, double az, double bx, double by, double bz) {
  return kPower ? __fma_rn(az, bz, __fma_rn(ay, by, __dmul_rn(ax, bx)))
                : __fma_rn(az, bz, __fma_rn(ax, bx, __dmul_rn(ay, by)));
}
__device__ __forceinline__ double minus_r2(double pp, double R) { return __dadd_rn(pp, -__dmul_rn(R, R)); }

// Exact distance from p to the nearest boundary, rounded down (conservative).
template <bool kPower>
__device__ __forceinline__ float safe_distance(const ShellModel& m, const Photon& ph) {
  const double r = sqrt(dot3<kPower>(ph.px, ph.py, ph.pz, ph.px, ph.py, ph.pz));
  double d = m.R_out - r;
  if (m.R_in > 0.0) d = fmin(d, r - m.R_in);
  return fmaxf(__double2float_rd(d) * 0.999999f, 0.0f);
}

// The segment from p along k to the next boundary: b = p . k, pp = r^2.  FP64 runs at 1/64 of
// the FP32 rate here and a dependent FP64 operation takes some 40 cycles, so the exact distance
// is formed only for a sub-step that may end at the boundary.  `lower` is a lower bound of it:
// r^2 - R_in^2 is taken in FP64 and rounded once, roots are formed without cancellation, and
// the margins cover the FP32 rounding (relative 1e-6; absolute 1e-6 for R_out^2 - r^2).
struct ShellSegment {
  float lower, c_in, bf;  // bound, r^2 - R_in^2, b
  __device__ __forceinline__ ShellSegment(const ShellModel& m, double b, double pp) {
    bf = (float)b;
    c_in = (float)(pp - m.R_in2);
    const float b2 = bf * bf, disc = b2 - c_in, err = 1e-6f * (b2 + fabsf(c_in));
    if (m.inv_in > 0.0f && bf < 0.0f && disc > -err) {  // may meet the inner sphere (before the outer one)
      lower = 0.999f * c_in * rcp_approx(sqrt_approx(fmaxf(disc, 0.0f) + err) - bf);
    } else {
      const float c_out = fmaxf(m.span - c_in - 1e-6f, 0.0f), q = sqrt_approx(b2 + c_out);
      lower = 0.999f * (bf >= 0.0f ? c_out * rcp_approx(q + bf + 1e-30f) : q - bf);
    }
  }
  // the distance and what is met there (1 outside, 2 cavity)
  static __device__ __forceinline__ double exact(const ShellModel& m, double b, double pp, int& next) {
    next = 1;
    if (m.R_in > 0.0 && b < 0.0) {
      const double disc = __fma_rn(b, b, -minus_r2(pp, m.R_in));
      if (disc > 0.0) {  // nearer than the outer sphere: -b - sqrt(disc) < -b < its distance
        next = 2;
        return fmax(-b - sqrt(disc), 0.0);
      }
    }
    return fmax(-b + sqrt(fmax(__fma_rn(b, b, -minus_r2(pp, m.R_out)), 0.0)), 0.0);
  }
  // Whether the point at s along the segment is certainly nearer than the sub-step to a
  // boundary: r - R_in = (r^2 - R_in^2) / (r + R_in) <= (r^2 - R_in^2) / (2 R_in), likewise
  // outside.
  __device__ __forceinline__ bool near_edge(const ShellModel& m, float s) const {
    const float t = __fmaf_rn(s, __fmaf_rn(2.0f, bf, s), c_in), e = 1e-6f;  // r'^2 - R_in^2
    return (m.inv_in > 0.0f && (t + e) * m.inv_in < 0.99f * m.ds_core) ||
           (m.span - t + e) * m.inv_out < 0.99f * m.ds_core;
  }
};

// The start of a step, shared by shell_event's fast paths and the core events in rounds (one
// definition, so both evaluate an event bit for bit alike): H(a, x) from the table-free
// polynomial in the core (|x| <= 2), else from the table; kH = kap0 H; the crossing at the
// start-point rate s = tau / (kH + kapd); dust is chosen when R (kH + kapd) >= kH (the
// channel of Sec. 3.4, probability kapd / (kH + kapd)).
struct StartStep { float kH, s; };
__device__ __forceinline__ float voigt_start(float a, float x, const float* __restrict__ Ktab) {
  return (fabsf(x) <= THOR_VCORE_X) ? voigt_core_poly(a, x) : voigt<false>(a, x, Ktab);
}
__device__ __forceinline__ StartStep start_step(const ShellModel& m, float H, float tau) {
  const float kH = __fmul_rn(m.kap0, H);
  return StartStep{kH, __fmul_rn(tau, rcp_approx(__fadd_rn(kH, m.kapd)))};
}
__device__ __forceinline__ bool dust_channel(const ShellModel& m, float kH, float R) {
  return __fmul_rn(R, __fadd_rn(kH, m.kapd)) >= kH;
}

// Free flight: sub-steps in the wing, four at a time while none of them ends the flight (the
// caller takes that one).  Their opacities do not depend on one another (x drifts
// monotonically), so they are formed side by side -- one at a time a flight is a chain of some
// 100 dependent instructions per sub-step -- and only depth and column are summed in order.
// (Out of line it took 14.0 instead of 11.7 ms on the Mg II sphere.)
struct FlyOut {
  float s, tau, col_hi, col_lo;
  uint32_t n;  // sub-steps done
};
static __device__ __forceinline__ FlyOut fly_wing(float kap0, float kapd, float a, float gam, float x0, float ds, float s,
                                               float bound, float tau, int most) {
  FlyOut o{s, tau, 0.0f, 0.0f, 0u};
  const float g = gam * 0.5f;
  while ((int)o.n < most && o.s + 4.25f * ds <= bound) {
    float e[5], kp[4];
    e[0] = o.s;
#pragma unroll
    for (int i = 0; i < 4; ++i) e[i + 1] = e[i] + ds;
    const float xa = __fmaf_rn(-g, e[0] + e[1], x0), xb = __fmaf_rn(-g, e[3] + e[4], x0);
    if (!(fminf(xa, xb) >= 6.0f || fmaxf(xa, xb) <= -6.0f)) break;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float x = __fmaf_rn(-g, e[i] + e[i + 1], x0);
      kp[i] = __fmaf_rn(kap0, voigt_wing<false>(a, x * x), kapd);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float dt = __fmul_rn(kp[i], e[i + 1] - e[i]);
      if (dt >= o.tau) return o;
      o.tau = __fsub_rn(o.tau, dt);
      o.s = e[i + 1];
      ++o.n;
    }
  }
  return o;
}

// One event.  Returns 0 = continues, 1 = escaped, 2 = absorbed by dust, 3 = capped, -1 =
// interrupted in flight (the same event goes on with the next call).
// The gas-frame frequency x is carried along the ray: in the homologous flow it drifts
// as x(s) = x0 - gam s in every direction, and a scattering leaves it at x_out at the
// same point.  A conservative safety distance to the shell boundaries lets events whose
// interaction lies inside the safety ball skip the FP64 ray-sphere geometry (the common
// case for photons trapped in the line core).
// Blocks of words an event may take: the third holds the channel, albedo and mixed-phase words.
__device__ __forceinline__ bool needs_block2(const ShellModel& m) {
  return m.kapd > 0.0f || m.kapdn > 0.0f || m.phase == PH_MIXED || m.n_lines == 2;
}

// The packet's next event, from what it takes of its random words.
__device__ int shell_event(const ShellModel& m, Photon& ph, const float* __restrict__ Ktab, const EventWords& w) {
  const bool resumed = ph.fly != kFlyNone;
  float tau_rem = resumed ? ph.fly_tau : w.tau;
  float s_seg = ph.fly;  // >= 0: resumed in a segment, there
  ph.fly = kFlyNone;
  int turn_steps = kFlySteps;
  float x_site, kH;
  for (;;) {
    if (ph.region) {  // empty cavity: straight to the inner sphere, lab X conserved
      anchor(ph);
      const double kx = ph.k.x, ky = ph.k.y, kz = ph.k.z;
      const double b = dot3<false>(ph.px, ph.py, ph.pz, kx, ky, kz);
      const double c = minus_r2(dot3<false>(ph.px, ph.py, ph.pz, ph.px, ph.py, ph.pz), m.R_in);
      const double s = -b + sqrt(fmax(__fma_rn(b, b, -c), 0.0));
      ph.px = __fma_rn(s, kx, ph.px); ph.py = __fma_rn(s, ky, ph.py); ph.pz = __fma_rn(s, kz, ph.pz);
      ph.region = 0;
      ph.x = __fmul_rn(__fmaf_rn(-m.vgrad, (float)(b + s), ph.X), m.inv_vth);
      ph.safe = 0.0f;
    }
    // ---- fast path: the next (sub-)step lies inside the safety ball
    if (s_seg >= 0.0f) {
      // resumed below
    } else if (m.gam == 0.0f) {
      const StartStep st0 = start_step(m, voigt_start(m.a, ph.x, Ktab), tau_rem);
      kH = st0.kH;
      const float s = st0.s;
      ++ph.steps;
      if (s <= ph.safe) {
        advance(ph, s);
        ph.safe = __fmaf_rd(-s, 1.000001f, ph.safe);
        x_site = ph.x;
        break;
      }
    } else if (ph.safe >= m.ds_core) {
      // Rate at the start of the step: a crossing within ds_core / 16 of the start is a
      // sub-step of its own, integrated with that rate (the common case in the core).
      const StartStep st0 = start_step(m, voigt_start(m.a, ph.x, Ktab), tau_rem);
      const float s0 = st0.s;
      if (s0 <= 0.0625f * m.ds_core) {
        ++ph.steps;
        advance(ph, s0);
        ph.safe = __fmaf_rd(-s0, 1.000001f, ph.safe);
        x_site = __fmaf_rn(-m.gam, s0, ph.x);
        kH = st0.kH;
        break;
      }
      const float ds = m.ds_core;
      const float xm = __fmaf_rn(-__fmul_rn(m.gam, 0.5f), ds, ph.x);
      const float kap = __fmaf_rn(m.kap0, voigt<false>(m.a, xm, Ktab), m.kapd);
      const float dtau = __fmul_rn(kap, ds);
      ++ph.steps;
      if (dtau >= tau_rem) {
        const float s = __fdividef(tau_rem, kap);
        advance(ph, s);
        ph.safe = __fmaf_rd(-s, 1.000001f, ph.safe);
        x_site = __fmaf_rn(-m.gam, s, ph.x);
        kH = __fmul_rn(m.kap0, voigt<false>(m.a, x_site, Ktab));
        break;
      }
      tau_rem = __fsub_rn(tau_rem, dtau);
      advance(ph, ds);
      ph.safe = __fmaf_rd(-ds, 1.000001f, ph.safe);
      ph.x = __fsub_rn(ph.x, __fmul_rn(m.gam, ds));
      if (--turn_steps <= 0) {
        ph.fly = kFlyBall; ph.fly_tau = tau_rem;
        return -1;
      }
      continue;
    }
    // ---- general path: sub-steps to the crossing or the next boundary, its distance exact
    // (FP64) where it counts
    anchor(ph);
    const double kx = ph.k.x, ky = ph.k.y, kz = ph.k.z;
    const double b = dot3<false>(ph.px, ph.py, ph.pz, kx, ky, kz);
    const double pp = dot3<false>(ph.px, ph.py, ph.pz, ph.px, ph.py, ph.pz);
    const ShellSegment seg(m, b, pp);
    const float x0 = ph.x;
    double S = 0.0;  // distance to the boundary, once needed (seg.exact), and what is there
    float Sf = 0.0f;
    int next = 1;
    float s_star = -1.0f;
    if (m.gam == 0.0f) {
      S = ShellSegment::exact(m, b, pp, next);
      Sf = (float)S;
      const float kap = __fadd_rn(kH, m.kapd), t = __fmul_rn(kap, Sf);
      if (t >= tau_rem) s_star = fminf(__fdiv_rn(tau_rem, kap), Sf);
      else tau_rem = __fsub_rn(tau_rem, t);
    } else {
      float s = fmaxf(s_seg, 0.0f);
      s_seg = kFlyNone;
      bool have = false;
      for (;;) {
        if (turn_steps <= 0) {
          ph.fly = s; ph.fly_tau = tau_rem;
          return -1;
        }
        --turn_steps;
        float s1 = s + m.ds_core;
        if (!have && !(s1 <= seg.lower)) {
          S = ShellSegment::exact(m, b, pp, next);
          Sf = (float)S;
          have = true;
        }
        if (have) {
          if (!(s < Sf)) break;
          s1 = fminf(Sf, s1);
        }
        const float xm = __fmaf_rn(-__fmul_rn(m.gam, 0.5f), s + s1, x0);
        const float kap = __fmaf_rn(m.kap0, voigt<false>(m.a, xm, Ktab), m.kapd);
        const float dtau = __fmul_rn(kap, s1 - s);
        ++ph.steps;
        if (dtau >= tau_rem) {
          s_star = __fadd_rn(s, __fdiv_rn(tau_rem, kap));
          if (have) s_star = fminf(s_star, Sf);
          break;
        }
        tau_rem = __fsub_rn(tau_rem, dtau);
        s = s1;
        const float bound = have ? Sf : seg.lower;
        if (turn_steps > 0 && s + 4.25f * m.ds_core <= bound && fabsf(xm) >= 6.0f) {
          const FlyOut f = fly_wing(m.kap0, m.kapd, m.a, m.gam, x0, m.ds_core, s, bound, tau_rem, turn_steps);
          s = f.s;
          tau_rem = f.tau;
          ph.steps += f.n;
          turn_steps -= (int)f.n + 1;
        }
      }
    }
    if (s_star >= 0.0f) {
      const double sd = s_star;
      ph.px = __fma_rn(sd, kx, ph.px); ph.py = __fma_rn(sd, ky, ph.py); ph.pz = __fma_rn(sd, kz, ph.pz);
      x_site = __fmaf_rn(-m.gam, s_star, x0);
      if (m.gam != 0.0f) kH = __fmul_rn(m.kap0, voigt<false>(m.a, x_site, Ktab));
      // the safety distance counts only from ds on: where it is certainly shorter (photons
      // trapped at the shell's edge, which come here event after event) its FP64 square root
      // is left out
      ph.safe = (m.gam != 0.0f && seg.near_edge(m, s_star)) ? 0.0f : safe_distance<false>(m, ph);
      break;
    }
    ph.px = __fma_rn(S, kx, ph.px); ph.py = __fma_rn(S, ky, ph.py); ph.pz = __fma_rn(S, kz, ph.pz);
    const float x_end = __fmaf_rn(-m.gam, Sf, x0);
    ph.X = __fmaf_rn(x_end, m.vth, __fmul_rn(m.vgrad, (float)(b + S)));  // lab frequency at the boundary
    if (next == 1) return 1;
    ph.region = 1;
  }
  ++ph.key.event;
  ph.x = x_site;
  // Interaction (Sec. 3.4): channel i with probability tau_i / sum_i tau_i.
  bool dust = false;
  if (m.kapd > 0.0f) dust = dust_channel(m, kH, w.channel);
  if (dust) {
    bool scat;
    if (m.albedo <= 0.0f) scat = false;
    else if (m.albedo >= 1.0f) scat = true;
    else scat = w.albedo < m.albedo;
    if (!scat) return 2;
    scatter_dust(m.g_hg, ph.k, w.Rm, w.cp, w.sp);  // gas-frame frequency unchanged
    ++ph.ndust;
    return 0;
  }
  // Eq. 7: the gas-frame frequency after the scattering, at the same point
  ph.x = scatter_resonant<kTurnShell, kTurnShellIso>(x_site, m.a, m.phase, ph.k, w, ph.key, ph.iters, nullptr,
                                                     m.xcrit);
  ++ph.nscat;
  if (m.max_scat && ph.nscat >= m.max_scat) {
    anchor(ph);
    const float b = (float)dot3<false>(ph.px, ph.py, ph.pz, ph.k.x, ph.k.y, ph.k.z);
    ph.X = __fmaf_rn(ph.x, m.vth, __fmul_rn(m.vgrad, b));
    return 3;
  }
  return 0;
}

// ---- core events in rounds (homologous shells) ---------------------------------------
// A packet trapped in the line core spends its life in one kind of event: the crossing lies
// within ds/16 of the start (start-point rate, Sec. 5.1 step limiter) inside the safety
// ball, the interaction is a resonant scattering at |x| <= 2 (Sec. 3.4), and the u_par
// sampler (Eq. 10) accepts within two trials.  In such an event only the frequency
// chain x -> H(a,x) -> s -> x_site -> u_par -> x_out depends on the packet's state; the
// optical depth, the sampler's uniforms, the perpendicular atom velocity (Eq. 5), mu and the
// azimuth are functions of the event's random words, which depend on nothing but the key,
// the photon id and the event number.
//
// What bounds it: a run lasts as long as its longest photon (1e6 to 1e7 core events one after
// another), so the time of one event in a warp with few packets is what counts, and that is
// its instructions at the issue rate of a lone warp.  So the events run in rounds: all 32
// lanes first evaluate everything that depends on words alone, one event of one packet
// per lane, for the next D events of the warp's P packets (P D <= kChainSlots), into shared
// memory; then the P lanes that own the packets run D events of the chain, each from one
// 64-byte slot.  The general event evaluates these events with the same helpers
// (start_step, dust_channel, u0_core, upar_q / atan_small, upar_trial, x_after_scatter) on
// the same words, so both paths give bit-identical results.
// Measured (GB300, 2070 MHz): a photon alone in a static sphere 0.345 us per event (0.47 us
// when its own lane formed the directions' angles and the words came by shuffle), at 1e3 K
// 0.40 us (1.76 us); 5000 photons in a sphere of tau0 = 1e4 78 ms (113 ms); 1e5 photons in an
// expanding shell of N_HI = 1e19 350-380 ms (535-580 ms), of 1e20 3.4 s (5.4 s).  The general events run for
// all the packets that wait for one, at most once per `depth` core events: a general event
// costs several core events, and one lane in sixty needs one at any time.
constexpr int kChainSlots = kWordSlots;  // events per warp and round
constexpr uint32_t kChainDepth = 32;  // ... and per packet, in warps with few packets
constexpr uint32_t kCrowdDepth = 16;  // ... and per packet, in the others (kept until a general event runs)
constexpr uint32_t kFirstDepth = 4;   // ... at first: doubled where a round runs full, halved where it mostly does not
// ... and in a served warp while another packet waits for a general event: the packets of a warp
// belong to several requests there, and with 16 core events to each general one a thin request's
// packets got one event in 17 of those a round is charged.  256 requests of up to N_HI = 1e21, 28
// per second: p50 28 -> 23 ms, p90 483 -> 429 ms, all at once no slower (64 requests 2.41 -> 2.44 s;
// depth 2 2.48 s, 1 2.78 s, 8 2.51 s).
constexpr uint32_t kSharedDepth = 4;
constexpr uint32_t kVoteEvents = 4;   // core events between two votes on whether any packet goes on
__device__ __forceinline__ void form_words(const ShellModel& m, const Photon& ph, WordBuf& wb, bool mine, int D,
                                           WordPos& at) {
  form_words(wb, ph.key, (needs_block2(m) ? kWordBlock2 : 0u) | (m.profile ? kWordLog : 0u), m.phase, m.xcrit, mine, D,
             at);
}

// Whether the packet's next event may be of the core kind (the cheap part of the test).
__device__ __forceinline__ bool chain_kind(const ShellModel& m, const Photon& ph) {
  return ph.fly == kFlyNone && !ph.region && m.phase != PH_MIXED && fabsf(ph.x) <= THOR_VCORE_X && (m.gam == 0.0f || ph.safe >= m.ds_core);
}

// One core event from its slot, committed where `go` holds and the event is of the core kind
// (by selects: a loop body of one basic block but for the rare second trial).  Returns
// whether it was committed.
__device__ __forceinline__ bool chain_event(const ShellModel& m, Photon& ph, const float4& wa, const float4& wb,
                                            const float4& wc, float channel, uint32_t e, bool go, uint32_t& second) {
  // ---- the frequency chain: rate at the start, crossing, gas-frame frequency at the site
  const float x0 = ph.x;  // (lanes that are not going evaluate what they have, and commit nothing)
  const StartStep st0 = start_step(m, voigt_core_poly(m.a, x0), wa.x);
  const float s0 = st0.s;
  const bool in_ball = (m.gam == 0.0f) ? (s0 <= ph.safe) : (ph.safe >= m.ds_core && s0 <= 0.0625f * m.ds_core);
  const float xs = (m.gam == 0.0f) ? x0 : __fmaf_rn(-m.gam, s0, x0);
  const bool dust = (m.kapd > 0.0f) && dust_channel(m, st0.kH, channel);
  // ---- u_par, first trial of the two-piece comparison function (as sample_upar)
  const float sgn = (xs < 0.0f) ? -1.0f : 1.0f;
  const float xr = fabsf(xs);
  const float u0 = u0_core(xr, m.a);
  const float q = upar_q(xr, m.a);
  // w1 = atan2(a, x - u0) as sample_upar forms it: from q where u0 > 0 and q is small, else the
  // series in a / x, else (within 20 a of line centre, and in cold gas) atan2f itself
  const bool split = u0 > 0.0f && q <= 0.05f, far = m.a <= 0.05f * (xr - u0);
  float w1 = split ? atan_small(q) : atan2_series(m.a, xr - u0);
  if (go && !split && !far) w1 = atan2f(m.a, xr - u0);
  const float u02 = __fmul_rn(u0, u0);
  const float mass = envelope_mass(w1, exp_fast(-u02));
  const float w1p = __fmul_rn(w1, 1.0f / kPiF);
  float u;
  bool accepted = upar_trial(xr, m.a, w1, w1p, mass, u02, wa.y, wa.z, wa.w, u);
  const bool kind = go && fabsf(x0) <= THOR_VCORE_X && in_ball && !dust && xr <= 2.0f;
  if (!accepted && kind) {  // rare: the second trial, from block 3 of the event as sample_upar takes it
    StreamKey r = ph.key;
    r.event = e;
    uint32_t b0, b1, b2, b3;
    r.block(3u, b0, b1, b2, b3);
    accepted = upar_trial(xr, m.a, w1, w1p, mass, u02, uni32(b0), uni32(b1), uni32(b2), u);
    second += accepted ? 1u : 0u;
  }
  const bool ok = kind && accepted;
  // ---- beside the chain: the outgoing direction (as scatter_resonant)
  float3 e1, e2;
  basis(ph.k.x, ph.k.y, ph.k.z, e1, e2);
  const float3 ko = turn<kTurnShell>(ph.k, e1, e2, wb.x, wb.y, wb.z, wb.w);
  // ---- commit
  ph.ox = ok ? __fmaf_rn(s0, ph.k.x, ph.ox) : ph.ox;  // advance(ph, s0)
  ph.oy = ok ? __fmaf_rn(s0, ph.k.y, ph.oy) : ph.oy;
  ph.oz = ok ? __fmaf_rn(s0, ph.k.z, ph.oz) : ph.oz;
  ph.safe = ok ? __fmaf_rd(-s0, 1.000001f, ph.safe) : ph.safe;
  const bool skip = xr < m.xcrit;
  const float perp = scatter_perp(wb.y, skip ? wc.z : wc.x, skip ? wc.w : wc.y, wb.z, wb.w);
  ph.x = ok ? x_after_perp(xs, sgn * u, wb.x, perp) : ph.x;
  ph.k.x = ok ? ko.x : ph.k.x;
  ph.k.y = ok ? ko.y : ph.k.y;
  ph.k.z = ok ? ko.z : ph.k.z;
  return ok;
}

// A round: up to D core events of every packet in `mine` lanes.  Called by all 32 lanes,
// converged.  `stuck` tells the lanes whose packet stopped before an event that is not of the
// core kind, or one scattering short of the cap (the general event runs that one, from slot
// at.cur).  Returns the events done.
__device__ __forceinline__ uint32_t chain_round(const ShellModel& m, Photon& ph, WordBuf& wb, bool mine, int D,
                                                WordPos& at, bool& stuck, int first_vote) {
  form_words(m, ph, wb, mine, D, at);
  const uint32_t left = m.max_scat ? (m.max_scat > ph.nscat + 1u ? m.max_scat - ph.nscat - 1u : 0u) : (uint32_t)D;
  const int lim = (int)min(left, (uint32_t)D);
  bool go = mine;
  uint32_t n = 0, second = 0;
  int d = 0;
  while (d < D) {
    const int end = min(D, d + (d ? (int)kVoteEvents : first_vote));
#pragma unroll 1
    for (; d < end; ++d) {
      const int s = d * at.P + at.rank;
      go = chain_event(m, ph, wb.a[s], wb.b[s], wb.c[s], wb.d[s].y, ph.key.event + 1u + (uint32_t)d, go && d < lim, second);
      n += go ? 1u : 0u;
    }
    if (!__any_sync(kFull, go)) break;
  }
  if (mine) {
    ph.key.event += n;
    ph.nscat += n;
    ph.steps += n;
    ph.iters += n + second;
    at.cur = (int)n;
  }
  stuck = mine && !go;
  return n;
}

// The depth of a warp's next round from that of the last: gas that is not thick enough for core
// events to follow one another (a crossing beyond ds/16 ends a round) would form slots and
// evaluate events for nothing.
__device__ __forceinline__ uint32_t next_depth(uint32_t depth, uint32_t most, unsigned tried, unsigned full) {
  if (2 * __popc(full) >= __popc(tried)) return min(2u * depth, most);
  return 8 * __popc(full) < __popc(tried) ? max(depth / 2u, 1u) : depth;
}

// Core events of a warp's packets until `depth` of them ran or the packet needs a general
// event (`general` then stays set).  Several rounds where the slots of one do not reach
// (P > kChainSlots / depth): the general events, which run for a few lanes at a time, come
// once per `depth` events.  Returns this lane's events; `at`: the slots of its last round, if
// no other round has overwritten them.
__device__ __forceinline__ uint32_t core_events(const ShellModel& m, Photon& ph, WordBuf& wb, bool active,
                                                uint32_t& depth_io, uint32_t most, bool& general, WordPos& at) {
  uint32_t n = 0;
  const uint32_t depth = min(depth_io, most);
  bool go = active && chain_kind(m, ph);
  const unsigned tried = __ballot_sync(kFull, go);
  for (uint32_t d = 0; d < depth; ) {
    const unsigned P = __popc(__ballot_sync(kFull, go));
    if (P == 0) break;
    // (one pass of the 32 lanes forms 32 slots anyway, and general events use what is left)
    const uint32_t D = min(max(depth - d, min(32u / P, most)), (uint32_t)(kChainSlots / P));
    bool stuck = false;
    n += chain_round(m, ph, wb, go, (int)D, at, stuck, (int)min(depth, kVoteEvents));
    go = go && !stuck;
    d += D;
  }
  general = active && !go;
  if (tried) depth_io = next_depth(depth, most, tried, __ballot_sync(kFull, go));
  return n;
}

// Slots for the next general event of the lanes in `general`, formed where they are not there
// yet: as many events ahead as one pass of the 32 lanes yields (at most kCrowdDepth).
__device__ __forceinline__ void general_words(const ShellModel& m, const Photon& ph, WordBuf& wb, bool general,
                                              WordPos& at) {
  if (!__any_sync(kFull, general && at.cur >= at.D)) return;
  const int P = __popc(__ballot_sync(kFull, general));
  form_words(m, ph, wb, general, min((int)kCrowdDepth, 32 / P), at);
}

// ---- power-law shells (Sec. 5.1) ---------------------------------------------------
// Gas state at a point q (FP32, |q| <= 1) for direction k: radius, r_hat . k, density
// relative to r = 1 and outflow speed.
struct PLState { float r, mur, nr, v, ir; };
__device__ __forceinline__ PLState pl_state(const ShellModel& m, float qx, float qy, float qz, float3 k) {
  const float r2 = __fmaf_rn(qx, qx, __fmaf_rn(qy, qy, qz * qz));
  PLState st;
  st.ir = rsqrtf(r2);
  st.r = r2 * st.ir;
  st.mur = __fmaf_rn(qx, k.x, __fmaf_rn(qy, k.y, qz * k.z)) * st.ir;
  const float lr = __log2f(st.r);
  st.nr = ex2_approx(m.ar * lr);
  st.v = m.v1 * ex2_approx(m.av * lr);
  return st;
}
// The same at the packet's position, which a scattering does not change: from the event
// before, where it was formed there (only the direction is new; the FP64 anchor's conversions
// are saved too).
__device__ __forceinline__ PLState pl_here(const ShellModel& m, Photon& ph) {
  if (ph.pl_ir == 0.0f) {
    ph.qx = (float)ph.px + ph.ox; ph.qy = (float)ph.py + ph.oy; ph.qz = (float)ph.pz + ph.oz;
    return pl_state(m, ph.qx, ph.qy, ph.qz, ph.k);
  }
  PLState st;
  st.ir = ph.pl_ir;
  st.r = ph.pl_r;
  st.mur = __fmaf_rn(ph.qx, ph.k.x, __fmaf_rn(ph.qy, ph.k.y, ph.qz * ph.k.z)) * st.ir;
  st.nr = ph.pl_nr;
  st.v = ph.pl_v;
  return st;
}
__device__ __forceinline__ void col_add(Photon& ph, float n, float d) {  // n d
  ph.col_lo = __fmaf_rn(n, d, ph.col_lo);
  if (ph.col_lo >= 0.00390625f) { ph.col_hi += ph.col_lo; ph.col_lo = 0.0f; }
}

// One event on a power-law shell; returns as shell_event.  The lab frequency X is the
// photon's frequency variable (the flow is not homologous, so x is evaluated from the
// local state).  A crossing predicted from the rate at the current point within
// min(safety distance, ds / 16) is taken with that rate (one Voigt evaluation, no FP64);
// otherwise sub-steps of at most ds (the global step limiter) use the midpoint state.
// Dust follows the gas and absorbs.
// Second transition of a doublet (Mg II H): its own offset X_2 = X + eps2 (c + X) on the
// scale of the first, and back.
constexpr float kCkms = 299792.458f;
__device__ __forceinline__ float to_line2(const ShellModel& m, float X) { return __fmaf_rn(m.eps2, kCkms + X, X); }
__device__ __forceinline__ float from_line2(const ShellModel& m, float X2) {
  return __fmaf_rn(-__fdividef(m.eps2, 1.0f + m.eps2), kCkms + X2, X2);
}

// X - v mu_r, the product rounded on its own (`apart`) or not: part of a history's bits.
__device__ __forceinline__ float x_offset(float X, const PLState& st, bool apart) {
  return apart ? __fsub_rn(X, __fmul_rn(st.v, st.mur)) : __fmaf_rn(-st.v, st.mur, X);
}
// fly_wing on a power-law shell, through the wings of its one or two lines, with the column.
static __device__ __forceinline__ FlyOut fly_power(const ShellModel* __restrict__ mp, float p0x, float p0y, float p0z,
                                                float3 k, float X, float s, float bound, float tau, float col_hi,
                                                float col_lo, int most) {
  const ShellModel& m = *mp;
  FlyOut o{s, tau, col_hi, col_lo, 0u};
  const float ds = m.ds_core;
  const bool two = m.n_lines == 2;
  while ((int)o.n < most && o.s + 4.25f * ds <= bound) {
    float e[5], kap[4], nr[4];
    e[0] = o.s;
    bool wing = true;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      e[i + 1] = e[i] + ds;
      const float sm = 0.5f * (e[i] + e[i + 1]);
      const PLState st = pl_state(m, __fmaf_rn(sm, k.x, p0x), __fmaf_rn(sm, k.y, p0y), __fmaf_rn(sm, k.z, p0z), k);
      nr[i] = st.nr;
      const float vk = __fmul_rn(st.v, st.mur);  // rounded as the caller's sub-step rounds it
      const float ax = fabsf(__fmul_rn(two ? __fsub_rn(X, vk) : __fmaf_rn(-st.v, st.mur, X), m.inv_vth));
      wing = wing && ax >= 6.0f;
      float H2 = 0.0f;
      if (two) {
        const float ax2 = fabsf(__fmul_rn(__fsub_rn(to_line2(m, X), vk), m.inv_vth));
        H2 = voigt_wing<false>(m.a2, ax2 * ax2);
        wing = wing && ax2 >= 6.0f;
      }
      kap[i] = __fmul_rn(st.nr, __fmaf_rn(m.kapn, voigt_wing<false>(m.a, ax * ax), __fmaf_rn(m.kapn2, H2, m.kapdn)));
    }
    if (!wing) return o;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float d = e[i + 1] - e[i], dt = __fmul_rn(kap[i], d);
      if (dt >= o.tau) return o;
      o.col_lo = __fmaf_rn(__fmul_rn(nr[i], m.invF), d, o.col_lo);
      if (o.col_lo >= 0.00390625f) { o.col_hi += o.col_lo; o.col_lo = 0.0f; }
      o.tau = __fsub_rn(o.tau, dt);
      o.s = e[i + 1];
      ++o.n;
    }
  }
  return o;
}

__device__ int shell_event_pl(const ShellModel& m, const ShellModel* mp, Photon& ph, const float* __restrict__ Ktab,
                              const EventWords& w) {
  const bool resumed = ph.fly != kFlyNone;
  float tau_rem = resumed ? ph.fly_tau : w.tau;
  float s_seg = ph.fly;
  ph.fly = kFlyNone;
  int turn_steps = kFlySteps;
  const bool two = m.n_lines == 2;
  float kH, kH2 = 0.0f, kD;
  PLState site;
  for (;;) {
    if (ph.region) {  // empty cavity: straight to the inner sphere, lab X conserved
      anchor(ph);
      const double kx = ph.k.x, ky = ph.k.y, kz = ph.k.z;
      const double b = dot3<true>(ph.px, ph.py, ph.pz, kx, ky, kz);
      const double c = minus_r2(dot3<true>(ph.px, ph.py, ph.pz, ph.px, ph.py, ph.pz), m.R_in);
      const double s = -b + sqrt(fmax(__fma_rn(b, b, -c), 0.0));
      ph.px = __fma_rn(s, kx, ph.px); ph.py = __fma_rn(s, ky, ph.py); ph.pz = __fma_rn(s, kz, ph.pz);
      ph.region = 0;
      ph.safe = 0.0f;
      ph.pl_ir = 0.0f;
    }
    float lower = 0.0f;  // of the distance to any boundary
    if (!(s_seg >= 0.0f)) {  // short step with the rate at the current point
      const PLState st = pl_here(m, ph);
      lower = fminf(1.0f - st.r, st.r - (float)m.R_in) - 1e-6f;
      const float x = __fmul_rn(x_offset(ph.X, st, true), m.inv_vth);
      const float H = voigt<false>(m.a, x, Ktab);
      const float H2 = (m.n_lines == 2) ? voigt<false>(m.a2, __fmul_rn(x_offset(to_line2(m, ph.X), st, true), m.inv_vth), Ktab)
                                         : 0.0f;
      const float kap = __fmul_rn(st.nr, __fmaf_rn(m.kapn, H, __fmaf_rn(m.kapn2, H2, m.kapdn)));
      const float s0 = __fdividef(tau_rem, kap);
      ++ph.steps;
      const bool is_short = s0 <= 0.0625f * m.ds_core;
      // the safety distance (an FP64 square root) is formed where it decides
      if (is_short && ph.safe == kSafePending) ph.safe = safe_distance<true>(m, ph);
      if (is_short && s0 <= ph.safe) {
        advance(ph, s0);
        ph.safe = __fmaf_rd(-s0, 1.000001f, ph.safe);
        col_add(ph, st.nr * m.invF, s0);
        kH = __fmul_rn(__fmul_rn(m.kapn, st.nr), H);
        kH2 = __fmul_rn(__fmul_rn(m.kapn2, st.nr), H2);
        kD = __fmul_rn(m.kapdn, st.nr);
        ph.qx = (float)ph.px + ph.ox; ph.qy = (float)ph.py + ph.oy; ph.qz = (float)ph.pz + ph.oz;
        site = pl_state(m, ph.qx, ph.qy, ph.qz, ph.k);
        break;
      }
    }
    // general path: sub-steps of <= ds to the crossing or the next boundary, its distance
    // exact (FP64) where it counts
    if (ph.ox != 0.0f || ph.oy != 0.0f || ph.oz != 0.0f || ph.pl_ir == 0.0f) {
      anchor(ph);
      ph.qx = (float)ph.px; ph.qy = (float)ph.py; ph.qz = (float)ph.pz;
    }
    const double kx = ph.k.x, ky = ph.k.y, kz = ph.k.z;
    double S = 0.0;
    float Sf = 0.0f;
    int next = 1;
    bool have = false;
    const float p0x = ph.qx, p0y = ph.qy, p0z = ph.qz;
    float s = fmaxf(s_seg, 0.0f), s_star = -1.0f;
    s_seg = kFlyNone;
    // one sub-step of opacity kap, density nr, [s, s1]: true where the crossing lies in it
    auto sub_step = [&](float s1, float kap, float nr) {
      const float dtau = __fmul_rn(kap, s1 - s);
      ++ph.steps;
      if (dtau >= tau_rem) {
        s_star = s + __fdividef(tau_rem, kap);
        if (have) s_star = fminf(s_star, Sf);
        col_add(ph, nr * m.invF, s_star - s);
        return true;
      }
      col_add(ph, nr * m.invF, s1 - s);
      tau_rem = __fsub_rn(tau_rem, dtau);
      s = s1;
      return false;
    };
    for (;;) {
      if (turn_steps <= 0) {
        ph.fly = s; ph.fly_tau = tau_rem;
        return -1;
      }
      --turn_steps;
      float s1 = s + m.ds_core;
      if (!have && !(s1 <= lower)) {  // the bound from the radius alone, then along the ray, then exact
        const double b = dot3<true>(ph.px, ph.py, ph.pz, kx, ky, kz);
        const double pp = dot3<true>(ph.px, ph.py, ph.pz, ph.px, ph.py, ph.pz);
        lower = ShellSegment(m, b, pp).lower;
        if (!(s1 <= lower)) {
          S = ShellSegment::exact(m, b, pp, next);
          Sf = (float)S;
          have = true;
        }
      }
      if (have) {
        if (!(s < Sf)) break;
        s1 = fminf(Sf, s1);
      }
      bool in_wing;
      {
        const float sm = 0.5f * (s + s1);
        const PLState st = pl_state(m, __fmaf_rn(sm, ph.k.x, p0x), __fmaf_rn(sm, ph.k.y, p0y),
                                    __fmaf_rn(sm, ph.k.z, p0z), ph.k);
        const float x = __fmul_rn(x_offset(ph.X, st, two), m.inv_vth);
        const float H = voigt<false>(m.a, x, Ktab);
        const float H2 = (m.n_lines == 2) ? voigt<false>(m.a2, __fmul_rn(x_offset(to_line2(m, ph.X), st, true), m.inv_vth), Ktab)
                                           : 0.0f;
        const float kap = __fmul_rn(st.nr, __fmaf_rn(m.kapn, H, __fmaf_rn(m.kapn2, H2, m.kapdn)));
        in_wing = fabsf(x) >= 6.0f;
        if (sub_step(s1, kap, st.nr)) {
          kH = __fmul_rn(__fmul_rn(m.kapn, st.nr), H);
          kH2 = __fmul_rn(__fmul_rn(m.kapn2, st.nr), H2);
          kD = __fmul_rn(m.kapdn, st.nr);
          break;
        }
      }
      const float bound = have ? Sf : lower;
      if (in_wing && turn_steps > 0 && s + 4.25f * m.ds_core <= bound) {
        const FlyOut f = fly_power(mp, p0x, p0y, p0z, ph.k, ph.X, s, bound, tau_rem, ph.col_hi, ph.col_lo, turn_steps);
        s = f.s;
        tau_rem = f.tau;
        ph.col_hi = f.col_hi;
        ph.col_lo = f.col_lo;
        ph.steps += f.n;
        turn_steps -= (int)f.n + 1;
      }
    }
    if (s_star >= 0.0f) {
      const double sd = s_star;
      ph.px = __fma_rn(sd, kx, ph.px); ph.py = __fma_rn(sd, ky, ph.py); ph.pz = __fma_rn(sd, kz, ph.pz);
      ph.safe = kSafePending;
      ph.qx = (float)ph.px; ph.qy = (float)ph.py; ph.qz = (float)ph.pz;
      site = pl_state(m, ph.qx, ph.qy, ph.qz, ph.k);
      break;
    }
    ph.px = __fma_rn(S, kx, ph.px); ph.py = __fma_rn(S, ky, ph.py); ph.pz = __fma_rn(S, kz, ph.pz);
    if (next == 1) return 1;  // escapes with its lab X
    ph.region = 1;
  }
  ++ph.key.event;
  ph.pl_r = site.r; ph.pl_ir = site.ir; ph.pl_nr = site.nr; ph.pl_v = site.v;
  // Interaction (Sec. 3.4): transition 1, transition 2 or dust in proportion to their
  // opacities (one uniform); dust absorbs.
  int ch = 0;
  if (kD > 0.0f || m.n_lines == 2) {
    const float u = w.channel, kt = __fadd_rn(__fadd_rn(kH, kH2), kD);
    ch = (u < __fdividef(kH, kt)) ? 0 : ((u < __fdividef(__fadd_rn(kH, kH2), kt)) ? 1 : 2);
  }
  if (ch == 2) return 2;
  float xo;
  if (ch == 0) {
    xo = scatter_resonant(__fmul_rn(x_offset(ph.X, site, false), m.inv_vth), m.a, m.phase, ph.k, w, ph.key, ph.iters, nullptr,
                          m.xcrit);
  } else {  // second transition: J = 1/2 upper level, isotropic
    EventWords wi = w;
    wi.mu = __fmaf_rn(2.0f, w.Rm, -1.0f);
    wi.st = sqrt_approx(fmaxf(0.0f, __fmaf_rn(-wi.mu, wi.mu, 1.0f)));
    xo = scatter_resonant(__fmul_rn(x_offset(to_line2(m, ph.X), site, false), m.inv_vth), m.a2, PH_ISO, ph.k, wi, ph.key,
                          ph.iters, nullptr, 0.0f);
  }
  // back to the lab frame with the new direction: X = x v_th + v(r) r_hat . k_out
  const float mur = __fmaf_rn(ph.qx, ph.k.x, __fmaf_rn(ph.qy, ph.k.y, ph.qz * ph.k.z)) / site.r;
  const float Xl = __fmaf_rn(xo, m.vth, site.v * mur);
  ph.X = (ch == 0) ? Xl : from_line2(m, Xl);
  ++ph.nscat;
  if (m.max_scat && ph.nscat >= m.max_scat) return 3;
  return 0;
}

__device__ __forceinline__ void tally_spectrum(const ShellModel& m, float X) {
  int bin;
  const float f = (X - m.X_min) * m.inv_dX;
  if (!(f >= 0.0f)) bin = m.n_bins;
  else if (f >= (float)m.n_bins) bin = m.n_bins + 1;
  else bin = (int)f;
  atomicAdd(&m.spectrum[bin], 1ull);
}

__device__ __forceinline__ void write_raw(const ShellModel& m, const Photon& ph, int status) {
  const unsigned long long j = ph.pid - m.id_base;
  if (m.raw_X) {
    m.raw_X[j] = ph.X;
    m.raw_nscat[j] = ph.nscat;
    m.raw_status[j] = (uint8_t)status;
  }
  if (m.raw_X0) m.raw_X0[j] = ph.X0;
  if (m.raw_col) m.raw_col[j] = ph.col_hi + ph.col_lo;
}

// Per-photon tally with global atomics (used where lanes may belong to different models).
__device__ __forceinline__ void finish_global(const ShellModel& m, const Photon& ph, int status) {
  Tally* T = m.tally;
  if (status == 1) { atomicAdd(&T->n_escaped, 1ull); tally_spectrum(m, ph.X); }
  else if (status == 2) atomicAdd(&T->n_absorbed, 1ull);
  else atomicAdd(&T->n_capped, 1ull);
  atomicAdd(&T->n_scat, (unsigned long long)ph.nscat);
  atomicAdd(&T->n_dust_scat, (unsigned long long)ph.ndust);
  atomicAdd(&T->n_upar_iters, (unsigned long long)ph.iters);
  atomicAdd(&T->n_steps, (unsigned long long)ph.steps);
  atomicAdd(&T->sum_scat2, (double)ph.nscat * (double)ph.nscat);
  atomicAdd(&T->n_done, 1ull);
  write_raw(m, ph, status);
}

struct LaneTally {
  unsigned long long esc = 0, abs = 0, cap = 0, scat = 0, dust = 0, iters = 0, steps = 0, done = 0;
  double scat2 = 0.0;
};

__device__ __forceinline__ unsigned long long warp_sum(unsigned long long v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(kFull, v, o);
  return v;
}
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(kFull, v, o);
  return v;
}

__device__ __forceinline__ void save_rec(const Photon& ph, PhotonRec& r) {
  r.px = ph.px; r.py = ph.py; r.pz = ph.pz;
  r.ox = ph.ox; r.oy = ph.oy; r.oz = ph.oz;
  r.X0 = ph.X0; r.col_hi = ph.col_hi; r.col_lo = ph.col_lo;
  r.kx = ph.k.x; r.ky = ph.k.y; r.kz = ph.k.z;
  r.fly = ph.fly; r.fly_tau = ph.fly_tau;
  r.x = ph.x; r.X = ph.X; r.safe = ph.safe;
  r.region = ph.region;
  r.nscat = ph.nscat; r.ndust = ph.ndust; r.iters = ph.iters; r.steps = ph.steps;
  r.event = ph.key.event;
  r.pid = ph.pid;
}

__device__ __forceinline__ void load_rec(const ShellModel& m, const PhotonRec& r, Photon& ph) {
  ph.px = r.px; ph.py = r.py; ph.pz = r.pz;
  ph.ox = r.ox; ph.oy = r.oy; ph.oz = r.oz;
  ph.X0 = r.X0; ph.col_hi = r.col_hi; ph.col_lo = r.col_lo;
  ph.k = make_float3(r.kx, r.ky, r.kz);
  ph.fly = r.fly; ph.fly_tau = r.fly_tau;
  ph.pl_ir = 0.0f;
  ph.x = r.x; ph.X = r.X; ph.safe = r.safe;
  ph.region = r.region;
  ph.nscat = r.nscat; ph.ndust = r.ndust; ph.iters = r.iters; ph.steps = r.steps;
  ph.pid = r.pid;
  ph.key.keys(((uint64_t)m.seed_hi << 32) | m.seed_lo, ph.pid);
  ph.key.event = r.event;
}

// ---- work sharing in the tail of a one-launch run (pool_take in thor_device.cuh) ----------
constexpr uint32_t kShareEvents = 256;  // a warp with several live packets checks for waiting warps this often
__device__ __forceinline__ long long share_take(const Compact& c) { return pool_take(c.share, c.ready, c.n_total); }

// Run-to-completion: all queue entries belong to one model (thor_run).  With kCompact,
// lanes first resume saved packets, and a warp whose sources are empty and whose live
// lanes drop below c.spill_below saves them and exits (tail compaction across launches).
template <bool kCompact, int kProfile>
__global__ void __launch_bounds__(256, 1) shell_run_kernel(const ShellModel* __restrict__ models, WorkQueue q,
                                                        Compact c, const float* __restrict__ gK) {
  __shared__ __align__(16) float sK[THOR_VOIGT_NINT * THOR_VOIGT_NCOEF];
  __shared__ ShellModel sm;
  extern __shared__ __align__(16) unsigned char dyn[];
  WordBuf& wb = reinterpret_cast<WordBuf*>(dyn)[threadIdx.x >> 5];
  load_ktab(sK, gK);
  if (threadIdx.x == 0) sm = models[q.model[0]];
  __syncthreads();
  const ShellModel m = sm;  // by value: the fields the event loop reads stay in registers
  const unsigned lane = threadIdx.x & 31u;
  Photon ph;
  bool active = false, done = (int)lane >= c.per_warp;  // lanes above per_warp stay idle
  bool drained = false;  // warp-uniform: a refill found the photon queue exhausted
  uint32_t depth = kFirstDepth;  // of the warp's next round of core events
  uint32_t ran = 0;  // events of the warp since the queue ran dry
  LaneTally lt;
  for (;;) {
    unsigned need = __ballot_sync(kFull, !active && !done);
    if (kCompact && need && c.n_resume) {  // saved packets first
      const int leader = __ffs(need) - 1;
      unsigned long long base = 0;
      if ((int)lane == leader) base = atomicAdd(c.resume_next, (unsigned long long)__popc(need));
      base = __shfl_sync(kFull, base, leader);
      if (!active && !done) {
        const unsigned long long g = base + __popc(need & ((1u << lane) - 1u));
        if (g < c.n_resume) { load_rec(m, c.resume[g], ph); active = true; }
      }
      need = __ballot_sync(kFull, !active && !done);
    }
    if (need) {
      const int leader = __ffs(need) - 1;
      unsigned long long base = 0;
      if ((int)lane == leader) base = atomicAdd(q.next, (unsigned long long)__popc(need));
      base = __shfl_sync(kFull, base, leader);
      if (base + __popc(need) > q.total) drained = true;
      if (!active && !done) {
        const unsigned long long g = base + __popc(need & ((1u << lane) - 1u));
        if (g < q.total) {
          ph.model = q.model[0];
          ph.pid = q.first_id[0] + g;
          shell_emit(m, ph);
          active = true;
        } else {
          done = true;
        }
      }
    }
    if (kCompact && c.spill_below > 0) {
      const unsigned live = __ballot_sync(kFull, active);
      if (drained && __popc(live) < c.spill_below) {
        if (live) {
          const int leader = __ffs(live) - 1;
          unsigned long long base = 0;
          if ((int)lane == leader) base = atomicAdd(c.n_spill, (unsigned long long)__popc(live));
          base = __shfl_sync(kFull, base, leader);
          if (active) save_rec(ph, c.spill[base + __popc(live & ((1u << lane) - 1u))]);
        }
        active = false;
        break;
      }
    }
    if (c.pool && drained) {
      const unsigned live = __ballot_sync(kFull, active);
      if (live == 0u) {  // an empty warp: take a packet that a crowded warp gives away
        long long got = -1;
        if (lane == 0) got = share_take(c);
        got = __shfl_sync(kFull, got, 0);
        if (got < 0) break;
        if (lane == 0) { load_rec(m, c.pool[got], ph); active = true; }
        continue;
      }
      // give packets away while empty warps wait, keeping the lowest lane's (short histories are over by then)
      if (__popc(live) >= 2 && ran >= kShareEvents) {
        const int leader = __ffs(live) - 1;
        long long give = 0;
        if ((int)lane == leader) give = pool_give_count(c.share, __popc(live));
        give = __shfl_sync(kFull, give, leader);
        if (give > 0) {
          // the `give` highest live lanes: their rank from the top
          const int from_top = __popc(live & ~((2u << lane) - 1u));
          const bool giver = active && from_top < (int)give;
          unsigned long long base = 0;
          if ((int)lane == leader) base = atomicAdd(&c.share[0], (unsigned long long)give);
          base = __shfl_sync(kFull, base, leader);
          if (giver) {
            const unsigned long long j = base + (unsigned long long)from_top;
            if (j < c.n_total) {  // an entry per photon
              save_rec(ph, c.pool[j]);
              if (pool_put(c.ready, j)) active = false;
            }
          }
        }
      }
    }
    if (__all_sync(kFull, !active)) break;
    const int n_live = __popc(__ballot_sync(kFull, active));
    const bool check_share = c.pool && drained && n_live >= 2;
    const bool chain = kProfile == 0 && n_live <= c.core_lanes;
    const uint32_t most = n_live <= c.burst_lanes || n_live <= kChainSlots / (int)kChainDepth ? kChainDepth : kCrowdDepth;
    uint32_t n_ev = 0;
    // events until some lane of the warp finishes its packet: the refill and spill checks
    // above run only when the set of live lanes changed
    bool fin;
    do {
      fin = false;
      bool general = active;  // lanes whose next event is a general one
      WordPos at;
      if (chain) core_events(m, ph, wb, active, depth, most, general, at);
      // packets whose next event is not of the core kind take general events: one, and more
      // while at least half of the warp's packets need them
      uint32_t n_gen = 0;
      do {
        general_words(m, ph, wb, general, at);
        if (general) {
          const EventWords w = read_words(wb, at.cur * at.P + at.rank);
          const int st = kProfile ? shell_event_pl(m, &sm, ph, sK, w) : shell_event(m, ph, sK, w);
          if (st >= 0) ++at.cur;
          if (st > 0) {
            if (st == 1) { ++lt.esc; tally_spectrum(m, ph.X); }
            else if (st == 2) ++lt.abs;
            else ++lt.cap;
            lt.scat += ph.nscat; lt.dust += ph.ndust; lt.iters += ph.iters; lt.steps += ph.steps; ++lt.done;
            lt.scat2 += (double)ph.nscat * (double)ph.nscat;
            write_raw(m, ph, st);
            if (c.pool) atomicAdd(&c.share[3], 1ull);
            active = false;
            fin = true;
          }
          general = active && !(chain && chain_kind(m, ph));
        }
      } while (!__any_sync(kFull, fin) && ++n_gen < kCrowdDepth &&
               (kProfile || 2 * __popc(__ballot_sync(kFull, general)) >= n_live));
      n_ev += chain ? most : n_gen;
      if (drained) ran += chain ? most : 8u * n_gen;  // (a turn on a power law may be 128 sub-steps)
    } while (!__any_sync(kFull, fin) && !(check_share && n_ev >= kShareEvents));
  }
  // flush lane tallies: warp reduce, one atomic per warp and field
  const unsigned long long e = warp_sum(lt.esc), a = warp_sum(lt.abs), cp = warp_sum(lt.cap),
                           s = warp_sum(lt.scat), d = warp_sum(lt.dust), it = warp_sum(lt.iters),
                           sp = warp_sum(lt.steps), dn = warp_sum(lt.done);
  const double s2 = warp_sum(lt.scat2);
  if (lane == 0 && dn) {
    Tally* T = m.tally;
    atomicAdd(&T->n_escaped, e); atomicAdd(&T->n_absorbed, a); atomicAdd(&T->n_capped, cp);
    atomicAdd(&T->n_scat, s); atomicAdd(&T->n_dust_scat, d); atomicAdd(&T->n_upar_iters, it);
    atomicAdd(&T->n_steps, sp); atomicAdd(&T->n_done, dn); atomicAdd(&T->sum_scat2, s2);
  }
}

// Time-sliced execution (serving): packets in flight live in a list (`in`): in.live[0]
// entries from the front, and in.live[2] priority entries from the back (packets of the
// requests the host marked as priority, the oldest ones).  The first priority packets, up
// to half of the warps, each run alone in a warp of their own (one packet per warp, so
// the longest histories of the oldest requests advance at the latency of a lone lane
// instead of behind divergent packets of other requests).  The remaining entries spread
// over the other warps: lane l of warp w resumes entry w + l * (their count).  Each lane
// runs at most `budget` events, finished lanes take new photons from the queue of admitted
// requests while the warp has fewer live packets than its limit (1 for a priority warp,
// per_warp otherwise), and what is still in flight is appended to `out`: priority packets
// from the back (out.live[3]), the others from the front (out.live[1]).
// kMixed: the round holds power-law models too (the event function is chosen per lane);
// otherwise only homologous shells, compiled without the power-law event.
template <bool kMixed>
__global__ void __launch_bounds__(256, 1) shell_slice_kernel(const ShellModel* __restrict__ models, WorkQueue q,
                                                          SlotState in, SlotState out, uint32_t budget,
                                                          const float* __restrict__ gK) {
  __shared__ __align__(16) float sK[THOR_VOIGT_NINT * THOR_VOIGT_NCOEF];
  extern __shared__ __align__(16) unsigned char dyn[];
  WordBuf& wb = reinterpret_cast<WordBuf*>(dyn)[threadIdx.x >> 5];
  load_ktab(sK, gK);
  int per_warp = 32;  // at most this many live packets per warp after a refill
  if (q.hdr) {
    q.total = q.hdr[0]; q.n_entries = (int32_t)q.hdr[1]; budget = (uint32_t)q.hdr[2];
    per_warp = (int)q.hdr[3];
  }
  const unsigned lane = threadIdx.x & 31u;
  const int64_t n_warps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const unsigned long long n_in = in.live[0], n_pri = in.live[2];
  // priority warps: [0, n_pw), one priority packet each; the rest of the priority list and
  // the front list spread over warps [n_pw, n_warps), at most 32 per warp.  Every stored
  // packet must find a lane: n_in + n_pri - n_pw <= 32 (n_warps - n_pw), i.e.
  // n_pw <= (32 n_warps - n_in - n_pri) / 31 (none when the list is full), and at most half
  // of the warps.
  const unsigned long long lanes = 32ull * (unsigned long long)n_warps;
  const unsigned long long fit = (lanes > n_in + n_pri) ? (lanes - n_in - n_pri) / 31ull : 0ull;
  const int64_t n_pw = (int64_t)min(min(n_pri, (unsigned long long)(n_warps / 2)), fit);
  const unsigned long long rest = n_in + (n_pri - (unsigned long long)n_pw);
  const int64_t n_rest_warps = n_warps - n_pw;
  const bool pri_warp = warp < n_pw;
  if (pri_warp) per_warp = 1;
  // A priority warp holds one packet and runs at a lone lane's latency, several times the
  // events a crowded warp runs in the same time: past the round's budget it goes on, up to
  // kPriBudget times the budget, while other warps of the round are still running (live[4]
  // counts those that finished), so the round lasts no longer for it.
  const int64_t n_regular = n_warps - n_pw;
  const uint32_t base_budget = budget;
  if (pri_warp) budget *= kPriBudget;
  int64_t slot = -1;
  if (pri_warp) {
    if (lane == 0) slot = in.n_slots - 1 - warp;
  } else {
    // contiguous entries per warp, counts differing by at most one: [w rest / W, (w+1) rest / W)
    // (the list arrives sorted by frequency bucket, so a warp's packets are of one kind)
    const unsigned long long wi = (unsigned long long)(warp - n_pw), W = (unsigned long long)n_rest_warps;
    const unsigned long long e = wi * rest / W + lane, e1 = (wi + 1) * rest / W;
    if (e < e1) slot = (e < n_in) ? (int64_t)e : in.n_slots - 1 - (int64_t)(n_pw + (e - n_in));
  }
  Photon ph;
  bool active = false, done = false;
  const SlotState& st = in;
  if (slot >= 0) {
    ph.model = st.model[slot];
    const ShellModel& m = models[ph.model];
    ph.pid = st.pid[slot];
    ph.key.keys(((uint64_t)m.seed_hi << 32) | m.seed_lo, ph.pid);
    ph.key.event = st.event[slot];
    ph.px = st.px[slot]; ph.py = st.py[slot]; ph.pz = st.pz[slot];
    ph.ox = st.ox[slot]; ph.oy = st.oy[slot]; ph.oz = st.oz[slot];
    ph.k = make_float3(st.kx[slot], st.ky[slot], st.kz[slot]);
    ph.X = st.X[slot];
    ph.x = st.x[slot];
    ph.safe = st.safe[slot];
    ph.X0 = 0.0f; ph.col_hi = 0.0f; ph.col_lo = 0.0f;  // raw records are not served
    ph.region = st.region[slot];
    ph.fly = st.fly[slot]; ph.fly_tau = st.fly_tau[slot];
    ph.pl_ir = 0.0f;
    ph.nscat = st.nscat[slot]; ph.ndust = st.ndust[slot]; ph.iters = st.iters[slot]; ph.steps = st.steps[slot];
    active = true;
  }
  uint32_t ev = 0;  // event iterations of this launch (warp-uniform)
  uint32_t depth = kFirstDepth;  // of the warp's next round of core events
  auto others_done = [&]() { return pri_warp && ev >= base_budget && (int64_t)vload(&in.live[4]) >= n_regular; };
  while (ev < budget && !others_done()) {
    const unsigned idle = __ballot_sync(kFull, !active && !done);
    const int room = per_warp - __popc(__ballot_sync(kFull, active));
    const bool take = ((idle >> lane) & 1u) && (int)__popc(idle & ((1u << lane) - 1u)) < room;
    const unsigned need = __ballot_sync(kFull, take);
    if (need) {
      const int leader = __ffs(need) - 1;
      unsigned long long base = 0;
      if ((int)lane == leader) base = atomicAdd(q.next, (unsigned long long)__popc(need));
      base = __shfl_sync(kFull, base, leader);
      if (take) {
        const unsigned long long g = base + __popc(need & ((1u << lane) - 1u));
        if (g < q.total) {
          const int e = find_entry(q, g);
          ph.model = q.model[e];
          ph.pid = q.first_id[e] + (g - q.prefix[e]);
          shell_emit(models[ph.model], ph);
          active = true;
        } else {
          done = true;
        }
      }
    }
    if (__all_sync(kFull, !active)) break;
    // The lane's model record, and the cancel flag, once per run of events: a request
    // cancelled on the host drops its packets here (the flag is set between launches).
    const ShellModel* mp = models + (active ? ph.model : 0);
    bool dropped = false;
    if (active && *(volatile const int32_t*)&mp->cancelled) {
      atomicAdd(&mp->tally->n_done, 1ull);
      active = false;
      dropped = true;
    }
    if (__any_sync(kFull, dropped)) { ++ev; continue; }  // refill the dropped lanes first
    const ShellModel mr = *mp;  // by value: the fields the event loop reads stay in registers
    // events until some lane finishes its packet or the budget is used (a warp is charged the
    // events of the lane that ran most of them)
    const int n_live = __popc(__ballot_sync(kFull, active));
    const bool chain = !(kMixed && mr.profile);  // this lane's packet runs core events in rounds
    bool fin;
    do {
      fin = false;
      bool general = active;
      const bool waiting = __any_sync(kFull, active && !(chain && chain_kind(mr, ph)));
      const uint32_t most = min(waiting                                       ? kSharedDepth
                                : n_live <= kChainSlots / (int)kChainDepth ? kChainDepth
                                                                           : kCrowdDepth,
                                budget - ev);
      WordPos at;
      uint32_t n = core_events(mr, ph, wb, active && chain, depth, most, general, at);
      if (kMixed) general = general || (active && !chain);
      uint32_t n_gen = 0;
      do {
        general_words(mr, ph, wb, general, at);
        if (general) {
          const EventWords w = read_words(wb, at.cur * at.P + at.rank);
          const int r = (kMixed && mr.profile) ? shell_event_pl(mr, mp, ph, sK, w) : shell_event(mr, ph, sK, w);
          if (r >= 0) ++at.cur;
          ++n;
          if (r > 0) { finish_global(mr, ph, r); active = false; fin = true; }
          general = active && !(chain && chain_kind(mr, ph));
        }
      } while (!__any_sync(kFull, fin) && ++n_gen < kCrowdDepth && n_gen + most < budget - ev &&
               2 * __popc(__ballot_sync(kFull, general)) >= n_live);
      ev += max(1u, __reduce_max_sync(kFull, n));
    } while (ev < budget && !__any_sync(kFull, fin) && !others_done());
  }
  if (!pri_warp && lane == 0) atomicAdd(&in.live[4], 1ull);  // this regular warp's round is over
  // append the packets still in flight to the next list (one atomic per warp and list):
  // priority packets from the back, the others from the front.  Priority: packets of the
  // requests the host marked (the oldest), and long-lived packets (more than kLongLived
  // events: photons trapped in the line core, whose histories set the requests' latency)
  const bool pri = active && ((ph.nscat + ph.ndust) >= kLongLived ||
                              *(volatile const int32_t*)&models[ph.model].priority);
  const unsigned live_f = __ballot_sync(kFull, active && !pri), live_b = __ballot_sync(kFull, pri);
  if (live_f | live_b) {
    const int lead_f = live_f ? __ffs(live_f) - 1 : 0, lead_b = live_b ? __ffs(live_b) - 1 : 0;
    unsigned long long base_f = 0, base_b = 0;
    if (live_f && (int)lane == lead_f) base_f = atomicAdd(&out.live[1], (unsigned long long)__popc(live_f));
    if (live_b && (int)lane == lead_b) base_b = atomicAdd(&out.live[3], (unsigned long long)__popc(live_b));
    base_f = __shfl_sync(kFull, base_f, lead_f);
    base_b = __shfl_sync(kFull, base_b, lead_b);
    if (active) {
      const unsigned mine = pri ? live_b : live_f;
      const unsigned long long r = (pri ? base_b : base_f) + __popc(mine & ((1u << lane) - 1u));
      const unsigned long long j = pri ? (unsigned long long)(out.n_slots - 1) - r : r;
      SlotState& o = out;
      o.model[j] = ph.model; o.pid[j] = ph.pid;
      o.event[j] = ph.key.event;
      o.px[j] = ph.px; o.py[j] = ph.py; o.pz[j] = ph.pz;
      o.ox[j] = ph.ox; o.oy[j] = ph.oy; o.oz[j] = ph.oz; o.safe[j] = ph.safe;
      o.kx[j] = ph.k.x; o.ky[j] = ph.k.y; o.kz[j] = ph.k.z;
      o.X[j] = ph.X; o.x[j] = ph.x; o.region[j] = (uint8_t)ph.region;
      o.fly[j] = ph.fly; o.fly_tau[j] = ph.fly_tau;
      o.nscat[j] = ph.nscat; o.ndust[j] = ph.ndust; o.iters[j] = ph.iters; o.steps[j] = ph.steps;
    }
  }
}

// ---- frequency pre-sorting of resident packets between served rounds ----------------
// Sorting packets by frequency before they are handed to warps groups those that take the
// same branches (the paper's pre-sorting, App. A.1 and Sec. 7.1): here, between rounds, the
// front list of `from` (from.live[1] packets) is copied into `to` by bucket -- line core
// (|x| <= 2), near wing (|x| <= 5), far wing, empty cavity -- and the resume hands each warp
// contiguous entries, so a warp's packets are of one kind (core packets then run the
// core events in step, wing packets the general event).  The back (priority)
// list is copied in place.  cnt[0..3]: bucket sizes, cnt[4..7]: cursors, zero on entry.
// The order inside a bucket does not matter: a packet's history does not depend on its
// warp or lane.
__device__ __forceinline__ int slot_bucket(const SlotState& s, int64_t i) {
  if (s.region[i]) return 3;
  const float ax = fabsf(s.x[i]);
  return ax <= 2.0f ? 0 : (ax <= 5.0f ? 1 : 2);
}
__device__ __forceinline__ void copy_slot(const SlotState& a, int64_t i, const SlotState& b, int64_t j) {
  b.px[j] = a.px[i]; b.py[j] = a.py[i]; b.pz[j] = a.pz[i];
  b.ox[j] = a.ox[i]; b.oy[j] = a.oy[i]; b.oz[j] = a.oz[i]; b.safe[j] = a.safe[i];
  b.kx[j] = a.kx[i]; b.ky[j] = a.ky[i]; b.kz[j] = a.kz[i]; b.X[j] = a.X[i]; b.x[j] = a.x[i];
  b.event[j] = a.event[i];
  b.fly[j] = a.fly[i]; b.fly_tau[j] = a.fly_tau[i];
  b.nscat[j] = a.nscat[i]; b.ndust[j] = a.ndust[i]; b.iters[j] = a.iters[i]; b.steps[j] = a.steps[i];
  b.model[j] = a.model[i]; b.pid[j] = a.pid[i]; b.region[j] = a.region[i];
}
__global__ void slot_hist_kernel(SlotState from, unsigned long long* __restrict__ cnt) {
  const unsigned long long n = from.live[1];
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const bool mine = (unsigned long long)i < n;
  const int key = mine ? slot_bucket(from, i) : 4;
  const unsigned peers = __match_any_sync(kFull, key);
  if (mine && (int)(threadIdx.x & 31u) == __ffs(peers) - 1) atomicAdd(&cnt[key], (unsigned long long)__popc(peers));
}
__global__ void slot_sort_kernel(SlotState from, SlotState to, unsigned long long* __restrict__ cnt) {
  const unsigned long long n = from.live[1], nb = from.live[3];
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const unsigned lane = threadIdx.x & 31u;
  const bool mine = (unsigned long long)i < n;
  const int key = mine ? slot_bucket(from, i) : 4;
  const unsigned peers = __match_any_sync(kFull, key);
  const int leader = __ffs(peers) - 1;
  unsigned long long base = 0;
  if (mine && (int)lane == leader) base = atomicAdd(&cnt[4 + key], (unsigned long long)__popc(peers));
  base = __shfl_sync(kFull, base, leader);
  if (mine) {
    unsigned long long off = 0;
    for (int k = 0; k < key; ++k) off += cnt[k];
    copy_slot(from, i, to, (int64_t)(off + base + __popc(peers & ((1u << lane) - 1u))));
  }
  if ((unsigned long long)i < nb) copy_slot(from, from.n_slots - 1 - i, to, to.n_slots - 1 - i);
}

}  // namespace

cudaError_t launch_slot_presort(SlotState from, SlotState to, unsigned long long* cnt, cudaStream_t s) {
  const unsigned grid = (unsigned)((from.n_slots + 255) / 256);
  cudaMemsetAsync(cnt, 0, 8 * sizeof(unsigned long long), s);
  slot_hist_kernel<<<grid, 256, 0, s>>>(from, cnt);
  slot_sort_kernel<<<grid, 256, 0, s>>>(from, to, cnt);
  return cudaGetLastError();
}

// Shared memory of a block: one buffer of event words per warp.
static size_t chain_bytes(int block) { return (size_t)(block / 32) * sizeof(WordBuf); }
template <class F>
static cudaError_t allow_chain(F* f) {  // 73 KB for the largest block: above the default limit
  return cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)chain_bytes(256));
}

int shell_grid(int block, int blocks_per_sm, bool sliced) {
  int dev = 0, sms = 0, occ = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  allow_chain(shell_slice_kernel<true>);
  allow_chain(shell_slice_kernel<false>);
  allow_chain(shell_run_kernel<true, 0>);
  allow_chain(shell_run_kernel<false, 0>);
  allow_chain(shell_run_kernel<true, 1>);
  allow_chain(shell_run_kernel<false, 1>);
  const size_t smem = chain_bytes(block);
  if (sliced) cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, shell_slice_kernel<true>, block, smem);
  else cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, shell_run_kernel<true, 0>, block, smem);
  if (occ < 1) occ = 1;
  const int b = (blocks_per_sm > 0 && blocks_per_sm < occ) ? blocks_per_sm : occ;
  return sms * b;
}

cudaError_t launch_shell_run(const ShellModel* d_models, WorkQueue q, const float* d_ktab, int grid, int block,
                             int profile, int per_warp, int core_lanes, int burst_lanes, cudaStream_t s,
                             const Compact* share) {
  Compact none{};
  if (share) {  // the work-sharing fields
    none.pool = share->pool;
    none.ready = share->ready;
    none.share = share->share;
    none.n_total = share->n_total;
  }
  none.per_warp = per_warp;
  none.core_lanes = core_lanes;
  none.burst_lanes = burst_lanes;
  if (profile) shell_run_kernel<false, 1><<<grid, block, chain_bytes(block), s>>>(d_models, q, none, d_ktab);
  else shell_run_kernel<false, 0><<<grid, block, chain_bytes(block), s>>>(d_models, q, none, d_ktab);
  return cudaGetLastError();
}

cudaError_t launch_shell_run_compact(const ShellModel* d_models, WorkQueue q, Compact c, const float* d_ktab,
                                     int grid, int block, int profile, cudaStream_t s) {
  if (profile) shell_run_kernel<true, 1><<<grid, block, chain_bytes(block), s>>>(d_models, q, c, d_ktab);
  else shell_run_kernel<true, 0><<<grid, block, chain_bytes(block), s>>>(d_models, q, c, d_ktab);
  return cudaGetLastError();
}

cudaError_t launch_shell_slice(const ShellModel* d_models, WorkQueue q, SlotState in, SlotState out, uint32_t budget,
                               const float* d_ktab, int grid, int block, bool mixed, cudaStream_t s) {
  const size_t smem = chain_bytes(block);
  if (mixed) shell_slice_kernel<true><<<grid, block, smem, s>>>(d_models, q, in, out, budget, d_ktab);
  else shell_slice_kernel<false><<<grid, block, smem, s>>>(d_models, q, in, out, budget, d_ktab);
  return cudaGetLastError();
}

}  // namespace thor
