// The implicit u-solve's state and its control: the update that the next sweep makes.  Plain functions of
// the state and the last sweep's residual, run by one device thread after each sweep; nothing here needs CUDA,
// so they compile for the host too.
#pragma once

#ifdef __CUDACC__
#define LBM_HD __host__ __device__ __forceinline__
#else
#define LBM_HD inline
#endif

namespace lbm {

// Device-resident state of one implicit u-solve (Sec. IX): which of the two
// j~ buffers is current, the sweep counter and the residual reductions.
struct UsolveState {
    unsigned long long resid_bits;  // atomicMax over |j~new - j~| (non-negative double bits)
    unsigned long long jmax_bits;   // atomicMax over |j~new|
    int cur;                        // buffer holding the current j~
    int iter;                       // sweeps of the solve in progress
    int iters_last;                 // sweeps of the last finished solve
    int iters_max;                  // largest sweep count since init
    double resid_last;              // residual of the last sweep: after a solve, its final one
    int converged;                  // 1 once the last solve met its tolerance
    int running;                    // 1 from k_us_begin until the control kernel stops the loop
    long long sweeps_total;         // sweeps since the last reset
    // the update of the next sweep: d = c1 d_prev + c2 (J(j~) - j~), j~ += d
    double c1, c2;
    double cheb_rho;                // Chebyshev recurrence variable
    double cheb_sigma, cheb_delta;  // this solve's spectrum [1 - g, 1] of I - A (theta = 1 - g/2)
    double gain;                    // this solve's bound g, from the density range of the state
    double resid_min;               // smallest residual of the solve so far (divergence guard)
    int mode;                       // 1: Chebyshev sweeps, 2: plain sweeps of a Chebyshev solve, 0: plain
                                    // relaxation
    int wsel;                       // pair 0: the warm-start buffer holding the newest j~ (see jwp)
    int tma;                        // 1 once a sweep of this solve loaded planes by tensor copies
    int opened;                     // how this solve (after it: the last one) opened, and what the choice for
                                    // the next one remembers: OpenedBits
};

// Plain sweeps inside Chebyshev-accelerated solves (32- and 64-bit storages).  J multiplies smooth modes by
// almost zero, so on the smooth residual of a steady flow one plain sweep does what takes Chebyshev five;
// on noise Chebyshev gains a factor 4 per sweep and plain 2.  Which of the two a flow is shows in the
// ratio q of a plain sweep's residual to the one before, and nowhere in a Chebyshev solve, which damps all modes
// alike.  So a solve opens with a plain update
//   - to find out, when solves have been short for a while (kCalm: two of at most kPlainOpenMost sweeps, or
//     several of one sweep more), kWait solves after the last such attempt that failed, and
//   - after a plainly opened one that was smooth (q below Chebyshev's own factor, or close to the tolerance by
//     then) and took no more sweeps than the last Chebyshev solve, which is taken anew every kRecheck solves where
//     the two may have come close.
// A cap on the sweeps that leaves no room for the sweep that an attempt can cost keeps a solve to Chebyshev.
// The second update is plain after a smooth solve, or near the tolerance; from then on updates are plain while they
// end the solve within two sweeps, or close to the tolerance, and otherwise Chebyshev's from there.  A Chebyshev
// solve that stalls close to the tolerance ends plainly: u of size 0.03 rounds at 2e-9 in FP32, and updates of
// 1.6 residuals met that rounding at the 5e-9 tolerance.  Long solves stay Chebyshev from first to last (ended
// plainly, the noisy start of a quench took 4 % fewer sweeps but left twice the error against FP64).
//
// Measured, sweeps per step, Chebyshev throughout / opening plainly after every Chebyshev solve of 4 or 5 sweeps and
// staying plain while the residual halves / these rules: 256^3 spinodal steps 6-25 5.95 / 6.35 / 5.95, steps 41-48
// 2.4 / 2.0 / 2.0; mean of 512^2 spinodals in a flow over 60 steps - / 4.90 / 4.34; 128^3 droplets in a flow over
// 200 steps 6 / 2.53 / 2.53.
enum OpenedBits { US_PLAIN = 1, US_SMOOTH = 2 };  // bits 4-7 calm, 8-15 count, 16-23 dear (usolve_open)
constexpr int kPlainOpenMost = 5, kCalm = 6, kWait = 4, kRecheck = 16;
constexpr double kPlainNear = 4.0, kStallNear = 2.0;

// A plain sweep's update is the residual itself.
LBM_HD void plain_sweep(UsolveState& u)
{
    u.c1 = 0.0;
    u.c2 = 1.0;
}

// First step of a Chebyshev semi-iteration from the current iterate: x += r / theta.
LBM_HD void cheb_first(UsolveState& u)
{
    u.mode = 1;
    u.cheb_rho = 1.0 / u.cheb_sigma;
    u.c1 = 0.0;
    u.c2 = 1.0 / (1.0 - u.cheb_delta);
}

// Whether the sweep leaves its update for the next one: only a Chebyshev sweep is followed by one that reads it
// (c1 != 0).  The vector is 12 of a plain FP32 sweep's 60 bytes per site.
LBM_HD bool keeps_update(const UsolveState& u) { return u.mode == 1; }

// A solve's start: spectrum bound g, and its first update.  `run` is the run's last solve, which a scratch
// solve reads too: what it does depends on the run's state alone.  cheb, omega, maxit: see DevSim.
LBM_HD void usolve_open(UsolveState& u, const UsolveState& run, int cheb, double omega, int maxit, double g)
{
    const int n = run.iters_last, last = run.opened;
    u.gain = g;
    u.cheb_delta = 0.5 * g;
    u.cheb_sigma = (1.0 - 0.5 * g) / (0.5 * g);
    u.iter = 0;
    u.resid_bits = 0ull;
    u.jmax_bits = 0ull;
    u.converged = 0;
    u.running = 1;
    u.tma = 0;
    u.resid_min = 1e300;
    u.resid_last = 1e300;
    int calm = last >> 4 & 15, count = last >> 8 & 255, dear = last >> 16 & 255;
    calm = n == 0 ? 0 : n <= kPlainOpenMost ? calm + 3 : n == kPlainOpenMost + 1 ? calm + 1 : 0;
    calm = calm < kCalm ? calm : kCalm;
    bool smooth = last & US_SMOOTH, plain;
    if (!(last & US_PLAIN)) {  // `dear`: sweeps of the last Chebyshev solve; count: solves until the next attempt
        dear = n < 255 ? n : 255;
        count = count > 0 ? count - 1 : 0;
        plain = smooth || (n <= kPlainOpenMost && calm == kCalm && count == 0);
    } else if (smooth && n <= dear) {  // count: solves since the last Chebyshev one
        count = n > 3 || (n > 1 && n == dear) ? count + 1 : 0;
        plain = count < kRecheck;
        if (!plain) count = 0;
    } else {
        smooth = plain = false;
        count = kWait;
    }
    plain = plain && cheb == 1 && n > 0 && maxit > 2 * kPlainOpenMost;
    u.opened = (plain ? US_PLAIN : 0) | (smooth ? US_SMOOTH : 0) | calm << 4 | count << 8 | dear << 16;
    if (plain) {
        u.mode = 2;
        plain_sweep(u);
    } else if (cheb) {
        cheb_first(u);
    } else {  // plain relaxation x += omega r (omega = 0: 2/(2 - g))
        u.mode = 0;
        u.c1 = 0.0;
        u.c2 = omega > 0.0 ? omega : 2.0 / (2.0 - g);
    }
}

// An accelerated solve's end after sweep u.iter: one that a plain opening brought there in two sweeps was smooth.
LBM_HD void usolve_end(UsolveState& u)
{
    if (u.iter == 2 && (u.opened & US_PLAIN)) u.opened |= US_SMOOTH;
}

// The next update of an accelerated solve that goes on after sweep u.iter, of residual r (finite) and tolerance lim:
// Chebyshev semi-iteration for the real spectrum [1 - g, 1] of I - A, or plain.  resid_last holds the residual of
// the sweep before.  A residual four times above the best one so far means the spectral bound was too small: plain
// sweeps from there on (mode 0).  (One thread, which waits for the few FP64 units at each operation: what decides
// comes in products, q = r / r0, and the cheapest first.)
LBM_HD void usolve_next(UsolveState& u, int cheb, double r, double lim)
{
    if (u.mode == 1 && r > 4.0 * u.resid_min) u.mode = 0;
    bool plain = u.mode == 0;
    if (cheb == 1) {
        const double r0 = u.resid_last;
        if (!(u.opened & US_PLAIN) || (u.mode != 2 && u.iter > 2)) {
            // stalled: no progress of the size that Chebyshev makes (its factor is below 1 / sigma)
            plain = plain || u.mode == 2 || (r <= kStallNear * lim && r > 0.5 * r0 && r * u.cheb_sigma > r0);
        } else if (u.iter == 1) {
            plain = (u.opened & US_SMOOTH) || r <= kPlainNear * lim;
        } else {
            // near: at the rounding of u, where q tells nothing (g bounds the plain sweeps left there), or halving;
            // smooth: q against Chebyshev's factor sigma - sqrt(sigma^2 - 1), to its second order in 1 / sigma
            const double sg = u.cheb_sigma;
            const bool near = r <= kPlainNear * lim && (u.gain <= 0.8 || r <= 0.5 * r0);
            if (u.iter == 2) {
                const bool smooth = near || r * (4.0 * sg * sg - 1.0) <= 2.0 * sg * r0;
                u.opened = (u.opened & ~US_SMOOTH) | (smooth ? US_SMOOTH : 0);
            }
            plain = plain || near || r * r * r <= lim * r0 * r0;  // q^2 r: the residual two sweeps on
        }
    }
    if (plain) {
        u.mode = u.mode == 0 ? 0 : 2;
        plain_sweep(u);
    } else if (u.mode == 2) {
        cheb_first(u);
    } else {
        const double rn = 1.0 / (2.0 * u.cheb_sigma - u.cheb_rho);
        u.c1 = rn * u.cheb_rho;
        u.c2 = 2.0 * rn / u.cheb_delta;
        u.cheb_rho = rn;
    }
}

}  // namespace lbm
