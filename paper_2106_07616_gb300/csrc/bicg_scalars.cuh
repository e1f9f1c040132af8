// bicg_scalars.cuh -- the scalar recurrences and decisions of a resident FP64
// BiCGSTAB solve (krylov_res.cu), one system: made by one thread of every CTA
// from the same totals.  Host and device, so that a host test can walk them.
#pragma once
#include <cmath>

#include "krylov.cuh"

namespace rbffd {

// As in krylov.cu: residual growth over the best that counts as a blow-up,
// restarts from the best iterate, restarts after a breakdown.
constexpr double BICG_BLOWUP2 = 1e20;  // squared
constexpr int BICG_BLOWUPS = 8, BICG_BREAKDOWNS = 3;
// A solve of BICG_CHECK_ITS iterations or more whose recurrence meets the
// tolerance is checked against its true residual, and restarted from there
// where that is over BICG_CHECK2^(1/2) times the tolerance, at most BICG_CHECKS
// times: after thousands of iterations the two part (a 19 920-row channel,
// 7 257 Jacobi iterations to 1e-12: fields 1.4e-8 off, against 4e-11 with a
// restart).  The check refines a solve that has met its tolerance: where the
// restart does not meet it again (no iterations left, a breakdown), the solve
// ends as met, with the best iterate since (bicg_end).
constexpr double BICG_CHECK2 = 100.0;
constexpr int BICG_CHECKS = 3, BICG_CHECK_ITS = 1000;

struct BicgScalars {
  double bnorm, tol2, rho, alpha, omega, beta, rr, best2;
  int it, restarts, blowups, state;
  int need_init;  // form r = b - A x before the next iteration
  int restore;    // from the best iterate
  int save;       // x is the best iterate, to be copied before it is updated
  int run, first, half;
  int checks, met;  // true-residual checks made; the recurrence met the tolerance
  int held;         // a checked iterate of finite residual is there to fall back on
  double met_rr;    // (r, r) of the recurrence when it last met the tolerance
};

// A system whose recurrence ran away (or became non-finite) restarts from its
// best iterate, a bounded number of times.
__host__ __device__ inline void bicg_blowup(BicgScalars &c, int final_state, int maxit) {
  if (c.blowups >= BICG_BLOWUPS || c.it >= maxit) {
    c.state = final_state;
  } else {
    c.blowups++;
    c.restore = c.need_init = 1;
  }
}

// The recurrence has met the tolerance.
__host__ __device__ inline void bicg_met(BicgScalars &c) {
  if (c.checks >= BICG_CHECKS || c.it < BICG_CHECK_ITS) {
    c.state = KRY_OK;
  } else {
    c.checks++;
    c.met = c.need_init = 1;
    c.met_rr = c.rr;
  }
}

__host__ __device__ inline void bicg_start(BicgScalars &c) {
  c.bnorm = c.rho = c.alpha = c.omega = 1.0;
  c.beta = c.rr = c.tol2 = c.met_rr = 0.0;
  c.best2 = 1e308;
  c.it = c.restarts = c.blowups = c.restore = c.save = c.half = c.checks = c.met = c.held = 0;
  c.state = KRY_RUNNING;
  c.need_init = c.first = c.run = 1;
}

// A (re)start takes x from the best iterate's copy (before the true residual
// is formed).  Where the copy is still to be made (s became non-finite right
// after an improvement: x has not been updated since), x is the best iterate.
__host__ __device__ inline bool bicg_from_copy(const BicgScalars &c) {
  return c.restore && !c.save;
}

// After a (re)start: (b, b) and (r, r) of the true residual.
__host__ __device__ inline void bicg_restarted(BicgScalars &c, double bb, double rr, double tol) {
  c.need_init = c.restore = 0;
  if (c.it == 0 && c.restarts == 0 && c.blowups == 0) {
    c.bnorm = sqrt(bb);
    c.tol2 = tol * tol * bb;
  }
  c.first = 1;
  if (c.met) {
    c.met = 0;
    c.best2 = 1e308;
    // the recurrence's residual is reported, as without the check
    if (rr <= BICG_CHECK2 * c.tol2) c.state = KRY_OK;
    else c.held |= rr == rr;
  }
  if (c.state == KRY_RUNNING) c.rr = rr;
  if (c.state == KRY_OK) {
  } else if (c.bnorm == 0.0) {
    c.rr = 0.0;
    c.state = KRY_OK;
    c.half = 3;  // x = 0
  } else if (!(rr == rr)) {
    c.state = KRY_DIVERGED;
  } else if (rr <= c.tol2) {
    c.state = KRY_OK;
  } else {
    if (rr < c.best2) {
      c.best2 = rr;
      c.save = 1;
    }
    c.rho = rr;
    if (rr == 0.0) c.state = KRY_NOCONV;
  }
}

// After v = A p^: (r^, v), and the tests of the iteration whose x and r were
// just formed, (r, r) and (r^, r).
__host__ __device__ inline void bicg_after_v(BicgScalars &c, double rhv, double rr, double rhr,
                                             int maxit) {
  const bool was_first = c.first != 0;
  c.first = c.save = 0;
  c.run = 0;
  if (!was_first) {
    c.rr = rr;
    if (!std::isfinite(rr)) {
      bicg_blowup(c, KRY_DIVERGED, maxit);
    } else if (rr <= c.tol2) {
      bicg_met(c);
    } else {
      bool go = true;
      if (rr < c.best2) {
        c.best2 = rr;
        c.save = 1;  // copied to xb before the next update of x
      } else if (rr > BICG_BLOWUP2 * c.best2) {
        bicg_blowup(c, KRY_NOCONV, maxit);
        go = false;
      }
      if (go && (c.omega == 0.0 || c.rho == 0.0)) {
        // breakdown: restart from the current x
        if (c.restarts >= BICG_BREAKDOWNS) {
          c.state = KRY_NOCONV;
        } else {
          c.restarts++;
          c.need_init = 1;
        }
        go = false;
      }
      if (go && c.it >= maxit) {
        c.state = KRY_NOCONV;
        go = false;
      }
      if (go) {
        // rho' came from two products that cancel; (r^, r) summed
        // directly replaces it (krylov.cu)
        c.rho = rhr;
        c.run = 1;
      }
    }
  } else {
    c.run = 1;
  }
  if (c.run) c.alpha = c.rho / rhv;
}

// After t = A s^: (s, s), (r^, s), (r^, t), whether (t, t) is zero, and the
// quotients om = (t, s) / (t, t), iom = 1 / om and ar = alpha / rho.
__host__ __device__ inline void bicg_after_t(BicgScalars &c, double ss, double rhs, double rht,
                                             bool tt_zero, double om, double iom, double ar,
                                             int maxit) {
  c.half = 0;
  if (!c.run) return;
  c.it++;
  if (!std::isfinite(ss)) {
    c.half = 2;  // non-finite s: restart from the best iterate
    bicg_blowup(c, KRY_DIVERGED, maxit);
  } else if (ss <= c.tol2) {
    c.half = 1;
    c.rr = ss;
    bicg_met(c);
  } else {
    c.omega = tt_zero ? 0.0 : om;
    const double rho_new = rhs - c.omega * rht;
    c.beta = (c.omega == 0.0 || c.rho == 0.0) ? 0.0 : rho_new * ar * iom;
    c.rho = rho_new;
  }
}

// The end of a solve: true when x has to be taken from the best iterate's copy.
// A solve that met its tolerance and was restarted from the true residual does
// not fail for what came after.
__host__ __device__ inline bool bicg_end(BicgScalars &c) {
  if (c.state == KRY_OK || c.state == KRY_RUNNING || !c.held) return false;
  c.state = KRY_OK;
  c.rr = c.met_rr;
  return !c.save;
}

}  // namespace rbffd
