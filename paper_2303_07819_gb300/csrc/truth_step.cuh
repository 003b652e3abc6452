// truth_step.cuh -- the wall law of the truth DEM.
#pragma once
#include "common.cuh"

namespace msd {

// Floe l against the rigid walls x = 0 and x = Lx (Sec. 4.4): the contact law
// of Eq. (2.2) with the wall as the partner, a floe at rest without spin, of
// unbounded radius and at least floe l's thickness.  Its edge is the wall
// line, so the overlap is delta = d - r_l (d: the centre's distance to the
// wall, dl and dr below), the lens becomes the segment the line cuts off with
// chord 2 sqrt(r_l^2 - d^2), and the normal n = (-1, 0) or (1, 0) points into
// the wall; the tangent t = (0, n_x).  Adds the force on l.
template <class R>
__device__ __forceinline__ void wall_add(R dl, R dr, R ul, R vl, R wl, R rl, R hl, const Phys<R> &P, R &fx,
                                         R &fy, R &tq, unsigned &deep)
{
#pragma unroll
    for (int side = 0; side < 2; side++) {
        const R d = side == 0 ? dl : dr;
        if (!(d < rl)) continue;
        const R nx = side == 0 ? R(-1) : R(1);
        const R delta = d - rl;
        const R c = d > -rl ? R(2) * sqrt(rl * rl - d * d) : R(2) * rl;
        const R hc = hl * P.inv_h_ref;
        const R vn = -ul * nx;                 // (wall - floe) velocity along n
        R Fn = c * hc * (P.E * delta + P.eta * vn);
        Fn = dmin(Fn, R(0));
        const R vt = -vl * nx - wl * rl;       // along t, minus the floe's rim speed
        R ft = c * hc * P.G * vt;
        const R cap = P.mu * (-Fn);
        ft = dmax(dmin(ft, cap), -cap);
        fx += Fn * nx;
        fy += ft * nx;
        tq += rl * ft;
        deep |= (delta < R(-0.5) * rl) ? 1u : 0u;
    }
}

}  // namespace msd
