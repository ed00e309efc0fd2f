// The laser field as the FP64 kernels evaluate it.
#pragma once

#include "tdb_internal.h"

namespace tdb {

// E(t) of eq:pumpf: E0 sin(omega t + phase) f(t) dir.
__device__ inline void field_at(const FieldDev& f, double t, double E[3]) {
    if (!f.on) {
        E[0] = E[1] = E[2] = 0.0;
        return;
    }
    double env = 1.0;
    if (f.envelope == 1) {
        const double x = t - f.t_center;
        env = exp(-x * x * 4.0 * 0.69314718055994530942 / (f.fwhm * f.fwhm));
    } else if (f.envelope == 2) {
        if (t >= 0.0 && t <= f.fwhm) {
            const double s = sin(3.14159265358979323846 * t / f.fwhm);
            env = s * s;
        } else {
            env = 0.0;
        }
    }
    const double a = f.E0 * sin(f.omega * t + f.phase) * env;
    E[0] = a * f.dir[0];
    E[1] = a * f.dir[1];
    E[2] = a * f.dir[2];
}

}  // namespace tdb
