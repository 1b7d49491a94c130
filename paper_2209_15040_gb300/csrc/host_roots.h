// Host-side roots of unity and stage-twiddle tables, shared by the plan
// builder and the allocation-free entry point (one generator for both).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <complex>
#include <unordered_map>

namespace wsfft {

// Cosine and sine of an angle of the first octant, evaluated in long double and
// rounded to both types.
struct OctantRoot {
    float cf = 0.f, sf = 0.f;
    double cd = 0.0, sd = 0.0;
};
// Those met so far: the tables of a plan repeat a few hundred angles thousands
// of times, at half a microsecond (128-bit long double) each.  Orders up to
// 4096 share a table of that order's octant, and one of its roots in float;
// longer ones are looked up by their angle in units of (pi/4) 2^-32.
struct RootMemo {
    static constexpr int LOG_ORDER = 12;
    OctantRoot near[(1 << (LOG_ORDER - 3)) + 1];
    bool known[(1 << (LOG_ORDER - 3)) + 1] = {};
    float2 circle[1 << LOG_ORDER];
    bool on_circle[1 << LOG_ORDER] = {};
    std::unordered_map<int64_t, OctantRoot> far;
};

// exp(-2*pi*i*m/n), n a power of two: the angle is reduced to the first octant by the
// eight-fold symmetry of the unit circle, evaluated in long double, then
// rounded to float (twiddles computed in higher precision and rounded once).
// With a memo each angle is evaluated once.
float2 host_root(int64_t m, int64_t n, RootMemo *memo = nullptr);
// the same root rounded to double
std::complex<double> host_root_d(int64_t m, int64_t n, RootMemo *memo = nullptr);

// Stage-twiddle table of the (N, E) register schedule (fft_core.cuh: stage
// s >= 1 reads w_{Ns*R}^{r*k} at sched_tw_offset(s) + (r-1)*Ns + k), plus one
// zero pad entry.  Writes at most `cap` entries to dst and returns how many
// it wrote, or -1 if the table does not fit.
int fill_stage_table(float2 *dst, int cap, int N, int E, RootMemo *memo = nullptr);

}  // namespace wsfft
