// plan.h -- the launch plan of the stencil kernels: which tile and how many z
// chunks for a grid.  Host arithmetic only (no CUDA call), shared by the FP32,
// binary16 and TTI kernels.
#pragma once

#include <limits.h>
#include <math.h>
#include <stdint.h>

namespace fdsweep {

// Time of `units` equal CTAs on nsm SMs with per_sm places each, in units of a
// CTA alone on its SM: k CTAs on an SM take sqrt(1 + (load k)^2).
inline double wave_cost(int64_t units, int nsm, int per_sm, double load) {
    const int64_t slots = (int64_t)nsm * per_sm;
    auto h = [&](double k) { return sqrt(1.0 + load * load * k * k); };
    const int64_t full = units / slots, rem = units - full * slots;
    double waves = (double)full * h(per_sm);
    if (rem) {
        // the last wave: between the mean and the fullest SM's load
        double k = (double)rem / nsm;
        if (k < 1.0) k = 1.0;
        waves += h(0.5 * (k + ceil(k)));
    }
    return waves;
}

// Number of z chunks into which the columns of a z-marching stencil launch
// are cut (1 .. nz).  A CTA marches `warmup` planes (in units of a full
// plane's time) before its chunk's first output, and the columns times the
// chunks fill the machine in waves of nsm * per_sm CTAs, so the launch lasts
// about
//   (chunk + warmup) * sum over the waves of h(CTAs per SM),
//   h(k) = sqrt(1 + (load k)^2),
// h being the time of one plane relative to a lone CTA's: constant (the
// latency of one plane's copy and arithmetic) while few CTAs share an SM,
// proportional to k once its throughput (shared memory, HBM) is used up.
// The count with the smallest estimate is taken.  Filling the slots and
// rounding the count up instead (a few CTAs then run a whole wave of their
// own) took 1.1x to 6x as long up to 384^3, measured on GB300 with one
// consumer thread as the producer: acoustic 64^3 so 4 20.1 against 7.2 us per
// step, 256^3 so 8 77 against 53, 384^3 so 8 170 against 142; TTI 48^3 so 4 85
// against 15, 256^3 so 8 382 against 301.
// `planes` (optional) receives the estimate.
inline int pick_z_chunks(int64_t cols, int nsm, int per_sm, int nz, double warmup, double load,
                         double *planes = nullptr) {
    const int64_t slots = (int64_t)nsm * per_sm;
    // beyond a few waves more chunks only add warm-up planes
    const int64_t most = 8 * slots / (cols > 0 ? cols : 1) + 8;
    int best = 1;
    double best_cost = 0.0;
    int last_chunk = 0;
    for (int n = 1; n <= nz && n <= most; ++n) {
        const int chunk = (nz + n - 1) / n;
        if (chunk == last_chunk) continue;
        last_chunk = chunk;
        const int64_t units = cols * ((nz + chunk - 1) / chunk);
        const double cost = (chunk + warmup) * wave_cost(units, nsm, per_sm, load);
        if (n == 1 || cost < best_cost) {
            best_cost = cost;
            best = n;
        }
    }
    if (planes) *planes = best_cost;
    return best;
}

// A candidate launch and what it costs (microseconds): `launch` + `lat` x the
// estimate of pick_z_chunks with load thr / lat; a block of a one-block kernel
// counts as one plane.
struct PlanEntry {
    int bx, by;       // tile of a CTA
    int bz;           // z points of a one-block kernel's CTA; 0: the CTA marches z
    int per_sm;       // CTAs that fit on an SM
    float launch, lat, thr;
    double warmup;    // planes before a chunk's first output
    int max_chunk;    // planes a chunk can have (shared memory)
    int long_chunk;   // planes a chunk has where the grid limit allows (0: max_chunk)
    bool spare;       // only where no other candidate can be launched
};

struct PlanChoice {
    int entry = -1;   // -1: no candidate can be launched
    int zchunk = 0, nzc = 0;
    double us = 0.0;
};

constexpr int kMaxGridYZ = 65535;
// z blocks of a launch up to which slices are left for its receiver blocks
constexpr int kMostColumnsZ = 60000;

// The launch of candidate e alone: its chunk and estimated time; false if its
// grid or a chunk would be too large.
inline bool plan_one(const PlanEntry &e, bool forced, int nx, int ny, int nz, int nshots, int nsm,
                     PlanChoice *c) {
    const int64_t ntx = (nx + e.bx - 1) / e.bx, nty = (ny + e.by - 1) / e.by;
    if (nty > kMaxGridYZ || nshots > kMaxGridYZ || e.max_chunk < 1) return false;
    const int64_t cols = ntx * nty * nshots;
    const double load = e.thr / e.lat;
    double planes = 0.0, penalty = 1.0;
    if (e.bz) {
        const int nzc = (nz + e.bz - 1) / e.bz;
        const double waves = (double)cols * nzc / ((double)nsm * e.per_sm);
        // A second wave of blocks hides nothing: only for a clear gain (TTI
        // 96^3 so 4 17.4 against 22.0 us, K1 128^3 so 8 14.9 against 9.8), and
        // never a third.
        if ((waves > 2.0 || (int64_t)nzc * nshots > kMostColumnsZ) && !forced) return false;
        if (waves > 1.0) penalty = 1.06;
        planes = wave_cost(cols * nzc, nsm, e.per_sm, load);
        c->zchunk = e.bz;
    } else {
        int nzc = pick_z_chunks(cols, nsm, e.per_sm, nz, e.warmup, load, &planes);
        const int fewest = (nz - 1) / e.max_chunk + 1;
        const int some = e.long_chunk ? (nz - 1) / e.long_chunk + 1 : fewest;
        if (nzc < some) nzc = some;
        const int room = kMostColumnsZ / nshots > 1 ? kMostColumnsZ / nshots : 1;
        if (nzc > room) nzc = room;
        // a chunk that fits comes before the receivers' slices (the sparse
        // kernel records where none is left)
        if (nzc < fewest) nzc = fewest;
        c->zchunk = (nz - 1) / nzc + 1;
    }
    c->nzc = (nz - 1) / c->zchunk + 1;
    c->us = (e.launch + e.lat * planes) * penalty;
    return (int64_t)nshots * c->nzc <= kMaxGridYZ;
}

// The candidate (`forced` >= 0: that one) and chunk count with the smallest
// estimated time among those that can be launched.
inline PlanChoice choose_plan(const PlanEntry *e, int n, int forced, int nx, int ny, int nz,
                              int nshots, int nsm) {
    PlanChoice best;
    for (int pass = 0; pass < 2 && best.entry < 0; ++pass)
        for (int i = 0; i < n; ++i) {
            if (forced >= 0 ? i != forced : e[i].spare != (pass == 1)) continue;
            PlanChoice c;
            if (!plan_one(e[i], forced >= 0, nx, ny, nz, nshots, nsm, &c)) continue;
            c.entry = i;
            if (best.entry < 0 || c.us < best.us) best = c;
        }
    return best;
}

// Checkpoint interval K, segments, imaging steps per launch G (the adjoint's
// ring has G + 1 levels) and shots of a batch B of a gradient over nsteps steps
// of nshots shots on fields of vol floats.
//   available  bytes the call can allocate: what is free on the device and what
//              the memory pool holds unused.  Both decisions below count the
//              same bytes, so that a call's batches (and with them the order of
//              its sums) do not depend on how far earlier calls grew the pool.
//   fixed      bytes of everything but the per-shot levels.
//   cap, most_steps  upper limits of B and G.
// A batch is kGradShots shots, or as many as have kGradBatchPoints points.
// checkpoint_every = 0 keeps the whole history of a batch (K = nsteps, no
// recomputation) where it takes at most an eighth of the device memory and a
// quarter of what is available (smaller batches where only kGradShots shots'
// does), and round(sqrt(nsteps)) steps otherwise.
// The imaging condition takes kGradShots shots per launch, and so does a batch
// of large grids; where eight shots leave the device idle a batch is as many as
// have kGradBatchPoints points.  59 steps, segments of 8, ms with batches of 8 /
// of 4e6 / 8e6 / 1.6e7 points: 64 shots of 40^3 so 16 18.6 / 9.6 / 8.6 / 8.6,
// 64 of 48^3 so 4 14.0 / 8.4 / 7.5 / 7.5, 32 of 64^3 9.2 / 7.2 / 7.0 / 6.2, 24
// of 80^3 so 8 14.7 / 14.5 / 13.8 / 12.8; from 96^3 on the same within 1 %.
constexpr int kGradShots = 8;
constexpr double kGradBatchPoints = 1.6e7;

struct GradientPlan {
    int K, nseg, G, B;
    int nfwd, nck;  // forward levels and checkpoint levels per shot
};

inline GradientPlan plan_gradient(int nsteps, int nshots, int64_t vol, int checkpoint_every,
                                  int cap, int most_steps, double total, double available,
                                  double fixed) {
    GradientPlan p;
    const double level = (double)vol * 4.0;
    double wide = ceil(kGradBatchPoints / (double)vol);
    if (wide > kMaxGridYZ / 4) wide = kMaxGridYZ / 4;  // shots lie along the grid's z
    int most = wide > kGradShots ? (wide < nshots ? (int)wide : nshots) : kGradShots;
    if (most > nshots) most = nshots;
    if (most > cap) most = cap;
    p.K = checkpoint_every > 0 ? checkpoint_every
                               : (int)lround(sqrt((double)(nsteps > 1 ? nsteps : 1)));
    const double history = (nsteps + 2) * level;  // of a shot
    const double keep = total / 8 < available / 4 ? total / 8 : available / 4;
    if (checkpoint_every == 0) {
        if (most > kGradShots && most * history > keep && kGradShots * history <= keep)
            most = kGradShots;
        if (most * history <= keep) p.K = nsteps;
    }
    if (p.K < 1) p.K = 1;
    if (nsteps > 0 && p.K > nsteps) p.K = nsteps;
    p.nseg = nsteps > 0 ? (nsteps - 1) / p.K + 1 : 0;
    p.nfwd = p.nseg > 1 ? 2 : 0;
    p.nck = p.nseg > 1 ? 2 * p.nseg : 0;
    p.G = p.K < most_steps ? p.K : most_steps;
    const double per_shot = ((double)p.nfwd + p.G + 1 + p.K + 2 + p.nck) * level;
    const double fit = (0.8 * available - fixed) / per_shot;
    p.B = fit >= most ? most : (int)fit;
    if (p.B < 1) {  // the least: one shot, two adjoint levels, one step per launch
        p.G = 1;
        p.B = 1;
    }
    return p;
}

}  // namespace fdsweep
