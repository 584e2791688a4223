// ctu_launch.h -- host-side launchers of the CTU kernels (internal).
#pragma once

#include <cuda_runtime.h>

#include "ctu_kernels.cuh"

namespace ctu {

// Scratch words (of the working precision) per unit of scratch stride:
// V (9), first-order fluxes F^n (3 x 9), running sum A = L_x (+ L_y) (9).
constexpr int SCRATCH_ARRAYS = 9 + 27 + 9;

// Optional per-kernel timing hook: mark(name) is called right before a
// launch and mark(nullptr) right after it, on the same stream.
struct ProfHook {
    virtual void mark(const char *name, cudaStream_t s) = 0;
    virtual ~ProfHook() {}
};

// Patches of identical shape, contiguous in the device patch table, with the
// thread-tile width along x (8, 16 or 32), the marching segment lengths (the
// sweeps', the first-order kernels') and the row widths of the x-tiled and ring
// kernels (group_widths).  A launch covers up to MAXG groups (GroupTable).
struct Group {
    int first, count;
    int n[3], N[3];
    int xw, seg, seg1;
    unsigned char sx, dx, rw;
};
inline void group_widths(Group &G, int ndim, bool f64, bool mt)
{
    G.sx = (unsigned char)sweepx_width(G.n, f64);
    G.dx = (unsigned char)div1x_width(G.n, ndim);
    G.rw = (unsigned char)ring_width(G.n, f64 ? 0.0 : mt ? 0.004 : 0.01);
}

// Marching segment lengths for a batch: of the first-order kernels (seg1) and,
// for the groups `pick` marks (the untuned ones), of the sweeps (seg), each the
// candidate with the least modelled time of its launches along y and z.  A
// thread marches L = seg + 2 cells (seg + 1), so long segments do the least
// work, but a small batch then leaves most of the chip idle behind a few
// serial chains.  With B blocks on S SMs, a step of the march takes a + k
// while k blocks share an SM (a: the latency part, in units of the throughput
// part of one block), at most `fit` of them, and the whole launch L times
//   floor(B / (fit S)) (a + fit) + (a + ceil(rest / S), if a rest is left),
// L the batch's mean, and no less than its longest march takes (a level of 162
// patches of 8^3 to 64^3 marched 64 cells without this, z and y 319 and 435 us;
// 16 with it, 230 and 254).
// Fitted on the GB300 to 11 lengths of 21 shapes: a = 1.5 in float32, 0.15 for
// float64 MHD, whose single block per SM already fills the FP64 pipe.  Against every
// candidate on 28 boxes: the sweeps within 3.5% of the fastest, 6% at two float64
// ones (64^3, 200 x 131 x 67), k_div1 within 3%.  k_pred takes k_div1's constants,
// though it does four times the work a cell, and is up to 17% (48^3) off its own
// best; the float64 relativistic k_div1 up to 26% (32^3).  us per step at the fixed
// 16 and at the model's choice: 2-D 128^2 float64 1326 and 369, 48^3 mixed 167 and
// 112, 64^3 mixed 208 and 180, 512^2 mixed 124 and 109, 256^3 mixed 5144 and 5026.
// Relativistic sweeps, fitted to 10 lengths of 16 boxes of the beam: a = 0.5
// in float32 and 2 in float64, and c L more (c = 0.5, 0.75), since pencils
// differ in their iterations and a long one finishes late; within 6% of the
// fastest in float64, within 11% in float32 (3% on average).  us of the sweep along
// z at 8 cells, at 16 and at the choice: 64^3 mixed 376, 580, 285; 128^3 mixed
// 1103, 1036, 1036; 64^3 float64 1068, 1280, 1068.
// The Taub-Mathews gas in float32 (float64 iterations, whose number differs most
// between pencils): c = 2, fitted to 15 lengths of 14 boxes, within 9% of the fastest
// (2% on average); us a step at c = 0.5 and 2: 48^3 5252 and 4219, 128^3 17390 and
// 16440, 130 x 70 x 50 9390 and 8460.
template <class Pick>
inline void choose_segments(Group *g, int ng, int ndim, bool f64, bool rel, bool tm, int sms, Pick pick)
{
    static const int cand[] = {1, 2, 3, 4, 6, 8, 12, 16, 24, 32, 48, 64};
    const double S = sms > 0 ? sms : 152;
    if (ndim < 2) return;
    for (int ring = 0; ring < 2; ++ring) {
        // the kernels' registers: 168 (three blocks), the float relativistic
        // ones 128 (four; the Taub-Mathews ones three, fitted at four), the float
        // first-order ones about 95 (five)
        const double fit = f64 ? 3.0 : ring ? 5.0 : rel ? 4.0 : 3.0;
        const double a = rel && !ring ? (f64 ? 2.0 : 0.5) : f64 && !rel ? 0.15 : 1.5;
        const double late = rel && !ring ? (f64 ? 0.75 : tm ? 2.0 : 0.5) : 0.0;
        int best = 0;
        double top = 0.0;
        for (int c : cand) {
            double t = 0.0;
            for (int D = 1; D < ndim; ++D) {
                double blocks = 0.0, steps = 0.0, longest = 0.0;
                for (int i = 0; i < ng; ++i) {
                    const Group &G = g[i];
                    const int seg = ring || pick(G) ? c : G.seg, len = seg < G.n[D] ? seg : G.n[D];
                    const double b = (double)G.count * (ring ? Tiles::div1(G.n, ndim, D, G.rw, seg)
                                                             : Tiles::sweep_m(G.n, D, G.xw, seg));
                    blocks += b;
                    steps += b * (len + (ring ? 1 : 2));
                    if (len + (ring ? 1 : 2) > longest) longest = len + (ring ? 1 : 2);
                }
                if (blocks <= 0.0) continue;
                const double k = blocks / S, full = (double)(long long)(k / fit), rest = k - full * fit;
                const double tail = rest > 1e-9 ? a + (double)(long long)(rest + 0.999999) : 0.0;
                const double mean = steps / blocks * (full * (a + fit) + tail + late);
                const double chain = longest * (a + (k < fit ? (double)(long long)(k + 0.999999) : fit));
                t += mean > chain ? mean : chain;
            }
            if (best == 0 || t < top) {
                top = t;
                best = c;
            }
        }
        for (int i = 0; i < ng; ++i)
            if (ring || pick(g[i])) (ring ? g[i].seg1 : g[i].seg) = best;
    }
}

struct LaunchInfo {
    const Group *groups;   // host array, largest patches first
    int ngroups;
    int recon;             // RECON_* kernel kind (reconstruction, reference-state tracing)
    int iface64;           // mixed path: 1 = float64 interface-state recovery
    int physics;           // PH_MHD or PH_SR
    void *scratch;         // SCRATCH_ARRAYS * sstride elements of R
    StepParams *sp;        // device per-step parameters
    ProfHook *prof;        // may be null
    int sms;               // streaming multiprocessors of the device (launch_rows)
};

// Enqueue one CTU step; returns the number of kernel launches.
template <class R> int launch_step(const StepArgs &a, const LaunchInfo &li, cudaStream_t s);
// Enqueue the CFL reduction of ctu_dt into *out.
template <class R> int launch_maxspeed(const StepArgs &a, const LaunchInfo &li, unsigned long long *out,
                                       cudaStream_t s);

// Per-(precision, physics, interface-mode) instantiations, one translation
// unit each.
template <class R, int IF64> int launch_step_impl(const StepArgs &a, const LaunchInfo &li, cudaStream_t s);
template <class R> int launch_step_sr(const StepArgs &a, const LaunchInfo &li, cudaStream_t s);
template <class R, int IF64, int G> int launch_step_var(const StepArgs &a, const LaunchInfo &li, cudaStream_t s);
template <class R, int IF64> int launch_step_mt(const StepArgs &a, const LaunchInfo &li, cudaStream_t s);

} // namespace ctu
