// Rules of the resident step kernel (lbm_resident.cu) that need no GPU to evaluate: plain C++ that
// the kernel, its launches and the CPU tests share.
#pragma once

#include <algorithm>
#include <new>
#include <vector>

#ifdef __CUDACC__
#define CMLBM_RULE __host__ __device__ __forceinline__
#else
#define CMLBM_RULE inline
#endif

namespace cmlbm {

constexpr int kResidentWarps = 16;   // warps of a block; one block per SM

// The carry row holds what the last row of a round pushed north, planes 2, 5 and 6 of the row above
// it, all columns of which the next round, whose first row that is, copies into place and then pushes.
// Two words of such a row come from nowhere in the round before: plane 5 of the first column beside a
// no-slip left side and plane 6 of the last one beside a no-slip right side, which the row's own node
// bounces back there in the round of the copy.  (A free-slip side mirrors populations 6 and 5 of the
// row below into the same words; they then come from the round before, and copy and pushes write
// different words, as they do everywhere else.)  The copy has nothing valid for the two: either it is
// over before the pushes, by a barrier in blocks at a walled side of a grid with a no-slip one (slip: the
// free-slip sides, bit 0 left, bit 1 right), or it leaves them out.  The two lattices take the barrier,
// the interface lattice alone the shorter copy, which each came out faster, through the registers of
// the whole loop also on grids without such sides: us a step at 256 x 1024 5.70 against 5.76, imposed
// flow 800 x 800 8.04 against 7.86 (the whole copy without a barrier: 5.69 and 7.94).
CMLBM_RULE bool carry_meets_pushes(int slip) { return (slip & 3) != 3; }
CMLBM_RULE bool carry_fills(int plane, int column, int width, bool noslip_left, bool noslip_right)
{
    return !(noslip_left && plane == 5 && column == 0) &&
           !(noslip_right && plane == 6 && column == width - 1);
}

// ---- plans ----------------------------------------------------------------------------------
struct GridSize {
    int nx, ny;
};

// A step of a launch, in units of one row for each of four warps: the exchange and the sums
// (kStepRows), the rows of the tallest block by fours (a warp of each quarter SM), and the start of
// every further round of 16.  One GB300, FP32, us a step of blocks of 2, 4, 8, 12, 16, 20, 24, 28, 32,
// 36 rows (all SMs, 4 strips): 2.6, 2.8, 3.3, 3.5, 4.0, 4.8, 5.3, 5.8, 6.5, 7.3; FP16 up to 32: 3.0,
// 3.3, 3.8, 4.6, 5.3, 6.6, 7.1, 7.7, 8.4.
inline double step_cost(int h)
{
    constexpr double kStepRows = 4.5, kRound = 0.6;
    return kStepRows + (h + 3) / 4 + kRound * ((h + kResidentWarps - 1) / kResidentWarps - 1);
}

// Waves of a batch: every case gets the fewest blocks of at most `cap` rows; cases of like block
// heights share a wave (its step takes as long as its tallest block), and the blocks a wave has left
// go to the cases with its tallest.
struct WavePart {
    int c, nstrip, nseg, h;
};
using Wave = std::vector<WavePart>;

inline int tallest(const Wave& wave)
{
    int h = 2;
    for (const WavePart& p : wave) h = std::max(h, p.h);
    return h;
}
inline int blocks_of(const Wave& wave)
{
    int n = 0;
    for (const WavePart& p : wave) n += p.nstrip * p.nseg;
    return n;
}
inline double waves_cost(const std::vector<Wave>& waves)
{
    double t = 0;
    for (const Wave& wave : waves) t += step_cost(tallest(wave));
    return t;
}

inline std::vector<Wave> waves_of(const std::vector<GridSize>& G, int nsm, int cap)
{
    std::vector<WavePart> parts;
    int smallest = nsm;
    for (int c = 0; c < (int)G.size(); ++c) {
        WavePart p = {c, (G[c].nx + 63) / 64, (G[c].ny + cap - 1) / cap, 0};
        p.h = (G[c].ny + p.nseg - 1) / p.nseg;
        if (p.nstrip * p.nseg > nsm) return {};
        smallest = std::min(smallest, p.nstrip * p.nseg);
        parts.push_back(p);
    }
    std::stable_sort(parts.begin(), parts.end(),
                     [](const WavePart& a, const WavePart& b) { return a.h > b.h; });
    std::vector<Wave> bins;
    std::vector<int> used;
    size_t open = 0;   // first wave that could still take a case
    for (const WavePart& p : parts) {
        while (open < bins.size() && used[open] + smallest > nsm) ++open;
        size_t w = open;
        while (w < bins.size() && used[w] + p.nstrip * p.nseg > nsm) ++w;
        if (w == bins.size()) {
            bins.push_back({});
            used.push_back(0);
        }
        bins[w].push_back(p);
        used[w] += p.nstrip * p.nseg;
    }
    for (size_t w = 0; w < bins.size(); ++w) {
        Wave& b = bins[w];
        for (;;) {
            WavePart* t = &b[0];
            for (WavePart& p : b)
                if (p.h > t->h) t = &p;
            // one segment more at a time shortens the tallest only now and then: go to the next
            // count that does
            int n = t->nseg + 1;
            while (n <= G[t->c].ny / 2 && (G[t->c].ny + n - 1) / n == t->h) ++n;
            if (n > G[t->c].ny / 2 || used[w] + (n - t->nseg) * t->nstrip > nsm) break;
            used[w] += (n - t->nseg) * t->nstrip;
            t->nseg = n;
            t->h = (G[t->c].ny + n - 1) / n;
        }
    }
    return bins;
}

// The taller its blocks, the less of a step a wave spends in the exchange; but a batch short of
// several full waves goes faster in one more wave of lower ones than in a last wave nearly empty.
// The block height cap with the shortest sum over the waves is taken (multiples of four, and what
// fits).  One GB300, FP32 drops of sides 32 - 256, us a step, always what fits / this: 30 cases 17.1 /
// 15.5, 45 25.0 / 23.8, 140 81.3 / 79.8; 16, 24, 64, 100 and 192 keep the same plan.
//
// The wave of the most blocks comes first: a device (or a part of one) on which not all its blocks
// can be resident refuses its launch, so that a run is either refused before any case has moved, or
// not at all.  Empty where a case does not fit or host memory runs out.
inline std::vector<Wave> batch_waves(const std::vector<GridSize>& G, int nsm, int fit)
try {
    std::vector<Wave> best = waves_of(G, nsm, fit);
    if (best.empty()) return best;
    double least = waves_cost(best);
    for (int cap = 8; cap < fit; cap += 4) {
        std::vector<Wave> other = waves_of(G, nsm, cap);
        if (other.empty() || waves_cost(other) >= least) continue;
        least = waves_cost(other);
        best.swap(other);
    }
    std::stable_sort(best.begin(), best.end(), [](const Wave& a, const Wave& b) {
        return blocks_of(a) > blocks_of(b);
    });
    return best;
} catch (const std::bad_alloc&) {
    return {};
}

// Whether a batch's run goes to the waves or to graph replays of one launch a step, from what either
// takes.  Waves: kWaveUnit us a step for each unit of their cost, and kWaveRun us a wave and run, in
// which it is launched and its part of the state read and written.  Replays of the default launch
// shape: by the strips of 64 columns, filled or not, times their rows, and by the strips (whose last
// segments are short).  One GB300, 96 - 2000 drops of sides 32 - 64, 32 - 256, 200 - 256 and 300 - 500
// (1.8 - 20.7 million nodes): the waves' steps within 3 % of this, the replays' within 3 % in FP32
// and 5 % in 16 bits (the waves are far ahead below that).  Measured, us a step, replays /
// waves: FP32 192 drops 134 / 107, 512 311 / 264, 60 of sides 300 - 500 260 / 239 (in runs of 16
// steps 286); FP16 192 drops 151 / 142, 512 340 / 351, 400 of sides 200 - 256 590 / 674, 2000 of
// sides 32 - 64 189 / 182.
constexpr double kWaveRun = 23.0;
inline double wave_unit(bool narrow) { return narrow ? 0.638 : 0.495; }

inline double waves_us(const std::vector<Wave>& waves, bool narrow)
{
    return wave_unit(narrow) * waves_cost(waves);
}
inline double replays_us(const std::vector<GridSize>& G, bool narrow)
{
    double nodes = 0, strips = 0;
    for (const GridSize& g : G) {
        strips += (g.nx + 63) / 64;
        nodes += 64.0 * ((g.nx + 63) / 64) * g.ny;
    }
    return narrow ? 27.6 + 24.1e-6 * nodes + 0.0171 * strips
                  : 18.2 + 22.4e-6 * nodes + 0.0188 * strips;
}
inline bool waves_pay(int steps, size_t nwaves, double waves_step, double replays_step)
{
    return steps * waves_step + kWaveRun * nwaves < steps * replays_step;
}

// A grid's segments.  Alone on the device a step is fastest over all SMs, each block a strip of 64
// columns by as few rows as that leaves; but a block has its SM to itself, so that several contexts on
// several streams then run one after another, where the small launches of graph replays ran side by
// side.  A context on a stream of its own therefore takes the most segments (the lowest blocks, the
// shortest step) with which neither it alone nor two, four or eight like it are slower than in the
// other forms, and where there are none (0) the other forms.  Their times are modelled from one
// GB300's: contexts alone, and eight side by side on eight streams.  All SMs / other forms / this, us
// for a step of each of 1, 2, 4, 8 contexts:
//   FP32 128 x 128   2.5 4.9 9.7 19.5 / 3.9 4.2 5.1 6.3 / 3.0 3.1 3.3 6.5
//   FP32 256 x 256   3.3 6.6 13.1 26.4 / 5.3 6.9 9.6 19.7 / 4.0 4.0 8.1 16.0
//   FP32 161 x 481   3.6 7.1 14.3 28.6 / 6.5 7.5 13.5 28.6 / 4.8 4.8 9.5 19.0
//   BF16 512 x 256   5.1 10.2 20.4 40.8 / 7.8 10.3 16.4 33.1 / the other forms
enum class Form { Fp32, Narrow, Flow };   // 32-bit and 16-bit storage; the interface lattice alone

inline double resident_step_us(Form form, int h)   // blocks of h rows; within 8 % of the kernel's
{
    const int rounds = (h + kResidentWarps - 1) / kResidentWarps;
    switch (form) {
    case Form::Narrow: return 2.7 + 0.15 * h + 0.7 * (rounds - 1);
    case Form::Flow: return 2.3 + 0.045 * h + 0.047 * std::max(0, h - 32);
    default: return 2.35 + 0.115 * h + 0.35 * (rounds - 1);
    }
}
struct OtherForms {
    double alone, share;   // us a step of one by itself, and of each of many side by side
};
inline OtherForms other_forms(Form form, double nodes)   // (nodes of whole strips)
{
    switch (form) {
    case Form::Narrow: return {4.2 + 27e-6 * nodes, 0.35 + 32e-6 * nodes};
    case Form::Flow: return {3.5 + 14.5e-6 * nodes, 0.35 + 18e-6 * nodes};
    default: return {3.4 + 31e-6 * nodes, 0.5 + 26e-6 * nodes};
    }
}
inline int most_segments(GridSize G, int nsm)
{
    return std::min(nsm / ((G.nx + 63) / 64), G.ny / 2);
}
inline int shared_segments(GridSize G, int nsm, int fit, Form form)
{
    const int nstrip = (G.nx + 63) / 64;
    const OtherForms other = other_forms(form, 64.0 * nstrip * G.ny);
    for (int nseg = most_segments(G, nsm); nseg >= 1; --nseg) {
        const int h = (G.ny + nseg - 1) / nseg;
        const double step = resident_step_us(form, h);
        if (h > fit || step > other.alone) break;
        const int at_once = nsm / (nstrip * nseg);
        bool no_slower = true;
        for (int k = 2; k <= 8; k *= 2)
            no_slower &= (k + at_once - 1) / at_once * step <= std::max(other.alone, k * other.share);
        if (no_slower) return nseg;
    }
    return 0;
}

// Steps of one launch.  While it runs nobody else gets its SMs, so a longer run is cut: 4096 steps
// take 10 - 35 ms, and what a launch costs beside its steps is 0.1 % of them or less (us a step in
// launches of 512 / 4096 steps: 64 x 64 2.234 / 2.213, 400 x 700 7.190 / 7.148).
constexpr int kResidentMaxSteps = 4096;

}  // namespace cmlbm
