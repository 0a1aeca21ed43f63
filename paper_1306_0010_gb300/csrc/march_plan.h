// march_plan.h -- planes per CTA of the split two-pass kernels (host code, used by rhd_api.cu and by a host test).
//
// A CTA marches its column tile through z; t0 + t1 k is the time (us) of one plane with k CTAs on an SM, t_full that
// with k_max of them in a long queue, and `start` the planes' worth of work that a chunk adds (the predictor's two
// halo planes, the corrector's first face).  A launch of more CTAs than fit at once ends with half a CTA's time on
// average.  Fitted to 3 .. 128 planes on 97x61x45, 64^3, 128^3, 200x150x120, 256^3, 300x250x200 and 512^3.  A small
// grid wants enough chunks to put two or three CTAs on every SM, a large one long chunks.  Predictor and corrector,
// us, with ghost layers on every face (FULL, minmod):
//     97x61x45   5 and 5 planes 22.6 and 30.8 (the model: 21.7 and 31.0); 16 each 32.7 and 63.4; 32 each 55.4 and 118
//     64^3       5 and 4 planes 22.8 and 26.8; 16 each 32.7 and 61.3; 32 each 55.7 and 115
//     256^3      130 and 20 planes 387 and 844; 32 each 379 and 875; 64 each 379 and 925
//     512^3      65 and 57 planes 2539 and 6474; 32 each 2576 and 6485; 128 each 2553 and 6493
#pragma once

namespace rhd {

struct MarchCost {
    double start, t0, t1, t_full;
    int k_max;
};
constexpr MarchCost kMarchPred = {2.2, 1.45, 0.52, 3.2, 4}, kMarchCorr = {1.2, 2.6, 1.2, 5.9, 3};

// ctas CTAs of at most `chunk` planes, `planes` in all
inline double march_time(const MarchCost& m, long long ctas, long long planes, int chunk, int n_sms)
{
    const long long slots = (long long)n_sms * m.k_max;
    const double longest = chunk + m.start;
    if (ctas <= slots) return longest * (m.t0 + m.t1 * (double)((ctas + n_sms - 1) / n_sms));
    return m.t_full * (((double)planes + m.start * (double)ctas) / (double)slots + 0.5 * longest);
}

// the chunk of the least time for a range of `tiles` column tiles and `planes` planes
inline int march_chunk(const MarchCost& m, long long tiles, int planes, int n_sms)
{
    int best = planes;
    double best_t = -1.0;
    for (int n = 1; n == 1 || 2 * n <= planes; ++n) {
        const int c = (planes + n - 1) / n;
        const double t = march_time(m, tiles * ((planes + c - 1) / c), tiles * planes, c, n_sms);
        if (best_t < 0.0 || t < best_t) {
            best_t = t;
            best = c;
        }
    }
    return best;
}

}  // namespace rhd
