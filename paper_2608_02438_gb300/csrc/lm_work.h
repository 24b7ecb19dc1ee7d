// lm_work.h -- which CTA of the LM head takes which (token chunk, vocabulary
// item): plain index arithmetic, for the kernels and for the host.
#ifndef XPRESS_LM_WORK_H
#define XPRESS_LM_WORK_H

#ifdef __CUDACC__
#define XP_HOST_DEVICE __host__ __device__ __forceinline__
#else
#define XP_HOST_DEVICE inline
#endif

namespace xp {

// G CTAs over NC token chunks, in groups of at most LM_GROUP chunks one after
// another.  In a group of n chunks CTA r takes its chunk r % n and every step-th
// vocabulary item of it, so that the CTAs that read the same rows of W_lm run side
// by side (one read from HBM per group), and each chunk has G / n CTAs, give or take
// one.  The CTAs of a chunk that has one fewer set the time, so a group is kept small
// enough for 152 CTAs (at most 9 % lost, with 14 chunks) and no smaller: each group
// reads W_lm again.  Measured with the Qwen3-8B head, groups of 16 / 8 / 19 / all
// chunks in one / one chunk at a time, ms: 2050 tokens 1.63 / 1.70 / 1.63 / 1.62 / -,
// 4352 3.50 / 3.63 / 3.74 / 3.75 / -, 9984 8.1 / 8.0 / 8.1 / 9.5 / 9.9, 19712 16.3 /
// 15.9 / 16.3 / 28.3 / 19.7, 39168 33.8 / 32.9 / 34.7 / 60 / 40.5.
constexpr int LM_GROUP = 16;

struct LmWork {
    int r, G, NC, groups;
    XP_HOST_DEVICE LmWork(int r_, int G_, int NC_) : r(r_), G(G_), NC(NC_)
    {
        const int most = G < LM_GROUP ? G : LM_GROUP;
        groups = (NC + most - 1) / most;                         // of sizes that differ by one at most
    }
    XP_HOST_DEVICE int begin(int g) const { return (int)((long long)NC * g / groups); }
    XP_HOST_DEVICE int count(int g) const { return begin(g + 1) - begin(g); }
    // of group g: the CTA's chunk, its first item (and the slot of its partials) and the step between its items
    XP_HOST_DEVICE int chunk(int g) const { return begin(g) + r % count(g); }
    XP_HOST_DEVICE int first(int g) const { return r / count(g); }
    XP_HOST_DEVICE int step(int g) const { return (G - 1 - r % count(g)) / count(g) + 1; }
    // CTAs that work on chunk c: their partials are a token's first so many
    XP_HOST_DEVICE int slots(int c) const
    {
        const int g = (int)(((long long)(c + 1) * groups - 1) / NC);
        return (G - 1 - (c - begin(g))) / count(g) + 1;
    }
};

}  // namespace xp

#endif
