/*
 * orbg_tables.cpp -- host-side tables of the query order, and GF(2) helpers.
 *
 * Every order this library decodes in is one of position weights: sorted
 * position j weighs rho_j >= 0 (basic ORBGRAND, Sec. III-B: rho_j = j; one
 * line, Sec. III-D: J_0 + beta j; m segments, Eq. relest_seg), and noise
 * patterns come in increasing weight R = sum of rho over the flipped
 * positions, then Hamming weight w, then positions lexicographically.  The
 * tables (orbg_internal.h) name every pattern of weight w >= 2 as a prefix,
 * its first w - 2 positions, and the pair of its last two, and give each
 * one's index in that order.
 */
#include <algorithm>
#include <cstdint>
#include <cstring>
#include <vector>

#include "orbg_internal.h"

namespace {

/* Patterns counted up to this many are counted exactly. */
constexpr uint64_t kCountMax = 1ull << 40;
/* Weights up to here are counted by one array over the weights. */
constexpr long kDenseMax = 4096;

/* One prefix during the build. */
struct Prefix {
    long R;        /* its weight */
    long m;        /* least weight of a pattern it starts */
    int32_t up;    /* the prefix without its last position, -1 for the empty one */
    int16_t q;     /* its last position, 0 for the empty one */
    uint8_t len;
    uint8_t extra; /* positions outside the sixteen lightest */
};

/* The patterns of an order given by position weights. */
struct Order {
    int n;
    const std::vector<long> &rho;   /* [n + 1], rho[j] of position j = 1..n */
    std::vector<long> x;            /* the weights ascending */
    explicit Order(int n_, const std::vector<long> &rho_) : n(n_), rho(rho_), x(rho_.begin() + 1,
                                                                               rho_.end())
    {
        std::sort(x.begin(), x.end());
    }
    /* patterns of weight <= R with least rank >= k (the empty one left out),
     * at least `most` if there are that many */
    uint64_t count_from(size_t k, long R, uint64_t most) const
    {
        const size_t end = (size_t)(std::upper_bound(x.begin() + (long)k, x.end(), R) - x.begin());
        uint64_t c = end - k;
        for (size_t i = k; i + 1 < end && c < most; i++) {
            if (x[i] + x[i + 1] > R)
                break;
            c += count_from(i + 1, R - x[i], most - c);
        }
        return c;
    }
    /* The least weight up to which there are at least `cap` patterns (the
     * heaviest pattern's if there are fewer in all), and the number of
     * patterns up to it. */
    long depth(uint64_t cap, uint64_t *patterns) const
    {
        long all = 0;
        for (long w : x)
            all += w;
        const long dense = std::min(all, kDenseMax);
        /* few weights first: a cap of 1,000 reaches weight 26 */
        for (long top = std::min(dense, 64l);; top = std::min(dense, 4 * top)) {
            std::vector<uint64_t> c((size_t)top + 1, 0);
            c[0] = 1;
            long reach = 0;
            for (long w : x) {
                reach = std::min(top, reach + w);
                for (long R = reach; R >= w; R--)
                    c[(size_t)R] = std::min(kCountMax, c[(size_t)R] + c[(size_t)(R - w)]);
            }
            uint64_t sum = 0;
            long last = 0;
            for (long R = 0; R <= top; R++) {
                if (!c[(size_t)R])
                    continue;
                sum = std::min(kCountMax, sum + c[(size_t)R]);
                last = R;
                if (sum >= cap || (top == all && R == all)) {
                    *patterns = sum;
                    return last;
                }
            }
            if (top == dense)
                break;
        }
        long lo = dense + 1, hi = all; /* the depth is in [lo, hi] */
        while (lo < hi) {
            const long mid = lo + (hi - lo) / 2;
            if (1 + count_from(0, mid, cap) >= cap)
                hi = mid;
            else
                lo = mid + 1;
        }
        *patterns = 1 + count_from(0, lo, kCountMax);
        return lo;
    }
};

struct TableBuilder {
    int n;
    std::vector<long> rho;          /* [n + 2] */
    long Rmax = 0;
    OrbgTables *out;
    std::vector<long> sufpair;      /* least pair weight over q < a < b */
    std::vector<long> gsum;         /* weight of each pair group */
    std::vector<uint8_t> is_light;  /* [n + 1] one of the sixteen lightest */
    std::vector<Prefix> pre;        /* in lexicographic (depth-first) order */
    bool monotone = true;

    void make_pairs()
    {
        std::vector<std::pair<long, uint32_t>> v;
        std::vector<long> least_from((size_t)n + 2, INT64_MAX / 4); /* over positions >= b */
        for (int b = n; b >= 1; b--)
            least_from[(size_t)b] = std::min(least_from[(size_t)b + 1], rho[(size_t)b]);
        for (int a = 1; a < n; a++)
            for (int b = a + 1; b <= n && rho[(size_t)a] + least_from[(size_t)b] <= Rmax; b++)
                if (rho[(size_t)a] + rho[(size_t)b] <= Rmax)
                    v.push_back({rho[(size_t)a] + rho[(size_t)b],
                                 (uint32_t)(a - 1) << 8 | (uint32_t)(b - 1)});
        std::sort(v.begin(), v.end());
        for (const auto &e : v) {
            if (gsum.empty() || gsum.back() != e.first)
                gsum.push_back(e.first);
            out->pairs.push_back((uint16_t)((e.second >> 8) | (e.second & 0xFFu) << 8));
            out->pgroup.push_back((uint16_t)(gsum.size() - 1));
            const size_t k = out->pgroup.size() - 1;
            const uint32_t first = k && out->pgroup[k] == out->pgroup[k - 1]
                                       ? out->pinfo[k - 1] >> 16
                                       : (uint32_t)k;
            out->pinfo.push_back((uint32_t)out->pgroup[k] | first << 16);
        }
        sufpair.assign((size_t)n + 2, INT64_MAX / 4);
        long least = INT64_MAX / 4; /* lightest single position after a */
        for (int a = n - 1; a >= 0; a--) {
            /* pairs with least position a + 1 */
            if (a + 2 <= n) {
                least = std::min(least, rho[(size_t)a + 2]);
                sufpair[(size_t)a] = std::min(sufpair[(size_t)a + 1], rho[(size_t)a + 1] + least);
            }
        }
    }

    /* every prefix that starts a pattern of weight <= Rmax */
    void make_prefixes()
    {
        struct Step {
            int id, v;
        };
        std::vector<Step> st;
        if (n < 2 || sufpair[0] > Rmax)
            return;
        pre.push_back(Prefix{0, sufpair[0], -1, 0, 0, 0});
        st.push_back(Step{0, 1});
        while (!st.empty()) {
            const int id = st.back().id, v = st.back().v;
            const long R = pre[(size_t)id].R;
            if (v + 2 > n || R + sufpair[(size_t)v] > Rmax ||
                (monotone && R + rho[(size_t)v] + sufpair[(size_t)v] > Rmax)) {
                st.pop_back(); /* no later position leads to a pattern either */
                continue;
            }
            st.back().v++;
            const long m = R + rho[(size_t)v] + sufpair[(size_t)v];
            if (m > Rmax)
                continue;
            Prefix p{R + rho[(size_t)v], m, id, (int16_t)v, (uint8_t)(pre[(size_t)id].len + 1),
                     (uint8_t)(pre[(size_t)id].extra + (is_light[(size_t)v] ? 0 : 1))};
            pre.push_back(p);
            st.push_back(Step{(int)pre.size() - 1, v + 1});
        }
    }

    /* A model's order is limited to patterns of 20 positions, and of 22 where
     * the last two can be written as a + j da, b - j db of one run of
     * patterns with bytes for a and b.  Is any pattern outside that?  (The
     * tables here have no such runs and would hold these patterns; the orders
     * that orbg_load_code_model has always refused stay refused.) */
    bool past_model_limit() const
    {
        for (const Prefix &p : pre) {
            if (p.len < ORBG_MAX_FLIPS - 3)
                continue;
            for (size_t k = 0; k < out->pairs.size();) {
                size_t e = k;
                std::vector<std::pair<int, int>> run;
                for (; e < out->pairs.size() && out->pgroup[e] == out->pgroup[k]; e++) {
                    const int a = (out->pairs[e] & 0xFF) + 1, b = (out->pairs[e] >> 8) + 1;
                    if (a > p.q)
                        run.push_back({a, b});
                }
                if (p.R + gsum[out->pgroup[k]] > Rmax)
                    break;
                for (size_t s = 0; s < run.size();) {
                    int da = 1, db = 1;
                    if (s + 1 < run.size()) {
                        da = run[s + 1].first - run[s].first;
                        db = run[s].second - run[s + 1].second;
                    }
                    if (da < 1 || db < 1)
                        da = db = 1;
                    size_t f = s + 1;
                    while (f < run.size() &&
                           run[f].first == run[s].first + da * (int)(f - s) &&
                           run[f].second == run[s].second - db * (int)(f - s))
                        f++;
                    const bool pairs = da == 1 && db == 1 &&
                                       run[s].first + run[s].second <= 255;
                    if (!pairs && (f - s < 2 || run[s].second > 255))
                        return true;
                    s = f;
                }
                k = e;
            }
        }
        return false;
    }

    /* positions of prefix id, ascending */
    int positions(int id, int *v) const
    {
        const int w = pre[(size_t)id].len;
        for (int i = w - 1; i >= 0; i--) {
            v[i] = pre[(size_t)id].q;
            id = pre[(size_t)id].up;
        }
        return w;
    }

    /* first query index of the patterns of weight R and more */
    std::vector<std::pair<long, uint32_t>> first_of; /* (weight, first index), ascending */
    uint32_t first_at(long R) const
    {
        const auto it = std::lower_bound(first_of.begin(), first_of.end(),
                                         std::make_pair(R, (uint32_t)0));
        return it == first_of.end() ? (uint32_t)out->patterns + 1u : it->second;
    }

    int build(bool model)
    {
        const int light_n = std::min(n, 16);
        std::vector<std::pair<long, int>> by;
        for (int j = 1; j <= n; j++) {
            by.push_back({rho[(size_t)j], j});
            monotone &= j == 1 || rho[(size_t)j] >= rho[(size_t)j - 1];
        }
        std::sort(by.begin(), by.end());
        is_light.assign((size_t)n + 1, 0);
        std::vector<int> bit((size_t)n + 1, 0);
        std::memset(out->light, 0, sizeof(out->light));
        for (int i = 0; i < light_n; i++) {
            const int j = by[(size_t)i].second;
            out->light[i] = (uint8_t)j; /* at most position 256 of n = 256, cut below */
            is_light[(size_t)j] = 1;
            bit[(size_t)j] = i;
            if (j > 255)
                is_light[(size_t)j] = 0, out->light[i] = 0; /* no prefix holds position 256 */
        }
        make_pairs();
        make_prefixes();
        if (model && past_model_limit())
            return -2;
        const uint32_t npre = (uint32_t)pre.size();
        /* the prefixes by the least weight they start; equal ones by the
         * loads they cost */
        std::vector<uint32_t> ord(npre);
        for (uint32_t i = 0; i < npre; i++)
            ord[i] = i;
        std::stable_sort(ord.begin(), ord.end(), [&](uint32_t a, uint32_t b) {
            return pre[a].m != pre[b].m ? pre[a].m < pre[b].m : pre[a].extra < pre[b].extra;
        });
        /* per last position q: the first group with a pair after q, and how
         * many pairs after q each group from there on holds */
        const uint32_t ngrp = (uint32_t)gsum.size();
        std::vector<std::vector<uint16_t>> after((size_t)n + 1);
        std::vector<uint32_t> g0((size_t)n + 1, 0);
        std::vector<uint32_t> place(npre); /* of lexicographic prefix i in the final order */
        out->pmeta.resize(2 * ((size_t)npre + 1));
        uint64_t rows = 0;
        for (uint32_t i = 0; i < npre; i++) {
            const Prefix &p = pre[ord[i]];
            place[ord[i]] = i;
            const size_t q = (size_t)p.q;
            if (after[q].empty()) {
                std::vector<uint16_t> c(ngrp, 0);
                for (size_t k = 0; k < out->pairs.size(); k++)
                    c[out->pgroup[k]] += (size_t)(out->pairs[k] & 0xFFu) + 1 > q;
                uint32_t g = 0;
                while (c[g] == 0)
                    g++;
                g0[q] = g;
                after[q].assign(c.begin() + g, c.end());
            }
            out->pmeta[2 * i] = (uint32_t)rows;
            out->pmeta[2 * i + 1] = (uint32_t)p.q | g0[q] << 16;
            const uint32_t g1 = (uint32_t)(std::upper_bound(gsum.begin(), gsum.end(), Rmax - p.R) -
                                           gsum.begin());
            rows += g1 - g0[q];
        }
        out->pmeta[2 * (size_t)npre] = (uint32_t)rows;
        out->pmeta[2 * (size_t)npre + 1] = 0;
        out->start.assign((size_t)rows, 0u);
        out->single.assign((size_t)n, 0u);
        /* the runs (prefix, group) and the single positions, ordered by
         * (weight, w); generated in lexicographic order, which a stable sort
         * keeps inside one (weight, w) */
        struct Run {
            uint32_t at;    /* entry of start[], or of single[] */
            uint16_t count; /* patterns; 0 marks a single position */
        };
        std::vector<Run> runs;
        std::vector<uint64_t> key;
        for (int j = 1; j <= n; j++)
            if (rho[(size_t)j] <= Rmax) {
                runs.push_back(Run{(uint32_t)j - 1u, 0});
                key.push_back((uint64_t)rho[(size_t)j] << 5 | 1u);
            }
        for (uint32_t l = 0; l < npre; l++) {
            const uint32_t i = place[l];
            const uint32_t lo = out->pmeta[2 * i], hi = out->pmeta[2 * i + 2];
            const size_t q = (size_t)pre[l].q;
            for (uint32_t k = lo; k < hi; k++) {
                const uint16_t c = after[q][k - lo];
                if (!c)
                    continue;
                runs.push_back(Run{k, c});
                key.push_back((uint64_t)(pre[l].R + gsum[g0[q] + (k - lo)]) << 5 |
                              (uint64_t)(pre[l].len + 2));
            }
        }
        std::vector<uint32_t> ro(runs.size());
        if (Rmax <= kDenseMax) {
            std::vector<uint32_t> c((size_t)(Rmax + 1) * 32 + 1, 0);
            for (uint64_t k : key)
                c[(size_t)k + 1]++;
            for (size_t k = 1; k < c.size(); k++)
                c[k] += c[k - 1];
            for (size_t r = 0; r < runs.size(); r++)
                ro[c[(size_t)key[r]]++] = (uint32_t)r;
        } else {
            for (size_t r = 0; r < runs.size(); r++)
                ro[r] = (uint32_t)r;
            std::stable_sort(ro.begin(), ro.end(),
                             [&](uint32_t a, uint32_t b) { return key[a] < key[b]; });
        }
        uint32_t t = 2; /* the zero pattern is query 1 */
        first_of.push_back({0, 1u});
        for (uint32_t r : ro) {
            const long R = (long)(key[r] >> 5);
            if (R != first_of.back().first)
                first_of.push_back({R, t});
            if (runs[r].count) {
                out->start[runs[r].at] = t;
                t += runs[r].count;
            } else {
                out->single[runs[r].at] = t++;
            }
        }
        /* the records the kernels read, 32 prefixes to a group */
        /* an even number of groups: a CTA's warps take two at a time */
        const uint32_t ng = (npre + 2 * ORBG_GROUP - 1) / (2 * ORBG_GROUP) * 2;
        out->npre = npre;
        for (uint32_t g = 0; g < ng; g++)
            out->gmeta.push_back(0xFFFFFFFFu), out->gmeta.push_back(0u);
        out->pre.assign((size_t)ng * ORBG_GROUP, 0);
        out->pre1.assign((size_t)ng * ORBG_GROUP, 0);
        uint32_t npre1 = npre; /* leading prefixes a phase-1 warp walks */
        int v[64];
        for (uint32_t i = 0; i < npre; i++) {
            const Prefix &p = pre[ord[i]];
            positions((int)ord[i], v);
            uint64_t rec = 0, rec1 = 0, ext = 0;
            int x = 0;
            for (int k = 0; k < p.len; k++) {
                if (is_light[(size_t)v[k]]) {
                    rec |= 1ull << bit[(size_t)v[k]];
                } else {
                    if (x < ORBG_PRE_POS)
                        rec |= (uint64_t)v[k] << (16 + 8 * x);
                    else
                        ext |= (uint64_t)v[k] << (8 * (x - ORBG_PRE_POS));
                    x++;
                }
                if (k < 8)
                    rec1 |= (uint64_t)v[k] << (8 * k);
            }
            if (p.len > 8 && npre1 == npre)
                npre1 = i;
            out->pre[i] = rec;
            out->pre1[i] = rec1;
            if (x > ORBG_PRE_POS) {
                out->pext.resize((size_t)ng * ORBG_GROUP, 0);
                out->pext[i] = ext;
            }
            uint32_t &gm = out->gmeta[2 * (size_t)(i / ORBG_GROUP) + 1];
            gm = std::max(gm & 0xFFu, (uint32_t)x) |
                 std::max(gm >> 8, (uint32_t)std::min<int>(p.len, 8)) << 8;
            if (i % ORBG_GROUP == 0)
                out->gmeta[2 * (size_t)(i / ORBG_GROUP)] = first_at(p.m);
        }
        npre1 = std::min<uint32_t>(npre1, ORBG_PRE1_MAX);
        const long past = Rmax + 1;
        const uint32_t npairs = (uint32_t)out->pairs.size();
        /* the first weight of a prefix that holds a position, and the pairs
         * below it */
        const long first = npre > 1 ? pre[ord[1]].m : past;
        uint32_t alone = 0;
        while (alone < npairs && gsum[out->pgroup[alone]] < first)
            alone++;
        if (alone >= ORBG_BAND2_PAIRS && npre <= ORBG_SCAN_PREFIXES && npre <= npairs / 2) {
            out->scan = 1;
            out->cut_pairs[0] = alone;
            out->cut_end[0] = first_at(first);
            /* then the pairs that prefixes of positions take, or all, if the
             * first ones are not */
            uint32_t most = 0, np = npairs;
            for (uint32_t i = 1; i < npre; i++)
                most = std::max(most, g0[(size_t)pre[ord[i]].q] + out->pmeta[2 * i + 2] -
                                          out->pmeta[2 * i]);
            while (alone == npairs && np > 0 && out->pgroup[np - 1] >= most)
                np--;
            out->cut_pairs[1] = np;
        }
        /* phase 1's bands: the pairs of the leading groups; the first weight
         * not covered by them and the leading prefixes; how many prefixes
         * and positions the patterns below it take */
        const uint32_t aim[ORBG_BANDS] = {ORBG_BAND1_PAIRS, ORBG_BAND2_PAIRS};
        const long lim1 = npre1 < npre ? pre[ord[npre1]].m : past;
        for (int k = 0; k < ORBG_BANDS; k++) {
            uint32_t np = std::min(aim[k], npairs);
            while (np > 0 && np < out->pairs.size() && out->pgroup[np] == out->pgroup[np - 1])
                np--;
            const long end =
                std::min(lim1, np < out->pairs.size() ? gsum[out->pgroup[np]] : past);
            out->band_pairs[k] = np;
            out->band_end[k] = first_at(end);
            uint32_t c = 0;
            while (c < npre1 && pre[ord[c]].m < end)
                c++;
            out->band_pre[k] = c;
            uint32_t top = 0;
            for (int j = 1; j <= n; j++)
                if (rho[(size_t)j] < end)
                    top = (uint32_t)j;
            for (uint32_t i = 0; i < np; i++)
                top = std::max(top, (uint32_t)(out->pairs[i] >> 8) + 1u);
            out->band_ranks[k] = top;
        }
        for (int j = 1; j <= n; j++)
            if (rho[(size_t)j] <= Rmax)
                out->ranks = (uint32_t)j;
        /* phase 2's cuts, likewise, where one CTA's set does not hold all
         * pairs */
        out->chunk = out->scan ? npre : (uint32_t)out->pairs.size();
        if (!out->scan && out->chunk > ORBG_PAIR_CHUNK) {
            out->chunk = ORBG_SPLIT_CHUNK;
            const uint32_t to[ORBG_CUTS] = {ORBG_LEAD_PAIRS, ORBG_SPLIT_CHUNK};
            for (int k = 0; k < ORBG_CUTS; k++) {
                uint32_t np = to[k];
                while (np > 0 && out->pgroup[np] == out->pgroup[np - 1])
                    np--;
                out->cut_pairs[k] = np;
                out->cut_end[k] = first_at(gsum[out->pgroup[np]]);
            }
        }
        make_flat();
        return 0;
    }

    /* Flat table: the leading patterns of weight <= ORBG_FLAT_POS, at most
     * ORBG_FLAT_MAX of them, in query order. */
    void make_flat()
    {
        const uint32_t most = (uint32_t)std::min<uint64_t>(out->patterns, ORBG_FLAT_MAX);
        std::vector<std::vector<int>> first((size_t)most);
        orbg_expand_tables(*out, n, most, [&](uint32_t t, const int *v, int w) {
            first[t - 1].assign(v, v + w);
        });
        uint32_t nflat = 0;
        while (nflat < first.size() && first[nflat].size() <= ORBG_FLAT_POS)
            nflat++;
        /* per step of 32 patterns: the ranks it needs in sorted order (its
         * largest position, non-decreasing over the steps; the table ends
         * before the first step needing more than ORBG_FLAT_RANKS) and its
         * largest Hamming weight */
        std::vector<uint8_t> need;
        int mx = 0;
        uint32_t keep = 0;
        for (uint32_t base = 0; base < nflat; base += 32) {
            const uint32_t end = std::min<uint32_t>(nflat, base + 32);
            int wmax = 0;
            for (uint32_t t = base; t < end; t++) {
                wmax = std::max(wmax, (int)first[t].size());
                for (int p : first[t])
                    mx = std::max(mx, p);
            }
            if (mx > ORBG_FLAT_RANKS)
                break;
            need.push_back((uint8_t)(mx | wmax << 5));
            keep = end;
        }
        nflat = keep;
        out->nflat = nflat;
        out->flat.assign((size_t)std::max<uint32_t>(nflat, 1) * 8, 0);
        for (uint32_t t = 0; t < nflat; t++) {
            uint8_t *e = &out->flat[(size_t)t * 8];
            for (size_t i = 0; i < first[t].size(); i++)
                e[i] = (uint8_t)first[t][i];
            e[7] = need[t / 32];
        }
    }
};

/* Some pattern of weight <= Rmax flips more than ORBG_MAX_FLIPS positions. */
bool too_heavy(const Order &o, long Rmax)
{
    long s = 0;
    for (int i = 0; i < o.n && i <= ORBG_MAX_FLIPS; i++)
        s += o.x[(size_t)i];
    return o.n > ORBG_MAX_FLIPS && s <= Rmax;
}

int build_order(int n, const std::vector<long> &rho, uint64_t patterns, long Rmax, bool model,
                OrbgTables *out)
{
    if (patterns >= 0xFFFFFFFFull)
        return -3;
    *out = OrbgTables();
    out->patterns = patterns;
    TableBuilder b;
    b.n = n;
    b.rho = rho;
    b.rho.push_back(0);
    b.Rmax = Rmax;
    b.out = out;
    return b.build(model);
}

}  // namespace

int orbg_build_tables(int n, uint64_t cap, OrbgTables *out, long J0, long beta)
{
    if (n < 1 || n > 256 || cap < 1 || J0 < 0 || beta < 1 || J0 > ORBG_MAX_LINE ||
        beta > ORBG_MAX_LINE)
        return -1;
    std::vector<long> rho((size_t)n + 1, 0);
    for (int j = 1; j <= n; j++)
        rho[(size_t)j] = J0 + beta * j;
    const Order o(n, rho);
    uint64_t patterns = 0;
    const long Rmax = o.depth(cap, &patterns);
    if (too_heavy(o, Rmax))
        return -2;
    /* lines stop at logistic weight ORBG_MAX_LOGISTIC */
    for (long w = 1; w <= n; w++) {
        const long W = std::max<long>(ORBG_MAX_LOGISTIC + 1, w * (w + 1) / 2);
        if (W <= w * (w + 1) / 2 + w * (n - w) && J0 * w + beta * W <= Rmax)
            return -2;
    }
    return build_order(n, rho, patterns, Rmax, false, out);
}

int orbg_build_tables_model(int n, uint64_t cap, const OrbgModel &md, OrbgTables *out)
{
    if (n < 1 || n > 256 || cap < 1 || md.m < 1 || md.m > ORBG_MAX_SEG || md.I[0] != 0 ||
        md.I[md.m] != n)
        return -1;
    for (int i = 0; i < md.m; i++)
        if (md.I[i + 1] <= md.I[i] || md.beta[i] < 1 || md.beta[i] > ORBG_MAX_MODEL ||
            md.J[i] < -md.beta[i] || md.J[i] > ORBG_MAX_MODEL)
            return -1;
    std::vector<long> rho((size_t)n + 1, 0);
    for (int i = 0; i < md.m; i++)
        for (int j = md.I[i] + 1; j <= md.I[i + 1]; j++)
            rho[(size_t)j] = md.J[i] + md.beta[i] * (long)(j - md.I[i]);
    const Order o(n, rho);
    uint64_t patterns = 0;
    const long Rmax = o.depth(cap, &patterns);
    /* position 256 does not fit a byte of a model's order */
    if (too_heavy(o, Rmax) || (n == 256 && rho[256] <= Rmax))
        return -2;
    return build_order(n, rho, patterns, Rmax, true, out);
}

void orbg_few_rows(OrbgTables *tb, int n, int r)
{
    /* phase 2: fewer pairs at a time, two cuts as for an order of many */
    if (r <= ORBG_FEW_ROWS && !tb->scan && tb->chunk > ORBG_FEW_CHUNK) {
        tb->chunk = ORBG_FEW_CHUNK;
        const uint32_t to[ORBG_CUTS] = {ORBG_BAND2_PAIRS, ORBG_FEW_CHUNK};
        for (int k = 0; k < ORBG_CUTS; k++) {
            uint32_t np = to[k];
            while (np > 0 && tb->pgroup[np] == tb->pgroup[np - 1])
                np--;
            tb->cut_pairs[k] = np;
            /* the empty prefix's first index of the group: the first pattern
             * that takes one of its pairs */
            tb->cut_end[k] = tb->start[tb->pgroup[np]];
        }
    }
    const uint32_t end = tb->band_end[0];
    if (r > ORBG_LONG_FLAT_ROWS || end <= tb->nflat + 1)
        return;
    std::vector<uint8_t> more((size_t)(end - 1 - tb->nflat) * 8, 0);
    bool fits = true;
    orbg_expand_tables(*tb, n, end - 1, [&](uint32_t t, const int *v, int w) {
        fits &= w <= ORBG_FLAT_POS && (w == 0 || v[w - 1] <= 255);
        if (t > tb->nflat && fits)
            for (int i = 0; i < w; i++)
                more[(size_t)(t - 1 - tb->nflat) * 8 + i] = (uint8_t)v[i];
    });
    if (!fits)
        return;
    tb->flat.resize((size_t)tb->nflat * 8);
    tb->flat.insert(tb->flat.end(), more.begin(), more.end());
    tb->long_end = end;
}

/* Calls f(t, positions, w) for every pattern of index t <= count: positions
 * 1-based, ascending.  Expanded from the tables the kernels read. */
void orbg_expand_tables(const OrbgTables &tb, int n, uint64_t count,
                        const std::function<void(uint32_t, const int *, int)> &f)
{
    int v[64];
    if (count >= 1)
        f(1u, v, 0);
    for (int j = 1; j <= n; j++)
        if (tb.single[(size_t)j - 1] && tb.single[(size_t)j - 1] <= count) {
            v[0] = j;
            f(tb.single[(size_t)j - 1], v, 1);
        }
    /* first pair of each group */
    std::vector<uint32_t> gfirst;
    for (size_t k = 0; k < tb.pairs.size(); k++)
        if (k == 0 || tb.pgroup[k] != tb.pgroup[k - 1])
            gfirst.push_back((uint32_t)k);
    gfirst.push_back((uint32_t)tb.pairs.size());
    for (uint32_t i = 0; i < tb.npre; i++) {
        if (tb.gmeta[2 * (size_t)(i / ORBG_GROUP)] > count)
            break;
        int w = 0;
        const uint64_t rec = tb.pre[i], ext = i < tb.pext.size() ? tb.pext[i] : 0;
        for (int b = 0; b < 16; b++)
            if (rec >> b & 1)
                v[w++] = tb.light[b];
        for (int k = 0; k < ORBG_PRE_POS; k++)
            if (rec >> (16 + 8 * k) & 0xFF)
                v[w++] = (int)(rec >> (16 + 8 * k) & 0xFF);
        for (int k = 0; k < 8; k++)
            if (ext >> (8 * k) & 0xFF)
                v[w++] = (int)(ext >> (8 * k) & 0xFF);
        std::sort(v, v + w);
        const int q = (int)(tb.pmeta[2 * (size_t)i + 1] & 0xFFFFu);
        const uint32_t g0 = tb.pmeta[2 * (size_t)i + 1] >> 16;
        for (uint32_t k = tb.pmeta[2 * (size_t)i]; k < tb.pmeta[2 * (size_t)i + 2]; k++) {
            const uint32_t g = g0 + (k - tb.pmeta[2 * (size_t)i]);
            uint32_t t = tb.start[k];
            if (t == 0)
                continue;
            for (uint32_t e = gfirst[g]; e < gfirst[g + 1]; e++) {
                if ((tb.pairs[e] & 0xFF) + 1 <= q)
                    continue;
                if (t <= count) {
                    v[w] = (tb.pairs[e] & 0xFF) + 1;
                    v[w + 1] = (tb.pairs[e] >> 8) + 1;
                    f(t, v, w + 2);
                }
                t++;
            }
        }
    }
}

/* ------------------------------------------------------------- GF(2) -- */

namespace {

struct BitMat {
    int rows, cols, words;
    std::vector<uint64_t> a;
    BitMat(const uint8_t *M, int r, int c) : rows(r), cols(c), words((c + 63) / 64),
                                             a((size_t)r * ((c + 63) / 64), 0) {
        for (int i = 0; i < r; i++)
            for (int j = 0; j < c; j++)
                if (M[(size_t)i * c + j])
                    a[(size_t)i * words + j / 64] |= 1ull << (j % 64);
    }
    bool get(int i, int j) const { return (a[(size_t)i * words + j / 64] >> (j % 64)) & 1; }
    void swap_rows(int i, int k) {
        for (int w = 0; w < words; w++)
            std::swap(a[(size_t)i * words + w], a[(size_t)k * words + w]);
    }
    void add_row(int dst, int src) {
        for (int w = 0; w < words; w++)
            a[(size_t)dst * words + w] ^= a[(size_t)src * words + w];
    }
    /* reduced row echelon form; returns pivot columns */
    std::vector<int> rref() {
        std::vector<int> piv;
        int r = 0;
        for (int c = 0; c < cols && r < rows; c++) {
            int p = -1;
            for (int i = r; i < rows; i++)
                if (get(i, c)) { p = i; break; }
            if (p < 0)
                continue;
            swap_rows(r, p);
            for (int i = 0; i < rows; i++)
                if (i != r && get(i, c))
                    add_row(i, r);
            piv.push_back(c);
            r++;
        }
        return piv;
    }
};

}  // namespace

int orbg_gf2_rank(const uint8_t *M, int rows, int cols)
{
    BitMat m(M, rows, cols);
    return (int)m.rref().size();
}

int orbg_gf2_nullspace(const uint8_t *M, int rows, int cols,
                       std::vector<uint8_t> *basis, int *dim)
{
    BitMat m(M, rows, cols);
    std::vector<int> piv = m.rref();
    std::vector<char> is_piv(cols, 0);
    for (int c : piv)
        is_piv[c] = 1;
    basis->clear();
    int d = 0;
    for (int f = 0; f < cols; f++) {
        if (is_piv[f])
            continue;
        std::vector<uint8_t> x(cols, 0);
        x[f] = 1;
        for (size_t i = 0; i < piv.size(); i++)
            x[piv[i]] = m.get((int)i, f) ? 1 : 0;
        basis->insert(basis->end(), x.begin(), x.end());
        d++;
    }
    *dim = d;
    return 0;
}
