/* Host check of what phase 2 leaves out at each stage of an order
 * (test_tables_host.py): the pairs a cut or a scan covers against every
 * pattern of the order, and the flat table past its first part. */
#include <algorithm>
#include <cstdint>
#include <map>
#include <vector>

#include "orbg_internal.h"

namespace {

int check(const OrbgTables &tb, int n)
{
    std::map<std::pair<int, int>, uint32_t> id;
    for (size_t k = 0; k < tb.pairs.size(); k++)
        id[{(tb.pairs[k] & 0xFF) + 1, (tb.pairs[k] >> 8) + 1}] = (uint32_t)k;
    const uint32_t npairs = (uint32_t)tb.pairs.size();
    const bool cuts = tb.scan || tb.chunk < npairs;
    if (tb.scan && (tb.chunk != tb.npre || tb.npre > ORBG_SCAN_PREFIXES ||
                    tb.cut_pairs[0] > npairs || tb.cut_pairs[1] > npairs))
        return 1;
    if (!tb.scan && (tb.chunk > ORBG_PAIR_CHUNK ||
                     (cuts && (tb.cut_pairs[0] > tb.chunk || tb.cut_pairs[1] > tb.chunk))))
        return 2;
    int bad = 0;
    orbg_expand_tables(tb, n, tb.patterns, [&](uint32_t t, const int *v, int w) {
        if (t > tb.nflat && t < tb.long_end) {
            const uint8_t *e = &tb.flat[(size_t)(t - 1) * 8];
            for (int i = 0; i < 8; i++)
                if (e[i] != (i < w ? v[i] : 0))
                    bad = 3;
        }
        if (w < 2 || !cuts)
            return;
        const uint32_t p = id[{v[w - 2], v[w - 1]}];
        if (tb.scan) {
            /* the first part: pairs alone, and all of them */
            if (t < tb.cut_end[0] && (w > 2 || p >= tb.cut_pairs[0]))
                bad = 4;
            /* the second: every other pattern's pair */
            if (p >= tb.cut_pairs[1] && (w > 2 || p >= tb.cut_pairs[0]))
                bad = 5;
            /* the empty prefix bounds a pair's hits from below */
            if (t < tb.start[tb.pgroup[p]])
                bad = 6;
        } else {
            for (int k = 0; k < ORBG_CUTS; k++)
                if (t < tb.cut_end[k] && p >= tb.cut_pairs[k])
                    bad = 7;
        }
    });
    return bad;
}

}  // namespace

/* J0, beta of m segments; r parity bits.  Returns 0, -1 for a refused order,
 * or the check that failed; what: 1 scan, 2 cuts, 4 a longer flat table. */
extern "C" int tables_check(int n, uint64_t cap, int m, const int *I, const int64_t *J,
                            const int64_t *beta, int r, int *what)
{
    OrbgModel md{};
    md.m = m;
    for (int i = 0; i <= m; i++)
        md.I[i] = I[i];
    for (int i = 0; i < m; i++) {
        md.J[i] = (long)J[i];
        md.beta[i] = (long)beta[i];
    }
    OrbgTables tb;
    if (orbg_build_tables_model(n, cap, md, &tb) != 0)
        return -1;
    orbg_few_rows(&tb, n, r);
    *what = (tb.scan ? 1 : tb.chunk < tb.pairs.size() ? 2 : 0) | (tb.long_end ? 4 : 0);
    return check(tb, n);
}
