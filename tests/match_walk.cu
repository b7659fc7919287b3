// Walks the shares of every block pair of a matching launch on the host.
// usage: match_walk SMS COUNT NQ NT [NQ NT ...]   (the sets are repeated up to COUNT problems)
// prints: whole_tiles pairs most_units fewest_units units_walked units_distinct units
#include <cstdio>
#include <cstdlib>
#include <set>
#include <vector>

#include "match_common.cuh"

using namespace latch;

int main(int argc, char** argv) {
    if (argc < 5) return 2;
    const int sms = atoi(argv[1]), count = atoi(argv[2]), sets = (argc - 3) / 2;
    MatchBatch* b = new MatchBatch();
    int32_t out0 = 0;
    for (int i = 0; i < count; ++i) {
        MatchProblem& P = b->p[i];
        P.nq = atoi(argv[3 + 2 * (i % sets)]);
        P.nt = atoi(argv[4 + 2 * (i % sets)]);
        P.out0 = out0;
        out0 += P.nq;
    }
    plan_match_batch(b, count, sms);
    std::set<std::vector<int64_t>> seen;
    int64_t most = 0, fewest = INT64_MAX, walked = 0;
    for (int64_t c = 0; c < b->grid; ++c) {
        int64_t mine = 0;
        for (Share s = first_share(*b, c); s.p < b->count;) {
            int32_t m = s.m, n = s.n;
            for (int64_t k = 0; k < s.left; ++k) {
                if (n == b->p[s.p].ntl) {
                    n = 0;
                    ++m;
                }
                seen.insert({s.p, m, n++});
            }
            mine += s.left;
            s = share_after(*b, s.p, m, c);
        }
        most = mine > most ? mine : most;
        fewest = mine < fewest ? mine : fewest;
        walked += mine;
    }
    printf("%d %lld %lld %lld %lld %lld %lld\n", b->whole_tiles, static_cast<long long>(b->grid),
           static_cast<long long>(most), static_cast<long long>(fewest), static_cast<long long>(walked),
           static_cast<long long>(seen.size()), static_cast<long long>(b->units));
    return 0;
}
