// The order of the mixed factorisation's launches on its two streams, tile by tile, from the
// library's own rule of which launch writes which tile (csrc/mixed_order.cuh).
//
// Every launch of factor_mixed gets a vector clock (its place on the main and on the side
// stream, joined by the events it waits for).  For each tile, any two launches that write it,
// or of which one writes and the other reads it, have to be ordered by these clocks, and each
// update (m, n, k) has to be applied once, after the panel of step k and before tile (m, n)
// is factored or solved.  Prints the number of unordered pairs, of updates applied late or not
// once, and of the accesses looked at.
#include <cstdio>
#include <cstdlib>
#include <map>
#include <set>
#include <utility>
#include <vector>

#include "mixed_order.cuh"

using namespace egs;

struct Clock {
    int v[2] = {0, 0};
    void join(const Clock &o)
    {
        for (int i = 0; i < 2; ++i) v[i] = o.v[i] > v[i] ? o.v[i] : v[i];
    }
};
struct Access {
    int stream;
    Clock c;
    bool write;
    int step, kind;  // kind 0: factored / solved (final), 1: update, 2: read as an operand
};

struct Model {
    Clock now[2];
    std::map<std::pair<int, int>, std::vector<Access>> acc;
    int stream = 0;
    void launch(int s)
    {
        stream = s;
        ++now[s].v[s];
    }
    void touch(int m, int n, bool write, int step, int kind) { acc[{m, n}].push_back({stream, now[stream], write, step, kind}); }
    Clock record(int s) const { return now[s]; }
    void wait(int s, const Clock &e) { now[s].join(e); }
};

static bool before(const Access &a, const Access &b) { return b.c.v[a.stream] >= a.c.v[a.stream]; }

// fp32: the FP32 mode (band outputs by slice products, the off-band solve behind ev_diag)
static void run(int T, int band, int xband, bool fp32, long &races, long &wrong, long &seen)
{
    enum { MAIN = 0, SIDE = 1 };
    Model M;
    Clock ev_col = M.record(MAIN);
    auto band_launch = [&](int part, int k) {
        std::set<std::pair<int, int>> rd;
        for (int64_t t = 0; t < order::band_tiles_of(part, k, band, xband, T); ++t) {
            int m, n;
            if (!order::band_tile(part, k, band, xband, T, t, m, n) || n > m) continue;
            M.touch(m, n, true, k, 1);
            rd.insert({m, k});
            rd.insert({n, k});
        }
        for (auto &r : rd) M.touch(r.first, r.second, false, k, 2);
    };
    auto update_launch = [&](int part, int k) {
        const int skip = fp32 ? 1 : 0;
        std::vector<std::pair<int, int>> tiles;
        if (part == order::kColumn) {
            for (int64_t t = 0; t < order::update_tiles_of(part, k, band, skip, T); ++t) {
                int m = k + 1 + (int)t, n = k + 1;
                if (m >= T) order::update_corner(k, band, T, t, m, n);
                tiles.push_back({m, n});
            }
        } else {
            for (int n = k + 2; n < T; ++n)
                for (int m = n; m < T; ++m) tiles.push_back({m, n});
            wrong += (long)tiles.size() != order::update_tiles_of(part, k, band, skip, T);
        }
        for (auto &t : tiles)
            if (order::update_tile(part, k, band, t.first, t.second, skip, xband)) M.touch(t.first, t.second, true, k, 1);
    };
    for (int k = 0; k < T; ++k) {
        const int nb = band - 1 < T - k - 1 ? band - 1 : T - k - 1;
        if (k == 0 || order::potrf_waits_for_column(band)) M.wait(SIDE, ev_col);
        M.launch(SIDE);  // POTRF
        M.touch(k, k, true, k, 0);
        const Clock ev_diag = M.record(SIDE);
        if (k > 0) M.wait(SIDE, ev_col);
        M.launch(SIDE);  // the band rows' solve and operands
        for (int m = k + 1; m <= k + nb; ++m) M.touch(m, k, true, k, 0);
        const Clock ev_panel = M.record(SIDE);
        if (k + 1 < T) {
            M.launch(SIDE);  // band x band
            band_launch(order::kBandBand, k);
        }
        if (k + 1 == T) break;
        M.wait(MAIN, fp32 ? ev_diag : ev_panel);
        M.launch(MAIN);  // off-band solve
        for (int m = k + 1 + nb; m < T; ++m) M.touch(m, k, true, k, 0);
        M.wait(MAIN, ev_panel);
        M.launch(MAIN);
        if (fp32) band_launch(order::kColumn, k);
        M.launch(MAIN);
        update_launch(order::kColumn, k);
        ev_col = M.record(MAIN);
        M.launch(MAIN);
        if (fp32) band_launch(order::kRest, k);
        M.launch(MAIN);
        update_launch(order::kRest, k);
    }
    for (auto &kv : M.acc) {
        const auto &v = kv.second;
        seen += (long)v.size();
        std::vector<int> applied(T, 0);
        const Access *fin = nullptr;
        for (auto &a : v)
            if (a.kind == 0) fin = &a;
        for (size_t i = 0; i < v.size(); ++i) {
            if (v[i].kind == 1) {
                ++applied[v[i].step];
                if (!fin || !before(v[i], *fin)) ++wrong;
            }
            for (size_t j = i + 1; j < v.size(); ++j)
                if ((v[i].write || v[j].write) && v[i].stream != v[j].stream && !before(v[i], v[j]) && !before(v[j], v[i]))
                    ++races;
        }
        for (int k = 0; k < kv.first.second; ++k) wrong += applied[k] != 1;
        for (int k = kv.first.second; k < T; ++k) wrong += applied[k] != 0;
    }
}

int main()
{
    long races = 0, wrong = 0, seen = 0;
    for (int T = 2; T <= 14; ++T)
        for (int band = 1; band < T && band <= 6; ++band)
            for (int xband = band; xband <= band + 3; ++xband)
                for (int fp32 = 0; fp32 < 2; ++fp32) {
                    long r = 0, w = 0;
                    run(T, band, xband, fp32 != 0, r, w, seen);
                    if ((r || w) && races + wrong == 0)
                        std::fprintf(stderr, "first at T %d band %d xband %d fp32 %d: %ld unordered, %ld wrong\n", T, band,
                                     xband, fp32, r, w);
                    races += r;
                    wrong += w;
                }
    std::printf("races=%ld wrong=%ld seen=%ld\n", races, wrong, seen);
    return 0;
}
