// Host-side check of the wide row kernel's gather lists (no GPU needed): every (cell, antenna, tap)
// contribution appears exactly once, in its band of 64 rows, under the lane that owns its cell pair;
// the odd-row bit follows the row; offsets stay inside the table; each cell pair is stored once; a
// layout wider than 128 cells is refused; the table does not depend on the host threads.
// Usage: wide_lists_check A K span_x span_y C   (exit status 0 when every check holds)
#include <cstdio>
#include <cstdlib>
#include <random>
#include <set>
#include <vector>

#include "epic_internal.cuh"

static long g_bad = 0;
#define CHECK(cond, ...)                  \
    do {                                  \
        if (!(cond)) {                    \
            if (g_bad < 10) {             \
                std::printf(__VA_ARGS__); \
                std::printf("\n");        \
            }                             \
            g_bad++;                      \
        }                                 \
    } while (0)

int main(int argc, char **argv)
{
    if (argc != 6) return 2;
    const int A = std::atoi(argv[1]), K = std::atoi(argv[2]), sx = std::atoi(argv[3]), sy = std::atoi(argv[4]),
              C = std::atoi(argv[5]);
    const int h = (K - 1) / 2, W = 12, S = 129;
    std::mt19937 rng(11u + A + sx);
    std::vector<short2> cells(static_cast<size_t>(C) * A);
    for (int c = 0; c < C; c++) {
        const int ox = 100 + 3 * c, oy = 90 - c;
        for (int a = 0; a < A; a++) {
            int x = static_cast<int>(rng() % (sx - 2 * h)), y = static_cast<int>(rng() % (sy - 2 * h));
            if (a == 0) x = y = 0;
            if (a == 1 % A) {
                x = sx - 2 * h - 1;
                y = sy - 2 * h - 1;
            }
            cells[static_cast<size_t>(c) * A + a] = make_short2(static_cast<short>(ox + h + x), static_cast<short>(oy + h + y));
        }
    }
    std::vector<int> chans(C);
    for (int i = 0; i < C; i++) chans[i] = C - 1 - i;
    int bands = 0, bands1 = 0;
    std::vector<uint32_t> tab, tab1;
    std::vector<int2> idx, idx1;
    std::vector<int4> chan, chan1;
    const int rc = epic::build_wide_lists(cells, A, K, chans, bands, tab, idx, chan);
    CHECK((rc == EPIC_OK) == (sx <= 128 && sy <= 128), "status %d", rc);
    if (rc == EPIC_OK) {
        CHECK(epic::build_wide_lists(cells, A, K, chans, bands1, tab1, idx1, chan1, 1) == EPIC_OK && tab1 == tab &&
                  bands1 == bands, "one host thread builds another table");
        CHECK(bands == (sy + 63) / 64, "%d bands", bands);
    }
    for (int ci = 0; ci < C && rc == EPIC_OK; ci++) {
        const int c = chans[ci], ox = 100 + 3 * c, oy = 90 - c;
        CHECK(A == 1 || (chan[ci].x == sy && chan[ci].y == sx), "channel %d: %d x %d", ci, chan[ci].x, chan[ci].y);
        std::multiset<long long> want, got;   // (row, column, antenna, tap)
        for (int a = 0; a < A; a++) {
            const short2 k = cells[static_cast<size_t>(c) * A + a];
            for (int dyi = 0; dyi < K; dyi++)
                for (int dx = 0; dx < K; dx++)
                    want.insert((static_cast<long long>((k.y + dyi - h - oy) * 256 + k.x + dx - h - ox) << 32) |
                                (static_cast<long long>(a) << 8) | (dyi * K + dx));
        }
        std::set<int> stored;
        for (int band = 0; band < bands; band++)
            for (int w = 0; w < W; w++) {
                const int2 ix = idx[(static_cast<size_t>(ci) * bands + band) * W + w];
                size_t off = static_cast<size_t>(ix.x);
                for (int b = 0; b < ix.y; b++) {
                    CHECK(off + 33 <= tab.size(), "channel %d: header outside the table", ci);
                    if (off + 33 > tab.size()) break;
                    const size_t d = tab[off];
                    CHECK(d >= 1 && off + 33 + 32 * d <= tab.size(), "channel %d: batch outside the table", ci);
                    if (off + 33 + 32 * d > tab.size()) break;
                    for (int l = 0; l < 32; l++) {
                        const uint32_t o = tab[off + 1 + l];
                        const int cell = static_cast<int>(o & 0x7FFFFFFFu), y = cell / S, x = cell % S;
                        if (o != ~0u) {
                            CHECK((o >> 31) == static_cast<uint32_t>(y & 1), "channel %d: odd-row bit", ci);
                            CHECK(y < 64 && x < 128 && x % 2 == 0, "channel %d: cell (%d, %d)", ci, y, x);
                            CHECK(stored.insert((band * 64 + y) * 256 + x).second, "channel %d: cell stored twice", ci);
                        }
                        for (size_t j = 0; j < d; j++) {
                            const uint32_t e = tab[off + 33 + 32 * j + l];
                            const long long a = e >> 8;
                            const int tp = static_cast<int>(e & 255u), dyi = tp / (K + 1), dxl = tp % (K + 1) - 1;
                            CHECK(a < A && tp <= K * (K + 1), "channel %d: entry out of range", ci);
                            if (tp == K * (K + 1)) continue;
                            CHECK(o != ~0u, "channel %d: entry under an empty lane", ci);
                            const long long at = (band * 64 + y) * 256 + x;
                            if (dxl >= 0) got.insert((at << 32) | (a << 8) | (dyi * K + dxl));
                            if (dxl + 1 < K) got.insert(((at + 1) << 32) | (a << 8) | (dyi * K + dxl + 1));
                        }
                    }
                    off += 33 + 32 * d;
                }
            }
        CHECK(want == got, "channel %d: contributions differ (%zu wanted, %zu listed)", ci, want.size(), got.size());
    }
    std::printf("%s: A=%d K=%d span=%d x %d, %zu words\n", g_bad ? "FAIL" : "ok", A, K, sx, sy, tab.size());
    return g_bad ? 1 : 0;
}
