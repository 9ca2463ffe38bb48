// Host-side check of the compact kernel's gather lists (no GPU needed): every (cell, antenna, tap)
// contribution appears exactly once, under the lane that owns its cell pair, relative to the first
// occupied cell; the odd-row bit follows the row; offsets stay inside the block; each cell pair is
// stored once; a layout wider than 64 cells is refused.
// Usage: compact_lists_check A K span C P   (exit status 0 when every check holds)
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
    const int A = std::atoi(argv[1]), K = std::atoi(argv[2]), span = std::atoi(argv[3]), C = std::atoi(argv[4]),
              P = std::atoi(argv[5]);
    const int h = (K - 1) / 2, N = 128;
    std::mt19937 rng(7u + A + span);
    std::vector<short2> cells(static_cast<size_t>(C) * A);
    for (int c = 0; c < C; c++) {
        // footprints span exactly `span` cells on both axes, from another corner in each channel
        const int ox = 5 + 3 * c, oy = 20 - c, in = span - 2 * h;
        for (int a = 0; a < A; a++) {
            int x = static_cast<int>(rng() % in), y = static_cast<int>(rng() % in);
            if (a == 0) x = y = 0;
            if (a == 1 % A) x = y = in - 1;
            cells[static_cast<size_t>(c) * A + a] = make_short2(static_cast<short>(ox + h + x), static_cast<short>(oy + h + y));
        }
    }
    std::vector<int> chans(C);
    for (int i = 0; i < C; i++) chans[i] = C - 1 - i;   // the group's order, not the plan's
    std::vector<uint16_t> tab;
    std::vector<int2> idx;
    std::vector<int4> chan;
    const int rc = epic::build_compact_lists(cells, A, K, P, chans, tab, idx, chan);
    const bool fits = span <= 64 && A <= 1024 && K * (K + 1) <= 62;
    CHECK((rc == EPIC_OK) == fits, "span %d: status %d", span, rc);
    for (int ci = 0; ci < C && rc == EPIC_OK; ci++) {
        const int c = chans[ci], ox = 5 + 3 * c, oy = 20 - c;
        const int4 ch = chan[2 * ci], org = chan[2 * ci + 1];
        CHECK(A == 1 || (ch.z == span && ch.w == span), "channel %d: %d x %d occupied", ci, ch.z, ch.w);
        CHECK(org.x == ox && org.y == oy, "channel %d: origin (%d, %d)", ci, org.x, org.y);
        std::multiset<long long> want, got;
        for (int a = 0; a < A; a++) {
            const short2 k = cells[static_cast<size_t>(c) * A + a];
            for (int dyi = 0; dyi < K; dyi++)
                for (int dx = 0; dx < K; dx++)
                    want.insert((static_cast<long long>((k.y + dyi - h - oy) * 65 + k.x + dx - h - ox) << 32) |
                                (static_cast<long long>(a) << 8) | (dyi * K + dx));
        }
        std::set<int> stored;
        const uint16_t *blk = tab.data() + ch.x;
        for (int w = 0; w < epic::kCompactGatherWarps; w++) {
            const int2 ix = idx[static_cast<size_t>(ci) * epic::kCompactGatherWarps + w];
            long long off = ix.x;
            for (int b = 0; b < ix.y; b++) {
                CHECK(off + 33 <= ch.y, "channel %d: header outside the block", ci);
                if (off + 33 > ch.y) break;
                const int d = blk[off];
                CHECK(d >= 1 && off + 33 + 32LL * d <= ch.y, "channel %d: batch outside the block", ci);
                if (off + 33 + 32LL * d > ch.y) break;
                for (int l = 0; l < 32; l++) {
                    const uint16_t o = blk[off + 1 + l];
                    const int cell = o & 0x7FFF;
                    if (o != 0xFFFFu) {
                        CHECK(((o >> 15) & 1) == ((cell / 65) & 1), "channel %d: odd-row bit", ci);
                        CHECK(cell / 65 < 64 && cell % 65 < 64 && (cell % 65) % 2 == 0, "channel %d: cell %d", ci, cell);
                        CHECK(stored.insert(cell).second, "channel %d: cell %d stored twice", ci, cell);
                    }
                    for (int j = 0; j < d; j++) {
                        const uint16_t e = blk[off + 33 + 32LL * j + l];
                        const long long a = e & 1023;
                        const int tp = e >> 10, dyi = tp / (K + 1), dxl = tp % (K + 1) - 1;
                        CHECK(a < A && tp <= K * (K + 1), "channel %d: entry out of range", ci);
                        if (tp == K * (K + 1)) continue;   // an empty step
                        CHECK(o != 0xFFFFu, "channel %d: entry under an empty lane", ci);
                        if (dxl >= 0) got.insert((static_cast<long long>(cell) << 32) | (a << 8) | (dyi * K + dxl));
                        if (dxl + 1 < K) got.insert((static_cast<long long>(cell + 1) << 32) | (a << 8) | (dyi * K + dxl + 1));
                    }
                }
                off += 33 + 32LL * d;
            }
        }
        CHECK(want == got, "channel %d: contributions differ (%zu wanted, %zu listed)", ci, want.size(), got.size());
    }
    std::printf("%s: A=%d K=%d span=%d, %zu words\n", g_bad ? "FAIL" : "ok", A, K, span, tab.size());
    return g_bad ? 1 : 0;
}
