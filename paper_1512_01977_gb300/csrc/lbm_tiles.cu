// Work plan of the batched step kernel: the (z-strip, row) space of every solve
// is cut into tiles (rows [j0, jend) of one strip of one solve) and the tiles
// are dealt to the CTAs of one launch, largest first, each to the CTA with the
// smallest load so far (longest-processing-time scheduling).  A tile costs its
// rows plus `fill` rows of pipeline fill (march2: kTileFillRows): the kernel marches 6 halo rows
// above the tile and its last stage trails the first by 12 rows.  Host code.
#include <algorithm>
#include <map>
#include <new>
#include <queue>
#include <vector>

#include "lbm_axi_batch.h"
#include "lbm_tiles.h"

namespace lbm {

namespace {

struct Cand {
    std::vector<Tile> tiles;
    std::vector<int> first;
    long long makespan = -1;
    int ncta = 0;
};

// Tiles of chunk height at most h (h <= 0: one tile per strip), rows split evenly.
void cut(const int* nz, const int* nr, int n, int strip, int h, std::vector<Tile>& out) {
    out.clear();
    for (int s = 0; s < n; s++) {
        const int strips = (nz[s] + strip - 1) / strip;
        const int c = h > 0 ? std::max(1, (nr[s] + h - 1) / h) : 1;
        const int q = nr[s] / c, r = nr[s] % c;
        for (int t = 0; t < strips; t++) {
            int j = 0;
            for (int k = 0; k < c; k++) {
                const int rows = q + (k < r ? 1 : 0);
                out.push_back(Tile{s, t, j, j + rows});
                j += rows;
            }
        }
    }
}

long long count_tiles(const int* nz, const int* nr, int n, int strip, int h) {
    long long t = 0;
    for (int s = 0; s < n; s++)
        t += (long long)((nz[s] + strip - 1) / strip) * std::max(1, (nr[s] + h - 1) / h);
    return t;
}

void deal(std::vector<Tile>& tiles, int slots, int fill, Cand& c) {
    std::vector<int> order(tiles.size());
    for (size_t i = 0; i < order.size(); i++) order[i] = (int)i;
    std::stable_sort(order.begin(), order.end(), [&](int a, int b) {
        return tiles[a].jend - tiles[a].j0 > tiles[b].jend - tiles[b].j0;
    });
    // min-heap of (load, cta)
    typedef std::pair<long long, int> L;
    std::priority_queue<L, std::vector<L>, std::greater<L>> heap;
    const int used = (int)std::min<size_t>((size_t)slots, tiles.size());
    for (int k = 0; k < used; k++) heap.push(L(0, k));
    std::vector<int> owner(tiles.size());
    std::vector<long long> load(used, 0);
    for (int i : order) {
        L top = heap.top();
        heap.pop();
        owner[i] = top.second;
        top.first += tiles[i].jend - tiles[i].j0 + fill;
        load[top.second] = top.first;
        heap.push(top);
    }
    // group by CTA; within a CTA keep the cut order (solve, strip, rows)
    std::vector<int> count(used + 1, 0);
    for (size_t i = 0; i < tiles.size(); i++) count[owner[i] + 1]++;
    for (int k = 0; k < used; k++) count[k + 1] += count[k];
    c.first = count;
    c.tiles.assign(tiles.size(), Tile{0, 0, 0, 0});
    std::vector<int> pos(count.begin(), count.end() - 1);
    for (size_t i = 0; i < tiles.size(); i++) c.tiles[pos[owner[i]]++] = tiles[i];
    c.makespan = 0;
    for (long long x : load) c.makespan = std::max(c.makespan, x);
    c.ncta = used;
}

// Chunk heights worth trying: whole strips, and the smallest height (>= 16 rows) whose tiles fill k = 1..4 waves.
std::vector<int> candidate_heights(const int* nz, const int* nr, int n, int strip, int slots, int max_nr) {
    std::vector<int> heights = {0};
    for (int k = 1; k <= 4; k++) {
        int lo = std::min(16, max_nr), hi = max_nr;
        if (count_tiles(nz, nr, n, strip, hi) > (long long)k * slots) continue;
        while (lo < hi) {
            const int mid = (lo + hi) / 2;
            if (count_tiles(nz, nr, n, strip, mid) <= (long long)k * slots) hi = mid;
            else lo = mid + 1;
        }
        heights.push_back(lo);
    }
    return heights;
}

// The largest load that deal() would give, from how many tiles there are of each height: slots of equal load are
// taken together, a few steps where the heap takes one per tile.  *ntiles: the number of tiles.
long long makespan_of(const int* nz, const int* nr, int n, int strip, int h, int slots, int fill, long long* ntiles) {
    std::map<int, long long, std::greater<int>> tall;  // height -> tiles
    *ntiles = 0;
    for (int s = 0; s < n; s++) {
        const long long strips = (nz[s] + strip - 1) / strip;
        const int c = h > 0 ? std::max(1, (nr[s] + h - 1) / h) : 1, q = nr[s] / c, r = nr[s] % c;
        if (r) tall[q + 1] += strips * r;
        tall[q] += strips * (c - r);
        *ntiles += strips * c;
    }
    std::map<long long, long long> loads;  // load -> slots
    loads[0] = std::min<long long>(slots, *ntiles);
    long long most = 0;
    for (const auto& t : tall)
        for (long long left = t.second; left > 0;) {
            const auto least = loads.begin();
            const long long load = least->first + t.first + fill, take = std::min(left, least->second);
            least->second -= take;
            if (least->second == 0) loads.erase(least);
            loads[load] += take;
            most = std::max(most, load);
            left -= take;
        }
    return most;
}

}  // namespace

int plan_tiles(const int* nz, const int* nr, int n, int strip, int slots, std::vector<Tile>& tiles,
               std::vector<int>& first, long long* makespan, int fill) {
    if (!nz || !nr || n < 1 || strip < 1 || slots < 1) return LBM_ERR_INVALID_ARG;
    int max_nr = 0;
    for (int s = 0; s < n; s++) {
        if (nz[s] < 1 || nr[s] < 1) return LBM_ERR_INVALID_ARG;
        max_nr = std::max(max_nr, nr[s]);
    }
    try {
        const std::vector<int> heights = candidate_heights(nz, nr, n, strip, slots, max_nr);
        Cand best;
        std::vector<Tile> cutv;
        for (int h : heights) {
            cut(nz, nr, n, strip, h, cutv);
            Cand c;
            deal(cutv, slots, fill, c);
            if (best.makespan < 0 || c.makespan < best.makespan ||
                (c.makespan == best.makespan && c.tiles.size() < best.tiles.size()))
                best = std::move(c);
        }
        tiles = std::move(best.tiles);
        first = std::move(best.first);
        if (makespan) *makespan = best.makespan;
    } catch (const std::bad_alloc&) {
        return LBM_ERR_OOM;
    }
    return LBM_OK;
}

// plan_tiles' choice of heights; which slot a tile would go to does not matter here, so nothing is dealt (plan_tiles
// and a sort took 0.98 ms for 4096 x 2048 and 1824 slots on the Grace host, all but 0.2 of which a solve's creation
// had not spent with 608 slots).
int plan_warp_tiles(const int* nz, const int* nr, int n, int slots, std::vector<Tile>& tiles) {
    if (!nz || !nr || n < 1 || slots < 1) return LBM_ERR_INVALID_ARG;
    int max_nr = 0;
    for (int s = 0; s < n; s++) {
        if (nz[s] < 1 || nr[s] < 1) return LBM_ERR_INVALID_ARG;
        max_nr = std::max(max_nr, nr[s]);
    }
    try {
        int best = 0;
        long long least = -1, fewest = 0;
        for (int h : candidate_heights(nz, nr, n, kWarpStrip, slots, max_nr)) {
            long long count;
            const long long m = makespan_of(nz, nr, n, kWarpStrip, h, slots, kWarpFillRows, &count);
            if (least < 0 || m < least || (m == least && count < fewest)) best = h, least = m, fewest = count;
        }
        cut(nz, nr, n, kWarpStrip, best, tiles);
        std::stable_sort(tiles.begin(), tiles.end(),
                         [](const Tile& a, const Tile& b) { return a.jend - a.j0 > b.jend - b.j0; });
    } catch (const std::bad_alloc&) {
        return LBM_ERR_OOM;
    }
    return LBM_OK;
}

}  // namespace lbm

extern "C" int lbm_axi_tile_plan(const int* nz, const int* nr, int n, int strip, int slots, int max_tiles,
                                 int* tiles_out, int* first_out, int* ntiles, int* ncta, long long* makespan) {
    if (!ntiles || !ncta || max_tiles < 0) return LBM_ERR_INVALID_ARG;
    std::vector<lbm::Tile> tiles;
    std::vector<int> first;
    long long ms = 0;
    const int rc = lbm::plan_tiles(nz, nr, n, strip, slots, tiles, first, &ms);
    if (rc != LBM_OK) return rc;
    *ntiles = (int)tiles.size();
    *ncta = (int)first.size() - 1;
    if (makespan) *makespan = ms;
    if ((int)tiles.size() > max_tiles || !tiles_out || !first_out) return LBM_ERR_INVALID_ARG;
    for (size_t i = 0; i < tiles.size(); i++) {
        tiles_out[4 * i] = tiles[i].solve;
        tiles_out[4 * i + 1] = tiles[i].strip;
        tiles_out[4 * i + 2] = tiles[i].j0;
        tiles_out[4 * i + 3] = tiles[i].jend;
    }
    for (size_t c = 0; c < first.size(); c++) first_out[c] = first[c];
    return LBM_OK;
}
