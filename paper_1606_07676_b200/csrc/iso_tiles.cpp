// Plan of the schedules whose intermediate blocks fit in shared memory: all phases of a tile of processes
// in one launch (iso_tiles.cuh).
#include <algorithm>
#include <cstring>
#include <list>
#include <map>

#include "iso_internal.h"

namespace iso {

namespace {

constexpr int64_t kTileSmem = 220 * 1024;   // shared memory of a CTA whose tile is one row wide, at most
constexpr int64_t kTileTarget = 72 * 1024;  // of wider ones: three CTAs of an SM
constexpr int64_t kTilePieces = 6000;       // units of a process that the tables describe at most

int64_t round16(int64_t x) { return (x + 15) / 16 * 16; }

// Largest power of two up to 16 that divides x.
int alignment16(int64_t x)
{
    int a = 16;
    while (a > 1 && (x & (a - 1))) a >>= 1;
    return a;
}

struct Hop {
    int stage;
    uint32_t kind;
    int64_t src_off, place_dst, recv_dst, len;
    const Part *p;
};
struct Piece {
    int stage;
    uint32_t kind;
    TileUnit u;
};

// Whether anything but the schedule was asked for: how it is cut into launches, or by which kernels it runs.  (One slab and
// one chain are what a single launch has: a plan read back from one request and asked for on another stays what it was.)
bool execution_asked_for(const Request &r)
{
    const Knobs &k = r.knobs;
    return r.per_phase || r.persistent || r.wave_request || r.slab_request > 1 || r.chains_request > 1 || r.graph_request || r.hybrid ||
           r.bulk_threshold_asked >= 0 || r.sender_side != 1 || k.slabs >= 0 || k.chains >= 0 || k.graph >= 0 || k.vec_threads ||
           k.vec_ctas_per_sm || k.words >= 0 || k.sender_side >= 0 || k.hybrid >= 0 || k.mixed >= 0 || k.bulk_chunk || k.bulk_tile;
}

// Blocks of several unit widths, or of none that asynchronous copies take.
bool mixed_widths(const Request &r)
{
    const int64_t all = r.send_stride | r.recv_stride | (int64_t)(uintptr_t)r.send | (int64_t)(uintptr_t)r.recv;
    int64_t least = 16, widest = 1;
    for (const Part &p : r.parts) {
        const int64_t at = (p.src_buf == ISO_BUF_SEND ? p.src_off : 0) | (p.dst_buf == ISO_BUF_RECV ? p.dst_off : 0);
        least = std::min<int64_t>(least, alignment16(all | p.len | at));
        widest = std::max<int64_t>(widest, std::min<int64_t>(alignment16(all), p.len));
    }
    return least < 4 || (least < 16 && widest > least);
}

// The schedule's hops as moves between send buffers, places and receive buffers.  Places: what a phase reads, in the
// order of the phases that write it, each where it lies in its source's 16-byte words.  False: the schedule is not
// like that.
bool collect_hops(const Request &r, std::vector<Hop> &hops, std::list<Part> &own, int64_t &place_stride)
{
    // What only passes from a send to a receive buffer may go through places too: the copies to a place are asynchronous, so
    // that the copies of several widths wait for memory once and not one after the other.  It costs places: 13-byte
    // blocks on 257x251 57 -> 43 microseconds, irregular sizes to 24 neighbours on 18x24 7.3 -> 5.7, but, with blocks of 1 KB among
    // them, to 26 on 27x19x31 100 -> 137.
    const bool staged = mixed_widths(r) && r.stats.bytes_moved < 250000000;
    using Key = std::pair<int, int64_t>;
    std::map<Key, int64_t> read_len, place;
    for (const Part &p : r.parts)
        if (p.src_buf != ISO_BUF_SEND) {
            auto it = read_len.emplace(Key{p.src_buf, p.src_off}, p.len);
            if (it.first->second != p.len) return false;
        }
    std::vector<std::pair<int64_t, int64_t>> written[2];
    int64_t at = 0;
    auto new_place = [&](int64_t src_off, int64_t len) {
        const int64_t start = round16(at - (src_off & 15)) + (src_off & 15);
        at = start + len;
        return start;
    };
    int stage = 0, last_phase = -1;
    for (const Part &p : r.parts) {
        Hop h{0, 0, p.src_off, -1, -1, p.len, &p};
        if (p.src_buf != ISO_BUF_SEND) {
            if (p.phase != last_phase) ++stage;
            last_phase = p.phase;
            h.stage = stage;
            auto it = place.find(Key{p.src_buf, p.src_off});
            if (it == place.end()) return false;
            h.src_off = it->second;
        }
        auto it = read_len.find(Key{p.dst_buf, p.dst_off});
        if (it != read_len.end()) {
            if (it->second != p.len) return false;
            h.place_dst = place[Key{p.dst_buf, p.dst_off}] = new_place(h.src_off, p.len);
        } else if (p.dst_buf == ISO_BUF_INTER) {
            return false;  // (nobody reads it)
        }
        if (p.dst_buf == ISO_BUF_RECV) h.recv_dst = p.dst_off;
        if (staged && h.stage == 0 && h.recv_dst >= 0) {
            if (h.place_dst < 0) h.place_dst = new_place(h.src_off, p.len);
            own.push_back(p);  // the way on, to the own receive buffer
            std::fill(own.back().shift, own.back().shift + ISO_MAX_DIMS, 0);
            hops.push_back(Hop{1, 0, h.place_dst, -1, h.recv_dst, p.len, &own.back()});
            h.recv_dst = -1;
        }
        written[p.dst_buf == ISO_BUF_RECV].push_back({p.dst_off, p.dst_off + p.len});
        hops.push_back(h);
    }
    // nothing may be written twice: whatever comes from the send buffers is copied at the beginning
    for (auto &w : written) {
        std::sort(w.begin(), w.end());
        for (size_t i = 1; i < w.size(); ++i)
            if (w[i].first < w[i - 1].second) return false;
    }
    for (Hop &h : hops) {
        if (h.stage == 0) h.kind = h.recv_dst < 0 ? TILE_FETCH : TILE_DELIVER;
        else h.kind = h.place_dst >= 0 ? TILE_BETWEEN : TILE_FORWARD;
    }
    place_stride = round16(at);
    return true;
}

// Threads of a CTA, by how many an SM holds for their shared memory (64 registers each: 1024 threads to an SM), three rows and
// more to a thread: 32^3 with 26 64-byte blocks, three CTAs, of 320 threads 26.5 microseconds, of 256 27.8, of 512 (two
// CTAs) 30, of 128 32; irregular sizes on 26x31x22, two of 512 177, of 256 201.
int64_t tile_threads(int64_t unit_rows, int64_t resident)
{
    const int64_t most = resident <= 2 ? kTileThreads : (resident == 3 ? 320 : kTileThreads / 2);
    return std::min<int64_t>(most, std::max<int64_t>(64, (unit_rows / 3 + 31) / 32 * 32));
}

}  // namespace

void plan_tiles(Request &r)
{
    const Comm &c = *r.comm;
    TilesPlan &F = r.tiles;
    F = TilesPlan{};
    if (r.knobs.tiles == 0 || r.alg != ISO_ALG_COMBINING || r.fusion < 1 || r.layout != ISO_LAYOUT_PACKED || r.stats.phases < 2) return;
    // (what runs as two chains of slabs, 100 MB to a launch and more, is bound by memory and keeps them)
    if (execution_asked_for(r) || r.chains > 1) return;
    if (r.send_stride >= (int64_t)1 << 31 || r.recv_stride >= (int64_t)1 << 31) return;
    int64_t bytes = 0;
    for (const Part &p : r.parts) bytes += p.len;
    if (bytes / 16 > kTilePieces) return;
    int64_t between = 1;  // (a first look, without the allgather's receive slots)
    for (int j = 0; j < c.d; ++j)
        for (const Part &p : r.parts)
            if (p.src_buf == ISO_BUF_INTER && p.dst_buf == ISO_BUF_INTER && p.shift[j]) {
                between *= c.dims[j];
                break;
            }
    if (between * r.inter_stride > kTileSmem) return;
    std::vector<Hop> hops;
    std::list<Part> own;
    if (!collect_hops(r, hops, own, F.place_stride)) return;

    // The dimensions of the hops from place to place, and what lies between them: a tile is complete along those.
    int m0 = c.d, m1 = -1;
    for (const Hop &h : hops)
        for (int j = 0; j < c.d && h.kind == TILE_BETWEEN; ++j)
            if (h.p->shift[j]) {
                m0 = std::min(m0, j);
                m1 = std::max(m1, j);
            }
    if (m1 < 0) m0 = 0;
    for (int j = 0; j < c.d; ++j) (j < m0 ? F.outer : (j <= m1 ? F.middle : F.inner)) *= c.dims[j];
    if (F.middle > kTileSmem || F.middle * F.place_stride > kTileSmem) return;
    int coord_of[ISO_MAX_DIMS];
    for (int j = 0; j < c.d; ++j) {
        coord_of[j] = -1;
        bool used = false;
        for (const Part &p : r.parts) used = used || p.shift[j] != 0 || p.check[j] != 0;
        if (!used) continue;
        F.mesh = F.mesh || !c.periodic[j];
        coord_of[j] = (int)F.coords.size();
        F.coords.push_back(j);
    }
    for (int j : F.coords)
        if (F.mesh && c.dims[j] > 65535) return;  // (on a mesh coordinates are kept in 16 bits)

    // units, in groups of one stage and one kind, of 16 bytes or of fewer
    const int send_align = std::min(alignment16(r.send_stride), alignment16((int64_t)(uintptr_t)r.send));
    const int recv_align = std::min(alignment16(r.recv_stride), alignment16((int64_t)(uintptr_t)r.recv));
    std::vector<Piece> pieces;
    int64_t apart = 0;  // units of a byte or two whose neighbours are wider: a sector of their own
    F.shifts.assign(1, TileShift{});
    auto before = [](const TileShift &x, const TileShift &y) { return std::memcmp(&x, &y, sizeof(x)) < 0; };  // (no padding)
    std::map<TileShift, uint32_t, decltype(before)> shift_index(before);
    for (const Hop &h : hops) {
        int a = h.stage == 0 ? send_align : 16;
        if (h.place_dst >= 0) a = std::min(a, alignment16(h.src_off - h.place_dst));
        if (h.recv_dst >= 0) a = std::min({a, recv_align, alignment16(h.src_off - h.recv_dst)});
        TileShift sh{};
        sh.between = h.kind == TILE_BETWEEN;
        for (int j = 0; j < c.d; ++j) {
            if (coord_of[j] < 0) continue;
            const int e = coord_of[j], v = h.p->shift[j];
            sh.wraps[e] = c.periodic[j] != 0;
            if (h.kind != TILE_FORWARD) {
                sh.c[e] = v;
                sh.check[e] = h.p->check[j];
            } else {  // seen from the process that sends it
                sh.c[e] = c.periodic[j] && v ? c.dims[j] - v : -v;
                sh.check[e] = c.periodic[j] ? 0 : h.p->check[j] - v;
            }
        }
        int n = 0;
        for (int e = 0; e < (int)F.coords.size(); ++e) {
            if (!sh.c[e]) continue;
            if (n < 2) {
                sh.first_two |= (uint32_t)e << (16 + 8 * n);
                (n == 0 ? sh.c_first : sh.c_second) = sh.c[e];
            }
            ++n;
        }
        sh.first_two |= (uint32_t)n | (sh.between ? 1u << 8 : 0u);
        const uint32_t index = shift_index.emplace(sh, (uint32_t)F.shifts.size()).first->second;
        if (index == F.shifts.size()) F.shifts.push_back(sh);
        for (int64_t x = 0; x < h.len;) {
            int w = a;
            while (w > 1 && (((h.src_off + x) & (w - 1)) || h.len - x < w)) w >>= 1;
            TileUnit u{};
            u.src_off = (uint32_t)(h.src_off + x);
            u.place_dst = h.place_dst >= 0 ? (int32_t)(h.place_dst + x) : -1;
            u.recv_dst = h.recv_dst >= 0 ? (int32_t)(h.recv_dst + x) : -1;
            u.shift = index;
            u.width = (uint8_t)w;
            // (asynchronous copies move at least 4 bytes)
            pieces.push_back(Piece{h.stage, h.kind == TILE_FETCH && w < 4 ? TILE_DELIVER : h.kind, u});
            x += w;
            apart += w < 4 && (a >= 4 || h.len < 4);
            if ((int64_t)pieces.size() > kTilePieces) return;
        }
    }
    std::stable_sort(pieces.begin(), pieces.end(), [](const Piece &x, const Piece &y) {
        if (x.stage != y.stage) return x.stage < y.stage;
        return x.kind != y.kind ? x.kind < y.kind : x.u.width > y.u.width;
    });
    // (A group costs a quarter of a microsecond whatever is in it, so the narrow widths go together: irregular sizes to 48 neighbours on
    // 20x27 8.4 -> 6.3, the 32^3 mesh with blocks of 1024, 32 and 1 bytes 147 -> 126.)
    F.unit = pieces.empty() ? 0 : (int)pieces[0].u.width;
    for (const Piece &q : pieces)
        if ((int)q.u.width != F.unit || F.unit < 4) F.unit = 0;
    for (const Piece &q : pieces) {
        const uint32_t width = F.unit ? (uint32_t)F.unit : (q.u.width == 16 ? 16u : 0u);
        if (F.groups.empty() || F.groups.back().stage != (uint32_t)q.stage || F.groups.back().kind != q.kind || F.groups.back().width != width)
            F.groups.push_back(TileGroup{q.kind, width, (uint32_t)q.stage, (uint32_t)F.units.size(), 0});
        ++F.groups.back().n;
        F.units.push_back(q.u);
    }
    for (TileGroup &g : F.groups) {
        bool eights = g.width == 0;  // (those have code of their own: 88-byte blocks on 17x12x10x17 26 microseconds, 30 without)
        for (uint32_t u = g.first; u < g.first + g.n; ++u) eights = eights && F.units[u].width == 8;
        if (eights) g.width = 8;
    }
    if (F.groups.empty() || (int)F.groups.size() > kTileGroups) return;

    // The width of a tile: the one with which the SM that has the most tiles has the least to do.  A unit of a row counts
    // one, and one more per tile for its descriptor; a partner of a row more, on a mesh (with its conditions) the most.  A copy of
    // the unit table in shared memory pays for itself unless the table is long and a CTA has many tiles (27x28x29 with 124 blocks of 192
    // bytes, two dimensions per phase, 2640 units 373 -> 234 microseconds without; 110x59 with 359 bytes, 752 units, 10.1 with and
    // 13.7 without).
    const int64_t units = (int64_t)F.units.size(), shifts = (int64_t)F.shifts.size(), table = units * (int64_t)sizeof(TileUnit);
    const int64_t per_row = F.place_stride + 4 * shifts + (F.mesh ? 2 * (int64_t)F.coords.size() : 0);
    auto copied = [&](int64_t tiles) { return units <= 1600 || tiles <= 2 * r.sm_count; };
    int64_t longest = 1;
    for (const TileGroup &g : F.groups) longest = std::max<int64_t>(longest, g.n);
    double least = 0;
    int64_t most_tiles = 0;
    for (int64_t w = 1; w <= F.inner; ++w) {
        const int64_t rows = F.middle * w, tiles = F.outer * ((F.inner + w - 1) / w);
        const int64_t smem = rows * per_row + (copied(tiles) ? table : 0) + 128;
        if (smem > (w == 1 ? kTileSmem : kTileTarget)) break;
        const int64_t per_sm = (tiles + r.sm_count - 1) / r.sm_count, resident = std::max<int64_t>(1, 228 * 1024 / (smem + 1024));
        const int64_t threads = tile_threads(longest * rows, resident);
        const double warps = (double)(std::min({resident, 1024 / threads, per_sm}) * threads / 32);
        const double cost = (double)per_sm * (double)(units * (rows + 1) + (F.mesh ? 6 : 2) * shifts * rows + 400) * (0.75 + 8.0 / warps);
        if (least != 0 && cost >= least) continue;
        least = cost;
        most_tiles = per_sm;
        F.width = w;
    }
    if (least == 0) return;
    F.intervals = (F.inner + F.width - 1) / F.width;
    F.rows_per_tile = F.middle * F.width;
    F.moved_at = (size_t)(F.rows_per_tile * F.place_stride);
    F.coords_at = F.moved_at + (size_t)(F.rows_per_tile * shifts) * 4;
    F.smem = F.coords_at + (F.mesh ? (size_t)(F.rows_per_tile * 2) * F.coords.size() : 0);
    if (copied(F.outer * F.intervals)) {
        F.units_at = (size_t)round16((int64_t)F.smem);
        F.smem = F.units_at + (size_t)table;
    }
    const int64_t resident = std::max<int64_t>(1, 228 * 1024 / ((int64_t)F.smem + 1024));
    F.threads = (int)tile_threads(longest * F.rows_per_tile, resident);
    F.grid = std::min<int64_t>(F.outer * F.intervals, std::min<int64_t>(resident, 1024 / F.threads) * r.sm_count);

    // Which is faster?  Both sides fitted to 402 calls of all sorts (2 to 5 phases, 3 to 600 microseconds; the times of either side
    // within some 30 % of these), in microseconds.  A launch costs 2.5, and what is moved nearly the rate of a copy, less of it
    // where blocks are not made of 16-byte units; where some go to the bulk kernel, which wants long launches, more.  A tile costs
    // what its rows' units do, and at least what the receive buffers take at 3.6 or 3.3 TB/s (31x22x22 with 342 neighbours, allgather of
    // 48 bytes, 71 against 60 in phases; 11x11x15x13 with 80, 152 bytes, 142 against 116).  The line lies where next to none of those calls lost: used for 260 of them, in 0.64 of
    // the time (a quarter took less than half).
    bool bulk = false;
    for (const LaunchPlan &L : r.launches) bulk = bulk || L.kernel == KERNEL_BULK;
    const double moved = (double)r.stats.bytes_moved / 6.537e6, received = (double)r.stats.bytes_min / 2.0 / (F.unit == 16 ? 3.6e6 : 3.3e6);
    const double per_phase = 2.5 * r.stats.phases + 2.2 * (double)(r.launches.size() - r.stats.phases) + (bulk ? 4.0 - 0.6 * r.stats.phases : 0.0) +
                             ((r.kind == ISO_KIND_ALLGATHER ? 0.84 : 0.76) + (F.unit == 16 ? 0.0 : (F.unit == 0 ? 0.4 : 0.82))) * moved;
    // (a byte or two between wider units is a sector of its own on either side: stencil blocks of 324, 18 and 1 bytes on 43x44x39 228
    // against 167)
    const double work = least * (1.0 + 4.0 * (double)apart / (double)units);
    const double in_tiles = std::max(1.3 + 0.23 * (double)F.groups.size() + 0.000215 * work + 0.3 * (double)most_tiles, received);
    F.on = r.knobs.tiles >= 1 || in_tiles < (F.unit == 0 ? 0.75 : 0.8) * per_phase;
}

}  // namespace iso
