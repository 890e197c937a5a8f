// Plan of the schedules whose intermediate blocks fit in shared memory: all phases of a tile of processes
// in one launch (iso_tiles.cuh).
#include <algorithm>
#include <cmath>
#include <cstring>
#include <list>

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
// order of the phases that write it, each where it lies in its source's 16-byte words; `staged`: what only passes from a send to
// a receive buffer as well.  False: the schedule is not like that.
bool collect_hops(const Request &r, bool staged, std::vector<Hop> &hops, std::list<Part> &own, int64_t &place_stride)
{
    struct Read { int64_t key, len, place; };  // what a phase reads, and its place once it has one
    std::vector<Read> reads;
    auto key_of = [](int buf, int64_t off) { return off * 4 + buf; };
    for (const Part &p : r.parts)
        if (p.src_buf != ISO_BUF_SEND) reads.push_back(Read{key_of(p.src_buf, p.src_off), p.len, -1});
    std::sort(reads.begin(), reads.end(), [](const Read &x, const Read &y) { return x.key != y.key ? x.key < y.key : x.len < y.len; });
    for (size_t i = 1; i < reads.size(); ++i)
        if (reads[i].key == reads[i - 1].key && reads[i].len != reads[i - 1].len) return false;
    reads.erase(std::unique(reads.begin(), reads.end(), [](const Read &x, const Read &y) { return x.key == y.key; }), reads.end());
    auto find = [&](int buf, int64_t off) -> Read * {
        const int64_t key = key_of(buf, off);
        auto it = std::lower_bound(reads.begin(), reads.end(), key, [](const Read &x, int64_t k) { return x.key < k; });
        return it != reads.end() && it->key == key ? &*it : nullptr;
    };
    std::vector<std::pair<int64_t, int64_t>> written[2];
    hops.reserve(2 * r.parts.size());
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
            const Read *from = find(p.src_buf, p.src_off);
            if (from->place < 0) return false;
            h.src_off = from->place;
        }
        if (Read *to = find(p.dst_buf, p.dst_off)) {
            if (to->len != p.len) return false;
            h.place_dst = to->place = new_place(h.src_off, p.len);
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

// How many tiles an SM works on at a time, and in how many turns.
struct Residency {
    int64_t per_sm, at_once, turns;
    Residency(int64_t tiles, int64_t smem, int64_t threads, int sm_count)
    {
        per_sm = (tiles + sm_count - 1) / sm_count;
        at_once = std::max<int64_t>(1, std::min({228 * 1024 / (smem + 1024), 1024 / threads, per_sm}));
        turns = (per_sm + at_once - 1) / at_once;
    }
};

// The plan's units, groups and tiles.  False: the schedule cannot run so.
bool build_plan(const Request &r, bool staged, TilesPlan &F)
{
    const Comm &c = *r.comm;
    F = TilesPlan{};
    std::vector<Hop> hops;
    std::list<Part> own;
    if (!collect_hops(r, staged, hops, own, F.place_stride)) return false;
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
    if (F.middle > kTileSmem || F.middle * F.place_stride > kTileSmem) return false;
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
        if (F.mesh && c.dims[j] > 65535) return false;  // (on a mesh coordinates are kept in 16 bits)

    // units, in groups of one stage and one kind, of 16 bytes or of fewer
    const int send_align = std::min(alignment16(r.send_stride), alignment16((int64_t)(uintptr_t)r.send));
    const int recv_align = std::min(alignment16(r.recv_stride), alignment16((int64_t)(uintptr_t)r.recv));
    std::vector<Piece> pieces;
    pieces.reserve(512);
    F.shifts.assign(1, TileShift{});
    size_t slots = 64;  // of a table of the shifts so far, by their bytes
    while (slots < 2 * hops.size() + 2) slots *= 2;
    std::vector<uint32_t> shift_at(slots, 0);
    auto index_of = [&](const TileShift &sh) {
        uint64_t words[sizeof(TileShift) / 8], hash = 0;  // (no padding)
        std::memcpy(words, &sh, sizeof(sh));
        for (uint64_t w : words) hash = (hash ^ w) * 0x9E3779B97F4A7C15ull, hash ^= hash >> 29;
        for (size_t at = hash & (slots - 1);; at = (at + 1) & (slots - 1)) {
            if (shift_at[at] == 0) {
                shift_at[at] = (uint32_t)F.shifts.size();
                F.shifts.push_back(sh);
            }
            if (std::memcmp(&F.shifts[shift_at[at]], &sh, sizeof(sh)) == 0) return shift_at[at];
        }
    };
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
        const uint32_t index = index_of(sh);
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
            if ((int64_t)pieces.size() > kTilePieces) return false;
        }
    }
    // (A group costs a quarter of a microsecond whatever is in it, so the narrow widths go together: irregular sizes to 48 neighbours on
    // 20x27 8.4 -> 6.3, the 32^3 mesh with blocks of 1024, 32 and 1 bytes 147 -> 126.)
    F.unit = pieces.empty() ? 0 : (int)pieces[0].u.width;
    int stages = 0;
    for (const Piece &q : pieces) {
        if ((int)q.u.width != F.unit || F.unit < 4) F.unit = 0;
        stages = std::max(stages, q.stage + 1);
    }
    // sorted by stage, kind and width, the wider ones first
    auto rank_of = [](const Piece &q) {
        const int narrow = q.u.width == 16 ? 0 : (q.u.width == 8 ? 1 : (q.u.width == 4 ? 2 : (q.u.width == 2 ? 3 : 4)));
        return (size_t)((q.stage * 4 + (int)q.kind) * 5 + narrow);
    };
    std::vector<uint32_t> first((size_t)stages * 20 + 1, 0);
    for (const Piece &q : pieces) ++first[rank_of(q) + 1];
    for (size_t k = 1; k < first.size(); ++k) first[k] += first[k - 1];
    F.units.resize(pieces.size());
    for (size_t k = 0; k + 1 < first.size(); ++k) {
        if (first[k] == first[k + 1]) continue;
        const uint32_t stage = (uint32_t)(k / 20), kind = (uint32_t)(k / 5 % 4);
        const uint32_t width = F.unit ? (uint32_t)F.unit : (k % 5 == 0 ? 16u : 0u);
        if (F.groups.empty() || F.groups.back().stage != stage || F.groups.back().kind != kind || F.groups.back().width != width)
            F.groups.push_back(TileGroup{kind, width, stage, first[k], 0});
        F.groups.back().n += first[k + 1] - first[k];
    }
    for (const Piece &q : pieces) F.units[first[rank_of(q)]++] = q.u;
    for (TileGroup &g : F.groups) {
        bool eights = g.width == 0;  // (those have code of their own: 88-byte blocks on 17x12x10x17 26 microseconds, 30 without)
        for (uint32_t u = g.first; u < g.first + g.n; ++u) eights = eights && F.units[u].width == 8;
        if (eights) g.width = 8;
    }
    if (F.groups.empty() || (int)F.groups.size() > kTileGroups) return false;

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
    for (int64_t w = 1; w <= F.inner; ++w) {
        const int64_t rows = F.middle * w, tiles = F.outer * ((F.inner + w - 1) / w);
        const int64_t smem = rows * per_row + (copied(tiles) ? table : 0) + 128;
        if (smem > (w == 1 ? kTileSmem : kTileTarget)) break;
        const int64_t threads = tile_threads(longest * rows, std::max<int64_t>(1, 228 * 1024 / (smem + 1024)));
        const Residency on(tiles, smem, threads, r.sm_count);
        const double warps = (double)(on.at_once * threads / 32);
        const double cost = (double)on.per_sm * (double)(units * (rows + 1) + (F.mesh ? 6 : 2) * shifts * rows + 400) * (0.75 + 8.0 / warps);
        if (least != 0 && cost >= least) continue;
        least = cost;
        F.width = w;
    }
    if (least == 0) return false;
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
    return true;
}

// What decides between tiles and a launch per phase, in microseconds: [0] for all-to-alls, [1] for allgathers.  Fitted to
// 8164 calls of all sorts (2 to 5 dimensions, tori and meshes, 64 to 131 072 processes, blocks of 1 to 4096 bytes) timed both ways and,
// where blocks can be staged, all three, for the least time lost by the choice, with a loss against phases or against the choice
// made before weighed fifteen times as much as a gain (sixty times for calls that were not in tiles before).  The estimates are within some
// 20 %.  Of the 8164 calls 6650 run in tiles, in 0.60 of their time in phases; 62 of those lose 5 % and more, at most 1.6 (before: 5446
// and 113, at most 2.3), and 61 calls take 5 % longer than by the choice before.  Fitted to one half, the other half loses as much.
struct TileCosts {
    double turn, load, move;                    // per turn of an SM: itself, a load from device and one from shared memory that others wait for
    double unit16, unit_one, unit_mixed, partner;  // per thousand on the busiest SM: a unit of a row of 16 bytes, of one narrower width and of one among
                                                   // several; a row's partner on a mesh
    double table, warps;                        // per thousand: a unit descriptor that is not copied to shared memory; how much dearer all that is with one warp
    double sector, cut, late;                   // per million: a 32-byte sector touched; of calls that receive more than 8 MB, a cut one of the receive
                                                // buffers and any of them
    double power;                               // of issue and memory: 1, one after the other, more, side by side
};
constexpr TileCosts kTileCosts[2] = {{1.68, 0.537, 0.244, 0.114, 0.009, 0.068, 0.863, 0.478, 13.5, 2.43, 3.17, 0.0, 1.04},
                                     {1.62, 0.459, 0.114, 0.235, 0.178, 0.306, 1.43, 0.526, 3.79, 0.0, 7.68, 8.92, 8.77}};
struct PhaseCosts {
    double phase, launch;         // a phase, and every launch of it but one
    double moved, bulk, mixed;    // per time of a copy: what is moved, and more where the bulk kernel does or widths are mixed
    double block, end, end_mesh;  // per million: a block of a hop, an end of one that does not fall on 16 bytes, that on a mesh more
    double word, word_mesh;       // per million: 4 bytes put together from words that lie otherwise, a 16-byte word on a mesh
};
constexpr PhaseCosts kPhaseCosts[2] = {{2.42, 6.12, 1.133, 1.413, 0.237, 1.448, 0.829, 0.997, 0.218, 0.901},
                                       {2.52, 2.76, 0.936, 0.883, 0.008, 0.026, 0.004, 0.228, 1.103, 0.529}};

// Send and receive buffers, as tiles go through them.
double memory_time(const Request &r)
{
    const bool allgather = r.kind == ISO_KIND_ALLGATHER;
    const TileCosts &k = kTileCosts[allgather];
    const double bytes = (double)r.stats.bytes_min / 2.0, P = (double)r.comm->P;
    double sent = 0, received = 0, cut = 0;  // sectors of a process
    for (const Part &p : r.parts) {
        if (p.src_buf == ISO_BUF_SEND) sent += (double)((p.src_off % 32 + p.len + 31) / 32);
        if (p.dst_buf != ISO_BUF_RECV) continue;
        received += (double)((p.dst_off % 32 + p.len + 31) / 32);
        cut += (p.dst_off % 32 != 0) + ((p.dst_off + p.len) % 32 != 0);
    }
    if (allgather) {  // (neighbouring blocks of the own receive buffer are stored together)
        received = bytes / 32.0 / P;
        cut = std::min(cut, received);
    }
    return 1e-6 * P * (k.sector * (sent + received) + std::max(0.0, 1.0 - 8e6 / std::max(1.0, bytes)) * (k.cut * cut + k.late * received));
}

double time_in_tiles(const Request &r, const TilesPlan &F, double memory)
{
    const TileCosts &k = kTileCosts[r.kind == ISO_KIND_ALLGATHER];
    const Residency on(F.outer * F.intervals, (int64_t)F.smem, F.threads, r.sm_count);
    const double warps = (double)(on.at_once * F.threads / 32);
    double loads = 0, moves = 0, units = 0;
    for (const TileGroup &g : F.groups) {  // (as upload_tiles deals them to threads)
        const int64_t passes = (g.n + F.threads - 1) / F.threads, owned = (g.n + passes - 1) / passes, slots = F.threads / owned;
        const int64_t at_a_time = F.unit == 0 || (F.mesh && F.unit == 16) ? 2 : 4, each = (F.rows_per_tile + slots - 1) / slots;
        const double chains = (double)(passes * ((each + at_a_time - 1) / at_a_time));
        if (g.kind == TILE_DELIVER) loads += chains;
        else if (g.kind != TILE_FETCH) moves += chains;
        units += (g.width == 16 ? k.unit16 : (F.unit == 0 ? k.unit_mixed : k.unit_one)) * (double)g.n;
    }
    if (F.mesh) units += k.partner * (double)F.shifts.size();
    const double latency = (double)on.turns * (k.turn + k.load * loads + k.move * moves);
    const double table = F.units_at ? 0.0 : k.table * (double)F.units.size();
    const double issue = 1e-3 * (double)on.per_sm * ((double)F.rows_per_tile * units + table) * (1.0 + k.warps / warps);
    return latency + std::pow(std::pow(issue, k.power) + std::pow(memory, k.power), 1.0 / k.power);
}

double time_in_phases(const Request &r, bool mesh, bool mixed)
{
    const PhaseCosts &k = kPhaseCosts[r.kind == ISO_KIND_ALLGATHER];
    const int64_t stride[3] = {r.send_stride, r.recv_stride, r.inter_stride};
    int64_t ends = 0, put_together = 0, words = 0;
    for (const Part &p : r.parts) {
        ends += (p.dst_off % 16 != 0) + ((p.dst_off + p.len) % 16 != 0);
        if (alignment16((p.src_off - p.dst_off) | stride[p.src_buf] | stride[p.dst_buf]) == 16) words += (p.dst_off % 16 + p.len + 15) / 16;
        else put_together += (p.dst_off % 4 + p.len + 3) / 4;
    }
    const double P = 1e-6 * (double)r.comm->P, copy = 1.0 / 6.5e6;
    return k.phase * r.stats.phases + k.launch * ((double)r.launches.size() - r.stats.phases) +
           copy * ((k.moved + (mixed ? k.mixed : 0.0)) * (double)r.stats.bytes_moved + k.bulk * (double)r.stats.bulk_bytes) +
           P * (k.block * (double)r.parts.size() + (k.end + (mesh ? k.end_mesh : 0.0)) * (double)ends + k.word * (double)put_together +
                (mesh ? k.word_mesh * (double)words : 0.0));
}

}  // namespace

void plan_tiles(Request &r)
{
    const Comm &c = *r.comm;
    TilesPlan &F = r.tiles;
    F = TilesPlan{};
    if (r.knobs.tiles == 0 || r.alg != ISO_ALG_COMBINING || r.fusion < 1 || r.layout != ISO_LAYOUT_PACKED || r.stats.phases < 2) return;
    // (What the library runs as two chains of slabs keeps them.  The faster way is the one or the other, in microseconds, chains and tiles:
    // 256x256 with 24 blocks of 512 bytes 328 and 258, of 2 KB 1348 and 1526, 48^3 with 26 of 64 bytes 127 and 76, 40^3 with 7 of
    // 500 bytes 203 and 288; the estimates below have not been fitted to such calls.)
    if (execution_asked_for(r) || r.chains > 1) return;
    const bool long_launches = (double)r.stats.bytes_moved / 2.0 > 2.0 * kSlabLaunchBytes * (double)r.launches.size();
    if ((r.slab_request == 1 || r.chains_request == 1) && r.kind != ISO_KIND_ALLGATHER && long_launches) return;  // (would be such a call)
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
    const bool forced = r.knobs.tiles >= 1;
    bool mesh = false;
    for (int j = 0; j < c.d; ++j) mesh = mesh || !c.periodic[j];
    const double memory = memory_time(r);
    // (less than any plan's estimate against more than that of the phases)
    if (!forced && kTileCosts[r.kind == ISO_KIND_ALLGATHER].turn + memory >= time_in_phases(r, mesh, true)) return;
    if (!build_plan(r, false, F)) return;
    double in_tiles = time_in_tiles(r, F, memory);
    if (mixed_widths(r)) {
        // What only passes from a send to a receive buffer may go through places too: the copies to a place are asynchronous, so
        // that the copies of several widths wait for memory once and not one after the other.  It costs places, and so rows per
        // tile: irregular sizes to 45 neighbours on 40x51 19.6 -> 14.1 microseconds, 164-byte blocks of 8 on a 39x51 mesh 4.9 -> 3.7,
        // but 41-byte blocks of 8 on 355x292 36.4 -> 50.5.  Of 3183 such calls five in six are staged; 255 would be 5 % faster the
        // other way, 36 15 % (by the bytes of the call, as before: 675 and 198).
        TilesPlan S;
        double t;
        if (r.knobs.tiles != 3 && build_plan(r, true, S) && ((t = time_in_tiles(r, S, memory)) < 1.1 * in_tiles || r.knobs.tiles == 2)) {
            F = std::move(S);
            in_tiles = t;
        }
    }
    F.on = forced || in_tiles < time_in_phases(r, F.mesh, F.unit == 0);
    if (!F.on) F = TilesPlan{};
}

}  // namespace iso
