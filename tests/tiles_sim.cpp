// Schedules whose phases run tile by tile in one launch (csrc/iso_tiles.cpp), executed on host memory
// the way the kernel does it, against the schedule's parts executed phase by phase: random tori, meshes,
// neighbourhoods, block sizes, displacements and buffer alignments.  Prints the number of plans compared.
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <random>
#include <set>

#include "iso_internal.h"

using namespace iso;

namespace {

using Bytes = std::vector<unsigned char>;

int64_t wrapped(const Comm &c, int64_t rank, const int *shift)  // source rank, or -1 outside a mesh
{
    int64_t r = 0;
    for (int j = 0; j < c.d; ++j) {
        int64_t x = rank / c.rank_stride[j] % c.dims[j] - shift[j];
        if (c.periodic[j]) x = (x % c.dims[j] + c.dims[j]) % c.dims[j];
        if (x < 0 || x >= c.dims[j]) return -1;
        r += x * c.rank_stride[j];
    }
    return r;
}

Bytes by_phases(const Request &r, const Bytes &send)
{
    const Comm &c = *r.comm;
    Bytes buf[3] = {send, Bytes(c.P * r.recv_stride, 0xA5), Bytes(c.P * r.inter_stride, 0x5A)};
    const int64_t stride[3] = {r.send_stride, r.recv_stride, r.inter_stride};
    for (const Part &p : r.parts)
        for (int64_t x = 0; x < c.P; ++x) {
            bool there = true;
            for (int j = 0; j < c.d; ++j) {
                const int64_t y = x / c.rank_stride[j] % c.dims[j] - p.check[j];
                if (!c.periodic[j]) there = there && y >= 0 && y < c.dims[j];
            }
            const int64_t s = there ? wrapped(c, x, p.shift) : -1;
            if (s >= 0)
                std::memcpy(&buf[p.dst_buf][x * stride[p.dst_buf] + p.dst_off], &buf[p.src_buf][s * stride[p.src_buf] + p.src_off], p.len);
        }
    return buf[1];
}

void require(bool ok, const char *what)
{
    if (ok) return;
    std::printf("failed: %s\n", what);
    std::exit(1);
}

Bytes by_tiles(const Request &r, const Bytes &send)
{
    const Comm &c = *r.comm;
    const TilesPlan &F = r.tiles;
    Bytes recv(c.P * r.recv_stride, 0xA5);
    std::set<int64_t> seen;
    for (int64_t tile = 0; tile < F.outer * F.intervals; ++tile) {
        const int64_t outer = tile / F.intervals, interval = tile % F.intervals;
        const int64_t width = std::min(F.width, F.inner - interval * F.width), rows = F.middle * width;
        require(rows > 0 && rows <= F.rows_per_tile, "rows of a tile");
        std::vector<int64_t> rank(rows);
        for (int64_t j = 0; j < rows; ++j) {
            rank[j] = outer * F.middle * F.inner + interval * F.width + j / width * F.inner + j % width;
            require(seen.insert(rank[j]).second, "a process in two tiles");
        }
        auto partner = [&](const TileShift &sh, int64_t j) -> int64_t {
            int64_t at = sh.between ? j : rank[j];
            for (size_t k = 0; k < F.coords.size(); ++k) {
                const int dim = F.coords[k];
                const int64_t x = rank[j] / c.rank_stride[dim] % c.dims[dim];
                const int64_t step = sh.between ? c.rank_stride[dim] / F.inner * width : c.rank_stride[dim];
                if (sh.c[k]) {
                    at -= sh.c[k] * step;
                    if (sh.wraps[k]) at += x < sh.c[k] ? c.dims[dim] * step : 0;
                    else if (x - sh.c[k] < 0 || x - sh.c[k] >= c.dims[dim]) return -1;
                }
                if (!sh.wraps[k] && (x - sh.check[k] < 0 || x - sh.check[k] >= c.dims[dim])) return -1;
            }
            return at;
        };
        Bytes places(F.rows_per_tile * F.place_stride + 1, 0x33);
        uint32_t stage = 0;
        Bytes before = places;  // what a stage reads, no group of it has written
        for (const TileGroup &g : F.groups) {
            require(g.stage >= stage && g.first + g.n <= F.units.size(), "order of the groups");
            if (g.stage != stage) before = places;
            stage = g.stage;
            for (uint32_t u = g.first; u < g.first + g.n; ++u) {
                const TileUnit &t = F.units[u];
                require(g.width == 0 ? t.width < 16 : t.width == g.width, "width");
                require(g.kind != TILE_FETCH || t.width >= 4, "asynchronous copies");
                for (int64_t j = 0; j < rows; ++j) {
                    const int64_t p = partner(F.shifts[t.shift], j);
                    if (p < 0) continue;
                    const bool global = g.kind == TILE_FETCH || g.kind == TILE_DELIVER;
                    const int64_t row = g.kind == TILE_FORWARD ? j : p;
                    require(global ? p < c.P && t.src_off + t.width <= r.send_stride : row < rows && t.src_off + t.width <= F.place_stride, "source");
                    const unsigned char *from = global ? &send[p * r.send_stride + t.src_off] : &before[row * F.place_stride + t.src_off];
                    const uintptr_t src_at = global ? (uintptr_t)r.send + p * r.send_stride + t.src_off : t.src_off;
                    require(src_at % t.width == 0, "alignment of a source");
                    if (g.kind != TILE_FORWARD && t.place_dst >= 0) {
                        require(t.place_dst + t.width <= F.place_stride && t.place_dst % t.width == 0, "place");
                        std::memcpy(&places[j * F.place_stride + t.place_dst], from, t.width);
                    }
                    if (t.recv_dst >= 0) {
                        const int64_t to = (g.kind == TILE_FORWARD ? p : rank[j]) * r.recv_stride + t.recv_dst;
                        require(t.recv_dst + t.width <= r.recv_stride && ((uintptr_t)r.recv + to) % t.width == 0, "receive buffer");
                        std::memcpy(&recv[to], from, t.width);
                    }
                }
            }
        }
    }
    require((int64_t)seen.size() == c.P, "every process in a tile");
    return recv;
}

// Calls read from standard input, a line each: kind, fusion level, d, the sides, whether each wraps, s, the vectors, the
// blocks' bytes.  Prints what the library chooses: the bytes of a row's places, or 0 where it does not run in tiles.
int choices()
{
    Comm c;
    Request r;
    while (std::scanf("%d %d %d", &r.kind, &r.fusion, &c.d) == 3) {
        auto number = [] {
            int x = 0;
            require(std::scanf("%d", &x) == 1, "a number");
            return x;
        };
        c.P = 1;
        for (int j = 0; j < c.d; ++j) c.dims[j] = number();
        for (int j = 0; j < c.d; ++j) c.periodic[j] = number();
        for (int j = c.d - 1; j >= 0; --j) c.rank_stride[j] = c.P, c.P *= c.dims[j];
        r.s = c.s = number();
        for (int k = 0; k < c.s * c.d; ++k) c.coords.push_back(number());
        int64_t at = 0;
        for (int i = 0; i < c.s; ++i) {
            r.len.push_back(number());
            r.sdispl.push_back(r.kind == ISO_KIND_ALLGATHER ? 0 : at);
            r.rdispl.push_back(at);
            at += r.len.back();
        }
        if (r.kind == ISO_KIND_ALLTOALLV) at = (at + 15) / 16 * 16;
        r.send_stride = r.kind == ISO_KIND_ALLGATHER ? r.len[0] : at;
        r.recv_stride = at;
        r.comm = &c;
        r.send = reinterpret_cast<const unsigned char *>((uintptr_t)4096);
        r.recv = reinterpret_cast<unsigned char *>((uintptr_t)1 << 40);
        default_dimension_order(r);
        require(build_schedule(r) == ISO_SUCCESS && lower_schedule(r, (uintptr_t)r.send, (uintptr_t)r.recv, 0) == ISO_SUCCESS, "schedule");
        plan_tiles(r);
        std::printf("%lld\n", r.tiles.on ? (long long)r.tiles.place_stride : 0LL);
        c = Comm();
        r = Request();
    }
    return 0;
}

// Sides above 65 535: on a mesh, where coordinates are kept in 16 bits, they stay out of tiles.
void long_sides()
{
    for (int mesh = 0; mesh < 2; ++mesh) {
        Comm c;
        c.d = 2;
        c.dims[0] = 70001, c.dims[1] = 3;
        c.P = 3 * 70001;
        c.rank_stride[0] = 3, c.rank_stride[1] = 1;
        c.periodic[0] = !mesh, c.periodic[1] = 1;
        c.coords = {-1, 1, 2, 0, 1, -1};
        Request r;
        r.comm = &c;
        r.s = c.s = 3;
        r.len = {16, 16, 16};
        r.sdispl = r.rdispl = {0, 16, 32};
        r.send_stride = r.recv_stride = 48;
        r.send = reinterpret_cast<const unsigned char *>((uintptr_t)4096);
        r.recv = reinterpret_cast<unsigned char *>((uintptr_t)1 << 40);
        r.knobs.tiles = 1;
        require(build_schedule(r) == ISO_SUCCESS && lower_schedule(r, (uintptr_t)r.send, (uintptr_t)r.recv, 0) == ISO_SUCCESS, "schedule");
        plan_tiles(r);
        require(r.tiles.on == !mesh, "long sides");
        Bytes send(c.P * r.send_stride);
        for (size_t k = 0; k < send.size(); ++k) send[k] = (unsigned char)(k * 2654435761u >> 13);
        if (r.tiles.on) require(by_tiles(r, send) == by_phases(r, send), "long sides, result");
    }
}

}  // namespace

int main(int argc, char **argv)
{
    if (argc > 1 && std::strcmp(argv[1], "choices") == 0) return choices();
    long_sides();
    std::mt19937 rng(argc > 1 ? std::atoi(argv[1]) : 1);
    auto pick = [&](int lo, int hi) { return (int)(rng() % (unsigned)(hi - lo + 1)) + lo; };
    int compared = 0;
    for (int trial = 0; trial < 400; ++trial) {
        Comm c;
        c.d = pick(2, 5);
        for (int j = 0; j < c.d; ++j) c.dims[j] = pick(1, c.d == 2 ? 12 : (c.d == 3 ? 7 : 4));
        const bool mesh = pick(0, 3) == 0;
        for (int j = c.d - 1; j >= 0; --j) {
            c.rank_stride[j] = c.P;
            c.P *= c.dims[j];
            c.periodic[j] = mesh ? pick(0, 1) : 1;
        }
        c.s = pick(1, 20);
        for (int k = 0; k < c.s * c.d; ++k) c.coords.push_back(pick(-3, 3));
        if (c.s > 2)
            for (int j = 0; j < c.d; ++j) {
                if (pick(0, 1)) c.coords[j] = 0;               // the zero vector, sometimes
                c.coords[c.d + j] = c.coords[2 * c.d + j];     // a repeated one
            }
        Request r;
        r.comm = &c;
        r.s = c.s;
        r.kind = pick(0, 2);
        r.fusion = pick(1, 3);
        const int sizes[] = {1, 2, 3, 4, 7, 8, 12, 13, 16, 24, 48, 64, 100, 131};
        const int m = sizes[pick(0, 13)];
        int64_t at_s = 0, at_r = 0;
        for (int i = 0; i < c.s; ++i) {
            const int64_t len = r.kind == ISO_KIND_ALLGATHER || pick(0, 1) ? m : (r.kind == ISO_KIND_ALLTOALL ? m : sizes[pick(0, 13)]);
            r.len.push_back(len);
            r.sdispl.push_back(r.kind == ISO_KIND_ALLGATHER ? 0 : at_s);
            r.rdispl.push_back(at_r);
            at_s += len;
            at_r += len + (r.kind == ISO_KIND_ALLTOALLV ? pick(0, 5) : 0);
        }
        r.send_stride = r.kind == ISO_KIND_ALLGATHER ? m : at_s;
        r.recv_stride = at_r;
        if (r.kind == ISO_KIND_ALLTOALLV && pick(0, 1)) r.send_stride = (at_s + 15) / 16 * 16, r.recv_stride = (at_r + 15) / 16 * 16;
        const int leads[] = {0, 0, 16, 1, 4, 8, 2};
        r.send = reinterpret_cast<const unsigned char *>((uintptr_t)4096 + leads[pick(0, 6)]);  // (only their alignment is looked at)
        r.recv = reinterpret_cast<unsigned char *>((uintptr_t)8192 + leads[pick(0, 6)]);
        r.knobs.tiles = pick(1, 3);
        default_dimension_order(r);
        if (build_schedule(r) != ISO_SUCCESS) require(false, "schedule");
        if (lower_schedule(r, (uintptr_t)r.send, (uintptr_t)r.recv, 0) != ISO_SUCCESS) require(false, "lowering");
        plan_tiles(r);
        if (!r.tiles.on) continue;
        Bytes send(c.P * r.send_stride);
        for (unsigned char &b : send) b = (unsigned char)rng();
        if (by_tiles(r, send) != by_phases(r, send)) {
            std::printf("trial %d: d %d kind %d fusion %d m %d mesh %d\n", trial, c.d, r.kind, r.fusion, m, (int)mesh);
            return 1;
        }
        ++compared;
    }
    std::printf("%d\n", compared);
    return 0;
}
