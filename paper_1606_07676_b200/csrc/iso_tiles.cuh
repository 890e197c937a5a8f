// Device code for schedules whose intermediate blocks fit in shared memory (sm_100a): all phases in one
// launch.
//
// A block's first hop reads a send buffer and its last one writes a receive buffer; only the hops in
// between go from one process's intermediate storage to another's.  So a CTA acts for a tile of processes that is complete along the dimensions of those middle hops and of any width
// along the others: it fetches what the first hops bring to the tile's processes into places in shared
// memory, runs the middle phases between the places with a barrier of the CTA as the ordering point, and
// sends the last hops from the places to the receive buffers of the processes they are bound for.  In two dimensions there are no
// middle hops at all.  Every hop is made, every phase of a block after the one before it; but the
// intermediate blocks never reach device memory, and there is one launch instead of one per phase.
//
// What bounds it.  Small calls: the latency of one chain of a global load, a shared-memory hop per phase and a
// global store, about a microsecond beside the launch, where a launch per phase costs 2.6 microseconds each
// (8^2 with 8-byte blocks 5.2 -> 3.1, 11x9x8 with 30 4-byte blocks 7.1 -> 3.1, 20x27 with 48 irregular ones 8.3 ->
// 6.8).  Large ones: the instructions per unit and row, 1.5 of four a cycle, with 0.42 of the warps there and most of them waiting for
// memory, shared memory or a barrier (32^3 with 26 64-byte blocks 35.8 -> 27.1, DRAM traffic 174 -> 65 MB during the kernel; allgather there
// 19.0 -> 13.5; 17x12x10x17 with 15 88-byte blocks 82 -> 34).  Why a thread owns a unit position and the partners of the
// rows are tabulated: with a division per row and dimension and a wrap test per unit and row the
// same 32^3 took 73, with coordinates in a table 30.  Clusters that share a tile (distributed shared memory) were
// slower than a launch per phase: 64x64x32 with 30 irregular blocks 2750 against 1300.
#pragma once

#include "iso_kernels.cuh"

namespace iso {

struct TileGroupDev {
    uint32_t kind, width;  // TILE_FETCH ..., bytes of its units (0: narrow ones)
    uint32_t first, n;     // units
    uint32_t owned, slots; // unit positions that threads own at a time, rows worked on at a time
    FastDivDev div_owned;
    uint32_t barrier;      // the next group reads places that this one or those before it have filled
};

struct TilesDev {
    const TileUnit *units;
    const TileShift *shifts;
    const unsigned char *send;
    unsigned char *recv;
    uint32_t send_stride, recv_stride;
    uint32_t n_units, n_shifts;
    uint32_t n_tiles, n_intervals;      // a tile is an interval of the inner ranks of one outer index
    uint32_t middle, inner, width;      // processes along the complete dimensions, behind them, and of an interval
    uint32_t rows_per_tile;             // (the last tile of an outer index may be narrower)
    uint32_t place_stride;              // bytes of a row's places in shared memory
    uint32_t moved_at, coords_at, units_at;  // where the rows' partners, their coordinates and (not 0) the unit table lie behind them
    uint32_t n_coords;                  // coordinates per row
    uint32_t n_groups;
    TileGroupDev group[kTileGroups];
    FastDivDev div_intervals, div_width, div_last_width, div_rows_per_tile;
    uint32_t size[ISO_MAX_DIMS], stride[ISO_MAX_DIMS], row_stride[ISO_MAX_DIMS];  // of the dimensions whose coordinates are kept; in
                                                                                 // ranks and in rows of a tile of width 1
    FastDivDev div_stride[ISO_MAX_DIMS], div_size[ISO_MAX_DIMS];
};

// A unit of W bytes from and to shared memory.
template <int W> __device__ __forceinline__ typename VecOf<W>::type load_shared(uint32_t a);
template <> __device__ __forceinline__ uint4 load_shared<16>(uint32_t a)
{
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a) : "memory");
    return v;
}
template <> __device__ __forceinline__ uint2 load_shared<8>(uint32_t a)
{
    uint2 v;
    asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(a) : "memory");
    return v;
}
template <> __device__ __forceinline__ uint32_t load_shared<4>(uint32_t a)
{
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
    return v;
}
template <> __device__ __forceinline__ uint16_t load_shared<2>(uint32_t a)
{
    uint16_t v;
    asm volatile("ld.shared.u16 %0, [%1];" : "=h"(v) : "r"(a) : "memory");
    return v;
}
template <> __device__ __forceinline__ uint8_t load_shared<1>(uint32_t a)
{
    uint32_t v;
    asm volatile("ld.shared.u8 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
    return (uint8_t)v;
}
__device__ __forceinline__ void store_shared(uint32_t a, const uint4 &v)
{
    asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(a), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}
__device__ __forceinline__ void store_shared(uint32_t a, const uint2 &v)
{
    asm volatile("st.shared.v2.u32 [%0], {%1, %2};" ::"r"(a), "r"(v.x), "r"(v.y) : "memory");
}
__device__ __forceinline__ void store_shared(uint32_t a, uint32_t v) { asm volatile("st.shared.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory"); }
__device__ __forceinline__ void store_shared(uint32_t a, uint16_t v) { asm volatile("st.shared.u16 [%0], %1;" ::"r"(a), "h"(v) : "memory"); }
__device__ __forceinline__ void store_shared(uint32_t a, uint8_t v)
{
    asm volatile("st.shared.u8 [%0], %1;" ::"r"(a), "r"((uint32_t)v) : "memory");
}
template <int W> __device__ __forceinline__ void copy_async_at(uint32_t place, const unsigned char *src)
{
    if (W == 16) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(place), "l"(src) : "memory");
    else asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(place), "l"(src), "n"(W) : "memory");
}

// The same for units of W bytes, or (W is kNarrow) of `width`: 8, 4, 2 or 1.
constexpr int kNarrow = 0;
template <int W> struct TileVec { using type = typename VecOf<W>::type; };
template <> struct TileVec<kNarrow> { using type = uint2; };
template <int W> __device__ __forceinline__ typename TileVec<W>::type unit_from_place(uint32_t a, uint32_t width)
{
    if constexpr (W != kNarrow) {
        return load_shared<W>(a);
    } else {
        uint2 v = make_uint2(0, 0);
        if (width == 8) v = load_shared<8>(a);
        else if (width == 4) v.x = load_shared<4>(a);
        else if (width == 2) v.x = load_shared<2>(a);
        else v.x = load_shared<1>(a);
        return v;
    }
}
template <int W> __device__ __forceinline__ void unit_to_place(uint32_t a, const typename TileVec<W>::type &v, uint32_t width)
{
    if constexpr (W != kNarrow) {
        store_shared(a, v);
    } else {
        if (width == 8) store_shared(a, v);
        else if (width == 4) store_shared(a, v.x);
        else if (width == 2) store_shared(a, (uint16_t)v.x);
        else store_shared(a, (uint8_t)v.x);
    }
}
template <int W> __device__ __forceinline__ typename TileVec<W>::type unit_from_device(const unsigned char *p, uint32_t width)
{
    if constexpr (W != kNarrow) {
        return *reinterpret_cast<const typename TileVec<W>::type *>(p);
    } else {
        uint2 v = make_uint2(0, 0);
        if (width == 8) v = *reinterpret_cast<const uint2 *>(p);
        else if (width == 4) v.x = *reinterpret_cast<const uint32_t *>(p);
        else if (width == 2) v.x = *reinterpret_cast<const uint16_t *>(p);
        else v.x = *p;
        return v;
    }
}
template <int W> __device__ __forceinline__ void unit_to_device(unsigned char *p, const typename TileVec<W>::type &v, uint32_t width)
{
    if constexpr (W != kNarrow) {
        *reinterpret_cast<typename TileVec<W>::type *>(p) = v;
    } else {
        if (width == 8) *reinterpret_cast<uint2 *>(p) = v;
        else if (width == 4) *reinterpret_cast<uint32_t *>(p) = v.x;
        else if (width == 2) *reinterpret_cast<uint16_t *>(p) = (uint16_t)v.x;
        else *p = (unsigned char)v.x;
    }
}

constexpr uint32_t kNobody = 0xffffffffu;  // no partner: outside a mesh

// What a thread needs to know about the unit it moves, beside the group's kind.
struct TileWalk {
    uint32_t src_off;
    int place_dst, recv_dst;
    uint32_t width;
    uint32_t partner;  // shared-memory address of the partner of the thread's first row
    uint32_t own;      // of that row's rank
    uint32_t row;      // that row
    int left;          // rows from it to the end of the CTA's
    uint32_t step;     // to the thread's next row
};

// Nothing but a place to fill: the copies of all rows are in flight at once.
template <int W, bool MESH>
__device__ __forceinline__ void fetch_tile(const TilesDev &L, uint32_t places_at, const TileWalk &t)
{
    const unsigned char *const src = L.send + t.src_off;
    const uint32_t place_step = t.step * L.place_stride;
    uint32_t partner = t.partner, to = places_at + t.row * L.place_stride + (uint32_t)t.place_dst;
#pragma unroll 4
    for (int left = t.left; left > 0; left -= (int)t.step) {
        const uint32_t r = load_shared<4>(partner);
        if (!MESH || r != kNobody) {
            const unsigned char *const from = src + (unsigned long long)r * L.send_stride;
            if constexpr (W != kNarrow) copy_async_at<W>(to, from);
            else if (t.width == 8) copy_async_at<8>(to, from);
            else copy_async_at<4>(to, from);  // (asynchronous copies move at least 4 bytes; narrower units are delivered)
        }
        partner += 4 * t.step;
        to += place_step;
    }
}

// The other kinds of a group's units, as one thread moves them.  What a row costs here is what the kernel costs: a
// table entry, an address, a load and a store.
template <int W, int R, uint32_t KIND, bool MESH>
__device__ __forceinline__ void walk_tile(const TilesDev &L, uint32_t places_at, const TileWalk &t)
{
    using V = typename TileVec<W>::type;
    const uint32_t place_step = t.step * L.place_stride;
    const unsigned char *const src = L.send + t.src_off;
    unsigned char *const dst = L.recv + t.recv_dst;
    uint32_t partner = t.partner, own = t.own;
    uint32_t from = places_at + t.row * L.place_stride + t.src_off, to = places_at + t.row * L.place_stride + (uint32_t)t.place_dst;
    const uint32_t from0 = places_at + t.src_off;
    int left = t.left;
    for (; left > 0; left -= R * (int)t.step) {
        V v[R];
        uint32_t r[R];
#pragma unroll
        for (int i = 0; i < R; ++i) {
            r[i] = kNobody;
            if (left > i * (int)t.step) r[i] = load_shared<4>(partner + 4 * i * t.step);
        }
#pragma unroll
        for (int i = 0; i < R; ++i) {
            const bool there = MESH ? r[i] != kNobody : left > i * (int)t.step;
            if (there) {
                if (KIND == TILE_DELIVER) {
                    v[i] = unit_from_device<W>(src + (unsigned long long)r[i] * L.send_stride, t.width);
                } else if (KIND == TILE_FORWARD) {
                    v[i] = unit_from_place<W>(from + i * place_step, t.width);
                } else {
                    v[i] = unit_from_place<W>(from0 + r[i] * L.place_stride, t.width);
                }
            }
        }
#pragma unroll
        for (int i = 0; i < R; ++i) {
            const bool there = MESH ? r[i] != kNobody : left > i * (int)t.step;
            if (there) {
                if (KIND == TILE_FORWARD) {
                    unit_to_device<W>(dst + (unsigned long long)r[i] * L.recv_stride, v[i], t.width);
                } else {
                    if (t.place_dst >= 0) unit_to_place<W>(to + i * place_step, v[i], t.width);
                    if (t.recv_dst >= 0)
                        unit_to_device<W>(dst + (unsigned long long)load_shared<4>(own + 4 * i * t.step) * L.recv_stride, v[i], t.width);
                }
            }
        }
        partner += 4 * R * t.step;
        own += 4 * R * t.step;
        from += R * place_step;
        to += R * place_step;
    }
}

template <int W, int R, bool MESH>
__device__ __forceinline__ void walk_group(const TilesDev &L, uint32_t kind, uint32_t places_at, const TileWalk &t)
{
    if (kind == TILE_FETCH) {
        fetch_tile<W, MESH>(L, places_at, t);
    } else if (kind == TILE_DELIVER) {
        walk_tile<W, R, TILE_DELIVER, MESH>(L, places_at, t);
    } else if (kind == TILE_BETWEEN) {
        walk_tile<W, R, TILE_BETWEEN, MESH>(L, places_at, t);
    } else {
        walk_tile<W, R, TILE_FORWARD, MESH>(L, places_at, t);
    }
}

// W: bytes of every unit, 0: 16, or fewer in some groups.  MESH: some dimensions are not periodic, and a row may
// have no partner for a shift.
// A thread owns a unit position of a group (a kind of move, 16 bytes or fewer) and walks down the rows (processes) of
// its CTA.  Which process a row's bytes come from or go to depends on the shift and the row alone: the CTA
// tabulates it for every tile.
template <int W, bool MESH>
__global__ void __launch_bounds__(kTileThreads, 2) iso_gather_tiles(const __grid_constant__ TilesDev L)
{
    extern __shared__ __align__(128) unsigned char places[];
    const uint32_t nthr = blockDim.x;
    const uint32_t places_at = (uint32_t)__cvta_generic_to_shared(places);
    uint32_t *const moved = reinterpret_cast<uint32_t *>(places + L.moved_at);  // [shift][row], shift 0: the row itself
    uint16_t *const coords = reinterpret_cast<uint16_t *>(places + L.coords_at);
    // the unit table (nothing that kernels produce): a copy in shared memory, or where it lies
    const uint4 *const table = reinterpret_cast<const uint4 *>(L.units);
    const bool copied = L.units_at != 0;
    if (copied)
        for (uint32_t k = threadIdx.x; k < L.n_units; k += nthr) *reinterpret_cast<uint4 *>(places + L.units_at + 16 * k) = __ldg(table + k);
    bool ordered = false;  // behind the previous kernel
    for (uint32_t tile = blockIdx.x; tile < L.n_tiles; tile += gridDim.x) {
        const uint32_t outer = fastdiv(L.div_intervals, tile), interval = tile - outer * L.n_intervals;
        const bool last = interval + 1 == L.n_intervals;
        const uint32_t width = last ? L.inner - interval * L.width : L.width;
        const uint32_t n_rows = L.middle * width;
        const uint32_t rank0 = outer * (L.middle * L.inner) + interval * L.width;
        auto rank_of = [&](uint32_t j) -> uint32_t {
            const uint32_t m = last ? fastdiv(L.div_last_width, j) : fastdiv(L.div_width, j);
            return rank0 + m * L.inner + (j - m * width);
        };
        auto coordinate = [&](uint32_t k, uint32_t r) -> uint32_t {
            const uint32_t t = fastdiv(L.div_stride[k], r);
            return t - fastdiv(L.div_size[k], t) * L.size[k];
        };
        if (!MESH) {
            // (a row's coordinates are worked out where a shift asks for them: one or two of them mostly, and nothing waits for a
            // table of them)
            for (uint32_t e = threadIdx.x; e < L.n_shifts * L.rows_per_tile; e += nthr) {
                const uint32_t s = fastdiv(L.div_rows_per_tile, e), j = e - s * L.rows_per_tile;
                if (j >= n_rows) continue;
                const uint32_t own = rank_of(j);
                const uint4 h = __ldg(reinterpret_cast<const uint4 *>(L.shifts + s));
                const uint32_t n = h.x & 0xffu;
                const bool between = (h.x & 0x100u) != 0;
                uint32_t r = between ? j : own;
                auto move = [&](uint32_t k, uint32_t c) {
                    const uint32_t step = between ? L.row_stride[k] * width : L.stride[k];
                    r -= c * step;
                    if (coordinate(k, own) < c) r += L.size[k] * step;
                };
                if (n > 2) {
                    for (uint32_t k = 0; k < L.n_coords; ++k) {
                        const uint32_t c = (uint32_t)__ldg(&L.shifts[s].c[k]);
                        if (c) move(k, c);
                    }
                } else {
                    if (n > 0) move((h.x >> 16) & 0xffu, h.y);
                    if (n > 1) move(h.x >> 24, h.z);
                }
                moved[e] = r;
            }
        } else {
            for (uint32_t j = threadIdx.x; j < n_rows; j += nthr) {
                const uint32_t r = rank_of(j);
                moved[j] = r;
                for (uint32_t k = 0; k < L.n_coords; ++k) coords[j * L.n_coords + k] = (uint16_t)coordinate(k, r);
            }
            __syncthreads();
            for (uint32_t e = threadIdx.x; e < (L.n_shifts - 1) * L.rows_per_tile; e += nthr) {
                const uint32_t s = fastdiv(L.div_rows_per_tile, e) + 1, j = e - (s - 1) * L.rows_per_tile;
                if (j >= n_rows) continue;
                const TileShift *const sh = L.shifts + s;
                const bool between = __ldg(&sh->between) != 0;
                uint32_t r = between ? j : moved[j];
                for (uint32_t k = 0; k < L.n_coords; ++k) {
                    const int c = __ldg(&sh->c[k]);
                    const int x = coords[j * L.n_coords + k];
                    bool there = true;
                    if (c) {
                        const uint32_t step = between ? L.row_stride[k] * width : L.stride[k];
                        r -= (uint32_t)c * step;
                        if (__ldg(&sh->wraps[k])) {
                            if (x < c) r += L.size[k] * step;
                        } else {
                            there = x - c >= 0 && x - c < (int)L.size[k];
                        }
                    }
                    const int y = x - __ldg(&sh->check[k]);
                    if (!there || y < 0 || y >= (int)L.size[k]) {
                        r = kNobody;
                        break;
                    }
                }
                moved[s * L.rows_per_tile + j] = r;
            }
        }
        __syncthreads();
        if (!ordered) {
            grid_dependency_wait();
            grid_launch_dependents();
            ordered = true;
        }
        for (uint32_t k = 0; k < L.n_groups; ++k) {
            const TileGroupDev &T = L.group[k];
            const uint32_t g = fastdiv(T.div_owned, threadIdx.x);
            if (g < T.slots && g < n_rows)
                for (uint32_t u = threadIdx.x - g * T.owned; u < T.n; u += T.owned) {
                    const uint4 a = copied ? load_shared<16>(places_at + L.units_at + 16 * (T.first + u)) : __ldg(table + (T.first + u));
                    TileWalk t;
                    t.src_off = a.x;
                    t.place_dst = (int)a.y;
                    t.recv_dst = (int)a.z;
                    t.own = places_at + L.moved_at + 4 * g;
                    t.partner = t.own + 4 * ((a.w & 0xffffffu) * L.rows_per_tile);
                    t.row = g;
                    t.left = (int)(n_rows - g);
                    t.step = T.slots;
                    t.width = a.w >> 24;
                    // (rows at a time: four, on a mesh two of 16 bytes, where four spill: 103 such calls of 8 microseconds and more in 0.81 of
                    // the time, an allgather of 96 bytes from 124 neighbours on 15x18x11 18.4 -> 11.2)
                    if (W != 0) walk_group<(W != 0 ? W : 16), (MESH && W == 16 ? 2 : 4), MESH>(L, T.kind, places_at, t);
                    else if (T.width == 16) walk_group<16, 2, MESH>(L, T.kind, places_at, t);
                    else if (!MESH && T.width == 8) walk_group<8, 2, MESH>(L, T.kind, places_at, t);  // (with it the mesh kernel spills: 126 -> 147)
                    else walk_group<kNarrow, 2, MESH>(L, T.kind, places_at, t);
                }
            if (T.barrier) {
                cp_async_commit();
                cp_async_wait<0>();
                __syncthreads();
            }
        }
        __syncthreads();  // the places are filled anew
    }
}

}  // namespace iso
