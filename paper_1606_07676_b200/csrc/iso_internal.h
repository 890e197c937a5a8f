// Internal host-side types of the isomorphic neighbourhood collectives library.
#pragma once

#include <cstdint>
#include <vector>

#include "iso.h"

namespace iso {

struct Comm {
    int refcount = 1;
    int d = 0;
    int s = 0;
    int dims[ISO_MAX_DIMS] = {0};
    int periodic[ISO_MAX_DIMS] = {0};
    int64_t P = 1;
    int64_t rank_stride[ISO_MAX_DIMS] = {0};  // ranks between neighbours along dimension j
    std::vector<int> coords;                  // s*d, as given by the caller
};

// One line of the executed schedule, before it is lowered to kernel launches.
struct Part {
    int phase = 0;
    int round = -1;
    int slot = 0;
    int src_buf = ISO_BUF_SEND;
    int dst_buf = ISO_BUF_RECV;
    int64_t src_off = 0;
    int64_t dst_off = 0;
    int64_t len = 0;
    int shift[ISO_MAX_DIMS] = {0};  // residue in [0,p_j) for periodic dimensions, signed for mesh ones
    int check[ISO_MAX_DIMS] = {0};  // mesh dimensions: process x takes part only if 0 <= x_j - check_j < p_j
};

// Exact unsigned 32-bit division by an invariant divisor (Granlund & Montgomery 1994,
// round-up method): q = (t + ((n - t) >> s1)) >> s2 with t = mulhi(m, n).
struct FastDiv {
    uint32_t m = 1, s1 = 0, s2 = 0, div = 1;
};
FastDiv make_fastdiv(uint32_t divisor);
inline uint32_t fastdiv_host(const FastDiv &f, uint32_t n)
{
    uint32_t t = (uint32_t)(((uint64_t)f.m * n) >> 32);
    return (t + ((n - t) >> f.s1)) >> f.s2;
}

// A part as one kernel launch sees it (after splitting into aligned pieces).
struct LoweredPart {
    Part p;            // offsets / len of this piece
    uint32_t first_unit = 0;
    uint32_t units = 0;
    int width = 16;    // bytes per unit of this piece (differs between pieces in a launch of mixed widths)
};

enum { KERNEL_VEC = 0, KERNEL_BULK = 1, KERNEL_FAN = 2 };

// Sender-side form of an allgather phase (Section III-B: a trie edge carries one block once):
// a parent block, read once from the process that holds it, and the places it is copied to.
struct FanDst {
    int buf = ISO_BUF_RECV;
    int64_t off = 0;
    int c = 0;  // the destination process is the source process shifted by +c along the phase's dimension, c in [0, p)
};
struct FanParent {
    int src_buf = ISO_BUF_SEND;
    int64_t src_off = 0;
    int64_t len = 0;
    std::vector<FanDst> dsts;  // at most kFanDsts
};
constexpr int kFanDsts = 4;  // destinations per descriptor; a parent with more is listed several times
constexpr int64_t kHybridMinBytes = 256;  // 16-byte-aligned pieces of a ragged row from which bulk copies take over
constexpr int kMaxOwnSlabs = 128;          // most slabs of dimension 0 the library chooses by itself
constexpr double kSlabLaunchBytes = 52e6;  // what one launch of a slab may write so that it and its reader share the L2
constexpr int kMaxVecUnits = 8192;  // unit positions per process in one vector launch
constexpr int kVecDepth = 8;        // cp.async ring slots per thread in the vector kernel
constexpr int kWideDepth = 12;      // the same in CTAs of more than 256 threads (one CTA per SM)
constexpr int kHybridDepth = 6;     // the same for the vector warps of a hybrid launch (most of the shared memory stages bulk copies)
constexpr size_t kHybridStageBytes = 128 * 1024;  // staging area of the bulk warps of a hybrid launch

// ---- launches of words (iso_words.cuh) ------------------------------------------------------
// Tables of a launch whose blocks are not made of whole, equally placed 16-byte units.  A chunk is
// what one warp moves per row (or group of rows): at most 32 aligned 16-byte words to load, and
// what they are stored as.

// One word to load, by lane.  In a whole or placed chunk (and in form 2) the lane may also store one.
struct alignas(16) LoadDev {
    long long src_term;      // rank_delta * source stride + offset of the block, or (with word 0) of the aligned word itself
                             // where that is the same place inside its word for all rows
    uint32_t len;            // bytes of the block (0: this lane loads nothing)
    int32_t word;            // index of this word, counted from the one that holds the byte at src_term
    int32_t c[ISO_MAX_DIMS]; // shift (non-periodic dimension: check value) along the launch's used dimensions
    long long dst_term;      // whole or placed chunk: the word, from the (aligned down) start of the row group; form 2: offset
                             // of the block
    uint8_t src_buf, dst_buf;
    uint8_t sub;             // which of the rows of the group
    uint8_t stores;          // whole or placed chunk, form 2: this lane stores a word
    uint8_t second, third;   // placed chunk: lanes that hold more bytes of the word (this lane itself: none)
    uint16_t mask;           // placed chunk: which bytes of the destination word this lane's word holds
};
static_assert(sizeof(LoadDev) == 64, "load descriptors are read as four 16-byte words");

// One aligned 4- or 8-byte word to store, put together from the chunk's loaded bytes.  A place counts
// from 16 bytes in front of the chunk's first slot, so that it is never negative.
struct alignas(8) FineDev {
    uint32_t a;  // place q0 (10 bits) and lane0 (5) of the first block, q1 (10) and lane1 (5) of the second:
                 // the byte of the block that falls on the word's byte 0, and a lane that loads the block
    uint32_t b;  // offset in units of 4 bytes behind the chunk's first word (16 bits), bytes from the first (4)
                 // and from the second block (4); no bytes: no word
};
// The same where more than two blocks meet in a 4-byte word: place (10) and lane (5) of every byte.
struct alignas(16) TinyDev {
    uint32_t a, b;  // bytes 0 and 1, bytes 2 and 3
    uint32_t off;   // offset in units of 4 bytes behind the chunk's first word
    uint32_t mask;
};

// How a chunk is stored.  WHOLE: every lane stores the word it has loaded.  PLACED: likewise, merged
// where need be with the words of one or two other lanes, every byte having the same place in both
// (for all rows).  ONE4, ONE8: 4- or 8-byte words, each out of one block.  TWO: 4-byte words out of one
// or two blocks.  TINY: likewise, byte by byte.
enum { CHUNK_WHOLE = 0, CHUNK_PLACED = 1, CHUNK_ONE4 = 2, CHUNK_ONE8 = 3, CHUNK_TWO = 4, CHUNK_TINY = 5 };

// Which warp does what: warp g of the grid works on entry g mod n, of the row groups dealt to it on
// those with index `turn` mod `turns`.  A chunk that costs more instructions per row has more entries.
struct alignas(16) EntryDev {
    uint32_t chunk, turn, turns;
    uint32_t first;      // index of the chunk's first FineDev or TinyDev (32 per pass)
    uint8_t passes;      // 32-word passes over its 4- or 8-byte words; placed chunk: most sources of a word
    uint8_t kind;        // CHUNK_*
    uint8_t dst_buf;
    uint8_t pad[5];
    long long dst_term;  // its first 4- or 8-byte word, from the (aligned down) start of the row group
};
static_assert(sizeof(EntryDev) == 32, "entries are read as two 16-byte words");

struct WordTables {
    int form = 0;          // 0: all alignments the same for every row, 1: not so, or a mesh, 2: long blocks of any alignment
    uint32_t rows_sub = 1; // forms 0, 1: rows described together (a row group)
    std::vector<LoadDev> loads;     // 32 per chunk
    std::vector<EntryDev> chunks;   // one per chunk (turn 0 of 1), before they are dealt to warps
    std::vector<FineDev> fine;
    std::vector<TinyDev> tiny;
    std::vector<EntryDev> entries;
};
constexpr int64_t kWordsLongBlock = 64;       // mean block length from which form 2 replaces form 1
constexpr int64_t kWordsMostGroup = 32 << 10; // bytes of a row group that the tables describe at most
constexpr int kWordsDepth = 16;               // words in flight per lane, as many as fit beside a coordinate table ...
constexpr int kWordsDepthCoded = 12;          // ... and where the codes of the stages have to fit into 64 bits
constexpr int kWordsThreads = 768;            // threads per SM, in one to three CTAs
constexpr int64_t kWordsSmallLaunch = 12 << 20;  // bytes up to which a launch of 16-byte units runs as words
constexpr int64_t kWordsScattered = 96 << 20;    // bytes from which one with scattered loads does
constexpr int kWordsPasses = 4;               // passes over a chunk's words at most
constexpr uint32_t kWordsPadFront = 16, kWordsPadBack = 48;  // shared memory around the ring that a shifted read may touch

struct LaunchPlan {
    int kernel = KERNEL_VEC;
    int width = 16;       // bytes per unit (vector kernel; 0: mixed, every piece has its own); chunk bytes (bulk kernel)
    int phase = 0;
    std::vector<LoweredPart> parts;
    uint32_t units_per_proc = 0;
    uint32_t uniform_units = 0;  // >0: every part has this many units
    int lookup_shift = 0;
    std::vector<uint16_t> lookup;  // unit >> lookup_shift -> index of the part holding that unit
    uint32_t chunk_units = 1;    // vector kernel: unit positions per row slot
    uint32_t rows_per_pass = 1;  // vector kernel: rows a CTA handles at the same time
    int tile_procs = 1;
    int threads = 256;
    int64_t grid = 0;
    size_t smem = 0;
    int n_used = 0;
    int used_dim[ISO_MAX_DIMS] = {0};
    int max_nnz = 0;       // most dimensions any one part shifts along
    bool compact = false;  // vector kernel: unit descriptors list only the shifted dimensions
    int64_t rows_hint = 0; // vector kernel: rows the grid holds at a time when CTAs cover whole rows (slab heuristic)
    int col_split = 1;     // vector kernel: column chunks of a row longer than a CTA, one CTA per chunk and row (1: none)
    std::vector<LaunchPlan> side;  // mixed-width vector launch: at most one bulk-copy plan for the long bodies of its rows,
                                   // run by one extra warp of the same CTAs
    bool words = false;           // vector launch whose blocks are not whole, equally placed 16-byte units
    WordTables tables;            // its tables (build_words)
    bool any_dims = false;        // without a coordinate table: the kernel for any number of dimensions
    std::vector<FanParent> fans;  // KERNEL_FAN: the launch as parents and their destinations (parts: the same copies, one per destination)
    // byte offsets of this launch's tables inside the request's device blob
    size_t parts_off = 0, lookup_off = 0, units_off = 0, fine_off = 0, tiny_off = 0, entries_off = 0;
};

// ---- all phases of a tile of processes in one launch (iso_tiles.cuh) ----------------------------
// One unit of a block's hop inside a process's payload.  A place is what a block with hops left (or a
// trie node with children) occupies in shared memory, the same for every row of a tile.
struct alignas(16) TileUnit {
    uint32_t src_off;                 // in the source process's send buffer (stage 0) or places
    int32_t place_dst, recv_dst;      // in the places, in the receive buffer (-1: not there)
    uint32_t shift : 24, width : 8;   // index of its shift, its bytes
};
static_assert(sizeof(TileUnit) == 16, "unit descriptors are read as 16-byte words");
// What is subtracted from a row's coordinates to find the process its bytes come from (or go to).  `c` along a periodic
// dimension in [0, p); `check` as in Part, for the row itself.
struct alignas(16) TileShift {
    uint32_t first_two;               // how many dimensions it moves along (8 bits), `between` (8), the first two of them (8 each)
    int32_t c_first, c_second;        // and the shifts along those
    int32_t between;                  // the partner is a row of the tile
    int32_t c[ISO_MAX_DIMS], check[ISO_MAX_DIMS];
    uint8_t wraps[ISO_MAX_DIMS];      // the dimension is periodic
    int32_t pad[2];
};
static_assert(sizeof(TileShift) == 16 + 9 * ISO_MAX_DIMS + 8, "compared byte by byte: no padding");
// What a group of units does.  FETCH: a send buffer's bytes to places, asynchronously.  DELIVER: likewise to the receive buffer
// (and places).  BETWEEN: from another row's places to the own ones (and the receive buffer).  FORWARD: from the own places to
// the receive buffer of another process.
enum : uint32_t { TILE_FETCH = 0, TILE_DELIVER = 1, TILE_BETWEEN = 2, TILE_FORWARD = 3 };
struct TileGroup {
    uint32_t kind = TILE_FETCH, width = 16, stage = 0, first = 0, n = 0;  // width 0: units of 8, 4, 2 and 1 bytes, the wider ones first
};
constexpr int kTileGroups = 40;
constexpr int kTileThreads = 512;  // of a CTA at most

struct TilesPlan {
    bool on = false;
    int64_t outer = 1, middle = 1, inner = 1;  // processes in front of, along and behind the dimensions of the middle hops
    int64_t width = 1, intervals = 1, rows_per_tile = 0, place_stride = 0, grid = 0;
    int threads = 256, unit = 16;  // unit: bytes of every unit (0: several widths)
    bool mesh = false;
    size_t smem = 0, units_at = 0, moved_at = 0, coords_at = 0;
    std::vector<int> coords;          // dimensions whose coordinates the units look at
    std::vector<TileUnit> units;
    std::vector<TileShift> shifts;    // the first: none
    std::vector<TileGroup> groups;    // stage 0: whatever the send buffers provide, then the phases that read places
    std::vector<unsigned char> args;  // the kernel's argument
};

// Experiment knobs, read from the environment ONCE, when a request is created, so that a
// persistent request keeps one plan however the environment changes between its starts.
// -1 (or 0 where stated) means "not set": the library's own choice applies.
struct Knobs {
    int pack_by_round = -1;   // ISO_PACK_BY_ROUND: intermediate places grouped by reading round (0/1)
    int lazy_final = -1;      // ISO_LAZY_FINAL: postpone every final hop to the last phase (0/1)
    int mixed = -1;           // ISO_MIXED: 0 = one launch per unit width instead of one of mixed widths
    int64_t bulk_chunk = 0;   // ISO_BULK_CHUNK: chunk bytes of the bulk kernel (0: automatic)
    int vec_threads = 0;      // ISO_VEC_THREADS: 256 or 512 for narrower CTAs (0: up to 1024)
    int vec_ctas_per_sm = 0;  // ISO_VEC_CTAS_PER_SM: CTAs per SM of the 256-thread shapes (0: automatic)
    int64_t bulk_tile = 0;    // ISO_BULK_TILE: processes per CTA of the bulk kernel (0: automatic)
    int host_slabs = -1;      // ISO_HOST_SLABS: slabs of the pipelined host-buffer path (-1: automatic)
    int graph = -1;           // ISO_GRAPH: graph replay on/off
    int slabs = -1;           // ISO_SLABS: slab count of Iso_Start
    int chains = -1;          // ISO_CHAINS
    bool no_pdl = false;      // ISO_NO_PDL: plain launches instead of programmatic dependent ones
    bool tune_log = false;    // ISO_TUNE_LOG: the tuner prints every plan it times
    int sender_side = -1;     // ISO_SENDER_SIDE: 0 never, 1 automatic, 2 wherever possible (allgather phases; -1: the request's setting)
    int hybrid = -1;          // ISO_HYBRID: 1 = long bodies of ragged rows through bulk warps, 0 = not (-1: the request's setting)
    bool col_split = true;    // ISO_COL_SPLIT=0: rows longer than a CTA are covered in passes instead of column chunks
    bool host_graph = true;   // ISO_HOST_GRAPH=0: the pipelined host-buffer path is never replayed from a graph
    bool coord_table = true;  // ISO_COORD_TABLE=0: row coordinates by division in every thread
    bool l2_keep = true;      // ISO_L2_KEEP=0: no eviction-priority hint on stores into the intermediate buffer
    int ag_order = -1;        // ISO_AG_ORDER=0/1: allgather visits the dimensions first-to-last / last-to-first
    int tiles = -1;           // ISO_TILES: 0 = never all phases of a tile in one launch, 1 = wherever possible, 2 and 3 = likewise, with
                              // all blocks going through places where widths are mixed and with none
    int words = -1;           // ISO_WORDS: 0 = no launches of words, 1 = wherever they can be (-1: chosen by the library)
};
Knobs read_knobs();

struct Request {
    Comm *comm = nullptr;
    Knobs knobs;
    int kind = ISO_KIND_ALLTOALL;
    int alg = ISO_ALG_COMBINING;
    int fusion = 1;
    int dim_order[ISO_MAX_DIMS] = {0, 1, 2, 3, 4, 5, 6, 7};  // allgather: dimension visited k-th (Section III-B)
    int64_t bulk_threshold = 512;        // in force (set by lower_schedule)
    int64_t bulk_threshold_asked = -1;   // Iso_request_set_bulk_threshold; -1: chosen by the library
    int layout = ISO_LAYOUT_PACKED;
    int slab_request = 0;     // slabs of dimension 0 Iso_Start runs one after the other (0: automatic, 1: none)
    bool persistent = false;  // run all phases in one cooperative launch when the schedule allows
    const unsigned char *send = nullptr;
    unsigned char *recv = nullptr;
    int s = 0;
    std::vector<int64_t> len, sdispl, rdispl;
    int64_t send_stride = 0, recv_stride = 0, inter_stride = 0;
    std::vector<Part> parts;           // schedule in execution order
    std::vector<LaunchPlan> launches;  // lowered schedule
    Iso_stats stats{};
    // device side (owned by iso_api.cu)
    bool dirty = true;
    void *d_blob = nullptr;                  // tables of the launches
    void *d_tiles = nullptr;                 // tables of the tiles
    bool launches_ready = false;             // the former and the intermediate buffer stand (not while nothing but starts in tiles ran)
    unsigned char *d_inter = nullptr;        // first usable byte (behind the leading guard band)
    unsigned char *d_inter_alloc = nullptr;  // the allocation: guard band, buffer, guard band
    int64_t d_inter_bytes = 0;
    int *d_err = nullptr;
    bool reports = false;  // the plan has kernels that may raise the error flag (bulk copies, waits on other CTAs)
    unsigned long long *d_counter = nullptr;  // grid-barrier arrivals (one-launch execution)
    unsigned long long epoch = 0;             // counter value at the next launch
    int multi_grid = 0;                       // > 0: one-launch execution with this grid
    size_t multi_smem = 0, multi_launches_off = 0;
    int *h_err = nullptr;
    void *last_stream = nullptr;
    bool started = false;
    std::vector<std::pair<long long, long long>> slab_plan;  // row ranges of the slabs (empty: whole torus at once)
    int64_t inter_rows = 0;            // processes the intermediate buffer holds
    std::vector<void *> host_streams;  // pipelined host-buffer path: two upload and two download streams
    std::vector<void *> slab_events;   // its events
    void *host_main_stream = nullptr;  // origin stream when that path is captured into a graph
    void *host_graph_exec = nullptr;   // cudaGraphExec_t of one pipelined host-buffer start
    const void *host_graph_hs = nullptr, *host_graph_hr = nullptr;  // the host buffers that graph copies from / to
    const void *host_last_hs = nullptr, *host_last_hr = nullptr;    // the host buffers of the last such start
    std::vector<void *> host_timing;   // timing events of its last call: uploads, downloads, whole call (begin, end each)
    bool host_timed = false;
    int host_slabs_used = 0;
    int sm_count = 148;  // a B200's; replaced by the current device's count before the first start
    int chains_request = 0;     // slabs to run side by side, as asked for (0: the library chooses)
    bool graph_request = false; // graph replay, as asked for
    int chains = 1;             // slabs that run side by side (each on its share of the SMs)
    struct ChainStream { int chain, priority; void *stream; };
    std::vector<ChainStream> chain_streams;  // for chains outside a graph: all but the first, by the priority of the caller's stream
    std::vector<void *> chain_events;        // fork and joins
    bool use_graph = false;     // Iso_Start replays a captured graph of the launches
    bool late_graph = false;    // likewise, but only from the third start on
    int plain_starts = 0;       // starts so far whose launches were enqueued one by one
    void *graph_exec = nullptr; // cudaGraphExec_t, built at the first Iso_Start after a change
    // pipelined one-launch execution (items = slab x launch, per-item completion counters)
    int wave_request = 0;       // 0: off, 1: one slab, n >= 2: n slabs of dimension 0
    bool wave_ok = false;       // the lowered schedule allows it (decided before the buffers are sized)
    int wave_slabs = 0;         // slabs in use (0: not in this mode)
    int wave_grid = 0;          // > 0: Iso_Start makes one cooperative launch of this many CTAs
    int wave_items = 0;
    size_t wave_smem = 0, wave_launches_off = 0, wave_items_off = 0;
    unsigned long long wave_run = 0;  // starts since the counters were last zeroed
    int wave_counters = 0;      // counters allocated in d_counter
    bool per_phase = false;     // one launch per phase was asked for (Iso_request_set_single_launch)
    TilesPlan tiles;            // all phases of a tile in one launch
    bool lean_tables = false;   // word tables of one row each, where the room for tables is short
    bool plain_units = false;   // no launches of words: every launch in units (Iso_neighbor_alltoall_static)
    bool hybrid = false;        // launches of mixed widths hand their long bodies to bulk warps (Iso_request_set_hybrid)
    int sender_side = 1;        // allgather phases in sender-side form: 0 never, 1 where measured faster, 2 wherever possible
    uint32_t wait_limit = 1u << 22;  // polls before a device-side wait on other CTAs gives up
    int skew_next = 0;          // testing: extra arrivals the next cooperative start waits for (one shot)
};

// Builds r.parts, r.inter_stride and the schedule statistics from r.comm, r.kind, r.alg,
// r.fusion and the block layout.  Returns an ISO_* code.
// Default visiting order of the allgather's prefix trie for this neighbourhood (fills r.dim_order).
void default_dimension_order(Request &r);
int build_schedule(Request &r);

// Splits parts into aligned pieces, groups them into kernel launches and fills the launch
// geometry.  `send_addr` / `recv_addr` / `inter_addr` are only used for their alignment.
int lower_schedule(Request &r, uintptr_t send_addr, uintptr_t recv_addr, uintptr_t inter_addr);

// Fills L.tables for the lowered launch L (L.words).  The addresses are only used for their alignment.
void build_words(const Request &r, LaunchPlan &L, uintptr_t send_addr, uintptr_t recv_addr, uintptr_t inter_addr);

// Whether Iso_Start runs all phases of a tile of processes in one launch, and how (fills r.tiles; the launches
// are lowered beside it, and set up when the host-buffer path asks for them).
void plan_tiles(Request &r);

// Checks the executed parts for hazards: every range inside its buffer, no write to the send
// buffer, and within a phase no written range overlapping another written or any read range.
int validate_schedule(const Request &r);

}  // namespace iso
