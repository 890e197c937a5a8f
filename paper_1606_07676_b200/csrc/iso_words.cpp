// Tables of the launches that move blocks of any size and placement in aligned 16-byte words
// (iso_words.cuh): which words a warp loads, which words it stores, and which bytes of the
// former make up the latter.
#include <algorithm>
#include <cstring>
#include <numeric>

#include "iso_internal.h"

namespace iso {

namespace {

// A run of bytes that is contiguous on both sides (the lowering may have cut it into pieces).
struct Block {
    int src_buf, dst_buf;
    int64_t src_off, dst_off, len;
    const Part *p;  // shift and check values
};

std::vector<Block> merged_blocks(const LaunchPlan &L, int d)
{
    std::vector<Block> b;
    for (const LoweredPart &lp : L.parts)
        b.push_back(Block{lp.p.src_buf, lp.p.dst_buf, lp.p.src_off, lp.p.dst_off, lp.p.len, &lp.p});
    std::sort(b.begin(), b.end(), [](const Block &x, const Block &y) {
        return x.dst_buf != y.dst_buf ? x.dst_buf < y.dst_buf : x.dst_off < y.dst_off;
    });
    size_t n = 0;
    for (size_t k = 0; k < b.size(); ++k) {
        if (n > 0) {
            Block &a = b[n - 1];
            if (a.dst_buf == b[k].dst_buf && a.src_buf == b[k].src_buf && a.dst_off + a.len == b[k].dst_off &&
                a.src_off + a.len == b[k].src_off && std::memcmp(a.p->shift, b[k].p->shift, sizeof(int) * d) == 0 &&
                std::memcmp(a.p->check, b[k].p->check, sizeof(int) * d) == 0) {
                a.len += b[k].len;
                continue;
            }
        }
        b[n++] = b[k];
    }
    b.resize(n);
    return b;
}

// The places inside a 16-byte word at which a block may start, over all rows.
struct Placement {
    int64_t lowest, highest;
};
Placement placement(int64_t addr, int64_t stride)
{
    const int64_t g = std::gcd<int64_t>(16, stride);
    const int64_t lowest = addr & (g - 1);  // g is a power of two
    return Placement{lowest, lowest + 16 - g};
}

// Deals warps to the chunks in proportion to what a row costs in them, so that all warps of a launch
// are done at the same time.  The weights are measured, in units of which a row of whole words costs
// 50: with equal shares the 27-point stencil of faces, edges and corners took 222 microseconds in three
// phases on a mesh, with these 166.
// (Placed chunks at 60, so that they got as many warps as whole ones: those warps finished last, 32^3 with
// blocks of 1024, 32 and 1 bytes in one pass 103.7 against 87.7 microseconds, the same on a mesh 169.0
// against 166.2, 64x64x32 with 30 blocks of 4 to 1024 bytes 1334 against 1316; anything from 70 to 100 is
// as good.)
void deal(WordTables &T)
{
    std::vector<uint32_t> cost;
    for (const EntryDev &ck : T.chunks) {
        uint32_t c = 50;
        if (ck.kind == CHUNK_PLACED) c = 80;
        if (ck.kind == CHUNK_ONE4 || ck.kind == CHUNK_ONE8) c = 40 + 8u * ck.passes;
        if (ck.kind == CHUNK_TWO) c = 75 + 45u * ck.passes;
        if (ck.kind == CHUNK_TINY) c = 75 + 90u * ck.passes;
        cost.push_back(c);
    }
    T.entries.clear();
    if (cost.empty()) return;
    const uint32_t least = *std::min_element(cost.begin(), cost.end());
    const uint32_t greatest = *std::max_element(cost.begin(), cost.end());
    const uint32_t unit = 4 * greatest <= 5 * least ? greatest : least / 4;  // entries in quarters of the cheapest chunk
    for (uint32_t k = 0; k < cost.size(); ++k) {
        const uint32_t turns = std::max<uint32_t>(1, (cost[k] + unit / 2) / unit);
        for (uint32_t t = 0; t < turns; ++t) {
            EntryDev e = T.chunks[k];
            e.chunk = k;
            e.turn = t;
            e.turns = turns;
            T.entries.push_back(e);
        }
    }
    // the entries of one chunk apart from one another, so that the warps that work on a row at the
    // same time are neighbours
    std::stable_sort(T.entries.begin(), T.entries.end(), [](const EntryDev &x, const EntryDev &y) {
        return (uint64_t)x.turn * y.turns < (uint64_t)y.turn * x.turns;
    });
}

struct Run { uint32_t block, sub; int64_t x; int begin, n; };  // bytes x .. x+n of a block, at `begin` in a word

// A destination word and its runs (runs[first] ...).
struct Word {
    int64_t at;  // from the (aligned down) start of the row group
    uint32_t first;
    uint8_t n, buf;
    bool in_place, full;  // 16-byte words: could be stored by the lanes that load it; all its bytes are in this launch
};

// Collects words of 4 or 8 bytes into chunks: one is closed when the next word would need more than 32
// loads, or be one too many.
struct FineChunks {
    WordTables &T;
    const std::vector<Run> &runs;
    const uint8_t plainest;  // the chunk's kind as long as every word has one block (TWO: two)
    EntryDev open{};
    uint32_t n_loads = 0, n_words = 0;
    uint32_t last_block = UINT32_MAX, last_slot = 0, last_sub = 0;  // what the last loads belong to
    int64_t first_k = 0, last_k = 0;
    Word words[32 * kWordsPasses];
    std::vector<uint32_t> places;  // place | lane << 10 of every run of the open chunk

    // range(run, k0, k1): the run's words, counted from the one that holds the block's first byte at its
    // lowest place, which is returned; load(run, k): the descriptor of its word k
    template <typename Range, typename Load>
    void add(const Word &w, Range range, Load load)
    {
        uint32_t need = 0, lb = last_block, ls = last_sub;
        int64_t lk = last_k, k0, k1;
        for (uint32_t j = w.first; j < w.first + w.n; ++j) {
            const Run &q = runs[j];
            range(q, k0, k1);
            const bool same = lb == q.block && ls == q.sub && k0 <= lk + 1;
            need += (uint32_t)(same ? std::max<int64_t>(0, k1 - lk) : k1 - k0 + 1);
            lk = same ? std::max(lk, k1) : k1;
            lb = q.block;
            ls = q.sub;
        }
        if (n_words == 32 * kWordsPasses || (n_words > 0 && (open.dst_buf != w.buf || w.at - words[0].at >= 4 << 16)) || n_loads + need > 32)
            close();
        if (n_words == 0) open.kind = plainest;
        open.dst_buf = w.buf;
        for (uint32_t j = w.first; j < w.first + w.n; ++j) {
            const Run &q = runs[j];
            const int64_t base = range(q, k0, k1);
            if (last_block != q.block || last_sub != q.sub || k0 > last_k + 1) {
                last_block = q.block;
                last_sub = q.sub;
                last_slot = n_loads;
                first_k = k0;
                last_k = k0 - 1;
            }
            while (last_k < k1) {
                T.loads.push_back(load(q, ++last_k));
                ++n_loads;
            }
            places.push_back((uint32_t)(16 + 16 * ((int64_t)last_slot - first_k) + q.x - q.begin + base) | last_slot << 10);
        }
        if (w.n > 2) open.kind = CHUNK_TINY;
        words[n_words++] = w;
    }

    void close()
    {
        if (n_words == 0) return;
        const bool tiny = open.kind == CHUNK_TINY;
        open.first = (uint32_t)(tiny ? T.tiny.size() : T.fine.size());
        open.passes = (uint8_t)((n_words + 31) / 32);
        open.dst_term = words[0].at;
        const uint32_t *place = places.data();
        for (uint32_t k = 0; k < n_words; ++k) {
            const Word &w = words[k];
            const uint32_t off = (uint32_t)((w.at - words[0].at) >> 2);
            if (tiny) {
                TinyDev t{};
                uint32_t byte[4] = {0, 0, 0, 0};
                for (uint32_t j = 0; j < w.n; ++j, ++place) {
                    const Run &q = runs[w.first + j];
                    for (int e = q.begin; e < q.begin + q.n; ++e) {
                        byte[e] = *place + (uint32_t)e;
                        t.mask |= 1u << e;
                    }
                }
                t.a = byte[0] | byte[1] << 15;
                t.b = byte[2] | byte[3] << 15;
                t.off = off;
                T.tiny.push_back(t);
            } else {
                FineDev f{};
                f.b = off;
                for (uint32_t j = 0; j < w.n; ++j, ++place) {  // one or two blocks
                    const Run &q = runs[w.first + j];
                    f.a |= *place << (15 * j);
                    f.b |= ((((1u << q.n) - 1u) << q.begin) & 15u) << (16 + 4 * j);
                }
                T.fine.push_back(f);
            }
        }
        T.fine.resize((T.fine.size() + 31) / 32 * 32, FineDev{});
        T.tiny.resize((T.tiny.size() + 31) / 32 * 32, TinyDev{});
        T.loads.resize((T.loads.size() + 31) / 32 * 32, LoadDev{});
        T.chunks.push_back(open);
        open = EntryDev{};
        places.clear();
        n_loads = n_words = 0;
        last_block = UINT32_MAX;
    }
};

}  // namespace

void build_words(const Request &r, LaunchPlan &L, uintptr_t send_addr, uintptr_t recv_addr, uintptr_t inter_addr)
{
    const Comm &c = *r.comm;
    const int64_t stride[3] = {r.send_stride, r.recv_stride, r.inter_stride};
    const int64_t addr[3] = {(int64_t)(send_addr & 15), (int64_t)(recv_addr & 15), (int64_t)(inter_addr & 15)};
    WordTables &T = L.tables;
    T = WordTables{};
    int used_index[ISO_MAX_DIMS];
    for (int j = 0; j < ISO_MAX_DIMS; ++j) used_index[j] = -1;
    for (int k = 0; k < L.n_used; ++k) used_index[L.used_dim[k]] = k;

    const std::vector<Block> blocks = merged_blocks(L, c.d);
    bool same_places[3];  // inside a word for all rows
    for (int k = 0; k < 3; ++k) same_places[k] = stride[k] % 16 == 0 && addr[k] == 0;
    auto at16 = [&](int buf) { return same_places[buf]; };
    bool fixed = true, dst_fixed = true;  // all buffers, all destinations are like that
    bool by4 = true, by8 = true;   // every address is a multiple of 4, of 8
    int64_t rows = 1, bytes = 0, words = 0, moving = 0, moving_bytes = 0;  // moving: blocks that are not, on either side
    for (const Block &b : blocks) {
        dst_fixed = dst_fixed && at16(b.dst_buf);
        if (!at16(b.src_buf) || !at16(b.dst_buf)) {
            fixed = false;
            ++moving;
            moving_bytes += b.len;
        }
        for (int64_t v : {stride[b.src_buf], stride[b.dst_buf], addr[b.src_buf], addr[b.dst_buf], b.src_off, b.dst_off, b.len}) {
            by4 = by4 && v % 4 == 0;
            by8 = by8 && v % 8 == 0;
        }
        rows = std::max<int64_t>(rows, 16 / std::gcd<int64_t>(16, stride[b.dst_buf]));
        bytes += b.len;
        words += (b.len + 23) / 16;
    }
    bool mesh = false;
    for (int k = 0; k < L.n_used; ++k) mesh = mesh || !c.periodic[L.used_dim[k]];
    // Form 1 describes `rows` rows in its tables: worth it where the blocks whose place varies are short
    // (several meet in a destination word) and the tables stay small.
    if (dst_fixed) rows = 1;
    if (fixed) T.form = mesh ? 1 : 0;
    else T.form = moving_bytes < kWordsLongBlock * moving && rows * bytes <= kWordsMostGroup && (rows == 1 || !r.lean_tables) ? 1 : 2;
    if (T.form == 2) {
        rows = 1;
    } else if (!r.lean_tables) {
        // Short rows: several of them share a chunk, so that its 32 loads are nearly all used (24 blocks of
        // 4 bytes are 24 loads, a quarter of the lanes idle) - as long as three warps per SM remain, and in
        // form 0, which knows no incomplete row group, where every slab is whole groups.  (Asking for 96
        // warps per SM instead: allgather of 24-byte blocks on 32^3 19.0 against 14.7 microseconds per start,
        // 8-byte blocks on 300x290 13.5 against 8.4, 12-byte blocks on 100x90 6.1 against 4.8; 26 64-byte
        // blocks, 104 words, one row to a group instead of four: 64^3 in one pass 168 against 150.)
        const int64_t whole = T.form == 1 ? 0 : (c.d >= 2 ? c.rank_stride[0] : c.P);
        auto uneven = [&]() {  // too few words, or a last chunk of which a good part is idle
            const int64_t n = rows * words;
            return n < 96 || ((n + 31) / 32 * 32 - n) * 100 > 7 * n;
        };
        while (uneven() && rows * 2 * bytes <= kWordsMostGroup && rows < 16 && whole % (rows * 2) == 0 &&
               c.P * words / 28 >= 3ll * r.sm_count)
            rows *= 2;
    }
    T.rows_sub = (uint32_t)rows;
    const int64_t grain = by8 ? 8 : 4;  // of the words that are smaller than 16 bytes

    std::vector<LoadDev> base(blocks.size());  // descriptors without a word
    for (size_t i = 0; i < blocks.size(); ++i) {
        const Block &b = blocks[i];
        LoadDev ld{};
        long long delta = 0;
        for (int j = 0; j < c.d; ++j) {
            const int value = c.periodic[j] ? b.p->shift[j] : b.p->check[j];
            delta -= (long long)b.p->shift[j] * c.rank_stride[j];
            if (value) ld.c[used_index[j]] = value;
        }
        ld.src_term = delta * stride[b.src_buf] + b.src_off;
        ld.len = (uint32_t)b.len;
        ld.dst_term = b.dst_off;
        ld.src_buf = (uint8_t)b.src_buf;
        ld.dst_buf = (uint8_t)b.dst_buf;
        base[i] = ld;
    }

    if (T.form == 2) {
        // A group of lanes per block: one per destination word, and one more that only loads.  What does not
        // fit into a chunk goes on in the next one, which costs a second lane that only loads, if that saves
        // an eighth of the chunks; else every block of up to 31 words has its lanes in one chunk.  (On 32^3 in
        // one pass 26 blocks of 252 bytes, 18 lanes each: 155.9 microseconds with one block to a chunk, 109.3
        // continued; 244 bytes, combining 327 against 251.  With 3 % fewer chunks, allgather of 919 bytes on
        // 5x5x8x5, 40.4 against 42.2.)
        auto lay_out = [&](int64_t least_room) {
            T.loads.clear();
            for (size_t i = 0; i < blocks.size(); ++i) {
                const Block &b = blocks[i];
                const LoadDev &ld = base[i];
                const int64_t n = (placement(addr[b.dst_buf] + b.dst_off, stride[b.dst_buf]).highest + b.len + 15) / 16;
                for (int64_t w = 0; w < n;) {
                    int64_t room = 32 - (int64_t)(T.loads.size() % 32);
                    if (n - w + 1 > room && room < least_room) {
                        T.loads.resize((T.loads.size() + 31) / 32 * 32, LoadDev{});
                        room = 32;
                    }
                    const int64_t take = std::min(room - 1, n - w);
                    for (int64_t k = 0; k <= take; ++k) {
                        T.loads.push_back(ld);
                        T.loads.back().word = (int32_t)(w + k);
                        T.loads.back().stores = k < take;
                    }
                    w += take;
                }
            }
            T.loads.resize((T.loads.size() + 31) / 32 * 32, LoadDev{});
        };
        lay_out(6);
        const size_t continued = T.loads.size();
        lay_out(32);
        if (continued * 8 <= T.loads.size() * 7) lay_out(6);
        T.chunks.resize(T.loads.size() / 32, EntryDev{});
        deal(T);
        return;
    }

    // Forms 0 and 1.  A destination word of 16 bytes whose bytes have the same place in one to three
    // source words, for all rows, can go into a placed chunk; everything else is cut into words of 4 or, where
    // everything is a multiple of 8, of 8 bytes.
    std::vector<Run> runs;
    std::vector<Word> words16;
    runs.reserve((size_t)(rows * (words + 2 * (int64_t)blocks.size())));
    words16.reserve((size_t)(rows * words));
    T.loads.reserve((size_t)(rows * words / 32 * 35 + 64));  // a few lanes of a chunk stay idle
    size_t n_in_place = 0, merged = 0, partial = 0;
    auto finish = [&]() {  // the last of words16 has all its runs
        if (words16.empty() || words16.back().n) return;
        Word &w = words16.back();
        w.n = (uint8_t)(runs.size() - w.first);
        w.in_place = w.n <= 3;  // every byte of the word has the same place in its source word
        int filled = 0;
        for (size_t j = w.first; j < runs.size(); ++j) {
            const Block &b = blocks[runs[j].block];
            w.in_place = w.in_place && at16(b.src_buf) && ((b.src_off + runs[j].x) & 15) == runs[j].begin;
            filled += runs[j].n;
        }
        w.full = filled == 16;
        n_in_place += w.in_place;
        merged += w.in_place && w.n > 1;
        partial += w.in_place && !w.full;
    };
    for (size_t lo = 0; lo < blocks.size();) {
        size_t hi = lo;
        while (hi < blocks.size() && blocks[hi].dst_buf == blocks[lo].dst_buf) ++hi;
        const int buf = blocks[lo].dst_buf;
        for (uint32_t sub = 0; sub < T.rows_sub; ++sub)
            for (size_t k = lo; k < hi; ++k) {
                const int64_t at = (int64_t)sub * stride[buf] + addr[buf] + blocks[k].dst_off, last = at + blocks[k].len;
                for (int64_t p = at; p < last;) {
                    const int64_t w = p & ~(int64_t)15, end = std::min(w + 16, last);
                    if (words16.empty() || words16.back().buf != buf || words16.back().at != w) {
                        finish();
                        words16.push_back(Word{w, (uint32_t)runs.size(), 0, (uint8_t)buf, false, false});
                    }
                    runs.push_back(Run{(uint32_t)k, sub, p - at, (int)(p - w), (int)(end - p)});
                    p = end;
                }
            }
        lo = hi;
    }
    finish();

    // Words that this launch fills only in part are cheaper as smaller words, unless there are next to
    // none (the end of a row): with them all placed the irregular collective of 4 to 1024 bytes took
    // 1642 instead of 1387 microseconds.  Where merged words are few, the words that are not get chunks
    // of their own, which need no merging (and where everything is a multiple of 4 bytes, the few are
    // cheaper in smaller words: one-pass irregular 735 against 685); where they are many, they stay
    // with their neighbours (118-byte blocks, one merged word in eight: 88 against 134 microseconds).
    // In one pass along three dimensions and more they stay with their neighbours further down: what is stored far from its
    // sector-mates costs more in the L2 (120-byte blocks of 342 neighbours on 24x22x23 204 against 380, 232 bytes of 124 on 16x26x24
    // 108 against 131, but 168 bytes of 8 along two dimensions on 525x492 147 against 127, irregular sizes on 64x64x32 705 against 679).
    const size_t few = L.n_used < 3 ? 12 : (by8 ? 36 : 20);
    const bool apart = merged * few < n_in_place, keep_partial = partial * 64 <= n_in_place;
    std::vector<uint32_t> plain, rest;  // of words16
    std::vector<Word> fine;
    std::vector<Run> fine_runs;
    for (uint32_t i = 0; i < words16.size(); ++i) {
        const Word &w = words16[i];
        if (w.in_place && (w.full || keep_partial)) {
            if (apart && w.full && w.n == 1) {
                plain.push_back(i);
                continue;
            }
            if (!apart || !by4) {
                rest.push_back(i);
                continue;
            }
        }
        for (uint32_t j = w.first; j < w.first + w.n; ++j) {
            const Run &q = runs[j];
            for (int at = q.begin; at < q.begin + q.n;) {
                const int start = at & ~((int)grain - 1), end = std::min(start + (int)grain, q.begin + q.n);
                if (fine.empty() || fine.back().buf != w.buf || fine.back().at != w.at + start)
                    fine.push_back(Word{w.at + start, (uint32_t)fine_runs.size(), 0, w.buf, false, false});
                ++fine.back().n;
                fine_runs.push_back(Run{q.block, q.sub, q.x + at - q.begin, at - start, end - at});
                at = end;
            }
        }
    }

    // Placed words in address order, so that the two halves of a 32-byte sector belong to one chunk: the
    // lanes that store first, then those that only load.
    for (const std::vector<uint32_t> *list : {&plain, &rest})
        for (size_t k = 0; k < list->size();) {
            auto word = [&](size_t i) -> const Word & { return words16[(*list)[i]]; };
            size_t n = 0, lanes = 0;
            while (k + n < list->size() && word(k + n).buf == word(k).buf && lanes + word(k + n).n <= 32) lanes += word(k + n++).n;
            if (k + n < list->size() && n > 1 && word(k + n).at % 32 != 0 && word(k + n).at == word(k + n - 1).at + 16) --n;
            const size_t first = T.loads.size();
            T.loads.resize(first + 32, LoadDev{});
            for (size_t e = 0; e < 32; ++e) T.loads[first + e].second = T.loads[first + e].third = (uint8_t)e;
            size_t extra = n;
            EntryDev ck{};
            ck.kind = CHUNK_WHOLE;
            ck.passes = 1;
            ck.dst_buf = word(k).buf;
            for (size_t e = 0; e < n; ++e) {
                const Word &w = word(k + e);
                for (uint32_t j = 0; j < w.n; ++j) {
                    const Run &q = runs[w.first + j];
                    const size_t lane = j == 0 ? e : extra++;
                    const uint8_t second = T.loads[first + lane].second, third = T.loads[first + lane].third;
                    LoadDev &ld = T.loads[first + lane];
                    ld = base[q.block];
                    ld.sub = (uint8_t)q.sub;
                    ld.src_term += q.x - q.begin;
                    ld.dst_term = w.at;
                    ld.mask = (uint16_t)(((1u << q.n) - 1u) << q.begin);
                    ld.second = second;
                    ld.third = third;
                    ld.stores = j == 0;
                    if (j == 1) T.loads[first + e].second = (uint8_t)lane;
                    if (j == 2) T.loads[first + e].third = (uint8_t)lane;
                }
                if (w.n > 1 || !w.full) ck.kind = CHUNK_PLACED;
                ck.passes = std::max(ck.passes, w.n);
            }
            T.chunks.push_back(ck);
            k += n;
        }

    FineChunks chunks{T, fine_runs, (uint8_t)(by8 ? CHUNK_ONE8 : (by4 ? CHUNK_ONE4 : CHUNK_TWO))};
    std::vector<Placement> places(blocks.size());
    for (size_t i = 0; i < blocks.size(); ++i) places[i] = placement(addr[blocks[i].src_buf] + blocks[i].src_off, stride[blocks[i].src_buf]);
    auto range = [&](const Run &q, int64_t &k0, int64_t &k1) -> int64_t {
        const Placement &pl = places[q.block];
        k0 = (pl.lowest + q.x) >> 4;
        k1 = (pl.highest + q.x + q.n - 1) >> 4;
        return at16(blocks[q.block].src_buf) ? pl.lowest : 0;  // (where it varies the kernel adds the row's own place)
    };
    auto load = [&](const Run &q, int64_t k) {
        LoadDev ld = base[q.block];
        ld.sub = (uint8_t)q.sub;
        if (at16(blocks[q.block].src_buf)) ld.src_term += k * 16 - (blocks[q.block].src_off & 15);  // the aligned word itself
        else ld.word = (int32_t)k;
        return ld;
    };
    for (const Word &w : fine) chunks.add(w, range, load);
    chunks.close();
    deal(T);
}

}  // namespace iso
