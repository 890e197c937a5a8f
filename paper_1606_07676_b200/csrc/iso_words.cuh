// Device code for launches whose blocks are not made of whole, equally placed 16-byte units
// (sm_100a): blocks of a few or of an odd number of bytes, irregular collectives, buffers whose
// process stride is not a multiple of 16.
//
// Such data used to move in units of the widest power of two that divides every offset: 4-byte
// units for a block of 12 bytes, 1-byte units for one of 13, each a load and a store of its own,
// which bounds the kernel by load/store instructions.  (Some still do, where that is the faster way:
// better_in_units in iso_schedule.cpp.)  Here
//   * a lane LOADS one aligned 16-byte word of a source row (cp.async into a ring of slots, as in
//     the aligned kernel), whatever part of the word its block needs;
//   * where every byte of a destination word has the same place in the words it comes from, a lane
//     stores 16 bytes: the word it has loaded itself, merged at the ends of a block with those of one or
//     two other lanes; everything else is stored in aligned 4- or 8-byte words, consecutive lanes
//     consecutive words, each put together from the bytes that the lanes of the warp have loaded (two
//     shared-memory reads and a shift per block that meets in the word).
// Loading and storing lanes belong to the same warp, so the hand-over costs a __syncwarp and the
// warps run independently of one another.  A warp owns one chunk of the payload of a row and walks
// down its rows.
//
// FORM says how source and destination are placed against each other:
//   0  every stride and base address is a multiple of 16 and all dimensions are periodic: the place of
//      every byte inside its word is the same for all rows, so shifts and masks come from the tables;
//   1  anything else, short blocks: the tables describe A consecutive rows (A * the destination's stride
//      is a multiple of 16), and the place of a source whose stride is not one, and whether it exists
//      at all, is worked out per row (a "code" per word in flight);
//   2  anything else, long blocks: a group of lanes per block, both alignments worked out per row;
//      16-byte stores, only the first and the last word of a block in part.
// An aligned word that holds one byte of a buffer never leaves the buffer's page, so words are
// loaded whole at the ends of a buffer too (iso.h says so: up to 15 bytes on either side are read and
// dropped); what is stored is exact to the byte.
#pragma once

#include "iso_kernels.cuh"

namespace iso {

// 16 bytes from any byte address of shared memory.
__device__ __forceinline__ uint4 lds_shifted(const unsigned char *p)
{
    const uint32_t a = (uint32_t)__cvta_generic_to_shared(p);
    const uint4 *w = reinterpret_cast<const uint4 *>(p - (a & 15u));
    const uint4 lo = w[0];
    if ((a & 15u) == 0) return lo;
    const uint4 hi = w[1];
    const bool two = (a & 8u) != 0, one = (a & 4u) != 0;
    const uint32_t y0 = two ? lo.z : lo.x, y1 = two ? lo.w : lo.y, y2 = two ? hi.x : lo.z;
    const uint32_t y3 = two ? hi.y : lo.w, y4 = two ? hi.z : hi.x, y5 = two ? hi.w : hi.y;
    const uint32_t z0 = one ? y1 : y0, z1 = one ? y2 : y1, z2 = one ? y3 : y2, z3 = one ? y4 : y3, z4 = one ? y5 : y4;
    const uint32_t b = (a & 3u) * 8u;
    return make_uint4(__funnelshift_r(z0, z1, b), __funnelshift_r(z1, z2, b), __funnelshift_r(z2, z3, b), __funnelshift_r(z3, z4, b));
}

// Bit k of the four bits of `m` spread to byte k.
__device__ __forceinline__ uint32_t byte_mask(uint32_t m) { return ((m * 0x00204081u) & 0x01010101u) * 0xffu; }

// 4 bytes from any byte address `at` behind `base` (a multiple of 4).
__device__ __forceinline__ uint32_t lds_shifted_4(const unsigned char *base, uint32_t at)
{
    const uint32_t *w = reinterpret_cast<const uint32_t *>(base + (at & ~3u));
    return __funnelshift_r(w[0], w[1], at * 8u);  // (the shift counts modulo 32)
}

// Exactly the bytes named by the four bits of `m`: the others belong to other launches, or to nobody.
__device__ __forceinline__ void store_4_masked(unsigned char *dst, uint32_t v, uint32_t m)
{
    if (m == 15u) {
        *reinterpret_cast<uint32_t *>(dst) = v;
        return;
    }
    if ((m & 3u) == 3u) {
        *reinterpret_cast<uint16_t *>(dst) = (uint16_t)v;
    } else {
        if (m & 1u) dst[0] = (unsigned char)v;
        if (m & 2u) dst[1] = (unsigned char)(v >> 8);
    }
    if ((m & 12u) == 12u) {
        *reinterpret_cast<uint16_t *>(dst + 2) = (uint16_t)(v >> 16);
    } else {
        if (m & 4u) dst[2] = (unsigned char)(v >> 16);
        if (m & 8u) dst[3] = (unsigned char)(v >> 24);
    }
}

__device__ __forceinline__ void store_16_masked(unsigned char *dst, const uint4 &v, uint32_t mask)
{
    if (mask == 0xffffu) {
        *reinterpret_cast<uint4 *>(dst) = v;
        return;
    }
    if (mask & 0x000fu) store_4_masked(dst, v.x, mask & 15u);
    if (mask & 0x00f0u) store_4_masked(dst + 4, v.y, (mask >> 4) & 15u);
    if (mask & 0x0f00u) store_4_masked(dst + 8, v.z, (mask >> 8) & 15u);
    if (mask & 0xf000u) store_4_masked(dst + 12, v.w, (mask >> 12) & 15u);
}

// `a` with the bytes of `b` where the masks (of whole bytes) are set.
__device__ __forceinline__ uint4 blend(const uint4 &a, const uint4 &b, const uint4 &k)
{
    return make_uint4((b.x & k.x) | (a.x & ~k.x), (b.y & k.y) | (a.y & ~k.y), (b.z & k.z) | (a.z & ~k.z), (b.w & k.w) | (a.w & ~k.w));
}
__device__ __forceinline__ uint4 byte_masks(uint32_t m)
{
    return make_uint4(byte_mask(m & 15u), byte_mask((m >> 4) & 15u), byte_mask((m >> 8) & 15u), byte_mask((m >> 12) & 15u));
}

// NU: shifted dimensions per block the kernel is compiled for (1 to 4, or ISO_MAX_DIMS for any number).
// MESH: some of them are not periodic.  TAB: the rows' coordinates come from a table in shared memory
// (the CTA fills it before it waits for the previous kernel), otherwise from exact divisions.
//
// A warp works on two rows at a time: what it waits for, beside device memory, is its own chain of
// shared-memory reads, shuffles and stores, and two rows are two such chains.  For the registers that
// takes, a CTA has 24 warps instead of 32; the ring holds sixteen words per lane, so that the bytes in
// flight per SM stay those of the aligned kernel (with eight or twelve instead, one-pass irregular
// sizes on 64x64x32 677 and 687 against 683 microseconds, 64^3 with 64-byte blocks 171 in all three).
template <int FORM, bool MESH, int NU, bool TAB>
__global__ void __launch_bounds__(kWordsThreads, 1) iso_gather_words(const __grid_constant__ LaunchDev L)
{
    extern __shared__ __align__(128) unsigned char smem_raw[];
    constexpr int DEPTH = FORM == 0 ? kWordsDepth : kWordsDepthCoded, R = 2;
    static_assert(FORM != 0 || !MESH, "a mesh needs codes");
    constexpr uint32_t NT = NU <= 1 ? 1 : (NU == 2 ? 2 : (NU <= 4 ? 4 : 8));  // table entries per row
    constexpr uint32_t kNone = 16;                                            // code of a block that has no source
    constexpr bool coded = FORM != 0;
    constexpr bool GROUPS = FORM != 2;  // the tables may describe several rows
    constexpr int kFew = 4;             // up to so many dimensions their wrap terms are kept in registers
    const uint32_t nthr = blockDim.x, nw = nthr >> 5, warp = threadIdx.x >> 5, lane = threadIdx.x & 31u;
    const uint32_t A = GROUPS ? L.rows_sub : 1;
    const uint32_t n_entries = L.n_entries;
    const uint32_t gw = blockIdx.x * nw + warp;
    const uint32_t slot = gw / n_entries;
    const uint32_t nslots = gridDim.x * nw / n_entries;
    // (ranks are below 2^31)
    const uint32_t s_lo = (uint32_t)L.row_lo / A, s_hi = ((uint32_t)L.row_hi + A - 1) / A;
    EntryDev en;
    {
        const uint4 *raw = reinterpret_cast<const uint4 *>(L.entries + (gw - slot * n_entries));
        reinterpret_cast<uint4 *>(&en)[0] = __ldg(raw);
        reinterpret_cast<uint4 *>(&en)[1] = __ldg(raw + 1);
    }
    const uint32_t s_first = s_lo + slot + en.turn * nslots, s_step = en.turns * nslots;  // this warp's row groups
    const bool active = slot < nslots && s_first < s_hi;
    unsigned char *const ring = smem_raw + kWordsPadFront + (size_t)threadIdx.x * 16;

    LoadDev ld;
    ld.len = 0;
    if (active) {
        const uint4 *raw = reinterpret_cast<const uint4 *>(L.loads + en.chunk * 32u + lane);
        uint4 *into = reinterpret_cast<uint4 *>(&ld);
        into[0] = __ldg(raw);
        into[1] = __ldg(raw + 1);
        if (NU > kFew) into[2] = __ldg(raw + 2);
        into[3] = __ldg(raw + 3);
    }
    uint32_t *const tab = reinterpret_cast<uint32_t *>(smem_raw + kWordsPadFront + (size_t)DEPTH * nthr * 16 + kWordsPadBack);
    const uint32_t first_slot = blockIdx.x * nw / n_entries;
    if (TAB) {
        const uint32_t per_it = L.tab_slots * A;
        const uint32_t entries = L.tab_iters * per_it;
        for (uint32_t j = threadIdx.x; j < entries; j += nthr) {
            const uint32_t it = j / per_it, rest = j - it * per_it;
            const uint32_t ls = rest / A;
            const unsigned long long r = (unsigned long long)(s_lo + first_slot + ls + it * nslots) * A + (rest - ls * A);
            if (r < (unsigned long long)L.P)
                for (int k = 0; k < L.n_used; ++k) {
                    const uint32_t t = fastdiv(L.div_rstride[k], (uint32_t)r);
                    tab[j * NT + k] = t - fastdiv(L.div_size[k], t) * L.used_size[k];
                }
        }
        __syncthreads();
    }
    grid_dependency_wait();
    grid_launch_dependents();
    if (!active) return;

    const long long stride_s = L.buf_stride[ld.src_buf];
    const uint32_t sub = GROUPS ? ld.sub : 0u;
    const unsigned char *src_ld = L.buf[ld.src_buf] + ld.src_term + ((long long)s_first * A + sub) * stride_s;
    const long long src_step = (long long)s_step * A * stride_s;
    const bool loads = ld.len != 0;
    const bool whole = FORM != 2 && en.kind == CHUNK_WHOLE, placed = FORM != 2 && en.kind == CHUNK_PLACED;
    const int db = FORM == 2 ? ld.dst_buf : en.dst_buf;
    const long long group_d = (long long)A * L.buf_stride[db];
    const bool keep = (whole || placed) && L.keep_inter && db == 2;  // ISO_BUF_INTER
    const uint64_t policy = keep ? l2_policy_evict_last() : 0;
    unsigned char *const base_d = FORM == 2 ? L.buf[db] + ld.dst_term
                                            : reinterpret_cast<unsigned char *>(reinterpret_cast<uintptr_t>(L.buf[db]) & ~(uintptr_t)15) +
                                                  (whole || placed ? ld.dst_term : en.dst_term);
    long long wrap_bytes[NU <= kFew ? NU : 1];
    if (NU <= kFew) {
#pragma unroll
        for (int e = 0; e < NU; ++e) wrap_bytes[e] = (long long)L.used_wrap[e] * stride_s;
    }

    // Loads this lane's word of row group s into a ring slot.  Returns where in its word the byte at
    // src_term lies, or kNone (forms 1, 2).
    const uint32_t tab_row = L.tab_slots * A * NT;
    uint32_t tab_at = ((slot - first_slot) * A + sub) * NT + en.turn * tab_row;
    const uint32_t tab_step = en.turns * tab_row;
    auto load = [&](uint32_t s, unsigned char *to) -> uint32_t {
        const uint32_t r = s * A + sub;
        uint32_t x[NU];
        if (TAB) {
            if (NU == 1) {
                x[0] = tab[tab_at];
            } else if (NU == 2) {
                const uint2 t = *reinterpret_cast<const uint2 *>(tab + tab_at);
                x[0] = t.x;
                x[NU > 1 ? 1 : 0] = t.y;
            } else {
#pragma unroll
                for (int e = 0; e < NU; e += 4) {
                    const uint4 t = *reinterpret_cast<const uint4 *>(tab + tab_at + e);
                    x[e] = t.x;
                    if (e + 1 < NU) x[e + 1] = t.y;
                    if (e + 2 < NU) x[e + 2] = t.z;
                    if (e + 3 < NU) x[e + 3] = t.w;
                }
            }
            tab_at += tab_step;
        } else {
#pragma unroll
            for (int e = 0; e < NU; ++e)
                if (NU <= kFew || e < L.n_used) {
                    const uint32_t t = fastdiv(L.div_rstride[e], r);
                    x[e] = t - fastdiv(L.div_size[e], t) * L.used_size[e];
                }
        }
        bool valid = true;
        if (FORM == 1) valid = r >= (uint32_t)L.row_lo && r < (uint32_t)L.row_hi;
        const unsigned char *src = src_ld;
        src_ld += src_step;
        uint32_t wraps = 0;
#pragma unroll
        for (int e = 0; e < NU; ++e)
            if (NU <= kFew || e < L.n_used) {
                const int c = ld.c[e];
                if (MESH && ((L.mesh_mask >> e) & 1)) {
                    const int y = (int)x[e] - c;
                    valid = valid && y >= 0 && y < (int)L.used_size[e];
                } else if ((int)x[e] < c) {
                    if (NU <= kFew) src += wrap_bytes[e < kFew ? e : 0];
                    else wraps += L.used_wrap[e];
                }
            }
        if (NU > kFew) src += (long long)wraps * stride_s;
        if (FORM == 0) {
            if (loads) cp_async<16>(to, src);
            return 0u;
        }
        const uint32_t mis = (uint32_t)(uintptr_t)src & 15u;
        int w = ld.word;
        if (FORM == 2) {
            const uint32_t dm = (uint32_t)(uintptr_t)(base_d + (long long)r * group_d) & 15u;
            if (mis < dm) --w;
        }
        if (loads && valid && w >= 0 && (uint32_t)w * 16u < mis + ld.len) cp_async<16>(to, src - mis + (long long)w * 16);
        return valid ? mis : kNone;
    };

    unsigned long long codes = 0;  // forms 1 and 2: five bits per stage in flight, the newest lowest
    uint32_t s_ld = s_first;
    const uint32_t stage_bytes = nthr * 16;
    auto load_two = [&](unsigned char *to) {
#pragma unroll
        for (int i = 0; i < R; ++i) {
            uint32_t code = kNone;
            if (s_ld < s_hi) code = load(s_ld, to + i * stage_bytes);
            s_ld += s_step;
            if (coded) codes = (codes << 5) | code;
        }
        cp_async_commit();
    };
#pragma unroll
    for (int i = 0; i < DEPTH; i += R) load_two(ring + i * stage_bytes);
    unsigned char *stage = ring;
    unsigned char *const stage_end = ring + DEPTH * stage_bytes;
    unsigned char *dst = base_d + (long long)s_first * group_d;
    const long long dst_step = (long long)s_step * group_d;
    auto refill = [&]() {
        load_two(stage);
        dst += R * dst_step;
        stage += R * stage_bytes;
        if (stage == stage_end) stage = ring;
    };
    auto code_of = [&](int i) -> uint32_t { return (uint32_t)(codes >> (5 * (DEPTH - 1 - i))) & 31u; };

    if (FORM == 2) {
        for (uint32_t s = s_first; s < s_hi; s += R * s_step) {
            cp_async_wait<DEPTH / R - 1>();
            __syncwarp();
            uint4 v[R];
            uint32_t mask[R];
            int x0[R];
#pragma unroll
            for (int i = 0; i < R; ++i) {
                const uint32_t code = code_of(i);
                const uint32_t dm = (uint32_t)(uintptr_t)(dst + i * dst_step) & 15u;
                x0[i] = ld.word * 16 - (int)dm;  // the block's byte that goes to byte 0 of the word
                const int lo = x0[i] < 0 ? -x0[i] : 0;
                const int left = (int)ld.len - x0[i];
                const int hi = left < 16 ? left : 16;
                mask[i] = 0;
                if (loads && ld.stores && code != kNone && hi > lo && s + i * s_step < s_hi) mask[i] = (0xffffu >> (16 - hi)) & (0xffffu << lo);
                if (mask[i]) v[i] = lds_shifted(stage + i * stage_bytes + ((code - dm) & 15u));
            }
#pragma unroll
            for (int i = 0; i < R; ++i)
                if (mask[i]) store_16_masked(dst + i * dst_step + x0[i], v[i], mask[i]);
            __syncwarp();
            refill();
        }
    } else if (whole) {
        constexpr int RW = 2 * R;  // nothing but copies: four rows at a time
        for (uint32_t s = s_first; s < s_hi; s += RW * s_step) {
            cp_async_wait<DEPTH / R - 2>();
            uint4 v[RW];
#pragma unroll
            for (int i = 0; i < RW; ++i) v[i] = *reinterpret_cast<const uint4 *>(stage + i * stage_bytes);
#pragma unroll
            for (int i = 0; i < RW; ++i)
                if (loads && (coded ? code_of(i) != kNone : s + i * s_step < s_hi)) {
                    if (keep) store_16_hinted(dst + i * dst_step, v[i], policy);
                    else *reinterpret_cast<uint4 *>(dst + i * dst_step) = v[i];
                }
            refill();
            refill();
        }
    } else if (placed) {
        // what is stored: this lane's bytes, those of the second and of the third lane
        const uint32_t m_own = loads ? (uint32_t)ld.mask : 0u;
        uint32_t m_second = __shfl_sync(0xffffffffu, m_own, ld.second), m_third = __shfl_sync(0xffffffffu, m_own, ld.third);
        if (ld.second == lane) m_second = 0;
        if (ld.third == lane) m_third = 0;
        const bool stores = loads && ld.stores;
        const uint4 k_second = byte_masks(m_second);
        const int to_second = ((int)ld.second - (int)lane) * 16, to_third = ((int)ld.third - (int)lane) * 16;
        for (uint32_t s = s_first; s < s_hi; s += R * s_step) {
            cp_async_wait<DEPTH / R - 1>();
            __syncwarp();
            uint4 v[R];
            uint32_t mask[R];
#pragma unroll
            for (int i = 0; i < R; ++i) {
                mask[i] = s + i * s_step < s_hi ? m_own | m_second | m_third : 0u;
                if (coded) {
                    const uint32_t code = code_of(i), code2 = __shfl_sync(0xffffffffu, code, ld.second), code3 = __shfl_sync(0xffffffffu, code, ld.third);
                    mask[i] = (code != kNone ? m_own : 0u) | (code2 != kNone ? m_second : 0u) | (code3 != kNone ? m_third : 0u);
                }
                const unsigned char *const own = stage + i * stage_bytes;
                v[i] = *reinterpret_cast<const uint4 *>(own);
                if (m_second) v[i] = blend(v[i], *reinterpret_cast<const uint4 *>(own + to_second), k_second);
            }
            if (en.passes > 2) {
#pragma unroll
                for (int i = 0; i < R; ++i)
                    if (m_third) v[i] = blend(v[i], *reinterpret_cast<const uint4 *>(stage + i * stage_bytes + to_third), byte_masks(m_third));
            }
#pragma unroll
            for (int i = 0; i < R; ++i)
                if (stores && mask[i]) {
                    if (keep && mask[i] == 0xffffu) store_16_hinted(dst + i * dst_step, v[i], policy);
                    else store_16_masked(dst + i * dst_step, v[i], mask[i]);
                }
            __syncwarp();
            refill();
        }
    } else {
        FineDev f[kWordsPasses];
#pragma unroll
        for (int p = 0; p < kWordsPasses; ++p) {
            f[p].a = f[p].b = 0;
            if (p < en.passes && en.kind != CHUNK_TINY) *reinterpret_cast<uint2 *>(&f[p]) = __ldg(reinterpret_cast<const uint2 *>(L.fine + en.first + 32u * p + lane));
        }
        // codes of the two rows (without codes: whether the row exists)
        uint32_t code[R];
        const unsigned char *bytes;  // 16 bytes in front of the chunk's first slot
        auto wait = [&](uint32_t s) {
            cp_async_wait<DEPTH / R - 1>();
            __syncwarp();
#pragma unroll
            for (int i = 0; i < R; ++i) code[i] = coded ? code_of(i) : (s + i * s_step < s_hi ? 0u : kNone);
            bytes = stage - lane * 16u - 16u;
        };
        auto advance = [&]() {
            __syncwarp();
            refill();
        };
        auto one_block = [&](auto word) {  // every word out of one block, no shift
            using V = decltype(word);
            for (uint32_t s = s_first; s < s_hi; s += R * s_step) {
                wait(s);
#pragma unroll
                for (int p = 0; p < kWordsPasses; ++p) {
                    if (p >= en.passes) break;
                    V v[R];
                    bool there[R];
#pragma unroll
                    for (int i = 0; i < R; ++i) {
                        const uint32_t mis = coded ? __shfl_sync(0xffffffffu, code[i], f[p].a >> 10) : code[i];
                        there[i] = (f[p].b & 0xf0000u) && mis != kNone;
                        if (there[i]) v[i] = *reinterpret_cast<const V *>(bytes + i * stage_bytes + (f[p].a & 1023u) + (coded ? mis : 0u));
                    }
#pragma unroll
                    for (int i = 0; i < R; ++i)
                        if (there[i]) *reinterpret_cast<V *>(dst + i * dst_step + (f[p].b & 0xffffu) * 4u) = v[i];
                }
                advance();
            }
        };
        if (en.kind == CHUNK_ONE8) {
            one_block(uint2{});
        } else if (en.kind == CHUNK_ONE4) {
            one_block(uint32_t{});
        } else if (en.kind == CHUNK_TWO) {
            for (uint32_t s = s_first; s < s_hi; s += R * s_step) {
                wait(s);
#pragma unroll
                for (int p = 0; p < kWordsPasses; ++p) {
                    if (p >= en.passes) break;
                    uint32_t v[R], m[R];
#pragma unroll
                    for (int i = 0; i < R; ++i) {
                        uint32_t m0 = (f[p].b >> 16) & 15u, m1 = (f[p].b >> 20) & 15u, mis0 = code[i], mis1 = code[i];
                        if (coded) {
                            mis0 = __shfl_sync(0xffffffffu, code[i], f[p].a >> 10);
                            mis1 = __shfl_sync(0xffffffffu, code[i], f[p].a >> 25);
                        }
                        if (mis0 == kNone) m0 = 0;
                        if (mis1 == kNone) m1 = 0;
                        m[i] = m0 | m1;
                        const unsigned char *const from = bytes + i * stage_bytes;
                        v[i] = lds_shifted_4(from, (f[p].a & 1023u) + (mis0 & 15u));
                        if (m1) {
                            const uint32_t second = byte_mask(m1);
                            v[i] = (v[i] & ~second) | (lds_shifted_4(from, ((f[p].a >> 15) & 1023u) + (mis1 & 15u)) & second);
                        }
                    }
#pragma unroll
                    for (int i = 0; i < R; ++i)
                        if (m[i]) store_4_masked(dst + i * dst_step + (f[p].b & 0xffffu) * 4u, v[i], m[i]);
                }
                advance();
            }
        } else {
            for (uint32_t s = s_first; s < s_hi; s += R * s_step) {
                wait(s);
                for (uint32_t p = 0; p < en.passes; ++p) {
                    const uint4 t = __ldg(reinterpret_cast<const uint4 *>(L.tiny + en.first + 32u * p + lane));
#pragma unroll
                    for (int i = 0; i < R; ++i) {
                        uint32_t v = 0, m = 0;
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            const uint32_t w = (e < 2 ? t.x : t.y) >> (15 * (e & 1));
                            const uint32_t mis = coded ? __shfl_sync(0xffffffffu, code[i], w >> 10) : code[i];
                            if ((t.w >> e & 1u) && mis != kNone) {
                                v |= (uint32_t)bytes[i * stage_bytes + (w & 1023u) + mis] << (8 * e);
                                m |= 1u << e;
                            }
                        }
                        if (m) store_4_masked(dst + i * dst_step + (size_t)t.z * 4, v, m);
                    }
                }
                advance();
            }
        }
    }
    cp_async_wait<0>();
}

}  // namespace iso
