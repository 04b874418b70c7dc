// The expander (paper Sec. 2.2, "Unfolding at load time"): one pass that turns every 48-bit code word into its
// decoded-field record - class id, gain bit, sign mask, per-coordinate level - in one of the layouts of include/llvq.h.
// Integer arithmetic only (the float estimates in llvq_unrank.cuh are corrected in integers), so the output is bit-exact.
//
// Bound: the gathers from the lists and instruction issue, not HBM (8 bytes in, 10 to 20 out a block).  The two types of
// class take different code, and codes come in random order, so a warp first finds the class of all 128 blocks of a
// tile (a lane a row), lists them by type in shared memory and then un-ranks 32 blocks of one type at a time, whatever
// their place; the codes wait in shared memory until the tile's words are gathered from them.  The small look-up tables
// are copied to shared memory once a CTA, while the previous kernel of the stream ends; one CTA a multiprocessor walks over
// the tiles.
// Measured (9728 x 2560 into the 14-byte layout, 1.04 M blocks): 35.2 us; 17408 x 5120 106 us, counted and expanded into the
// 10-byte layout 171.  A lane a row with a 64-bit division a coordinate and candidate took 484 and 4700 (10-byte layout) us, one odd
// coordinate at a time 45.  24 or 28 warps a CTA instead of 32: 47 and 50 us against 38.  A multiprocessor's memory that is not shared is the
// L1 cache the lists are read through, so the shared tables are kept to 20 KB and a warp's scratch to 2 KB (with 51 and 3.6 KB
// 33 % of the lists' sectors come from the cache, and 37 % now; with 104 KB of tables 53 us).  The gathers were 85 % of the
// load unit's time: the parts of a class stand in tables of their own, where 32-byte records lay in one of four banks.
#include "llvq_internal.cuh"
#include "llvq_unrank.cuh"

namespace llvq {
namespace {

constexpr int kExpandWarps = 32;
constexpr int kExpandThreads = kExpandWarps * 32;
// A tile under construction.  Until a block is un-ranked, its first two words of codes hold the rank in its class (47 bits),
// the class << 47 and the gain << 56, the third the class's flags.
struct WarpScratch {
    uint32_t nat[4][3][32];                // [block of the piece][codes of eight coordinates][row, see `cell`]
    uint16_t hdr[4][32];                   // its header
    uint32_t exceptions[4];                // 10-byte layout: rows of a block without a window
    uint8_t place[128];                    // 32 * block + row: odd type from the front, even from the back
    // neighbouring words' rows lie eight banks apart: the four lanes of a quad read two words of a block, or of two
    __device__ __forceinline__ uint32_t &cell(int q, int j, int row) { return nat[q][j][row ^ ((q + j) & 1) << 3]; }
};
constexpr int kExpandSmem = kUnrankSharedBytes + kExpandWarps * (int)sizeof(WarpScratch);

__device__ __forceinline__ void copy_blob(uint8_t *to, const uint8_t *from, int bytes) {
    for (int i = threadIdx.x * 16; i < bytes; i += blockDim.x * 16)
        *reinterpret_cast<uint4 *>(to + i) = __ldg(reinterpret_cast<const uint4 *>(from + i));
}

__device__ __forceinline__ bool code_names_point(uint64_t code, uint64_t num_points) {
    return (code >> 48) == 0 && (code & ((1ull << kIndexBits) - 1)) < num_points;
}

// two header pairs (each two 16-bit fields of which the low byte counts) -> four bytes
__device__ __forceinline__ uint32_t bytes4(uint32_t a, uint32_t b) {
    return (a & 0xffu) | ((a >> 8) & 0xff00u) | ((b & 0xffu) << 16) | ((b << 8) & 0xff000000u);
}

// The window base of the 10-byte layout for a block's 24 four-bit codes (three words of eight nibbles): the
// smallest o in 3..6 with o <= the smallest code and the largest code <= o + 7; 0 if there is none.
__device__ __forceinline__ uint32_t window_base(const uint32_t cw[3]) {
    uint32_t lo = 15u, hi = 0u;
#pragma unroll 1
    for (int n = 0; n < 32; n += 4)
#pragma unroll
        for (int j = 0; j < 3; j++) {
            const uint32_t u = (cw[j] >> n) & 15u;
            lo = min(lo, u);
            hi = max(hi, u);
        }
    const uint32_t o = max(3u, hi > 7u ? hi - 7u : 0u);
    return o <= min(6u, lo) ? o : 0u;
}
// the same for a block that is known to have one: it is 3 and one more for every one of 11, 12, 13 that a code reaches
__device__ __forceinline__ uint32_t window_base_of_fitting(const uint32_t cw[3]) {
    uint32_t r11 = 0, r12 = 0, r13 = 0;
#pragma unroll
    for (int j = 0; j < 3; j++) {
        const uint32_t low = cw[j] & 0x77777777u, high = cw[j] & 0x88888888u;
        r11 |= (low + 0x55555555u) & high;
        r12 |= (low + 0x44444444u) & high;
        r13 |= (low + 0x33333333u) & high;
    }
    return 3u + (r11 != 0u) + (r12 != 0u) + (r13 != 0u);
}

__device__ __forceinline__ void unrank(const UnrankView &v, const UnrankDesc &d, uint64_t r, Point &p) {
    if (d.flags & 1u) unrank_odd(v, d, r, p); else unrank_even(v, d, r, p);
}

// LAYOUT = LLVQ_PLANES, LLVQ_PLANES13 (the same code words, the header one byte) or LLVQ_PLANES10X (tiles of
// three-bit window codes, the blocks a window cannot hold listed in the exception table; the leftover blocks as in
// LLVQ_PLANES13).  A warp's piece is a tile (four blocks of a row group), the pair after the tiles or the single at the end
// (see include/llvq.h).  For LLVQ_PLANES10X `index` holds, on entry, every tile's first entry in the table (or the
// capacity, where that is less), and `capacity` is the number of entries the table has room for.
template <int LAYOUT>
__global__ void __launch_bounds__(kExpandThreads, 1)
expand_planes_kernel(UnrankView global, uint64_t num_points, const uint64_t *__restrict__ codes, int64_t rows, int64_t nb, uint32_t total_pieces,
                     uint8_t *__restrict__ out, uint32_t *bad_count, uint32_t *ctx_bad, const uint32_t *index, uint4 *table, uint32_t capacity) {
    constexpr bool COMPACT = LAYOUT != LLVQ_PLANES, OVERLAY = LAYOUT == LLVQ_PLANES10X;
    constexpr int kCell = COMPACT ? kCell13Bytes : kCellBytes, kTile = OVERLAY ? kTile10Bytes : (COMPACT ? kTile13Bytes : kTileBytes);
    extern __shared__ __align__(16) uint8_t smem[];
    copy_blob(smem, global.blob, kUnrankSharedBytes);
    UnrankView v = global;
    v.blob = smem;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    WarpScratch &s = reinterpret_cast<WarpScratch *>(smem + kUnrankSharedBytes)[warp];
    // the tables are the library's: they are copied while the previous kernel of the stream ends
    asm volatile("griddepcontrol.wait;" ::: "memory");
    __syncthreads();

    const uint32_t tiles = (uint32_t)(nb / kTileCells), left = (uint32_t)(nb % kTileCells);
    const uint32_t pieces = tiles + (left >= 2 ? 1 : 0) + (left & 1);
    const int g = lane >> 2, t = lane & 3;
    uint32_t bad = 0;
    // The CTA's pieces (every gridDim-th), a warp a piece and round.  A piece is a chain of some ten microseconds, however few
    // run: where the last round has work for half of the warps or a quarter, two or four share a piece, each its blocks
    // (500 x 1000: 7.5 us; before the tables were made smaller 8.3, 14.8 without; 17408 x 5120: 117, 121; a last round of 26 pieces,
    // 9728 x 2560: 38.0, 37.9).
    // `own` = the blocks of the piece that are this warp's, a bit each, and 16 (0: no piece left), `share` = log2 of the warps on it.
    const uint32_t mine = (total_pieces - blockIdx.x + gridDim.x - 1) / gridDim.x, full = mine / kExpandWarps * kExpandWarps;
    const int last_share = mine - full <= kExpandWarps / 4 ? 2 : (mine - full <= kExpandWarps / 2 ? 1 : 0);
    uint32_t base = 0, piece = 0, own = 0;
    int share = 0;
    // a piece's codes are loaded while the piece before it is un-ranked
    uint64_t code[4];
    auto next_piece = [&]() {
        uint32_t at = base + warp;
        own = 15u;
        if (base >= full) {
            share = last_share;
            at = base + (warp >> share);
            own = share == 0 ? 15u : (share == 1 ? 3u << (2 * (warp & 1)) : 1u << (warp & 3));
        }
        base += kExpandWarps;
        piece = at * gridDim.x + blockIdx.x;
        const uint32_t rg = piece / pieces, u = piece % pieces;
        const int64_t row = (int64_t)rg * kRowsPerGroup + lane;
        const int64_t b0 = u < tiles ? (int64_t)u * kTileCells : (left >= 2 && u == tiles ? (int64_t)tiles * kTileCells : nb - 1);
        own = at < mine ? (own & (u < tiles ? 15u : (left >= 2 && u == tiles ? 3u : 1u))) | 16u : 0u;
        const uint32_t load = row < rows ? own : 0u;
#pragma unroll
        for (int q = 0; q < 4; q++) code[q] = (load >> q & 1u) ? __ldg(codes + row * nb + b0 + q) : 0ull;
    };
    next_piece();
    while (own) {                                                  // the same for all warps that share a piece
        const int now_share = share, part = warp & ((1 << share) - 1);
        const uint32_t now_own = own;
        WarpScratch &n = (&s)[-part];                              // where the piece's codes wait
        auto meet = [&]() {                                        // the warps that share the piece
            if (now_share == 0) __syncwarp();
            else asm volatile("bar.sync %0, %1;" ::"r"(warp >> now_share), "r"(32 << now_share) : "memory");
        };
        if (now_share) meet();                                     // the first warp's last piece is written
        const uint32_t rg = piece / pieces, u = piece % pieces;
        const bool row_exists = (int64_t)rg * kRowsPerGroup + lane < rows;
        uint8_t *grp = out + (size_t)rg * ((size_t)tiles * kTile + (size_t)left * kCell);
        const bool is_tile = u < tiles;
        const bool is_pair = !is_tile && left >= 2 && u == tiles;
        const bool single = !is_tile && !is_pair;
        uint32_t next_entry = 0;                                   // OVERLAY: where this tile's next exception goes
        if (OVERLAY && is_tile) next_entry = index[(size_t)rg * tiles + u];

        // ---- class of every block, listed by type
        int n_odd = 0, n_even = 0;
        if (OVERLAY && lane < 4 && (now_own >> lane & 1u)) n.exceptions[lane] = 0;
#pragma unroll
        for (int q = 0; q < 4; q++) {
            if (!(now_own >> q & 1u)) continue;
            const bool valid = row_exists && code_names_point(code[q], num_points);
            bool odd = false;
            if (valid) {
                const uint64_t idx = code[q] & ((1ull << kIndexBits) - 1);
                const int c = find_class(v, idx);
                const uint32_t flags = blob_at<uint32_t>(v, kUnrankFlags, c);
                odd = flags & 1u;
                const uint64_t entry = (idx - blob_at<uint64_t>(v, kUnrankBase, c)) | (uint64_t)c << 47 | ((code[q] >> kIndexBits) & 1) << 56;
                n.cell(q, 0, lane) = (uint32_t)entry;
                n.cell(q, 1, lane) = (uint32_t)(entry >> 32);
                n.cell(q, 2, lane) = flags;
            } else {
                bad += row_exists;
                // the empty record
                const uint32_t zero_code = OVERLAY && is_tile ? 0u : 0x88888888u;
#pragma unroll
                for (int j = 0; j < 3; j++) n.cell(q, j, lane) = zero_code;
                n.hdr[q][lane] = COMPACT ? 0u : (uint16_t)kEmptyClass;
            }
            const uint32_t of_odd = __ballot_sync(0xffffffffu, valid && odd), of_even = __ballot_sync(0xffffffffu, valid && !odd);
            const uint32_t before = (1u << lane) - 1u;
            if (valid) s.place[odd ? n_odd + __popc(of_odd & before) : 127 - n_even - __popc(of_even & before)] = (uint8_t)(32 * q + lane);
            n_odd += __popc(of_odd);
            n_even += __popc(of_even);
        }
        __syncwarp();
        next_piece();

        // ---- un-rank: 32 blocks of a type at a time
        auto finish = [&](uint32_t place, uint64_t entry, const UnrankDesc &d, const Point &p, bool odd) {
            const uint32_t q = place >> 5, row = place & 31u;
            const uint32_t cls = (uint32_t)(entry >> 47) & 511u, gain = (uint32_t)(entry >> 56) & 1u;
            uint32_t cw[3];
#pragma unroll
            for (int j = 0; j < 3; j++) cw[j] = point_codes(p, j, odd);
            const uint32_t shell = (d.flags >> 16) & 15u;
            uint32_t hdr = COMPACT ? shell | (uint32_t)odd << 4 | gain << 5 : cls | gain << 9;
            if (OVERLAY && is_tile) {
                const uint32_t window = d.flags >> 20;
                const uint32_t o = window == kWindowAlways ? window_base_of_fitting(cw) : (window == kWindowDepends ? window_base(cw) : 0u);
                if (o) {
                    // no borrow between nibbles: every code is at least o
#pragma unroll
                    for (int j = 0; j < 3; j++) cw[j] -= o * 0x11111111u;
                    // the short record's header byte: the shell above, and below it window, parity and gain mixed with the shell
                    hdr = ((o - 3u) | (uint32_t)odd << 2 | gain << 3) ^ shell | shell << 4;
                } else {
                    atomicOr(&n.exceptions[q], 1u << row);
                }
            }
#pragma unroll
            for (int j = 0; j < 3; j++) n.cell(q, j, row) = cw[j];
            n.hdr[q][row] = (uint16_t)hdr;
        };
        auto waiting = [&](uint32_t place) -> uint64_t { return n.cell(place >> 5, 0, place & 31u) | (uint64_t)n.cell(place >> 5, 1, place & 31u) << 32; };
#pragma unroll 1
        for (int i = lane; i < n_odd; i += 32) {
            const uint32_t place = s.place[i];
            const uint64_t entry = waiting(place);
            UnrankDesc d;                                          // nothing else of it is read
            d.flags = n.cell(place >> 5, 2, place & 31u);
            Point p;
            unrank_odd(v, d, entry & ((1ull << 47) - 1), p);
            finish(place, entry, d, p, true);
        }
#pragma unroll 1
        for (int i = lane; i < n_even; i += 32) {
            const uint32_t place = s.place[127 - i];
            const uint64_t entry = waiting(place);
            const uint32_t cls = (uint32_t)(entry >> 47) & 511u;
            const UnrankPerms perms = blob_at<UnrankPerms>(v, kUnrankPerms, cls);
            const UnrankFirsts firsts = blob_at<UnrankFirsts>(v, kUnrankFirsts, cls);
            const UnrankDesc d = {n.cell(place >> 5, 2, place & 31u), perms.perm_a, perms.perm_b, perms.inv_a, perms.inv_b,
                                  firsts.a_golay & 0xffffu, firsts.b, firsts.a_golay >> 16};
            Point p;
            unrank_even(v, d, entry & ((1ull << 47) - 1), p);
            finish(place, entry, d, p, false);
        }
        meet();
        if (part) break;                                           // a shared piece is the last
        if (OVERLAY && is_tile) {
            // the tile's exceptions go to the table in the order block, row, and leave an empty short record
#pragma unroll 1
            for (int q = 0; q < 4; q++) {
                const uint32_t rows_out = n.exceptions[q];
                if ((rows_out >> lane) & 1u) {
                    const uint32_t at = next_entry + __popc(rows_out & ((1u << lane) - 1u));
                    if (at < capacity)
                        table[at] = make_uint4(n.hdr[q][lane] | (uint32_t)lane << 8 | (u * kTileCells + q) << 13, n.cell(q, 0, lane), n.cell(q, 1, lane), n.cell(q, 2, lane));
                    n.cell(q, 0, lane) = n.cell(q, 1, lane) = n.cell(q, 2, lane) = 0u;
                    n.hdr[q][lane] = 0;
                }
                next_entry += __popc(rows_out);
            }
            __syncwarp();
        }

        // ---- gather the words of the piece: lane 4g+t
        // the word of codes that holds positions kappa0..kappa0+3 (kappa0 = 4t + a multiple of 16: the half of the word is t & 1)
        // of row (m, e, g) in the half-step whose slots are blocks q0, q0+1
        auto codes_at = [&](int q0, int m, int e, int kappa0) -> uint32_t {
            const int slot = kappa0 / 24, i0 = kappa0 % 24;
            const int r = single ? 16 * slot + 8 * e + g : 16 * m + 8 * e + g;
            return n.cell(single ? q0 : q0 + slot, i0 >> 3, r);
        };
        auto header = [&](int q0, int m, int e, int slot) -> uint32_t {
            const int r = single ? 16 * slot + 8 * e + g : 16 * m + 8 * e + g;
            return n.hdr[single ? q0 : q0 + slot][r];
        };
        const uint32_t half_sel = (t & 1) ? 0x7362u : 0x5140u;
        // the lane's four nibbles of x to the low nibbles of four bytes, those of y to the high nibbles
        auto pair_up = [&](uint32_t x, uint32_t y) -> uint32_t {
            const uint32_t even = (x & 0x0f0f0f0fu) | ((y << 4) & 0xf0f0f0f0u), odd = ((x >> 4) & 0x0f0f0f0fu) | (y & 0xf0f0f0f0u);
            return __byte_perm(even, odd, half_sel);
        };
        auto half_step = [&](int q0, int m, uint32_t w[3], uint32_t &hw) {
            w[0] = pair_up(codes_at(q0, m, 0, 4 * t), codes_at(q0, m, 0, 16 + 4 * t));
            w[1] = pair_up(codes_at(q0, m, 1, 4 * t), codes_at(q0, m, 1, 16 + 4 * t));
            w[2] = pair_up(codes_at(q0, m, 0, 32 + 4 * t), codes_at(q0, m, 1, 32 + 4 * t));
            hw = header(q0, m, 0, t >> 1) | header(q0, m, 1, t >> 1) << 16;
        };
        if (OVERLAY && is_tile) {
            // Group(h, e, c): byte i = code i of row (m, e, g) at positions 16c + 4t + i (c < 2) or 32 + 4t + i of half-step h
            auto group = [&](int h, int e, int c) -> uint32_t {
                const uint32_t x = codes_at(2 * (h >> 1), h & 1, e, (c < 2 ? 16 * c : 32) + 4 * t);
                return __byte_perm(x & 0x0f0f0f0fu, (x >> 4) & 0x0f0f0f0fu, half_sel);
            };
            uint32_t V[9], hw[4];
#pragma unroll
            for (int k = 0; k < 8; k++) V[k] = group(k >> 1, k & 1, 0) | group(k >> 1, k & 1, 1) << 3;
            V[8] = group(0, 0, 2) | group(1, 0, 2) << 3;
            // the six groups left go to bits 6, 7: the low two bits of Xk to Vk, its third bit to V(6 + k / 2)
            const uint32_t X[6] = {group(0, 1, 2), group(1, 1, 2), group(2, 0, 2), group(2, 1, 2), group(3, 0, 2), group(3, 1, 2)};
#pragma unroll
            for (int k = 0; k < 6; k++) {
                V[k] |= (X[k] & 0x03030303u) << 6;
                V[6 + (k >> 1)] |= ((X[k] >> 2) & 0x01010101u) << (6 + (k & 1));
            }
#pragma unroll
            for (int h = 0; h < 4; h++) hw[h] = header(2 * (h >> 1), h & 1, 0, t >> 1) | header(2 * (h >> 1), h & 1, 1, t >> 1) << 16;
            uint8_t *tile = grp + (size_t)u * kTile;
            *reinterpret_cast<uint4 *>(tile + 16 * lane) = make_uint4(V[0], V[1], V[2], V[3]);
            *reinterpret_cast<uint4 *>(tile + 512 + 16 * lane) = make_uint4(V[4], V[5], V[6], V[7]);
            *reinterpret_cast<uint32_t *>(tile + 1024 + 4 * lane) = V[8];
            if ((t & 1) == 0) *reinterpret_cast<uint2 *>(tile + 1152 + 8 * (lane >> 1)) = make_uint2(bytes4(hw[0], hw[1]), bytes4(hw[2], hw[3]));
        } else if (is_tile) {
            uint32_t w[12], hw[4];
#pragma unroll
            for (int h = 0; h < 4; h++) half_step(2 * (h >> 1), h & 1, w + 3 * h, hw[h]);
            uint8_t *tile = grp + (size_t)u * kTile;
#pragma unroll
            for (int j = 0; j < 3; j++)
                *reinterpret_cast<uint4 *>(tile + 512 * j + 16 * lane) = make_uint4(w[4 * j], w[4 * j + 1], w[4 * j + 2], w[4 * j + 3]);
            if ((t & 1) == 0) {
                if (COMPACT) *reinterpret_cast<uint2 *>(tile + 1536 + 8 * (lane >> 1)) = make_uint2(bytes4(hw[0], hw[1]), bytes4(hw[2], hw[3]));
                else *reinterpret_cast<uint4 *>(tile + 1536 + 16 * (lane >> 1)) = make_uint4(hw[0], hw[1], hw[2], hw[3]);
            }
        } else if (is_pair) {
            uint8_t *pair = grp + (size_t)tiles * kTile;
            uint32_t hw[2];
#pragma unroll
            for (int m = 0; m < 2; m++) {
                uint32_t w[3];
                half_step(0, m, w, hw[m]);
#pragma unroll
                for (int q = 0; q < 3; q++) *reinterpret_cast<uint32_t *>(pair + 128 * (3 * m + q) + 4 * lane) = w[q];
                if (!COMPACT && (t & 1) == 0) *reinterpret_cast<uint32_t *>(pair + 768 + 8 * (lane >> 1) + 4 * m) = hw[m];
            }
            if (COMPACT && (t & 1) == 0) *reinterpret_cast<uint32_t *>(pair + 768 + 4 * (lane >> 1)) = bytes4(hw[0], hw[1]);
        } else {
            uint8_t *one = grp + (size_t)tiles * kTile + (left == 3 ? 2 * kCell : 0);
            uint32_t w[3], hw;
            half_step(0, 0, w, hw);
#pragma unroll
            for (int q = 0; q < 3; q++) *reinterpret_cast<uint32_t *>(one + 128 * q + 4 * lane) = w[q];
            if ((t & 1) == 0) {
                if (COMPACT) *reinterpret_cast<uint16_t *>(one + 384 + 2 * (lane >> 1)) = (uint16_t)((hw & 0xffu) | ((hw >> 8) & 0xff00u));
                else *reinterpret_cast<uint32_t *>(one + 384 + 4 * (lane >> 1)) = hw;
            }
        }
        __syncwarp();                                              // the scratch is free for the next piece
    }
    bad = __reduce_add_sync(0xffffffffu, bad);
    if (bad && lane == 0) {
        atomicAdd(ctx_bad, bad);                                   // the context's own count: llvq_status reports it
        if (bad_count) atomicAdd(bad_count, bad);
    }
}

// One-hot layout: a warp a cell (32 rows of a block column), a lane a row.
__global__ void __launch_bounds__(kExpandThreads, 1)
expand_onehot_kernel(UnrankView global, DeviceTables T, const uint64_t *__restrict__ codes, int64_t rows, int64_t nb, int64_t cells,
                     uint8_t *__restrict__ out, uint32_t *bad_count, uint32_t *ctx_bad) {
    extern __shared__ __align__(16) uint8_t smem[];
    copy_blob(smem, global.blob, kUnrankSharedBytes);
    UnrankView v = global;
    v.blob = smem;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    __syncthreads();
    uint32_t bad = 0;
    for (int64_t cell_id = (int64_t)warp * gridDim.x + blockIdx.x; cell_id < cells; cell_id += (int64_t)kExpandWarps * gridDim.x) {
        const int64_t rg = cell_id / nb, b = cell_id % nb, row = rg * kRowsPerGroup + lane;
        uint32_t smask = 0, mask[4] = {0, 0, 0, 0}, cls = kEmptyClass, gain = 0;
        if (row < rows) {
            const uint64_t code = __ldg(codes + row * nb + b), idx = code & ((1ull << kIndexBits) - 1);
            if (code_names_point(code, T.num_points)) {
                cls = (uint32_t)find_class(v, idx);
                gain = (uint32_t)(code >> kIndexBits) & 1u;
                const UnrankDesc d = far_at<UnrankDesc>(v, kUnrankDescs, cls);
                const uint32_t odd = d.flags & 1u;
                Point p;
                unrank(v, d, idx - blob_at<uint64_t>(v, kUnrankBase, cls), p);
                const int nd = T.desc[cls].ndist;
#pragma unroll
                for (int j = 0; j < 3; j++) smask |= gather8(p.neg[j]) << (8 * j);
#pragma unroll
                for (int l = 1; l < 5; l++) {
                    // magnitude 2j + 1 (odd type) or 2h: the nibbles that equal the level's
                    const uint32_t level = (uint32_t)(T.desc[cls].dist[l] - odd) >> 1;
#pragma unroll
                    for (int j = 0; j < 3; j++) {
                        const uint32_t x = p.mag[j] ^ (level * 0x11111111u);
                        if (l < nd) mask[l - 1] |= (gather8((x | x >> 1 | x >> 2) & 0x11111111u) ^ 0xffu) << (8 * j);
                    }
                }
            } else {
                bad++;
            }
        }
        uint32_t *cell = reinterpret_cast<uint32_t *>(out + (size_t)cell_id * kOneHotCellBytes);
        cell[0 * 32 + lane] = smask | (cls & 255u) << 24;
        cell[1 * 32 + lane] = mask[0] | (cls >> 8) << 24 | gain << 25;
        cell[2 * 32 + lane] = mask[1];
        cell[3 * 32 + lane] = mask[2];
        cell[4 * 32 + lane] = mask[3];
    }
    bad = __reduce_add_sync(0xffffffffu, bad);
    if (bad && lane == 0) {
        atomicAdd(ctx_bad, bad);
        if (bad_count) atomicAdd(bad_count, bad);
    }
}

// ---- the exception table of the 10-byte layout is filled in a fixed order, so its entries' places are known before
// they are written.  A warp a tile counts the tile's exceptions (lane = row): a bit of the class guide says of nearly every
// index (59 in 60 of the synthetic stream) that its classes hold none, the class settles most others, and only one block in
// some thousands is un-ranked (from the tables in global memory).  So the count streams the codes: bound HBM, 8 bytes a
// block.  INDEX: the count goes to the index entry after the tile's (the running sum over the index then gives every
// tile's first entry); else the counts are added up in total[0], and the last CTA (total[1] counts them) writes the sum to
// `host`, page-locked memory, and leaves both at zero.
// Blocks to look at wait in a list until there are thirty-two or the warp's tiles are through: a look's chain of dependent
// reads (3 us) is then paid once a warp, not once a tile.
constexpr int kCountWarps = 8;
template <bool INDEX>
__global__ void __launch_bounds__(kCountWarps * 32)
overlay_count_kernel(UnrankView v, uint64_t num_points, const uint64_t *__restrict__ codes, int64_t rows, int64_t nb, uint32_t total_tiles,
                     uint32_t *index, unsigned long long *total, volatile unsigned long long *host) {
    __shared__ uint32_t window[kGuideSlots / 32];
    __shared__ uint64_t list_all[kCountWarps][160];                // index of a block to look at
    __shared__ uint32_t tile_all[kCountWarps][160];                // and its tile
    for (int i = threadIdx.x; i < kGuideSlots / 32; i += blockDim.x) window[i] = __ldg(reinterpret_cast<const uint32_t *>(v.blob + kUnrankWindow) + i);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint64_t *list = list_all[warp];
    uint32_t *tile_of = tile_all[warp];
    const uint32_t tiles = (uint32_t)(nb / kTileCells);
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    __syncthreads();
    uint32_t sum = 0;
    int listed = 0;
    // looks at the last (at most 32) blocks of the list
    auto look = [&]() {
        __syncwarp();
        const int n = min(listed, 32);
        listed -= n;
        if (lane < n) {
            const uint64_t idx = list[listed + lane];
            const int c = find_class(v, idx);
            const UnrankDesc d = blob_at<UnrankDesc>(v, kUnrankDescs, c);
            bool exception = d.flags >> 20 == kWindowNever;
            if (d.flags >> 20 == kWindowDepends) {
                Point p;
                unrank(v, d, idx - blob_at<uint64_t>(v, kUnrankBase, c), p);
                const bool odd = d.flags & 1u;
                const uint32_t cw[3] = {point_codes(p, 0, odd), point_codes(p, 1, odd), point_codes(p, 2, odd)};
                exception = window_base(cw) == 0u;
            }
            if (exception) {
                if (INDEX) atomicAdd(index + tile_of[listed + lane] + 1, 1u);
                else sum++;
            }
        }
        __syncwarp();
    };
    uint64_t code[4], next[4];
    auto load = [&](uint32_t tile, uint64_t (&to)[4]) {
        const uint32_t rg = tile / tiles, u = tile - rg * tiles;
        const int64_t row = (int64_t)rg * kRowsPerGroup + lane;
#pragma unroll
        for (int q = 0; q < 4; q++) to[q] = (row < rows && tile < total_tiles) ? __ldcs(codes + row * nb + (int64_t)u * kTileCells + q) : ~0ull;
    };
    uint32_t tile = blockIdx.x * kCountWarps + warp;
    const uint32_t stride = kCountWarps * gridDim.x;
    load(tile, next);
    for (; tile < total_tiles; tile += stride) {
#pragma unroll
        for (int q = 0; q < 4; q++) code[q] = next[q];
        load(tile + stride, next);
        if (INDEX && lane == 0) index[(size_t)tile + 1] = 0u;      // before any addition to it, which the look's barrier puts behind
#pragma unroll
        for (int q = 0; q < 4; q++) {
            const uint64_t idx = code[q] & ((1ull << kIndexBits) - 1);
            const int slot = guide_slot(idx);
            const bool wanted = code_names_point(code[q], num_points) && ((window[slot >> 5] >> (slot & 31)) & 1u);
            const uint32_t votes = __ballot_sync(0xffffffffu, wanted);
            if (wanted) {
                const int at = listed + __popc(votes & ((1u << lane) - 1u));
                list[at] = idx;
                tile_of[at] = tile;
            }
            listed += __popc(votes);
        }
        while (listed >= 32) look();                               // at most 31 stay, and a tile adds at most 128
    }
    if (listed > 0) look();
    if (!INDEX) {
        sum = __reduce_add_sync(0xffffffffu, sum);
        if (lane == 0 && sum) {
            atomicAdd(total, (unsigned long long)sum);
            __threadfence();
        }
        __syncthreads();                                           // the CTA's sums are in
        if (threadIdx.x == 0 && atomicAdd(total + 1, 1ull) == gridDim.x - 1) {
            __threadfence();
            *host = atomicExch(total, 0ull);
            atomicExch(total + 1, 0ull);
        }
    }
}

// One CTA, between the count and the expansion: index[i + 1] = counts of the tiles up to i (index[0] = 0), in place, no
// further than the capacity (so that no reader looks past the table; an expansion that starts there writes nothing);
// the entries that will find no room are counted, and the bytes between the parts of the buffer zeroed.
__global__ void __launch_bounds__(1024) overlay_index_kernel(uint8_t *out, size_t records_end, size_t index_offset, size_t table_offset,
                                                             int64_t n, uint32_t capacity, uint32_t *overflow) {
    constexpr int kEach = 8, kRound = 1024 * kEach;                // entries a thread and a round
    uint32_t *index = reinterpret_cast<uint32_t *>(out + index_offset);
    __shared__ uint32_t warp_sum[32], staged[kRound + kRound / kEach];     // a word's pad after eight: consecutive threads' eights start in different banks
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    uint32_t carry = 0;                                            // the same in every thread
    uint32_t c[kEach];
    auto load = [&](int64_t base) {                                // a round's entries, neighbours to neighbours
#pragma unroll
        for (int j = 0; j < kEach; j++) {
            const int64_t at = base + j * 1024 + tid;
            c[j] = at < n ? index[at + 1] : 0u;
        }
    };
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    load(0);
    for (int64_t base = 0; base < n; base += kRound) {
#pragma unroll
        for (int j = 0; j < kEach; j++) staged[(j * 1024 + tid) + (j * 1024 + tid) / kEach] = c[j];
        __syncthreads();
        load(base + kRound);
        uint32_t mine = 0;
#pragma unroll
        for (int j = 0; j < kEach; j++) mine += staged[tid * (kEach + 1) + j];
        uint32_t incl = mine;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const uint32_t up = __shfl_up_sync(0xffffffffu, incl, off);
            if (lane >= off) incl += up;
        }
        if (lane == 31) warp_sum[warp] = incl;
        __syncthreads();
        const uint32_t w = warp_sum[lane];
        uint32_t run = carry + incl - mine + __reduce_add_sync(0xffffffffu, lane < warp ? w : 0u);
        carry += __reduce_add_sync(0xffffffffu, w);
#pragma unroll
        for (int j = 0; j < kEach; j++) {
            run += staged[tid * (kEach + 1) + j];
            staged[tid * (kEach + 1) + j] = min(run, capacity);
        }
        __syncthreads();
#pragma unroll
        for (int j = 0; j < kEach; j++) {
            const int64_t at = base + j * 1024 + tid;
            if (at < n) index[at + 1] = staged[(j * 1024 + tid) + (j * 1024 + tid) / kEach];
        }
        __syncthreads();                                           // the shared words are free for the next round
    }
    if (tid == 0) {
        index[0] = 0;
        if (carry > capacity) atomicAdd(overflow, carry - capacity);
    }
    for (size_t i = records_end + tid; i < index_offset; i += blockDim.x) out[i] = 0;
    for (size_t i = index_offset + (size_t)(n + 1) * 4 + tid; i < table_offset; i += blockDim.x) out[i] = 0;
}

// CTAs of a grid whose warps walk over `work` pieces: `per_sm` a multiprocessor, or one a piece if there are fewer
unsigned grid_for(const llvq_ctx *ctx, int64_t work, int per_sm = 1) {
    const int64_t most = (int64_t)ctx->sm_count * per_sm;
    return (unsigned)(work < most ? work : most);
}

// Launches with programmatic stream serialization, if the context has it switched on.  The kernels wait for their
// predecessor ahead of all they read but the library's tables.  The expansions let no kernel start before they end: what
// follows may be a GEMV of another context, which reads records ahead of its own wait.
template <typename... P, typename... A>
cudaError_t launch(const llvq_ctx *ctx, void (*kernel)(P...), unsigned grid, int threads, int smem, cudaStream_t s, A... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = (size_t)smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = ctx->use_pdl ? 1 : 0;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

}  // namespace

int expand_configure() {
    const int bytes = kExpandSmem;
    if (cudaFuncSetAttribute(expand_planes_kernel<LLVQ_PLANES>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) != cudaSuccess) return -1;
    if (cudaFuncSetAttribute(expand_planes_kernel<LLVQ_PLANES13>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) != cudaSuccess) return -1;
    if (cudaFuncSetAttribute(expand_planes_kernel<LLVQ_PLANES10X>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) != cudaSuccess) return -1;
    return cudaFuncSetAttribute(expand_onehot_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kUnrankSharedBytes) == cudaSuccess ? 0 : -1;
}

cudaError_t launch_overlay_count(const llvq_ctx *ctx, const uint64_t *codes, int64_t rows, int64_t nb, unsigned long long *counter,
                                 unsigned long long *host, cudaStream_t s) {
    const int64_t groups = (rows + kRowsPerGroup - 1) / kRowsPerGroup, tiles = nb / kTileCells;
    if (tiles == 0) return cudaSuccess;
    return launch(ctx, overlay_count_kernel<false>, grid_for(ctx, (groups * tiles + kCountWarps - 1) / kCountWarps, 8), kCountWarps * 32, 0, s, ctx->unrank,
                  ctx->dev.num_points, codes, rows, nb, groups * tiles, nullptr, counter, host);
}

cudaError_t launch_expand(const llvq_ctx *ctx, int layout, const uint64_t *codes, int64_t rows, int64_t nb,
                          void *out, size_t out_bytes, uint32_t *bad_count, cudaStream_t s) {
    const int64_t groups = (rows + kRowsPerGroup - 1) / kRowsPerGroup;
    uint8_t *o8 = (uint8_t *)out;
    const UnrankView v = ctx->unrank;
    const uint64_t points = ctx->dev.num_points;
    if (layout == LLVQ_ONEHOT)
        return launch(ctx, expand_onehot_kernel, grid_for(ctx, groups * nb), kExpandThreads, kUnrankSharedBytes, s, v, ctx->dev, codes, rows, nb, groups * nb, o8,
                      bad_count, ctx->bad_codes);
    const int64_t left = nb % kTileCells, tiles = nb / kTileCells;
    const int64_t pieces = groups * (tiles + (left >= 2 ? 1 : 0) + (left & 1));
    const unsigned grid = grid_for(ctx, pieces);
    if (layout == LLVQ_PLANES10X) {
        const size_t index_offset = overlay_index_offset(rows, nb), table_offset = overlay_table_offset(rows, nb);
        uint32_t *index = reinterpret_cast<uint32_t *>(o8 + index_offset);
        uint4 *table = reinterpret_cast<uint4 *>(o8 + table_offset);
        const size_t room = (out_bytes - table_offset) / 16;
        const uint32_t capacity = room > 0xffffffffull ? 0xffffffffu : (uint32_t)room;
        // count the tiles' exceptions into the index, turn the counts into first entries, expand
        if (tiles > 0) {
            const cudaError_t r = launch(ctx, overlay_count_kernel<true>, grid_for(ctx, (groups * tiles + kCountWarps - 1) / kCountWarps, 8), kCountWarps * 32, 0, s, v, points,
                                         codes, rows, nb, groups * tiles, index, nullptr, nullptr);
            if (r != cudaSuccess) return r;
        }
        const cudaError_t r = launch(ctx, overlay_index_kernel, 1u, 1024, 0, s, o8, (size_t)groups * overlay_group_bytes(nb), index_offset, table_offset, groups * tiles,
                                     capacity, ctx->overflow);
        if (r != cudaSuccess) return r;
        return launch(ctx, expand_planes_kernel<LLVQ_PLANES10X>, grid, kExpandThreads, kExpandSmem, s, v, points, codes, rows, nb, pieces, o8, bad_count, ctx->bad_codes, index,
                      table, capacity);
    }
    if (layout == LLVQ_PLANES13)
        return launch(ctx, expand_planes_kernel<LLVQ_PLANES13>, grid, kExpandThreads, kExpandSmem, s, v, points, codes, rows, nb, pieces, o8, bad_count, ctx->bad_codes, nullptr,
                      nullptr, 0u);
    return launch(ctx, expand_planes_kernel<LLVQ_PLANES>, grid, kExpandThreads, kExpandSmem, s, v, points, codes, rows, nb, pieces, o8, bad_count, ctx->bad_codes, nullptr, nullptr,
                  0u);
}

}  // namespace llvq
