// pgz_kernels.cu -- sm_103a kernels of the two-pass parallel gzip decompression
// (Kerbiriou & Chikhi, arXiv 1905.07224, Section "Full file decompression in
// two passes (pugz)").
//
//   k_sync      pass 1a: per part, the first bit of [lo, hi) where a DEFLATE
//               block starts (Section "Detection of DEFLATE block start
//               positions", Appendix "DEFLATE block decompression checks"):
//               each warp of the part's team filters windows of 1024 bit
//               offsets (32 per lane, bit-parallel header tests), the survivors'
//               headers are checked one per lane, and the lowest valid
//               candidate's whole block is then decoded as the final check --
//               into the part's own copy map, so pass 1 resumes after it.
//   k_inflate   pass 1b: the blocks of part i up to the next part's block
//               start.  One team (a block of 2 to 16 warps) per part: the lanes
//               decode segments of a DEFLATE block in parallel and meet (see
//               par_block), then write the tokens' copy map: where a token's
//               output starts, its byte or the distance to its source.  No
//               symbol is read, so no window is kept.
//   k_exec      pass 1c: decode(C_i, w^_i) (Algorithm "DEFLATE decompression"
//               with the symbolic context [U_0..U_32767]) finished from the
//               copy map, in place: one block per part, the last 32 KiB of the
//               part's symbols in shared memory.  A source before the part
//               start p < 0 is the placeholder U_{32768+p}, computed, not
//               stored.
//   k_plan      output offsets of the parts (prefix of their lengths), error
//               aggregation, ISIZE and capacity checks.
//   k_chain_*   pass 2a: w_{i+1} from w_i and the tail of D_i (Section "Full
//               file decompression in two passes").  Each part's tail is a map
//               from w_i to w_{i+1} whose entries are bytes or indices; maps
//               compose, so groups of parts (and groups of groups) are composed
//               in parallel, then expanded level by level.
//   k_translate pass 2b: U_j -> w_i[j] for every symbol, written to the
//               final output with 8-byte aligned stores (HBM-bound).
//   k_crc       CRC-32 (RFC 1952) of the output: raw CRCs of 32-byte pieces,
//               combined by multiplication with x^(8n) mod P in GF(2) and
//               XOR-accumulated per member.
//   k_finalize  finished CRC-32 against the trailer.
//
// No kernel waits on another block or warp; every read of the compressed
// data, the symbol scratch and the output is bounds-checked.
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cuda_runtime.h>

#include "pgz_internal.h"
#include "../../include/pgz.h"

namespace pgz {
namespace {

constexpr uint32_t FULL = 0xffffffffu;
constexpr int LB = 10;          // literal/length lookup bits
constexpr int DB = 9;            // distance lookup bits
constexpr uint32_t kPoly = 0xEDB88320u;

// RFC 1951 3.2.7: order of the code-length code lengths
__constant__ uint8_t c_clorder[19] = {16, 17, 18, 0, 8, 7, 9, 6, 10, 5, 11, 4, 12, 3, 13, 2, 14, 1, 15};
// CRC-32 tables (filled by upload_crc_tables)
__constant__ uint32_t c_crc_tab[4][256];   // [0][b]: register after byte b from a zero register; [k]: k more zero bytes
__constant__ uint32_t c_x8[5][256];        // [d][v]: x^(8 v 256^d) mod P
__constant__ uint32_t c_lane_shift[32];    // x^(8*kPiece*k) mod P
__constant__ uint32_t c_seg_shift[4][256]; // [j][b]: (byte b at byte j of a register) x^(8*kCrcSeg) mod P

// Lookup entry of either code, one layout, so that a lane's step is the same
// for both: bits 0-4 the bits to drop (code and extra bits; both codes of two
// literals), 5-8 the code's length (the first literal's), 9-11 the kind, 12-31
// the payload -- LIT: the token (bytes in its low 16 bits, their count above),
// two literals when both codes fit the lookup width; LEN, DIST: the base to
// which the extra bits are added.
// Kinds from K_EOB on (bit 11 of the entry set) are rare: they end a parse, or need the longer codes.
enum : uint32_t { K_LIT = 0, K_LEN = 1, K_DIST = 2, K_EOB = 4, K_LONG = 5, K_BAD = 6 };
constexpr uint32_t kRare = 4u << 9;

// Shared memory of a team: the NW warps of one block, all on one part.
template <int NW>
struct TeamSmem {
    static constexpr uint32_t T = 32 * NW;
    // longest segment of a lane, in words; odd, so that the lanes' equal places lie in different banks
    static constexpr uint32_t kSegWords = NW <= 4 ? 29 : (NW == 8 ? 25 : 15);
    // token starts of a lane that the lanes before it can meet: every second one
    static constexpr uint32_t kList = NW <= 8 ? 48 : 40;
    // a round's words, or a block's header (at most 4510 bits) and its first round's
    static constexpr uint32_t kBits = T * kSegWords + 160;
    uint32_t tab[(1 << LB) + (1 << DB)];   // literal/length entries, then distance entries
    // the two codes (0 literal/length, 1 distance): entries of the symbols in (length, value) order, the
    // distance code's from kDistEnt on; ends of the codes of each length, left-aligned in 15 bits; index of a
    // length's first entry minus its first code
    static constexpr uint32_t kDistEnt = 288;
    uint32_t ent[kDistEnt + 32];
    uint32_t lim[2][16];
    int32_t sb[2][16];
    uint32_t allowed[8];
    uint32_t table_kind;
    // a header's results, a round's results
    int32_t h_status;
    uint32_t h_hlit, h_hdist, h_bits;
    uint16_t r_next[T], r_j[T];            // the lane a lane met (T: none), and at which of its tokens
    uint8_t r_cnt[T];                      // a lane's listed token starts
    uint32_t r_exc[NW], r_sum[NW], r_flags, r_end;
    // block-start search
    static constexpr uint32_t kCand = 4;                           // valid headers a warp reports per step
    static constexpr uint32_t kScanWindows = NW <= 8 ? 16 : 8;     // windows of 1024 bits a warp filters per step
    uint32_t c_n[NW], c_done[NW], c_at[NW][kCand];
    uint64_t c_resume[NW];
    int32_t q;                             // queue position
    union {
        uint8_t list[kList][T];            // every second token start of each lane's own parse, from its segment's
                                           // start, modulo 256 (a token takes at most 48 bits)
        struct {                           // a header's code-length code, its symbols, the lengths and their counts
            uint16_t cl[128], hs[320];
            uint8_t lens[320];
            uint32_t cnt[2][16];
        };
    };
    uint32_t bits[kBits + 2];              // staged words of the compressed data (during the block-start search, its
                                           // table of Kraft sums takes the last 256)
    __device__ __forceinline__ uint16_t* kraft3() { return reinterpret_cast<uint16_t*>(bits + kBits + 2 - 256); }
};

__device__ __forceinline__ uint64_t shfl64(uint64_t v, int src) {
    uint32_t lo = __shfl_sync(FULL, (uint32_t)v, src), hi = __shfl_sync(FULL, (uint32_t)(v >> 32), src);
    return ((uint64_t)hi << 32) | lo;
}

// ---------------------------------------------------------------------------
// bit input: RFC 1951 3.1.1, LSB first; 32-bit words, bounds-checked, staged in
// shared memory.  Each lane of the parallel decoder reads at its own place: a
// load from global memory there would stall the whole warp on whichever lane's
// line is missing, at every step.
// ---------------------------------------------------------------------------
struct Input {
    const uint32_t* w;   // the member's bytes as 32-bit words (4-byte aligned)
    const uint8_t* b;
    uint64_t nbytes;
    uint64_t nfull;      // words wholly inside the member

    __device__ __forceinline__ Input(const uint8_t* gz, uint64_t len)
        : w(reinterpret_cast<const uint32_t*>(gz)), b(gz), nbytes(len), nfull(len >> 2) {}
    __device__ __forceinline__ uint32_t word(uint64_t i) const {
        if (i < nfull) return __ldg(w + i);
        uint32_t v = 0;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const uint64_t p = i * 4 + k;
            if (p < nbytes) v |= (uint32_t)__ldg(b + p) << (8 * k);
        }
        return v;
    }
};

// n words of the input from word w0 on into S.bits, by the whole team (zeros past the member's end)
template <int NW>
__device__ void stage(TeamSmem<NW>& S, const Input& in, uint64_t w0, uint32_t n) {
    constexpr uint32_t T = 32 * NW;
    __syncthreads();
    uint32_t i = threadIdx.x;
    if (w0 + n <= in.nfull) {
        for (; i + 7 * T < n; i += 8 * T) {
            uint32_t v[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) v[k] = __ldg(in.w + w0 + i + k * T);
#pragma unroll
            for (int k = 0; k < 8; ++k) S.bits[i + k * T] = v[k];
        }
    }
    for (; i < n; i += T) S.bits[i] = in.word(w0 + i);
    __syncthreads();
}

// a reader at bit p of the staged words: 32 bits from p on in x()
struct Bits {
    uint32_t p, w0, w1;
    __device__ __forceinline__ void seek(const uint32_t* bits, uint32_t at) {
        p = at;
        w0 = bits[at >> 5];
        w1 = bits[(at >> 5) + 1];
    }
    __device__ __forceinline__ uint32_t x() const { return __funnelshift_r(w0, w1, p); }
    __device__ __forceinline__ void drop(const uint32_t* bits, uint32_t n) {   // n <= 32
        const uint32_t q = p + n;
        if ((q ^ p) >> 5) {
            w0 = w1;
            w1 = bits[(q >> 5) + 1];
        }
        p = q;
    }
};

// ---------------------------------------------------------------------------
// canonical Huffman codes (RFC 1951 3.2.2)
// ---------------------------------------------------------------------------
// entries of the two codes (RFC 1951 3.2.5): length codes 257..285 and distance codes 0..29 by their rule --
// four (two) codes per number of extra bits
__device__ __forceinline__ uint32_t lit_entry(uint32_t s, uint32_t L) {
    if (s < 256) return ((0x10000u | s) << 12) | (K_LIT << 9) | (L << 5) | L;
    if (s == 256) return (K_EOB << 9) | (L << 5) | L;
    if (s > 285) return (K_BAD << 9) | 1u;
    const uint32_t k = s - 257;
    if (k < 8) return ((k + 3) << 12) | (K_LEN << 9) | (L << 5) | L;
    if (k == 28) return (258u << 12) | (K_LEN << 9) | (L << 5) | L;
    const uint32_t E = (k - 4) >> 2;
    return ((((4 + (k & 3u)) << E) + 3) << 12) | (K_LEN << 9) | (L << 5) | (L + E);
}
__device__ __forceinline__ uint32_t dist_entry(uint32_t s, uint32_t L) {
    if (s > 29) return (K_BAD << 9) | 1u;
    if (s < 4) return ((s + 1) << 12) | (K_DIST << 9) | (L << 5) | L;
    const uint32_t E = (s - 2) >> 1;
    return ((((2 + (s & 1u)) << E) + 1) << 12) | (K_DIST << 9) | (L << 5) | (L + E);
}

// the code that prefixes v (15 code bits, first bit most significant): its length (MAX + 1: none so short) from the
// ends of the codes of each length
template <int MAX>
__device__ __forceinline__ uint32_t code_length(uint32_t v, const uint32_t* lim) {
    uint32_t L = 1;
#pragma unroll
    for (int l = 1; l <= MAX; ++l) L += v >= lim[l];
    return L;
}

// a code longer than the lookup width (or none) of code d: its entry
template <int NW>
__device__ __forceinline__ uint32_t long_entry(const TeamSmem<NW>& S, uint32_t x, uint32_t d) {
    const uint32_t v = __brev(x) >> 17;
    const uint32_t* lim = S.lim[d];
    uint32_t L = DB + 1;
#pragma unroll
    for (int l = DB + 1; l <= 15; ++l) L += v >= lim[l];
    if (L > 15) return (K_BAD << 9) | 1u;
    return S.ent[(int32_t)(v >> (15 - L)) + S.sb[d][L]];
}

// One warp: code ends of n code lengths whose counts per length are known, and the entries of the symbols in
// (length, value) order, from ent[off] on.
template <typename Make>
__device__ __forceinline__ void sort_code(const uint8_t* lens, int n, uint32_t* cnt, uint32_t* lim, int32_t* sb,
                                          uint32_t* ent, uint32_t off, Make make, int lane) {
    uint32_t code = 0, prev = 0, my_off = 0;
#pragma unroll
    for (int L = 1; L <= 15; ++L) {
        const uint32_t c = cnt[L];
        code = (code + prev) << 1;
        prev = c;
        if (lane == L) {
            lim[L] = (code + c) << (15 - L);
            sb[L] = (int32_t)off - (int32_t)code;
            my_off = off;
        }
        off += c;
    }
    __syncwarp();
    if (lane < 16) cnt[lane] = my_off;             // next index of each length
    __syncwarp();
    for (int s0 = 0; s0 < n; s0 += 32) {
        const int s = s0 + lane;
        const uint32_t l = (s < n) ? lens[s] : 0u;
        if (!__any_sync(FULL, l != 0)) continue;       // most values of a byte do not occur in a text
        const uint32_t peers = __match_any_sync(FULL, l);
        const uint32_t rank = __popc(peers & ((1u << lane) - 1u));
        const uint32_t base = cnt[l];
        if (s < n && l) ent[base + rank] = make((uint32_t)s, l);
        __syncwarp();
        if (rank == 0 && l) cnt[l] = base + __popc(peers);
        __syncwarp();
    }
}

// Both codes of a block from their lengths (S.lens: hlit literal/length, then hdist distance lengths), by the
// whole team: counts, then one warp per code sorts, then every thread fills its share of the lookup table by
// the ends of the codes.  A sum of lengths at most 1 has been checked (or is that of the fixed code).
template <int NW>
__device__ void build_tables(TeamSmem<NW>& S, uint32_t hlit, uint32_t hdist) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid < 32) S.cnt[tid >> 4][tid & 15] = 0;
    __syncthreads();
    for (uint32_t s = tid; s < hlit + hdist; s += 32 * NW) {
        const uint32_t l = S.lens[s];
        if (l) atomicAdd(&S.cnt[s >= hlit][l], 1u);
    }
    __syncthreads();
    if (warp == 0) sort_code(S.lens, (int)hlit, S.cnt[0], S.lim[0], S.sb[0], S.ent, 0, lit_entry, lane);
    if (warp == 1)
        sort_code(S.lens + hlit, (int)hdist, S.cnt[1], S.lim[1], S.sb[1], S.ent, TeamSmem<NW>::kDistEnt, dist_entry, lane);
    __syncthreads();
    for (uint32_t x = tid; x < (1u << LB); x += 32 * NW) {         // x: stream bits, the first least significant
        const uint32_t v = __brev(x) >> 17;                        // the same, left-aligned in 15 bits
        const uint32_t L = code_length<LB>(v, S.lim[0]);
        uint32_t e = K_LONG << 9;
        if (L <= LB) {
            e = S.ent[(int32_t)(v >> (15 - L)) + S.sb[0][L]];
            if (((e >> 9) & 7u) == K_LIT) {                        // a second literal inside the lookup width?
                const uint32_t v2 = (v << L) & 0x7fffu, L2 = code_length<LB>(v2, S.lim[0]);
                if (L + L2 <= LB) {
                    const uint32_t e2 = S.ent[(int32_t)(v2 >> (15 - L2)) + S.sb[0][L2]];
                    if (((e2 >> 9) & 7u) == K_LIT)
                        e = (0x20000u << 12) | ((e2 & 0xff000u) << 8) | (e & 0xff000u) | (K_LIT << 9) | (L << 5) | (L + L2);
                }
            }
        }
        S.tab[x] = e;
    }
    for (uint32_t x = tid; x < (1u << DB); x += 32 * NW) {
        const uint32_t v = __brev(x) >> 17;
        const uint32_t L = code_length<DB>(v, S.lim[1]);
        S.tab[(1 << LB) + x] = L <= DB ? S.ent[(int32_t)(v >> (15 - L)) + S.sb[1][L]] : K_LONG << 9;
    }
    __syncthreads();
}

// A dynamic block's header up to its code lengths, by one warp (RFC 1951
// 3.2.7).  Reading of valid codes, as its producer zlib uses them: code-length
// code complete; literal/length code complete or one code of length 1, with an
// end-of-block code; distance code complete, one code of length 1, or empty.
template <int NW>
__device__ int read_lengths(TeamSmem<NW>& S, Bits& br, int lane, uint32_t& hlit, uint32_t& hdist) {
    uint32_t x = br.x();
    hlit = (x & 31u) + 257;
    hdist = ((x >> 5) & 31u) + 1;
    const uint32_t hclen = ((x >> 10) & 15u) + 4;
    br.drop(S.bits, 14);
    if (hlit > 286 || hdist > 30) return CE_DATA;
    // lane k reads the k-th code-length length; lane s then holds that of symbol s
    uint32_t mine = 0;
    const uint32_t n1 = hclen < 10 ? hclen : 10;
    if ((uint32_t)lane < n1) mine = (br.x() >> (3 * lane)) & 7;
    br.drop(S.bits, 3 * n1);
    if (hclen > 10) {
        if ((uint32_t)lane >= 10 && (uint32_t)lane < hclen) mine = (br.x() >> (3 * (lane - 10))) & 7;
        br.drop(S.bits, 3 * (hclen - 10));
    }
    uint32_t len = 0;
#pragma unroll
    for (int k = 0; k < 19; ++k) {
        const uint32_t l = __shfl_sync(FULL, mine, k);
        if (lane == c_clorder[k]) len = l;
    }
    if (__reduce_add_sync(FULL, len ? 128u >> len : 0u) != 128u) return CE_DATA;   // complete
    uint32_t lim[8], base[8], code = 0, off = 0, prev = 0, at = 0;
#pragma unroll
    for (int L = 1; L <= 7; ++L) {
        const uint32_t m = __ballot_sync(FULL, len == (uint32_t)L), c = __popc(m);
        code = (code + prev) << 1;
        prev = c;
        lim[L] = (code + c) << (7 - L);
        base[L] = off - code;
        if (len == (uint32_t)L) at = off + __popc(m & ((1u << lane) - 1u));
        off += c;
    }
    if (len) S.ent[at] = (uint32_t)lane;
    __syncwarp();
    // entry: bits 0-3 the bits to drop (code and repeat count), 4-6 the code's length, 7-10 the least repeat
    // count, 11-15 the symbol
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const uint32_t x = (uint32_t)lane + 32u * k, v = __brev(x) >> 25;
        uint32_t L = 1, b = base[1];
#pragma unroll
        for (int l = 1; l <= 6; ++l)
            if (v >= lim[l]) {
                L = l + 1;
                b = base[l + 1];
            }
        const uint32_t y = S.ent[(v >> (7 - L)) + b];
        const uint32_t ex = y < 16 ? 0u : (y == 16 ? 2u : (y == 17 ? 3u : 7u));
        S.cl[x] = (uint16_t)((L + ex) | (L << 4) | ((y < 16 ? 1u : (y == 18 ? 11u : 3u)) << 7) | (y << 11));
    }
    __syncwarp();
    // the chain of symbols, kept as short as it can be (every lane the same): symbol | repeat count << 5
    const uint32_t total = hlit + hdist;
    uint32_t i = 0, n = 0;
    while (i < total) {
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            if (u && i >= total) break;
            const uint32_t w = br.x(), e = S.cl[w & 127u], drop = e & 15u;
            const uint32_t rep = ((e >> 7) & 15u) + ((w & ((1u << drop) - 1u)) >> ((e >> 4) & 7u));
            br.drop(S.bits, drop);
            if (lane == 0) S.hs[n] = (uint16_t)((e >> 11) | (rep << 5));
            ++n;
            i += rep;
        }
    }
    if (i != total) return CE_DATA;
    __syncwarp();
    // the lengths, 32 symbols at a time: places by a prefix sum of the counts, a repeat's value from the last
    // symbol before it that is no repeat
    // (a run of zeros would take up to 138 turns: they are written beforehand)
    uint32_t at0 = 0, prev_val = 0xffu;
    bool bad = false;
    for (int k = lane; k < 320 / 4; k += 32) reinterpret_cast<uint32_t*>(S.lens)[k] = 0;
    __syncwarp();
    for (uint32_t k0 = 0; k0 < n; k0 += 32) {
        const uint32_t h = k0 + lane < n ? S.hs[k0 + lane] : 0u, y = h & 31u, rep = h >> 5;
        uint32_t incl = rep;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t x = __shfl_up_sync(FULL, incl, d);
            if (lane >= d) incl += x;
        }
        const uint32_t own = __ballot_sync(FULL, y != 16) & (FULL >> (31 - lane));   // values at or before mine
        const uint32_t from = __shfl_sync(FULL, y < 16 ? y : 0u, own ? 31 - __clz(own) : 0);
        const uint32_t val = own ? from : prev_val;
        bad |= val == 0xffu && rep;                    // a repeat before the first length
        const uint32_t at1 = at0 + incl - rep;
        for (uint32_t j = 0; j < (val ? rep : 0u); ++j) S.lens[at1 + j] = (uint8_t)val;
        at0 += __shfl_sync(FULL, incl, 31);
        prev_val = __shfl_sync(FULL, val, 31);
    }
    if (__any_sync(FULL, bad)) return CE_DATA;
    __syncwarp();
    // Kraft sums (units of 2^-15) with the counts above bit 20, longest lengths
    uint32_t kl = 0, kd = 0, ml = 0, md = 0;
    for (uint32_t k = lane; k < total; k += 32) {
        const uint32_t l = S.lens[k];
        const uint32_t v = l ? (1u << 20 << 3) + (32768u >> l) : 0u;
        if (k < hlit) {
            kl += v;
            ml = max(ml, l);
        } else {
            kd += v;
            md = max(md, l);
        }
    }
    kl = __reduce_add_sync(FULL, kl);
    kd = __reduce_add_sync(FULL, kd);
    ml = __reduce_max_sync(FULL, ml);
    md = __reduce_max_sync(FULL, md);
    const uint32_t sl = kl & 0x7fffffu, nl = kl >> 23, sd = kd & 0x7fffffu, nd = kd >> 23;
    if (S.lens[256] == 0) return CE_DATA;
    if (!(sl == 32768u || (nl == 1 && ml == 1))) return CE_DATA;
    if (!(sd == 32768u || nd == 0 || (nd == 1 && md == 1))) return CE_DATA;
    return CE_OK;
}

// the header of a dynamic block (at bit `at` of the staged words) and its tables; *bits: the header's bits
template <int NW>
__device__ int read_dynamic(TeamSmem<NW>& S, uint32_t at, uint32_t* bits) {
    if (threadIdx.x < 32) {
        uint32_t hlit = 0, hdist = 0;
        Bits br;
        br.seek(S.bits, at);
        const int st = read_lengths<NW>(S, br, threadIdx.x, hlit, hdist);
        if (threadIdx.x == 0) {
            S.h_status = st;
            S.h_hlit = hlit;
            S.h_hdist = hdist;
            S.h_bits = br.p - at;
            S.table_kind = 0;
        }
    }
    __syncthreads();
    const int st = S.h_status;
    *bits = S.h_bits;
    if (st) {
        __syncthreads();                       // S.h_* may be rewritten
        return st;
    }
    build_tables<NW>(S, S.h_hlit, S.h_hdist);
    return CE_OK;
}

// the fixed code of RFC 1951 3.2.6
template <int NW>
__device__ void build_fixed(TeamSmem<NW>& S) {
    __syncthreads();
    for (int s = threadIdx.x; s < 320; s += 32 * NW)
        S.lens[s] = (uint8_t)(s < 144 ? 8 : s < 256 ? 9 : s < 280 ? 7 : s < 288 ? 8 : 5);
    if (threadIdx.x == 0) S.table_kind = 1;
    __syncthreads();
    build_tables<NW>(S, 288, 32);
}

// ---------------------------------------------------------------------------
// copy map of one part: what the block decoder writes and k_exec turns into
// symbols in place.  At the position where a token's output starts, a u16: a
// byte (each literal), or kPH | (distance - 1) (a match), and the position's bit
// in the start bits (zero before the run); a match also starts anew at every
// multiple of kRestart positions inside it, so that k_exec finds the code in
// force without looking back.  The other positions hold nothing.
// ---------------------------------------------------------------------------
constexpr uint32_t kRestart = 256;

struct OutState {
    uint16_t* sym;     // the part's copy map
    uint32_t* start;   // its start bits
    uint64_t cap;
    uint64_t n;        // positions so far (uniform)
    uint64_t hi;       // positions written, or tried (uniform): n, or more after a failed block
    bool known;        // the context before the part is empty (member start)
    bool neg;          // a match of this lane reaches before the part start (a placeholder source)
};

__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

__device__ __forceinline__ bool allowed_has(const uint32_t* a, uint32_t b) { return (a[b >> 5] >> (b & 31)) & 1u; }

// The entry of the next Huffman symbol at 32 bits x: of a distance when `pend`
// (the length of a match whose distance is next), else of a literal or length.
// One table and one entry layout, so that the lanes of a warp take the same step
// whatever their symbols' kinds.
template <int NW>
__device__ __forceinline__ uint32_t symbol_entry(const TeamSmem<NW>& S, uint32_t x, uint32_t pend) {
    uint32_t e = S.tab[pend ? (1u << LB) + (x & ((1u << DB) - 1u)) : (x & ((1u << LB) - 1u))];
    if (((e >> 9) & 7u) == K_LONG) e = long_entry<NW>(S, x, pend ? 1u : 0u);
    return e;
}
__device__ __forceinline__ uint32_t entry_kind(uint32_t e) { return (e >> 9) & 7u; }
// base and extra bits of a length or distance
__device__ __forceinline__ uint32_t entry_value(uint32_t e, uint32_t x) {
    return (e >> 12) + ((x & ((1u << (e & 31u)) - 1u)) >> ((e >> 5) & 15u));
}

// The first tokens of a candidate's block, by one warp whose lanes decode the
// same bits: a false candidate fails after a few tokens (its literals must be
// allowed bytes), before the whole block is decoded in parallel.  A prefix that
// reaches the end of the block is left to the parallel decoder to judge.
constexpr int kTrialTokens = 24;

template <int NW>
__device__ int trial_prefix(const TeamSmem<NW>& S, uint32_t at) {
    uint32_t dist = 0;                                 // 1: a distance is next
    Bits br;
    br.seek(S.bits, at);
#pragma unroll 1
    for (int ntok = 0; ntok < kTrialTokens; ++ntok) {
        const uint32_t x = br.x();
        const uint32_t e = symbol_entry<NW>(S, x, dist), k = entry_kind(e);
        if (k == K_BAD) return CE_DATA;
        if (k == K_EOB) return CE_OK;
        if (k == K_LIT) {
            if (!allowed_has(S.allowed, (e >> 12) & 0xffu)) return CE_BYTE;
            if ((e >> 29) & 1u)
                if (!allowed_has(S.allowed, (e >> 20) & 0xffu)) return CE_BYTE;
        }
        dist = k == K_LEN;
        br.drop(S.bits, e & 31u);
    }
    return CE_OK;
}

// ---------------------------------------------------------------------------
// parallel decoding of one Huffman block by the T = 32 NW lanes of a team.
// Round, over a stretch of the block staged in shared memory:
//  A. lane k parses its own segment of `seg` bits from bit start + k*seg with
//     the block's codes (a guess: it may begin inside a code), keeping its tokens
//     and listing where the first of them start;
//  B. it parses on through the next segments until it reaches a token start
//     listed by some lane j > k (nearly always k+1): from there the two parses are
//     identical (Huffman codes resynchronise), so lane j's tokens from that one
//     on are the block's, and the lanes between hold nothing.  Lane 0 starts at
//     a known token start, so the lanes on the path 0 -> next(0) -> ... hold the
//     block's tokens, up to the first that meets nobody (the block's end, or the
//     round's);
//  C. each lane on the path drops its tokens before its meeting point; a prefix
//     sum of the output lengths gives its place in the output, and it writes the
//     copy map of its tokens.
// The next round starts where the last lane of the path stopped.
// Tokens are kept in global memory, row by row over the lanes: the stores wait
// for nothing, and in C the lanes read along together.
// seg follows the length of the part's previous block, so that its rounds have
// few lanes left over.
// ---------------------------------------------------------------------------
constexpr uint32_t kSegWordsMin = 3;

// token: bits 16-24 the output length, bit 31 a match (bits 0-14 distance - 1), else one or two bytes
__device__ __forceinline__ uint32_t token_len(uint32_t t) { return (t >> 16) & 0x1ffu; }

enum : uint32_t { PS_OK = 0, PS_EOB = 1, PS_ERR = 2, PS_SYNC = 3, PS_NOSYNC = 4, PS_CAP = 5 };

// A lane's parse and what it has found so far.
struct LaneParse {
    uint32_t p;           // bit of the staged words
    uint32_t n, out_len;  // tokens kept (rows of T), their output length
    uint32_t st;
};

__device__ __forceinline__ void st_global_if(bool on, uint32_t* a, uint32_t v) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %0, 0;\n\t@p st.global.u32 [%1], %2;\n\t}" ::"r"((uint32_t)on), "l"(a), "r"(v)
                 : "memory");
}
__device__ __forceinline__ void st_global_u16_if(bool on, uint16_t* a, uint32_t v) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %0, 0;\n\t@p st.global.u16 [%1], %2;\n\t}" ::"r"((uint32_t)on), "l"(a),
                 "h"((uint16_t)v)
                 : "memory");
}
__device__ __forceinline__ void or_shared_if(bool on, uint32_t a, uint32_t v) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %0, 0;\n\t@p red.shared.or.b32 [%1], %2;\n\t}" ::"r"((uint32_t)on), "r"(a),
                 "r"(v)
                 : "memory");
}

// The token at P.p of a lane with `go` (two literals at once if PAIRS), kept in tok[P.n]; go becomes false at a
// symbol that ends the parse (P.p stays at it; P.st says why).  One step for a literal, a match, or two literals, and
// no branch but one for the rare entries: a step's time is the chain of its three shared-memory reads (the words, the
// first entry, the distance's).  Against a branch for every kind, search and decoding of a 1 MiB file took 443 us for
// 493, of a 256 MiB file 2086 for 2120.
template <int NW, bool PAIRS>
__device__ __forceinline__ void next_token(const TeamSmem<NW>& S, LaneParse& P, bool& go, uint32_t* tok) {
    const uint32_t* w = S.bits + (P.p >> 5);
    const uint32_t w0 = w[0], w1 = w[1], w2 = w[2];
    const uint32_t x = __funnelshift_r(w0, w1, P.p);
    uint32_t e = S.tab[x & ((1u << LB) - 1u)];
    uint32_t q = (P.p & 31u) + (e & 31u);
    uint32_t y = __funnelshift_r(q < 32 ? w0 : w1, q < 32 ? w1 : w2, q);   // the bits after the code
    uint32_t d = S.tab[(1u << LB) + (y & ((1u << DB) - 1u))];
    bool len = e & (K_LEN << 9);
    if (go && ((e | (len ? d : 0u)) & kRare)) {
        if (entry_kind(e) == K_LONG) {
            e = long_entry<NW>(S, x, 0);
            q = (P.p & 31u) + (e & 31u);
            y = __funnelshift_r(q < 32 ? w0 : w1, q < 32 ? w1 : w2, q);
            d = S.tab[(1u << LB) + (y & ((1u << DB) - 1u))];
        }
        len = entry_kind(e) == K_LEN;
        if (len && entry_kind(d) == K_LONG) d = long_entry<NW>(S, y, 1);
        const uint32_t kind = len ? entry_kind(d) : entry_kind(e);
        if (kind >= K_EOB) {
            P.st = kind == K_EOB ? PS_EOB : PS_ERR;
            go = false;
        }
    }
    const uint32_t lit = PAIRS ? e >> 12 : 0x10000u | ((e >> 12) & 0xffu);
    const uint32_t t = len ? 0x80000000u | (entry_value(e, x) << 16) | (entry_value(d, y) - 1u) : lit;
    const uint32_t drop = len ? (e & 31u) + (d & 31u) : (PAIRS ? e & 31u : (e >> 5) & 15u);
    st_global_if(go, tok + P.n, t);
    P.p += go ? drop : 0u;
    P.out_len += go ? token_len(t) : 0u;
    P.n += go ? 32u * NW : 0u;
}

// In the loops below the lanes of a warp take every step together (the vote every second one): left to themselves,
// lanes that took different branches run apart for the rest of the loop, and the warp does each group's steps in
// turn.

// A: the tokens that start before p0 + seg, kept in tok[0], tok[T], ... up to tok[cap]
template <int NW>
__device__ __forceinline__ void parse_own(TeamSmem<NW>& S, LaneParse& P, uint32_t tl, uint32_t seg, uint32_t* tok,
                                          uint32_t cap) {
    constexpr uint32_t T = 32 * NW;
    const uint32_t p0 = P.p, p1 = p0 + seg;
    uint8_t* list = &S.list[0][0] + tl;
    bool go = true;
    do {
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            if (go && !(P.n & T) && P.n < 2 * TeamSmem<NW>::kList * T) list[P.n / 2] = (uint8_t)(P.p - p0);
            next_token<NW, true>(S, P, go, tok);
            go = go && P.p < p1 && P.n < cap;
        }
    } while (__any_sync(FULL, go));
    if (P.st == PS_OK && P.p < p1) P.st = PS_CAP;
}

// B: on through the segments after lane tl's (rel: the place in the first), literals one at a time, until a listed
// token start; m and j: that lane and list entry.  A parse that meets nobody over kMeetBits bits gives up (a lane past
// the block's end can otherwise go on to the round's).
constexpr uint32_t kMeetBits = 8192;

template <int NW>
__device__ __forceinline__ void parse_on(TeamSmem<NW>& S, LaneParse& P, bool go, uint32_t tl, uint32_t seg, uint32_t rel,
                                         uint32_t* tok, uint32_t cap, uint32_t& m, uint32_t& j) {
    constexpr uint32_t T = 32 * NW;
    const uint32_t give_up = min(T, tl + 2 + kMeetBits / seg);
    m = min(tl + 1, T - 1);
    j = 0;
    uint32_t at = 0, cnt = S.r_cnt[m];                 // place of entry j of lane m's list; its entries
    uint32_t nx = S.list[1][m];                        // its next entry
    while (__any_sync(FULL, go)) {
        if (go && rel >= seg) {                        // the next lane's segment
            rel -= seg;
            ++m;
            if (m >= give_up) {
                P.st = PS_NOSYNC;
                go = false;
            } else {
                j = at = 0;
                cnt = S.r_cnt[m];
                nx = S.list[1][m];
            }
        }
        if (go && P.n >= cap) {
            P.st = PS_NOSYNC;
            go = false;
        }
#pragma unroll
        for (int u = 0; u < 2; ++u) {                  // along the list, to the first entry at or after rel
            const bool adv = go && at < rel && j + 1 < cnt;
            at += adv ? (nx - at) & 255u : 0u;
            j += adv ? 1u : 0u;
            if (adv && j + 1 < cnt) nx = S.list[j + 1][m];
        }
        const bool behind = at < rel && j + 1 < cnt;   // not there yet: no token in this step
        if (go && at == rel) {
            P.st = PS_SYNC;
            go = false;
        }
        bool step = go && !behind;
        const bool was = step;
        const uint32_t p = P.p;
        next_token<NW, false>(S, P, step, tok);
        rel += P.p - p;
        go = go && (step || !was);
    }
}

// output length of the tokens [0, z)
template <int NW>
__device__ __forceinline__ uint32_t tokens_length(const uint32_t* tok, uint32_t z) {
    constexpr uint32_t T = 32 * NW;
    uint32_t len = 0;
    for (uint32_t n = 0; __any_sync(FULL, n < z); n += 4 * T) {
        uint32_t t[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) t[k] = n + k * T < z ? tok[n + k * T] : 0u;
#pragma unroll
        for (int k = 0; k < 4; ++k) len += token_len(t[k]);
    }
    return len;
}

// whether every literal among the tokens [n, z) is an allowed byte
template <int NW>
__device__ __noinline__ bool tokens_allowed(const TeamSmem<NW>& S, const uint32_t* tok, uint32_t n, uint32_t z) {
    bool ok = true;
    for (; n < z; n += 32 * NW) {
        const uint32_t t = tok[n];
        if (!(t >> 31))
            ok &= allowed_has(S.allowed, t & 0xffu) && (token_len(t) < 2 || allowed_has(S.allowed, (t >> 8) & 0xffu));
    }
    return ok;
}

// C: the copy map of the tokens [n, z), from position base + pos on (map and words from position base on, a multiple
// of kRestart).  Only the places where a token starts are written
// (a u16 each, and its start bit): k_exec spreads the matches, many threads to each.  The start bits go to shared
// memory (SHARED: words from the round's first on), when the round's fit there, else to the part's own words.
// Returns false if (check) a literal is not an allowed byte.
template <int NW, bool SHARED>
__device__ __forceinline__ bool write_map(const TeamSmem<NW>& S, const uint32_t* tok, uint32_t n, uint32_t z,
                                          uint16_t* map, uint32_t* words, uint32_t pos, uint32_t base, bool check, bool& neg) {
    constexpr uint32_t T = 32 * NW;
    constexpr int kAhead = 4;
    const uint32_t words_a = SHARED ? (uint32_t)__cvta_generic_to_shared(words) : 0u;
    auto set = [&](bool on, uint32_t word, uint32_t bits) {
        if (SHARED) or_shared_if(on, words_a + 4 * word, bits);
        else if (on) atomicOr(words + word, bits);
    };
    bool ok = true;
    uint32_t nx[kAhead];
#pragma unroll
    for (int k = 0; k < kAhead; ++k) nx[k] = n + k * T < z ? tok[n + k * T] : 0u;
    while (__any_sync(FULL, n < z)) {
        uint32_t q[kAhead];
#pragma unroll
        for (int k = 0; k < kAhead; ++k) q[k] = nx[k];
        n += kAhead * T;
#pragma unroll
        for (int k = 0; k < kAhead; ++k) nx[k] = n + k * T < z ? tok[n + k * T] : 0u;
#pragma unroll
        for (int k = 0; k < kAhead; ++k) {
            const uint32_t t = q[k], len = token_len(t), d = t & 0x7fffu;   // (len 0: past the lane's last token)
            const bool match = t >> 31, two = !match && len > 1;
            const uint32_t code = match ? kPH | d : t & 0xffu, b1 = (t >> 8) & 0xffu;
            if (check && !match && len) ok &= allowed_has(S.allowed, code) && (!two || allowed_has(S.allowed, b1));
            neg |= match && base + pos <= d;
            set(len != 0, pos >> 5, (two ? 3u : 1u) << (pos & 31u));
            st_global_u16_if(len != 0, map + pos, code);
            st_global_u16_if(two, map + pos + 1, b1);
            const uint32_t r = (pos | (kRestart - 1)) + 1, e = pos + len;
            if (r < e || (two && !(~pos & 31u))) {
                // the match starts anew at every multiple of kRestart; the second literal's bit is the next word's
                if (match) {
                    for (uint32_t a = r; a < e; a += kRestart) {
                        map[a] = (uint16_t)code;
                        set(true, a >> 5, 1u);
                    }
                } else {
                    set(true, (pos >> 5) + 1, 1u);
                }
            }
            pos = e;
        }
    }
    return ok;
}

// What a part's blocks share.
struct TeamState {
    uint32_t* tok;       // the team's tokens: row k holds every lane's k-th
    uint32_t cap;        // rows
    uint32_t est;        // bits of the part's previous block (0: not known)
    uint32_t segw_lim;   // longest segment in words, shortened while tokens fill the rows first
};

// The tokens of a Huffman block whose tables are in S, from bit `pos` of the
// member on; [s0, s1) are the staged words.
template <int NW>
__device__ int par_block(TeamSmem<NW>& S, const Input& in, uint64_t s0, uint64_t s1, uint64_t& pos, TeamState& ts,
                         OutState& o, bool check, uint64_t max_block, uint64_t end_bit, uint64_t& block_n) {
    constexpr uint32_t T = 32 * NW, kSegWords = TeamSmem<NW>::kSegWords;
    const uint32_t tl = threadIdx.x, lane = tl & 31, warp = tl >> 5;
    const uint64_t block0 = pos;
    for (;;) {
        uint32_t segw = ts.segw_lim;
        if (ts.est) {                                  // what is expected to be left, in equal rounds
            const uint64_t done = pos - block0;
            uint32_t left = done < ts.est ? ts.est - (uint32_t)done : ts.est >> 4;
            left = (left + left / 32) / 32 + 1;
            const uint32_t rounds = (left + T * segw - 1) / (T * segw);
            segw = min(segw, max(5u, (left / rounds + T - 1) / T) | 1u);
        }
        const uint32_t seg = 32 * segw, need = T * segw + 4;   // a token may end 48 bits past the last segment
        const uint64_t w = pos >> 5;
        if (w < s0 || w + need > s1) {
            s0 = w;
            s1 = w + TeamSmem<NW>::kBits;
            stage<NW>(S, in, s0, TeamSmem<NW>::kBits);
        }
        const uint64_t base = s0 << 5;                 // member bit of staged bit 0
        const uint32_t start = (uint32_t)(pos - base), p0 = start + tl * seg;
        LaneParse P{p0, 0, 0, PS_OK};
        uint32_t* tok = ts.tok + tl;
        const uint32_t cap = ts.cap * T;
        __syncthreads();                               // the lists' place is free
        parse_own<NW>(S, P, tl, seg, tok, cap);
        S.r_cnt[tl] = (uint8_t)min((P.n / T + 1) / 2, TeamSmem<NW>::kList);
        __syncthreads();
        uint32_t m, j;
        parse_on<NW>(S, P, P.st == PS_OK && tl + 1 < T, tl, seg, P.p - p0 - seg, tok, cap, m, j);
        const bool met = P.st == PS_SYNC;
        const uint32_t n = P.n;
        S.r_next[tl] = (uint16_t)(met ? m : T);
        S.r_j[tl] = (uint16_t)(2 * j);
        const uint32_t exc = __ballot_sync(FULL, !met || m != tl + 1);
        if (lane == 0) S.r_exc[warp] = exc;
        __syncthreads();
        // the path from lane 0 (uniform): runs of lanes that met the next one, up to a lane that met another or
        // nobody (the last)
        uint32_t path = 0, last = 0, pred = tl - 1;    // my warp's lanes on the path; mine's predecessor
        for (uint32_t cur = 0;;) {
            uint32_t v = cur >> 5, x = S.r_exc[v] & (FULL << (cur & 31));
            while (!x) {                               // ends: the team's last lane met nobody
                if (v == warp) path |= FULL << (cur & 31);
                cur = 32 * ++v;
                x = S.r_exc[v];
            }
            const uint32_t e = 32 * v + (uint32_t)(__ffs(x) - 1);
            if (v == warp) path |= (FULL << (cur & 31)) & (FULL >> (31 - (e & 31)));
            const uint32_t nx = S.r_next[e];
            if (nx >= T) {
                last = e;
                break;
            }
            if (nx == tl) pred = e;
            cur = nx;
        }
        const bool mine = (path >> lane) & 1u;
        // my tokens before my predecessor's meeting point are not the block's
        const uint32_t skip = mine && tl ? T * S.r_j[pred] : 0u;
        const uint32_t skipped = tokens_length<NW>(tok, skip);
        const uint32_t len = mine ? P.out_len - skipped : 0u;
        uint32_t incl = len;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t x = __shfl_up_sync(FULL, incl, d);
            if ((int)lane >= d) incl += x;
        }
        if (lane == 31) S.r_sum[warp] = incl;
        if (tl == last) {
            S.r_flags = P.st;
            Bits b;
            b.seek(S.bits, P.p);
            S.r_end = P.p + (P.st == PS_EOB ? symbol_entry<NW>(S, b.x(), 0) & 31u : 0u);
        }
        __syncthreads();
        uint32_t before = 0, total = 0;
#pragma unroll
        for (int v = 0; v < NW; ++v) {
            const uint32_t x = S.r_sum[v];
            if (v < (int)warp) before += x;
            total += x;                                // lanes off the path add nothing
        }
        const uint32_t st = S.r_flags;
        const uint64_t round_end = base + S.r_end;
        int err = CE_OK;
        if (st == PS_ERR) err = CE_DATA;
        else if (max_block && block_n + total >= max_block) err = CE_SIZE;
        else if (o.n + total > o.cap) err = CE_OVERFLOW;
        if (err) {
            // a false candidate is told by its literals before it is given more room
            if (__syncthreads_or(err == CE_OVERFLOW && check && mine && !tokens_allowed<NW>(S, tok, skip, n)))
                return CE_BYTE;
            return err;
        }
        bool neg = false;
        o.hi = max(o.hi, o.n + total);
        // the round's start bits, in the lists' place if they fit
        const uint32_t pos0 = (uint32_t)o.n, map0 = pos0 & ~(kRestart - 1);
        const uint32_t nw = (uint32_t)((o.n + total + 31) / 32) - map0 / 32;
        uint32_t* sb = nw <= sizeof(S.list) / 4 ? reinterpret_cast<uint32_t*>(&S.list[0][0]) : nullptr;
        if (sb) {
            for (uint32_t k = tl; k < nw; k += T) sb[k] = 0;
            __syncthreads();
        }
        const uint32_t to = mine ? n : skip, at = pos0 + before + incl - len;
        const bool ok = sb ? write_map<NW, true>(S, tok, skip, to, o.sym + map0, sb, at - map0, map0, check, neg)
                           : write_map<NW, false>(S, tok, skip, to, o.sym, o.start, at, 0, check, neg);
        const bool bad = __syncthreads_or(!ok);
        if (sb)
            for (uint32_t k = tl; k < nw; k += T) {
                uint32_t* g = o.start + (map0 >> 5) + k;
                if (k <= (pos0 - map0) >> 5 || k + 1 == nw) atomicOr(g, sb[k]);   // words shared with other rounds
                else *g = sb[k];
            }
        o.neg |= neg;
        if (bad) return CE_BYTE;
        if (o.known && __syncthreads_or(neg)) return CE_DIST;
        o.n += total;
        block_n += total;
        if (round_end > end_bit) return CE_TRUNC;
        pos = round_end;
        if (st == PS_EOB) {
            ts.est = (uint32_t)min(round_end - block0, (uint64_t)0xfffffffu);
            ts.segw_lim = min(kSegWords, 2 * ts.segw_lim + 1);
            return CE_OK;
        }
        if (st == PS_CAP) ts.segw_lim = max(kSegWordsMin, segw / 2 | 1u);
    }
}

// a stored block; pos is after its three header bits
template <int NW>
__device__ int stored_block(const Input& in, uint64_t& pos, OutState& o, bool check, const uint32_t* allowed,
                            uint64_t end_bit, uint64_t& block_n) {
    const uint64_t p = (pos + 7) & ~7ull;
    if (p + 32 > end_bit) return CE_TRUNC;
    const uint64_t byte = p >> 3;
    const uint8_t* g = in.b;
    const uint32_t len = (uint32_t)__ldg(g + byte) | ((uint32_t)__ldg(g + byte + 1) << 8);
    const uint32_t nlen = (uint32_t)__ldg(g + byte + 2) | ((uint32_t)__ldg(g + byte + 3) << 8);
    if ((len ^ 0xffffu) != nlen) return CE_DATA;
    if (p + 32 + 8ull * len > end_bit) return CE_TRUNC;
    if (o.n + len > o.cap) return CE_OVERFLOW;
    bool bad = false;
    for (uint32_t j = threadIdx.x; j < len; j += 32 * NW) {
        const uint32_t v = __ldg(g + byte + 4 + j);
        if (check && !allowed_has(allowed, v)) bad = true;
        o.sym[o.n + j] = (uint16_t)v;
    }
    if (len) {                                  // every position a start
        const uint32_t a = (uint32_t)o.n, z = a + len;
        for (uint32_t k = (a >> 5) + threadIdx.x; k <= (z - 1) >> 5; k += 32 * NW) {
            const uint32_t lo = k == a >> 5 ? FULL << (a & 31u) : FULL, hi = k == (z - 1) >> 5 ? FULL >> (31u - ((z - 1) & 31u)) : FULL;
            atomicOr(o.start + k, lo & hi);
        }
    }
    o.hi = max(o.hi, o.n + len);
    if (__syncthreads_or(bad)) return CE_BYTE;
    o.n += len;
    block_n += len;
    pos = p + 32 + 8ull * len;
    return CE_OK;
}

// The block at bit `pos`, which moves past it.  candidate: the block must be a
// non-final dynamic block (the block-start checks); min/max_block bound its
// size; check: its literals must be allowed bytes.  Huffman blocks are decoded
// by the whole team in parallel (par_block); a candidate block start first runs
// a short serial prefix, so that false candidates fail after a few tokens.
template <int NW>
__device__ int one_block(TeamSmem<NW>& S, const Input& in, uint64_t& pos, TeamState& ts, OutState& o, bool check,
                         uint64_t min_block, uint64_t max_block, bool candidate, uint64_t end_bit, uint32_t& final) {
    const uint64_t s0 = pos >> 5, s1 = s0 + TeamSmem<NW>::kBits;
    // a candidate's header and prefix first; its block's words follow if they pass
    const uint32_t ns = candidate ? 256u : TeamSmem<NW>::kBits;
    stage<NW>(S, in, s0, ns);
    uint32_t at = (uint32_t)pos & 31u;
    const uint32_t h = __funnelshift_r(S.bits[0], S.bits[1], at) & 7u;
    final = h & 1u;
    const uint32_t type = h >> 1;
    pos += 3;
    at += 3;
    if (pos > end_bit) return CE_TRUNC;
    if (candidate) {
        if (final) return CE_FINAL;
        if (type != 2) return CE_TYPE;
    }
    uint64_t block_n = 0;
    int st = CE_OK;
    if (type == 0) {
        st = stored_block<NW>(in, pos, o, check, S.allowed, end_bit, block_n);
    } else if (type == 3) {
        st = CE_DATA;
    } else {
        if (type == 1) {
            if (S.table_kind != 1) build_fixed<NW>(S);
        } else {
            uint32_t bits = 0;
            st = read_dynamic<NW>(S, at, &bits);
            pos += bits;
            at += bits;
            if (st == CE_OK && pos > end_bit) st = CE_TRUNC;
        }
        if (st == CE_OK && candidate) {
            if (threadIdx.x < 32) {
                const int t = trial_prefix<NW>(S, at);
                if (threadIdx.x == 0) S.h_status = t;
            }
            __syncthreads();
            st = S.h_status;
            __syncthreads();
        }
        if (st == CE_OK)
            st = par_block<NW>(S, in, s0, candidate ? s0 : s1, pos, ts, o, check, max_block, end_bit, block_n);
    }
    if (st == CE_OK && max_block && block_n >= max_block) st = CE_SIZE;
    if (st == CE_OK && block_n < min_block) st = CE_SIZE;
    return st;
}

// ---------------------------------------------------------------------------
// block-start candidates.  Per bit offset p, in order of cost:
//  1. BFINAL = 0, BTYPE = 10, HLIT <= 29, HDIST <= 29: bit-parallel over the
//     32 offsets of a lane;
//  2. the code-length code is complete: sum of 2^-l over its lengths is 1,
//     from a 512-entry table of three-field sums;
//  3. the dynamic header is valid (the checks of read_lengths), up to 32 listed
//     offsets at a time, one per lane (headers_ok).
// The full block decode then follows in k_sync, lowest offset first.  Stages
// 1-3 are implied by the complete checks, so no offset that passes those is
// dropped here.
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t fsr(uint32_t lo, uint32_t hi, uint32_t s) { return __funnelshift_r(lo, hi, s); }

// 3-field Kraft sums in units of 2^-7: kraft3[a | b << 3 | c << 6]
__device__ __forceinline__ uint32_t kraft1(uint32_t l) { return l ? (128u >> l) : 0u; }

__device__ uint32_t cl_complete(const uint16_t* kraft3, uint32_t w0, uint32_t w1, uint32_t w2, uint32_t w3, uint32_t k) {
    // bits of the window from offset k + 13 (HCLEN) onward; k < 32
    const uint32_t q = k + 13;                   // < 45
    const uint32_t a0 = q < 32 ? fsr(w0, w1, q) : fsr(w1, w2, q - 32);
    const uint32_t hclen = (a0 & 15u) + 4;
    const uint32_t q1 = q + 4, q2 = q + 34;      // 10 fields, then 9 fields
    const uint32_t f1 = q1 < 32 ? fsr(w0, w1, q1) : fsr(w1, w2, q1 - 32);
    const uint32_t f2 = q2 < 64 ? fsr(w1, w2, q2 - 32) : fsr(w2, w3, q2 - 64);
    const uint64_t fields = (uint64_t)(f1 & 0x3fffffffu) | ((uint64_t)(f2 & 0x7ffffffu) << 30);
    const uint64_t x = fields & ((1ull << (3 * hclen)) - 1ull);
    uint32_t kr = 0;
#pragma unroll
    for (int g = 0; g < 7; ++g) kr += kraft3[(x >> (9 * g)) & 511u];
    return kr == 128u;
}

// The whole dynamic-header check of up to 32 candidates by one warp, one per
// lane (mine: its bit of the staged words; the caller has checked that its
// code-length code is complete).  The warp first builds each candidate's lookup
// table of the code-length code, one candidate at a time (128 bytes: length,
// symbol << 3), in tabs, candidate i's at i mod kTabs; then every lane reads its
// candidate's lengths symbol by symbol, the checks of read_lengths made as they
// come, nearly every false candidate failing long before its end.  Returns the
// lanes whose headers are valid.  Bound by instruction issue, half of it in the
// tables: filled by one lane per symbol a code of one bit took 64 turns of the
// loop (k_sync of a 256 MiB file 750 us, now 690; of 96 files 1160, now 1100).
__device__ uint32_t headers_ok(const uint32_t* bits, uint8_t* tabs, uint32_t kTabs, uint32_t n, uint32_t mine,
                               uint64_t base_bit, uint64_t end_bit, int lane) {
    uint32_t ok = 0, order = 19;                           // place of symbol `lane` among the code's lengths
#pragma unroll
    for (uint32_t k = 0; k < 19; ++k)
        if (lane == c_clorder[k]) order = k;
    for (uint32_t c0 = 0; c0 < n; c0 += kTabs) {
        const uint32_t c1 = min(n, c0 + kTabs);
        __syncwarp();
        for (uint32_t c = c0; c < c1; ++c) {
            Bits br;
            br.seek(bits, __shfl_sync(FULL, mine, (int)c) + 3);
            const uint32_t hclen = ((br.x() >> 10) & 15u) + 4;
            br.drop(bits, 14);
            const uint32_t f1 = br.x();
            br.drop(bits, 30);
            const uint32_t f2 = br.x();
            // length of symbol `lane`
            const uint32_t len = order < hclen ? (order < 10 ? f1 >> (3 * order) : f2 >> (3 * (order - 10))) & 7u : 0u;
            uint32_t code = 0, prev = 0, first = 0;        // first code of my length
            uint32_t rank = 0;
#pragma unroll
            for (uint32_t L = 1; L <= 7; ++L) {
                const uint32_t m = __ballot_sync(FULL, len == L);
                code = (code + prev) << 1;
                prev = __popc(m);
                if (len == L) {
                    first = code;
                    rank = __popc(m & ((1u << lane) - 1u));
                }
            }
            uint8_t* tab = tabs + 128 * (c - c0);
            // the warp fills the many entries of a short code together, each lane the few of its long one
            const uint32_t lo = len ? __brev(first + rank) >> (32 - len) : 128u, val = len | ((uint32_t)lane << 3);
            for (uint32_t m = __ballot_sync(FULL, len - 1u < 3u); m; m &= m - 1u) {
                const int src = __ffs((int)m) - 1;
                const uint32_t sval = __shfl_sync(FULL, val, src), slen = sval & 7u;
                for (uint32_t v = __shfl_sync(FULL, lo, src) + ((uint32_t)lane << slen); v < 128; v += 32u << slen)
                    tab[v] = (uint8_t)sval;
            }
            if (len > 3)
                for (uint32_t v = lo; v < 128; v += 1u << len) tab[v] = (uint8_t)val;
        }
        __syncwarp();
        bool go = (uint32_t)lane >= c0 && (uint32_t)lane < c1;
        const uint8_t* tab = tabs + 128 * (go ? lane - c0 : 0);
        Bits br;
        br.seek(bits, mine + 3);
        const uint32_t x0 = br.x();
        const uint32_t hlit = (x0 & 31u) + 257, total = hlit + ((x0 >> 5) & 31u) + 1, hclen = ((x0 >> 10) & 15u) + 4;
        go = go && hlit <= 286 && total - hlit <= 30;
        br.seek(bits, go ? mine + 17 + 3 * hclen : 0);
        bool good = go;
        uint32_t i = 0, prev = 0, kl = 0, kd = 0;          // Kraft sums (units of 2^-15), codes of length 1 at bit 20
        bool eob = false;
        while (__any_sync(FULL, go)) {
            const uint32_t x = br.x(), e = tab[x & 127u], l = e & 7u, sym = e >> 3, y = x >> l;
            const uint32_t ex = sym < 16 ? 0u : (sym == 16 ? 2u : (sym == 17 ? 3u : 7u));
            const uint32_t rep = (sym < 16 ? 1u : (sym == 18 ? 11u : 3u)) + (y & ((1u << ex) - 1u));
            const uint32_t val = sym < 16 ? sym : (sym == 16 ? prev : 0u);
            prev = val;
            const uint32_t e2 = i + rep;
            const uint32_t nlit = i < hlit ? min(e2, hlit) - i : 0u, w = val ? 32768u >> val : 0u;
            const bool bad = (sym == 16 && i == 0) || e2 > total;
            if (go) {
                kl += nlit * w;
                kd += (rep - nlit) * w;
                eob |= val && i <= 256 && 256 < e2;
                good = !bad && kl <= 32768u && kd <= 32768u && (eob || e2 <= 256);   // e2 > 256: no end of block
                i = e2;
                go = good && i < total;
            }
            br.drop(bits, go ? l + ex : 0u);
        }
        // complete, or one code of length 1 (a sum of one half can also be that of longer codes: the team's own
        // check of the header tells), or no distance code at all
        good = good && eob && (kl == 32768u || kl == 16384u) && (kd == 32768u || kd == 16384u || kd == 0);
        ok |= __ballot_sync(FULL, good && base_bit + br.p <= end_bit);
    }
    return ok;
}

// One step of the search from bit `next`: each warp filters kScanWindows
// consecutive windows of 1024 bits (each lane tests 32 offsets with bit masks,
// then the completeness of the code-length code); the survivors are gathered,
// one per lane, and their whole headers are checked at once, one per lane.  A
// warp that finds valid headers stops there.  The results are in S.c_*: per warp
// the offsets from T (the step's first window) whose headers are valid, lowest
// first, and the bit where its search resumes.

template <int NW>
__device__ void scan_step(TeamSmem<NW>& S, const Input& in, uint64_t next, uint64_t hi, uint64_t end_bit) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    constexpr uint32_t kScanWindows = TeamSmem<NW>::kScanWindows;
    constexpr uint32_t kWords = NW * kScanWindows * 32 + 148;      // the windows, and a header after the last bit
    static_assert(kWords + 256 <= TeamSmem<NW>::kBits + 2, "a step's words are staged at once");
    const uint64_t T0 = next & ~1023ull;
    uint16_t* kraft3 = S.kraft3();
    __syncthreads();
    for (uint32_t v = threadIdx.x; v < 512; v += 32 * NW)
        kraft3[v] = (uint16_t)(kraft1(v & 7) + kraft1((v >> 3) & 7) + kraft1(v >> 6));
    stage<NW>(S, in, T0 >> 5, kWords);
    const uint64_t lo_w = T0 + (uint64_t)warp * (kScanWindows * 1024u);
    uint64_t end_w = min(hi, lo_w + kScanWindows * 1024u);
    uint64_t at = max(next, lo_w);             // this warp's first bit not yet filtered
    // the warps' header tables take the place between the step's words and the Kraft sums
    constexpr uint32_t kTabs = (TeamSmem<NW>::kBits + 2 - 256 - kWords) / NW / 32;
    static_assert(kTabs >= 4, "a header table is 32 words");
    uint8_t* tabs = reinterpret_cast<uint8_t*>(S.bits + kWords + warp * (32 * kTabs));
    uint32_t found = 0, mine = 0;
    uint32_t pass = 0;
    while (!pass && at < end_w) {
        uint32_t n = 0;                        // offsets listed
        while (n < 32 && at < end_w) {
            const uint64_t T = at & ~1023ull;
            const uint64_t base = T + 32ull * (uint64_t)lane;
            const uint32_t* wp = S.bits + (uint32_t)((base - T0) >> 5);
            const uint32_t w0 = wp[0], w1 = wp[1], w2 = wp[2], w3 = wp[3];
            const uint64_t x = (uint64_t)w0 | ((uint64_t)w1 << 32);
            uint64_t y = ~x & ~(x >> 1) & (x >> 2);                // BFINAL = 0, BTYPE = 10
            y &= ~((x >> 4) & (x >> 5) & (x >> 6) & (x >> 7));     // HLIT <= 29
            y &= ~((x >> 9) & (x >> 10) & (x >> 11) & (x >> 12));  // HDIST <= 29
            uint32_t m = (uint32_t)y;
            if (base < at) {
                const uint64_t d = at - base;
                m = d >= 32 ? 0u : (m & (~0u << d));
            }
            if (base + 32 > end_w) m = base >= end_w ? 0u : (m & ((1u << (uint32_t)(end_w - base)) - 1u));
            uint32_t c = 0;
            for (uint32_t mm = m; mm; mm &= mm - 1) {
                const uint32_t k = __ffs(mm) - 1;
                if (cl_complete(kraft3, w0, w1, w2, w3, k)) c |= 1u << k;
            }
            // list the survivors lowest first (lanes cover increasing offsets) while there is room
            uint64_t resume = T + 1024;
            for (uint32_t bl = __ballot_sync(FULL, c != 0); bl; bl = __ballot_sync(FULL, c != 0)) {
                const int l = __ffs(bl) - 1;
                const uint32_t cl = __shfl_sync(FULL, c, l);
                const uint32_t k = __ffs(cl) - 1;
                const uint64_t pos = T + 32ull * (uint64_t)l + k;
                if (n == 32) {                                    // full: this window resumes here
                    resume = pos;
                    break;
                }
                if (lane == l) c &= c - 1;
                if ((uint32_t)lane == n) mine = (uint32_t)(pos - T0);
                ++n;
            }
            at = resume;
        }
        pass = headers_ok(S.bits, tabs, kTabs, n, mine, T0, end_bit, lane);
    }
    constexpr uint32_t kCand = TeamSmem<NW>::kCand;
    found = __popc(pass);
    const uint32_t ix = __popc(pass & ((1u << lane) - 1u));
    if (((pass >> lane) & 1u) && ix < kCand) S.c_at[warp][ix] = mine;
    if (found > kCand) {                       // the search resumes at the first one left out
        at = T0 + __shfl_sync(FULL, mine, (int)__fns(pass, 0, kCand + 1));
        end_w = ~0ull;
        found = kCand;
    }
    if (lane == 0) {
        S.c_n[warp] = found;
        S.c_done[warp] = at >= end_w;
        S.c_resume[warp] = at;
    }
    __syncthreads();
}

template <int NW>
__device__ __forceinline__ TeamSmem<NW>& team_smem() {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    return *reinterpret_cast<TeamSmem<NW>*>(smem_raw);
}

// Work queue of the pass-1 kernels: each resident team takes the next queue
// position until the parts run out, so parts of uneven work (many members of
// different sizes in one launch) balance over the teams.  Position q holds
// part order[q] (the parts with the most expected output first, so that the
// short ones fill the end of the launch), or part q without an order.  The
// counter is zero before the launch.
template <int NW>
__device__ __forceinline__ int next_part(TeamSmem<NW>& S, uint32_t* queue) {
    __syncthreads();
    if (threadIdx.x == 0) S.q = (int)min(atomicAdd(queue, 1u), 0x7fffffffu);
    __syncthreads();
    return S.q;
}

template <int NW>
__device__ __forceinline__ void init_smem(TeamSmem<NW>& S, const KParams& p) {
    if (threadIdx.x < 8) S.allowed[threadIdx.x] = p.allowed[threadIdx.x];
    if (threadIdx.x == 0) S.table_kind = 0;
    __syncthreads();
}

// ---------------------------------------------------------------------------
// k_sync: block start of each part and its first block; k_inflate: the rest of each part
// ---------------------------------------------------------------------------
template <int NW>
__device__ __forceinline__ TeamState team_state(uint32_t* tok, const KParams& p, uint32_t est) {
    return TeamState{tok + (uint64_t)blockIdx.x * (32 * NW) * p.tok_rows, p.tok_rows, est, TeamSmem<NW>::kSegWords};
}

// the start bits of a block that failed
template <int NW>
__device__ void clear_starts(OutState& o) {
    __syncthreads();
    for (uint64_t k = threadIdx.x; k < (o.hi + 31) / 32; k += 32 * NW) o.start[k] = 0;
    o.hi = 0;
    __syncthreads();
}

// The block start of part c and its first block (Section "Detection of DEFLATE block start positions").
template <int NW>
__device__ void sync_part(TeamSmem<NW>& S, const FileDesc& F, ChunkDesc& C, uint16_t* symbuf,
                          uint32_t* start_bits, uint32_t* tok, const KParams& p) {
    init_smem<NW>(S, p);
    OutState o{symbuf + C.sym_base, start_bits + C.sym_base / 32, C.cap, 0, 0, C.index == 0 && C.lo <= F.s0_bit, false};
    const Input in(F.gz, F.gz_len);
    TeamState ts = team_state<NW>(tok, p, 0);
    uint32_t state = CS_EMPTY, err = CE_OK, final = 0;
    uint64_t sync = kNone, resume = 0;
    if (C.disabled) {
        state = CS_EMPTY;
    } else if (o.known || C.given) {          // the member start (empty context) or a known block start
        sync = resume = C.lo;
        const int st = one_block<NW>(S, in, resume, ts, o, false, 0, 0, false, F.end_bit, final);
        if (st) {
            state = CS_ERROR;
            err = (uint32_t)st;
        } else {
            state = CS_FOUND;
        }
    } else {
        const uint64_t hi = min(C.hi, F.end_bit);
        uint64_t next = C.lo;
        bool go = true;
        while (go && next < hi) {
            scan_step<NW>(S, in, next, hi, F.end_bit);
            const uint64_t T0 = next & ~1023ull;
            next = T0 + NW * TeamSmem<NW>::kScanWindows * 1024ull;
            for (int w = 0; w < NW && go; ++w) {
                const uint32_t n = S.c_n[w];
                for (uint32_t k = 0; k < n; ++k) {
                    const uint64_t cand = T0 + S.c_at[w][k];
                    uint64_t pos = cand;
                    o.n = 0;
                    o.neg = false;
                    ts = team_state<NW>(tok, p, 0);
                    const int st = one_block<NW>(S, in, pos, ts, o, true, p.min_block, p.max_block, true, F.end_bit,
                                                 final);
                    if (st == CE_OK) {
                        state = CS_FOUND;
                        sync = cand;
                        resume = pos;
                        go = false;
                        break;
                    }
                    clear_starts<NW>(o);
                    if (st == CE_OVERFLOW) {     // the candidate's block does not fit: cannot judge it here
                        state = CS_ERROR;
                        err = CE_OVERFLOW;
                        sync = cand;
                        go = false;
                        break;
                    }
                }
                if (go && !S.c_done[w]) {        // that warp's search stopped short: the next step starts there
                    next = S.c_resume[w];
                    break;
                }
            }
            __syncthreads();                     // S.c_* may be rewritten
        }
    }
    const bool neg = __syncthreads_or(o.neg);
    if (threadIdx.x == 0) {
        C.err = err;
        C.sync = sync;
        C.resume = resume;
        C.n = state == CS_FOUND ? o.n : 0;
        C.nph = 0;
        C.last_ph = 0;
        C.det = kNone;
        C.anyph = neg && state == CS_FOUND;
        C.blocks = state == CS_FOUND ? 1u : 0u;
        C.final = final && state == CS_FOUND;
        C.confirmed = (state == CS_FOUND && (o.known || C.given || final || p.confirm_blocks == 0)) ? 1u : 0u;
        C.end = resume;
        C.state = state;
    }
}

// Where part c's decoding stops: the start of the next part that holds one (`sync` is final after k_sync and
// never written by k_inflate, whose other warps rewrite `state`); parts merged into their predecessor hold
// none.
__device__ __forceinline__ uint64_t find_stop(const FileDesc& F, const ChunkDesc* chunks, int c, uint64_t stop_hint) {
    for (int j = c + 1; j < F.chunk0 + F.nchunks; ++j) {
        const uint64_t sj = chunks[j].sync;
        if (sj != kNone) return sj;
    }
    return stop_hint;
}

// Pass 1 of part c from the end of its first block up to the next part's block start.
template <int NW>
__device__ void inflate_part(TeamSmem<NW>& S, const FileDesc* __restrict__ files, ChunkDesc* chunks, int c,
                             uint16_t* symbuf, uint32_t* start_bits, uint32_t* tok, const KParams& p) {
    ChunkDesc& C = chunks[c];
    if (C.state != CS_FOUND) return;
    if (C.probe) {                    // a streamed segment's end: the block start found is all it gives
        __syncthreads();
        if (threadIdx.x == 0) {
            C.state = CS_DONE;
            C.n = 0;
            C.anyph = 0;
            C.blocks = 0;
            C.final = 0;
            C.confirmed = 0;
            C.end = C.sync;
        }
        return;
    }
    const FileDesc& F = files[C.file];
    const uint64_t stop = find_stop(F, chunks, c, C.stop_hint);
    OutState o{symbuf + C.sym_base, start_bits + C.sym_base / 32, C.cap, C.n, C.n, C.index == 0 && C.sync == F.s0_bit, false};
    uint32_t blocks = C.blocks, final = C.final, err = CE_OK, confirmed = C.confirmed;
    uint64_t end = C.resume;
    // the confirmation (Section "Detection of DEFLATE block start positions") covers the start's block and
    // the confirm_blocks blocks after it; they are decoded with the literal checks
    const uint32_t window = (uint32_t)p.confirm_blocks + 1u;
    if (final) {
        if (stop != kNone && !F.open_end) err = CE_CHAIN;
    } else if (!(stop != kNone && C.resume == stop) || (C.confirm_ext && !confirmed)) {
        init_smem<NW>(S, p);
        TeamState ts = team_state<NW>(tok, p, (uint32_t)min(C.resume - C.sync, (uint64_t)0xfffffffu));
        const Input in(F.gz, F.gz_len);
        uint64_t bit = C.resume;
        // past the stop (confirm_ext): blocks decoded only to finish the confirmation; the part's own
        // output, end and status are those at the stop
        bool past = false;
        uint32_t err_stop = CE_OK;
        uint64_t n_stop = 0, end_stop = 0;
        for (;;) {
            const uint64_t pos = bit;
            if (!past && stop != kNone && pos >= stop) {
                err_stop = pos != stop ? (uint32_t)CE_CHAIN : (uint32_t)CE_OK;
                if (!C.confirm_ext || blocks >= window) {
                    err = err_stop;
                    break;
                }
                past = true;
                n_stop = o.n;
                end_stop = pos;
            }
            if (past && blocks >= window) break;
            const bool check = !o.known && blocks < window;
            uint32_t fin = 0;
            const int st = one_block<NW>(S, in, bit, ts, o, check, 0, 0, false, F.end_bit, fin);
            if (st) {
                err = (check && st != CE_OVERFLOW) ? (uint32_t)CE_CONFIRM : (uint32_t)st;
                break;
            }
            ++blocks;
            if (fin) {
                if (blocks <= window) confirmed = 1;
                if (past) break;
                final = 1;
                if (stop != kNone && !F.open_end) err = CE_CHAIN;   // an open member may end before the next part
                break;
            }
        }
        end = bit;
        if (blocks >= window && err != CE_CONFIRM) confirmed = 1;
        if (past) {
            if (err == CE_OK) err = err_stop;
            if (err != CE_CONFIRM && err != CE_OVERFLOW) {
                o.n = n_stop;
                end = end_stop;
            }
        }
    }
    const bool neg = __syncthreads_or(o.neg);
    if (err == CE_OK && final && F.mode != 2 && !F.open_end) {   // the trailer must follow the final block
        if (((end + 7) >> 3) + 8 != F.gz_len) err = CE_TRAIL;
    }
    if (threadIdx.x == 0) {
        C.state = err ? CS_ERROR : CS_DONE;
        C.err = err;
        C.n = o.n;
        C.anyph = C.anyph | (neg ? 1u : 0u);
        C.blocks = blocks;
        C.final = final;
        C.confirmed = confirmed;
        C.end = end;
    }
}

// Launch bounds of the pass-1 kernels, the blocks per SM that the registers are to allow (MB): with many parts what
// shared memory holds, 11 teams of 2 warps (80 registers a thread) and 7 of 4 (72; 64, for an eighth team that does not
// fit, spilled).  Larger teams are for few parts, where a part's own time counts: 3 of 8 warps (80 registers; at 4,
// with 64, they spilled; files of 305 to 611 parts take the same time either way).  Teams of 16 have two forms: 2 per
// SM (64 registers) and, where the parts fill at most half of the SMs, 1 per SM (128), k_sync + k_inflate: 1 MiB file
// 433 -> 389 us, 64 KiB 161 -> 145, eight byte ranges 2380 -> 2130.
// With 9 bits of distance lookup instead of 8 fewer steps take the rare branch: k_inflate of a 256 MiB file 1343 ->
// 1251 us.
constexpr int pass1_min_blocks(int nw) { return nw == 2 ? 11 : (nw == 4 ? 7 : (nw == 8 ? 3 : 2)); }

// the teams that pass1_min_blocks counts on fit the 228 KiB of an SM (1 KiB of it reserved per block)
template <int NW>
constexpr bool team_fits() { return pass1_min_blocks(NW) * (sizeof(TeamSmem<NW>) + 1024) <= 228 * 1024; }
static_assert(team_fits<2>() && team_fits<4>() && team_fits<8>() && team_fits<16>(), "more teams than shared memory holds");

template <int NW, int MB = pass1_min_blocks(NW)>
__global__ void __launch_bounds__(32 * NW, MB)
    k_sync(const FileDesc* __restrict__ files, ChunkDesc* chunks, int nchunks, uint16_t* symbuf, uint32_t* start_bits,
           uint32_t* tok, uint32_t* queue, const uint32_t* __restrict__ order, KParams p) {
    TeamSmem<NW>& S = team_smem<NW>();
    for (;;) {
        const int q = next_part<NW>(S, queue);
        if (q >= nchunks) return;
        const int c = order ? (int)__ldg(order + q) : q;
        sync_part<NW>(S, files[chunks[c].file], chunks[c], symbuf, start_bits, tok, p);
    }
}

template <int NW, int MB = pass1_min_blocks(NW)>
__global__ void __launch_bounds__(32 * NW, MB)
    k_inflate(const FileDesc* __restrict__ files, ChunkDesc* chunks, int nchunks, uint16_t* symbuf, uint32_t* start_bits,
              uint32_t* tok, uint32_t* queue, const uint32_t* __restrict__ order, KParams p) {
    TeamSmem<NW>& S = team_smem<NW>();
    for (;;) {
        const int q = next_part<NW>(S, queue);
        if (q >= nchunks) return;
        const int c = order ? (int)__ldg(order + q) : q;
        inflate_part<NW>(S, files, chunks, c, symbuf, start_bits, tok, p);
    }
}

// ---------------------------------------------------------------------------
// k_exec: the copy map of each part into its symbols, in place
// ---------------------------------------------------------------------------
// One block of NT threads per part, in passes of 8 NT positions (a thread takes
// 8 consecutive ones: one 16-byte load, one 16-byte store; a warp's 256 begin at
// a multiple of kRestart, so the code in force at each comes from the start
// bits and codes of its own lanes).  The last 32 KiB of the part's symbols live
// in a ring in shared memory, the pass itself in a stage beside it.  A
// position's stage entry is its symbol when the source lies before the pass
// (read from the ring; U_j when it lies before the part), else kPtr | the
// source's index inside the pass.  After one barrier every thread follows its
// own pointers; each step shortens the chain the next reader follows (an entry
// is replaced by the entry it points to), an entry only ever changes to an
// earlier source or to its symbol, and indices strictly decrease, so the chase
// needs no further barrier and ends, overlapping copies included.  The pass's
// symbols then go to the ring, whose places they take are no longer read.
// Bound: instruction issue (0.60 G warp instructions, all but a few with 32 threads, for the 509 M symbols of 64
// members: about 37 a position).  0.74 ms for the 1024 parts of a 256 MiB file (364 G symbols/s); 1.05 ms with a branch per
// position and entry in the chase, whose loads then wait for one another.
constexpr uint32_t kPtr = 0x4000u;    // neither a byte nor a placeholder; the index takes 14 bits

template <int NT>
constexpr size_t exec_smem() { return (kWin + 8 * NT) * sizeof(uint16_t); }

__device__ __forceinline__ uint32_t lds_u16(uint32_t a) {
    uint16_t v;
    asm volatile("ld.volatile.shared.u16 %0, [%1];" : "=h"(v) : "r"(a));
    return v;
}

template <int NT>
__global__ void __launch_bounds__(NT, NT == 512 ? 2 : 3)
    k_exec(const FileDesc* __restrict__ files, ChunkDesc* chunks, int nchunks, uint16_t* symbuf,
           const uint32_t* __restrict__ start_bits, uint32_t* queue, const uint32_t* __restrict__ order, int tail) {
    extern __shared__ __align__(16) uint16_t ring[];     // kWin symbols, then the stage
    __shared__ int s_q;
    constexpr uint32_t P = 8 * NT;
    static_assert(kWin % P == 0 && P <= kPtr, "whole passes in the ring, indices in 14 bits");
    uint16_t* stage = ring + kWin;
    const uint32_t ring_a = (uint32_t)__cvta_generic_to_shared(ring), stage_a = ring_a + 2 * kWin;
    static_assert(kRestart == 256, "a warp's positions of a pass");
    const uint32_t t8 = 8u * threadIdx.x;
    const uint32_t below = (1u << (threadIdx.x & 31)) - 1u;
    for (;;) {
        __syncthreads();
        if (threadIdx.x == 0) s_q = (int)min(atomicAdd(queue, 1u), 0x7fffffffu);
        __syncthreads();
        const int q = s_q;
        if (q >= nchunks) return;
        ChunkDesc& C = chunks[order ? (int)__ldg(order + q) : q];
        if (C.state != CS_DONE || C.n == 0) continue;
        const uint32_t n = (uint32_t)C.n;
        uint16_t* sym = symbuf + C.sym_base;
        // the determined tail when the configuration asks for it; decoding from a bit offset keeps every
        // symbol as u16 (its caller asks for the symbols themselves)
        const bool track = tail && files[C.file].mode != 1;
        uint32_t det = 0xffffffffu, ph_end = 0;      // tail start; end of the last pass that held a placeholder
        const uint8_t* start = reinterpret_cast<const uint8_t*>(start_bits) + C.sym_base / 8;
        uint4 nx = make_uint4(0, 0, 0, 0);
        uint32_t nst = 0;
        if (t8 < n) {
            nx = *reinterpret_cast<const uint4*>(sym + t8);
            nst = start[t8 >> 3];
        }
        for (uint32_t A = 0; A < n; A += P) {
            const uint32_t p0 = A + t8;
            uint32_t w4[4] = {nx.x, nx.y, nx.z, nx.w}, st = nst;
            if (p0 + P < n) {
                nx = *reinterpret_cast<const uint4*>(sym + p0 + P);
                nst = start[(p0 + P) >> 3];
            }
            if (A + P > n) {                         // the last pass: byte 0 past the part's end
                const uint32_t nv = p0 < n ? min(n - p0, 8u) : 0u;
                st = (st & ((1u << nv) - 1u)) | (0xffu & (0xffu << nv));
#pragma unroll
                for (uint32_t k = 0; k < 4; ++k)
                    w4[k] = 2 * k + 1 < nv ? w4[k] : (2 * k < nv ? w4[k] & 0xffffu : 0u);
            }
            // the last code of the lanes below is in force at my first position
            const uint32_t top = st ? 31u - __clz(st) : 0u;
            const uint32_t last = (top < 4 ? (top < 2 ? w4[0] : w4[1]) : (top < 6 ? w4[2] : w4[3])) >> (16u * (top & 1u));
            const uint32_t has = __ballot_sync(FULL, st != 0) & below;
            uint32_t code = __shfl_sync(FULL, last, has ? 31 - __clz(has) : 0) & 0xffffu;
            // (selections, not branches: the eight loads of a thread are in flight together, here and below)
            uint32_t e[8], ptr[8];
            int32_t q[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const uint32_t c = (u & 1) ? w4[u >> 1] >> 16 : w4[u >> 1] & 0xffffu;
                code = (st >> u) & 1u ? c : code;
                e[u] = code;
                q[u] = (int32_t)(p0 + u) - 1 - (int32_t)(code & 0x7fffu);   // a match's source
                ptr[u] = lds_u16(ring_a + 2u * ((uint32_t)q[u] & (kWin - 1u)));
            }
            uint32_t open = 0;
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const bool match = e[u] >> 15, in = match && q[u] >= (int32_t)A;
                const uint32_t val = q[u] < 0 ? ((uint32_t)q[u] & 0x7fffu) | kPH : ptr[u], rel = (uint32_t)q[u] - A;
                e[u] = in ? kPtr | rel : (match ? val : e[u]);
                ptr[u] = stage_a + 2u * (in ? rel : t8 + u);                // a resolved entry reads itself
                open |= in;
            }
            uint4 v4;
            auto pack = [&]() {
                v4.x = e[0] | (e[1] << 16);
                v4.y = e[2] | (e[3] << 16);
                v4.z = e[4] | (e[5] << 16);
                v4.w = e[6] | (e[7] << 16);
            };
            pack();
            *reinterpret_cast<uint4*>(stage + t8) = v4;
            __syncthreads();
            while (__any_sync(FULL, open)) {
                open = 0;
#pragma unroll
                for (int u = 0; u < 8; ++u) e[u] = lds_u16(ptr[u]);
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    const bool more = (e[u] & 0xc000u) == kPtr;
                    ptr[u] = more ? stage_a - 2u * kPtr + 2u * e[u] : ptr[u];
                    open |= more;
                }
                pack();
                *reinterpret_cast<uint4*>(stage + t8) = v4;   // a thread's entries change only by its own hand
            }
            *reinterpret_cast<uint4*>(ring + ((A + t8) & (kWin - 1u))) = v4;
            if (det == 0xffffffffu && track && A >= ph_end + kWin) det = A;
            if (track) {
                const uint32_t any = (v4.x | v4.y | v4.z | v4.w) & (kPH | (kPH << 16));
                if (__syncthreads_or((int)any)) ph_end = A + P;
            } else {
                __syncthreads();
            }
            if (p0 < n) {
                if (det != 0xffffffffu) {            // bytes at det + position, always behind the map still unread
                    uint2 b;
                    b.x = __byte_perm(v4.x, v4.y, 0x6420);
                    b.y = __byte_perm(v4.z, v4.w, 0x6420);
                    *reinterpret_cast<uint2*>(reinterpret_cast<uint8_t*>(sym) + det + p0) = b;
                } else {
                    *reinterpret_cast<uint4*>(sym + p0) = v4;
                }
            }
        }
        if (threadIdx.x == 0 && det != 0xffffffffu) C.det = det;
    }
}

// ---------------------------------------------------------------------------
// k_plan: output offsets, error aggregation, length checks (one block per member)
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(1024) k_plan(FileDesc* files, ChunkDesc* chunks) {
    FileDesc& F = files[blockIdx.x];
    __shared__ uint64_t part[1024];
    __shared__ uint32_t bad, fin;
    __shared__ int any_final;
    const int t = threadIdx.x;
    if (t == 0) {
        bad = 0xffffffffu;
        fin = 0xffffffffu;
        any_final = 0;
    }
    __syncthreads();
    // an open member ends with the first part that decoded its final block; the parts after it lie in
    // what follows the member (the next member, or other data) and are dropped
    if (F.open_end)
        for (int i = t; i < F.nchunks; i += 1024) {
            const ChunkDesc& C = chunks[F.chunk0 + i];
            if (C.state == CS_DONE && C.final) atomicMin(&fin, (uint32_t)i);
        }
    __syncthreads();
    uint64_t carry = F.out_base;
    for (int b0 = 0; b0 < F.nchunks; b0 += 1024) {
        const int c = F.chunk0 + b0 + t;
        uint64_t n = 0;
        if (b0 + t < F.nchunks && (uint32_t)(b0 + t) > fin) {
            chunks[c].state = CS_EMPTY;
        } else if (b0 + t < F.nchunks) {
            ChunkDesc& C = chunks[c];
            if (C.state == CS_DONE) {
                n = C.n;
                if (C.final) atomicOr(&any_final, 1);
            } else if (C.state == CS_ERROR) {
                atomicMin(&bad, (uint32_t)(b0 + t));
            }
        }
        part[t] = n;
        __syncthreads();
        for (int d = 1; d < 1024; d <<= 1) {          // inclusive scan
            const uint64_t v = t >= d ? part[t - d] : 0;
            __syncthreads();
            part[t] += v;
            __syncthreads();
        }
        if (b0 + t < F.nchunks) chunks[c].out_off = carry + part[t] - n;
        carry += part[1023];
        __syncthreads();
    }
    if (t == 0) {
        const uint64_t total = carry - F.out_base;
        F.total = total;
        F.bad_chunk = bad;
        F.crc_acc = 0;
        F.member_end = F.gz_len;
        uint32_t st = PGZ_OK;
        if (F.open_end && fin != 0xffffffffu && bad == 0xffffffffu) {   // the member's own trailer
            const uint64_t me = ((chunks[F.chunk0 + fin].end + 7) >> 3) + 8;
            if (me > F.gz_len) {
                st = PGZ_E_DATA;
            } else {
                const uint8_t* tr = F.gz + me - 8;
                F.crc_expect = tr[0] | ((uint32_t)tr[1] << 8) | ((uint32_t)tr[2] << 16) | ((uint32_t)tr[3] << 24);
                F.isize_expect = tr[4] | ((uint32_t)tr[5] << 8) | ((uint32_t)tr[6] << 16) | ((uint32_t)tr[7] << 24);
                F.member_end = me;
            }
        }
        if (st == PGZ_OK) {
            if (bad != 0xffffffffu) {
                F.bad_err = chunks[F.chunk0 + bad].err;
                st = F.bad_err == CE_TRAIL ? PGZ_E_UNSUPPORTED : PGZ_E_DATA;
            } else if (!any_final && (F.mode == 0 || F.mode == 1 || (F.mode == 3 && F.last_seg))) {
                st = PGZ_E_DATA;
            } else if (F.mode != 2 && total > F.out_cap) {
                st = PGZ_E_CAPACITY;
            } else if (F.mode == 0 && (uint32_t)total != F.isize_expect) {
                st = PGZ_E_ISIZE;
            } else if (F.mode == 3 && F.last_seg && (uint32_t)(F.out_before + total) != F.isize_expect) {
                st = PGZ_E_ISIZE;
            }
        }
        F.status = st;
    }
}

// ---------------------------------------------------------------------------
// pass 2a: the window chain
// map of part c: entry k of w_{c+1} is D_c[n-32768+k] if that exists (a byte
// or U_j -> w_c[j]), else w_c[k+n]
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint16_t map_entry(const uint16_t* d, uint64_t n, uint64_t det, uint32_t k) {
    const int64_t t = (int64_t)n - (int64_t)kWin + (int64_t)k;
    if (t < 0) return (uint16_t)(kPH | (uint32_t)(k + n));
    return (uint64_t)t >= det ? reinterpret_cast<const uint8_t*>(d)[det + (uint64_t)t] : d[t];   // det: the tail
}

// The items of a run of the chain, in order: PARTS, the finished parts c0 .. c0 + n - 1 of the plan (others hold
// nothing and are skipped), else the composed maps c0 .. at `maps`.
template <bool PARTS>
struct ChainItem {
    const uint16_t* d = nullptr;
    uint64_t n = 0, det = 0;
    int c = 0;                    // the item (past the last: end)
    __device__ __forceinline__ void find(int from, int end, const ChunkDesc* chunks, const uint16_t* base) {
        c = from;
        if (!PARTS) {
            d = base + (uint64_t)c * kWin;
            return;
        }
        for (; c < end; ++c) {
            const ChunkDesc& C = chunks[c];
            if (C.state == CS_DONE && C.n != 0) {
                d = base + C.sym_base;
                n = C.n;
                det = C.det;
                return;
            }
        }
    }
    // whole entries in memory, entry k at plain()[k] (a part with 32 Ki u16 symbols or more): loads without a branch
    __device__ __forceinline__ bool is_plain() const { return !PARTS || (n >= kWin && det >= n); }
    __device__ __forceinline__ const uint16_t* plain() const { return PARTS ? d + (n - kWin) : d; }
    __device__ __forceinline__ uint32_t entry(uint32_t k) const { return PARTS ? map_entry(d, n, det, k) : d[k]; }
};

// Each thread handles the entries tid + 1024 j, j < 32.  A step's 32 loads of a thread were issued during the step
// before (each register is refilled as soon as its entry is used), so a step costs its shared-memory gathers, about
// 3 us, and not the latency of the symbols.
constexpr int kChainPer = kWin / 1024;

// m: the entries of `it`, if it is an item (else left alone)
template <bool PARTS>
__device__ __forceinline__ void chain_fill(uint32_t (&m)[kChainPer], const ChainItem<PARTS>& it, int end) {
    if (it.c >= end) return;
    if (it.is_plain()) {
        const uint16_t* p = it.plain() + threadIdx.x;
#pragma unroll
        for (int j = 0; j < kChainPer; ++j) m[j] = p[1024 * j];
    } else {
#pragma unroll
        for (int j = 0; j < kChainPer; ++j) m[j] = it.entry(threadIdx.x + 1024u * j);
    }
}

// One step: put(k, e) for every entry e = m[j] of k = tid + 1024 j, and m refilled with the next item's (next.c <
// end) entries on the way.
template <bool PARTS, typename Put>
__device__ __forceinline__ void chain_step(uint32_t (&m)[kChainPer], const ChainItem<PARTS>& next, int end, Put put) {
    if (next.c < end && next.is_plain()) {
        const uint16_t* p = next.plain() + threadIdx.x;
#pragma unroll
        for (int j = 0; j < kChainPer; ++j) {
            const uint32_t e = m[j];
            m[j] = p[1024 * j];
            put(threadIdx.x + 1024u * j, e);
        }
    } else {
#pragma unroll
        for (int j = 0; j < kChainPer; ++j) put(threadIdx.x + 1024u * j, m[j]);
        chain_fill<PARTS>(m, next, end);
    }
}

// the composed map of each group's items; the last group of a member has no successor, so no one reads its map
template <bool PARTS>
__global__ void __launch_bounds__(1024) k_chain_compose(const FileDesc* __restrict__ files,
                                                        const ChunkDesc* __restrict__ chunks, const int32_t* g0,
                                                        const int32_t* gn, const int32_t* gfile,
                                                        const uint16_t* __restrict__ src, uint16_t* gmaps) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    uint16_t* acc = reinterpret_cast<uint16_t*>(smem_raw);
    uint16_t* tmp = acc + kWin;
    const int g = blockIdx.x;
    const FileDesc& F = files[gfile[g]];
    if (F.status != PGZ_OK || g + 1 == (PARTS ? F.group0 + F.ngroups : F.super0 + F.nsupers)) return;
    const uint32_t tid = threadIdx.x;
    const int end = g0[g] + gn[g];
    uint16_t* dst = gmaps + (uint64_t)g * kWin;
    ChainItem<PARTS> it;
    it.find(g0[g], end, chunks, src);
    if (it.c >= end) {
        for (uint32_t k = tid; k < kWin; k += 1024) dst[k] = (uint16_t)(kPH | k);
        return;
    }
    uint32_t m[kChainPer];
    chain_fill<PARTS>(m, it, end);
    bool have = false;
    for (;;) {
        it.find(it.c + 1, end, chunks, src);
        const bool more = it.c < end;
        uint16_t* to = more ? tmp : dst;
        if (have)
            chain_step<PARTS>(m, it, end, [&](uint32_t k, uint32_t e) {
                const uint32_t w = acc[e & (kWin - 1)];
                to[k] = (uint16_t)((e & kPH) ? w : e);
            });
        else
            chain_step<PARTS>(m, it, end, [&](uint32_t k, uint32_t e) { to[k] = (uint16_t)e; });
        if (!more) return;
        __syncthreads();
        uint16_t* x = acc;
        acc = tmp;
        tmp = x;
        have = true;
    }
}

// Resolved windows along each group's items, from the window before its first: out[item] = the window before that
// item (PARTS: every part of the group, skipped ones too).  win (null: each member's own start, FileDesc::win0 or
// nothing) holds the groups' first windows.  T: bytes, or u16 symbols, for a member decoded from an unknown context
// (then null: that context itself, entry k the placeholder U_k).
template <bool PARTS, typename T>
__global__ void __launch_bounds__(1024) k_chain_expand(const FileDesc* __restrict__ files,
                                                       const ChunkDesc* __restrict__ chunks, const int32_t* g0,
                                                       const int32_t* gn, const int32_t* gfile,
                                                       const uint16_t* __restrict__ src, const T* win, T* out) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T* W = reinterpret_cast<T*>(smem_raw);
    T* W2 = W + kWin;
    const int g = blockIdx.x;
    const FileDesc& F = files[gfile[g]];
    if (F.status != PGZ_OK) return;
    const uint32_t tid = threadIdx.x;
    const int c0 = g0[g], end = c0 + gn[g];
    ChainItem<PARTS> it;
    it.find(c0, end, chunks, src);
    uint32_t m[kChainPer];
    chain_fill<PARTS>(m, it, end - 1);                   // the last item's own map leads out of the group
    constexpr uint32_t kVec = kWin * sizeof(T) / 16;     // a window in 16-byte words
    if (sizeof(T) == 2 && !win) {
        for (uint32_t k = tid; k < kWin; k += 1024) W[k] = (T)(kPH | k);
    } else {
        const T* ws = win ? win + (uint64_t)g * kWin : reinterpret_cast<const T*>(F.win0);
        for (uint32_t k = tid; k < kVec; k += 1024)
            reinterpret_cast<uint4*>(W)[k] = ws ? reinterpret_cast<const uint4*>(ws)[k] : make_uint4(0, 0, 0, 0);
    }
    __syncthreads();
    int c = c0;                                          // next item whose window is not written
    for (;;) {
        const int last = min(it.c, end - 1);             // the items up to the next finished part share this window
        for (; c <= last; ++c)
            for (uint32_t k = tid; k < kVec; k += 1024)
                reinterpret_cast<uint4*>(out + (uint64_t)c * kWin)[k] = reinterpret_cast<const uint4*>(W)[k];
        if (c >= end) return;
        it.find(it.c + 1, end, chunks, src);
        chain_step<PARTS>(m, it, end - 1, [&](uint32_t k, uint32_t e) {
            const uint32_t w = W[e & (kWin - 1)];
            W2[k] = (T)((e & kPH) ? w : e);
        });
        __syncthreads();
        T* x = W;
        W = W2;
        W2 = x;
    }
}

// The symbols of a member decoded from a bit offset in several parts, relative to the context before its first part:
// part c's U_j is entry j of its u16 window.  sym_out and byte_out (nullable; placeholders as `fill`) receive them in
// order; res[0], res[1]: placeholders left, one past the last.  kAtSplit blocks per part.  Coalesced loads and stores
// of one symbol a thread: about 3 symbols a cycle and SM, a tenth of the time of the decoding before it.
constexpr int kAtSplit = 2;

__global__ void __launch_bounds__(512) k_resolve_at(const FileDesc* __restrict__ files, const ChunkDesc* __restrict__ chunks,
                                                    const uint16_t* __restrict__ sym, const uint16_t* __restrict__ windows,
                                                    uint16_t* sym_out, uint8_t* byte_out, uint8_t fill,
                                                    unsigned long long* res) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    uint16_t* W = reinterpret_cast<uint16_t*>(smem_raw);
    const int c = blockIdx.x / kAtSplit;
    const ChunkDesc& C = chunks[c];
    if (files[C.file].status != PGZ_OK || C.state != CS_DONE || C.n == 0) return;
    const uint32_t n = (uint32_t)C.n, per = (n + kAtSplit - 1) / kAtSplit, a = (blockIdx.x % kAtSplit) * per;
    if (C.anyph)
        for (uint32_t k = threadIdx.x; k < kWin / 8; k += blockDim.x)
            reinterpret_cast<uint4*>(W)[k] = reinterpret_cast<const uint4*>(windows + (uint64_t)c * kWin)[k];
    __syncthreads();
    const uint16_t* s = sym + C.sym_base;
    const uint32_t z = min(n, a + per);
    uint32_t cnt = 0;
    uint64_t last = 0;
#pragma unroll 4
    for (uint32_t i = a + threadIdx.x; i < z; i += blockDim.x) {
        uint32_t v = s[i];
        if (v & kPH) v = W[v & (kWin - 1)];
        const uint64_t P = C.out_off + i;
        sym_out[P] = (uint16_t)v;
        if (byte_out) byte_out[P] = (v & kPH) ? fill : (uint8_t)v;
        if (v & kPH) {
            ++cnt;
            last = P + 1;
        }
    }
    cnt = __reduce_add_sync(FULL, cnt);
    for (int d = 16; d; d >>= 1) last = max(last, shfl64(last, (threadIdx.x & 31) ^ d));
    if ((threadIdx.x & 31) == 0 && cnt) {
        atomicAdd(&res[0], (unsigned long long)cnt);
        atomicMax(&res[1], (unsigned long long)last);
    }
}

// ---------------------------------------------------------------------------
// pass 2b: translation U_j -> w_i[j], 8 symbols per thread per step
// ---------------------------------------------------------------------------

// Persistent: block b translates units b, b + gridDim.x, ... (a unit is a part, or
// a piece of one when there are few parts: 18 us for the 8 parts of a 1 MiB file
// with one block each); the part's
// window w_i is copied into shared memory (only if the part produced a
// placeholder) while the block's previous unit is translated (two tables).  The shared table is the window followed by the 256 byte
// values, so a symbol s (a byte b < 0x100, or 0x8000 | j for U_j) becomes
// T[s ^ 0x8000]: window byte j for a placeholder, b for a byte, with no
// branch.  Parts without any placeholder pack their bytes with byte
// permutations.
//
// A warp writes a contiguous run of slices of 512 symbols, a lane 16
// symbols (two 16-byte loads) of each; the loads of the next slice are in
// flight while a slice is translated.
// Output bytes P..P+15 of a lane (P = out_off + symbol index) go out as the
// two aligned 8-byte words from P - m (m = out_off mod 8); the m bytes before
// P come from the previous lane (lane 31's from the previous slice), the m
// bytes after P + 15 - m are the next lane's first word.  Partial slices and
// the first slice of a warp's run take byte stores where a neighbour is
// missing.
constexpr int kTransThreads = 512;
constexpr uint32_t kTransSlice = 512;                  // symbols per slice (16 per lane)
constexpr size_t kTransSmem = 2 * (kWin + 256);         // two window tables

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}

// 8 symbols -> 8 bytes (symbols past nv are taken as byte 0)
__device__ __forceinline__ uint64_t translate8(const uint8_t* T, uint4 q, uint32_t nv, bool ph) {
    uint32_t w4[4] = {q.x, q.y, q.z, q.w};
    if (nv < 8) {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            if (2u * k >= nv) w4[k] = 0;
            else if (2u * k + 1 >= nv) w4[k] &= 0xffffu;
        }
    }
    uint32_t b0, b1;
    if (!ph) {
        b0 = __byte_perm(w4[0], w4[1], 0x6420);
        b1 = __byte_perm(w4[2], w4[3], 0x6420);
    } else {
        uint32_t pr[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const uint32_t w = w4[k] ^ 0x80008000u;
            pr[k] = (uint32_t)T[w & 0xffffu] | ((uint32_t)T[w >> 16] << 8);
        }
        b0 = __byte_perm(pr[0], pr[1], 0x5410);
        b1 = __byte_perm(pr[2], pr[3], 0x5410);
    }
    return (uint64_t)b0 | ((uint64_t)b1 << 32);
}

// 8 bytes of the determined tail as they are (bytes past nv taken as 0)
__device__ __forceinline__ uint64_t tail8(uint4 q, uint32_t nv) {
    const uint64_t v = (uint64_t)q.x | ((uint64_t)q.y << 32);
    return nv >= 8 ? v : (nv ? v & (~0ull >> (64 - 8 * nv)) : 0ull);
}

__global__ void __launch_bounds__(kTransThreads, 2) k_translate(const FileDesc* __restrict__ files, ChunkDesc* chunks,
                                                                int nchunks, const uint16_t* __restrict__ sym,
                                                                const uint8_t* __restrict__ windows,
                                                                const uint8_t* __restrict__ fillw, int split) {
    extern __shared__ __align__(16) uint8_t Wbuf[];      // two tables of kWin + 256 bytes (kTransSmem)
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
    if (threadIdx.x < 256) {
        Wbuf[kWin + threadIdx.x] = (uint8_t)threadIdx.x;
        Wbuf[2 * kWin + 256 + threadIdx.x] = (uint8_t)threadIdx.x;
    }
    const int nwork = nchunks * split;                   // unit w: piece w % split of part w / split
    // the window of unit w's part goes into table `buf` by asynchronous copies, one group per unit
    auto fetch = [&](int w, int buf) {
        if (w < nwork) {
            const int c = w / split;
            const ChunkDesc& C = chunks[c];
            if (files[C.file].status == PGZ_OK && C.state == CS_DONE && C.n != 0 && C.anyph) {
                const uint8_t* src = fillw ? fillw : windows + (uint64_t)c * kWin;
                const uint32_t dst = smem_u32(Wbuf + buf * (kWin + 256));
                for (uint32_t k = threadIdx.x; k < kWin / 16; k += blockDim.x) cp_async16(dst + 16 * k, src + 16 * k);
            }
        }
        cp_async_commit();
    };
    fetch(blockIdx.x, 0);
    int buf = 0;
    for (int w = blockIdx.x; w < nwork; w += gridDim.x, buf ^= 1) {
        fetch(w + gridDim.x, buf ^ 1);                    // the next unit's window, while this one runs
        cp_async_wait<1>();                               // this unit's window (this thread's copies) ...
        __syncthreads();                                  // ... and everyone else's
        const uint8_t* W = Wbuf + buf * (kWin + 256);
        const ChunkDesc& C = chunks[w / split];
        const FileDesc& F = files[C.file];
        const bool ph = C.anyph != 0;
        if (F.status == PGZ_OK && C.state == CS_DONE && C.n != 0) {   // uniform per block
        const uint16_t* s = sym + C.sym_base;
        // output byte P of the member goes to out[P - out_lo] when out_lo <= P < out_hi
        uint8_t* out = F.out;
        const uint64_t lo = F.out_lo, hi = F.out_hi;
        const bool vec = F.out_lo == 0 && F.out_hi == kNone && ((reinterpret_cast<uintptr_t>(out) & 7) == 0);
        const uint32_t m = (uint32_t)(C.out_off & 7), sh = 8u * m;
        const uint32_t n32 = (uint32_t)C.n;
        // the part's slices, those that hold output bytes in [lo, hi) only, in equal runs over the units' warps
        uint32_t s0 = 0, nsl = (n32 + kTransSlice - 1) / kTransSlice;
        if (lo > C.out_off) s0 = (uint32_t)min((lo - C.out_off) / kTransSlice, (uint64_t)nsl);
        if (hi < C.out_off + n32) nsl = hi > C.out_off ? (uint32_t)((hi - C.out_off + kTransSlice - 1) / kTransSlice) : 0u;
        const uint32_t cnt = nsl > s0 ? nsl - s0 : 0u, runs = (uint32_t)(nwarp * split);
        const uint32_t per = (cnt + runs - 1) / runs, run = (uint32_t)(w % split) * nwarp + (uint32_t)warp;
        const uint32_t j0 = s0 + min(cnt, per * run), j1 = s0 + min(cnt, per * (run + 1));
        // the determined tail (symbols from det32 on are bytes at byte det32 + k; det32 is a multiple of 8, so
        // each 8-symbol half lies wholly before or wholly inside it): copied, not translated
        const uint32_t det32 = C.det < (uint64_t)n32 ? (uint32_t)C.det : 0xffffffffu;
        const uint8_t* tb = reinterpret_cast<const uint8_t*>(s) + (det32 == 0xffffffffu ? 0u : det32);
        auto load_half = [&](uint32_t j, uint32_t i0, uint4& a) {
            if (!(j < j1 && i0 < n32)) {
                a = make_uint4(0, 0, 0, 0);
            } else if (i0 >= det32) {
                const uint2 v = *reinterpret_cast<const uint2*>(tb + i0);
                a = make_uint4(v.x, v.y, 0, 0);
            } else {
                a = *reinterpret_cast<const uint4*>(s + i0);
            }
        };
        // loads of slice j + 1 are in flight while slice j is translated
        auto load = [&](uint32_t j, uint4& a, uint4& b) {
            const uint32_t i = j * kTransSlice + 16u * (uint32_t)lane;
            load_half(j, i, a);
            load_half(j, i + 8, b);
        };
        uint4 n0, n1;
        load(j0, n0, n1);
        uint64_t carry = 0;                               // lane 31's second word of the previous slice
        for (uint32_t j = j0; j < j1; ++j) {
            const uint4 q0 = n0, q1 = n1;
            load(j + 1, n0, n1);
            const uint32_t i = j * kTransSlice + 16u * (uint32_t)lane;
            const bool full = (j + 1) * kTransSlice <= n32;   // uniform: every lane holds 16 symbols
            const uint32_t nv = full ? 16u : (i < n32 ? min(n32 - i, 16u) : 0u);
            const uint64_t v0 = i >= det32 ? tail8(q0, nv < 8 ? nv : 8u) : translate8(W, q0, nv < 8 ? nv : 8u, ph);
            const uint64_t v1 = i + 8 >= det32 ? tail8(q1, nv > 8 ? nv - 8 : 0u)
                                               : translate8(W, q1, nv > 8 ? nv - 8 : 0u, ph);
            const uint64_t P = C.out_off + i;
            if (!vec || !full) {          // each lane stores its own bytes (clipped to [lo, hi) when !vec)
                for (uint32_t k = 0; k < nv; ++k) {
                    const uint64_t q = P + k;
                    if (q >= lo && q < hi) out[q - lo] = (uint8_t)((k < 8 ? v0 : v1) >> (8 * (k & 7)));
                }
                continue;
            }
            if (m == 0) {
                *reinterpret_cast<uint64_t*>(out + P) = v0;
                *reinterpret_cast<uint64_t*>(out + P + 8) = v1;
                continue;
            }
            uint64_t prev = __shfl_up_sync(FULL, v1, 1);
            if (lane == 0) prev = carry;
            carry = shfl64(v1, 31);
            const bool have_prev = lane > 0 || j > j0;    // the previous slice of this run was full
            if (have_prev) {
                *reinterpret_cast<uint64_t*>(out + P - m) = (v0 << sh) | (prev >> (64 - sh));
            } else {
                for (uint32_t k = 0; k < 8 - m; ++k) out[P + k] = (uint8_t)(v0 >> (8 * k));
            }
            *reinterpret_cast<uint64_t*>(out + P + 8 - m) = (v1 << sh) | (v0 >> (64 - sh));
            // my last m bytes start the next lane's first word; lane 31 writes them itself unless
            // the next slice is full and in this run
            if (lane == 31) {
                const bool next_full = j + 1 < j1 && (j + 2) * kTransSlice <= n32;
                if (!next_full)
                    for (uint32_t k = 16 - m; k < 16; ++k) out[P + k] = (uint8_t)(v1 >> (8 * (k - 8)));
            }
        }
        }
        __syncthreads();                                  // table `buf` is refilled two parts later
    }
    cp_async_wait<0>();
}

// placeholder count of every part and one past its last placeholder (for
// statistics and inspection; not on the decompression path)
__global__ void __launch_bounds__(256) k_count_ph(ChunkDesc* chunks, int nchunks, const uint16_t* __restrict__ sym) {
    __shared__ unsigned long long s_n, s_last;
    for (int c = blockIdx.x; c < nchunks; c += gridDim.x) {
        ChunkDesc& C = chunks[c];
        __syncthreads();
        if (threadIdx.x == 0) {
            s_n = 0;
            s_last = 0;
        }
        __syncthreads();
        const uint64_t n0 = C.state == CS_DONE ? C.n : 0;
        const uint64_t n = n0 < C.det ? n0 : C.det;        // a determined tail holds no placeholder
        const uint16_t* p = sym + C.sym_base;
        unsigned long long cnt = 0, last = 0;
        for (uint64_t i = threadIdx.x; i < n; i += blockDim.x)
            if (p[i] & kPH) {
                ++cnt;
                last = i + 1;
            }
        for (int d = 16; d; d >>= 1) {
            cnt += __shfl_xor_sync(FULL, cnt, d);
            last = max(last, __shfl_xor_sync(FULL, last, d));
        }
        if ((threadIdx.x & 31) == 0) {
            atomicAdd(&s_n, cnt);
            atomicMax(&s_last, last);
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            C.nph = s_n;
            C.last_ph = s_last;
        }
    }
}

// ---------------------------------------------------------------------------
// CRC-32 in GF(2): reflected representation, bit 31-k = coefficient of x^k
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t gf2_mul(uint32_t a, uint32_t b) {
    uint32_t p = 0;
#pragma unroll
    for (int k = 0; k < 32; ++k) {
        p ^= b & (0u - ((a >> (31 - k)) & 1u));
        b = (b >> 1) ^ (kPoly & (0u - (b & 1u)));
    }
    return p;
}

// x^(8n) mod P, n < 2^40: a product of one power per byte of n (a multiplication is a serial chain, so their number
// counts: with powers of two, one per set bit of n, k_crc took 22 us for 1 MiB and 85 us for 256 MiB, now 8 and 71)
__device__ uint32_t xpow8(uint64_t n) {
    uint32_t r = c_x8[0][n & 255u];
    for (int d = 1; d < 5; ++d) {
        const uint32_t v = (uint32_t)(n >> (8 * d)) & 255u;
        if (v) r = gf2_mul(r, c_x8[d][v]);
    }
    return r;
}

constexpr uint32_t kPiece = 32;       // bytes per lane and segment
constexpr uint32_t kCrcSeg = 32 * kPiece;   // bytes per warp step (one piece per lane)
constexpr int kCrcAhead = 3;          // segments whose loads are in flight while one is folded
constexpr int kCrcThreads = 1024;     // one block per SM
// Four byte tables, then the segment shift's four byte tables (4 KiB).  REPL: one copy of the first four per lane
// (128 KiB), so that the lookups of a warp never share a bank: 72 us instead of 126 for 256 MiB; else one copy (4 KiB),
// whose lookups conflict but which is filled at once: for 1 MiB (one segment per warp) 8 us instead of 13.  At 12.6 MB
// (three) the copies take 18 us, the single tables 23.
template <bool REPL>
constexpr size_t crc_smem() { return ((REPL ? 32 : 1) * 4 * 256 + 4 * 256) * sizeof(uint32_t); }
constexpr uint64_t kCrcRepl = 3;      // segments per warp from which the copies pay

// Slicing by four (four table lookups per 32-bit word, RFC 1952 CRC in the
// reflected form): with x = r ^ w, the register after the word's four bytes
// is T3[x0] ^ T2[x1] ^ T1[x2] ^ T0[x3], where Tk is the byte table followed
// by k zero bytes.  With copies, entry b of table k of lane l is at word
// 32 * (256 k + b) + l.
template <bool REPL>
struct CrcTable {
    const uint32_t* t;      // with copies: this lane's
    __device__ __forceinline__ uint32_t at(uint32_t i) const { return t[REPL ? 32u * i : i]; }
    __device__ __forceinline__ uint32_t word(uint32_t r, uint32_t w) const {
        const uint32_t x = r ^ w;
        return at(768u + (x & 0xffu)) ^ at(512u + ((x >> 8) & 0xffu)) ^ at(256u + ((x >> 16) & 0xffu)) ^ at(x >> 24);
    }
};

// raw CRC register (zero start) of a whole piece held in registers
template <bool REPL>
__device__ __forceinline__ uint32_t crc_piece(const CrcTable<REPL>& T, const uint4 (&v)[kPiece / 16]) {
    uint32_t r = 0;
#pragma unroll
    for (int q = 0; q < (int)(kPiece / 16); ++q) {
        r = T.word(r, v[q].x);
        r = T.word(r, v[q].y);
        r = T.word(r, v[q].z);
        r = T.word(r, v[q].w);
    }
    return r;
}

// raw CRC register (zero start) of n bytes at p, byte by byte
template <bool REPL>
__device__ __forceinline__ uint32_t crc_bytes(const CrcTable<REPL>& T, const uint8_t* p, uint64_t n) {
    uint32_t r = 0;
    for (uint64_t i = 0; i < n; ++i) r = T.at((r ^ p[i]) & 0xffu) ^ (r >> 8);
    return r;
}

// r times x^(8 kCrcSeg) mod P: by linearity, the XOR of the products of r's four bytes, each looked up in
// its own table (Y + 256 j: byte j of the register, in place, times the constant)
__device__ __forceinline__ uint32_t crc_shift_seg(const uint32_t* Y, uint32_t r) {
    return Y[r & 0xffu] ^ Y[256u + ((r >> 8) & 0xffu)] ^ Y[512u + ((r >> 16) & 0xffu)] ^ Y[768u + (r >> 24)];
}

// Each warp takes a contiguous run of segments and walks the members it
// covers.  Within a member, lane l's pieces (bytes 32 l .. 32 l + 31 of each
// segment) are folded across the run's full segments by Horner's rule,
// acc_l <- acc_l x^(8 kCrcSeg) + R(piece), so that at the end acc_l
// x^(8 kPiece (31 - l)), summed over the lanes, is the raw CRC of those
// segments (R(A||B) = R(A) x^(8|B|) + R(B)); that sum is shifted to the end
// of the member once and XOR-accumulated there.  The loads of the next
// kCrcAhead segments are in flight while a segment is folded (a warp's
// 32-byte pieces are one 1 KiB stretch, so each load instruction reads few
// lines).  A member's last segment, when shorter, is done byte by byte with
// per-lane shifts, and so is a member whose output is not 16-byte aligned.
template <bool REPL>
__global__ void __launch_bounds__(kCrcThreads, 1) k_crc(FileDesc* files, int nfiles, uint64_t total_seg,
                                                        const uint64_t* seg0, uint64_t segs_per_warp) {
    extern __shared__ uint32_t T[];                       // 4 x 256 words (x 32 copies), then 4 x 256 (the segment shift)
    __shared__ uint32_t LS[32];
    constexpr int kCopies = REPL ? 32 : 1;
    for (int k = threadIdx.x; k < 4 * 256 * kCopies; k += blockDim.x) T[k] = c_crc_tab[k / (256 * kCopies)][k / kCopies & 255];
    uint32_t* Y = T + 4 * 256 * kCopies;
    for (int k = threadIdx.x; k < 4 * 256; k += blockDim.x) Y[k] = c_seg_shift[k >> 8][k & 255];
    if (threadIdx.x < 32) LS[threadIdx.x] = c_lane_shift[threadIdx.x];
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const CrcTable<REPL> Tl{T + (REPL ? lane : 0)};
    const uint64_t w = (uint64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const uint64_t s_begin = w * segs_per_warp;
    if (s_begin >= total_seg) return;
    const uint64_t s_end = s_begin + segs_per_warp < total_seg ? s_begin + segs_per_warp : total_seg;
    int f;
    {
        int lo = 0, hi = nfiles - 1;                      // member holding the run's first segment
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (seg0[mid] <= s_begin) lo = mid;
            else hi = mid - 1;
        }
        f = lo;
    }
    // this lane's part of a raw CRC that ends `shift` bytes before the end of member f: summed over the warp,
    // shifted to the end, accumulated
    auto add = [&](uint32_t r, uint64_t shift) {
        for (int d = 16; d; d >>= 1) r ^= __shfl_xor_sync(FULL, r, d);
        if (lane == 0) atomicXor(&files[f].crc_acc, shift ? gf2_mul(r, xpow8(shift)) : r);
    };
    for (uint64_t sg = s_begin; sg < s_end; ++f) {        // one member of the run per step
        const uint64_t m_end = f + 1 < nfiles ? seg0[f + 1] : ~0ull;
        if (sg >= m_end) continue;                        // a member with no segment
        const uint64_t g_end = m_end < s_end ? m_end : s_end;
        const FileDesc& F = files[f];
        const uint64_t i0 = sg - seg0[f], i1 = g_end - seg0[f];   // the member's segments [i0, i1) in this run
        sg = g_end;
        if (F.status != PGZ_OK || (F.mode != 0 && F.mode != 3)) continue;
        const uint64_t D = F.total;
        const uint8_t* out = F.out;
        const uint64_t nfull = D / kCrcSeg;
        const uint64_t ie = i1 < nfull ? i1 : nfull;      // full segments [i0, ie)
        const uint8_t* base = out + (uint64_t)kPiece * lane;
        if (i0 < ie) {
            uint32_t acc = 0;
            if ((reinterpret_cast<uintptr_t>(out) & 15) == 0) {
                uint4 v[kCrcAhead + 1][kPiece / 16];
                auto load = [&](uint64_t i, uint4 (&dst)[kPiece / 16]) {
                    if (i < ie) {
                        const uint4* p = reinterpret_cast<const uint4*>(base + i * kCrcSeg);
#pragma unroll
                        for (int q = 0; q < (int)(kPiece / 16); ++q) dst[q] = p[q];
                    }
                };
#pragma unroll
                for (int k = 0; k < kCrcAhead; ++k) load(i0 + k, v[k]);
                for (uint64_t i = i0; i < ie; i += kCrcAhead + 1) {
#pragma unroll
                    for (int k = 0; k <= kCrcAhead; ++k) {
                        if (i + k < ie) {
                            load(i + k + kCrcAhead, v[(k + kCrcAhead) % (kCrcAhead + 1)]);
                            const uint32_t r = crc_piece(Tl, v[k]);
                            acc = i + k > i0 ? crc_shift_seg(Y, acc) ^ r : r;
                        }
                    }
                }
            } else {
                for (uint64_t i = i0; i < ie; ++i) {
                    const uint32_t r = crc_bytes(Tl, base + i * kCrcSeg, kPiece);
                    acc = i > i0 ? crc_shift_seg(Y, acc) ^ r : r;
                }
            }
            add(gf2_mul(acc, LS[31 - lane]), D - ie * kCrcSeg);
        }
        if (i0 <= nfull && nfull < i1 && D > nfull * kCrcSeg) {   // the member's last segment, shorter
            const uint64_t pa = nfull * kCrcSeg + (uint64_t)kPiece * lane;
            const uint64_t pb = pa + kPiece < D ? pa + kPiece : D;
            uint32_t r = 0;
            if (pa < pb) r = gf2_mul(crc_bytes(Tl, out + pa, pb - pa), xpow8(D - pb));
            add(r, 0);
        }
    }
}

__global__ void k_finalize(FileDesc* files, int nfiles) {
    const int f = blockIdx.x * blockDim.x + threadIdx.x;
    if (f >= nfiles) return;
    FileDesc& F = files[f];
    if (F.status != PGZ_OK) return;
    if (F.mode == 3) {
        // register after the segment, from the register the earlier segments left (R_I(M) = I x^(8|M|) + R_0(M))
        const uint32_t reg = F.crc_acc ^ gf2_mul(F.crc_in, xpow8(F.total));
        F.crc = reg;
        if (F.last_seg && (reg ^ 0xffffffffu) != F.crc_expect) F.status = PGZ_E_CRC;
        return;
    }
    if (F.mode != 0) return;
    // register after D bytes from the initial all-ones register, then inverted
    const uint32_t crc = F.crc_acc ^ gf2_mul(0xffffffffu, xpow8(F.total)) ^ 0xffffffffu;
    F.crc = crc;
    if (crc != F.crc_expect) F.status = PGZ_E_CRC;
}

// ---------------------------------------------------------------------------
// DNA sequences in a block with undetermined characters (Appendix "Heuristic
// extraction of DNA sequences in DEFLATE block"): the maximal non-overlapping
// substrings matching T D+ (U+ D+)* T, T a newline or an undetermined
// character, D a nucleotide, U an undetermined character.  Within a maximal
// run of D/U symbols there is at most one: from the first D preceded by a T
// to the last D followed by a T (outside the run, only a newline is a T), if
// the first comes before the last.  k_seq_classes turns the symbols into three
// bit arrays (D, U, newline; coalesced, at the rate of the loads);
// k_sequences then walks each run a word of 32 symbols at a time, from the
// thread of the word it starts in.  Walking the symbols themselves, 1024 to a
// thread, took 3.4 ms for 4.9 M symbols: the runs of a block whose context is
// unknown are thousands of symbols long.
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t seq_class(uint16_t s) {      // 0 other, 1 D, 2 U, 3 newline
    if (s & kPH) return 2;
    const uint32_t b = s & 0xffu;
    if (b == 'A' || b == 'C' || b == 'G' || b == 'T' || b == 'N') return 1;
    return b == '\n' ? 3 : 0;
}

constexpr uint32_t kSeqPer = 8;      // words of 32 symbols per warp

// bits: nw words of D, then of U, then of newlines (bits past n are zero)
__global__ void __launch_bounds__(256) k_seq_classes(const uint16_t* __restrict__ sym, uint64_t n, uint64_t nw,
                                                     uint32_t* bits) {
    const uint32_t lane = threadIdx.x & 31;
    const uint64_t w0 = (((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * kSeqPer;
    uint16_t s[kSeqPer];
#pragma unroll
    for (uint32_t k = 0; k < kSeqPer; ++k) {
        const uint64_t i = 32 * (w0 + k) + lane;
        s[k] = i < n ? sym[i] : 0;
    }
#pragma unroll
    for (uint32_t k = 0; k < kSeqPer; ++k) {
        const uint32_t c = seq_class(s[k]);
        const uint32_t d = __ballot_sync(FULL, c == 1), u = __ballot_sync(FULL, c == 2), l = __ballot_sync(FULL, c == 3);
        if (lane < 3 && w0 + k < nw) bits[lane * nw + w0 + k] = lane == 0 ? d : (lane == 1 ? u : l);
    }
}

__global__ void __launch_bounds__(256) k_sequences(const uint32_t* __restrict__ bits, uint64_t nw, uint32_t min_len,
                                                   uint64_t* spans, uint64_t max_spans, unsigned long long* counts) {
    const uint32_t *D = bits, *U = bits + nw, *N = bits + 2 * nw;
    const uint64_t t = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= nw) return;
    const uint32_t r0 = D[t] | U[t];
    const uint32_t rp = t ? (D[t - 1] | U[t - 1]) >> 31 : 0u, np = t ? N[t - 1] >> 31 : 0u;
    for (uint32_t starts = r0 & ~((r0 << 1) | rp); starts; starts &= starts - 1) {
        const uint32_t b = __ffs(starts) - 1;
        const bool open_left = b ? (N[t] >> (b - 1)) & 1u : np;
        uint64_t first = ~0ull, last = ~0ull, u_after = ~0ull;   // u_after: the first U after `first`
        uint32_t m = FULL << b;                                  // the run's symbols in word w
        uint32_t follows = open_left ? 1u << b : 0u;             // symbols of w that follow a T: what the word before,
                                                                 // or the newline before the run, tells
        for (uint64_t w = t;; ++w) {
            const uint32_t d = D[w], u = U[w], l = N[w], r = d | u;
            const uint32_t stop = ~r & m;                        // the run ends at its lowest bit
            const uint32_t in = stop ? m & ((stop & (0u - stop)) - 1u) : m;
            const uint32_t next = w + 1 < nw ? (U[w + 1] | N[w + 1]) & 1u : 0u;
            const uint32_t s = d & in & (((u & in) << 1) | follows);
            const uint32_t e = d & in & (((u | l) >> 1) | (next << 31));
            const uint64_t base = 32 * w;
            if (first == ~0ull && s) first = base + (uint32_t)__ffs(s) - 1;
            if (e) last = base + 31u - (uint32_t)__clz(e);
            if (first != ~0ull && u_after == ~0ull) {
                const uint32_t ua = u & in & (first >= base ? FULL << (uint32_t)(first - base) : FULL);
                if (ua) u_after = base + (uint32_t)__ffs(ua) - 1;
            }
            if (stop || w + 1 >= nw) break;
            follows = u >> 31;
            m = FULL;
        }
        if (first != ~0ull && last != ~0ull && last >= first && last - first + 1 >= min_len) {
            const unsigned long long k = atomicAdd(&counts[0], 1ull);
            const bool und = u_after < last;
            if (und) atomicAdd(&counts[1], 1ull);
            if (k < max_spans) {
                spans[2 * k] = first;
                spans[2 * k + 1] = (last - first + 1) | (und ? (1ull << 63) : 0ull);
            }
        }
    }
}

// The first kHeadBytes bytes and the last 8 of every member of a batch, one warp per member, so that the host reads
// all of them with one copy (the caller has made sure that they lie in device memory).
__global__ void __launch_bounds__(128) k_heads(const MemberRef* __restrict__ in, int n, uint8_t* out) {
    const int m = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (m >= n) return;
    const uint8_t* gz = in[m].gz;
    const uint64_t len = in[m].len;
    uint8_t* o = out + (uint64_t)m * (kHeadBytes + 8);
    for (uint32_t k = lane; k < kHeadBytes; k += 32) o[k] = k < len ? gz[k] : 0;
    if (lane < 8 && len >= 8) o[kHeadBytes + lane] = gz[len - 8 + lane];
}

}  // namespace

// ---------------------------------------------------------------------------
// host wrappers
// ---------------------------------------------------------------------------
void launch_heads(const MemberRef* in, int n, uint8_t* out, cudaStream_t s) {
    if (n > 0) k_heads<<<(n + 3) / 4, 128, 0, s>>>(in, n, out);
}

uint64_t sequence_words(uint64_t n) { return 3 * ((n + 31) / 32); }

void launch_sequences(const uint16_t* sym, uint64_t n, uint32_t min_len, uint32_t* bits, uint64_t* spans,
                      uint64_t max_spans, unsigned long long* counts, cudaStream_t s) {
    cudaMemsetAsync(counts, 0, 2 * sizeof(unsigned long long), s);
    if (n == 0) return;
    const uint64_t nw = (n + 31) / 32, per_block = 8 * kSeqPer;
    k_seq_classes<<<(unsigned)((nw + per_block - 1) / per_block), 256, 0, s>>>(sym, n, nw, bits);
    k_sequences<<<(unsigned)((nw + 255) / 256), 256, 0, s>>>(bits, nw, min_len, spans, max_spans, counts);
}

// resident teams of a size on the current device (both pass-1 kernels have the same launch bounds and shared
// memory); also raises the kernels' dynamic shared-memory limit once
template <int NW>
static int pass1_resident_t() {
    static int cached[64] = {};
    int dev = 0;
    cudaGetDevice(&dev);
    const int slot = dev >= 0 && dev < 64 ? dev : 0;
    if (!cached[slot]) {
        const int smem = (int)sizeof(TeamSmem<NW>);
        int sms = 0, per_sm_a = 0, per_sm_b = 0;
        auto raise = [smem](auto kernel) {
            return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) == cudaSuccess;
        };
        bool ok = raise(k_sync<NW>) && raise(k_inflate<NW>);
        if constexpr (NW == 16) ok = ok && raise(k_sync<NW, 1>) && raise(k_inflate<NW, 1>);
        ok = ok &&
            cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess &&
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm_a, k_sync<NW>, 32 * NW, smem) == cudaSuccess &&
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm_b, k_inflate<NW>, 32 * NW, smem) == cudaSuccess;
        const int v = std::max(1, sms) * std::max(1, std::min(per_sm_a, per_sm_b));
        if (!ok) {
            cudaGetLastError();
            return v;                            // not cached: asked again once a device answers
        }
        cached[slot] = v;
    }
    return cached[slot];
}

static int pass1_resident(int nw) {
    switch (nw) {
        case 2: return pass1_resident_t<2>();
        case 8: return pass1_resident_t<8>();
        case 16: return pass1_resident_t<16>();
        default: return pass1_resident_t<4>();
    }
}

// Rows of the teams' token buffers: twice the tokens of a segment of ordinary text (about 8 bits each).  Data of
// fewer bits a token ends its rounds early and shortens its segments.
static uint32_t team_rows(int nw) { return nw <= 8 ? 384 : 256; }

// Warps per part: with few parts the largest team whose launch still holds every part at once (the time of a part
// falls with its team's size: 8 parts of a 1 MiB file take 0.20 ms of block-start search and 0.19 ms of decoding with
// teams of 16, against 0.86 and 1.36 ms with one warp each); with more parts than that the configured size, whose
// rounds spend less on lanes left over.  Teams of 8 instead of two teams of 16 on an SM are faster for
// one call (160 parts of a 12 MiB text: 1.14 ms against 1.23) but slower for runs side by side (40 requests served in
// 4 slots: 1.64 against 1.55).
int pass1_team(int nchunks, int wpb) {
    const int base = wpb == 2 || wpb == 8 ? wpb : 4;
    for (int nw = 16; nw > base; nw >>= 1)
        if (nchunks <= pass1_resident(nw)) return nw;
    return base;
}

int pass1_parts(int wpb) { return pass1_resident(wpb == 2 || wpb == 8 ? wpb : 4); }

static int pass1_grid(int nchunks, int nw) { return std::min(nchunks, pass1_resident(nw)); }

uint64_t token_words(int nchunks, int wpb) {
    if (nchunks <= 0) return 0;
    const int nw = pass1_team(nchunks, wpb);
    return (uint64_t)pass1_grid(nchunks, nw) * 32 * nw * team_rows(nw);
}

template <int NW>
static void launch_pass1_t(bool sync, const FileDesc* files, ChunkDesc* chunks, int nchunks, uint16_t* sym,
                           uint32_t* start, uint32_t* tok, uint32_t* queue, const uint32_t* order, const KParams& p, cudaStream_t s) {
    const int grid = pass1_grid(nchunks, NW);
    KParams q = p;
    if (!p.team) q.tok_rows = team_rows(NW);
    auto launch = [&](auto kernel) {
        kernel<<<grid, 32 * NW, sizeof(TeamSmem<NW>), s>>>(files, chunks, nchunks, sym, start, tok, queue, order, q);
    };
    if constexpr (NW == 16) {                    // the form with more registers (see pass1_min_blocks)
        if (nchunks <= pass1_resident(16) / 4) return launch(sync ? k_sync<NW, 1> : k_inflate<NW, 1>);
    }
    launch(sync ? k_sync<NW> : k_inflate<NW>);
}

static void launch_pass1_any(bool sync, const FileDesc* files, ChunkDesc* chunks, int nchunks, uint16_t* sym,
                             uint32_t* start, uint32_t* tok, uint32_t* queue, const uint32_t* order, const KParams& p,
                             cudaStream_t s) {
    if (nchunks <= 0) return;
    switch (p.team ? p.team : pass1_team(nchunks, p.wpb)) {
        case 2: launch_pass1_t<2>(sync, files, chunks, nchunks, sym, start, tok, queue, order, p, s); break;
        case 8: launch_pass1_t<8>(sync, files, chunks, nchunks, sym, start, tok, queue, order, p, s); break;
        case 16: launch_pass1_t<16>(sync, files, chunks, nchunks, sym, start, tok, queue, order, p, s); break;
        default: launch_pass1_t<4>(sync, files, chunks, nchunks, sym, start, tok, queue, order, p, s); break;
    }
}

void launch_sync(const FileDesc* files, ChunkDesc* chunks, int nchunks, uint16_t* sym, uint32_t* start, uint32_t* tok,
                 uint32_t* queue, const uint32_t* order, const KParams& p, cudaStream_t s) {
    launch_pass1_any(true, files, chunks, nchunks, sym, start, tok, queue, order, p, s);
}

void launch_inflate(const FileDesc* files, ChunkDesc* chunks, int nchunks, uint16_t* sym, uint32_t* start,
                    uint32_t* tok, uint32_t* queue, const uint32_t* order, const KParams& p, cudaStream_t s) {
    launch_pass1_any(false, files, chunks, nchunks, sym, start, tok, queue, order, p, s);
}

// k_exec's resident blocks on the current device (0 if it cannot be asked)
template <int NT>
static int exec_resident() {
    static int cached[64] = {};
    int dev = 0, sms = 0, per_sm = 0;
    cudaGetDevice(&dev);
    const int slot = dev >= 0 && dev < 64 ? dev : 0;
    if (!cached[slot]) {
        if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess &&
            cudaFuncSetAttribute(k_exec<NT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)exec_smem<NT>()) ==
                cudaSuccess &&
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_exec<NT>, NT, exec_smem<NT>()) == cudaSuccess)
            cached[slot] = sms * per_sm;
        else
            cudaGetLastError();
    }
    return cached[slot];
}

template <int NT>
static void launch_exec_t(const FileDesc* files, ChunkDesc* chunks, int nchunks, uint16_t* sym, uint32_t* start, uint32_t* queue,
                          const uint32_t* order, const KParams& p, cudaStream_t s) {
    const int cap = std::max(1, exec_resident<NT>());
    k_exec<NT><<<std::min(nchunks, cap), NT, exec_smem<NT>(), s>>>(files, chunks, nchunks, sym, start, queue, order, p.tail);
}

void launch_exec(const FileDesc* files, ChunkDesc* chunks, int nchunks, uint16_t* sym, uint32_t* start, uint32_t* queue,
                 const uint32_t* order, const KParams& p, cudaStream_t s) {
    if (nchunks <= 0) return;
    // With at most one part per SM, blocks of 512 threads: half the passes of a part (file of 8 parts: 53 us, against
    // 59 us with 256).  With more, 256: three fit an SM (two of 512), and shorter passes hold fewer sources inside
    // them, so they take fewer chase steps (1024 parts of 256 MiB: 737 us, against 873 us with 512 and 996 us with
    // 1024).
    if (nchunks <= exec_resident<512>() / 2) launch_exec_t<512>(files, chunks, nchunks, sym, start, queue, order, p, s);
    else launch_exec_t<256>(files, chunks, nchunks, sym, start, queue, order, p, s);
}

void launch_plan(FileDesc* files, ChunkDesc* chunks, int nfiles, cudaStream_t s) {
    if (nfiles <= 0) return;
    k_plan<<<nfiles, 1024, 0, s>>>(files, chunks);
}

// Parts -> group maps -> (supergroup maps ->) the windows before the first items, member by member, then group by
// group (through the supergroups), then part by part.
template <typename T>
static void launch_chain_t(const FileDesc* files, const ChunkDesc* chunks, int nfiles, const ChainPlan& C,
                           const uint16_t* sym, uint16_t* gmaps, T* wstart, T* windows, cudaStream_t s) {
    if (C.ngroups <= 0) return;
    constexpr int kSmem = 2 * kWin * (int)sizeof(T);
    static bool attr[64] = {};                            // the shared-memory limits are raised per device
    int dev = 0;
    cudaGetDevice(&dev);
    const int slot = dev >= 0 && dev < 64 ? dev : 0;
    if (!attr[slot]) {
        const auto raise = [](const void* f, int n) {
            return cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, n) == cudaSuccess;
        };
        attr[slot] = raise((const void*)k_chain_compose<true>, 4 * kWin) &&
                     raise((const void*)k_chain_compose<false>, 4 * kWin) &&
                     raise((const void*)k_chain_expand<true, T>, kSmem) &&
                     raise((const void*)k_chain_expand<false, T>, kSmem);
    }
    if (C.many) k_chain_compose<true><<<C.ngroups, 1024, 4 * kWin, s>>>(files, chunks, C.g0, C.gn, C.gfile, sym, gmaps);
    const T* first = nullptr;
    if (C.deep) {
        uint16_t* smaps = gmaps + (uint64_t)C.ngroups * kWin;
        T* swin = wstart + (uint64_t)C.ngroups * kWin;
        k_chain_compose<false><<<C.nsupers, 1024, 4 * kWin, s>>>(files, chunks, C.s0, C.sn, C.sfile, gmaps, smaps);
        k_chain_expand<false, T><<<nfiles, 1024, kSmem, s>>>(files, chunks, C.f0, C.fn, C.ffile, smaps, nullptr, swin);
        first = swin;
    }
    if (C.many)
        k_chain_expand<false, T><<<C.nsupers, 1024, kSmem, s>>>(files, chunks, C.s0, C.sn, C.sfile, gmaps, first, wstart);
    k_chain_expand<true, T><<<C.ngroups, 1024, kSmem, s>>>(files, chunks, C.g0, C.gn, C.gfile, sym,
                                                           C.many ? wstart : nullptr, windows);
}

void launch_chain(const FileDesc* files, const ChunkDesc* chunks, int nfiles, const ChainPlan& C, const uint16_t* sym,
                  uint16_t* gmaps, uint8_t* wstart, uint8_t* windows, cudaStream_t s) {
    launch_chain_t<uint8_t>(files, chunks, nfiles, C, sym, gmaps, wstart, windows, s);
}

void launch_resolve_at(const FileDesc* files, const ChunkDesc* chunks, int nchunks, const ChainPlan& C,
                       const uint16_t* sym, uint16_t* gmaps, uint16_t* wstart, uint16_t* windows, uint16_t* sym_out,
                       uint8_t* byte_out, uint8_t fill, unsigned long long* res, cudaStream_t s) {
    if (nchunks <= 0) return;
    launch_chain_t<uint16_t>(files, chunks, 1, C, sym, gmaps, wstart, windows, s);
    static bool attr[64] = {};
    int dev = 0;
    cudaGetDevice(&dev);
    const int slot = dev >= 0 && dev < 64 ? dev : 0;
    if (!attr[slot])
        attr[slot] = cudaFuncSetAttribute(k_resolve_at, cudaFuncAttributeMaxDynamicSharedMemorySize, 2 * kWin) == cudaSuccess;
    cudaMemsetAsync(res, 0, 2 * sizeof(unsigned long long), s);
    k_resolve_at<<<nchunks * kAtSplit, 512, 2 * kWin, s>>>(files, chunks, sym, windows, sym_out, byte_out, fill, res);
}

int chain_group_size(int n) {
    if (n <= 12) return n;
    const double g = n <= 64 ? std::sqrt((double)n) : std::cbrt((double)n);
    return (int)std::ceil(g);
}
int chain_super_size(int ngroups) {
    return ngroups <= 12 ? ngroups : (int)std::ceil(std::sqrt((double)ngroups));
}

void launch_translate(const FileDesc* files, ChunkDesc* chunks, int nchunks, uint64_t max_cap,
                      const uint16_t* sym, const uint8_t* windows, const uint8_t* fillw, cudaStream_t s) {
    if (nchunks <= 0) return;
    static int resident[64] = {};                         // blocks of k_translate that fit on the device at once
    int dev = 0;
    cudaGetDevice(&dev);
    const int slot = dev >= 0 && dev < 64 ? dev : 0;
    if (!resident[slot]) {
        int sms = 0, per_sm = 0;
        if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess &&
            cudaFuncSetAttribute(k_translate, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTransSmem) ==
                cudaSuccess &&
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_translate, kTransThreads, kTransSmem) == cudaSuccess &&
            sms > 0 && per_sm > 0)
            resident[slot] = sms * per_sm;
        else
            cudaGetLastError();
    }
    const int cap = resident[slot] ? resident[slot] : 152 * 2;
    // pieces of a part: enough units for the resident blocks, each piece worth its window's copy
    const uint64_t pieces = std::max<uint64_t>(1, max_cap / (2 * kWin));
    const int split = (int)std::min<uint64_t>({(uint64_t)std::max(1, cap / nchunks), pieces, 16});
    const int grid = std::min(nchunks * split, cap);
    k_translate<<<grid, kTransThreads, kTransSmem, s>>>(files, chunks, nchunks, sym, windows, fillw, split);
}

uint64_t crc_segment_bytes() { return kCrcSeg; }

void launch_count_ph(ChunkDesc* chunks, int nchunks, const uint16_t* sym, cudaStream_t s) {
    if (nchunks <= 0) return;
    k_count_ph<<<nchunks < 1216 ? nchunks : 1216, 256, 0, s>>>(chunks, nchunks, sym);
}

void launch_crc(FileDesc* files, int nfiles, uint64_t total_seg, const uint64_t* seg0, cudaStream_t s) {
    if (nfiles <= 0 || total_seg == 0) return;
    static int sms[64] = {};
    int dev = 0;
    cudaGetDevice(&dev);
    const int slot = dev >= 0 && dev < 64 ? dev : 0;
    if (!sms[slot]) {
        int n = 0;
        if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess && n > 0) sms[slot] = n;
        else cudaGetLastError();
        cudaFuncSetAttribute(k_crc<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)crc_smem<true>());
    }
    const uint64_t n = (uint64_t)(sms[slot] ? sms[slot] : 152);
    const uint64_t spw = (total_seg + n * (kCrcThreads / 32) - 1) / (n * (kCrcThreads / 32));   // one block per SM
    if (spw >= kCrcRepl) {
        const uint64_t wpb = kCrcThreads / 32, warps = (total_seg + spw - 1) / spw;
        k_crc<true><<<(unsigned)((warps + wpb - 1) / wpb), kCrcThreads, crc_smem<true>(), s>>>(files, nfiles, total_seg,
                                                                                              seg0, spw);
    } else {
        const uint64_t wpb = 8, warps = (total_seg + spw - 1) / spw;
        k_crc<false><<<(unsigned)((warps + wpb - 1) / wpb), 32 * wpb, crc_smem<false>(), s>>>(files, nfiles, total_seg,
                                                                                             seg0, spw);
    }
}

void launch_finalize(FileDesc* files, int nfiles, cudaStream_t s) {
    if (nfiles <= 0) return;
    k_finalize<<<(nfiles + 127) / 128, 128, 0, s>>>(files, nfiles);
}


// CRC-32 constants from the polynomial (RFC 1952 section 8)
static uint32_t h_mul(uint32_t a, uint32_t b) {
    uint32_t p = 0;
    for (int k = 0; k < 32; ++k) {
        if ((a >> (31 - k)) & 1u) p ^= b;
        b = (b & 1u) ? (b >> 1) ^ kPoly : (b >> 1);
    }
    return p;
}

void upload_crc_tables() {
    uint32_t tab[4][256], x2k[64], ls[32], x8[5][256];
    for (uint32_t b = 0; b < 256; ++b) {
        uint32_t r = b;
        for (int k = 0; k < 8; ++k) r = (r & 1u) ? (r >> 1) ^ kPoly : (r >> 1);
        tab[0][b] = r;
    }
    for (int k = 1; k < 4; ++k)                // k further zero bytes
        for (uint32_t b = 0; b < 256; ++b) tab[k][b] = (tab[k - 1][b] >> 8) ^ tab[0][tab[k - 1][b] & 0xffu];
    x2k[0] = 0x40000000u;                      // x
    for (int k = 1; k < 64; ++k) x2k[k] = h_mul(x2k[k - 1], x2k[k - 1]);
    for (int d = 0; d < 5; ++d) {              // powers of x^(8 256^d)
        x8[d][0] = 0x80000000u;
        for (int v = 1; v < 256; ++v) x8[d][v] = h_mul(x8[d][v - 1], x2k[3 + 8 * d]);
    }
    for (int l = 0; l < 32; ++l) {             // x^(8*kPiece*l)
        uint64_t e = 8ull * kPiece * (uint64_t)l;
        uint32_t r = 0x80000000u;
        for (int k = 0; e; ++k, e >>= 1)
            if (e & 1) r = h_mul(r, x2k[k]);
        ls[l] = r;
    }
    uint32_t xseg = 0x80000000u;
    {
        uint64_t e = 8ull * kCrcSeg;
        for (int k = 0; e; ++k, e >>= 1)
            if (e & 1) xseg = h_mul(xseg, x2k[k]);
    }
    uint32_t seg[4][256];                      // multiplication by x^(8*kCrcSeg), byte by byte (it is linear)
    for (int j = 0; j < 4; ++j)
        for (uint32_t b = 0; b < 256; ++b) seg[j][b] = h_mul(b << (8 * j), xseg);
    cudaMemcpyToSymbol(c_crc_tab, tab, sizeof tab);
    cudaMemcpyToSymbol(c_x8, x8, sizeof x8);
    cudaMemcpyToSymbol(c_lane_shift, ls, sizeof ls);
    cudaMemcpyToSymbol(c_seg_shift, seg, sizeof seg);
}

}  // namespace pgz
