// ea_tile.cuh -- the common end of a worker or server tile: given the residual-corrected input u
// of the tile's 4096 coordinates (16 per thread, in registers or parked in shared memory), form
// the group scale, encode and pack the message, and keep the residual e = u - Q(u) (Algorithm 1 /
// Algorithm 2).
#pragma once

#include "ea_device.cuh"

namespace ea {

// Per-warp results of group_partials, by parity of the reduction's turn.
struct PartRed {
    DF red[2][kWarps];
    uint32_t redm[2][kWarps];
};

struct TileSmem {
    DF red256[kThreads];  // per-thread partial pairs of the l1 scale
    PartRed parts;
    TileGroups tg;        // PASS_STASH, PASS_LAZY: the groups of a tile that holds several
    uint32_t redm[kWarps];
    float bcastf;
    float csc[kChunks];  // PASS_SHORT: the scale of each chunk
    int64_t part;        // PASS_STASH, PASS_LAZY: the tile's first partial norm (thread 0 writes and reads it)
    float qtab[256];  // the uniform grid's fl(i / L) of the tile's own quantizer (build_qtab)
};

// Slot k of this thread in tile `tile`: coordinates 4q .. 4q+3.  Consecutive threads own
// consecutive float4 slots, so every warp access is one contiguous 512-byte segment.
__device__ __forceinline__ int64_t slot_of(int64_t tile, int k)
{
    return tile * (kTile / 4) + k * kThreads + threadIdx.x;
}

// Where a tile's u comes from: this thread's registers (16 values), or shared memory, one float4 per
// slot at ls = k * kThreads + threadIdx.x.
struct URegs {
    float (*u)[4];
    __device__ __forceinline__ void get(int k, float (&o)[4]) const
    {
#pragma unroll
        for (int i = 0; i < 4; ++i) o[i] = u[k][i];
    }
};
struct USmem {
    const float4 *p;
    __device__ __forceinline__ void get(int k, float (&o)[4]) const
    {
        const float4 v = p[k * kThreads + threadIdx.x];
        o[0] = v.x, o[1] = v.y, o[2] = v.z, o[3] = v.w;
    }
};

// The scale of a tile's encode: one for the tile (a float), or one per chunk (short blocks), read
// once per slot by each warp.
struct ChunkScales {
    const float *csc;
};
__device__ __forceinline__ float slot_scale(float s, int) { return s; }
__device__ __forceinline__ float slot_scale(ChunkScales s, int k) { return s.csc[k * kWarps + (threadIdx.x >> 5)]; }
template <class Scale>
constexpr bool kPerSlot = false;
template <>
constexpr bool kPerSlot<ChunkScales> = true;

// For every group of Q that meets [lo, hi) (a range of tile `tile`), reduce this CTA's part of it
// -- |u| summed (compensated, to ~2^-44) for the scaled sign, max |u| for Example 1's grid -- over
// u read through `src` (shared memory) and store it as the group's partial for this tile.  One barrier per
// group: the warps' results go to pr by turn & 1 and thread 0 combines them in warp order.  tg: the
// tile's groups in shared memory, or null.  All threads call it.
template <int QK>
__device__ __forceinline__ void group_partials(const USmem &src, int64_t tile, int64_t lo, int64_t hi, int64_t d,
                                               const QParams &q, const TileRef &ref, const TileGroups *tg,
                                               double *partials, PartRed &pr, int &turn)
{
    const Grouping &G = q.grp;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t tl = tile * kTile;
    const int end = static_cast<int>(hi - tl);
    const bool cached = tg != nullptr && tg->nb <= kTileBounds;
#pragma unroll 1
    for (int64_t gi = (ref.ng() == 1 || lo == tl) ? ref.g0 : group_of(G, lo, ref.g0);; ++gi, ++turn) {
        const int i0 = static_cast<int>(gi - ref.g0);
        int a = 0, b = kTile;  // the group's part of the range, from the tile's start
        if (cached) {
            if (i0 > 0) a = tg->b[i0 - 1];
            if (i0 < tg->nb) b = tg->b[i0];
        } else if (ref.ng() > 1) {
            a = static_cast<int>(max(group_begin(G, gi, d) - tl, static_cast<int64_t>(0)));
            b = static_cast<int>(min(group_end(G, gi, d) - tl, static_cast<int64_t>(kTile)));
        }
        a = max(a, static_cast<int>(lo - tl));
        const bool last = b >= end;
        b = min(b, end);
        const int par = turn & 1;
        DF acc{0.0f, 0.0f};
        float mx = 0.0f;
#pragma unroll 1
        for (int k = 0; k < kSlots; ++k) {
            const int x = 4 * (k * kThreads + threadIdx.x);
            float u[4];
            src.get(k, u);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                if (x + i < a || x + i >= b) continue;
                if constexpr (QK == QK_SIGN) df_accumulate(acc, fabsf(u[i]));
                else mx = fmaxf(mx, fabsf(u[i]));
            }
        }
        if constexpr (QK == QK_SIGN) {
#pragma unroll 1
            for (int o = 16; o > 0; o >>= 1) {
                const DF w{__shfl_down_sync(0xffffffffu, acc.hi, o), __shfl_down_sync(0xffffffffu, acc.lo, o)};
                acc = df_add(acc, w);
            }
            if (lane == 0) pr.red[par][warp] = acc;
        } else {
            const uint32_t m = __reduce_max_sync(0xffffffffu, __float_as_uint(mx));  // exact on bit patterns
            if (lane == 0) pr.redm[par][warp] = m;
        }
        compute_sync();
        if (threadIdx.x == 0) {
            double part;
            if constexpr (QK == QK_SIGN) {
                DF t = pr.red[par][0];
#pragma unroll 1
                for (int w = 1; w < kWarps; ++w) t = df_add(t, pr.red[par][w]);
                part = static_cast<double>(t.hi) + static_cast<double>(t.lo);
            } else {
                uint32_t t = pr.redm[par][0];
#pragma unroll 1
                for (int w = 1; w < kWarps; ++w) t = max(t, pr.redm[par][w]);
                part = static_cast<double>(__uint_as_float(t));
            }
            partials[ref.part() + i0] = part;
        }
        if (last) {
            ++turn;  // the next call, too, writes the other half of pr while thread 0 may still read this one
            break;
        }
    }
}

// PASS_SHORT: the scales of the tile's blocks of 2^sh chunks, from u read through `src`, into
// sm.csc (one per chunk) and scales[].  A warp reduces its four chunks at once: for the scaled sign
// the compensated pairs of four slots are exchanged by halves, so that five shuffle levels take six
// pair additions (each lane keeps 2, 1, then 1 pair) instead of twenty.  Warp 0 then combines the
// 32 chunk results, one per lane, over the blocks.  Two barriers; all 256 threads call it.
template <int QK, class USrc>
__device__ __forceinline__ void chunk_scales(const USrc &src, int64_t tile, int64_t d, int sh, float *scales,
                                             TileSmem &sm)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    auto shfl = [](DF v, int o) { return DF{__shfl_xor_sync(0xffffffffu, v.hi, o), __shfl_xor_sync(0xffffffffu, v.lo, o)}; };
    static_assert(kSlots == 4 && kChunks == 32, "two halvings over the slots; one chunk per lane of warp 0");
    if constexpr (QK == QK_SIGN) {
        DF p[kSlots];
#pragma unroll
        for (int k = 0; k < kSlots; ++k) {
            float uk[4];
            src.get(k, uk);
            p[k] = DF{0.0f, 0.0f};
#pragma unroll
            for (int i = 0; i < 4; ++i) df_accumulate(p[k], fabsf(uk[i]));  // invalid u are 0
        }
        const bool h16 = lane & 16, h8 = lane & 8;
        const DF a = df_add(h16 ? p[2] : p[0], shfl(h16 ? p[0] : p[2], 16));
        const DF b = df_add(h16 ? p[3] : p[1], shfl(h16 ? p[1] : p[3], 16));
        DF c = df_add(h8 ? b : a, shfl(h8 ? a : b, 8));  // lane: slot lane / 8
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) c = df_add(c, shfl(c, o));
        if ((lane & 7) == 0) sm.red256[(lane >> 3) * kWarps + warp] = c;
    } else {
#pragma unroll
        for (int k = 0; k < kSlots; ++k) {
            float uk[4];
            src.get(k, uk);
            const float mx = fmaxf(fmaxf(fabsf(uk[0]), fabsf(uk[1])), fmaxf(fabsf(uk[2]), fabsf(uk[3])));
            const uint32_t m = __reduce_max_sync(0xffffffffu, __float_as_uint(fmaxf(0.0f, mx)));
            if (lane == 0) sm.red256[k * kWarps + warp].hi = __uint_as_float(m);
        }
    }
    compute_sync();
    if (warp == 0) {
        const int64_t base = tile * kTile + ((lane >> sh) << (sh + kLog2Chunk));  // the block's first coordinate
        const int64_t left = d - base;
        const int len = left < (kChunk << sh) ? static_cast<int>(left) : kChunk << sh;
        float s = 0.0f;
        if constexpr (QK == QK_SIGN) {
            DF v = sm.red256[lane];
            for (int o = 1; o < (1 << sh); o <<= 1) v = df_add(v, shfl(v, o));
            s = sign_scale(v, len);
        } else {
            s = sm.red256[lane].hi;
            for (int o = 1; o < (1 << sh); o <<= 1) s = fmaxf(s, __shfl_xor_sync(0xffffffffu, s, o));
        }
        sm.csc[lane] = s;
        if (len > 0 && (lane & ((1 << sh) - 1)) == 0) scales[tile * (kChunks >> sh) + (lane >> sh)] = s;
    }
    compute_sync();
}

// Example 1's grid index of u (|u| <= s, s > 0) without a division.  z = RN(u / s) and y = RN(z L)
// are stood in for by z' = RN(u r), y' = RN(z' L) with r = RN(1 / s), which the caller computes
// once per tile.  For s in [2^-125, 2^125] the relative errors of r, z', z and the two products
// (each at most 2^-24, |z| <= 1) give |y' - y| <= 5.01 * 2^-24 * L, below the margin m = L * 2^-20.
// The index changes only where y crosses a half-integer (round to nearest even) or, for the
// stochastic rule, an integer or the draw U; when y' is farther than m from every such point, y
// lies on the same side of each and gets the same index (so does u = 0, where y' = y = 0).
// Returns false otherwise, and for r = NaN, which the caller passes for scales outside the range:
// the caller then takes the index from unif_index, whose division gives z itself.
template <bool STO>
__device__ __forceinline__ bool unif_index_fast(float u, float r, float Lf, float m, float U, int &qi)
{
    const float y = __fmul_rn(__fmul_rn(u, r), Lf);
    if constexpr (STO) {
        const float f = floorf(y);
        const float fr = __fsub_rn(y, f);  // exact: |y| <= L + 1 < 2^23
        qi = static_cast<int>(f) + (U < fr ? 1 : 0);
        // u = 0 gives y' = y = 0 and index 0 exactly
        return (fr > m && fr < __fsub_rn(1.0f, m) && fabsf(__fsub_rn(U, fr)) > m) || u == 0.0f;
    } else {
        const float rn = rintf(y);
        qi = static_cast<int>(rn);
        return fabsf(__fsub_rn(y, rn)) < __fsub_rn(0.5f, m);
    }
}

// Variants of the per-coordinate encode, chosen once per tile: the uniform grid's zero scale
// (every q = 0), deterministic or stochastic rounding, decode from the fl(i/L) table or by division.
enum EncVar : int { ENC_PLAIN = 0, ENC_UZERO, ENC_UDET_TAB, ENC_UDET_DIV, ENC_USTO_TAB, ENC_USTO_DIV };

// Encode u (valid coordinates only) with its scale, store codes (all lanes) and the residual.
// FULL: the whole tile lies inside [0, d), so no coordinate needs a bounds check.
// BITS: the code width as a compile-time constant (0: code_bits of the kind, or q.bits).
// Only the coordinates of [lo, d) are encoded and stored (lo: 0, or the start of a word and a slot).
template <int QK, bool FULL, bool BALLOT, int VAR, int BITS, class USrc, class Scale>
__device__ __forceinline__ void encode_store_v(const USrc &src, Scale sc, int64_t tile, int64_t d,
                                               const QParams &q, uint32_t *words, float *resid, int ef,
                                               uint64_t seed, uint32_t id, uint32_t t, const float *qtab,
                                               int64_t lo = 0)
{
    constexpr bool STO = VAR == ENC_USTO_TAB || VAR == ENC_USTO_DIV;
    constexpr bool TAB = VAR == ENC_UDET_TAB || VAR == ENC_USTO_TAB;
    constexpr bool GRID = VAR != ENC_PLAIN && VAR != ENC_UZERO;
    const int bits = BITS ? BITS : code_bits<QK>(q);
    const int L = (QK == QK_UNIF) ? unif_L(bits) : 0;
    const float Lf = static_cast<float>(L);
    float s = 0.0f, r = 0.0f, m = 0.0f;
    auto take_scale = [&](int k) {  // a zero scale gives r = NaN, and unif_index then index 0
        s = slot_scale(sc, k);
        if (GRID) r = (s >= 0x1p-125f && s <= 0x1p125f) ? __frcp_rn(s) : __int_as_float(0x7fc00000);
    };
    if (GRID) m = __fmul_rn(Lf, 0x1p-20f);
    if constexpr (!kPerSlot<Scale>) take_scale(0);
#pragma unroll
    for (int k = 0; k < kSlots; ++k) {
        const int64_t qs = slot_of(tile, k);
        const int64_t j0 = 4 * qs;
        if constexpr (kPerSlot<Scale>) take_scale(k);
        float U[4] = {0.f, 0.f, 0.f, 0.f};
        if (STO && (FULL || j0 < d)) uniforms4(seed, id, t, j0, U);
        float uk[4];
        src.get(k, uk);
        uint32_t c[4];
        float e[4];
        int qi[4] = {0, 0, 0, 0};
        if (GRID) {
            // Example 1 with s > 0: the index of y = RN(RN(u / s) L) (see unif_index_fast)
            bool ok[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) ok[i] = unif_index_fast<STO>(uk[i], r, Lf, m, U[i], qi[i]);
            if (!(ok[0] && ok[1] && ok[2] && ok[3])) {
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    if (!ok[i]) qi[i] = unif_index(uk[i], s, Lf, STO, U[i]);
            }
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            float dec = 0.0f;
            uint32_t code = 0u;
            if (VAR == ENC_PLAIN) {
                code = encode1<QK>(uk[i], s, q, Lf, L, U[i], dec, qtab);
            } else if (VAR == ENC_UZERO) {
                code = static_cast<uint32_t>(L);  // Example 1: Q = 0 when the scale is 0
            } else {
                dec = __fmul_rn(s, TAB ? qtab[qi[i] + L] : __fdiv_rn(static_cast<float>(qi[i]), Lf));
                code = static_cast<uint32_t>(qi[i] + L);
            }
            c[i] = (FULL || j0 + i < d) ? code : 0u;
            e[i] = ef ? __fsub_rn(uk[i], dec) : 0.0f;
        }
        store_codes4<FULL, BALLOT>(words, qs, bits, c, lo, d);
        if (ef && (FULL || (j0 >= lo && j0 < d))) store4<FULL>(resid, qs, d, e);
    }
}

// Example 1 with a compile-time width: for b <= 8 the caller passes qtab (fl(i/L) of the tile's
// quantizer) and the decode is a table read; 16-bit grids divide.
template <int QK, bool FULL, bool BALLOT, int BITS, class USrc, class Scale>
__device__ __forceinline__ void encode_store_unif(const USrc &u, Scale sc, int64_t tile, int64_t d,
                                                  const QParams &q, uint32_t *words, float *resid, int ef,
                                                  uint64_t seed, uint32_t id, uint32_t t, const float *qtab,
                                                  int64_t lo = 0)
{
    constexpr bool tab = BITS <= 8;
    bool zero = false;
    if constexpr (!kPerSlot<Scale>) zero = !(sc > 0.0f);
    if (zero)
        encode_store_v<QK, FULL, BALLOT, ENC_UZERO, BITS>(u, sc, tile, d, q, words, resid, ef, seed, id, t, qtab, lo);
    else if (q.stochastic)
        encode_store_v<QK, FULL, BALLOT, tab ? ENC_USTO_TAB : ENC_USTO_DIV, BITS>(u, sc, tile, d, q, words, resid, ef,
                                                                               seed, id, t, qtab, lo);
    else
        encode_store_v<QK, FULL, BALLOT, tab ? ENC_UDET_TAB : ENC_UDET_DIV, BITS>(u, sc, tile, d, q, words, resid, ef,
                                                                               seed, id, t, qtab, lo);
}

// Encode and store a tile; the variant (and a configured code width) is chosen once per tile.
template <int QK, bool FULL, bool BALLOT, class USrc, class Scale>
__device__ __forceinline__ void encode_store(const USrc &u, Scale sc, int64_t tile, int64_t d,
                                             const QParams &q, uint32_t *words, float *resid, int ef,
                                             uint64_t seed, uint32_t id, uint32_t t, const float *qtab,
                                             int64_t lo = 0)
{
    if constexpr (QK == QK_UNIF) {
        switch (q.bits) {  // the widths ea_init accepts
        case 2: encode_store_unif<QK, FULL, BALLOT, 2>(u, sc, tile, d, q, words, resid, ef, seed, id, t, qtab, lo); break;
        case 4: encode_store_unif<QK, FULL, BALLOT, 4>(u, sc, tile, d, q, words, resid, ef, seed, id, t, qtab, lo); break;
        case 8: encode_store_unif<QK, FULL, BALLOT, 8>(u, sc, tile, d, q, words, resid, ef, seed, id, t, qtab, lo); break;
        default: encode_store_unif<QK, FULL, BALLOT, 16>(u, sc, tile, d, q, words, resid, ef, seed, id, t, qtab, lo); break;
        }
    } else if constexpr (QK == QK_POW2) {
        if (q.bits == 4)
            encode_store_v<QK, FULL, BALLOT, ENC_PLAIN, 4>(u, sc, tile, d, q, words, resid, ef, seed, id, t, qtab, lo);
        else
            encode_store_v<QK, FULL, BALLOT, ENC_PLAIN, 8>(u, sc, tile, d, q, words, resid, ef, seed, id, t, qtab, lo);
    } else {
        encode_store_v<QK, FULL, BALLOT, ENC_PLAIN, 0>(u, sc, tile, d, q, words, resid, ef, seed, id, t, qtab, lo);
    }
}

// The tile's end when the tile is one scale group (or Q has no scale) and u sits in shared memory
// (USmem layout); l1 / mx are this thread's partial sum / maximum of |u| over its valid coordinates.
template <int QK, bool FULL, bool BALLOT>
__device__ __forceinline__ void finish_tile_smem(const float4 *ubuf, DF l1, float mx, int64_t tile, int64_t d,
                                                 const QParams &q, uint32_t *words, float *scales, float *resid,
                                                 int ef, uint64_t seed, uint32_t id, uint32_t t, TileSmem &sm)
{
    float s = 0.0f;
    if constexpr (has_scale<QK>()) {
        const int64_t tile_lo = tile * kTile;
        const int64_t tile_hi = min(tile_lo + static_cast<int64_t>(kTile), d);
        if constexpr (QK == QK_SIGN)
            s = block_sign_scale(l1, tile_hi - tile_lo, sm.red256, &sm.bcastf);
        else
            s = block_max_all(mx, sm.redm);
        if (threadIdx.x == 0) scales[tile] = s;
    }
    encode_store<QK, FULL, BALLOT>(USmem{ubuf}, s, tile, d, q, words, resid, ef, seed, id, t,
                                   (QK == QK_UNIF && q.bits <= 8) ? sm.qtab : nullptr);
}

// PASS_LAZY on a tile that lies inside one scale group, as a compile-time refinement chosen per tile
// by the worker's kernel (the general form's group lookups cost registers: with Adam at the worker,
// a single form for both spilled 92 bytes a thread, and ResNet-18's messages took 5% longer).
constexpr int PASS_LAZY_ONE = 16;
constexpr int PASS_STASH_ONE = 17;  // likewise PASS_STASH, where the caller knows it
// PASS_STASH with a streaming hint on the stores of u (stash_is_kept).  The direct server (PASS = -1) stores
// so too: 62 segments, 60,000,001 x 1, Adam at the server, the round 871 us with that u kept, 800 us so.
constexpr int PASS_STASH_STREAM = 18;

// The tile's end for a quantizer with scale groups, u read through `src` (URegs or USmem).
//   PASS_FUSED: the tile is exactly one scale group (blocks of 4096): reduce, encode, store.
//   PASS_SHORT: the tile is several groups of whole chunks: the same with a scale per chunk.
//   PASS_STASH: store u in resid and one partial norm per (tile, group) for finalize/encode.
// BALLOT: pack 1-bit codes with __ballot_sync (worker kernels) or with shuffles (the server, whose
// tile loop is instruction-bound).
// PASS: PASS_FUSED, PASS_SHORT or PASS_STASH as a compile-time constant (the other path is then not compiled
// in), or -1 to follow `pass`.
// ref (PASS_STASH, PASS_LAZY): the tile's groups; sm.part, and sm.tg where they are several, are set
// by the caller.  src is then USmem, or u is in shared memory (only the one-group forms take URegs).
template <int QK, bool FULL = false, bool BALLOT = true, int PASS = -1, class USrc>
__device__ __forceinline__ void finish_tile(const USrc &src, int64_t tile, int64_t d, const QParams &q,
                                            uint32_t *words, float *scales, float *resid, int ef, int pass,
                                            uint64_t seed, uint32_t id, uint32_t t, double *partials,
                                            TileSmem &sm, const TileRef &ref)
{
    if constexpr (PASS >= 0) pass = PASS;
    if constexpr (!has_scale<QK>()) {
        encode_store<QK, FULL, BALLOT>(src, 0.0f, tile, d, q, words, resid, ef, seed, id, t, nullptr);
        return;
    } else {
        const int64_t tile_lo = tile * kTile;
        const int64_t tile_hi = min(tile_lo + static_cast<int64_t>(kTile), d);
        if (pass == PASS_FUSED) {
            float s;
            if constexpr (QK == QK_SIGN) {
                DF acc{0.0f, 0.0f};
#pragma unroll
                for (int k = 0; k < kSlots; ++k) {
                    float uk[4];
                    src.get(k, uk);
#pragma unroll
                    for (int i = 0; i < 4; ++i) df_accumulate(acc, fabsf(uk[i]));  // invalid u are 0
                }
                s = block_sign_scale(acc, tile_hi - tile_lo, sm.red256, &sm.bcastf);
            } else {
                float mx = 0.0f;
#pragma unroll
                for (int k = 0; k < kSlots; ++k) {
                    float uk[4];
                    src.get(k, uk);
#pragma unroll
                    for (int i = 0; i < 4; ++i) mx = fmaxf(mx, fabsf(uk[i]));
                }
                s = block_max_all(mx, sm.redm);
            }
            if (threadIdx.x == 0) scales[tile] = s;
            // sm.qtab was filled by build_qtab before the reduction's barrier
            encode_store<QK, FULL, BALLOT>(src, s, tile, d, q, words, resid, ef, seed, id, t,
                                           (QK == QK_UNIF && q.bits <= 8) ? sm.qtab : nullptr);
            return;
        }
        if (pass == PASS_SHORT) {
            chunk_scales<QK>(src, tile, d, chunk_shift(q.grp), scales, sm);
            encode_store<QK, FULL, BALLOT>(src, ChunkScales{sm.csc}, tile, d, q, words, resid, ef, seed, id, t,
                                           (QK == QK_UNIF && q.bits <= 8) ? sm.qtab : nullptr);
            return;
        }
        // PASS_STASH: u into resid for encode_kernel.  PASS_LAZY (scaled sign): u into resid, where
        // the residual is formed from it and the scale later (lazy_residual; without error feedback
        // the residual stays 0), and the codes now: the sign of u needs no scale.  PASS_LAZY_ONE forms
        // the norm on the way.
        constexpr bool lazy = PASS == PASS_LAZY || PASS == PASS_LAZY_ONE;
        constexpr bool one = PASS == PASS_LAZY_ONE || PASS == PASS_STASH_ONE;
        DF all{0.0f, 0.0f};
#pragma unroll
        for (int k = 0; k < kSlots; ++k) {
            const int64_t qs = slot_of(tile, k);
            float uk[4];
            src.get(k, uk);
            if constexpr (PASS == PASS_LAZY_ONE)
#pragma unroll
                for (int i = 0; i < 4; ++i) df_accumulate(all, fabsf(uk[i]));  // u beyond d is 0
            if constexpr (!lazy) {
                if (FULL || 4 * qs < d) {
                    if constexpr (PASS < 0 || PASS == PASS_STASH_STREAM) store4<FULL>(resid, qs, d, uk);
                    else store4_kept<FULL>(resid, qs, d, uk);
                }
            } else {
                if (ef && (FULL || 4 * qs < d)) store4<FULL>(resid, qs, d, uk);
            }
            if constexpr (lazy && QK == QK_SIGN) {
                uint32_t c[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    float dec;
                    const uint32_t code = encode1<QK>(uk[i], 0.0f, q, 0.0f, 0, 0.0f, dec);
                    c[i] = (FULL || 4 * qs + i < d) ? code : 0u;
                }
                store_codes4<FULL, BALLOT>(words, qs, 1, c, 0, d);
            }
        }
        if (one || ref.ng() == 1) {
            if constexpr (QK == QK_SIGN) {
                if constexpr (PASS != PASS_LAZY_ONE)
#pragma unroll
                    for (int k = 0; k < kSlots; ++k) {
                        float uk[4];
                        src.get(k, uk);
#pragma unroll
                        for (int i = 0; i < 4; ++i) df_accumulate(all, fabsf(uk[i]));
                    }
                const DF tot = block_sum_lane0(all, sm.red256);
                if (threadIdx.x == 0) partials[sm.part] = static_cast<double>(tot.hi) + static_cast<double>(tot.lo);
            } else {
                float mx = 0.0f;
#pragma unroll
                for (int k = 0; k < kSlots; ++k) {
                    float uk[4];
                    src.get(k, uk);
#pragma unroll
                    for (int i = 0; i < 4; ++i) mx = fmaxf(mx, fabsf(uk[i]));
                }
                mx = block_max_warp0(mx, sm.redm);
                if (threadIdx.x == 0) partials[sm.part] = static_cast<double>(mx);
            }
            return;
        }
        if constexpr (!one) {
            int turn = 0;
            group_partials<QK>(src, tile, tile_lo, tile_hi, d, q, ref, &sm.tg, partials, sm.parts, turn);
        }
    }
}

// PASS_LAZY (scaled sign): where the residual e = u - Q(u) of a kept u is formed -- u - (u >= 0 ? s
// : -s), s the scale of the coordinate's group in the previous message (scales).  This is
// e <- u - Q(u) of Algorithm 1 / Algorithm 2 with the same binary32 operations, evaluated where the
// residual is next read.  LazyScale holds a tile's scale when the tile lies in one group (loaded
// once, early), else the group to start the per-coordinate lookups from.
struct LazyScale {
    int64_t g1, hint;  // the tile's one group (-1: several), the tile's first group
    float s1;          // the scale of g1
};

__device__ __forceinline__ LazyScale lazy_scale_of_tile(const TileRef &ref, const float *scales)
{
    LazyScale ls;
    ls.g1 = ref.ng() == 1 ? ref.g0 : -1;
    ls.hint = ref.g0;
    ls.s1 = ls.g1 >= 0 ? scales[ls.g1] : 0.0f;
    return ls;
}

// The residual of the kept u of coordinates j0 .. j0+3 (in place in e); coordinates >= d unchanged.  tg:
// the tile's groups.
template <bool FULL>
__device__ __forceinline__ void lazy_residual4(const QParams &q, const float *scales, const LazyScale &ls,
                                               const TileGroups &tg, int64_t tile, int64_t j0, int64_t d, float (&e)[4])
{
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        if (FULL || j0 + i < d) {
            const float s = ls.g1 >= 0 ? ls.s1 : scales[tile_group_of(q.grp, tg, tile, j0 + i)];
            float dec;
            (void)encode1<QK_SIGN>(e[i], s, q, 0.0f, 0, 0.0f, dec);
            e[i] = __fsub_rn(e[i], dec);
        }
    }
}

// The same for all of this thread's slots of tile `tile`.  ONE: the tile lies inside one group.  buf: the
// threads' slots of shared memory, through which a tile of several groups goes one slot at a time.
template <bool FULL, bool ONE>
__device__ __forceinline__ void lazy_residual(const QParams &q, const float *scales, const LazyScale &ls,
                                              const TileGroups &tg, float4 *buf, int64_t tile, int64_t d,
                                              float (&e)[kSlots][4])
{
    if (ONE || ls.g1 >= 0) {  // one branch for the tile
#pragma unroll
        for (int k = 0; k < kSlots; ++k) {
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                float dec;
                (void)encode1<QK_SIGN>(e[k][i], ls.s1, q, 0.0f, 0, 0.0f, dec);
                if (FULL || 4 * slot_of(tile, k) + i < d) e[k][i] = __fsub_rn(e[k][i], dec);
            }
        }
        return;
    }
#pragma unroll
    for (int k = 0; k < kSlots; ++k) buf[k * kThreads + threadIdx.x] = to_f4(e[k]);
#pragma unroll 1
    for (int k = 0; k < kSlots; ++k) {
        float v[4];
        to_arr(buf[k * kThreads + threadIdx.x], v);
        lazy_residual4<FULL>(q, scales, ls, tg, tile, 4 * slot_of(tile, k), d, v);
        buf[k * kThreads + threadIdx.x] = to_f4(v);
    }
#pragma unroll
    for (int k = 0; k < kSlots; ++k) to_arr(buf[k * kThreads + threadIdx.x], e[k]);
}

}  // namespace ea
