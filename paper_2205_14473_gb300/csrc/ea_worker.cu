// ea_worker.cu -- worker compress (Algorithm 2), the two-pass scale kernels, and x <- x - Q_s(w).
#include "ea_grouped.cuh"

namespace ea {

// One tile of worker_kernel; FULL: the tile lies inside [0, d) (every tile but a ragged last one).
// Each slot's u goes to ubuf (only this thread reads it again), so that no register holds u across
// the scale's reduction and more CTAs fit on an SM.
// ref: the tile's groups (PASS_STASH, PASS_LAZY), looked up by the caller.
template <int MODE, int QK, bool FULL, int PASS>
__device__ __forceinline__ void worker_tile(const WorkerArgs &a, const WorkerBufs &p, int64_t tile, float4 *ubuf,
                                            TileSmem &sm, const TileRef &ref)
{
    const int64_t d = a.d;
    constexpr bool lazy = PASS == PASS_LAZY || PASS == PASS_LAZY_ONE;
    LazyScale ls{};
    if constexpr (lazy)
        if (a.lazy_in) {
            if constexpr (PASS == PASS_LAZY_ONE) ls.s1 = p.scales[ref.g0];
            else ls = lazy_scale_of_tile(ref, p.scales);
        }
    float g[kSlots][4], e[kSlots][4], m[kSlots][4], v[kSlots][4];
#pragma unroll
    for (int k = 0; k < kSlots; ++k) {
        const int64_t q = slot_of(tile, k);
        load4<FULL>(p.g, q, d, g[k]);
        load4<FULL>(p.e, q, d, e[k]);
        if (MODE == MODE_W) {
            load4<FULL>(p.m, q, d, m[k]);
            load4<FULL>(p.v, q, d, v[k]);
        }
    }
    // the grid's fl(i/L) table, built while the loads are in flight (read after the scale
    // reduction's barrier)
    build_qtab<QK>(a.q, sm.qtab);
    if constexpr (lazy) {
        // e holds the previous round's u: its residual is u - Q(u) with the previous scales
        if (a.lazy_in) lazy_residual<FULL, PASS == PASS_LAZY_ONE>(a.q, p.scales, ls, sm.tg, ubuf, tile, d, e);
    }
#pragma unroll
    for (int k = 0; k < kSlots; ++k) {
        const int64_t q = slot_of(tile, k);
        const int64_t j0 = 4 * q;
        float u[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            float step = g[k][i];
            if (MODE == MODE_W) step = adam_step(g[k][i], m[k][i], v[k][i], a.hp);
            u[i] = (FULL || j0 + i < d) ? __fadd_rn(step, e[k][i]) : 0.0f;
        }
        ubuf[k * kThreads + threadIdx.x] = make_float4(u[0], u[1], u[2], u[3]);
        if (MODE == MODE_W && (FULL || j0 < d)) {
            store4<FULL>(p.m, q, d, m[k]);
            store4<FULL>(p.v, q, d, v[k]);
        }
    }
    finish_tile<QK, FULL, true, PASS>(USmem{ubuf}, tile, d, a.q, p.words, p.scales, p.e, a.ef, a.pass, a.seed,
                                      a.id + blockIdx.y, a.t, p.partials, sm, ref);
}

// Algorithm 2 for one worker on one 4096-coordinate tile.  With Adam at the worker:
//   v <- beta2 v + (1-beta2) g^2, m <- beta1 m + (1-beta1) g, u = alpha m / sqrt(v) + e;
// with Adam at the server: u = g + e.  Then Q_w(u) and e <- u - Q_w(u) (finish_tile).
// HBM traffic per coordinate: 16 B read + 12 B written + b/8 B of code (Adam at the worker).
// Resident CTAs per SM the registers are sized for: four with Adam at the server (g and e per
// coordinate), three with Adam at the worker.  Measured: the server-side-Adam uniform grid runs
// faster at four CTAs with a few bytes of spill than at three without, and the worker-side-Adam
// uniform grid faster at three (80 registers, a few bytes of spill) than at two.
// One CTA per tile and worker (blockIdx.y), a worker's tiles next to each other: the workers of one
// launch leave no idle SMs between them, where a launch each drains the chip n times and a small
// vector fills a part of it.  Rounds with a launch per worker and with one for all: 500 coordinates,
// ten workers 83 and 20 us; ResNet-18, sixteen 981 and 820 us; 110,000,000, eight 4199 and 3995 us.
// PASS_LAZY for the scaled sign: the same tile, the codes stored with the partial norms and u kept
// in e (see lazy_residual); one launch per message plus finalize_kernel.
template <int MODE, class Workers>
__global__ void __launch_bounds__(kThreads, MODE == MODE_S ? 4 : 3)
    worker_lazy_kernel(const __grid_constant__ WorkerArgs a, const __grid_constant__ Workers ws)
{
    __shared__ TileSmem sm;
    __shared__ float4 ubuf[kSlots * kThreads];
    pdl_trigger();
    const WorkerBufs &p = ws.at(blockIdx.y);
    const CtaTile ct = cta_tile(a.q.grp, a.d);
    if (ct.tile < 0) return;
    if (threadIdx.x == 0) sm.part = ct.ref.part();
    if (ct.plain) {
        pdl_wait();
        worker_tile<MODE, QK_SIGN, true, PASS_LAZY_ONE>(a, p, plain_tile(), ubuf, sm, ct.ref);
        return;
    }
    if (ct.ref.ng() > 1) {
        cache_tile_groups(a.q.grp, ct.tile, a.d, sm.tg);
        __syncthreads();
    }
    pdl_wait();
    worker_tile<MODE, QK_SIGN, false, PASS_LAZY>(a, p, ct.tile, ubuf, sm, ct.ref);
}

template <int MODE, int QK, class Workers>
__global__ void __launch_bounds__(kThreads, MODE == MODE_S ? 4 : 3)
    worker_kernel(const __grid_constant__ WorkerArgs a, const __grid_constant__ Workers ws)
{
    __shared__ TileSmem sm;
    __shared__ float4 ubuf[kSlots * kThreads];
    pdl_trigger();
    const WorkerBufs &p = ws.at(blockIdx.y);
    const int64_t tile = plain_tile();  // the ragged one first, see cta_tile
    TileRef ref{};
    if (has_scale<QK>() && a.pass == PASS_STASH) {
        ref = tile_ref(a.q.grp, tile, a.d);
        if (threadIdx.x == 0) sm.part = ref.part();
        if (ref.ng() > 1) {
            cache_tile_groups(a.q.grp, tile, a.d, sm.tg);
            __syncthreads();
        }
    }
    pdl_wait();
    // the scale pass as a compile-time constant: each instantiation carries only its own path
    const bool full = (tile + 1) * kTile <= a.d;
    if (a.pass == PASS_FUSED) {
        if (full) worker_tile<MODE, QK, true, PASS_FUSED>(a, p, tile, ubuf, sm, ref);
        else worker_tile<MODE, QK, false, PASS_FUSED>(a, p, tile, ubuf, sm, ref);
    } else if (has_scale<QK>() && a.pass == PASS_SHORT) {
        if (full) worker_tile<MODE, QK, true, PASS_SHORT>(a, p, tile, ubuf, sm, ref);
        else worker_tile<MODE, QK, false, PASS_SHORT>(a, p, tile, ubuf, sm, ref);
    } else {
        if (full) worker_tile<MODE, QK, true, PASS_STASH>(a, p, tile, ubuf, sm, ref);
        else worker_tile<MODE, QK, false, PASS_STASH>(a, p, tile, ubuf, sm, ref);
    }
}

// PASS_STASH of the uniform grid with streaming stores of u (WorkerArgs::keep = 0).  A kernel of its own: as
// a path more in worker_kernel it made that one 2 to 5% longer for messages of 1 to 5 million coordinates.
template <int MODE>
__global__ void __launch_bounds__(kThreads, MODE == MODE_S ? 4 : 3)
    worker_stream_kernel(const __grid_constant__ WorkerArgs a, const __grid_constant__ WorkerOne ws)
{
    __shared__ TileSmem sm;
    __shared__ float4 ubuf[kSlots * kThreads];
    pdl_trigger();
    const WorkerBufs &p = ws.at(0);
    const int64_t tile = plain_tile();
    const TileRef ref = tile_ref(a.q.grp, tile, a.d);
    if (threadIdx.x == 0) sm.part = ref.part();
    if (ref.ng() > 1) {
        cache_tile_groups(a.q.grp, tile, a.d, sm.tg);
        __syncthreads();
    }
    pdl_wait();
    if ((tile + 1) * kTile <= a.d) worker_tile<MODE, QK_UNIF, true, PASS_STASH_STREAM>(a, p, tile, ubuf, sm, ref);
    else worker_tile<MODE, QK_UNIF, false, PASS_STASH_STREAM>(a, p, tile, ubuf, sm, ref);
}

// Phase one of a grouped worker tile: u of the coordinate range [lo, hi) of tile `tile` (0
// elsewhere) into ub, with m and v updated and stored in the range (Adam at the worker).
// FULL: the range is the whole tile.  All four slots' loads are issued at once (the kernel's
// register budget is sized for it), so that enough bytes are in flight per SM.
template <int MODE, bool FULL>
__device__ __forceinline__ void worker_u_range(const WorkerArgs &a, const WorkerBufs &p, int64_t tile, int64_t lo,
                                               int64_t hi, float4 *ub)
{
    constexpr int H = kSlots;
#pragma unroll
    for (int h = 0; h < kSlots; h += H) {
        float g[H][4], e[H][4], m[H][4], v[H][4];
        bool in[H];
#pragma unroll
        for (int k = 0; k < H; ++k) {
            const int64_t q = slot_of(tile, h + k);
            in[k] = FULL || (4 * q >= lo && 4 * q < hi);
#pragma unroll
            for (int i = 0; i < 4; ++i) g[k][i] = e[k][i] = m[k][i] = 0.0f, v[k][i] = 1.0f;
            if (in[k]) {
                load4<FULL>(p.g, q, hi, g[k]);
                load4<FULL>(p.e, q, hi, e[k]);
                if (MODE == MODE_W) {
                    load4<FULL>(p.m, q, hi, m[k]);
                    load4<FULL>(p.v, q, hi, v[k]);
                }
            }
        }
#pragma unroll
        for (int k = 0; k < H; ++k) {
            const int64_t q = slot_of(tile, h + k);
            const int64_t j0 = 4 * q;
            float u[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                float step = g[k][i];
                if (MODE == MODE_W) step = adam_step(g[k][i], m[k][i], v[k][i], a.hp);
                u[i] = (in[k] && (FULL || j0 + i < hi)) ? __fadd_rn(step, e[k][i]) : 0.0f;
            }
            ub[(h + k) * kThreads + threadIdx.x] = make_float4(u[0], u[1], u[2], u[3]);
            if (MODE == MODE_W && in[k]) {
                store4<FULL>(p.m, q, hi, m[k]);
                store4<FULL>(p.v, q, hi, v[k]);
            }
        }
    }
}

// Algorithm 2 for scale groups that span tiles, in one cooperative pass (PASS_GROUPED; see
// GroupPlan): for each wave, every CTA computes u of its tiles into shared memory (phase one) and
// publishes the partial norms; once a group's scale is ready, the tiles are encoded from shared
// memory and e <- u - Q_w(u) stored (phase two).  HBM traffic per coordinate as worker_kernel's:
// no second read of u.
template <int MODE, int QK>
__global__ void __launch_bounds__(kThreads, MODE == MODE_S ? 4 : 2) worker_grouped_kernel(const WorkerGroupedArgs ga)
{
    const WorkerArgs &a = ga.a;
    const WorkerBufs &p = ga.p;
    extern __shared__ __align__(16) float4 uslot[];  // a.gp.slots tiles of u
    __shared__ GroupSmem gs;
    build_qtab<QK>(a.q, gs.qtab);
    __syncthreads();
    const GroupPlan &gp = a.gp;
    int turn = 0;  // reductions so far (the same count in every thread)
    for (int w = 0; w < static_cast<int>(gp.n_waves); ++w) {
        const int64_t c0 = gp.cuts[w], c1 = gp.cuts[w + 1];
        const int t0 = static_cast<int>(c0 / kTile) + blockIdx.x;   // tiles < 2^28 (d <= 2^40)
        const int t_end = static_cast<int>((c1 - 1) / kTile) + 1;
        int k = 0;
        for (int tile = t0; tile < t_end; tile += gridDim.x, ++k) {
            float4 *ub = uslot + k * (kThreads * kSlots);
            const int64_t tl = static_cast<int64_t>(tile) * kTile, lo = max(c0, tl), hi = min(c1, tl + kTile);
            if (lo == tl && hi == tl + kTile) worker_u_range<MODE, true>(a, p, tile, lo, hi, ub);
            else worker_u_range<MODE, false>(a, p, tile, lo, hi, ub);
            group_partials<QK>(USmem{ub}, tile, lo, hi, a.d, a.q, tile_ref(a.q.grp, tile, a.d), nullptr, p.partials,
                               gs.parts, turn);
        }
        if (!wave_barrier(gp, w, a.status, gs)) return;
        encode_wave<QK>(uslot, t0, t_end, c0, c1, a.d, a.q, p.words, p.partials, p.scales, p.e, a.ef, a.seed, a.id, a.t, gs);
    }
}

// One CTA per scale group (blockIdx.x) and message (blockIdx.y): combine the group's per-tile
// partial norms in a fixed order and write the group scale (Example 1: ||.||_inf; scaled sign:
// ||.||_1 / |group|).
template <int QK>
__global__ void __launch_bounds__(kThreads) finalize_kernel(const FinalizeArgs a)
{
    __shared__ double red[kWarps];
    pdl_trigger();
    pdl_wait();
    const int64_t gi = blockIdx.x;
    const double *partials = a.partials + static_cast<int64_t>(blockIdx.y) * a.partials_stride;
    float *scales = a.scales + static_cast<int64_t>(blockIdx.y) * a.scales_stride;
    const int64_t pb = a.q.grp.pair_base[gi], pe = a.q.grp.pair_base[gi + 1];
    // eight loads in flight per thread: a whole vector's partials (7,325 at d = 30,000,000) are a chain of
    // L2 latencies otherwise (8.0 us, 7.0 us so).
    constexpr int U = 8;
    double acc = 0.0;
    for (int64_t p = pb + threadIdx.x; p < pe; p += U * kThreads) {
        double v[U];
#pragma unroll
        for (int i = 0; i < U; ++i) v[i] = p + i * kThreads < pe ? partials[p + i * kThreads] : 0.0;  // norms >= 0
#pragma unroll
        for (int i = 0; i < U; ++i) acc = (QK == QK_SIGN) ? __dadd_rn(acc, v[i]) : fmax(acc, v[i]);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const double w = __shfl_down_sync(0xffffffffu, acc, o);
        acc = (QK == QK_SIGN) ? __dadd_rn(acc, w) : fmax(acc, w);
    }
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = red[0];
        for (int w = 1; w < kWarps; ++w) t = (QK == QK_SIGN) ? __dadd_rn(t, red[w]) : fmax(t, red[w]);
        const int64_t len = group_end(a.q.grp, gi, a.d) - group_begin(a.q.grp, gi, a.d);
        scales[gi] = (QK == QK_SIGN) ? sign_scale(t, len) : static_cast<float>(t);
    }
}

// Second pass, one CTA per tile: encode the stashed input with its group's scale and leave the
// residual u - Q(u) in its place.  The first pass takes the tiles last first and this one first first, so
// that it begins with what was written last; u that was stored without a streaming hint (stash_is_kept) is
// in part still in L2 then, and what is overwritten there was never written to memory.  Whole-vector 8-bit
// grid, 30,000,000 x 4: the round 1042 us with both passes in one order, streaming hints and two CTAs per SM
// here, 903 us with opposite orders, no hint and four CTAs.
template <int QK, bool FULL>
__device__ __forceinline__ void encode_one_group(const EncodeArgs &a, float s, int64_t tile, const float *qtab)
{
    float u[kSlots][4];
#pragma unroll
    for (int k = 0; k < kSlots; ++k) load4<FULL>(a.buf, slot_of(tile, k), a.d, u[k]);
    encode_store<QK, FULL, true>(URegs{u}, s, tile, a.d, a.q, a.words, a.buf, a.ef, a.seed, a.id, a.t, qtab);
    if (!a.ef) {  // without error feedback the residual is 0: clear the stash of u
        const float z[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int k = 0; k < kSlots; ++k)
            if (FULL || 4 * slot_of(tile, k) < a.d) store4<FULL>(a.buf, slot_of(tile, k), a.d, z);
    }
}

template <int QK>
__global__ void __launch_bounds__(kThreads, 4) encode_kernel(const EncodeArgs a)
{
    __shared__ float qtab_s[256];
    __shared__ TileGroups tg;
    pdl_trigger();
    const float *qtab = build_qtab<QK>(a.q, qtab_s);
    const int64_t tile = blockIdx.x;
    const int64_t d = a.d;
    const Grouping &G = a.q.grp;
    const TileRef ref = tile_ref(G, tile, d);
    if (ref.ng() > 1) cache_tile_groups(G, tile, d, tg);
    __syncthreads();
    pdl_wait();
    // a tile inside one group (the common case) has one scale: the fused tile encode
    if (ref.ng() == 1) {
        const float s = a.scales[ref.g0];
        if ((tile + 1) * kTile <= d) encode_one_group<QK, true>(a, s, tile, qtab);
        else encode_one_group<QK, false>(a, s, tile, qtab);
        return;
    }
    const int L = (QK == QK_UNIF) ? unif_L(a.q.bits) : 0;
    const float Lf = static_cast<float>(L);
#pragma unroll 1
    for (int k = 0; k < kSlots; ++k) {
        const int64_t qs = slot_of(tile, k);
        const int64_t j0 = 4 * qs;
        float u[4];
        load4(a.buf, qs, d, u);
        float U[4] = {0.f, 0.f, 0.f, 0.f};
        if (QK == QK_UNIF && a.q.stochastic && j0 < d) uniforms4(a.seed, a.id, a.t, j0, U);
        uint32_t c[4];
        float e[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            float dec = 0.0f;
            c[i] = 0u;
            if (j0 + i < d) {
                const float s = a.scales[tile_group_of(G, tg, tile, j0 + i)];
                c[i] = encode1<QK>(u[i], s, a.q, Lf, L, U[i], dec, qtab);
            }
            e[i] = a.ef ? __fsub_rn(u[i], dec) : 0.0f;
        }
        store_codes4(a.words, qs, a.q.bits, c, 0, d);
        if (j0 < d) store4(a.buf, qs, d, e);
    }
}

// x <- x - dec(Q_s message) on one tile (Algorithm 1 and Algorithm 2); HBM traffic per coordinate:
// 4 B read + 4 B written + b/8 B of code.  BITS: the code width as a compile-time constant.  The
// loads of x and of the raw code words are issued first; the fl(i/L) table of the uniform grid
// (b <= 8) is built while they are in flight, and the codes are unpacked after its barrier.
// SCALES: where a coordinate's scale is.  AS_TILE: 4096-blocks, one per tile (then no group lookup is
// compiled in; that instantiation measured 4% faster than one carrying the lookup as well);
// AS_SLOT: power-of-two blocks of 128 and more, one per warp and slot, loaded with the slot;
// AS_ANY: a group lookup.
enum ApplyScales : int { AS_TILE, AS_SLOT, AS_ANY };
template <int QK, bool FULL, int BITS, int SCALES>
__device__ __forceinline__ void apply_tile(const ApplyArgs &a, int64_t tile, const TileRef &ref, const TileGroups &tg,
                                           float *qtab_s)
{
    const int64_t d = a.d;
    const Grouping &G = a.q.grp;
    constexpr int bits = BITS;
    const int L = (QK == QK_UNIF) ? unif_L(bits) : 0;
    const float Lf = static_cast<float>(L);
    float x[kSlots][4];
    float s_slot[kSlots];
    uint4 raw[kSlots];  // the slot's code bits: .x for b <= 8, .x .y for b = 16, all four for b = 32
#pragma unroll
    for (int k = 0; k < kSlots; ++k) {
        const int64_t q = slot_of(tile, k);
        load4<FULL>(a.x, q, d, x[k]);
        raw[k] = make_uint4(0u, 0u, 0u, 0u);
        if (FULL || 4 * q < d) {
            if constexpr (has_scale<QK>() && SCALES == AS_SLOT) s_slot[k] = a.scales[(4 * q) >> G.log2G];
            if constexpr (bits <= 8) {
                raw[k].x = a.words[(q * bits) >> 3];
            } else if constexpr (bits == 16) {
                const uint2 w = reinterpret_cast<const uint2 *>(a.words)[q];
                raw[k].x = w.x, raw[k].y = w.y;
            } else {
                raw[k] = reinterpret_cast<const uint4 *>(a.words)[q];
            }
        }
    }
    const float *qtab = nullptr;
    if constexpr (QK == QK_UNIF && bits <= 8) {
        qtab = build_qtab<QK>(a.q, qtab_s);
        __syncthreads();
    }
    // one scale for the whole tile: 4096-blocks, or a tile inside one group
    const int64_t g1 = (!has_scale<QK>() || SCALES == AS_SLOT) ? 0 : SCALES == AS_TILE ? tile : FULL || ref.ng() == 1 ? ref.g0 : -1;
    const bool tile_scale = SCALES != AS_ANY || FULL || g1 >= 0;
    const float s_tile = (has_scale<QK>() && SCALES != AS_SLOT && tile_scale) ? a.scales[g1] : 0.0f;
#pragma unroll
    for (int k = 0; k < kSlots; ++k) {
        const int64_t q = slot_of(tile, k);
        const int64_t j0 = 4 * q;
        if (!FULL && j0 >= d) continue;
        uint32_t c[4];
        if constexpr (bits <= 8) {
            const int sh = static_cast<int>((q * bits) & 7) * 4;
#pragma unroll
            for (int i = 0; i < 4; ++i) c[i] = (raw[k].x >> (sh + i * bits)) & ((1u << bits) - 1u);
        } else if constexpr (bits == 16) {
            c[0] = raw[k].x & 0xffffu, c[1] = raw[k].x >> 16, c[2] = raw[k].y & 0xffffu, c[3] = raw[k].y >> 16;
        } else {
            c[0] = raw[k].x, c[1] = raw[k].y, c[2] = raw[k].z, c[3] = raw[k].w;
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            if (FULL || j0 + i < d) {
                float s = SCALES == AS_SLOT ? s_slot[k] : s_tile;
                if (has_scale<QK>() && !tile_scale) s = a.scales[tile_group_of(G, tg, tile, j0 + i)];
                x[k][i] = __fsub_rn(x[k][i], decode1<QK>(c[i], s, a.q, Lf, L, qtab));
            }
        }
        store4<FULL>(a.x, q, d, x[k]);
    }
}

// AS_TILE and AS_SLOT take any whole tile, AS_ANY one inside one group; the rest is the general form.
template <int QK, int BITS>
__device__ __forceinline__ void apply_body(const ApplyArgs &a, const CtaTile &ct, const TileGroups &tg, float *qtab_s)
{
    if ((ct.tile + 1) * kTile <= a.d && a.q.grp.gkind == GK_BLOCK && a.q.grp.G == kTile)
        apply_tile<QK, true, BITS, AS_TILE>(a, plain_tile(), ct.ref, tg, qtab_s);
    else if (has_scale<QK>() && (ct.tile + 1) * kTile <= a.d && a.q.grp.gkind == GK_BLOCK && a.q.grp.log2G >= kLog2Chunk)
        apply_tile<QK, true, BITS, AS_SLOT>(a, plain_tile(), ct.ref, tg, qtab_s);
    else if (ct.plain)
        apply_tile<QK, true, BITS, AS_ANY>(a, plain_tile(), ct.ref, tg, qtab_s);
    else
        apply_tile<QK, false, BITS, AS_ANY>(a, ct.tile, ct.ref, tg, qtab_s);
}

// One CTA per 4096-tile; the code width is dispatched once per CTA.
template <int QK>
__global__ void __launch_bounds__(kThreads) apply_kernel(const ApplyArgs a)
{
    __shared__ float qtab_s[256];
    pdl_trigger();
    __shared__ TileGroups tg;
    const CtaTile ct = cta_tile(a.q.grp, a.d);
    if (ct.tile < 0) return;
    const bool per_slot = a.q.grp.gkind == GK_BLOCK && a.q.grp.log2G >= kLog2Chunk && (ct.tile + 1) * kTile <= a.d;
    if (has_scale<QK>() && !per_slot && ct.ref.ng() > 1) {
        cache_tile_groups(a.q.grp, ct.tile, a.d, tg);
        __syncthreads();
    }
    pdl_wait();
    if constexpr (QK == QK_UNIF) {
        switch (a.q.bits) {  // the widths ea_init accepts
        case 2: apply_body<QK, 2>(a, ct, tg, qtab_s); break;
        case 4: apply_body<QK, 4>(a, ct, tg, qtab_s); break;
        case 8: apply_body<QK, 8>(a, ct, tg, qtab_s); break;
        default: apply_body<QK, 16>(a, ct, tg, qtab_s); break;
        }
    } else if constexpr (QK == QK_POW2) {
        if (a.q.bits == 4) apply_body<QK, 4>(a, ct, tg, qtab_s);
        else apply_body<QK, 8>(a, ct, tg, qtab_s);
    } else {
        apply_body<QK, QK == QK_SIGN ? 1 : 32>(a, ct, tg, qtab_s);
    }
}

__global__ void fill_kernel(float *p, int64_t count, float value)
{
    for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < count;
         i += static_cast<int64_t>(gridDim.x) * blockDim.x)
        p[i] = value;
}

// ------------------------------------------------------------------------------- launchers

template <int MODE, class Workers>
static cudaError_t launch_worker_mode(const WorkerArgs &a, const Workers &w, int count, cudaStream_t s, bool overlap)
{
    const bool lazy = a.pass == PASS_LAZY;
    const dim3 grid(static_cast<unsigned>(a.n_tiles + (lazy ? a.q.grp.n_slow : 0)), static_cast<unsigned>(count)),
        block(kThreads);
    if (lazy && a.q.kind != QK_SIGN) return cudaErrorNotSupported;
    if (lazy) return launch_pdl(worker_lazy_kernel<MODE, Workers>, grid, block, 0, s, overlap, kCarveoutPercent, a, w);
    switch (a.q.kind) {
    case QK_SIGN: return launch_pdl(worker_kernel<MODE, QK_SIGN, Workers>, grid, block, 0, s, overlap, kCarveoutPercent, a, w);
    case QK_UNIF: return launch_pdl(worker_kernel<MODE, QK_UNIF, Workers>, grid, block, 0, s, overlap, kCarveoutPercent, a, w);
    case QK_POW2: return launch_pdl(worker_kernel<MODE, QK_POW2, Workers>, grid, block, 0, s, overlap, kCarveoutPercent, a, w);
    default: return launch_pdl(worker_kernel<MODE, QK_IDENT, Workers>, grid, block, 0, s, overlap, kCarveoutPercent, a, w);
    }
}

cudaError_t launch_worker(int mode, const WorkerArgs &a, const WorkerBufs *w, int count, cudaStream_t s, bool overlap)
{
    if (count == 1) {
        const WorkerOne one{w[0]};
        if (a.pass == PASS_STASH && a.q.kind == QK_UNIF && !a.keep) {
            const dim3 grid(static_cast<unsigned>(a.n_tiles)), block(kThreads);
            return mode == MODE_W
                       ? launch_pdl(worker_stream_kernel<MODE_W>, grid, block, 0, s, overlap, kCarveoutPercent, a, one)
                       : launch_pdl(worker_stream_kernel<MODE_S>, grid, block, 0, s, overlap, kCarveoutPercent, a, one);
        }
        return mode == MODE_W ? launch_worker_mode<MODE_W>(a, one, 1, s, overlap)
                              : launch_worker_mode<MODE_S>(a, one, 1, s, overlap);
    }
    if (count < 1 || count > kWorkerBatch) return cudaErrorInvalidValue;
    WorkerList list{};
    std::copy(w, w + count, list.w);
    return mode == MODE_W ? launch_worker_mode<MODE_W>(a, list, count, s, overlap)
                          : launch_worker_mode<MODE_S>(a, list, count, s, overlap);
}

// The grouped kernel exists for the uniform grid (a scaled-sign message takes PASS_LAZY).
cudaError_t worker_grouped_shape(int mode, int qk, GroupedShape *out)
{
    const int w = mode == MODE_W ? 2 : 4;  // the kernels' launch bounds
    if (qk != QK_UNIF) return cudaErrorNotSupported;
    return mode == MODE_W ? grouped_shape(worker_grouped_kernel<MODE_W, QK_UNIF>, w, out)
                          : grouped_shape(worker_grouped_kernel<MODE_S, QK_UNIF>, w, out);
}

cudaError_t launch_worker_grouped(int mode, const WorkerArgs &a, const WorkerBufs &p, int grid, cudaStream_t s)
{
    const int slots = a.gp.slots;
    if (a.q.kind != QK_UNIF) return cudaErrorNotSupported;
    return mode == MODE_W ? grouped_launch(worker_grouped_kernel<MODE_W, QK_UNIF>, WorkerGroupedArgs{a, p}, grid, slots, s)
                          : grouped_launch(worker_grouped_kernel<MODE_S, QK_UNIF>, WorkerGroupedArgs{a, p}, grid, slots, s);
}

cudaError_t launch_finalize(const FinalizeArgs &a, cudaStream_t s, bool overlap)
{
    const dim3 grid(static_cast<unsigned>(a.q.grp.n_groups), static_cast<unsigned>(a.n_msgs > 1 ? a.n_msgs : 1)),
        block(kThreads);
    if (a.q.kind == QK_SIGN) return launch_pdl(finalize_kernel<QK_SIGN>, grid, block, 0, s, overlap, kCarveoutPercent, a);
    return launch_pdl(finalize_kernel<QK_UNIF>, grid, block, 0, s, overlap, kCarveoutPercent, a);
}

cudaError_t launch_encode(const EncodeArgs &a, cudaStream_t s, bool overlap)
{
    const dim3 grid(static_cast<unsigned>(a.n_tiles)), block(kThreads);
    if (a.q.kind == QK_SIGN) return launch_pdl(encode_kernel<QK_SIGN>, grid, block, 0, s, overlap, kCarveoutPercent, a);
    return launch_pdl(encode_kernel<QK_UNIF>, grid, block, 0, s, overlap, kCarveoutPercent, a);
}

// The residual u - Q(u) of the u kept by PASS_LAZY, into a.out, one CTA per tile (a view of it).
__global__ void __launch_bounds__(kThreads) lazy_resid_kernel(const ResidArgs a)
{
    __shared__ TileGroups tg;
    __shared__ float4 buf[kSlots * kThreads];
    pdl_trigger();
    const int64_t tile = blockIdx.x;
    const TileRef ref = tile_ref(a.q.grp, tile, a.d);
    if (ref.ng() > 1) cache_tile_groups(a.q.grp, tile, a.d, tg);
    __syncthreads();
    pdl_wait();
    const bool full = (tile + 1) * kTile <= a.d;
    const LazyScale ls = lazy_scale_of_tile(ref, a.scales);
    float u[kSlots][4];
#pragma unroll
    for (int k = 0; k < kSlots; ++k) load4(a.u, slot_of(tile, k), a.d, u[k]);
    if (full) lazy_residual<true, false>(a.q, a.scales, ls, tg, buf, tile, a.d, u);
    else lazy_residual<false, false>(a.q, a.scales, ls, tg, buf, tile, a.d, u);
#pragma unroll
    for (int k = 0; k < kSlots; ++k)
        if (4 * slot_of(tile, k) < a.d) store4(a.out, slot_of(tile, k), a.d, u[k]);
}

cudaError_t launch_lazy_resid(const ResidArgs &a, cudaStream_t s, bool overlap)
{
    const dim3 grid(static_cast<unsigned>((a.d + kTile - 1) / kTile)), block(kThreads);
    if (a.q.kind != QK_SIGN) return cudaErrorNotSupported;
    return launch_pdl(lazy_resid_kernel, grid, block, 0, s, overlap, kCarveoutPercent, a);
}

cudaError_t launch_apply(const ApplyArgs &a, cudaStream_t s, bool overlap)
{
    const dim3 grid(static_cast<unsigned>((a.d + kTile - 1) / kTile + a.q.grp.n_slow)), block(kThreads);
    switch (a.q.kind) {
    case QK_SIGN: return launch_pdl(apply_kernel<QK_SIGN>, grid, block, 0, s, overlap, kCarveoutPercent, a);
    case QK_UNIF: return launch_pdl(apply_kernel<QK_UNIF>, grid, block, 0, s, overlap, kCarveoutPercent, a);
    case QK_POW2: return launch_pdl(apply_kernel<QK_POW2>, grid, block, 0, s, overlap, kCarveoutPercent, a);
    default: return launch_pdl(apply_kernel<QK_IDENT>, grid, block, 0, s, overlap, kCarveoutPercent, a);
    }
}

cudaError_t launch_fill(float *p, int64_t count, float value, cudaStream_t s)
{
    if (count <= 0) return cudaSuccess;
    const int64_t want = (count + 255) / 256;
    fill_kernel<<<static_cast<unsigned>(want < 152 * 64 ? want : 152 * 64), 256, 0, s>>>(p, count, value);
    return cudaGetLastError();
}

}  // namespace ea
