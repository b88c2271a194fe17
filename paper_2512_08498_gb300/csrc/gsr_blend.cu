// gsr_blend.cu -- per-pixel compositing (forward) and its adjoint (backward).
//
// One persistent launch per direction covers every (view, tile) of the batch:
// work comes from an atomic tile counter, so views of uneven size and tiles of
// uneven list length share one grid of (SMs x resident blocks).  A tile has
// 256 pixels; a warp takes one of its 8x8 pixel blocks and waits for no other
// warp.
//
// Culling: every record carries a conservative box outside which its
// binary32 alpha is certainly below 1/255 (see alpha_box in
// gsr_preprocess.cu) and a threshold of its exponent.  A forward warp walks only
// the entries that can touch its block, in list order, and records which 8x4
// halves composited each entry; the backward walks exactly those.  Skipped
// pairs would have been skipped by the 1/255 rule anyway, so every decision
// (blend, skip, stop, contributor count) is unchanged.
//
// Forward, front to back (binary32 decisions per the contract):
//   P2 = dx (qa dx + qb dy) + qc dy^2           (= log2 of the Gaussian)
//   skip if P2 > 0; alpha = min(0.99, sigma 2^P2); skip if alpha < 1/255;
//   T' = T (1 - alpha); stop (entry not blended) if T' < 1e-4;
//   C += c alpha T, D += z alpha T, T = T'.
// Backward, back to front from the saved T_final and contributor count:
//   T_k = T_{k+1} / (1 - alpha_k) and suffix sums S of the later terms give
//   dL/dalpha_k = sum_ch dC (c T_k - S_C / (1 - alpha_k))
//               + dD (z T_k - S_D / (1 - alpha_k)) + dA T_final / (1 - alpha_k),
//   evaluated as T_k (dC . c + dD z) - X / (1 - alpha_k) with the single
//   running scalar X = dC . S_C + dD S_D - dA T_final;
//   then the chain to (u, v, qa, qb, qc, sigma, colour, z), reduced over the
//   block's pixels through per-warp slot buffers and added to the per-record
//   gradient.
#include <type_traits>

#include "gsr_common.cuh"
#include "gsr_kernels.h"

namespace gsr {

constexpr int kTilePixels = 256;

// Largest value of the quadratic form P(x, y) = x (qa x + qb y) + qc y^2
// (negative definite) over the rectangle [x0, x1] x [y0, y1] of pixel
// offsets, up to rounding.  The unconstrained maximum is at the origin; when
// the origin lies outside, the maximum lies on a face that faces it, and
// along a face P is a parabola with its vertex at y = ky x (x = kx y), so two
// clamped candidates cover every case: each is a point of the rectangle, and
// together they include the maximiser.
__device__ __forceinline__ float rect_max_form(float x0, float x1, float y0, float y1, float qa, float qb, float qc,
                                               float kx, float ky)
{
    const float xe = fminf(fmaxf(0.0f, x0), x1);
    const float y1c = fminf(fmaxf(ky * xe, y0), y1);
    const float ye = fminf(fmaxf(0.0f, y0), y1);
    const float x2c = fminf(fmaxf(kx * ye, x0), x1);
    const float p1 = __fmaf_rn(xe, __fmaf_rn(qa, xe, __fmul_rn(qb, y1c)), __fmul_rn(__fmul_rn(qc, y1c), y1c));
    const float p2 = __fmaf_rn(x2c, __fmaf_rn(qa, x2c, __fmul_rn(qb, ye)), __fmul_rn(__fmul_rn(qc, ye), ye));
    return fmaxf(p1, p2);
}

// ---------------------------------------------------------------------------
// forward
// ---------------------------------------------------------------------------
// One warp renders one 8x8 pixel block of a tile, two horizontally adjacent
// pixels per lane, and nothing in it waits for another warp.  The tile's list
// is walked in chunks of 32 entries.  Per chunk: the records (64 bytes each)
// arrive by asynchronous copies issued one chunk ahead; each lane tests one
// entry against the block (alpha box, then the maximum of the exponent over the
// block); the survivors' walk values are written densely to shared memory; the
// walk evaluates each survivor at the lane's two pixels.
//
// Bound by instruction issue (about 90 % of the slots; DRAM idle).  Against one
// pixel per lane with the tile's eight 8x4 warps in step (a barrier per 256
// staged entries, 82 % of the slots): a record's loads, dy and the row's products
// serve two pixels, the barriers and the batch bookkeeping are gone, and a block
// stops fetching as soon as its own pixels have stopped; it walks more idle
// lanes (8x8 blocks composite 69 % of the walked lanes on the 1M-Gaussian
// six-camera rig, 8x4 blocks 77 %).  Rig 2.04 -> 1.63 ms, 30-view window (with
// pair counters) 9.8 -> 7.35 ms, 60-view road 29.1 -> 21.6 ms.  Packed pairs
// (fma.rn.f32x2 over the two pixels) take the issue slots of the two scalar
// operations on this part and need their operands twice: 1.69 ms on the rig.
constexpr int kFwdWarps = 4;            // warps per block (they share nothing)
constexpr int kFwdThreads = 32 * kFwdWarps;
constexpr int kChunk = 32;              // list entries per step: one per lane
constexpr int kBlk = 8;                 // the pixel block's side
constexpr int kBlocksPerTile = kTilePixels / (kBlk * kBlk);

// A surviving record as the walk reads it.
struct DenseRec {
    float4 q[3];   // {u, v, qa, qb}, {qc, sigma, r, g}, {b, z, -, -}
};

struct FwdSmem {
    float4 raw[2][kChunk][4];        // staged records, 16-byte pieces swizzled (see raw_piece)
    DenseRec dense[kChunk];          // the chunk's survivors
    uint8_t entry[kChunk];           // a survivor's position in the chunk
    uint2 own;                       // see next_block
    unsigned long long stat[3];      // the warp's walked entries, examined and composited pairs
};

// Piece q of lane l's record: lanes l and l + 2 would otherwise meet in a bank.
__device__ __forceinline__ int raw_piece(int l, int q) { return q ^ ((l >> 1) & 3); }

__device__ __forceinline__ void stage_record(float4* dst, const float4* src, int lane)
{
#pragma unroll
    for (int q = 0; q < 4; ++q)
        asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst + raw_piece(lane, q))), "l"(src + q)
                     : "memory");
}

// Whether a record can reach alpha >= 1/255 at a pixel centre of the block at
// (X0, Y0).  Two conservative tests: the record's alpha box against the
// block, then the maximum of the record's exponent over the block against
// its culling threshold (record slot 11).  The corner offsets are rounded
// exactly as the blend rounds each pixel's offset, so every pixel's rounded
// offset lies in the tested rectangle.
__device__ __forceinline__ bool block_hit(const float4& r0, float qc, float thr_cull, const float4& bb, float X0, float Y0)
{
    bool hit = bb.x <= X0 + (kBlk - 0.5f) && bb.y >= X0 + 0.5f && bb.z <= Y0 + (kBlk - 0.5f) && bb.w >= Y0 + 0.5f;
    if (hit && thr_cull > -3.0e38f) {
        const float kx = -r0.w / (2.0f * r0.z), ky = -r0.w / (2.0f * qc);
        const float x0 = __fsub_rn(__fadd_rn(X0, 0.5f), r0.x);
        const float x1 = __fsub_rn(__fadd_rn(X0, kBlk - 0.5f), r0.x);
        const float y0 = __fsub_rn(__fadd_rn(Y0, 0.5f), r0.y);
        const float y1 = __fsub_rn(__fadd_rn(Y0, kBlk - 0.5f), r0.y);
        hit = rect_max_form(x0, x1, y0, y1, r0.z, r0.w, qc, kx, ky) >= thr_cull;
    }
    return hit;
}

// One entry at a lane's two pixels (same row, so dy and its products are
// equal) up to alpha (independent of T).  2^P2 is the contract's exp2_nonpos
// bit for bit wherever a pixel can composite: the upper clamp (P2 <= 0) is
// left out because the entry is refused there anyway, and the final scaling by
// 2^n adds n to the exponent field, which differs from the product only below
// 2^-126, far under the 1/255 threshold.
struct FwdPair {
    float P0, P1;      // P2 at the two pixels
    float al0, al1;
    float r, g, b, z;  // colour, depth
};

__device__ __forceinline__ float exp2_walk(float P)
{
    const float y = fmaxf(P, -126.0f);
    const float j = __fadd_rn(y, 0x1.8p23f);
    const float f = __fsub_rn(y, __fsub_rn(j, 0x1.8p23f));
    return __int_as_float(__float_as_int(exp2_poly(f)) + (__float_as_int(j) << 23));
}

__device__ __forceinline__ FwdPair fwd_pair(const DenseRec& d, float px0, float px1, float py)
{
    FwdPair e;
    const float4 q0 = d.q[0], q1 = d.q[1];
    const float2 q2 = *reinterpret_cast<const float2*>(&d.q[2]);
    const float dx0 = __fsub_rn(px0, q0.x), dx1 = __fsub_rn(px1, q0.x), dy = __fsub_rn(py, q0.y);
    const float t = __fmul_rn(q0.w, dy), s = __fmul_rn(__fmul_rn(q1.x, dy), dy);
    e.P0 = __fmaf_rn(dx0, __fmaf_rn(q0.z, dx0, t), s);
    e.P1 = __fmaf_rn(dx1, __fmaf_rn(q0.z, dx1, t), s);
    e.al0 = fminf(GSR_ALPHA_MAX, __fmul_rn(q1.y, exp2_walk(e.P0)));
    e.al1 = fminf(GSR_ALPHA_MAX, __fmul_rn(q1.y, exp2_walk(e.P1)));
    e.r = q1.z; e.g = q1.w; e.b = q2.x; e.z = q2.y;
    return e;
}

// The next pixel block of a warp.  The warps of a block of threads share one
// tile's blocks (state: tile << 32 | next block), so the records a warp
// stages are mostly in L1 for the other three (the 65M-record road gathers from
// 4 GB: with independent warps its forward took 37 ms, 22 ms with the sharing).  A warp that finds the tile
// exhausted takes a new one from the global queue and installs it; if another
// warp installed one meanwhile, it renders its own tile alone.  No warp waits.
// (The first tile is installed for all: four warps that each took one left a
// small image's tiles to a quarter of the blocks, 93 us instead of 31 on
// 256 x 256 pixels.)
__device__ __forceinline__ uint2 next_block(unsigned long long* shared, uint2* own, unsigned int* work)
{
    const uint2 o = *own;   // a tile held alone: {tile, next block}
    if (o.y < kBlocksPerTile) {
        own->y = o.y + 1u;
        return o;
    }
    for (;;) {
        const unsigned long long old = *reinterpret_cast<volatile unsigned long long*>(shared);
        const unsigned int b = (unsigned int)old;
        if (b < kBlocksPerTile) {
            if (atomicCAS(shared, old, old + 1ull) == old) return make_uint2((unsigned int)(old >> 32), b);
            continue;
        }
        const unsigned int t = atomicAdd(work, 1u);
        if (atomicCAS(shared, old, ((unsigned long long)t << 32) | 1ull) != old) *own = make_uint2(t, 1u);
        return make_uint2(t, 0u);
    }
}

// First 32-bit word of a tile's composited-entry masks: kMaskWords words per
// chunk of 32 list positions, word 2 blk + h the entries that some pixel of
// the upper (h = 0) or lower 8x4 half of block blk composited.  A tile's
// chunks start at its range's first position / 32 plus the tile id (plus the
// tile count in the second list region), so no two tiles' words overlap:
// floor((x + n) / 32) - floor(x / 32) + 1 >= ceil(n / 32).
constexpr int kMaskWords = 2 * kBlocksPerTile;
__device__ __forceinline__ size_t mask_base(uint32_t first, uint32_t tile, uint32_t region2, int64_t n_tiles)
{
    return (size_t)kMaskWords * ((size_t)(first / kChunk) + tile + (first >= region2 ? (size_t)n_tiles : (size_t)0));
}

// COUNT: keep the per-pixel examined and composited counts (statistics only;
// a separate instantiation because the running counts lengthen the walk).
// 80 registers, six blocks per SM (at 72 the walk spills: 6 % slower).
template <int BX, bool COUNT>
__global__ void __launch_bounds__(kFwdThreads, 6)
blend_fwd_kernel(const __grid_constant__ Table Tb, BlendFwdArgs a)
{
    if (earlier_wait_timed_out(a.status)) return;
    constexpr int BY = kTilePixels / BX, BPR = BX / kBlk;   // blocks per tile row
    __shared__ __align__(128) FwdSmem s_warp[kFwdWarps];
    __shared__ unsigned long long s_queue;
    if (threadIdx.x == 0) s_queue = (unsigned long long)atomicAdd(a.work, 1u) << 32;   // the first tile
    const int lane = threadIdx.x & 31;
    FwdSmem& S = s_warp[threadIdx.x >> 5];
    if (lane == 0) {
        S.own = make_uint2(0u, kBlocksPerTile);
        S.stat[0] = S.stat[1] = S.stat[2] = 0ull;
    }
    __syncthreads();
    if (a.round == 2 && a.counters[kCntOpenTiles] == 0ull) return;
    bool prefix_all = false;   // the first round's lists are the full ones
    if (a.round == 1) {
        const int64_t n_vis = (int64_t)a.counters[kCntVisible];
        prefix_all = prefix_records(n_vis, a.prefix) == n_vis;
    }
    const uint32_t lt_mask = (1u << lane) - 1u;

    for (;;) {
        uint2 next = make_uint2(0u, 0u);
        if (lane == 0) next = next_block(&s_queue, &S.own, a.work);
        const unsigned int tile = __shfl_sync(0xffffffffu, next.x, 0), blk = __shfl_sync(0xffffffffu, next.y, 0);
        if ((int64_t)tile >= Tb.n_tiles) break;
        if (a.round == 2 && !((a.open_tiles[tile >> 5] >> (tile & 31u)) & 1u)) continue;
        const int view = find_view_of_tile(Tb, tile);
        const DevView& V = Tb.v[view];
        const int lt = (int)(tile - V.tile_base);
        const int bx0 = (lt % V.TX) * BX + (int)(blk % BPR) * kBlk, by0 = (lt / V.TX) * BY + (int)(blk / BPR) * kBlk;
        const int px = bx0 + 2 * (lane & 3), py = by0 + (lane >> 2);
        const uint2 rg = a.ranges[tile];
        const int n = (int)(rg.y - rg.x);
        const float fx = __fadd_rn((float)px, 0.5f), fy = __fadd_rn((float)py, 0.5f);
        const float fx1 = __fadd_rn(fx, 1.0f);
        float Cr0 = 0.0f, Cr1 = 0.0f, Cg0 = 0.0f, Cg1 = 0.0f, Cb0 = 0.0f, Cb1 = 0.0f, D0 = 0.0f, D1 = 0.0f;
        // transmittance, negated once the pixel has stopped (or if it lies
        // outside the image): a negative T passes no stop test, so nothing more
        // is composited
        float T0 = py < V.H && px < V.W ? 1.0f : -1.0f, T1 = py < V.H && px + 1 < V.W ? 1.0f : -1.0f;
        uint32_t last0 = 0, last1 = 0, exam0 = (uint32_t)n, exam1 = (uint32_t)n, nblend = 0;
        auto all_stopped = [&]() { return __all_sync(0xffffffffu, T0 < 0.0f && T1 < 0.0f); };
        // list positions up to the end of the chunk in which every pixel had
        // stopped (0: they did not)
        int satpos = 0;
        unsigned int walked = 0;
        uint2* words = a.wmask ? reinterpret_cast<uint2*>(a.wmask + mask_base(rg.x, tile, a.region2, Tb.n_tiles)) + blk
                               : nullptr;
        const uint32_t* vals = a.vals + rg.x;
        bool all = all_stopped();   // a block outside the image

        uint32_t kn = 0;   // record of this lane's entry of the next chunk
        if (lane < n) stage_record(S.raw[0][lane], a.rec + 4 * (size_t)vals[lane], lane);
        asm volatile("cp.async.commit_group;" ::: "memory");
        if (kChunk + lane < n) kn = vals[kChunk + lane];
        for (int c0 = 0; c0 < n && !all; c0 += kChunk) {
            const int s = (c0 / kChunk) & 1;
            if (c0 + kChunk + lane < n) stage_record(S.raw[s ^ 1][lane], a.rec + 4 * (size_t)kn, lane);
            asm volatile("cp.async.commit_group;" ::: "memory");
            if (c0 + 2 * kChunk + lane < n) kn = vals[c0 + 2 * kChunk + lane];
            asm volatile("cp.async.wait_group 1;" ::: "memory");
            // each lane reads the record it staged itself
            const float4* R = S.raw[s][lane];
            bool hit = false, indefinite = false;
            float4 r0, r1, r2;
            if (c0 + lane < n) {
                r0 = R[raw_piece(lane, 0)];
                r1 = R[raw_piece(lane, 1)];
                r2 = R[raw_piece(lane, 2)];
                hit = block_hit(r0, r1.x, r2.w, R[raw_piece(lane, 3)], (float)bx0, (float)by0);
                indefinite = hit && !(r2.w > -3.0e38f);
            }
            const uint32_t hits = __ballot_sync(0xffffffffu, hit);
            const int m = __popc(hits), rank = __popc(hits & lt_mask);
            if (hit) {
                DenseRec& d = S.dense[rank];
                float4* q = reinterpret_cast<float4*>(&d);
                q[0] = r0;
                q[1] = make_float4(r1.x, r1.y, r2.x, r2.y);
                q[2] = make_float4(r2.z, r1.z, 0.0f, 0.0f);
                S.entry[rank] = (uint8_t)lane;
            } else if ((m & 1) && lane == 31 - __clz(~hits)) {
                // an odd survivor count is padded with a record that composites
                // nowhere (sigma = 0); m is odd, so some lane is no hit
                float4* q = reinterpret_cast<float4*>(&S.dense[m]);
#pragma unroll
                for (int i = 0; i < 3; ++i) q[i] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            }
            __syncwarp();
            // Branch-free: after exact culling nearly every walked entry
            // composites somewhere in the block, so every lane evaluates it and
            // the decisions select the updates (a zero weight leaves C and D
            // bit-identical).  Entries are taken two at a time: the second's
            // alpha does not depend on T, so it overlaps the first's update.
            // Bit p of w0 / w1: the pixel composited the chunk's survivor p.
            uint32_t w0 = 0, w1 = 0, x0 = 0, x1 = 0, bit = 1u;
            const bool live0 = T0 > 0.0f, live1 = T1 > 0.0f;
            // TEST_P: whether P2 > 0 has to be tested.  A record with a culling
            // threshold has a negative definite form of condition below 1e5,
            // whose binary32 value is within 8 2^-24 cond < 5 % of the exact one
            // and so never positive.
            auto step = [&](const FwdPair& e, uint32_t b, auto TEST_P) {
                const float n0 = __fmul_rn(T0, __fsub_rn(1.0f, e.al0)), n1 = __fmul_rn(T1, __fsub_rn(1.0f, e.al1));
                const bool pass0 = (!TEST_P.value || e.P0 <= 0.0f) && e.al0 >= GSR_ALPHA_MIN;
                const bool pass1 = (!TEST_P.value || e.P1 <= 0.0f) && e.al1 >= GSR_ALPHA_MIN;
                const bool bl0 = pass0 && n0 >= GSR_T_STOP, bl1 = pass1 && n1 >= GSR_T_STOP;
                const float g0 = bl0 ? e.al0 * T0 : 0.0f, g1 = bl1 ? e.al1 * T1 : 0.0f;
                Cr0 = fmaf(e.r, g0, Cr0); Cr1 = fmaf(e.r, g1, Cr1);
                Cg0 = fmaf(e.g, g0, Cg0); Cg1 = fmaf(e.g, g1, Cg1);
                Cb0 = fmaf(e.b, g0, Cb0); Cb1 = fmaf(e.b, g1, Cb1);
                D0 = fmaf(e.z, g0, D0); D1 = fmaf(e.z, g1, D1);
                if constexpr (COUNT) {
                    if (pass0 && !bl0) x0 |= b;
                    if (pass1 && !bl1) x1 |= b;
                }
                if (pass0) T0 = bl0 ? n0 : -fabsf(T0);
                if (pass1) T1 = bl1 ? n1 : -fabsf(T1);
                if (bl0) w0 |= b;
                if (bl1) w1 |= b;
            };
            int i = 0;
            auto walk = [&](auto TEST_P) {
                while (i < m && !all) {
                    // the warp vote that ends the walk once every pixel has
                    // stopped is taken after every fourth pair (a stopped pixel
                    // passes nothing, so the extra entries change no result)
                    const int e = min(i + 8, m);
                    for (; i < e; i += 2) {
                        const FwdPair e0 = fwd_pair(S.dense[i], fx, fx1, fy);
                        const FwdPair e1 = fwd_pair(S.dense[i + 1], fx, fx1, fy);
                        step(e0, bit, TEST_P);
                        step(e1, bit << 1, TEST_P);
                        bit <<= 2;
                    }
                    all = all_stopped();
                }
            };
            if (__any_sync(0xffffffffu, indefinite)) walk(std::true_type{});
            else walk(std::false_type{});
            walked += (unsigned)min(i, m);
            // a pixel's last composited entry is the highest set bit; one OR
            // over each half of the warp says which survivors some pixel of its
            // 8x4 half composited, spread back to the chunk's positions
            if (w0) last0 = (uint32_t)(c0 + S.entry[31 - __clz(w0)] + 1);
            if (w1) last1 = (uint32_t)(c0 + S.entry[31 - __clz(w1)] + 1);
            if constexpr (COUNT) {
                // the lowest bit of x0 / x1: the entry that stopped the pixel
                if (live0 && x0) exam0 = (uint32_t)(c0 + S.entry[__ffs(x0) - 1] + 1);
                if (live1 && x1) exam1 = (uint32_t)(c0 + S.entry[__ffs(x1) - 1] + 1);
                nblend += __popc(w0) + __popc(w1);
            }
            if (words) {
                const uint32_t own = w0 | w1;
                const uint32_t up = __reduce_or_sync(0xffffffffu, lane < 16 ? own : 0u);
                const uint32_t lo = __reduce_or_sync(0xffffffffu, lane < 16 ? 0u : own);
                const uint32_t mu = __ballot_sync(0xffffffffu, hit && ((up >> rank) & 1u));
                const uint32_t ml = __ballot_sync(0xffffffffu, hit && ((lo >> rank) & 1u));
                if (lane == 0) words[(size_t)(c0 / kChunk) * kBlocksPerTile] = make_uint2(mu, ml);
            }
            __syncwarp();   // the dense records are rewritten by the next chunk
            if (all) satpos = min(c0 + kChunk, n);
        }
        // no copy is left in flight into the buffers the next block stages
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        // A first round's tile is final when its pixels all stopped within
        // the prefix lists (or those were the full lists); otherwise the
        // second round renders it again over its full list.
        const bool saturated = all;
        const bool final_block = a.round != 1 || saturated || prefix_all;
        if (lane == 0) {
            if (!final_block) {
                const size_t item = (size_t)tile * kBlocksPerTile + blk;
                atomicOr(a.open_blocks + (item >> 5), 1u << (item & 31u));
                const uint32_t bit = 1u << (tile & 31u);
                if (!(atomicOr(a.open_tiles + (tile >> 5), bit) & bit)) atomicAdd(a.counters + kCntOpenTiles, 1ull);
            }
            if (a.hist) {
                // the tile's last block records the share of the depth-ordered
                // records the tile needed before every pixel stopped, weighted
                // by its (estimated full) list length
                uint2* need = a.tile_need + tile;   // {largest satpos, blocks that finished}
                const uint32_t never = 0xffffffffu;
                atomicMax(&need->x, saturated ? (uint32_t)satpos : never);
                __threadfence();
                if (atomicAdd(&need->y, 1u) == kBlocksPerTile - 1) {
                    const uint32_t most = atomicMax(&need->x, 0u);
                    const unsigned long long n_vis = a.counters[kCntVisible];
                    int bucket = kSatBuckets;
                    if (most != never && most > 0u && n_vis > 0ull) {
                        const uint32_t k = vals[most - 1];
                        bucket = sat_bucket((float)(a.depthpos[k] + 1u) / (float)n_vis);
                    }
                    unsigned long long len = (unsigned long long)n;
                    if (a.round == 1) {
                        const unsigned long long n_pre = (unsigned long long)prefix_records((int64_t)n_vis, a.prefix);
                        if (n_pre > 0ull) len = len * n_vis / n_pre;
                    }
                    const bool open = a.round == 1 && most == never && !prefix_all;
                    if (len && !open) atomicAdd(a.hist + bucket, len);
                    *need = make_uint2(0u, 0u);   // for a second round
                }
            }
        }
        if (!final_block) continue;
        // statistics are taken by the round that finishes the block
        const size_t item = (size_t)tile * kBlocksPerTile + blk;
        if (a.round != 2 || ((a.open_blocks[item >> 5] >> (item & 31u)) & 1u)) {
            if (lane == 0) S.stat[0] += walked;
            if constexpr (COUNT) {
                unsigned long long exam = 0;
                if (py < V.H && px < V.W) exam += exam0;
                if (py < V.H && px + 1 < V.W) exam += exam1;
                exam = warp_sum(exam);
                nblend = __reduce_add_sync(0xffffffffu, nblend);
                if (lane == 0) {
                    S.stat[1] += exam;
                    S.stat[2] += nblend;
                }
            }
        }
        if (py < V.H) {
            const int64_t hw = (int64_t)V.W * V.H;
            const int64_t off = (int64_t)py * V.W + px;
            const int64_t pix = V.pix_base + off;
            float* rgb = a.rgb + 3 * V.pix_base;
            auto put = [&](int64_t o, float T, float C0, float C1, float C2, float Dz, uint32_t last) {
                rgb[off + o] = C0 + T * Tb.bg[0];
                rgb[hw + off + o] = C1 + T * Tb.bg[1];
                rgb[2 * hw + off + o] = C2 + T * Tb.bg[2];
                a.depth[pix + o] = Dz;
                a.alpha[pix + o] = 1.0f - T;
                a.tfinal[pix + o] = T;
                a.ncontrib[pix + o] = last;
            };
            if (px < V.W) put(0, fabsf(T0), Cr0, Cg0, Cb0, D0, last0);
            if (px + 1 < V.W) put(1, fabsf(T1), Cr1, Cg1, Cb1, D1, last1);
        }
    }
    if (lane == 0) {
        if (S.stat[0]) atomicAdd(a.counters + kCntWarpFwd, 2ull * S.stat[0]);   // in units of 32 pixels
        if (S.stat[1]) atomicAdd(a.counters + kCntFwdPairs, S.stat[1]);
        if (S.stat[2]) atomicAdd(a.counters + kCntBlended, S.stat[2]);
    }
}

// ---------------------------------------------------------------------------
// backward
// ---------------------------------------------------------------------------
// One warp takes one 8x8 pixel block, two horizontally adjacent pixels per
// lane as in the forward, and nothing in it waits for another warp.  The
// block's composited entries come from the forward's mask words, 32 list
// positions at a time from the back; their records (48 bytes) are staged
// densely, last entry first, by asynchronous copies issued one chunk ahead, and
// walked in groups of kSlots.
//
// Reduction over the block's 64 pixels, transposed.  For each walked entry
// every lane stores, for its two pixels, gP = dL/dP2 and w = alpha T (both zero
// where the pixel does not composite the entry), and per group four lanes sum
// one entry over two pixel rows each.  The record gradient needs
//   sum gP dx, sum gP dy, sum gP dx^2, sum gP dx dy, sum gP dy^2,
//   sum gP / sigma (= sum dL/dalpha G where alpha is not clamped),
//   sum w dD, sum w dC (three channels),
// with dx = px - u the same for every pixel up to the pixel's offset inside
// the block: dx = xo - ux, xo = x - 3.5, ux = u minus the block centre (same
// for y).  So a lane keeps the six moments M = sum gP {1, xo, yo, xo^2, xo yo,
// yo^2} (constant weights) and shifts them once per entry:
//   sum gP dx = Mx - ux M0, sum gP dx^2 = Mxx - 2 ux Mx + ux^2 M0,
//   sum gP dx dy = Mxy - ux My - uy Mx + ux uy M0 (and y alike).
// The shifted form has the rounding error of the direct sums (bounded by
// the sums of |gP| dx^2 both ways).  Two shuffle steps add the four lanes, and
// they add the record's ten sums to memory in binary64: a record's blocks
// each add once (the tile's eight warps used to be summed in shared memory
// first), and in binary32 the longer chain of additions showed in the
// gradients of Gaussians that cover many tiles (1.6 times the error).
//
// Bound by instruction issue (81 % of the slots) with the shared-memory pipe close
// behind (71 %: slot stores and the reduction's reads).  Against the tile's eight
// 8x4 warps in step (batches of 128 records with two barriers each, sums of a
// record over the warps in shared memory): a record's loads and row products serve
// two pixels, one test covers the alpha thresholds and the clamp, and the record
// sums, their flush and the barriers are gone.  1M-Gaussian six-camera rig 2.62 ->
// 2.09 ms, 30-view window 11.5 -> 8.7, 60-view road 36.8 -> 28.1.  Summing w dC over
// a lane's pixels in the walk instead of storing w (no reads of dC in the
// reduction): 2.13 ms on the rig; binary32 additions to memory: 2.02 ms.
// Keeping a non-finite upstream gradient to its pixel (S.odd) costs 0.04 ms there.
// Where a batch's blocks do not fill the chip or a few lists are very long, the
// walk of twice the pixels per warp is the longer chain: 0.066 -> 0.105 ms on 20k
// Gaussians at 640 x 384 (the forward 0.061 -> 0.087).
constexpr int kSlots = 8;
constexpr int kLeft = kSlots;                  // dense positions kept for the entries left over from a chunk
constexpr int kDense = kLeft + kChunk;

struct BwdSmem {
    // row e: the group's entry e; 16-byte piece c of a row (pixels 4c .. 4c + 3
    // in row-major order) is stored at piece c ^ e, so that the reads of the same
    // piece of eight rows land in eight different bank groups
    float4 gp[kSlots][16], wg[kSlots][16];
    float4 dcd[4][17];                         // (dC, dD) of the pixels, 16 per quarter and one of padding
    // {u, v, qa, qb}, {qc, sigma, z, record}, {r, g, b, culling threshold}
    float4 dense[2][kDense][3];
    uint2 own;                                 // see next_block
    unsigned odd;                              // lanes with an upstream gradient that is not finite
    unsigned long long stat[2];                // contributor counts, composited (8x4 block, entry) pairs
};

__device__ __forceinline__ float rcp_approx(float x)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

__device__ __forceinline__ float ex2_approx(float x)
{
    float r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// Sums over the row of eight pixels g: {1, xo, xo^2}, by the symmetry of xo.
__device__ __forceinline__ void row_moments(const float4& a, const float4& b, float& r, float& x1, float& x2)
{
    const float s0 = a.w + b.x, s1 = a.z + b.y, s2 = a.y + b.z, s3 = a.x + b.w;
    const float d0 = b.x - a.w, d1 = b.y - a.z, d2 = b.z - a.y, d3 = b.w - a.x;
    r = (s0 + s1) + (s2 + s3);
    x1 = fmaf(3.5f, d3, fmaf(2.5f, d2, fmaf(1.5f, d1, 0.5f * d0)));
    x2 = fmaf(12.25f, s3, fmaf(6.25f, s2, fmaf(2.25f, s1, 0.25f * s0)));
}

// Adds the group's n entries (dense records D) to the records' gradients.
// Zero weights are left out of the sums where some pixel's upstream gradient is
// not finite (S.odd).
template <bool DEPTH>
__device__ __forceinline__ void reduce_group(const BwdSmem& S, const float4 (*D)[3], int n, int lane, float cx, float cy,
                                             double* __restrict__ grad_rec, int64_t cap)
{
    const int e = lane & (kSlots - 1), q = lane >> 3;     // entry, pixel rows 2q and 2q + 1
    float ra, xa, xxa, rb, xb, xxb;
    row_moments(S.gp[e][(4 * q) ^ e], S.gp[e][(4 * q + 1) ^ e], ra, xa, xxa);
    row_moments(S.gp[e][(4 * q + 2) ^ e], S.gp[e][(4 * q + 3) ^ e], rb, xb, xxb);
    const float ya = 2.0f * (float)q - 3.5f, yb = ya + 1.0f;
    const float m0 = ra + rb, mx = xa + xb, mxx = xxa + xxb;
    const float my = fmaf(ya, ra, yb * rb), mxy = fmaf(ya, xa, yb * xb), myy = fmaf(ya * ya, ra, (yb * yb) * rb);
    float sd = 0.0f, s0 = 0.0f, s1 = 0.0f, s2 = 0.0f;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        const float4 t = S.wg[e][(4 * q + c) ^ e];
        const float w4[4] = {t.x, t.y, t.z, t.w};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float4 d = S.dcd[q][4 * c + j];
            s0 = fmaf(w4[j], d.x, s0);
            s1 = fmaf(w4[j], d.y, s1);
            s2 = fmaf(w4[j], d.z, s2);
            if constexpr (DEPTH) sd = fmaf(w4[j], d.w, sd);
        }
    }
    if (S.odd != 0u) {
        sd = s0 = s1 = s2 = 0.0f;
#pragma unroll 1
        for (int i = 0; i < 16; ++i) {
            const float4 t = S.wg[e][(4 * q + (i >> 2)) ^ e], d = S.dcd[q][i];
            const float w = (i & 2) ? ((i & 1) ? t.w : t.z) : ((i & 1) ? t.y : t.x);
            if (w == 0.0f) continue;
            s0 = fmaf(w, d.x, s0);
            s1 = fmaf(w, d.y, s1);
            s2 = fmaf(w, d.z, s2);
            if constexpr (DEPTH) sd = fmaf(w, d.w, sd);
        }
    }
    const float4 q0 = D[e][0], q1 = D[e][1];
    const float ux = q0.x - cx, uy = q0.y - cy;
    const float sx = fmaf(-ux, m0, mx), sy = fmaf(-uy, m0, my);
    const float sxx = fmaf(ux * ux, m0, fmaf(-2.0f * ux, mx, mxx));
    const float sxy = fmaf(ux * uy, m0, fmaf(-ux, my, fmaf(-uy, mx, mxy)));
    const float syy = fmaf(uy * uy, m0, fmaf(-2.0f * uy, my, myy));
    // lanes with bit 3 clear end with {sx, sy, sxx, sxy}, the others with
    // {syy, m0, sd, s0, s1, s2}
    const bool hi = lane & 8;
    const float a[4] = {sx, sy, sxx, sxy}, b[6] = {syy, m0, sd, s0, s1, s2};
    float v[6];
#pragma unroll
    for (int i = 0; i < 4; ++i) v[i] = (hi ? b[i] : a[i]) + __shfl_xor_sync(0xffffffffu, hi ? a[i] : b[i], 8);
#pragma unroll
    for (int i = 4; i < 6; ++i) v[i] = b[i] + __shfl_xor_sync(0xffffffffu, b[i], 8);
#pragma unroll
    for (int i = 0; i < 6; ++i) v[i] += __shfl_xor_sync(0xffffffffu, v[i], 16);
    // the record's coefficients, ln2 and the sign of the mean gradient; the
    // sum of dL/dalpha G over the pixels where alpha is not clamped = sum gP / sigma
    const bool last = lane & 16;
    float o0, o1, o2 = 0.0f;
    if (!hi) {
        o0 = last ? GSR_LN2 * v[2] : -GSR_LN2 * (2.0f * q0.z * v[0] + q0.w * v[1]);
        o1 = last ? GSR_LN2 * v[3] : -GSR_LN2 * (q0.w * v[0] + 2.0f * q1.x * v[1]);
    } else {
        o0 = last ? v[3] : GSR_LN2 * v[0];
        o1 = last ? v[4] : __fdividef(v[1], q1.y);
        o2 = last ? v[5] : v[2];
    }
    if (e < n) {
        const size_t k = __float_as_uint(q1.w);
        double* p = grad_rec + 8 * k + (hi ? 2 : 0) + (last ? 1 : 0);
        atomicAdd(p, (double)o0);
        atomicAdd(p + 4, (double)o1);
        if (hi && (DEPTH || last)) atomicAdd(grad_rec + 8 * (size_t)cap + 2 * k + (last ? 1 : 0), (double)o2);
    }
}

// DEPTH: an upstream depth gradient is given (else its terms are zero).
template <int BX, bool DEPTH>
__global__ void __launch_bounds__(kFwdThreads, 6)
blend_bwd_kernel(const __grid_constant__ Table Tb, BlendBwdArgs a)
{
    if (earlier_wait_timed_out(a.status)) return;
    constexpr int BY = kTilePixels / BX, BPR = BX / kBlk;   // blocks per tile row
    __shared__ __align__(128) BwdSmem s_warp[kFwdWarps];
    __shared__ unsigned long long s_queue;
    if (threadIdx.x == 0) s_queue = (unsigned long long)atomicAdd(a.work, 1u) << 32;   // the first tile
    const int lane = threadIdx.x & 31;
    BwdSmem& S = s_warp[threadIdx.x >> 5];
    if (lane == 0) {
        S.own = make_uint2(0u, kBlocksPerTile);
        S.stat[0] = S.stat[1] = 0ull;
    }
    __syncthreads();
    // this lane's two pixels in a slot row: piece (lane >> 1) ^ e, half lane & 1
    float2* const gp = reinterpret_cast<float2*>(S.gp) + (lane & 1);
    float2* const wg = reinterpret_cast<float2*>(S.wg) + (lane & 1);

    for (;;) {
        uint2 next = make_uint2(0u, 0u);
        if (lane == 0) next = next_block(&s_queue, &S.own, a.work);
        const unsigned int tile = __shfl_sync(0xffffffffu, next.x, 0), blk = __shfl_sync(0xffffffffu, next.y, 0);
        if ((int64_t)tile >= Tb.n_tiles) break;
        const int view = find_view_of_tile(Tb, tile);
        const DevView& V = Tb.v[view];
        const int lt = (int)(tile - V.tile_base);
        const int bx0 = (lt % V.TX) * BX + (int)(blk % BPR) * kBlk, by0 = (lt / V.TX) * BY + (int)(blk / BPR) * kBlk;
        const uint2 rg = a.ranges[tile];
        const float fx = __fadd_rn((float)(bx0 + 2 * (lane & 3)), 0.5f), fy = __fadd_rn((float)(by0 + (lane >> 2)), 0.5f);
        const float fx1 = __fadd_rn(fx, 1.0f);
        float T[2] = {1.0f, 1.0f}, X[2] = {0.0f, 0.0f};
        float4 dc[2] = {make_float4(0.0f, 0.0f, 0.0f, 0.0f), make_float4(0.0f, 0.0f, 0.0f, 0.0f)};   // dC, dD
        int lst[2] = {0, 0};
        {
            const int px = bx0 + 2 * (lane & 3), py = by0 + (lane >> 2);
            const int64_t hw = (int64_t)V.W * V.H;
            const int64_t off = (int64_t)py * V.W + px;
            const int64_t pix = V.pix_base + off;
            const float* g = a.dl_rgb + 3 * V.pix_base;
#pragma unroll
            for (int p = 0; p < 2; ++p) {
                if (py >= V.H || px + p >= V.W) continue;
                T[p] = a.tfinal[pix + p];
                lst[p] = (int)a.ncontrib[pix + p];
                dc[p].x = g[off + p]; dc[p].y = g[hw + off + p]; dc[p].z = g[2 * hw + off + p];
                if constexpr (DEPTH) dc[p].w = a.dl_depth[pix + p];
                const float dA = a.dl_alpha ? a.dl_alpha[pix + p] : 0.0f;
                // X = dC . S_C + dD S_D - dA T_final, S the suffix sums of the
                // later colour and depth terms (S_C starts at T_final bg): then
                // dL/dalpha_k = T_k (dC . c_k + dD z_k) - X / (1 - alpha_k)
                X[p] = T[p] * (dc[p].x * Tb.bg[0] + dc[p].y * Tb.bg[1] + dc[p].z * Tb.bg[2] - dA);
            }
        }
        const int warp_last = (int)__reduce_max_sync(0xffffffffu, (unsigned)max(lst[0], lst[1]));
        if (warp_last == 0) continue;
        // A pixel whose upstream gradient is not finite spoils the gradients of
        // the entries that it composites and no others of the block: such a
        // block takes the exact path, which selects instead of multiplying by
        // zero.
        const unsigned odd = __ballot_sync(0xffffffffu, !(fabsf(X[0]) + fabsf(X[1]) <= 3.0e38f) ||
                                                     !(fabsf(dc[0].x) + fabsf(dc[0].y) + fabsf(dc[0].z) + fabsf(dc[0].w) <= 3.0e38f) ||
                                                     !(fabsf(dc[1].x) + fabsf(dc[1].y) + fabsf(dc[1].z) + fabsf(dc[1].w) <= 3.0e38f));
        if (lane == 0) S.odd = odd;
        S.dcd[lane >> 3][2 * (lane & 7)] = dc[0];
        S.dcd[lane >> 3][2 * (lane & 7) + 1] = dc[1];
        {
            const unsigned long long c = warp_sum((unsigned long long)lst[0] + (unsigned long long)lst[1]);
            if (lane == 0) S.stat[0] += c;
        }
        const float cx = (float)(bx0 + kBlk / 2), cy = (float)(by0 + kBlk / 2);
        const uint2* words = reinterpret_cast<const uint2*>(a.wmask + mask_base(rg.x, tile, a.region2, Tb.n_tiles)) + blk;
        const uint32_t* vals = a.vals + rg.x;
        const int n = (int)(rg.y - rg.x);

        // stage the composited entries of a chunk behind the left-over places
        auto stage = [&](float4 (*dst)[3], uint32_t m, uint32_t k) {
            if ((m >> lane) & 1u) {
                float4* d = dst[kLeft + __popc(m >> lane >> 1)];
                const float4* src = a.rec + 4 * (size_t)k;
#pragma unroll
                for (int i = 0; i < 3; ++i)
                    asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(smem_u32(d + i)), "l"(src + i) : "memory");
            }
            asm volatile("cp.async.commit_group;" ::: "memory");
        };
        auto load_val = [&](int c) { return c >= 0 && c * kChunk + lane < n ? vals[c * kChunk + lane] : 0u; };
        auto load_words = [&](int c) { return c >= 0 ? words[(size_t)c * kBlocksPerTile] : make_uint2(0u, 0u); };
        const int c_last = (warp_last - 1) / kChunk;
        uint2 wd = load_words(c_last), wn = load_words(c_last - 1);
        uint32_t kc = load_val(c_last), kn = load_val(c_last - 1);
        stage(S.dense[c_last & 1], wd.x | wd.y, kc);
        int left = 0;             // entries of earlier chunks not walked yet
        int staged = 0;           // entries staged before this chunk
        // a pixel takes part from its own last composited entry on: the
        // position of that entry in the walk
        int start[2] = {0x7fffffff, 0x7fffffff};
        bool indefinite = false;  // among the left-over entries or the chunk's
        unsigned int walked = 0;
        // (one more turn walks what is left over)
        for (int c = c_last; c >= 0 || (c == -1 && left > 0); --c) {
            const int s = c & 1;
            const uint32_t m = wd.x | wd.y;
            walked += __popc(wd.x) + __popc(wd.y);
            stage(S.dense[s ^ 1], wn.x | wn.y, kn);
            const uint32_t kcur = kc;
            wd = wn;
            kc = kn;
            wn = load_words(c - 2);
            kn = load_val(c - 2);
            asm volatile("cp.async.wait_group 1;" ::: "memory");
            bool ind = false;
            if ((m >> lane) & 1u) {
                // the lane's own record: its index takes the place of an
                // unused value
                float4* d = S.dense[s][kLeft + __popc(m >> lane >> 1)];
                d[1].w = __uint_as_float(kcur);
                ind = !(d[2].w > -3.0e38f);
            }
            indefinite = __any_sync(0xffffffffu, ind || (lane == 0 && S.odd != 0u)) || (left > 0 && indefinite);
#pragma unroll
            for (int p = 0; p < 2; ++p)
                if (lst[p] > 0 && (lst[p] - 1) / kChunk == c) start[p] = staged + __popc(m >> ((lst[p] - 1) & 31) >> 1);
            __syncwarp();
            const int avail = left + __popc(m);
            int o = kLeft - left, walk = avail / kSlots * kSlots;
            if (c < 0) {
                // the block's last group is filled up with records that
                // composite nowhere (sigma = 0)
                if (lane < 3 * (kSlots - left)) (&S.dense[s][kLeft][0])[lane] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                __syncwarp();
                walk = kSlots;
            }
            for (const int end = o + walk; o < end; o += kSlots) {
                const float4 (*D)[3] = S.dense[s] + o;
                const int rel0 = start[0] - (staged + o - kLeft), rel1 = start[1] - (staged + o - kLeft);
                // One entry at the lane's two pixels up to alpha.  The value of
                // 2^P2 here only feeds the adjoint, so the hardware approximation
                // (ex2.approx, a few ulp from 2^x, as is the contract's
                // polynomial) serves; the decisions that must be the forward's --
                // alpha >= 1/255 and the 0.99 clamp -- are re-taken with the
                // contract's exponential whenever alpha lies within 1.1e-6 of
                // either threshold (3e-4 relative at 1/255: several times what
                // the approximations can differ by).  Clamped pixels and records
                // that need the P2 > 0 test take that path too.
                struct Entry {
                    float P[2], sa[2], cdot[2];
                    float sig;
                };
                auto eval = [&](int e) {
                    Entry t;
                    const float4 q0 = D[e][0], q1 = D[e][1], q2 = D[e][2];
                    const float dx0 = __fsub_rn(fx, q0.x), dx1 = __fsub_rn(fx1, q0.x), dy = __fsub_rn(fy, q0.y);
                    const float tt = __fmul_rn(q0.w, dy), ss = __fmul_rn(__fmul_rn(q1.x, dy), dy);
                    t.P[0] = __fmaf_rn(dx0, __fmaf_rn(q0.z, dx0, tt), ss);
                    t.P[1] = __fmaf_rn(dx1, __fmaf_rn(q0.z, dx1, tt), ss);
                    t.sig = q1.y;
#pragma unroll
                    for (int p = 0; p < 2; ++p) {
                        t.sa[p] = __fmul_rn(q1.y, ex2_approx(t.P[p]));
                        t.cdot[p] = dc[p].x * q2.x + dc[p].y * q2.y + dc[p].z * q2.z;
                        if constexpr (DEPTH) t.cdot[p] += dc[p].w * q1.z;
                    }
                    return t;
                };
                auto near = [&](const Entry& t) {
                    return t.sa[0] > GSR_ALPHA_MAX - 1.1e-6f || fabsf(t.sa[0] - GSR_ALPHA_MIN) <= 1.1e-6f ||
                           t.sa[1] > GSR_ALPHA_MAX - 1.1e-6f || fabsf(t.sa[1] - GSR_ALPHA_MIN) <= 1.1e-6f;
                };
                // A pixel that does not composite the entry takes alpha = 0: its T
                // and X stay, and gP and w are zero.
                auto step = [&](const Entry& t, int e, auto EXACT) {
                    float gP[2], w[2];
#pragma unroll
                    for (int p = 0; p < 2; ++p) {
                        const bool active = e >= (p ? rel1 : rel0);
                        float al, alg;   // alpha; alpha where it has a derivative
                        if constexpr (EXACT.value) {
                            const float sa = __fmul_rn(t.sig, exp2_walk(t.P[p]));
                            al = active && t.P[p] <= 0.0f && fminf(GSR_ALPHA_MAX, sa) >= GSR_ALPHA_MIN
                                     ? fminf(GSR_ALPHA_MAX, sa) : 0.0f;
                            alg = sa < GSR_ALPHA_MAX ? al : 0.0f;
                        } else {
                            al = active && t.sa[p] >= GSR_ALPHA_MIN ? t.sa[p] : 0.0f;
                            alg = al;
                        }
                        const float iom = rcp_approx(1.0f - al);   // 1 - al >= 0.01; 1 for al = 0
                        const float ga = iom * fmaf(T[p], t.cdot[p], -X[p]);
                        T[p] = T[p] * iom;
                        w[p] = al * T[p];
                        gP[p] = EXACT.value && alg == 0.0f ? 0.0f : ga * alg;
                        X[p] = fmaf(w[p], t.cdot[p], X[p]);
                    }
                    const int at = (16 * e + ((lane >> 1) ^ e)) * 2;
                    gp[at] = make_float2(gP[0], gP[1]);
                    wg[at] = make_float2(w[0], w[1]);
                };
                // two entries at a time: the second's alpha (independent of T
                // and X) overlaps the first's update
#pragma unroll
                for (int e = 0; e < kSlots; e += 2) {
                    const Entry t0 = eval(e), t1 = eval(e + 1);
                    if (__any_sync(0xffffffffu, indefinite || near(t0) || near(t1))) {
                        step(t0, e, std::true_type{});
                        step(t1, e + 1, std::true_type{});
                    } else {
                        step(t0, e, std::false_type{});
                        step(t1, e + 1, std::false_type{});
                    }
                }
                __syncwarp();
                reduce_group<DEPTH>(S, D, min(kSlots, kLeft + __popc(m) - o), lane, cx, cy, a.grad_rec, a.rec_cap);
                __syncwarp();
            }
            staged += __popc(m);
            left = max(0, avail - walk);
            // the entries left over go in front of the next chunk's
            if (lane < 3 * left) (&S.dense[s ^ 1][0][0])[3 * (kLeft - left) + lane] = (&S.dense[s][0][0])[3 * o + lane];
            __syncwarp();
        }
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        if (lane == 0) S.stat[1] += walked;
    }
    if (lane == 0) {
        if (S.stat[0]) atomicAdd(a.counters + kCntBwdPairs, S.stat[0]);
        if (S.stat[1]) atomicAdd(a.counters + kCntWarpBwd, S.stat[1]);
    }
}

// ---------------------------------------------------------------------------
// dispatch
// ---------------------------------------------------------------------------
template <int BX, bool COUNT>
static void fwd_launch(const Table& T, const BlendFwdArgs& a, int num_sms, cudaStream_t s)
{
    auto kern = blend_fwd_kernel<BX, COUNT>;
    // function attributes and occupancy are per device
    static std::atomic<int> per_sm_dev[kMaxDevices];
    const int per_sm = per_device_once(per_sm_dev, [&] {
        int n = 0;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kern, kFwdThreads, 0);
        return n < 1 ? 1 : n;
    });
    int64_t grid = (int64_t)num_sms * per_sm;
    const int64_t want = (T.n_tiles * kBlocksPerTile + kFwdWarps - 1) / kFwdWarps;
    if (grid > want) grid = want;
    if (grid < 1) return;
    GSR_COUNT_LAUNCH();
    kern<<<(unsigned)grid, kFwdThreads, 0, s>>>(T, a);
}

template <int BX>
static void fwd_one(const Table& T, const BlendFwdArgs& a, int num_sms, cudaStream_t s)
{
    if (a.count_pairs) fwd_launch<BX, true>(T, a, num_sms, s);
    else fwd_launch<BX, false>(T, a, num_sms, s);
}

template <int BX, bool DEPTH>
static void bwd_launch(const Table& T, const BlendBwdArgs& a, int num_sms, cudaStream_t s)
{
    auto kern = blend_bwd_kernel<BX, DEPTH>;
    static std::atomic<int> per_sm_dev[kMaxDevices];
    const int per_sm = per_device_once(per_sm_dev, [&] {
        int n = 0;
        // six blocks of 36 KB fit an SM only with all of the unified L1 as shared memory
        cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, (int)cudaSharedmemCarveoutMaxShared);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kern, kFwdThreads, 0);
        return n < 1 ? 1 : n;
    });
    int64_t grid = (int64_t)num_sms * per_sm;
    if (grid > T.n_tiles) grid = T.n_tiles;
    if (grid < 1) return;
    GSR_COUNT_LAUNCH();
    kern<<<(unsigned)grid, kFwdThreads, 0, s>>>(T, a);
}

template <int BX>
static void bwd_one(const Table& T, const BlendBwdArgs& a, int num_sms, cudaStream_t s)
{
    if (a.dl_depth) bwd_launch<BX, true>(T, a, num_sms, s);
    else bwd_launch<BX, false>(T, a, num_sms, s);
}

bool blend_supported(int tw, int th, int batch)
{
    const bool shape = (tw == 16 && th == 16) || (tw == 32 && th == 8) || (tw == 8 && th == 32);
    const bool b = batch == 128 || batch == 256 || batch == 512;
    return shape && b;
}

// (both directions stage chunks of 32 entries per warp whatever the configured batch)
void launch_blend_fwd(const Table& T, const BlendFwdArgs& a, int num_sms, cudaStream_t s)
{
    if (T.tile_w == 16) fwd_one<16>(T, a, num_sms, s);
    else if (T.tile_w == 32) fwd_one<32>(T, a, num_sms, s);
    else fwd_one<8>(T, a, num_sms, s);
}

size_t blend_mask_bytes(int64_t list_span, int64_t n_tiles)
{
    return ((size_t)(list_span / kChunk) + 2 * (size_t)n_tiles + 1) * kMaskWords * sizeof(uint32_t);
}

void launch_blend_bwd(const Table& T, const BlendBwdArgs& a, int num_sms, cudaStream_t s)
{
    if (T.tile_w == 16) bwd_one<16>(T, a, num_sms, s);
    else if (T.tile_w == 32) bwd_one<32>(T, a, num_sms, s);
    else bwd_one<8>(T, a, num_sms, s);
}

}  // namespace gsr
