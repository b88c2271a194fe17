// gsr_blend.cu -- per-pixel compositing (forward) and its adjoint (backward).
//
// One persistent launch per direction covers every (view, tile) of the batch:
// work comes from an atomic tile counter, so views of uneven size and tiles of
// uneven list length share one grid of (SMs x resident blocks).  A tile has
// 256 pixels.  The backward, and the forward's tile form, give the tile to a block
// of eight warps over 8x4 pixels each and walk the list in batches of BATCH
// records, each gathered into shared memory with one bulk async copy
// (cp.async.bulk, the TMA engine) per record (64 bytes; the backward stages only
// the 48 it reads), completing on an mbarrier, double-buffered so the gather of
// batch b+1 overlaps the arithmetic of batch b.  The forward's warp form gives an
// 8x8 pixel block to a warp that waits for no other (see below).
//
// Culling: every record carries a conservative box outside which its
// binary32 alpha is certainly below 1/255 (see alpha_box in
// gsr_preprocess.cu) and a threshold of its exponent.  A forward warp walks only
// the entries that can touch its pixels, in list order, and records which 8x4
// blocks composited each entry; the backward walks exactly those.  Skipped
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
//   warp through per-warp slot buffers (one entry per lane pair, see
//   slots_reduce), over the CTA in shared memory, and added to the
//   per-record gradient with one vector atomic per 16 bytes.
#include <algorithm>
#include <type_traits>

#include "gsr_common.cuh"
#include "gsr_kernels.h"

namespace gsr {

constexpr int kBlendThreads = 256;
constexpr int kWarps = kBlendThreads / 32;

template <int BX, int BY>
struct TileShape {
    static_assert(BX * BY == kBlendThreads, "tile must hold 256 pixels");
    static constexpr int WX = 8, WY = 4;          // warp footprint
    static constexpr int WPR = BX / WX;           // warps per tile row
    __device__ static int lx(int tid) { return ((tid >> 5) % WPR) * WX + (tid & 7); }
    __device__ static int ly(int tid) { return ((tid >> 5) / WPR) * WY + ((tid & 31) >> 3); }
};

// Gather `cnt` records (list positions [first, first + cnt)) into dst.
template <int NQ>
__device__ __forceinline__ void issue_batch(const uint32_t* vals, const float4* rec, uint32_t first, int cnt,
                                            float4* dst, uint64_t* bar, uint32_t* idx_out)
{
    const int tid = threadIdx.x;
    if (tid == 0) mbar_arrive_expect_tx(bar, (uint32_t)cnt * NQ * 16u);
    for (int t = tid; t < cnt; t += kBlendThreads) {
        const uint32_t k = vals[first + t];
        if (idx_out) idx_out[t] = k;
        bulk_g2s(dst + NQ * t, rec + 4 * (size_t)k, NQ * 16, bar);
    }
}

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
// composited-entry masks
// ---------------------------------------------------------------------------
constexpr int kChunk = 32;              // list entries per mask word
constexpr int kBlk = 8;                 // a pixel block's side
constexpr int kBlocksPerTile = kBlendThreads / (kBlk * kBlk);

// First 32-bit word of a tile's composited-entry masks: kMaskWords words per
// chunk of 32 list positions, word 2 blk + h the entries that some pixel of
// the upper (h = 0) or lower 8x4 half of block blk composited.  A tile's
// chunks start at its range's first position / 32 plus the tile id (plus the
// tile count in the second list region), so no two tiles' words overlap:
// floor((x + n) / 32) - floor(x / 32) + 1 >= ceil(n / 32).  (The sum fits 32 bits:
// a tile has eight pixels and more but at the edges, of 28 bytes each.)
constexpr int kMaskWords = 2 * kBlocksPerTile;
__device__ __forceinline__ size_t mask_base(uint32_t first, uint32_t tile, uint32_t region2, int64_t n_tiles)
{
    return (size_t)kMaskWords * (first / kChunk + tile + (first >= region2 ? (uint32_t)n_tiles : 0u));
}
// The word of the 8x4 pixels of warp w of a tile-wide block, WPR warps per tile row.
template <int WPR>
__device__ __forceinline__ int mask_word(int w) { return 2 * ((w / WPR / 2) * WPR + w % WPR) + ((w / WPR) & 1); }

// ---------------------------------------------------------------------------
// forward
// ---------------------------------------------------------------------------
// Two forms, the same results bit for bit.
//   warp form  one warp per 8x8 pixel block, two pixels per lane, no waits
//              between warps (below): fewer instructions per pair.
//   tile form  the tile's eight 8x4 warps in step, a pixel per lane: twice the
//              warps on a tile and the shorter chain per list entry.
// The sum of the work decides for the warp form, the longest lists' chains for the
// tile form.  So the lists choose, on the device: the warp form if the longest one
// has at most 1 / kWarpFormShare of the instances per resident block (the kernels
// that make the lists see it as they go).  Times of the two (tile, warp form; ms)
// around that line, by instances per resident block over longest list, from 4096
// tiles on:
//   share 3.9  six 1600x900 views, 1M Gaussians      2.10  1.63
//   share 1.9  1237x701 and smaller, 32x8 tiles      0.263 0.229
//   share 1.9  24 views of 606x348                   0.351 0.353
//   share 1.5  18 1080p views of the road, 300k      3.20  2.90
//   share 1.0  one view of 1242x995                  0.090 0.123
//   share 0.8  24 views of 400x225, 300k             1.08  1.38
//   share 0.2  24 views up to 994x845 of the road    1.40  2.97
// With fewer tiles there is little to gain (3840 tiles at share 2.6: 0.193 and
// 0.175; 2300 at 2.0: 0.107 and 0.114), and small images would feel the second
// launch (the form not taken returns after 4 us).
constexpr int64_t kWarpFormMinTiles = 4096;
constexpr double kWarpFormShare = 1.5;
__device__ __forceinline__ bool warp_form(const BlendFwdArgs& a) { return a.long_list && *a.long_list == 0ull; }

// ---- tile form
// A block has one thread per pixel and takes the next tile from the counter.  The
// list is walked in batches of BATCH records, each gathered into shared memory with
// one bulk async copy per record, completing on an mbarrier, double-buffered so
// that the gather of batch b+1 overlaps the arithmetic of batch b.  After a batch
// lands, each record's box is tested against the eight warps' 8x4 pixel blocks, and
// each warp walks only the entries that can touch its pixels.

// Bit w of mask[t]: record t can reach alpha >= 1/255 at a pixel centre of
// warp w.  Two conservative tests: the record's alpha box against the warp's
// block, then the maximum of the record's exponent over the block against
// its culling threshold (record slot 11).  The corner offsets are rounded
// exactly as the blend rounds each pixel's offset, so every pixel's rounded
// offset lies in the tested rectangle.
template <int BX, int BY>
__device__ __forceinline__ void warp_masks(const float4* B, int cnt, int tx0, int ty0, uint8_t* s_mask)
{
    using TS = TileShape<BX, BY>;
    for (int t = threadIdx.x; t < cnt; t += kBlendThreads) {
        const float4 r0 = B[4 * t];
        const float qc = B[4 * t + 1].x;
        const float thr_cull = B[4 * t + 2].w;
        const float4 bb = B[4 * t + 3];
        const float kx = -r0.w / (2.0f * r0.z), ky = -r0.w / (2.0f * qc);
        uint32_t m = 0;
#pragma unroll 1
        for (int w = 0; w < kWarps; ++w) {
            const float X0 = (float)(tx0 + (w % TS::WPR) * TS::WX);
            const float Y0 = (float)(ty0 + (w / TS::WPR) * TS::WY);
            bool hit = bb.x <= X0 + (TS::WX - 0.5f) && bb.y >= X0 + 0.5f && bb.z <= Y0 + (TS::WY - 0.5f) &&
                       bb.w >= Y0 + 0.5f;
            if (hit && thr_cull > -3.0e38f) {
                const float x0 = __fsub_rn(__fadd_rn(X0, 0.5f), r0.x);
                const float x1 = __fsub_rn(__fadd_rn(X0, TS::WX - 0.5f), r0.x);
                const float y0 = __fsub_rn(__fadd_rn(Y0, 0.5f), r0.y);
                const float y1 = __fsub_rn(__fadd_rn(Y0, TS::WY - 0.5f), r0.y);
                hit = rect_max_form(x0, x1, y0, y1, r0.z, r0.w, qc, kx, ky) >= thr_cull;
            }
            m |= (uint32_t)hit << w;
        }
        s_mask[t] = (uint8_t)m;
    }
}

// This warp's entries of the batch, in list order; returns their number.
__device__ __forceinline__ int warp_list(const uint8_t* s_mask, int cnt, int w, int lane, uint16_t* list)
{
    int nl = 0;
    const uint32_t lt = (1u << lane) - 1u;
    for (int base = 0; base < cnt; base += 32) {
        const int t = base + lane;
        const bool bit = t < cnt && ((s_mask[t] >> w) & 1u);
        const uint32_t bal = __ballot_sync(0xffffffffu, bit);
        if (bit) list[nl + __popc(bal & lt)] = (uint16_t)t;
        nl += __popc(bal);
    }
    __syncwarp();
    return nl;
}

// One (pixel, entry) pair of the forward up to alpha (independent of T).
struct TilePair {
    int k;
    float P2, al;
    float4 c;      // colour, depth
};

__device__ __forceinline__ TilePair tile_pair(const float4* B, int k, float pxf, float pyf)
{
    TilePair e;
    e.k = k;
    const float4 r0 = B[4 * k];
    const float4 r1 = B[4 * k + 1];
    const float4 r2 = B[4 * k + 2];
    const float dx = __fsub_rn(pxf, r0.x), dy = __fsub_rn(pyf, r0.y);
    e.P2 = __fmaf_rn(dx, __fmaf_rn(r0.z, dx, __fmul_rn(r0.w, dy)), __fmul_rn(__fmul_rn(r1.x, dy), dy));
    e.al = fminf(GSR_ALPHA_MAX, __fmul_rn(r1.y, exp2_nonpos(fminf(e.P2, 0.0f))));
    e.c = make_float4(r2.x, r2.y, r2.z, r1.z);
    return e;
}

// Four blocks per SM: 64 registers (the two-entry walk would otherwise take
// 72 and leave room for three).  COUNT: keep the per-pixel examined and
// composited counts (statistics only; a separate instantiation because the
// two running counts cost about 6 % of the walk).
template <int BX, int BY, int BATCH, bool COUNT>
__global__ void __launch_bounds__(kBlendThreads, 4)
blend_fwd_tile_kernel(const __grid_constant__ Table Tb, BlendFwdArgs a)
{
    if (earlier_wait_timed_out(a.status) || warp_form(a)) return;
    using TS = TileShape<BX, BY>;
    extern __shared__ __align__(128) float4 s_buf[];     // [2][BATCH][4]
    __shared__ __align__(8) uint64_t s_bar[2];
    __shared__ unsigned int s_item;
    __shared__ uint8_t s_mask[BATCH];
    __shared__ uint16_t s_list[kWarps][BATCH];
    __shared__ __align__(16) uint8_t s_wb[kWarps][BATCH]; // per warp: composited each entry of the batch
    // per tile (kept in shared memory, off the walk's registers): the warps'
    // walked entries, and the list entries up to the end of the batch in
    // which every pixel had stopped (0: they did not)
    __shared__ unsigned int s_witer[kWarps];
    __shared__ int s_satpos;
    __shared__ int s_prefix_all;   // the first round's lists are the full ones
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    if (tid == 0) {
        mbar_init(&s_bar[0], 1);
        mbar_init(&s_bar[1], 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        const int64_t n_vis = (int64_t)a.counters[kCntVisible];
        s_prefix_all = prefix_records(n_vis, a.prefix) == n_vis;
    }
    for (int t = tid; t < kWarps * BATCH / 4; t += kBlendThreads) reinterpret_cast<uint32_t*>(&s_wb[0][0])[t] = 0u;
    __syncthreads();
    uint32_t par0 = 0u, par1 = 0u;
    const int lx = TS::lx(tid), ly = TS::ly(tid);
    unsigned long long exam_total = 0, blended_total = 0;
    unsigned int witer = 0;
    bool failed = false;
    uint16_t* L = s_list[w];
    if (a.round == 2 && a.counters[kCntOpenTiles] == 0ull) return;

    for (;;) {
        if (tid == 0) s_item = atomicAdd(a.work, 1u);
        __syncthreads();
        const unsigned int item = s_item;
        __syncthreads();
        if ((int64_t)item >= Tb.n_tiles || failed) break;
        if (a.round == 2 && !((a.open_tiles[item >> 5] >> (item & 31u)) & 1u)) continue;
        if (lane == 0) s_witer[w] = 0u;
        if (tid == 0) s_satpos = 0;
        const int view = find_view_of_tile(Tb, item);
        const DevView& V = Tb.v[view];
        const int lt = (int)(item - V.tile_base);
        const int tx0 = (lt % V.TX) * BX, ty0 = (lt / V.TX) * BY;
        const int px = tx0 + lx, py = ty0 + ly;
        const bool inside = px < V.W && py < V.H;
        const uint2 rg = a.ranges[item];
        const int n = (int)(rg.y - rg.x);
        const int nb = (n + BATCH - 1) / BATCH;
        const float pxf = __fadd_rn((float)px, 0.5f), pyf = __fadd_rn((float)py, 0.5f);
        float T = 1.0f, C0 = 0.0f, C1 = 0.0f, C2 = 0.0f, D = 0.0f;
        uint32_t last = 0, exam = (uint32_t)n, nblend = 0;
        bool done = !inside;

        if (nb > 0) issue_batch<4>(a.vals, a.rec, rg.x, min(BATCH, n), s_buf, &s_bar[0], nullptr);
        for (int b = 0; b < nb; ++b) {
            const int s = b & 1;
            if (b + 1 < nb)
                issue_batch<4>(a.vals, a.rec, rg.x + (b + 1) * BATCH, min(BATCH, n - (b + 1) * BATCH),
                            s_buf + (size_t)(s ^ 1) * BATCH * 4, &s_bar[s ^ 1], nullptr);
            const bool ok = mbar_wait_bounded(&s_bar[s], s ? par1 : par0, a.status, a.wait_ns);
            if (s) par1 ^= 1u; else par0 ^= 1u;
            if (__syncthreads_or(!ok)) {
                failed = true;
                if (b + 1 < nb) mbar_wait_bounded(&s_bar[s ^ 1], s ? par0 : par1, a.status, a.wait_ns);
                break;
            }
            const int cnt = min(BATCH, n - b * BATCH);
            const float4* B = s_buf + (size_t)s * BATCH * 4;
            warp_masks<BX, BY>(B, cnt, tx0, ty0, s_mask);
            __syncthreads();
            const int nl = warp_list(s_mask, cnt, w, lane, L);
            // Structured body and a warp vote per entry: the vote reconverges
            // the warp every iteration (lanes would otherwise drift apart under
            // independent thread scheduling) and ends the batch for the warp
            // once all of its pixels are done.
            if (!__all_sync(0xffffffffu, done)) {
                // Branch-free: after exact culling nearly every walked entry
                // composites somewhere in the warp, so every lane evaluates it
                // and the decisions select the updates (a zero weight leaves C
                // and D bit-identical).  Entries are taken two at a time: the
                // second's alpha does not depend on T, so it overlaps the
                // first's update; the warp vote that ends the walk once every
                // pixel has stopped is taken after every second pair (a done
                // pixel passes nothing, so the extra entries change no result).
                // Returns whether this pixel composited the entry.
                auto step = [&](const TilePair& e) {
                    const float Tn = __fmul_rn(T, __fsub_rn(1.0f, e.al));
                    const bool pass = !done && e.P2 <= 0.0f && e.al >= GSR_ALPHA_MIN;
                    const bool stop = pass && Tn < GSR_T_STOP;
                    const bool blended_now = pass && !stop;
                    const float wgt = blended_now ? e.al * T : 0.0f;
                    C0 = fmaf(e.c.x, wgt, C0);
                    C1 = fmaf(e.c.y, wgt, C1);
                    C2 = fmaf(e.c.z, wgt, C2);
                    D = fmaf(e.c.w, wgt, D);
                    T = blended_now ? Tn : T;
                    if constexpr (COUNT) {
                        exam = stop ? (uint32_t)(b * BATCH + e.k + 1) : exam;
                        nblend += blended_now ? 1u : 0u;
                    }
                    done = done || stop;
                    return blended_now;
                };
                // Bit p of a lane's wb is its own decision for the p-th entry of
                // a group of 32.  Per group: the pixel's last composited entry
                // is the highest set bit, and one OR over the warp publishes
                // which entries some pixel of the warp composited (entry
                // L[i0 + l] by lane l).
                auto publish = [&](uint32_t wb, int i0, int cnt) {
                    if (wb) last = (uint32_t)(b * BATCH + L[i0 + 31 - __clz(wb)] + 1);
                    const uint32_t any = __reduce_or_sync(0xffffffffu, wb);
                    if (lane < cnt && ((any >> lane) & 1u)) s_wb[w][L[i0 + lane]] = 1;
                };
                int i = 0;
                bool all = false;
                // whole groups of 32 entries, bit positions fixed at compile time
                for (; i + 32 <= nl; i += 32) {
                    uint32_t wb = 0;
                    int p = 0;
#pragma unroll
                    for (; p < 32; p += 2) {
                        const TilePair e0 = tile_pair(B, L[i + p], pxf, pyf);
                        const TilePair e1 = tile_pair(B, L[i + p + 1], pxf, pyf);
                        if (step(e0)) wb |= 1u << p;
                        if (step(e1)) wb |= 2u << p;
                        if ((p & 2) && __all_sync(0xffffffffu, done)) { p += 2; all = true; break; }
                    }
                    publish(wb, i, p);
                    if (all) { i += p; break; }
                }
                if (!all) {
                    // the last (fewer than 32) entries
                    uint32_t wb = 0;
                    int p = 0;
                    for (; i + p + 1 < nl; p += 2) {
                        const TilePair e0 = tile_pair(B, L[i + p], pxf, pyf);
                        const TilePair e1 = tile_pair(B, L[i + p + 1], pxf, pyf);
                        if (step(e0)) wb |= 1u << p;
                        if (step(e1)) wb |= 2u << p;
                        if (__all_sync(0xffffffffu, done)) { p += 2; all = true; break; }
                    }
                    if (!all && i + p < nl) {
                        if (step(tile_pair(B, L[i + p], pxf, pyf))) wb |= 1u << p;
                        ++p;
                    }
                    publish(wb, i, p);
                    i += p;
                }
                if (lane == 0) s_witer[w] += (unsigned)i;
                // The warp's mask words of the batch (the backward walks only those
                // entries, and reads no further than a warp's last composited one:
                // a warp whose pixels have all stopped writes no more).  A lane
                // packs kLaneBits flags (bytes of 0 or 1) into bits, the lanes of a
                // word put theirs together.  (Ballots after the block's barrier,
                // one warp per 32 entries: 44 us on a view of 296 x 176, 42 so; 0.98
                // and 0.94 ms on six of 224 x 118 with lists of 0.3 M entries.)
                if (a.wmask) {
                    constexpr int kLaneBits = BATCH / 32, kLanes = 32 / kLaneBits;
                    __syncwarp();
                    uint32_t* const f = reinterpret_cast<uint32_t*>(s_wb[w]) + lane * (kLaneBits / 4);
                    uint32_t word = 0u;
                    if (nl > 0) {
#pragma unroll
                        for (int q = 0; q < kLaneBits / 4; ++q) {
                            word |= ((f[q] * 0x01020408u >> 24) & 15u) << (4 * q);
                            f[q] = 0u;
                        }
                        word <<= kLaneBits * (lane % kLanes);
#pragma unroll
                        for (int o = 1; o < kLanes; o *= 2) word |= __shfl_xor_sync(0xffffffffu, word, o);
                    }
                    const int c = lane / kLanes;
                    if (lane % kLanes == 0 && c * kChunk < cnt)
                        a.wmask[mask_base(rg.x, s_item, a.region2, Tb.n_tiles) +
                                (size_t)(b * (BATCH / kChunk) + c) * kMaskWords + mask_word<TS::WPR>(w)] = word;
                }
            }
            const bool all_done = __syncthreads_and(done);
            if (all_done) {
                if (tid == 0) s_satpos = b * BATCH + cnt;
                // drain the prefetched batch before leaving the tile
                if (b + 1 < nb) {
                    const bool ok2 = mbar_wait_bounded(&s_bar[s ^ 1], s ? par0 : par1, a.status, a.wait_ns);
                    if (s) par0 ^= 1u; else par1 ^= 1u;
                    if (__syncthreads_or(!ok2)) failed = true;
                }
                break;
            }
        }
        // A first round's tile is final when its pixels all stopped within
        // the prefix lists (or those were the full lists); otherwise the
        // second round renders it again over its full list.
        const bool saturated = __syncthreads_and(done);   // (also publishes s_witer and s_satpos)
        const bool final_tile = a.round != 1 || saturated || s_prefix_all;
        // (thread 0 re-reads the tile and its range: nothing of them stays
        // live in registers across the walk)
        if (!final_tile) {
            if (tid == 0 && !failed) {
                const unsigned int it = s_item;
                atomicOr(a.open_tiles + (it >> 5), 1u << (it & 31u));
                atomicAdd(a.counters + kCntOpenTiles, 1ull);
            }
            continue;
        }
        if (lane == 0) witer += s_witer[w];
        if (tid == 0 && a.hist && !failed) {
            // the share of the depth-ordered records the tile needed before
            // every pixel stopped, weighted by its (estimated full) list length
            const uint2 r = a.ranges[s_item];
            const unsigned long long n_vis = a.counters[kCntVisible];
            int bucket = kSatBuckets;
            if (saturated && s_satpos > 0 && n_vis > 0ull) {
                const uint32_t k = a.vals[r.x + s_satpos - 1];
                bucket = sat_bucket((float)(a.depthpos[k] + 1u) / (float)n_vis);
            }
            unsigned long long len = r.y - r.x;
            if (a.round == 1) {
                const unsigned long long n_pre = (unsigned long long)prefix_records((int64_t)n_vis, a.prefix);
                if (n_pre > 0ull) len = len * n_vis / n_pre;
            }
            if (len) atomicAdd(a.hist + bucket, len);
        }
        if (inside) {
            const int64_t hw = (int64_t)V.W * V.H;
            const int64_t off = (int64_t)py * V.W + px;
            const int64_t pix = V.pix_base + off;
            float* rgb = a.rgb + 3 * V.pix_base;
            rgb[off] = C0 + T * Tb.bg[0];
            rgb[hw + off] = C1 + T * Tb.bg[1];
            rgb[2 * hw + off] = C2 + T * Tb.bg[2];
            a.depth[pix] = D;
            a.alpha[pix] = 1.0f - T;
            a.tfinal[pix] = T;
            a.ncontrib[pix] = last;
            if constexpr (COUNT) {
                exam_total += exam;
                blended_total += nblend;
            }
        }
    }
    exam_total = warp_sum(exam_total);
    blended_total = warp_sum(blended_total);
    if (lane == 0 && exam_total) atomicAdd(a.counters + kCntFwdPairs, exam_total);
    if (lane == 0 && blended_total) atomicAdd(a.counters + kCntBlended, blended_total);
    if (lane == 0 && witer) atomicAdd(a.counters + kCntWarpFwd, (unsigned long long)witer);
}

// ---- warp form
// One warp renders one 8x8 pixel block of a tile, two horizontally adjacent
// pixels per lane, and nothing in it waits for another warp.  The tile's list
// is walked in chunks of 32 entries.  Per chunk: the records (64 bytes each)
// arrive by asynchronous copies issued one chunk ahead; each lane tests one
// entry against the block (alpha box, then the maximum of the exponent over the
// block); the survivors' walk values are written densely to shared memory; the
// walk evaluates each survivor at the lane's two pixels.
//
// Bound by instruction issue (88 % of the slots; DRAM 3 %).  Against one
// pixel per lane with the tile's eight 8x4 warps in step (a barrier per 256
// staged entries, 85 % of the slots for 22 % more instructions): a record's loads, dy and the row's products
// serve two pixels, the barriers and the batch bookkeeping are gone, and a block
// stops fetching as soon as its own pixels have stopped; it walks more idle
// lanes (8x8 blocks composite 69 % of the walked lanes on the 1M-Gaussian
// six-camera rig, 8x4 blocks 77 %).  Rig 2.04 -> 1.63 ms, 30-view window (with
// pair counters) 9.8 -> 7.35 ms, 60-view road 29.1 -> 21.6 ms.  Packed pairs
// (fma.rn.f32x2 over the two pixels) take the issue slots of the two scalar
// operations on this part and need their operands twice: 1.69 ms on the rig.
constexpr int kFwdWarps = 4;            // warps per block (they share a tile, see next_block)
constexpr int kFwdThreads = 32 * kFwdWarps;

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

// COUNT: keep the per-pixel examined and composited counts (statistics only;
// a separate instantiation because the running counts lengthen the walk).
// 80 registers, six blocks per SM (at 72 the walk spills: 6 % slower).
template <int BX, bool COUNT>
__global__ void __launch_bounds__(kFwdThreads, 6)
blend_fwd_warp_kernel(const __grid_constant__ Table Tb, BlendFwdArgs a)
{
    if (earlier_wait_timed_out(a.status) || !warp_form(a)) return;
    constexpr int BY = kBlendThreads / BX, BPR = BX / kBlk;   // blocks per tile row
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
                // in steps of the tile form's batch, which the choice of the
                // first round's fraction was fitted to: finer steps made it take
                // two rounds where one is faster (30k Gaussians on a view of
                // 1280 x 900: 0.66 -> 0.76 ms)
                const uint32_t steps = ((uint32_t)satpos + a.stat_batch - 1u) / a.stat_batch;
                atomicMax(&need->x, saturated ? min(steps * a.stat_batch, (uint32_t)n) : never);
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

// Backward reduction over a warp's 32 pixels, transposed.  For each walked
// entry every lane stores two scalars in its warp's slot buffer -- gP =
// dL/dP2 and w = alpha T (both zero where the pixel does not composite the
// entry) -- and every kSlots entries the warp reduces the buffer with one
// entry per lane pair, so a lane sums over pixels serially instead of the
// warp summing ten values per entry with shuffles.  The record gradient needs
//   sum gP dx, sum gP dy, sum gP dx^2, sum gP dx dy, sum gP dy^2,
//   sum gP / sigma (= sum dL/dalpha G where alpha is not clamped),
//   sum w dD, sum w dC (three channels),
// with dx = px - u the same for every pixel up to the pixel's offset inside
// the 8x4 block: dx = xo - ux, xo = x - 3.5 (x = lane & 7), ux = u minus the
// block centre (same for y with yo = (lane >> 3) - 1.5).  So the warp keeps
// the six moments M = sum gP {1, xo, yo, xo^2, xo yo, yo^2} (constant
// weights) and shifts them once per entry:
//   sum gP dx = Mx - ux M0, sum gP dx^2 = Mxx - 2 ux Mx + ux^2 M0,
//   sum gP dx dy = Mxy - ux My - uy Mx + ux uy M0 (and y alike).
// The shifts cancel: the rounding error is bounded by a few 2^-24 of the sums of
// |gP| (|xo| + |ux|)^2 (|yo| <= 1.5 in the 8x4 block), not of |gP| dx^2; a record on
// one corner pixel shows it (tests/test_gpu_record_sums.py).  Per-pixel dC, dD come
// from s_dcd.
constexpr int kSlots = 16;
// Shared record sums: 10 floats per record at an odd stride, so lanes
// adding to (or flushing) different records hit different banks.
constexpr int kSumStride = 11;
constexpr int kSlotStride = 32;   // floats per slot row: 32 pixels
// 16-byte chunk c of slot row r is stored at chunk c ^ (r & 7): a row's
// stores stay a permutation of its 32 banks, and the 16-byte reads of the
// same chunk from eight different rows land in eight different bank groups.
__device__ __forceinline__ int slot_chunk(int c, int r) { return c ^ (r & 7); }
// The float of slot row r that holds pixel (lane) l: chunk l / 4, element l % 4.
__device__ __forceinline__ int slot_col(int l, int r) { return l ^ ((r & 7) << 2); }

// Slot j holds the entry at position i0 - j of the warp's walk list L.
template <typename LT>
__device__ __forceinline__ void slots_reduce(const float* __restrict__ sgp, const float* __restrict__ swg,
                                             const float4* __restrict__ sdcd, int n, int lane, const LT* L,
                                             int i0, const float4* B, float cxw, float cyw, float* s_grad)
{
    const int e = lane & (kSlots - 1), h = lane >> 4;     // entry slot, pixel half (block rows 2h, 2h + 1)
    const float* gp = sgp + e * kSlotStride;
    const float* wg = swg + e * kSlotStride;
    float g[16];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        const float4 t = *reinterpret_cast<const float4*>(gp + 4 * slot_chunk(4 * h + c, e));
        g[4 * c] = t.x; g[4 * c + 1] = t.y; g[4 * c + 2] = t.z; g[4 * c + 3] = t.w;
    }
    float r0 = 0.0f, r1 = 0.0f, mxx = 0.0f, mx0 = 0.0f, mx1 = 0.0f;
#pragma unroll
    for (int x = 0; x < 8; ++x) {
        const float xo = (float)x - 3.5f;
        r0 += g[x];
        r1 += g[8 + x];
        mxx = fmaf(xo * xo, g[x] + g[8 + x], mxx);
        mx0 = fmaf(xo, g[x], mx0);
        mx1 = fmaf(xo, g[8 + x], mx1);
    }
    const float y0 = 2.0f * (float)h - 1.5f, y1 = y0 + 1.0f;
    float v[10];
    v[0] = r0 + r1;
    v[1] = mx0 + mx1;
    v[2] = fmaf(y0, r0, y1 * r1);
    v[3] = mxx;
    v[4] = fmaf(y0, mx0, y1 * mx1);
    v[5] = fmaf(y0 * y0, r0, (y1 * y1) * r1);
    float sd = 0.0f, s0 = 0.0f, s1 = 0.0f, s2 = 0.0f;
    const float4* dcd = sdcd + 16 * h;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        const float4 t = *reinterpret_cast<const float4*>(wg + 4 * slot_chunk(4 * h + c, e));
        const float w4[4] = {t.x, t.y, t.z, t.w};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float4 d = dcd[4 * c + j];
            s0 = fmaf(w4[j], d.x, s0);
            s1 = fmaf(w4[j], d.y, s1);
            s2 = fmaf(w4[j], d.z, s2);
            sd = fmaf(w4[j], d.w, sd);
        }
    }
    v[6] = sd; v[7] = s0; v[8] = s1; v[9] = s2;
#pragma unroll
    for (int j = 0; j < 10; ++j) v[j] += __shfl_xor_sync(0xffffffffu, v[j], 16);
    if (e >= n) return;
    const uint32_t k = L[i0 - e];
    // layout of a record's sums: du dv dqa dqb dqc dsig dz dr dg db
    float* sg = s_grad + k * kSumStride;
    if (h == 0) {
        const float4 r = B[3 * k];
        const float ux = r.x - cxw, uy = r.y - cyw;
        const float m0 = v[0];
        atomicAdd(sg + 0, fmaf(-ux, m0, v[1]));
        atomicAdd(sg + 1, fmaf(-uy, m0, v[2]));
        atomicAdd(sg + 2, fmaf(ux * ux, m0, fmaf(-2.0f * ux, v[1], v[3])));
        atomicAdd(sg + 3, fmaf(ux * uy, m0, fmaf(-ux, v[2], fmaf(-uy, v[1], v[4]))));
        atomicAdd(sg + 4, fmaf(uy * uy, m0, fmaf(-2.0f * uy, v[2], v[5])));
    } else {
        atomicAdd(sg + 5, v[0]);
        atomicAdd(sg + 6, v[6]);
        atomicAdd(sg + 7, v[7]);
        atomicAdd(sg + 8, v[8]);
        atomicAdd(sg + 9, v[9]);
    }
}

// ---------------------------------------------------------------------------
// backward
// ---------------------------------------------------------------------------
// The part of one (pixel, entry) pair of the backward that does not depend
// on the running T and X: alpha, its decisions and the colour/depth dot.
struct BwdPair {
    int k;
    bool front;    // P2 <= 0
    bool near;     // alpha within 1e-6 relative of a threshold (see bwd_refine)
    bool contrib;
    float P2m, sa, al, iom, cdot;
};

__device__ __forceinline__ BwdPair bwd_pair(const float4* B, int k, float pxf, float pyf, float dC0, float dC1,
                                            float dC2, float dD)
{
    BwdPair e;
    e.k = k;
    const float4 r0 = B[3 * k];
    const float4 r1 = B[3 * k + 1];
    const float4 r2 = B[3 * k + 2];
    const float dx = __fsub_rn(pxf, r0.x), dy = __fsub_rn(pyf, r0.y);
    const float P2 = __fmaf_rn(dx, __fmaf_rn(r0.z, dx, __fmul_rn(r0.w, dy)), __fmul_rn(__fmul_rn(r1.x, dy), dy));
    // The value of 2^P2 here only feeds the adjoint, so the hardware
    // approximation (ex2.approx, a few ulp from 2^x, as is the contract's
    // polynomial) serves; the two decisions that must be the forward's --
    // alpha >= 1/255 and the 0.99 clamp -- are re-taken with the contract's
    // exponential whenever alpha lies near either threshold.  One test covers
    // both: (sa - 1/255)(sa - 0.99) is within 1.1e-6 of zero for sa within
    // about 1.1e-6 of either root (0.99 - 1/255 = 0.986), i.e. 1.1e-6 relative
    // at 0.99 and 3e-4 relative at 1/255 -- several times what the two
    // approximations can differ by (the rounding of the product is below
    // 3e-8 there).
    e.front = P2 <= 0.0f;
    e.P2m = fminf(P2, 0.0f);
    float G;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(G) : "f"(e.P2m));
    e.sa = __fmul_rn(r1.y, G);
    e.near = fabsf(__fmaf_rn(e.sa, __fsub_rn(e.sa, GSR_ALPHA_MIN + GSR_ALPHA_MAX), GSR_ALPHA_MIN * GSR_ALPHA_MAX)) <=
             1.1e-6f;
    e.cdot = dC0 * r2.x + dC1 * r2.y + dC2 * r2.z + dD * r1.z;
    return e;
}

// The contract's exponential for the (rare) pairs near a threshold.  Taken
// once per pair of entries on a warp vote, so the common case pays one vote
// instead of a divergent branch per entry.
__device__ __forceinline__ void bwd_refine(const float4* B, BwdPair& e1, BwdPair& e0)
{
    if (__any_sync(0xffffffffu, e1.near || e0.near)) {
        if (e1.near) e1.sa = __fmul_rn(B[3 * e1.k + 1].y, exp2_nonpos(e1.P2m));
        if (e0.near) e0.sa = __fmul_rn(B[3 * e0.k + 1].y, exp2_nonpos(e0.P2m));
    }
}

// The decisions and 1 / (1 - alpha) from the (refined) alpha.
__device__ __forceinline__ void bwd_finish(BwdPair& e, int lim)
{
    e.al = fminf(GSR_ALPHA_MAX, e.sa);
    e.contrib = e.k < lim && e.front && e.al >= GSR_ALPHA_MIN;
    e.iom = __fdividef(1.0f, 1.0f - e.al);   // 1 - al >= 0.01
}

// Dynamic shared memory of the backward: [2][BATCH][3] float4 records (the
// first 48 bytes of each: mean, conic, opacity, depth, colour),
// [BATCH][kSumStride] record sums, then per warp the slot buffers of gP and
// w ([kSlots][kSlotStride] floats each) and the pixels' (dC, dD) (32 float4):
// 55 KB at BATCH = 128, so four blocks share an SM.
template <int BATCH>
constexpr size_t bwd_smem_bytes()
{
    return (size_t)2 * BATCH * 48 + (size_t)BATCH * kSumStride * sizeof(float) +
           (size_t)kWarps * (2 * kSlots * kSlotStride * sizeof(float) + 32 * sizeof(float4));
}

template <int BX, int BY, int BATCH>
__global__ void __launch_bounds__(kBlendThreads, 4)
blend_bwd_kernel(const __grid_constant__ Table Tb, BlendBwdArgs a)
{
    if (earlier_wait_timed_out(a.status)) return;
    using TS = TileShape<BX, BY>;
    extern __shared__ __align__(128) float4 s_buf[];     // layout: see bwd_smem_bytes
    __shared__ __align__(8) uint64_t s_bar[2];
    __shared__ unsigned int s_item;
    __shared__ uint32_t s_idx[2][BATCH];
    __shared__ uint32_t s_maxlast;
    __shared__ int s_wlast[kWarps];   // the warps' last composited entries (off the walk's registers)
    using ListT = typename std::conditional<(BATCH <= 256), uint8_t, uint16_t>::type;
    __shared__ ListT s_list[kWarps][BATCH];
    float* s_grad = reinterpret_cast<float*>(s_buf + 2 * BATCH * 3);
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    float* s_slots = s_grad + BATCH * kSumStride;
    float* sgp = s_slots + (size_t)w * 2 * kSlots * kSlotStride;   // this warp's gP slots
    float* swg = sgp + kSlots * kSlotStride;                          // and its w slots
    float4* sdcd = reinterpret_cast<float4*>(s_slots + (size_t)kWarps * 2 * kSlots * kSlotStride) + 32 * w;
    if (tid == 0) {
        mbar_init(&s_bar[0], 1);
        mbar_init(&s_bar[1], 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    for (int i = tid; i < BATCH * kSumStride; i += kBlendThreads) s_grad[i] = 0.0f;
    __syncthreads();
    uint32_t par0 = 0u, par1 = 0u;
    const int lx = TS::lx(tid), ly = TS::ly(tid);
    unsigned long long pairs_total = 0, witer = 0;
    bool failed = false;
    ListT* L = s_list[w];

    for (;;) {
        if (tid == 0) { s_item = atomicAdd(a.work, 1u); s_maxlast = 0; }
        __syncthreads();
        const unsigned int item = s_item;
        if ((int64_t)item >= Tb.n_tiles || failed) break;
        const int view = find_view_of_tile(Tb, item);
        const DevView& V = Tb.v[view];
        const int lt = (int)(item - V.tile_base);
        const int tx0 = (lt % V.TX) * BX, ty0 = (lt / V.TX) * BY;
        const int px = tx0 + lx, py = ty0 + ly;
        const bool inside = px < V.W && py < V.H;
        const uint2 rg = a.ranges[item];
        const float pxf = __fadd_rn((float)px, 0.5f), pyf = __fadd_rn((float)py, 0.5f);
        float Tcur = 1.0f, Tf = 1.0f, dC0 = 0, dC1 = 0, dC2 = 0, dD = 0, dA = 0;
        uint32_t mylast = 0;
        if (inside) {
            const int64_t hw = (int64_t)V.W * V.H;
            const int64_t off = (int64_t)py * V.W + px;
            const int64_t pix = V.pix_base + off;
            Tf = a.tfinal[pix];
            Tcur = Tf;
            mylast = a.ncontrib[pix];
            const float* g = a.dl_rgb + 3 * V.pix_base;
            dC0 = g[off]; dC1 = g[hw + off]; dC2 = g[2 * hw + off];
            if (a.dl_depth) dD = a.dl_depth[pix];
            if (a.dl_alpha) dA = a.dl_alpha[pix];
        }
        pairs_total += mylast;
        sdcd[lane] = make_float4(dC0, dC1, dC2, dD);   // read by the slot reduction (after __syncwarp)
        const float cxw = (float)(tx0 + (w % TS::WPR) * TS::WX + TS::WX / 2);
        const float cyw = (float)(ty0 + (w / TS::WPR) * TS::WY + TS::WY / 2);
        const int warp_last = (int)__reduce_max_sync(0xffffffffu, mylast);
        if (lane == 0) {
            s_wlast[w] = warp_last;
            if (warp_last) atomicMax(&s_maxlast, (uint32_t)warp_last);
        }
        __syncthreads();
        const int maxlast = (int)s_maxlast;
        const int nb = (maxlast + BATCH - 1) / BATCH;
        // X = dC . S_C + dD S_D - dA T_final, S the suffix sums of the later
        // colour and depth terms (S_C starts at T_final bg): then
        // dL/dalpha_k = T_k (dC . c_k + dD z_k) - X / (1 - alpha_k).
        float X = Tf * (dC0 * Tb.bg[0] + dC1 * Tb.bg[1] + dC2 * Tb.bg[2] - dA);

        // batches from the back: the q-th processed batch covers list positions [bb*BATCH, ...)
        if (nb > 0) {
            const int bb = nb - 1;
            issue_batch<3>(a.vals, a.rec, rg.x + bb * BATCH, min(BATCH, maxlast - bb * BATCH), s_buf, &s_bar[0],
                        s_idx[0]);
        }
        for (int q = 0; q < nb; ++q) {
            const int s = q & 1;
            const int bb = nb - 1 - q;
            const int cnt = min(BATCH, maxlast - bb * BATCH);
            // exactly the (warp, entry) pairs the forward composited: lane j
            // holds the mask word of the batch's entries 32 j .., read before the
            // wait (past the warp's last composited entry none was written)
            uint32_t mword = 0u;
            if (lane < BATCH / kChunk && bb * BATCH + kChunk * lane < s_wlast[w])
                mword = a.wmask[mask_base(rg.x, item, a.region2, Tb.n_tiles) +
                                (size_t)(bb * (BATCH / kChunk) + lane) * kMaskWords + mask_word<TS::WPR>(w)];
            const bool ok = mbar_wait_bounded(&s_bar[s], s ? par1 : par0, a.status, a.wait_ns);
            if (s) par1 ^= 1u; else par0 ^= 1u;
            // (this barrier also orders the previous batch's flush before the
            // reuse of its buffers and sums)
            if (__syncthreads_or(!ok)) {
                failed = true;
                break;
            }
            if (q + 1 < nb) {
                const int nbb = bb - 1;
                issue_batch<3>(a.vals, a.rec, rg.x + nbb * BATCH, min(BATCH, maxlast - nbb * BATCH),
                            s_buf + (size_t)(s ^ 1) * BATCH * 3, &s_bar[s ^ 1], s_idx[s ^ 1]);
            }
            const float4* B = s_buf + (size_t)s * BATCH * 3;
            int nl = 0;
            {
                const uint32_t lt = (1u << lane) - 1u;
#pragma unroll
                for (int j = 0; j < BATCH / 32; ++j) {
                    if (32 * j < cnt) {
                        const uint32_t bal = __shfl_sync(0xffffffffu, mword, j);
                        if ((bal >> lane) & 1u) L[nl + __popc(bal & lt)] = (ListT)(32 * j + lane);
                        nl += __popc(bal);
                    }
                }
                __syncwarp();
            }
            witer += nl;
            const int lim = (int)mylast - bb * BATCH;   // this pixel's entries k < lim
            // The walk is back to front: each entry's adjoint needs T and X as
            // left by the entry after it.  Branch-free: every lane evaluates
            // the pair, and a lane that does not composite it stores zero gP
            // and w into slot s of its warp's buffers.  Entries are taken two
            // at a time so that the second's alpha (independent of T and X)
            // overlaps the first's.
            auto step = [&](const BwdPair& e, int s) {
                const float Tk = Tcur * e.iom;
                const float wgt = e.contrib ? e.al * Tk : 0.0f;
                // the clamped alpha (sa >= 0.99) has no derivative
                const float ga = (e.contrib && e.sa < GSR_ALPHA_MAX) ? Tk * e.cdot - e.iom * X : 0.0f;
                // dL/dP2 / ln2; the record's coefficients, ln2 and the sign of
                // the mean gradient are applied once per record when the
                // shared sums are flushed
                const float gP = ga * e.al;
                X = fmaf(wgt, e.cdot, X);
                Tcur = e.contrib ? Tk : Tcur;
                const int at = s * kSlotStride + slot_col(lane, s);
                sgp[at] = gP;
                swg[at] = wgt;
            };
            auto pair = [&](int i1, int s) {
                BwdPair e1 = bwd_pair(B, L[i1], pxf, pyf, dC0, dC1, dC2, dD);
                BwdPair e0 = bwd_pair(B, L[i1 - 1], pxf, pyf, dC0, dC1, dC2, dD);
                bwd_refine(B, e1, e0);
                bwd_finish(e1, lim);
                bwd_finish(e0, lim);
                step(e1, s);
                step(e0, s + 1);
            };
            int i = nl - 1;
            // whole groups of kSlots entries, slot indices fixed at compile time
            for (; i >= kSlots - 1; i -= kSlots) {
#pragma unroll
                for (int p = 0; p < kSlots; p += 2) pair(i - p, p);
                __syncwarp();
                slots_reduce(sgp, swg, sdcd, kSlots, lane, L, i, B, cxw, cyw, s_grad);
                __syncwarp();
            }
            // the last (fewer than kSlots) entries
            const int i0 = i;      // list position of slot 0's entry
            int slot = 0;          // entries in the slot buffers (warp-uniform)
            for (; i >= 1; i -= 2, slot += 2) pair(i, slot);
            if (i == 0) {
                BwdPair e = bwd_pair(B, L[0], pxf, pyf, dC0, dC1, dC2, dD);
                if (__any_sync(0xffffffffu, e.near) && e.near) e.sa = __fmul_rn(B[3 * e.k + 1].y, exp2_nonpos(e.P2m));
                bwd_finish(e, lim);
                step(e, slot);
                ++slot;
            }
            if (slot) {
                __syncwarp();
                slots_reduce(sgp, swg, sdcd, slot, lane, L, i0, B, cxw, cyw, s_grad);
                __syncwarp();
            }
            __syncthreads();
            for (int t = tid; t < cnt; t += kBlendThreads) {
                float* sg = s_grad + t * kSumStride;
                // sums of gP dx, gP dy -> d(u, v); gP dx^2, gP dx dy, gP dy^2 -> d(qa, qb, qc)
                const float4 q0 = B[3 * t];
                const float qc = B[3 * t + 1].x, sig = B[3 * t + 1].y;
                const float sx = sg[0], sy = sg[1];
                const float4 v0 = make_float4(-GSR_LN2 * (2.0f * q0.z * sx + q0.w * sy),
                                              -GSR_LN2 * (q0.w * sx + 2.0f * qc * sy), GSR_LN2 * sg[2],
                                              GSR_LN2 * sg[3]);
                // sum dL/dalpha G over the pixels where alpha is not clamped = sum gP / sigma
                const float4 v1 = make_float4(GSR_LN2 * sg[4], sg[5] / sig, sg[6], 0.0f);
                const float4 v2 = make_float4(sg[7], sg[8], sg[9], 0.0f);
                const uint32_t k = s_idx[s][t];
                if (v0.x != 0.0f || v0.y != 0.0f || v0.z != 0.0f || v0.w != 0.0f || v1.x != 0.0f || v1.y != 0.0f ||
                    v1.z != 0.0f || v2.x != 0.0f || v2.y != 0.0f || v2.z != 0.0f) {
                    atomicAdd(a.grad_rec + 3 * (size_t)k, v0);
                    atomicAdd(a.grad_rec + 3 * (size_t)k + 1, v1);
                    atomicAdd(a.grad_rec + 3 * (size_t)k + 2, v2);
                }
#pragma unroll
                for (int c = 0; c < 10; ++c) sg[c] = 0.0f;
            }
        }
        __syncthreads();   // every thread has read s_item / s_maxlast of this tile; the flush is done
    }
    pairs_total = warp_sum(pairs_total);
    if (lane == 0 && pairs_total) atomicAdd(a.counters + kCntBwdPairs, pairs_total);
    if (lane == 0 && witer) atomicAdd(a.counters + kCntWarpBwd, witer);
}

// ---------------------------------------------------------------------------
// dispatch
// ---------------------------------------------------------------------------
template <int BX, int BY, int BATCH, bool COUNT>
static void fwd_tile_launch(const Table& T, const BlendFwdArgs& a, int num_sms, cudaStream_t s)
{
    auto kern = blend_fwd_tile_kernel<BX, BY, BATCH, COUNT>;
    const size_t smem = (size_t)2 * BATCH * kRecordBytes;
    // function attributes and occupancy are per device
    static std::atomic<int> per_sm_dev[kMaxDevices];
    const int per_sm = per_device_once(per_sm_dev, [&] {
        int n = 0;
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kern, kBlendThreads, smem);
        return n < 1 ? 1 : n;
    });
    int64_t grid = (int64_t)num_sms * per_sm;
    if (grid > T.n_tiles) grid = T.n_tiles;
    if (grid < 1) return;
    GSR_COUNT_LAUNCH();
    kern<<<(unsigned)grid, kBlendThreads, smem, s>>>(T, a);
}

template <int BX, int BY, int BATCH>
static void fwd_tile_one(const Table& T, const BlendFwdArgs& a, int num_sms, cudaStream_t s)
{
    if (a.count_pairs) fwd_tile_launch<BX, BY, BATCH, true>(T, a, num_sms, s);
    else fwd_tile_launch<BX, BY, BATCH, false>(T, a, num_sms, s);
}

// Blocks of the warp form resident on the device.
template <int BX, bool COUNT>
static int fwd_warp_resident(int num_sms)
{
    static std::atomic<int> per_sm_dev[kMaxDevices];
    return num_sms * per_device_once(per_sm_dev, [&] {
        int n = 0;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, blend_fwd_warp_kernel<BX, COUNT>, kFwdThreads, 0);
        return n < 1 ? 1 : n;
    });
}

template <int BX, bool COUNT>
static void fwd_warp_launch(const Table& T, const BlendFwdArgs& a, int num_sms, cudaStream_t s)
{
    const int64_t grid = std::min<int64_t>(fwd_warp_resident<BX, COUNT>(num_sms), T.n_tiles);
    GSR_COUNT_LAUNCH();
    blend_fwd_warp_kernel<BX, COUNT><<<(unsigned)grid, kFwdThreads, 0, s>>>(T, a);
}

template <int BX>
static void fwd_warp_one(const Table& T, const BlendFwdArgs& a, int num_sms, cudaStream_t s)
{
    if (a.count_pairs) fwd_warp_launch<BX, true>(T, a, num_sms, s);
    else fwd_warp_launch<BX, false>(T, a, num_sms, s);
}

template <int BX, int BY, int BATCH>
static void bwd_one(const Table& T, const BlendBwdArgs& a, int num_sms, cudaStream_t s)
{
    auto kern = blend_bwd_kernel<BX, BY, BATCH>;
    const size_t smem = bwd_smem_bytes<BATCH>();
    // function attributes and occupancy are per device
    static std::atomic<int> per_sm_dev[kMaxDevices];
    const int per_sm = per_device_once(per_sm_dev, [&] {
        int n = 0;
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        // all of the unified L1 as shared memory: four blocks of the
        // 128-record variant fit (the kernel keeps records in shared memory,
        // not in L1)
        cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, (int)cudaSharedmemCarveoutMaxShared);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kern, kBlendThreads, smem);
        return n < 1 ? 1 : n;
    });
    int64_t grid = (int64_t)num_sms * per_sm;
    if (grid > T.n_tiles) grid = T.n_tiles;
    if (grid < 1) return;
    GSR_COUNT_LAUNCH();
    kern<<<(unsigned)grid, kBlendThreads, smem, s>>>(T, a);
}

bool blend_supported(int tw, int th, int batch)
{
    const bool shape = (tw == 16 && th == 16) || (tw == 32 && th == 8) || (tw == 8 && th == 32);
    const bool b = batch == 128 || batch == 256 || batch == 512;
    return shape && b;
}

#define GSR_DISPATCH(FN, T, batch, ...)                                                          \
    do {                                                                                         \
        const int tw_ = (T).tile_w, th_ = (T).tile_h;                                            \
        if (tw_ == 16 && th_ == 16) {                                                            \
            if (batch == 128) FN<16, 16, 128>(T, __VA_ARGS__);                                   \
            else if (batch == 256) FN<16, 16, 256>(T, __VA_ARGS__);                              \
            else FN<16, 16, 512>(T, __VA_ARGS__);                                                \
        } else if (tw_ == 32 && th_ == 8) {                                                      \
            if (batch == 128) FN<32, 8, 128>(T, __VA_ARGS__);                                    \
            else if (batch == 256) FN<32, 8, 256>(T, __VA_ARGS__);                               \
            else FN<32, 8, 512>(T, __VA_ARGS__);                                                 \
        } else {                                                                                 \
            if (batch == 128) FN<8, 32, 128>(T, __VA_ARGS__);                                    \
            else if (batch == 256) FN<8, 32, 256>(T, __VA_ARGS__);                               \
            else FN<8, 32, 512>(T, __VA_ARGS__);                                                 \
        }                                                                                        \
    } while (0)

int blend_fwd_list_parts(const Table& T, bool count_pairs, int num_sms)
{
    if (T.n_tiles < kWarpFormMinTiles) return 0;
    const int resident = T.tile_w == 16 ? (count_pairs ? fwd_warp_resident<16, true>(num_sms) : fwd_warp_resident<16, false>(num_sms))
                       : T.tile_w == 32 ? (count_pairs ? fwd_warp_resident<32, true>(num_sms) : fwd_warp_resident<32, false>(num_sms))
                                        : (count_pairs ? fwd_warp_resident<8, true>(num_sms) : fwd_warp_resident<8, false>(num_sms));
    return (int)(kWarpFormShare * resident);
}

// Both forms are launched where the warp form may be taken; the lists decide on
// the device which of the two returns at once (a second round of two takes the
// first one's form).
void launch_blend_fwd(const Table& T, int batch, BlendFwdArgs a, int num_sms, cudaStream_t s)
{
    a.stat_batch = (uint32_t)batch;
    if (a.long_list) {
        if (T.tile_w == 16) fwd_warp_one<16>(T, a, num_sms, s);
        else if (T.tile_w == 32) fwd_warp_one<32>(T, a, num_sms, s);
        else fwd_warp_one<8>(T, a, num_sms, s);
    }
    GSR_DISPATCH(fwd_tile_one, T, batch, a, num_sms, s);
}

size_t blend_mask_bytes(int64_t list_span, int64_t n_tiles)
{
    return ((size_t)(list_span / kChunk) + 2 * (size_t)n_tiles + 1) * kMaskWords * sizeof(uint32_t);
}

void launch_blend_bwd(const Table& T, int batch, const BlendBwdArgs& a, int num_sms, cudaStream_t s)
{
    GSR_DISPATCH(bwd_one, T, batch, a, num_sms, s);
}

}  // namespace gsr
