// gsr_freq.cu -- frequency-based scheduling (Sec. 3.3, Eq. 9-12) for a batch
// of images.
//
//   X(I) = sum over frequencies (i, j) of || DFT(I)(i, j) ||_2     (Eq. 10, 11)
//
// the unnormalised 2-D DFT of each colour channel, the norm taken over the
// three channels at each frequency.  Then r = X(I) / X(I~) (Eq. 9) weights
// the frames drawn for optimisation and r' = X(I^n) / X(I~) (Eq. 12), I^n the
// ground truth at downsampling factor n, raises the level when below tau_f.
//
// The DFT is a mixed-radix Stockham transform in as few passes as the composite
// radices 16, 15, 12, 10, 9, 8, 6, 5, 4, 3, 2 give (1600 = 16 10 10, 900 = 10 10
// 9), after a direct pass for each other prime, in two passes over each image:
//   rows     two real rows of a channel packed as one complex sequence; after
//            the transform the Hermitian split gives both rows' spectra for
//            k = 0 .. W/2 (the other half is their conjugate mirror), written
//            to a half-spectrum buffer [3][H][W/2 + 1];
//   columns  C adjacent columns of that buffer, one channel after the other,
//            transformed along y; |F_c|^2 summed over the channels in shared
//            memory, then sqrt and summed with weight 2 for the columns whose
//            mirror k' = W - k is not stored (1 for k = 0 and k = W/2).
// The first pass of a transform loads from memory, the last one of a column
// adds |F_c|^2, so only the passes between them go through shared memory.
// Box downsampling (I^n) is applied while loading the rows.  Values are FP32
// (twiddles from a host table computed in double); the magnitudes are summed
// per thread in FP32 and across threads and blocks in FP64.
//
// Bound by latency: barriers and the index arithmetic around them (issue slots
// 49-55 %, DRAM 14-25 %).  Against radix-4, 2, 3 and 5 passes (five for 1600 and
// 900) with separate load and magnitude steps, a direct pass per output and four
// columns per item whatever the image: 18 images of 1600 x 900 columns 282 ->
// 200 us, rows 246 -> 249; nine images of 333 x 251 and smaller (prime heights)
// columns 122 -> 44 us.  The radix-16 passes need the padding (rows 296 us
// without).
#include <algorithm>
#include <cmath>
#include <vector>

#include "gsr_common.cuh"
#include "gsr_kernels.h"

namespace gsr {

// Largest blocks; a launch takes as many threads as its largest pass has
// butterflies (whole warps), so that a pass is one round where it can be.
constexpr int kRowThreads = 512;
constexpr int kColThreads = 512;

static uint32_t recip32(int d) { return d <= 1 ? 0u : (uint32_t)((((uint64_t)1 << 32) + (uint64_t)d - 1) / (uint64_t)d); }

// The fewest passes over the composite radices for n = 2^a 3^b 5^c (ties to the
// larger first radix), by the exponents; false if a pass more than
// 2 kFftMaxStages were needed.
static bool fft_radices(int n, int* radix, int& k)
{
    static constexpr struct { int r, e[3]; } kRadix[] = {
        {16, {4, 0, 0}}, {15, {0, 1, 1}}, {12, {2, 1, 0}}, {10, {1, 0, 1}}, {9, {0, 2, 0}}, {8, {3, 0, 0}},
        {6, {1, 1, 0}}, {5, {0, 0, 1}}, {4, {2, 0, 0}}, {3, {0, 1, 0}}, {2, {1, 0, 0}}};
    int e[3] = {0, 0, 0};
    const int base[3] = {2, 3, 5};
    for (int i = 0; i < 3; ++i)
        while (n % base[i] == 0) { n /= base[i]; ++e[i]; }
    if (n != 1) return false;
    // best[x]: passes of 2^x0 3^x1 5^x2 and the first one's radix
    struct Best { int passes, first; };
    const int ny = e[1] + 1, nz = e[2] + 1;
    std::vector<Best> best((size_t)(e[0] + 1) * ny * nz, Best{0, -1});
    auto at = [&](int x, int y, int z) -> Best& { return best[((size_t)x * ny + y) * nz + z]; };
    for (int x = 0; x <= e[0]; ++x)
        for (int y = 0; y <= e[1]; ++y)
            for (int z = 0; z <= e[2]; ++z) {
                if (x + y + z == 0) continue;
                Best& b = at(x, y, z);
                b.passes = 1 << 20;
                for (int i = 0; i < (int)(sizeof(kRadix) / sizeof(kRadix[0])); ++i) {
                    const int* r = kRadix[i].e;
                    if (r[0] > x || r[1] > y || r[2] > z) continue;
                    const int p = 1 + at(x - r[0], y - r[1], z - r[2]).passes;
                    if (p < b.passes) b = Best{p, i};
                }
            }
    if (at(e[0], e[1], e[2]).passes > 2 * kFftMaxStages) return false;
    for (k = 0; e[0] + e[1] + e[2] > 0;) {
        const auto& r = kRadix[at(e[0], e[1], e[2]).first];
        radix[k++] = r.r;
        for (int i = 0; i < 3; ++i) e[i] -= r.e[i];
    }
    return true;
}

bool fft_plan(int n, FftPlan* P)
{
    if (n < 1 || n > kFreqMaxDim) return false;
    int radix[2 * kFftMaxStages];
    int k = 0, rest = n;
    for (int p : {2, 3, 5})
        while (rest % p == 0) rest /= p;
    const int smooth = n / rest;
    // other primes first: their direct pass then needs no twiddles
    for (int p = 7; rest > 1 && k < kFftMaxStages; p += 2)
        while (rest % p == 0 && k < kFftMaxStages) { radix[k++] = p; rest /= p; }
    int ks = 0, rs[2 * kFftMaxStages];
    if (rest != 1 || !fft_radices(smooth, rs, ks) || k + ks > kFftMaxStages) return false;
    for (int i = 0; i < ks; ++i) radix[k++] = rs[i];
    P->n = n;
    P->n_stages = k;
    int Ns = 1;
    for (int i = 0; i < k; ++i) {
        FftStage& S = P->st[i];
        S.R = radix[i]; S.Ns = Ns; S.m = n / S.R; S.step = n / (Ns * S.R);
        S.mag_m = recip32(S.m); S.mag_ns = recip32(Ns);
        Ns *= S.R;
    }
    return true;
}

// x / d for x < 2^16, d < 2^16, by the reciprocal ceil(2^32 / d) (0 for d = 1)
__device__ __forceinline__ int udiv16(int x, uint32_t mag) { return mag ? (int)__umulhi((uint32_t)x, mag) : x; }

__device__ __forceinline__ float2 cmul(float2 a, float2 b)
{
    return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 csub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ float2 mul_ni(float2 a) { return make_float2(a.y, -a.x); }   // -i a

// R-point forward DFTs, y_q = sum_r v_r exp(-2 pi i q r / R), in place.
template <int R> __device__ __forceinline__ void butterfly(float2* v);

template <> __device__ __forceinline__ void butterfly<2>(float2* v)
{
    const float2 a = v[0], b = v[1];
    v[0] = cadd(a, b); v[1] = csub(a, b);
}

template <> __device__ __forceinline__ void butterfly<4>(float2* v)
{
    const float2 t0 = cadd(v[0], v[2]), t1 = csub(v[0], v[2]);
    const float2 t2 = cadd(v[1], v[3]), t3 = mul_ni(csub(v[1], v[3]));
    v[0] = cadd(t0, t2); v[2] = csub(t0, t2);
    v[1] = cadd(t1, t3); v[3] = csub(t1, t3);
}

template <> __device__ __forceinline__ void butterfly<3>(float2* v)
{
    constexpr float h = 0.8660254037844386f;   // sin(2 pi / 3)
    const float2 s = cadd(v[1], v[2]), d = csub(v[1], v[2]);
    const float2 m = make_float2(v[0].x - 0.5f * s.x, v[0].y - 0.5f * s.y);
    const float2 rot = mul_ni(make_float2(h * d.x, h * d.y));   // -i sin(2 pi/3) d
    v[0] = cadd(v[0], s);
    v[1] = cadd(m, rot);
    v[2] = csub(m, rot);
}

template <> __device__ __forceinline__ void butterfly<5>(float2* v)
{
    constexpr float c1 = 0.30901699437494745f, c2 = -0.8090169943749475f;   // cos(2 pi k / 5), k = 1, 2
    constexpr float s1 = 0.9510565162951535f, s2 = 0.5877852522924731f;     // sin(2 pi k / 5)
    const float2 a0 = v[0];
    const float2 p1 = cadd(v[1], v[4]), d1 = csub(v[1], v[4]);
    const float2 p2 = cadd(v[2], v[3]), d2 = csub(v[2], v[3]);
    const float2 m1 = make_float2(a0.x + c1 * p1.x + c2 * p2.x, a0.y + c1 * p1.y + c2 * p2.y);
    const float2 m2 = make_float2(a0.x + c2 * p1.x + c1 * p2.x, a0.y + c2 * p1.y + c1 * p2.y);
    const float2 r1 = mul_ni(make_float2(s1 * d1.x + s2 * d2.x, s1 * d1.y + s2 * d2.y));
    const float2 r2 = mul_ni(make_float2(s2 * d1.x - s1 * d2.x, s2 * d1.y - s1 * d2.y));
    v[0] = cadd(a0, cadd(p1, p2));
    v[1] = cadd(m1, r1); v[4] = csub(m1, r1);
    v[2] = cadd(m2, r2); v[3] = csub(m2, r2);
}

// cos and sin of 2 pi t / N for t < N, rounded once (series in double, at
// compile time).
template <int N>
struct UnitRoots {
    float c[N], s[N];
    constexpr UnitRoots() : c(), s()
    {
        for (int t = 0; t < N; ++t) {
            // angle folded into [-pi, pi]
            const double x = 2.0 * 3.14159265358979323846 * (double)(2 * t > N ? t - N : t) / (double)N;
            double tc = 1.0, ts = x, sc = 1.0, ss = x;
            for (int i = 1; i < 20; ++i) {
                tc *= -x * x / (double)((2 * i - 1) * (2 * i));
                ts *= -x * x / (double)((2 * i) * (2 * i + 1));
                sc += tc;
                ss += ts;
            }
            c[t] = (float)sc;
            s[t] = (float)ss;
        }
    }
};

// N1 N2-point DFT from N1- and N2-point ones: input n = N2 n1 + n2, output
// k = k1 + N1 k2, twiddles W_N^(n2 k1) between the two.
template <int N1, int N2>
__device__ __forceinline__ void dft_composite(float2* v)
{
    constexpr int N = N1 * N2;
    constexpr UnitRoots<N> w;
    float2 t[N];
#pragma unroll
    for (int n2 = 0; n2 < N2; ++n2) {
        float2 u[N1];
#pragma unroll
        for (int n1 = 0; n1 < N1; ++n1) u[n1] = v[N2 * n1 + n2];
        butterfly<N1>(u);
#pragma unroll
        for (int k1 = 0; k1 < N1; ++k1) {
            const int e = n2 * k1;
            t[N2 * k1 + n2] = e == 0 ? u[k1] : cmul(u[k1], make_float2(w.c[e], -w.s[e]));
        }
    }
#pragma unroll
    for (int k1 = 0; k1 < N1; ++k1) {
        butterfly<N2>(t + N2 * k1);
#pragma unroll
        for (int k2 = 0; k2 < N2; ++k2) v[k1 + N1 * k2] = t[N2 * k1 + k2];
    }
}
template <> __device__ __forceinline__ void butterfly<6>(float2* v) { dft_composite<2, 3>(v); }
template <> __device__ __forceinline__ void butterfly<8>(float2* v) { dft_composite<2, 4>(v); }
template <> __device__ __forceinline__ void butterfly<9>(float2* v) { dft_composite<3, 3>(v); }
template <> __device__ __forceinline__ void butterfly<10>(float2* v) { dft_composite<2, 5>(v); }
template <> __device__ __forceinline__ void butterfly<12>(float2* v) { dft_composite<3, 4>(v); }
template <> __device__ __forceinline__ void butterfly<15>(float2* v) { dft_composite<3, 5>(v); }
template <> __device__ __forceinline__ void butterfly<16>(float2* v) { dft_composite<4, 4>(v); }

// Where element i of a sequence lies in its shared-memory buffer: one place of
// padding per 16, because the first pass of radix 16 writes at a stride of 16
// (the row pass takes 296 us without, 249 with).
__device__ __forceinline__ int fft_at(int i) { return i + (i >> 4); }
// (fft_span(n), the length of such a buffer, is in gsr_kernels.h)

// One Stockham pass over nseq sequences of length n.  Butterfly j (of
// m = n / R) of sequence s takes its inputs from load(s, j + r m), r < R,
// twiddled by W_{Ns R}^{r (j mod Ns)}, and gives its R outputs to
// store(s, (j - j mod Ns) R + j mod Ns + q Ns, value), q < R; Ns is the product
// of the radices of the earlier passes.  One twiddle is loaded per butterfly,
// its powers formed by complex products w^(2i) = w^i w^i, w^(2i+1) = w^(2i) w.
// Consecutive threads take consecutive sequences if SEQ_FAST (the columns,
// adjacent in memory), else consecutive butterflies.
template <int R, bool SEQ_FAST, typename Load, typename Store>
__device__ __forceinline__ void fft_pass(int nseq, const FftStage& S, const float2* __restrict__ tw, Load load, Store store)
{
    const int m = S.m, Ns = S.Ns, step = S.step;
    const uint32_t mag_m = S.mag_m, mag_ns = S.mag_ns;
    for (int t = threadIdx.x; t < nseq * m; t += blockDim.x) {
        int s, j;
        if (SEQ_FAST) { j = t / nseq; s = t - j * nseq; }
        else { s = udiv16(t, mag_m); j = t - s * m; }
        const int jb = udiv16(j, mag_ns), jm = j - jb * Ns;
        float2 v[R];
#pragma unroll
        for (int r = 0; r < R; ++r) v[r] = load(s, j + r * m);
        if (jm != 0) {
            float2 w[R];
            w[1] = __ldg(tw + jm * step);
#pragma unroll
            for (int r = 2; r < R; ++r) w[r] = (r & 1) ? cmul(w[r - 1], w[1]) : cmul(w[r / 2], w[r / 2]);
#pragma unroll
            for (int r = 1; r < R; ++r) v[r] = cmul(v[r], w[r]);
        }
        butterfly<R>(v);
        const int o = jb * Ns * R + jm;
#pragma unroll
        for (int q = 0; q < R; ++q) store(s, o + q * Ns, v[q]);
    }
}

// The same pass for a prime radix R > 5, the R-point DFT by its definition
// with the outputs q and R - q taken together: from s_r = x_r + x_{R-r} and
// d_r = x_r - x_{R-r} (x the twiddled inputs, r <= h = (R - 1) / 2),
//   X_q, X_{R-q} = x_0 + sum_r s_r cos(2 pi q r / R) -+ i sum_r d_r sin(2 pi q r / R),
// a quarter of the products of the separate sums.  a holds the sequences
// (stored back to back) and is overwritten with s and d.
template <typename Store>
__device__ void fft_pass_prime(float2* __restrict__ a, int nseq, int n, const FftStage& S, const float2* __restrict__ tw,
                               Store store)
{
    const int R = S.R, m = S.m, Ns = S.Ns, step = S.step, h = (R - 1) / 2, root = n / R;
    const int per = h * m, per_out = (h + 1) * m;
    for (int t = threadIdx.x; t < nseq * per; t += blockDim.x) {
        const int s = t / per, u = t - s * per;
        const int r = u / m + 1, j = u - (r - 1) * m;
        const int jb = udiv16(j, S.mag_ns), jm = j - jb * Ns;
        float2* x = a + s * fft_span(n);
        float2 &xp = x[fft_at(j + r * m)], &xq = x[fft_at(j + (R - r) * m)];
        float2 p = xp, q = xq;
        if (jm != 0) {
            p = cmul(p, __ldg(tw + r * jm * step));
            q = cmul(q, __ldg(tw + (R - r) * jm * step));
        }
        xp = cadd(p, q);
        xq = csub(p, q);
    }
    __syncthreads();
    for (int t = threadIdx.x; t < nseq * per_out; t += blockDim.x) {
        const int s = t / per_out, u = t - s * per_out;
        const int q = u / m, j = u - q * m;
        const int jb = udiv16(j, S.mag_ns), jm = j - jb * Ns;
        const float2* x = a + s * fft_span(n);
        const float2 x0 = x[fft_at(j)];
        float2 c = x0, d = make_float2(0.0f, 0.0f);
        int idx = 0;
#pragma unroll 4
        for (int r = 1; r <= h; ++r) {
            idx += q;
            if (idx >= R) idx -= R;
            const float2 w = __ldg(tw + idx * root);   // cos, -sin
            const float2 sr = x[fft_at(j + r * m)], dr = x[fft_at(j + (R - r) * m)];
            c.x = fmaf(sr.x, w.x, c.x);
            c.y = fmaf(sr.y, w.x, c.y);
            d.x = fmaf(dr.y, -w.y, d.x);    // -i d sin
            d.y = fmaf(dr.x, w.y, d.y);
        }
        const int o = jb * Ns * R + jm;
        store(s, o + q * Ns, cadd(c, d));
        if (q > 0) store(s, o + (R - q) * Ns, csub(c, d));
    }
}

// Pass st of plan P over nseq sequences.  A prime pass reads from `a` (first
// filled through load if it is the plan's first pass).
template <bool SEQ_FAST, typename Load, typename Store>
__device__ __forceinline__ void fft_stage(const FftPlan& P, int st, int nseq, float2* a, Load load, Store store)
{
    const FftStage& S = P.st[st];
    switch (S.R) {
    case 16: fft_pass<16, SEQ_FAST>(nseq, S, P.tw, load, store); break;
    case 15: fft_pass<15, SEQ_FAST>(nseq, S, P.tw, load, store); break;
    case 12: fft_pass<12, SEQ_FAST>(nseq, S, P.tw, load, store); break;
    case 10: fft_pass<10, SEQ_FAST>(nseq, S, P.tw, load, store); break;
    case 9: fft_pass<9, SEQ_FAST>(nseq, S, P.tw, load, store); break;
    case 8: fft_pass<8, SEQ_FAST>(nseq, S, P.tw, load, store); break;
    case 6: fft_pass<6, SEQ_FAST>(nseq, S, P.tw, load, store); break;
    case 5: fft_pass<5, SEQ_FAST>(nseq, S, P.tw, load, store); break;
    case 4: fft_pass<4, SEQ_FAST>(nseq, S, P.tw, load, store); break;
    case 3: fft_pass<3, SEQ_FAST>(nseq, S, P.tw, load, store); break;
    case 2: fft_pass<2, SEQ_FAST>(nseq, S, P.tw, load, store); break;
    default:
        if (st == 0) {
            for (int t = threadIdx.x; t < nseq * P.n; t += blockDim.x) {
                const int x = SEQ_FAST ? t / nseq : t % P.n, s = SEQ_FAST ? t - x * nseq : t / P.n;
                a[s * fft_span(P.n) + fft_at(x)] = load(s, x);
            }
            __syncthreads();
        }
        fft_pass_prime(a, nseq, P.n, S, P.tw, store);
        break;
    }
    __syncthreads();
}

// Transform nseq sequences: the first pass takes its inputs through load, the
// last gives its outputs to store, the ones between run in shared memory (a and
// b, nseq fft_span(n) places each).  All threads of the block call it; it ends with a
// barrier.
template <bool SEQ_FAST, typename Load, typename Store>
__device__ __forceinline__ void fft_run(const FftPlan& P, int nseq, float2* a, float2* b, Load load, Store store)
{
    const int n = fft_span(P.n), last = P.n_stages - 1;
    if (last < 0) {   // length 1
        for (int s = threadIdx.x; s < nseq; s += blockDim.x) store(s, 0, load(s, 0));
        __syncthreads();
        return;
    }
    if (last == 0) {
        fft_stage<SEQ_FAST>(P, 0, nseq, a, load, store);
        return;
    }
    // (a prime first pass stages its inputs in a, so its outputs go to b)
    fft_stage<SEQ_FAST>(P, 0, nseq, a, load, [=](int s, int i, float2 v) { b[s * n + fft_at(i)] = v; });
    float2 *src = b, *dst = a;
    for (int st = 1; st < last; ++st) {
        float2 *from = src, *to = dst;
        fft_stage<false>(P, st, nseq, from, [=](int s, int i) { return from[s * n + fft_at(i)]; },
                         [=](int s, int i, float2 v) { to[s * n + fft_at(i)] = v; });
        src = to;
        dst = from;
    }
    float2* from = src;
    fft_stage<false>(P, last, nseq, from, [=](int s, int i) { return from[s * n + fft_at(i)]; }, store);
}

__device__ __forceinline__ int image_of(const FreqTable& T, int64_t item, bool rows)
{
    int lo = 0, hi = T.n_images - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        const int64_t base = rows ? T.img[mid].row_base : T.img[mid].col_base;
        if (base <= item) lo = mid; else hi = mid - 1;
    }
    return lo;
}

// Row pass: item = (image, row pair, group of I.RC channels).  Rows y0 = 2p and
// y0 + 1 of a channel (box-averaged over factor x factor source pixels) are the
// real and imaginary parts of one sequence Z; their spectra are
// A(k) = (Z(k) + conj Z(-k)) / 2 and B(k) = (Z(k) - conj Z(-k)) / (2i).
__global__ void __launch_bounds__(kRowThreads, 2)
dft_rows_kernel(const __grid_constant__ FreqTable T, float2* __restrict__ inter)
{
    extern __shared__ float2 sm[];   // two buffers of the group's rows
    for (int64_t item = blockIdx.x; item < T.row_items; item += gridDim.x) {
        const FreqImage& I = T.img[image_of(T, item, true)];
        const int64_t local = item - I.row_base;
        const int RC = I.RC, per = 3 / RC;
        const int c0 = (int)(local % per) * RC, y0 = 2 * (int)(local / per);
        const int Wd = I.Wd, f = I.factor;
        const int64_t W = I.W, hw = (int64_t)I.H * I.W;
        const bool two = y0 + 1 < I.Hd;
        const float* __restrict__ r0 = I.src + c0 * hw + (int64_t)y0 * f * W;
        const FftPlan& P = T.plan[I.row_plan];
        const int span = fft_span(Wd);
        float2 *a = sm, *b = sm + RC * span;
        // the last pass reads the buffer its predecessor wrote (b, a, b, ...) and
        // writes the other; a single pass writes b
        float2* z = (P.n_stages & 1) ? b : a;
        if (f != 1) {
            // the means of f x f source pixels, staged in a
            const float inv = 1.0f / (float)(f * f);
            for (int t = threadIdx.x; t < RC * Wd; t += blockDim.x) {
                const int c = t / Wd, x = t - c * Wd;
                float p0 = 0.0f, p1 = 0.0f;
                for (int dy = 0; dy < f; ++dy) {
                    const float* q = r0 + c * hw + dy * W + (int64_t)x * f;
                    for (int dx = 0; dx < f; ++dx) p0 += __ldg(q + dx);
                    if (two)
                        for (int dx = 0; dx < f; ++dx) p1 += __ldg(q + (int64_t)f * W + dx);
                }
                a[c * span + fft_at(x)] = make_float2(p0 * inv, p1 * inv);
            }
            __syncthreads();
        }
        fft_run<false>(P, RC, a, b,
                       [=](int c, int x) {
                           if (f != 1) return a[c * span + fft_at(x)];
                           const float* q = r0 + c * hw + x;
                           return make_float2(__ldg(q), two ? __ldg(q + W) : 0.0f);
                       },
                       [=](int c, int k, float2 v) { z[c * span + fft_at(k)] = v; });
        for (int c = 0; c < RC; ++c) {
            float2* o = inter + I.inter + ((int64_t)(c0 + c) * I.Hd + y0) * I.Wh;
            const float2* zc = z + c * span;
            for (int k = threadIdx.x; k < I.Wh; k += blockDim.x) {
                const float2 z1 = zc[fft_at(k)], z2 = zc[fft_at(k == 0 ? 0 : Wd - k)];
                o[k] = make_float2(0.5f * (z1.x + z2.x), 0.5f * (z1.y - z2.y));
                if (two) o[I.Wh + k] = make_float2(0.5f * (z1.y + z2.y), 0.5f * (z2.x - z1.x));
            }
        }
        __syncthreads();   // the buffers are rewritten by the next item
    }
}

// Column pass: item = (image, C adjacent half-spectrum columns).  Shared
// memory: two C x Hd complex buffers and C x Hd floats of sum_c |F_c|^2.
__global__ void __launch_bounds__(kColThreads, 2)
dft_cols_kernel(const __grid_constant__ FreqTable T, const float2* __restrict__ inter, double* __restrict__ xacc)
{
    extern __shared__ float2 sm[];
    __shared__ double s_red[kColThreads / 32];
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    for (int64_t item = blockIdx.x; item < T.col_items; item += gridDim.x) {
        const int ii = image_of(T, item, false);
        const FreqImage& I = T.img[ii];
        const int Hd = I.Hd, Wh = I.Wh;
        const int k0 = (int)(item - I.col_base) * I.C;
        const int nc = min(I.C, Wh - k0), ne = nc * Hd;
        float2* a = sm;
        float2* b = sm + I.C * fft_span(Hd);
        float* acc = reinterpret_cast<float*>(sm + 2 * I.C * fft_span(Hd));
        for (int e = tid; e < ne; e += blockDim.x) acc[e] = 0.0f;
        __syncthreads();
        for (int c = 0; c < 3; ++c) {
            // the last pass adds |F_c|^2 where a thread's butterflies put their
            // outputs, the same places for every channel
            const float2* __restrict__ plane = inter + I.inter + (int64_t)c * Hd * Wh + k0;
            fft_run<true>(T.plan[I.col_plan], nc, a, b, [=](int kk, int y) { return __ldg(plane + (int64_t)y * Wh + kk); },
                          [=](int kk, int y, float2 v) { acc[kk * Hd + y] += v.x * v.x + v.y * v.y; });
        }
        float part = 0.0f;
        for (int q = 0; q < nc; ++q) {
            const int k = k0 + q;
            const float w = (k == 0 || 2 * k == I.Wd) ? 1.0f : 2.0f;
            float sq = 0.0f;
            for (int y = tid; y < Hd; y += blockDim.x) sq += sqrtf(acc[q * Hd + y]);
            part += w * sq;
        }
        double d = (double)part;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) d += __shfl_xor_sync(0xffffffffu, d, o);
        if (lane == 0) s_red[wid] = d;
        __syncthreads();
        if (tid == 0) {
            double s = 0.0;
            for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += s_red[w];
            atomicAdd(xacc + ii, s);
        }
        __syncthreads();   // s_red and the buffers are rewritten by the next item
    }
}

__global__ void dft_finalize_kernel(const double* __restrict__ xacc, float* __restrict__ x, int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) x[i] = (float)xacc[i];
}

// Scheduler decisions in binary32 (one block): r = x_gt / x_rendered,
// r' = x_gt_level / x_rendered, level-up iff r' < tau_f; frame weights r
// (NaN -> 0, capped at 1e30; all 1 if none is positive), cumulative sums in
// frame order, and for each uniform u the first frame whose cumulative weight
// exceeds u * total (else the last frame of positive weight).
__global__ void __launch_bounds__(256)
frequency_schedule_kernel(int n, const float* __restrict__ x_gt, const float* __restrict__ x_gl,
                          const float* __restrict__ x_r, float tau, const float* __restrict__ u, int ns,
                          float* __restrict__ r, float* __restrict__ rl, int32_t* __restrict__ up,
                          int32_t* __restrict__ samples)
{
    __shared__ float s_c[kFreqMaxFrames];
    __shared__ int s_last;
    const int tid = threadIdx.x;
    for (int f = tid; f < n; f += blockDim.x) {
        const float rv = __fdiv_rn(x_gt[f], x_r[f]);
        if (r) r[f] = rv;
        if (x_gl) {
            const float lv = __fdiv_rn(x_gl[f], x_r[f]);
            if (rl) rl[f] = lv;
            if (up) up[f] = lv < tau ? 1 : 0;
        }
        s_c[f] = isnan(rv) ? 0.0f : fminf(rv, 1e30f);
    }
    __syncthreads();
    if (tid == 0) {
        bool any = false;
        for (int f = 0; f < n; ++f) any = any || s_c[f] > 0.0f;
        float c = 0.0f;
        int last = -1;
        for (int f = 0; f < n; ++f) {
            const float w = any ? s_c[f] : 1.0f;
            if (w > 0.0f) last = f;
            c = __fadd_rn(c, w);
            s_c[f] = c;
        }
        s_last = last;
    }
    __syncthreads();
    if (!samples) return;
    const float total = s_c[n - 1];
    for (int k = tid; k < ns; k += blockDim.x) {
        const float t = __fmul_rn(u[k], total);
        int lo = 0, hi = n;   // first f with c_f > t (cumulative sums do not decrease)
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if (s_c[mid] > t) hi = mid; else lo = mid + 1;
        }
        samples[k] = lo < n ? lo : s_last;
    }
}

template <typename K>
static int resident_blocks(K kernel, int threads, int smem)
{
    int n = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kernel, threads, smem) != cudaSuccess || n < 1) n = 1;
    return n;
}

void launch_dft_energy(const FreqTable& T, float2* inter, double* xacc, int row_smem, int col_smem, int row_threads,
                       int col_threads, int num_sms, cudaStream_t s)
{
    static std::atomic<int> attr_set[kMaxDevices];
    per_device_once(attr_set, [] {
        cudaFuncSetAttribute(dft_rows_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 100 * 1024);
        cudaFuncSetAttribute(dft_cols_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 100 * 1024);
        return 1;
    });
    row_threads = std::min(kRowThreads, std::max(64, (row_threads + 31) / 32 * 32));
    col_threads = std::min(kColThreads, std::max(64, (col_threads + 31) / 32 * 32));
    if (T.row_items > 0) {
        int64_t grid = (int64_t)num_sms * resident_blocks(dft_rows_kernel, row_threads, row_smem);
        if (grid > T.row_items) grid = T.row_items;
        GSR_COUNT_LAUNCH();
        dft_rows_kernel<<<(unsigned)grid, row_threads, row_smem, s>>>(T, inter);
    }
    if (T.col_items > 0) {
        int64_t grid = (int64_t)num_sms * resident_blocks(dft_cols_kernel, col_threads, col_smem);
        if (grid > T.col_items) grid = T.col_items;
        GSR_COUNT_LAUNCH();
        dft_cols_kernel<<<(unsigned)grid, col_threads, col_smem, s>>>(T, inter, xacc);
    }
}

void launch_dft_finalize(const double* xacc, float* x, int n, cudaStream_t s)
{
    if (n <= 0) return;
    GSR_COUNT_LAUNCH();
    dft_finalize_kernel<<<(n + 255) / 256, 256, 0, s>>>(xacc, x, n);
}

void launch_frequency_schedule(int n_frames, const float* x_gt, const float* x_gt_level, const float* x_rendered,
                               float tau_f, const float* uniforms, int n_samples, float* r, float* r_level,
                               int32_t* level_up, int32_t* samples, cudaStream_t s)
{
    GSR_COUNT_LAUNCH();
    frequency_schedule_kernel<<<1, 256, 0, s>>>(n_frames, x_gt, x_gt_level, x_rendered, tau_f, uniforms, n_samples,
                                                r, r_level, level_up, samples);
}

}  // namespace gsr
