// FP32 FSR at S = 32 with a CTA of four or two warps on one support block, for
// calls with few blocks in flight: the 32 x 32 spectrum is spread over 128
// threads, 8 components each (or 64 threads, 16 each).
//
// What bounds it: the K iterations of a block are a serial chain (the argmax
// of Eq. (8) needs the residual of Eq. (12), which needs the last argmax), so
// such a call pays the latency of one iteration K times.  One warp per block
// (fsr_block.cuh) walks 32 components per lane in every iteration; here the
// update and the objective of a thread are 8 independent components, and one
// CTA barrier per iteration joins the warps' maxima.  Four warps have the
// shortest chain, two need fewer issue slots per block: which one a launch
// takes goes by its blocks per SM (fsr_launch.h).
//
// The arithmetic of every component, of both transforms, of the objective and
// of the target pixels is that of fsr_block.cuh operation by operation, and
// so is the selection rule: the results are the same bit for bit.
//
// Spectrum layout (four warps): warp w holds rows 8w .. 8w + 7, lane (r, g) of
// it the columns g, g + 4, g + 8, g + 12 of row 8w + r (r = lane / 4, g = lane %
// 4) and those 16 further on, as pairs for packed f32x2 operations.  A stored W
// row has 48 entries (Re W[c], Re W[c + 16], Im W[c], Im W[c + 16]) of 16 bytes;
// a quarter-warp reads 2 rows of 4 consecutive entries, which the row stride of
// 52 entries puts on distinct banks for every shift (u, v).  The rows are
// stored twice (64 of them), so the shifted entry W[k-u][l-v] of a thread is
// one subtraction away from a fixed address: no wrap of either index on the
// chain from the pick to the W loads.
//
// Measured (a block alone on an SM, cycles at 1.98 GHz): one iteration takes
// 1,130 with one warp per block, 385 with four: about 40 the W load, 50 the
// update, objective and maximum, 65 two warp reductions, 90 the barrier and the
// candidates through shared memory; the rest is issue.  What a thread may
// publish, and the target pixels of the previous pick, are computed while the
// reductions and loads run.  A branch in this chain costs 40 to 60 cycles even
// when every thread goes the same way, so the loop has none.  Scalar
// components instead of pairs: 457; 8 and 16 warps per block: 480-600.  With two
// warps and 8 CTAs per SM the 128 registers do not hold the DC phase's rows beside
// the state: 84 bytes are spilled (B = 16: up to 164), over one local load and store
// per warp and iteration.
//
// Transforms (four warps): the radix-2 decimation-in-time FFT of length 32
// splits over the warps.  Warp q takes the inputs of rows (columns) = brev2(q)
// mod 4, does
// the three stages inside its 8 points in registers, and after one exchange
// through shared memory the last two stages of the points t, t + 8, t + 16,
// t + 24 for t = 2q, 2q + 1.  A thread so runs about 200 instructions per
// transform where a lane of the one-warp kernel runs 1,200 of straight code,
// most of whose time a block that runs alone spends fetching instructions.
#pragma once

#include <type_traits>

#include "fsr_launch.h"

namespace fsrk {
namespace coop {

// Shape of the kernel with N warps per block.
template <int N>
struct Cfg {
    static_assert(N == 4 || N == 2, "4 or 2 warps per block");
    static constexpr int T = 32 * N;             // threads per block
    static constexpr int G = N;                  // lanes per row
    static constexpr int NP = S / G / 2;         // pairs (l, l + 16) per thread
    static constexpr int RPW = S / N;            // rows per warp
    static constexpr int WS = N == 4 ? 52 : 50;  // W row stride (16-byte entries)
    // 4 warps: rows stored twice, the shifted row is one subtraction away; 2
    // warps: once, so that 8 CTAs share an SM (28 KB, 128 registers)
    static constexpr bool TWICE = N == 4;
    static constexpr int MIN_CTAS = N == 4 ? 1 : 8;
    static constexpr int PTS = S / N;            // points of a transform per thread
    static constexpr int TT = PTS / N;           // groups of N points in its last stages
    static constexpr unsigned DIV = 65536 / WS + 1;   // off / WS = (off * DIV) >> 16 for off < S * WS
    static constexpr bool div_ok() {
        for (unsigned o = 0; o < (unsigned)(S * WS); ++o)
            if ((o * DIV) >> 16 != o / WS) return false;
        return true;
    }
};
static_assert(Cfg<4>::div_ok() && Cfg<2>::div_ok(), "division by multiplication");
constexpr int AS = S + 1;                // row stride of the transform buffers (float2)
constexpr int H1 = S / 2 + 1;            // w_f quadrant: indices 0 .. S/2

template <int N>
struct Smem {
    // the transforms' exchange buffer and A (support (f, w), first transform,
    // spectrum Z), then the W rows
    ulonglong2 W[(Cfg<N>::TWICE ? 2 : 1) * S * Cfg<N>::WS];
    float4 slot[2][N];                   // candidates of the warps: maximum, shift offset, coefficient
    float w0[S / 2 * S / 2];             // Eq. (5), one quadrant (symmetric)
    float wf[H1 * H1];                   // Eq. (9), one quadrant (symmetric)
    float2 cs[S];                        // cos, sin of 2 pi t / S
    unsigned flags[N];                  // per warp: 1 = a pixel of the support is available, 2 = an unknown target pixel
    unsigned dmax[N];
};

static_assert(2 * sizeof(float2) * S * AS <= sizeof(Smem<2>::W), "the transforms fit the W area");

__device__ __forceinline__ int fold(int m) { return m < S / 2 ? m : S - 1 - m; }   // w0: m and S-1-m are alike
__device__ __forceinline__ int foldf(int k) { return k <= S / 2 ? k : S - k; }      // w_f: k and S-k are alike

// The tables of the CTA: pairs (m, n) with m <= n, both ways round.  Not
// unrolled: a CTA that runs one block fetches this code cold, and the fetch is
// most of its time.  The entries beyond one per thread go to another warp for
// each table.
template <int N>
__device__ __forceinline__ void tables(const MethodArgs& mth, Smem<N>* sm) {
    constexpr int T = Cfg<N>::T;
    const int tid = threadIdx.x;
    constexpr int EF = H1 * (H1 + 1) / 2;          // w_f: 153 pairs, rows r and 16 - r side by side
#pragma unroll 1
    for (int base = 0; base < EF; base += T) {
        const int i = base + (base + T > EF ? (tid + T - 32) % T : tid);
        if (i >= EF) continue;
        const int r = i / (H1 + 1), c = i % (H1 + 1);
        const bool first = c < H1 - r;
        const int m = first ? r : H1 - 1 - r, n = first ? r + c : c - 1;
        sm->wf[m * H1 + n] = sm->wf[n * H1 + m] = wf_value<float>(mth, m, n);
    }
    constexpr int H = S / 2, EW = H * (H + 1) / 2;   // w0: 136 pairs, rows r and 15 - r side by side
#pragma unroll 1
    for (int base = 0; base < EW; base += T) {
        const int i = base + (base + T > EW ? (tid + T - 64) % T : tid);
        if (i >= EW) continue;
        const int r = i / (H + 1), c = i % (H + 1);
        const bool first = c < H - r;
        const int m = first ? r : H - 1 - r, n = first ? r + c : c - 1;
        sm->w0[m * H + n] = sm->w0[n * H + m] = w0_value<float>(mth, m, n);
    }
    if (tid < S) sm->cs[tid] = make_float2(float(cos_2pi32(tid)), float(sin_2pi32(tid)));
}

// One butterfly of the FFT, twiddle e^{-j 2 pi tw / 32} = c + j s, rounded as in
// fft32.  c = 1, s = -0 and c = 0, s = -1 give its multiplication-free cases.
__device__ __forceinline__ void butterfly(float2& a, float2& b, float c, float s, int tw) {
    float xr, xi;
    twiddle(b.x, b.y, c, s, tw, xr, xi);
    b.x = __fsub_rn(a.x, xr);
    b.y = __fsub_rn(a.y, xi);
    a.x = __fadd_rn(a.x, xr);
    a.y = __fadd_rn(a.y, xi);
}
__device__ __forceinline__ void butterfly_one(float2& a, float2& b) {   // twiddle 1
    const float2 x = b;
    b = make_float2(__fsub_rn(a.x, x.x), __fsub_rn(a.y, x.y));
    a = make_float2(__fadd_rn(a.x, x.x), __fadd_rn(a.y, x.y));
}
__device__ __forceinline__ void butterfly_mj(float2& a, float2& b) {    // twiddle -j
    const float2 x = make_float2(b.y, -b.x);
    b = make_float2(__fsub_rn(a.x, x.x), __fsub_rn(a.y, x.y));
    a = make_float2(__fadd_rn(a.x, x.x), __fadd_rn(a.y, x.y));
}

// the low `bits` bits of i reversed
__device__ __forceinline__ constexpr int brev(int i, int bits) {
    int r = 0;
    for (int b = 0; b < bits; ++b) r |= ((i >> b) & 1) << (bits - 1 - b);
    return r;
}
// index of point i of warp q (bit-reversed position PTS q + i); q2: q's bits reversed
template <int N>
__device__ __forceinline__ constexpr int in_index(int q2, int i) {
    return N * brev(i, N == 4 ? 3 : 4) + q2;
}

// the first stages on the PTS points of a thread, exchange through X, the
// last ones.  On return e[tt][p] is output TT q + tt + PTS p.
template <int N>
__device__ __forceinline__ void fft32_split(float2 (&x)[Cfg<N>::PTS], float2 (&e)[Cfg<N>::TT][N], float2* X,
                                            const float2* cs, int q, int lane) {
    constexpr int PTS = Cfg<N>::PTS, TT = Cfg<N>::TT;
#pragma unroll
    for (int half = 1; half < PTS; half *= 2)
#pragma unroll
        for (int j = 0; j < PTS; j += 2 * half)
#pragma unroll
            for (int t = 0; t < half; ++t) {
                const int tw = t * (16 / half);
                if (tw == 0) butterfly_one(x[j + t], x[j + t + half]);
                else if (tw == 8) butterfly_mj(x[j + t], x[j + t + half]);
                else butterfly(x[j + t], x[j + t + half], float(cos_2pi32(tw)), float(-sin_2pi32(tw)), tw);
            }
#pragma unroll
    for (int i = 0; i < PTS; ++i) X[(PTS * q + i) * AS + lane] = x[i];
    __syncthreads();
#pragma unroll
    for (int tt = 0; tt < TT; ++tt) {
        const int t = TT * q + tt;
#pragma unroll
        for (int p = 0; p < N; ++p) e[tt][p] = X[(t + PTS * p) * AS + lane];
        const float2 c1 = cs[t];
        if constexpr (N == 4) {
            const float2 c2 = cs[2 * t], c9 = cs[t + 8];
            butterfly(e[tt][0], e[tt][1], c2.x, -c2.y, 2 * t);
            butterfly(e[tt][2], e[tt][3], c2.x, -c2.y, 2 * t);
            butterfly(e[tt][0], e[tt][2], c1.x, -c1.y, t);
            butterfly(e[tt][1], e[tt][3], c9.x, -c9.y, t + 8);
        } else {
            butterfly(e[tt][0], e[tt][1], c1.x, -c1.y, t);
        }
    }
}

// A thread's lowest component holding its maximum mb, among the n components
// o with values (r, i): the half that has it, the lower one first.
template <int n>
__device__ __forceinline__ void halve(const float (&o)[n], const float (&r)[n], const float (&i)[n], unsigned mb,
                                      unsigned unit, unsigned& at, float& br, float& bi) {
    if constexpr (n == 1) {
        br = r[0];
        bi = i[0];
    } else {
        float m = o[0];
#pragma unroll
        for (int j = 1; j < n / 2; ++j) m = fmaxf(m, o[j]);
        const bool h = __float_as_uint(m) == mb;
        float o2[n / 2], r2[n / 2], i2[n / 2];
#pragma unroll
        for (int j = 0; j < n / 2; ++j) {
            o2[j] = h ? o[j] : o[j + n / 2];
            r2[j] = h ? r[j] : r[j + n / 2];
            i2[j] = h ? i[j] : i[j + n / 2];
        }
        at += h ? 0u : unit * (n / 2);
        halve<n / 2>(o2, r2, i2, mb, unit, at, br, bi);
    }
}
template <int n>
__device__ __forceinline__ float max_of(const float (&o)[n]) {
    if constexpr (n == 4) return fmaxf(max3(o[0], o[1], o[2]), o[3]);
    else return max3(max3(o[0], o[1], o[2]), max3(o[3], o[4], o[5]), fmaxf(o[6], o[7]));
}

// One block by the whole CTA.  Every thread reaches every barrier.  BUILD: the
// CTA's tables are built here, while the pixel loads are in flight.
template <int B, int N, bool REUSE, bool BUILD>
__device__ __forceinline__ void block(const ImageArgs& im, int by, int bx, const MethodArgs& mth, Smem<N>* sm,
                                      unsigned long long* empty, float delta) {
    using C = Cfg<N>;
    constexpr int T = C::T, G = C::G, NP = C::NP, WS = C::WS, PTS = C::PTS, TT = C::TT;
    constexpr int PT = (B * B + T - 1) / T;   // target pixels per thread
    const int tid = threadIdx.x, lane = tid & 31, q = tid >> 5;
    const int L = mth.L, y0 = by * B - L, x0 = bx * B - L;
    const long long blk = (long long)by * im.nbx + bx;
    int16_t* seq = im.seq ? im.seq + (size_t)blk * im.K : nullptr;
    const int q2 = N == 4 ? ((q & 1) << 1) | (q >> 1) : q;   // the bits of q reversed
    float2* X = reinterpret_cast<float2*>(sm->W);
    float2* A = X + S * AS;

    // ---- a1: PTS pixels of column `lane` per thread, and the target pixels ----
    float f[PTS];
    unsigned kn = 0, re = 0;
    {
        const int xc = x0 + lane;
        const bool xin = (unsigned)xc < (unsigned)im.W;
        const int pbx = xin ? xc / B : 0;
#pragma unroll
        for (int i = 0; i < PTS; ++i) {
            const int y = y0 + in_index<N>(q2, i);
            bool known = false, reused = false;
            float fv = 0.f, pv = 0.f;
            if (xin && (unsigned)y < (unsigned)im.H) {
                const size_t off = (size_t)y * im.pitch + xc;
                known = __ldg(im.mask + off) != 0;
                fv = __ldg(im.img + off);
                if constexpr (REUSE) {
                    const int pby = y / B;
                    const bool earlier = pby < by || (pby == by && pbx < bx);
                    // earlier targets were written by other CTAs, of earlier launches or
                    // of this one (their rows' progress acquired): read through L2
                    if (earlier) pv = __ldcg(im.out + off);
                    reused = !known && earlier;
                }
            }
            f[i] = known ? fv : (reused ? pv : 0.f);   // select: unknown values never enter arithmetic
            kn |= known ? 1u << i : 0u;
            re |= reused ? 1u << i : 0u;
        }
    }
    float tv[PT];          // value of a known target pixel
    bool tk[PT], tin[PT];  // known; in the image
    unsigned need = 0;
#pragma unroll
    for (int p = 0; p < PT; ++p) {
        const int i = tid + T * p;
        const int ty = by * B + i / B, tx = bx * B + i % B;
        tin[p] = i < B * B && ty < im.H && tx < im.W;
        tk[p] = true;
        tv[p] = 0.f;
        if (tin[p]) {
            const size_t off = (size_t)ty * im.pitch + tx;
            tk[p] = __ldg(im.mask + off) != 0;
            tv[p] = __ldg(im.img + off);
        }
        need |= tk[p] ? 0u : 2u;
    }
    if constexpr (BUILD) tables(mth, sm);
    const unsigned avail = kn | re;
    __syncthreads();   // the tables are complete, the buffers free
    float wv[PTS];
#pragma unroll
    for (int i = 0; i < PTS; ++i) {
        const int m = in_index<N>(q2, i);
        const float w0 = sm->w0[fold(m) * (S / 2) + fold(lane)];
        // Eq. (5): w0 on known pixels, delta w0 on re-used ones, 0 elsewhere
        wv[i] = ((kn >> i) & 1u) ? w0 : (((re >> i) & 1u) ? delta * w0 : 0.f);
        A[m * AS + lane] = make_float2(f[i], wv[i]);
    }
    need = __reduce_or_sync(FULL, need | (avail ? 1u : 0u));
    if (lane == 0) sm->flags[q] = need;
    __syncthreads();
    need = sm->flags[0] | sm->flags[1];
    if constexpr (N == 4) need |= sm->flags[2] | sm->flags[3];

    float gacc[PT];
#pragma unroll
    for (int p = 0; p < PT; ++p) gacc[p] = 0.f;
    const int K = im.K;
    if (!(need & 1u)) {
        if (tid == 0) empty_block(seq, K, empty);
    } else if (K > 0 && ((need & 2u) || seq != nullptr)) {   // all targets known: copied, whatever the model
        // ---- a2: sums over the column in row order, then over the columns
        //      (every warp for itself: no barrier); weighted mean ----
        float sw = 0.f, sfw = 0.f;
#pragma unroll
        for (int m = 0; m < S; ++m) {
            const float2 fw = A[m * AS + lane];
            sw = __fadd_rn(sw, fw.y);
            sfw = __fmaf_rn(fw.y, fw.x, sfw);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            sw += __shfl_xor_sync(FULL, sw, o);
            sfw += __shfl_xor_sync(FULL, sfw, o);
        }
        const float mu = sfw / sw;
        float2 x[PTS];
        unsigned dmax = 0;
#pragma unroll
        for (int i = 0; i < PTS; ++i) {
            const bool av = (avail >> i) & 1u;
            const float d = __fsub_rn(f[i], mu);
            x[i] = make_float2(av ? __fmul_rn(d, wv[i]) : 0.f, wv[i]);
            const unsigned ab = __float_as_uint(d) & 0x7fffffffu;
            dmax = (av && ab > dmax) ? ab : dmax;
        }
        dmax = __reduce_max_sync(FULL, dmax);
        if (lane == 0) sm->dmax[q] = dmax;
        __syncthreads();
        dmax = max(sm->dmax[0], sm->dmax[1]);
        if constexpr (N == 4) dmax = max(dmax, max(sm->dmax[2], sm->dmax[3]));
        unsigned aexp = (dmax >> 23) + 1u;             // exponent field of alpha = 2^e
        aexp = (dmax >= 0x00800000u && dmax < 0x7e000000u) ? aexp : 127u;
        const float alpha = __uint_as_float(aexp << 23);
        const float inv2alpha = __uint_as_float((253u - aexp) << 23);   // 1 / (2 alpha)
#pragma unroll
        for (int i = 0; i < PTS; ++i) x[i].y *= alpha;

        // ---- a3: over the rows (lane n = column n), then over the columns (lane k = row k) ----
#pragma unroll 1
        for (int pass = 0; pass < 2; ++pass) {
            float2 e[TT][N];
            fft32_split<N>(x, e, X, sm->cs, q, lane);
            // first transform out by rows k, then back in by columns; the second stays transposed
            const int sk = pass == 0 ? AS : 1, sl = pass == 0 ? 1 : AS;
#pragma unroll
            for (int tt = 0; tt < TT; ++tt)
#pragma unroll
                for (int p = 0; p < N; ++p) A[(TT * q + tt + PTS * p) * sk + lane * sl] = e[tt][p];
            __syncthreads();
            if (pass == 0) {
#pragma unroll
                for (int i = 0; i < PTS; ++i) x[i] = A[lane * AS + in_index<N>(q2, i)];
            }
        }

        // ---- Q and W of this thread's components ----
        const int k = C::RPW * q + lane / G, g = lane % G;
        f32x2 zr[NP], zi[NP], wf[NP], wur[NP], wui[NP];   // wu: the unshifted W row
#pragma unroll
        for (int j = 0; j < NP; ++j) {
            float qr[2], qi[2], wr[2], wi[2], f2[2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int l = g + G * j + S / 2 * h;
                const float2 a = A[k * AS + l], c = A[((S - k) & (S - 1)) * AS + ((S - l) & (S - 1))];
                wr[h] = (a.y + c.y) * inv2alpha;
                wi[h] = (c.x - a.x) * inv2alpha;
                qr[h] = (a.x + c.x) * 0.5f;
                qi[h] = (a.y - c.y) * 0.5f;
                f2[h] = sm->wf[foldf(k) * H1 + foldf(l)];
            }
            zr[j] = pack2(qr[0], qr[1]);
            zi[j] = pack2(qi[0], qi[1]);
            wf[j] = pack2(f2[0], f2[1]);
            wur[j] = pack2(wr[0], wr[1]);
            wui[j] = pack2(wi[0], wi[1]);
        }
        __syncthreads();   // Z is read no more: the W rows go there
#pragma unroll
        for (int j = 0; j < NP; ++j) {
            // entries l, l + 16 (the halves change places) and l + 32, in rows k and k + 32
            float r0, r1, i0, i1;
            unpack2(wur[j], r0, r1);
            unpack2(wui[j], i0, i1);
            const ulonglong2 e = make_ulonglong2(wur[j], wui[j]);
            const ulonglong2 x = make_ulonglong2(pack2(r1, r0), pack2(i1, i0));
            ulonglong2* w = sm->W + k * WS + g + G * j;
            w[0] = w[S] = e;
            w[S / 2] = x;
            if constexpr (C::TWICE) {
                w[S * WS] = w[S * WS + S] = e;
                w[S * WS + S / 2] = x;
            }
        }
        __syncthreads();
        float w00, w16;
        unpack2(sm->W[0].x, w00, w16);
        const float cg = mth.gamma * (1.f / w00);
        int pm[PT], pn[PT];
#pragma unroll
        for (int p = 0; p < PT; ++p) {
            pm[p] = L + (tid + T * p) / B;
            pn[p] = L + (tid + T * p) % B;
        }
        // W[k-u][l-v], l = g
        const ulonglong2* wbase = sm->W + (C::TWICE ? (k + S) * WS : 0) + g + S;
        auto shifted = [&](unsigned o) {
            if constexpr (C::TWICE) return wbase - o;   // u rows and v entries before W[k][g]
            const int u = (int)((o * C::DIV) >> 16), v = (int)(o - (unsigned)u * WS);
            return wbase + ((k - u) & (S - 1)) * WS - v;
        };
        const unsigned off0 = (unsigned)(k * WS + g);
        float cr = 0.f, ci = 0.f;
        unsigned off;   // u * WS + v
        float olo[NP] = {}, ohi[NP] = {};   // objectives of the pairs' halves
        float2 csn[PT];
#pragma unroll
        for (int p = 0; p < PT; ++p) csn[p] = make_float2(0.f, 0.f);
        // the last pick's share of the target pixels (sparse inverse of G)
        auto target = [&]() {
#pragma unroll
            for (int p = 0; p < PT; ++p) gacc[p] = fma_rn(cr, csn[p].x, fma_rn(-ci, csn[p].y, gacc[p]));
        };

        // a5, a6 for the objectives of the values (vr, vi): the warp's
        // maximum (objectives are >= +0: their bits order like the values)
        // and its lowest index, then the four warps' candidates.  What a
        // thread may publish is formed while the reductions run: its lowest
        // component holding its own maximum, by halving.
        auto pick = [&](int nu, const f32x2 (&vr)[NP], const f32x2 (&vi)[NP]) {
            const float mlo = max_of(olo), mhi = max_of(ohi);
            const float m = fmaxf(mlo, mhi);
            const unsigned mb = __float_as_uint(m);
            const unsigned Mw = __reduce_max_sync(FULL, mb);
            target();   // of the previous pick
            const bool h1 = __float_as_uint(mlo) == mb;   // columns < 16
            float o1[NP], r1[NP], i1[NP], br, bi;
#pragma unroll
            for (int j = 0; j < NP; ++j) {
                float r0, rx, i0, ix;
                unpack2(vr[j], r0, rx);
                unpack2(vi[j], i0, ix);
                o1[j] = h1 ? olo[j] : ohi[j];
                r1[j] = h1 ? r0 : rx;
                i1[j] = h1 ? i0 : ix;
            }
            // index u * S + v as the offset u * WS + v: the same order
            unsigned boff = off0 + (h1 ? 0u : S / 2);
            halve<NP>(o1, r1, i1, mb, (unsigned)G, boff, br, bi);
            const unsigned lo = __reduce_min_sync(FULL, mb == Mw ? boff : 0xffffffffu);
            // c = gamma p (Eq. 10)
            const float4 mine = make_float4(m, __uint_as_float(boff), br * cg, bi * cg);
            float4* sl = sm->slot[nu & 1];
            if (mb == Mw && boff == lo) sl[q] = mine;
            __syncthreads();   // one barrier per iteration: the slots alternate
            // rows ascend with the warp, so the first maximum has the lowest index
            float4 c0 = sl[0];
            const float4 c1 = sl[1];
            if constexpr (N == 4) {
                float4 c2 = sl[2];
                const float4 c3 = sl[3];
                if (__float_as_uint(c1.x) > __float_as_uint(c0.x)) c0 = c1;
                if (__float_as_uint(c3.x) > __float_as_uint(c2.x)) c2 = c3;
                if (__float_as_uint(c2.x) > __float_as_uint(c0.x)) c0 = c2;
            } else {
                if (__float_as_uint(c1.x) > __float_as_uint(c0.x)) c0 = c1;
            }
            off = __float_as_uint(c0.y);
            cr = c0.z;
            ci = c0.w;
        };
        // the recorded index, and the target pixels' phases of the pick (used
        // by target() in the next one)
        // (in every thread: a branch to the warps that have target pixels costs
        // 50 cycles of the iteration)
        auto note = [&](int nu, auto rec) {
            const int u = (int)((off * C::DIV) >> 16), v = (int)(off - (unsigned)u * WS);
            if constexpr (rec.value) {
                if (tid == 0) seq[nu] = (int16_t)(u * S + v);
            }
#pragma unroll
            for (int p = 0; p < PT; ++p) csn[p] = sm->cs[(u * pm[p] + v * pn[p]) & (S - 1)];
        };

        // ---- a4-a8: the DC phase, R = a W + Q, then the plain loop; rec: the
        //      selected indices are recorded ----
        auto iterate = [&](auto rec) {
            int nu = 0;
            {
                float ar = mu, ai = 0.f;
                for (;;) {
                    const f32x2 ar2 = pack2(ar, ar), ai2 = pack2(ai, ai), nai2 = pack2(-ai, -ai);
                    f32x2 rr[NP], ri[NP];
#pragma unroll
                    for (int j = 0; j < NP; ++j) {
                        rr[j] = ffma2(ar2, wur[j], ffma2(nai2, wui[j], zr[j]));
                        ri[j] = ffma2(ar2, wui[j], ffma2(ai2, wur[j], zi[j]));
                        unpack2(objective2(rr[j], ri[j], wf[j]), olo[j], ohi[j]);
                    }
                    pick(nu, rr, ri);
                    if (nu + 1 == K || off != 0) {
#pragma unroll
                        for (int j = 0; j < NP; ++j) {   // fold a W into Q
                            zr[j] = rr[j];
                            zi[j] = ri[j];
                        }
                        break;
                    }
                    note(nu++, rec);
                    ar -= cr;
                    ai -= ci;
                }
            }
            for (;;) {   // the pick of iteration nu is not applied yet
                if (nu + 1 == K) break;
                const ulonglong2* row = shifted(off);   // a7 (Eq. 12) and the next objective
                const f32x2 ncr2 = pack2(-cr, -cr), ci2 = pack2(ci, ci), nci2 = pack2(-ci, -ci);
                constexpr int NL = 4;
#pragma unroll
                for (int j0 = 0; j0 < NP; j0 += NL) {
                    ulonglong2 w[NL];
#pragma unroll
                    for (int j = 0; j < NL; ++j) w[j] = row[G * (j0 + j)];
                    if (j0 == 0) note(nu++, rec);   // while the loads are under way
#pragma unroll
                    for (int j = 0; j < NL; ++j) {
                        f32x2 &a = zr[j0 + j], &b = zi[j0 + j];
                        a = ffma2(ncr2, w[j].x, ffma2(ci2, w[j].y, a));
                        b = ffma2(ncr2, w[j].y, ffma2(nci2, w[j].x, b));
                        unpack2(objective2(a, b, wf[j0 + j]), olo[j0 + j], ohi[j0 + j]);
                    }
                }
                pick(nu, zr, zi);
            }
            note(nu, rec);
            target();
        };
        if (seq != nullptr) iterate(std::true_type{});
        else iterate(std::false_type{});
    }

    // ---- a9 ----
#pragma unroll
    for (int p = 0; p < PT; ++p) {
        const int i = tid + T * p;
        if (tin[p]) {
            const int ty = by * B + i / B, tx = bx * B + i % B;
            im.out[(size_t)ty * im.pitch + tx] = tk[p] ? tv[p] : gacc[p];
        }
    }
}

// One block per CTA, the grid sized to the work.  INLINE: one image whose
// arguments are kernel parameters; else images and block prefix sums of a
// work table in device memory.
template <int B, int N, bool INLINE>
__global__ void __launch_bounds__(Cfg<N>::T, Cfg<N>::MIN_CTAS) fsr_coop_kernel(const __grid_constant__ BatchArgs a,
                                                     const __grid_constant__ ImageArgs one) {
    extern __shared__ __align__(16) unsigned char smem[];
    Smem<N>* sm = reinterpret_cast<Smem<N>*>(smem);
    const long long item = blockIdx.x;
    if constexpr (INLINE) {
        const int by = (int)item / one.nbx;
        block<B, N, false, true>(one, by, (int)item - by * one.nbx, a.mth, sm, a.empty, 0.f);
    } else {
        int lo = 0, hi = a.n - 1;   // image of this entry: last i with first[i] <= item
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (__ldg(a.first + mid) <= item) lo = mid;
            else hi = mid - 1;
        }
        const ImageArgs im = a.images[lo];
        const int blk = (int)(item - __ldg(a.first + lo));
        const int by = blk / im.nbx;
        block<B, N, false, true>(im, by, blk - by * im.nbx, a.mth, sm, a.empty, 0.f);
    }
}

// Re-use form: one launch per wavefront (see fsr_reuse_kernel), a CTA per block.
template <int B, int NSEG>
__global__ void __launch_bounds__(Cfg<4>::T) fsr_coop_reuse_kernel(const __grid_constant__ ReuseLaunchN<NSEG> a) {
    extern __shared__ __align__(16) unsigned char smem[];
    Smem<4>* sm = reinterpret_cast<Smem<4>*>(smem);
    tables(a.mth, sm);
    // a programmatic dependent of the previous wavefront: nothing of the
    // image or the output is read before that one has completed
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int j = blockIdx.x;
    int s = 0;   // the segment (image) of block j
    if constexpr (NSEG > 1) {
        while (s + 1 < a.nseg && a.seg[s + 1].first <= j) ++s;
    }
    const ReuseSeg& sg = a.seg[s];
    const int by = sg.by_lo + (j - sg.first);
    block<B, 4, true, false>(sg.im, by, a.t - a.slope * by, a.mth, sm, a.empty, a.delta);
}

// Re-use form in one launch: a CTA takes block rows in order and works through
// a row from left to right; row by of an image runs `lag` = ceil(L / B) + 1
// blocks behind row by - 1, the same dependency as the wavefront launches
// (every earlier block of the raster order whose target meets the support is
// complete), so the results are the same bit for bit.  Against a launch per
// wavefront it saves the launch and the tables on the chain, and no block
// waits for the slowest of its wavefront.
//
// Rows are claimed in order from a counter, row r of every image before row
// r + 1 of any (images by falling row count), so the row a CTA waits for is
// held by a CTA that already runs: the waits end whatever the grid size.
// Progress of row g is published in ring[g % kRowRing] as (g + 1) << 32 |
// blocks done (0xffffffff: all); a larger tag in the slot means the row is
// long done, and a row takes its slot over only from a finished one.
constexpr int kRowRing = 2048;
constexpr int kRowImages = 48;
struct RowsArgs {
    MethodArgs mth;
    float delta;
    int lag, n, rows;            // rows of all images together
    unsigned long long* ring;    // kRowRing entries, then the row counter and the finished blocks: zero at launch
    unsigned long long limit_ns; // of the waits
    unsigned* status;
    unsigned long long* empty;
    ImageArgs im[kRowImages];    // by falling number of block rows
    int nby[kRowImages];
};
static_assert(sizeof(RowsArgs) <= 4096, "row launch parameters must fit the 4 KB parameter space");

__device__ __forceinline__ unsigned long long ld_acquire(const unsigned long long* p) {
    unsigned long long v;
    asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_release(unsigned long long* p, unsigned long long v) {
    asm volatile("st.release.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

// One thread: wait (bounded) until slot shows row g with at least `need`
// blocks done, or a later row.  The wait gives up when no block of the launch
// has finished for limit_ns (row_limit_ns: more than any block takes).  The
// row waited for may itself stand still for much longer, behind all rows
// between it and the one at work, and those may be of an image with other
// sizes and iterations than this one's: 300 rows of two blocks each, K = 100,
// start 13 ms after one another's first.
__device__ __forceinline__ bool row_wait(const RowsArgs& a, unsigned g, unsigned need) {
    const unsigned long long* slot = a.ring + g % (unsigned)kRowRing;
    unsigned long long t0 = 0, last = 0;
    for (unsigned it = 0;; ++it) {
        const unsigned long long v = ld_acquire(slot);
        const unsigned tag = (unsigned)(v >> 32);
        if (tag > g + 1u || (tag == g + 1u && (unsigned)v >= need)) return true;
        __nanosleep(64);
        if ((it & 63u) == 0u) {
            const unsigned long long done = ld_acquire(a.ring + kRowRing + 1);
            unsigned long long t;
            asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
            if (it == 0u || done != last) t0 = t;   // the clock starts again with every block that finishes
            else if (t - t0 > a.limit_ns) return false;
            last = done;
        }
    }
}

template <int B>
__global__ void __launch_bounds__(Cfg<4>::T) fsr_coop_rows_kernel(const __grid_constant__ RowsArgs a) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int s_row, s_ok;
    Smem<4>* sm = reinterpret_cast<Smem<4>*>(smem);
    tables(a.mth, sm);
    for (;;) {
        if (threadIdx.x == 0) s_row = (int)atomicAdd(a.ring + kRowRing, 1ull);
        __syncthreads();
        const int g = s_row;
        if (g >= a.rows) return;
        // row r of image i: g = (rows r' < r of all images) + i
        auto before = [&](int r) {
            int t = 0;
            for (int i = 0; i < a.n; ++i) t += min(a.nby[i], r);
            return t;
        };
        int lo = 0, hi = a.nby[0] - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (before(mid) <= g) lo = mid;
            else hi = mid - 1;
        }
        const int r = lo, first = before(r), i = g - first;
        const int prev = r > 0 ? before(r - 1) + i : 0;   // row r - 1 of this image
        const ImageArgs im = a.im[i];
        unsigned long long* slot = a.ring + g % kRowRing;
        const unsigned long long tag = (unsigned long long)(g + 1) << 32;
        if (threadIdx.x == 0) {
            s_ok = g < kRowRing || row_wait(a, (unsigned)(g - kRowRing), 0xffffffffu);
            if (s_ok) st_release(slot, tag);
        }
        __syncthreads();
        for (int bx = 0; bx < im.nbx; ++bx) {
            // the row above, while thread 0 publishes the last block
            if (threadIdx.x == Cfg<4>::T - 1 && r > 0 && s_ok &&
                !row_wait(a, (unsigned)prev, (unsigned)min(bx + a.lag, im.nbx)))
                s_ok = 0;
            __syncthreads();
            if (!s_ok) {
                if (threadIdx.x == 0) atomicOr(a.status, kStatusRowWait);
                return;
            }
            block<B, 4, true, false>(im, r, bx, a.mth, sm, a.empty, a.delta);
            __syncthreads();
            // (release at the end of a barrier: the CTA's pixels come before it)
            if (threadIdx.x == 0) {
                st_release(slot, tag | (bx + 1 == im.nbx ? 0xffffffffu : (unsigned)(bx + 1)));
                atomicAdd(a.ring + kRowRing + 1, 1ull);
            }
        }
    }
}

}  // namespace coop
}  // namespace fsrk
