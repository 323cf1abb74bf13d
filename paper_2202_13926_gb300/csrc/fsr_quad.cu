// FP32 FSR with the 4 x 4 support (B <= 4; the smallest support of the study of
// Sec. IV, Fig. 3): one lane per block, 32 blocks per warp.
//
// What bounds this support is the pick: with 4 lanes per block and a row in
// each, block maximum, row, column and coefficient took three times the
// instructions of the 16 components' arithmetic.  With the whole spectrum in
// one lane the pick needs no other lane: no shuffle, ballot or barrier in the
// iteration.
//   * Components l and l + 2 of a row are a pair in two adjacent registers,
//     updated by packed f32x2 operations (the same roundings as the scalar
//     ones): half the issue slots.
//   * A stored W row is 5 entries (Re W[c], Re W[c + 2], Im W[c], Im W[c + 2])
//     of 16 bytes, so the shifted row of Eqs. (12), (14), (15) is 2 entries from
//     c = 4 - v: no column wrap.  The entries of 8 blocks are interleaved: the
//     lanes of a quarter-warp, each with its own shift, never meet on a bank.
//   * The picks are summed in G (one entry per pick, [component][lane] in shared
//     memory: no conflicts) and inverted at the end: the sparse inverse would
//     touch the 16 target pixels of the lane in every iteration.
//   * R = a W + Q while only the DC component is selected (DC phase).  Its pass
//     is an update pass with shift (0, 0) and coefficient -a whose result is
//     not stored (the same operations); at the end of the phase one that is
//     stored folds a W into Q.  So blocks in and out of the phase share passes.
// The transforms (a1-a3) run on groups of 4 lanes, 8 blocks at a time: support
// by columns, weighted mean mu removed, x = (f - mu) w and alpha w packed into
// z = x + j alpha w, two in-register FFTs with a transpose through shared
// memory; R_w and W from Z[k][l] and conj Z[-k][-l] with commutative operations
// (exactly Hermitian, as in the oracle).
//
// Measured (K = 100, B = 4), 4 lanes per block -> this: 1280 x 720 128 -> 90 us,
// 480 x 480 72 -> 50 us, 64 x 64 48 -> 43 us, 1080p 250 -> 182 us; 16.1 -> 10.7
// instructions per block and iteration (129 per warp, of 8 blocks, then; 344, of
// 32, now).  What bounds it now: the issue slots and the latency of one
// iteration's chain (0.4 us) at 3 warps per scheduler (issue active 66 %).
#include "fsr_launch.h"

namespace fsrk {
namespace {

constexpr int SZ = 4;
constexpr int HP = SZ / 2;              // pairs (l, l + 2) per row
constexpr int BPW = 32;                 // blocks per warp
constexpr int IL = 8;                   // blocks interleaved
constexpr int EW = SZ + HP - 1;         // W row: entries
constexpr int BPR = 32 / SZ;            // blocks per round of the transforms
constexpr int TS = SZ + 1;              // transpose stride (float2)
static_assert(EW % 2 == 1 && BPR == IL, "layout");
static_assert(BPR * SZ * TS * 8 <= BPR * SZ * EW * 16, "the transposes fit the W rows of the round's blocks");

// shared memory: tables (bytes), then per warp the W rows, G and the queue
constexpr size_t kW0Off = 0;
constexpr size_t kWfOff = kW0Off + 4 * SZ * SZ;
constexpr size_t kWarp0Off = 128;
constexpr size_t kGOff = (size_t)16 * BPW * SZ * EW;
constexpr size_t kQOff = kGOff + (size_t)8 * SZ * SZ * 32;
constexpr size_t kPerWarp = (kQOff + 8 * (BPW + 32) + 127) & ~(size_t)127;
constexpr size_t smem_bytes(int warps) { return kWarp0Off + kPerWarp * (size_t)warps; }

// entry e of block b's W rows
__device__ __forceinline__ int entry(int b, int e) { return (b / IL) * SZ * EW * IL + e * IL + b % IL; }

template <int N>
__host__ __device__ constexpr int bit_reverse(int i) {
    int r = 0;
    for (int b = 1, rb = N >> 1; b < N; b <<= 1, rb >>= 1)
        if (i & b) r |= rb;
    return r;
}

// In-register radix-2 decimation-in-time FFT of length N, natural order in
// and out, X[k] = sum_m x[m] e^{-j 2 pi k m / N}.
template <int N>
__device__ __forceinline__ void fftn(float (&re)[N], float (&im)[N]) {
    float ar[N], ai[N];
#pragma unroll
    for (int i = 0; i < N; ++i) {
        ar[i] = re[bit_reverse<N>(i)];
        ai[i] = im[bit_reverse<N>(i)];
    }
#pragma unroll
    for (int half = 1; half < N; half *= 2) {
#pragma unroll
        for (int j = 0; j < N; j += 2 * half) {
#pragma unroll
            for (int t = 0; t < half; ++t) {
                const int tw = t * (N / 2 / half);   // e^{-j 2 pi tw / N}
                const float br = ar[j + t + half], bi = ai[j + t + half];
                float xr, xi;
                if (tw == 0) {
                    xr = br;
                    xi = bi;
                } else if (tw == N / 4) {   // times -j
                    xr = bi;
                    xi = -br;
                } else {
                    const float c = float(cos_2pi32(tw * (32 / N))), s = float(-sin_2pi32(tw * (32 / N)));
                    xr = br * c - bi * s;
                    xi = br * s + bi * c;
                }
                ar[j + t + half] = ar[j + t] - xr;
                ai[j + t + half] = ai[j + t] - xi;
                ar[j + t] = ar[j + t] + xr;
                ai[j + t] = ai[j + t] + xi;
            }
        }
    }
#pragma unroll
    for (int i = 0; i < N; ++i) {
        re[i] = ar[i];
        im[i] = ai[i];
    }
}

// reductions inside a group of SZ lanes
__device__ __forceinline__ unsigned group_umax(unsigned v) {
#pragma unroll
    for (int s = SZ / 2; s > 0; s >>= 1) v = max(v, (unsigned)__shfl_xor_sync(FULL, v, s));
    return v;
}
__device__ __forceinline__ float group_sum(float v) {
#pragma unroll
    for (int s = SZ / 2; s > 0; s >>= 1) v += __shfl_xor_sync(FULL, v, s);
    return v;
}

// Re g at the 16 pixels of the support from G (entries [u * 4 + v][lane])
__device__ __forceinline__ void inverse4(const float2* G, float (&g)[16]) {
    float2 h[4][4];   // h[u][n] = sum_v G[u][v] j^(v n)
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        float2 a[4];
#pragma unroll
        for (int v = 0; v < 4; ++v) a[v] = G[(u * 4 + v) * 32];
        const float2 s02 = make_float2(a[0].x + a[2].x, a[0].y + a[2].y), d02 = make_float2(a[0].x - a[2].x, a[0].y - a[2].y);
        const float2 s13 = make_float2(a[1].x + a[3].x, a[1].y + a[3].y), d13 = make_float2(a[1].x - a[3].x, a[1].y - a[3].y);
        h[u][0] = make_float2(s02.x + s13.x, s02.y + s13.y);
        h[u][1] = make_float2(d02.x - d13.y, d02.y + d13.x);
        h[u][2] = make_float2(s02.x - s13.x, s02.y - s13.y);
        h[u][3] = make_float2(d02.x + d13.y, d02.y - d13.x);
    }
#pragma unroll
    for (int n = 0; n < 4; ++n) {
        const float s02 = h[0][n].x + h[2][n].x, d02 = h[0][n].x - h[2][n].x;
        const float s13 = h[1][n].x + h[3][n].x, d13 = h[1][n].y - h[3][n].y;   // Re(j z) = -Im z
        g[n] = s02 + s13;
        g[4 + n] = d02 - d13;
        g[8 + n] = s02 - s13;
        g[12 + n] = d02 + d13;
    }
}

// The work list: entries that need the iteration queue up (queue: BPW + 32
// entries) until there are `per` of them, then run(n) works on queue[0 .. n-1],
// n <= per <= BPW.
template <int B, class F>
__device__ __forceinline__ void for_queued_blocks(const BatchArgs& a, int warps, int per, long long* queue, int lane,
                                                  F&& run) {
    int nq = 0;
    long long pos = 0, end = 0, seen = 0;   // the part of the list this warp has taken and not scanned yet
    bool more = true;
    for (;;) {
        while (nq < per && more) {
            if (pos >= end) {
                const int take = guided_take(a, seen, warps, a.chunk * per);
                unsigned long long base = 0;
                if (lane == 0) base = atomicAdd(a.counter, (unsigned long long)take);
                base = __shfl_sync(FULL, base, 0);
                more = base < (unsigned long long)a.total;
                if (!more) break;
                seen = pos = (long long)base;
                end = min(pos + take, a.total);
            }
            const int n = (int)min(end - pos, 32ll);
            // (one round of the grid holds every block: nothing is gained by
            // sorting out the copies first)
            const unsigned todo = a.total > (long long)warps * per ? scan_targets<B>(a, pos, n, lane)
                                                                   : 0xffffffffu >> (32 - n);
            if ((todo >> lane) & 1u) queue[nq + __popc(todo & ((1u << lane) - 1u))] = pos + lane;
            nq += __popc(todo);
            pos += n;
        }
        if (nq == 0) break;
        __syncwarp();
        const int nblk = min(nq, per);
        run(nblk);
        __syncwarp();
        nq -= nblk;   // at most 31 left
        long long rest = 0;
        if (lane < nq) rest = queue[nblk + lane];
        __syncwarp();
        if (lane < nq) queue[lane] = rest;
        __syncwarp();
    }
}

template <int B>
__device__ __forceinline__ void run_blocks(const BatchArgs& a, int nblk, const float* __restrict__ sw0,
                                           const float* __restrict__ swf, unsigned char* area, int lane) {
    ulonglong2* Wd = reinterpret_cast<ulonglong2*>(area);   // (Re pair, Im pair)
    float2* G = reinterpret_cast<float2*>(area + kGOff) + lane;       // this lane's [component][lane]
    const long long* queue = reinterpret_cast<const long long*>(area + kQOff);
    const int L = a.mth.L;

    f32x2 zr[SZ][HP], zi[SZ][HP];   // pairs (l, l + 2) of the rows
#pragma unroll
    for (int r = 0; r < SZ; ++r)
#pragma unroll
        for (int j = 0; j < HP; ++j) zr[r][j] = zi[r][j] = 0;
    float mu = 0.f, W0 = 1.f;
    int K = 0;
    int16_t* seq = nullptr;
    bool active = false;

    // ---- a1-a3, BPR blocks at a time: lane ts of group i holds column ts,
    //      then row ts, of block r * BPR + i ----
#pragma unroll 1
    for (int round = 0; round * BPR < nblk; ++round) {
        const int ts = lane % SZ, i = lane / SZ, gs = lane - ts;
        const int bb = round * BPR + i;
        const bool valid = bb < nblk;
        float pr[SZ], pi[SZ];
        unsigned known = 0;
        int imK = 0;
        int16_t* sq = nullptr;
        {
            ImageArgs im;
            long long blk = 0;
            im.img = nullptr; im.mask = nullptr; im.H = im.W = im.pitch = 0; im.nbx = 1; im.seq = nullptr; im.K = 0;
            if (valid) {
                const long long item = queue[bb];
                const int lo = image_of(a, item);
                im = a.images[lo];
                blk = item - __ldg(a.first + lo);
            }
            imK = im.K;
            sq = im.seq ? im.seq + (size_t)blk * im.K : nullptr;
            const int by = (int)(blk / im.nbx), bx = (int)(blk - (long long)by * im.nbx);
            const int y0 = by * B - L, x = bx * B - L + ts;
#pragma unroll
            for (int m = 0; m < SZ; ++m) {
                const int y = y0 + m;
                float f = 0.f;
                if ((unsigned)y < (unsigned)im.H && (unsigned)x < (unsigned)im.W) {
                    const size_t off = (size_t)y * im.pitch + x;
                    const float fv = __ldg(im.img + off);
                    if (__ldg(im.mask + off) != 0) {
                        known |= 1u << m;
                        f = fv;
                    }
                }
                pr[m] = f;   // unknown values never enter arithmetic
            }
        }
        float sw = 0.f, sfw = 0.f;
#pragma unroll
        for (int m = 0; m < SZ; ++m) {
            const float w = ((known >> m) & 1u) ? sw0[m * SZ + ts] : 0.f;
            sw += w;
            sfw += w * pr[m];
        }
        sw = group_sum(sw);
        sfw = group_sum(sfw);
        const unsigned kb = (__ballot_sync(FULL, known != 0) >> gs) & ((1u << SZ) - 1u);
        const bool act = valid && kb != 0u;
        const float mub = act ? sfw / sw : 0.f;
        unsigned dmax = 0;
#pragma unroll
        for (int m = 0; m < SZ; ++m) {
            const bool kn = (known >> m) & 1u;
            const float w = kn ? sw0[m * SZ + ts] : 0.f;
            const float d = pr[m] - mub;
            pr[m] = kn ? d * w : 0.f;
            pi[m] = w;
            const unsigned ab = __float_as_uint(d) & 0x7fffffffu;
            dmax = (kn && ab > dmax) ? ab : dmax;
        }
        // alpha = 2^e >= max |f - mu|: both halves of z = x + j alpha w have one
        // magnitude through the shared FFT; powers of two are undone exactly
        dmax = group_umax(dmax);
        unsigned aexp = (dmax >> 23) + 1u;
        aexp = (dmax >= 0x00800000u && dmax < 0x7e000000u) ? aexp : 127u;
        const float alpha = __uint_as_float(aexp << 23);
        const float inv2alpha = __uint_as_float((253u - aexp) << 23);
#pragma unroll
        for (int m = 0; m < SZ; ++m) pi[m] *= alpha;

        // FFT over m (lane ts holds column ts), transpose, FFT over n; the
        // buffer lies in the W rows of this round's blocks
        float2* tb = reinterpret_cast<float2*>(Wd + round * BPR * SZ * EW) + i * SZ * TS;
        fftn<SZ>(pr, pi);
        __syncwarp();   // the W rows of the previous blocks are read no more
#pragma unroll
        for (int k = 0; k < SZ; ++k) tb[k * TS + ts] = make_float2(pr[k], pi[k]);
        __syncwarp();
#pragma unroll
        for (int n = 0; n < SZ; ++n) {
            const float2 v = tb[ts * TS + n];
            pr[n] = v.x;
            pi[n] = v.y;
        }
        __syncwarp();
        fftn<SZ>(pr, pi);   // lane k = ts holds Z[k][0..S-1]

        // Q[k][l] = (Z[k][l] + conj Z[-k][-l]) / 2,  W[k][l] = (Z[k][l] - conj Z[-k][-l]) / (2j alpha)
        const int src = gs + ((SZ - ts) & (SZ - 1));
        float wr[SZ], wi[SZ];
#pragma unroll
        for (int l = 0; l <= SZ / 2; ++l) {
            const int l2 = (SZ - l) & (SZ - 1);
            const float cr = __shfl_sync(FULL, pr[l2], src);
            const float ci = __shfl_sync(FULL, pi[l2], src);
            float dr = cr, di = ci;
            if (l2 != l) {
                dr = __shfl_sync(FULL, pr[l], src);
                di = __shfl_sync(FULL, pi[l], src);
            }
            const float ar = pr[l], ai = pi[l];
            wr[l] = (ai + ci) * inv2alpha;
            wi[l] = (cr - ar) * inv2alpha;
            pr[l] = (ar + cr) * 0.5f;
            pi[l] = (ai - ci) * 0.5f;
            if (l2 != l) {
                const float br = pr[l2], bi = pi[l2];
                wr[l2] = (bi + di) * inv2alpha;
                wi[l2] = (dr - br) * inv2alpha;
                pr[l2] = (br + dr) * 0.5f;
                pi[l2] = (bi - di) * 0.5f;
            }
        }
        // Q to the lanes of the iteration, then the W rows in its place
#pragma unroll
        for (int l = 0; l < SZ; ++l) tb[ts * TS + l] = make_float2(pr[l], pi[l]);
        __syncwarp();
        const bool mine = lane / BPR == round;   // this lane's block is of this round
        {
            const float2* qb = reinterpret_cast<const float2*>(Wd + round * BPR * SZ * EW) + (lane % BPR) * SZ * TS;
            if (mine) {
#pragma unroll
                for (int r = 0; r < SZ; ++r)
#pragma unroll
                    for (int j = 0; j < HP; ++j) {
                        const float2 q0 = qb[r * TS + j], q1 = qb[r * TS + j + HP];
                        zr[r][j] = pack2(q0.x, q1.x);
                        zi[r][j] = pack2(q0.y, q1.y);
                    }
            }
        }
        __syncwarp();
#pragma unroll
        for (int c = 0; c < EW; ++c)
            Wd[entry(bb, ts * EW + c)] =
                make_ulonglong2(pack2(wr[c % SZ], wr[(c + HP) % SZ]), pack2(wi[c % SZ], wi[(c + HP) % SZ]));
        // the block's scalars
        const int sl = (lane % BPR) * SZ;
        const float w00 = __shfl_sync(FULL, wr[0], sl), mus = __shfl_sync(FULL, mub, sl);
        const int Ks = __shfl_sync(FULL, imK, sl), as = __shfl_sync(FULL, act ? 1 : 0, sl);
        const unsigned long long sqs = __shfl_sync(FULL, (unsigned long long)sq, sl);
        if (mine) {
            W0 = w00;
            mu = mus;
            K = Ks;
            active = as != 0;
            seq = reinterpret_cast<int16_t*>(sqs);
        }
        if (valid && !act && ts == 0) empty_block(sq, imK, a.empty);
    }
    __syncwarp();

    // ---- a4-a8 ----
    f32x2 wf[SZ][HP];
#pragma unroll
    for (int r = 0; r < SZ; ++r)
#pragma unroll
        for (int j = 0; j < HP; ++j) {
            const float* w = swf + r * SZ + j;
            wf[r][j] = pack2(w[0], w[HP]);
        }
    const ulonglong2* Wb = Wd + entry(lane, 0);   // this block's W rows (entry stride IL)
#pragma unroll
    for (int e = 0; e < SZ * SZ; ++e) G[e * 32] = make_float2(0.f, 0.f);
    const float cg = active ? a.mth.gamma * (1.f / W0) : 0.f;   // c = R[u,v] gamma / W[0,0] (Eqs. 10, 11)
    int left = active ? K : 0;                                  // iterations still to commit
    float ar = mu, ai = 0.f;      // DC phase: R = a W + Q
    int u = 0, v = 0;             // shift and coefficient of the next pass: the DC objective
    float cr = -ar, ci = -ai;
    unsigned rm[SZ];              // row maxima (objectives are >= +0: their bits order like the values)

    // Eq. (12) and the objectives; keep: the rows stay as they were (DC phase)
    auto pass = [&](bool mixed, bool keep) {
        const f32x2 ncr2 = pack2(-cr, -cr), ci2 = pack2(ci, ci), nci2 = pack2(-ci, -ci);
        const int s = (SZ - v) & (SZ - 1);
#pragma unroll
        for (int r = 0; r < SZ; ++r) {
            const ulonglong2* row = Wb + (((r - u) & (SZ - 1)) * EW + s) * IL;
            float m = 0.f;
#pragma unroll
            for (int j = 0; j < HP; ++j) {
                const ulonglong2 w = row[j * IL];
                const f32x2 nr = ffma2(ncr2, w.x, ffma2(ci2, w.y, zr[r][j]));
                const f32x2 ni = ffma2(ncr2, w.y, ffma2(nci2, w.x, zi[r][j]));
                float o0, o1;
                unpack2(objective2(nr, ni, wf[r][j]), o0, o1);
                m = j == 0 ? fmaxf(o0, o1) : max3(m, o0, o1);
                if (!mixed || !keep) {
                    zr[r][j] = nr;
                    zi[r][j] = ni;
                }
            }
            rm[r] = __float_as_uint(m);
        }
    };
    // a5: block maximum, the lowest row holding it, its lowest column
    int pu = 0, pv = 0;
    float pr = 0.f, pi = 0.f;   // the pick and its value
    auto select = [&](bool mixed, bool keep) {
        unsigned c2 = 0;   // of columns 0 and 2: 0 column 0 has M, 1 column 2, 2 neither
        const unsigned M = max(max(rm[0], rm[1]), max(rm[2], rm[3]));
        // all rows in this lane: the lowest with M by selects
        const bool hi = rm[0] != M && rm[1] != M;
        const bool odd = hi ? rm[2] != M : rm[0] != M;
        pu = (hi ? 2 : 0) + (odd ? 1 : 0);
        f32x2 qr[HP], qi[HP];
#pragma unroll
        for (int j = 0; j < HP; ++j) {
            const f32x2 r0 = odd ? zr[1][j] : zr[0][j], r1 = odd ? zr[3][j] : zr[2][j];
            const f32x2 i0 = odd ? zi[1][j] : zi[0][j], i1 = odd ? zi[3][j] : zi[2][j];
            const f32x2 w0 = odd ? wf[1][j] : wf[0][j], w1 = odd ? wf[3][j] : wf[2][j];
            qr[j] = hi ? r1 : r0;
            qi[j] = hi ? i1 : i0;
            if (mixed && keep) {   // DC phase: the rows hold Q
                const ulonglong2 w = Wb[(pu * EW + j) * IL];
                const f32x2 ar2 = pack2(ar, ar), ai2 = pack2(ai, ai), nai2 = pack2(-ai, -ai);
                const f32x2 q = qr[j];
                qr[j] = ffma2(ar2, w.x, ffma2(nai2, w.y, q));
                qi[j] = ffma2(ar2, w.y, ffma2(ai2, w.x, qi[j]));
            }
            float o0, o1, a0, a1, b0, b1;
            unpack2(objective2(qr[j], qi[j], hi ? w1 : w0), o0, o1);
            unpack2(qr[j], a0, a1);
            unpack2(qi[j], b0, b1);
            // columns j, j + 2: the lowest column wins
            const bool h0 = __float_as_uint(o0) == M, h1 = __float_as_uint(o1) == M;
            if (j == 0) {
                pv = h0 ? 0 : 2;
                pr = h0 ? a0 : a1;
                pi = h0 ? b0 : b1;
                c2 = h0 ? 0u : (h1 ? 1u : 2u);
            } else {
                const bool t0 = h0 && c2 != 0u, t1 = h1 && !h0 && c2 == 2u;
                pv = t0 ? 1 : t1 ? 3 : pv;
                pr = t0 ? a0 : t1 ? a1 : pr;
                pi = t0 ? b0 : t1 ? b1 : pi;
            }
        }
    };
    // a6 (Eqs. 10, 11): c = gamma p into G (over S^2), the recorded index
    auto commit = [&](float dr, float di) {
        if (seq != nullptr) *seq++ = (int16_t)(pu * SZ + pv);
        float2 g = G[(pu * SZ + pv) * 32];
        g.x += dr;
        g.y += di;
        G[(pu * SZ + pv) * 32] = g;
        --left;
    };

    // While a block of the warp is in its DC phase or leaves it (fold: the
    // pass that stores a W + Q; its pick is then still to be applied).
    bool dc = true, fold = false;
    while (__any_sync(FULL, left > 0 && (dc || fold))) {
        pass(true, dc);
        const int ou = pu, ov = pv;
        const float orr = pr, oi = pi;
        select(true, dc);
        if (fold) {
            pu = ou;
            pv = ov;
            pr = orr;
            pi = oi;
            fold = false;
            u = pu;
            v = pv;
            cr = pr * cg;
            ci = pi * cg;
        } else {
            const float dr = pr * cg, di = pi * cg;
            if (left > 0) commit(dr, di);
            u = pu;
            v = pv;
            cr = dr;
            ci = di;
            if (dc) {
                if ((pu | pv) == 0) {
                    ar -= dr;
                    ai -= di;
                } else {
                    dc = false;
                    fold = true;
                }
                u = v = 0;
                cr = -ar;
                ci = -ai;
            }
        }
    }
    int trips = left;
#pragma unroll
    for (int s = 16; s > 0; s >>= 1) trips = max(trips, __shfl_xor_sync(FULL, trips, s));
    // (a block that is done keeps iterating on values nobody reads)
    for (; trips > 0; --trips) {
        pass(false, false);
        select(false, false);
        u = pu;
        v = pv;
        cr = pr * cg;
        ci = pi * cg;
        if (left > 0) commit(cr, ci);
    }

    // ---- a9: write-back of the B x B target ----
    if (lane < nblk) {
        const long long item = queue[lane];
        const int lo = image_of(a, item);
        const ImageArgs* im = a.images + lo;
        const int nbx = im->nbx, pitch = im->pitch;
        const long long blk = item - __ldg(a.first + lo);
        const int by = (int)(blk / nbx), bx = (int)(blk - (long long)by * nbx);
        float g[SZ * SZ];
        inverse4(G, g);
        constexpr int LB = (SZ - B) / 2;   // = L: the target's place in the support
#pragma unroll
        for (int q = 0; q < B * B; ++q) {
            const int ty = by * B + q / B, tx = bx * B + q % B;
            if (ty < im->H && tx < im->W) {
                const size_t off = (size_t)ty * pitch + tx;
                const bool kn = __ldg(im->mask + off) != 0;
                im->out[off] = kn ? __ldg(im->img + off) : g[(LB + q / B) * SZ + LB + q % B];
            }
        }
    }
    __syncwarp();
}

// 12 warps per SM (3 CTAs of 4, 146 registers): 1280 x 720 94 us at the time; 10 warps 103,
// 14 (2 CTAs of 7, 128 registers) 117.
constexpr int kWarpsQuad = 4;
constexpr int kCtasQuad = 3;

// per: blocks a warp works on at once.
template <int B>
__global__ void __launch_bounds__(kWarpsQuad * 32, kCtasQuad) fsr_quad_kernel(const BatchArgs a, int per) {
    extern __shared__ __align__(128) unsigned char smem[];
    float* sw0 = reinterpret_cast<float*>(smem + kW0Off);
    float* swf = reinterpret_cast<float*>(smem + kWfOff);
    const int lane = threadIdx.x & 31;
    unsigned char* area = smem + kWarp0Off + kPerWarp * (threadIdx.x >> 5);

    // tables: Eq. (5) without the known-set factor, Eq. (9)
    const float hs = float(SZ) / 2.f;
    for (int i = threadIdx.x; i < SZ * SZ; i += blockDim.x) {
        const int m = i / SZ, n = i % SZ;
        const float dm = float(m) - float(SZ - 1) / 2.f, dn = float(n) - float(SZ - 1) / 2.f;
        sw0[i] = powf(a.mth.rho, sqrtf(dm * dm + dn * dn));
        float wfv = 1.f;
        if (a.mth.freq_weight) {
            const float kt = hs - fabsf(float(m) - hs), lt = hs - fabsf(float(n) - hs);
            const float r = sqrtf(kt * kt / float(SZ * SZ) + lt * lt / float(SZ * SZ));
            const float b = 1.f - sqrtf(2.f) * r;
            wfv = b * b;
        }
        swf[i] = wfv;
    }
    __syncthreads();

    long long* queue = reinterpret_cast<long long*>(area + kQOff);
    for_queued_blocks<B>(a, (int)gridDim.x * kWarpsQuad, per, queue, lane,
                         [&](int nblk) { run_blocks<B>(a, nblk, sw0, swf, area, lane); });
}

template <int B>
cudaError_t configure_one() {
    return cudaFuncSetAttribute(fsr_quad_kernel<B>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)smem_bytes(kWarpsQuad));
}

template <int B>
cudaError_t launch_one(const BatchArgs& a, int chunk, int sm_count, cudaStream_t stream) {
    const size_t smem = smem_bytes(kWarpsQuad);
    // A warp takes 32 blocks at a time, or fewer (whole rounds of the
    // transforms) while that still gives each of an SM's four schedulers a
    // warp: a small image then pays one round of transforms and not four.
    const long long slots = 4ll * sm_count;
    const long long even = ((a.total + slots - 1) / slots + BPR - 1) / BPR * BPR;
    const int per = even < BPW ? (int)even : BPW;
    int grid = 0;
    const long long take = (long long)per * chunk;
    cudaError_t e = persistent_grid(fsr_quad_kernel<B>, kWarpsQuad, smem, (a.total + take - 1) / take, sm_count, &grid);
    if (e != cudaSuccess) return e;
    fsr_quad_kernel<B><<<grid, kWarpsQuad * 32, smem, stream>>>(a, per);
    return cudaGetLastError();
}

}  // namespace

cudaError_t configure_quad() {
    const cudaError_t e = configure_one<2>();
    return e != cudaSuccess ? e : configure_one<4>();
}

// FP32, S = 4
cudaError_t launch_quad(const BatchArgs& a, int B, int chunk, int sm_count, cudaStream_t stream) {
    if (B == 2) return launch_one<2>(a, chunk, sm_count, stream);
    if (B == 4) return launch_one<4>(a, chunk, sm_count, stream);
    return cudaErrorNotSupported;
}

}  // namespace fsrk
