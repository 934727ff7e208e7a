// FP32 overlap-save Toeplitz product for the large single-CTA blocks (2^14 and 2^15 reals):
// a persistent, warp-specialised kernel (see toeplitz.cuh for the tiles and the product).
//
// A block's input is gathered from the map through the pointing, which waits on memory; its
// transforms wait on issue slots and shared memory.  Run one after the other by the same
// threads (one 136 KB block per SM) neither uses what the other leaves idle: the gather took
// 40 % of a block's time, transforms and product 49 %, stores 11 %.  Here a CTA walks over its
// blocks with two kinds of warps: the gather warps form P x of the next block into a scratch
// buffer of the CTA (two of B floats in global memory, read back through L2, which writes most
// of them to memory all the same: 127 MB of DRAM writes a launch, 67 of them output) while the
// transform warps work on the current one; one CTA-wide barrier per block swaps them.  A CTA's
// blocks are consecutive windows: where their distance is a multiple of four, the 2 lambda
// positions that two windows share are copied from buffer to buffer instead of gathered twice.
//
// Measured (I/Q/U, 2^24 samples, lambda = 4096, 736 blocks): 153 -> 118 us, of which 11 us are
// the first block's gather (nothing to overlap it with); per block 38k cycles of transform,
// 40k of gather beside it.  T, 2^26 samples, lambda = 1024: 405 -> 291 us.  Bound by the
// latency of shared memory and barriers in the transform and of L2 in the gather.
//
// Transform of N = 2^LOGN packed points, in place (no second copy of the block fits):
//   forward   natural order in, bit-reversed out: sub-block b of 2^l takes the twiddle of its
//             own roots (x^2m - w^2 = (x^m - w)(x^m + w)), the same for all its points,
//   inverse   bit-reversed in, natural out (decimation in time).
// Passes: radix 16 (inputs from the scratch buffer), 16, 16, then a middle pass that does the
// last forward radix RM = N / 4096, the spectrum product and the first inverse radix RM in
// registers (a thread holds the sub-blocks of bins k0 and 4096 - k0, which contain every
// mirrored pair k, N - k of theirs), then 16, 16, 16, whose results go straight to global
// memory: six trips of the block through shared memory where separate load, product and store
// phases took eight and a half.  The 16-point butterflies run two at a time on packed FP32
// (f32x2).  After the first pass a block of N / 16 points belongs to a warp (or half a warp)
// until the last one, but for the middle pass, which mirrors blocks 2^m .. 2^(m+1) - 1 onto
// themselves: the passes between need barriers of 32 to 256 threads only, so that some warps
// load while others compute.  Twiddles come from tables formed in FP64.
#include "toeplitz.cuh"

namespace mm {

// ------------------------------------------------------------------------- layout
// Threads of the transform role: two 16-point butterflies each; as many gather.  Registers:
// the launch gives every thread 64, and the roles share them out again, 88 and 40.
template <int LOGN> __host__ __device__ constexpr int ws_nf() { return (1 << LOGN) / 32; }
template <int LOGN> __host__ __device__ constexpr int ws_threads() { return 2 * ws_nf<LOGN>(); }
constexpr int WS_REG_FFT = 88, WS_REG_GATHER = 40;

// Shared layout: two planes of N floats (real parts, imaginary parts), two floats of padding
// after every 32, so that the passes' 8-byte accesses meet no bank conflicts; then the
// twiddle tables of the inner passes (float4 entries): powers t^1 .. t^15 by power and class,
// (c, c, s, s) for forward pass 2, whose two butterflies share a class, and (c, c', s, s') of
// two neighbouring positions for the inverse passes; (c, s) of t and t^4 for forward pass 3.
// Behind them, in global memory only: (t, t^4) of two neighbouring positions for the last
// pass, by thread, and t and its square root, the split's
// twiddle, of the middle pass's tasks.
template <int LOGN>
struct WsTab {
    static constexpr int N = 1 << LOGN;
    static constexpr int NF = N / 32;
    static constexpr int RM = N / 4096;           // radix of the middle pass: 2 or 4
    static constexpr int F2 = 0;                  // per block of N / 16
    static constexpr int F3 = F2 + 15 * 16;       // per block of N / 256
    static constexpr int I3 = F3 + 256;           // per pair of positions below RM
    static constexpr int I2 = I3 + 15 * RM / 2;   // per pair of positions below 16 RM
    static constexpr int LT = I2 + 15 * RM * 8;   // global: last pass
    static constexpr int MT = LT + 2 * NF;        // global: middle pass
    static constexpr size_t BYTES = sizeof(float4) * LT;
    static constexpr int PLANE = N + N / 16;
    static constexpr size_t DATA = sizeof(float) * 2 * PLANE;
};
constexpr int WS_TASKS = 2048;                    // pairs of sub-blocks in the middle pass

static int brv(int v, int bits) {
    int r = 0;
    for (int i = 0; i < bits; ++i) r |= ((v >> i) & 1) << (bits - 1 - i);
    return r;
}

// Sub-blocks of RM bins that a task of the middle pass holds: positions p and pm of 4096,
// whose bins are k0 + 4096 s and 4096 - k0 + 4096 s (k0 = bit-reversed p).  Negation of k0
// keeps the highest set bit of p and flips those below it, so within [2^m, 2^(m+1)) the
// partner runs backwards: neighbouring tasks hold neighbouring sub-blocks.  Positions 0 and 1
// (k0 = 0 and 2048) are their own partners; task 0 holds both.  hb: highest power of two <=
// task (0 for task 0).
__host__ __device__ inline void ws_task(int task, int hb, int& p, int& pm) {
    p = task + hb;
    pm = task == 0 ? 1 : 5 * hb - 1 - task;
}
static void ws_task_host(int task, int& p, int& pm) {
    int hb = 0;
    if (task > 0)
        for (hb = 1; 2 * hb <= task;) hb *= 2;
    ws_task(task, hb, p, pm);
}

// Tables in WsTab's order.
std::vector<float> ws_tables(int logn) {
    const int N = 1 << logn, RM = N / 4096;
    std::vector<float> out;
    auto cs = [&](double turns, bool sine) {
        const double th = 2.0 * 3.14159265358979323846 * turns;
        out.push_back((float)(sine ? std::sin(th) : std::cos(th)));
    };
    auto two = [&](double a, double b) {   // (c_a, c_b, s_a, s_b)
        cs(a, false);
        cs(b, false);
        cs(a, true);
        cs(b, true);
    };
    auto one = [&](double a) {   // (c, s)
        cs(a, false);
        cs(a, true);
    };
    // block b of 2^l, radix 16: t = exp(-pi i brv_l(b) / 2^(l+3))
    for (int r = 1; r < 16; ++r)
        for (int b = 0; b < 16; ++b) two(-r * brv(b, 4) / 256.0, -r * brv(b, 4) / 256.0);
    for (int b = 0; b < 256; ++b) {
        one(-brv(b, 8) / 4096.0);
        one(-4 * brv(b, 8) / 4096.0);
    }
    // position j of a block of 16 S, radix 16, parts exchanged: t = exp(-2 pi i j / (16 S))
    for (int S : {RM, 16 * RM})
        for (int r = 1; r < 16; ++r)
            for (int j = 0; j < S; j += 2) two(-r * j / (16.0 * S), -r * (j + 1) / (16.0 * S));
    for (int r : {1, 4})
        for (int j = 0; j < N / 16; j += 2) two(-(double)r * j / N, -(double)r * (j + 1) / N);
    for (int task = 0; task < WS_TASKS; ++task) {
        int p, pm;
        ws_task_host(task, p, pm);
        one(-(double)brv(p, 12) / N);
        one(-0.5 * (double)brv(p, 12) / N);
    }
    return out;
}

// Spectra / 4 (split_chain) in the order of the middle pass, per PSD: two arrays
// [WS_TASKS][RM], of the bins k0 + 4096 s of a task's first sub-block and of their partners
// N - k; then [RM], the first RM / 2 bins of sub-block 1 (task 0) and their partners.
int64_t ws_spectrum_size(int logn) { return (int64_t)(2 * WS_TASKS + 1) * ((1 << logn) / 4096); }

void ws_append_spectrum(const std::vector<double>& h, int logn, std::vector<float>& out) {
    const int N = 1 << logn, RM = N / 4096;
    const int64_t part = (int64_t)WS_TASKS * RM;
    const size_t at = out.size();
    out.resize(at + (size_t)ws_spectrum_size(logn));
    float* o = out.data() + at;
    for (int task = 0; task < WS_TASKS; ++task) {
        int p, pm;
        ws_task_host(task, p, pm);
        const int k0 = brv(p, 12);
        for (int e = 0; e < RM; ++e) {
            o[(int64_t)task * RM + e] = (float)(0.25 * h[(size_t)(k0 + 4096 * e)]);
            o[part + (int64_t)task * RM + e] = (float)(0.25 * h[(size_t)(N - k0 - 4096 * e)]);
        }
    }
    for (int e = 0; e < RM / 2; ++e) {
        o[2 * part + e] = (float)(0.25 * h[(size_t)(2048 + 4096 * e)]);
        o[2 * part + RM / 2 + e] = (float)(0.25 * h[(size_t)(N - 2048 - 4096 * e)]);
    }
}

// ---------------------------------------------------------------------- butterflies
constexpr float WS_C1 = 0.92387953251128675613f, WS_S1 = 0.38268343236508977173f, WS_H = 0.70710678118654752440f;

__device__ __forceinline__ float2 mulc(float2 a, float2 b) {
    return make_float2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x));
}

// ------------------------------------------------- two butterflies at a time (f32x2)
// Blackwell's packed FP32 instructions work on two values per register pair: half the issue
// slots of scalar code, which is what bounds the passes.  The two lanes are two neighbouring
// butterflies, the parts of a value two register pairs.
typedef unsigned long long f2;
__device__ __forceinline__ f2 pk(float a, float b) {
    f2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ float2 upk(f2 a) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(a));
    return r;
}
__device__ __forceinline__ f2 add2(f2 a, f2 b) {
    f2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f2 sub2(f2 a, f2 b) {
    f2 r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f2 mul2(f2 a, f2 b) {
    f2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) {
    f2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
struct cx2 {
    f2 re, im;
};
__device__ __forceinline__ cx2 add2(cx2 a, cx2 b) { return {add2(a.re, b.re), add2(a.im, b.im)}; }
__device__ __forceinline__ cx2 sub2(cx2 a, cx2 b) { return {sub2(a.re, b.re), sub2(a.im, b.im)}; }
__device__ __forceinline__ cx2 mul2(cx2 a, cx2 w) {
    return {sub2(mul2(a.re, w.re), mul2(a.im, w.im)), fma2(a.re, w.im, mul2(a.im, w.re))};
}
__device__ __forceinline__ cx2 entry2(float4 e) { return {pk(e.x, e.y), pk(e.z, e.w)}; }

// forward 4-point DFT, natural order in and out
__device__ __forceinline__ void dft4x2(cx2& a0, cx2& a1, cx2& a2, cx2& a3) {
    const cx2 t0 = add2(a0, a2), t1 = sub2(a0, a2), t2 = add2(a1, a3), d = sub2(a1, a3);
    a0 = add2(t0, t2);
    a2 = sub2(t0, t2);
    a1 = {add2(t1.re, d.im), sub2(t1.im, d.re)};
    a3 = {sub2(t1.re, d.im), add2(t1.im, d.re)};
}

// forward 16-point DFT, natural order in and out (4 x 4, as dft16 in toeplitz.cuh)
__device__ __forceinline__ void dft16x2(cx2* v) {
    const cx2 w1 = {pk(WS_C1, WS_C1), pk(-WS_S1, -WS_S1)}, w3 = {pk(WS_S1, WS_S1), pk(-WS_C1, -WS_C1)};
    const f2 h = pk(WS_H, WS_H);
#pragma unroll
    for (int n = 0; n < 4; ++n) dft4x2(v[n], v[4 + n], v[8 + n], v[12 + n]);
    auto w2 = [&](cx2 a) -> cx2 {   // (1 - i) / sqrt 2
        return {mul2(h, add2(a.re, a.im)), mul2(h, sub2(a.im, a.re))};
    };
    // element n + 4 k: W16^(n k)
    v[5] = mul2(v[5], w1);
    v[9] = w2(v[9]);
    v[13] = mul2(v[13], w3);
    v[6] = w2(v[6]);
    {
        const cx2 t = v[14];   // W16^6 = -i (1 - i) / sqrt 2
        v[14] = {mul2(h, sub2(t.im, t.re)), mul2(pk(-WS_H, -WS_H), add2(t.re, t.im))};
    }
    v[7] = mul2(v[7], w3);
    {
        const cx2 t = v[11];   // W16^6
        v[11] = {mul2(h, sub2(t.im, t.re)), mul2(pk(-WS_H, -WS_H), add2(t.re, t.im))};
    }
    {
        const cx2 t = v[15];   // W16^9 = -w1
        v[15] = mul2(t, cx2{pk(-WS_C1, -WS_C1), pk(WS_S1, WS_S1)});
    }
    // W16^4 = -i on element 10, taken in the second stage
    const cx2 t10 = v[10];
    v[10] = {t10.im, sub2(pk(0.f, 0.f), t10.re)};
#pragma unroll
    for (int k = 0; k < 4; ++k) dft4x2(v[4 * k], v[4 * k + 1], v[4 * k + 2], v[4 * k + 3]);
    // outputs k + 4 m sit at 4 k + m
#pragma unroll
    for (int k = 0; k < 4; ++k)
#pragma unroll
        for (int m = k + 1; m < 4; ++m) {
            const cx2 t = v[4 * k + m];
            v[4 * k + m] = v[4 * m + k];
            v[4 * m + k] = t;
        }
}

// v[r] *= t^r from a table of powers of NCL classes
template <int NCL>
__device__ __forceinline__ void scale_table(cx2* v, const float4* e) {
#pragma unroll
    for (int r = 1; r < 16; ++r) v[r] = mul2(v[r], entry2(e[(r - 1) * NCL]));
}
// v[r] *= t^r from t and t^4: at most four roundings
__device__ __forceinline__ void scale_powers(cx2* v, cx2 t, cx2 t4) {
    cx2 w[4], W = t4;
    w[1] = t;
    w[2] = mul2(t, t);
    w[3] = mul2(t, w[2]);
#pragma unroll
    for (int b = 1; b < 4; ++b) v[b] = mul2(v[b], w[b]);
#pragma unroll
    for (int a = 1; a < 4; ++a) {
        v[4 * a] = mul2(v[4 * a], W);
#pragma unroll
        for (int b = 1; b < 4; ++b) v[4 * a + b] = mul2(v[4 * a + b], mul2(W, w[b]));
        if (a == 1) W = mul2(t4, t4);
        if (a == 2) W = mul2(t4, W);
    }
}

__host__ __device__ constexpr int brv4(int r) { return ((r & 1) << 3) | ((r & 2) << 1) | ((r & 4) >> 1) | ((r & 8) >> 3); }

template <int ID, int COUNT>
__device__ __forceinline__ void named_sync() {
    asm volatile("bar.sync %0, %1;" ::"n"(ID), "n"(COUNT) : "memory");
}

// Barrier of the warps whose N / 16-point blocks mirror each other in the middle pass: 0, 1,
// 2-3, 4-7, 8-15.
__device__ __forceinline__ void group_sync(int warp) {
    if (warp < 2) {
        __syncwarp();
    } else {
        const int id = warp < 4 ? 3 : warp < 8 ? 4 : 5, count = warp < 4 ? 64 : warp < 8 ? 128 : 256;
        asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(count) : "memory");
    }
}

// --------------------------------------------------------------------- input of a block
// y[pb .. pe) = the samples at times pb + d .., by NT threads of rank g.  Load modes 0-3 as
// in load_block, mode 3 with the packed map; mode 6: the I/Q/U map unpacked.  U positions in
// flight per thread, the pixel indices of the next U requested before the current ones'
// weights and map values are used; no branch stands between the loads of a round.
constexpr int WS_IQU = 6;

// L2 prefetch of the streamed inputs of positions [p, min(p + WS_PF, pe)) of a segment.  The
// gather warps ask for a chunk one chunk ahead of its use: a whole block ahead (60 MB over the
// SMs) was evicted again before it was read.
constexpr int WS_PF = 4096;

template <int MODE>
__device__ __forceinline__ void ws_prefetch(const TzArgs<float>& A, int64_t roff, int p, int pe, int64_t d) {
    const int64_t n = min(WS_PF, pe - p);
    if (n <= 0) return;
    if constexpr (MODE == 0) l2_prefetch(A.y + roff + d + p, n * 4);
    else if constexpr (MODE == 2) l2_prefetch(A.yd + roff + d + p, n * 8);
    else {
        l2_prefetch(A.pixc + d + p, n * 4);
        if constexpr (MODE != 1) l2_prefetch(A.w + d + p, n * 8);
    }
}

// Slot of block position p in the input buffer: even positions (real parts) first, then odd.
template <int B>
__device__ __forceinline__ int ws_slot(int p) { return (p & 1) * (B / 2) + (p >> 1); }

// One round: positions s + u NT, u < U, whose pixel indices are in q, into y[u NT / 2] (their
// slots: ws_slot); END: those from pe on are left out (they read the last sample).
template <int MODE, int NT, int U, bool END>
__device__ __forceinline__ void ws_round(const TzArgs<float>& A, const float* __restrict__ x,
                                         const float2* __restrict__ pw, float* __restrict__ y, int s, int pe,
                                         const int (&q)[U]) {
    float r[U];
    if constexpr (MODE == 1) {
#pragma unroll
        for (int u = 0; u < U; ++u) r[u] = __ldg(x + max(q[u], 0));
    } else {
        float2 w[U];
        float m[U][3];
#pragma unroll
        for (int u = 0; u < U; ++u) w[u] = __ldg(pw + (END ? min(s + u * NT, pe - 1) : s + u * NT));
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if constexpr (MODE == 3) {
                const float4 v = __ldg(A.x4 + max(q[u], 0));
                m[u][0] = v.x;
                m[u][1] = v.y;
                m[u][2] = v.z;
            } else {
                const float* xq = x + 3 * (int64_t)max(q[u], 0);
                m[u][0] = __ldg(xq);
                m[u][1] = __ldg(xq + 1);
                m[u][2] = __ldg(xq + 2);
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) r[u] = fmaf(w[u].y, m[u][2], fmaf(w[u].x, m[u][1], m[u][0]));
    }
#pragma unroll
    for (int u = 0; u < U; ++u)
        if (!END || s + u * NT < pe) y[u * (NT / 2)] = q[u] >= 0 ? r[u] : 0.f;
}

template <int B, int MODE, int NT>
__device__ __forceinline__ void ws_fill_segment(const TzArgs<float>& A, int64_t roff, float* __restrict__ y, int pb,
                                                int pe, int64_t d, int g) {
    constexpr int U = MODE == 3 || MODE == WS_IQU ? 4 : 8;
    const int last = pe - 1;
    if constexpr (MODE == 0 || MODE == 2) {
        const float* yt = A.y + roff + d;
        const double* yd = A.yd + roff + d;
#pragma unroll 1
        for (int s = pb + g; s < pe; s += NT * U) {
            if (g == 0 && (s - pb) % WS_PF < NT * U) ws_prefetch<MODE>(A, roff, s + WS_PF, pe, d);
            float v[U];
            double dv[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int p = min(s + u * NT, last);
                if constexpr (MODE == 0) v[u] = __ldg(yt + p);
                else dv[u] = __ldg(yd + p);
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if constexpr (MODE == 2) v[u] = (float)dv[u];
                if (s + u * NT < pe) y[ws_slot<B>(s) + u * (NT / 2)] = v[u];
            }
        }
    } else {
        const int32_t* __restrict__ pq = A.pixc + d;
        const float2* __restrict__ pw = A.w + d;
        const float* __restrict__ x = A.x + roff;
        int s = pb + g;
        int q[U];
#pragma unroll
        for (int u = 0; u < U; ++u) q[u] = __ldg(pq + min(s + u * NT, last));
        // whole rounds; the indices of the round after are requested first (PIXC_PAD: they may
        // lie past the last sample)
#pragma unroll 1
        for (; s + (U - 1) * NT < pe; s += NT * U) {
            if (g == 0 && (s - pb) % WS_PF < NT * U) ws_prefetch<MODE>(A, roff, s + WS_PF, pe, d);
            int qn[U];
#pragma unroll
            for (int u = 0; u < U; ++u) qn[u] = __ldg(pq + s + (U + u) * NT);
            ws_round<MODE, NT, U, false>(A, x, pw, y + ws_slot<B>(s), s, pe, q);
#pragma unroll
            for (int u = 0; u < U; ++u) q[u] = qn[u];
        }
        if (s < pe) ws_round<MODE, NT, U, true>(A, x, pw, y + ws_slot<B>(s), s, pe, q);
    }
}

// y[0 .. B) = the block's positions: its segments, and zeros around them.  prev: null, or the
// input of the window before this one in the same run (Tile::cont = the windows' distance),
// whose last positions are this one's first: they are copied instead of gathered again.
template <int B, int MODE, int NT>
__device__ __forceinline__ void ws_fill(const TzArgs<float>& A, const Tile* tp, int64_t roff, float* __restrict__ y,
                                        const float* prev, int g) {
    int at = 0;
    if (prev != nullptr) {
        const int lv = tp->cont;   // a multiple of 4
        at = B - lv;
        // slots come in pairs: 2 g of either plane from slot 2 g + lv / 2
        constexpr int U = 8;
#pragma unroll 1
        for (int m = 2 * g; m < at; m += 2 * NT * U) {
            float2 v[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int mu = min(m + 2 * NT * u, at - 2);
                v[u] = __ldcg(reinterpret_cast<const float2*>(prev + (mu < at / 2 ? mu : mu - at / 2 + B / 2) + lv / 2));
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int mu = min(m + 2 * NT * u, at - 2);   // past the end: the last pair again
                *reinterpret_cast<float2*>(y + (mu < at / 2 ? mu : mu - at / 2 + B / 2)) = v[u];
            }
        }
    }
#pragma unroll 1
    for (int sg = 0; sg < TILE_SEGS; ++sg) {
        const int pb = min(max(tp->pb[sg], at), B), pe = min(tp->pe[sg], B);   // unused segments: empty
        for (int p = at + g; p < pb; p += NT) y[ws_slot<B>(p)] = 0.f;
        if (pb < pe) ws_fill_segment<B, MODE, NT>(A, roff, y, pb, pe, tp->d[sg], g);
        at = max(at, pe);
    }
    for (int p = at + g; p < B; p += NT) y[ws_slot<B>(p)] = 0.f;
}

// The blocks of a CTA: units of `span` consecutive tiles of one right-hand side (unit u: tiles
// from span (u / R) on, right-hand side u % R), the CTA's units gridDim.x apart.
struct WsWalk {
    int unit, tile, end;
    __device__ __forceinline__ void start(int u, int span, int ntiles, int R) {
        unit = u;
        tile = (u / R) * span;
        end = min(tile + span, ntiles);
    }
    __device__ __forceinline__ bool valid(int units) const { return unit < units; }
    __device__ __forceinline__ void next(int span, int ntiles, int R) {
        if (++tile == end) start(unit + gridDim.x, span, ntiles, R);
    }
};

// ------------------------------------------------------------------- transform of a block
__host__ __device__ __forceinline__ constexpr int ws_pad(int i) { return i + 2 * (i >> 5); }
__device__ __forceinline__ f2 ld2(const float* p) { return *reinterpret_cast<const f2*>(p); }
__device__ __forceinline__ void st2(float* p, f2 v) { *reinterpret_cast<f2*>(p) = v; }

// Two neighbouring 16-point butterflies at positions s + r STRIDE (planes re and im = re +
// PLANE): forward, natural positions in, bit-reversed bins out; inverse, bit-reversed in,
// natural out.  The inverse works on values with their parts exchanged, swap(z) = i conj(z),
// on which the inverse transform is the forward one.
template <int STRIDE, int PLANE, bool INV, typename F>
__device__ __forceinline__ void ws_load16(const float* s, cx2* v, F&& scale) {
#pragma unroll
    for (int r = 0; r < 16; ++r) {
        const int o = ws_pad((INV ? brv4(r) : r) * STRIDE);
        v[r] = {ld2(s + o), ld2(s + PLANE + o)};
    }
    scale(v);
    dft16x2(v);
}
template <int STRIDE, int PLANE, bool INV>
__device__ __forceinline__ void ws_store16(float* s, const cx2* v) {
#pragma unroll
    for (int r = 0; r < 16; ++r) {
        const int o = ws_pad((INV ? r : brv4(r)) * STRIDE);
        st2(s + o, v[r].re);
        st2(s + PLANE + o, v[r].im);
    }
}
template <int STRIDE, int PLANE, bool INV, typename F>
__device__ __forceinline__ void ws_pass16(float* s, F&& scale) {
    cx2 v[16];
    ws_load16<STRIDE, PLANE, INV>(s, v, scale);
    ws_store16<STRIDE, PLANE, INV>(s, v);
}

// RM floats of one task
template <int RM> struct FloatN;
template <> struct FloatN<2> { using type = float2; };
template <> struct FloatN<4> { using type = float4; };
template <int RM>
__device__ __forceinline__ void ldn(float (&d)[RM], const float* p) {
    using V = typename FloatN<RM>::type;
    const V v = __ldg(reinterpret_cast<const V*>(p));
    d[0] = v.x;
    d[1] = v.y;
    if constexpr (RM == 4) {
        d[2] = v.z;
        d[3] = v.w;
    }
}

// RM-point forward DFT
template <int RM>
__device__ __forceinline__ void dftm(float2* v) {
    if constexpr (RM == 4) dft4<float>(v[0], v[1], v[2], v[3]);
    else bfly2<float>(v[0], v[1]);
}

// split_chain (toeplitz.cuh) for two bin pairs at a time, V unconjugated: w = exp(-i pi k / N)
__device__ __forceinline__ void chain2(cx2& u1, cx2& u2, cx2 w, f2 h1, f2 h2) {
    const cx2 E = {add2(u1.re, u2.re), sub2(u1.im, u2.im)};
    const cx2 F = {sub2(u1.re, u2.re), add2(u1.im, u2.im)};   // O = -i F
    const cx2 WO = {fma2(w.re, F.im, mul2(w.im, F.re)), sub2(mul2(w.im, F.im), mul2(w.re, F.re))};
    const cx2 Z1 = {mul2(h1, add2(E.re, WO.re)), mul2(h1, add2(E.im, WO.im))};
    const cx2 Z2 = {mul2(h2, sub2(E.re, WO.re)), mul2(h2, sub2(E.im, WO.im))};
    const cx2 S = add2(Z1, Z2), D = sub2(Z1, Z2);
    const cx2 P = {fma2(w.re, D.re, mul2(w.im, D.im)), sub2(mul2(w.re, D.im), mul2(w.im, D.re))};   // conj(W) D
    u1 = {sub2(S.re, P.im), add2(S.im, P.re)};
    u2 = {add2(S.re, P.im), sub2(P.re, S.im)};
}

// the same for one pair
__device__ __forceinline__ void chain1(float2& u1, float2& u2, float2 w, float h1, float h2) {
    float2 V1, V2;
    split_chain<float>(u1, u2, w.x, -w.y, h1, h2, V1, V2);
    u1 = make_float2(V1.x, -V1.y);
    u2 = make_float2(V2.x, -V2.y);
}

// Sub-blocks sa and sb of one task: last forward radix, product, first inverse radix.
// tw = (t, exp(-i pi k0 / N)).
template <int RM, int PLANE>
__device__ __forceinline__ void ws_middle(float* sa, float* sb, float4 tw, const float (&h1)[RM], const float (&h2)[RM],
                                          bool self, const float* __restrict__ b1) {
    float2 va[RM], vb[RM];
#pragma unroll
    for (int r = 0; r < RM; r += 2) {
        const float2 xa = *reinterpret_cast<const float2*>(sa + r), ya = *reinterpret_cast<const float2*>(sa + PLANE + r);
        const float2 xb = *reinterpret_cast<const float2*>(sb + r), yb = *reinterpret_cast<const float2*>(sb + PLANE + r);
        va[r] = make_float2(xa.x, ya.x);
        va[r + 1] = make_float2(xa.y, ya.y);
        vb[r] = make_float2(xb.x, yb.x);
        vb[r + 1] = make_float2(xb.y, yb.y);
    }
    const float2 t = make_float2(tw.x, tw.y);
    // the second sub-block's root is exp(-2 pi i (4096 - k0) / N) = exp(-2 pi i / RM) conj(t)
    // (task 0: exp(-2 pi i 2048 / N) instead, t = 1 for the first)
    float2 u = RM == 4 ? make_float2(-t.y, -t.x) : make_float2(-t.x, t.y);
    if (self) u = RM == 4 ? make_float2(WS_H, -WS_H) : make_float2(0.f, -1.f);
    va[1] = mulc(va[1], t);
    vb[1] = mulc(vb[1], u);
    if constexpr (RM == 4) {
        const float2 t2 = mulc(t, t), u2 = mulc(u, u);
        va[2] = mulc(va[2], t2);
        va[3] = mulc(va[3], mulc(t, t2));
        vb[2] = mulc(vb[2], u2);
        vb[3] = mulc(vb[3], mulc(u, u2));
    }
    dftm<RM>(va);
    dftm<RM>(vb);
    // twiddle of bin k0 + 4096 s: exp(-i pi k0 / N) times exp(-i pi s / RM)
    if (!self) {
        const float2 w0 = make_float2(tw.z, tw.w);
        float2 w1 = RM == 4 ? mulc(w0, make_float2(WS_H, -WS_H)) : make_float2(w0.y, -w0.x);
        cx2 w = {pk(w0.x, w1.x), pk(w0.y, w1.y)};
#pragma unroll
        for (int s = 0; s < RM; s += 2) {
            const int m = RM - 1 - s;
            cx2 a = {pk(va[s].x, va[s + 1].x), pk(va[s].y, va[s + 1].y)};
            cx2 b = {pk(vb[m].x, vb[m - 1].x), pk(vb[m].y, vb[m - 1].y)};
            if (s == 2) w = {pk(w0.y, w1.y), pk(-w0.x, -w1.x)};   // times -i
            chain2(a, b, w, pk(h1[s], h1[s + 1]), pk(h2[s], h2[s + 1]));
            const float2 ar = upk(a.re), ai = upk(a.im), br = upk(b.re), bi = upk(b.im);
            va[s] = make_float2(ar.x, ai.x);
            va[s + 1] = make_float2(ar.y, ai.y);
            vb[m] = make_float2(br.x, bi.x);
            vb[m - 1] = make_float2(br.y, bi.y);
        }
    } else {
        // k0 = 0: bins 0 and N/2 are their own partners, else s and RM - s; k0 = 2048: s and
        // RM - 1 - s
        float2 x = va[0];
        chain1(va[0], x, make_float2(1.f, 0.f), h1[0], h2[0]);
        x = va[RM / 2];
        chain1(va[RM / 2], x, make_float2(0.f, -1.f), h1[RM / 2], h2[RM / 2]);
        if constexpr (RM == 4) {
            chain1(va[1], va[3], make_float2(WS_H, -WS_H), h1[1], h2[1]);
            chain1(vb[0], vb[3], make_float2(WS_C1, -WS_S1), __ldg(b1), __ldg(b1 + 2));
            chain1(vb[1], vb[2], make_float2(WS_S1, -WS_C1), __ldg(b1 + 1), __ldg(b1 + 3));
        } else {
            chain1(vb[0], vb[1], make_float2(WS_H, -WS_H), __ldg(b1), __ldg(b1 + 1));
        }
    }
#pragma unroll
    for (int s = 0; s < RM; ++s) {
        va[s] = make_float2(va[s].y, va[s].x);
        vb[s] = make_float2(vb[s].y, vb[s].x);
    }
    dftm<RM>(va);
    dftm<RM>(vb);
#pragma unroll
    for (int r = 0; r < RM; r += 2) {
        *reinterpret_cast<float2*>(sa + r) = make_float2(va[r].x, va[r + 1].x);
        *reinterpret_cast<float2*>(sa + PLANE + r) = make_float2(va[r].y, va[r + 1].y);
        *reinterpret_cast<float2*>(sb + r) = make_float2(vb[r].x, vb[r + 1].x);
        *reinterpret_cast<float2*>(sb + PLANE + r) = make_float2(vb[r].y, vb[r + 1].y);
    }
}

template <int LOGN>
__device__ __forceinline__ void ws_transform(const TzArgs<float>& A, const Tile* tp, int rhs, const float* y,
                                             const float* __restrict__ Hall, const float4* __restrict__ gtab,
                                             float* a, const float4* tab, int tid) {
    using TB = WsTab<LOGN>;
    constexpr int N = TB::N, NF = TB::NF, RM = TB::RM, PLANE = TB::PLANE;
    constexpr int S1 = N / 16, S2 = 16 * RM, S3 = RM;    // strides of the radix-16 passes
    const int warp = tid >> 5;
    // forward 1: positions 2 tid and 2 tid + 1, no twiddles
    {
        cx2 v[16];
        const float* yt = y + 2 * tid;
#pragma unroll
        for (int r = 0; r < 16; ++r) {
            const float2 re = __ldcg(reinterpret_cast<const float2*>(yt + r * S1));
            const float2 im = __ldcg(reinterpret_cast<const float2*>(yt + N + r * S1));
            v[r] = {pk(re.x, re.y), pk(im.x, im.y)};
        }
        dft16x2(v);
        ws_store16<S1, PLANE, false>(a + ws_pad(2 * tid), v);
    }
    named_sync<2, NF>();
    // forward 2 and 3
    const int b2 = tid / (S2 / 2), j2 = tid % (S2 / 2);
    float* const s2 = a + b2 * ws_pad(S1) + ws_pad(2 * j2);
    ws_pass16<S2, PLANE, false>(s2, [&](cx2* v) { scale_table<16>(v, tab + TB::F2 + b2); });
    __syncwarp();
    const int b3 = tid / (S3 / 2), j3 = tid % (S3 / 2);
    float* const s3 = a + b3 * ws_pad(S2) + 2 * j3;
    ws_pass16<S3, PLANE, false>(s3, [&](cx2* v) {
        const float4 e = tab[TB::F3 + b3];
        scale_powers(v, {pk(e.x, e.x), pk(e.y, e.y)}, {pk(e.z, e.z), pk(e.w, e.w)});
    });
    // middle: the spectrum values of a task are requested one task ahead
    {
        constexpr int TPT = WS_TASKS / NF;
        const float* H = Hall + tp->psd * ((int64_t)(2 * WS_TASKS + 1) * RM);
        const float4* mt = gtab + TB::MT;
        int task = warp * (32 * TPT) + (tid & 31);
        float h1[RM], h2[RM];
        ldn<RM>(h1, H + task * RM);
        ldn<RM>(h2, H + (WS_TASKS + task) * RM);
        float4 t = __ldg(mt + task);
        group_sync(warp);
#pragma unroll 1
        for (int i = 0; i < TPT; ++i) {
            float n1[RM], n2[RM];
            float4 nt;
            if (i + 1 < TPT) {
                ldn<RM>(n1, H + (task + 32) * RM);
                ldn<RM>(n2, H + (WS_TASKS + task + 32) * RM);
                nt = __ldg(mt + task + 32);
            }
            int p, pm;
            ws_task(task, task == 0 ? 0 : 1 << (31 - __clz(task)), p, pm);
            ws_middle<RM, PLANE>(a + ws_pad(RM * p), a + ws_pad(RM * pm), t, h1, h2, task == 0, H + 2 * WS_TASKS * RM);
#pragma unroll
            for (int s = 0; s < RM; ++s) {
                h1[s] = n1[s];
                h2[s] = n2[s];
            }
            t = nt;
            task += 32;
        }
    }
    group_sync(warp);
    // inverse 3 and 2
    ws_pass16<S3, PLANE, true>(s3, [&](cx2* v) { scale_table<RM / 2>(v, tab + TB::I3 + j3); });
    __syncwarp();
    ws_pass16<S2, PLANE, true>(s2, [&](cx2* v) { scale_table<8 * RM>(v, tab + TB::I2 + j2); });
    const float4 l1 = __ldg(gtab + TB::LT + tid), l4 = __ldg(gtab + TB::LT + NF + tid);
    named_sync<2, NF>();
    // inverse 1; packed point m holds the reals 2m (plane im) and 2m + 1 (plane re), stored at
    // their times
    cx2 v[16];
    ws_load16<S1, PLANE, true>(a + ws_pad(2 * tid), v, [&](cx2* x) { scale_powers(x, entry2(l1), entry2(l4)); });
    // outputs: positions [lo, hi) of a segment, relative to this thread's first point; written
    // from registers where four of them are an aligned word, of at most two segments
    const int base = 4 * tid, lend = A.lambda + tp->nout;
    float* zo = A.z + rhs * A.out_stride + base;
    const bool two = max(tp->pb[1], A.lambda) < min(tp->pe[1], lend);
    const bool fast = ((reinterpret_cast<uintptr_t>(zo + tp->d[0]) |
                        reinterpret_cast<uintptr_t>(zo + (two ? tp->d[1] : tp->d[0]))) & 15) == 0 &&
                      lend <= tp->pb[2];
    if (fast) {
#pragma unroll 1
        for (int g = 0; g < (two ? 2 : 1); ++g) {
            float* z = zo + tp->d[g];
            const int lo = max(tp->pb[g], A.lambda) - base, hi = min(tp->pe[g], lend) - base;
            if (lo >= hi) continue;   // a segment without outputs
#pragma unroll
            for (int r = 0; r < 16; ++r) {
                const float2 e = upk(v[r].im), w = upk(v[r].re);   // even, odd positions
                const int p = 2 * r * S1;
                if (p >= lo && p + 3 < hi) {
                    *reinterpret_cast<float4*>(z + p) = make_float4(e.x, w.x, e.y, w.y);
                } else if (p + 3 >= lo && p < hi) {
                    if (p >= lo) z[p] = e.x;
                    if (p + 1 >= lo && p + 1 < hi) z[p + 1] = w.x;
                    if (p + 2 >= lo && p + 2 < hi) z[p + 2] = e.y;
                    if (p + 3 < hi) z[p + 3] = w.y;
                }
            }
        }
    } else {
        // back to where they came from (read above, by this thread alone), then one by one
        ws_store16<S1, PLANE, true>(a + ws_pad(2 * tid), v);
        named_sync<2, NF>();
        const Tile tile = *tp;
        float* zt = A.z + rhs * A.out_stride;
        for (int n = tid; n < tile.nout; n += NF) {
            const int p = n + A.lambda;
            store_out<float>(tile, zt, A.lambda, n, a[(p & 1 ? 0 : PLANE) + ws_pad(p >> 1)]);
        }
    }
}

template <int LOGN, int MODE>
__global__ void __launch_bounds__(ws_threads<LOGN>(), 1 << (14 - LOGN))
    toeplitz_ws_kernel(TzArgs<float> A, int ntiles, int span, int units, const float4* __restrict__ gtab,
                       const float* __restrict__ H, float* scratch) {
    using TB = WsTab<LOGN>;
    constexpr int B = 2 << LOGN, NF = TB::NF, NG = NF, NT = NF + NG;
    griddep_wait();   // launched as a dependent launch: the previous kernel's outputs
    if (A.done != nullptr && *(volatile const int*)A.done) return;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float* a = reinterpret_cast<float*>(smem_raw);
    float4* tab = reinterpret_cast<float4*>(smem_raw + TB::DATA);
    const int tid = threadIdx.x;
    for (int i = tid; i < (int)(TB::BYTES / sizeof(float4)); i += NT) tab[i] = __ldg(gtab + i);
    __shared__ Tile tsh[2];   // descriptors of the blocks in the two buffers
    float* y0 = scratch + (int64_t)blockIdx.x * 2 * B;
    WsWalk w;
    w.start(blockIdx.x, span, ntiles, A.R);
    // the first block is everybody's
    if (tid == 0) tsh[0] = A.tiles[w.tile];
    ws_fill<B, MODE, NT>(A, A.tiles + w.tile, (w.unit % A.R) * A.in_stride, y0, nullptr, tid);
    __syncthreads();
    if (tid < NF) {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(WS_REG_FFT));
        for (int it = 0; w.valid(units); ++it) {
            ws_transform<LOGN>(A, tsh + (it & 1), w.unit % A.R, y0 + (it & 1) * B, H, gtab, a, tab, tid);
            named_sync<1, NT>();
            w.next(span, ntiles, A.R);
        }
    } else {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(WS_REG_GATHER));
        for (int it = 0; w.valid(units); ++it) {
            const int unit = w.unit;
            w.next(span, ntiles, A.R);
            if (w.valid(units)) {
                const Tile* tp = A.tiles + w.tile;
                float* y = y0 + ((it + 1) & 1) * B;
                if (tid == NF) tsh[(it + 1) & 1] = *tp;
                const float* prev = w.unit == unit && tp->cont != 0 ? y0 + (it & 1) * B : nullptr;
                ws_fill<B, MODE, NG>(A, tp, (w.unit % A.R) * A.in_stride, y, prev, tid - NF);
            }
            named_sync<1, NT>();
        }
    }
}

bool ws_supported(int logn) { return logn == 13 || logn == 14; }

// CTAs launched at most: the resident ones (one of 2^15 reals, two of 2^14, per SM)
static int ws_ctas(int logn, int num_sms) { return num_sms << (14 - logn); }
// Two buffers of B floats per CTA: 262 KB per SM for either block.  One set per plan: all of
// its launches, of its own block and the batch's, run one after the other on its stream.
size_t ws_scratch_floats(int num_sms) { return (size_t)ws_ctas(14, num_sms) * 2 * (size_t(2) << 14); }

template <int LOGN>
static void ws_launch(const TzArgs<float>& A, const ToeplitzDev& tz, int num_sms, int mode, cudaStream_t s) {
    using TB = WsTab<LOGN>;
    static_assert(TB::BYTES % sizeof(float4) == 0, "tables are copied as float4");
    void (*kern)(TzArgs<float>, int, int, int, const float4*, const float*, float*) = nullptr;
    switch (mode) {
        case 0: kern = toeplitz_ws_kernel<LOGN, 0>; break;
        case 1: kern = toeplitz_ws_kernel<LOGN, 1>; break;
        case 2: kern = toeplitz_ws_kernel<LOGN, 2>; break;
        case 3: kern = A.x4 != nullptr ? toeplitz_ws_kernel<LOGN, 3> : toeplitz_ws_kernel<LOGN, WS_IQU>; break;
        default: throw Error{MM_ERR_ARG, "unsupported Toeplitz load mode"};
    }
    const size_t smem = TB::DATA + TB::BYTES;
    // the rest of the SM's 256 KB is the L1 that the gathers of the map live on
    const int per_sm = (int)((smem + 1024) << (14 - LOGN));
    ensure_smem_attr((const void*)kern, (int)smem, "cudaFuncSetAttribute(toeplitz ws)", (per_sm * 100 + 228 * 1024 - 1) / (228 * 1024));
    // units of consecutive tiles: one right-hand side spreads its tiles evenly over the CTAs;
    // of many, at most eight tiles at a time, so that the CTAs at work read the same pointing
    const int ctas = ws_ctas(LOGN, num_sms);
    const int64_t items = (int64_t)tz.ntiles * A.R;
    int span = (int)((items + ctas - 1) / ctas);
    if (A.R > 1) span = std::min(8, std::max(1, span / 4));
    const int units = (int)(((int64_t)tz.ntiles + span - 1) / span * A.R);
    launch_pdl(kern, (unsigned)std::min(units, ctas), ws_threads<LOGN>(), smem, s, A, tz.ntiles, span, units,
               static_cast<const float4*>(tz.ws_tab), static_cast<const float*>(tz.ws_H), tz.ws_scratch);
    note_launch();
}

void launch_toeplitz_ws(const TzArgs<float>& A, const ToeplitzDev& tz, int num_sms, int mode, cudaStream_t s) {
    if (tz.logn == 14) ws_launch<14>(A, tz, num_sms, mode, s);
    else if (tz.logn == 13) ws_launch<13>(A, tz, num_sms, mode, s);
    else throw Error{MM_ERR_ARG, "unsupported FFT length"};
}

}  // namespace mm
