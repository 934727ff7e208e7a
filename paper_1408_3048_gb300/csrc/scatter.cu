// P^T z from the sliced layout of the pixel-sorted samples (the CSR forms, with a fixed
// number of lanes per pixel, are in pointing.cu).
//
// Eight consecutive observed pixels form a slice, four lanes to a pixel: step j of a slice
// holds, lane by lane, samples 4 j .. 4 j + 3 of each of its pixels in time order (index -1
// past a pixel's last sample).  A warp walks over a slice's steps, so its index and weight
// reads are contiguous, its lanes' sums need no tree but the last one over four lanes, and
// the time-domain values that it reads in one step lie close together in time: a raster
// passes neighbouring pixels one after the other.  The CSR forms spread a pixel's samples
// over a warp: every load of theirs went to as many places as the pixel has visits (a
// different 2 MB page each in a long run), and each pixel paid a 32-lane tree.
// Measured against the 32-lane form (time inside A x): T, 2^26 samples on 512 x 512 pixels
// 264 -> 98 us (537 MB, 0.81 of the copy bandwidth); I/Q/U circles, 1.6e7 samples on 303079
// pixels 99 -> 63 us; I/Q/U in FP64, 2^22 samples 106 -> 39 us; 64 right-hand sides on 2^22
// samples 481 -> 318 us.  I/Q/U in FP32 on 65536 pixels of 256 samples: 47.6 -> 52.8 us, so
// there the 32-lane form stays (scatter_sliced in plan_host.cpp has the rule and its figures).
//
// Few pixels with many samples: the S warps of a slice take consecutive parts of its steps and
// add them in order through shared memory.  Every sum has a fixed order: bit-reproducible.
#include <algorithm>

#include "mm_internal.h"
#include "pcg.cuh"

namespace mm {

constexpr int SL_PIX = 8;     // pixels per slice
constexpr int SL_U = 8;       // steps in flight

template <typename T> struct W2;
template <> struct W2<double> { using type = double2; };
template <> struct W2<float> { using type = float2; };

// ------------------------------------------------------------------------------- build
// entry (step, lane) of slice s: its sample, weight pair (FP64) and angle
__global__ void slice_fill_kernel(const int32_t* __restrict__ off, const int32_t* __restrict__ tsort,
                                  const double2* __restrict__ w64, const float* __restrict__ ang,
                                  const int32_t* __restrict__ sl_off, int nslices, int npix,
                                  int32_t* __restrict__ st, double2* __restrict__ sw64, float2* __restrict__ sw32,
                                  float* __restrict__ sang) {
    const int lane = threadIdx.x & 31, warps = blockDim.x >> 5;
    for (int s = blockIdx.x * warps + (threadIdx.x >> 5); s < nslices; s += gridDim.x * warps) {
        const int q = s * SL_PIX + (lane >> 2), sub = lane & 3;
        const int b = q < npix ? off[q] : 0, hits = q < npix ? off[q + 1] - b : 0;
        const int o0 = sl_off[s], o1 = sl_off[s + 1];
        for (int o = o0; o < o1; ++o) {
            const int k = 4 * (o - o0) + sub;
            const bool in = k < hits;
            const int64_t e = (int64_t)o * 32 + lane;
            st[e] = in ? tsort[b + k] : -1;
            if (sw64 != nullptr) {
                const double2 w = in ? w64[b + k] : make_double2(0.0, 0.0);
                sw64[e] = w;
                if (sw32 != nullptr) sw32[e] = make_float2((float)w.x, (float)w.y);
                if (sang != nullptr) sang[e] = in ? ang[b + k] : 0.f;
            }
        }
    }
}

void launch_slice_fill(const Plan& P, int32_t* st, double2* sw64, float2* sw32, float* sang, cudaStream_t s) {
    const int g = std::max(1, std::min((P.sl_count + 7) / 8, P.num_sms * 8));
    slice_fill_kernel<<<g, 256, 0, s>>>(P.csr_off, P.tsort, P.wsort64, P.asort32, P.sl_off, P.sl_count, P.npix_obs, st,
                                        sw64, sw32, sang);
    check_cuda(cudaGetLastError(), "slice fill launch");
    note_launch();
}

// ----------------------------------------------------------------------------- scatter
// Sum of a lane's values: FP32 in exact pairs (batches of SL_U added plainly first), FP64 in
// batches too, so that the number of roundings in a row stays small.
template <typename T> struct Acc {
    T hi = 0, lo = 0;
    __device__ __forceinline__ void add(T v) {
        if constexpr (sizeof(T) == 4) pair_add(hi, lo, v, 0.f);
        else hi += v;
    }
    __device__ __forceinline__ void merge(T h, T l) {
        if constexpr (sizeof(T) == 4) pair_add(hi, lo, h, l);
        else hi += h;
    }
    __device__ __forceinline__ void lanes(int o) {
        const T h = __shfl_xor_sync(0xffffffffu, hi, o);
        T l = 0;
        if constexpr (sizeof(T) == 4) l = __shfl_xor_sync(0xffffffffu, lo, o);
        merge(h, l);
    }
    __device__ __forceinline__ T total() const { return hi + lo; }
};

struct SlicedDot {
    const void* p;      // T[n]
    double* part;       // [gridDim.x]
    unsigned* count;
    double* pq;
};

// Resident 256-thread blocks asked for: eight for FP32 temperature (32 registers a thread; 116
// us at its own 40, 98 at 32, for 2^26 samples), else five (48 registers keep a batch's loads
// together: at 36 the I/Q/U form with its dot product took 68 us where it took 57).
template <typename T, int NC, int WPB>
__host__ __device__ constexpr int sl_min_blocks() { return WPB != 8 ? 1 : sizeof(T) == 4 && NC == 1 ? 8 : 5; }

template <typename T, int NC, bool DOT, bool ANG, int WPB>
__global__ void __launch_bounds__(WPB * 32, (sl_min_blocks<T, NC, WPB>())) sliced_scatter_kernel(const int32_t* __restrict__ sl_off,
                                                                  const int32_t* __restrict__ st,
                                                                  const typename W2<T>::type* __restrict__ sw,
                                                                  const float* __restrict__ sang, const T* __restrict__ z,
                                                                  T* __restrict__ w, int nslices, int npix, int S,
                                                                  const int* done, SlicedDot sd) {
    using V2 = typename W2<T>::type;
    griddep_wait();   // launched as a dependent launch: the previous kernel's outputs
    if (done != nullptr && *(volatile const int*)done) return;
    __shared__ T comb[WPB > 1 ? WPB : 1][SL_PIX][2 * NC];   // parts 1 .. S - 1 of their slices
    const int lane = threadIdx.x & 31, wi = threadIdx.x >> 5;
    const int part = wi % S, grp = wi / S, G = WPB / S;
    DotAcc<T> dacc;   // DOT: lanes 0, 4, ... of the first parts, slices ascending
    for (int sb = blockIdx.x * G; sb < nslices; sb += gridDim.x * G) {
        const int s = sb + grp;
        int j0 = 0, j1 = 0;
        if (s < nslices) {
            const int o0 = sl_off[s], o1 = sl_off[s + 1];
            const int per = (o1 - o0 + S - 1) / S;
            j0 = o0 + part * per;
            j1 = min(o1, j0 + per);
        }
        // DOT: this lane's pixel of p, requested ahead of the walk
        const int q = s * SL_PIX + (lane >> 2);
        const bool mine = (lane & 3) == 0 && part == 0 && s < nslices && q < npix;
        T pv[NC];
        if constexpr (DOT) {
#pragma unroll
            for (int c = 0; c < NC; ++c) pv[c] = mine ? static_cast<const T*>(sd.p)[(int64_t)q * NC + c] : (T)0;
        }
        Acc<T> a[NC];
        const int64_t e0 = (int64_t)j0 * 32 + lane;
        const int32_t* pt = st + e0;
        const float* pa = sang + e0;
        const V2* pw = sw + e0;
        // batches of SL_U steps; a last one reads on into the entries behind (SL_PAD) and
        // leaves them out
        for (int left = j1 - j0; left > 0; left -= SL_U) {
            T v[SL_U];
            V2 ww[SL_U];
            int t[SL_U];
#pragma unroll
            for (int u = 0; u < SL_U; ++u) t[u] = __ldg(pt + u * 32);
            if constexpr (NC == 3) {
#pragma unroll
                for (int u = 0; u < SL_U; ++u) {
                    if constexpr (ANG) ww[u].x = __ldg(pa + u * 32);
                    else ww[u] = __ldg(pw + u * 32);
                }
            }
#pragma unroll
            for (int u = 0; u < SL_U; ++u) v[u] = z[u < left ? max(t[u], 0) : 0];
            T b0 = 0, b1 = 0, b2 = 0;
#pragma unroll
            for (int u = 0; u < SL_U; ++u) {
                const T x = t[u] >= 0 && u < left ? v[u] : (T)0;
                b0 += x;
                if constexpr (NC == 3) {
                    if constexpr (ANG) {
                        // (the angle's rounding is then all: 1e-7.  The fast sine and cosine save
                        // 4 of 63 us on the circle scan.)
                        float sv, cv;
                        sincospif(ww[u].x, &sv, &cv);
                        b1 += cv * x;
                        b2 += sv * x;
                    } else {
                        b1 += ww[u].x * x;
                        b2 += ww[u].y * x;
                    }
                }
            }
            a[0].add(b0);
            if constexpr (NC == 3) {
                a[1].add(b1);
                a[2].add(b2);
            }
            pt += SL_U * 32;
            pa += SL_U * 32;
            pw += SL_U * 32;
        }
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            a[c].lanes(1);
            a[c].lanes(2);
        }
        if (S > 1) {   // uniform over the block
            const int px = lane >> 2;
            if ((lane & 3) == 0 && part > 0) {
#pragma unroll
                for (int c = 0; c < NC; ++c) {
                    comb[wi][px][2 * c] = a[c].hi;
                    comb[wi][px][2 * c + 1] = a[c].lo;
                }
            }
            __syncthreads();
            if ((lane & 3) == 0 && part == 0)
                for (int p = 1; p < S; ++p)
#pragma unroll
                    for (int c = 0; c < NC; ++c) a[c].merge(comb[wi + p][px][2 * c], comb[wi + p][px][2 * c + 1]);
            __syncthreads();
        }
        if (mine) {
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                const T r = a[c].total();
                w[(int64_t)q * NC + c] = r;
                if constexpr (DOT) dacc.add(pv[c], r);
            }
        }
    }
    if constexpr (DOT) {
        // a warp's pixels by a tree over its lanes, warps in order, then the last block to finish
        // adds the blocks in order
        __shared__ double wacc[WPB];
        __shared__ double wsum[WPB];
        __shared__ bool last;
        Acc<T> d;
        if constexpr (sizeof(T) == 4) {
            d.hi = dacc.hi;
            d.lo = dacc.lo;
        } else {
            d.hi = dacc.s;
        }
#pragma unroll
        for (int o = 4; o < 32; o <<= 1) d.lanes(o);
        if (lane == 0) wacc[wi] = (double)d.hi + (double)d.lo;
        __syncthreads();
        if (threadIdx.x == 0) {
            double b = 0.0;
            for (int i = 0; i < WPB; ++i) b += wacc[i];
            sd.part[blockIdx.x] = b;
            __threadfence();
            last = atomicAdd(sd.count, 1u) == gridDim.x - 1;
        }
        __syncthreads();
        if (last) {
            __threadfence();
            const int per = (gridDim.x + WPB - 1) / WPB;
            const int i1 = min((int)gridDim.x, (wi + 1) * per);
            double x = 0.0;
            for (int i = wi * per + lane; i < i1; i += 32) x += __ldcg(sd.part + i);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
            if (lane == 0) wsum[wi] = x;
            __syncthreads();
            if (threadIdx.x == 0) {
                double tot = 0.0;
                for (int i = 0; i < WPB; ++i) tot += wsum[i];
                *sd.pq = tot;
                *sd.count = 0;
            }
        }
    }
}

// Warps per slice.  One column: enough of them for half the chip's warps, each with at least a
// batch of steps.  (More parts shorten the last, partly filled wave of blocks but also the slices'
// runs: four warps per slice on 8192 slices of 64 steps took 51 us, one 47.)
// groups: of a batch's right-hand sides, each a walk over every slice by warps with several loads
// in flight for a step.  Half as many of them are enough, and from a quarter on only long walks
// gain, most of all by the first split, which changes the kernel (A x in us by parts, I/Q/U; 512
// walks of 64 steps 1: 83, 4: 72, 8: 70; of 256 287, 203, 170; 1024 of 128 1: 259, 2: 227, 4: 187;
// 2048 of 64 1: 158, 2: 160, of 128 323, 317, of 256 504, 498; T, of 64 128, 120, of 256 446, 369;
// 4096 of 64 1: 253, 2: 282).
int sliced_parts(const Plan& P, int groups) {
    const int64_t steps = P.sl_count > 0 ? P.sl_steps / P.sl_count : 0;
    int S = 1;
    if (groups == 0) {
        while (S < 32 && (int64_t)P.sl_count * S < (int64_t)P.num_sms * 32 && steps / (2 * S) >= SL_U) S *= 2;
        return S;
    }
    const int64_t walks = (int64_t)P.sl_count * groups;
    while (S < 32 && walks * S < (int64_t)P.num_sms * 16) {
        const int least = walks * S < (int64_t)P.num_sms * 8 ? SL_U : S == 1 && P.ncomp == 3 ? 64 : 32;
        if (steps / (2 * S) < least) break;
        S *= 2;
    }
    return S;
}

// Blocks: up to SL_BLOCKS per SM, several times what is resident, so that an SM that is done
// takes the next one (a grid of just the resident blocks, each walking over its share, left
// whole rounds of some of them to the end: 99 to 127 us for the same work).
static int sliced_blocks(const Plan& P, int wpb, int S) {
    const int G = wpb / S;
    return std::max(1, std::min((P.sl_count + G - 1) / G, P.num_sms * SL_BLOCKS));
}

template <typename T, int NC, bool DOT, bool ANG>
static void sliced_launch(const Plan& P, const typename W2<T>::type* sw, const float* sang, const T* z, T* w,
                          const int* done, SlicedDot sd, cudaStream_t s) {
    const int S = sliced_parts(P);
    const int32_t* so = P.sl_off;
    const int32_t* st = P.sl_t;
    if (S <= 8)
        launch_pdl(sliced_scatter_kernel<T, NC, DOT, ANG, 8>, (unsigned)sliced_blocks(P, 8, S), 256, 0, s, so, st, sw, sang,
                   z, w, P.sl_count, P.npix_obs, S, done, sd);
    else
        launch_pdl(sliced_scatter_kernel<T, NC, DOT, ANG, 32>, (unsigned)sliced_blocks(P, 32, S), 1024, 0, s, so, st, sw,
                   sang, z, w, P.sl_count, P.npix_obs, S, done, sd);
    check_cuda(cudaGetLastError(), "scatter launch");
    note_launch();
}

template <typename T>
void launch_scatter_sliced(const Plan& P, const T* z, T* w, const T* p, double* part, unsigned* count, double* pq,
                           const int* done, cudaStream_t s) {
    const SlicedDot sd{p, part, count, pq};
    const typename W2<T>::type* none = nullptr;
    if (P.ncomp == 1) {
        if (p != nullptr) sliced_launch<T, 1, true, false>(P, none, nullptr, z, w, done, sd, s);
        else sliced_launch<T, 1, false, false>(P, none, nullptr, z, w, done, sd, s);
        return;
    }
    if constexpr (sizeof(T) == 4) {
        if (P.sl_ang != nullptr) {
            if (p != nullptr) sliced_launch<T, 3, true, true>(P, none, P.sl_ang, z, w, done, sd, s);
            else sliced_launch<T, 3, false, true>(P, none, P.sl_ang, z, w, done, sd, s);
            return;
        }
        if (p != nullptr) sliced_launch<T, 3, true, false>(P, P.sl_w32, nullptr, z, w, done, sd, s);
        else sliced_launch<T, 3, false, false>(P, P.sl_w32, nullptr, z, w, done, sd, s);
    } else {
        if (p != nullptr) sliced_launch<T, 3, true, false>(P, P.sl_w64, nullptr, z, w, done, sd, s);
        else sliced_launch<T, 3, false, false>(P, P.sl_w64, nullptr, z, w, done, sd, s);
    }
}
template void launch_scatter_sliced<double>(const Plan&, const double*, double*, const double*, double*, unsigned*,
                                            double*, const int*, cudaStream_t);
template void launch_scatter_sliced<float>(const Plan&, const float*, float*, const float*, double*, unsigned*,
                                           double*, const int*, cudaStream_t);

// ------------------------------------------------------------- many right-hand sides
// The same walk for RC right-hand sides at a time (grid.y; four in FP32, two in FP64): a step's
// indices and weights are read once for them.
constexpr int SL_BU = 4;

// a += steps [j, j1) of a slice; z0: the first right-hand side of the group
template <typename T, int NC, int RC>
__device__ __forceinline__ void batch_walk(Acc<T> (&a)[RC][NC], int j, int j1, const int32_t* __restrict__ st,
                                           const typename W2<T>::type* __restrict__ sw, const T* __restrict__ z0, int r0,
                                           int64_t nt, int R, int lane) {
    using V2 = typename W2<T>::type;
    for (; j < j1; j += SL_BU) {
        int t[SL_BU];
        V2 ww[SL_BU];
#pragma unroll
        for (int u = 0; u < SL_BU; ++u) {
            const int64_t e = (int64_t)min(j + u, j1 - 1) * 32 + lane;
            t[u] = j + u < j1 ? __ldg(st + e) : -1;
            if constexpr (NC == 3) ww[u] = __ldg(sw + e);
        }
        T v[RC][SL_BU];
#pragma unroll
        for (int r = 0; r < RC; ++r) {
            const T* z = z0 + (r0 + r < R ? (size_t)r * nt : 0);
#pragma unroll
            for (int u = 0; u < SL_BU; ++u) v[r][u] = z[max(t[u], 0)];
        }
#pragma unroll
        for (int r = 0; r < RC; ++r) {
            T b[NC] = {};
#pragma unroll
            for (int u = 0; u < SL_BU; ++u) {
                const T x = t[u] >= 0 ? v[r][u] : (T)0;
                b[0] += x;
                if constexpr (NC == 3) {
                    b[1] += ww[u].x * x;
                    b[2] += ww[u].y * x;
                }
            }
#pragma unroll
            for (int c = 0; c < NC; ++c) a[r][c].add(b[c]);
        }
    }
}

template <typename T, int NC, int RC>
__global__ void __launch_bounds__(256) sliced_batch_kernel(const int32_t* __restrict__ sl_off,
                                                           const int32_t* __restrict__ st,
                                                           const typename W2<T>::type* __restrict__ sw,
                                                           const T* __restrict__ Z, T* __restrict__ W, int nslices,
                                                           int npix, int64_t nt, int64_t n, int R, const int* done) {
    if (done != nullptr && *(volatile const int*)done) return;
    const int lane = threadIdx.x & 31, warps = blockDim.x >> 5;
    const int r0 = blockIdx.y * RC;
    const T* z0 = Z + (size_t)r0 * nt;
    for (int s = blockIdx.x * warps + (threadIdx.x >> 5); s < nslices; s += gridDim.x * warps) {
        Acc<T> a[RC][NC];
        const int j1 = sl_off[s + 1];
        batch_walk<T, NC, RC>(a, sl_off[s], j1, st, sw, z0, r0, nt, R, lane);
        const int q = s * SL_PIX + (lane >> 2);
#pragma unroll
        for (int r = 0; r < RC; ++r)
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                a[r][c].lanes(1);
                a[r][c].lanes(2);
                if ((lane & 3) == 0 && q < npix && r0 + r < R) W[(size_t)(r0 + r) * n + (int64_t)q * NC + c] = a[r][c].total();
            }
    }
}

// S warps per slice as above, where few pixels and few columns have too few slices for the chip
// (T, 64 pixels of 8192 samples, two columns: A x 505 -> 67 us, with the 32-lane form 103).  With
// S = 1 it took 346 us where the kernel above takes 319 (64 columns, 2^22 I/Q/U samples).
template <typename T, int NC, int RC, int WPB>
__global__ void __launch_bounds__(WPB * 32) sliced_batch_parts_kernel(const int32_t* __restrict__ sl_off,
                                                                      const int32_t* __restrict__ st,
                                                                      const typename W2<T>::type* __restrict__ sw,
                                                                      const T* __restrict__ Z, T* __restrict__ W,
                                                                      int nslices, int npix, int64_t nt, int64_t n, int R,
                                                                      int S, const int* done) {
    if (done != nullptr && *(volatile const int*)done) return;
    __shared__ T comb[WPB][SL_PIX][RC][2 * NC];   // parts 1 .. S - 1 of their slices
    const int lane = threadIdx.x & 31, wi = threadIdx.x >> 5;
    const int part = wi % S, G = WPB / S;
    const int r0 = blockIdx.y * RC;
    const T* z0 = Z + (size_t)r0 * nt;
    for (int sb = blockIdx.x * G; sb < nslices; sb += gridDim.x * G) {   // uniform over the block
        const int s = sb + wi / S;
        Acc<T> a[RC][NC];
        if (s < nslices) {
            const int o0 = sl_off[s], o1 = sl_off[s + 1], per = (o1 - o0 + S - 1) / S;
            const int j0 = min(o1, o0 + part * per);
            batch_walk<T, NC, RC>(a, j0, min(o1, j0 + per), st, sw, z0, r0, nt, R, lane);
        }
        const int px = lane >> 2, q = s * SL_PIX + px;
#pragma unroll
        for (int r = 0; r < RC; ++r)
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                a[r][c].lanes(1);
                a[r][c].lanes(2);
                if ((lane & 3) == 0 && part > 0) {
                    comb[wi][px][r][2 * c] = a[r][c].hi;
                    comb[wi][px][r][2 * c + 1] = a[r][c].lo;
                }
            }
        __syncthreads();
        if ((lane & 3) == 0 && part == 0 && s < nslices && q < npix)
#pragma unroll
            for (int r = 0; r < RC; ++r)
#pragma unroll
                for (int c = 0; c < NC; ++c) {
                    for (int p = 1; p < S; ++p) a[r][c].merge(comb[wi + p][px][r][2 * c], comb[wi + p][px][r][2 * c + 1]);
                    if (r0 + r < R) W[(size_t)(r0 + r) * n + (int64_t)q * NC + c] = a[r][c].total();
                }
        __syncthreads();
    }
}

template <typename T, int WPB>
static void sliced_batch_parts(const Plan& P, const typename W2<T>::type* sw, const T* Z, T* W, int R, int S,
                               const int* done, cudaStream_t s) {
    constexpr int RC = sizeof(T) == 4 ? 4 : 2;
    const int G = WPB / S;
    const int gx = std::max(1, std::min((P.sl_count + G - 1) / G, P.num_sms * 8));
    const dim3 grid((unsigned)gx, (unsigned)((R + RC - 1) / RC));
    auto kern = P.ncomp == 1 ? sliced_batch_parts_kernel<T, 1, RC, WPB> : sliced_batch_parts_kernel<T, 3, RC, WPB>;
    kern<<<grid, WPB * 32, 0, s>>>(P.sl_off, P.sl_t, sw, Z, W, P.sl_count, P.npix_obs, P.nt, P.n, R, S, done);
}

template <typename T>
void launch_batch_scatter_sliced(const Plan& P, const T* Z, T* W, int R, const int* done, cudaStream_t s) {
    constexpr int RC = sizeof(T) == 4 ? 4 : 2;
    const typename W2<T>::type* sw = nullptr;
    if constexpr (sizeof(T) == 4) sw = P.sl_w32;
    else sw = P.sl_w64;
    const int S = sliced_parts(P, (R + RC - 1) / RC);
    if (S == 1) {
        const int gx = std::max(1, std::min((P.sl_count + 7) / 8, P.num_sms * 8));
        const dim3 grid((unsigned)gx, (unsigned)((R + RC - 1) / RC));
        auto kern = P.ncomp == 1 ? sliced_batch_kernel<T, 1, RC> : sliced_batch_kernel<T, 3, RC>;
        kern<<<grid, 256, 0, s>>>(P.sl_off, P.sl_t, sw, Z, W, P.sl_count, P.npix_obs, P.nt, P.n, R, done);
    } else if (S <= 8) {
        sliced_batch_parts<T, 8>(P, sw, Z, W, R, S, done, s);
    } else {
        sliced_batch_parts<T, 32>(P, sw, Z, W, R, S, done, s);
    }
    check_cuda(cudaGetLastError(), "batch scatter launch");
    note_launch();
}
template void launch_batch_scatter_sliced<float>(const Plan&, const float*, float*, int, const int*, cudaStream_t);
template void launch_batch_scatter_sliced<double>(const Plan&, const double*, double*, int, const int*, cudaStream_t);

}  // namespace mm
