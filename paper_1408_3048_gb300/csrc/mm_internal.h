// Internal declarations shared by the translation units of libmm.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <array>
#include <string>
#include <utility>
#include <vector>

#include "../../include/mm.h"

namespace mm {

// entries of -1 behind the pixel indices: a gather that asks for its next indices ahead of
// time reads up to this many past the last sample
constexpr int PIXC_PAD = 8192;
// entries behind the sliced scatter's last step that its last batches read and leave out
constexpr int SL_PAD = 1024;
constexpr int SL_BLOCKS = 32;   // blocks of a scatter per SM, at most

// ---------------------------------------------------------------------------------
// Overlap-save tile of the single-right-hand-side Toeplitz kernels: a block of B real
// positions holding up to TILE_SEGS segments of samples.  Segment g covers block positions
// [pb[g], pe[g]) and position p in it holds the sample of time p + d[g]; every other
// position is 0.  The segments of one tile come from consecutive stationary intervals of
// one PSD, separated in the block by at least lambda zeros, so the band product of one
// interval never reaches another (Eq. 4: no coupling between intervals).  The valid
// outputs are block positions [lambda, lambda + nout); those inside a segment are stored
// at their time.  Unused segments have pb = pe = TILE_NONE.
constexpr int TILE_SEGS = 3;
constexpr int32_t TILE_NONE = 0x7fffffff;
struct Tile {
    int64_t d[TILE_SEGS];
    int32_t pb[TILE_SEGS];
    int32_t pe[TILE_SEGS];
    int32_t nout;
    int32_t psd;
    int32_t cont;   // positions from the window of the tile before, of the same run, to this one's, a
                    // multiple of 4 (0: none)
    int32_t unused;
};

// Tile of the batched kernels: block of B real samples [in0, in0 + B) of one interval
// producing the valid outputs [out0, out0 + nout) (out0 = in0 + lambda); samples outside
// [ibeg, iend) read as 0.
struct SpanTile {
    int64_t out0;
    int64_t ibeg;
    int64_t iend;
    int32_t nout;
    int32_t psd;
};

// Device tables of one arithmetic precision (T = double or float).
struct ToeplitzDev {
    int logn = 0;            // complex FFT length N = 2^logn, real block B = 2N
    int cluster = 1;         // CTAs per tile (2 or 4: split across a thread-block cluster)
    int ntiles = 0;
    Tile* tiles = nullptr;   // [ntiles]
    void* twiddle = nullptr; // T[B/4 + 1]: cos(2 pi k / B) (FP32: cluster blocks)
    void* ptw = nullptr;     // T2[...]: per-pass twiddles of the N-point FFT (not FP32)
    // FP32 blocks of 2^14 and 2^15 reals (toeplitz_ws.cu): twiddle tables, spectra in the kernel's
    // order, and the plan's input buffers
    void* ws_tab = nullptr;
    void* ws_H = nullptr;
    float* ws_scratch = nullptr;
    void* H = nullptr;       // T[npsd][split_size(N)]: kernel spectrum / N (fold_split_spectrum);
                             // FP32: T[npsd][N + 1], divided by another 4 (split_chain)
};

struct CoarseDev {
    int k = 0;                   // kept dimension
    double* Z64 = nullptr;       // [k][n]
    double* AZ64 = nullptr;      // [k][n]
    float* Z32 = nullptr;        // [k][n]
    float* AZ32 = nullptr;       // [k][n]
    double* Einv = nullptr;      // [k][k] E^-1 = L^-T L^-1 from the Cholesky factor (row-major)
    std::vector<double> ritz;    // k smallest Ritz values
};

// Scratch and state of the PCG driver.
struct PcgDev {
    int64_t n = 0;
    int nblocks = 0;             // cooperative grid size
    double* partial = nullptr;   // [nblocks][2 + KMAX] block partial sums
    double* scal = nullptr;      // [16] device scalars (see pcg.cu)
    int* flags = nullptr;        // [8] done / status / iteration / barrier words
    unsigned* barrier = nullptr; // grid barrier word
    void* x = nullptr;           // vectors, sized for double
    void* r = nullptr;
    void* p = nullptr;
    void* q = nullptr;
    void* z = nullptr;
    double* hist_alpha = nullptr;  // [maxhist]
    double* hist_beta = nullptr;   // [maxhist]
    double* hist_rz = nullptr;     // [maxhist]
    double* hist_rr = nullptr;     // [maxhist]
    int maxhist = 0;
    double* sc_part = nullptr;     // [scatter blocks] p^T q partials of the fused scatter
    unsigned* sc_count = nullptr;  // arrival counter of that scatter's last-block sum
};

// Per-stage CUDA-event timers (enabled by mm_profile).
enum { ST_TZ64 = 0, ST_TZ32 = 1, ST_SC64 = 2, ST_SC32 = 3, ST_PCG64 = 4, ST_PCG32 = 5, ST_TZDF = 6, ST_COUNT = 8 };
struct Prof {
    bool on = false;
    struct Pending {
        int stage;
        cudaEvent_t a, b;
    };
    std::vector<Pending> pending;
    std::vector<cudaEvent_t> pool;
    double ms[ST_COUNT] = {0, 0, 0, 0, 0, 0, 0, 0};
    int64_t launches[ST_COUNT] = {0, 0, 0, 0, 0, 0, 0, 0};
};

struct Plan {
    // problem
    int64_t nt = 0;
    int32_t npix_sky = 0;
    int32_t ncomp = 1;
    int32_t K = 0;
    int32_t npsd = 0;
    int32_t lambda = 0;
    int32_t window = MM_WINDOW_GAUSS;
    double fsamp = 100.0;
    double rcond_min = 1e-6;
    cudaStream_t stream = 0;
    int device = 0;                // device current when the plan was made
    int num_sms = 0;
    int scatter_lpp = 32;          // scatter lanes per pixel (32, 16 or 8; the pixel tile)
    int64_t L_grid = 0;

    // observed pixels
    int32_t npix_obs = 0;
    int64_t n = 0;
    int64_t nkept = 0;
    std::vector<int32_t> h_obs2sky, h_hits;
    std::vector<std::vector<double>> rows;   // [npsd][lambda+1]
    std::vector<int64_t> h_ioff;
    std::vector<int32_t> h_ipsd;

    // device pointing (time order) and pixel-sorted CSR
    int32_t* pixc = nullptr;       // [nt] observed index or -1
    double2* w64 = nullptr;        // [nt] (cos, sin), pol only
    float2* w32 = nullptr;         // [nt]
    int32_t* csr_off = nullptr;    // [npix_obs + 1]
    int32_t* tsort = nullptr;      // [nkept] sample index, pixel-major, ascending t
    double2* wsort64 = nullptr;    // [nkept] weights in sorted order (pol)
    float2* wsort32 = nullptr;     // [nkept]
    float* asort32 = nullptr;      // [nkept] angle / pi of the sorted weights when every weight
                                   // pair has unit norm (the FP32 scatter reads 4 bytes, not 8)
    // sliced layout of the sorted samples (scatter.cu), or null: slices of eight pixels, step j
    // of a slice = 32 entries (four samples of each of its pixels); the sorted weight arrays
    // above that no scatter reads any more are then freed once the plan is built.  Batches of
    // four or more use it, smaller ones as the FP32 scatter of one right-hand side.
    bool sl_f64 = false, sl_f32 = false;   // the scatters of one right-hand side use it
    int32_t sl_count = 0;          // slices
    int64_t sl_steps = 0;          // steps in all
    int32_t* sl_off = nullptr;     // [sl_count + 1] first step
    int32_t* sl_t = nullptr;       // [sl_steps][32] sample index, -1: none
    double2* sl_w64 = nullptr;     // [sl_steps][32] weights (pol)
    float2* sl_w32 = nullptr;
    float* sl_ang = nullptr;       // angles, where asort32 exists
    int64_t* ioff = nullptr;       // [K+1]
    int32_t* ipsd = nullptr;       // [K]
    double* t0 = nullptr;          // [npsd] diagonal of each row

    ToeplitzDev tz64, tz32;
    float* ws_scratch = nullptr;   // input buffers of the persistent kernel (toeplitz_ws.cu), or null
    ToeplitzDev tzdf;              // double-float tables (refinement residual)
    std::vector<std::vector<double>> spec;   // spectra of the rows while tables are built (N = spec_n), if few
    int64_t spec_n = 0;
    mutable std::array<std::array<int64_t, 20>, 2> tile_count;   // by layout and logn, -1: not counted yet
    Plan() {
        for (auto& c : tile_count) c.fill(-1);
    }

    // block-Jacobi: inverse blocks, symmetric packed (a00 a01 a02 a11 a12 a22) or 1
    double* bd64 = nullptr;        // [npix_obs][ncomp == 3 ? 6 : 1]
    float* bd32 = nullptr;

    // time-domain scratch
    double* tod64 = nullptr;       // [nt]
    float* tod32 = nullptr;        // [nt]
    float4* map4 = nullptr;        // [npix_obs] FP32 I/Q/U map packed per pixel (ncomp 3): the
                                   // layout the Toeplitz gather reads in one 16-byte load
    double* dbuf = nullptr;        // [nt] staging for host data
    double* b64 = nullptr;         // [n] last right-hand side
    bool have_b = false;

    CoarseDev coarse;
    PcgDev pcg;
    Prof prof;

    std::string err;
};

// profiling helpers (api.cu): begin returns a slot (or -1 when off), end closes it
int prof_begin(Plan& P, int stage);
void prof_end(Plan& P, int slot);
void prof_flush(Plan& P);   // after a stream synchronisation

// error helpers ----------------------------------------------------------------------
struct Error {
    mm_status st;
    std::string msg;
};

void check_cuda(cudaError_t e, const char* what);   // throws Error{MM_ERR_CUDA}
// cudaFuncSetAttribute(kern, MaxDynamicSharedMemorySize, bytes) once per kernel and
// device (thread-safe; the attribute is per device, so a second GPU gets its own call);
// carveout: also the preferred shared-memory share of the SM's 228 KB in percent (-1: default)
void ensure_smem_attr(const void* kern, int bytes, const char* what, int carveout = -1);
// Runs f and turns what it throws into a status: sets P->err (P may be null) and the
// calling thread's last-error message (mm_last_error(NULL)).  Nothing leaves it.
mm_status run_guarded(Plan* P, void (*f)(void*), void* ctx);
// No-allocation scratch of mm_apply_A_static (apply_static.cu): looks up the device
// address of the library's static array on the current device (called by mm_plan with
// the plan's device current) and returns it / its size.
void static_scratch_setup(int device);
void* static_scratch_ptr(int device);
size_t static_scratch_bytes();
void note_launch(int kernels = 1);                   // process-wide kernel launch counter

// Launch with programmatic dependent launch: the kernel may be scheduled before the
// previous kernel in the stream has finished, and must execute griddep_wait() before it
// reads anything that kernel wrote (the wait returns once that kernel has completed and
// its writes are visible).  Only kernels that wait first are launched this way.
template <typename... KA, typename... A>
void launch_pdl(void (*kern)(KA...), unsigned grid, unsigned block, size_t smem, cudaStream_t s, A&&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    check_cuda(cudaLaunchKernelEx(&cfg, kern, std::forward<A>(args)...), "kernel launch (dependent)");
}

#ifdef __CUDACC__
// Wait for the kernel before this one in the stream (programmatic dependent launch);
// returns at once for a kernel launched the ordinary way.
__device__ __forceinline__ void griddep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
#endif
void* dmalloc(size_t bytes);                         // throws Error{MM_ERR_OOM}
void dfree(void* p);

// host numerics (plan.cpp) -------------------------------------------------------------
void host_fft(std::vector<double>& re, std::vector<double>& im, bool inverse);
std::vector<double> toeplitz_row(double sigma, double fknee, double alpha, int64_t L,
                                 double fsamp, int lam, int window);
bool symbol_positive(const std::vector<double>& t);
std::vector<std::vector<double>> toeplitz_row_derivatives(double sigma, double fknee, double alpha, int64_t L,
                                                          double fsamp, int lam, int window);
std::vector<double> overlap_save_spectrum(const std::vector<double>& t, int64_t N);
// values of a folded spectrum: alpha [N], beta [N/2 + 1], the number of chained bins
__host__ __device__ constexpr int64_t split_size(int64_t N) { return N + N / 2 + 2; }
constexpr double SPLIT_RATIO = 0.25;   // of H_k and H_{N-k}: below it a pair of bins is chained
// cos(2 pi k / B), k = 0..B/4: the quarter wave (sin from the other end)
std::vector<double> quarter_wave(int64_t B);
void fold_split_spectrum(const std::vector<double>& h, int64_t N, const std::vector<double>& quarter, double* out);
// per-pass Stockham twiddles of an N = 2^logn point FFT as interleaved (cos, sin)
std::vector<double> pass_twiddle_table(int logn);
double rcond_sym3(const double B[6]);
bool scatter_sliced(int ncomp, int bytes, int64_t nt, int64_t nkept, int64_t npix, double padded);

// kernels (launchers) --------------------------------------------------------------------
// Toeplitz overlap-save (toeplitz_f64.cu / toeplitz_f32.cu)
template <typename T>
void launch_toeplitz(const Plan& P, const ToeplitzDev& tz, const T* y_tod, const T* x_map,
                     T* z, const int* done, cudaStream_t s);
// R right-hand sides in one launch: RHS r reads y_tod + r in_stride (or x_map + r in_stride)
// and writes z + r out_stride
template <typename T>
void launch_toeplitz_rhs(const Plan& P, const ToeplitzDev& tz, const T* y_tod, const T* x_map, int R,
                         int64_t in_stride, T* z, int64_t out_stride, const int* done, cudaStream_t s);
// General form: d_tod (FP64 time domain) alone is rounded to T (FP32 only); with x_map the
// input is d - P x (FP64 only: the residual data of b - A x; right-hand side r: x + r in_stride,
// d + r d_stride).
template <typename T>
void launch_toeplitz_any(const Plan& P, const ToeplitzDev& tz, const T* y_tod, const double* d_tod, const T* x_map,
                         int R, int64_t in_stride, T* z, int64_t out_stride, const int* done, cudaStream_t s,
                         int64_t d_stride = 0);
// Double-float N^-1 on FP64 data (toeplitz_df.cu): y (time domain) given, or else the
// residual data d - P x; output z FP64 [nt] (R right-hand sides as for launch_toeplitz_rhs)
void launch_toeplitz_df(const Plan& P, const double* y, const double* d, const double* x, int R, int64_t in_stride,
                        double* z, int64_t out_stride, cudaStream_t s, int64_t d_stride = 0);
// FP32 I/Q/U N^-1 P x with the gather reading x from P.map4; pack: first write x into
// P.map4 (one small kernel), else P.map4 already holds x (the FP32 PCG kernels keep it)
void launch_toeplitz_f32_packed(const Plan& P, const float* x, bool pack, float* z, const int* done,
                                cudaStream_t s);
bool ws_supported(int logn);
std::vector<float> ws_tables(int logn);
void ws_append_spectrum(const std::vector<double>& h, int logn, std::vector<float>& out);
size_t ws_scratch_floats(int num_sms);
template <typename T>
size_t toeplitz_smem_bytes(int logn);
template <typename T>
int toeplitz_max_logn();          // largest single-CTA FFT (the cluster kernels add one or two)

// pointing (pointing.cu)
template <typename T>
void launch_gather(const Plan& P, const T* x, T* y, cudaStream_t s);
template <typename T>
void launch_scatter(const Plan& P, const T* z, T* w, const int* done, cudaStream_t s);
// w = P^T z and, fused, *pq = p^T w (FP64, fixed summation order: warp partials over their
// pixels, block partials in part[], summed in block order by the last block to finish,
// which also resets *count to 0).  part holds SL_BLOCKS doubles per SM.
template <typename T>
void launch_scatter_dot(const Plan& P, const T* z, T* w, const T* p, double* part, unsigned* count, double* pq,
                        const int* done, cudaStream_t s);
int scatter_blocks(const Plan& P);
// whether launch_scatter<T> sums from the sliced layout
template <typename T>
bool use_sliced(const Plan& P) { return P.sl_off != nullptr && (sizeof(T) == 8 ? P.sl_f64 : P.sl_f32); }
// the same from the sliced layout (P.sl_off != nullptr); p null: no dot product
void launch_slice_fill(const Plan& P, int32_t* st, double2* sw64, float2* sw32, float* sang, cudaStream_t s);
template <typename T>
void launch_scatter_sliced(const Plan& P, const T* z, T* w, const T* p, double* part, unsigned* count, double* pq,
                           const int* done, cudaStream_t s);
template <typename T>
void launch_batch_scatter_sliced(const Plan& P, const T* Z, T* W, int R, const int* done, cudaStream_t s);
int sliced_parts(const Plan& P, int groups = 0);   // warps per slice; groups of a batch, 0: one column
void launch_bd_build(const Plan& P, double* bd64, float* bd32, cudaStream_t s);
// merged a priori coarse space Z_S (Sec. 3.3.1), r groups of consecutive intervals, into
// Z [r][n] FP64 (zeroed here)
void launch_apriori(const Plan& P, int r, double* Z, cudaStream_t s);
template <typename T>
void launch_bd_apply(const Plan& P, const T* r, T* z, cudaStream_t s);
void launch_angles(const double2* w, float* ang, int64_t n, unsigned* bad, cudaStream_t s);
void launch_convert_f64_to_f32(const double* a, float* b, int64_t n, cudaStream_t s);
void launch_convert_f32_to_f64(const float* a, double* b, int64_t n, cudaStream_t s);
// gradient helpers (grad.cu)
void launch_sub_time(const double* a, const double* b, double* out, int64_t n, cudaStream_t s);
void launch_interval_dot(const double* u, const double* w, const int64_t* ioff, int K, double* part,
                         cudaStream_t s);

}  // namespace mm
