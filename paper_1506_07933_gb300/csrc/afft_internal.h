// afft_internal.h -- shared host/device declarations of the CUDA library.
//
// One 3-D transform is three "stages" (Algorithm 1 of AccFFT, with the
// process grid P0 = P1 = 1): batched 1-D FFTs along the contiguous axis N2,
// then along N1, then along N0 (reverse order for the backward transform).
// Each stage is one kernel launch.  A stage transforms every line of length n
// with a Stockham autosort FFT made of radix-R passes (R in 16, 15, 12, 10, 9, 8, 6, 5, 4, 3, 2);
// StageDesc carries that factorisation and the offsets of each pass's twiddle
// table in the plan's device buffer.
#pragma once

#include <cstddef>
#include <cstdint>

#include <cuda_runtime.h>

struct afft_plan;

namespace afft {

constexpr int kMaxPasses = 16;
constexpr int kMaxLine = 4096;     // longest line a single CTA transforms

struct StageDesc {
    int n;                         // line length in complex points
    int npass;                     // number of radix passes (0 when n == 1)
    int radix[kMaxPasses];         // radix of each pass
    int ns[kMaxPasses];            // product of the radices of the earlier passes
    // first twiddle of each pass (complex entries); entry (k, r), k < ns and 1 <= r < radix, of the
    // pass is at (r - 1) ns + k, or in the k-major tables of the generic families at k (radix - 1) + r - 1
    int tw_off[kMaxPasses];
    int ld;                        // r2c/c2r stage: stride between half-spectrum lines, in complex
                                   // elements; 0 means compact (M + 1 for a line of M points)
    // FP64 plans: the same twiddle tables as float-float values (hi, lo floats),
    // or null to compute in FP64 (specialised kernels then use float-float)
    const void *twdf;              // this axis' tables, same offsets as `tw`
    const void *post_df;           // the r2c/c2r table w_{2M}^k
    // split-precision plans: the tensor-core fragments of the 16-point DFT matrix
    // (both directions, see fft_split.cuh), else null
    const unsigned *mma;
    // contiguous c2c stage of a blocked plan: the lines of `in` (blk_in) or of `out` (blk_out)
    // lie in the layout [n1 / blk][planes][blk][n], line q = plane * n1 + j at line
    // ((j / blk) * planes + plane) * blk + j % blk; blk = 0: row-major on both sides
    int blk, blk_in, blk_out;
    long long blk_n1, blk_planes;
    unsigned *err;                 // set by a kernel whose bounded wait ran out (null: not reported)
    // 1: the CTAs take their line blocks (or tiles) in reverse order, last first, so that a stage
    // following one that wrote the same array front to back starts on the part still in L2
    int rev;
};

// Block (or tile) i of n in the order a stage walks them.
__host__ __device__ inline long long stage_order(long long i, long long n, int rev) { return rev ? n - 1 - i : i; }

// Line of the blocked layout holding row-major line q (see StageDesc::blk).
__host__ __device__ inline long long blocked_line(const StageDesc &d, long long q)
{
    const long long pl = q / d.blk_n1, j = q - pl * d.blk_n1;
    return ((j / d.blk) * d.blk_planes + pl) * d.blk + j % d.blk;
}

// Butterflies a thread carries per pass for radix R: at most 16 complex
// values in registers (15 for radix 3 and 5; the pipelined tiles have counts of their own, up to 20
// values, see PipeShape).  The host picks the thread
// count so that threads * bmax(R) covers every butterfly of every pass.
__host__ __device__ constexpr int bmax_for_radix(int r)
{
    return r >= 16 ? 1 : (r == 3 ? 5 : (r == 5 ? 3 : 16 / r));
}

// Radix passes of a generic line of n points: the power-of-two part as evenly sized radix-16/8/4/2
// passes (radix 16 runs on the tensor cores in split precision), then one pass per factor 3 and 5.
// Writes at most kMaxPasses radices to r and returns their number (0 for n == 1).
inline int basic_sequence(long long n, int *r)
{
    int k = 0, a = 0;
    while (n % 2 == 0) { n /= 2; ++a; }
    const int passes = (a + 3) / 4;
    for (int i = 0; i < passes; ++i) r[k++] = 1 << (a / passes + (i < a % passes ? 1 : 0));
    while (n % 3 == 0) { n /= 3; r[k++] = 3; }
    while (n % 5 == 0) { n /= 5; r[k++] = 5; }
    return k;
}

// Radix passes for a line of n points of the mixed generic family: the fewest passes of radices up to
// 16 (every pass is a round trip through shared memory), and among those the smallest largest
// radix, then the smallest sum, in descending order.  A generic CTA has kGenericThreads threads and
// holds at least one line, so radices whose butterflies of one line do not fit it are left out (9
// carries one butterfly per thread where 3 carries five: 2430 points take 15 6 3 3 3, not 9 9 6 5);
// the three lengths that no sequence fits (3888, 4000, 4050) get one that the launch shapes refuse.
// Writes at most kMaxPasses radices to r and returns their number (0 for n == 1, -1 when n is not
// 2/3/5-smooth).
constexpr int kGenericThreads = 256;

inline int radix_sequence(long long n, int *r)
{
    static constexpr int kRadices[] = {16, 15, 12, 10, 9, 8, 6, 5, 4, 3, 2};
    if (n == 1) return 0;
    struct Search {
        long long n;
        bool fit;                  // only radices that fit the CTA
        int best[kMaxPasses], cur[kMaxPasses], best_max = 1 << 30, best_sum = 1 << 30;
        void go(long long m, int left, int at, int hi, int sum)
        {
            if (left == 0) {
                if (m != 1 || cur[0] > best_max || (cur[0] == best_max && sum >= best_sum)) return;
                best_max = cur[0];
                best_sum = sum;
                for (int i = 0; i < at; ++i) best[i] = cur[i];
                return;
            }
            for (int R : kRadices) {
                if (R > hi || m % R != 0) continue;
                if (fit && n > (long long)kGenericThreads * R * bmax_for_radix(R)) continue;
                cur[at] = R;
                go(m / R, left - 1, at + 1, R, sum + R);
            }
        }
    };
    for (const bool fit : {true, false})
        for (int k = 1; k <= 8; ++k) {   // lines of at most 4096 points need at most seven
            Search s;
            s.n = n;
            s.fit = fit;
            s.go(n, k, 0, 16, 0);
            if (s.best_sum < (1 << 30)) {
                for (int i = 0; i < k; ++i) r[i] = s.best[i];
                return k;
            }
        }
    return -1;
}

// Threads that hold every butterfly of each pass of `lines` lines.
inline int line_threads(const int *radix, int npass, long long n, int lines)
{
    long long req = lines;   // copy path (n == 1)
    for (int p = 0; p < npass; ++p) {
        const int per = bmax_for_radix(radix[p]);
        const long long t = ((long long)lines * (n / radix[p]) + per - 1) / per;
        req = t > req ? t : req;
    }
    return (int)(req < 32 ? 32 : (req + 31) / 32 * 32);
}

// Whether a generic line of n points runs the mixed family (radix_sequence) or the basic one
// (basic_sequence); elem: bytes per complex value.  Both were measured at every smooth length from
// 1080 to 4096 on 320 to 640 MB.
//  * The mixed sequence must have fewer passes (3125, 3200 and 3456 points, the same passes in both,
//    lose 2 to 9%; 2000 = 10 8 5 5 against 16 5 5 5 lost 4 to 20%).
//  * complex64 passes are bound by shared memory and barriers, so their time goes as passes over
//    points resident per SM, and wide radices give a line fewer threads.  With that quotient up to 1.2
//    times the basic one the mixed family measured 0.55 to 0.98 (2700 points N2 1074 -> 594 us, N0 1109
//    -> 784 us; 1440 points N0 1054 -> 800 us); above, lost or equal (1.88: 1920 points N0 701 ->
//    946 us; 1.5: 1800 points N0 846 -> 1000 us, 1280 points N2 557 -> 600 us).  A strided tile that
//    halves its columns reads half the bytes per row: its quotient counts 1.25 times (1600 points N0,
//    1.0 x 1.25, 852 -> 930 us).
//  * complex128 passes are bound by the FP64 pipe: two radix-9 butterflies with their inner twiddles and
//    idle lanes cost what four radix-3 passes do (1458 = 9 9 6 3: N2 3475 -> 3690 us, 1215 = 15 9 9: r2c
//    3884 -> 4150 us); the other lengths measured 0.78 to 1.04 (2592 points N0 3977 -> 3200 us, 1920
//    points N0 2780 -> 2880 us).
// regs: registers per thread of the kernel (255 in the four-step kernel, where the same quotient told
// complex64 halves of 72 and 75 points, 0.67 and measured 0.75 to 0.91 on the transform, from 50, 60
// and 100, 1.33 and measured 1.22 to 1.36; complex128 ones lose 2 to 7% and stay with the basic family).
inline bool mixed_pays(long long n, int elem, bool contiguous, int regs = 128)
{
    int basic[kMaxPasses], mixed[kMaxPasses];
    const int nb = basic_sequence(n, basic), nm = radix_sequence(n, mixed);
    if (nm <= 0 || nm >= nb) return false;
    if (elem == 16) {
        if (regs > 128) return false;
        int nines = 0;
        for (int p = 0; p < nm; ++p) nines += mixed[p] == 9;
        return nines < 2;
    }
    constexpr int kSmem = 227 * 1024;   // an SM's shared memory
    int lines[2];
    double cost[2];
    for (int m = 0; m < 2; ++m) {
        const int *r = m ? mixed : basic, np = m ? nm : nb;
        int l = contiguous ? (int)(4096 / n > 1 ? 4096 / n : 1) : 128 / elem;
        while (l > 1 && (line_threads(r, np, n, l) > kGenericThreads || n * l * elem > kSmem))
            l = contiguous ? (l + 1) / 2 : l / 2;
        const int by_regs = 65536 / (regs * line_threads(r, np, n, l)), by_smem = (int)(kSmem / (n * l * elem + 1024));
        const int ctas = by_regs < by_smem ? by_regs : by_smem;
        lines[m] = l;
        cost[m] = (double)np / ((double)l * (ctas > 1 ? ctas : 1));
    }
    if (!contiguous && lines[1] < lines[0]) cost[1] *= 1.25;
    return cost[1] <= 1.2 * cost[0] * (1 + 1e-9);
}

// Rows per TMA box when a line of n rows is loaded in boxes of at most 256
// rows: the largest divisor of n not above 256, so the boxes tile the line
// exactly; an even one where n is even and takes several boxes, so that boxes of 64-byte
// rows start 128-byte aligned in shared memory (used identically by the kernels and by the
// host's tensor maps).
__host__ __device__ constexpr int tma_box_rows(int n)
{
    if (n <= 256) return n;
    int r = 256;
    while (r > 1 && (n % r != 0 || (n % 2 == 0 && r % 2 != 0))) --r;
    return r;
}

// Elements of a contiguous stage's shared tile of `points` values, 128-byte rows of `row` values
// (pad: one spare value after each row, see SmemTile), rounded up to whole rows.
__host__ __device__ constexpr int contig_tile_elems(int points, int row, bool pad)
{
    const int e = pad ? points + points / row + 1 : points;
    return (e + row - 1) / row * row;
}

struct Launch {
    int lines;                     // lines (columns) per CTA
    int log2_lines;                // log2(lines) for the strided stage (lines is a power of 2)
    int threads;                   // threads per CTA
    int c2r_threads;               // contiguous stage: threads per CTA of the c2r kernel
    size_t smem;                   // dynamic shared memory bytes
    long long blocks;              // grid size
    long long tiles_per_outer;     // strided stage: CTAs per outer slab
};

// Entry points of one kernel family (a specialised line length, or the
// generic kernels), indexed by KS_*.  Signatures, with V = float2 / double2
// and T its real type:
//   strided: (const V *in, V *out, StageDesc d, const V *tw, long long W,
//             long long tiles_per_outer, int log2_lines)
//   contig:  (const V *in, V *out, StageDesc d, const V *tw, long long nlines,
//             int lines, T scale)
//   r2c:     (const T *in, V *out, StageDesc d, const V *tw, const V *post_tw,
//             long long nlines, int lines)
//   c2r:     (const V *in, T *out, StageDesc d, const V *tw, const V *post_tw,
//             long long nlines, int lines, T scale)
enum { KS_STRIDED_FWD = 0, KS_STRIDED_BWD, KS_CONTIG_FWD, KS_CONTIG_BWD, KS_R2C, KS_C2R, KS_COUNT };

// Pipelined strided kernels (persistent CTAs, double-buffered tiles), indexed
// by PIPE_*.  Signature: (const V *in, V *out, CUtensorMap map, const V *tw,
// long long W, long long tiles_per_outer, long long ntiles, unsigned *err,
// const void *twdf, const unsigned *mma, int rev) (twdf: the float-float
// twiddles of an FP64 plan, or null; mma: the tensor-core DFT-16 table of a
// split-precision plan, or null; rev: walk the tiles last to first, see
// StageDesc::rev); the TMA variants read through `map`, a [outer][n][W] view,
// the cp.async ones through `in`; the blocked variants (pipe_blk, TMA) read a
// 4-D map [n / R][outer][R][W] with one box per tile (the blocked c2c
// workspace, or the rows of a [outer][n][W] array grouped by R).  The row-pair
// kernels (pipe_rp) take the same arguments.
enum { PIPE_FWD_TMA = 0, PIPE_FWD_CPASYNC, PIPE_BWD_TMA, PIPE_BWD_CPASYNC, PIPE_COUNT };

struct KernelSet {
    int n;                         // line length (0 for the generic family)
    int npass;
    int radix[kMaxPasses];         // the compile-time radix sequence of a specialised family
    const void *fn[KS_COUNT];
    int max_threads;               // largest CTA the kernels were compiled for
    bool generic;
    bool split;                    // radix-16 passes on the tensor cores
    bool smooth;                   // a family of AFFT_SMOOTH_PLANS
    bool contig_pad;               // the contiguous kernels pad their shared tile (contig_tile_elems)
    const void *pipe[PIPE_COUNT];  // null when the family has no pipelined strided kernel
    const void *pipe_blk[2];       // its blocked-row TMA variants ([0] forward, [1] backward)
    // generic family only: second half of a four-step line, (const V *in, V *out,
    // StageDesc d, const V *tw, const V *wn, long long W, long long tiles_per_outer,
    // int log2_lines, int nb, T scale); [0] forward, [1] backward
    const void *four[2];
    // generic family only: (V *x, long long planes, int n0, int n1, int nhp, int nh)
    const void *poisson_mult;
    // fused Poisson N0 stage (forward DFTs, 1/|k|^2, inverse DFTs) on pipelined tiles:
    // (const V *in, V *out, CUtensorMap map, const V *tw, long long W,
    // long long tiles_per_outer, long long ntiles, unsigned *err, const void *twdf,
    // int n1, int nhp, int nh, int rev, const V *twr, const void *twrdf) (twr, twrdf: the twiddle
    // tables of the reversed radix sequence); [0] TMA, [1] cp.async
    const void *poisson[2];
    int poisson_smem;              // its dynamic shared memory
    int pipe_lines;                // columns per tile of the pipelined kernel
    int pipe_threads;              // its (compile-time) CTA size
    int pipe_smem;                 // its dynamic shared memory (two tile buffers)
    // complex64 families: the pipelined kernels for rows of odd width, read as row pairs
    // through TMA ([0] forward, [1] backward; the first ten arguments of pipe[], see
    // k_strided_pipe_rp), their shared memory and CTA size; null / 0 elsewhere
    const void *pipe_rp[2];
    const void *pipe_rp_early[2];  // the same with the load buffer released after the first pass
    int pipe_smem_rp;
    int pipe_threads_rp;
    bool rp_all_pairs;             // every row-pair pass works on column pairs (radices <= 8)
};

// Specialised kernels for line length n, or nullptr.
const KernelSet *spec_kernels_f32(int n);
const KernelSet *spec_kernels_f64(int n);
// The strided kernels of AFFT_STRIDED_PLANS_F32 / _F64 (lengths whose strided stages prefer another
// radix sequence than their contiguous ones; no contiguous kernels), or nullptr.
const KernelSet *strided_kernels_f32(int n);
const KernelSet *strided_kernels_f64(int n);
// The families of AFFT_SMOOTH_PLANS (the other 2/3/5-smooth lengths up to 1024), or nullptr.
const KernelSet *smooth_kernels_f32(int n);
const KernelSet *smooth_kernels_f64(int n);
// Generic kernels (any n whose radix plan the host builds): radices of basic_sequence, and with the
// radices of radix_sequence too (mixed; no Poisson kernel).
const KernelSet *generic_kernels_f32();
const KernelSet *generic_kernels_f64();
const KernelSet *mixed_kernels_f32();
const KernelSet *mixed_kernels_f64();
// Generic complex64 kernels whose radix-16 passes run on the tensor cores
// (split-precision plans), and the device table of their DFT-16 fragments
// (kSplitTableBytes, written by split_fragments on `stream`).
// Failure-detection self-test (selftest.cu): one CTA waits at most limit_ns on
// an mbarrier that nothing completes, then sets *err.
cudaError_t launch_wait_probe(unsigned *err, unsigned long long limit_ns, cudaStream_t stream);
const KernelSet *generic_kernels_split();

// What the persistent multi-plan executor (queue.cu) reads from a plan.
struct PlanView {
    long long n[3], batch, nh;
    int kind, precision, axes;
    const void *tw;            // twiddle tables (complex of the plan's precision)
    int tw_base[3];            // first twiddle of each axis' tables
    int line_n[3];             // line length of each axis' stages (n0, n1, n2 or n2/2)
    bool specialised[3];       // the axis runs a specialised (compile-time radix) family
    int radix[3][kMaxPasses];  // that family's radix sequence (npass entries)
    int npass[3];
    bool four_step;            // some axis is split four-step
    int post_off;              // r2c: first entry of the w_{n2}^k table
    void *work;                // r2c workspace (n0 n1 nh complex per transform)
    int device;
};
bool plan_view(const afft_plan *p, PlanView *v);
const KernelSet *spec_kernels_split(int n);
// the mma.sync fragments (2 directions x 32 lanes x 32 words), then the tcgen05 operands
// F_hi, F_lo of both directions in the canonical shared-memory layout (2 x 2 x 2 KB)
constexpr size_t kSplitTableBytes = 2 * 32 * 32 * sizeof(unsigned) + 2 * 2 * 32 * 64;
cudaError_t split_fragments(unsigned *table, cudaStream_t stream);

}  // namespace afft
