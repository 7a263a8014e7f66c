// kernels.cuh -- device kernels of the bispectrum-multipole estimator and
// their launch helpers.  Internal to libbisp.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "plan.hpp"

namespace bisp {

template <typename R> struct Cx;
template <> struct Cx<float> { using T = float2; };
template <> struct Cx<double> { using T = double2; };

// Ring table as a kernel argument (membership by the integer test of
// build_rings).
struct RingArg {
    int nr;
    int64_t e3sq[kMaxRings + 1];   // (3 e_r)^2
    int maxc[kMaxRings];
};

// Twiddle table of the transforms, computed on the host in double.  A stage of
// a transform of length F x 2^q (F = 1, 3, 5, 7) that starts from Ns = F x 2^s
// interleaved results (s = 0, 3, 6, ..; Ns <= 512) takes, with w_R = exp(-2 pi i
// / (R Ns)), w_8^(rk) in [r - 1][k] (r = 1 .. 7), then w_4^(rk) (r = 1 .. 3), then
// w_2^k, k < Ns: 11 Ns values, each run contiguous in k.
template <typename C> struct Twiddles {
    const C *t;
    // first element of length family F, and of its stage Ns = F x 2^s (relative)
    static BISP_HD constexpr int offset(int F)
    {
        return 11 * (F == 1 ? 0 : (F == 3 ? 585 : (F == 5 ? 804 : 1169)));
    }
    static BISP_HD constexpr int stage(int F, int s) { return 11 * F * (((1 << s) - 1) / 7); }
};
constexpr int kTwiddles = 11 * 1680;             // F = 1: Ns = 1 .. 512; 3: 3 .. 192; 5: 5 .. 320; 7: 7 .. 448
void make_twiddles(double2 *t);                  // fills kTwiddles values

// Side lengths of the plan's reduction grids, by level index.
struct GridArg {
    int M[kMaxLevels];
};

// Fields of a batched launch: gridDim.y = nf; field f reads its input fs_in
// bytes and writes its output fs_out bytes past field f - 1's (kernels whose
// buffers all lie in one per-field workspace region use fs_in for both).
struct Batch {
    unsigned nf = 1;
    int64_t fs_in = 0, fs_out = 0;
};

// Step-I job: one (plane, ring) field on one reduction grid.
struct Job {
    int32_t n, r;
    int64_t out_off;   // complex elements into the destination store
};

// The reduction grids of a Step-I launch: grid i's jobs take the blocks from
// blk0 on, ntile blocks of rt rows (first pass) or columns (second) per job.  The
// caller fills M, rt (0: the default), jobs and njobs.
struct StepGrid {
    int M, rt;
    const Job *jobs;
    int64_t njobs;
    int ntile, lgw;
    unsigned blk0;
};
struct StepGrids {
    int n = 0;
    StepGrid g[kMaxLevels];
};

struct StepIIArgs {
    const Group *groups;
    const Tile *tiles;
    const Unit *units;
    const int64_t *doff;     // [kMaxLevels][nz+1][kMaxRings]
    int nz1;                 // planes stored: 0 .. nz1 - 1
    int nr;                  // rings per plane
    int64_t x_chunk;         // grid points of one unit
    double *partials;
    int64_t fs;              // bytes between the workspace regions of the fields of a batch
};

// The kernels of an estimate follow one another on a stream, each reading what the
// one before wrote, and at small N_g each lasts a few us: they are launched with
// programmatic stream serialisation, so that a kernel's blocks are placed while the
// last blocks of the one before still run.  Every kernel so launched, and the first of
// an estimate, calls grid_begin before it reads or writes global memory that another
// kernel writes or reads: the next kernel may be placed from here on; this one
// goes on when every kernel before it has completed (each waits so, also blocks
// without work) and its writes are visible.  Pointers that such memory is read through
// are not __restrict__: the compiler may then neither take the read-only path, which is
// for data that nobody writes while the kernel lasts, nor move loads before the wait.
// (The plan's tables are, and the input of an estimate's first kernel, which is launched
// the ordinary way.)
// 32^3 (11 kernels) 79 -> 59 us, 48^3 x 3 202 -> 177, 64^3 173 -> 161; from 128^3 on, 2% of Step I.
__device__ __forceinline__ void grid_begin()
{
    asm volatile("griddepcontrol.launch_dependents;\ngriddepcontrol.wait;\n" ::: "memory");
}
template <typename... P, typename... A>
cudaError_t launch_next(void (*k)(P...), dim3 grid, unsigned threads, size_t smem, cudaStream_t s, A &&...args)
{
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t c{};
    c.gridDim = grid;
    c.blockDim = dim3(threads);
    c.dynamicSmemBytes = smem;
    c.stream = s;
    c.attrs = &at;
    c.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&c, k, P(args)...);
    return e == cudaSuccess ? e : cudaGetLastError();
}

// --- launch helpers (kernels.cu); all return cudaGetLastError() --------------

// z pass of the forward 3D transform: real rows of length ng -> kept
// frequencies [0, nkeep) written transposed as out[k][row].  clear: an int of each
// output region set to zero (a memset of its own cost as much as a small kernel).
template <typename R>
cudaError_t launch_fft_z_real(const R *in, typename Cx<R>::T *out, int ng, int64_t rows, int nkeep,
                              const Twiddles<typename Cx<R>::T> &tw, const Batch &fb, cudaStream_t s, int rt = 0,
                              int *clear = nullptr);

// Batched row transforms written transposed: in[b][nrow][M] -> out[b][M][nrow],
// times scale; zero_dc clears element [0][0] of batch 0.
template <typename R>
cudaError_t launch_fft_rows_T(const typename Cx<R>::T *in, typename Cx<R>::T *out, int M, int nrow,
                              int64_t nb, R scale, bool zero_dc,
                              const Twiddles<typename Cx<R>::T> &tw, const Batch &fb, cudaStream_t s,
                              int rt = 0);

// Real fields out[f][p][z], f < nf, p < M^2, from half spectra in[f][k][p], k < nkeep
// <= M/2 along the line of sight (of k = 0 the real part counts).  M even, at most 128.
template <typename R>
cudaError_t launch_fft_z_back(const typename Cx<R>::T *in, R *out, int M, int nkeep, int64_t nf,
                              const Twiddles<typename Cx<R>::T> &tw, cudaStream_t s);

// Step I, first pass: for every job of the grids, ring r of plane n of Delta
// (planes [nz+1][ng][ng]), folded onto the M x M grid, transformed along u_y,
// written in place order [u_x][k_y] at out + out_off; rows that hold no member
// of the ring are not written.  unit = true uses Delta = 1 (the unit fields of
// Eq. 2FT).  scale: optional factors [nz1][kMaxRings] of the members' values
// (one field's; the next field's lie fb.fs_in bytes further).
template <typename R>
cudaError_t launch_ring_gather(const typename Cx<R>::T *planes, int ng, const RingArg &rings, StepGrids gs, bool unit,
                               typename Cx<R>::T *out, const Twiddles<typename Cx<R>::T> &tw, const Batch &fb,
                               cudaStream_t s, const float *scale = nullptr);

// Power-of-two factor of every (plane, ring) field D(r, n), [nz1][kMaxRings]
// (see k_ring_scale): with it, every |D| on the grid is at most kFieldBound.
// The tensor-core Step II splits the scaled values into FP16 parts; Step I's
// first pass applies the factors (launch_ring_gather's scale).
constexpr float kFieldBound = 250.0f;
cudaError_t launch_ring_scale(const float2 *planes, int ng, int nz1, const RingArg &rings, float *scale,
                              const Batch &fb, cudaStream_t s);

// Step I second pass: the M x M field of every job, as the first pass left it,
// transformed along u_x in place, in strips of columns: [k_x][k_y].  Rows
// that hold no member of the job's ring are taken as zero without being read.
template <typename R>
cudaError_t launch_fft_cols(typename Cx<R>::T *out, StepGrids gs, const RingArg &rings,
                            const Twiddles<typename Cx<R>::T> &tw, const Batch &fb, cudaStream_t s);

// Step II: partial triple sums of units, one block per unit, one launch per
// block class (units [lo[c], hi[c]) run in blocks of 2^c warps with
// kStep2ClassSmem[c] bytes of shared memory; a whole estimate passes
// lo = class_begin, hi = class_begin + 1).
template <typename R>
cudaError_t launch_step2(const StepIIArgs &a, const typename Cx<R>::T *dstore, const int64_t *lo, const int64_t *hi,
                         int nf, cudaStream_t s);

// Step II on tcgen05 (FP32 fields; step2_tc.cu).
struct TcArgs {
    const TcTile *tiles;
    const TcRow *rows;
    const int32_t *slots;
    const TcLane *lanes;
    const TcUnit *units;
    const int64_t *doff;     // [kMaxLevels][nz+1][kMaxRings]
    int nz1, nr;
    int64_t x_chunk;
    double *partials;
    const float *scale;      // field 0's power-of-two factors of the stored fields [nz1][kMaxRings]
    int *status;             // field 0's status word, set to 1 by a block whose wait ran out
    int64_t fs;              // bytes between the workspace regions of the fields of a batch
    int wait_spins;          // polls before an abortable wait gives up
};

// Polls of an mbarrier before a tensor-core Step-II wait gives up (the plan's
// default; estimator_set_wait_limit lowers it to test the give-up path).
constexpr int kDefaultWaitSpins = 1 << 22;

// Device address of estimator_estimate_static's scratch array on the current
// device (noalloc.cu), and the device a plan lives on (abi.cu).
int static_scratch_address(void **out);
int plan_device(const bisp_plan *p);

// One launch per column class: units [lo[c], hi[c]), one block per unit
// with kTcSmem bytes of shared memory.
cudaError_t launch_step2_tc(const TcArgs &a, const float2 *dstore, const int64_t *lo, const int64_t *hi, int nf,
                            cudaStream_t s);

// Allow the kernels their dynamic shared memory once (kernels.cu and
// step2_tc.cu), so that estimates are plain stream work.
cudaError_t init_kernel_attributes();
cudaError_t init_step2_tc_attributes();

// S[c0 + j] = (ng/M)^2 sum_k partials[part0 + k ncombo + j]
template <typename A>
cudaError_t launch_reduce_partials(const Group *groups, int64_t ngroups, const double *partials,
                                   int ng, double *S, const Batch &fb, cudaStream_t s);

// Binning epilogue of Eq. bs_lm2_1 for the moments of even l_lo .. l_hi
// (out and den: [nbins][moments of those l]).  mode 0: B = sqrt((2l+1)/4pi)
// num / (V N_g^2 den) from S and den; mode 1: den from the triangle counts.
// fp32_weights: the Y_lm of each record in FP32 (sums stay in W).
// The records are walked in chunks of one bin each (one warp per chunk, FP64
// partial sums per moment in `partial` [nchunks][moments of l <= l_hi]),
// then each bin adds its chunks in a fixed order (a block per bin, or per
// fin_bins_per_block of them).
struct EpiArgs {
    const Record *rec;                    // fp32_weights: not read (recf is)
    const RecordF *recf;
    const int64_t *chunk_lo, *chunk_hi;   // record range of each chunk
    int64_t nchunks;
    const int64_t *bin_chunk;             // [nbins + 1]: first chunk of each bin
    int64_t nbins;
    double *partial;                      // field 0's partial sums
    int64_t fs_part;                      // bytes between the fields' partial sums
};
template <typename W>
cudaError_t launch_epilogue(int mode, const EpiArgs &e, const double *value, int l_lo, int l_hi, const double *den,
                            double norm, double *out, const Batch &fb, cudaStream_t s, bool fp32_weights = false);

// The same (mode 0) for all views of a plan in one launch per pass: the views do
// not depend on one another, and at a few thousand chunks each a launch is short
// and leaves most of the GPU idle.  blk0, fin0 and per are the launcher's.
struct EpiView {
    const int64_t *chunk_lo, *chunk_hi, *bin_chunk;
    int64_t nchunks, nbins;
    double *partial;                      // this view's own [nchunks][moments of l <= l_hi]
    const double *den;
    double *out;
    int l_hi, lm_lo, nlm;                 // first moment and moments written
    unsigned blk0, fin0;                  // first block of the chunks' and of the bins' launch
};
struct EpiViews {
    int n;
    const Record *rec;
    const RecordF *recf;
    int64_t per;                          // bins of a block of the bins' launch
    EpiView v[5];                         // even l <= 8
};
template <typename W>
cudaError_t launch_epilogue_views(EpiViews ev, const double *value, double norm, const Batch &fb, cudaStream_t s,
                                  bool fp32_weights);

// The records' FP32 form.
cudaError_t launch_records_f(const Record *rec, RecordF *recf, int64_t n, cudaStream_t s);

// Y_lm normalisations nlm[l][m] and the prefactors sqrt((2l+1)/(4 pi)).
cudaError_t set_ylm_constants(const double nlm[9][9], const double pref[9], cudaStream_t s);

// Welford update of per-element count, mean and squared deviations with
// nf fields B[f][0 .. n-1] (non-finite values skipped).
cudaError_t launch_stats_update(const double *B, int nf, int64_t n, int64_t *count, double *mean, double *m2,
                                cudaStream_t s);

// N_tri of unordered ring triples from the unit fields (Eq. Ntri2), FP64.
// triples[4 t .. 4 t + 3] = (r1, r2, r3, level index into grids.M).
cudaError_t launch_ntri(const double2 *ifields, const int64_t *ioff, const int32_t *triples,
                        int64_t ntriples, const GridArg &grids, double *raw, cudaStream_t s);

// Sizes of dynamic shared memory (bytes) of the transform kernels.
// Rows of length M a transform block holds: each of its two shared-memory
// buffers takes about `bytes` (1 .. 256 rows).  rt = 0 passed to the
// launchers above selects this with the default 16 KB; the plan's autotuner
// passes its own choice.
size_t fft_rows_per_block(int M, size_t elem, size_t bytes = 16384);
// Elements from one row of a transform's shared-memory buffer to the next.  An
// element's place in its row is its index with the low four bits exchanged
// (spos in kernels.cu), so a row takes a multiple of 16; what is added to it
// spreads the rows over the banks (16 of 8 bytes, or 8 of 16) where a warp's
// lanes run across `across` rows first and along them second.
template <typename C> inline __host__ __device__ constexpr int fft_stride(int M, int across)
{
    const int banks = 128 / int(sizeof(C));
    return ((M + 15) & ~15) + (across >= banks ? 1 : (2 * across >= banks ? 2 : (4 * across >= banks ? 4 : banks / 2)));
}

}  // namespace bisp
