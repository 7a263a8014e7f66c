// kernels.cu -- CUDA kernels of the bispectrum-multipole estimator
// (Gill & Bharadwaj, arXiv:2405.14513, Sec. II) for sm_103a.
//
//   k_fft_z_real    forward transform along the line of sight (real rows),
//                   keeping planes 0..N_g/3, written plane-major
//   k_fft_rows_T    batched row transforms written transposed (the y and x
//                   passes of the forward transform)
//   k_fft_z_back    real fields from their half spectra, along the line of sight
//                   (the shell estimator's fields)
//   k_ring_gather   Step I first pass: ring mask (and fold onto the M x M
//                   reduction grid) fused into the load, transform along u_y
//   k_fft_cols      Step I second pass: transform along u_x, in place
//   k_ring_scale    power-of-two factors of the D fields (tensor-core Step II)
//   k_step2         Step II: partial triple sums sum_x D1 D2 D3 (Eq. fftbs)
//   k_reduce        partial sums -> S per combination, grid normalisation
//   k_epi_part, k_epi_fin  Y_lm weights, (k1, mu, t) binning and the ratio of
//                   Eq. bs_lm2_1; or the plan-time denominators
//   k_ntri          N_tri = M^-2 sum_y I1 I2 I3 on the unit fields (Eq. Ntri2)
//
// All transforms use exp(-i k.x), the sign of Eq. iFT.  Transform lengths
// are 2^q, 3 x 2^q, 5 x 2^q or 7 x 2^q (N_g and the reduction grids of the
// plan); the twiddle tables (Twiddles) are computed on the host in double.
#include "kernels.cuh"

#include <algorithm>
#include <cmath>
#include <type_traits>

namespace bisp {

namespace {

__device__ __forceinline__ float2 cmul(float2 a, float2 b)
{
    return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__device__ __forceinline__ double2 cmul(double2 a, double2 b)
{
    return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double2 cadd(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 csub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ double2 csub(double2 a, double2 b) { return make_double2(a.x - b.x, a.y - b.y); }
template <typename C> __device__ __forceinline__ C cmk(double re, double im);
template <> __device__ __forceinline__ float2 cmk<float2>(double re, double im) { return make_float2(float(re), float(im)); }
template <> __device__ __forceinline__ double2 cmk<double2>(double re, double im) { return make_double2(re, im); }

// Field f = blockIdx.y of a batched launch: its buffers sit fs bytes apart.
template <typename T> __device__ __forceinline__ T *field_ptr(T *p, int64_t fs)
{
    return reinterpret_cast<T *>(reinterpret_cast<char *>(p) + int64_t(blockIdx.y) * fs);
}
template <typename T> __device__ __forceinline__ const T *field_ptr(const T *p, int64_t fs)
{
    return reinterpret_cast<const T *>(reinterpret_cast<const char *>(p) + int64_t(blockIdx.y) * fs);
}

// t = q d + r along t = t0, t0 + step, ...: quotient and remainder kept
// incrementally (one division per thread rather than one per element)
struct DivIter {
    int q, r, dq, dr, d;
    __device__ __forceinline__ DivIter(int t0, int step, int d_) : d(d_)
    {
        q = t0 / d;
        r = t0 - q * d;
        dq = step / d;
        dr = step - dq * d;
    }
    __device__ __forceinline__ void next()
    {
        q += dq;
        r += dr;
        if (r >= d) {
            r -= d;
            ++q;
        }
    }
};

// Shared-memory position of element i of a transform row: the low four bits
// exchanged with those of i / 8, so that runs of 16 elements and elements 8 or 64
// apart (the strided stores of the first radix-8 stages) each fall in different
// banks.  (A padding slot after every 8 elements, which this replaces, made runs
// take two accesses where one will do: the kernels were bound by them, up to 93% of
// the L1's wavefronts.)
__device__ __forceinline__ int spos(int i) { return i ^ ((i >> 3) & 15); }

// a + c x and c x for a constant c of a butterfly.  FINE: FP32 takes it in two parts, c
// rounded and what that leaves.  A rounded constant is off the same way in every
// butterfly (1/sqrt(2) by 1.7e-8 of itself, and most points of a transform meet it two
// or three times), which makes all amplitudes smaller alike, and a triple product takes
// that three times: with rounded constants the planes of Delta were 4e-8 (24^3) to 7e-8
// (96^3) too small, so 2e-8 to 5e-8 (what is left comes from the twiddles), and B's
// errors against 64 bits fell by 6 to 15% (the shell estimator's by 20 to 40%).  Step I
// keeps to one part: with two there as well the estimate of 384^3 x 10 took 63.5 ms
// instead of 63.1.
struct Const {
    double c;
    __host__ __device__ constexpr Const operator-() const { return Const{-c}; }
};
template <bool FINE> __device__ __forceinline__ float muladd(Const k, float x, float a)
{
    const float h = float(k.c), l = float(k.c - double(h));
    return fmaf(h, x, FINE ? fmaf(l, x, a) : a);
}
template <bool FINE> __device__ __forceinline__ double muladd(Const k, double x, double a) { return fma(k.c, x, a); }
template <bool FINE> __device__ __forceinline__ float mul(Const k, float x)
{
    const float h = float(k.c), l = float(k.c - double(h));
    return FINE ? fmaf(h, x, l * x) : h * x;
}
template <bool FINE> __device__ __forceinline__ double mul(Const k, double x) { return k.c * x; }

// DFT of R values in registers, X_m = sum_r v_r exp(-2 pi i r m / R), in place.
template <int R, bool FINE, typename C> __device__ __forceinline__ void dft(C (&v)[R])
{
    using Rr = decltype(v[0].x);
    if constexpr (R == 2) {
        const C t = csub(v[0], v[1]);
        v[0] = cadd(v[0], v[1]);
        v[1] = t;
    } else if constexpr (R == 3) {
        constexpr Const h{0.86602540378443864676};   // sqrt(3)/2
        const Rr sx = v[1].x + v[2].x, sy = v[1].y + v[2].y, dx = v[1].x - v[2].x, dy = v[1].y - v[2].y;
        const Rr mx = v[0].x - Rr(0.5) * sx, my = v[0].y - Rr(0.5) * sy;
        v[0].x += sx; v[0].y += sy;
        v[1].x = muladd<FINE>(h, dy, mx); v[1].y = muladd<FINE>(-h, dx, my);
        v[2].x = muladd<FINE>(-h, dy, mx); v[2].y = muladd<FINE>(h, dx, my);
    } else if constexpr (R == 4) {
        const C s02 = cadd(v[0], v[2]), d02 = csub(v[0], v[2]), s13 = cadd(v[1], v[3]), d13 = csub(v[1], v[3]);
        v[0] = cadd(s02, s13);
        v[2] = csub(s02, s13);
        v[1] = d02;                                // d02 -/+ i d13
        v[1].x += d13.y; v[1].y -= d13.x;
        v[3] = d02;
        v[3].x -= d13.y; v[3].y += d13.x;
    } else if constexpr (R == 5) {
        // w = exp(-2 pi i/5):
        //   y_0 = v0 + s1 + s2,  s1 = v1 + v4,  s2 = v2 + v3,  d1 = v1 - v4,  d2 = v2 - v3,
        //   y_1, y_4 = v0 + c1 s1 + c2 s2 -/+ i (n1 d1 + n2 d2),
        //   y_2, y_3 = v0 + c2 s1 + c1 s2 -/+ i (n2 d1 - n1 d2),
        // c_m = cos(2 pi m/5), n_m = sin(2 pi m/5)
        const Rr c1 = Rr(0.30901699437494742410), c2 = Rr(-0.80901699437494742410);
        const Rr n1 = Rr(0.95105651629515357212), n2 = Rr(0.58778525229247312917);
        const C s1 = cadd(v[1], v[4]), s2 = cadd(v[2], v[3]), d1 = csub(v[1], v[4]), d2 = csub(v[2], v[3]);
        C a1, a2, b1, b2;
        a1.x = v[0].x + c1 * s1.x + c2 * s2.x; a1.y = v[0].y + c1 * s1.y + c2 * s2.y;
        a2.x = v[0].x + c2 * s1.x + c1 * s2.x; a2.y = v[0].y + c2 * s1.y + c1 * s2.y;
        b1.x = n1 * d1.x + n2 * d2.x; b1.y = n1 * d1.y + n2 * d2.y;
        b2.x = n2 * d1.x - n1 * d2.x; b2.y = n2 * d1.y - n1 * d2.y;
        // -i b = (b.y, -b.x)
        v[0].x = v[0].x + s1.x + s2.x; v[0].y = v[0].y + s1.y + s2.y;
        v[1].x = a1.x + b1.y; v[1].y = a1.y - b1.x;
        v[2].x = a2.x + b2.y; v[2].y = a2.y - b2.x;
        v[3].x = a2.x - b2.y; v[3].y = a2.y + b2.x;
        v[4].x = a1.x - b1.y; v[4].y = a1.y + b1.x;
    } else if constexpr (R == 7) {
        // by the same pairing: s_k = v_k + v_{7-k},  d_k = v_k - v_{7-k}  (k = 1, 2, 3),
        //   y_m, y_{7-m} = v0 + sum_k cos(2 pi mk/7) s_k -/+ i sum_k sin(2 pi mk/7) d_k  (m = 1, 2, 3)
        const Rr c1 = Rr(0.62348980185873353053), c2 = Rr(-0.22252093395631440429), c3 = Rr(-0.90096886790241912624);
        const Rr n1 = Rr(0.78183148246802980871), n2 = Rr(0.97492791218182360702), n3 = Rr(0.43388373911755812048);
        const C s1 = cadd(v[1], v[6]), s2 = cadd(v[2], v[5]), s3 = cadd(v[3], v[4]);
        const C d1 = csub(v[1], v[6]), d2 = csub(v[2], v[5]), d3 = csub(v[3], v[4]);
        C am[3], bm[3];
        am[0].x = v[0].x + c1 * s1.x + c2 * s2.x + c3 * s3.x; am[0].y = v[0].y + c1 * s1.y + c2 * s2.y + c3 * s3.y;
        am[1].x = v[0].x + c2 * s1.x + c3 * s2.x + c1 * s3.x; am[1].y = v[0].y + c2 * s1.y + c3 * s2.y + c1 * s3.y;
        am[2].x = v[0].x + c3 * s1.x + c1 * s2.x + c2 * s3.x; am[2].y = v[0].y + c3 * s1.y + c1 * s2.y + c2 * s3.y;
        bm[0].x = n1 * d1.x + n2 * d2.x + n3 * d3.x; bm[0].y = n1 * d1.y + n2 * d2.y + n3 * d3.y;
        bm[1].x = n2 * d1.x - n3 * d2.x - n1 * d3.x; bm[1].y = n2 * d1.y - n3 * d2.y - n1 * d3.y;
        bm[2].x = n3 * d1.x - n1 * d2.x + n2 * d3.x; bm[2].y = n3 * d1.y - n1 * d2.y + n2 * d3.y;
        v[0].x = v[0].x + s1.x + s2.x + s3.x; v[0].y = v[0].y + s1.y + s2.y + s3.y;
#pragma unroll
        for (int m = 0; m < 3; ++m) {
            // -i b = (b.y, -b.x)
            v[m + 1].x = am[m].x + bm[m].y; v[m + 1].y = am[m].y - bm[m].x;
            v[6 - m].x = am[m].x - bm[m].y; v[6 - m].y = am[m].y + bm[m].x;
        }
    } else {
        static_assert(R == 8, "radix");
        // a radix-2 step (pairs r, r + 4; the odd half turned by
        // exp(-2 pi i r / 8)) followed by two 4-point transforms
        constexpr Const r2{0.70710678118654752440};  // 1/sqrt(2)
        C e[4], o[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            e[r] = cadd(v[r], v[r + 4]);
            o[r] = csub(v[r], v[r + 4]);
        }
        // o_1 exp(-i pi/4), o_2 (-i), o_3 exp(-3 i pi/4)
        const C t1 = o[1], t3 = o[3];
        o[1].x = mul<FINE>(r2, t1.x + t1.y); o[1].y = mul<FINE>(r2, t1.y - t1.x);
        const Rr x2 = o[2].x;
        o[2].x = o[2].y; o[2].y = -x2;
        o[3].x = mul<FINE>(r2, t3.y - t3.x); o[3].y = -mul<FINE>(r2, t3.x + t3.y);
        dft<4, FINE>(e);
        dft<4, FINE>(o);
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            v[2 * m] = e[m];
            v[2 * m + 1] = o[m];
        }
    }
}

// Rows of a transform block: nr rows of length M = F x 2^p, on the threads
// either along the row (consecutive threads take consecutive elements) or, ACROSS,
// across 2^lgw >= nr rows (consecutive threads take the same element of
// consecutive rows).
struct FftRows {
    int M, p, nr, lgw;
};

// One Stockham stage of radix R on every row: out[q R Ns + k + m Ns] =
// sum_r w^(rk) x[j + r M/R] exp(-2 pi i rm / R) with j = q Ns + k and
// w = exp(-2 pi i / (R Ns)) (tw: its table [r - 1][k], null in a first
// stage); get(row, i) and put(row, i, value) read and write an element.  Every
// index split is a shift, or a shift and a division by the constant F.
template <typename C, int F, bool ACROSS, bool FINE, int R, typename G, typename S>
__device__ __forceinline__ void fft_stage(const FftRows &fr, int Ns, int s, const C *__restrict__ tw, G get, S put)
{
    constexpr int LR = R == 8 ? 3 : (R == 4 ? 2 : (R == 2 ? 1 : 0));
    auto divF = [](int x) { return F == 1 ? x : int(unsigned(x) / unsigned(F)); };
    const int nb = R == F ? 1 << fr.p : F << (fr.p - LR);     // butterflies per row
    const int total = ACROSS ? nb << fr.lgw : nb * fr.nr;
    for (int t = threadIdx.x; t < total; t += blockDim.x) {
        int row, j;
        if (ACROSS) {
            row = t & ((1 << fr.lgw) - 1);
            j = t >> fr.lgw;
            if (row >= fr.nr) continue;
        } else {
            row = R == F ? t >> fr.p : divF(t >> (fr.p - LR));
            j = t - row * nb;
        }
        int q = j, k = 0;
        if (Ns > 1) {
            q = divF(j >> s);
            k = j - q * Ns;
        }
        C v[R];
#pragma unroll
        for (int r = 0; r < R; ++r) v[r] = get(row, j + r * nb);
        if (tw) {
#pragma unroll
            for (int r = 1; r < R; ++r) v[r] = cmul(v[r], __ldg(tw + (r - 1) * Ns + k));
        }
        dft<R, FINE>(v);
        const int d0 = q * R * Ns + k;
#pragma unroll
        for (int m = 0; m < R; ++m) put(row, d0 + m * Ns, v[m]);
    }
}

// Stockham transform X_k = sum_j x_j exp(-2 pi i jk / M) of the block's rows:
// one radix-F stage first when F > 1, then radix-8 stages and, for what is
// left of the power of two, one radix-4 or radix-2 stage.  The first stage
// takes its elements from `load` and the last hands them to `store` (SMEM:
// leaves them in the returned buffer instead, block synchronised), so that
// between global memory and the registers a transform of three stages (2^q up to
// 512, F x 2^q with q up to 6) crosses shared memory twice, not four times.  a, b:
// buffers of nr rows of stride P.  Every thread of the block takes part.
template <typename C, int F, bool ACROSS, bool SMEM, bool FINE, typename G, typename S>
__device__ __forceinline__ C *fft_block(const FftRows &fr, int P, C *a, C *b, const C *__restrict__ tw, G load, S store)
{
    auto from = [&](C *x) { return [x, P](int row, int i) { return x[row * P + spos(i)]; }; };
    auto into = [&](C *x) { return [x, P](int row, int i, const C &v) { x[row * P + spos(i)] = v; }; };
    constexpr int R1 = F > 1 ? F : 8;
    int Ns = R1, s = F > 1 ? 0 : 3;                 // Ns = F 2^s
    if (F == 1 && fr.M == 8) {
        if constexpr (SMEM) {
            fft_stage<C, F, ACROSS, FINE, R1>(fr, 1, 0, nullptr, load, into(a));
            __syncthreads();
        } else {
            fft_stage<C, F, ACROSS, FINE, R1>(fr, 1, 0, nullptr, load, store);
        }
        return a;
    }
    fft_stage<C, F, ACROSS, FINE, R1>(fr, 1, 0, nullptr, load, into(a));
    __syncthreads();
    const C *w = tw + Twiddles<C>::offset(F);
    for (;; s += 3) {
        const int lg = fr.p - s;                    // what is left: 2^lg
        const C *w8 = w + Twiddles<C>::stage(F, s);
        if (lg > 3) {
            fft_stage<C, F, ACROSS, FINE, 8>(fr, Ns, s, w8, from(a), into(b));
            __syncthreads();
            C *t = a;
            a = b;
            b = t;
            Ns *= 8;
            continue;
        }
        if constexpr (SMEM) {
            if (lg == 3) fft_stage<C, F, ACROSS, FINE, 8>(fr, Ns, s, w8, from(a), into(b));
            else if (lg == 2) fft_stage<C, F, ACROSS, FINE, 4>(fr, Ns, s, w8 + 7 * Ns, from(a), into(b));
            else fft_stage<C, F, ACROSS, FINE, 2>(fr, Ns, s, w8 + 10 * Ns, from(a), into(b));
            __syncthreads();
        } else {
            if (lg == 3) fft_stage<C, F, ACROSS, FINE, 8>(fr, Ns, s, w8, from(a), store);
            else if (lg == 2) fft_stage<C, F, ACROSS, FINE, 4>(fr, Ns, s, w8 + 7 * Ns, from(a), store);
            else fft_stage<C, F, ACROSS, FINE, 2>(fr, Ns, s, w8 + 10 * Ns, from(a), store);
        }
        return b;
    }
}

// fft_block of rows of length M = 2^q, 3 x 2^q, 5 x 2^q or 7 x 2^q
// (block-uniform dispatch).  STEP1 = false: of 2^q or 3 x 2^q, the lengths of N_g, with
// the butterflies' constants in two parts (see muladd)
template <typename C, bool ACROSS, bool SMEM, bool STEP1, typename G, typename S>
__device__ __forceinline__ C *fft_any(int M, int nr, int lgw, int P, C *a, C *b, const C *__restrict__ tw, G load, S store)
{
    const FftRows fr{M, __ffs(M) - 1, nr, lgw};
    const int odd = M >> fr.p;
    if constexpr (STEP1) {
        if (odd == 7) return fft_block<C, 7, ACROSS, SMEM, false>(fr, P, a, b, tw, load, store);
        if (odd == 5) return fft_block<C, 5, ACROSS, SMEM, false>(fr, P, a, b, tw, load, store);
    }
    if (odd == 3) return fft_block<C, 3, ACROSS, SMEM, !STEP1>(fr, P, a, b, tw, load, store);
    return fft_block<C, 1, ACROSS, SMEM, !STEP1>(fr, P, a, b, tw, load, store);
}

// no store: the transform's result stays in shared memory
struct NoStore {
    template <typename C> __device__ void operator()(int, int, const C &) const {}
};

// ---------------------------------------------------------------------------
template <typename R>
__global__ void __launch_bounds__(256)
k_fft_z_real(const R *__restrict__ in, typename Cx<R>::T *__restrict__ out, int M, int64_t rows,
             int nkeep, int rt, Twiddles<typename Cx<R>::T> tw, int64_t fs_in, int64_t fs_out, int *clear)
{
    using C = typename Cx<R>::T;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    grid_begin();
    in = field_ptr(in, fs_in);
    out = field_ptr(out, fs_out);
    if (clear && blockIdx.x == 0 && threadIdx.x == 0) *field_ptr(clear, fs_out) = 0;
    const int P = fft_stride<C>(M, rt);
    C *a = reinterpret_cast<C *>(smem_raw);
    C *b = a + rt * P;
    // two real rows a, b share a transform of a + i b (the number of rows is
    // even): half the transforms of a kernel that is bound by its shared-memory
    // accesses (forward transform, 384^3 x 10: 4.5 -> 3.4 ms)
    const int64_t row0 = int64_t(blockIdx.x) * 2 * rt;
    const int npair = int(min(int64_t(rt), (rows - row0) / 2));
    const R *src = in + row0 * M;
    const C *res = fft_any<C, false, true, false>(
        M, npair, 0, P, a, b, tw.t,
        [&](int r, int i) {
            C v;
            v.x = src[2 * r * M + i];
            v.y = src[(2 * r + 1) * M + i];
            return v;
        },
        NoStore{});
    // A_k = (X_k + conj X_{M-k}) / 2,  B_k = (X_k - conj X_{M-k}) / (2 i)
    DivIter st(threadIdx.x, blockDim.x, npair);
    for (int t = threadIdx.x; t < nkeep * npair; t += blockDim.x, st.next()) {
        const int k = st.q, r = st.r;
        const C x = res[r * P + spos(k)], y = res[r * P + spos(k == 0 ? 0 : M - k)];
        C *o = out + int64_t(k) * rows + row0 + 2 * r;
        C u, v;
        u.x = R(0.5) * (x.x + y.x); u.y = R(0.5) * (x.y - y.y);
        v.x = R(0.5) * (x.y + y.y); v.y = R(0.5) * (y.x - x.x);
        o[0] = u;
        o[1] = v;
    }
}

template <typename R>
__global__ void __launch_bounds__(256)
k_fft_rows_T(const typename Cx<R>::T *in, typename Cx<R>::T *__restrict__ out, int M,
             int nrow, int ntile, R scale, int zero_dc, int rt, Twiddles<typename Cx<R>::T> tw, int64_t fs)
{
    using C = typename Cx<R>::T;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    grid_begin();
    in = field_ptr(in, fs);
    out = field_ptr(out, fs);
    const int P = fft_stride<C>(M, rt);
    C *a = reinterpret_cast<C *>(smem_raw);
    C *b = a + rt * P;
    const int64_t bt = blockIdx.x / ntile;
    const int tile = int(blockIdx.x - bt * ntile);
    const int row0 = tile * rt;
    const int nr = min(rt, nrow - row0);
    const C *src = in + bt * int64_t(M) * nrow + int64_t(row0) * M;
    const C *res = fft_any<C, false, true, false>(M, nr, 0, P, a, b, tw.t, [&](int r, int i) { return src[r * M + i]; },
                                                  NoStore{});
    C *dst = out + bt * int64_t(M) * nrow;
    DivIter st(threadIdx.x, blockDim.x, nr);
    for (int t = threadIdx.x; t < M * nr; t += blockDim.x, st.next()) {
        const int k = st.q, r = st.r;
        C v = res[r * P + spos(k)];
        v.x *= scale;
        v.y *= scale;
        if (zero_dc && bt == 0 && row0 + r == 0 && k == 0) v = cmk<C>(0.0, 0.0);
        dst[int64_t(k) * nrow + row0 + r] = v;
    }
}

// Real fields of half spectra in[f][k][p], k < nkeep along the line of sight, p the
// M^2 points of a plane: out[f][p][z] = Re A_0 + sum over 0 < k < nkeep of
// 2 Re(A_k exp(-2 pi i kz / M)) (A_{-k} = conj A_k).  Two rows A, B share a transform
// of A + i B, neighbours of one field, so that a field's rounding errors are those
// of its own size whatever the other fields hold.  A block takes w = 2^lgw pairs: the
// threads run across them, so that the loads are runs of 2 w elements of a plane, and
// the rows leave shared memory whole.  Bound by instruction issue (23 fields of 128^3,
// 0.14 ms: 72% of the slots, shared memory 54%, DRAM 24%; 64^3: 60%, and barriers).
template <typename R>
__global__ void __launch_bounds__(256)
k_fft_z_back(const typename Cx<R>::T *in, R *__restrict__ out, int M, int nkeep, int ntile, int lgw,
             Twiddles<typename Cx<R>::T> tw)
{
    using C = typename Cx<R>::T;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    grid_begin();
    const int w = 1 << lgw, npos = M * M;
    const int P = fft_stride<C>(M, w);
    C *a = reinterpret_cast<C *>(smem_raw);
    C *b = a + w * P;
    const int64_t f = blockIdx.x / ntile;
    const int p0 = int(blockIdx.x - f * ntile) * 2 * w;
    const int nr = min(w, (npos - p0) / 2);        // pairs of rows (npos is even)
    const C *src = in + f * nkeep * npos + p0;
    auto load = [&](int r, int i) {
        const bool neg = 2 * i > M;                // A_{i - M} = conj A_{M - i}
        const int k = neg ? M - i : i;
        if (k >= nkeep) return cmk<C>(0.0, 0.0);
        const C *q = src + int64_t(k) * npos + 2 * r;
        const C u = q[0], v = q[1];
        C x;
        if (k == 0) {                              // real
            x.x = u.x;
            x.y = v.x;
        } else {
            x.x = neg ? u.x + v.y : u.x - v.y;
            x.y = neg ? v.x - u.y : v.x + u.y;
        }
        return x;
    };
    const C *res = fft_any<C, true, true, false>(M, nr, lgw, P, a, b, tw.t, load, NoStore{});
    R *dst = out + (f * npos + p0) * M;
    DivIter st(threadIdx.x, blockDim.x, M);
    for (int t = threadIdx.x; t < 2 * nr * M; t += blockDim.x, st.next()) {
        const C v = res[(st.q >> 1) * P + spos(st.r)];
        dst[t] = (st.q & 1) ? v.y : v.x;
    }
}

// scale[n][r] = the power of two 2^e with 2^e sum (|Re Delta| + |Im Delta|)
// in (kFieldBound / 2, kFieldBound], the sum over ring r of plane n.  No
// |D(r, n, x)| 2^e exceeds that sum, so a product of two scaled fields stays
// below 62500, inside FP16, while a typical value (the root mean square of a
// Gaussian field is about the bound over the square root of the ring's mode
// count) stays near or above 1/2 up to N_g = 1024, so that the low part of an
// FP16 pair keeps its 11 bits.  One block per (ring, plane), eight lanes per row
// u_x, 32 rows at a time: the loads of a row are a few runs of u_y, so the
// kernel is bound by their latency (a warp per row took 0.3 ms a field at
// 384^3, this one a tenth of it).  Every sum is in a fixed order.  Empty or
// non-finite rings get 1.
__global__ void __launch_bounds__(256)
k_ring_scale(const float2 *planes, int ng, RingArg rings, float *__restrict__ scale, int64_t fs)
{
    grid_begin();
    planes = field_ptr(planes, fs);
    scale = field_ptr(scale, fs);
    const int r = blockIdx.x % rings.nr, n = blockIdx.x / rings.nr;
    const float2 *pl = planes + int64_t(n) * ng * ng;
    // members: lo <= |u|^2 < hi (9 |u|^2 is compared with squares of 3 e_r)
    const int lo = int((rings.e3sq[r] + 8) / 9), hi = int((rings.e3sq[r + 1] + 8) / 9);
    const int mc = rings.maxc[r], grp = threadIdx.x >> 3, sub = threadIdx.x & 7;
    float sum = 0.0f;
#pragma unroll 2
    for (int ux = -mc + grp; ux <= mc; ux += 32) {
        const float2 *row = pl + int64_t(ux < 0 ? ux + ng : ux) * ng;
        // |u_y| from just inside the inner edge on (members are tested exactly)
        const int in2 = lo - ux * ux, out2 = hi - ux * ux;
        const int first = in2 > 0 ? max(0, int(sqrtf(float(in2))) - 1) : 0;
        for (int a = first + sub; a * a < out2; a += 8) {
            if (a * a < in2) continue;
            const float2 v = row[a];
            const float2 w = a == 0 ? make_float2(0.0f, 0.0f) : row[ng - a];
            sum += (fabsf(v.x) + fabsf(v.y)) + (fabsf(w.x) + fabsf(w.y));
        }
    }
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_down_sync(0xffffffffu, sum, o);
    __shared__ float wsum[8];
    if ((threadIdx.x & 31) == 0) wsum[threadIdx.x >> 5] = sum;
    __syncthreads();
    if (threadIdx.x != 0) return;
    float b = 0.0f;
    for (int w = 0; w < 8; ++w) b += wsum[w];
    b *= 1.0f / kFieldBound;
    int e = 0;
    if (b > 0.0f && isfinite(b)) {
        const float m = frexpf(b, &e);             // b = m 2^e, 1/2 <= m < 1
        e = m == 0.5f ? 1 - e : -e;                // the largest e with b 2^e <= 1
        e = max(-100, min(100, e));
    }
    scale[n * kMaxRings + r] = ldexpf(1.0f, e);
}

// rows that the lanes of a first-pass warp run across: several where a row is short
__host__ __device__ __forceinline__ constexpr int gather_across(int M) { return M >= 128 ? 16 : 2; }

// the grid of a Step-I block (the grids of a launch in order of their blocks)
__device__ __forceinline__ const StepGrid &grid_of_block(const StepGrids &gs)
{
    int i = 0;
    while (i + 1 < gs.n && blockIdx.x >= gs.g[i + 1].blk0) ++i;
    return gs.g[i];
}

template <typename R, bool UNIT>
__global__ void __launch_bounds__(256)
k_ring_gather(const typename Cx<R>::T *planes, int ng, const __grid_constant__ RingArg rings,
              const __grid_constant__ StepGrids gs, typename Cx<R>::T *__restrict__ out,
              Twiddles<typename Cx<R>::T> tw, const float *scale, int64_t fs)
{
    using C = typename Cx<R>::T;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    grid_begin();
    planes = field_ptr(planes, fs);
    out = field_ptr(out, fs);
    scale = scale ? field_ptr(scale, fs) : scale;
    const StepGrid &gr = grid_of_block(gs);
    const int M = gr.M, rt = gr.rt;
    const int P = fft_stride<C>(M, gather_across(M));
    C *a = reinterpret_cast<C *>(smem_raw);
    C *b = a + rt * P;
    const int blk = int(blockIdx.x - gr.blk0), jb = blk / gr.ntile;
    const Job J = gr.jobs[jb];
    const C *pl = planes + int64_t(J.n) * ng * ng;
    // members: lo <= |u|^2 < hi (9 |u|^2 is compared with squares of 3 e_r)
    const int lo = int((rings.e3sq[J.r] + 8) / 9), hi = int((rings.e3sq[J.r + 1] + 8) / 9);
    const int mc = rings.maxc[J.r];
    const R fac = scale ? R(scale[J.n * kMaxRings + J.r]) : R(1);
    const int row0 = (blk - jb * gr.ntile) * rt;
    const int nr = min(rt, M - row0);
    // rows i hold ring members only where |u_x| <= maxc for u_x = i or i - M;
    // a block of rows without members is zero after the transform too, and
    // the column pass reads such rows as zero without loading them
    if (row0 > mc && row0 + nr - 1 < M - mc) return;
    // element (row, j): members u with u_x = i or i - M and u_y = j or j - M
    // (mod M folding; |u_x|, |u_y| <= maxc < M, so no other alias exists)
    auto load = [&](int row, int j) {
        const int i = row0 + row;
        R vr = 0, vi = 0;
#pragma unroll
        for (int ca = 0; ca < 2; ++ca) {
            const int ux = ca ? i - M : i;
            if (ux > mc || ux < -mc) continue;
            const C *prow = pl + int64_t(ux < 0 ? ux + ng : ux) * ng;
#pragma unroll
            for (int cb = 0; cb < 2; ++cb) {
                const int uy = cb ? j - M : j;
                if (uy > mc || uy < -mc) continue;
                const int q = ux * ux + uy * uy;
                if (q < lo || q >= hi) continue;
                if (UNIT) {
                    vr += R(1);
                } else {
                    const C v = prow[uy < 0 ? uy + ng : uy];
                    vr += v.x * fac;
                    vi += v.y * fac;
                }
            }
        }
        C v;
        v.x = vr;
        v.y = vi;
        return v;
    };
    // whole rows (u_x, k_y) of the job's M x M field in place: coalesced
    C *dst = out + J.out_off + int64_t(row0) * M;
    fft_any<C, false, false, true>(M, nr, 0, P, a, b, tw.t, load, [&](int row, int k, const C &v) { dst[row * M + k] = v; });
}

// Step I second pass: transforms along the first axis of each job's M x M
// field (rows u_x of the gather's output), in place: a strip of w columns k_y
// per block, of all the columns of the grid's jobs one after another (a block of a
// small grid takes several jobs' columns), read (by the first stage) and written
// (by the last) in runs of consecutive elements of every row, so the D field
// comes out as [k_x][k_y].  The threads run across the strip first: the runs are
// whole 32-byte sectors for w >= 4, the lanes of a warp take few different
// twiddles, and a thread's column is the same throughout.
template <typename R>
__global__ void __launch_bounds__(256)
k_fft_cols(typename Cx<R>::T *out, const __grid_constant__ StepGrids gs,
           const __grid_constant__ RingArg rings, Twiddles<typename Cx<R>::T> tw, int64_t fs)
{
    using C = typename Cx<R>::T;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    grid_begin();
    out = field_ptr(out, fs);
    const StepGrid &gr = grid_of_block(gs);
    const int M = gr.M, w = gr.rt;
    const int P = fft_stride<C>(M, w);
    C *a = reinterpret_cast<C *>(smem_raw);
    C *b = a + w * P;
    const int64_t c0 = int64_t(blockIdx.x - gr.blk0) * w, cols = gr.njobs * M;
    const int nc = int(min(int64_t(w), cols - c0));
    // this thread's column (of the grid's jobs' M each)
    const int64_t c = min(c0 + (threadIdx.x & (w - 1)), cols - 1);
    const int64_t jb = c / M;
    const Job J = gr.jobs[jb];
    const int mc = rings.maxc[J.r];             // rows mc < i < M - mc hold no ring member: zero
    C *f = out + J.out_off + (c - jb * M);
    auto load = [&](int, int i) { return (i <= mc || i >= M - mc) ? f[i * M] : cmk<C>(0.0, 0.0); };
    fft_any<C, true, false, true>(M, nc, gr.lgw, P, a, b, tw.t, load, [&](int, int k, const C &v) { f[k * M] = v; });
}

// ---------------------------------------------------------------------------
// Step II (Eq. fftbs): S(r1, r2, r3) = sum over the M x M grid of
// D(r1, n1) D(r2, n2) D(r3, n3), for every combination of a plane pair.
//
// One block per unit: an x chunk of one group (plane pair and grid) and up
// to NW of its tiles, one tile per warp.  The block stages the unit's rings
// of the three planes for TX grid points at a time in shared memory
// ([slot][x], x contiguous), double-buffered with cp.async.  The lanes of a
// warp take consecutive grid points, so every shared-memory load is
// conflict free.  Per point a lane forms the 8 row products
// P_i = D(r1_i, n1) D(r2_i, n2) once and accumulates Re(P_i D(w0 + j, n3))
// for the 8 r3 of the tile's window: 64 sums in registers over the whole
// chunk, reduced across the warp at the end.  Negative planes enter through
// D(r, -n) = conj D(r, n) as sign factors.  Blocks of 4, 8 and 16 warps
// (unit classes) let small units share an SM.
//
// A tile's 64 entries are a quarter to a half combinations (64^3 23%, 256^3
// 54%): FP32 computes them all (a test costs as much as the two FMAs), FP64,
// bound by its pipe of two lanes a clock and SM, tests each entry (the mask is
// uniform over the warp) and leaves the others out.
//
// FP32 is bound by instruction issue (66-71% of the slots), of which the FMAs of a
// tile are a third: so the staging and the addresses are kept lean (stages of a
// constant 64 or 128 points, slot addresses in registers, one piece column per
// thread, signs on sign bits), and the warps that a unit's tiles leave over take
// turns at the points (128^3: 61% of the warp slots had a tile).  Without these
// 128^3 took 6.3 ms and 96^3 x 2 3.6 ms, with them 3.8 and 2.1 (128^3 with the
// store's base address in registers 3.5); FP64 at 64^3 4.3 and 2.2 ms, most of it
// from the entries left out.
// (The asm statements below clobber memory at the barriers' sides only, so
// the loads of a stage may move among each other.)
template <typename C> __device__ __forceinline__ C lds_complex(uint32_t a)
{
    C v;
    if constexpr (sizeof(C) == 8) asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(a));
    else asm volatile("ld.shared.v2.f64 {%0, %1}, [%2];" : "=d"(v.x), "=d"(v.y) : "r"(a));
    return v;
}
// x, with the other sign where bit = 0x80000000
__device__ __forceinline__ float flip_sign(float x, uint32_t bit) { return __uint_as_float(__float_as_uint(x) ^ bit); }
__device__ __forceinline__ double flip_sign(double x, uint32_t bit)
{
    return __hiloint2double(__double2hiint(x) ^ int(bit), __double2loint(x));
}

template <typename R, int NW>
__global__ void __launch_bounds__(32 * NW, (sizeof(R) == 8 ? 8 : 16) / NW)
k_step2(StepIIArgs args, int64_t unit0, const typename Cx<R>::T *dstore, int smem_bytes)
{
    grid_begin();
    dstore = field_ptr(dstore, args.fs);
    // an address of its own to the compiler, which otherwise works out that of every
    // copy from the kernel's arguments anew (128^3: 3.79 -> 3.49 ms)
    asm volatile("" : "+l"(dstore));
    args.partials = field_ptr(args.partials, args.fs);
    using C = typename Cx<R>::T;
    constexpr int NT = 32 * NW;
    constexpr bool SKIP = sizeof(R) == 8;     // see above
    constexpr int PER16 = 16 / sizeof(C);     // complex values per 16-byte copy
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const Unit U = args.units[unit0 + blockIdx.x];
    const Group G = args.groups[U.group];
    const int lev = G.lev;
    const int64_t M2 = int64_t(G.M) * G.M;
    const int64_t x0 = int64_t(U.chunk) * args.x_chunk;
    const int64_t x1 = min(M2, x0 + args.x_chunk);
    const int nq0 = U.rhi[0] - U.rlo[0] + 1, nq1 = U.rhi[1] - U.rlo[1] + 1, nq2 = U.rhi[2] - U.rlo[2] + 1;
    const int ns = nq0 + nq1 + nq2;

    int64_t *offs = reinterpret_cast<int64_t *>(smem_raw);
    const size_t off = (size_t(ns) * sizeof(int64_t) + 127) & ~size_t(127);
    C *buf = reinterpret_cast<C *>(smem_raw + off);
    // grid points per stage: 64 (the plan saw to it that they fit), 128 where
    // they do; constants, so that the slots' addresses are a base and an immediate
    const bool wide = off + 2 * size_t(ns) * 128 * sizeof(C) <= size_t(smem_bytes);

    for (int s = threadIdx.x; s < ns; s += NT) {
        const int q = s < nq0 ? 0 : (s < nq0 + nq1 ? 1 : 2);
        const int r = U.rlo[q] + s - (q == 0 ? 0 : (q == 1 ? nq0 : nq0 + nq1));
        const int n = q == 0 ? G.n1 : (q == 1 ? G.n2 : G.n3);
        offs[s] = r < args.nr ? args.doff[(size_t(lev) * args.nz1 + (n < 0 ? -n : n)) * kMaxRings + r] : -1;
    }
    __syncthreads();

    // signs of conj(D) for negative planes (n1 >= 0): with D2 -> (b.x, g2 b.y),
    // D3 -> (c.x, g3 c.y):  Re(P D3) = Pr c.x + Pi (-g3 c.y); applied to the
    // fields' sign bits
    const uint32_t flip2 = G.n2 < 0 ? 0x80000000u : 0u, flip3 = G.n3 < 0 ? 0u : 0x80000000u;

    // tile of the warp, and which of the tile's warps it is: a unit with fewer
    // tiles than warps gives each tile nw2 of them, which take turns at 32 points
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int ntile2 = 1;
    while (ntile2 < U.nt) ntile2 *= 2;
    const int nw2 = NW / ntile2, tile = warp & (ntile2 - 1), turn = warp / ntile2;
    const bool active = tile < U.nt;
    Tile T;
    if (active) T = args.tiles[U.t0 + tile];
    R a[kTileRows * kTileCols];
#pragma unroll
    for (int i = 0; i < kTileRows * kTileCols; ++i) a[i] = R(0);

    // the stage loop, TX points a stage
    auto run = [&](auto txc) {
        constexpr int TX = decltype(txc)::value;
        constexpr int per = TX / PER16;               // 16-byte pieces per slot row
        static_assert(NT % per == 0, "a thread copies one piece of its slots");
        const uint32_t buf0 = uint32_t(__cvta_generic_to_shared(buf)), stage_bytes = uint32_t(ns * TX * sizeof(C));
        const int nstage = int((x1 - x0 + TX - 1) / TX);
        auto issue = [&](int st) {
            const uint32_t dst = buf0 + (st & 1) * stage_bytes;
            const C *src = dstore + x0 + int64_t(st) * TX;
            const int nx = int(min(int64_t(TX), x1 - x0 - int64_t(st) * TX));
            // the thread's piece of every (NT / per)-th slot
            const int c = int(threadIdx.x % per) * PER16;
            uint32_t d = dst + 16 * threadIdx.x;
            for (int s = threadIdx.x / per; s < ns; s += NT / per, d += 16 * NT) {
                const int64_t o = offs[s];
                if (o >= 0 && c < nx)
                    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(src + c + o));
                else
                    asm volatile("st.shared.v4.b32 [%0], {%1, %1, %1, %1};\n" ::"r"(d), "r"(0) : "memory");
            }
            asm volatile("cp.async.commit_group;\n" ::: "memory");
        };
        // shared-memory addresses of the tile's slots in stage buffer 0 (this
        // lane's point), kept: the compiler would rebuild them from their bytes
        // for every stage
        uint32_t a1[kTileRows], a2[kTileRows], a3 = 0;
        if (active) {
            a3 = buf0 + uint32_t((T.s3 * TX + lane) * sizeof(C));
#pragma unroll
            for (int i = 0; i < kTileRows; ++i) {
                a1[i] = buf0 + uint32_t((T.s1[i] * TX + lane) * sizeof(C));
                a2[i] = buf0 + uint32_t((T.s2[i] * TX + lane) * sizeof(C));
                asm volatile("" : "+r"(a1[i]), "+r"(a2[i]));
            }
        }
        issue(0);
        for (int st = 0; st < nstage; ++st) {
            if (st + 1 < nstage) {
                issue(st + 1);
                asm volatile("cp.async.wait_group 1;\n" ::: "memory");
            } else {
                asm volatile("cp.async.wait_group 0;\n" ::: "memory");
            }
            __syncthreads();
            const int nx = int(min(int64_t(TX), x1 - (x0 + int64_t(st) * TX)));
            if (active) {
#pragma unroll 1
                for (int x = 32 * turn; x < nx; x += 32 * nw2) {      // 32 points, one per lane
                    const uint32_t at = (st & 1) * stage_bytes + uint32_t(x * sizeof(C));
                    C w[kTileCols];
#pragma unroll
                    for (int j = 0; j < kTileCols; ++j) {
                        w[j] = lds_complex<C>(a3 + at + uint32_t(j * TX * sizeof(C)));
                        w[j].y = flip_sign(w[j].y, flip3);
                    }
#pragma unroll
                    for (int i = 0; i < kTileRows; ++i) {
                        // FP64: entries that are no combination are left out
                        const uint32_t live = SKIP ? (T.mask[i / 4] >> (8 * (i % 4))) & 255u : 255u;
                        if (SKIP && live == 0) continue;
                        const C u = lds_complex<C>(a1[i] + at);
                        const C v = lds_complex<C>(a2[i] + at);
                        const R vy = flip_sign(v.y, flip2);
                        const R pr = fma(u.x, v.x, -(u.y * vy));
                        const R pi = fma(u.x, vy, u.y * v.x);
#pragma unroll
                        for (int j = 0; j < kTileCols; ++j) {
                            if (SKIP && !((live >> j) & 1u)) continue;
                            R &acc = a[i * kTileCols + j];
                            acc = fma(pr, w[j].x, acc);
                            acc = fma(pi, w[j].y, acc);
                        }
                    }
                }
            }
            __syncthreads();
        }
    };
    if (wide) run(std::integral_constant<int, 128>{});
    else run(std::integral_constant<int, 64>{});
    // butterfly reduction across the warp: after the step with offset o the
    // lane keeps the half of its sums selected by (lane & o); at the end lane
    // l holds the sums of tile entries 2 l and 2 l + 1
#pragma unroll
    for (int o = 16, n = kTileRows * kTileCols / 2; o >= 1; o >>= 1, n >>= 1) {
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int k = 0; k < kTileRows * kTileCols / 2; ++k) {
            if (k >= n) break;
            const R keep = up ? a[k + n] : a[k];
            const R give = up ? a[k] : a[k + n];
            a[k] = keep + __shfl_xor_sync(0xffffffffu, give, o);
        }
    }
    // the warps of a tile: their sums in order, in FP64 (the stages' buffers
    // are free after the loop's last barrier)
    double sum[2] = {double(a[0]), double(a[1])};
    if (nw2 > 1) {
        double *sh = reinterpret_cast<double *>(buf);
        if (turn > 0) {
            sh[64 * warp + 2 * lane] = sum[0];
            sh[64 * warp + 2 * lane + 1] = sum[1];
        }
        __syncthreads();
        if (turn > 0) return;
        for (int g = 1; g < nw2; ++g)
#pragma unroll
            for (int k = 0; k < 2; ++k) sum[k] += sh[64 * (warp + g * ntile2) + 2 * lane + k];
    }
    if (!active) return;
    double *dst = args.partials + G.part0 + int64_t(U.chunk) * G.ncombo;
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const int idx = 2 * lane + k;
        if ((T.mask[idx >> 5] >> (idx & 31)) & 1u) dst[T.coff[idx / kTileCols] + (idx % kTileCols)] = sum[k];
    }
}

template <typename A>
__global__ void __launch_bounds__(256)
k_reduce(const Group *__restrict__ groups, int64_t ngroups, const double *partials, int ng,
         double *__restrict__ S, int64_t fs)
{
    grid_begin();
    partials = field_ptr(partials, fs);
    S = field_ptr(S, fs);
    // one warp per group: groups hold 14 (64^3) to 140 (512^3) combinations
    const int64_t g = int64_t(blockIdx.x) * 8 + (threadIdx.x >> 5);
    if (g >= ngroups) return;
    const Group G = groups[g];
    const double f = double(ng) / double(G.M);
    const A scale = A(f * f);
    for (int j = threadIdx.x & 31; j < G.ncombo; j += 32) {
        const double *p = partials + G.part0 + j;
        A s = A(0);
#pragma unroll 4
        for (int k = 0; k < G.nchunk; ++k) s += A(p[int64_t(k) * G.ncombo]);
        S[G.c0 + j] = double(s * scale);
    }
}

// Y_lm normalisation sqrt((2l+1)/(4 pi) (l-m)!/(l+m)!), and the prefactor
// sqrt((2l+1)/(4 pi)) of Eq. bs_lm2_1, set by set_ylm_constants.
__constant__ double c_nlm[9][9];
__constant__ double c_pref[9];
// Legendre recurrence ratios (2l+1)/(l+1-m) and (l+m)/(l+1-m), l, m <= 8
__constant__ double c_rec[2][9][9];
// the same in FP32, so that the FP32 weights take them as operands
__constant__ float c_nlm_f[9][9];
__constant__ float c_rec_f[2][9][9];
template <typename Y> __device__ __forceinline__ Y nlm_of(int l, int m)
{
    if constexpr (sizeof(Y) == 4) return c_nlm_f[l][m]; else return Y(c_nlm[l][m]);
}
template <typename Y> __device__ __forceinline__ Y rec_of(int k, int l, int m)
{
    if constexpr (sizeof(Y) == 4) return c_rec_f[k][l][m]; else return Y(c_rec[k][l][m]);
}

__global__ void __launch_bounds__(256)
k_records_f(const Record *__restrict__ rec, RecordF *__restrict__ recf, int64_t n)
{
    for (int64_t k = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; k < n; k += int64_t(gridDim.x) * blockDim.x) {
        const Record r = rec[k];
        recf[k] = RecordF{r.s_index, r.flags, float(r.pz), float(r.cphi)};
    }
}

// w 2^-896, exactly, for a normal (or zero) w: the float's sign, exponent
// field and mantissa moved to a double's, three integer operations.
__device__ __forceinline__ double widen_scaled(float w)
{
    const int u = __float_as_int(w);
    return __hiloint2double((u >> 3) & int(0x8FFFFFFFu), u << 29);
}

// W: type of the sums over records; Y: type the Y_lm of each record are
// computed in (FP32 for the FP32-transform paths, whose tolerance is 1e-4;
// FP64 for the FP64 path and the plan-time denominators).  The moments
// written are lm_lo .. (LMAX/2 + 1)^2 - 1 (even l from l_lo = 2 sqrt(lm_lo)),
// nlm_out = that count per bin, for out and den alike.
//
// One warp per chunk.  With FP32 weights and FP64 sums the slow FP64 pipe (two
// lanes a clock and SM) bounds it, so a record costs it one FMA per moment and
// two products: the weight is widened in the integer pipe (as w 2^-896; 2^448 goes
// to the value and 2^448 to the sum, so neither can overflow below 1e173) where
// a conversion instruction took as long as the FMA, and the orientation is read
// as FP32 and the recurrences' constants are FP32 operands in constant memory.
// The next record's value and the one after's record are loaded ahead.  With
// conversions of all of these, and one thread per bin in k_epi_fin: 512^3 (1.1e8
// records) 7.5 -> 3.2 ms, 256^3 1.21 -> 0.52 ms; 64^3, mostly for its shorter chunks
// (bin_chunk_len), 184 -> 26 us.
template <typename W, typename Y, int LMAX>
__device__ __forceinline__ void
epi_part(int mode, const Record *__restrict__ rec, const RecordF *__restrict__ recf,
         const int64_t *__restrict__ chunk_lo, const int64_t *__restrict__ chunk_hi, int64_t nchunks, int64_t ch,
         const double *value, double *__restrict__ partial, int64_t fs_in, int64_t fs_part)
{
    constexpr bool F32 = sizeof(Y) == 4;                  // FP32 weights (mode 0 only)
    constexpr bool WIDEN = F32 && sizeof(W) == 8;
    using Rec = typename std::conditional<F32, RecordF, Record>::type;
    const Rec *recs;
    if constexpr (F32) recs = recf; else recs = rec;
    value = field_ptr(value, fs_in);
    partial = field_ptr(partial, fs_part);
    constexpr int NLM = (LMAX / 2 + 1) * (LMAX / 2 + 1);
    const int lane = threadIdx.x & 31;
    if (ch >= nchunks) return;   // whole warps leave together
    W acc[NLM];
#pragma unroll
    for (int i = 0; i < NLM; ++i) acc[i] = W(0);
    const int64_t k1 = chunk_hi[ch];
    int64_t k = chunk_lo[ch] + lane;
    auto load_value = [&](const Rec &r, int64_t at) { return mode == 0 ? value[r.s_index] : value[at]; };
    Rec R{}, Rn{};
    double val = 0.0;
    if (k < k1) {
        R = recs[k];
        if (k + 32 < k1) Rn = recs[k + 32];
        val = load_value(R, k);
    }
    for (; k < k1; k += 32) {
        double val_n = 0.0;
        Rec Rnn{};
        if (k + 64 < k1) Rnn = recs[k + 64];
        if (k + 32 < k1) val_n = load_value(Rn, k + 32);
        const Y x = Y(R.pz), c = Y(R.cphi);
        const W mult = (R.flags & 1) ? W(1) : W(2);
        const W v = W(val) * (WIDEN ? W(0x1p448) * mult : mult);
        const bool deg = (R.flags & 2) != 0;
        const Y s = sqrt(max(Y(0), Y(1) - x * x));
        Y pmm = Y(1), tm1 = Y(1), tm2 = Y(1);   // P_m^m; cos(m phi), cos((m-1) phi)
#pragma unroll
        for (int m = 0; m <= LMAX; ++m) {
            Y tm;
            if (m == 0) tm = Y(1);
            else if (m == 1) tm = c;
            else tm = Y(2) * c * tm1 - tm2;
            if (m > 0) pmm *= -Y(2 * m - 1) * s;
            Y plm1 = Y(0), pl = pmm;                 // P_{l-1}^m, P_l^m at l = m
#pragma unroll
            for (int l = m; l <= LMAX; ++l) {
                if ((l & 1) == 0) {
                    const Y y = nlm_of<Y>(l, m) * pl;
                    const int idx = (l >> 1) * (l >> 1) + m;
                    if (F32 || mode == 0) {
                        const Y w = deg ? (m == 0 ? y : Y(0)) : y * tm;
                        if constexpr (WIDEN) acc[idx] = fma(widen_scaled(w), v, acc[idx]);
                        else acc[idx] += W(w) * v;
                    } else {
                        acc[idx] += W(y) * W(y) * v;
                    }
                }
                // P_{l+1}^m = ((2l+1) x P_l^m - (l+m) P_{l-1}^m) / (l+1-m), with
                // the two ratios from constant memory (no division per record)
                const Y pn = rec_of<Y>(0, l, m) * x * pl - rec_of<Y>(1, l, m) * plm1;
                plm1 = pl;
                pl = pn;
            }
            tm2 = tm1;
            tm1 = tm;
        }
        R = Rn;
        Rn = Rnn;
        val = val_n;
    }
    // Sums across the warp: while more than one sum is left, the step of
    // distance o gives half of them away (the lanes with bit o keep the upper
    // half), so NLM sums cost about NLM exchanges and not 5 NLM; then plain
    // halving steps.  At the end lane l holds sum (l's bits from the top).
    constexpr int P2 = NLM <= 1 ? 1 : (NLM <= 4 ? 4 : (NLM <= 16 ? 16 : 32));
    W red[P2];
#pragma unroll
    for (int i = 0; i < P2; ++i) red[i] = i < NLM ? acc[i] : W(0);
    int idx = 0;
#pragma unroll
    for (int o = 16, n = P2; o >= 1; o >>= 1) {
        if (n > 1) {
            n >>= 1;
            const bool up = (lane & o) != 0;
#pragma unroll
            for (int k = 0; k < P2 / 2; ++k) {
                if (k >= n) break;
                const W keep = up ? red[k + n] : red[k];
                const W give = up ? red[k] : red[k + n];
                red[k] = keep + __shfl_xor_sync(0xffffffffu, give, o);
            }
            if (up) idx += n;
        } else {
            red[0] += __shfl_xor_sync(0xffffffffu, red[0], o);
        }
    }
    if ((lane & (32 / P2 - 1)) == 0 && idx < NLM) partial[ch * NLM + idx] = double(red[0]) * (WIDEN ? 0x1p448 : 1.0);
}

template <typename W, typename Y, int LMAX>
__global__ void __launch_bounds__(256)
k_epi_part(int mode, const Record *__restrict__ rec, const RecordF *__restrict__ recf,
           const int64_t *__restrict__ chunk_lo, const int64_t *__restrict__ chunk_hi, int64_t nchunks,
           const double *value, double *__restrict__ partial, int64_t fs_in, int64_t fs_part)
{
    grid_begin();
    epi_part<W, Y, LMAX>(mode, rec, recf, chunk_lo, chunk_hi, nchunks, (int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5,
                         value, partial, fs_in, fs_part);
}

// The view that block blockIdx.x of a launch over all views works on
template <bool FIN> __device__ __forceinline__ const EpiView &view_of_block(const EpiViews &ev)
{
    int i = 0;
    while (i + 1 < ev.n && blockIdx.x >= (FIN ? ev.v[i + 1].fin0 : ev.v[i + 1].blk0)) ++i;
    return ev.v[i];
}

// k_epi_part (mode 0) for several views in one launch
template <typename W, typename Y>
__global__ void __launch_bounds__(256)
k_epi_part_views(const __grid_constant__ EpiViews ev, const double *value, int64_t fs_in)
{
    grid_begin();
    const EpiView &v = view_of_block<false>(ev);
    const int64_t ch = int64_t(blockIdx.x - v.blk0) * 8 + (threadIdx.x >> 5);
    auto run = [&](auto lmax) {
        epi_part<W, Y, decltype(lmax)::value>(0, ev.rec, ev.recf, v.chunk_lo, v.chunk_hi, v.nchunks, ch, value, v.partial,
                                              fs_in, fs_in);
    };
    switch (v.l_hi) {
    case 0: run(std::integral_constant<int, 0>{}); break;
    case 2: run(std::integral_constant<int, 2>{}); break;
    case 4: run(std::integral_constant<int, 4>{}); break;
    case 6: run(std::integral_constant<int, 6>{}); break;
    default: run(std::integral_constant<int, 8>{}); break;
    }
}

// The bins b0 .. b1 - 1 of a block (see fin_bins_per_block): their chunks' partial sums
// added up, then (mode 0) the ratio of Eq. bs_lm2_1 or (mode 1) the sum itself.  The sum
// of a moment: kFinSplit running sums take the bin's chunks in turn, and are added in
// order (the same for every LMAX, so that a moment does not depend on the others binned
// with it).  They take kFinSplit threads per moment, so that none walks many chunks
// alone (64^3, up to 80 of them: 14 us); of several bins, those of at most kFinSplit
// chunks take one thread per moment, which comes to the same.  A block per bin
// throughout was bound by the launch of empty blocks where bins are many, one thread per
// bin by its strided stores (64^3, 3e6 bins of 4 moments, the binning: 3.1 ms and 0.52;
// so 0.24 ms).
constexpr int kFinSplit = 8;
template <int LMAX> constexpr int fin_threads()
{
    const int n = (LMAX / 2 + 1) * (LMAX / 2 + 1);
    return n <= 4 ? 32 : (n <= 16 ? 128 : 256);
}
template <int LMAX>
__device__ __forceinline__ void
epi_fin(int mode, const int64_t *__restrict__ bin_chunk, const double *partial,
        const double *__restrict__ den, double norm, double *__restrict__ out, int64_t fs_part, int64_t fs_out,
        int lm_lo, int nlm_out, int64_t b0, int64_t b1, double *red)
{
    partial = field_ptr(partial, fs_part);
    out = field_ptr(out, fs_out);
    constexpr int NLM = (LMAX / 2 + 1) * (LMAX / 2 + 1);
    constexpr int P2 = fin_threads<LMAX>() / kFinSplit;     // at least NLM
    auto store = [&](int64_t b, int i, double v) {
        const int64_t o = b * nlm_out + (i - lm_lo);
        if (mode == 0) {
            const double d = den[o];
            int l = 0;
            while ((l / 2 + 1) * (l / 2 + 1) <= i) l += 2;
            out[o] = d > 0.0 ? c_pref[l] * v * norm / d : __longlong_as_double(0x7ff8000000000000LL);
        } else {
            out[o] = v;
        }
    };
    const bool several = b1 - b0 > 1;
    const int64_t total = several ? (b1 - b0) * nlm_out : 0;
    bool more = !several;                                   // a bin of more chunks seen
    for (int64_t t = threadIdx.x; t < total; t += blockDim.x) {
        const int64_t q = t / nlm_out, b = b0 + q, c0 = bin_chunk[b], c1 = bin_chunk[b + 1];
        if (c1 - c0 > kFinSplit) {
            more = true;
            continue;
        }
        const int i = lm_lo + int(t - q * nlm_out);
        double v = 0.0;
        for (int64_t ch = c0; ch < c1; ++ch) v += partial[ch * NLM + i];
        store(b, i, v);
    }
    if (several && !__syncthreads_or(more)) return;
    const int i = threadIdx.x % P2, sub = threadIdx.x / P2;
    for (int64_t b = b0; b < b1; ++b) {                     // (the same bins for every thread)
        const int64_t c0 = bin_chunk[b], c1 = bin_chunk[b + 1];
        if (several && c1 - c0 <= kFinSplit) continue;
        double v = 0.0;
        if (sub < kFinSplit) {                              // (a launch may have threads to spare)
            if (i < NLM)
#pragma unroll 4
                for (int64_t ch = c0 + sub; ch < c1; ch += kFinSplit) v += partial[ch * NLM + i];
            red[threadIdx.x] = v;
        }
        __syncthreads();
        if (sub == 0 && i >= lm_lo && i < NLM) {
            for (int k = 1; k < kFinSplit; ++k) v += red[k * P2 + i];
            store(b, i, v);
        }
        if (several) __syncthreads();
    }
}

template <int LMAX>
__global__ void __launch_bounds__(256)
k_epi_fin(int mode, const int64_t *__restrict__ bin_chunk, int64_t nbins, int64_t per, const double *partial,
          const double *__restrict__ den, double norm, double *__restrict__ out, int64_t fs_part, int64_t fs_out,
          int lm_lo, int nlm_out)
{
    __shared__ double red[fin_threads<LMAX>()];
    grid_begin();
    const int64_t b0 = int64_t(blockIdx.x) * per;
    epi_fin<LMAX>(mode, bin_chunk, partial, den, norm, out, fs_part, fs_out, lm_lo, nlm_out, b0, min(nbins, b0 + per), red);
}

// k_epi_fin (mode 0) for several views in one launch
__global__ void __launch_bounds__(256)
k_epi_fin_views(const __grid_constant__ EpiViews ev, double norm, int64_t fs_part, int64_t fs_out)
{
    __shared__ double red[256];
    grid_begin();
    const EpiView &v = view_of_block<true>(ev);
    const int64_t b0 = int64_t(blockIdx.x - v.fin0) * ev.per, b1 = min(v.nbins, b0 + ev.per);
    auto run = [&](auto lmax) {
        epi_fin<decltype(lmax)::value>(0, v.bin_chunk, v.partial, v.den, norm, v.out, fs_part, fs_out, v.lm_lo, v.nlm, b0, b1, red);
    };
    switch (v.l_hi) {
    case 0: run(std::integral_constant<int, 0>{}); break;
    case 2: run(std::integral_constant<int, 2>{}); break;
    case 4: run(std::integral_constant<int, 4>{}); break;
    case 6: run(std::integral_constant<int, 6>{}); break;
    default: run(std::integral_constant<int, 8>{}); break;
    }
}

// Running statistics of estimates over fields: Welford's update (mean and
// sum of squared deviations, FP64) of element i with B[f][i], f < nf, in
// field order; non-finite values (empty bins) are skipped.
__global__ void __launch_bounds__(256)
k_stats_update(const double *__restrict__ B, int nf, int64_t n, int64_t *__restrict__ count,
               double *__restrict__ mean, double *__restrict__ m2)
{
    const int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if (i >= n) return;
    int64_t c = count[i];
    double m = mean[i], s = m2[i];
    for (int f = 0; f < nf; ++f) {
        const double x = B[int64_t(f) * n + i];
        if (!isfinite(x)) continue;
        ++c;
        const double d = x - m;
        m += d / double(c);
        s += d * (x - m);
    }
    count[i] = c;
    mean[i] = m;
    m2[i] = s;
}

__global__ void __launch_bounds__(256)
k_ntri(const double2 *__restrict__ I, const int64_t *__restrict__ ioff, const int32_t *__restrict__ tri,
       GridArg grids, double *__restrict__ raw)
{
    __shared__ double red[8];
    const int r1 = tri[4 * blockIdx.x], r2 = tri[4 * blockIdx.x + 1], r3 = tri[4 * blockIdx.x + 2];
    const int lev = tri[4 * blockIdx.x + 3];
    const int64_t M2 = int64_t(grids.M[lev]) * grids.M[lev];
    const double2 *a = I + ioff[lev * kMaxRings + r1];
    const double2 *b = I + ioff[lev * kMaxRings + r2];
    const double2 *c = I + ioff[lev * kMaxRings + r3];
    double s = 0;
    for (int64_t y = threadIdx.x; y < M2; y += blockDim.x) {
        const double2 p = cmul(cmul(a[y], b[y]), c[y]);
        s += p.x;
    }
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0;
        for (int w = 0; w < int(blockDim.x >> 5); ++w) t += red[w];
        raw[blockIdx.x] = t / double(M2);
    }
}

}  // namespace

size_t fft_rows_per_block(int M, size_t elem, size_t bytes)
{
    size_t rt = bytes / (size_t(M) * elem);
    if (rt < 1) rt = 1;
    if (rt > 256) rt = 256;
    return rt;
}

template <typename R>
cudaError_t launch_fft_z_real(const R *in, typename Cx<R>::T *out, int ng, int64_t rows, int nkeep,
                              const Twiddles<typename Cx<R>::T> &tw, const Batch &fb, cudaStream_t s, int rt, int *clear)
{
    using C = typename Cx<R>::T;
    if (rt <= 0) rt = int(fft_rows_per_block(ng, sizeof(C)));
    rt = std::max(1, int(std::min<int64_t>(rt, rows / 2)));        // pairs of rows
    const size_t smem = size_t(2) * rt * fft_stride<C>(ng, rt) * sizeof(C);
    const int64_t nblk = (rows / 2 + rt - 1) / rt;
    k_fft_z_real<R><<<dim3(unsigned(nblk), fb.nf), 256, smem, s>>>(in, out, ng, rows, nkeep, rt, tw, fb.fs_in,
                                                                   fb.fs_out, clear);
    return cudaGetLastError();
}

template <typename R>
cudaError_t launch_fft_rows_T(const typename Cx<R>::T *in, typename Cx<R>::T *out, int M, int nrow,
                              int64_t nb, R scale, bool zero_dc,
                              const Twiddles<typename Cx<R>::T> &tw, const Batch &fb, cudaStream_t s, int rt)
{
    using C = typename Cx<R>::T;
    if (rt <= 0) rt = int(fft_rows_per_block(M, sizeof(C)));
    rt = std::min(rt, nrow);
    const size_t smem = size_t(2) * rt * fft_stride<C>(M, rt) * sizeof(C);
    const int ntile = (nrow + rt - 1) / rt;
    const int64_t nblk = nb * ntile;
    if (nblk == 0) return cudaSuccess;
    return launch_next(k_fft_rows_T<R>, dim3(unsigned(nblk), fb.nf), 256, smem, s, in, out, M, nrow, ntile, scale,
                       zero_dc ? 1 : 0, rt, tw, fb.fs_in);
}

template <typename R>
cudaError_t launch_fft_z_back(const typename Cx<R>::T *in, R *out, int M, int nkeep, int64_t nf,
                              const Twiddles<typename Cx<R>::T> &tw, cudaStream_t s)
{
    using C = typename Cx<R>::T;
    const int lgw = sizeof(R) == 4 ? 4 : 3, w = 1 << lgw;      // 256 bytes of a plane per load
    const size_t smem = size_t(2) * w * fft_stride<C>(M, w) * sizeof(C);
    if (M % 2 || 2 * nkeep > M + 1 || smem > 48 * 1024) return cudaErrorInvalidValue;
    const int ntile = (M * M / 2 + w - 1) / w;
    const int64_t nblk = nf * ntile;
    if (nblk > 0x7FFFFFFF) return cudaErrorInvalidValue;
    if (nblk == 0) return cudaSuccess;
    return launch_next(k_fft_z_back<R>, unsigned(nblk), 256, smem, s, in, out, M, nkeep, ntile, lgw, tw);
}

// Shared-memory buffers of a Step-I transform of length M: its stages hand the
// data on between the first, from global memory, and the last, to it.
static int fft_buffers(int M)
{
    const int lg = __builtin_ctz(unsigned(M)), odd = M >> lg;
    const int stages = odd > 1 ? 1 + (lg + 2) / 3 : (lg + 2) / 3;
    return stages > 2 ? 2 : 1;
}

// The blocks of a Step-I launch over several grids, and its shared memory.
template <typename C> static cudaError_t step_blocks(StepGrids &gs, bool cols, unsigned *nblk, size_t *smem)
{
    int64_t blk = 0;
    *smem = 0;
    for (int i = 0; i < gs.n; ++i) {
        StepGrid &g = gs.g[i];
        if (g.rt <= 0) g.rt = cols ? 8 : int(fft_rows_per_block(g.M, sizeof(C)));
        g.rt = std::min(g.rt, g.M);
        if (cols) {                              // strips of a power of two
            g.lgw = 0;
            while ((2 << g.lgw) <= g.rt) ++g.lgw;
            g.rt = 1 << g.lgw;
        }
        g.ntile = (g.M + g.rt - 1) / g.rt;
        g.blk0 = unsigned(blk);
        blk += cols ? (g.njobs * g.M + g.rt - 1) / g.rt : g.njobs * g.ntile;
        *smem = std::max(*smem, size_t(fft_buffers(g.M)) * g.rt * fft_stride<C>(g.M, cols ? g.rt : gather_across(g.M)) * sizeof(C));
    }
    if (blk > 0x7FFFFFFF || *smem > 227 * 1024) return cudaErrorInvalidValue;
    *nblk = unsigned(blk);
    return cudaSuccess;
}

// Threads of a Step-I block: 128 up to M = 256, whose tiles give more threads
// little to do in a stage and whose blocks are then finer to place (all grids of
// 64^3 63 -> 49 us with the columns of several jobs per block, of 128^3 x 16 5.0 ->
// 4.0 ms); 256 above (at 512^3, 128 for all took 29.9 ms, 256 27.0).
static unsigned step_threads(const StepGrids &gs)
{
    int m = 0;
    for (int i = 0; i < gs.n; ++i) m = std::max(m, gs.g[i].M);
    return m <= 256 ? 128 : 256;
}

template <typename R>
cudaError_t launch_ring_gather(const typename Cx<R>::T *planes, int ng, const RingArg &rings, StepGrids gs, bool unit,
                               typename Cx<R>::T *out, const Twiddles<typename Cx<R>::T> &tw, const Batch &fb,
                               cudaStream_t s, const float *scale)
{
    unsigned nblk;
    size_t smem;
    if (cudaError_t e = step_blocks<typename Cx<R>::T>(gs, false, &nblk, &smem); e != cudaSuccess) return e;
    if (nblk == 0) return cudaSuccess;
    const dim3 grid(nblk, fb.nf);
    const unsigned threads = step_threads(gs);
    return launch_next(unit ? k_ring_gather<R, true> : k_ring_gather<R, false>, grid, threads, smem, s, planes, ng, rings, gs,
                       out, tw, scale, fb.fs_in);
}

cudaError_t launch_ring_scale(const float2 *planes, int ng, int nz1, const RingArg &rings, float *scale,
                              const Batch &fb, cudaStream_t s)
{
    return launch_next(k_ring_scale, dim3(unsigned(nz1 * rings.nr), fb.nf), 256, 0, s, planes, ng, rings, scale, fb.fs_in);
}

template <typename R>
cudaError_t launch_fft_cols(typename Cx<R>::T *out, StepGrids gs, const RingArg &rings,
                            const Twiddles<typename Cx<R>::T> &tw, const Batch &fb, cudaStream_t s)
{
    unsigned nblk;
    size_t smem;
    if (cudaError_t e = step_blocks<typename Cx<R>::T>(gs, true, &nblk, &smem); e != cudaSuccess) return e;
    if (nblk == 0) return cudaSuccess;
    return launch_next(k_fft_cols<R>, dim3(nblk, fb.nf), step_threads(gs), smem, s, out, gs, rings, tw, fb.fs_in);
}

template <typename R, int NW>
cudaError_t launch_step2_class(const StepIIArgs &a, const typename Cx<R>::T *dstore, int64_t u0, int64_t n,
                               size_t smem, int nf, cudaStream_t s)
{
    if (n == 0) return cudaSuccess;
    return launch_next(k_step2<R, NW>, dim3(unsigned(n), nf), 32 * NW, smem, s, a, u0, dstore, int(smem));
}

template <typename R>
cudaError_t launch_step2(const StepIIArgs &a, const typename Cx<R>::T *dstore, const int64_t *lo, const int64_t *hi,
                         int nf, cudaStream_t s)
{
    if constexpr (sizeof(R) == 4) {
        cudaError_t e = launch_step2_class<R, 4>(a, dstore, lo[2], hi[2] - lo[2], kStep2ClassSmem[2], nf, s);
        if (e == cudaSuccess)
            e = launch_step2_class<R, 8>(a, dstore, lo[3], hi[3] - lo[3], kStep2ClassSmem[3], nf, s);
        if (e == cudaSuccess)
            e = launch_step2_class<R, 16>(a, dstore, lo[4], hi[4] - lo[4], kStep2ClassSmem[4], nf, s);
        return e;
    }
    // FP64: register tiles, blocks of at most 8 warps (register file)
    cudaError_t e = launch_step2_class<R, 4>(a, dstore, lo[2], hi[2] - lo[2], kStep2ClassSmem[2], nf, s);
    if (e == cudaSuccess)
        e = launch_step2_class<R, 8>(a, dstore, lo[3], hi[3] - lo[3], kStep2ClassSmem[3], nf, s);
    if (e == cudaSuccess && hi[4] != lo[4]) e = cudaErrorInvalidValue;
    return e;
}

template <typename A>
cudaError_t launch_reduce_partials(const Group *groups, int64_t ngroups, const double *partials, int ng,
                                   double *S, const Batch &fb, cudaStream_t s)
{
    if (ngroups == 0) return cudaSuccess;
    return launch_next(k_reduce<A>, dim3(unsigned((ngroups + 7) / 8), fb.nf), 256, 0, s, groups, ngroups, partials, ng, S, fb.fs_in);
}

template <typename W, typename Y, int LMAX>
cudaError_t epilogue_l(int mode, const EpiArgs &e, const double *value, const double *den, double norm, double *out,
                       const Batch &fb, int lo, int n, cudaStream_t s)
{
    const int64_t per = fin_bins_per_block(e.nbins);
    const dim3 g1(unsigned((e.nchunks * 32 + 255) / 256), fb.nf), g2(unsigned((e.nbins + per - 1) / per), fb.nf);
    cudaError_t st = cudaSuccess;
    if (e.nchunks > 0)
        st = launch_next(k_epi_part<W, Y, LMAX>, g1, 256, 0, s, mode, e.rec, e.recf, e.chunk_lo, e.chunk_hi, e.nchunks, value,
                         e.partial, fb.fs_in, e.fs_part);
    if (st == cudaSuccess)
        st = launch_next(k_epi_fin<LMAX>, g2, per > 1 ? 256 : fin_threads<LMAX>(), 0, s, mode, e.bin_chunk, e.nbins, per, e.partial,
                         den, norm, out, e.fs_part, fb.fs_out, lo, n);
    return st;
}

template <typename W, typename Y>
cudaError_t epilogue_lmax(int mode, const EpiArgs &e, const double *value, int l_lo, int l_hi, const double *den,
                          double norm, double *out, const Batch &fb, cudaStream_t s)
{
    const int lo = (l_lo / 2) * (l_lo / 2), n = (l_hi / 2 + 1) * (l_hi / 2 + 1) - lo;
    switch (l_hi) {
    case 0: return epilogue_l<W, Y, 0>(mode, e, value, den, norm, out, fb, lo, n, s);
    case 2: return epilogue_l<W, Y, 2>(mode, e, value, den, norm, out, fb, lo, n, s);
    case 4: return epilogue_l<W, Y, 4>(mode, e, value, den, norm, out, fb, lo, n, s);
    case 6: return epilogue_l<W, Y, 6>(mode, e, value, den, norm, out, fb, lo, n, s);
    case 8: return epilogue_l<W, Y, 8>(mode, e, value, den, norm, out, fb, lo, n, s);
    default: return cudaErrorInvalidValue;
    }
}

template <typename W>
cudaError_t launch_epilogue(int mode, const EpiArgs &e, const double *value, int l_lo, int l_hi, const double *den,
                            double norm, double *out, const Batch &fb, cudaStream_t s, bool fp32_weights)
{
    if (e.nbins == 0) return cudaSuccess;
    if (l_lo < 0 || l_lo > l_hi || (l_lo & 1)) return cudaErrorInvalidValue;
    if (fp32_weights && mode != 0) return cudaErrorInvalidValue;
    if (fp32_weights) return epilogue_lmax<W, float>(mode, e, value, l_lo, l_hi, den, norm, out, fb, s);
    return epilogue_lmax<W, W>(mode, e, value, l_lo, l_hi, den, norm, out, fb, s);
}

template <typename W>
cudaError_t launch_epilogue_views(EpiViews ev, const double *value, double norm, const Batch &fb, cudaStream_t s,
                                  bool fp32_weights)
{
    int64_t bins = 0;
    for (int i = 0; i < ev.n; ++i) bins += ev.v[i].nbins;
    ev.per = fin_bins_per_block(bins);
    // (a view has fewer than 2^31 chunks, as a plan has fewer combinations: 5 x 2^28 blocks)
    unsigned blk = 0, fin = 0;
    int threads = ev.per > 1 ? 256 : 32;
    for (int i = 0; i < ev.n; ++i) {
        EpiView &v = ev.v[i];
        if (v.l_hi < 0 || v.l_hi > 8 || (v.l_hi & 1)) return cudaErrorInvalidValue;
        v.blk0 = blk;
        v.fin0 = fin;
        blk += unsigned((v.nchunks + 7) / 8);
        fin += unsigned((v.nbins + ev.per - 1) / ev.per);
        threads = std::max(threads, v.l_hi < 4 ? fin_threads<2>() : (v.l_hi < 8 ? fin_threads<6>() : fin_threads<8>()));
    }
    if (fin == 0) return cudaSuccess;
    if (blk > 0) {
        const cudaError_t e = launch_next(fp32_weights ? k_epi_part_views<W, float> : k_epi_part_views<W, W>, dim3(blk, fb.nf),
                                          256, 0, s, ev, value, fb.fs_in);
        if (e != cudaSuccess) return e;
    }
    return launch_next(k_epi_fin_views, dim3(fin, fb.nf), threads, 0, s, ev, norm, fb.fs_in, fb.fs_out);
}

cudaError_t launch_records_f(const Record *rec, RecordF *recf, int64_t n, cudaStream_t s)
{
    if (n == 0) return cudaSuccess;
    k_records_f<<<unsigned(std::min<int64_t>((n + 255) / 256, 152 * 16)), 256, 0, s>>>(rec, recf, n);
    return cudaGetLastError();
}

// Every kernel that takes more than 48 KB of dynamic shared memory is
// allowed the 227 KB maximum once, up front, so that the launches of an
// estimate are plain stream work (capturable in a CUDA graph).
cudaError_t init_kernel_attributes()
{
    const int mx = 227 * 1024;
    cudaError_t e = cudaSuccess;
    auto set = [&](const void *f) {
        if (e == cudaSuccess) e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, mx);
    };
    set((const void *)k_fft_z_real<float>);
    set((const void *)k_fft_z_real<double>);
    set((const void *)k_fft_rows_T<float>);
    set((const void *)k_fft_rows_T<double>);
    set((const void *)k_fft_cols<float>);
    set((const void *)k_fft_cols<double>);
    set((const void *)k_ring_gather<float, false>);
    set((const void *)k_ring_gather<float, true>);
    set((const void *)k_ring_gather<double, false>);
    set((const void *)k_ring_gather<double, true>);
    set((const void *)k_step2<float, 4>);
    set((const void *)k_step2<float, 8>);
    set((const void *)k_step2<float, 16>);
    set((const void *)k_step2<double, 4>);
    set((const void *)k_step2<double, 8>);
    return e;
}

cudaError_t launch_stats_update(const double *B, int nf, int64_t n, int64_t *count, double *mean, double *m2,
                                cudaStream_t s)
{
    if (n == 0 || nf == 0) return cudaSuccess;
    k_stats_update<<<unsigned((n + 255) / 256), 256, 0, s>>>(B, nf, n, count, mean, m2);
    return cudaGetLastError();
}

cudaError_t launch_ntri(const double2 *ifields, const int64_t *ioff, const int32_t *triples, int64_t ntriples,
                        const GridArg &grids, double *raw, cudaStream_t s)
{
    if (ntriples == 0) return cudaSuccess;
    k_ntri<<<unsigned(ntriples), 256, 0, s>>>(ifields, ioff, triples, grids, raw);
    return cudaGetLastError();
}

cudaError_t set_ylm_constants(const double nlm[9][9], const double pref[9], cudaStream_t s)
{
    double rec[2][9][9] = {};
    for (int l = 0; l <= 8; ++l)
        for (int m = 0; m <= l; ++m) {
            rec[0][l][m] = double(2 * l + 1) / double(l + 1 - m);
            rec[1][l][m] = double(l + m) / double(l + 1 - m);
        }
    cudaError_t e = cudaMemcpyToSymbolAsync(c_nlm, nlm, sizeof(double) * 81, 0, cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) e = cudaMemcpyToSymbolAsync(c_pref, pref, sizeof(double) * 9, 0, cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) e = cudaMemcpyToSymbolAsync(c_rec, rec, sizeof(rec), 0, cudaMemcpyHostToDevice, s);
    float nlm_f[9][9], rec_f[2][9][9];
    for (int l = 0; l < 9; ++l)
        for (int m = 0; m < 9; ++m) {
            nlm_f[l][m] = float(nlm[l][m]);
            for (int k = 0; k < 2; ++k) rec_f[k][l][m] = float(rec[k][l][m]);
        }
    if (e == cudaSuccess) e = cudaMemcpyToSymbolAsync(c_nlm_f, nlm_f, sizeof(nlm_f), 0, cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) e = cudaMemcpyToSymbolAsync(c_rec_f, rec_f, sizeof(rec_f), 0, cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);   // the tables above live on this stack
    return e;
}

// explicit instantiations
template cudaError_t launch_fft_z_real<float>(const float *, float2 *, int, int64_t, int, const Twiddles<float2> &, const Batch &, cudaStream_t, int, int *);
template cudaError_t launch_fft_z_real<double>(const double *, double2 *, int, int64_t, int, const Twiddles<double2> &, const Batch &, cudaStream_t, int, int *);
template cudaError_t launch_fft_rows_T<float>(const float2 *, float2 *, int, int, int64_t, float, bool, const Twiddles<float2> &, const Batch &, cudaStream_t, int);
template cudaError_t launch_fft_rows_T<double>(const double2 *, double2 *, int, int, int64_t, double, bool, const Twiddles<double2> &, const Batch &, cudaStream_t, int);
template cudaError_t launch_fft_z_back<float>(const float2 *, float *, int, int, int64_t, const Twiddles<float2> &, cudaStream_t);
template cudaError_t launch_fft_z_back<double>(const double2 *, double *, int, int, int64_t, const Twiddles<double2> &, cudaStream_t);
template cudaError_t launch_ring_gather<float>(const float2 *, int, const RingArg &, StepGrids, bool, float2 *, const Twiddles<float2> &, const Batch &, cudaStream_t, const float *);
template cudaError_t launch_ring_gather<double>(const double2 *, int, const RingArg &, StepGrids, bool, double2 *, const Twiddles<double2> &, const Batch &, cudaStream_t, const float *);
template cudaError_t launch_fft_cols<float>(float2 *, StepGrids, const RingArg &, const Twiddles<float2> &, const Batch &, cudaStream_t);
template cudaError_t launch_fft_cols<double>(double2 *, StepGrids, const RingArg &, const Twiddles<double2> &, const Batch &, cudaStream_t);
template cudaError_t launch_step2<float>(const StepIIArgs &, const float2 *, const int64_t *, const int64_t *, int,
                                         cudaStream_t);
template cudaError_t launch_step2<double>(const StepIIArgs &, const double2 *, const int64_t *, const int64_t *, int,
                                          cudaStream_t);
template cudaError_t launch_reduce_partials<float>(const Group *, int64_t, const double *, int, double *, const Batch &, cudaStream_t);
template cudaError_t launch_reduce_partials<double>(const Group *, int64_t, const double *, int, double *, const Batch &, cudaStream_t);
template cudaError_t launch_epilogue<float>(int, const EpiArgs &, const double *, int, int, const double *, double,
                                            double *, const Batch &, cudaStream_t, bool);
template cudaError_t launch_epilogue<double>(int, const EpiArgs &, const double *, int, int, const double *, double,
                                             double *, const Batch &, cudaStream_t, bool);
template cudaError_t launch_epilogue_views<float>(EpiViews, const double *, double, const Batch &, cudaStream_t, bool);
template cudaError_t launch_epilogue_views<double>(EpiViews, const double *, double, const Batch &, cudaStream_t, bool);

}  // namespace bisp
