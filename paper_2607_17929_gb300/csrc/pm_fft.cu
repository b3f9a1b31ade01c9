// Pencil-staged 3D FFT for the metric solves (Sec. 2.3 transforms a 3D
// field as a sequence of 1D FFTs along x, y and z; here every sequence of
// 1D transforms runs from shared memory on one GPU).
//
// Layout: real fields [z][y][x]; half spectra [kz][ky][kx] with
// kx in [0, N/2].  Forward: x pass (two real rows packed as one complex
// line, r2c split), y pass, z pass.  Inverse: z, y, then x (c2r).  No
// normalisation: the Fourier solve applies 1/N^3.
//
// Every mesh size that a context accepts (2^a 3^b, a >= 3, up to 1024) has its passes compiled for it: the points
// of a line stay in registers through all radix stages and consecutive stages exchange them through shared memory
// (pm_fft_core.cuh).  Sizes outside the powers of two and 192 used to take a run-time plan whose stages went through
// shared memory: at 288^3 mixed a field's three forward passes 0.77 -> 0.18 ms, its inverse ones 0.69 -> 0.18.
#include "pm_fft_core.cuh"
#include "pm_internal.cuh"

namespace pm {

namespace {

// ---------------------------------------------------------------------------
// Compile-time-N passes (register-resident radix stages, see pm_fft_core.cuh).
// ---------------------------------------------------------------------------
// Shapes of the FP32 column passes for power-of-two sizes >= 64 (ZP: the z
// pass, whose points are a whole plane apart, else the y pass): points per
// thread, lines per block (the line width sets the contiguous row segment)
// and the threads per SM the register budget must allow.  Shape 0 is the one
// timed best at 512^3; fft_tune_shapes picks among the three per context.
struct ColShape {
    int p, l, tpsm;
};
constexpr int NCOLSHAPES = 3;
constexpr ColShape kColY[NCOLSHAPES] = {{32, 8, 512}, {16, 8, 1024}, {8, 8, 1536}};
constexpr ColShape kColZ[NCOLSHAPES] = {{16, 16, 1024}, {8, 16, 1536}, {16, 8, 1024}};

template <class T, int N, bool ZP = false, int V = 0> struct Lines {
    static constexpr bool tuned = sizeof(T) == 4 && N % 3 != 0 && N >= 64 && N <= 512;
    static constexpr ColShape sh = ZP ? kColZ[V] : kColY[V];
    static constexpr int CP = tuned && sh.p != 8 ? sh.p : 0;  // 0: default points per thread
    static constexpr int TL = fftc::Geo<N>::TL;
    static constexpr int TLC = fftc::Geo<N, CP>::TL;
    // lines per block of the column passes: 64-byte row segments by default, >= 128 threads
    static constexpr int col0 = tuned ? sh.l : (sizeof(T) == 4 ? 8 : 4);
    static constexpr int col1 = col0 * TLC < 128 ? 128 / TLC : col0;
    static constexpr int col = col1 * TLC > 1024 ? 1024 / TLC : col1;
    // Row pairs per block of the x passes: 256 threads, 128 for sizes with a factor of three.  Those hold
    // 24 points a thread, few warps fit an SM, and every exchange stops the whole block: smaller blocks
    // leave others to run meanwhile (one r2c launch of 9 fields / one c2r launch of 5, us, with 256 and with 128
    // threads: FP32 192^3 170 / 97 and 152 / 88; 288^3 614 / 343 and 568 / 330; 72^3 16.7 / 18.6 and 16.5 / 14.5;
    // FP64 192^3 1836 / 959 and 1720 / 878; 64 threads gain no more).  With 8 points a thread they gain nothing
    // (256^3 220 / 131 and 223 / 128, 512^3 1759 / 1002 and 1816 / 1016).
    static constexpr int row_threads = N % 3 == 0 && TL <= 128 ? 128 : 256;
    static constexpr int row = TL >= 256 ? 1 : row_threads / TL;
    // resident blocks per SM the register allocation must allow
    static constexpr int tpsm = tuned ? sh.tpsm : (fftc::Geo<N>::P == 8 ? (sizeof(T) == 4 ? 1536 : 1024) : 0);
    static constexpr int col_min_blocks = tpsm / (TLC * col) > 0 ? tpsm / (TLC * col) : 1;
};

template <class T, int N, bool ZP, int V> size_t col_fast_smem()
{
    using G = fftc::Geo<N>;
    return sizeof(typename Cplx<T>::type) * (G::TWN + (size_t)N * Lines<T, N, ZP, V>::col);  // TWN does not depend on P
}
template <class T, int N> size_t row_fast_smem()
{
    using G = fftc::Geo<N>;
    return sizeof(typename Cplx<T>::type) * (G::TWN + (size_t)Lines<T, N>::row * fftc::RowIdx<N>::pitch);
}

template <class T, int N, int DIR, bool ZP, int V>
__global__ void __launch_bounds__(Lines<T, N, ZP, V>::TLC * Lines<T, N, ZP, V>::col, Lines<T, N, ZP, V>::col_min_blocks)
k_col_fast(const __grid_constant__ Ptrs ptrs, const typename Cplx<T>::type *__restrict__ twg)
{
    using C = typename Cplx<T>::type;
    constexpr int CP = Lines<T, N, ZP, V>::CP;
    using G = fftc::Geo<N, CP>;
    constexpr int L = Lines<T, N, ZP, V>::col;
    extern __shared__ __align__(16) unsigned char smem[];
    C *tw = reinterpret_cast<C *>(smem);
    C *buf = tw + G::TWN;
    for (int i = threadIdx.x; i < G::TWN; i += blockDim.x) tw[i] = twg[i];
    // strides and line counts are compile-time constants of N and the pass, so every point's address is the
    // thread's base plus an immediate (no per-point address registers, no spills)
    constexpr int H = N / 2 + 1;
    constexpr int SJ = ZP ? N * H : H;          // point stride
    constexpr int NLINES = N * H;               // lines (kz, kx) or (ky, kx)
    const int l = threadIdx.x % L, t = threadIdx.x / L;
    const int g = (int)blockIdx.x * L + l;
    const bool ok = g < NLINES;
    // y: line (kz, kx) starts at kz N H + kx; z: line (ky, kx) at ky H + kx = g
    const int base = ok ? (ZP ? g : (g / H) * (N * H) + g % H) : 0;
    C *data = reinterpret_cast<C *>(ptrs.p[blockIdx.y]) + base + (int64_t)t * SJ;
    C v[G::P];
#pragma unroll
    for (int i = 0; i < G::P; i++)
        v[i] = ok ? data[(int64_t)fftc::in_pos<N, CP>(0, i) * SJ] : fftc::mk<C>(0, 0);
    __syncthreads();
    fftc::fft<C, N, DIR, CP>(v, t, buf, tw, fftc::ColIdx{L, l});
    if (ok) {
#pragma unroll
        for (int i = 0; i < G::P; i++) data[(int64_t)fftc::out_pos<N, CP>(0, i) * SJ] = v[i];
    }
}

template <class T, int N>
__global__ void __launch_bounds__(fftc::Geo<N>::TL * Lines<T, N>::row)
k_r2c_fast(const __grid_constant__ Ptrs in, const __grid_constant__ Ptrs out, const typename Cplx<T>::type *__restrict__ twg, int64_t npairs)
{
    using C = typename Cplx<T>::type;
    using G = fftc::Geo<N>;
    constexpr int L = Lines<T, N>::row, H = N / 2 + 1;
    extern __shared__ __align__(16) unsigned char smem[];
    C *tw = reinterpret_cast<C *>(smem);
    C *buf = tw + G::TWN;
    for (int i = threadIdx.x; i < G::TWN; i += blockDim.x) tw[i] = twg[i];
    const int t = threadIdx.x % G::TL, l = threadIdx.x / G::TL;
    const int64_t pair = (int64_t)blockIdx.x * L + l;
    const bool ok = pair < npairs;
    const T *src = reinterpret_cast<const T *>(in.p[blockIdx.y]);
    C *dst = reinterpret_cast<C *>(out.p[blockIdx.y]);
    const T *ra = src + 2 * pair * N, *rb = ra + N;
    C v[G::P];
#pragma unroll
    for (int i = 0; i < G::P; i++) {
        const int j = fftc::in_pos<N>(t, i);
        v[i] = ok ? fftc::mk<C>(ra[j], rb[j]) : fftc::mk<C>(0, 0);
    }
    __syncthreads();
    const fftc::RowIdx<N> ix{l * fftc::RowIdx<N>::pitch};
    fftc::fft<C, N, -1>(v, t, buf, tw, ix);
#pragma unroll
    for (int i = 0; i < G::P; i++) buf[ix(fftc::out_pos<N>(t, i))] = v[i];
    __syncthreads();
    if (!ok) return;
    C *oa = dst + 2 * pair * H, *ob = oa + H;
    const T half = (T)0.5;
    for (int k = t; k < H; k += G::TL) {
        const C zk = buf[ix(k)], zn = buf[ix((N - k) % N)];
        oa[k] = fftc::mk<C>(half * (zk.x + zn.x), half * (zk.y - zn.y));
        ob[k] = fftc::mk<C>(half * (zk.y + zn.y), -half * (zk.x - zn.x));
    }
}

template <class T, int N>
__global__ void __launch_bounds__(fftc::Geo<N>::TL * Lines<T, N>::row)
k_c2r_fast(const __grid_constant__ Ptrs in, const __grid_constant__ Ptrs out, const typename Cplx<T>::type *__restrict__ twg, int64_t npairs)
{
    using C = typename Cplx<T>::type;
    using G = fftc::Geo<N>;
    constexpr int L = Lines<T, N>::row, H = N / 2 + 1;
    extern __shared__ __align__(16) unsigned char smem[];
    C *tw = reinterpret_cast<C *>(smem);
    C *buf = tw + G::TWN;
    for (int i = threadIdx.x; i < G::TWN; i += blockDim.x) tw[i] = twg[i];
    const int t = threadIdx.x % G::TL, l = threadIdx.x / G::TL;
    const int64_t pair = (int64_t)blockIdx.x * L + l;
    const bool ok = pair < npairs;
    const C *src = reinterpret_cast<const C *>(in.p[blockIdx.y]);
    T *dst = reinterpret_cast<T *>(out.p[blockIdx.y]);
    const fftc::RowIdx<N> ix{l * fftc::RowIdx<N>::pitch};
    const C *ia = src + 2 * pair * H, *ib = ia + H;
    constexpr int NK = (H + G::TL - 1) / G::TL;
    C As[NK], Bs[NK];
#pragma unroll
    for (int q = 0; q < NK; q++) {
        const int k = t + q * G::TL;
        As[q] = (ok && k < H) ? ia[k] : fftc::mk<C>(0, 0);
        Bs[q] = (ok && k < H) ? ib[k] : fftc::mk<C>(0, 0);
    }
#pragma unroll
    for (int q = 0; q < NK; q++) {
        const int k = t + q * G::TL;
        if (k >= H) break;
        C A = As[q], B = Bs[q];
        if (k == 0 || 2 * k == N) {
            A.y = 0;
            B.y = 0;
        }
        buf[ix(k)] = fftc::mk<C>(A.x - B.y, A.y + B.x);
        if (k > 0 && 2 * k < N) buf[ix(N - k)] = fftc::mk<C>(A.x + B.y, B.x - A.y);
    }
    __syncthreads();
    C v[G::P];
#pragma unroll
    for (int i = 0; i < G::P; i++) v[i] = buf[ix(fftc::in_pos<N>(t, i))];
    __syncthreads();
    fftc::fft<C, N, +1>(v, t, buf, tw, ix);
    if (!ok) return;
    T *wa = dst + 2 * pair * N, *wb = wa + N;
#pragma unroll
    for (int i = 0; i < G::P; i++) {
        const int j = fftc::out_pos<N>(t, i);
        wa[j] = v[i].x;
        wb[j] = v[i].y;
    }
}

template <class T, int N> struct FastPasses {
    static void attrs()
    {
        static DeviceOnce once;
        once_on_device(once, [] {
            set_col<0>();
            if constexpr (Lines<T, N>::tuned) {
                set_col<1>();
                set_col<2>();
            }
            allow_smem(k_r2c_fast<T, N>, row_fast_smem<T, N>());
            allow_smem(k_c2r_fast<T, N>, row_fast_smem<T, N>());
        });
    }
    template <int V> static void set_col()
    {
        allow_smem(k_col_fast<T, N, -1, false, V>, col_fast_smem<T, N, false, V>());
        allow_smem(k_col_fast<T, N, 1, false, V>, col_fast_smem<T, N, false, V>());
        allow_smem(k_col_fast<T, N, -1, true, V>, col_fast_smem<T, N, true, V>());
        allow_smem(k_col_fast<T, N, 1, true, V>, col_fast_smem<T, N, true, V>());
    }
    template <bool ZP, int V>
    static void cols_t(Ctx &c, int nf, const Ptrs &p, int dir)
    {
        constexpr int64_t nl = (int64_t)N * (N / 2 + 1);   // lines of a y or z pass
        constexpr int L = Lines<T, N, ZP, V>::col;
        constexpr int threads = Lines<T, N, ZP, V>::TLC * L;
        dim3 grid((unsigned)((nl + L - 1) / L), nf);
        const auto *tw = reinterpret_cast<const typename Cplx<T>::type *>(c.tw2);
        const size_t sm = col_fast_smem<T, N, ZP, V>();
        if (dir < 0)
            k_col_fast<T, N, -1, ZP, V><<<grid, threads, sm, c.stream>>>(p, tw);
        else
            k_col_fast<T, N, 1, ZP, V><<<grid, threads, sm, c.stream>>>(p, tw);
        c.launches++;
    }
    template <bool ZP>
    static void cols_v(Ctx &c, int nf, const Ptrs &p, int dir)
    {
        const int v = Lines<T, N>::tuned ? c.col_shape[ZP ? 1 : 0] : 0;
        if constexpr (Lines<T, N>::tuned) {
            if (v == 1) return cols_t<ZP, 1>(c, nf, p, dir);
            if (v == 2) return cols_t<ZP, 2>(c, nf, p, dir);
        }
        cols_t<ZP, 0>(c, nf, p, dir);
    }
    // y pass (ZP false): lines (kz, kx), points a row apart; z pass: lines (ky, kx), points a plane apart
    template <bool ZP> static void cols(Ctx &c, int nf, const Ptrs &p, int dir) { cols_v<ZP>(c, nf, p, dir); }
    static void rows(Ctx &c, int nf, const Ptrs &pi, const Ptrs &po, int dir)
    {
        constexpr int L = Lines<T, N>::row;
        const int64_t npairs = (int64_t)N * N / 2;
        dim3 grid((unsigned)((npairs + L - 1) / L), nf);
        const auto *tw = reinterpret_cast<const typename Cplx<T>::type *>(c.tw2);
        if (dir < 0)
            k_r2c_fast<T, N><<<grid, fftc::Geo<N>::TL * L, row_fast_smem<T, N>(), c.stream>>>(pi, po, tw, npairs);
        else
            k_c2r_fast<T, N><<<grid, fftc::Geo<N>::TL * L, row_fast_smem<T, N>(), c.stream>>>(pi, po, tw, npairs);
        c.launches++;
    }
};

}  // namespace

template <class T>
void fft_forward(Ctx &c, int nf, const void *const *real_in, void *const *spec_out)
{
    const int N = c.N;
    Ptrs pi{}, po{};
    for (int i = 0; i < nf; i++) {
        pi.p[i] = const_cast<void *>(real_in[i]);
        po.p[i] = spec_out[i];
    }
    auto fast = [&]<int NN>() {
        using F = FastPasses<T, NN>;
        F::attrs();
        F::rows(c, nf, pi, po, -1);
        c.mark(EV_FWD_X);
        F::template cols<false>(c, nf, po, -1);
        c.mark(EV_FWD_Y);
        F::template cols<true>(c, nf, po, -1);
        c.mark(EV_FWD_Z);
    };
    with_mesh_size(N, fast);
}

template <class T>
void fft_inverse(Ctx &c, int nf, void *const *spec_in, void *const *real_out)
{
    const int N = c.N;
    Ptrs pi{}, po{};
    for (int i = 0; i < nf; i++) {
        pi.p[i] = spec_in[i];
        po.p[i] = real_out[i];
    }
    auto fast = [&]<int NN>() {
        using F = FastPasses<T, NN>;
        F::attrs();
        F::template cols<true>(c, nf, pi, +1);
        c.mark(EV_INV_Z);
        F::template cols<false>(c, nf, pi, +1);
        c.mark(EV_INV_Y);
        F::rows(c, nf, pi, po, +1);
        c.mark(EV_INV_X);
    };
    with_mesh_size(N, fast);
}

template <class T>
bool fft_shapes_tunable(const Ctx &c)
{
    bool t = false;
    with_mesh_size(c.N, [&]<int NN>() { t = Lines<T, NN>::tuned; });
    return t;
}

// Time the column-pass shapes of one pass on the context's spectra (9 forward and 5 inverse line
// transforms, as in a step) and keep the fastest.  pass 0: y, 1: z.
template <class T>
int tune_col_pass(Ctx &c, int pass)
{
    const int N = c.N;
    Ptrs p{};
    for (int i = 0; i < 9; i++) p.p[i] = reinterpret_cast<typename Cplx<T>::type *>(c.spec) + (size_t)i * c.nh;
    cudaEvent_t e0, e1;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    float best = 1e30f;
    int best_v = 0;
    for (int v = 0; v < NCOLSHAPES; v++) {
        c.col_shape[pass] = v;
        auto run = [&]() {
            with_mesh_size(N, [&]<int NN>() {
                using F = FastPasses<T, NN>;
                if (pass == 0) {
                    F::template cols<false>(c, 9, p, -1);
                    F::template cols<false>(c, 5, p, +1);
                } else {
                    F::template cols<true>(c, 9, p, -1);
                    F::template cols<true>(c, 5, p, +1);
                }
            });
        };
        run();   // warm-up (and the first launch of a new shape)
        cudaEventRecord(e0, c.stream);
        for (int r = 0; r < 3; r++) run();
        cudaEventRecord(e1, c.stream);
        cudaEventSynchronize(e1);
        float ms = 0.f;
        cudaEventElapsedTime(&ms, e0, e1);
        if (ms < best) {
            best = ms;
            best_v = v;
        }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    c.col_shape[pass] = best_v;
    return best_v;
}

template <class T>
bool fft_tune_shapes(Ctx &c, int force_y, int force_z)
{
    if (!fft_shapes_tunable<T>(c)) {
        c.col_shape[0] = c.col_shape[1] = 0;
        return false;
    }
    with_mesh_size(c.N, [&]<int NN>() { FastPasses<T, NN>::attrs(); });
    if (force_y < 0 || force_z < 0) {
        // the spectra hold nothing between steps; clear them so the timed transforms see finite data
        cudaMemsetAsync(c.spec, 0, 9 * 2 * sizeof(T) * (size_t)c.nh, c.stream);
    }
    if (force_y >= 0) c.col_shape[0] = force_y;
    else tune_col_pass<T>(c, 0);
    if (force_z >= 0) c.col_shape[1] = force_z;
    else tune_col_pass<T>(c, 1);
    return true;
}

template bool fft_tune_shapes<float>(Ctx &, int, int);
template bool fft_tune_shapes<double>(Ctx &, int, int);

void fast_twiddles(int n, std::vector<double> &re_im)
{
    re_im.clear();
    const long double pi = 3.141592653589793238462643383279502884L;
    for (int s = 1; s < fftc::nstages(n); s++) {
        const int Ns = fftc::span_before(n, s), R = fftc::radix_at(n, s);
        for (int k = 0; k < Ns; k++)
            for (int r = 1; r < R; r++) {
                const long double ang = -2.0L * pi * (long double)(r * k) / (long double)(Ns * R);
                re_im.push_back((double)cosl(ang));
                re_im.push_back((double)sinl(ang));
            }
    }
}

template void fft_forward<double>(Ctx &, int, const void *const *, void *const *);
template void fft_forward<float>(Ctx &, int, const void *const *, void *const *);
template void fft_inverse<double>(Ctx &, int, void *const *, void *const *);
template void fft_inverse<float>(Ctx &, int, void *const *, void *const *);

}  // namespace pm
