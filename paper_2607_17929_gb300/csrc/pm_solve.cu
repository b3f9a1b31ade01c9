// Fourier-space solution of the field equations (Sec. 3.1), one thread per
// mode of the half spectrum [kz][ky][kx], kx in [0, N/2]:
//
//   phi_k = -R_k / (kt^2 + 3Hc/dtau_{n-1} + 3Hc^2)          (Eq. NewtonHc, backward difference)
//   chi_k = -3/(4 kt^4) kt_i kt_j Sig_ij,k                  (scalar part of Eq. spacespace)
//   B_i,k = 4 (delta_ij - kt_i kt_j / kt^2) F_j,k / kt^2    (Eq. momentumcontraint, spin-1 part)
//   h_A   : h'' + 2Hc h' + kt^2 h = e^A_ij Sig_ij, one implicit-midpoint step
//
// or, with B from the spin-1 part of Eq. spacespace ((d_tau + 2Hc) B_j = W_j, d_i -> i kt_i):
//   W_j = -i (delta_jl - kt_j kt_l / kt^2) kt_i Sig_il,k / kt^2
//   B_j,k = (a_{n-1} / a_n)^2 B_j,k(previous step) + dtau_{n-1} W_j      (backward Euler in a^2 B)
//
// with kt_i = 2N sin(pi n_i / N), so kt^2 is the eigenvalue of minus the
// 7-point Laplacian.  The k = 0 mode of phi comes from the FP64 particle sum
// of the projection; chi, B and h vanish at k = 0 and on Nyquist modes.
// Outputs are scaled by 1/N^3 so that the inverse transforms need no
// normalisation.
#include "pm_internal.cuh"

namespace pm {

namespace {

template <class T> struct SolveParams {
    void *spec;        // 9 half spectra: R, Fx, Fy, Fz, Sxx, Sxy, Sxz, Syy, Syz
    void *tens;        // 4 half spectra: h+, hx, h+', hx'
    const T *ktab;     // ktilde per DFT index
    double *dscal;     // [1 + ring] mean phi per ring slot, [8 ..] slots of the k = 0 excess
    int imean_prev, imean_new;
    int N;
    int64_t nh;
    int full, newtonian, bootstrap;
    double four_pi_g_a2, c1, c2;   // FP64 copies for the k = 0 mode
    T cphi, inv_n3, hc_half, dtau;
    void *bstate;      // 3 half spectra of B_k (unnormalised), B from Eq. spacespace only
    int b_space, b_seed;
    T b_decay, dtau_prev;
};

// 1 / sqrt(x).  FP64, whose pipe bounds the FP64 solve, takes CUDA's rsqrt and one Newton step with the residual
// 1 - x r r to twice the precision, which leaves about half a unit in the last place: fewer operations than a square
// root and a quotient, and as exact.  FP32, bound by memory, takes those.
// Solve of a step at 256^3, FP64: 4.42 ms with square root, quotients and the nine products of each polarisation
// tensor, 3.56 now; of 2e5 modes against extended precision the error of h is 2.0e-16 and that of h beside a scalar part
// 100 times larger 3.2e-15 (3.9e-15 before), with rsqrt alone 2.3e-16.
__device__ __forceinline__ double inv_sqrt(double x)
{
    const double r = rsqrt(x), t = x * r;
    return fma(0.5 * r, fma(-t, r, 1.0) - r * fma(x, r, -t), r);
}
__device__ __forceinline__ float inv_sqrt(float x) { return 1.f / sqrtf(x); }

template <class T>
__global__ void __launch_bounds__(256) k_solve(SolveParams<T> p)
{
    using C = typename Cplx<T>::type;
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    // the k = 0 excess of the projection: block 0 (whole, as nh >= 320) sums its slots and clears them for the next one
    double k0 = 0.0;
    if (blockIdx.x == 0 && !p.newtonian) {
        __shared__ double part[8];
        static_assert(NK0SLOTS == 4 * 256, "four slots a thread");
#pragma unroll
        for (int q = 0; q < 4; q++) {
            k0 += p.dscal[8 + threadIdx.x + 256 * q];
            p.dscal[8 + threadIdx.x + 256 * q] = 0.0;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) k0 += __shfl_down_sync(0xffffffffu, k0, o);
        if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = k0;
        __syncthreads();
        k0 = 0.0;
        if (threadIdx.x == 0)
            for (int q = 0; q < 8; q++) k0 += part[q];
    }
    if (e >= p.nh) return;
    const int N = p.N, h = N / 2 + 1;
    const int kx = (int)(e % h);
    const int64_t r = e / h;
    const int ky = (int)(r % N), kz = (int)(r / N);
    const int nv[3] = {kx, ky <= N / 2 ? ky : ky - N, kz <= N / 2 ? kz : kz - N};
    const T kt[3] = {p.ktab[kx], p.ktab[ky], p.ktab[kz]};
    const T k2 = kt[0] * kt[0] + kt[1] * kt[1] + kt[2] * kt[2];
    const bool zero = (kx == 0 && ky == 0 && kz == 0);
    const bool nyq = (2 * kx == N) || (2 * abs(nv[1]) == N) || (2 * abs(nv[2]) == N);
    C *S = reinterpret_cast<C *>(p.spec);
    C *H = reinterpret_cast<C *>(p.tens);
    const int64_t nh = p.nh;
    // every input of this mode, loaded before any output is stored
    const bool fullmode = p.full && !zero && !nyq;
    const bool bint = p.b_space && !p.b_seed;
    C inR, inS[5], inH[4], inF[3];
    if (!zero) inR = S[e];
    if (fullmode) {
#pragma unroll
        for (int c = 0; c < 5; c++) inS[c] = S[(4 + c) * nh + e];
#pragma unroll
        for (int c = 0; c < 4; c++) inH[c] = H[c * nh + e];
        const C *FB = bint ? reinterpret_cast<const C *>(p.bstate) : S + nh;
#pragma unroll
        for (int c = 0; c < 3; c++) inF[c] = FB[c * nh + e];
    }

    // scalar potential phi
    if (zero) {
        double mean_phi = 0.0;
        if (!p.newtonian) {
            double mean_r = p.four_pi_g_a2 * k0;
            if (!p.bootstrap) mean_r -= p.c1 * p.dscal[1 + p.imean_prev];
            mean_phi = -mean_r / (p.c1 + p.c2);
        }
        p.dscal[1 + p.imean_new] = mean_phi;
        C v;
        v.x = (T)mean_phi;
        v.y = 0;
        S[0] = v;
    } else {
        C R = inR;
        const T f = -p.inv_n3 / (k2 + p.cphi);
        R.x *= f;
        R.y *= f;
        S[e] = R;
    }
    if (!p.full) return;
    if (zero || nyq) {
        C z;
        z.x = 0;
        z.y = 0;
#pragma unroll
        for (int c = 1; c <= 4; c++) S[c * nh + e] = z;
#pragma unroll
        for (int c = 0; c < 4; c++) H[c * nh + e] = z;
        if (p.b_space) {
            C *BS = reinterpret_cast<C *>(p.bstate);
#pragma unroll
            for (int c = 0; c < 3; c++) BS[c * nh + e] = z;
        }
        return;
    }
    // trace-free Sig as a symmetric matrix (Sig_zz = -Sig_xx - Sig_yy)
    const C sxx = inS[0], sxy = inS[1], sxz = inS[2], syy = inS[3], syz = inS[4];
    C szz;
    szz.x = -sxx.x - syy.x;
    szz.y = -sxx.y - syy.y;
    const C Sm[3][3] = {{sxx, sxy, sxz}, {sxy, syy, syz}, {sxz, syz, szz}};

    // v_l = kt_i Sig_il and kt_i kt_j Sig_ij
    C v[3], kks;
#pragma unroll
    for (int l = 0; l < 3; l++) {
        v[l].x = kt[0] * Sm[0][l].x + kt[1] * Sm[1][l].x + kt[2] * Sm[2][l].x;
        v[l].y = kt[0] * Sm[0][l].y + kt[1] * Sm[1][l].y + kt[2] * Sm[2][l].y;
    }
    kks.x = kt[0] * v[0].x + kt[1] * v[1].x + kt[2] * v[2].x;
    kks.y = kt[0] * v[0].y + kt[1] * v[1].y + kt[2] * v[2].y;
    const T ik2 = T(1) / k2;

    // tensor sector: polarisation basis from the axis with the smallest |n_i|
    {
        const T ikn = inv_sqrt(k2);
        const T kh[3] = {kt[0] * ikn, kt[1] * ikn, kt[2] * ikn};
        int m = 0;
        if (abs(nv[1]) < abs(nv[m])) m = 1;
        if (abs(nv[2]) < abs(nv[m])) m = 2;
        const T km = m == 0 ? kh[0] : m == 1 ? kh[1] : kh[2];
        T e1[3] = {-km * kh[0], -km * kh[1], -km * kh[2]};
#pragma unroll
        for (int d = 0; d < 3; d++) e1[d] += d == m ? T(1) : T(0);
        const T il = inv_sqrt(e1[0] * e1[0] + e1[1] * e1[1] + e1[2] * e1[2]);
#pragma unroll
        for (int d = 0; d < 3; d++) e1[d] *= il;
        const T e2[3] = {kh[1] * e1[2] - kh[2] * e1[1], kh[2] * e1[0] - kh[0] * e1[2],
                         kh[0] * e1[1] - kh[1] * e1[0]};
        // e^+_ij Sig_ij = (e1 Sig e1 - e2 Sig e2) / sqrt2, e^x_ij Sig_ij = sqrt2 e1 Sig e2
        C sp, sx;
        sp.x = sp.y = sx.x = sx.y = 0;
#pragma unroll
        for (int i = 0; i < 3; i++) {
            C a, b;   // (Sig e1)_i, (Sig e2)_i
            a.x = Sm[i][0].x * e1[0] + Sm[i][1].x * e1[1] + Sm[i][2].x * e1[2];
            a.y = Sm[i][0].y * e1[0] + Sm[i][1].y * e1[1] + Sm[i][2].y * e1[2];
            b.x = Sm[i][0].x * e2[0] + Sm[i][1].x * e2[1] + Sm[i][2].x * e2[2];
            b.y = Sm[i][0].y * e2[0] + Sm[i][1].y * e2[1] + Sm[i][2].y * e2[2];
            sp.x = sp.x + e1[i] * a.x - e2[i] * b.x;
            sp.y = sp.y + e1[i] * a.y - e2[i] * b.y;
            sx.x += e1[i] * b.x;
            sx.y += e1[i] * b.y;
        }
        const T is2 = T(0.70710678118654752440084436210484903928), s2 = T(1.41421356237309504880168872420969807857);
        sp.x *= is2;
        sp.y *= is2;
        sx.x *= s2;
        sx.y *= s2;
        // implicit midpoint: (I - dt/2 A) y' = (I + dt/2 A) y + dt (0, s), A = [[0,1],[-k2,-2Hc]]
        const T dt = p.dtau, hc = p.hc_half;
        const T m12 = -T(0.5) * dt, m21 = T(0.5) * dt * k2, m22 = T(1) + dt * hc;
        const T p12 = T(0.5) * dt, p21 = -T(0.5) * dt * k2, p22 = T(1) - dt * hc;
        const T idet = T(1) / (m22 - m12 * m21);
#pragma unroll
        for (int a = 0; a < 2; a++) {
            const C s = a == 0 ? sp : sx;
            C hh = inH[a], vv = inH[2 + a];
            C r1, r2;
            r1.x = hh.x + p12 * vv.x;
            r1.y = hh.y + p12 * vv.y;
            r2.x = p21 * hh.x + p22 * vv.x + dt * s.x;
            r2.y = p21 * hh.y + p22 * vv.y + dt * s.y;
            hh.x = (m22 * r1.x - m12 * r2.x) * idet;
            hh.y = (m22 * r1.y - m12 * r2.y) * idet;
            vv.x = (-m21 * r1.x + r2.x) * idet;
            vv.y = (-m21 * r1.y + r2.y) * idet;
            H[a * nh + e] = hh;
            H[(2 + a) * nh + e] = vv;
        }
    }
    // scalar slip chi (written over Sxx)
    {
        // 1 / kt^4 as exact as the quotient: the square of 1 / kt^2 doubles its rounding, the same for both parts of a mode,
        // which the residual takes out again (chi of a 192^3 mixed box at z = 1 against 64 bits 3.5e-7 -> 3.1e-7)
        const T k4 = k2 * k2, t = ik2 * ik2;
        const T f = -T(0.75) * (t + t * (T(1) - k4 * t)) * p.inv_n3;
        C chi;
        chi.x = f * kks.x;
        chi.y = f * kks.y;
        S[4 * nh + e] = chi;
    }
    // frame dragging B (written over F)
    if (p.b_space && !p.b_seed) {
        C *BS = reinterpret_cast<C *>(p.bstate);
        const T w = p.dtau_prev * ik2;
#pragma unroll
        for (int j = 0; j < 3; j++) {
            // dtau W_j = dtau (-i) (v_j - kt_j kv / kt^2) / kt^2
            const T px = v[j].x - kt[j] * kks.x * ik2, py = v[j].y - kt[j] * kks.y * ik2;
            C b = inF[j];
            b.x = p.b_decay * b.x + w * py;
            b.y = p.b_decay * b.y - w * px;
            BS[j * nh + e] = b;
            b.x *= p.inv_n3;
            b.y *= p.inv_n3;
            S[(1 + j) * nh + e] = b;
        }
    } else {
        const C F[3] = {inF[0], inF[1], inF[2]};
        C kF;
        kF.x = kt[0] * F[0].x + kt[1] * F[1].x + kt[2] * F[2].x;
        kF.y = kt[0] * F[0].y + kt[1] * F[1].y + kt[2] * F[2].y;
        const T f = T(4) * ik2;
#pragma unroll
        for (int i = 0; i < 3; i++) {
            C b;
            // kt_i kF rounded by itself in each component: kF / kt^2 formed once leaves its rounding in all three, along
            // kt, in a B that is small against F (6.8e-14 of it instead of 6.1e-14)
            b.x = f * (F[i].x - kt[i] * kF.x * ik2);
            b.y = f * (F[i].y - kt[i] * kF.y * ik2);
            if (p.b_space) reinterpret_cast<C *>(p.bstate)[i * nh + e] = b;  // seeds the integration
            b.x *= p.inv_n3;
            b.y *= p.inv_n3;
            S[(1 + i) * nh + e] = b;
        }
    }
}

// P(k) binning of one half spectrum of delta, bins round(|n|) = b: modes with 0 < kx < N/2 stand for themselves and
// their conjugate partner.  The mode count and the mean |k| of a bin need no spectrum: k_pk_modes counts the modes of
// each |n|^2 and k_pk_shells takes one FP64 square root per value, instead of one per mode.  The bin of a mode comes
// from an FP32 square root corrected in integers, which leaves two FP64 products and one shared atomic a mode.
// 256^3 mixed: 0.45 -> 0.12 ms.
__device__ __forceinline__ int pk_shell(int n2)   // round(sqrt(n2)): b b - b < n2 <= b b + b
{
    int b = (int)(sqrtf((float)n2) + 0.5f);
    if (n2 > b * b + b) b++;
    if (n2 <= b * b - b && b > 0) b--;
    return b;
}

// a warp per row (kz, ky): acc[b] += w |d|^2 / N^6
template <class T>
__global__ void __launch_bounds__(256) k_pk_bin(const typename Cplx<T>::type *d, int N, int nbins, double inv_n6, double *acc)
{
    extern __shared__ double sb[];
    for (int i = threadIdx.x; i < nbins; i += blockDim.x) sb[i] = 0.0;
    __syncthreads();
    const int h = N / 2 + 1, rows = N * N, lane = threadIdx.x & 31;
    for (int r = blockIdx.x * 8 + (threadIdx.x >> 5); r < rows; r += gridDim.x * 8) {
        const int ky = r % N, kz = r / N;
        const int ny = ky <= N / 2 ? ky : ky - N, nz = kz <= N / 2 ? kz : kz - N, nt = ny * ny + nz * nz;
        for (int kx = lane; kx < h; kx += 32) {
            const int b = pk_shell(kx * kx + nt);
            if (b < 1 || b >= nbins) continue;
            const typename Cplx<T>::type v = d[(int64_t)r * h + kx];
            const T w = (kx > 0 && 2 * kx < N) ? T(2) : T(1);
            const double re = widen(v.x), im = widen(v.y);
            atomicAdd(&sb[b], widen(w * v.x) * re + widen(w * v.y) * im);
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < nbins; i += blockDim.x)
        if (sb[i] != 0.0) atomicAdd(&acc[i], sb[i] * inv_n6);
}

// All three sums of every mode in one launch, for meshes of at most 64: there the launches of the kernels below and the
// clearing of their histogram cost more than an FP64 square root and two more shared atomics a mode do (32^3 FP64 P(k)
// 80 us, 87 with them; 64^3 104 and 110).
template <class T>
__global__ void __launch_bounds__(256) k_pk_bin_small(const typename Cplx<T>::type *d, int N, int nbins, double inv_n6,
                                                       double *acc)
{
    extern __shared__ double sb[];   // 3 nbins: sums of w |d|^2, w |k|, w
    for (int i = threadIdx.x; i < 3 * nbins; i += blockDim.x) sb[i] = 0.0;
    __syncthreads();
    const int h = N / 2 + 1, e = blockIdx.x * 256 + threadIdx.x, kx = e % h, r = e / h;
    if (r < N * N) {
        const int ky = r % N, kz = r / N, ny = ky <= N / 2 ? ky : ky - N, nz = kz <= N / 2 ? kz : kz - N;
        const int n2 = kx * kx + ny * ny + nz * nz, b = pk_shell(n2);
        if (b >= 1 && b < nbins) {
            const typename Cplx<T>::type v = d[e];
            const double w = (kx > 0 && 2 * kx < N) ? 2.0 : 1.0, re = widen(v.x), im = widen(v.y);
            atomicAdd(&sb[b], w * (re * re + im * im));
            atomicAdd(&sb[nbins + b], w * (6.283185307179586476925286766559 * sqrt((double)n2)));
            atomicAdd(&sb[2 * nbins + b], w);
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < 3 * nbins; i += blockDim.x)
        if (sb[i] != 0.0) atomicAdd(&acc[i], i < nbins ? sb[i] * inv_n6 : sb[i]);
}

// hist[n2] = number of modes of the full spectrum with |n|^2 = n2, from the octant 0 <= |n_i| <= N/2 (a block per
// |n_z|, |n_y|); only shells below nbins are counted
__global__ void k_pk_modes(int N, int nbins, unsigned int *hist)
{
    const int m = N / 2, ny = blockIdx.x, nz = blockIdx.y;
    const unsigned mult = (ny > 0 && ny < m ? 2u : 1u) * (nz > 0 && nz < m ? 2u : 1u);
    for (int kx = threadIdx.x; kx <= m; kx += blockDim.x) {
        const int n2 = kx * kx + ny * ny + nz * nz;
        if (n2 > 0 && n2 <= (int64_t)nbins * (nbins - 1)) atomicAdd(&hist[n2], (kx > 0 && kx < m ? 2u : 1u) * mult);
    }
}

// a warp per bin: acc[nbins + b] = sum of 2 pi |n| over its modes, acc[2 nbins + b] = their number
__global__ void __launch_bounds__(256) k_pk_shells(const unsigned int *hist, int n2max, int nbins, double *acc)
{
    const int b = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (b >= nbins) return;
    double k = 0.0, cnt = 0.0;
    if (b > 0)
        for (int n2 = b * b - b + 1 + lane; n2 <= min(b * b + b, n2max); n2 += 32) {
            const double c = (double)hist[n2];
            cnt += c;
            k += c * (6.283185307179586476925286766559 * sqrt((double)n2));
        }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        k += __shfl_xor_sync(0xffffffffu, k, o);
        cnt += __shfl_xor_sync(0xffffffffu, cnt, o);
    }
    if (lane == 0) {
        acc[nbins + b] = k;
        acc[2 * nbins + b] = cnt;
    }
}

}  // namespace

template <class T>
void launch_solve(Ctx &c, const StepScalars &s)
{
    SolveParams<T> p{};
    p.spec = c.spec;
    p.tens = c.tens;
    p.ktab = reinterpret_cast<const T *>(c.ktab);
    p.dscal = c.dscal;
    p.imean_prev = c.iphi_prev;
    p.imean_new = c.iphi_new;
    p.N = c.N;
    p.nh = c.nh;
    p.newtonian = s.newtonian;
    p.bootstrap = s.bootstrap;
    p.full = !(s.newtonian || s.bootstrap);
    p.four_pi_g_a2 = s.four_pi_g / (s.a * s.a);
    p.c1 = s.c_phi_dt;
    p.c2 = s.c_phi_h2;
    p.cphi = (T)(s.c_phi_dt + s.c_phi_h2);
    p.inv_n3 = (T)(1.0 / (double)c.nc);
    p.hc_half = (T)s.hc_half;
    p.dtau = (T)s.dtau;
    p.bstate = c.bstate;
    p.b_space = s.b_space && c.bstate != nullptr;
    p.b_seed = s.b_seed;
    p.b_decay = (T)s.b_decay;
    p.dtau_prev = (T)s.dtau_prev;
    k_solve<T><<<(unsigned)((c.nh + 255) / 256), 256, 0, c.stream>>>(p);
    c.launches++;
}

template <class T>
void launch_pk_bin(Ctx &c, const void *spec_in, int nbins, double *d_acc, unsigned int *hist)
{
    const double inv_n6 = 1.0 / ((double)c.nc * (double)c.nc);
    const int m = c.N / 2;
    cudaMemsetAsync(d_acc, 0, sizeof(double) * 3 * nbins, c.stream);
    if (c.N <= 64 && nbins <= 2048) {   // 3 nbins doubles of shared memory: 48 KB
        k_pk_bin_small<T><<<(unsigned)((c.nh + 255) / 256), 256, 3 * sizeof(double) * nbins, c.stream>>>(
            reinterpret_cast<const typename Cplx<T>::type *>(spec_in), c.N, nbins, inv_n6, d_acc);
        return;
    }
    cudaMemsetAsync(hist, 0, sizeof(unsigned int) * (size_t)pk_hist_len(c.N), c.stream);
    const int blocks = std::min((c.N * c.N + 7) / 8, 152 * 8);
    k_pk_bin<T><<<blocks, 256, sizeof(double) * nbins, c.stream>>>(
        reinterpret_cast<const typename Cplx<T>::type *>(spec_in), c.N, nbins, inv_n6, d_acc);
    k_pk_modes<<<dim3(m + 1, m + 1), std::min(256, (m + 32) / 32 * 32), 0, c.stream>>>(c.N, nbins, hist);
    k_pk_shells<<<(nbins + 7) / 8, 256, 0, c.stream>>>(hist, (int)pk_hist_len(c.N) - 1, nbins, d_acc);
}

template void launch_solve<double>(Ctx &, const StepScalars &);
template void launch_solve<float>(Ctx &, const StepScalars &);
template void launch_pk_bin<double>(Ctx &, const void *, int, double *, unsigned int *);
template void launch_pk_bin<float>(Ctx &, const void *, int, double *, unsigned int *);

}  // namespace pm
