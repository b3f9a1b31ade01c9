// Particle-mesh kernels: stress-energy projection, gather + kick + drift,
// counting sort by cell, particle I/O.
//
// Projection (Sec. 2.1 "particle-mesh projection", Eqs. matterstress):
// particles are kept sorted by cell.  A CTA owns a column of mesh vertices and
// marches along z, one plane of cells at a time.  A warp takes an x-row of
// cells: a lane forms the charges of one of its particles, then sums, for one
// vertex, over the particles of the two cells beside it; the sums of
// neighbouring planes meet in registers and those of neighbouring rows through
// shared memory.  No global atomics, and every mesh value is written once.
// The same kernel assembles the configuration-space sources of the field
// equations from phi_{n-1}, chi_{n-1}, phi_{n-2}.
#include <algorithm>
#include <cmath>
#include <type_traits>

#include "pm_internal.cuh"
#include "pm_rows.cuh"

namespace pm {

namespace {


// Accumulator of the T^00 charge, whose sums cancel against the uniform
// background in R.  FP64: plain double.  Mixed: float-float with Knuth's
// TwoSum, which loses nothing of a term whatever its size and the sum's, and
// the roundings of the high word summed up in the low one: about 48
// significant bits, and as many less as that word's own roundings come to
// (n terms: at most 2^-24 of their share, n 2^-24 of the sum).  The other
// components have no such cancellation and are summed in the field type.
template <class T> struct Acc;
template <> struct Acc<double> {
    double s;
    __device__ __forceinline__ void zero() { s = 0.0; }
    __device__ __forceinline__ void add(double x) { s += x; }
    __device__ __forceinline__ void add_product(double a, double b) { s = fma(a, b, s); }
    __device__ __forceinline__ double hi() const { return s; }
    __device__ __forceinline__ double lo() const { return 0.0; }
};
template <> struct Acc<float> {
    float s, c;
    __device__ __forceinline__ void zero() { s = 0.f; c = 0.f; }
    __device__ __forceinline__ void add(float x)
    {
        float t = __fadd_rn(s, x);
        float bp = __fsub_rn(t, s);
        float e = __fadd_rn(__fsub_rn(s, __fsub_rn(t, bp)), __fsub_rn(x, bp));
        s = t;
        c = __fadd_rn(c, e);
    }
    __device__ __forceinline__ void add_product(float a, float b) { add(__fmul_rn(a, b)); }
    __device__ __forceinline__ void add_two(float x, float lo)
    {
        add(x);
        c = __fadd_rn(c, lo);
    }
    __device__ __forceinline__ float hi() const { return s; }
    __device__ __forceinline__ float lo() const { return c; }
};

// 1 / sqrt(x) and a / b: the hardware approximations (a few ulp) in the mixed form, whose
// FP32 rounding already sets the error; CUDA's rsqrt (1 ulp) in FP64
__device__ __forceinline__ float rsqrt_t(float x) { return rsqrtf(x); }
__device__ __forceinline__ double rsqrt_t(double x) { return rsqrt(x); }
__device__ __forceinline__ float div_t(float a, float b) { return __fdividef(a, b); }

template <class T> __device__ __forceinline__ T mulr(T a, T b);
template <> __device__ __forceinline__ float mulr<float>(float a, float b) { return __fmul_rn(a, b); }
template <> __device__ __forceinline__ double mulr<double>(double a, double b) { return __dmul_rn(a, b); }

__device__ __forceinline__ int wrapi(int i, int n) { return i < 0 ? i + n : (i >= n ? i - n : i); }

template <class T> struct DepParams {
    const Particle<T> *part;
    const int32_t *start;
    const T *phi1;   // phi_{n-1}
    const T *chi1;   // chi_{n-1}
    const T *phi2;   // phi_{n-2}
    Ptrs out;        // R, Fx, Fy, Fz, Sxx, Sxy, Sxz, Syy, Syz
    double *k0slots; // NK0SLOTS partial sums of the k = 0 excess
    int N;
    int nrow, ncol;  // vertices of a tile along x and y
    int ntx, nty;    // tiles along x and y
    int tz;          // vertices of a tile along z
    int cyclic;      // one tile along x: the cell x0 - 1 is the row's last
    int newtonian;
    T a, a2, mass;
    T G;             // 4piG a^-2 N^3 (Newtonian: 4piG a^-1 N^3)
    T rb_hi, rb_lo;  // expected per-vertex charge sum of a uniform load, float-float split
    T c1, c2;        // 3Hc/dtau_{n-1}, 3Hc^2
    T inv_dt2;       // 1/dtau_{n-2}
    T halfN;         // N/2 (centred difference 1/(2 dx))
    int full_hc;     // R -= Nl, the remainder of Eq. fullHc
    int write_f;     // F_i is needed (momentum-constraint B)
    T hc, n2;        // Hc(a_n), N^2 (7-point Laplacian 1/dx^2)
    double inv_g;    // 1 / (4piG a^-2 N^3): Nl's share of the k = 0 sum
};

// e^x - 1 - x without cancellation: its Taylor series through x^9 / 9! for small |x| (truncation below
// 1e-8 relative in FP32 for |x| < 1/2 and below 1e-20 in FP64 for |x| < 1e-2), expm1(x) - x beyond.
template <class T> __device__ __forceinline__ T expm1_minus_x(T x)
{
    constexpr T lim = sizeof(T) == 4 ? T(0.5) : T(1e-2);
    if (fabs(x) >= lim) return expm1(x) - x;
    T s = T(1.0 / 362880.0);
    s = s * x + T(1.0 / 40320.0);
    s = s * x + T(1.0 / 5040.0);
    s = s * x + T(1.0 / 720.0);
    s = s * x + T(1.0 / 120.0);
    s = s * x + T(1.0 / 24.0);
    s = s * x + T(1.0 / 6.0);
    s = s * x + T(0.5);
    return s * x * x;
}

// Nonlinear remainder of Eq. fullHc at one vertex from phi_{n-1} (ph, and its six neighbours up/dn along
// each axis), chi_{n-1} (ch) and phi_{n-2}:
//   Nl = (e^{2phi} - 1) Lap phi - 1/2 e^{2phi} |grad phi|^2
//      + 3/2 [Hc^2 (e^x - 1 - x) - 2 Hc phi' (e^x - 1) + phi'^2 e^x],  x = -2 psi,
// the bracket being (Hc - phi')^2 e^{-2psi} - Hc^2 + 2 Hc phi' + 2 Hc^2 psi regrouped so that no term
// of size Hc^2 cancels.
template <class T>
__device__ __forceinline__ T hc_remainder(T ph, const T (&up)[3], const T (&dn)[3], T ch, T phi2, const DepParams<T> &p)
{
    T lap = T(-6) * ph, g2 = T(0);
#pragma unroll
    for (int d = 0; d < 3; d++) {
        lap += up[d] + dn[d];
        const T g = (up[d] - dn[d]) * p.halfN;
        g2 += g * g;
    }
    lap *= p.n2;
    const T psi = ph - ch;
    const T dphi = (ph - phi2) * p.inv_dt2;
    const T x = T(-2) * psi;
    const T em = expm1(x);
    const T e2p = exp(T(2) * ph);
    return expm1(T(2) * ph) * lap - T(0.5) * e2p * g2 +
           T(1.5) * (p.hc * p.hc * expm1_minus_x(x) - T(2) * p.hc * dphi * em + dphi * dphi * (em + T(1)));
}

// ---------------------------------------------------------------------------
// Mass deposit of the Newtonian mode in FP32: a particle's charge is its mass, so a vertex needs only the offsets
// of its 8 cells' particles.  One CTA per 8^3 tile of vertices stages the offsets of the 9^3 cells [x0 - 1, x0 + 8)
// in cell order, and each thread sums its vertex's products one by one with TwoSum, rows (z, y), (z, y - 1),
// (z - 1, y), (z - 1, y - 1), cells x - 1 then x.  This order is kept: the force correction feeds R through BF16
// layers, where a change in the last bit of R changes the momenta by 1e-3 of their size, so a faster summation
// order (the columns below need 0.33 ms at 288^3 with 201^3 particles) is not taken here.
// What bounds it: instruction issue of the 8 dependent sums per vertex.  Staging: in an even tile each thread takes
// the particles of its two cells, else every 512th particle, whose row it finds by halving the 81 rows' offsets (a
// row's cells follow each other in memory).  256^3 at z = 50 0.37 ms with the search alone, 0.35 with both; with its
// own cells alone, and the warp for full ones, z = 1 0.65 and 128^3 with 16 a cell 2.0, with both 0.57 and 0.71.
// The general tile kernel before it, which staged whole charge records, took 0.52 ms at 256^3, z = 50.
// ---------------------------------------------------------------------------
constexpr int MT = 8, MR = MT + 1, MCELLS = MR * MR * MR, MTHREADS = MT * MT * MT;
constexpr int MEVEN = 5;    // particles of two cells up to which a thread stages those of its own

template <class I> struct MassSmem {
    float4 rec[MCAP];                         // f
    I off[MCELLS + 1];                        // exclusive scan of the cells' counts
    I base[2][MR * MR];                       // particle j of the tile is base[..][its row] + j: [0] for a row's first cell
    I warp[MTHREADS / 32];
};

// I: type of the tile's offsets (mass_wide)
template <class I> __device__ __forceinline__ void mass_tile(const DepParams<float> &p, const int b)
{
    __shared__ MassSmem<I> sm;
    const int N = p.N, nt = N / MT, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int x0 = (b % nt) * MT, y0 = ((b / nt) % nt) * MT, z0 = (b / (nt * nt)) * MT;
    // first particle and count of cells 2 tid and 2 tid + 1, then the exclusive scan of the counts
    int n[2] = {0, 0}, s[2] = {0, 0};
#pragma unroll
    for (int q = 0; q < 2; q++) {
        const int i = 2 * tid + q;
        if (i < MCELLS) {
            const int sx = i % MR, sy = (i / MR) % MR, sz = i / (MR * MR);
            const int g = (wrapi(z0 - 1 + sz, N) * N + wrapi(y0 - 1 + sy, N)) * N + wrapi(x0 - 1 + sx, N);
            s[q] = __ldg(p.start + g);
            n[q] = __ldg(p.start + g + 1) - s[q];
        }
    }
    I inc = (I)n[0] + n[1];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const I v = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += v;
    }
    if (lane == 31) sm.warp[wid] = inc;
    __syncthreads();
    I before = 0, total = 0;
#pragma unroll
    for (int w = 0; w < MTHREADS / 32; w++) {
        const I v = sm.warp[w];
        before += w < wid ? v : 0;
        total += v;
    }
    const I e = before + inc - n[0] - n[1];
    if (2 * tid <= MCELLS) sm.off[2 * tid] = e;
    if (2 * tid + 1 <= MCELLS) sm.off[2 * tid + 1] = e + n[0];
#pragma unroll
    for (int q = 0; q < 2; q++) {   // the row's cells after its first one follow each other in memory, too
        const int i = 2 * tid + q;
        if (i < MCELLS && i % MR < 2) sm.base[i % MR][i / MR] = s[q] - (q ? e + n[0] : e);
    }
    const bool even = !__syncthreads_or(n[0] + n[1] > MEVEN) && total <= MCAP;

    const int ox = tid % MT, oy = (tid / MT) % MT, oz = tid / (MT * MT);
    Acc<float> acc;
    acc.zero();
    for (I lo = 0; lo < total; lo += MCAP) {
        const I hi = min(total, lo + MCAP);
        auto stage = [&](I i, int to) {
            const float *q = reinterpret_cast<const float *>(p.part + i);
            const float2 xy = __ldg(reinterpret_cast<const float2 *>(q + 2));
            sm.rec[to] = make_float4(xy.x, xy.y, __ldg(q + 4), 0.f);
        };
        if (even) {   // a thread those of its two cells
#pragma unroll 1
            for (int k = 0; k < n[0] + n[1]; k++) stage(k < n[0] ? s[0] + k : s[1] + (k - n[0]), (int)e + k);
        } else        // a thread every 512th, its row by halving
            for (int k = tid; k < (int)(hi - lo); k += MTHREADS) {
                const I j = lo + k;
                int row = 0;
#pragma unroll
                for (int half = 64; half > 0; half >>= 1)
                    if (row + half < MR * MR && sm.off[MR * (row + half)] <= j) row += half;
                stage(sm.base[j >= sm.off[MR * row + 1]][row] + j, k);
            }
        __syncthreads();
        // vertex o receives from cells o - d, d in {0,1}^3, weight (d ? f : 1 - f) per axis; the x-neighbours
        // (region x = ox and ox + 1) are adjacent in the particle order
#pragma unroll
        for (int dz = 0; dz < 2; dz++)
#pragma unroll
            for (int dy = 0; dy < 2; dy++) {
                const int ts = ox + MR * ((oy + 1 - dy) + MR * (oz + 1 - dz));   // cell with dx = 1
                const I mid = sm.off[ts + 1];                                  // first particle with dx = 0
                const I je = min(sm.off[ts + 2], hi);
                for (I j = max(sm.off[ts], lo); j < je; j++) {
                    const float4 f = sm.rec[(int)(j - lo)];
                    const float wyz = (dy ? f.y : 1.f - f.y) * (dz ? f.z : 1.f - f.z);
                    const float w = (j < mid ? f.x : 1.f - f.x) * wyz;
                    acc.add(mulr(w, p.mass));
                }
            }
        __syncthreads();
    }
    const int go = ((z0 + oz) * N + (y0 + oy)) * N + (x0 + ox);
    // the uniform background is removed before rounding
    reinterpret_cast<float *>(p.out.p[0])[go] = p.G * ((acc.hi() - p.rb_hi) + (acc.lo() - p.rb_lo));
}

template <class I> __global__ void __launch_bounds__(MTHREADS, 4) k_mass(const __grid_constant__ DepParams<float> p)
{
    mass_tile<I>(p, blockIdx.x);
}

// ---------------------------------------------------------------------------
// Deposit.  A CTA owns the vertices [x0, x0 + nrow) x [y0, y0 + ncol) x [z0, z0 + tz) and visits the cells
// that reach them, one more in front along each axis, plane by plane along z.  Warp w takes the x-row of cells
// y = y0 - 1 + w, whose particles are consecutive in memory:
//  - lane i forms the weights and the 9 charges of the i-th particle of the row (32 at a time) and leaves them
//    in shared memory, so that this work is even whatever the cells hold;
//  - lane l, the vertex x0 + l, sums over the particles of the cells x - 1 and x, again consecutive, the shares
//    of the row's four (y, z) corner lines: two of them belong to plane z, where the sums of the plane before
//    wait in registers, and two to plane z + 1;
//  - shared memory carries the y + 1 sums to the next row's warp, which then holds whole vertices.
// What bounds it: instruction issue (FP32) and the FP64 pipe (FP64).  A particle's charges are formed once per
// CTA that needs them (about 1.2 times: (nrow + 1)/nrow, (ncol + 1)/ncol and (tz + 1)/tz), its record is read
// by two vertex lanes, and a vertex costs 36 products per particle of two cells, in packed pairs in FP32, or, where a
// cell is full, 3 per lane (crowd_sums).  Against 8^3 vertex tiles that
// stage the charges of 9^3 cells and let each vertex gather from 8 cells (a record read 8 times, potentials, ranges
// and a scan set up per tile), at 512^3 mixed 6.9 -> 3.9 ms early (sums of one plane in registers, 40 of them, so
// 20 warps an SM), at 256^3 FP64 15.3 -> 8.1, late (192^3, z = 1, cells of up to 55 particles) 0.59 -> 0.58; at 4 and 16
// particles a cell (128^3) FP32 0.45 -> 0.49 and 1.66 -> 1.95, FP64 7.9 -> 8.2 and 33.8 -> 20.0.  A cell per lane with its
// 8 corners in registers was faster early (3.4 ms) but ran as long as its row's fullest cell (late 0.78 ms).
// ---------------------------------------------------------------------------
constexpr int DROWS = 10;                 // rows of cells of a tile along y, one warp each
constexpr int DTY = DROWS - 1;            // and of vertices, at most
constexpr int DEP_THREADS = 32 * DROWS;
constexpr int DPX = 34, DPY = DTY + 2;    // staged potentials: x0 - 1 .. x0 + nrow, y0 - 1 .. y0 + ncol
constexpr int DPN = DPX * DPY;
constexpr int DRING = 5;                  // staged planes: z - 1 .. z + 2, and the one being fetched
constexpr int NDEPSHAPES = 2;

// sums exchanged per vertex: T00 (two words in FP32) and the other 8 charges
template <class T, bool FULL> constexpr int dep_words() { return (sizeof(T) == 4 ? 2 : 1) + (FULL ? 8 : 0); }
// words of a particle's weights and charges; DEN: its weights in two words instead of charges
template <bool FULL, bool DEN> constexpr int dep_rec() { return FULL || DEN ? 17 : 9; }
// staged particle records (the first 32 of a row, two planes), exchange rows (two planes), weights and charges,
// staged potentials
template <class T, bool FULL, bool DEN> constexpr size_t dep_smem()
{
    return 2 * DEP_THREADS * sizeof(Particle<T>) +
           sizeof(T) * 32 * DROWS * (2 * dep_words<T, FULL>() + dep_rec<FULL, DEN>()) + sizeof(T) * (FULL ? 2 * DRING * DPN : 0);
}

// (hi, lo) += (h, l) of another sum, TwoSum on the high words
template <class T> __device__ __forceinline__ void acc_merge(Acc<T> &s, const Acc<T> &o)
{
    s.add(o.hi());
    if constexpr (sizeof(T) == 4) s.c += o.c;
}
// Two values side by side.  FP32 takes the packed instructions, one for both values, each rounded as the scalar one's.
template <class T> struct Pair;
template <> struct Pair<float> {
    uint64_t v;
    static __device__ __forceinline__ Pair of(float a, float b)
    {
        Pair r;
        asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(a), "f"(b));
        return r;
    }
    __device__ __forceinline__ float get(int k) const
    {
        float a, b;
        asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
        return k ? b : a;
    }
};
template <> struct Pair<double> {
    double a, b;
    static __device__ __forceinline__ Pair of(double a, double b) { return {a, b}; }
    __device__ __forceinline__ double get(int k) const { return k ? b : a; }
};
__device__ __forceinline__ Pair<float> operator+(Pair<float> x, Pair<float> y)
{
    Pair<float> r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(x.v), "l"(y.v));
    return r;
}
__device__ __forceinline__ Pair<float> operator-(Pair<float> x, Pair<float> y)
{
    Pair<float> r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(x.v), "l"(y.v));
    return r;
}
__device__ __forceinline__ Pair<float> operator*(Pair<float> x, Pair<float> y)
{
    Pair<float> r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(x.v), "l"(y.v));
    return r;
}
__device__ __forceinline__ Pair<float> fma(Pair<float> x, Pair<float> y, Pair<float> z)
{
    Pair<float> r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(x.v), "l"(y.v), "l"(z.v));
    return r;
}
__device__ __forceinline__ Pair<double> operator+(Pair<double> x, Pair<double> y) { return {x.a + y.a, x.b + y.b}; }
__device__ __forceinline__ Pair<double> fma(Pair<double> x, Pair<double> y, Pair<double> z)
{
    return {::fma(x.a, y.a, z.a), ::fma(x.b, y.b, z.b)};
}
// four staged values (FP64: in two parts, 32 records apart)
__device__ __forceinline__ void pairs(const float4 *v, Pair<float> (&p)[2])
{
    const ulonglong2 a = *reinterpret_cast<const ulonglong2 *>(v);
    p[0].v = a.x;
    p[1].v = a.y;
}
__device__ __forceinline__ void pairs(const double2 *v, Pair<double> (&p)[2])
{
    p[0] = {v[0].x, v[0].y};
    p[1] = {v[32].x, v[32].y};
}

// Acc of two sums side by side
template <class T> struct AccPair;
template <> struct AccPair<double> {
    Pair<double> s;
    __device__ __forceinline__ void zero() { s = {0.0, 0.0}; }
    __device__ __forceinline__ void add_product(Pair<double> a, Pair<double> b) { s = fma(a, b, s); }
    __device__ __forceinline__ void merge(const double *h, const double *) { s = s + Pair<double>{h[0], h[1]}; }
    __device__ __forceinline__ Acc<double> get(int k) const { return {s.get(k)}; }
};
template <> struct AccPair<float> {
    Pair<float> s, c;
    __device__ __forceinline__ void zero() { s = c = Pair<float>::of(0.f, 0.f); }
    __device__ __forceinline__ void add_two(Pair<float> x, Pair<float> lo)
    {
        add(x);
        c = c + lo;
    }
    __device__ __forceinline__ void add(Pair<float> x)
    {
        const Pair<float> t = s + x, b = t - s, e = (s - (t - b)) + (x - b);
        s = t;
        c = c + e;
    }
    __device__ __forceinline__ void add_product(Pair<float> a, Pair<float> b) { add(a * b); }
    __device__ __forceinline__ void merge(const float *h, const float *l) { add_two(Pair<float>::of(h[0], h[1]), Pair<float>::of(l[0], l[1])); }
    __device__ __forceinline__ Acc<float> get(int k) const { return {s.get(k), c.get(k)}; }
};

// Cell, offset and momentum of one particle.
template <class T> struct PartFU {
    int cell;
    T f[3], u[3];
};
// from its 16-byte parts, `step` parts apart
__device__ __forceinline__ PartFU<float> unpack(const float4 *q, int step)
{
    const float4 a = q[0], b = q[step];
    return {__float_as_int(a.x), {a.z, a.w, b.x}, {b.y, b.z, b.w}};
}
__device__ __forceinline__ PartFU<double> unpack(const double2 *q, int step)
{
    const double2 a = q[0], b = q[step], c = q[2 * step], d = q[3 * step];
    return {__double2loint(a.x), {a.y, b.x, b.y}, {c.x, c.y, d.x}};
}

// The FP32 weights of charges() with the low words that make them exact to 2^-48 (w above its rounding).
__device__ __forceinline__ void weights_lo(const PartFU<float> &P, const float (&w)[8], float (&lo)[8])
{
    float g[3], ge[3];   // 1 - f in two words
#pragma unroll
    for (int d = 0; d < 3; d++) {
        g[d] = 1.f - P.f[d];
        ge[d] = __fsub_rn(__fsub_rn(1.f, g[d]), P.f[d]);
    }
#pragma unroll
    for (int i = 0; i < 4; i++) {
        const float a = i & 1 ? P.f[1] : g[1], ae = i & 1 ? 0.f : ge[1], b = i & 2 ? P.f[2] : g[2], be = i & 2 ? 0.f : ge[2];
        const float p = __fmul_rn(a, b), e = __fmaf_rn(a, b, -p) + (a * be + ae * b);
        lo[i] = __fmaf_rn(g[0], p, -w[i]) + (g[0] * e + ge[0] * p);
        lo[4 + i] = __fmaf_rn(P.f[0], p, -w[4 + i]) + P.f[0] * e;
    }
}

// Charges of one particle and its 8 CIC weights (w[4 dx + dy + 2 dz]).  lo/up: the staged potentials of the
// cell's lower and upper plane at its corner (0, 0); chi DRING DPN values after phi.  ex receives the excess of the T^00 charge over a particle at rest (the k = 0 mode).
template <class T, bool FULL>
__device__ __forceinline__ void charges(const DepParams<T> &p, const PartFU<T> &P, const T *lo, const T *up, T (&w)[8],
                                        T &q00, T (&q)[8], T &ex)
{
    const T fx = P.f[0], fy = P.f[1], fz = P.f[2];
    const T gx = T(1) - fx, gy = T(1) - fy, gz = T(1) - fz;
    const T yz[4] = {gy * gz, fy * gz, gy * fz, fy * fz};
#pragma unroll
    for (int i = 0; i < 4; i++) {
        w[i] = gx * yz[i];
        w[4 + i] = fx * yz[i];
    }
    if (!FULL && p.newtonian) {
        q00 = p.mass;
        ex = T(0);
        return;
    }
    T ph = 0, ch = 0;
    if constexpr (FULL) {
#pragma unroll
        for (int i = 0; i < 8; i++) {
            const T *s = (i & 2 ? up : lo) + (i >> 2) + (i & 1 ? DPX : 0);
            ph += w[i] * s[0];
            ch += w[i] * s[DRING * DPN];
        }
    }
    const T ux = P.u[0], uy = P.u[1], uz = P.u[2];
    const T u2 = ux * ux + uy * uy + uz * uz;
    const T e2 = p.a2 + u2;
    const T iE = rsqrt_t(e2);
    // E = a + u^2 / (E + a): the approximate E enters only the small term, so E keeps the
    // accuracy of a (the T^00 charge cancels against the background in R)
    T dE;
    if constexpr (sizeof(T) == 4) {
        dE = div_t(u2, e2 * iE + p.a);
    } else {   // a Newton step for dE (dE + 2 a) = u^2 from E - a: as accurate as the quotient, and fewer operations
        const T E0 = e2 * iE, d0 = E0 - p.a;
        dE = d0 - T(0.5) * (iE * (d0 * (E0 + p.a) - u2));
    }
    const T E = p.a + dE;
    const T v2 = u2 * iE * iE;
    const T m = p.mass;
    const T mE = m * E, g = ph * (T(3) + v2);
    q00 = mE + mE * g;
    ex = m * dE + mE * g;
    if constexpr (FULL) {
        const T wv = m * (T(1) + T(4) * ph - ch);
        q[0] = wv * ux;
        q[1] = wv * uy;
        q[2] = wv * uz;
        const T ws = m * iE * (T(1) + ph * (T(3) - v2));
        const T sx = ws * ux, sy = ws * uy;
        const T tr3 = ws * u2 * T(1.0 / 3.0);
        q[3] = sx * ux - tr3;
        q[4] = sx * uy;
        q[5] = sx * uz;
        q[6] = sy * uy - tr3;
        q[7] = sy * uz;
    }
}

// sum over the warp, in every lane
template <class T> __device__ __forceinline__ Acc<T> warp_sum(Acc<T> v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        Acc<T> b;
        b.s = __shfl_xor_sync(0xffffffffu, v.s, o);
        if constexpr (sizeof(T) == 4) b.c = __shfl_xor_sync(0xffffffffu, v.c, o);
        acc_merge(v, b);
    }
    return v;
}

// values to and from 16-byte parts
__device__ __forceinline__ float4 pack(const float *v) { return make_float4(v[0], v[1], v[2], v[3]); }
__device__ __forceinline__ double2 pack(const double *v) { return make_double2(v[0], v[1]); }
__device__ __forceinline__ void unpackv(const float4 &a, float *v)
{
    v[0] = a.x;
    v[1] = a.y;
    v[2] = a.z;
    v[3] = a.w;
}
__device__ __forceinline__ void unpackv(const double2 &a, double *v)
{
    v[0] = a.x;
    v[1] = a.y;
}

template <class T> __device__ __forceinline__ void cp_async_word(T *s, const T *g)
{
    const unsigned a = (unsigned)__cvta_generic_to_shared(s);
    if constexpr (sizeof(T) == 4) asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(a), "l"(g));
    else asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(a), "l"(g));
}

// The field-equation sources of one vertex: dS the T^00 sum over the background, s the other 8 sums,
// dn/md/up the staged potentials at the vertex in planes z - 1, z and z + 1.
template <class T>
__device__ __forceinline__ void dep_epilogue(const DepParams<T> &p, const T *dn, const T *md, const T *up, T phi2, T dS,
                                             const T (&s)[8], int g, Acc<T> &k0)
{
    constexpr int CH = DRING * DPN;
    const T ph = md[0], ch = md[CH];
    const T pu[3] = {md[1], md[DPX], up[0]}, pd[3] = {md[-1], md[-DPX], dn[0]};
    const T cu[3] = {md[CH + 1], md[CH + DPX], up[CH]}, cd[3] = {md[CH - 1], md[CH - DPX], dn[CH]};
    T nl = T(0);
    if (p.full_hc) {
        nl = hc_remainder<T>(ph, pu, pd, ch, phi2, p);
        k0.add(-nl * (T)p.inv_g);   // the k = 0 mode carries the mean of -Nl
    }
    reinterpret_cast<T *>(p.out.p[0])[g] = p.G * dS - p.c1 * ph - p.c2 * ch - nl;
    // with dc = 2 dx d chi and b = 2 dx d psi (psi = phi - chi):
    //   2 TF[2 d_i phi d_j phi - d_i(phi + psi) d_j(phi + psi)] = N^2/2 TF[dc_i dc_j - 2 b_i b_j]
    T dc[3], b[3], hc[3], hb[3];
#pragma unroll
    for (int d = 0; d < 3; d++) {
        dc[d] = cu[d] - cd[d];
        b[d] = (pu[d] - pd[d]) - dc[d];
        hc[d] = T(0.5) * p.n2 * dc[d];
        hb[d] = p.n2 * b[d];
    }
    if (p.write_f) {
        const T f = (ph - phi2) * p.inv_dt2 * p.halfN;   // phi' / (2 dx)
#pragma unroll
        for (int d = 0; d < 3; d++) reinterpret_cast<T *>(p.out.p[1 + d])[g] = p.G * s[d] - f * b[d];
    }
    const T G4 = T(4) * p.G;
    auto quad = [&](int i, int j) { return hc[i] * dc[j] - hb[i] * b[j]; };
    const T qxx = quad(0, 0), qyy = quad(1, 1), tr3 = (qxx + qyy + quad(2, 2)) * T(1.0 / 3.0);
    reinterpret_cast<T *>(p.out.p[4])[g] = G4 * s[3] - (qxx - tr3);
    reinterpret_cast<T *>(p.out.p[5])[g] = hb[0] * b[1] + (G4 * s[4] - hc[0] * dc[1]);
    reinterpret_cast<T *>(p.out.p[6])[g] = hb[0] * b[2] + (G4 * s[5] - hc[0] * dc[2]);
    reinterpret_cast<T *>(p.out.p[7])[g] = G4 * s[6] - (qyy - tr3);
    reinterpret_cast<T *>(p.out.p[8])[g] = hb[1] * b[2] + (G4 * s[7] - hc[1] * dc[2]);
}

// A vertex lane's sums in one plane, of its own row of vertices and of the one at y + 1: T00 of both, the others by row.
template <class T> struct RowSums {
    AccPair<T> t00;
    Pair<T> q[2][4];
    __device__ __forceinline__ void zero()
    {
        t00.zero();
#pragma unroll
        for (int i = 0; i < 2; i++)
#pragma unroll
            for (int j = 0; j < 4; j++) q[i][j] = Pair<T>::of(T(0), T(0));
    }
};

// The particles of a warp's row of cells in one plane: those of the cell x0 - 1, then those of the others.
// Particle i of the row is p.part[i < nh ? sh + i : sr + i]; a vertex lane's particles are prev .. end - 1, of
// the cell at x - 1 below mid and of its own from there on.
struct DepRow {
    int sh, nh, sr, total;
    int prev, mid, end;
    int wrap;   // cyclic rows: lane 0's particles of the row's last cell are wrap .. total - 1
};

// A thread's view of its tile.
template <class T, bool FULL, bool DEN> struct DepCol {
    static constexpr int PQ = sizeof(Particle<T>) / 16;    // 16-byte parts of a record
    static constexpr int VT = 16 / sizeof(T);              // values in 16 bytes
    static constexpr int W = dep_words<T, FULL>(), R = dep_rec<FULL, DEN>();
    using V = std::conditional_t<sizeof(T) == 4, float4, double2>;
    // Particles of one cell in a group of 32 from which the warp sums them together, and the row's particles from which
    // it looks for such cells (a load of one per cell, whose rows it would only slow down, has 32).  A vertex lane takes
    // 36 products a particle one after another, for two cells: with 16 particles a cell 29 of 32 lanes wait for it.  The
    // warp takes 3 a particle and some 100 instructions a cell; FP64, where an instruction costs the same for one lane as
    // for all, four cells at a time.  Deposit at 128^3 without and with it, and of the 8^3 tiles before the columns:
    // FP32 16 a cell 3.25, 1.94 (1.66), 4 a cell 0.47, 0.49 (0.45), a tenth of the mass in cells of 1000 0.42, 0.26
    // (0.36); FP64 77.6, 19.9 (33.8), 10.2, 8.2 (7.9), 6.9, 2.8 (5.9) ms.  From 4 or 7 particles on FP32 is slower
    // (4 a cell 0.78, 0.54), and from 10 on FP64 (16 a cell 28).
    static constexpr int CROWD = sizeof(T) == 8 ? 4 : 10, CROWDED_ROW = 48;

    const DepParams<T> &p;
    V *stage;            // the row's first 32 records in this and the next plane, [par][part][thread]
    T *xch, *rec, *ring;
    int z0, nz, row;     // row: y N + x0
    int nx;              // vertices of the row, 0 for a warp without one
    int halo;            // index of the cell x0 - 1 relative to row
    int go[2];           // staged potentials: where this thread's two entries of a plane come from (-1: none)
    int sc;              // ring slot of plane z; plane z + i is in slot sc + i modulo DRING
    Acc<T> k0;           // this thread's share of the k = 0 excess (float-float in the mixed form)

    __device__ __forceinline__ int slot(int i) const { return sc + i >= DRING ? sc + i - DRING : sc + i; }
    __device__ __forceinline__ void fetch(int slot, int z)
    {
        if constexpr (FULL) {
            const int base = wrapi(z, p.N) * (p.N * p.N);
            T *s = ring + slot * DPN + threadIdx.x;
#pragma unroll
            for (int q = 0; q < 2; q++)
                if (go[q] >= 0) {
                    cp_async_word(s + q * DEP_THREADS, p.phi1 + (base + go[q]));
                    cp_async_word(s + q * DEP_THREADS + DRING * DPN, p.chi1 + (base + go[q]));
                }
        }
    }
    // the start and end of a lane's cell and of the cell x0 - 1
    __device__ __forceinline__ int4 bounds(int z) const
    {
        if (nx == 0) return make_int4(0, 0, 0, 0);
        const int32_t *c = p.start + (wrapi(z, p.N) * (p.N * p.N) + row);   // N^3 <= 2^30
        const int l = min((int)threadIdx.x & 31, nx - 1);
        return make_int4(__ldg(c + l), __ldg(c + l + 1), __ldg(c + halo), __ldg(c + halo + 1));
    }
    __device__ __forceinline__ DepRow range(const int4 &v) const
    {
        const int lane = threadIdx.x & 31;
        DepRow r;
        r.sh = v.z;
        r.nh = p.cyclic ? 0 : v.w - v.z;
        r.sr = __shfl_sync(0xffffffffu, v.x, 0) - r.nh;
        r.total = __shfl_sync(0xffffffffu, v.y, 31) - r.sr;
        r.mid = v.x - r.sr;
        r.end = v.y - r.sr;
        r.prev = __shfl_up_sync(0xffffffffu, r.mid, 1);
        r.wrap = lane == 0 && p.cyclic ? v.z - r.sr : r.total;
        if (lane == 0) r.prev = 0;
        if (lane >= nx) r.prev = r.mid = r.end;   // nothing
        return r;
    }
    // the row's records from c0 on, 32 at most, into part `par` of the stage
    __device__ __forceinline__ void fetch_row(int par, const DepRow &r, int c0 = 0)
    {
        const int i = c0 + (threadIdx.x & 31);
        if (i < r.total) {
            const V *g = reinterpret_cast<const V *>(p.part + (i < r.nh ? r.sh + i : r.sr + i));
#pragma unroll
            for (int q = 0; q < PQ; q++) {
                const unsigned a = (unsigned)__cvta_generic_to_shared(stage + (par * PQ + q) * DEP_THREADS + threadIdx.x);
                asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(a), "l"(g + q) : "memory");
            }
        }
    }

    // The sums of records n0 .. n1 - 1 of the staged group, all of one cell, to the cell's 8 corners, into sum
    // [side][value][line]: a lane forms the T00 sum of a quarter of them for one corner, and two of the other sums of all
    // of them.
    __device__ __forceinline__ void crowd_sums(int n0, int n1, T *sum) const
    {
        const int lane = threadIdx.x & 31, side = lane & 1, line = (lane >> 1) & 3, part = lane >> 3;
        const T *wt = rec + (side * (4 / VT) + line / VT) * (32 * VT) + line % VT, *r0 = rec + 32 * (R - 1);
        Acc<T> t;
        t.zero();
#pragma unroll 2
        for (int n = n0 + part; n < n1; n += 4) {
            if constexpr (DEN) t.add_two(wt[n * VT], wt[2 * 32 * VT + n * VT]);
            else t.add_product(wt[n * VT], r0[n]);
        }
#pragma unroll
        for (int k = 8; k < 32; k *= 2) {
            Acc<T> b;
            b.s = __shfl_xor_sync(0xffffffffu, t.s, k);
            if constexpr (sizeof(T) == 4) b.c = __shfl_xor_sync(0xffffffffu, t.c, k);
            acc_merge(t, b);
        }
        T *d = sum + side * (4 * W) + line;
        if (part == 0) {
            d[0] = t.hi();
            if constexpr (sizeof(T) == 4) d[4] = t.lo();
        }
        if constexpr (FULL) {
            const T *q = rec + (8 / VT + 2 * part / VT) * (32 * VT) + 2 * part % VT;
            Pair<T> qs = Pair<T>::of(T(0), T(0));
#pragma unroll 4
            for (int n = n0; n < n1; n++) {
                const T w = wt[n * VT];
                qs = fma(Pair<T>::of(w, w), *reinterpret_cast<const Pair<T> *>(q + n * VT), qs);
            }
            d[4 * (W - 8 + 2 * part)] = qs.get(0);
            d[4 * (W - 7 + 2 * part)] = qs.get(1);
        }
    }
    // adds what crowd_sums left for one side of a cell
    __device__ __forceinline__ void crowd_add(const T *v, RowSums<T> &A, RowSums<T> &B) const
    {
#pragma unroll
        for (int k = 0; k < 2; k++) {
            RowSums<T> &S = k ? B : A;
            S.t00.merge(v + 2 * k, v + 4 + 2 * k);
            if constexpr (FULL) {
#pragma unroll
                for (int i = 0; i < 2; i++)
#pragma unroll
                    for (int j = 0; j < 4; j++) {
                        const T *u = v + 4 * (W - 8 + 2 * j) + 2 * k + i;
                        S.q[i][j] = S.q[i][j] + Pair<T>::of(u[0], u[4]);
                    }
            }
        }
    }

    // One plane of cells, z = z0 + iz; PAR = iz & 1.  r: its rows, rn: those of the next plane (replaced by the
    // ones after it).  A: the sums of plane z (on entry what the plane before put there), B: those of plane z + 1.
    template <int PAR> __device__ __forceinline__ void plane(int iz, DepRow &r, DepRow &rn, RowSums<T> &A, RowSums<T> &B)
    {
        const int z = z0 + iz, w = threadIdx.x >> 5, lane = threadIdx.x & 31;
        const int cells = z * (p.N * p.N) + row;       // first cell of the row (used for 0 <= z < N)
        const bool out = iz >= 0 && w > 0 && lane < nx;
        const int col = w * DPX + lane + 1;            // the vertex in a staged plane
        T f2 = 0;
        if (FULL && out) f2 = __ldg(p.phi2 + cells + lane);
        int4 nb = make_int4(0, 0, 0, 0);
        if (iz + 2 < nz) nb = bounds(z + 2);
        // this row's first records, copied since the plane before (the potentials fetched there may still be under way)
        asm volatile("cp.async.wait_group 1;" ::: "memory");
        fetch_row(PAR ^ 1, rn);
        asm volatile("cp.async.commit_group;" ::: "memory");
        const T *lo = ring + sc * DPN + w * DPX, *up = ring + slot(1) * DPN + w * DPX;
        B.zero();
        V *rv = reinterpret_cast<V *>(rec);            // [part][32]: weights dx = 0, dx = 1, T00 and the other charges
        const int base = wrapi(z, p.N) * (p.N * p.N) + row - 1;
        for_groups(r.total, [&](int c0) {
            const int i = c0 + lane;
            PartFU<T> P{};
            if (c0 > 0) asm volatile("cp.async.wait_group 0;" ::: "memory");
            int cx = 0;                                // the cell's lower corner in the row's staged potentials
            if (i < r.total) {
                P = unpack(stage + PAR * PQ * DEP_THREADS + threadIdx.x, DEP_THREADS);
                if (i >= r.nh) cx = P.cell - base;
            }
            T wt[8], q00, q[8], ex;
            charges<T, FULL>(p, P, lo + cx, up + cx, wt, q00, q, ex);
            if (iz >= 0 && w > 0 && i >= r.nh && i < r.total) k0.add(ex);
            __syncwarp();
            if (r.total - c0 > 32) {   // the row's next records, over those used above
                fetch_row(PAR, r, c0 + 32);
                asm volatile("cp.async.commit_group;" ::: "memory");
            }
#pragma unroll
            for (int k = 0; k < 8 / VT; k++) rv[32 * k + lane] = pack(wt + VT * k);
            if constexpr (FULL) {
#pragma unroll
                for (int k = 0; k < 8 / VT; k++) rv[32 * (8 / VT + k) + lane] = pack(q + VT * k);
            }
            if constexpr (DEN) {
                float wlo[8];
                weights_lo(P, wt, wlo);
#pragma unroll
                for (int k = 0; k < 2; k++) rv[32 * (2 + k) + lane] = pack(wlo + 4 * k);
            }
            T *r0 = rec + 32 * (R - 1);
            r0[lane] = q00;
            __syncwarp();
            // particles n0 .. n1 - 1 of the chunk, those below nm from the cell at x - 1
            auto gather = [&](int n0, int n1, int nm) {
#pragma unroll(FULL ? 1 : 2)
                for (int n = n0; n < n1; n++) {
                    Pair<T> w[2], c[2];
                    const V *v = rv + n + (n < nm ? 32 * (4 / VT) : 0);
                    pairs(v, w);
                    if constexpr (DEN) {
                        pairs(v + 64, c);
                        A.t00.add_two(w[0], c[0]);
                        B.t00.add_two(w[1], c[1]);
                    } else {
                        const T t = r0[n];
                        A.t00.add_product(w[0], Pair<T>::of(t, t));
                        B.t00.add_product(w[1], Pair<T>::of(t, t));
                    }
                    if constexpr (FULL) {
                        Pair<T> ww[2][2];
#pragma unroll
                        for (int i = 0; i < 2; i++)
#pragma unroll
                            for (int k = 0; k < 2; k++) ww[k][i] = Pair<T>::of(w[k].get(i), w[k].get(i));
#pragma unroll
                        for (int h = 0; h < 2; h++) {
                            pairs(rv + 32 * (8 / VT + h * 4 / VT) + n, c);
#pragma unroll
                            for (int j = 0; j < 2; j++)
#pragma unroll
                                for (int i = 0; i < 2; i++) {
                                    A.q[i][2 * h + j] = fma(ww[0][i], c[j], A.q[i][2 * h + j]);
                                    B.q[i][2 * h + j] = fma(ww[1][i], c[j], B.q[i][2 * h + j]);
                                }
                        }
                    }
                }
            };
            int g0 = r.prev, g1 = r.end, g2 = r.wrap;
            if (r.total >= CROWDED_ROW) {   // cells with many particles in this group: by the whole warp
                const int own0 = max(r.mid - c0, 0), own1 = min(r.end - c0, 32);
                unsigned m = __ballot_sync(0xffffffffu, own1 - own0 >= CROWD);
                const int n1 = min(r.nh - c0, 32);
                const bool front = n1 >= CROWD;   // the cell x0 - 1
                if (lane == 0 ? front : (m >> (lane - 1)) & 1) g0 = r.mid;
                if ((m >> lane) & 1) g1 = r.mid;
                if ((m >> (nx - 1)) & 1) g2 = r.total;
                T *sum = xch + (PAR * DROWS + w) * (32 * W);   // this row's part of the exchange, free until the barrier
                if constexpr (sizeof(T) == 8) {   // four cells at a time, the cell x0 - 1 among the first
                    int f = 0;
                    if (front) crowd_sums(0, n1, sum + 8 * W * f++);
                    while (f || m) {
                        unsigned now = m;
                        for (int k = f; m && k < 4; k++) {
                            const int o = __ffs(m) - 1;
                            m &= m - 1;
                            crowd_sums(__shfl_sync(0xffffffffu, own0, o), __shfl_sync(0xffffffffu, own1, o), sum + 8 * W * k);
                        }
                        now &= ~m;
                        __syncwarp();
                        // where this vertex's shares of its own cell and of the one at x - 1 are
                        auto slot = [&](int o) { return (now >> o) & 1 ? f + __popc(now & ((1u << o) - 1)) : -1; };
                        const int own = slot(lane);
                        int prev = lane > 0 ? slot(lane - 1) : f ? 0 : p.cyclic ? slot(nx - 1) : -1;
                        if (lane >= nx) prev = -1;
                        if (own >= 0 || prev >= 0) crowd_add(own >= 0 ? sum + 8 * W * own : sum + 8 * W * prev + 4 * W, A, B);
                        if (own >= 0 && prev >= 0) crowd_add(sum + 8 * W * prev + 4 * W, A, B);
                        __syncwarp();
                        f = 0;
                    }
                } else if (front || m) {   // one at a time: fewer registers
                    int o = -1, e0 = 0, e1 = n1;
                    while (true) {
                        if (o >= 0 || front) {
                            crowd_sums(e0, e1, sum);
                            __syncwarp();
                            const int next = p.cyclic && o == nx - 1 ? 0 : o + 1;
                            if (lane == o || (lane == next && lane < nx)) crowd_add(sum + (lane == o ? 0 : 4 * W), A, B);
                            __syncwarp();
                        }
                        if (!m) break;
                        o = __ffs(m) - 1;
                        m &= m - 1;
                        e0 = __shfl_sync(0xffffffffu, own0, o);
                        e1 = __shfl_sync(0xffffffffu, own1, o);
                    }
                }
            }
            gather(max(g0 - c0, 0), min(g1 - c0, 32), r.mid - c0);
            if (p.cyclic) gather(max(g2 - c0, 0), min(r.total - c0, 32), 32);   // lane 0: the row's last cell
            __syncwarp();
        });
        T *xo = xch + (PAR * DROWS + w) * (32 * W) + lane;
        if (iz >= 0) {   // the sums for the row at y + 1
            const Acc<T> t = A.t00.get(1);
            xo[0] = t.hi();
            if constexpr (sizeof(T) == 4) xo[32] = t.lo();
            if constexpr (FULL) {
#pragma unroll
                for (int j = 0; j < 8; j++) xo[(W - 8 + j) * 32] = A.q[1][j / 2].get(j & 1);
            }
        }
        asm volatile("cp.async.wait_group 1;" ::: "memory");   // the potentials of plane z + 2
        __syncthreads();
        if (iz + 2 < nz) fetch(slot(3), z + 3);   // into the slot of plane z - 2, last read before the barrier
        asm volatile("cp.async.commit_group;" ::: "memory");
        r = rn;
        rn = range(nb);
        if (out) {
            const T *xi = xo - 32 * W;
            Acc<T> S = A.t00.get(0), S2;
            S2.s = xi[0];
            if constexpr (sizeof(T) == 4) S2.c = xi[32];
            acc_merge(S, S2);
            // R: the uniform background a*Omega_m is removed before rounding
            const T dS = (S.hi() - p.rb_hi) + (S.lo() - p.rb_lo);
            const int g = cells + lane;
            if constexpr (DEN) {
                // the contrast N^3 / n_part (S - n_part / N^3) in two words
                S.add(-p.rb_hi);
                const float l = S.lo() - p.rb_lo;
                const float sum = __fadd_rn(S.hi(), l), low = __fsub_rn(l, __fsub_rn(sum, S.hi())), x = __fmul_rn(p.G, sum);
                reinterpret_cast<T *>(p.out.p[0])[g] = x + (__fmaf_rn(p.G, sum, -x) + (p.G * low + p.c1 * sum));
            } else if constexpr (!FULL) {
                reinterpret_cast<T *>(p.out.p[0])[g] = p.G * dS;
            } else {
                T s[8];
#pragma unroll
                for (int j = 0; j < 8; j++) s[j] = A.q[0][j / 2].get(j & 1) + xi[(W - 8 + j) * 32];
                dep_epilogue(p, ring + slot(DRING - 1) * DPN + col, ring + sc * DPN + col, ring + slot(1) * DPN + col, f2, dS,
                             s, g, k0);
            }
        }
        sc = slot(1);
    }
};

// The deposit of tile b of the box described by p.
template <class T, bool FULL, bool DEN = false>
__device__ __forceinline__ void deposit_tile(const DepParams<T> &p, const int b)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const int N = p.N, tid = threadIdx.x, w = tid >> 5;
    using C = DepCol<T, FULL, DEN>;
    C c{p};
    c.stage = reinterpret_cast<typename C::V *>(smem);
    c.rec = reinterpret_cast<T *>(smem + 2 * DEP_THREADS * sizeof(Particle<T>)) + w * (32 * C::R);
    c.xch = reinterpret_cast<T *>(smem + 2 * DEP_THREADS * sizeof(Particle<T>)) + DROWS * (32 * C::R);
    c.ring = c.xch + 2 * DROWS * (32 * C::W);              // phi, chi [DRING][DPN]
    const int x0 = (b % p.ntx) * p.nrow, y0 = ((b / p.ntx) % p.nty) * p.ncol;
    const int nx = min(p.nrow, N - x0), ny = min(p.ncol, N - y0);
    c.z0 = (b / (p.ntx * p.nty)) * p.tz;
    c.nz = min(p.tz, N - c.z0);
    c.nx = w <= ny ? nx : 0;
    c.row = (w <= ny ? wrapi(y0 - 1 + w, N) : 0) * N + x0;
    c.halo = x0 > 0 ? -1 : N - 1;
#pragma unroll
    for (int q = 0; q < 2; q++) {   // entries tid and tid + DEP_THREADS of a plane (nx + 2 columns, ny + 2 rows used)
        const int e = tid + q * DEP_THREADS;
        const int ey = e / DPX, ex = e - ey * DPX;
        c.go[q] = ey < ny + 2 && ex < nx + 2 ? wrapi(y0 - 1 + ey, N) * N + wrapi(x0 - 1 + ex, N) : -1;
    }
    static_assert(DPN <= 2 * DEP_THREADS, "two entries a thread");
    // before the first plane of cells (z0 - 1): planes z0 - 1 .. z0 + 1 of the potentials and its first records
    c.fetch(0, c.z0 - 1);
    c.fetch(1, c.z0);
    c.fetch(2, c.z0 + 1);
    DepRow r = c.range(c.bounds(c.z0 - 1)), rn = c.range(c.bounds(c.z0));
    c.fetch_row(1, r);
    asm volatile("cp.async.commit_group;" ::: "memory");
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    asm volatile("cp.async.commit_group;" ::: "memory");   // an empty group: plane() leaves one pending
    c.sc = 0;
    c.k0.zero();
    RowSums<T> A, B;
    A.zero();
    __syncthreads();
    for (int iz = -1; iz < c.nz; iz += 2) {
        c.template plane<1>(iz, r, rn, A, B);
        if (iz + 1 == c.nz) break;
        c.template plane<0>(iz + 1, r, rn, B, A);
    }

    // k = 0 excess: warp reduction of the (hi, lo) pairs with TwoSum, one FP64 atomic per warp into a slot
    if (!p.newtonian) {
        const Acc<T> k0 = warp_sum(c.k0);
        if ((tid & 31) == 0)
            atomicAdd(&p.k0slots[(blockIdx.x * DROWS + w) & (NK0SLOTS - 1)], (double)k0.hi() + (double)k0.lo());
    }
}

template <class T, bool FULL> constexpr int dep_ctas() { return sizeof(T) == 4 ? (FULL ? 2 : 3) : (FULL ? 1 : 2); }

template <class T, bool FULL>
__global__ void __launch_bounds__(DEP_THREADS, dep_ctas<T, FULL>()) k_project(const __grid_constant__ DepParams<T> p)
{
    deposit_tile<T, FULL>(p, blockIdx.x);
}

// The CIC density contrast of the P(k) diagnostic in FP32 contexts: the columns above with the weights and the sums
// in two words.  In place of FP64 weights and atomics on the FP64 pipe: 256^3 at z = 3 0.98 (with clearing and the
// final pass) -> 0.48 ms.  FP64 contexts take k_density_acc.
__global__ void __launch_bounds__(DEP_THREADS, 2) k_contrast(const __grid_constant__ DepParams<float> p)
{
    deposit_tile<float, false, true>(p, blockIdx.x);
}

// Several boxes in one launch (the batched ensemble): CTA j deposits tile j - first[i] of box i, the box whose
// range [first[i], first[i+1]) holds j.  The boxes' parameters travel by value in the kernel's parameter space.
constexpr int MAXBATCH = 48;
template <class T> struct DepBatch {
    int nbox;
    int first[MAXBATCH + 1];
    DepParams<T> box[MAXBATCH];
};
static_assert(sizeof(DepBatch<double>) < 32000, "kernel parameter space");

template <class T, bool FULL>
__global__ void __launch_bounds__(DEP_THREADS, dep_ctas<T, FULL>()) k_project_batch(const __grid_constant__ DepBatch<T> q)
{
    int i = 0;
    while (i + 1 < q.nbox && (int)blockIdx.x >= q.first[i + 1]) i++;
    deposit_tile<T, FULL>(q.box[i], (int)blockIdx.x - q.first[i]);
}

template <class I>
__global__ void __launch_bounds__(MTHREADS, 4) k_mass_batch(const __grid_constant__ DepBatch<float> q)
{
    int i = 0;
    while (i + 1 < q.nbox && (int)blockIdx.x >= q.first[i + 1]) i++;
    mass_tile<I>(q.box[i], (int)blockIdx.x - q.first[i]);
}

// ---------------------------------------------------------------------------
// Gather + kick + drift (Eqs. kick, drift to first order, Sec. 3.1):
//   du_i/dtau = -E d_i psi - (u^2/E) d_i phi - u_j d_i B_j,  E = sqrt(a_n^2 + u^2)
//   dx^i/dtau = (u_i/E')(1 + 3 phi - chi - phi u'^2/E'^2) + B_i,  E' at a_{n+1/2}
// with mesh gradients (f(x+dx) - f(x-dx)) / (2 dx) interpolated by CIC, i.e. a
// 4x2x2 stencil per direction.  Newtonian mode: du = -a grad phi, dx = u/a.
// The new cell of each particle is counted for the sort.
// ---------------------------------------------------------------------------
template <class T> struct KdParams {
    Particle<T> *part;
    const int32_t *start;
    int32_t *count;
    const T *phi, *chi, *Bx, *By, *Bz;
    int N;
    int nrow, ntx, tz;   // cells of a tile along x, tiles along x, cells along z
    T a, a2, a_half2, inv_a_half, dt_kick, dt_drift_N, halfN;
    T kick_N;            // dt_kick N/2
    const float *corr;   // force correction [cell][8] (CORR)
    T corr_scale;
};

// A CTA owns the cells [x0, x0 + nrow) x [y0, y0 + 8) x [z0, z0 + tz) and marches along z; warp w takes the row of
// cells y0 + w, whose particles are consecutive in memory, one per lane.  The fields on the plane's vertices
// [x0 - 1, x0 + nrow + 1] x [y0 - 1, y0 + 9] and the planes z - 1 .. z + 2 sit in a ring of five, one plane of which
// is loaded while the warps work on the plane before.
// What bounds it: the shared-memory pipe (a particle reads 32 vertices of 20 bytes, 5 of its 8 wavefronts) and, in
// FP64, the FP64 pipe.  Against 8^3 tiles of 11^3 vertices, one search and three integer divisions per particle, and
// the gradients of five fields kept in 20 registers (512^3 mixed 5.15 ms, 256^3 FP64 14.0, 288^3 Newtonian 0.52):
// 3.55 ms, 8.8, 0.30.  Rows that hold more than 32 particles make their CTA's other warps wait where they are not shared
// (192^3 at z = 1: 0.33 -> 0.35).  Two planes between barriers, records staged in shared memory instead of registers, four CTAs of 64
// registers an SM, two of 128: 0.58, 0.48, 0.61, 0.52 ms against 0.46 at 256^3 (the first two take L1 from the loads).
constexpr int KROWS = 8, KD_THREADS = 32 * KROWS;
constexpr int KPX = 32 + 3, KPN = KPX * (KROWS + 3);   // vertices of a plane
constexpr int KRING = 5;
constexpr int KUNEVEN = 96;   // FP32: particles of a row from which its tile's warps share their rows
constexpr int KLD = (KPN + KD_THREADS - 1) / KD_THREADS;   // vertices of a plane per thread

// phi, chi, B_x, B_y of one vertex in one 16-byte (FP32) or two 16-byte (FP64) loads
template <class T> struct alignas(4 * sizeof(T) >= 16 ? 16 : 4 * sizeof(T)) Vtx4 {
    T phi, chi, bx, by;
};

template <class T, bool NEWT> constexpr size_t kd_smem()
{
    return KRING * KPN * sizeof(T) * (NEWT ? 1 : 5);
}

// Accumulate the centred-difference gradient of one vertex value s at stencil offset (kx, ky, kz) in {0..3}^3
// (offset -1 .. +2 from the cell); terms whose weight is identically zero are skipped at compile time.
template <int kx, int ky, int kz, class T>
__device__ __forceinline__ void stencil_acc(T s, const T *Wx, const T *Wy, const T *Wz, const T *Gx, const T *Gy,
                                            const T *Gz, T (&g)[3])
{
    constexpr bool cx = (kx == 1 || kx == 2), cy = (ky == 1 || ky == 2), cz = (kz == 1 || kz == 2);
    if constexpr (cy && cz) g[0] += Gx[kx] * (Wy[ky] * Wz[kz]) * s;
    if constexpr (cx && cz) g[1] += Gy[ky] * (Wx[kx] * Wz[kz]) * s;
    if constexpr (cx && cy) g[2] += Gz[kz] * (Wx[kx] * Wy[ky]) * s;
}

// Newtonian: the gradient of phi from the vertex planes pl[kz] (at stencil offset (0, 0)), vertex by vertex
template <int I, class T>
__device__ __forceinline__ void gather_phi(const T *const (&pl)[4], const T *Wx, const T *Wy, const T *Wz, const T *Gx,
                                           const T *Gy, const T *Gz, T (&g)[3])
{
    if constexpr (I < 64) {
        constexpr int kx = I % 4, ky = (I / 4) % 4, kz = I / 16;
        constexpr bool cx = (kx == 1 || kx == 2), cy = (ky == 1 || ky == 2), cz = (kz == 1 || kz == 2);
        if constexpr ((int)!cx + (int)!cy + (int)!cz <= 1)
            stencil_acc<kx, ky, kz>(pl[kz][kx + KPX * ky], Wx, Wy, Wz, Gx, Gy, Gz, g);
        gather_phi<I + 1>(pl, Wx, Wy, Wz, Gx, Gy, Gz, g);
    }
}

// The relativistic gather.  The kick is minus the gradient of one scalar,
//   s = (E + u^2/E) phi - E chi + u_j B_j      (coefficients c[5] of phi, chi, B of this particle),
// so each of the 32 stencil vertices is first reduced to s (5 products) and only s is differenced and
// interpolated, axis by axis (68 operations instead of the 280 of five fields' three gradients, and 3 sums
// instead of 15).  FP64 takes s/E in 4 operations a vertex, the small terms first, and multiplies the gradient by E:
// 256^3 11.1 -> 8.8 ms, with carry_cells().  FP32 does not miss the operation and was slower with each order of the
// four (0.46 -> 0.48 to 0.53 ms at 256^3).  g: 2 dx grad s (s/E); val: phi, chi, B at the particle.
template <class T>
__device__ __forceinline__ void gather_s(const Vtx4<T> *const (&sv)[4], const T *const (&sb)[4], const T (&c)[5], T fx, T fy,
                                         T fz, T (&g)[3], T (&val)[5])
{
    const T gx = T(1) - fx, gy = T(1) - fy, gz = T(1) - fz;
    // scalar at vertex (kx, ky) of plane kz; at the 8 corners of the cell the fields' values gather, too
    auto at = [&](int kz, int v, T w, bool corner) {
        const Vtx4<T> a = sv[kz][v];
        const T b = sb[kz][v];
        if (corner) {
            val[0] += w * a.phi;
            val[1] += w * a.chi;
            val[2] += w * a.bx;
            val[3] += w * a.by;
            val[4] += w * b;
        }
        if constexpr (sizeof(T) == 8) return c[0] * a.phi + (c[4] * b + (c[3] * a.by + (c[2] * a.bx - a.chi)));
        else return c[0] * a.phi + c[1] * a.chi + (c[2] * a.bx + c[3] * a.by + c[4] * b);
    };
    auto line = [&](int kz, int v) {   // interpolated along x between kx = 1 and 2 (v: the vertex at kx = 1)
        const T s1 = at(kz, v, T(0), false), s2 = at(kz, v + 1, T(0), false);
        return s1 + fx * (s2 - s1);
    };
    T pz[4], px[2], py[2];   // per plane: s; its difference along x; along y
#pragma unroll
    for (int kz = 0; kz < 4; kz++) {
        if (kz == 0 || kz == 3) {
            const T v1 = line(kz, 1 + KPX), v2 = line(kz, 1 + 2 * KPX);
            pz[kz] = v1 + fy * (v2 - v1);
            continue;
        }
        const T wz = kz == 1 ? gz : fz;
        T v[4], d[2];
        v[0] = line(kz, 1);
        v[3] = line(kz, 1 + 3 * KPX);
#pragma unroll
        for (int ky = 1; ky < 3; ky++) {
            const T wyz = (ky == 1 ? gy : fy) * wz;
            const T s0 = at(kz, KPX * ky, T(0), false), s1 = at(kz, KPX * ky + 1, gx * wyz, true),
                    s2 = at(kz, KPX * ky + 2, fx * wyz, true), s3 = at(kz, KPX * ky + 3, T(0), false);
            const T a = s2 - s0, b = s3 - s1;
            v[ky] = s1 + fx * (s2 - s1);
            d[ky - 1] = a + fx * (b - a);
        }
        pz[kz] = v[1] + fy * (v[2] - v[1]);
        px[kz - 1] = d[0] + fy * (d[1] - d[0]);
        const T a = v[2] - v[0], b = v[3] - v[1];
        py[kz - 1] = a + fy * (b - a);
    }
    g[0] = px[0] + fz * (px[1] - px[0]);
    g[1] = py[0] + fz * (py[1] - py[0]);
    const T a = pz[2] - pz[0], b = pz[3] - pz[1];
    g[2] = a + fz * (b - a);
}

// u += dtau_kick a c(x_p) of a force correction c, interpolated by CIC: k_corr_kick's arithmetic in the Newtonian mode
template <class T>
__device__ __forceinline__ void add_correction(const KdParams<T> &p, int x, int y, int z, T fx, T fy, T fz, T (&u)[3])
{
    const int n = p.N;
    const int xp = x + 1 == n ? 0 : x + 1, yp = y + 1 == n ? 0 : y + 1, zp = z + 1 == n ? 0 : z + 1;
    const T wx[2] = {T(1) - fx, fx}, wy[2] = {T(1) - fy, fy}, wz[2] = {T(1) - fz, fz};
    T cv[3] = {0, 0, 0};
#pragma unroll
    for (int dz = 0; dz < 2; dz++)
#pragma unroll
        for (int dy = 0; dy < 2; dy++) {
            const T wyz = wy[dy] * wz[dz];
            const int row = ((dz ? zp : z) * n + (dy ? yp : y)) * n;
#pragma unroll
            for (int dx = 0; dx < 2; dx++) {
                const T w = wx[dx] * wyz;
                const float4 c4 = __ldg(reinterpret_cast<const float4 *>(p.corr) + 2 * ((int64_t)row + (dx ? xp : x)));
                cv[0] += w * (T)c4.x;
                cv[1] += w * (T)c4.y;
                cv[2] += w * (T)c4.z;
            }
        }
    const T f = p.a * p.corr_scale;
#pragma unroll
    for (int k = 0; k < 3; k++) u[k] += p.dt_kick * f * cv[k];
}

// An offset v that left its cell in FP64: f = v - floor(v) (0 and the next cell where that rounds to 1), carry the
// cells crossed.  3 FP64 additions instead of floor, two comparisons and two conversions, all of which take the FP64
// pipe: v + 1.5 2^52, rounded down, holds floor(v) in its low word.  False (f and carry of no use) at N cells or more.
__device__ __forceinline__ bool carry_cells(double v, int N, double &f, int &carry)
{
    const double M = 6755399441055744.0;   // 1.5 2^52
    const double r = __dadd_rd(v, M), g = v - (r - M);
    const int lo = __double2loint(r), hi = __double2hiint(g) & 0x7fffffff;   // no -0
    const bool one = hi >= 0x3ff00000;
    f = __hiloint2double(one ? 0 : hi, one ? 0 : __double2loint(g));
    carry = lo + one;
    return __double2hiint(r) == 0x43380000 + (lo >> 31) && lo < N && lo > -N;
}
__device__ __forceinline__ bool carry_cells(float, int, float &, int &) { return false; }

// The particles of the rows of cells of a plane, for the warps to share in groups of 32 where a row has more than 32, or
// all rows so few that most lanes would be idle.  FP64, where an instruction takes the pipe as long for one lane as for 32,
// always keeps this table (128^3, own rows and shared ones: z = 1 1.89 -> 1.46 ms, half a particle a cell 1.21 -> 0.72,
// 0.05 0.98 -> 0.36, a tenth of the mass in cells of 1000 2.39 -> 1.44; from 192 particles a plane on, 6 of 8 full groups,
// there is nothing to gain).  FP32 is slower with it at one particle a cell (256^3 0.46 -> 0.52), so only the relativistic
// kernel takes it, in tiles with a row of more than KUNEVEN (128^3, clumps as above 0.196 -> 0.110, of 300 0.157 -> 0.106,
// 192^3 at z = 1 0.358 -> 0.349); to look for one costs the other tiles 2% (512^3 3.47 -> 3.55).  In the Newtonian kernel,
// half as long, both forms together spill and cost 19%.
struct alignas(16) KickRows {
    int end[KROWS];   // particles of the rows up to this one
    int off[KROWS];   // particle j of all rows' is off[its row] + j
    int shared;       // the warps share them

    // by a whole warp, whose lane l < KROWS has row l's particles s .. e - 1
    __device__ __forceinline__ void set(int s, int e)
    {
        const int lane = threadIdx.x & 31, n = lane < KROWS ? e - s : 0;
        int sum = n;
#pragma unroll
        for (int o = 1; o < KROWS; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, sum, o);
            if (lane >= o) sum += v;
        }
        const bool full = __any_sync(0xffffffffu, n > 32);
        if (lane < KROWS) {
            end[lane] = sum;
            off[lane] = e - sum;
        }
        if (lane == KROWS - 1) shared = full || sum <= 24 * KROWS;
    }
    // particle j of all rows' and its row; i = -1: none
    __device__ __forceinline__ void find(unsigned j, int &i, int &r) const
    {
        const int4 a = *reinterpret_cast<const int4 *>(end), b = *reinterpret_cast<const int4 *>(end + 4);
        r = (j >= (unsigned)a.x) + (j >= (unsigned)a.y) + (j >= (unsigned)a.z) + (j >= (unsigned)a.w) +
            (j >= (unsigned)b.x) + (j >= (unsigned)b.y) + (j >= (unsigned)b.z);
        i = j < (unsigned)b.w ? off[r] + (int)j : -1;
    }
    // a lane's first particle: `group` 32 of all rows' where they are shared
    __device__ __forceinline__ void first(int w, int group, int &i, int &r) const
    {
        if (shared) {
            find(32 * group + (threadIdx.x & 31), i, r);
        } else {
            const int j = (w > 0 ? end[w - 1] : 0) + (threadIdx.x & 31);
            r = w;
            i = j < end[w] ? off[w] + j : -1;
        }
    }
};
static_assert(KROWS == 8, "find() compares with 7 ends");

// CORR: with the force correction of a Newtonian context.  SHARED: with a table of the rows
template <class T, bool NEWT, bool CORR, bool SHARED>
__device__ __forceinline__ void kick_tile(const KdParams<T> &p, const int b)
{
    extern __shared__ __align__(16) unsigned char smem[];
    constexpr bool FP64 = sizeof(T) == 8;
    constexpr int PQ = sizeof(Particle<T>) / 16;
    using V = std::conditional_t<FP64, double2, float4>;
    T *ring = reinterpret_cast<T *>(smem);
    Vtx4<T> *sv = reinterpret_cast<Vtx4<T> *>(ring);                           // [KRING][KPN]
    T *sb = NEWT ? ring : ring + 4 * KRING * KPN;                              // B_z (Newtonian: phi) [KRING][KPN]
    const int N = p.N, tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const int x0 = (b % p.ntx) * p.nrow, y0 = ((b / p.ntx) % (N / KROWS)) * KROWS, z0 = b / (p.ntx * (N / KROWS)) * p.tz;
    const int nx = min(p.nrow, N - x0), nz = min(p.tz, N - z0);

    // this thread's vertices of a plane: where they come from (-1: none)
    int go[KLD];
#pragma unroll
    for (int q = 0; q < KLD; q++) {
        const int e = tid + q * KD_THREADS, ey = e / KPX, ex = e - ey * KPX;
        go[q] = e < KPN && ex < nx + 3 ? wrapi(y0 - 1 + ey, N) * N + wrapi(x0 - 1 + ex, N) : -1;
    }
    Vtx4<T> va[NEWT ? 1 : KLD];
    T vb[KLD];
    auto load = [&](int z) {
        const int base = wrapi(z, N) * (N * N);
#pragma unroll
        for (int q = 0; q < KLD; q++)
            if (go[q] >= 0) {
                const int g = base + go[q];
                if constexpr (NEWT) {
                    vb[q] = __ldg(p.phi + g);
                } else {
                    va[q].phi = __ldg(p.phi + g);
                    va[q].chi = __ldg(p.chi + g);
                    va[q].bx = __ldg(p.Bx + g);
                    va[q].by = __ldg(p.By + g);
                    vb[q] = __ldg(p.Bz + g);
                }
            }
    };
    auto keep = [&](int slot) {
#pragma unroll
        for (int q = 0; q < KLD; q++)
            if (go[q] >= 0) {
                if constexpr (!NEWT) sv[slot * KPN + tid + q * KD_THREADS] = va[q];
                sb[slot * KPN + tid + q * KD_THREADS] = vb[q];
            }
    };
    for (int i = 0; i < 4; i++) {   // planes z0 - 1 .. z0 + 2
        load(z0 - 1 + i);
        keep(i);
    }
    const int32_t *st = p.start + z0 * (N * N) + y0 * N + x0;
    __shared__ KickRows rows[SHARED ? 4 : 1];
    // this lane's first particle of a plane, fetched a plane ahead
    V nxt[PQ];
    auto fetch = [&](int i) {
#pragma unroll
        for (int q = 0; q < PQ; q++) nxt[q] = reinterpret_cast<const V *>(p.part + i)[q];
    };
    int i0 = -1, r0 = w;                  // SHARED: that particle and its row
    int s0 = 0, e0 = 0, s1 = 0, e1 = 0;   // else this warp's row in this plane and the next
    if constexpr (SHARED) {   // the rows of a plane are counted two planes ahead, by a warp after the other
        const int32_t *q = st + w * (N * N) + (lane % KROWS) * N;
        if (w < 2 && w < nz) rows[w].set(__ldg(q), __ldg(q + nx));
        __syncthreads();
        rows[0].first(w, (w + z0) % KROWS, i0, r0);
        if (i0 >= 0) fetch(i0);
    } else {
        const int32_t *q = st + w * N;
        s0 = __ldg(q);
        e0 = __ldg(q + nx);
        if (nz > 1) {
            s1 = __ldg(q + N * N);
            e1 = __ldg(q + N * N + nx);
        }
        if (lane < e0 - s0) fetch(s0 + lane);
        __syncthreads();
    }

    int sc = 0;   // slot of plane z - 1
    for (int iz = 0; iz < nz; iz++) {
        const int z = z0 + iz;
        if (iz + 1 < nz) load(z + 3);
        const bool ahead = iz + 2 < nz && (!SHARED || w == iz % KROWS);
        int s2 = 0, e2 = 0;
        if (ahead) {
            const int32_t *q = st + (iz + 2) * (N * N) + (SHARED ? lane % KROWS : w) * N;
            s2 = __ldg(q);
            e2 = __ldg(q + nx);
        }
        V rec[PQ];
#pragma unroll
        for (int q = 0; q < PQ; q++) rec[q] = nxt[q];
        int i = i0, r = r0;
        if constexpr (SHARED) {
            i0 = -1;
            if (iz + 1 < nz) rows[(iz + 1) % 4].first(w, (w + z + 1) % KROWS, i0, r0);
            if (i0 >= 0) fetch(i0);
        } else {
            if (lane < e1 - s1) fetch(s1 + lane);
        }
        auto record = [&](int i) {
#pragma unroll
            for (int q = 0; q < PQ; q++) rec[q] = reinterpret_cast<const V *>(p.part + i)[q];
        };
        // particle i, in row r
        auto move = [&](int i, int r) {
            Particle<T> P = *reinterpret_cast<const Particle<T> *>(rec);
            const int cx = P.cell - (z * (N * N) + (y0 + r) * N + x0);
            const int vo = r * KPX + cx;   // vertex at stencil offset (0, 0) in its plane
            const T fx = P.f[0], fy = P.f[1], fz = P.f[2];
            T u[3] = {P.u[0], P.u[1], P.u[2]};
            T dx[3];
            int slot[4];
#pragma unroll
            for (int k = 0; k < 4; k++) slot[k] = (sc + k >= KRING ? sc + k - KRING : sc + k) * KPN + vo;
            const T *const pb[4] = {sb + slot[0], sb + slot[1], sb + slot[2], sb + slot[3]};
            if constexpr (CORR) add_correction(p, x0 + cx, y0 + r, z, fx, fy, fz, u);
            if constexpr (NEWT) {
                const T hn = p.halfN;
                const T Wx[4] = {0, T(1) - fx, fx, 0}, Wy[4] = {0, T(1) - fy, fy, 0}, Wz[4] = {0, T(1) - fz, fz, 0};
                const T Gx[4] = {-(T(1) - fx) * hn, -fx * hn, (T(1) - fx) * hn, fx * hn};
                const T Gy[4] = {-(T(1) - fy) * hn, -fy * hn, (T(1) - fy) * hn, fy * hn};
                const T Gz[4] = {-(T(1) - fz) * hn, -fz * hn, (T(1) - fz) * hn, fz * hn};
                T grd[3] = {0, 0, 0};
                gather_phi<0>(pb, Wx, Wy, Wz, Gx, Gy, Gz, grd);
#pragma unroll
                for (int d = 0; d < 3; d++) u[d] -= p.dt_kick * p.a * grd[d];
#pragma unroll
                for (int d = 0; d < 3; d++) dx[d] = mulr(mulr(p.dt_drift_N, u[d]), p.inv_a_half);   // no FMA with the offset
            } else {
                const T u2 = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
                const T e2 = p.a2 + u2;
                const T iE = rsqrt_t(e2);
                const T E = e2 * iE, by = sizeof(T) == 8 ? iE : T(1);
                const T c[5] = {sizeof(T) == 8 ? T(1) + u2 * (iE * iE) : E + u2 * iE, -E, u[0] * by, u[1] * by, u[2] * by};
                const Vtx4<T> *const pv[4] = {sv + slot[0], sv + slot[1], sv + slot[2], sv + slot[3]};
                T val[5] = {0, 0, 0, 0, 0}, g[3];
                gather_s(pv, pb, c, fx, fy, fz, g, val);
                const T dtk = sizeof(T) == 8 ? p.kick_N * E : p.kick_N;
#pragma unroll
                for (int d = 0; d < 3; d++) u[d] -= dtk * g[d];
                const T v2 = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
                const T iEd = rsqrt_t(p.a_half2 + v2);
                // (1 + (3 - v^2/E^2) phi - chi) / E, v^2 = E^2 - a^2
                const T fac = ((T(1) - val[1]) + val[0] * (T(2) + p.a_half2 * (iEd * iEd))) * iEd;
#pragma unroll
                for (int d = 0; d < 3; d++) dx[d] = p.dt_drift_N * (u[d] * fac + val[2 + d]);
            }
            const T fo[3] = {fx, fy, fz};
            const int io[3] = {x0 + cx, y0 + r, z};
            int inew[3];
            bool near = sizeof(T) == 8;
            if constexpr (sizeof(T) == 8) {
#pragma unroll
                for (int d = 0; d < 3; d++) {
                    int carry;
                    near &= carry_cells(fo[d] + dx[d], N, P.f[d], carry);
                    inew[d] = wrapi(io[d] + carry, N);   // |carry| <= N
                }
            }
            if (!near) {
#pragma unroll
                for (int d = 0; d < 3; d++) {
                    T f = fo[d] + dx[d];
                    T fl = floor(f);
                    f -= fl;
                    // a finite move is far below N cells; anything else (NaN, Inf) keeps the cell
                    int carry = (fabs(fl) < (T)N) ? (int)fl : 0;
                    if (f >= T(1)) {
                        f = T(0);
                        carry += 1;
                    }
                    inew[d] = wrapi(io[d] + carry, N);   // |carry| <= N
                    P.f[d] = f;
                }
            }
#pragma unroll
            for (int d = 0; d < 3; d++) P.u[d] = u[d];
            P.cell = (inew[2] * N + inew[1]) * N + inew[0];
            p.part[i] = P;
            atomicAdd(&p.count[P.cell], 1);
        };
        if constexpr (SHARED) {
            const KickRows &now = rows[iz % 4];
            for (unsigned c = 32 * ((unsigned)(w + z) % KROWS);;) {
                if (i >= 0) move(i, r);
                if (!now.shared || (c += 32 * KROWS) >= (unsigned)now.end[KROWS - 1]) break;
                now.find(c + lane, i, r);
                if (i >= 0) record(i);
            }
            if (ahead) rows[(iz + 2) % 4].set(s2, e2);
        } else {
            // (unsigned: a particle number plus 32 can pass 2^31 - 1)
            for (unsigned k = (unsigned)s0 + lane; k < (unsigned)e0; k += 32) {
                if (k >= (unsigned)s0 + 32) record(k);
                move(k, w);
            }
        }
        // plane z + 3 into the slot of plane z - 2, last read before the barrier of the plane before
        if (iz + 1 < nz) keep(sc + 4 >= KRING ? sc + 4 - KRING : sc + 4);
        __syncthreads();
        if constexpr (!SHARED) {
            s0 = s1;
            e0 = e1;
            s1 = s2;
            e1 = e2;
        }
        sc = sc + 1 == KRING ? 0 : sc + 1;
    }
}

// Whether a row of the tile has more than KUNEVEN particles, for the whole CTA.
template <class T> __device__ __forceinline__ bool kick_uneven(const KdParams<T> &p, const int b)
{
    const int N = p.N, x0 = (b % p.ntx) * p.nrow, y0 = ((b / p.ntx) % (N / KROWS)) * KROWS, z0 = b / (p.ntx * (N / KROWS)) * p.tz;
    const int nx = min(p.nrow, N - x0), nz = min(p.tz, N - z0);
    int most = 0;
    for (int r = threadIdx.x; r < KROWS * nz; r += KD_THREADS) {
        const int32_t *q = p.start + ((z0 + r / KROWS) * N + y0 + r % KROWS) * N + x0;
        most = max(most, __ldg(q + nx) - __ldg(q));
    }
    return __syncthreads_or(most > KUNEVEN);
}

template <class T, bool NEWT, bool CORR = false>
__device__ __forceinline__ void kick_cells(const KdParams<T> &p, const int b)
{
    if constexpr (sizeof(T) == 8) kick_tile<T, NEWT, CORR, true>(p, b);
    else if constexpr (NEWT) kick_tile<T, NEWT, CORR, false>(p, b);
    else if (kick_uneven(p, b)) kick_tile<T, NEWT, CORR, true>(p, b);
    else kick_tile<T, NEWT, CORR, false>(p, b);
}

// CTAs an SM holds: the relativistic FP32 kernel needs 80 registers, the Newtonian one 64, FP64 128
template <class T, bool NEWT> constexpr int kd_ctas() { return sizeof(T) == 4 ? (NEWT ? 4 : 3) : 2; }

template <class T, bool NEWT>
__global__ void __launch_bounds__(KD_THREADS, kd_ctas<T, NEWT>()) k_kick_drift(const __grid_constant__ KdParams<T> p)
{
    kick_cells<T, NEWT>(p, blockIdx.x);
}

// The Newtonian kick with a force correction: one pass over the particles instead of k_corr_kick's before it
// (256^3 mixed, both kicks: 0.50 -> 0.42 ms).
template <class T>
__global__ void __launch_bounds__(KD_THREADS, sizeof(T) == 4 ? 3 : 2) k_kick_corrected(const __grid_constant__ KdParams<T> p)
{
    kick_cells<T, true, true>(p, blockIdx.x);
}

template <class T> struct KdBatch {
    int nbox;
    int first[MAXBATCH + 1];
    KdParams<T> box[MAXBATCH];
};
static_assert(sizeof(KdBatch<double>) < 32000, "kernel parameter space");

template <class T, bool NEWT>
__global__ void __launch_bounds__(KD_THREADS, kd_ctas<T, NEWT>()) k_kick_batch(const __grid_constant__ KdBatch<T> q)
{
    int i = 0;
    while (i + 1 < q.nbox && (int)blockIdx.x >= q.first[i + 1]) i++;
    kick_cells<T, NEWT>(q.box[i], (int)blockIdx.x - q.first[i]);
}

// ---------------------------------------------------------------------------
// Counting sort by cell: exclusive scan of the per-cell counts, then scatter.
// The scan takes two passes over the counts.  A scan tile is SCAN_ROUNDS rounds of one 16-byte
// vector per thread; a round covers 4 * SCAN_T consecutive counts, so each warp load and store is
// 512 contiguous bytes.  The first pass writes each tile's sum.  The second reads its tile again,
// adds up the sums of the tiles before it (32 KB at 512^3, read from L2 in 16-byte vectors) and
// writes the exclusive offsets; the last tile also writes the total.
// ---------------------------------------------------------------------------
constexpr int SCAN_T = 1024, SCAN_ROUNDS = 4;
constexpr int SCAN_TILE = SCAN_T * 4 * SCAN_ROUNDS;

// The four counts at cnt[base .. base + 4), zero past n; base is a multiple of 4 (16-byte aligned).
__device__ __forceinline__ int4 scan_load4(const int32_t *cnt, int64_t n, int64_t base)
{
    int4 q = make_int4(0, 0, 0, 0);
    if (base + 4 <= n) {
        q = *reinterpret_cast<const int4 *>(cnt + base);
    } else {
        if (base < n) q.x = cnt[base];
        if (base + 1 < n) q.y = cnt[base + 1];
        if (base + 2 < n) q.z = cnt[base + 2];
    }
    return q;
}

__global__ void __launch_bounds__(SCAN_T) k_scan_reduce(const int32_t *cnt, int64_t n, int32_t *bsum)
{
    __shared__ int wsum[SCAN_T / 32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int64_t t0 = (int64_t)blockIdx.x * SCAN_TILE + 4 * (int64_t)threadIdx.x;
    int4 q[SCAN_ROUNDS];
#pragma unroll
    for (int r = 0; r < SCAN_ROUNDS; r++) q[r] = scan_load4(cnt, n, t0 + (int64_t)r * 4 * SCAN_T);
    int s = 0;
#pragma unroll
    for (int r = 0; r < SCAN_ROUNDS; r++) s += q[r].x + q[r].y + q[r].z + q[r].w;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) wsum[wid] = s;
    __syncthreads();
    if (wid == 0) {
        int t = wsum[lane];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        if (lane == 0) bsum[blockIdx.x] = t;
    }
}

__global__ void __launch_bounds__(SCAN_T, 2) k_scan_down(const int32_t *cnt, int64_t n, const int32_t *bsum,
                                                       int32_t *start)
{
    static_assert(SCAN_T == 1024, "32 warps: one lane of warp 0 per warp");
    __shared__ int wex[SCAN_ROUNDS][SCAN_T / 32];   // exclusive offset of each warp in each round
    __shared__ int wpre[SCAN_T / 32];
    __shared__ int tile_end;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int tile = (int)blockIdx.x;
    const int64_t t0 = (int64_t)tile * SCAN_TILE + 4 * (int64_t)threadIdx.x;
    int v[SCAN_ROUNDS], inc[SCAN_ROUNDS];
#pragma unroll
    for (int r = 0; r < SCAN_ROUNDS; r++) {
        const int4 q = scan_load4(cnt, n, t0 + (int64_t)r * 4 * SCAN_T);
        inc[r] = v[r] = q.x + q.y + q.z + q.w;
    }
    // this thread's share of the sums of tiles 0 .. tile-1
    int pre = 0;
    const int nv = tile >> 2;
    for (int i = (int)threadIdx.x; i < nv; i += SCAN_T) {
        const int4 b = reinterpret_cast<const int4 *>(bsum)[i];
        pre += b.x + b.y + b.z + b.w;
    }
    if ((int)threadIdx.x < (tile & 3)) pre += bsum[4 * nv + (int)threadIdx.x];
    // inclusive warp scans of the thread sums of every round, and the warp sum of pre
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
#pragma unroll
        for (int r = 0; r < SCAN_ROUNDS; r++) {
            const int y = __shfl_up_sync(0xffffffffu, inc[r], o);
            if (lane >= o) inc[r] += y;
        }
        pre += __shfl_xor_sync(0xffffffffu, pre, o);
    }
    if (lane == 31) {
#pragma unroll
        for (int r = 0; r < SCAN_ROUNDS; r++) wex[r][wid] = inc[r];
    }
    if (lane == 0) wpre[wid] = pre;
    __syncthreads();
    if (wid == 0) {
        int w[SCAN_ROUNDS], z[SCAN_ROUNDS];
#pragma unroll
        for (int r = 0; r < SCAN_ROUNDS; r++) z[r] = w[r] = wex[r][lane];
        int p = wpre[lane];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
#pragma unroll
            for (int r = 0; r < SCAN_ROUNDS; r++) {
                const int y = __shfl_up_sync(0xffffffffu, z[r], o);
                if (lane >= o) z[r] += y;
            }
            p += __shfl_xor_sync(0xffffffffu, p, o);
        }
        // round r starts after the tiles before this one and after rounds 0 .. r-1 of this tile
        int carry = p;
#pragma unroll
        for (int r = 0; r < SCAN_ROUNDS; r++) {
            wex[r][lane] = carry + z[r] - w[r];
            carry += __shfl_sync(0xffffffffu, z[r], 31);
        }
        if (lane == 0) tile_end = carry;
    }
    __syncthreads();
    // the counts again (from L1: this CTA read them above), to keep two CTAs of registers per SM
#pragma unroll
    for (int r = 0; r < SCAN_ROUNDS; r++) {
        const int64_t base = t0 + (int64_t)r * 4 * SCAN_T;
        const int4 q = scan_load4(cnt, n, base);
        const int e = wex[r][wid] + inc[r] - v[r];
        const int4 o = make_int4(e, e + q.x, e + q.x + q.y, e + q.x + q.y + q.z);
        if (base + 4 <= n) {
            *reinterpret_cast<int4 *>(start + base) = o;
        } else {
            if (base < n) start[base] = o.x;
            if (base + 1 < n) start[base + 1] = o.y;
            if (base + 2 < n) start[base + 2] = o.z;
        }
    }
    if (tile == (int)gridDim.x - 1 && threadIdx.x == 0) start[n] = tile_end;
}

template <class T>
__global__ void __launch_bounds__(256) k_scatter(const Particle<T> *in, Particle<T> *out, int64_t np,
                                                 const int32_t *start, int32_t *count)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= np) return;
    const Particle<T> P = in[i];
    const int r = atomicSub(&count[P.cell], 1) - 1;
    out[start[P.cell] + r] = P;
}

// ---------------------------------------------------------------------------
// f64 <-> f32 conversions, integer parts and fractions on the integer pipes.  The FP64 pipe, which also runs the
// conversion instructions, takes 16 cycles a warp instruction here: with them the load spent 1.02 ms on
// 256^3 particles and the store 0.46, with these 0.23 and 0.21 (the bytes take 0.20).  Every result is the one of
// the FP64 instructions, rounded to nearest even; what is not in the common range takes those, out of line, since
// the compiler would otherwise run both and select.
// ---------------------------------------------------------------------------
__device__ __noinline__ double position_any(int c, float f, double inv_n) { return ((double)c + (double)f) * inv_n; }
__device__ __noinline__ double wrap_unit(double x)
{
    if (!isfinite(x)) x = 0.0;   // keeps the cell index valid; the caller rejects the input
    x -= floor(x);
    return x >= 1.0 ? 0.0 : x;
}

// Integer part (returned) and fraction of s in [0, 2^10].
__device__ __forceinline__ int split(double s, double &f)
{
    const uint64_t b = (uint64_t)__double_as_longlong(s);
    const int e = (int)(b >> 52) - 1023;
    if (e < 0) {
        f = s;
        return 0;
    }
    const uint64_t m = (b & 0xfffffffffffffull) | 0x10000000000000ull;
    const uint64_t r = m & ((0x10000000000000ull >> e) - 1);   // the fraction is r 2^(e - 52)
    f = 0.0;
    if (r) {
        const int lead = __clzll((long long)r) - 11;           // its exponent is e - lead
        f = __longlong_as_double((long long)(((uint64_t)(e - lead + 1022) << 52) + (r << lead)));
    }
    return (int)(m >> (52 - e));
}
__device__ __forceinline__ int split(double s, float &f)
{
    const uint64_t b = (uint64_t)__double_as_longlong(s);
    const int e = (int)(b >> 52) - 1023;
    if (e < 0) {
        f = f64_to_f32(s);
        return 0;
    }
    const uint64_t m = (b & 0xfffffffffffffull) | 0x10000000000000ull;
    const int c = (int)(m >> (52 - e));
    const uint64_t r = m & ((0x10000000000000ull >> e) - 1);   // the fraction is r 2^(e - 52)
    f = 0.f;
    if (r) {
        const int top = 63 - __clzll((long long)r), x = top + e - 52;   // its exponent, -52 .. -1
        const uint64_t v = r << (63 - top);   // leading bit at 63; 24 bits kept, ties to even
        const uint64_t q = (v + 0x7fffffffffull + ((v >> 40) & 1));
        // a carry out of bit 63 is the next power of two, whose mantissa is zero
        const uint32_t mant = q < v ? 0x1000000u : (uint32_t)(q >> 40);
        f = __uint_as_float(((uint32_t)(x + 126) << 23) + mant);
    }
    return c;
}

// (c + f) / N of a cell index below 2^10 and an offset in [0, 1); inv_n = 1 / N, scaled = 2^-42 / N
__device__ __forceinline__ double position(int c, double f, double inv_n, double) { return ((double)c + f) * inv_n; }
__device__ __forceinline__ double position(int c, float f, double inv_n, double scaled)
{
    const uint32_t b = __float_as_uint(f), e = b >> 23;
    if (e - 108u < 19u || b == 0) {   // f = 0 or in [2^-19, 1): a multiple of 2^-42, so 2^42 (c + f) is one below 2^52
        const uint64_t m = b == 0 ? 0 : (uint64_t)((b & 0x7fffffu) | 0x800000u) << (e - 108u);
        const uint64_t n = ((uint64_t)c << 42) | m;
        return (__longlong_as_double((long long)(0x4330000000000000ull | n)) - 4503599627370496.0) * scaled;
    }
    return position_any(c, f, inv_n);
}

// f64_to_f32 where the particle type is f32
__device__ __forceinline__ void narrow(double d, float &f) { f = f64_to_f32(d); }
__device__ __forceinline__ void narrow(double d, double &f) { f = d; }

// ---------------------------------------------------------------------------
// Particle I/O: f64 (x, y, z) rows <-> cell + offset records.
// ---------------------------------------------------------------------------
template <class T>
__global__ void k_load(const double *pos, const double *mom, int64_t first, int64_t cnt, int N,
                       Particle<T> *out, int32_t *count, int *nonfinite)
{
    const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= cnt) return;
    // all six values before the branches below: the arrays may be pinned host memory, and a load that comes later
    // crosses the link again for a line that has left L1
    // (384^3 from pinned memory 13.6 ms, 19.7 with the loads between the branches)
    double xs[3], us[3];
#pragma unroll
    for (int d = 0; d < 3; d++) {
        xs[d] = pos[3 * k + d];
        us[d] = mom[3 * k + d];
    }
    Particle<T> P{};
    int ic[3];
    bool bad = false;
#pragma unroll
    for (int d = 0; d < 3; d++) {
        double x = xs[d];
        const double u = us[d];
        const uint32_t xh = (uint32_t)__double2hiint(x);
        bad |= (xh & 0x7ff00000u) == 0x7ff00000u || ((uint32_t)__double2hiint(u) & 0x7ff00000u) == 0x7ff00000u;
        if (xh >= 0x3ff00000u) x = wrap_unit(x);   // not in [0, 1)
        int c = split(x * N, P.f[d]);
        if (c >= N) c -= N;
        ic[d] = c;
        if (P.f[d] >= T(1)) {  // rounding of the offset to the storage type
            P.f[d] = T(0);
            ic[d] = c + 1 == N ? 0 : c + 1;
        }
        narrow(u, P.u[d]);
    }
    if (bad) *nonfinite = 1;
    P.cell = (ic[2] * N + ic[1]) * N + ic[0];
    P.id = (uint32_t)(first + k);
    out[first + k] = P;
    atomicAdd(&count[P.cell], 1);
}

// Packed host records (cell, 3 f32 offsets, 3 f32 momenta; 28 bytes) -> device records, checked.  A block
// takes PK_P records (14336 bytes) and moves them between the caller's array and shared memory with 16-byte
// accesses at consecutive addresses (the array may be pinned host memory read across the CPU-GPU link, where
// narrow accesses waste most of each transfer); vec = 0 (an array not 16-byte aligned) uses 4-byte accesses.
constexpr int PK_P = 512;
constexpr int PK_VEC = PK_P * (int)sizeof(pm_packed_particle) / 16;
static_assert(sizeof(pm_packed_particle) == 28 && PK_P * 28 % 16 == 0, "packed record");

__device__ __forceinline__ void pk_copy(uint4 *dst, const uint4 *src, int bytes, int vec)
{
    const int nv = vec ? bytes / 16 : 0;
    for (int v = threadIdx.x; v < nv; v += blockDim.x) dst[v] = src[v];
    for (int w = nv * 4 + threadIdx.x; w < bytes / 4; w += blockDim.x)
        reinterpret_cast<uint32_t *>(dst)[w] = reinterpret_cast<const uint32_t *>(src)[w];
}

// one packed record as the particle it stands for; a record with a cell outside [0, nc), an offset outside
// [0, 1) or a non-finite momentum is flagged (*bad = 1) and kept at a valid cell and offset
__device__ __forceinline__ Particle<float> unpack_record(const pm_packed_particle &q, uint32_t id, int64_t nc, int *bad)
{
    Particle<float> P;
    P.cell = q.cell;
    P.id = id;
    bool ok = q.cell >= 0 && (int64_t)q.cell < nc;
#pragma unroll
    for (int d = 0; d < 3; d++) {
        P.f[d] = q.f[d];
        P.u[d] = q.u[d];
        ok = ok && q.f[d] >= 0.f && q.f[d] < 1.f && isfinite(q.u[d]);
    }
    if (!ok) {   // keeps the cell index valid; the caller rejects the input
        *bad = 1;
        P.cell = 0;
        P.f[0] = P.f[1] = P.f[2] = 0.f;
    }
    return P;
}

__global__ void __launch_bounds__(256) k_load_packed(const pm_packed_particle *in, int64_t first, int64_t cnt,
                                                     int64_t nc, Particle<float> *out, int32_t *count, int *bad, int vec)
{
    __shared__ uint4 sb[PK_VEC];
    const int64_t base = (int64_t)blockIdx.x * PK_P;
    const int nb = (int)min((int64_t)PK_P, cnt - base);
    pk_copy(sb, reinterpret_cast<const uint4 *>(in + base), nb * 28, vec);
    __syncthreads();
    const pm_packed_particle *sq = reinterpret_cast<const pm_packed_particle *>(sb);
    for (int j = threadIdx.x; j < nb; j += blockDim.x) {
        const Particle<float> P = unpack_record(sq[j], (uint32_t)(first + base + j), nc, bad);
        out[first + base + j] = P;
        atomicAdd(&count[P.cell], 1);
    }
}

// The two passes of a counting sort straight from packed records in device memory: the histogram (with the
// record checks), then, after the scan, each record placed at its cell's slot as a particle.  Against loading
// the records into the particle buffer and sorting that, the particle buffer is written once and not read.
__global__ void __launch_bounds__(256) k_count_packed(const pm_packed_particle *in, int64_t cnt, int64_t nc,
                                                      int32_t *count, int *bad, int vec)
{
    __shared__ uint4 sb[PK_VEC];
    const int64_t base = (int64_t)blockIdx.x * PK_P;
    const int nb = (int)min((int64_t)PK_P, cnt - base);
    pk_copy(sb, reinterpret_cast<const uint4 *>(in + base), nb * 28, vec);
    __syncthreads();
    const pm_packed_particle *sq = reinterpret_cast<const pm_packed_particle *>(sb);
    for (int j = threadIdx.x; j < nb; j += blockDim.x)
        atomicAdd(&count[unpack_record(sq[j], 0u, nc, bad).cell], 1);
}

__global__ void __launch_bounds__(256) k_scatter_packed(const pm_packed_particle *in, int64_t cnt, int64_t nc,
                                                        const int32_t *start, int32_t *count, Particle<float> *out,
                                                        int *bad, int vec)
{
    __shared__ uint4 sb[PK_VEC];
    const int64_t base = (int64_t)blockIdx.x * PK_P;
    const int nb = (int)min((int64_t)PK_P, cnt - base);
    pk_copy(sb, reinterpret_cast<const uint4 *>(in + base), nb * 28, vec);
    __syncthreads();
    const pm_packed_particle *sq = reinterpret_cast<const pm_packed_particle *>(sb);
    for (int j = threadIdx.x; j < nb; j += blockDim.x) {
        const Particle<float> P = unpack_record(sq[j], (uint32_t)(base + j), nc, bad);
        const int r = atomicSub(&count[P.cell], 1) - 1;
        out[start[P.cell] + r] = P;
    }
}

// Device records in id order -> packed records (same staging as the load).
__global__ void __launch_bounds__(256) k_store_packed(const Particle<float> *byid, int64_t first, int64_t cnt,
                                                      pm_packed_particle *out, int vec)
{
    __shared__ uint4 sb[PK_VEC];
    const int64_t base = (int64_t)blockIdx.x * PK_P;
    const int nb = (int)min((int64_t)PK_P, cnt - base);
    pm_packed_particle *sq = reinterpret_cast<pm_packed_particle *>(sb);
    for (int j = threadIdx.x; j < nb; j += blockDim.x) {
        const Particle<float> P = byid[first + base + j];
        pm_packed_particle q;
        q.cell = P.cell;
#pragma unroll
        for (int d = 0; d < 3; d++) {
            q.f[d] = P.f[d];
            q.u[d] = P.u[d];
        }
        sq[j] = q;
    }
    __syncthreads();
    pk_copy(reinterpret_cast<uint4 *>(out + base), sb, nb * 28, vec);
}

template <class T>
__global__ void k_unpermute(const Particle<T> *in, Particle<T> *out, int64_t np)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= np) return;
    const Particle<T> P = in[i];
    out[P.id] = P;
}

// Particle records (in id order) -> f64 positions and momenta [k][3].  A block stages 512
// particles in shared memory and writes them with 16-byte stores at consecutive addresses, which
// keeps the writes full-line even when the destination is pinned host memory across the link.
constexpr int ST_P = 512;
template <class T>
__global__ void __launch_bounds__(256) k_store(const Particle<T> *byid, int64_t first, int64_t cnt, int N,
                                               double inv_n, double scaled, double *pos, double *mom, int vec)
{
    __shared__ double sp[3 * ST_P], su[3 * ST_P];
    const int64_t base = (int64_t)blockIdx.x * ST_P;
    const int nb = (int)min((int64_t)ST_P, cnt - base);
    for (int j = threadIdx.x; j < nb; j += blockDim.x) {
        const Particle<T> P = byid[first + base + j];
        const int ic[3] = {P.cell % N, (P.cell / N) % N, P.cell / (N * N)};
#pragma unroll
        for (int d = 0; d < 3; d++) {
            sp[3 * j + d] = position(ic[d], P.f[d], inv_n, scaled);
            su[3 * j + d] = widen(P.u[d]);
        }
    }
    __syncthreads();
    const int nv = 3 * nb;
    double *dst[2] = {pos ? pos + 3 * base : nullptr, mom ? mom + 3 * base : nullptr};
    const double *src[2] = {sp, su};
#pragma unroll
    for (int a = 0; a < 2; a++) {
        if (!dst[a]) continue;
        if (vec) {
            double2 *o = reinterpret_cast<double2 *>(dst[a]);
            for (int v = threadIdx.x; v < nv / 2; v += blockDim.x) o[v] = make_double2(src[a][2 * v], src[a][2 * v + 1]);
            if ((nv & 1) && threadIdx.x == 0) dst[a][nv - 1] = src[a][nv - 1];
        } else {
            for (int v = threadIdx.x; v < nv; v += blockDim.x) dst[a][v] = src[a][v];
        }
    }
}

// CIC density contrast N^3 / n_part sum w - 1 of FP64 contexts, a particle per thread.  Bound by the FP64 atomics, which
// take about as long whatever the cells hold: 128^3 P(k) 0.38 ms at z = 50 and at z = 1, 0.49 with a tenth of the mass in
// cells of 10^4.  The columns of the deposit, whose warps wait for their fullest cell on the FP64 pipe, took 0.42, 0.65
// and 4.3.
__global__ void k_density_acc(const Particle<double> *part, int64_t np, int N, double q, double *rho)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= np) return;
    const Particle<double> P = part[i];
    const int ix = P.cell % N, iy = (P.cell / N) % N, iz = P.cell / (N * N);
#pragma unroll
    for (int v = 0; v < 8; v++) {
        const int dx = v & 1, dy = v >> 1 & 1, dz = v >> 2;
        const double w = (dx ? P.f[0] : 1 - P.f[0]) * (dy ? P.f[1] : 1 - P.f[1]) * (dz ? P.f[2] : 1 - P.f[2]);
        atomicAdd(&rho[((int64_t)wrapi(iz + dz, N) * N + wrapi(iy + dy, N)) * N + wrapi(ix + dx, N)], q * w);
    }
}

__global__ void k_density_fin(double *rho, int64_t n)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) rho[i] -= 1.0;
}

template <class T> __global__ void k_to_f64(const T *s, double *d, int64_t n)
{
    // four values a thread: with one, starting the blocks takes longer than the copy
    const int64_t i = (int64_t)blockIdx.x * (4 * 256) + threadIdx.x;
    T v[4];
#pragma unroll
    for (int k = 0; k < 4; k++)
        if (i + 256 * k < n) v[k] = s[i + 256 * k];
#pragma unroll
    for (int k = 0; k < 4; k++)
        if (i + 256 * k < n) d[i + 256 * k] = widen(v[k]);
}

template <class T> __global__ void k_from_f64(const double *s, T *d, int64_t n)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) d[i] = (T)s[i];
}

__global__ void k_check_finite(const double *d, int64_t n, int *flag)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n && !isfinite(d[i])) *flag = 1;
}

inline unsigned nblk(int64_t n, int t) { return (unsigned)((n + t - 1) / t); }

}  // namespace

// Tiles of the deposit.  Along x the vertices are split evenly over as few warps as hold them: 31, so that a row
// of a nearly uniform load has 32 particles, or a whole row of up to 32, whose neighbour at x0 - 1 is its own last
// cell.  Along z a tile of tz vertices visits tz + 1 planes of cells and takes about two more to start; tz makes
// the number of waves times that smallest (64^3 mixed: 6, one wave, 17 us against 28 with one-plane tiles;
// 512^3: 57; longer ones cost more in L2 than they save).  Shape 1 halves it.
template <class T> void dep_tiles(DepParams<T> &p, bool full, int shape)
{
    const int N = p.N;
    p.cyclic = N <= 32;
    p.ntx = p.cyclic ? 1 : (N + 30) / 31;
    p.nrow = (N + p.ntx - 1) / p.ntx;
    p.nty = (N + DTY - 1) / DTY;
    p.ncol = (N + p.nty - 1) / p.nty;
    const int slots = 152 * (sizeof(T) == 4 ? (full ? dep_ctas<float, true>() : dep_ctas<float, false>())
                                            : (full ? dep_ctas<double, true>() : dep_ctas<double, false>()));
    int64_t best = INT64_MAX;
    for (int tz = 1; tz <= std::min(N, 64); tz++) {
        const int64_t waves = ((int64_t)p.ntx * p.nty * ((N + tz - 1) / tz) + slots - 1) / slots;
        if (waves * (tz + 3) < best) {
            best = waves * (tz + 3);
            p.tz = tz;
        }
    }
    if (shape == 1 && p.tz > 1) p.tz = (p.tz + 1) / 2;
}

inline bool dep_full(const StepScalars &s) { return !(s.newtonian || s.bootstrap); }

template <class T> DepParams<T> dep_params(const Ctx &c, const StepScalars &s)
{
    DepParams<T> p{};
    p.part = reinterpret_cast<const Particle<T> *>(c.part[c.cur]);
    p.start = c.start;
    p.phi1 = reinterpret_cast<const T *>(c.phi[c.iphi_prev]);
    p.chi1 = reinterpret_cast<const T *>(c.chi);
    p.phi2 = reinterpret_cast<const T *>(c.phi[c.iphi_prev2]);
    for (int i = 0; i < 9; i++) p.out.p[i] = reinterpret_cast<T *>(c.src) + (size_t)i * c.nc;
    p.k0slots = c.dscal + 8;
    p.N = c.N;
    p.newtonian = s.newtonian;
    dep_tiles(p, dep_full(s), c.dep_shape);
    p.a = (T)s.a;
    p.a2 = (T)(s.a * s.a);
    p.mass = (T)s.mass;
    const double n3 = (double)c.nc;
    double rb;
    if (s.newtonian) {
        p.G = (T)(s.four_pi_g / s.a * n3);
        rb = s.omega_m / n3;
    } else {
        p.G = (T)(s.four_pi_g / (s.a * s.a) * n3);
        rb = s.a * s.omega_m / n3;
    }
    p.rb_hi = (T)rb;
    p.rb_lo = (T)(rb - (double)p.rb_hi);
    p.c1 = (T)s.c_phi_dt;
    p.c2 = (T)s.c_phi_h2;
    p.inv_dt2 = (T)s.inv_dtau_prev2;
    p.halfN = (T)(0.5 * c.N);
    p.full_hc = s.full_hc;
    p.write_f = !(s.b_space && !s.b_seed);
    p.hc = (T)s.hc;
    p.n2 = (T)((double)c.N * (double)c.N);
    p.inv_g = 1.0 / (s.four_pi_g / (s.a * s.a) * n3);
    return p;
}

template <class T, bool FULL> void dep_attrs()
{
    static DeviceOnce once;
    once_on_device(once, [] {
        allow_smem(k_project<T, FULL>, dep_smem<T, FULL, false>());
        if constexpr (sizeof(T) == 8 || FULL) allow_smem(k_project_batch<T, FULL>, dep_smem<T, FULL, false>());
    });
}

// the mixed Newtonian mode takes k_mass
template <class T> bool dep_mass(const DepParams<T> &p) { return sizeof(T) == 4 && p.newtonian; }
template <class T> int dep_ntiles(const DepParams<T> &p)
{
    return dep_mass(p) ? (p.N / MT) * (p.N / MT) * (p.N / MT) : p.ntx * p.nty * ((p.N + p.tz - 1) / p.tz);
}

template <class T>
void launch_project(Ctx &c, const StepScalars &s)
{
    const DepParams<T> p = dep_params<T>(c, s);
    if (dep_full(s)) {
        dep_attrs<T, true>();
        k_project<T, true><<<dep_ntiles(p), DEP_THREADS, dep_smem<T, true, false>(), c.stream>>>(p);
    } else if (!dep_mass(p)) {
        dep_attrs<T, false>();
        k_project<T, false><<<dep_ntiles(p), DEP_THREADS, dep_smem<T, false, false>(), c.stream>>>(p);
    } else if constexpr (sizeof(T) == 4) {
        (mass_wide(c.N, c.np) ? k_mass<int64_t> : k_mass<int>)<<<dep_ntiles(p), MTHREADS, 0, c.stream>>>(p);
    }
    c.launches++;
}

// One deposit launch over several boxes of one precision, all relativistic or all Newtonian (batches of MAXBATCH).
template <class T>
void launch_project_batch(Ctx *const *cs, const StepScalars *ss, int n, bool full, cudaStream_t st)
{
    for (int b0 = 0; b0 < n; b0 += MAXBATCH) {
        const int nb = std::min(MAXBATCH, n - b0);
        thread_local DepBatch<T> q;   // host staging of the launch parameters (copied at launch)
        q.nbox = nb;
        q.first[0] = 0;
        for (int i = 0; i < nb; i++) {
            Ctx &c = *cs[b0 + i];
            q.box[i] = dep_params<T>(c, ss[b0 + i]);
            q.first[i + 1] = q.first[i] + dep_ntiles(q.box[i]);
            c.launches++;
        }
        if (full) {
            dep_attrs<T, true>();
            k_project_batch<T, true><<<q.first[nb], DEP_THREADS, dep_smem<T, true, false>(), st>>>(q);
        } else if constexpr (sizeof(T) == 4) {
            bool wide = false;
            for (int i = 0; i < nb; i++) wide |= mass_wide(cs[b0 + i]->N, cs[b0 + i]->np);
            (wide ? k_mass_batch<int64_t> : k_mass_batch<int>)<<<q.first[nb], MTHREADS, 0, st>>>(q);
        } else {
            dep_attrs<T, false>();
            k_project_batch<T, false><<<q.first[nb], DEP_THREADS, dep_smem<T, false, false>(), st>>>(q);
        }
    }
}

// Tiles of the kick: rows of up to 32 cells, as long along z as makes the number of waves times (tz + 2) smallest
// (the fields of three more planes are loaded than cells are visited).  A wave is counted with the relativistic kernel's
// CTAs (three an SM in FP32) for the Newtonian one, too, which holds four: with four, 128^3 and 192^3 gain 1-4%, 144^3 and
// 288^3 lose 3-4% (0.336 -> 0.346 ms).
template <class T> KdParams<T> kd_params(const Ctx &c, const StepScalars &s)
{
    KdParams<T> p{};
    p.part = reinterpret_cast<Particle<T> *>(c.part[c.cur]);
    p.start = c.start;
    p.count = c.count;
    const T *B = reinterpret_cast<const T *>(c.B);
    p.phi = reinterpret_cast<const T *>(c.phi[c.iphi_new]);
    p.chi = reinterpret_cast<const T *>(c.chi);
    p.Bx = B;
    p.By = B + c.nc;
    p.Bz = B + 2 * c.nc;
    p.N = c.N;
    p.ntx = (c.N + 31) / 32;
    p.nrow = (c.N + p.ntx - 1) / p.ntx;
    const int slots = 152 * kd_ctas<T, false>();
    int64_t best = INT64_MAX;
    for (int tz = 1; tz <= std::min(c.N, 64); tz++) {
        const int64_t waves = ((int64_t)p.ntx * (c.N / KROWS) * ((c.N + tz - 1) / tz) + slots - 1) / slots;
        if (waves * (tz + 2) < best) {
            best = waves * (tz + 2);
            p.tz = tz;
        }
    }
    p.a = (T)s.a;
    p.a2 = (T)(s.a * s.a);
    p.a_half2 = (T)(s.a_half * s.a_half);
    p.inv_a_half = (T)(1.0 / s.a_half);
    p.dt_kick = (T)s.dtau_kick;
    p.dt_drift_N = (T)(s.dtau * c.N);
    p.halfN = (T)(0.5 * c.N);
    p.kick_N = p.dt_kick * p.halfN;
    return p;
}

template <class T> int kd_ntiles(const KdParams<T> &p) { return p.ntx * (p.N / KROWS) * ((p.N + p.tz - 1) / p.tz); }

template <class T, bool NEWT> void kd_attrs()
{
    static DeviceOnce once;
    once_on_device(once, [] {
        allow_smem(k_kick_drift<T, NEWT>, kd_smem<T, NEWT>());
        allow_smem(k_kick_batch<T, NEWT>, kd_smem<T, NEWT>());
    });
}

template <class T>
void launch_kick_drift(Ctx &c, const StepScalars &s)
{
    KdParams<T> p = kd_params<T>(c, s);
    if (s.newtonian && c.corr) {
        static DeviceOnce once;
        once_on_device(once, [] { allow_smem(k_kick_corrected<T>, kd_smem<T, true>()); });
        p.corr = static_cast<const float *>(c.corr);
        p.corr_scale = (T)c.corr_scale;
        k_kick_corrected<T><<<kd_ntiles(p), KD_THREADS, kd_smem<T, true>(), c.stream>>>(p);
    } else if (s.newtonian) {
        kd_attrs<T, true>();
        k_kick_drift<T, true><<<kd_ntiles(p), KD_THREADS, kd_smem<T, true>(), c.stream>>>(p);
    } else {
        kd_attrs<T, false>();
        k_kick_drift<T, false><<<kd_ntiles(p), KD_THREADS, kd_smem<T, false>(), c.stream>>>(p);
    }
    c.launches++;
}

// One gather + kick + drift launch over several boxes of one precision, all relativistic or all Newtonian (batches
// of MAXBATCH).
template <class T>
void launch_kick_batch(Ctx *const *cs, const StepScalars *ss, int n, bool full, cudaStream_t st)
{
    for (int b0 = 0; b0 < n; b0 += MAXBATCH) {
        const int nb = std::min(MAXBATCH, n - b0);
        thread_local KdBatch<T> q;
        q.nbox = nb;
        q.first[0] = 0;
        for (int i = 0; i < nb; i++) {
            Ctx &c = *cs[b0 + i];
            q.box[i] = kd_params<T>(c, ss[b0 + i]);
            q.first[i + 1] = q.first[i] + kd_ntiles(q.box[i]);
            c.launches++;
        }
        if (full) {
            kd_attrs<T, false>();
            k_kick_batch<T, false><<<q.first[nb], KD_THREADS, kd_smem<T, false>(), st>>>(q);
        } else {
            kd_attrs<T, true>();
            k_kick_batch<T, true><<<q.first[nb], KD_THREADS, kd_smem<T, true>(), st>>>(q);
        }
    }
}

// Time the deposit of the context's current state with each column length and keep the fastest.  The trial
// deposits write into the spectrum buffer, which holds nothing between steps (9 half spectra hold more than
// 9 real fields), so the sources the caller can read stay as they were; the k = 0 slots they also add to are
// cleared again.
template <class T>
int tune_deposit_shape(Ctx &c, const StepScalars &s)
{
    void *const src = c.src;
    c.src = c.spec;
    cudaEvent_t e0, e1;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    float best = 1e30f;
    int best_v = 0;
    for (int v = 0; v < NDEPSHAPES; v++) {
        c.dep_shape = v;
        launch_project<T>(c, s);   // warm-up (and the first launch of the shape)
        cudaEventRecord(e0, c.stream);
        for (int r = 0; r < 3; r++) launch_project<T>(c, s);
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
    cudaMemsetAsync(c.dscal + 8, 0, sizeof(double) * NK0SLOTS, c.stream);
    c.src = src;
    c.dep_shape = best_v;
    return best_v;
}

void launch_scan(Ctx &c)
{
    const int64_t nb = (c.nc + SCAN_TILE - 1) / SCAN_TILE;
    k_scan_reduce<<<(unsigned)nb, SCAN_T, 0, c.stream>>>(c.count, c.nc, c.blocksum);
    k_scan_down<<<(unsigned)nb, SCAN_T, 0, c.stream>>>(c.count, c.nc, c.blocksum, c.start);
    c.launches += 2;
}

template <class T>
void launch_sort(Ctx &c)
{
    launch_scan(c);
    c.mark(EV_SCAN);
    const int o = 1 - c.cur;
    k_scatter<T><<<nblk(c.np, 256), 256, 0, c.stream>>>(reinterpret_cast<const Particle<T> *>(c.part[c.cur]),
                                                         reinterpret_cast<Particle<T> *>(c.part[o]), c.np,
                                                         c.start, c.count);
    c.launches++;
    c.cur = o;
}

template <class T>
void launch_load_particles(Ctx &c, const double *d_pos, const double *d_mom, int64_t first, int64_t count,
                           int *d_nonfinite)
{
    k_load<T><<<nblk(count, 256), 256, 0, c.stream>>>(d_pos, d_mom, first, count, c.N,
                                                      reinterpret_cast<Particle<T> *>(c.part[c.cur]), c.count,
                                                      d_nonfinite);
}

template <class T>
void launch_store_particles_scatter(Ctx &c, double *, double *)
{
    const int o = 1 - c.cur;
    k_unpermute<T><<<nblk(c.np, 256), 256, 0, c.stream>>>(reinterpret_cast<const Particle<T> *>(c.part[c.cur]),
                                                           reinterpret_cast<Particle<T> *>(c.part[o]), c.np);
}

template <class T>
void launch_store_particles(Ctx &c, double *d_pos, double *d_mom, int64_t first, int64_t count)
{
    const int o = 1 - c.cur;
    // 16-byte stores need 16-byte aligned arrays (the block offsets are multiples of 3 * 512 doubles)
    const int vec = ((reinterpret_cast<uintptr_t>(d_pos) | reinterpret_cast<uintptr_t>(d_mom)) & 15) == 0;
    k_store<T><<<nblk(count, ST_P), 256, 0, c.stream>>>(reinterpret_cast<const Particle<T> *>(c.part[o]), first,
                                                        count, c.N, 1.0 / (double)c.N,
                                                        std::ldexp(1.0 / (double)c.N, -42), d_pos, d_mom, vec);
}

void launch_load_packed(Ctx &c, const pm_packed_particle *in, int64_t first, int64_t count, int *d_bad)
{
    const int vec = (reinterpret_cast<uintptr_t>(in) & 15) == 0;
    k_load_packed<<<nblk(count, PK_P), 256, 0, c.stream>>>(in, first, count, c.nc,
                                                           reinterpret_cast<Particle<float> *>(c.part[c.cur]), c.count,
                                                           d_bad, vec);
}

void launch_put_packed_sorted(Ctx &c, const pm_packed_particle *in, int *d_bad)
{
    const int vec = (reinterpret_cast<uintptr_t>(in) & 15) == 0;
    const unsigned nb = nblk(c.np, PK_P);
    k_count_packed<<<nb, 256, 0, c.stream>>>(in, c.np, c.nc, c.count, d_bad, vec);
    launch_scan(c);
    const int o = 1 - c.cur;
    k_scatter_packed<<<nb, 256, 0, c.stream>>>(in, c.np, c.nc, c.start, c.count,
                                               reinterpret_cast<Particle<float> *>(c.part[o]), d_bad, vec);
    c.launches += 2;
    c.cur = o;
}

void launch_store_packed(Ctx &c, pm_packed_particle *out, int64_t first, int64_t count)
{
    const int vec = (reinterpret_cast<uintptr_t>(out) & 15) == 0;
    k_store_packed<<<nblk(count, PK_P), 256, 0, c.stream>>>(
        reinterpret_cast<const Particle<float> *>(c.part[1 - c.cur]), first, count, out, vec);
}

// CIC mass density contrast delta = rho / omega_m - 1
template <> void launch_density<double>(Ctx &c, void *real_out)
{
    double *rho = static_cast<double *>(real_out);
    cudaMemsetAsync(rho, 0, sizeof(double) * c.nc, c.stream);
    k_density_acc<<<nblk(c.np, 256), 256, 0, c.stream>>>(reinterpret_cast<const Particle<double> *>(c.part[c.cur]), c.np, c.N,
                                                         (double)c.nc / (double)c.np, rho);
    k_density_fin<<<nblk(c.nc, 256), 256, 0, c.stream>>>(rho, c.nc);
}

template <> void launch_density<float>(Ctx &c, void *real_out)
{
    DepParams<float> p{};
    p.part = reinterpret_cast<const Particle<float> *>(c.part[c.cur]);
    p.start = c.start;
    p.out.p[0] = real_out;
    p.N = c.N;
    p.newtonian = 1;
    p.mass = 1.f;
    dep_tiles(p, false, 0);
    const double mean = (double)c.np / (double)c.nc, q = (double)c.nc / (double)c.np;
    p.G = (float)q;
    p.c1 = (float)(q - (double)p.G);
    p.rb_hi = (float)mean;
    p.rb_lo = (float)(mean - (double)p.rb_hi);
    static DeviceOnce once;
    constexpr size_t bytes = dep_smem<float, false, true>();
    once_on_device(once, [] { allow_smem(k_contrast, bytes); });
    k_contrast<<<p.ntx * p.nty * ((p.N + p.tz - 1) / p.tz), DEP_THREADS, bytes, c.stream>>>(p);
}

template <class T>
void launch_to_f64(Ctx &c, const void *src, double *dst, int64_t n)
{
    k_to_f64<T><<<nblk(n, 4 * 256), 256, 0, c.stream>>>(reinterpret_cast<const T *>(src), dst, n);
}

template <class T>
void launch_from_f64(Ctx &c, const double *src, void *dst, int64_t n)
{
    k_from_f64<T><<<nblk(n, 256), 256, 0, c.stream>>>(src, reinterpret_cast<T *>(dst), n);
}

template <class T>
void launch_check_finite(Ctx &c, const double *d, int64_t n, int *d_flag)
{
    k_check_finite<<<nblk(n, 256), 256, 0, c.stream>>>(d, n, d_flag);
}

#define PM_INST(T)                                                                          \
    template void launch_project<T>(Ctx &, const StepScalars &);                            \
    template void launch_project_batch<T>(Ctx *const *, const StepScalars *, int, bool, cudaStream_t); \
    template void launch_kick_batch<T>(Ctx *const *, const StepScalars *, int, bool, cudaStream_t); \
    template int tune_deposit_shape<T>(Ctx &, const StepScalars &);                         \
    template void launch_kick_drift<T>(Ctx &, const StepScalars &);                         \
    template void launch_sort<T>(Ctx &);                                                    \
    template void launch_load_particles<T>(Ctx &, const double *, const double *, int64_t,  \
                                           int64_t, int *);                                 \
    template void launch_store_particles<T>(Ctx &, double *, double *, int64_t, int64_t);   \
    template void launch_store_particles_scatter<T>(Ctx &, double *, double *);             \
    template void launch_to_f64<T>(Ctx &, const void *, double *, int64_t);                 \
    template void launch_from_f64<T>(Ctx &, const double *, void *, int64_t);               \
    template void launch_check_finite<T>(Ctx &, const double *, int64_t, int *);
PM_INST(double)
PM_INST(float)

}  // namespace pm
