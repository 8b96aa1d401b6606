// lqcd_split.cu -- persistent batched solver for single- and double-precision
// inner storage (the half formats and the Schwarz-preconditioned solves run in
// lqcd_solver.cu's k_solve).
//
// The same solve as k_solve: an outer double defect correction around
// BiCGstab or the geometric series on every system at once, one cooperative
// launch, a software barrier per system.  What bounds it, and what follows:
//   * small systems (up to a few thousand sites): the length of a phase, a
//     half-lattice hopping sweep between two barriers.  One thread per site
//     makes that eight dependent neighbour reads and 2000 instructions.  LPS
//     warps share 32 sites instead: warp d of a site group sums the hops of
//     its own directions (LPS = 2: forward or backward, 4: half of those,
//     8: one hop), the partial sums meet in shared memory and each warp
//     finishes its own spin components.  No warp diverges: its directions
//     are compile-time constants in its branch.
//   * larger systems: L2 traffic and instruction fetch.  One thread per site
//     (LPS = 1) with the loads of a hop issued before the arithmetic of the
//     previous one, one copy of the hopping code for all sweeps of an
//     iteration (four copies overran the instruction cache and made a sweep
//     1.5 times longer), vectors and links in tiles of 32 sites, phases,
//     barriers and reductions kept apart so that no more than a few of the
//     128 registers spill (4-16 bytes a kernel, 32 a reduction; spilled
//     vectors tripled the L2 writes).
//   * everywhere: the dot products of an iteration are FP64 sums and its
//     scalars double, whatever the storage.  FP64 issues two lanes per cycle
//     and SM, so a site's term (a word's, in an element-wise phase) is summed
//     in the storage arithmetic first.
// Measured (ms per solve to 1e-12, one thread per site without the above ->
// this kernel): 12x6^3 global 4.65 -> 2.61, 32x16^3 global 30.7 -> 24.0, its
// 8 slabs 4.77 -> 3.83, 64x32^3 global 579 -> 358, 32x24^3 series 9.37 -> 7.70;
// double precision at 16x8^3 (two solves and the force) 34.9 -> 5.70.
#include <algorithm>

#include "lqcd_solve.cuh"

namespace {

// ---------------------------------------------------------------------------
// sums: FP64 over sites, warps and CTAs, of per-site terms in the storage
// arithmetic.  The FP64 pipe issues two lanes per cycle and SM, so a sum
// enters it as late as that allows.
// ---------------------------------------------------------------------------
// what a thread adds up in an element-wise phase, word by word: a pair of
// floats in single precision (no FP64 instruction per word), one conversion
// at the end
template <class T>
struct Local;
template <>
struct Local<float> {
    float h, l;
    __device__ __forceinline__ void add(float x)
    {
        float s, e;
        df_two_sum(h, x, s, e);
        h = s;
        l += e;
    }
    __device__ __forceinline__ double value() const { return (double)h + (double)l; }
    static __device__ __forceinline__ Local zero() { return Local{0.f, 0.f}; }
};
template <>
struct Local<double> {
    double h;
    __device__ __forceinline__ void add(double x) { h += x; }
    __device__ __forceinline__ double value() const { return h; }
    static __device__ __forceinline__ Local zero() { return Local{0.0}; }
};

// warp sums of N = 1, 2 or 4 quantities, halving the quantities a lane
// carries with every step (N = 4: six additions instead of twenty): every
// lane returns the sum of quantity lane * N / 32
template <int N>
__device__ __forceinline__ double warp_sum(double (&v)[N])
{
    const int lane = threadIdx.x & 31;
    int m = 16;
#pragma unroll
    for (int n = N / 2; n >= 1; n >>= 1, m >>= 1) {
        const bool up = (lane & m) != 0;
#pragma unroll
        for (int k = 0; k < n; ++k) {
            const double x = up ? v[n + k] : v[k];
            v[k] = x + __shfl_xor_sync(0xffffffffu, up ? v[k] : v[n + k], m);
        }
    }
    for (; m >= 1; m >>= 1) v[0] += __shfl_xor_sync(0xffffffffu, v[0], m);
    return v[0];
}

// the scalars of the recurrences, in double; the vectors take them rounded to
// the storage arithmetic
__device__ __forceinline__ cx<double> cdiv(cx<double> a, cx<double> b)
{
    const double d = 1.0 / (b.re * b.re + b.im * b.im);
    return d * cjmul(b, a);
}
template <class T>
__device__ __forceinline__ cx<T> sround(cx<double> a)
{
    return mk((T)a.re, (T)a.im);
}
template <class T>
__device__ __forceinline__ bool fin2(cx<T> a) { return isfinite(a.re) && isfinite(a.im); }

// ---------------------------------------------------------------------------
// barrier of the CTAs of one group (bounded, as in k_solve) and the sums
// that go with it.  Warp 0 does both alone: it adds the CTA's sums, arrives,
// waits, adds the group's sums and hands them to f (on lane 0), so a
// reducing barrier costs the CTA two __syncthreads.
// ---------------------------------------------------------------------------
struct Group {
    int grp, cin, cps;  // group, CTA in the group, CTAs per group
    unsigned epoch;
    int rb;
};

__device__ __forceinline__ bool group_wait(const SolveArgs& A, Group& G)
{
    unsigned* bar = A.bar + (size_t)G.grp * BAR_STRIDE;
    const unsigned target = G.epoch * (unsigned)G.cps;
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(bar) : "memory");
    const long long t0 = clock64();
    for (int n = 1; ld_acquire(bar) < target; ++n) {
        if (clock64() - t0 > A.spin_limit) {
            atomicExch(A.status, LQCD_ERR_TIMEOUT);
            atomicCAS(A.sticky, 0, LQCD_ERR_TIMEOUT);
            return false;
        }
        if ((n & 15) == 0 && *(volatile int*)A.status == LQCD_ERR_TIMEOUT) return false;
    }
    return true;
}

__device__ __noinline__ bool group_sync(const SolveArgs& A, Group& G)
{
    __shared__ int s_ok;
    __syncthreads();
    ++G.epoch;
    if (G.cps == 1) return true;
    if (threadIdx.x == 0) s_ok = group_wait(A, G);
    __syncthreads();
    return s_ok != 0;
}

// (Not inlined: with their registers the phases would spill.)
// f receives the group's sums of the N quantities v on thread 0.  The CTAs'
// partials lie quantity by quantity: warp k adds those of quantity k, four
// loads in flight per lane.
template <int NW, int N, class F>
__device__ __noinline__ bool group_reduce(const SolveArgs& A, Group& G, double (&v)[N], F f)
{
    static_assert(N <= NW && N <= SPLIT_NQ, "one warp per quantity");
    __shared__ double sh[N][NW], tot[N];
    __shared__ int s_ok;
    constexpr int LQ = 32 / N;  // lanes per quantity
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    {
        const double x = warp_sum<N>(v);
        if (lane % LQ == 0) sh[lane / LQ][w] = x;
    }
    __syncthreads();
    ++G.epoch;
    if (G.cps == 1) {
        if (w < N) {
            double q[1] = {0.0};
            if (lane < NW) q[0] = sh[w][lane];
            q[0] = warp_sum<1>(q);
            if (lane == 0) tot[w] = q[0];
        }
        __syncthreads();
        if (threadIdx.x == 0) f(tot);
        __syncthreads();
        return true;
    }
    double* part = A.part + ((size_t)G.rb * gridDim.x + (size_t)G.grp * G.cps) * SPLIT_NQ;
    if (w == 0) {
        // lane LQ k + j adds every LQ-th warp's sum of quantity k
        double x = 0.0;
#pragma unroll
        for (int j = 0; j < (NW + LQ - 1) / LQ; ++j) {
            const int i = lane % LQ + j * LQ;
            if (i < NW) x += sh[lane / LQ][i];
        }
#pragma unroll
        for (int m = LQ / 2; m >= 1; m >>= 1)
            if (m < NW) x += __shfl_xor_sync(0xffffffffu, x, m);
        if (lane % LQ == 0) part[(size_t)(lane / LQ) * G.cps + G.cin] = x;
        __syncwarp();
        if (lane == 0) s_ok = group_wait(A, G);
    }
    __syncthreads();
    if (w < N) {
        const double* p = part + (size_t)w * G.cps;
        double q[1] = {0.0};
        for (int c = lane; c < G.cps; c += 128) {
            double u[4];
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if (c + 32 * k < G.cps) u[k] = __ldcg(p + c + 32 * k);
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if (c + 32 * k < G.cps) q[0] += u[k];
        }
        q[0] = warp_sum<1>(q);
        if (lane == 0) tot[w] = q[0];
    }
    G.rb ^= 1;
    __syncthreads();
    if (threadIdx.x == 0) f(tot);
    __syncthreads();
    return s_ok != 0;
}

// ---------------------------------------------------------------------------
// inner vectors: words of two (single) or one (double) complex numbers
// ---------------------------------------------------------------------------
template <int P>
struct Word;
template <>
struct Word<PREC32> {
    typedef float4 W;
    static constexpr int N = 6;
};
template <>
struct Word<PREC64> {
    typedef double2 W;
    static constexpr int N = 12;
};

// The inner vectors are stored in tiles of 32 sites, [Vh/32][N][32] words
// (Vh rounded up): one address and constant offsets reach all words of a
// site.  tile_at: the place of word 0 of site i, word k is 32 k further.
template <int P>
__device__ __forceinline__ size_t tile_at(int i)
{
    return (size_t)i + (size_t)(i >> 5) * (32 * (Word<P>::N - 1));
}

__device__ __forceinline__ float4 wzero(float4) { return make_float4(0.f, 0.f, 0.f, 0.f); }
__device__ __forceinline__ double2 wzero(double2) { return make_double2(0.0, 0.0); }
// y + a x
__device__ __forceinline__ float4 waxpy(cx<float> a, float4 x, float4 y)
{
    return make_float4(y.x + a.re * x.x - a.im * x.y, y.y + a.re * x.y + a.im * x.x, y.z + a.re * x.z - a.im * x.w,
                       y.w + a.re * x.w + a.im * x.z);
}
__device__ __forceinline__ double2 waxpy(cx<double> a, double2 x, double2 y)
{
    return make_double2(y.x + a.re * x.x - a.im * x.y, y.y + a.re * x.y + a.im * x.x);
}
// |a|^2, Re <a, b> and Im <a, b> of a word
__device__ __forceinline__ float wnorm(float4 a) { return a.x * a.x + a.y * a.y + a.z * a.z + a.w * a.w; }
__device__ __forceinline__ double wnorm(double2 a) { return a.x * a.x + a.y * a.y; }
__device__ __forceinline__ float wdot_re(float4 a, float4 b) { return a.x * b.x + a.y * b.y + a.z * b.z + a.w * b.w; }
__device__ __forceinline__ float wdot_im(float4 a, float4 b) { return a.x * b.y - a.y * b.x + a.z * b.w - a.w * b.z; }
__device__ __forceinline__ double wdot_re(double2 a, double2 b) { return a.x * b.x + a.y * b.y; }
__device__ __forceinline__ double wdot_im(double2 a, double2 b) { return a.x * b.y - a.y * b.x; }

__device__ __forceinline__ void put(Spinor<float>& s, int k, float4 w)
{
    s.c[(2 * k) / 3][(2 * k) % 3] = mk(w.x, w.y);
    s.c[(2 * k + 1) / 3][(2 * k + 1) % 3] = mk(w.z, w.w);
}
__device__ __forceinline__ void put(Spinor<double>& s, int k, double2 w) { s.c[k / 3][k % 3] = mk(w.x, w.y); }

// ---------------------------------------------------------------------------
// the hops of one warp
// ---------------------------------------------------------------------------
// one hop's loads, kept as the words that were read
template <int P>
struct Raw {
    static constexpr int NL = P == PREC32 ? 3 : 9;
    typename Word<P>::W s[Word<P>::N], l[NL];
    bool use, neg;
};

// hop H: direction mu = 3 - H / 2, forward (even H) or backward
template <int P, int H>
__device__ __forceinline__ void hop_fetch(const Geo& g, int mode, int pout, int i, const int x[4], int lex,
                                          const typename Word<P>::W* in, const GaugeF& U, Raw<P>& R)
{
    typedef typename Word<P>::W W;
    constexpr int MU = 3 - H / 2, DIR = H & 1;
    const int stride = MU == 3 ? 1 : MU == 2 ? g.L[3] : MU == 1 ? g.L[3] * g.L[2] : g.V3;
    const bool wrap = DIR ? x[MU] == 0 : x[MU] == g.L[MU] - 1;
    int nl = DIR ? lex - stride : lex + stride;
    if (wrap) nl += DIR ? g.L[MU] * stride : -g.L[MU] * stride;
    R.use = MU != 0 || t_hop_kept(g, mode, DIR ? x[0] : x[0] + 1);
    R.neg = MU == 0 && wrap && g.bc_t < 0;
    // a dropped hop reads the own index instead of another system's site
    const int j = R.use ? nl >> 1 : i;
    const W* sp = in + tile_at<P>(j);
#pragma unroll
    for (int k = 0; k < Word<P>::N; ++k) R.s[k] = sp[32 * k];
    constexpr int NL = Raw<P>::NL;
    const int mp = MU * 2 + (DIR ? 1 - pout : pout), li = DIR ? j : i;
    const W* lp = (const W*)U.v + (P == PREC32 ? (size_t)mp * link32_block(U.Vh) + link32_at(li) : (size_t)mp * NL * U.Vh + li);
#pragma unroll
    for (int k = 0; k < NL; ++k) R.l[k] = __ldg(lp + (P == PREC32 ? (size_t)(32 * k) : (size_t)k * U.Vh));
}

// rows 0 and 1 of the link as read, entry c of row 2
__device__ __forceinline__ cx<float> link_entry(const float4 (&l)[3], int r, int c)
{
    const int e = 3 * r + c;
    return e & 1 ? mk(l[e >> 1].z, l[e >> 1].w) : mk(l[e >> 1].x, l[e >> 1].y);
}
__device__ __forceinline__ cx<float> link_row2(const float4 (&l)[3], int c)
{
    const int j = (c + 1) % 3, k = (c + 2) % 3;
    return conjx(link_entry(l, 0, j) * link_entry(l, 1, k) - link_entry(l, 0, k) * link_entry(l, 1, j));
}
__device__ __forceinline__ cx<double> link_entry(const double2 (&l)[9], int r, int c)
{
    return mk(l[3 * r + c].x, l[3 * r + c].y);
}
__device__ __forceinline__ cx<double> link_row2(const double2 (&l)[9], int c) { return link_entry(l, 2, c); }

using ::cfma;
__device__ __forceinline__ cx<float> cfma(cx<float> a, cx<float> b, cx<float> c)
{
    return mk(fmaf(-a.im, b.im, fmaf(a.re, b.re, c.re)), fmaf(a.im, b.re, fmaf(a.re, b.im, c.im)));
}
template <class T>
__device__ __forceinline__ cx<T> cmul1(cx<T> a, cx<T> b)
{
    return mk(fma(-a.im, b.im, a.re * b.re), fma(a.im, b.re, a.re * b.im));
}

// adds hop H: the neighbour is projected, and the link applied and the result
// accumulated colour by colour (row by row, column by column for U^dag), so
// that besides acc only the half spinor and rows 0-1 of the link are live.
// FIRST: acc is set instead (with a warp per hop, adding to zero would be 192
// of a site's 1200 additions and multiply-adds: a series at 64x32^3 in double,
// bound by their number, took 131 instead of 123 ms)
template <int P, int H, bool FIRST>
__device__ __forceinline__ void hop_add(const Raw<P>& R, Spinor<typename Real<P>::T>& acc)
{
    typedef typename Real<P>::T T;
    constexpr int MU = 3 - H / 2, DAG = H & 1, sg = DAG ? +1 : -1;
    if (MU == 0 && !R.use) {
        if (FIRST) {
#pragma unroll
            for (int s = 0; s < 4; ++s)
#pragma unroll
                for (int c = 0; c < 3; ++c) acc.c[s][c] = mk(T(0), T(0));
        }
        return;
    }
    HalfSp<T> h;
    {
        Spinor<T> s;
#pragma unroll
        for (int k = 0; k < Word<P>::N; ++k) put(s, k, R.s[k]);
        project(MU, sg, s, h);
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        cx<T> w0, w1;
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            const int r = DAG ? j : c, q = DAG ? c : j;
            cx<T> u = r == 2 ? link_row2(R.l, q) : link_entry(R.l, r, q);
            if (DAG) u = conjx(u);
            w0 = j ? cfma(u, h.c[0][j], w0) : cmul1(u, h.c[0][j]);
            w1 = j ? cfma(u, h.c[1][j], w1) : cmul1(u, h.c[1][j]);
        }
        if (MU == 0 && R.neg) {
            w0 = -w0;
            w1 = -w1;
        }
        if (FIRST) set_recon1(MU, sg, w0, w1, acc, c);
        else accum_recon1(MU, sg, w0, w1, acc, c);
    }
}

// hops H, H + STEP, .. (N of them): the loads of a hop are issued before the
// arithmetic of the one before it
template <int P, int H, int STEP, int N, bool FIRST = true>
struct Hops {
    static __device__ __forceinline__ void run(const Geo& g, int mode, int pout, int i, const int x[4], int lex,
                                               const typename Word<P>::W* in, const GaugeF& U, Raw<P>& R,
                                               Spinor<typename Real<P>::T>& acc)
    {
        if constexpr (N > 1) {
            Raw<P> Q;
            hop_fetch<P, H + STEP>(g, mode, pout, i, x, lex, in, U, Q);
            hop_add<P, H, FIRST>(R, acc);
            Hops<P, H + STEP, STEP, N - 1, false>::run(g, mode, pout, i, x, lex, in, U, Q, acc);
        } else {
            hop_add<P, H, FIRST>(R, acc);
        }
    }
    static __device__ __forceinline__ void start(const Geo& g, int mode, int pout, int i, const int x[4], int lex,
                                                 const typename Word<P>::W* in, const GaugeF& U,
                                                 Spinor<typename Real<P>::T>& acc)
    {
        Raw<P> R;
        hop_fetch<P, H>(g, mode, pout, i, x, lex, in, U, R);
        run(g, mode, pout, i, x, lex, in, U, R, acc);
    }
};

// partial sum of the hopping term at (pout, i) over the directions of warp d
template <int P, int LPS>
__device__ __forceinline__ void hop_part(const Geo& g, int mode, int pout, int i, int d, const typename Word<P>::W* in,
                                         const GaugeF& U, Spinor<typename Real<P>::T>& acc)
{
    int x[4];
    eo_coords(g, pout, i, x);
    const int lex = lex_of(g, x);
#define LQ_H(H, STEP, N) Hops<P, H, STEP, N>::start(g, mode, pout, i, x, lex, in, U, acc)
    if constexpr (LPS == 1) {
        LQ_H(0, 1, 8);
    } else if constexpr (LPS == 2) {
        if (d == 0) LQ_H(0, 2, 4);
        else LQ_H(1, 2, 4);
    } else if constexpr (LPS == 4) {
        switch (d) {
            case 0: LQ_H(0, 2, 2); break;
            case 1: LQ_H(1, 2, 2); break;
            case 2: LQ_H(4, 2, 2); break;
            default: LQ_H(5, 2, 2); break;
        }
    } else {
        switch (d) {
            case 0: LQ_H(0, 1, 1); break;
            case 1: LQ_H(1, 1, 1); break;
            case 2: LQ_H(2, 1, 1); break;
            case 3: LQ_H(3, 1, 1); break;
            case 4: LQ_H(4, 1, 1); break;
            case 5: LQ_H(5, 1, 1); break;
            case 6: LQ_H(6, 1, 1); break;
            default: LQ_H(7, 1, 1); break;
        }
    }
#undef LQ_H
}

// The partial sums of a site group's LPS warps meet in shared memory; warp d
// receives the components [d NC, (d + 1) NC) of the sum (LPS = 8: warps 0..3).
// The buffer is used alternately in two halves: a warp that writes a half
// again has passed the barrier after the other half, which its partners
// reached after they had read this one.
template <class T, int LPS>
struct Xchg {
    static constexpr int PARTS = LPS < 4 ? LPS : 4;
    static constexpr int NC = 12 / PARTS;
    T* buf;  // [2][NW][24][32]
    int w, d, sg, lane, half;
    __device__ __forceinline__ bool fin() const { return d < PARTS; }
    __device__ __forceinline__ void combine(int nw, const Spinor<T>& acc, cx<T> out[NC])
    {
        if constexpr (LPS == 1) {
#pragma unroll
            for (int k = 0; k < 12; ++k) out[k] = acc.c[k / 3][k % 3];
            return;
        }
        T* b = buf + (size_t)half * nw * 24 * 32;
        half ^= 1;
        T* mine = b + (size_t)w * 24 * 32 + lane;
#pragma unroll
        for (int q = 0; q < PARTS; ++q)
            if (q != d) {
#pragma unroll
                for (int k = 0; k < NC; ++k) {
                    const cx<T> v = acc.c[(q * NC + k) / 3][(q * NC + k) % 3];
                    mine[(2 * (q * NC + k)) * 32] = v.re;
                    mine[(2 * (q * NC + k) + 1) * 32] = v.im;
                }
            } else {
#pragma unroll
                for (int k = 0; k < NC; ++k) out[k] = acc.c[(q * NC + k) / 3][(q * NC + k) % 3];
            }
        asm volatile("bar.sync %0, %1;" ::"r"(1 + sg), "r"(LPS * 32) : "memory");
        if (fin()) {
#pragma unroll
            for (int p = 1; p < LPS; ++p) {
                const int o = d ^ p;  // warp of the group
                const T* s = b + (size_t)(sg * LPS + o) * 24 * 32 + (size_t)(2 * d * NC) * 32 + lane;
#pragma unroll
                for (int k = 0; k < NC; ++k) out[k] = out[k] + mk(s[(2 * k) * 32], s[(2 * k + 1) * 32]);
            }
        }
    }
};

__device__ __forceinline__ void store_split(float4* p, double x, double y)
{
    const df a = df_split(x), b = df_split(y);
    *p = make_float4(a.hi, b.hi, a.lo, b.lo);
}

// part d (NC complex numbers) of the spinor whose word 0 is *v; single
// precision stores two complex numbers per float4
template <int NC>
__device__ __forceinline__ void load_part(const float4* v, int d, cx<float> o[NC])
{
    if constexpr (NC != 3) {
#pragma unroll
        for (int k = 0; k < NC / 2; ++k) {
            const float4 w = v[32 * (NC / 2 * d + k)];
            o[2 * k] = mk(w.x, w.y);
            o[2 * k + 1] = mk(w.z, w.w);
        }
    } else {
        const float2* v2 = (const float2*)v;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const int c = 3 * d + k;
            const float2 w = v2[64 * (c >> 1) + (c & 1)];
            o[k] = mk(w.x, w.y);
        }
    }
}
template <int NC>
__device__ __forceinline__ void store_part(float4* v, int d, const cx<float> o[NC])
{
    if constexpr (NC != 3) {
#pragma unroll
        for (int k = 0; k < NC / 2; ++k)
            v[32 * (NC / 2 * d + k)] = make_float4(o[2 * k].re, o[2 * k].im, o[2 * k + 1].re, o[2 * k + 1].im);
    } else {
        float2* v2 = (float2*)v;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const int c = 3 * d + k;
            v2[64 * (c >> 1) + (c & 1)] = make_float2(o[k].re, o[k].im);
        }
    }
}
template <int NC>
__device__ __forceinline__ void load_part(const double2* v, int d, cx<double> o[NC])
{
#pragma unroll
    for (int k = 0; k < NC; ++k) {
        const double2 w = v[32 * (d * NC + k)];
        o[k] = mk(w.x, w.y);
    }
}
template <int NC>
__device__ __forceinline__ void store_part(double2* v, int d, const cx<double> o[NC])
{
#pragma unroll
    for (int k = 0; k < NC; ++k) v[32 * (d * NC + k)] = make_double2(o[k].re, o[k].im);
}

template <int NC, class T>
__device__ __forceinline__ void pdot(const cx<T> a[NC], const cx<T> b[NC], T& re, T& im)
{
    re = im = 0;
#pragma unroll
    for (int k = 0; k < NC; ++k) {
        re += a[k].re * b[k].re + a[k].im * b[k].im;
        im += a[k].re * b[k].im - a[k].im * b[k].re;
    }
}
template <int NC, class T>
__device__ __forceinline__ T pnorm(const cx<T> a[NC])
{
    T s = 0;
#pragma unroll
    for (int k = 0; k < NC; ++k) s += a[k].re * a[k].re + a[k].im * a[k].im;
    return s;
}

// ---------------------------------------------------------------------------
// the kernel
// ---------------------------------------------------------------------------
template <int P, int LPS, int BS>
constexpr int split_smem()
{
    return LPS == 1 ? 0 : 2 * (BS / 32) * 24 * 32 * (int)sizeof(typename Real<P>::T);
}

// x, unknown to the compiler: the addresses of one phase are computed in it
// instead of being held in registers (and spilled) through all the others
__device__ __forceinline__ int opaque(int x)
{
    asm volatile("" : "+r"(x));
    return x;
}

// first site of the g-th group of 32 of a system, in the tiled order: a CTA's
// consecutive groups form a compact block of the lattice, whose hops meet in
// its L1 (a run of sites shares a spinor between 8 / 3.5 of its readers, a
// 4 x 4 tile between 8 / 2.5)
__device__ __forceinline__ int group_site(const SolveArgs& A, int g)
{
    if (!A.tiled) return g * 32;
    const int q = g & ((1 << A.lt[2]) - 1), i1 = (g >> A.lt[2]) & ((1 << A.lt[1]) - 1);
    const int i0 = (g >> (A.lt[1] + A.lt[2])) & ((1 << A.lt[0]) - 1);
    const int t = g >> (A.lt[0] + A.lt[1] + A.lt[2]);
    const int tq = t & ((1 << A.nt[1]) - 1), t1 = (t >> A.nt[1]) & ((1 << A.nt[0]) - 1), t0 = t >> (A.nt[0] + A.nt[1]);
    const int x0 = (t0 << A.lt[0]) + i0, x1 = (t1 << A.lt[1]) + i1;
    return (((((x0 << (A.nt[0] + A.lt[1])) + x1) << A.nt[1]) + tq) << (A.lt[2] + 5)) + (q << 5);
}

// Near a critical point the BiCGstab recurrence stalls: its residual stops
// falling for thousands of iterations, or for good, as rounding has it.  An
// inner solve that has gone `window` iterations without a new smallest |r|^2
// ends, and the outer cycle restarts it from the true residual of its best
// iterate (kept whenever |r| has halved), so a restart never adds a correction
// that is worse than its start.  It ends only where it has gained something,
// and where a cycle ended so has gained less than 1 / 0.3 the window doubles: a
// plateau that is longer than the window is waited out at the second or third
// try, and twelve decades take at most 23 such cycles and 7 doublings, fewer
// than the outer cycles allowed.  Iterations to 1e-12, four sources at 8x4^3
// near criticality (kappa = 0.15): double 2200-3100, single storage 3800-4700;
// restarted from the current iterate after a fixed 200: 2600-3900 and
// 6200-8600; not restarted: 11 600 to no convergence, and no convergence.
constexpr int STALL = 200;
constexpr double STALL_GAIN = 0.3;

// (site, word) items of the element-wise phases, B of them at a time so that
// their loads are in flight together: act(site, word, load(site, word)).  An
// item past the end repeats the last load and is not acted on.
template <int B, int NWD, int NW, class LD, class ACT>
__device__ __forceinline__ void for_words(const SolveArgs& A, int warp, int lane, int g0, int ngr, int base, LD load,
                                          ACT act)
{
    const int n = NWD * ngr;
    lane = opaque(lane);
    for (int u = warp; u < n; u += NW * B) {
        decltype(load(0, 0)) val[B];
        int i[B];
        bool in[B];
#pragma unroll
        for (int b = 0; b < B; ++b) {
            const int v = min(u + b * NW, n - 1), j = group_site(A, g0 + v / NWD) + lane;
            in[b] = u + b * NW < n && j < A.nsite;
            i[b] = base + min(j, A.nsite - 1);
            val[b] = load(i[b], v % NWD);
        }
#pragma unroll
        for (int b = 0; b < B; ++b)
            if (in[b]) act(i[b], (u + b * NW) % NWD, val[b]);
    }
}
template <class W>
struct W2 { W x, y; };
template <class W>
struct W3 { W r, v, p; };
template <class W>
struct W5 { W s, t, p, e, rh; };

template <int P, int LPS, int BS, int MINB, int METHOD>
__global__ void __launch_bounds__(BS, MINB) k_split(const __grid_constant__ SolveArgs A)
{
    typedef typename Real<P>::T T;
    typedef typename Word<P>::W W;
    constexpr int NWORD = Word<P>::N;
    constexpr int NW = BS / 32, SG = NW / LPS;
    // the residual sweeps read x, as df pairs (xs) around a single-precision
    // iteration, and their intermediate t64 in the same storage
    constexpr int PT = P == PREC64 ? PREC64 : PRECDS;
    typedef typename Real<PT>::T TR;
    typedef Xchg<T, LPS> X;
    constexpr int NC = X::NC;
    extern __shared__ __align__(16) unsigned char split_dyn[];
    __shared__ struct {
        double bn2, rn2, itol2;
        cx<double> rho, d, om;
        cx<T> alpha, omega, beta;  // rounded to the storage arithmetic
        // |r|^2: at the inner start, now, the smallest so far, that of the iterate
        // kept in A.eb; iterations since the smallest
        double start, rr, best, kept;
        int since, window, stalled, keep, use_kept;
        int idone, it, itc;
    } S;
    __shared__ double sums[METHOD == SOLVER_BICGSTAB ? 3 : 1][BS];

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    Group G;
    G.cps = A.cps;
    G.grp = blockIdx.x / A.cps;
    G.cin = blockIdx.x - G.grp * A.cps;
    G.epoch = 0;
    G.rb = 0;
    X xc;
    xc.buf = (T*)split_dyn;
    xc.w = warp;
    xc.d = LPS == 1 ? 0 : warp % LPS;
    xc.sg = warp / LPS;
    xc.lane = lane;
    xc.half = 0;
    const int d = xc.d;
    const int Vh = A.g.Vh;
    const GaugeF UP = A.UP;
    // the CTA's sites of a system, in groups of 32
    const int g0 = G.cin * (A.chunk >> 5);
    const int ngr = max(0, min(A.chunk >> 5, ((A.nsite + 31) >> 5) - g0));

#define V_(f) ((W*)A.f.v)
#define WORDS A, warp, lane, g0, ngr, base
// word k of site i: of an inner vector, of a double field
#define TW(i, k) (tile_at<P>(i) + 32 * (k))
#define DW(i, c) ((size_t)(c) * Vh + (i))
#define SYNC_OR_RETURN \
    if (!group_sync(A, G)) return
// sites of the CTA, a group of 32 per LPS warps; lanes past the end repeat the last site and store nothing
#define FOR_GROUPS                                                                \
    for (int gr_ = xc.sg; gr_ < ngr; gr_ += SG)                                   \
        if (const int j_ = group_site(A, g0 + gr_) + opaque(lane), i = base + min(j_, A.nsite - 1); true) \
            if (const bool on = j_ < A.nsite; true)                                    \
                if (const size_t at = tile_at<P>(i); true)
// (site, colour) items of the double sweeps
#define FOR_ITEMS                                                            \
    for (int u_ = warp; u_ < 3 * ngr; u_ += NW)                               \
        if (const int j_ = group_site(A, g0 + u_ / 3) + opaque(lane), r_ = u_ % 3; j_ < A.nsite)   \
            if (const int i = base + j_; true)
    for (int sys = G.grp; sys < A.nsys; sys += A.ngrp) {
        const int base = A.mode == MODE_INTRA ? (A.slab0 + sys * A.slabstep) * A.g.Sh : 0;
        const bool leader = G.cin == 0 && tid == 0;
        const double2* bb = (const double2*)A.b.v;
        double2* xx = (double2*)A.x.v;
        double2* r6 = (double2*)A.r64.v;
        const SpinorF xs = P == PREC64 ? A.x : A.s;

        // ---- |b|^2; from x = 0: r64 = b
        {
            double q[1] = {0.0};
            for_words<2, 12, NW>(
                WORDS, [&](int i, int c) { return __ldg(bb + DW(i, c)); },
                [&](int i, int c, double2 v) {
                    const size_t a = DW(i, c);
                    if (A.guess) {
                        if (P == PREC32) store_split((float4*)xs.v + a, xx[a].x, xx[a].y);
                    } else {
                        r6[a] = v;
                        xx[a] = make_double2(0.0, 0.0);
                    }
                    q[0] += v.x * v.x + v.y * v.y;
                });
            if (!group_reduce<NW, 1>(A, G, q, [&](const double(&n)[1]) {
                    S.bn2 = S.rn2 = n[0];
                    S.it = 0;
                    S.window = STALL;
                    S.stalled = 0;
                }))
                return;
        }
        // b = 0: the solution is 0, whatever the guess
        bool fresh = A.guess != 0;
        if (fresh && !(S.bn2 > 0.0)) {
            fresh = false;
            for (int u = warp; u < 12 * ngr; u += NW) {
                const int j = group_site(A, g0 + u / 12) + lane;
                if (j < A.nsite) xx[(size_t)(u % 12) * Vh + (base + j)] = make_double2(0.0, 0.0);
            }
        }

        int outer = 0, final_flag = F_DONE;
        for (;;) {
            // ---- x is new: r64 = b - diag x + k2 H_eo H_oe x in double-float (single
            // inner precision) or double arithmetic
            if (fresh) {
                FOR_ITEMS
                {
                    cx<TR> h[4];
                    hop_colour<PT, false>(A.g, A.mode, 0, 1, i, r_, xs, A.U64, h);
#pragma unroll
                    for (int s = 0; s < 4; ++s) store_comp<PT>(A.t64, 3 * s + r_, i, h[s]);
                }
                SYNC_OR_RETURN;
                double q[1] = {0.0};
                FOR_ITEMS
                {
                    cx<TR> h[4];
                    hop_colour<PT, false>(A.g, A.mode, 0, 0, i, r_, A.t64, A.U64, h);
#pragma unroll
                    for (int s = 0; s < 4; ++s) {
                        const size_t o = (size_t)(3 * s + r_) * Vh + i;
                        const double2 b2 = __ldg(bb + o), x2 = xx[o];
                        const double re = b2.x - A.diag * x2.x + A.k2 * as_double(h[s].re);
                        const double im = b2.y - A.diag * x2.y + A.k2 * as_double(h[s].im);
                        r6[o] = make_double2(re, im);
                        q[0] += re * re + im * im;
                    }
                }
                if (!group_reduce<NW, 1>(A, G, q, [&](const double(&n)[1]) {
                        // (S.rn2: the residual that the last inner solve started from)
                        if (S.stalled && !(n[0] <= STALL_GAIN * STALL_GAIN * S.rn2)) S.window *= 2;
                        S.stalled = 0;
                        S.rn2 = n[0];
                    })) return;
            }
            {
                // every CTA of the group takes the same decision from the same sums
                const bool nan = !isfinite(S.rn2);
                const bool conv = !(S.rn2 > A.tol * A.tol * S.bn2) || !(S.bn2 > 0.0);
                int f = nan ? F_NAN : conv ? F_DONE : F_ACTIVE;
                if (f == F_ACTIVE && (outer >= A.max_outer || S.it >= A.max_iter)) f = F_MAXIT;
                if (f != F_ACTIVE) {
                    final_flag = f;
                    break;
                }
            }
            ++outer;
            // ---- inner start: r = rh = p = r64 / |r64|, e = 0 (series: r = p)
            {
                Local<T> loc = Local<T>::zero();
                const double sc = 1.0 / sqrt(S.rn2);
                for_words<2, NWORD, NW>(
                    WORDS,
                    [&](int i, int k) {
                        // single precision: word k holds the complex numbers 2 k and 2 k + 1
                        if constexpr (P == PREC32) return W2<double2>{r6[DW(i, 2 * k)], r6[DW(i, 2 * k + 1)]};
                        else return r6[DW(i, k)];
                    },
                    [&](int i, int k, auto d) {
                        const size_t a = TW(i, k);
                        W w;
                        if constexpr (P == PREC32)
                            w = make_float4((float)(sc * d.x.x), (float)(sc * d.x.y), (float)(sc * d.y.x),
                                            (float)(sc * d.y.y));
                        else
                            w = make_double2(sc * d.x, sc * d.y);
                        V_(r)[a] = w;
                        V_(p)[a] = w;
                        if constexpr (METHOD == SOLVER_BICGSTAB) {
                            V_(rh)[a] = w;
                            V_(e)[a] = wzero(W());
                        }
                        loc.add(wnorm(w));
                    });
                double q[1] = {loc.value()};
                if (!group_reduce<NW, 1>(A, G, q, [&](const double(&n)[1]) {
                        S.rho = mk(n[0], 0.0);
                        S.start = S.rr = S.best = S.kept = n[0];
                        S.since = S.keep = S.use_kept = 0;
                        S.idone = 0;
                        S.itc = 0;
                        const double need = 0.5 * A.tol * sqrt(S.bn2 / fmax(S.rn2, 1e-300));
                        const double it = fmax(A.inner_tol, need);
                        S.itol2 = it * it;
                    }))
                    return;
            }

            if constexpr (METHOD == SOLVER_SERIES) {
                // ---- p <- (r + k2 H_eo H_oe p) / diag from p = r, the residual
                // reduced every second iteration (as in k_solve)
                const T k2 = (T)A.k2, dinv = (T)(1.0 / A.diag);
                for (;;) {
                    const bool chk = (S.itc & 1) || S.itc + 1 >= A.max_inner || S.it + 1 >= A.max_iter;
                    double q[1] = {0.0};
#pragma unroll 1
                    for (int par = 1; par >= 0; --par) {
                        const W* in = par ? V_(p) : V_(tmp);
                        FOR_GROUPS
                        {
                            Spinor<T> acc;
                            cx<T> o[NC];
                            hop_part<P, LPS>(A.g, A.mode, par, i, d, in, UP, acc);
                            xc.combine(NW, acc, o);
                            if (xc.fin() && on) {
                                if (par) {
                                    store_part<NC>(V_(tmp) + at, d, o);
                                } else {
                                    cx<T> pp[NC], rr[NC];
                                    load_part<NC>(V_(p) + at, d, pp);
                                    load_part<NC>(V_(r) + at, d, rr);
#pragma unroll
                                    for (int k = 0; k < NC; ++k) {
                                        o[k] = dinv * (rr[k] + k2 * o[k]);
                                        pp[k] = o[k] - pp[k];
                                    }
                                    store_part<NC>(V_(p) + at, d, o);
                                    if (chk) q[0] += (double)pnorm<NC>(pp);
                                }
                            }
                        }
                        if (par) SYNC_OR_RETURN;
                    }
                    if (!chk) {
                        SYNC_OR_RETURN;
                        if (tid == 0) {
                            S.it += 1;
                            S.itc += 1;
                        }
                        __syncthreads();
                        continue;
                    }
                    if (!group_reduce<NW, 1>(A, G, q, [&](const double(&n)[1]) {
                            S.it += 1;
                            S.itc += 1;
                            const double res2 = A.diag * A.diag * n[0];
                            if (!(res2 > S.itol2) || S.itc >= A.max_inner || S.it >= A.max_iter) S.idone = 1;
                            // a series that grows cannot converge: reported as not converged
                            if (!isfinite(res2) || (S.itc >= 16 && res2 > 1e6)) {
                                S.idone = 1;
                                S.it = A.max_iter;
                            }
                        }))
                        return;
                    if (S.idone) break;
                }
            } else {
                // ---- BiCGstab, seven barriers an iteration, three of them reducing:
                //   0  tmp = H_oe p        1  v = A p, <rh, v> -> alpha      s = r - alpha v
                //   2  tmp = H_oe s        3  t = A s, <t, s>, |t|^2 -> omega
                //   e += alpha p + omega s, r = s - omega t, <rh, r>, |r|^2 -> beta
                //   p = r + beta (p - omega v)
                // (<rh, r> and |r|^2 also follow from sums over s and t, without the
                // last reduction, but lose what one step reduces the residual by.)
                // One copy of the hopping code serves all four sweeps: it has to
                // fit the instruction cache.
                const T k2 = (T)A.k2, dg = (T)A.diag;
                bool stop = false;
                for (;;) {
#pragma unroll 1
                    for (int ph = 0; ph < 4; ++ph) {
                        const W* in = ph == 0 ? V_(p) : ph == 2 ? V_(r) : V_(tmp);
                        // the thread's sums wait in shared memory: six registers less in the hops
                        bool some = false;
                        FOR_GROUPS
                        {
                            Spinor<T> acc;
                            cx<T> o[NC];
                            hop_part<P, LPS>(A.g, A.mode, 1 - (ph & 1), i, d, in, UP, acc);
                            xc.combine(NW, acc, o);
                            if (xc.fin() && on) {
                                if (!(ph & 1)) {
                                    store_part<NC>(V_(tmp) + at, d, o);
                                } else {
                                    cx<T> y[NC], z[NC];
                                    load_part<NC>((ph == 1 ? V_(p) : V_(r)) + at, d, y);
#pragma unroll
                                    for (int k = 0; k < NC; ++k) o[k] = dg * y[k] - k2 * o[k];
                                    store_part<NC>((ph == 1 ? V_(v) : V_(t)) + at, d, o);
                                    T n[3];
                                    if (ph == 1) {
                                        load_part<NC>(V_(rh) + at, d, z);
                                        pdot<NC>(z, o, n[0], n[1]);
                                    } else {
                                        pdot<NC>(o, y, n[0], n[1]);
                                        n[2] = pnorm<NC>(o);
                                    }
#pragma unroll
                                    for (int k = 0; k < 3; ++k)
                                        if (k < 2 || ph == 3) sums[k][tid] = some ? sums[k][tid] + (double)n[k] : (double)n[k];
                                    some = true;
                                }
                            }
                        }
                        if (!(ph & 1)) {
                            SYNC_OR_RETURN;
                        } else if (ph == 1) {
                            double q[2] = {some ? sums[0][tid] : 0.0, some ? sums[1][tid] : 0.0};
                            if (!group_reduce<NW, 2>(A, G, q, [&](const double(&n)[2]) {
                                    const cx<double> dn = mk(n[0], n[1]);
                                    const cx<T> al = sround<T>(cdiv(S.rho, dn));
                                    S.d = dn;
                                    if (!fin2(al) || (n[0] == 0.0 && n[1] == 0.0)) {
                                        S.idone = 1;
                                        S.use_kept = S.kept < S.start && S.kept < S.rr;
                                    } else {
                                        S.alpha = al;
                                    }
                                }))
                                return;
                            if (S.idone) {  // the sums gave no step
                                stop = true;
                                break;
                            }
                            const cx<T> mal = -S.alpha;
                            for_words<3, NWORD, NW>(
                                WORDS, [&](int i, int k) { return W2<W>{V_(r)[TW(i, k)], V_(v)[TW(i, k)]}; },
                                [&](int i, int k, W2<W> w) { V_(r)[TW(i, k)] = waxpy(mal, w.y, w.x); });
                            SYNC_OR_RETURN;
                        } else {
                            double q[4] = {some ? sums[0][tid] : 0.0, some ? sums[1][tid] : 0.0, some ? sums[2][tid] : 0.0, 0.0};
                            if (!group_reduce<NW, 4>(A, G, q, [&](const double(&n)[4]) {
                                    const double inv = 1.0 / n[2];
                                    cx<double> om = mk(n[0] * inv, n[1] * inv);
                                    if (!(n[2] > 0.0) || !fin2(sround<T>(om))) {
                                        om = mk(0.0, 0.0);
                                        S.idone = 1;  // keep alpha p, stop afterwards
                                    }
                                    S.om = om;
                                    S.omega = sround<T>(om);
                                }))
                                return;
                        }
                    }
                    if (stop) break;
                    constexpr int B = P == PREC32 ? 3 : 2;
                    {
                        const cx<T> al = S.alpha, om = S.omega;
                        Local<T> l0 = Local<T>::zero(), l1 = l0, l2 = l0;
                        for_words<B, NWORD, NW>(
                            WORDS,
                            [&](int i, int k) {
                                const size_t a = TW(i, k);
                                return W5<W>{V_(r)[a], V_(t)[a], V_(p)[a], V_(e)[a], V_(rh)[a]};
                            },
                            [&](int i, int k, W5<W> w) {
                                const size_t a = TW(i, k);
                                V_(e)[a] = waxpy(om, w.s, waxpy(al, w.p, w.e));
                                const W rr = waxpy(-om, w.t, w.s);
                                V_(r)[a] = rr;
                                l0.add(wdot_re(w.rh, rr));
                                l1.add(wdot_im(w.rh, rr));
                                l2.add(wnorm(rr));
                            });
                        double q[4] = {l0.value(), l1.value(), l2.value(), 0.0};
                        if (!group_reduce<NW, 4>(A, G, q, [&](const double(&n)[4]) {
                                S.it += 1;
                                S.itc += 1;
                                const cx<double> rn = mk(n[0], n[1]);
                                const double rr = n[2];
                                // far above its start (1) the recurrence has diverged: keep the
                                // correction so far, the outer cycle recomputes the residual
                                if (S.itc >= A.max_inner || S.it >= A.max_iter || !(rr > S.itol2) || !fin2(rn) ||
                                    rr > 1e8)
                                    S.idone = 1;
                                S.rr = rr;
                                S.keep = rr < 0.25 * S.kept;
                                if (S.keep) S.kept = rr;
                                if (rr < S.best) {
                                    S.best = rr;
                                    S.since = 0;
                                } else if (++S.since >= S.window && S.kept < S.start && !S.idone) {
                                    S.idone = S.stalled = 1;
                                }
                                if (!S.idone) {
                                    // beta = (rn / rho) (alpha / omega) with alpha = rho / d
                                    S.beta = sround<T>(cdiv(rn, S.d * S.om));
                                    if (!fin2(S.beta)) S.idone = 1;
                                    S.rho = rn;
                                }
                                S.use_kept = S.kept < S.start && S.kept < rr;
                            }))
                            return;
                    }
                    if (S.idone) break;
                    if (S.keep)
                        for_words<B, NWORD, NW>(
                            WORDS, [&](int i, int k) { return V_(e)[TW(i, k)]; },
                            [&](int i, int k, W w) { V_(eb)[TW(i, k)] = w; });
                    {
                        const cx<T> om = S.omega, be = S.beta;
                        for_words<B, NWORD, NW>(
                            WORDS,
                            [&](int i, int k) {
                                const size_t a = TW(i, k);
                                return W3<W>{V_(r)[a], V_(v)[a], V_(p)[a]};
                            },
                            [&](int i, int k, W3<W> w) { V_(p)[TW(i, k)] = waxpy(be, waxpy(-om, w.v, w.p), w.r); });
                    }
                    SYNC_OR_RETURN;
                }
            }

            // ---- x += |r64| e
            {
                const double sc = sqrt(S.rn2);
                const W* ev = METHOD == SOLVER_SERIES ? V_(p) : S.use_kept ? V_(eb) : V_(e);
                for_words<2, 12, NW>(
                    WORDS,
                    [&](int i, int c) {
                        W2<double2> r;
                        r.x = xx[DW(i, c)];
                        if constexpr (P == PREC32) {
                            const float2 w = ((const float2*)ev)[TW(i, c >> 1) * 2 + (c & 1)];
                            r.y = make_double2(w.x, w.y);
                        } else {
                            r.y = ev[TW(i, c)];
                        }
                        return r;
                    },
                    [&](int i, int c, W2<double2> w) {
                        const size_t a = DW(i, c);
                        const double re = w.x.x + sc * w.y.x, im = w.x.y + sc * w.y.y;
                        xx[a] = make_double2(re, im);
                        if (P == PREC32) store_split((float4*)xs.v + a, re, im);
                    });
            }
            SYNC_OR_RETURN;
            fresh = true;
        }

        if (leader) {
            A.iters[sys] = S.it;
            A.resid[sys] = S.bn2 > 0.0 ? sqrt(S.rn2 / S.bn2) : 0.0;
            if (sys == 0) *A.outer_out = outer;
            const int err = final_flag == F_NAN ? LQCD_ERR_NAN : final_flag == F_MAXIT ? LQCD_ERR_NOCONVERGE : 0;
            if (err) {
                atomicCAS(A.status, 0, err);
                atomicCAS(A.sticky, 0, err);
            }
            atomicAdd(A.acc, (unsigned long long)S.it);
            atomicAdd(A.acc + (METHOD == SOLVER_SERIES ? 3 : 1), (unsigned long long)S.it * (unsigned long long)A.nsite);
            atomicAdd(A.acc + 2, (unsigned long long)outer * (unsigned long long)A.nsite);
        }
        __syncthreads();  // S belongs to the next system from here on
    }
#undef V_
#undef SYNC_OR_RETURN
#undef FOR_GROUPS
#undef FOR_ITEMS
#undef WORDS
#undef TW
#undef DW
}

}  // namespace

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
namespace {

struct Variant {
    const void* fn[2];  // BiCGstab, series
    int prec, lps, bs, smem;
};

template <int P, int LPS, int BS, int MINB>
constexpr Variant variant()
{
    return Variant{{(const void*)k_split<P, LPS, BS, MINB, SOLVER_BICGSTAB>,
                    (const void*)k_split<P, LPS, BS, MINB, SOLVER_SERIES>},
                   P, LPS, BS, split_smem<P, LPS, BS>()};
}

enum { V_F64 = 0, V_8, V_4, V_2, V_1, V_1W };
const Variant variants[SPLIT_NVAR] = {variant<PREC64, 8, 256, 2>(), variant<PREC32, 8, 256, 2>(),
                                      variant<PREC32, 4, 256, 2>(), variant<PREC32, 2, 256, 2>(),
                                      variant<PREC32, 1, 256, 2>(), variant<PREC32, 1, 512, 1>()};

// The kernel for `groups` groups of 32 sites over all systems.  Double
// precision is bound by the FP64 pipe: eight warps a group, two CTAs per SM so
// that one computes while the other's loads or barriers are under way (at
// 128 registers a thread; one CTA of 255 registers: 64x32^3 global 206 ms
// instead of 171, its series 123 / 99.5, 32x16^3 global 13.7 / 12.6; one thread
// per site: 198, 112, 15.5).  Single precision, measured (ms per solve, LPS 8 / 4 / 2 / 1):
// 41 groups 1.72 / 1.84 / 2.09 / 2.42, 128 groups 1.97 / 1.96 / 2.20 / 2.77, 250
// groups 2.39 / 2.07 / 2.26 / 2.81, 540 groups 2.88 / 2.60 / 2.43 / 2.79, 648
// groups 3.39 / 3.03 / 2.94 / 2.91, 1024 groups 3.69 / 3.33 / 2.97 / 2.98, 2048
// groups 5.83 / 5.01 / 4.53 / 4.22: LPS 8 while every group has an SM of its own,
// then 4 and 2 while the groups still fit the SMs side by side.  From 2432
// groups on (more than two CTAs of eight groups per SM) one CTA of 512 threads
// per SM halves the barrier's arrivals (2450 groups 5.64 against 5.74, 3072
// groups 6.15 / 6.37, 6912 groups 13.44 / 13.49).
int pick(int prec, int groups, int num_sms)
{
    if (prec == PREC64) return V_F64;
    if (8 * groups <= 7 * num_sms) return V_8;
    if (groups <= 2 * num_sms) return V_4;
    if (groups <= 4 * num_sms) return V_2;
    return groups <= 16 * num_sms ? V_1 : V_1W;
}

// How many of the systems a launch works on at a time.  What a series iteration
// of all of them reads and writes again (three vectors of 96 bytes a site and
// 384 of links) may not fit the L2; a part of the systems does, and the sweeps
// are bound by L2 traffic.  Full waves only (a divisor of the number of systems;
// an uneven last wave leaves SMs idle: eight systems of 32000 sites by three
// 6.68 ms, by four 5.81, at once 6.41), each within three quarters of the L2 and
// wide enough to fill the chip.  Measured (ms at 66 iterations, at once -> in
// these waves): 8 x 30976 sites 6.34 -> 5.39, 8 x 55296 10.87 -> 10.54, 4 x 131072
// 12.27 -> 11.51, 4 x 55296 5.26 -> 5.17 (122 iterations: 8.02 -> 7.64),
// 8 x 131072 23.8 -> 23.3; with few iterations the waves' start and end weigh
// more (38: 4 x 55296 3.83 -> 3.85, 8 x 131072 17.0 -> 17.4).  BiCGstab, seven
// vectors, runs at once: waves 0-29 % slower (10 x 27648 5.07 ms, by four 6.5;
// 4 x 46080 3.69, by two 3.92; the best of them, 8 x 30976 by four, 2 % faster).
int systems_at_once(const SolveArgs& A, int prec, int method, int num_sms, int l2)
{
    const double set = (3 * 96.0 + 384.0) * A.nsite;
    if (prec != PREC32 || method != SOLVER_SERIES || set * A.nsys <= l2) return A.nsys;
    int at = A.nsys;
    while (at > 1 && (A.nsys % at != 0 || set * at > 0.75 * l2)) --at;
    return set * at <= 0.75 * l2 && (A.nsite + 31) / 32 * at >= 20 * num_sms ? at : A.nsys;
}

}  // namespace

cudaError_t split_init(int num_sms, int occ[SPLIT_NVAR][2], int* gmax, int* l2)
{
    *gmax = 0;
    int dev;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(l2, cudaDevAttrL2CacheSize, dev);
    if (e != cudaSuccess) return e;
    for (int k = 0; k < SPLIT_NVAR; ++k)
        for (int m = 0; m < 2; ++m) {
            const Variant& v = variants[k];
            e = cudaFuncSetAttribute(v.fn[m], cudaFuncAttributeMaxDynamicSharedMemorySize, v.smem);
            if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ[k][m], v.fn[m], v.bs, v.smem);
            if (e != cudaSuccess) return e;
            if (occ[k][m] < 1) return cudaErrorLaunchOutOfResources;
            *gmax = std::max(*gmax, occ[k][m] * num_sms);
        }
    return cudaSuccess;
}

SplitPlan split_plan(SolveArgs& A, int prec, int method, int spt, int num_sms, const int occ[SPLIT_NVAR][2],
                     int l2)
{
    const int G = (A.nsite + 31) / 32;
    A.ngrp = systems_at_once(A, prec, method, num_sms, l2);
    const int k = pick(prec, G * A.ngrp, num_sms), m = method == SOLVER_SERIES ? 1 : 0;
    const Variant& v = variants[k];
    const int SG = v.bs / 32 / v.lps;  // groups a CTA holds side by side
    const int want = spt <= 0 ? G : (G + SG * spt - 1) / (SG * spt);
    auto groups_per_cta = [&](int per_sm) {
        A.cps = std::max(1, std::min(per_sm * num_sms / A.ngrp, want));
        return (G + A.cps - 1) / A.cps;
    };
    // Double precision: the FP64 pipe of the SM with the most groups sets the
    // time, so one CTA per SM where two would leave that SM with over a tenth
    // more groups (420 groups by two 3.61 ms, by one 3.11; 1024: 6.94 / 6.51,
    // 2048, where both give 14: 12.6 / 13.7)
    int per_sm = occ[k][m];
    if (prec == PREC64 && per_sm > 1) {
        auto most = [&](int n) {
            const int gpc = groups_per_cta(n), ctas = (G + gpc - 1) / gpc * A.ngrp;
            return (ctas + num_sms - 1) / num_sms * gpc;
        };
        if (11 * most(1) < 10 * most(per_sm)) per_sm = 1;
    }
    const int gpc = groups_per_cta(per_sm);
    A.cps = (G + gpc - 1) / gpc;
    A.chunk = gpc * 32;
    // tiles of 16 groups where the CTAs make several passes (64x32^3: 420
    // against 454 ms) and whole planes are whole groups; a single pass is no
    // faster for it (32x16^3: 23.0 against 22.3)
    A.tiled = 0;
    const Geo& g = A.g;
    const int plane = g.L[2] * g.L[3] / 2;
    if (gpc > SG && g.lg[0] && plane >= 32) {
        int left = 4;
        auto take = [&](int n, int most) {
            int l = 0;
            while (l < most && l < left && n % (2 << l) == 0) ++l;
            left -= l;
            return l;
        };
        A.lt[0] = take(A.nsite / (g.L[1] * plane), 2);
        A.lt[1] = take(g.L[1], 2);
        A.lt[2] = take(plane / 32, 4);
        A.nt[0] = g.lg[1] - A.lt[1];
        A.nt[1] = g.lg[2] + g.lg[3] - 6 - A.lt[2];
        A.tiled = 1;
    }
    return SplitPlan{v.fn[m], A.cps * A.ngrp, v.bs, v.smem};
}
