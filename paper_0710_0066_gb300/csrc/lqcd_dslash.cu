// lqcd_dslash.cu -- the hopping term of eq. (2) as one sweep over the output
// sites of one parity: out = a x + c H_{p,1-p} in, optionally restricted to
// the hops inside one x0-slab (W1) or between slabs (the blocks B, C of M),
// and to the output sites of the slabs of one colour.
//
// One thread per output site.  Every neighbour is read as a full spinor
// with 128-bit (single: float4, half: uint4) or 2x64-bit (double2) loads of
// consecutive sites, spin-projected to a half spinor, multiplied by the
// (rebuilt) link and accumulated; the output is written once.
#include <algorithm>

#include "lqcd_common.cuh"

namespace {

// block size chosen at run time (lqcd_autotune), at most HOP_BS_MAX
constexpr int HOP_BS_MAX = 256;

// acc += sc (1 + sg gamma_mu) psi rebuilt from its upper half w (the
// multiplication by sc fused into the accumulation)
__device__ __forceinline__ void accum_recon_sc(int mu, int sg, const HalfSp<float>& w, float sc, Spinor<float>& acc)
{
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        cx<float> l0, l1;
        switch (mu) {
            case 0: l0 = -w.c[0][i]; l1 = -w.c[1][i]; break;
            case 1: l0 = mul_i(w.c[1][i]); l1 = mul_i(w.c[0][i]); break;
            case 2: l0 = w.c[1][i]; l1 = -w.c[0][i]; break;
            default: l0 = mul_i(w.c[0][i]); l1 = mul_mi(w.c[1][i]); break;
        }
        const float sl = sg < 0 ? -sc : sc;
        acc.c[0][i] = mk(acc.c[0][i].re + sc * w.c[0][i].re, acc.c[0][i].im + sc * w.c[0][i].im);
        acc.c[1][i] = mk(acc.c[1][i].re + sc * w.c[1][i].re, acc.c[1][i].im + sc * w.c[1][i].im);
        acc.c[2][i] = mk(acc.c[2][i].re + sl * l0.re, acc.c[2][i].im + sl * l0.im);
        acc.c[3][i] = mk(acc.c[3][i].re + sl * l1.re, acc.c[3][i].im + sl * l1.im);
    }
}

// the hopping term at one output site for half storage: each neighbour is
// converted without its per-site scale, projected and multiplied by the
// link, and the scale (with the x0 boundary sign) enters once, in the
// accumulation: the same sum as hop_site<PREC16> with 24 fewer
// multiplications per hop
__device__ __forceinline__ void hop_site_h16(const Geo& g, int mode, int dag, int pout, int i, const SpinorF& in,
                                             const GaugeF& U, Spinor<float>& acc)
{
#pragma unroll
    for (int s = 0; s < 4; ++s)
#pragma unroll
        for (int c = 0; c < 3; ++c) acc.c[s][c] = mk(0.f, 0.f);
    int x[4];
    eo_coords(g, pout, i, x);
    const int lex = lex_of(g, x);
    int stride = 1;
    const int pin = 1 - pout;
    const uint4* pv = (const uint4*)in.v;
    auto ld = [&](int j, Spinor<float>& sp) -> float {
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const uint4 d = __ldg(pv + (size_t)k * in.N + j);
            const unsigned w[4] = {d.x, d.y, d.z, d.w};
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const float2 v = __half22float2(*reinterpret_cast<const __half2*>(&w[q]));
                const int cc = 4 * k + q;
                sp.c[cc / 3][cc % 3] = mk(v.x, v.y);
            }
        }
        return __ldg(in.nrm + j);
    };
#pragma unroll
    for (int mu = 3; mu >= 0; --mu) {
        {
            int nl = lex + stride;
            const bool wrap = (x[mu] == g.L[mu] - 1);
            if (wrap) nl -= g.L[mu] * stride;
            bool use = true;
            if (mu == 0) use = t_hop_kept(g, mode, x[0] + 1);
            else if (mode == MODE_CROSS || mode == MODE_CROSS2) use = false;
            if (use) {
                Spinor<float> ps;
                float sc = ld(nl >> 1, ps);
                Su3<float> u;
                load_link<PREC16>(U, mu, pout, i, u);
                HalfSp<float> h, w;
                const int sg = dag ? +1 : -1;
                project(mu, sg, ps, h);
                su3_mul_half(u, h, w);
                if (mu == 0 && wrap && g.bc_t < 0) sc = -sc;
                accum_recon_sc(mu, sg, w, sc, acc);
            }
        }
        {
            int nl = lex - stride;
            const bool wrap = (x[mu] == 0);
            if (wrap) nl += g.L[mu] * stride;
            bool use = true;
            if (mu == 0) use = t_hop_kept(g, mode, x[0]);
            else if (mode == MODE_CROSS || mode == MODE_CROSS2) use = false;
            if (use) {
                Spinor<float> ps;
                float sc = ld(nl >> 1, ps);
                Su3<float> u;
                load_link<PREC16>(U, mu, pin, nl >> 1, u);
                HalfSp<float> h, w;
                const int sg = dag ? -1 : +1;
                project(mu, sg, ps, h);
                su3_dagmul_half(u, h, w);
                if (mu == 0 && wrap && g.bc_t < 0) sc = -sc;
                accum_recon_sc(mu, sg, w, sc, acc);
            }
        }
        stride *= g.L[mu];
    }
}

// The warp's 32 results to the C-ABI layout, double[site][4][3][2]: each
// lane's 24 numbers pass through shared memory (rows of 13: no bank conflict
// beyond the width) so that the stores run along the sites.  Stored straight
// from the lanes, 192 bytes apart, every 32-byte sector is written in two
// halves.  S: the type a result fits exactly; `i`, `on` per lane.
// An operator call is bound by HBM; its C-ABI field alone is 192 bytes a site
// each way, so passes over it are what counts: packing to double, converting,
// sweeping, converting back, unpacking and the clearing of a result that is
// written in full moved 1900 bytes a site in single precision, packing
// straight to the sweep's storage and this store 864.  A call at 64x32^3 in
// single precision 506 -> 178 us, at 32x24^3 in half precision 117 -> 44 us.
template <class S>
struct Pair {
    S re, im;
};
template <class S, int NC, class T>
__device__ __forceinline__ void abi_store(Pair<S>* sh, double2* abi, int i, bool on, const Spinor<T>& acc)
{
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int c0 = 0; c0 < 12; c0 += NC) {
        __syncwarp();
#pragma unroll
        for (int k = 0; k < NC; ++k) {
            const cx<T> v = acc.c[(c0 + k) / 3][(c0 + k) % 3];
            sh[lane * (NC + 1) + k] = Pair<S>{(S)v.re, (S)v.im};
        }
        __syncwarp();
#pragma unroll
        for (int k = 0; k < NC; ++k) {
            const int e = k * 32 + lane, site = e / NC, c = e % NC;
            const int j = __shfl_sync(0xffffffffu, i, site);
            const bool ok = __shfl_sync(0xffffffffu, (int)on, site) != 0;
            const Pair<S> v = sh[site * (NC + 1) + c];
            if (ok) abi[(size_t)j * 12 + c0 + c] = make_double2((double)v.re, (double)v.im);
        }
    }
}

// complex numbers of a site that pass through shared memory at a time, and
// the shared memory of a block
template <int P>
constexpr int abi_chunk()
{
    return P == PREC64 ? 6 : 12;
}
template <int P>
constexpr int abi_smem(int bs)
{
    return bs * (abi_chunk<P>() + 1) * 2 * (int)sizeof(typename Real<P>::T);
}

template <int P, bool ABI>
__device__ __forceinline__ void hop_body(Geo g, int mode, int dag, int pout, int colour, SpinorF out, SpinorF in,
                                         GaugeF U, double a, SpinorF x, double c, int nsites, double2* abi)
{
    typedef typename Real<P>::T T;
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    const bool on = t < nsites;
    if (!ABI && !on) return;
    int i = on ? t : nsites - 1;
    bool mine = true;
    if (colour >= 0) {
        // with ABI every site: first the colour's, then zeros on the other
        // slabs (the sites in their own order would give one SM two blocks of
        // work and the next none: 16^4 in double 0.168 ms instead of 0.131)
        const int half = (g.nb / 2) * g.Sh;
        mine = !ABI || i < half;
        const int u = mine ? i : i - half, k = u / g.Sh;
        i = ((mine ? colour : 1 - colour) + 2 * k) * g.Sh + (u - k * g.Sh);
    }
    Spinor<T> acc;
    if (mine) {
        if constexpr (P == PREC16)
            hop_site_h16(g, mode, dag, pout, i, in, U, acc);
        else
            hop_site<P>(g, mode, dag, pout, i, in, U, acc);
        const T cc = (T)c;
        if (x.v) {
            Spinor<T> xs;
            load_spinor<P>(x, i, xs);
            const T aa = (T)a;
#pragma unroll
            for (int s = 0; s < 4; ++s)
#pragma unroll
                for (int q = 0; q < 3; ++q) acc.c[s][q] = aa * xs.c[s][q] + cc * acc.c[s][q];
        } else {
#pragma unroll
            for (int s = 0; s < 4; ++s)
#pragma unroll
                for (int q = 0; q < 3; ++q) acc.c[s][q] = cc * acc.c[s][q];
        }
    } else {
#pragma unroll
        for (int s = 0; s < 4; ++s)
#pragma unroll
            for (int q = 0; q < 3; ++q) acc.c[s][q] = mk(T(0), T(0));
    }
    if constexpr (ABI) {
        // half storage rounds the result to the storage format: through it
        extern __shared__ __align__(16) unsigned char hop_dyn[];
        constexpr int NC = abi_chunk<P>();
        if constexpr (P == PREC16 || P == PRECBF) round_spinor<P>(acc);
        abi_store<T, NC>((Pair<T>*)hop_dyn + (threadIdx.x >> 5) * 32 * (NC + 1), abi, i, on, acc);
    } else {
        store_spinor<P>(out, i, acc);
    }
}

template <int P, bool ABI>
__global__ void __launch_bounds__(HOP_BS_MAX) k_hop(Geo g, int mode, int dag, int pout, int colour, SpinorF out,
                                               SpinorF in, GaugeF U, double a, SpinorF x, double c, int nsites,
                                               double2* abi)
{
    hop_body<P, ABI>(g, mode, dag, pout, colour, out, in, U, a, x, c, nsites, abi);
}

// The double-float sweep: bound by issue and by the length of its dependent
// chains, so a site is three items, one per colour of the result: warp
// 3 k + r takes colour r of 32 sites.  (A neighbour is split and projected
// once per colour, out of L1.)  Small lattices gain most, one thread per site
// left the chip idle there: trajectory at 8x4^3 24.0 -> 20.6 ms, at 32x16^3
// 321 -> 319 ms.
__global__ void __launch_bounds__(HOP_BS_MAX, 3) k_hop_df(Geo g, int mode, int dag, int pout, int colour, SpinorF out,
                                                     SpinorF in, GaugeF U, double a, SpinorF x, double c, int nsites)
{
    const int w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, k = w / 3, r = w - 3 * k;
    const int t = 32 * k + (threadIdx.x & 31);
    if (t >= nsites) return;
    const int q = colour < 0 ? 0 : t / g.Sh;
    const int i = colour < 0 ? t : (colour + 2 * q) * g.Sh + (t - q * g.Sh);
    cx<df> acc[4];
    hop_colour<PRECDF, true>(g, mode, dag, pout, i, r, in, U, acc);
    const df aa(a), cc(c);
#pragma unroll
    for (int s = 0; s < 4; ++s) {
        cx<df> v = cc * acc[s];
        if (x.v) v = aa * load_comp<PRECDF, true>(x, 3 * s + r, i) + v;
        ((double2*)out.v)[(size_t)(3 * s + r) * out.N + i] = make_double2(as_double(v.re), as_double(v.im));
    }
}

}  // namespace

// algorithmic DRAM bytes of one output site: the output, the input site and
// the eight links, each moved once (neighbour spinors reused from cache)
double hop_site_bytes(int prec, bool with_x, bool abi)
{
    const bool dbl = prec == PREC64 || prec == PRECDF;
    const double sp = dbl ? 192.0 : prec == PREC32 ? 96.0 : prec == PREC16 ? 52.0 : 48.0;
    const double lk = dbl ? 144.0 : prec == PREC32 ? 48.0 : 24.0;
    return sp + (abi ? 192.0 : sp) + 8.0 * lk + (with_x ? sp : 0.0);
}

int hop_sweep(lqcd_ctx* h, int prec, int mode, int dag, int pout, int colour, SpinorF out, SpinorF in,
              double a, SpinorF x, double c, double2* abi)
{
    const Geo& g = h->g;
    const int nsites = colour < 0 || abi ? g.Vh : (g.nb / 2) * g.Sh;
    const int bs = std::min(std::max(h->tune.hop_bs[prec == PRECDF ? PREC64 : prec], 32), HOP_BS_MAX);  // whole warps
    const int nb = (nsites + bs - 1) / bs;
    GaugeF U = gauge_view(h, prec);
    cudaEvent_t ev;
    prof_begin(h, 0, &ev);
#define HOP(P)                                                                                                     \
    do {                                                                                                           \
        if (abi)                                                                                                   \
            k_hop<P, true><<<nb, bs, abi_smem<P>(bs), h->stream>>>(g, mode, dag, pout, colour, out, in, U, a, x, c, \
                                                                   nsites, abi);                                   \
        else                                                                                                       \
            k_hop<P, false><<<nb, bs, 0, h->stream>>>(g, mode, dag, pout, colour, out, in, U, a, x, c, nsites, abi); \
    } while (0)
    if (prec == PREC64) HOP(PREC64);
    else if (prec == PRECDF)
        k_hop_df<<<((nsites + 31) / 32 * 96 + bs - 1) / bs, bs, 0, h->stream>>>(g, mode, dag, pout, colour, out, in, U, a, x, c, nsites);
    else if (prec == PREC32) HOP(PREC32);
    else if (prec == PREC16) HOP(PREC16);
    else HOP(PRECBF);
#undef HOP
    h->launches += 1;
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) {
        h->err = std::string("hop kernel: ") + cudaGetErrorString(e);
        return LQCD_ERR_CUDA;
    }
    prof_end(h, 0, ev, hop_site_bytes(prec, x.v != nullptr, abi != nullptr) * nsites);
    return LQCD_OK;
}
