// Wilson hopping term ("dslash") on one parity, with fused epilogues.
//
//   out_p(x) = epi( sum_mu (1 - g_mu) U_mu(x) in(x+mu) + (1 + g_mu) U_mu(x-mu)^dag in(x-mu) )
//
// (the matrix-vector product the paper identifies as the dominant cost of
// every Krylov solver, Sec. 3 and Sec. 5; even-odd splitting makes each
// application touch one parity of output and the other of input, Sec. 5).
//
// One thread per output site (launches that reduce stride over the sites
// with one wave of blocks).  Every neighbour spinor is spin-projected to
// a half spinor (two colour vectors) before the SU(3) multiply and
// reconstructed afterwards, which is the 1320-flop form of the operator.
// The adjoint (DAG) swaps the projectors, since H^dag = g5 H g5.  The t
// boundary sign multiplies the half spinor of hops that cross t = Lt-1 <-> 0.
//
// Epilogues, in the compute precision:
//   EPI_NONE     out = a * D
//   EPI_CLOVINV  out = a * Cl D                  (Cl = A^{-1} of the output parity)
//   EPI_XPAY     out = Cl y + a * D               (Cl = A, or 1 without clover)
//   EPI_CG       s = Cl y + a * D; r -= alpha s  (s never stored); x += alpha p unless A.x is null
// and optionally (RED) the grid sum of |out|^2 (|r|^2 for EPI_CG) in FP64.
#pragma once
#include "core.cuh"

namespace lqcd {

enum Epi { EPI_NONE = 0, EPI_CLOVINV = 1, EPI_XPAY = 2, EPI_CG = 3 };

struct DslashArgs {
    Geom g;
    int par;                 // output parity
    void* out;               // output fields (EPI_CG: unused)
    size_t out_rb;           // bytes between right-hand sides
    const void* in;          // input fields, parity 1 - par
    size_t in_rb;
    const void* gauge;       // gauge copy of this precision / recon
    const void* clov;        // clover field of the output parity, or nullptr (= 1)
    const void* y;           // EPI_XPAY / EPI_CG: field of the output parity
    size_t y_rb;
    double a;                // coefficient of the hopping term
    // reductions (RED): per rhs r, partials + r * part_rs, tickets[r], red + r * red_rs
    double* partials;
    size_t part_rs;
    unsigned* tickets;
    double* red;
    size_t red_rs;
    // EPI_CG: x, r in the accumulation precision; p in P; scalars per rhs
    void* x;
    void* r;
    size_t acc_rb;
    const void* p;
    size_t p_rb;
    const double* scal;      // per rhs: scal + r * scal_rs
    size_t scal_rs;
    int s_num, s_num2;       // alpha = (scal[s_num] + scal[s_num2]) / (scal[s_den] + scal[s_den2])
    int s_den, s_den2;
    const int* skip;         // per rhs: nonzero = converged, do nothing (may be nullptr)
    int sites_per_thread;    // reducing launches: grid of Vh / (block * this); 0 = one wave of blocks
    int nrhs;                // right-hand sides of the launch (set by the launcher)
    int plain;               // not under the predecessor's tail (see launch_dslash)
};

// ---- spin projection (1 + S g_mu), S = -1 or +1, onto two colour vectors
template <int MU, int S, class R>
__device__ __forceinline__ void project(const R v[24], R h[12])
{
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const R p0r = v[2 * c], p0i = v[2 * c + 1];
        const R p1r = v[2 * (3 + c)], p1i = v[2 * (3 + c) + 1];
        const R p2r = v[2 * (6 + c)], p2i = v[2 * (6 + c) + 1];
        const R p3r = v[2 * (9 + c)], p3i = v[2 * (9 + c) + 1];
        R h0r, h0i, h1r, h1i;
        if (MU == 0) {        // h0 = p0 + S i p3, h1 = p1 + S i p2
            h0r = p0r - S * p3i; h0i = p0i + S * p3r;
            h1r = p1r - S * p2i; h1i = p1i + S * p2r;
        } else if (MU == 1) { // h0 = p0 - S p3, h1 = p1 + S p2
            h0r = p0r - S * p3r; h0i = p0i - S * p3i;
            h1r = p1r + S * p2r; h1i = p1i + S * p2i;
        } else if (MU == 2) { // h0 = p0 + S i p2, h1 = p1 - S i p3
            h0r = p0r - S * p2i; h0i = p0i + S * p2r;
            h1r = p1r + S * p3i; h1i = p1i - S * p3r;
        } else {              // h0 = p0 + S p2, h1 = p1 + S p3
            h0r = p0r + S * p2r; h0i = p0i + S * p2i;
            h1r = p1r + S * p3r; h1i = p1i + S * p3i;
        }
        h[2 * c] = h0r; h[2 * c + 1] = h0i;
        h[2 * (3 + c)] = h1r; h[2 * (3 + c) + 1] = h1i;
    }
}

// ---- reconstruct the lower spins from the two rotated colour vectors
template <int MU, int S, class R>
__device__ __forceinline__ void accumulate(R acc[24], const R w[12])
{
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const R w0r = w[2 * c], w0i = w[2 * c + 1];
        const R w1r = w[2 * (3 + c)], w1i = w[2 * (3 + c) + 1];
        acc[2 * c] += w0r; acc[2 * c + 1] += w0i;
        acc[2 * (3 + c)] += w1r; acc[2 * (3 + c) + 1] += w1i;
        R r2r, r2i, r3r, r3i;
        if (MU == 0) {        // r2 = -S i w1, r3 = -S i w0
            r2r = S * w1i; r2i = -S * w1r;
            r3r = S * w0i; r3i = -S * w0r;
        } else if (MU == 1) { // r2 = S w1, r3 = -S w0
            r2r = S * w1r; r2i = S * w1i;
            r3r = -S * w0r; r3i = -S * w0i;
        } else if (MU == 2) { // r2 = -S i w0, r3 = S i w1
            r2r = S * w0i; r2i = -S * w0r;
            r3r = -S * w1i; r3i = S * w1r;
        } else {              // r2 = S w0, r3 = S w1
            r2r = S * w0r; r2i = S * w0i;
            r3r = S * w1r; r3i = S * w1i;
        }
        acc[2 * (6 + c)] += r2r; acc[2 * (6 + c) + 1] += r2i;
        acc[2 * (9 + c)] += r3r; acc[2 * (9 + c) + 1] += r3i;
    }
}

// Both hops of a direction in one, from the sum s = w_f + w_b of the forward
// and the backward product and their difference d; S is the forward sign (the
// backward hop's lower spins are those of -w_b under it).
// FP64: s costs nothing where the backward products are chained onto w_f, d =
// 2 w_f - s takes 12 multiply-adds, and the first direction is assigned: 192
// additions of the 864 FP64 operations of a site's hops become 120, on the
// pipe that bounds the kernel (93 % busy).  24^4 hop 282 -> 274 us, Schur
// operator 716 -> 700; 16^4 with 16 rhs, full operator, 2126 -> 2078.
template <int MU, int S, class R>
__device__ __forceinline__ void accumulate_pair(R acc[24], const R s[12], const R d[12])
{
    constexpr int from[4] = {1, 1, 0, 0};         // lower spin 2 is made of d's vector 1 (mu = 0, 1) or 0
    constexpr bool turned = MU == 0 || MU == 2;  // by -S i or S i, else by a sign
    constexpr int s2 = MU == 0 || MU == 2 ? -S : S, s3 = MU == 0 || MU == 1 ? -S : S;
#pragma unroll
    for (int k = 0; k < 12; ++k) acc[k] = MU == 0 ? s[k] : acc[k] + s[k];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const R* const x2 = d + 2 * (3 * from[MU] + c);
        const R* const x3 = d + 2 * (3 * (1 - from[MU]) + c);
        // s i (re + i im) = -s im + i s re
        const R r2r = turned ? -s2 * x2[1] : s2 * x2[0], r2i = turned ? s2 * x2[0] : s2 * x2[1];
        const R r3r = turned ? -s3 * x3[1] : s3 * x3[0], r3i = turned ? s3 * x3[0] : s3 * x3[1];
        R* const a2 = acc + 2 * (6 + c);
        R* const a3 = acc + 2 * (9 + c);
        a2[0] = MU == 0 ? r2r : a2[0] + r2r;
        a2[1] = MU == 0 ? r2i : a2[1] + r2i;
        a3[0] = MU == 0 ? r3r : a3[0] + r3r;
        a3[1] = MU == 0 ? r3i : a3[1] + r3i;
    }
}

// w = U h (ADJ = false) or U^dag h (ADJ = true) for both colour vectors of h.
// Each real product is its own multiply-add into the running sum (one
// fused instruction each; a - b*c contracts with the sign folded in).
// PACK (FP32 only): the same products as packed two-lane instructions.
template <bool ADJ, bool PACK = false, class R>
__device__ __forceinline__ void su3_mul_half(const R u[18], const R h[12], R w[12])
{
    if constexpr (PACK && sizeof(R) == 4) {
        // FP32: the two colour vectors share every link entry, so lane s of
        // a packed pair carries colour vector s through the same sequence of
        // products (per lane the same roundings as the scalar form below)
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            float2 re, im;
#pragma unroll
            for (int b = 0; b < 3; ++b) {
                const int k = ADJ ? 2 * (3 * b + a) : 2 * (3 * a + b);
                const float2 ur = make_float2(u[k], u[k]);
                const float2 ui = make_float2(u[k + 1], u[k + 1]);
                const float2 nui = make_float2(-u[k + 1], -u[k + 1]);
                const float2 hr = make_float2(h[2 * b], h[2 * (3 + b)]);
                const float2 hi = make_float2(h[2 * b + 1], h[2 * (3 + b) + 1]);
                if (b == 0) {
                    re = __fmul2_rn(ur, hr);
                    im = __fmul2_rn(ur, hi);
                } else {
                    re = __ffma2_rn(ur, hr, re);
                    im = __ffma2_rn(ur, hi, im);
                }
                if (ADJ) {
                    re = __ffma2_rn(ui, hi, re);
                    im = __ffma2_rn(nui, hr, im);
                } else {
                    re = __ffma2_rn(nui, hi, re);
                    im = __ffma2_rn(ui, hr, im);
                }
            }
            w[2 * a] = re.x;
            w[2 * a + 1] = im.x;
            w[2 * (3 + a)] = re.y;
            w[2 * (3 + a) + 1] = im.y;
        }
        return;
    }
#pragma unroll
    for (int s = 0; s < 2; ++s) {
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            R re, im;
#pragma unroll
            for (int b = 0; b < 3; ++b) {
                const int k = ADJ ? 2 * (3 * b + a) : 2 * (3 * a + b);
                const R ur = u[k], ui = u[k + 1];
                const R hr = h[2 * (3 * s + b)], hi = h[2 * (3 * s + b) + 1];
                if (b == 0) {
                    re = ur * hr;
                    im = ur * hi;
                } else {
                    re += ur * hr;
                    im += ur * hi;
                }
                if (ADJ) {  // conj(u): (ur - i ui)(hr + i hi)
                    re += ui * hi;
                    im -= ui * hr;
                } else {
                    re -= ui * hi;
                    im += ui * hr;
                }
            }
            w[2 * (3 * s + a)] = re;
            w[2 * (3 * s + a) + 1] = im;
        }
    }
}

// w += U^dag h for both colour vectors, the products chained onto w.
// (Apart from su3_mul_half: a shared body moved the FP32 kernels' schedules,
// 5 % of a 16^4 CG iteration with FP16 spinors.)
__device__ __forceinline__ void su3_adjoint_add(const double u[18], const double h[12], double w[12])
{
#pragma unroll
    for (int s = 0; s < 2; ++s) {
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            double re = w[2 * (3 * s + a)], im = w[2 * (3 * s + a) + 1];
#pragma unroll
            for (int b = 0; b < 3; ++b) {
                const double ur = u[2 * (3 * b + a)], ui = u[2 * (3 * b + a) + 1];
                const double hr = h[2 * (3 * s + b)], hi = h[2 * (3 * s + b) + 1];
                re += ur * hr;
                im += ur * hi;
                re += ui * hi;
                im -= ui * hr;
            }
            w[2 * (3 * s + a)] = re;
            w[2 * (3 * s + a) + 1] = im;
        }
    }
}

// ---- the neighbour's spinor of a hop, as it is stored
// load(), then project<MU, S>() onto the two colour vectors, and, after the
// link product, add<MU, S>() into the sum.  flip: the hop crosses the
// antiperiodic t boundary.
template <int PS>
struct HopSpinor {
    typedef typename RealT<PS>::type R;
    R v[24];
    bool flip;
    __device__ __forceinline__ void load(const void* base, int stride, int j) { SpinorIO<PS>::load(base, stride, j, v); }
    template <int MU, int S>
    __device__ __forceinline__ void project_to(R h[12]) const
    {
        project<MU, S>(v, h);
        if (flip) {
#pragma unroll
            for (int k = 0; k < 12; ++k) h[k] = -h[k];
        }
    }
    template <int MU, int S>
    __device__ __forceinline__ void add(R acc[24], const R w[12]) const
    {
        accumulate<MU, S>(acc, w);
    }
};

// Half precision: 12 packed complex values q and the site's norm n.  The
// projection is formed from the packed halves (two mixed-precision adds a
// value), and the norm, with the boundary sign, multiplies the products where
// they are added to the sum (a multiply-add instead of an add): 48 instructions
// of the FMA pipe a hop where decoding, scaling and projecting took 84.
template <int MU, int S>
__device__ __forceinline__ void accumulate_scaled(float acc[24], const float w[12], float n)
{
    const float f = S * n;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const float w0r = w[2 * c], w0i = w[2 * c + 1], w1r = w[2 * (3 + c)], w1i = w[2 * (3 + c) + 1];
        float* const a0 = acc + 2 * c;
        float* const a1 = acc + 2 * (3 + c);
        float* const a2 = acc + 2 * (6 + c);
        float* const a3 = acc + 2 * (9 + c);
        a0[0] += n * w0r;
        a0[1] += n * w0i;
        a1[0] += n * w1r;
        a1[1] += n * w1i;
        if (MU == 0) {
            a2[0] += f * w1i;
            a2[1] -= f * w1r;
            a3[0] += f * w0i;
            a3[1] -= f * w0r;
        } else if (MU == 1) {
            a2[0] += f * w1r;
            a2[1] += f * w1i;
            a3[0] -= f * w0r;
            a3[1] -= f * w0i;
        } else if (MU == 2) {
            a2[0] += f * w0i;
            a2[1] -= f * w0r;
            a3[0] -= f * w1i;
            a3[1] += f * w1r;
        } else {
            a2[0] += f * w0r;
            a2[1] += f * w0i;
            a3[0] += f * w1r;
            a3[1] += f * w1i;
        }
    }
}

template <int ISBF>
struct HopSpinorHalf {
    uint32_t q[12];
    float n;
    bool flip;
    __device__ __forceinline__ void set(const uint4 s[3])
    {
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            q[4 * k] = s[k].x; q[4 * k + 1] = s[k].y; q[4 * k + 2] = s[k].z; q[4 * k + 3] = s[k].w;
        }
    }
    __device__ __forceinline__ void load(const void* base, int stride, int j)
    {
        const uint4* p = static_cast<const uint4*>(base);
        n = ld_plain(reinterpret_cast<const float*>(p + (size_t)3 * stride) + j);
        uint4 s[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) s[k] = ld_plain(p + (size_t)k * stride + j);
        set(s);
    }
    // h0 = q0 + e0 q_a, h1 = q1 + e1 q_b with e = +-1 (REAL) or +-i
    template <bool PLUS>
    __device__ __forceinline__ static void real_pair(uint32_t x, uint32_t y, float& re, float& im)
    {
        const float yr = half_value<ISBF, 0>(y), yi = half_value<ISBF, 1>(y);
        re = PLUS ? add_half<ISBF, 0>(x, yr) : half_minus<ISBF, 0>(x, yr);
        im = PLUS ? add_half<ISBF, 1>(x, yi) : half_minus<ISBF, 1>(x, yi);
    }
    template <bool PLUS>
    __device__ __forceinline__ static void imag_pair(uint32_t x, uint32_t y, float& re, float& im)
    {
        const float yr = half_value<ISBF, 0>(y), yi = half_value<ISBF, 1>(y);
        re = PLUS ? half_minus<ISBF, 0>(x, yi) : add_half<ISBF, 0>(x, yi);
        im = PLUS ? add_half<ISBF, 1>(x, yr) : half_minus<ISBF, 1>(x, yr);
    }
    template <int MU, int S>
    __device__ __forceinline__ void project_to(float h[12]) const
    {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const uint32_t p0 = q[c], p1 = q[3 + c], p2 = q[6 + c], p3 = q[9 + c];
            float* const h0 = h + 2 * c;
            float* const h1 = h + 2 * (3 + c);
            if (MU == 0) {  // p0 + S i p3, p1 + S i p2
                imag_pair<(S > 0)>(p0, p3, h0[0], h0[1]);
                imag_pair<(S > 0)>(p1, p2, h1[0], h1[1]);
            } else if (MU == 1) {  // p0 - S p3, p1 + S p2
                real_pair<(S < 0)>(p0, p3, h0[0], h0[1]);
                real_pair<(S > 0)>(p1, p2, h1[0], h1[1]);
            } else if (MU == 2) {  // p0 + S i p2, p1 - S i p3
                imag_pair<(S > 0)>(p0, p2, h0[0], h0[1]);
                imag_pair<(S < 0)>(p1, p3, h1[0], h1[1]);
            } else {  // p0 + S p2, p1 + S p3
                real_pair<(S > 0)>(p0, p2, h0[0], h0[1]);
                real_pair<(S > 0)>(p1, p3, h1[0], h1[1]);
            }
        }
    }
    template <int MU, int S>
    __device__ __forceinline__ void add(float acc[24], const float w[12]) const
    {
        accumulate_scaled<MU, S>(acc, w, scale());
    }
    __device__ __forceinline__ float scale() const { return flip ? -n : n; }
};
template <> struct HopSpinor<P16> : HopSpinorHalf<0> {};
template <> struct HopSpinor<PB16> : HopSpinorHalf<1> {};

// Are links read through the read-only path?  The two kinds of load give the
// compiler different schedules: read-only ones are faster with links and
// spinors in the same storage (CG iteration at 24^3 x 48, FP32, us, plain /
// read-only: recon-12 292 / 285; FP16 hop 23.1 / 22.7) and with 16-bit spinors
// and recon-18 (a CG solve by 1 to 2 %); with 16-bit spinors and recon-12 plain
// ones are, where the others spill (241 / 244; 16^4 by 3 %), and with 16-bit
// links and FP32 spinors (FP16 recon-12 hop by 3 %).
template <int PG, int PS, int RECON>
__host__ __device__ constexpr bool fixed_links()
{
    return (PG == PS && PG != P64) || (PG == P32 && RECON == 18);
}

// w = U P q (backward: U^dag P q) for the neighbour's spinor q: forward hops
// (BWD false) use (1 - g_mu), backward ones (1 + g_mu), swapped by DAG; the
// link is U_mu at checkerboard index lidx of parity lpar.  hop_term adds it.
// 16-bit links with FP32 spinors are decoded by conversions in the forward
// operator and by adds in its adjoint (and with BF16 recon-18): the values are
// the same and neither pipe is full, but the compiler's schedules differ by
// several per cent.  42 x 32^2 x 48, 4 rhs, us, by adds / by conversions: BF16
// recon-12 hop 265 / 250, Schur operator 658 / 642, adjoint full operator 555 /
// 576; BF16 recon-18 hop 281 / 284; FP16 recon-18 full operator 646 / 604,
// adjoint 600 / 605; FP16 recon-12 Schur operator 658 / 622, adjoint 641 / 648.
template <int PG, int PS, int RECON, int MU, bool DAG, bool BWD, bool PACK>
__device__ __forceinline__ void hop_product(const DslashArgs& A, const HopSpinor<PS>& q, int lpar, int lidx,
                                            typename RealT<PS>::type w[12])
{
    typename RealT<PS>::type h[12], u[18];
    q.template project_to<MU, (BWD != DAG) ? +1 : -1>(h);
    constexpr bool FIXED = fixed_links<PG, PS, RECON>();
    if constexpr (PG == P16 || PG == PB16)
        GaugeIO<PG, RECON>::template load<FIXED, !DAG && (PG == P16 || RECON == 12)>(A.gauge, A.g.stride, lpar, MU, lidx, u);
    else GaugeIO<PG, RECON>::template load<FIXED>(A.gauge, A.g.stride, lpar, MU, lidx, u);
    su3_mul_half<BWD, PACK>(u, h, w);
}
template <int PG, int PS, int RECON, int MU, bool DAG, bool BWD, bool PACK>
__device__ __forceinline__ void hop_term(const DslashArgs& A, const HopSpinor<PS>& q, int lpar, int lidx,
                                         typename RealT<PS>::type acc[24])
{
    typename RealT<PS>::type w[12];
    hop_product<PG, PS, RECON, MU, DAG, BWD, PACK>(A, q, lpar, lidx, w);
    q.template add<MU, (BWD != DAG) ? +1 : -1>(acc, w);
}

// FP64: sum and difference of the products of both hops of direction MU at
// site i, from the neighbours jf and jb (flips: across the antiperiodic boundary).
template <int RECON, int MU, bool DAG>
__device__ __forceinline__ void hop_pair(const DslashArgs& A, const char* in, int i, int jf, int jb, bool flip_f, bool flip_b,
                                         double sum[12], double d[12])
{
    HopSpinor<P64> q;
    double wf[12], h[12], u[18];
    q.load(in, A.g.stride, jf);
    q.flip = flip_f;
    hop_product<P64, P64, RECON, MU, DAG, false, false>(A, q, A.par, i, wf);
    q.load(in, A.g.stride, jb);
    q.flip = flip_b;
    q.project_to<MU, DAG ? -1 : +1>(h);
    GaugeIO<P64, RECON>::load(A.gauge, A.g.stride, 1 - A.par, MU, jb, u);
#pragma unroll
    for (int k = 0; k < 12; ++k) sum[k] = wf[k];
    su3_adjoint_add(u, h, sum);
#pragma unroll
    for (int k = 0; k < 12; ++k) d[k] = 2.0 * wf[k] - sum[k];
}

// PG: storage of links and clover; PS: storage of spinor fields; the
// arithmetic is in RealT<PS> (FP64 only when everything is FP64).
// HALO (sub-domain interior pass): a hop across the local boundary of a
// cut direction is left out; it arrives later as a face.
template <int PG, int PS, int RECON, int MU, bool DAG, bool HALO = false, bool PACK = false>
__device__ __forceinline__ void hop_dir(const DslashArgs& A, const char* in, int i, int full, const int c[4],
                                        int stepmu, typename RealT<PS>::type acc[24])
{
    const int L = A.g.L[MU];
    const int fwd = (c[MU] == L - 1) ? full - (L - 1) * stepmu : full + stepmu;
    const int bwd = (c[MU] == 0) ? full + (L - 1) * stepmu : full - stepmu;
    const bool tb = (MU == 3) && A.g.tanti;
    const bool cut = HALO && ((A.g.part >> MU) & 1);
    HopSpinor<PS> q;
    if constexpr (PS == P64 && !HALO) {
        double sum[12], d[12];
        hop_pair<RECON, MU, DAG>(A, in, i, fwd >> 1, bwd >> 1, tb && c[3] == L - 1, tb && c[3] == 0, sum, d);
        accumulate_pair<MU, DAG ? +1 : -1>(acc, sum, d);
        return;
    }
    if (!(cut && c[MU] == L - 1)) {
        q.load(in, A.g.stride, fwd >> 1);
        q.flip = tb && c[3] == L - 1;
        hop_term<PG, PS, RECON, MU, DAG, false, PACK>(A, q, A.par, i, acc);
    }
    if (!(cut && c[MU] == 0)) {
        q.load(in, A.g.stride, bwd >> 1);
        q.flip = tb && c[3] == 0;
        hop_term<PG, PS, RECON, MU, DAG, true, PACK>(A, q, 1 - A.par, bwd >> 1, acc);
    }
}

// ---- software-pipelined gather for half-precision spinors + recon-12 links
// The packed 16-bit data of hop d+1 (3 x uint4 + norm, 3 x uint2) is loaded
// before hop d is decoded and computed, so that two hops' loads are in
// flight per thread: half-precision loads move few bytes each, and one hop
// at a time does not cover DRAM latency.
template <int RECON>
struct HalfHopRaw {
    uint4 s[3];
    float n;
    uint32_t u[RECON == 12 ? 6 : 9];  // packed half2: two (recon-12) or three rows
};

struct HopPlan {
    int nb[8];      // neighbour checkerboard index per hop (2 mu: forward, 2 mu + 1: backward)
    int lidx[8];    // link index (the site itself forward, the neighbour backward)
    unsigned flip;  // bit h: the hop crosses the antiperiodic t boundary
};

template <int RECON>
__device__ __forceinline__ void load_half_hop(const char* in, const void* gauge, int stride, int par,
                                              const HopPlan& hp, int h, HalfHopRaw<RECON>& r)
{
    const uint4* sp = reinterpret_cast<const uint4*>(in);
    const int j = hp.nb[h];
    r.n = ld_plain(reinterpret_cast<const float*>(sp + (size_t)3 * stride) + j);
#pragma unroll
    for (int k = 0; k < 3; ++k) r.s[k] = ld_plain(sp + (size_t)k * stride + j);
    const int mu = h >> 1, lpar = (h & 1) ? 1 - par : par;
    if constexpr (RECON == 12) {
        const uint2* lp = static_cast<const uint2*>(gauge) + (size_t)((lpar * 4 + mu) * 3) * stride + hp.lidx[h];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const uint2 q = ld_fixed(lp + (size_t)k * stride);
            r.u[2 * k] = q.x;
            r.u[2 * k + 1] = q.y;
        }
    } else {
        const uint32_t* lp = static_cast<const uint32_t*>(gauge) + (size_t)((lpar * 4 + mu) * 9) * stride + hp.lidx[h];
#pragma unroll
        for (int k = 0; k < 9; ++k) r.u[k] = ld_fixed(lp + (size_t)k * stride);
    }
}

template <int ISBF, int RECON, int MU, bool BWD, bool DAG, bool PACK>
__device__ __forceinline__ void half_hop_product(const HalfHopRaw<RECON>& r, HopSpinorHalf<ISBF>& q, bool flip, float w[12])
{
    float h[12], u[18];
    q.set(r.s);
    q.n = r.n;
    q.flip = flip;
#pragma unroll
    for (int k = 0; k < (RECON == 12 ? 6 : 9); ++k) {
        const float2 a = halves<ISBF>(r.u[k]);
        u[2 * k] = a.x;
        u[2 * k + 1] = a.y;
    }
    if constexpr (RECON == 12) reconstruct_row2(u);
    q.template project_to<MU, (BWD != DAG) ? +1 : -1>(h);
    su3_mul_half<BWD, PACK>(u, h, w);
}
template <int ISBF, int RECON, int MU, bool BWD, bool DAG, bool PACK>
__device__ __forceinline__ void compute_half_hop(const HalfHopRaw<RECON>& r, bool flip, float acc[24])
{
    HopSpinorHalf<ISBF> q;
    float w[12];
    half_hop_product<ISBF, RECON, MU, BWD, DAG, PACK>(r, q, flip, w);
    q.template add<MU, (BWD != DAG) ? +1 : -1>(acc, w);
}

template <int ISBF, int RECON, bool DAG, bool PACK, int H>
__device__ __forceinline__ void half_pipeline_step(const char* in, const void* gauge, int stride, int par,
                                                   const HopPlan& hp, HalfHopRaw<RECON> (&buf)[2], float acc[24])
{
    if constexpr (H < 7) load_half_hop<RECON>(in, gauge, stride, par, hp, H + 1, buf[(H + 1) & 1]);
    compute_half_hop<ISBF, RECON, H / 2, (H & 1) != 0, DAG, PACK>(buf[H & 1], (hp.flip >> H) & 1u, acc);
    if constexpr (H < 7) half_pipeline_step<ISBF, RECON, DAG, PACK, H + 1>(in, gauge, stride, par, hp, buf, acc);
}

template <int ISBF, int RECON, bool DAG, bool PACK>
__device__ __forceinline__ void hop_all_half(const DslashArgs& A, const char* in, int i, int full, const int c[4],
                                             float acc[24])
{
    HopPlan hp;
    hp.flip = 0u;
    int step = 1;
#pragma unroll
    for (int mu = 0; mu < 4; ++mu) {
        const int L = A.g.L[mu];
        const int fwd = (c[mu] == L - 1) ? full - (L - 1) * step : full + step;
        const int bwd = (c[mu] == 0) ? full + (L - 1) * step : full - step;
        hp.nb[2 * mu] = fwd >> 1;
        hp.nb[2 * mu + 1] = bwd >> 1;
        hp.lidx[2 * mu] = i;
        hp.lidx[2 * mu + 1] = bwd >> 1;
        step *= L;
    }
    if (A.g.tanti) {
        if (c[3] == A.g.L[3] - 1) hp.flip |= 1u << 6;
        if (c[3] == 0) hp.flip |= 1u << 7;
    }
    HalfHopRaw<RECON> buf[2];
    load_half_hop<RECON>(in, A.gauge, A.g.stride, A.par, hp, 0, buf[0]);
    half_pipeline_step<ISBF, RECON, DAG, PACK, 0>(in, A.gauge, A.g.stride, A.par, hp, buf, acc);
}

// Threads per block are at most DSLASH_MAX_BLOCK; DSLASH_MIN_BLOCKS resident
// blocks per SM caps the registers so that enough warps are in flight to
// cover the latency of the neighbour gathers.
#ifndef LQCD_DSLASH_MINB
#define LQCD_DSLASH_MINB 4  // <= 128 registers; 4, 5, 6 measured within 5% on 32^3x64
#endif
#define DSLASH_MAX_BLOCK 128
#define DSLASH_WIDE 2    // internal: the warp-per-direction kernel
#define DSLASH_STAGED 1  // a "block size" that selects the shared-memory staged kernel (LQCD_BLOCK_STAGED)
// The CG step alpha = |r|^2 / |Mp|^2; once r is exactly zero (an exact
// solution inside a check interval) both vanish: no step instead of 0/0.  An
// FP64 division is some fifteen instructions of a pipe with 1/63 of FP32's
// rate, so the gathering kernel does it once a block, not once a site (CG
// iteration at 16^4, 12 FP16-spinor rhs: 206 -> 202 us; 32^3 x 64 FP32 746 ->
// 740).  The warp-per-direction kernel does it in its epilogue threads, beside
// the hops and before the barrier, the persistent kernel once a tile and thread.
template <int PS>
__device__ __forceinline__ typename RealT<AccumP<PS>::value>::type cg_alpha(const DslashArgs& A, int rhs)
{
    typedef typename RealT<AccumP<PS>::value>::type RA;
    const double* sc = A.scal + rhs * A.scal_rs;
    const double den = sc[A.s_den] + sc[A.s_den2];
    return den > 0.0 ? (RA)((sc[A.s_num] + sc[A.s_num2]) / den) : (RA)0;
}

// Epilogue at output site i of right-hand side rhs for the hopping term
// acc; nrm accumulates |out|^2 (|r|^2 for EPI_CG, whose step is alpha).
template <int PG, int PS, bool DAG, int EPI, bool RED>
__device__ __forceinline__ void dslash_epilogue(const DslashArgs& A, int rhs, int i, typename RealT<PS>::type acc[24],
                                                double& nrm, typename RealT<AccumP<PS>::value>::type alpha)
{
    typedef typename RealT<PS>::type R;
    const R a = (R)A.a;
    if (EPI == EPI_NONE) {
#pragma unroll
        for (int k = 0; k < 24; ++k) acc[k] *= a;
    } else if (EPI == EPI_CLOVINV) {
        if (A.clov) {
            R t[24];
            clover_apply_site<PG, PG == PS>(A.clov, A.g.stride, i, acc, t);
#pragma unroll
            for (int k = 0; k < 24; ++k) acc[k] = a * t[k];
        } else {
#pragma unroll
            for (int k = 0; k < 24; ++k) acc[k] *= a;
        }
    } else {  // EPI_XPAY, EPI_CG
        R yv[24], t[24];
        SpinorIO<PS>::load(static_cast<const char*>(A.y) + rhs * A.y_rb, A.g.stride, i, yv);
        if (A.clov) {
            clover_apply_site<PG, PG == PS>(A.clov, A.g.stride, i, yv, t);
        } else {
#pragma unroll
            for (int k = 0; k < 24; ++k) t[k] = yv[k];
        }
#pragma unroll
        for (int k = 0; k < 24; ++k) acc[k] = t[k] + a * acc[k];
    }
    if constexpr (EPI == EPI_CG) {
        typedef typename RealT<AccumP<PS>::value>::type RA;
        RA rv[24];
        char* rb = static_cast<char*>(A.r) + rhs * A.acc_rb;
        SpinorIO<AccumP<PS>::value>::load(rb, A.g.stride, i, rv);
        RA n = 0;
#pragma unroll
        for (int k = 0; k < 24; ++k) {
            rv[k] -= alpha * (RA)acc[k];
            n += rv[k] * rv[k];
        }
        nrm += (double)n;
        SpinorIO<AccumP<PS>::value>::store(rb, A.g.stride, i, rv);
        if (A.x) {  // (uniform; a deferred x is added by cg_x_kernel)
            R pv[24];
            RA xv[24];
            SpinorIO<PS>::load(static_cast<const char*>(A.p) + rhs * A.p_rb, A.g.stride, i, pv);
            char* xb = static_cast<char*>(A.x) + rhs * A.acc_rb;
            SpinorIO<AccumP<PS>::value>::load(xb, A.g.stride, i, xv);
#pragma unroll
            for (int k = 0; k < 24; ++k) xv[k] += alpha * (RA)pv[k];
            SpinorIO<AccumP<PS>::value>::store(xb, A.g.stride, i, xv);
        }
    } else {
        SpinorIO<PS>::store(static_cast<char*>(A.out) + rhs * A.out_rb, A.g.stride, i, acc);
        if (RED) {
            R n = 0;
#pragma unroll
            for (int k = 0; k < 24; ++k) n += acc[k] * acc[k];
            nrm += (double)n;
        }
    }
}

// Packed link products: in the launches that neither reduce nor update, and
// with all operands in 16 bits in every launch.  In the reducing launches the
// packed form is slower with FP32 links (CG iteration 24^3 x 48, us: FP32 263
// scalar, 271 packed; FP16 spinors 232 / 253) and faster with 16-bit ones
// (FP16 217 / 198, 12 rhs 2079 / 2041).  The results are the same.
template <int PG, int PS, int EPI, bool RED>
__host__ __device__ constexpr bool packed_products()
{
    return !(RED || EPI == EPI_CG) || ((PG == P16 || PG == PB16) && PS == PG);
}

// True if site c of a sub-domain has a neighbour across a cut boundary.
__device__ __forceinline__ bool on_cut_face(const Geom& g, const int c[4])
{
    bool f = false;
#pragma unroll
    for (int mu = 0; mu < 4; ++mu)
        if (((g.part >> mu) & 1) && (c[mu] == 0 || c[mu] == g.L[mu] - 1)) f = true;
    return f;
}

// The hopping term and epilogue at output site i of right-hand side rhs;
// nrm accumulates |out|^2 (|r|^2 for EPI_CG).  HALO: the interior pass of a
// sub-domain; a site with a neighbour across a cut boundary stores its
// partial sum unfinished (no epilogue) for the face pass to complete.
template <int PG, int PS, int RECON, bool DAG, int EPI, bool RED, bool HALO = false>
__device__ __forceinline__ void dslash_site(const DslashArgs& A, int rhs, int i, double& nrm,
                                            typename RealT<AccumP<PS>::value>::type alpha)
{
    typedef typename RealT<PS>::type R;
    int c[4];
    cb_coords(A.g, i, A.par, c);
    const int full = full_index(A.g, c);
    const char* in = static_cast<const char*>(A.in) + rhs * A.in_rb;
    R acc[24];
#pragma unroll
    for (int k = 0; k < 24; ++k) acc[k] = 0;
    constexpr bool PACK = packed_products<PG, PS, EPI, RED>();
    if constexpr ((PS == P16 || PS == PB16) && PG == PS) {
        static_assert(!HALO, "sub-domain hops use the generic gather");
        hop_all_half<PS == PB16 ? 1 : 0, RECON, DAG, PACK>(A, in, i, full, c, acc);
    } else {
        hop_dir<PG, PS, RECON, 0, DAG, HALO, PACK>(A, in, i, full, c, 1, acc);
        hop_dir<PG, PS, RECON, 1, DAG, HALO, PACK>(A, in, i, full, c, A.g.L[0], acc);
        hop_dir<PG, PS, RECON, 2, DAG, HALO, PACK>(A, in, i, full, c, A.g.L[0] * A.g.L[1], acc);
        hop_dir<PG, PS, RECON, 3, DAG, HALO, PACK>(A, in, i, full, c, A.g.L[0] * A.g.L[1] * A.g.L[2], acc);
    }
    if (HALO && on_cut_face(A.g, c)) {
        SpinorIO<PS>::store(static_cast<char*>(A.out) + rhs * A.out_rb, A.g.stride, i, acc);
        return;
    }
    dslash_epilogue<PG, PS, DAG, EPI, RED>(A, rhs, i, acc, nrm, alpha);
}

// One-dimensional grid: block b serves right-hand side b % nrhs and site
// block b / nrhs, so that the blocks of all right-hand sides for the same
// sites run together and share each link (and clover) read through L2.
// (Applying each loaded link to several right-hand sides in one thread was
// measured slower: the extra accumulators cost occupancy in a kernel whose
// neighbour gathers are latency-bound.)
template <int PG, int PS, int RECON, bool DAG, int EPI, bool RED>
__global__ void __launch_bounds__(DSLASH_MAX_BLOCK, (PG == P64 ? 1 : LQCD_DSLASH_MINB))
    dslash_kernel(const DslashArgs A)
{
    const int rhs = (int)(blockIdx.x % (unsigned)A.nrhs);
    const int sb = (int)(blockIdx.x / (unsigned)A.nrhs), nsb = (int)(gridDim.x / (unsigned)A.nrhs);
    pdl_wait();
    if (A.skip && A.skip[rhs]) return;  // uniform over the rhs: no block of it reduces
    double nrm = 0.0;
    typename RealT<AccumP<PS>::value>::type alpha = 0;
    if constexpr (EPI == EPI_CG) {
        __shared__ typename RealT<AccumP<PS>::value>::type alpha_s;
        if (threadIdx.x == 0) alpha_s = cg_alpha<PS>(A, rhs);
        __syncthreads();
        alpha = alpha_s;
    }
    if constexpr (RED || EPI == EPI_CG) {
        // grid-stride: the launcher runs one wave of blocks, so that each
        // block's partial sum covers many sites
        for (int i = sb * blockDim.x + threadIdx.x; i < A.g.Vh; i += nsb * blockDim.x)
            dslash_site<PG, PS, RECON, DAG, EPI, RED>(A, rhs, i, nrm, alpha);
        pdl_start_next();
        double v[1] = {nrm};
        block_reduce_finalize<1>(v, A.partials + rhs * A.part_rs, A.tickets + rhs, A.red + rhs * A.red_rs, sb, nsb);
    } else {
        const int i = sb * blockDim.x + threadIdx.x;
        if (i < A.g.Vh) dslash_site<PG, PS, RECON, DAG, EPI, RED>(A, rhs, i, nrm, alpha);
        pdl_start_next();
    }
}

// Launch helper: ceil(Vh / block) x nrhs blocks, one site per thread; for
// launches that reduce (fused norms, fused CG update) at most one wave of
// resident blocks, so that each block's partial sum covers more sites and the
// deterministic two-stage reduction handles 608 instead of 8192 partials at
// 32^3x64 (measured: solve 4 % faster; plain launches are faster with the
// full grid).
template <int PG, int PS, int RECON, bool DAG, int EPI, bool RED>
cudaError_t launch_dslash_t(const DslashArgs& A, int nrhs, int block, cudaStream_t s)
{
    static int wave[DSLASH_MAX_BLOCK / 32 + 1];  // per block size, 0 = not yet queried
    const int bi = block / 32;
    if ((RED || EPI == EPI_CG) && wave[bi] == 0) {
        int dev = 0, sms = 0, per_sm = 0;
        cudaError_t e = cudaGetDevice(&dev);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (e == cudaSuccess)
            e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, dslash_kernel<PG, PS, RECON, DAG, EPI, RED>,
                                                              block, 0);
        if (e != cudaSuccess) return e;
        wave[bi] = per_sm > 0 && sms > 0 ? per_sm * sms : 1 << 30;
    }
    int gx = (A.g.Vh + block - 1) / block;
    if (RED || EPI == EPI_CG) {
        if (A.sites_per_thread > 0) {
            const long per_block = (long)block * A.sites_per_thread;
            gx = (int)((A.g.Vh + per_block - 1) / per_block);
        } else if (gx > wave[bi]) {
            gx = wave[bi];
        }
    }
    if ((long)gx * nrhs > 0x7fffffffL) return cudaErrorInvalidConfiguration;
    DslashArgs Ar = A;
    Ar.nrhs = nrhs;
    if (A.plain) {
        dslash_kernel<PG, PS, RECON, DAG, EPI, RED><<<gx * nrhs, block, 0, s>>>(Ar);
        return cudaGetLastError();
    }
    return launch_dependent(dslash_kernel<PG, PS, RECON, DAG, EPI, RED>, false, gx * nrhs, block, s, 0, Ar);
}

// ---------------------------------------------------------------------------
// The hopping term with a warp per direction (launches of few sites, see
// wide_default).  A block takes 32 sites of one right-hand side: warps 0 to 3
// each form the products U P v of both hops of one direction and put their
// two colour vectors into shared memory; warp 4 (spins 0, 1) and warp 5
// (spins 2, 3) meanwhile load the epilogue's operands (and form Cl y), then
// add the eight products in the gathering kernel's order and run the epilogue
// on their chiral half.
//
// Why: with few sites nothing is bound by bandwidth.  A thread per site runs
// the loads and products of its eight hops one after another (registers keep
// it from having all loads in flight), a chain that is mostly L2 latency, on
// a GPU that is nearly empty; in FP64 the chain is 1100 instructions at one
// per 64 cycles and scheduler.  Here the chain is two hops, one barrier and
// the epilogue, over six times the warps.  Every sum runs over the same terms
// in the same order, so that the fields are those of the gathering kernel bit
// for bit (the norms' grid sums are grouped per 32 sites).  A warp per hop
// (320 threads) was as fast below 2048 sites and 20 to 30 % slower at 10368;
// four hops a warp slower below 4096.
enum { WIDE_SITES = 32, WIDE_THREADS = 192 };

template <class R> struct Pair;
template <> struct Pair<float> { typedef float2 type; };
template <> struct Pair<double> { typedef double2 type; };

// The products of the eight hops (two colour vectors each) of the block's 32
// sites, the neighbours' norms (half precision) and what the epilogue warps exchange.
template <int PS>
struct WideShared {
    typedef typename RealT<PS>::type R;
    typename Pair<R>::type w[8 * 6][32];
    float n[PS == P16 || PS == PB16 ? 8 : 1][32];
    R ex[3][32];
};

// The product of hop H (2 mu + backward) at site i.
template <int PG, int PS, int RECON, bool DAG, bool PACK, int H>
__device__ __forceinline__ void wide_hop(const DslashArgs& A, const char* in, int i, int full, const int c[4],
                                         WideShared<PS>& sh)
{
    typedef typename RealT<PS>::type R;
    constexpr int MU = H / 2;
    constexpr bool BWD = (H & 1) != 0;
    const int L = A.g.L[MU];
    const int step = (MU > 0 ? A.g.L[0] : 1) * (MU > 1 ? A.g.L[1] : 1) * (MU > 2 ? A.g.L[2] : 1);
    const bool edge = BWD ? c[MU] == 0 : c[MU] == L - 1;
    const int nb = BWD ? (edge ? full + (L - 1) * step : full - step) : (edge ? full - (L - 1) * step : full + step);
    const int j = nb >> 1;
    const bool flip = MU == 3 && A.g.tanti && edge;
    HopSpinor<PS> q;
    R w[12];
    if constexpr ((PS == P16 || PS == PB16) && PG == PS) {
        HopPlan hp;
        hp.nb[H] = j;
        hp.lidx[H] = BWD ? j : i;
        HalfHopRaw<RECON> raw;
        load_half_hop<RECON>(in, A.gauge, A.g.stride, A.par, hp, H, raw);
        half_hop_product<PS == PB16 ? 1 : 0, RECON, MU, BWD, DAG, PACK>(raw, q, flip, w);
    } else {
        q.load(in, A.g.stride, j);
        q.flip = flip;
        hop_product<PG, PS, RECON, MU, DAG, BWD, PACK>(A, q, BWD ? 1 - A.par : A.par, BWD ? j : i, w);
    }
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int k = 0; k < 6; ++k) {
        sh.w[6 * H + k][lane].x = w[2 * k];
        sh.w[6 * H + k][lane].y = w[2 * k + 1];
    }
    if constexpr (PS == P16 || PS == PB16) sh.n[H][lane] = q.scale();
}

// both hops of direction MU
template <int PG, int PS, int RECON, bool DAG, bool PACK, int MU>
__device__ __forceinline__ void wide_hops(const DslashArgs& A, const char* in, int i, int full, const int c[4],
                                          WideShared<PS>& sh)
{
    if constexpr (PS == P64) {  // their sum and difference in place of the two products
        const int L = A.g.L[MU];
        const int step = (MU > 0 ? A.g.L[0] : 1) * (MU > 1 ? A.g.L[1] : 1) * (MU > 2 ? A.g.L[2] : 1);
        const bool top = c[MU] == L - 1, bottom = c[MU] == 0, tb = MU == 3 && A.g.tanti;
        const int fwd = top ? full - (L - 1) * step : full + step, bwd = bottom ? full + (L - 1) * step : full - step;
        double w[2][12];
        hop_pair<RECON, MU, DAG>(A, in, i, fwd >> 1, bwd >> 1, tb && top, tb && bottom, w[0], w[1]);
#pragma unroll
        for (int k = 0; k < 12; ++k) sh.w[12 * MU + k][threadIdx.x & 31] = make_double2(w[k / 6][2 * (k % 6)], w[k / 6][2 * (k % 6) + 1]);
    } else {
        wide_hop<PG, PS, RECON, DAG, PACK, 2 * MU>(A, in, i, full, c, sh);
        wide_hop<PG, PS, RECON, DAG, PACK, 2 * MU + 1>(A, in, i, full, c, sh);
    }
}

template <bool DAG, int MU>
__device__ __forceinline__ void wide_sum_pairs(const WideShared<P64>& sh, double acc[24])
{
    const int lane = threadIdx.x & 31;
    double w[2][12];
#pragma unroll
    for (int k = 0; k < 12; ++k) {
        const double2 t = sh.w[12 * MU + k][lane];
        w[k / 6][2 * (k % 6)] = t.x;
        w[k / 6][2 * (k % 6) + 1] = t.y;
    }
    accumulate_pair<MU, DAG ? +1 : -1>(acc, w[0], w[1]);  // (as below, one half is used)
    if constexpr (MU < 3) wide_sum_pairs<DAG, MU + 1>(sh, acc);
}

template <int PS, bool DAG, int H>
__device__ __forceinline__ void wide_sum(const WideShared<PS>& sh, typename RealT<PS>::type acc[24])
{
    typedef typename RealT<PS>::type R;
    constexpr int S = ((H & 1) != 0) != DAG ? +1 : -1;
    const int lane = threadIdx.x & 31;
    R w[12];
#pragma unroll
    for (int q = 0; q < 6; ++q) {
        const typename Pair<R>::type t = sh.w[6 * H + q][lane];
        w[2 * q] = t.x;
        w[2 * q + 1] = t.y;
    }
    // (of acc the caller uses one half; the other is dead code)
    if constexpr (PS == P16 || PS == PB16) accumulate_scaled<H / 2, S>(acc, w, sh.n[H][lane]);
    else accumulate<H / 2, S>(acc, w);
    if constexpr (H < 7) wide_sum<PS, DAG, H + 1>(sh, acc);
}

// What an epilogue warp holds before the barrier, for its half B of the site.
template <int PS, int EPI>
struct WideOperands {
    typedef typename RealT<PS>::type R;
    typedef typename RealT<AccumP<PS>::value>::type RA;
    R t[EPI >= EPI_XPAY ? 12 : 1];            // Cl y
    R cl[EPI == EPI_CLOVINV ? 36 : 1];        // block of Cl
    R p[EPI == EPI_CG ? 12 : 1];
    RA x[EPI == EPI_CG ? 12 : 1], r[EPI == EPI_CG ? 12 : 1], alpha;
};

template <int PG, int PS, int EPI, int B>
__device__ __forceinline__ void wide_operands(const DslashArgs& A, int rhs, int i, WideOperands<PS, EPI>& o)
{
    typedef typename RealT<PS>::type R;
    if constexpr (EPI == EPI_CLOVINV) {
        if (A.clov) CloverIO<PG>::template load_block<PG == PS>(A.clov, A.g.stride, i, B, o.cl);
    }
    if constexpr (EPI >= EPI_XPAY) {
        R yv[12];
        SpinorIO<PS>::template load_half<B>(static_cast<const char*>(A.y) + rhs * A.y_rb, A.g.stride, i, yv);
        if (A.clov) {
            R cl[36];
            CloverIO<PG>::template load_block<PG == PS>(A.clov, A.g.stride, i, B, cl);
            hermitian6_apply<R>(cl, yv, o.t);
        } else {
#pragma unroll
            for (int k = 0; k < 12; ++k) o.t[k] = yv[k];
        }
    }
    if constexpr (EPI == EPI_CG) {
        constexpr int PA = AccumP<PS>::value;
        o.alpha = cg_alpha<PS>(A, rhs);
        if (A.x) {
            SpinorIO<PS>::template load_half<B>(static_cast<const char*>(A.p) + rhs * A.p_rb, A.g.stride, i, o.p);
            SpinorIO<PA>::template load_half<B>(static_cast<const char*>(A.x) + rhs * A.acc_rb, A.g.stride, i, o.x);
        }
        SpinorIO<PA>::template load_half<B>(static_cast<const char*>(A.r) + rhs * A.acc_rb, A.g.stride, i, o.r);
    }
}

// Sum, epilogue and store of half B; both epilogue warps run this together
// (they exchange the half's norm and largest component).
// Returns the site's |out|^2 (|r|^2) in the thread of half 1: its FP32 sum
// runs over the 24 components in order, so half 1 continues from half 0's.
template <int PG, int PS, bool DAG, int EPI, bool RED, int B>
__device__ __forceinline__ double wide_finish(const DslashArgs& A, int rhs, int i, bool live,
                                              WideShared<PS>& sh, WideOperands<PS, EPI>& o)
{
    typedef typename RealT<PS>::type R;
    typedef typename RealT<AccumP<PS>::value>::type RA;
    constexpr bool HALF = PS == P16 || PS == PB16;
    constexpr bool NORM = RED || EPI == EPI_CG;
    const int lane = threadIdx.x & 31;
    R full[24], out[12];
#pragma unroll
    for (int k = 0; k < 24; ++k) full[k] = 0;
    if constexpr (PS == P64) wide_sum_pairs<DAG, 0>(sh, full);
    else wide_sum<PS, DAG, 0>(sh, full);
    const R* acc = full + 12 * B;
    const R a = (R)A.a;
    if constexpr (EPI == EPI_NONE) {
#pragma unroll
        for (int k = 0; k < 12; ++k) out[k] = acc[k] * a;
    } else if constexpr (EPI == EPI_CLOVINV) {
        if (A.clov) {
            R t[12];
            hermitian6_apply<R>(o.cl, acc, t);
#pragma unroll
            for (int k = 0; k < 12; ++k) out[k] = a * t[k];
        } else {
#pragma unroll
            for (int k = 0; k < 12; ++k) out[k] = acc[k] * a;
        }
    } else {
#pragma unroll
        for (int k = 0; k < 12; ++k) out[k] = o.t[k] + a * acc[k];
    }
    if constexpr (EPI == EPI_CG) {
#pragma unroll
        for (int k = 0; k < 12; ++k) o.r[k] -= o.alpha * (RA)out[k];
        if (live) {
            constexpr int PA = AccumP<PS>::value;
            if (A.x) {
#pragma unroll
                for (int k = 0; k < 12; ++k) o.x[k] += o.alpha * (RA)o.p[k];
                SpinorIO<PA>::template store_half<B>(static_cast<char*>(A.x) + rhs * A.acc_rb, A.g.stride, i, o.x);
            }
            SpinorIO<PA>::template store_half<B>(static_cast<char*>(A.r) + rhs * A.acc_rb, A.g.stride, i, o.r);
        }
    } else if constexpr (!HALF) {
        if (live) SpinorIO<PS>::template store_half<B>(static_cast<char*>(A.out) + rhs * A.out_rb, A.g.stride, i, out);
    }
    R big = 0, n = 0;
    if constexpr (HALF && EPI != EPI_CG) {
#pragma unroll
        for (int k = 0; k < 12; ++k) big = fmaxf(big, fabsf(out[k]));
        sh.ex[B][lane] = big;
    }
    if constexpr (NORM) {
        if (B == 0) {
#pragma unroll
            for (int k = 0; k < 12; ++k) n += EPI == EPI_CG ? (R)o.r[k] * (R)o.r[k] : out[k] * out[k];
            sh.ex[2][lane] = n;
        }
    }
    if constexpr ((HALF && EPI != EPI_CG) || NORM) asm volatile("bar.sync 1, 64;" ::: "memory");
    if constexpr (HALF && EPI != EPI_CG) {
        big = fmaxf(big, sh.ex[1 - B][lane]);
        if (live)
            SpinorIO<PS>::template store_half<B>(static_cast<char*>(A.out) + rhs * A.out_rb, A.g.stride, i, out, big);
    }
    if constexpr (NORM) {
        if (B == 1) {
            n = sh.ex[2][lane];
#pragma unroll
            for (int k = 0; k < 12; ++k) n += EPI == EPI_CG ? (R)o.r[k] * (R)o.r[k] : out[k] * out[k];
        }
    }
    return B == 1 && live ? (double)n : 0.0;
}

// One-dimensional grid as in dslash_kernel: block b serves right-hand side
// b % nrhs and site block b / nrhs.
template <int PG, int PS, int RECON, bool DAG, int EPI, bool RED>
__global__ void __launch_bounds__(WIDE_THREADS, (PG == P64 ? 1 : 3)) dslash_wide_kernel(const DslashArgs A)
{
    __shared__ WideShared<PS> sh;
    const int rhs = (int)(blockIdx.x % (unsigned)A.nrhs);
    const int sb = (int)(blockIdx.x / (unsigned)A.nrhs), nsb = (int)(gridDim.x / (unsigned)A.nrhs);
    constexpr bool PACK = packed_products<PG, PS, EPI, RED>();  // the gathering kernel's choice
    const int warp = threadIdx.x >> 5;
    const int i = sb * WIDE_SITES + (threadIdx.x & 31);
    const bool live = i < A.g.Vh;
    int c[4];
    cb_coords(A.g, i, A.par, c);
    const int full = full_index(A.g, c);
    pdl_wait();
    if (A.skip && A.skip[rhs]) return;  // uniform over the rhs: no block of it reduces
    WideOperands<PS, EPI> o;
    if (warp < 4) {
        if (live) {
            const char* in = static_cast<const char*>(A.in) + rhs * A.in_rb;
            switch (warp) {
            case 0: wide_hops<PG, PS, RECON, DAG, PACK, 0>(A, in, i, full, c, sh); break;
            case 1: wide_hops<PG, PS, RECON, DAG, PACK, 1>(A, in, i, full, c, sh); break;
            case 2: wide_hops<PG, PS, RECON, DAG, PACK, 2>(A, in, i, full, c, sh); break;
            default: wide_hops<PG, PS, RECON, DAG, PACK, 3>(A, in, i, full, c, sh); break;
            }
        }
    } else if (live) {
        if (warp == 4) wide_operands<PG, PS, EPI, 0>(A, rhs, i, o);
        else wide_operands<PG, PS, EPI, 1>(A, rhs, i, o);
    }
    __syncthreads();
    double nrm = 0.0;
    if (warp == 4) nrm = wide_finish<PG, PS, DAG, EPI, RED, 0>(A, rhs, i, live, sh, o);
    else if (warp == 5) nrm = wide_finish<PG, PS, DAG, EPI, RED, 1>(A, rhs, i, live, sh, o);
    pdl_start_next();
    if constexpr (RED || EPI == EPI_CG) {
        double v[1] = {nrm};
        block_reduce_finalize<1>(v, A.partials + rhs * A.part_rs, A.tickets + rhs, A.red + rhs * A.red_rs, sb, nsb);
    }
}

template <int PG, int PS, int RECON, bool DAG, int EPI, bool RED>
cudaError_t launch_wide_t(const DslashArgs& A, int nrhs, cudaStream_t s)
{
    const long blocks = (long)((A.g.Vh + WIDE_SITES - 1) / WIDE_SITES) * nrhs;
    if (blocks > 0x7fffffffL) return cudaErrorInvalidConfiguration;
    DslashArgs Ar = A;
    Ar.nrhs = nrhs;
    if (A.plain) {
        dslash_wide_kernel<PG, PS, RECON, DAG, EPI, RED><<<(unsigned)blocks, WIDE_THREADS, 0, s>>>(Ar);
        return cudaGetLastError();
    }
    return launch_dependent(dslash_wide_kernel<PG, PS, RECON, DAG, EPI, RED>, true, (unsigned)blocks, WIDE_THREADS, s, 0, Ar);
}

// ---------------------------------------------------------------------------
// Shared-memory staged hop (plain launches, FP32 links): a block takes a
// tile of STG_TY x STG_TZ x STG_TT rows (y, z, t) of all Lx/2 checkerboard
// sites, one site per thread, and first copies the input spinors of the
// tile and of its six faces (the rows one step outside in y, z and t) into
// shared memory with asynchronous 16-byte copies, which hold no registers
// while in flight; every neighbour is then read from shared memory (x
// neighbours lie in the site's own row).  Faces are copied from the
// periodically wrapped rows.  Rows of the staging buffer: the tile's
// interior r = (tl TZ + zl) TY + yl, then y-, y+ (index tl TZ + zl), z-, z+
// (tl TY + yl), t-, t+ (zl TY + yl).
enum {
    STG_TY = 4, STG_TZ = 2, STG_TT = 2, STG_NIN = STG_TY * STG_TZ * STG_TT,
    STG_FY = STG_TZ * STG_TT, STG_FZ = STG_TY * STG_TT, STG_FT = STG_TY * STG_TZ,
    STG_NROW = STG_NIN + 2 * (STG_FY + STG_FZ + STG_FT), STG_MAXLXH = 16
};

__host__ __device__ inline bool staged_supported(const Geom& g)
{
    return g.part == 0 && g.Lxh <= STG_MAXLXH && g.L[1] % STG_TY == 0 && g.L[2] % STG_TZ == 0 &&
           g.L[3] % STG_TT == 0;
}

// Bytes of the staging buffer for spinor storage PS and Lx/2 = lxh.
__host__ __device__ inline size_t staged_smem_bytes(int PS, int lxh)
{
    const size_t ns = (size_t)STG_NROW * lxh;
    return PS == P32 ? ns * 96 : ns * 52;
}

// Checkerboard row index ((t Lz + z) Ly + y) of staging row r of the tile
// with origin (y0, z0, t0).
__device__ __forceinline__ int stg_row_global(const Geom& g, int r, int y0, int z0, int t0)
{
    int yl, zl, tl;
    if (r < STG_NIN) {
        yl = r % STG_TY;
        zl = (r / STG_TY) % STG_TZ;
        tl = r / (STG_TY * STG_TZ);
    } else if (r < STG_NIN + 2 * STG_FY) {
        const int q = r - STG_NIN, f = q % STG_FY;
        yl = q < STG_FY ? -1 : STG_TY;
        zl = f % STG_TZ;
        tl = f / STG_TZ;
    } else if (r < STG_NIN + 2 * (STG_FY + STG_FZ)) {
        const int q = r - STG_NIN - 2 * STG_FY, f = q % STG_FZ;
        zl = q < STG_FZ ? -1 : STG_TZ;
        yl = f % STG_TY;
        tl = f / STG_TY;
    } else {
        const int q = r - STG_NIN - 2 * (STG_FY + STG_FZ), f = q % STG_FT;
        tl = q < STG_FT ? -1 : STG_TT;
        yl = f % STG_TY;
        zl = f / STG_TY;
    }
    int y = y0 + yl, z = z0 + zl, t = t0 + tl;
    y = y < 0 ? y + g.L[1] : (y >= g.L[1] ? y - g.L[1] : y);
    z = z < 0 ? z + g.L[2] : (z >= g.L[2] ? z - g.L[2] : z);
    t = t < 0 ? t + g.L[3] : (t >= g.L[3] ? t - g.L[3] : t);
    return (t * g.L[2] + z) * g.L[1] + y;
}

__device__ __forceinline__ void cp_async16(void* dst, const void* src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}
__device__ __forceinline__ void cp_async4(void* dst, const void* src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}

// A staged spinor (row-major staging rows, the field's chunk order).
__device__ __forceinline__ void load_staged(const unsigned char* sm, int ns, int j, HopSpinor<P32>& q)
{
    const float4* p = reinterpret_cast<const float4*>(sm);
#pragma unroll
    for (int k = 0; k < 6; ++k) {
        const float4 c = p[k * ns + j];
        q.v[4 * k] = c.x;
        q.v[4 * k + 1] = c.y;
        q.v[4 * k + 2] = c.z;
        q.v[4 * k + 3] = c.w;
    }
}
template <int ISBF>
__device__ __forceinline__ void load_staged(const unsigned char* sm, int ns, int j, HopSpinorHalf<ISBF>& q)
{
    const uint4* p = reinterpret_cast<const uint4*>(sm);
    q.n = reinterpret_cast<const float*>(p + 3 * ns)[j];
    const uint4 s[3] = {p[j], p[ns + j], p[2 * ns + j]};
    q.set(s);
}

// One hop direction of the staged kernel: the neighbours' staging indices
// jf, jb, the backward link's checkerboard index bwd_cb.
template <int PG, int PS, int RECON, int MU, bool DAG>
__device__ __forceinline__ void hop_dir_staged(const DslashArgs& A, const unsigned char* sm, int ns, int i, int jf,
                                               int jb, int bwd_cb, bool flipf, bool flipb, float acc[24])
{
    HopSpinor<PS> q;
    load_staged(sm, ns, jf, q);
    q.flip = flipf;
    hop_term<PG, PS, RECON, MU, DAG, false, true>(A, q, A.par, i, acc);
    load_staged(sm, ns, jb, q);
    q.flip = flipb;
    hop_term<PG, PS, RECON, MU, DAG, true, true>(A, q, 1 - A.par, bwd_cb, acc);
}

// Block b: right-hand side b % nrhs, tile b / nrhs (y fastest, then z, t);
// blockDim = STG_NIN * Lx/2.  Same arithmetic, in the same order, as the
// gathering kernel's plain launches.
template <int PG, int PS, int RECON, bool DAG, int EPI>
__global__ void __launch_bounds__(STG_NIN * STG_MAXLXH, 2) dslash_staged_kernel(const DslashArgs A)
{
    extern __shared__ __align__(16) unsigned char stg_smem[];
    const Geom& g = A.g;
    const int rhs = (int)(blockIdx.x % (unsigned)A.nrhs);
    if (A.skip && A.skip[rhs]) return;  // uniform over the block
    const int tile = (int)(blockIdx.x / (unsigned)A.nrhs);
    const int nty = g.L[1] / STG_TY, ntz = g.L[2] / STG_TZ;
    const int y0 = (tile % nty) * STG_TY, z0 = ((tile / nty) % ntz) * STG_TZ, t0 = (tile / (nty * ntz)) * STG_TT;
    const int lxh = g.Lxh, ns = STG_NROW * lxh;
    const int xh = threadIdx.x % lxh, rl = threadIdx.x / lxh;  // this thread's site in the tile
    const char* in = static_cast<const char*>(A.in) + rhs * A.in_rb;

    // stage: thread (rl, xh) copies column xh of rows rl, rl + NIN, ... of every chunk
    constexpr int NCH = PS == P32 ? 6 : 3;
    for (int q = rl; q < NCH * STG_NROW; q += STG_NIN) {
        const int k = q / STG_NROW, r = q - k * STG_NROW;
        const int gi = stg_row_global(g, r, y0, z0, t0) * lxh + xh;
        cp_async16(stg_smem + ((size_t)k * ns + r * lxh + xh) * 16, in + ((size_t)k * g.stride + gi) * 16);
    }
    if constexpr (PS != P32) {  // the per-site norms
        for (int r = rl; r < STG_NROW; r += STG_NIN) {
            const int gi = stg_row_global(g, r, y0, z0, t0) * lxh + xh;
            cp_async4(stg_smem + (size_t)3 * ns * 16 + (size_t)(r * lxh + xh) * 4,
                      in + (size_t)3 * g.stride * 16 + (size_t)gi * 4);
        }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();

    const int yl = rl % STG_TY, zl = (rl / STG_TY) % STG_TZ, tl = rl / (STG_TY * STG_TZ);
    int c[4];
    c[1] = y0 + yl;
    c[2] = z0 + zl;
    c[3] = t0 + tl;
    c[0] = 2 * xh + ((c[1] + c[2] + c[3] + A.par) & 1);
    const int i = ((c[3] * g.L[2] + c[2]) * g.L[1] + c[1]) * lxh + xh;
    const int full = full_index(g, c);
    const int row = rl * lxh;
    float acc[24];
#pragma unroll
    for (int k = 0; k < 24; ++k) acc[k] = 0.f;
    // staging indices of the eight neighbours and checkerboard indices of the backward links
    {
        const int xf = c[0] == g.L[0] - 1 ? 0 : c[0] + 1, xb = c[0] == 0 ? g.L[0] - 1 : c[0] - 1;
        const int bwd = c[0] == 0 ? full + (g.L[0] - 1) : full - 1;
        hop_dir_staged<PG, PS, RECON, 0, DAG>(A, stg_smem, ns, i, row + (xf >> 1), row + (xb >> 1), bwd >> 1, false,
                                              false, acc);
    }
    {
        const int s1 = g.L[0];
        const int jf = (yl + 1 < STG_TY ? rl + 1 : STG_NIN + STG_FY + tl * STG_TZ + zl) * lxh + xh;
        const int jb = (yl > 0 ? rl - 1 : STG_NIN + tl * STG_TZ + zl) * lxh + xh;
        const int bwd = c[1] == 0 ? full + (g.L[1] - 1) * s1 : full - s1;
        hop_dir_staged<PG, PS, RECON, 1, DAG>(A, stg_smem, ns, i, jf, jb, bwd >> 1, false, false, acc);
    }
    {
        const int s2 = g.L[0] * g.L[1];
        constexpr int bz = STG_NIN + 2 * STG_FY;
        const int jf = (zl + 1 < STG_TZ ? rl + STG_TY : bz + STG_FZ + tl * STG_TY + yl) * lxh + xh;
        const int jb = (zl > 0 ? rl - STG_TY : bz + tl * STG_TY + yl) * lxh + xh;
        const int bwd = c[2] == 0 ? full + (g.L[2] - 1) * s2 : full - s2;
        hop_dir_staged<PG, PS, RECON, 2, DAG>(A, stg_smem, ns, i, jf, jb, bwd >> 1, false, false, acc);
    }
    {
        const int s3 = g.L[0] * g.L[1] * g.L[2];
        constexpr int bt = STG_NIN + 2 * (STG_FY + STG_FZ);
        const int jf = (tl + 1 < STG_TT ? rl + STG_TY * STG_TZ : bt + STG_FT + zl * STG_TY + yl) * lxh + xh;
        const int jb = (tl > 0 ? rl - STG_TY * STG_TZ : bt + zl * STG_TY + yl) * lxh + xh;
        const int bwd = c[3] == 0 ? full + (g.L[3] - 1) * s3 : full - s3;
        const bool tb = g.tanti != 0;
        hop_dir_staged<PG, PS, RECON, 3, DAG>(A, stg_smem, ns, i, jf, jb, bwd >> 1, tb && c[3] == g.L[3] - 1,
                                              tb && c[3] == 0, acc);
    }
    double nrm = 0.0;
    dslash_epilogue<PG, PS, DAG, EPI, false>(A, rhs, i, acc, nrm, 0);
}

template <int PG, int PS, int RECON, bool DAG, int EPI>
cudaError_t launch_staged_t(const DslashArgs& A, int nrhs, cudaStream_t s)
{
    // the largest buffer (Lx/2 = 16) is allowed once per instantiation and device
    static bool attr[64] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64 || !attr[dev]) {
        e = cudaFuncSetAttribute(dslash_staged_kernel<PG, PS, RECON, DAG, EPI>,
                                 cudaFuncAttributeMaxDynamicSharedMemorySize, (int)staged_smem_bytes(PS, STG_MAXLXH));
        if (e != cudaSuccess) return e;
        if (dev >= 0 && dev < 64) attr[dev] = true;
    }
    const long tiles = (long)(A.g.L[1] / STG_TY) * (A.g.L[2] / STG_TZ) * (A.g.L[3] / STG_TT);
    if (tiles * nrhs > 0x7fffffffL) return cudaErrorInvalidConfiguration;
    DslashArgs Ar = A;
    Ar.nrhs = nrhs;
    dslash_staged_kernel<PG, PS, RECON, DAG, EPI>
        <<<(unsigned)(tiles * nrhs), STG_NIN * A.g.Lxh, staged_smem_bytes(PS, A.g.Lxh), s>>>(Ar);
    return cudaGetLastError();
}

// Runtime dispatch over (recon, dag, epi, red) for fixed storage precisions.
// block == DSLASH_STAGED: the staged kernel where it applies (plain launches
// with FP32 links on an uncut lattice whose extents fit its tiles), else the
// gathering kernel with its default block.
template <int PG, int PS>
cudaError_t dispatch_dslash_p(const DslashArgs& A, int recon, bool dag, int epi, bool red, int nrhs, int block,
                              cudaStream_t s)
{
    if (block == DSLASH_STAGED) {
        if constexpr (PG == P32 && PS != P64) {
            if (!red && epi != EPI_CG && recon == 12 && staged_supported(A.g)) {
#define LQ_SCASE(DG, EP) \
    if (dag == DG && epi == EP) return launch_staged_t<PG, PS, 12, DG, EP>(A, nrhs, s);
                LQ_SCASE(false, EPI_NONE)
                LQ_SCASE(false, EPI_CLOVINV)
                LQ_SCASE(false, EPI_XPAY)
                LQ_SCASE(true, EPI_NONE)
                LQ_SCASE(true, EPI_CLOVINV)
                LQ_SCASE(true, EPI_XPAY)
#undef LQ_SCASE
            }
        }
        block = DSLASH_MAX_BLOCK;
    }
#define LQ_CASE(RC, DG, EP, RD)                                                              \
    if (recon == RC && dag == DG && epi == EP && red == RD)                                 \
        return block == DSLASH_WIDE ? launch_wide_t<PG, PS, RC, DG, EP, RD>(A, nrhs, s)       \
                                    : launch_dslash_t<PG, PS, RC, DG, EP, RD>(A, nrhs, block, s);
#define LQ_EPIS(RC, DG)                  \
    LQ_CASE(RC, DG, EPI_NONE, false)     \
    LQ_CASE(RC, DG, EPI_CLOVINV, false)  \
    LQ_CASE(RC, DG, EPI_XPAY, false)     \
    LQ_CASE(RC, DG, EPI_XPAY, true)      \
    LQ_CASE(RC, DG, EPI_CG, true)
    if constexpr (PG == P64) {
        LQ_EPIS(18, false)
        LQ_EPIS(18, true)
    } else {
        LQ_EPIS(12, false)
        LQ_EPIS(12, true)
        LQ_EPIS(18, false)
        LQ_EPIS(18, true)
    }
#undef LQ_EPIS
#undef LQ_CASE
    return cudaErrorInvalidValue;
}

}  // namespace lqcd
