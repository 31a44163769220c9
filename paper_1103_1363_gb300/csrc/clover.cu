// Clover term A(x) = 1 + i kappa csw sum_{mu<nu} sigma_{mu nu} Fhat_{mu nu}(x):
// build from the four-leaf field strength, invert, round to every held
// precision, and apply.  Build and inversion run in FP64 (the FP64 residual
// of the mixed-precision solver needs A to FP64 accuracy).  The leaf
// products are per-site SU(3) matrix products, the memory-bound kernel the
// paper uses as its example of the information-flow model (Sec. 3, Eq. (3)).
#include "internal.h"

namespace lqcd {

// 3x3 complex matrices as 18 doubles, row-major, (re, im) interleaved.
// Entry (i, j) of a, or of a^dag.
template <bool DAGGER>
__device__ __forceinline__ void m3_entry(const double a[18], int i, int j, double& re, double& im)
{
    const int k = DAGGER ? 2 * (3 * j + i) : 2 * (3 * i + j);
    re = a[k];
    im = DAGGER ? -a[k + 1] : a[k + 1];
}

// out (+)= s op(a) op(b), op = dagger where the flag says so, s = +1 or -1;
// one multiply-add per real product.
template <bool DA, bool DB, bool ACC, int S>
__device__ __forceinline__ void m3_mul(const double a[18], const double b[18], double out[18])
{
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            double re = ACC ? out[2 * (3 * i + j)] : 0.0, im = ACC ? out[2 * (3 * i + j) + 1] : 0.0;
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                double ar, ai, br, bi;
                m3_entry<DA>(a, i, k, ar, ai);
                m3_entry<DB>(b, k, j, br, bi);
                re += S * ar * br;
                re -= S * ai * bi;
                im += S * ar * bi;
                im += S * ai * br;
            }
            out[2 * (3 * i + j)] = re;
            out[2 * (3 * i + j) + 1] = im;
        }
}

// g = a b - (a b)^dag as 9 reals: the imaginary diagonal, then the complex
// entries (1,0), (2,0), (2,1).
__device__ __forceinline__ void m3_mul_anti(const double a[18], const double b[18], double g[9])
{
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        double im = 0.0;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            im += a[2 * (3 * i + k)] * b[2 * (3 * k + i) + 1];
            im += a[2 * (3 * i + k) + 1] * b[2 * (3 * k + i)];
        }
        g[i] = 2.0 * im;
    }
    int q = 3;
#pragma unroll
    for (int i = 1; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < i; ++j) {
            double re = 0.0, im = 0.0;
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const double ur = a[2 * (3 * i + k)], ui = a[2 * (3 * i + k) + 1];
                const double vr = b[2 * (3 * k + j)], vi = b[2 * (3 * k + j) + 1];
                const double sr = a[2 * (3 * j + k)], si = a[2 * (3 * j + k) + 1];
                const double tr = b[2 * (3 * k + i)], ti = b[2 * (3 * k + i) + 1];
                re += ur * vr;  // (a b)_ij - conj((a b)_ji)
                re -= ui * vi;
                re -= sr * tr;
                re += si * ti;
                im += ur * vi;
                im += ui * vr;
                im += sr * ti;
                im += si * tr;
            }
            g[q++] = re;
            g[q++] = im;
        }
}

// Checkerboard index of the site DM steps along MU and DN along NU from c (each -1, 0 or 1).
template <int MU, int DM, int NU, int DN>
__device__ __forceinline__ int cb_shift(const Geom& g, const int c[4])
{
    int d[4] = {c[0], c[1], c[2], c[3]};
    if (DM > 0) d[MU] = d[MU] == g.L[MU] - 1 ? 0 : d[MU] + 1;
    if (DM < 0) d[MU] = d[MU] == 0 ? g.L[MU] - 1 : d[MU] - 1;
    if (DN > 0) d[NU] = d[NU] == g.L[NU] - 1 ? 0 : d[NU] + 1;
    if (DN < 0) d[NU] = d[NU] == 0 ? g.L[NU] - 1 : d[NU] - 1;
    return full_index(g, d) >> 1;
}

// Field strength.  With the staples of the link (x, mu) in the mu-nu plane,
//   T(x) = U_nu(x+mu) U_mu(x+nu)^dag U_nu(x)^dag - U_nu(x+mu-nu)^dag U_mu(x-nu)^dag U_nu(x-nu),
// the sum Q of the four plaquette leaves at x (all circulating mu -> nu) has
//   Q - Q^dag = anti(U_mu(x) T(x)) + anti(T(x-mu) U_mu(x-mu)),  anti(X) = X - X^dag:
// a leaf and its adjoint have opposite anti-parts, so the lower staple enters
// with a minus sign, and the two leaves behind x hold the staples of x - mu.
// This kernel forms both terms at the link's own site, for one plane and
// site a thread: six 3x3 products (four whole, two of which only the
// anti-Hermitian part is formed) where the four leaves took twelve, and six
// times the threads of a thread per site, which small lattices need.
//
// The bound is the FP64 pipe (1.256 TFLOP/s measured: a warp's multiply-add
// occupies it for 15 cycles), so the count of FP64 instructions is what
// matters: about 650 a plane and site here.  The terms go through scratch
// (2 x 9 doubles a plane and site, 864 bytes written and read a site, a
// tenth of the time).  At 16^3 x 32: 810 us; the four leaves per site,
// with their twelve products and arrays in local memory, took 3218 us.
enum { CLOVER_PLANES = 6, CLOVER_TERM = 9 };

// element q of term `which` (0: at x, 1: for x + mu) of a plane, at site i of parity par
__device__ __forceinline__ size_t term_at(const Geom& g, int plane, int which, int q, int par, int i)
{
    return ((size_t)((plane * 2 + which) * CLOVER_TERM + q) * 2 + par) * g.stride + i;
}

template <int MU, int NU>
__device__ __forceinline__ void plane_terms(const Geom& g, const void* gauge, int plane, int par, int i, double* terms)
{
    typedef GaugeIO<P64, 18> IO;
    int c[4];
    cb_coords(g, i, par, c);
    double u[18], v[18], m[18], t[18], q[9];
    // upper staple
    IO::load(gauge, g.stride, par, NU, i, u);
    IO::load(gauge, g.stride, 1 - par, MU, cb_shift<MU, 0, NU, 1>(g, c), v);
    m3_mul<false, false, false, 1>(u, v, m);
    IO::load(gauge, g.stride, 1 - par, NU, cb_shift<MU, 1, NU, 0>(g, c), u);
    m3_mul<false, true, false, 1>(u, m, t);
    // minus the lower one
    IO::load(gauge, g.stride, 1 - par, MU, cb_shift<MU, 0, NU, -1>(g, c), u);
    IO::load(gauge, g.stride, par, NU, cb_shift<MU, 1, NU, -1>(g, c), v);
    m3_mul<false, false, false, 1>(u, v, m);
    IO::load(gauge, g.stride, 1 - par, NU, cb_shift<MU, 0, NU, -1>(g, c), u);
    m3_mul<true, false, true, -1>(m, u, t);
    IO::load(gauge, g.stride, par, MU, i, u);
    m3_mul_anti(u, t, q);
#pragma unroll
    for (int k = 0; k < CLOVER_TERM; ++k) terms[term_at(g, plane, 0, k, par, i)] = q[k];
    m3_mul_anti(t, u, q);
#pragma unroll
    for (int k = 0; k < CLOVER_TERM; ++k) terms[term_at(g, plane, 1, k, par, i)] = q[k];
}

// blockIdx.y: plane (xy, xz, xt, yz, yt, zt); blockIdx.z: parity.
__global__ void __launch_bounds__(64) clover_terms_kernel(Geom g, const void* gauge, double* terms)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int plane = blockIdx.y, par = blockIdx.z;
    if (i >= g.Vh) return;
    switch (plane) {
    case 0: plane_terms<0, 1>(g, gauge, 0, par, i, terms); break;
    case 1: plane_terms<0, 2>(g, gauge, 1, par, i, terms); break;
    case 2: plane_terms<0, 3>(g, gauge, 2, par, i, terms); break;
    case 3: plane_terms<1, 2>(g, gauge, 3, par, i, terms); break;
    case 4: plane_terms<1, 3>(g, gauge, 4, par, i, terms); break;
    default: plane_terms<2, 3>(g, gauge, 5, par, i, terms); break;
    }
}

// Packed position of the real part of entry (r, s), r > s, of a 6x6 Hermitian block.
__host__ __device__ constexpr int herm6_at(int r, int s) { return 6 + r * (r - 1) + 2 * s; }

// Inverse of a packed Hermitian block by Gauss-Jordan with partial pivoting
// (rows); false if a pivot is below 1e-12.  The general case: indexed rows
// live in local memory.
__device__ __noinline__ bool invert_pivoting(const double c[36], double out[36])
{
    double m[6][6][2], inv[6][6][2];
    for (int r = 0; r < 6; ++r)
        for (int s = 0; s < 6; ++s) {
            const int k = r > s ? herm6_at(r, s) : herm6_at(s, r);
            m[r][s][0] = r == s ? c[r] : c[k];
            m[r][s][1] = r == s ? 0.0 : r > s ? c[k + 1] : -c[k + 1];
            inv[r][s][0] = (r == s) ? 1.0 : 0.0;
            inv[r][s][1] = 0.0;
        }
    bool ok = true;
    for (int col = 0; col < 6; ++col) {
        int piv = col;
        double best = hypot(m[col][col][0], m[col][col][1]);
        for (int r = col + 1; r < 6; ++r) {
            const double v = hypot(m[r][col][0], m[r][col][1]);
            if (v > best) { best = v; piv = r; }
        }
        if (best < 1e-12) { ok = false; break; }
        if (piv != col)
            for (int s = 0; s < 6; ++s)
                for (int q = 0; q < 2; ++q) {
                    double tmp = m[col][s][q]; m[col][s][q] = m[piv][s][q]; m[piv][s][q] = tmp;
                    tmp = inv[col][s][q]; inv[col][s][q] = inv[piv][s][q]; inv[piv][s][q] = tmp;
                }
        // scale the pivot row by 1 / m[col][col]
        const double pr = m[col][col][0], pi = m[col][col][1];
        const double den = pr * pr + pi * pi;
        const double ir = pr / den, ii = -pi / den;
        for (int s = 0; s < 6; ++s) {
            double xr = m[col][s][0], xi = m[col][s][1];
            m[col][s][0] = xr * ir - xi * ii;
            m[col][s][1] = xr * ii + xi * ir;
            xr = inv[col][s][0]; xi = inv[col][s][1];
            inv[col][s][0] = xr * ir - xi * ii;
            inv[col][s][1] = xr * ii + xi * ir;
        }
        for (int r = 0; r < 6; ++r) {
            if (r == col) continue;
            const double fr = m[r][col][0], fi = m[r][col][1];
            for (int s = 0; s < 6; ++s) {
                m[r][s][0] -= fr * m[col][s][0] - fi * m[col][s][1];
                m[r][s][1] -= fr * m[col][s][1] + fi * m[col][s][0];
                inv[r][s][0] -= fr * inv[col][s][0] - fi * inv[col][s][1];
                inv[r][s][1] -= fr * inv[col][s][1] + fi * inv[col][s][0];
            }
        }
    }
    for (int r = 0; r < 6; ++r) {
        out[r] = inv[r][r][0];
        for (int s = 0; s < r; ++s) {
            out[herm6_at(r, s)] = inv[r][s][0];
            out[herm6_at(r, s) + 1] = inv[r][s][1];
        }
    }
    return ok;
}

// The same elimination where no row has to be exchanged: the pivots are the
// diagonal entries.  Swept in place the matrix stays Hermitian up to the sign
// of the entries between swept and unswept rows (M_kj = -conj(M_jk)), so the
// lower triangle in registers is enough: 60 multiply-adds and one division a
// pivot, against 290 and the pivot search's square roots.  False, with c
// destroyed, as soon as partial pivoting would exchange rows or the pivot is
// below 1e-12: the caller then takes invert_pivoting.
__device__ __forceinline__ bool invert_in_place(double c[36])
{
    bool ok = true;
#pragma unroll
    for (int k = 0; k < 6; ++k) {
        const double dk = c[k], d2 = dk * dk;
        double vr[6], vi[6];  // column k of the matrix
#pragma unroll
        for (int i = 0; i < 6; ++i) {
            if (i > k) {
                vr[i] = c[herm6_at(i, k)];
                vi[i] = c[herm6_at(i, k) + 1];
                ok = ok && d2 >= vr[i] * vr[i] + vi[i] * vi[i];
            } else if (i < k) {
                vr[i] = -c[herm6_at(k, i)];
                vi[i] = c[herm6_at(k, i) + 1];
            }
        }
        ok = ok && d2 >= 1e-24;
        const double p = 1.0 / dk;
#pragma unroll
        for (int i = 0; i < 6; ++i) {
            if (i == k) continue;
            const double tr = p * vr[i], ti = p * vi[i];
            // M_ij -= p v_i M_kj, M_kj = conj(v_j) for j > k and -conj(v_j) for j < k
#pragma unroll
            for (int j = 0; j < i; ++j) {
                if (j == k) continue;
                const int e = herm6_at(i, j);
                if (j > k) {
                    c[e] -= tr * vr[j];
                    c[e] -= ti * vi[j];
                    c[e + 1] += tr * vi[j];
                    c[e + 1] -= ti * vr[j];
                } else {
                    c[e] += tr * vr[j];
                    c[e] += ti * vi[j];
                    c[e + 1] -= tr * vi[j];
                    c[e + 1] += ti * vr[j];
                }
            }
            if (i > k) {
                c[i] -= tr * vr[i];
                c[i] -= ti * vi[i];
                c[herm6_at(i, k)] = -tr;
                c[herm6_at(i, k) + 1] = -ti;
            } else {
                c[i] += tr * vr[i];
                c[i] += ti * vi[i];
                c[herm6_at(k, i)] = -tr;  // p M_ki, M_ki = -conj(v_i)
                c[herm6_at(k, i) + 1] = ti;
            }
        }
        c[k] = p;
    }
    return ok;
}

// Where the blocks of A and A^{-1} go: per storage precision the field of
// both parities (nullptr: not held) and the bytes of one parity.
struct CloverOut {
    char* a[4];
    char* inv[4];
    size_t pb[4];
};

// Block b of site i, rounded to each held precision (through FP32 for the
// 16-bit ones, whose 36 halves a block are nine 8-byte pieces of the uint4 chunks).
__device__ __forceinline__ void store_rounded(char* const dst[4], const size_t pb[4], int stride, int par, int i, int b,
                                              const double c[36])
{
    CloverIO<P64>::store_block(dst[P64] + par * pb[P64], stride, i, b, c);
    float f[36];
#pragma unroll
    for (int k = 0; k < 36; ++k) f[k] = (float)c[k];
    if (dst[P32]) CloverIO<P32>::store_block(dst[P32] + par * pb[P32], stride, i, b, f);
#pragma unroll
    for (int P = P16; P <= PB16; ++P) {
        if (!dst[P]) continue;
        uint2* p = reinterpret_cast<uint2*>(dst[P] + par * pb[P]);
#pragma unroll
        for (int k = 0; k < 9; ++k) {
            const int piece = 9 * b + k;  // of the site's 18; two to a chunk
            p[((size_t)(piece >> 1) * stride + i) * 2 + (piece & 1)] =
                make_uint2(f2h(f[4 * k], f[4 * k + 1], P == PB16), f2h(f[4 * k + 2], f[4 * k + 3], P == PB16));
        }
    }
}

// Field strength terms -> A = 1 + i kc sum sigma Fhat, its inverse, and both
// in every held precision, in one pass.  Thread = (site, chiral block):
// threads 0..31 of a block of 64 take block 0 of 32 sites, 32..63 block 1
// (the second read of the terms hits L1).  sigma in the DeGrand-Rossi basis,
// worked out from (i/2)[g_mu, g_nu] (every sigma_{mu nu} commutes with g5):
// xy and zt are diagonal, diag(1,-1) and -+diag(1,-1) in the two blocks; xz
// and yt have (1,0) entries i and +-i; xt and yz have -+1 and 1.
// kc = kappa csw; Fhat = (Q - Q^dag)/8 made traceless.  FP64-bound like the
// terms: about 630 instructions a block.  At 16^3 x 32: 335 us; the
// inversion from memory (1570 us, local memory and pivot search) and the
// rounding passes (47 us) were kernels of their own.
__global__ void __launch_bounds__(64) clover_finish_kernel(Geom g, const double* __restrict__ terms, double kc,
                                                           CloverOut o, int* errw)
{
    const int b = threadIdx.x >> 5;
    const int i = blockIdx.x * 32 + (threadIdx.x & 31);
    const int par = blockIdx.y;
    if (i >= g.Vh) return;
    int c[4];
    cb_coords(g, i, par, c);
    const int back[3] = {cb_shift<0, -1, 1, 0>(g, c), cb_shift<1, -1, 0, 0>(g, c), cb_shift<2, -1, 0, 0>(g, c)};
    auto field = [&](int plane, int mu, double f[9]) {
#pragma unroll
        for (int q = 0; q < CLOVER_TERM; ++q)
            f[q] = terms[term_at(g, plane, 0, q, par, i)] + terms[term_at(g, plane, 1, q, 1 - par, back[mu])];
    };
    // e = F_xy + s F_zt, pp = F_yz + s F_xt, rr = F_xz - s F_yt with s = -1, +1 in the two blocks
    const double s = b ? 1.0 : -1.0;
    double e[9], pp[9], rr[9], f[9];
    field(0, 0, e);
    field(5, 2, f);
#pragma unroll
    for (int q = 0; q < 9; ++q) e[q] += s * f[q];
    field(3, 1, pp);
    field(2, 0, f);
#pragma unroll
    for (int q = 0; q < 9; ++q) pp[q] += s * f[q];
    field(1, 0, rr);
    field(4, 1, f);
#pragma unroll
    for (int q = 0; q < 9; ++q) rr[q] -= s * f[q];
    const double k8 = 0.125 * kc;
    auto scale = [&](double v[9]) {  // times k8, traceless
        const double tr = (v[0] + v[1] + v[2]) * (1.0 / 3.0);
#pragma unroll
        for (int q = 0; q < 9; ++q) v[q] = k8 * (q < 3 ? v[q] - tr : v[q]);
    };
    scale(e);
    scale(pp);
    scale(rr);
    double blk[36];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        // diagonal spin blocks 1 +- i e: the diagonal of e is imaginary
        blk[a] = 1.0 - e[a];
        blk[3 + a] = 1.0 + e[a];
#pragma unroll
        for (int q = 0; q < a; ++q) {
            const int l = a == 1 ? 3 : 5 + 2 * q;  // entry (a, q) of the 9 reals
            blk[herm6_at(a, q)] = -e[l + 1];
            blk[herm6_at(a, q) + 1] = e[l];
            blk[herm6_at(3 + a, 3 + q)] = e[l + 1];
            blk[herm6_at(3 + a, 3 + q) + 1] = -e[l];
        }
        // spin (1, 0): i pp - rr, with entry (c, a) = -conj of entry (a, c)
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            const int hi = a > q ? a : q, lo = a > q ? q : a;
            const int l = hi == 1 ? 3 : 5 + 2 * lo;
            double re, im;
            if (a == q) {
                re = -pp[a];
                im = -rr[a];
            } else if (a > q) {
                re = -pp[l + 1] - rr[l];
                im = pp[l] - rr[l + 1];
            } else {
                re = rr[l] - pp[l + 1];
                im = -pp[l] - rr[l + 1];
            }
            blk[herm6_at(3 + a, q)] = re;
            blk[herm6_at(3 + a, q) + 1] = im;
        }
    }
    store_rounded(o.a, o.pb, g.stride, par, i, b, blk);
    if (!invert_in_place(blk)) {
        double src[36];
        const double2* p = reinterpret_cast<const double2*>(o.a[P64] + par * o.pb[P64]) + (size_t)(18 * b) * g.stride + i;
        for (int k = 0; k < 18; ++k) {  // the block that this thread has just stored
            const double2 v = p[(size_t)k * g.stride];
            src[2 * k] = v.x;
            src[2 * k + 1] = v.y;
        }
        if (!invert_pivoting(src, blk)) atomicOr(errw, ERRW_CLOVER_SINGULAR);
    }
    store_rounded(o.inv, o.pb, g.stride, par, i, b, blk);
}

lqcd_status clover_build(lqcd_ctx* c, double kappa, double csw)
{
    // the field strength terms go through the solver vectors: 2 parities x 108 doubles a site
    static_assert(2 * CLOVER_PLANES * 2 * CLOVER_TERM * sizeof(double) <= NV64 * 2 * 192, "terms exceed the solver vectors");
    double* terms = reinterpret_cast<double*>(c->vec64);
    const int block = 64;
    clover_terms_kernel<<<dim3((c->g.Vh + block - 1) / block, CLOVER_PLANES, 2), block, 0, c->stream>>>(
        c->g, c->gauge[P64], terms);
    LQ_CUDA(cudaGetLastError());
    c->launches++;
    CloverOut o;
    for (int P = 0; P < 4; ++P) {
        o.a[P] = c->holds(P) ? static_cast<char*>(c->clov[P]) : nullptr;
        o.inv[P] = c->holds(P) ? static_cast<char*>(c->clovinv[P]) : nullptr;
        o.pb[P] = c->clov_parity_bytes(P);
    }
    clover_finish_kernel<<<dim3((c->g.Vh + 31) / 32, 2), block, 0, c->stream>>>(c->g, terms, kappa * csw, o, c->errw);
    LQ_CUDA(cudaGetLastError());
    c->launches++;
    return LQCD_OK;
}

// out = Cl in for one parity, Cl = A or A^{-1} stored in PG, spinors in PS.
template <int PG, int PS>
__global__ void clover_apply_kernel(Geom g, char* out, const char* in, const char* cl, size_t rb)
{
    typedef typename RealT<PS>::type R;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int rhs = blockIdx.y;
    if (i >= g.Vh) return;
    R v[24], w[24];
    SpinorIO<PS>::load(in + rhs * rb, g.stride, i, v);
    clover_apply_site<PG>(cl, g.stride, i, v, w);
    SpinorIO<PS>::store(out + rhs * rb, g.stride, i, w);
}

lqcd_status clover_apply_launch(lqcd_ctx* c, void* out, const void* in, int parity, int inverse, int mode, int nrhs,
                                size_t rb)
{
    const int block = 128;
    dim3 grid((c->g.Vh + block - 1) / block, nrhs);
    const int pg = mode_pg(mode);
    const char* cl = static_cast<const char*>(inverse ? c->clovinv[pg] : c->clov[pg]) + parity * c->clov_parity_bytes(pg);
    char* o = static_cast<char*>(out);
    const char* i = static_cast<const char*>(in);
    switch (mode) {
    case P64: clover_apply_kernel<P64, P64><<<grid, block, 0, c->stream>>>(c->g, o, i, cl, rb); break;
    case P32: clover_apply_kernel<P32, P32><<<grid, block, 0, c->stream>>>(c->g, o, i, cl, rb); break;
    case P16: clover_apply_kernel<P16, P16><<<grid, block, 0, c->stream>>>(c->g, o, i, cl, rb); break;
    case PB16: clover_apply_kernel<PB16, PB16><<<grid, block, 0, c->stream>>>(c->g, o, i, cl, rb); break;
    case MODE_F16_LINKS: clover_apply_kernel<P16, P32><<<grid, block, 0, c->stream>>>(c->g, o, i, cl, rb); break;
    case MODE_BF16_LINKS: clover_apply_kernel<PB16, P32><<<grid, block, 0, c->stream>>>(c->g, o, i, cl, rb); break;
    case MODE_F16_SPINORS: clover_apply_kernel<P32, P16><<<grid, block, 0, c->stream>>>(c->g, o, i, cl, rb); break;
    case MODE_BF16_SPINORS: clover_apply_kernel<P32, PB16><<<grid, block, 0, c->stream>>>(c->g, o, i, cl, rb); break;
    default: return fail(LQCD_ERR_INVALID, "clover apply: bad precision mode");
    }
    LQ_CUDA(cudaGetLastError());
    c->launches++;
    return LQCD_OK;
}

}  // namespace lqcd
