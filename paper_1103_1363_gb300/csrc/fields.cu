// Layout and precision conversions: canonical FP64 spinors and links to the
// parity-split structure-of-arrays fields of every precision, and back.
#include "internal.h"

namespace lqcd {

// ---- canonical spinors <-> fields
// A canonical site is one stretch of memory (192 bytes in FP64, 96 in FP32),
// the sites of one parity every other one; a field is planes over the sites.
// Writing canonical sites goes through shared memory, FIELD_SITES sites a
// block, so that consecutive threads write consecutive 16-byte pieces of a
// site: a thread per site wrote half sectors (16 FP64 spinors of 16^4: 168 us,
// 2.4 TB/s; now 74, 5.4 TB/s).  Reading them does not need it: L1 holds the
// rest of a line for the thread's next load, 72 us against 87 when staged.
// blockIdx.y: right-hand side, blockIdx.z: parity (par < 0: both, the odd field
// fb bytes after the even one).
enum { FIELD_SITES = 128 };

// Staging of FIELD_SITES sites of N 16-byte pieces (an odd pitch N + 1: the
// eight lanes of a 16-byte access phase hit different banks).
template <class T, int N>
struct SiteStage {
    static_assert(sizeof(T) == 16 && N % 2 == 0, "16-byte pieces, an odd pitch");
    T v[FIELD_SITES][N + 1];
    int full[FIELD_SITES];  // canonical site index, -1 past the end
    // this thread's site; returns its checkerboard index
    __device__ __forceinline__ int set_site(const Geom& g, int par)
    {
        const int i = blockIdx.x * FIELD_SITES + threadIdx.x;
        int c[4];
        cb_coords(g, i, par, c);
        full[threadIdx.x] = i < g.Vh ? full_index(g, c) : -1;
        return i;
    }
    // f(piece in shared memory, index of the piece in the canonical array)
    template <class F>
    __device__ __forceinline__ void each_piece(F f)
    {
#pragma unroll
        for (int q = 0; q < N; ++q) {
            const int e = q * FIELD_SITES + threadIdx.x, site = e / N, k = e - site * N;
            if (full[site] >= 0) f(v[site][k], (size_t)full[site] * N + k);
        }
    }
};

template <int P>
__global__ void __launch_bounds__(FIELD_SITES) pack_kernel(Geom g, int par0, const double* __restrict__ canon,
                                                           size_t canon_rb, char* out, size_t out_rb, size_t fb)
{
    typedef typename RealT<P>::type R;
    const int i = blockIdx.x * FIELD_SITES + threadIdx.x;
    const int rhs = blockIdx.y, par = par0 < 0 ? (int)blockIdx.z : par0;
    if (i >= g.Vh) return;
    int c[4];
    cb_coords(g, i, par, c);
    const double2* src = reinterpret_cast<const double2*>(reinterpret_cast<const char*>(canon) + rhs * canon_rb) +
                         (size_t)full_index(g, c) * 12;
    R v[24];
#pragma unroll
    for (int k = 0; k < 12; ++k) {
        const double2 d = src[k];
        v[2 * k] = (R)d.x;
        v[2 * k + 1] = (R)d.y;
    }
    SpinorIO<P>::store(out + rhs * out_rb + (par0 < 0 ? par * fb : 0), g.stride, i, v);
}

template <int P>
__global__ void __launch_bounds__(FIELD_SITES) unpack_kernel(Geom g, int par0, double* canon, size_t canon_rb,
                                                             const char* in, size_t in_rb, size_t fb)
{
    typedef typename RealT<P>::type R;
    __shared__ SiteStage<double2, 12> st;
    const int rhs = blockIdx.y, par = par0 < 0 ? (int)blockIdx.z : par0;
    double2* dst = reinterpret_cast<double2*>(reinterpret_cast<char*>(canon) + rhs * canon_rb);
    const int i = st.set_site(g, par);
    if (i < g.Vh) {
        R v[24];
        SpinorIO<P>::load(in + rhs * in_rb + (par0 < 0 ? par * fb : 0), g.stride, i, v);
#pragma unroll
        for (int k = 0; k < 12; ++k) st.v[threadIdx.x][k] = make_double2((double)v[2 * k], (double)v[2 * k + 1]);
    }
    __syncthreads();
    st.each_piece([&](double2& s, size_t at) { dst[at] = s; });
}

// FP64 full internal field = canonical a - b (b may be null: 0).
__global__ void __launch_bounds__(FIELD_SITES) pack_difference_kernel(Geom g, const double* __restrict__ a,
                                                                      const double* __restrict__ b, size_t canon_rb,
                                                                      char* out, size_t out_rb, size_t fb)
{
    const int i = blockIdx.x * FIELD_SITES + threadIdx.x;
    const int rhs = blockIdx.y, par = blockIdx.z;
    if (i >= g.Vh) return;
    int c[4];
    cb_coords(g, i, par, c);
    const size_t off = rhs * canon_rb / sizeof(double) + (size_t)full_index(g, c) * 24;
    double v[24];
#pragma unroll
    for (int k = 0; k < 12; ++k) {
        const double2 p = reinterpret_cast<const double2*>(a + off)[k];
        const double2 q = b ? reinterpret_cast<const double2*>(b + off)[k] : make_double2(0.0, 0.0);
        v[2 * k] = p.x - q.x;
        v[2 * k + 1] = p.y - q.y;
    }
    SpinorIO<P64>::store(out + rhs * out_rb + par * fb, g.stride, i, v);
}

// FP64 full internal field -> canonical FP32 complex spinor.
__global__ void __launch_bounds__(FIELD_SITES) unpack_f32_kernel(Geom g, float* canon, size_t canon_rb, const char* in,
                                                                 size_t in_rb, size_t fb)
{
    __shared__ SiteStage<float4, 6> st;
    const int rhs = blockIdx.y, par = blockIdx.z;
    float4* dst = reinterpret_cast<float4*>(reinterpret_cast<char*>(canon) + rhs * canon_rb);
    const int i = st.set_site(g, par);
    if (i < g.Vh) {
        double v[24];
        SpinorIO<P64>::load(in + rhs * in_rb + par * fb, g.stride, i, v);
#pragma unroll
        for (int k = 0; k < 6; ++k)
            st.v[threadIdx.x][k] = make_float4((float)v[4 * k], (float)v[4 * k + 1], (float)v[4 * k + 2], (float)v[4 * k + 3]);
    }
    __syncthreads();
    st.each_piece([&](float4& s, size_t at) { dst[at] = s; });
}

// Canonical links of the slices t0 <= t < t1 (the array starts at site (t0, 0,
// 0, 0)) to the field of every held precision (out[P], nullptr: not held).  A
// block stages GAUGE_SITES sites' four links, 576 bytes in one stretch each,
// in shared memory, once for all precisions; then a thread takes one link.
// (A pass per precision with a thread per link on both sides: FP64 and FP32
// recon-12 at 16^3 x 32 33 + 22 us, now 33.)
enum { GAUGE_SITES = 32 };
struct GaugeOut {
    void* out[4];
};

template <int RECON>
__global__ void __launch_bounds__(4 * GAUGE_SITES) gauge_pack_kernel(Geom g, const double* __restrict__ slice, int t0,
                                                                     int t1, int aligned, GaugeOut o)
{
    __shared__ double2 st[GAUGE_SITES][37];  // 36 pieces a site
    __shared__ int full[GAUGE_SITES];
    const int per_t = g.Vh / g.L[3];
    const int n = per_t * (t1 - t0);
    const int par = blockIdx.y;
    const int idx0 = blockIdx.x * GAUGE_SITES;
    if (threadIdx.x < GAUGE_SITES) {
        const int idx = idx0 + threadIdx.x;
        int c[4];
        cb_coords(g, idx + t0 * per_t, par, c);
        full[threadIdx.x] = idx < n ? full_index(g, c) - t0 * per_t * 2 : -1;
    }
    __syncthreads();
    for (int e = threadIdx.x; e < GAUGE_SITES * 36; e += 4 * GAUGE_SITES) {
        const int site = e / 36, k = e - site * 36;
        if (full[site] < 0) continue;
        const size_t at = (size_t)full[site] * 36 + k;
        if (aligned) st[site][k] = ld_fixed(reinterpret_cast<const double2*>(slice) + at);
        else st[site][k] = make_double2(ld_fixed(slice + 2 * at), ld_fixed(slice + 2 * at + 1));
    }
    __syncthreads();
    const int site = threadIdx.x % GAUGE_SITES, mu = threadIdx.x / GAUGE_SITES;
    if (idx0 + site >= n) return;
    const int i = idx0 + site + t0 * per_t;  // checkerboard index (t is the slowest coordinate)
    double u[18];
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        const double2 d = st[site][9 * mu + k];
        u[2 * k] = d.x;
        u[2 * k + 1] = d.y;
    }
    GaugeIO<P64, 18>::store(o.out[P64], g.stride, par, mu, i, u);
    float f[18];
#pragma unroll
    for (int k = 0; k < 18; ++k) f[k] = (float)u[k];
    if (o.out[P32]) GaugeIO<P32, RECON>::store(o.out[P32], g.stride, par, mu, i, f);
    if (o.out[P16]) GaugeIO<P16, RECON>::store(o.out[P16], g.stride, par, mu, i, f);
    if (o.out[PB16]) GaugeIO<PB16, RECON>::store(o.out[PB16], g.stride, par, mu, i, f);
}

template <int PIN, int POUT>
__global__ void convert_kernel(Geom g, char* out, size_t out_rb, const char* in, size_t in_rb, int nfield,
                               double* partials, size_t part_rs, unsigned* tickets, double* red, size_t red_rs)
{
    typedef typename RealT<PIN>::type RI;
    typedef typename RealT<POUT>::type RO;
    const int rhs = blockIdx.y;
    double nrm = 0.0;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < g.Vh; i += gridDim.x * blockDim.x) {
        for (int f = 0; f < nfield; ++f) {
            RI v[24];
            RO w[24];
            SpinorIO<PIN>::load(in + rhs * in_rb + f * spinor_field_bytes(PIN, g.stride), g.stride, i, v);
#pragma unroll
            for (int k = 0; k < 24; ++k) {
                w[k] = (RO)v[k];
                nrm += (double)v[k] * (double)v[k];
            }
            SpinorIO<POUT>::store(out + rhs * out_rb + f * spinor_field_bytes(POUT, g.stride), g.stride, i, w);
        }
    }
    if (partials) {
        double v[1] = {nrm};
        block_reduce_finalize<1>(v, partials + rhs * part_rs, tickets + rhs, red + rhs * red_rs);
    }
}

// blocks over the sites of one parity, right-hand sides, parities (parity < 0: both)
static dim3 field_grid(const lqcd_ctx* c, int parity, int nrhs)
{
    return dim3((c->g.Vh + FIELD_SITES - 1) / FIELD_SITES, nrhs, parity < 0 ? 2 : 1);
}

lqcd_status pack_spinor(lqcd_ctx* c, void* internal, const double* canon, int parity, int P, int nrhs,
                        size_t internal_rb, size_t canon_rb)
{
    const dim3 grid = field_grid(c, parity, nrhs);
    char* out = static_cast<char*>(internal);
    const size_t fb = spinor_field_bytes(P, c->g.stride);
#define LQ_PK(PP) pack_kernel<PP><<<grid, FIELD_SITES, 0, c->stream>>>(c->g, parity, canon, canon_rb, out, internal_rb, fb)
    switch (P) {
    case P64: LQ_PK(P64); break;
    case P32: LQ_PK(P32); break;
    case P16: LQ_PK(P16); break;
    default: LQ_PK(PB16); break;
    }
#undef LQ_PK
    LQ_CUDA(cudaGetLastError());
    c->launches++;
    return LQCD_OK;
}

lqcd_status unpack_spinor(lqcd_ctx* c, double* canon, const void* internal, int parity, int P, int nrhs,
                          size_t internal_rb, size_t canon_rb)
{
    const dim3 grid = field_grid(c, parity, nrhs);
    const char* in = static_cast<const char*>(internal);
    const size_t fb = spinor_field_bytes(P, c->g.stride);
#define LQ_UP(PP) unpack_kernel<PP><<<grid, FIELD_SITES, 0, c->stream>>>(c->g, parity, canon, canon_rb, in, internal_rb, fb)
    switch (P) {
    case P64: LQ_UP(P64); break;
    case P32: LQ_UP(P32); break;
    case P16: LQ_UP(P16); break;
    default: LQ_UP(PB16); break;
    }
#undef LQ_UP
    LQ_CUDA(cudaGetLastError());
    c->launches++;
    return LQCD_OK;
}

lqcd_status pack_difference(lqcd_ctx* c, void* internal, const double* a, const double* b, int nrhs,
                            size_t internal_rb, size_t canon_rb)
{
    pack_difference_kernel<<<field_grid(c, -1, nrhs), FIELD_SITES, 0, c->stream>>>(
        c->g, a, b, canon_rb, static_cast<char*>(internal), internal_rb, c->field_bytes(P64));
    LQ_CUDA(cudaGetLastError());
    c->launches++;
    return LQCD_OK;
}

lqcd_status unpack_spinor_f32(lqcd_ctx* c, float* canon, const void* internal, int nrhs, size_t internal_rb,
                              size_t canon_rb)
{
    unpack_f32_kernel<<<field_grid(c, -1, nrhs), FIELD_SITES, 0, c->stream>>>(
        c->g, canon, canon_rb, static_cast<const char*>(internal), internal_rb, c->field_bytes(P64));
    LQ_CUDA(cudaGetLastError());
    c->launches++;
    return LQCD_OK;
}

lqcd_status gauge_pack(lqcd_ctx* c, const double* slice, int t0, int t1)
{
    const int n = c->g.Vh / c->g.L[3] * (t1 - t0);
    const dim3 grid((n + GAUGE_SITES - 1) / GAUGE_SITES, 2);
    const int aligned = (reinterpret_cast<uintptr_t>(slice) & 15) == 0;  // links may start at any double
    GaugeOut o;
    for (int P = 0; P < 4; ++P) o.out[P] = c->holds(P) ? c->gauge[P] : nullptr;
    if (c->cfg.recon == 12) gauge_pack_kernel<12><<<grid, 4 * GAUGE_SITES, 0, c->stream>>>(c->g, slice, t0, t1, aligned, o);
    else gauge_pack_kernel<18><<<grid, 4 * GAUGE_SITES, 0, c->stream>>>(c->g, slice, t0, t1, aligned, o);
    LQ_CUDA(cudaGetLastError());
    c->launches++;
    return LQCD_OK;
}

template <int PIN>
static cudaError_t convert_out(lqcd_ctx* c, dim3 grid, int block, char* out, int Pout, size_t out_rb,
                               const char* in, size_t in_rb, int nfield, double* red, size_t red_rs)
{
    double* part = red ? c->partials : nullptr;
#define LQ_C(PO) convert_kernel<PIN, PO><<<grid, block, 0, c->stream>>>(c->g, out, out_rb, in, in_rb, nfield, part, c->part_rs, c->tickets, red, red_rs)
    switch (Pout) {
    case P64: LQ_C(P64); break;
    case P32: LQ_C(P32); break;
    case P16: LQ_C(P16); break;
    default: LQ_C(PB16); break;
    }
#undef LQ_C
    return cudaGetLastError();
}

// Convert nrhs fields (nf = 1: one parity, nf = 2: full) between precisions;
// with norm_slot >= 0 also write |in|^2 (FP64) to scal[rhs][norm_slot].
lqcd_status convert_field(lqcd_ctx* c, void* out, int Pout, const void* in, int Pin, int nrhs, size_t out_rb,
                          size_t in_rb, int nf, int norm_slot)
{
    const int block = 256;
    int nb = (c->g.Vh + block - 1) / block;
    if (nb > 4 * 152) nb = 4 * 152;
    dim3 grid(nb, nrhs);
    char* o = static_cast<char*>(out);
    const char* i = static_cast<const char*>(in);
    double* red = norm_slot >= 0 ? c->scal + norm_slot : nullptr;
    cudaError_t e;
    switch (Pin) {
    case P64: e = convert_out<P64>(c, grid, block, o, Pout, out_rb, i, in_rb, nf, red, SC_PER_RHS); break;
    case P32: e = convert_out<P32>(c, grid, block, o, Pout, out_rb, i, in_rb, nf, red, SC_PER_RHS); break;
    case P16: e = convert_out<P16>(c, grid, block, o, Pout, out_rb, i, in_rb, nf, red, SC_PER_RHS); break;
    default: e = convert_out<PB16>(c, grid, block, o, Pout, out_rb, i, in_rb, nf, red, SC_PER_RHS); break;
    }
    LQ_CUDA(e);
    c->launches++;
    return LQCD_OK;
}

}  // namespace lqcd
