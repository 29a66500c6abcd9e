// layout.cu -- canonical complex128 fields <-> the library's SoA formats.
//
// Canonical: spinor [site][spin][colour], gauge [site][mu][row][col], complex
// as (re, im) doubles, site s = x + Lx*(y + Ly*(z + Lz*t)); half fields hold
// the sites of one parity at index s >> 1.
//
// Spinors: F64 (12 x 16 B chunks), F32 (6 x 16 B), F16/BF16 (3 x 16 B plus an
// FP32 per-site scale = the largest |component|; the stored values are
// component / scale rounded to nearest even).  Links: rows 0 and 1 only for
// 12-real storage (row 2 is rebuilt in the kernels, exact for SU(3)); links
// are never scaled (|U_ij| <= 1).
#include "fx.cuh"
#include "internal.h"

namespace wl {

Geom make_geom(const int dims[4], const double ph[4][2]) {
    Geom g;
    long long V = 1;
    for (int mu = 0; mu < 4; mu++) {
        g.L[mu] = dims[mu];
        V *= dims[mu];
        for (int z = 0; z < 2; z++) {
            g.ph[mu][z] = ph[mu][z];
            g.pf[mu][z] = (float)ph[mu][z];
        }
    }
    g.Vh = (int)(V / 2);
    g.stride = round_up(g.Vh, 64);
    for (int k = 0; k < 3; k++) div_magic(dims[k], g.dm[k], g.ds[k]);
    return g;
}

long long spinor_field_bytes(Prec p, int stride) {
    switch (p) {
        case P_F64: return SpinorFmt<P_F64>::field_bytes(stride);
        case P_F32: return SpinorFmt<P_F32>::field_bytes(stride);
        default: return SpinorFmt<P_F16>::field_bytes(stride);
    }
}

long long gauge_block_bytes(Prec p, int recon, int stride) {
    int per_link = (p == P_F64 ? 8 : p == P_F32 ? 4 : 2) * recon;
    return (long long)per_link * stride;
}

long long gauge_bytes(Prec p, int recon, int stride) { return 8 * gauge_block_bytes(p, recon, stride); }

void SpinorField::alloc(Prec p, int sub, int nr, const Geom& geom) {
    prec = p;
    subset = sub;
    nrhs = nr;
    g = geom;
    pbytes = (spinor_field_bytes(p, g.stride) + 255) / 256 * 256;
    buf.alloc((size_t)pbytes * nparity() * nrhs);
}

void SpinorField::alloc_fx(int sub, int nr, const Geom& geom, int fields) {
    prec = P_F64;
    subset = sub;
    nrhs = nr;
    g = geom;
    pbytes = fx_spinor_bytes(g.stride) * fields;
    buf.alloc((size_t)pbytes * nparity() * nrhs);
}

// ---------------------------------------------------------------------------
// spinors
// ---------------------------------------------------------------------------
// Parity of the site with canonical index s.
__device__ __forceinline__ int site_parity(int s, const Geom& g) {
    const int r = div_by(s, g, 0), r2 = div_by(r, g, 1), t = div_by(r2, g, 2);
    return ((s - r * g.L[0]) + (r - r2 * g.L[1]) + (r2 - t * g.L[2]) + t) & 1;
}

// Canonical <-> SoA over all right-hand sides in one launch: blockIdx.y is the
// right-hand side.  Both are bound by their bytes; one launch of 21 us per
// right-hand side reached 4.5 TB/s on 24^3 x 48 F32 and, on 16^3 x 32 BF16, spent 12 x 7.4 us on
// what the bytes allow in 37.  They are launched like the hops (launch_dep).  A launch bound of 256
// threads on the import made it 4 us slower on 32^3 x 64 F32 (50 to 54 us).
template <int SP>
__global__ void pack_spinor_kernel(const double2* __restrict__ canon, char* base,
                                                          long long pbytes, long long rstep, int subset, Geom g) {
    using SF = SpinorFmt<SP>;
    using T = typename SF::real;
    pdl_wait();
    const int n = subset == 2 ? 2 * g.Vh : g.Vh;
    canon += (long long)blockIdx.y * n * 12;
    base += blockIdx.y * rstep;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const int p = subset == 2 ? site_parity((int)i, g) : 0;
        const int h = (int)(subset == 2 ? i >> 1 : i);
        cpx<T> v[12];
        const double2* src = canon + i * 12;
#pragma unroll
        for (int k = 0; k < 12; k++) {
            double2 d = __ldg(src + k);
            v[k] = {(T)d.x, (T)d.y};
        }
        SF::store(base + (subset == 2 ? p * pbytes : 0), g.stride, h, v);
    }
    pdl_trigger();
}

// Each block converts its sites into shared memory and then writes their
// canonical 192 bytes as one contiguous run (consecutive threads, consecutive
// 16-byte words), instead of 12 strided stores per thread.
constexpr int kUnpackBlock = 128;

template <int SP>
__global__ void __launch_bounds__(kUnpackBlock) unpack_spinor_kernel(double2* __restrict__ canon, const char* base,
                                                                     long long pbytes, long long rstep, int subset,
                                                                     Geom g) {
    using SF = SpinorFmt<SP>;
    using T = typename SF::real;
    __shared__ double2 stage[kUnpackBlock * 12];
    pdl_wait();
    const int n = subset == 2 ? 2 * g.Vh : g.Vh;
    canon += (long long)blockIdx.y * n * 12;
    base += blockIdx.y * rstep;
    // block-uniform trip count: every thread reaches both barriers
    for (long long i0 = (long long)blockIdx.x * kUnpackBlock; i0 < n; i0 += (long long)gridDim.x * kUnpackBlock) {
        const long long i = i0 + threadIdx.x;
        if (i < n) {
            const int p = subset == 2 ? site_parity((int)i, g) : 0;
            const int h = (int)(subset == 2 ? i >> 1 : i);
            cpx<T> v[12];
            SF::load(base + (subset == 2 ? p * pbytes : 0), g.stride, h, v);
#pragma unroll
            for (int k = 0; k < 12; k++) stage[threadIdx.x * 12 + k] = make_double2((double)v[k].re, (double)v[k].im);
        }
        __syncthreads();
        const int words = (int)(n - i0 < kUnpackBlock ? n - i0 : kUnpackBlock) * 12;
        double2* dst = canon + i0 * 12;
        for (int e = threadIdx.x; e < words; e += kUnpackBlock) dst[e] = stage[e];
        __syncthreads();
    }
    pdl_trigger();
}

static int grid_for(long long n, int block) {
    long long b = (n + block - 1) / block;
    long long cap = 64LL * device_sm_count();
    if (b > cap) b = cap;
    return (int)(b < 1 ? 1 : b);
}

// n_rhs consecutive right-hand sides from `rhs` on; canon: theirs, back to back.
void pack_spinor(const SpinorField& f, int rhs, int n_rhs, const double* canon, cudaStream_t st) {
    const dim3 block(256), grid(grid_for(f.subset == 2 ? 2LL * f.g.Vh : (long long)f.g.Vh, 256), n_rhs);
    char* base = static_cast<char*>(f.block(f.subset == 2 ? 0 : f.subset, rhs));
    const double2* src = reinterpret_cast<const double2*>(canon);
    switch (f.prec) {
        case P_F64: launch_dep(pack_spinor_kernel<P_F64>, grid, block, st, src, base, f.pbytes, f.rstep(), f.subset, f.g); break;
        case P_F32: launch_dep(pack_spinor_kernel<P_F32>, grid, block, st, src, base, f.pbytes, f.rstep(), f.subset, f.g); break;
        case P_F16: launch_dep(pack_spinor_kernel<P_F16>, grid, block, st, src, base, f.pbytes, f.rstep(), f.subset, f.g); break;
        case P_BF16: launch_dep(pack_spinor_kernel<P_BF16>, grid, block, st, src, base, f.pbytes, f.rstep(), f.subset, f.g); break;
    }
}

void unpack_spinor(const SpinorField& f, int rhs, int n_rhs, double* canon, cudaStream_t st) {
    const dim3 block(kUnpackBlock), grid(grid_for(f.subset == 2 ? 2LL * f.g.Vh : (long long)f.g.Vh, kUnpackBlock), n_rhs);
    const char* base = static_cast<const char*>(f.block(f.subset == 2 ? 0 : f.subset, rhs));
    double2* dst = reinterpret_cast<double2*>(canon);
    switch (f.prec) {
        case P_F64: launch_dep(unpack_spinor_kernel<P_F64>, grid, block, st, dst, base, f.pbytes, f.rstep(), f.subset, f.g); break;
        case P_F32: launch_dep(unpack_spinor_kernel<P_F32>, grid, block, st, dst, base, f.pbytes, f.rstep(), f.subset, f.g); break;
        case P_F16: launch_dep(unpack_spinor_kernel<P_F16>, grid, block, st, dst, base, f.pbytes, f.rstep(), f.subset, f.g); break;
        case P_BF16: launch_dep(unpack_spinor_kernel<P_BF16>, grid, block, st, dst, base, f.pbytes, f.rstep(), f.subset, f.g); break;
    }
}

// ---------------------------------------------------------------------------
// links
// ---------------------------------------------------------------------------
template <int GP, int R>
__device__ __forceinline__ void store_link(char* base, int stride, int blk, int i, const double2 u[9]) {
    if (GP == P_F64) {
        double2* b = reinterpret_cast<double2*>(base) + (size_t)blk * (R / 2) * stride + i;
#pragma unroll
        for (int c = 0; c < R / 2; c++) b[(size_t)c * stride] = u[c];
    } else if (GP == P_F32 && R == 18) {
        float2* b = reinterpret_cast<float2*>(base) + (size_t)blk * 9 * stride + i;
#pragma unroll
        for (int c = 0; c < 9; c++) b[(size_t)c * stride] = make_float2((float)u[c].x, (float)u[c].y);
    } else if (GP == P_F32 && R == 12) {
        float4* b = reinterpret_cast<float4*>(base) + (size_t)blk * 3 * stride + i;
#pragma unroll
        for (int c = 0; c < 3; c++)
            b[(size_t)c * stride] = make_float4((float)u[2 * c].x, (float)u[2 * c].y, (float)u[2 * c + 1].x,
                                                (float)u[2 * c + 1].y);
    } else if (R == 18) {  // F16 / BF16, 18 reals: rows of 16, 16 and 4 bytes
        using LT = LowT<GP == P_F16 ? P_F16 : P_BF16>;
        char* b = base + (size_t)blk * 36 * stride;
        unsigned int w[9];
#pragma unroll
        for (int k = 0; k < 9; k++) w[k] = LT::from_f2((float)u[k].x, (float)u[k].y);
        reinterpret_cast<uint4*>(b)[i] = make_uint4(w[0], w[1], w[2], w[3]);
        reinterpret_cast<uint4*>(b + 16LL * stride)[i] = make_uint4(w[4], w[5], w[6], w[7]);
        reinterpret_cast<unsigned int*>(b + 32LL * stride)[i] = w[8];
    } else {  // F16 / BF16, 12 reals
        using LT = LowT<GP == P_F16 ? P_F16 : P_BF16>;
        uint2* b = reinterpret_cast<uint2*>(base) + (size_t)blk * 3 * stride + i;
#pragma unroll
        for (int c = 0; c < 3; c++) {
            uint2 d;
            d.x = LT::from_f2((float)u[2 * c].x, (float)u[2 * c].y);
            d.y = LT::from_f2((float)u[2 * c + 1].x, (float)u[2 * c + 1].y);
            b[(size_t)c * stride] = d;
        }
    }
}

template <int GP, int R>
__global__ void pack_gauge_kernel(const double2* __restrict__ canon, char* base, Geom g) {
    const long long V = 2LL * g.Vh;
    for (long long s = blockIdx.x * (long long)blockDim.x + threadIdx.x; s < V; s += (long long)gridDim.x * blockDim.x) {
        const int p = site_parity((int)s, g);
        const int h = (int)(s >> 1);
#pragma unroll
        for (int mu = 0; mu < 4; mu++) {
            double2 u[9];
            const double2* src = canon + (s * 4 + mu) * 9;
#pragma unroll
            for (int k = 0; k < 9; k++) u[k] = src[k];
            store_link<GP, R>(base, g.stride, p * 4 + mu, h, u);
        }
    }
}

// F64 links in fixed point (fx.cuh): nine words per link whatever R, the third row
// rebuilt for R = 12; a link out of range is marked, and with COUNT counted.  DBL: the doubles too.  (The counter's ten
// registers in a stateless call's pack would leave three blocks an SM: M on 16^3 x 32 98 -> 103 us.)
template <int R, bool DBL, bool COUNT>
__global__ void pack_gauge_fx_kernel(const double2* __restrict__ canon, char* base, uint4* fx, Geom g,
                                     unsigned long long* bad) {
    const long long V = 2LL * g.Vh;
    unsigned misfits = 0;
    for (long long s = blockIdx.x * (long long)blockDim.x + threadIdx.x; s < V; s += (long long)gridDim.x * blockDim.x) {
        const int p = site_parity((int)s, g);
        const int h = (int)(s >> 1);
#pragma unroll
        for (int mu = 0; mu < 4; mu++) {
            double2 u[9];
            const double2* src = canon + (s * 4 + mu) * 9;
#pragma unroll
            for (int k = 0; k < R / 2; k++) u[k] = src[k];
            if (DBL) store_link<P_F64, R>(base, g.stride, p * 4 + mu, h, u);
            FxCplx f[3][3];
            unsigned mx = 0;
#pragma unroll
            for (int k = 0; k < R / 2; k++) {
                const unsigned rh = (unsigned)__double2hiint(u[k].x), ih = (unsigned)__double2hiint(u[k].y);
                mx = max(mx, max(rh << 1, ih << 1));
                f[k / 3][k % 3] = FxCplx{fx_link(rh, (unsigned)__double2loint(u[k].x)),
                                         fx_link(ih, (unsigned)__double2loint(u[k].y))};
            }
            bool fits = mx <= kFxLinkHi;
            if (R == 12) {
                fx_recon_row2(f);  // a third row of rows that are no SU(3) ones can be larger
#pragma unroll
                for (int k = 0; k < 3; k++) fits = fits && fx_limb_fits(f[2][k].re.h) && fx_limb_fits(f[2][k].im.h);
            }
            if (!fits) f[0][0].re.h = (int)kFxBadLink;
            if (COUNT) misfits += !fits;
            uint4* b = fx + (size_t)(p * 4 + mu) * 9 * g.stride + h;
#pragma unroll
            for (int k = 0; k < 9; k++) {
                const FxCplx& z = f[k / 3][k % 3];
                b[(size_t)k * g.stride] =
                    make_uint4((unsigned)z.re.h, (unsigned)z.re.l, (unsigned)z.im.h, (unsigned)z.im.l);
            }
        }
    }
    if (COUNT) {
        misfits = __reduce_add_sync(0xffffffffu, misfits);
        if (misfits && (threadIdx.x & 31) == 0) atomicAdd(bad, (unsigned long long)misfits);
    }
}

bool pack_gauge_fx(GaugeField& gf, const double* canon, cudaStream_t st) {
    DevBuf bad(sizeof(unsigned long long));
    WL_CUDA(cudaMemsetAsync(bad.p, 0, bad.bytes, st));
    pack_gauge(gf, canon, st, bad.as<unsigned long long>());
    unsigned long long n = 0;
    WL_CUDA(cudaMemcpyAsync(&n, bad.p, sizeof(n), cudaMemcpyDeviceToHost, st));
    WL_CUDA(cudaStreamSynchronize(st));
    return n * 12 <= 8ULL * gf.g.Vh;
}

void pack_gauge(GaugeField& gf, const double* canon, cudaStream_t st, unsigned long long* bad) {
    const long long V = 2LL * gf.g.Vh;
    const int block = 256, grid = grid_for(V, block);
    const double2* src = reinterpret_cast<const double2*>(canon);
    char* base = gf.buf.as<char>();
    const Prec p = gf.prec;
    const int R = gf.recon;
    if (p == P_F64 && gf.fx.p) {
        uint4* fx = gf.fx.as<uint4>();
        auto pack = [&](auto RR, auto DBL) {
            constexpr int r = decltype(RR)::value;
            constexpr bool d = decltype(DBL)::value;
            if (bad) pack_gauge_fx_kernel<r, d, true><<<grid, block, 0, st>>>(src, base, fx, gf.g, bad);
            else pack_gauge_fx_kernel<r, d, false><<<grid, block, 0, st>>>(src, base, fx, gf.g, bad);
        };
        using std::bool_constant;
        using std::integral_constant;
        if (R == 18 && base) pack(integral_constant<int, 18>{}, bool_constant<true>{});
        else if (R == 18) pack(integral_constant<int, 18>{}, bool_constant<false>{});
        else if (base) pack(integral_constant<int, 12>{}, bool_constant<true>{});
        else pack(integral_constant<int, 12>{}, bool_constant<false>{});
        WL_LAUNCH_CHECK();
        return;
    }
    if (p == P_F64 && R == 18) pack_gauge_kernel<P_F64, 18><<<grid, block, 0, st>>>(src, base, gf.g);
    else if (p == P_F64 && R == 12) pack_gauge_kernel<P_F64, 12><<<grid, block, 0, st>>>(src, base, gf.g);
    else if (p == P_F32 && R == 18) pack_gauge_kernel<P_F32, 18><<<grid, block, 0, st>>>(src, base, gf.g);
    else if (p == P_F32 && R == 12) pack_gauge_kernel<P_F32, 12><<<grid, block, 0, st>>>(src, base, gf.g);
    else if (p == P_F16 && R == 12) pack_gauge_kernel<P_F16, 12><<<grid, block, 0, st>>>(src, base, gf.g);
    else if (p == P_BF16 && R == 12) pack_gauge_kernel<P_BF16, 12><<<grid, block, 0, st>>>(src, base, gf.g);
    else if (p == P_F16 && R == 18) pack_gauge_kernel<P_F16, 18><<<grid, block, 0, st>>>(src, base, gf.g);
    else if (p == P_BF16 && R == 18) pack_gauge_kernel<P_BF16, 18><<<grid, block, 0, st>>>(src, base, gf.g);
    else throw Error(7, "unsupported link precision / storage");
    WL_LAUNCH_CHECK();
}

}  // namespace wl
