// dslash_fx.cu -- launches of the FP64 hopping term on the integer pipe
// (dslash_fx.cuh).
#include <algorithm>

#include "dslash_fx.cuh"

namespace wl {

namespace {

constexpr int kSiteThreads = 128;  // of hop_kernel_fx1: two per site
constexpr int kSiteBlocks = 4;     // per SM
constexpr int kSplitBlocks = 4;

FxField soa(const void* p, long long pstep, long long rstep, int stride) {
    return FxField{static_cast<char*>(const_cast<void*>(p)), pstep, rstep, 1, stride, 0};
}
// A canonical field: half fields by half-site index, full ones by site.
FxField canonical(const void* p, int full) {
    return FxField{static_cast<char*>(const_cast<void*>(p)), 0, 0, 12, 1, full};
}

template <bool OUTFX, bool RED>
void launch_site(const FxParams& P, int blocks, int ny, cudaStream_t st) {
    auto k = hop_kernel_fx1<OUTFX, RED, kSiteThreads, kSiteBlocks>;
    // and the turns' masks of sites to be done over (a field of more turns than fit does not fit the device's memory)
    const int turns = RED ? (int)((P.g.Vh + (long long)blocks * (kSiteThreads / 2) - 1) / ((long long)blocks * (kSiteThreads / 2))) : 0;
    const int smem = (int)sizeof(FxSlots<kSiteThreads>) + turns * (kSiteThreads / 32) * (int)sizeof(unsigned short);
    WL_REQUIRE(smem <= 48 * 1024, "too few blocks for a reducing hop of this lattice");
    launch_dep_smem(k, dim3(blocks * P.nrhs, ny), dim3(kSiteThreads), smem, st, P);
}

template <bool FXL, bool RED>
void launch_split(const FxParams& P, int tiles, int ny, cudaStream_t st) {
    // up to one tile per SM, eight warps a tile are faster (8^4 with the Python call of then: 8.2
    // against 10.3 us); beyond, four (16^3 x 32: 43 against 48 us)
    if (tiles * ny * P.nrhs <= device_sm_count())
        launch_dep(hop_kernel_fx<FXL, RED, 8, 2>, dim3(tiles * P.nrhs, ny), dim3(256), st, P);
    else launch_dep(hop_kernel_fx<FXL, RED, 4, kSplitBlocks>, dim3(tiles * P.nrhs, ny), dim3(128), st, P);
}

}  // namespace

long long fx_spinor_bytes(int stride) { return (fx_field_bytes(stride) + 255) / 256 * 256; }

bool fx_site_kernel(const Geom& g, int nrhs, int full) {
    return (long long)g.Vh * std::max(nrhs, 1) * (full ? 2 : 1) >= kFxSiteMin;
}

int launch_hop_fx(const HopLaunch& L, cudaStream_t st) {
    const GaugeField& gf = *L.gauge;
    const Geom& g = gf.g;
    const int nrhs = L.nrhs > 1 ? L.nrhs : 1, ny = L.full ? 2 : 1;
    const long long s = g.stride;
    WL_REQUIRE(!L.xpay || L.x, "xpay needs a field");
    WL_REQUIRE(!L.red || !L.full, "reducing hop launches are single-parity");
    FxParams P;
    WL_REQUIRE(!L.canon || nrhs == 1, "canonical fields: one right-hand side");
    P.out = L.canon & kCanonOut ? canonical(L.out, L.full) : soa(L.out, L.full ? L.out_pstep : 0, L.out_rstep, g.stride);
    P.in = L.canon & kCanonIn ? canonical(L.in, L.full) : soa(L.in, L.full ? L.in_pstep : 0, L.in_rstep, g.stride);
    P.nat = P.in;
    P.x = L.canon & kCanonX ? canonical(L.x, L.full) : soa(L.x, L.full ? L.x_pstep : 0, L.x_rstep, g.stride);
    P.u = FxLinks{gf.fx.as<const char>(), 36 * s, 9 * s, 1, g.stride, 0};
    P.un_recon = gf.recon;
    if (gf.canon) {
        P.un = FxLinks{reinterpret_cast<const char*>(gf.canon), 0, 9, 36, 1, 1};
        if (!gf.fx.p) P.u = P.un;
    } else {
        const long long w = gf.recon / 2 * s;
        P.un = FxLinks{gf.buf.as<const char>(), 4 * w, w, 1, g.stride, 0};
    }
    P.g = g;
    P.nrhs = nrhs;
    P.skip_stride = L.skip_stride;
    P.out_parity = L.out_parity;
    P.full = L.full;
    P.xpay = L.xpay;
    P.dag = L.dagger != 0;
    P.a = L.a;
    P.scaled = !L.xpay && L.a != 1.0;
    P.red = L.red ? *L.red : RedArgs{};
    P.skip = L.skip;
    const bool site = gf.fx.p && (L.fx_in || (L.fx_tmp && fx_site_kernel(g, nrhs, L.full)));
    WL_REQUIRE(site || !L.fx_out, "a fixed-point output needs the site kernel");
    const int sites = site ? kSiteThreads / 2 : 32;
    int cap = 0;
    if (L.red) cap = std::min(L.grid_cap, device_sm_count() * (site ? kSiteBlocks : kSplitBlocks));
    const int blocks = hop_grid_blocks(g, sites, cap);
    WL_REQUIRE(!L.red || blocks <= L.red->slot_cap, "reduction capacity below the grid size");
    if (!site) {
        if (!gf.fx.p) {
            WL_REQUIRE(gf.recon == 18 && !L.red, "links as doubles: 18 reals, no reduction");
            launch_split<false, false>(P, blocks, ny, st);
        } else if (L.red) {
            launch_split<true, true>(P, blocks, ny, st);
        } else {
            launch_split<true, false>(P, blocks, ny, st);
        }
        return blocks;
    }
    if (L.fx_in) {
        P.in = soa(L.fx_in, L.full ? L.fx_pstep : 0, L.fx_rstep, g.stride);
        P.nat.p = nullptr;  // the hop that wrote it left the sites out of range as doubles
    } else {
        launch_dep(fx_pack_kernel, dim3((g.Vh + 127) / 128 * nrhs, ny), dim3(128), st, P.in,
                   static_cast<char*>(L.fx_tmp), L.fx_pstep, L.fx_rstep, nrhs, 0, ny, g, L.skip, L.skip_stride);
        P.in = soa(L.fx_tmp, L.full ? L.fx_pstep : 0, L.fx_rstep, g.stride);
    }
    if (L.fx_out) {
        WL_REQUIRE(!L.red && !L.xpay && L.a == 1.0, "a fixed-point output is the plain hop");
        launch_site<true, false>(P, blocks, ny, st);
    } else if (L.red) {
        launch_site<false, true>(P, blocks, ny, st);
    } else {
        launch_site<false, false>(P, blocks, ny, st);
    }
    return blocks;
}

}  // namespace wl
