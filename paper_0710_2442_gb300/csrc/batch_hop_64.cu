// batch_hop_64.cu -- the batched FP64 hopping term (corrections, prologue and
// epilogue of the loop problems) in block fixed point, tile by tile.
#include "batch_impl.cuh"
#include "dslash_fx.cuh"

namespace wl {
namespace bt {

// A block of four warps works through its tile 32 sites at a time (fx_tile, the small-lattice
// kernel's work).  The FP64 stencil it replaces took 128 us for a 16^3 x 32
// problem's hop on its FP64 arithmetic, and a correction waits for two of them; F16 batch of
// 8 x 8^4, 4 x 12^4 and 2 x 16^3 x 32 problems 23.4 -> 19.6 ms.  One block a
// tile, without a loop over tiles: the call to fx_redo costs a loop around it spills (the hop 86 -> 123 us).
__global__ void __launch_bounds__(128, 4) bhop_fx_kernel(const BatchArgs A, const BOp op) {
    __shared__ FxTile T;
    __shared__ FxParams P;
    __shared__ unsigned redo[16];  // of the tile's groups (at most 512 sites)
    const int t = blockIdx.x;
    const int pid = __ldg(A.tile_prob + t);
    if (!tile_active(A, op, pid)) return;
    const BatchProb& Pr = A.probs[pid];
    const int p = op.out_parity;
    char* out = Pr.f[op.f_out] + p * Pr.fp[op.f_out];
    const char* x = op.f_x >= 0 ? Pr.f[op.f_x] + p * Pr.fp[op.f_x] : nullptr;
    const int vh = Pr.g.Vh, stride = Pr.g.stride;
    const int h0 = (t - Pr.tile0) * A.tile, h1 = min(h0 + A.tile, vh);
    // outer is written only by the correction finisher, a later kernel
    if (op.zero_first && __ldcg(&A.state[pid].outer) == 0) {  // the hop term is zero
        for (int i = threadIdx.x; i < 12 * (h1 - h0); i += blockDim.x) {
            const long long at = (long long)(i / (h1 - h0)) * stride + h0 + i % (h1 - h0);
            reinterpret_cast<double2*>(out)[at] =
                x ? reinterpret_cast<const double2*>(x)[at] : make_double2(0.0, 0.0);
        }
        return;
    }
    if (threadIdx.x == 0) {
        const long long s = stride;
        P.out = FxField{out, 0, 0, 1, stride, 0};
        P.in = FxField{Pr.f[op.f_in] + (1 - p) * Pr.fp[op.f_in], 0, 0, 1, stride, 0};
        P.nat = P.in;
        P.x = FxField{const_cast<char*>(x), 0, 0, 1, stride, 0};
        P.u = FxLinks{Pr.g64, 36 * s, 9 * s, 1, stride, 0};
        P.un = FxLinks{Pr.canon, 0, 9, 36, 1, 1};
        P.un_recon = 18;
        P.g = Pr.g;
        P.nrhs = 1;
        P.full = 0;
        P.dag = 0;
        P.xpay = x != nullptr;
        P.a = coef_of(op.coef, Pr.kappa);
        P.scaled = !x && op.coef != 0;
    }
    __syncthreads();
    unsigned any = 0;
    double none = 0.0;
    for (int h = h0; h < h1; h += 32) {
        const unsigned m = fx_tile<true, false, 4>(P, T, p, 0, h, h1, none);
        if (threadIdx.x == 0) redo[(h - h0) >> 5] = m;
        any |= m;
        __syncthreads();
    }
    if (!any) return;
    for (int h = h0; h < h1; h += 32) fx_tile_redo<4>(P, T, p, 0, h, redo[(h - h0) >> 5]);
}

void launch_bhop_fx(const BatchArgs& A, const BOp& o, cudaStream_t st) {
    WL_REQUIRE(o.fin == BF_NONE, "the batched FP64 hop has no fused reduction");
    if (A.ntiles) bhop_fx_kernel<<<A.ntiles, 128, 0, st>>>(A, o);
}

}  // namespace bt
}  // namespace wl
