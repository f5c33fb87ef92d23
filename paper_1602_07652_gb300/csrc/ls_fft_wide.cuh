// ls_fft_wide.cuh -- the LS-apply's three passes (Sec. 2) for 16-byte complex values: FP64
// (double2) and double-float (cdp: packed FP32x2 components), specialised on P = 2^LP.
//
// Both are bound by arithmetic -- FP64 by its pipe (about 1/64 of the FP32 rate), double-float
// by FP32 issue slots (a complex sum is 11 packed instructions, a product 19) -- so the
// transforms leave out what a zero-padded convolution does not need: the first forward stage
// sees only its lower 4 of 8 inputs (x, z < n <= P/2) and the last inverse stage computes only
// those outputs, a third and a sixth of a stage's additions.  Everything a transform does is
// fixed at compile time: Stockham stages of radix 8 (the last forward / first inverse stage
// takes the remaining radix), a thread owning one transform's 8 elements per stage in 32
// registers, so that 1024 threads share an SM (64 registers; the column pass of P = 4096 then
// spills 172 bytes in double-float and 88 in FP64, the others at most 72); every twiddle is a
// table load.  The generic passes these replace had a run-time plan, 2-column tiles at 128 registers (512 threads an SM) and no
// pruning.  One column per transform touches 16 bytes of a row, half a sector; the other half
// is the next column's and comes from L2, and the passes are far from the memory bound.
// The passes are launched programmatically, each starting its successor when only its
// stores are left.
// Double-float: 2048^2 1129 -> 971 us, 512^2 75 -> 58, 100^2 41 -> 21, and 2048^2 -> 759 with
// packed components and twiddles stage by stage (FMA pipe 60 to 74 per cent busy); FP64: 2048^2
// 4158 -> 3634 us, 1024^2 917 -> 852 (FP64 pipe 86 per cent busy), 100^2 53 -> 34.
#pragma once

#include "ls_fft_common.cuh"
#include "ls_dfloat.cuh"

namespace {

template <int LP>
struct GeoW {
    static constexpr int P = 1 << LP, E = 8, T = P / E;    // threads per transform
    static constexpr int THREADS = T >= 128 ? T : 128, G = THREADS / T;
    static constexpr int NS = (LP + 2) / 3, LRL = LP - 3 * (NS - 1);   // stages, log2 of the last radix
    static constexpr int SLOTS = P + P / 8;                // a padding slot every 8 elements
    static constexpr int MINB = (LRL == 1 ? 768 : 1024) / THREADS;   // (a last radix of 2 needs 80 registers)
    static constexpr size_t smem = (size_t)G * SLOTS * 16;
};
__device__ __forceinline__ int pad8(int i) { return i + (i >> 3); }

// Twiddles stage by stage, exp(-2 pi i k r / 2^(LS+LR)) at [offset of the stage][r - 1][k], the
// forward stages in the first P entries and the inverse ones in the next P: a warp's factors
// are consecutive.  In the one table exp(-2 pi i m / P) they lie up to a line apart, and a
// load took up to 32 wavefronts of the LSU (half of the double-float column pass's).
constexpr int wide_tw_off(bool inverse, int lrl, int S) {   // offset of stage S >= 1
    int o = 0;
    for (int s = 1; s < S; ++s) o += 7 << (inverse ? lrl + 3 * (s - 1) : 3 * s);
    return o;
}

// One stage: v[e R + r] *= exp(-DIR 2 pi i k r / 2^(LS+LR)), then the DFTs; tw: the stage's factors
template <int LR, int LS, int DIR, int LP, bool HZ, typename C, typename W>
__device__ __forceinline__ void stage_w(C (&v)[8], int j, const W* __restrict__ tw) {
    constexpr int R = 1 << LR, T = GeoW<LP>::T;
#pragma unroll
    for (int e = 0; e < 8 / R; ++e) {
        if constexpr (LS > 0) {
            const int k = (j + e * T) & ((1 << LS) - 1);
#pragma unroll
            for (int r = 1; r < R; ++r) {
                W w = ldg_c(&tw[((r - 1) << LS) + k]);
                if (DIR < 0) w.y = -w.y;
                v[e * R + r] = v[e * R + r] * w;
            }
        }
        dft_reg<R, DIR, HZ>(&v[e * R]);
    }
}

// outputs of a stage (radix 2^LR, Ns = 2^LS) -> inputs of the next (radix 2^LRN)
template <int LR, int LS, int LRN, int LP, bool FIRST, typename C>
__device__ __forceinline__ void exchange_w(C (&v)[8], C* buf, int j) {
    constexpr int R = 1 << LR, RN = 1 << LRN, T = GeoW<LP>::T, P = GeoW<LP>::P;
    if (!FIRST) __syncthreads();
#pragma unroll
    for (int e = 0; e < 8 / R; ++e) {
        const int b = j + e * T;
        const int base = ((b >> LS) << (LS + LR)) + (b & ((1 << LS) - 1));
#pragma unroll
        for (int r = 0; r < R; ++r) buf[pad8(base + (r << LS))] = v[e * R + r];
    }
    __syncthreads();
#pragma unroll
    for (int e = 0; e < 8 / RN; ++e)
#pragma unroll
        for (int r = 0; r < RN; ++r) v[e * RN + r] = buf[pad8(j + e * T + r * (P / RN))];
}

// Forward: in v[t] = x[j + t T] (t < 4; the rest is zero), out v[e R + r] = X[j + e T + r P/R], R = 2^LRL
template <int LP, int S, bool FIRST, typename C, typename W>
__device__ __forceinline__ void fwd_w(C (&v)[8], C* buf, int j, const W* __restrict__ tw) {
    using Gm = GeoW<LP>;
    constexpr int LR = S < Gm::NS - 1 ? 3 : Gm::LRL;
    if constexpr (S > 0) exchange_w<3, 3 * (S - 1), LR, LP, FIRST && S == 1>(v, buf, j);
    stage_w<LR, 3 * S, +1, LP, S == 0>(v, j, tw + wide_tw_off(false, Gm::LRL, S));
    if constexpr (S + 1 < Gm::NS) fwd_w<LP, S + 1, FIRST>(v, buf, j, tw);
}
// Inverse (unnormalised): the layout fwd_w leaves -> v[t] = x[j + t T]
template <int LP, int S, bool FIRST, typename C, typename W>
__device__ __forceinline__ void inv_w(C (&v)[8], C* buf, int j, const W* __restrict__ tw) {
    using Gm = GeoW<LP>;
    constexpr int LR = S == 0 ? Gm::LRL : 3, LS = S == 0 ? 0 : Gm::LRL + 3 * (S - 1);
    if constexpr (S > 0) {
        constexpr int LRP = S == 1 ? Gm::LRL : 3, LSP = S == 1 ? 0 : Gm::LRL + 3 * (S - 2);
        exchange_w<LRP, LSP, LR, LP, FIRST && S == 1>(v, buf, j);
    }
    stage_w<LR, LS, -1, LP, false>(v, j, tw + Gm::P + wide_tw_off(true, Gm::LRL, S));
    if constexpr (S + 1 < Gm::NS) inv_w<LP, S + 1, FIRST>(v, buf, j, tw);
}

template <int LP, typename C, typename W, class Src>
__global__ void __launch_bounds__(GeoW<LP>::THREADS, GeoW<LP>::MINB) k_wide_rows_fwd(int n, Src src, C* __restrict__ X,
                                                                                 const W* __restrict__ tw) {
    using Gm = GeoW<LP>;
    constexpr int T = Gm::T, R = 1 << Gm::LRL;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int grp = threadIdx.x / T, j = threadIdx.x % T;
    C* buf = reinterpret_cast<C*>(smem_raw) + grp * Gm::SLOTS;
    const int z = blockIdx.x * Gm::G + grp;
    pdl_wait();
    C v[8];
#pragma unroll
    for (int t = 0; t < 4; ++t) {
        const int x = j + t * T;
        v[t] = (z < n && x < n) ? src.template load<C>(z, x) : czero<C>();
    }
    fwd_w<LP, 0, true>(v, buf, j, tw);
    pdl_trigger();
    if (z >= n) return;
    C* o = X + (size_t)z * Gm::P;
#pragma unroll
    for (int e = 0; e < 8 / R; ++e)
#pragma unroll
        for (int r = 0; r < R; ++r) o[j + e * T + r * (Gm::P / R)] = v[e * R + r];
}

template <int LP, typename C, typename W>
__global__ void __launch_bounds__(GeoW<LP>::THREADS, GeoW<LP>::MINB) k_wide_cols(int n, C* __restrict__ X,
                                                                             const W* __restrict__ ghat,
                                                                             const W* __restrict__ tw) {
    using Gm = GeoW<LP>;
    constexpr int P = Gm::P, T = Gm::T, R = 1 << Gm::LRL;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int grp = threadIdx.x / T, j = threadIdx.x % T;
    C* buf = reinterpret_cast<C*>(smem_raw) + grp * Gm::SLOTS;
    // columns kx and P - kx, which share a row of the quadrant, run side by side
    const int lin = blockIdx.x * Gm::G + grp;
    const int kx = (lin & 1) ? (P - 1 - (lin >> 1)) : (lin >> 1);
    C* col = X + kx;
    const W* g = ghat + (size_t)(kx <= P / 2 ? kx : P - kx) * (P / 2 + 1);
    pdl_wait();
    C v[8];
#pragma unroll
    for (int t = 0; t < 4; ++t) {
        const int z = j + t * T;
        v[t] = z < n ? col[(size_t)z * P] : czero<C>();
    }
    fwd_w<LP, 0, true>(v, buf, j, tw);
#pragma unroll
    for (int e = 0; e < 8 / R; ++e)
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int kz = j + e * T + r * (P / R);
            v[e * R + r] = v[e * R + r] * ldg_c(&g[kz <= P / 2 ? kz : P - kz]);
        }
    inv_w<LP, 0, false>(v, buf, j, tw);
    pdl_trigger();
#pragma unroll
    for (int t = 0; t < 4; ++t) {
        const int z = j + t * T;
        if (z < n) col[(size_t)z * P] = v[t];
    }
}

template <int LP, typename C, typename W, class Dst>
__global__ void __launch_bounds__(GeoW<LP>::THREADS, GeoW<LP>::MINB) k_wide_rows_inv(int n, const C* X, Dst dst,
                                                                                 const W* __restrict__ tw) {
    using Gm = GeoW<LP>;
    constexpr int T = Gm::T, R = 1 << Gm::LRL;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int grp = threadIdx.x / T, j = threadIdx.x % T;
    C* buf = reinterpret_cast<C*>(smem_raw) + grp * Gm::SLOTS;
    const int z = blockIdx.x * Gm::G + grp;
    pdl_wait();
    C v[8];
    const C* xr = X + (size_t)(z < n ? z : 0) * Gm::P;
#pragma unroll
    for (int e = 0; e < 8 / R; ++e)
#pragma unroll
        for (int r = 0; r < R; ++r) v[e * R + r] = xr[j + e * T + r * (Gm::P / R)];
    inv_w<LP, 0, true>(v, buf, j, tw);
    pdl_trigger();
    if (z >= n) return;
#pragma unroll
    for (int t = 0; t < 4; ++t) {
        const int x = j + t * T;
        if (x < n) dst.template store<C>(z, x, v[t]);
    }
}

template <int LP, typename C, typename W, class Src, class Dst>
int wide_lp(ls_handle* h, const Src& src, const Dst& dst, const W* ghat, const W* tw) {
    using Gm = GeoW<LP>;
    const int n = h->n;
    C* X = static_cast<C*>(h->fftws);
    const dim3 rows((unsigned)((n + Gm::G - 1) / Gm::G)), threads(Gm::THREADS);
    LS_TRY(ls_launch_pdl(h, k_wide_rows_fwd<LP, C, W, Src>, rows, threads, Gm::smem, n, src, X, tw));
    LS_TRY(ls_launch_pdl(h, k_wide_cols<LP, C, W>, dim3(Gm::P / Gm::G), threads, Gm::smem, n, X, ghat, tw));
    return ls_launch_pdl(h, k_wide_rows_inv<LP, C, W, Dst>, rows, threads, Gm::smem, n, static_cast<const C*>(X), dst, tw);
}

template <typename C, typename W, class Src, class Dst>
int wide_apply(ls_handle* h, const Src& src, const Dst& dst, const W* ghat, const W* tw) {
    switch (h->lp) {
        case 6: return wide_lp<6, C>(h, src, dst, ghat, tw);
        case 7: return wide_lp<7, C>(h, src, dst, ghat, tw);
        case 8: return wide_lp<8, C>(h, src, dst, ghat, tw);
        case 9: return wide_lp<9, C>(h, src, dst, ghat, tw);
        case 10: return wide_lp<10, C>(h, src, dst, ghat, tw);
        case 11: return wide_lp<11, C>(h, src, dst, ghat, tw);
        case 12: return wide_lp<12, C>(h, src, dst, ghat, tw);
        default: return LS_EINVAL;
    }
}

// dynamic shared memory above 48 KB (P = 4096 only)
template <typename C, typename W, class Src, class Dst>
int wide_optin() {
    using Gm = GeoW<12>;
    static_assert(GeoW<11>::smem <= 48 * 1024, "only P = 4096 needs the opt-in");
    LS_CUDA(cudaFuncSetAttribute(k_wide_rows_fwd<12, C, W, Src>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Gm::smem));
    LS_CUDA(cudaFuncSetAttribute(k_wide_cols<12, C, W>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Gm::smem));
    LS_CUDA(cudaFuncSetAttribute(k_wide_rows_inv<12, C, W, Dst>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Gm::smem));
    return LS_OK;
}

}  // namespace
