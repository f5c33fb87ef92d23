// ls_sweep.cu -- local solves, trace injection, Algorithms 1 and 2 (Sec. 3.4-3.5).
//
// Strip data layout: the extended layer l of a direction is stored block by
// block along the long axis: element (r, i) (local row r, column i) at i*q + r,
// so one column of the strip -- one block of the block-tridiagonal C^l -- is q
// contiguous values.  Every strip keeps its right-hand side and its solution, so
// the traces a neighbour needs (two rows next to the interface) are read in place.
//
// Algorithm 1 (Gauss-Seidel preconditioner), with the index reading of the
// oracle (layers l = 0..L-1 from small z up; local row "1" = r = E, row "n^l" =
// r = E + t - 1):
//   downward, l = L-1..0:  g^l = chi g;  if l < L-1:
//        g^l[n]   -= C^l_{n,n+1} w^{l+1}_1,   g^l[n+1] += C^l_{n+1,n} w^{l+1}_0   (eq. pde_GRF_down)
//        w^l = (C^l)^{-1} g^l
//   upward, l = 1..L-1 (keeping g^l), with the up-going traces of the layer below:
//        g^l[1] -= C^l_{1,0} (v^{l-1}_n - w^l_0),  g^l[0] += C^l_{0,1} v^{l-1}_{n+1};  v^l = (C^l)^{-1} g^l
//   (the top injection of layer l-1 reproduces the down-going wave in its row n but
//   cancels it in its extension row n+1; w^l_0, the continuation of layer l's own
//   down-sweep solution below it, is that wave, so the injected pair is the
//   up-going field in both rows.  v^0 = w^0: layer 0 receives nothing upward.)
//   v = rows 1..n of every v^l.
// Algorithm 2: u1 = Alg. 1 on horizontal layers; e = g - C u1; u2 = Alg. 1 on
// vertical layers (the transposed grid); v = u1 + u2.
//
// Local solve (C^l)^{-1} b by the block cyclic reduction factors of ls_factor.cu:
//   forward  level 0:  y_j = D_j^{-1} b_j (odd j);  b_j -= W_j y_{j-1} + E_j y_{j+1} (even j)
//            level k:  b_j -= F_j b_{j-1} + G_j b_{j+1} (even j of level k),  y_j = D_j^{-1} b_j (odd j)
//   level c: x = S_c^{-1} b (the reduced system's precomputed inverse)
//   backward level k:  x_j = y_j - P_j x_{j-1} - Q_j x_{j+1} (odd j)
//            level 0:  x_j = y_j - D_j^{-1} (W_j x_{j-1} + E_j x_{j+1}) (odd j)
// Each kernel is one launch per level over all blocks of that level.
//
// Batches: every kernel takes nb right-hand sides at once (batch member b's
// strips at offset b * SB, its grid vectors at offset b * N).  A reduction step
// loads each factor matrix once and applies it to all nb vectors, so a batch
// shares both the factor traffic and the chain of dependent launches.
#include <vector>

#include "ls_internal.cuh"
#include "ls_strip.cuh"

namespace {

constexpr int kMvThreads = 256;

// Right-hand side of a local solve, block i (a strip column), row r, member b: the gathered
// field plus the injections of Algorithm 1, formed where level 0 reads it, so that the chain
// of a sweep holds no kernels but the reduction steps.  Rows E+t-1 and E+t take the traces of
// the layer above (its down-sweep solution, which stays in place until the upward sweep has
// passed this layer), rows E-1 and E those of the layer below (upward sweep only).
template <typename T>
struct RhsSrc {
    using C = cpx_t<T>;
    const C* rhs;      // gathered g^l; member b at + b * SB (never written by the solve)
    const C* inj;      // cinj of layer l: [slot][dx+1][i]
    const C* above;    // solution of layer l + 1, or null
    const C* below;    // solution of layer l - 1 (upward sweep), or null
    const C* tself;    // w^l_0 of the down sweep (upward sweep); member b at + b * TB
    C* tsave;          // where w^{l+1}_0 is kept for the upward sweep (down sweep), or null
    size_t SB, TB;
    int n, q, E, t;
    __device__ __forceinline__ C load(int i, int r, int b) const {
        const size_t mo = (size_t)b * SB;
        C val = rhs[mo + (size_t)i * q + r];
        if (above) {
            if (r == E + t - 1) {  // -C^l_{n,n+1} w^{l+1}_1 ; w^{l+1}_1 = row E of layer l+1
                for (int dx = -1; dx <= 1; ++dx)
                    if (i + dx >= 0 && i + dx < n)
                        val = cfms(inj[(size_t)(0 * 3 + dx + 1) * n + i], above[mo + (size_t)(i + dx) * q + E], val);
            } else if (r == E + t) {  // +C^l_{n+1,n} w^{l+1}_0 ; w^{l+1}_0 = row E-1 of layer l+1
                for (int dx = -1; dx <= 1; ++dx)
                    if (i + dx >= 0 && i + dx < n)
                        val = cfma(inj[(size_t)(1 * 3 + dx + 1) * n + i], above[mo + (size_t)(i + dx) * q + E - 1], val);
            }
        }
        if (below) {
            if (r == E) {  // -C^l_{1,0} (v^{l-1}_n - w^l_0) ; v^{l-1}_n = row E+t-1 of layer l-1
                for (int dx = -1; dx <= 1; ++dx) {
                    if (i + dx < 0 || i + dx >= n) continue;
                    const C p0 = below[mo + (size_t)(i + dx) * q + E + t - 1] - tself[(size_t)b * TB + i + dx];
                    val = cfms(inj[(size_t)(2 * 3 + dx + 1) * n + i], p0, val);
                }
            } else if (r == E - 1) {  // +C^l_{0,1} v^{l-1}_{n+1} ; v^{l-1}_{n+1} = row E+t of layer l-1
                for (int dx = -1; dx <= 1; ++dx) {
                    if (i + dx < 0 || i + dx >= n) continue;
                    val = cfma(inj[(size_t)(3 * 3 + dx + 1) * n + i], below[mo + (size_t)(i + dx) * q + E + t], val);
                }
            }
        }
        return val;
    }
    __device__ __forceinline__ void keep_trace(int i, int b) const {
        if (tsave) tsave[(size_t)b * TB + i] = above[(size_t)b * SB + (size_t)i * q + E - 1];
    }
};

// The tridiagonal couplings of level 0 (blocks W_i, E_i) of one strip: [i][dz+1][r]
template <typename T>
struct Couple {
    const cpx_t<T>* cw;
    const cpx_t<T>* ce;
};

// One reduction step.  A CTA takes one block j of the level and a chunk of R of its rows (S
// chunks a block) for NB (>= nb) batch members:
//   out_b = base_b + sum_t M_t v_{t,b}
//   MODE 0 (level 0 odd):     x_j = D^{-1} b_j
//   MODE 1 (forward, k >= 1): even j: x_j = x_j - F x_{j-1} - G x_{j+1};  odd j: y_j = D^{-1} x_j
//   MODE 2 (backward):        x_j = y_j - P x_{j-1} - Q x_{j+1}   (odd j, levels >= 1)
//   MODE 3 (top block):       x_0 = D^{-1} x_0   (S = 1; only to build the reduced inverse)
//   MODE 4 (level 0 back):    x_j = x_j - D^{-1} (W_j x_{j-1} + E_j x_{j+1})   (odd j)
//   MODE 6 (level c):         x = S_c^{-1} y over all nc unknowns of the level
// (the even blocks of level 0: k_cr_even)
//
// What bounds a step is latency: a local solve is a chain of dependent steps, most over a few
// blocks.  On GB300 a chain of trivial kernels takes 1.0 us a link, and handing partial sums
// from CTA to CTA through global memory adds 2.5 us.  So
//   * a level with few blocks is split by rows, which needs no sums across CTAs.  No CTA
//     writes what another one reads: D^{-1} b of the odd blocks is taken on the forward way,
//     into y, where it is off the backward chain and frees x_j for writing;
//   * thread (cg, rr) takes row rr of the chunk and columns cg, cg + CG, ... (CG = 256 / R):
//     no lane idles on rows past q (FP64 runs at 1/64 of the FP32 rate: at q = 70 rows padded
//     to warps cost 37 per cent), and the CG partial sums meet in shared memory;
//   * every step is launched programmatically and loads its first PF columns per thread and
//     its coupling tables (constant data) while its predecessor runs; the register window then
//     stays PF columns ahead of the products.  A step lets its successor start at once (one
//     FP32 member: bytes are short), when it has its vectors, or (FP64, few CTAs) at its end:
//     a successor placed while CTAs still run fills the idle SMs first, two or three CTAs
//     each, and the FP64 pipe of those then holds everyone up (a 64^2 FP64 solve: 53 us with
//     the trigger at once, 41 after the vectors, 36 at the end; at 400^2 145, 144 and 154 us,
//     so steps of more CTAs keep the second form).
// A local solve inside Algorithm 2 of one field (gathers and scatters included) went from 124 to
// 73 us (768^2, FP32), from 219 to 146 us (400^2, FP64: 27 million multiply-adds, 50 us at the
// FP64 rate) and from 82 to 36 us (64^2, FP64).
template <typename T>
struct CrStep {
    using C = cpx_t<T>;
    int q, k, nk;                  // strip height, level, blocks of the level
    int S, R;                      // row chunks per block (MODE 6: in all), rows of a chunk
    int nlead;                     // MODE 1: CTAs on even blocks (the odd blocks' follow)
    const C* pool;                 // first matrix of the strip (q x q, column-major)
    size_t off_a, off_b, off_c;    // level offsets (matrices): D^{-1}; F or P; G or Q
    C* x;                          // strip vectors; member b at + b * SB
    C* y;                          // y_j of the odd blocks of levels >= 1; at level c, its right-hand side
    size_t SB, YB;                 // member strides
    size_t pool_strip, x_strip;    // strip blockIdx.y (elements; the set-up runs all strips at once)
    int nb;
    bool early;                    // let the successor start at once (one FP32 member, a chain alone)
    bool to_y;                     // MODE 1: the even results go to y (the last level before c)
    const C* inv;                  // MODE 6: S_c^{-1} (nc x nc, column-major), blocks j << c
    int nc, c;
    RhsSrc<T> src;                 // MODE 0, k_cr_even
    Couple<T> cp;                  // MODE 4, k_cr_even
};

template <int MODE> constexpr int cr_mats() { return MODE == 1 || MODE == 2 ? 2 : 1; }   // matrices, a vector each
template <int MODE> constexpr int cr_tabs() { return MODE == 4 ? 1 : 0; }                // coupling tables
// columns a thread keeps in flight: 24 (FP64 32) registers of matrix entries, so that (FP32) four CTAs
// share an SM: 768^2, one member, 71 us a solve against 80 with 40 registers, 78 with five
// CTAs of 48 and 89 with three of 80
template <typename T, int MODE> constexpr int cr_prefetch() { return (sizeof(T) == 8 ? 8 : 12) / cr_mats<MODE>(); }
template <typename T, int NB> constexpr int cr_min_ctas() { return sizeof(T) == 8 ? (NB <= 2 ? 3 : 2) : (NB <= 4 ? 4 : 3); }
// shared memory: vectors (q or nc long) | partial sums | couplings
template <typename T, int MODE, int NB>
constexpr size_t cr_smem(int q, int nc) {
    return sizeof(cpx_t<T>) * ((size_t)cr_mats<MODE>() * NB * (MODE == 6 ? nc : q) + (size_t)kMvThreads * NB +
                               (size_t)cr_tabs<MODE>() * 6 * q);
}

template <typename T, int MODE, int NB>
__global__ void __launch_bounds__(kMvThreads, (cr_min_ctas<T, NB>())) k_cr_step(CrStep<T> a) {
    using C = cpx_t<T>;
    constexpr int NM = cr_mats<MODE>(), PF = cr_prefetch<T, MODE>();
    const bool early = sizeof(T) == 4 && NB == 1 && a.early;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    if (early) pdl_trigger();
    const int q = a.q, ncol = MODE == 6 ? a.nc : q;
    C* vin = reinterpret_cast<C*>(smem_raw);     // [NM][NB][ncol]
    C* red = vin + (size_t)NM * NB * ncol;       // [CG][NB][R]
    C* tab = red + kMvThreads * NB;              // MODE 4: [W, E][dz+1][q]
    const int tid = threadIdx.x;
    const int b0 = blockIdx.z * NB, nb = a.nb - b0 < NB ? a.nb - b0 : NB;
    const C* pool = a.pool + blockIdx.y * a.pool_strip;
    C* x = a.x + blockIdx.y * a.x_strip + (size_t)b0 * a.SB;
    C* y = a.y + blockIdx.y * a.x_strip + (size_t)b0 * a.YB;
    // block and matrices
    const size_t qq = (size_t)q * q;
    const size_t s = (size_t)q << a.k;           // elements between neighbouring blocks of the level
    bool odd = MODE == 0 || MODE == 2 || MODE == 4;
    int bid = blockIdx.x;
    if (MODE == 1 && bid >= a.nlead) {
        odd = true;
        bid -= a.nlead;
    }
    const int idx = MODE == 6 ? 0 : bid / a.S, sp = bid - idx * a.S;
    const int j = 2 * idx + (odd ? 1 : 0);
    const bool hw = j >= 1, he = j + 1 < a.nk;
    const C* Ms[NM];
    int vb[NM], nm = 1;                          // the vectors' blocks (level index), matrices present
    if (MODE == 6) {
        Ms[0] = a.inv;
        vb[0] = 0;
    } else if (NM == 1 || (MODE != 2 && odd)) {
        Ms[0] = pool + (a.off_a + idx) * qq;
        vb[0] = j;
    } else {                                     // the neighbours that exist
        const C* M0 = pool + (a.off_b + idx) * qq;
        const C* M1 = pool + (a.off_c + idx) * qq;
        Ms[0] = hw ? M0 : M1;
        vb[0] = hw ? j - 1 : j + 1;
        nm = (hw && he) ? 2 : 1;
        Ms[NM - 1] = nm == 2 ? M1 : Ms[0];
        vb[NM - 1] = nm == 2 ? j + 1 : vb[0];
    }
    const int R = a.R, r0 = sp * R, nr = (MODE == 6 ? a.nc : q) - r0 < R ? (MODE == 6 ? a.nc : q) - r0 : R;
    const int CG = kMvThreads / R, cg = tid / R, rr = tid - cg * R;
    const bool act = cg < CG && rr < nr;
    C pre[PF][NM];
    auto load_col = [&](C (&m)[NM], int c) {
#pragma unroll
        for (int t = 0; t < NM; ++t)
            m[t] = (act && c < ncol && t < nm) ? __ldg(&Ms[t][(size_t)c * ncol + r0 + rr]) : czero<C>();
    };
#pragma unroll
    for (int u = 0; u < PF; ++u) load_col(pre[u], cg + u * CG);
    if constexpr (cr_tabs<MODE>() > 0) {
        for (int w = tid; w < 6 * q; w += kMvThreads)
            tab[w] = __ldg(w < 3 * q ? &a.cp.cw[(size_t)j * 3 * q + w] : &a.cp.ce[(size_t)j * 3 * q + (w - 3 * q)]);
        __syncthreads();
    }
    pdl_wait();

    // In the set-up's FP64 steps on the identity's columns most vectors are still zero on the
    // forward way: their products are left out.
    constexpr bool kSparse = sizeof(T) == 8 && NB == 8;
    bool nonzero = false;
    // vectors, row r = tid % 128, members and slots alternating between the halves of the CTA
    if constexpr (MODE == 6) {
        for (int c = tid; c < ncol; c += kMvThreads) {
            const int jb = c / q;
            const size_t e = (((size_t)jb << a.c) - jb) * q + c;   // (jb << c) * q + c % q
#pragma unroll
            for (int b = 0; b < NB; ++b) vin[(size_t)b * ncol + c] = b < nb ? y[b * a.YB + e] : czero<C>();
        }
    } else {
        const int r = tid & 127;
#pragma unroll
        for (int p = 0; p < NM * NB; ++p) {
            const int v = p / NB, b = p % NB;
            if ((p & 1) != (tid >> 7) || r >= q) continue;
            C val = czero<C>();
            if (b < nb && v < nm) {
                const C* xb = x + (size_t)b * a.SB;
                if (MODE == 0) val = a.src.load(j, r, b0 + b);
                if (MODE == 1 || MODE == 2 || MODE == 3) {
                    val = xb[(size_t)vb[v] * s + r];
                    if (MODE == 2 || !(odd || MODE == 3)) val = -val;
                }
                if (MODE == 4) {   // -(W x_{j-1} + E x_{j+1})
#pragma unroll
                    for (int dz = -1; dz <= 1; ++dz) {
                        const int rz = r + dz;
                        if (rz < 0 || rz >= q) continue;
                        val = cfma(tab[(dz + 1) * q + r], xb[(size_t)(j - 1) * q + rz], val);
                        if (he) val = cfma(tab[(dz + 4) * q + r], xb[(size_t)(j + 1) * q + rz], val);
                    }
                    val = -val;
                }
            }
            vin[(size_t)p * q + r] = val;
            if (kSparse) nonzero = nonzero || val.x != T(0) || val.y != T(0);
        }
        if (MODE == 0 && sp == 0 && tid < nb) a.src.keep_trace(j, b0 + tid);
    }
    // what the result is added to (the first of this thread's outputs: fetched ahead)
    const int nout = nb * nr;
    auto base_of = [&](int b, int r) {
        if (MODE == 2) return y[(size_t)b * a.YB + (size_t)j * s + r];
        if ((MODE == 1 && !odd) || MODE == 4) return x[(size_t)b * a.SB + (size_t)j * s + r];
        return czero<C>();
    };
    C base = czero<C>();
    if (tid < nout) base = base_of(NB == 1 ? 0 : tid / nr, r0 + (NB == 1 ? tid : tid % nr));
    int cend = ncol;
    if (kSparse) cend = __syncthreads_or(nonzero) ? ncol : 0;
    else __syncthreads();
    if (!early && !(sizeof(T) == 8 && gridDim.x <= 304)) pdl_trigger();   // else at its end
    C part[NB];
#pragma unroll
    for (int b = 0; b < NB; ++b) part[b] = czero<C>();
    for (int c0 = cg; c0 < cend; c0 += CG * PF) {
#pragma unroll
        for (int u = 0; u < PF; ++u) {
            const int c = c0 + u * CG;
            if (c < ncol) {
#pragma unroll
                for (int t = 0; t < NM; ++t)
                    if (t < nm) {
#pragma unroll
                        for (int b = 0; b < NB; ++b)
                            part[b] = cfma(pre[u][t], vin[((size_t)t * NB + b) * ncol + c], part[b]);
                    }
            }
            load_col(pre[u], c + CG * PF);
        }
    }
    if (act) {
#pragma unroll
        for (int b = 0; b < NB; ++b) red[((size_t)cg * NB + b) * R + rr] = part[b];
    }
    __syncthreads();
    // the CG partial sums in two stages (about sqrt(CG) dependent adds each, in a fixed order):
    // FP64 adds take tens of cycles, and a chain of 32 of them 2 us
    auto add_up = [&](int first, int step, int b, int rc) {
        C sum = red[((size_t)first * NB + b) * R + rc];
#pragma unroll 4
        for (int g = first + step; g < CG; g += step) sum = sum + red[((size_t)g * NB + b) * R + rc];
        return sum;
    };
    const int G1 = CG >= 25 ? 6 : (CG >= 9 ? 4 : CG);
    if (G1 < CG) {
        for (int o = tid; o < G1 * nout; o += kMvThreads) {
            const int g = o / nout, w = o - g * nout, b = NB == 1 ? 0 : w / nr, rc = w - b * nr;
            red[((size_t)g * NB + b) * R + rc] = add_up(g, G1, b, rc);
        }
        __syncthreads();
    }
    for (int o = tid; o < nout; o += kMvThreads) {
        const int b = NB == 1 ? 0 : o / nr, rc = o - b * nr, r = r0 + rc;
        C sum = red[(size_t)b * R + rc];
#pragma unroll 6
        for (int g = 1; g < G1; ++g) sum = sum + red[((size_t)g * NB + b) * R + rc];
        C* xb = x + (size_t)b * a.SB;
        C* yb = y + (size_t)b * a.YB;
        if (o != tid) base = base_of(b, r);
        if (MODE == 6) {
            const int jb = r / q;
            xb[(((size_t)jb << a.c) - jb) * q + r] = sum;
        } else if (MODE == 1) {
            const size_t e = (size_t)j * s + r;
            if (odd) {
                yb[e] = sum;
            } else {
                sum = base + sum;
                if (a.to_y) yb[e] = sum;
                else xb[e] = sum;
            }
        } else if (MODE == 2 || MODE == 4) {
            xb[(size_t)j * s + r] = base + sum;
        } else {   // MODE 0, 3
            xb[(size_t)j * s + r] = sum;
        }
    }
}

// Level-0 even blocks: x_i = b_i - W_i y_{i-1} - E_i y_{i+1}, one thread per row and member.  A
// link of its own in the chain, of about 2 us.  Formed where level 1 reads the blocks instead, it
// is computed up to three times per block, again in every row chunk and for every member, and its
// tables take shared memory: a field of Algorithm 2 on FP32 steps, that form -> this one, ms:
// 768^2 3.42 -> 3.33 (one field), 1.99 -> 1.83 (a batch of 2), 1.12 -> 0.96 (8); 32 fields of
// 2048^2 in chunks of 8 on four streams 4.66 -> 3.44.
template <typename T>
__global__ void __launch_bounds__(128) k_cr_even(CrStep<T> a) {
    const int i = 2 * blockIdx.x, b = blockIdx.y, q = a.q, n = a.src.n;
    const int r = threadIdx.x < q ? threadIdx.x : q - 1;
    const cpx_t<T>* wi = a.cp.cw + (size_t)i * 3 * q + r;
    const cpx_t<T>* ei = a.cp.ce + (size_t)i * 3 * q + r;
    cpx_t<T> w[3], e[3], xw[3], xe[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        w[d] = __ldg(&wi[(size_t)d * q]);
        e[d] = __ldg(&ei[(size_t)d * q]);
    }
    pdl_trigger();
    pdl_wait();
    if (threadIdx.x >= q) return;
    if (r == 0) a.src.keep_trace(i, b);
    cpx_t<T>* xb = a.x + (size_t)b * a.SB;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        const int rz = r + d - 1;
        const bool in = rz >= 0 && rz < q;
        xw[d] = in && i >= 1 ? xb[(size_t)(i - 1) * q + rz] : czero<cpx_t<T>>();
        xe[d] = in && i + 1 < n ? xb[(size_t)(i + 1) * q + rz] : czero<cpx_t<T>>();
    }
    cpx_t<T> val = a.src.load(i, r, b);
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        if (r + d - 1 < 0 || r + d - 1 >= q) continue;
        if (i >= 1) val = cfms(w[d], xw[d], val);
        if (i + 1 < n) val = cfms(e[d], xe[d], val);
    }
    xb[(size_t)i * q + r] = val;
}

// the identity, nc x nc per strip (the right-hand sides of the reduced inverse)
__global__ void k_identity(size_t total, int nc, double2* A) {
    for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (size_t)gridDim.x * blockDim.x) {
        const size_t w = e % ((size_t)nc * nc);
        A[e] = make_double2(w / nc == w % nc ? 1.0 : 0.0, 0.0);
    }
}
__global__ void k_inverse32(size_t total, const double2* __restrict__ a, float2* __restrict__ b) {
    for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (size_t)gridDim.x * blockDim.x)
        b[e] = ccast<float2>(a[e]);
}

// level 0, even blocks: b_j -= W_j y_{j-1} + E_j y_{j+1} (tabulated tridiagonal couplings)
template <typename T>
__global__ void k_l0_even(int q, int nblk, const cpx_t<T>* __restrict__ cw, const cpx_t<T>* __restrict__ ce,
                          cpx_t<T>* __restrict__ x, size_t SB) {
    using C = cpx_t<T>;
    const int j = 2 * blockIdx.x;
    const int r = threadIdx.x;
    if (r >= q) return;
    C* xb = x + (size_t)blockIdx.y * SB;
    C acc = xb[(size_t)j * q + r];
    const C* wj = cw + (size_t)j * 3 * q;
    const C* ej = ce + (size_t)j * 3 * q;
#pragma unroll
    for (int dz = -1; dz <= 1; ++dz) {
        const int rr = r + dz;
        if (rr < 0 || rr >= q) continue;
        if (j >= 1) acc = cfms(wj[(dz + 1) * q + r], xb[(size_t)(j - 1) * q + rr], acc);
        if (j + 1 < nblk) acc = cfms(ej[(dz + 1) * q + r], xb[(size_t)(j + 1) * q + rr], acc);
    }
    xb[(size_t)j * q + r] = acc;
}

// g^l = chi_{Omega^l} g (+ injection from the layer above), copied to the solution buffer.
// Batch member b = blockIdx.z: strips at + b * SB, traces at + b * TB, grid vector at + b * N.
// A tiled transpose: a CTA of 32 x 8 threads takes 32 strip rows r x 32 columns i; it
// reads the rows of g that fall in Omega^l along x (coalesced) into shared memory and
// writes the strip's block layout (column i = q contiguous values) along r (coalesced).
// The injected rows (eq. pde_GRF_down) are computed in the strip's precision.
// TR: g is the field of the other direction (the vertical layers' grid is the transpose
// of the field's): strip row r, column i is g[i][l t - E + r], contiguous along r, so the
// reads go straight to the strip layout without the shared-memory tile.
constexpr int kGatherTile = 32;
template <typename T, bool TR, typename GF = double2>
__global__ void __launch_bounds__(256) k_gather(StripGeom g, const cpx_t<T>* __restrict__ inj, int l,
                                                const GF* __restrict__ gf, cpx_t<T>* __restrict__ rhs,
                                                cpx_t<T>* __restrict__ sol, const cpx_t<T>* __restrict__ above,
                                                cpx_t<T>* __restrict__ trace_above, size_t SB, size_t TB) {
    using C = cpx_t<T>;
    __shared__ C tile[kGatherTile][kGatherTile + 1];   // [r - r0][i - i0]
    const int q = g.q, n = g.n, E = g.E, t = g.t;
    const size_t b = blockIdx.z;
    const int i0 = blockIdx.x * kGatherTile, r0 = blockIdx.y * kGatherTile;
    gf += b * (size_t)n * n;
    rhs += b * SB;
    sol += b * SB;
    if (above) {
        above += b * SB;
        trace_above += b * TB;
    }
    const int tx = threadIdx.x, ty = threadIdx.y;
    const GF z0 = {};
    GF v[kGatherTile / 8];
    if constexpr (TR) {
#pragma unroll
        for (int u = 0; u < kGatherTile / 8; ++u) {   // rows of Omega^l (E <= r < E + t), along r
            const int i = i0 + ty + 8 * u, r = r0 + tx;
            v[u] = (r >= E && r < E + t && i < n) ? __ldg(&gf[(size_t)i * n + (l * t - E + r)]) : z0;
        }
    } else {
#pragma unroll
        for (int u = 0; u < kGatherTile / 8; ++u) {   // rows of Omega^l (E <= r < E + t), along x
            const int r = r0 + ty + 8 * u, i = i0 + tx;
            v[u] = (r >= E && r < E + t && i < n) ? __ldg(&gf[(size_t)(l * t - E + r) * n + i]) : z0;
        }
#pragma unroll
        for (int u = 0; u < kGatherTile / 8; ++u) tile[ty + 8 * u][tx] = ccast<C>(v[u]);
        __syncthreads();
    }
#pragma unroll
    for (int u = 0; u < kGatherTile / 8; ++u) {   // strip columns, along r
        const int i = i0 + ty + 8 * u, r = r0 + tx;
        if (i >= n || r >= q) continue;
        const size_t e = (size_t)i * q + r;
        C cv = TR ? ccast<C>(v[u]) : tile[tx][ty + 8 * u];
        if (above) {
            if (r == 0) trace_above[i] = above[(size_t)i * q + E - 1];  // w^{l+1}_0, kept for the upward sweep
            const C* c0 = inj + (size_t)l * 12 * n;  // slots 0, 1 of layer l: [slot][dx+1][i]
            if (r == E + t - 1) {  // -C^l_{n,n+1} w^{l+1}_1 ; w^{l+1}_1 = row E of layer l+1
                for (int dx = -1; dx <= 1; ++dx)
                    if (i + dx >= 0 && i + dx < n)
                        cv = cfms(c0[(size_t)(0 * 3 + dx + 1) * n + i], above[(size_t)(i + dx) * q + E], cv);
            } else if (r == E + t) {  // +C^l_{n+1,n} w^{l+1}_0 ; w^{l+1}_0 = row E-1 of layer l+1
                for (int dx = -1; dx <= 1; ++dx)
                    if (i + dx >= 0 && i + dx < n)
                        cv = cfma(c0[(size_t)(1 * 3 + dx + 1) * n + i], above[(size_t)(i + dx) * q + E - 1], cv);
            }
        }
        rhs[e] = cv;
        sol[e] = cv;
    }
}

// The same tiles for all layers of a sweep at once, without the injections (the reduction
// steps on the CUDA cores add them where level 0 reads the right-hand side): blockIdx.x =
// (member * L + layer) * column tiles + tile.
template <typename T, bool TR, typename GF = double2>
__global__ void __launch_bounds__(256) k_gather_all(StripGeom g, int L, const GF* __restrict__ gf,
                                                    cpx_t<T>* __restrict__ rhs, size_t SB) {
    using C = cpx_t<T>;
    __shared__ C tile[kGatherTile][kGatherTile + 1];   // [r - r0][i - i0]
    const int q = g.q, n = g.n, E = g.E, t = g.t;
    const int it = (n + kGatherTile - 1) / kGatherTile, bl = blockIdx.x / it, b = bl / L, l = bl - b * L;
    const int i0 = (blockIdx.x - bl * it) * kGatherTile, r0 = blockIdx.y * kGatherTile;
    gf += (size_t)b * n * n;
    rhs += (size_t)b * SB + (size_t)l * n * q;
    const int tx = threadIdx.x, ty = threadIdx.y;
    const GF z0 = {};
    GF v[kGatherTile / 8];
#pragma unroll
    for (int u = 0; u < kGatherTile / 8; ++u) {   // rows of Omega^l (E <= r < E + t), along r (TR) or x
        const int i = i0 + (TR ? ty + 8 * u : tx), r = r0 + (TR ? tx : ty + 8 * u);
        const size_t e = TR ? (size_t)i * n + (l * t - E + r) : (size_t)(l * t - E + r) * n + i;
        v[u] = (r >= E && r < E + t && i < n) ? __ldg(&gf[e]) : z0;
    }
    if constexpr (!TR) {
#pragma unroll
        for (int u = 0; u < kGatherTile / 8; ++u) tile[ty + 8 * u][tx] = ccast<C>(v[u]);
        __syncthreads();
    }
#pragma unroll
    for (int u = 0; u < kGatherTile / 8; ++u) {   // strip columns, along r
        const int i = i0 + ty + 8 * u, r = r0 + tx;
        if (i < n && r < q) rhs[(size_t)i * q + r] = TR ? ccast<C>(v[u]) : tile[tx][ty + 8 * u];
    }
}

// Upward sweep: sol = g^l (a device copy of rhs made just before) plus the injection
// from the layer below, which touches only the two rows E - 1 and E; one thread per
// (column i, row) of those, batch member b = blockIdx.y.
template <typename T>
__global__ void k_inject_up(StripGeom g, const cpx_t<T>* __restrict__ inj, int l, const cpx_t<T>* __restrict__ rhs,
                            cpx_t<T>* __restrict__ sol, const cpx_t<T>* __restrict__ below,
                            const cpx_t<T>* __restrict__ trace_self, size_t SB, size_t TB) {
    using C = cpx_t<T>;
    const int o = blockIdx.x * blockDim.x + threadIdx.x;
    const int q = g.q, n = g.n, E = g.E, t = g.t;
    if (o >= 2 * n) return;
    const size_t b = blockIdx.y;
    rhs += b * SB;
    sol += b * SB;
    below += b * SB;
    trace_self += b * TB;
    const int i = o >> 1, r = (o & 1) ? E : E - 1;
    const size_t e = (size_t)i * q + r;
    C val = rhs[e];   // the injection in the strip's precision
    const C* c0 = inj + (size_t)l * 12 * n;  // slots 2, 3 of layer l: [slot][dx+1][i]
    if (r == E) {  // -C^l_{1,0} (v^{l-1}_n - w^l_0) ; v^{l-1}_n = row E+t-1 of layer l-1
        for (int dx = -1; dx <= 1; ++dx) {
            if (i + dx < 0 || i + dx >= n) continue;
            const C p0 = below[(size_t)(i + dx) * q + E + t - 1] - trace_self[i + dx];
            val = cfms(c0[(size_t)(2 * 3 + dx + 1) * n + i], p0, val);
        }
    } else {  // +C^l_{0,1} v^{l-1}_{n+1} ; v^{l-1}_{n+1} = row E+t of layer l-1
        for (int dx = -1; dx <= 1; ++dx) {
            if (i + dx < 0 || i + dx >= n) continue;
            val = cfma(c0[(size_t)(3 * 3 + dx + 1) * n + i], below[(size_t)(i + dx) * q + E + t], val);
        }
    }
    sol[e] = val;
}

// v = rows 1..n of every layer's solution (concatenation); blocks as in k_gather_all, whose tiled
// transpose this is the other way round: reads along r, writes along x.
template <typename T, typename OF = double2>
__global__ void __launch_bounds__(256) k_scatter(StripGeom g, int L, const cpx_t<T>* __restrict__ sol,
                                                 size_t strip_stride, size_t SB, OF* __restrict__ v) {
    using C = cpx_t<T>;
    __shared__ C tile[kGatherTile][kGatherTile + 1];   // [i - i0][row - r0]
    const int q = g.q, n = g.n, t = g.t;
    const int it = (n + kGatherTile - 1) / kGatherTile, bl = blockIdx.x / it, b = bl / L, l = bl - b * L;
    const int i0 = (blockIdx.x - bl * it) * kGatherTile, r0 = blockIdx.y * kGatherTile;
    sol += (size_t)b * SB + (size_t)l * strip_stride + g.E;
    v += (size_t)b * n * n + (size_t)l * t * n;
    const int tx = threadIdx.x, ty = threadIdx.y;
#pragma unroll
    for (int u = 0; u < kGatherTile / 8; ++u) {
        const int i = i0 + ty + 8 * u, r = r0 + tx;
        if (i < n && r < t) tile[ty + 8 * u][tx] = sol[(size_t)i * q + r];
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < kGatherTile / 8; ++u) {
        const int r = r0 + ty + 8 * u, i = i0 + tx;
        if (i < n && r < t) v[(size_t)r * n + i] = ccast<OF>(tile[tx][ty + 8 * u]);
    }
}

// The same for the other direction's field, added to a field of this one:
// v[i][z] = u[i][z] + (row z of the layers' solutions)[i]  (the vertical sweep's result
// transposed back and added to the horizontal one, Algorithm 2); along z, coalesced.
// FP32 fields are added in FP32 (the same sum as in FP64 rounded to FP32).
template <typename T, typename AF = double2, typename OF = double2>
__global__ void k_scatter_tadd(StripGeom g, const cpx_t<T>* __restrict__ sol, size_t strip_stride, size_t SB,
                               const AF* __restrict__ u, OF* __restrict__ v) {
    const int n = g.n, z = blockIdx.x * blockDim.x + threadIdx.x, i = blockIdx.y;
    if (z >= n) return;
    const size_t b = blockIdx.z;
    const int l = z / g.t, r = z - l * g.t + g.E;
    const size_t o = (b * n + i) * (size_t)n + z;
    const cpx_t<T> w = sol[b * SB + (size_t)l * strip_stride + (size_t)i * g.q + r];
    if constexpr (sizeof(T) == 4 && sizeof(AF) == 8 && sizeof(OF) == 8) v[o] = u[o] + w;
    else v[o] = ccast<OF>(ccast<double2>(u[o]) + ccast<double2>(w));
}

// natural strip layout (q rows x n, x fastest) <-> block layout (i*q + r)
template <typename T>
__global__ void k_strip_in(int n, int q, const double2* __restrict__ b, cpx_t<T>* __restrict__ x) {
    const size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= (size_t)n * q) return;
    const int i = (int)(e / q), r = (int)(e % q);
    x[e] = ccast<cpx_t<T>>(b[(size_t)r * n + i]);
}
template <typename T>
__global__ void k_strip_out(int n, int q, const cpx_t<T>* __restrict__ x, double2* __restrict__ b) {
    const size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= (size_t)n * q) return;
    const int r = (int)(e / n), i = (int)(e % n);
    b[e] = ccast<double2>(x[(size_t)i * q + r]);
}


StripGeom geom_of(const ls_handle* h) { return StripGeom{h->n, h->t, h->E, h->q, h->opts.shift / h->omega}; }

// Row chunks per block of a reduction step: levels with few blocks are split until about
// kCtas CTAs run, down to chunks of min_rows: 8 rows (64 contiguous bytes of an FP32 column), and
// 4 of the reduced inverse in FP64, whose few rows would leave FP64 pipes idle.  The handle's
// cr_split switches the splitting of the levels off (1 CTA per block); the reduced inverse is one
// product of up to 700 rows, not a block, and is always split: on the three CTAs that its rows
// need at least, it was the longest step of the solve (unsplit levels, a field of Algorithm 2, ms:
// 64^2 FP64 2.47 -> 0.52, 400^2 FP64 10.7 -> 6.9, 256^2 FP32 1.80 -> 1.01).
// Chains that run side by side on the lanes share the SMs, and their CTAs fill them without
// splitting: the target is divided by the chains, down to about one CTA per SM and level (cr_share),
// and a step starts its successor only when it has its vectors, so that CTAs that wait do not
// keep another chain's from their slots.  A field of Algorithm 2 on FP32 steps, 32 fields, ms:
// chunks of 1 on eight lanes at 256^2 0.29 -> 0.15, 1024^2 2.60 -> 2.22, of 4 0.12 -> 0.065 and
// 1.12 -> 0.90; FP64, 16 fields in chunks of 1, 128^2 0.43 -> 0.25, 400^2 2.48 -> 2.22.  Two
// chains keep 304 CTAs (768^2, chunks of 8: 0.576, against 0.606 with 152 and 0.642 with 608).
constexpr int kCtas = 608;
int cr_share(const ls_handle* h) { return h->chains >= 4 ? 4 : (h->chains >= 2 ? 2 : 1); }
template <typename T>
void cr_split(CrStep<T>& a, int rows, int blocks, int min_rows, int ctas) {
    int S = ctas / blocks;
    if (S < 1) S = 1;
    if (S > rows / min_rows) S = rows / min_rows;
    if (S < (rows + kMvThreads - 1) / kMvThreads) S = (rows + kMvThreads - 1) / kMvThreads;   // R <= kMvThreads
    a.R = (rows + S - 1) / S;
    a.S = (rows + a.R - 1) / a.R;
}

// Unknowns of the reduced system whose inverse replaces the levels from c on.  Larger means
// fewer dependent steps and more bytes a solve (nc^2 entries instead of about 2.5 q^2 per
// block): 8 blocks of 84 rows are one 3.6 MB (FP32) product of 2.5 us instead of seven steps
// of 2.8 us; 16 blocks would read 14 MB to save two more.  For thin strips 700 unknowns are many
// blocks, and building their inverse shows in ls_factor (512^2 in 512 layers of q = 5, FP64: 0.27
// -> 1.14 s, 1.0 -> 7.4 GB), which six applications of Algorithm 2 pay back (247 -> 87 ms each).
constexpr int kInverseMax = 700;

template <typename T, int MODE, int NB>
int cr_launch(ls_handle* h, const CrStep<T>& a, unsigned grid, unsigned strips = 1, unsigned groups = 1) {
    return ls_launch_pdl(h, k_cr_step<T, MODE, NB>, dim3(grid, strips, groups), dim3(kMvThreads),
                         cr_smem<T, MODE, NB>(a.q, a.nc), a);
}

template <typename T, int NB>
int cr_solve_nb(ls_handle* h, int dir, int l, cpx_t<T>* x, size_t SB, int nb, const RhsSrc<T>& src) {
    using C = cpx_t<T>;
    const DirFactors& F = h->fac[dir];
    const int q = h->q, n = h->n;
    const size_t qq = (size_t)q * q;
    const CrLevel& l0 = F.lev[0];
    const ls_handle::SweepLane& W = h->lanes[h->lane];
    CrStep<T> a{};
    a.q = q;
    if constexpr (sizeof(T) == 4) a.pool = F.pool32 + (size_t)l * F.mats_per_strip * qq;
    else a.pool = F.pool64 + (size_t)l * F.mats_per_strip * qq;
    a.x = x;
    a.y = static_cast<C*>(W.cr_y);
    a.SB = SB;
    a.YB = (size_t)n * q;
    a.nb = nb;
    a.early = h->chains == 1;
    a.src = src;
    a.cp = Couple<T>{static_cast<const C*>(F.cw) + (size_t)l * n * 3 * q,
                     static_cast<const C*>(F.ce) + (size_t)l * n * 3 * q};
    a.nc = F.inv_nc;
    a.c = F.inv_c;
    a.inv = static_cast<const C*>(F.inv) + (size_t)l * a.nc * a.nc;
    auto level = [&](int k, int blocks) {
        const CrLevel& lv = F.lev[k];
        a.k = k;
        a.nk = lv.nk;
        a.off_a = lv.off_dinv;
        a.to_y = k == a.c - 1;
        cr_split(a, q, blocks, 8, h->cr_split ? kCtas / cr_share(h) : 0);
        a.nlead = lv.neven * a.S;
        return (unsigned)(blocks * a.S);
    };
    LS_TRY((cr_launch<T, 0, NB>(h, a, level(0, l0.nodd))));
    for (int k = 1; k < a.c; ++k) {
        const unsigned grid = level(k, F.lev[k].nk);
        a.off_b = F.lev[k].off_f;
        a.off_c = F.lev[k].off_g;
        if (k == 1) LS_TRY(ls_launch_pdl(h, k_cr_even<T>, dim3((unsigned)l0.neven, (unsigned)nb), dim3(128), 0, a));
        LS_TRY((cr_launch<T, 1, NB>(h, a, grid)));
    }
    cr_split(a, a.nc, 1, sizeof(T) == 8 ? 4 : 8, kCtas);
    LS_TRY((cr_launch<T, 6, NB>(h, a, (unsigned)a.S)));
    for (int k = a.c - 1; k >= 1; --k) {
        if (!F.lev[k].nodd) continue;
        const unsigned grid = level(k, F.lev[k].nodd);
        a.off_b = F.lev[k].off_p;
        a.off_c = F.lev[k].off_q;
        LS_TRY((cr_launch<T, 2, NB>(h, a, grid)));
    }
    const unsigned grid = level(0, l0.nodd);
    return cr_launch<T, 4, NB>(h, a, grid);
}

// The same local solve with the reduction steps on the tensor cores (ls_cr_mma.cu):
// every step a TF32 GEMM over the whole batch (up to 32 right-hand sides), the
// level-0 even update on the CUDA cores as above.
int cr_solve_tc(ls_handle* h, int dir, int l, float2* x, size_t SB, int nb) {
    const DirFactors& F = h->fac[dir];
    const int q = h->q, n = h->n;
    const CrLevel& l0 = F.lev[0];
    const float2* cw = static_cast<const float2*>(F.cw) + (size_t)l * n * 3 * q;
    const float2* ce = static_cast<const float2*>(F.ce) + (size_t)l * n * 3 * q;
    const int thr = (q + 31) / 32 * 32;
    // levels >= dense_c as one product with the reduced system's inverse, where it is built
    const bool dense = h->tc_dense && F.dense_nc && h->lanes[h->lane].dense_part;
    const int ktop = dense ? F.dense_c : F.K;
    if (l0.nodd) LS_TRY(ls_cr_tc_step(h, dir, l, 0, 0, l0.nk, (unsigned)l0.nodd, l0.off_dinv, 0, 0, x, SB, nb, cw, ce));
    LS_LAUNCH(h, k_l0_even<float>, dim3(l0.neven, nb), thr, 0, q, n, cw, ce, x, SB);
    for (int k = 1; k < ktop; ++k) {
        const CrLevel& lv = F.lev[k];
        LS_TRY(ls_cr_tc_step(h, dir, l, 1, k, lv.nk, (unsigned)lv.neven, 0, lv.off_f, lv.off_g, x, SB, nb, cw, ce));
    }
    if (dense) LS_TRY(ls_cr_dense_apply(h, dir, l, x, SB, nb));
    else LS_TRY(ls_cr_tc_step(h, dir, l, 3, 0, 1, 1u, F.off_top, 0, 0, x, SB, nb, cw, ce));
    for (int k = ktop - 1; k >= 1; --k) {
        const CrLevel& lv = F.lev[k];
        if (!lv.nodd) continue;
        LS_TRY(ls_cr_tc_step(h, dir, l, 2, k, lv.nk, (unsigned)lv.nodd, lv.off_dinv, lv.off_p, lv.off_q, x, SB, nb, cw,
                             ce));
    }
    if (l0.nodd) LS_TRY(ls_cr_tc_step(h, dir, l, 4, 0, l0.nk, (unsigned)l0.nodd, l0.off_dinv, 0, 0, x, SB, nb, cw, ce));
    return LS_OK;
}

// Where the reduction steps of a pass over nb right-hand sides run: on the tensor cores
// always (cr_tc 2), or for batches past the CUDA-core steps' sweet spot (cr_tc 1: at least 5
// right-hand sides; a one-matrix product per step does not fill them)
template <typename T>
bool cr_on_tensor_cores(const ls_handle* h, int nb) {
    return sizeof(T) == 4 && h->tc_ready && (h->cr_tc == 2 || (h->cr_tc == 1 && nb >= 5));
}

// Local solve on the CUDA cores: x = (C^l)^{-1} of the right-hand side src (which x must not
// overlap).  The batch template is the smallest supported NB >= nb (FP64 keeps NB <= 4 for
// registers).
template <typename T>
int cr_solve(ls_handle* h, int dir, int l, cpx_t<T>* x, size_t SB, int nb, const RhsSrc<T>& src) {
    if (nb <= 1) return cr_solve_nb<T, 1>(h, dir, l, x, SB, nb, src);
    if (nb <= 2) return cr_solve_nb<T, 2>(h, dir, l, x, SB, nb, src);
    if (nb <= 4) return cr_solve_nb<T, 4>(h, dir, l, x, SB, nb, src);
    if constexpr (sizeof(T) == 4) return cr_solve_nb<T, 8>(h, dir, l, x, SB, nb, src);
    return LS_EINVAL;
}

// The downward and upward sweeps with the local solves on the tensor cores (solutions in the
// lane's ssol; see sweep_impl).
template <typename GF>
int sweep_tc(ls_handle* h, int dir, const GF* g, int nb, bool tr) {
    const int n = h->n, q = h->q, L = h->L;
    const size_t sstride = (size_t)n * q;
    const size_t SB = (size_t)L * sstride, TB = (size_t)L * n;
    const ls_handle::SweepLane& W = h->lanes[h->lane];
    float2* rhs = static_cast<float2*>(W.srhs);
    float2* sol = static_cast<float2*>(W.ssol);
    float2* trc = static_cast<float2*>(W.strace);
    const float2* cinj = static_cast<const float2*>(h->fac[dir].cinj);
    const StripGeom geo = geom_of(h);
    const dim3 gg((unsigned)((n + kGatherTile - 1) / kGatherTile), (unsigned)((q + kGatherTile - 1) / kGatherTile), nb);
    const dim3 gb(kGatherTile, 8);
    for (int l = L - 1; l >= 0; --l) {  // downward sweep
        const float2* above = l < L - 1 ? sol + (l + 1) * sstride : nullptr;
        float2* tabove = l < L - 1 ? trc + (size_t)(l + 1) * n : nullptr;
        if (tr)
            LS_LAUNCH(h, (k_gather<float, true, GF>), gg, gb, 0, geo, cinj, l, g, rhs + l * sstride, sol + l * sstride,
                      above, tabove, SB, TB);
        else
            LS_LAUNCH(h, (k_gather<float, false, GF>), gg, gb, 0, geo, cinj, l, g, rhs + l * sstride, sol + l * sstride,
                      above, tabove, SB, TB);
        LS_TRY(cr_solve_tc(h, dir, l, sol + l * sstride, SB, nb));
    }
    const dim3 gi((unsigned)((2 * n + 255) / 256), nb);
    for (int l = 1; l < L; ++l) {  // upward sweep: sol = rhs, then the two injected rows
        LS_CUDA(cudaMemcpy2DAsync(sol + l * sstride, sizeof(float2) * SB, rhs + l * sstride, sizeof(float2) * SB,
                                  sizeof(float2) * sstride, nb, cudaMemcpyDeviceToDevice, h->stream));
        LS_LAUNCH(h, k_inject_up<float>, gi, 256, 0, geo, cinj, l, rhs + l * sstride, sol + l * sstride,
                  sol + (l - 1) * sstride, trc + (size_t)l * n, SB, TB);
        LS_TRY(cr_solve_tc(h, dir, l, sol + l * sstride, SB, nb));
    }
    return LS_OK;
}

// tr: g and v are fields of the other direction's grid (read and written transposed);
// add: v = add + the result (tr only).  GF, OF, AF: element types of g, v and add
// (double2; float2 for the mixed Algorithm 2's intermediate fields, which hold FP32
// values either way).
template <typename T, typename GF = double2, typename OF = double2, typename AF = double2>
int sweep_impl(ls_handle* h, int dir, const GF* g, OF* v, int nb, bool tr = false, const AF* add = nullptr) {
    using C = cpx_t<T>;
    const int n = h->n, q = h->q, L = h->L;
    const size_t sstride = (size_t)n * q;
    const size_t SB = (size_t)L * sstride, TB = (size_t)L * n;
    const ls_handle::SweepLane& W = h->lanes[h->lane];
    C* rhs = static_cast<C*>(W.srhs);
    C* sol = static_cast<C*>(W.ssol);
    C* trc = static_cast<C*>(W.strace);
    const DirFactors& F = h->fac[dir];
    const StripGeom geo = geom_of(h);
    const dim3 gg((unsigned)((n + kGatherTile - 1) / kGatherTile), (unsigned)((q + kGatherTile - 1) / kGatherTile), nb);
    const dim3 gb(kGatherTile, 8);
    const C* cinj = static_cast<const C*>(F.cinj);
    bool tc = false;
    if constexpr (sizeof(T) == 4) {
        tc = cr_on_tensor_cores<T>(h, nb);
        if (tc) LS_TRY((sweep_tc<GF>(h, dir, g, nb, tr)));
    }
    if (!tc) {
        const dim3 ga(gg.x * (unsigned)(nb * L), gg.y);
        if (tr) LS_LAUNCH(h, (k_gather_all<T, true, GF>), ga, gb, 0, geo, L, g, rhs, SB);
        else LS_LAUNCH(h, (k_gather_all<T, false, GF>), ga, gb, 0, geo, L, g, rhs, SB);
        RhsSrc<T> src{};
        src.SB = SB;
        src.TB = TB;
        src.n = n;
        src.q = q;
        src.E = h->E;
        src.t = h->t;
        auto layer = [&](int l, bool up) {
            src.rhs = rhs + l * sstride;
            src.inj = cinj + (size_t)l * 12 * n;
            src.above = l < L - 1 ? sol + (l + 1) * sstride : nullptr;
            src.below = up ? sol + (l - 1) * sstride : nullptr;
            src.tself = trc + (size_t)l * n;
            src.tsave = !up && l < L - 1 ? trc + (size_t)(l + 1) * n : nullptr;
            return cr_solve<T>(h, dir, l, sol + l * sstride, SB, nb, src);
        };
        for (int l = L - 1; l >= 0; --l) LS_TRY(layer(l, false));   // downward sweep
        for (int l = 1; l < L; ++l) LS_TRY(layer(l, true));         // upward sweep
    }
    if (tr && add) {
        LS_LAUNCH(h, (k_scatter_tadd<T, AF, OF>), dim3((unsigned)((n + 255) / 256), (unsigned)n, (unsigned)nb), 256, 0,
                  geo, sol, sstride, SB, add, v);
        return LS_OK;
    }
    LS_LAUNCH(h, (k_scatter<T, OF>), dim3(gg.x * (unsigned)(nb * L), (unsigned)((h->t + kGatherTile - 1) / kGatherTile)),
              gb, 0, geo, L, sol, sstride, SB, v);
    return LS_OK;
}

template <typename T, int NB, int... MODES>
int smem_optin_modes(int q) {
    cudaError_t e = cudaSuccess;
    auto one = [&](auto kern, size_t sz) {
        if (e == cudaSuccess && sz > 48 * 1024)
            e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sz);
    };
    (one(k_cr_step<T, MODES, NB>, cr_smem<T, MODES, NB>(q, kInverseMax)), ...);
    LS_CUDA(e);
    return LS_OK;
}
template <typename T, int NB>
int smem_optin_nb(int q) { return smem_optin_modes<T, NB, 0, 1, 2, 4, 6>(q); }
// (a kernel's limit is the process's, not the handle's: always that of the tallest strip, so that
// a handle of shorter strips does not lower it under another one)
int smem_optin(bool mixed) {
    constexpr int q = 112;
    if (mixed) {
        LS_TRY((smem_optin_nb<float, 1>(q)));
        LS_TRY((smem_optin_nb<float, 2>(q)));
        LS_TRY((smem_optin_nb<float, 4>(q)));
        LS_TRY((smem_optin_nb<float, 8>(q)));
    } else {
        LS_TRY((smem_optin_nb<double, 1>(q)));
        LS_TRY((smem_optin_nb<double, 2>(q)));
        LS_TRY((smem_optin_nb<double, 4>(q)));
    }
    return smem_optin_modes<double, 8, 1, 2, 3>(q);   // the reduced inverse
}

}  // namespace

// Workspace of the current lane for batches of up to nb right-hand sides (grown on
// demand; the lane's graphs, made for smaller buffers, are dropped).
static void lane_graphs_free(ls_handle::SweepLane& W) {
    for (int b = 0; b <= kMaxBatch; ++b) {
        for (auto& G : W.graphs[b]) {
            if (G.exec) cudaGraphExecDestroy(G.exec);
            if (G.graph) cudaGraphDestroy(G.graph);
            G = ls_handle::SweepLane::Graph{};
        }
    }
}

int ls_sweep_reserve(ls_handle* h, int nb) {
    ls_handle::SweepLane& W = h->lanes[h->lane];
    if (nb <= W.nb_cap) return LS_OK;
    lane_graphs_free(W);
    const size_t cnt = (size_t)h->L * h->n * h->q * nb;
    const size_t es = h->prec == LS_MIXED ? sizeof(float2) : sizeof(double2);
    const size_t N = (size_t)h->n * h->n;
    void* ptrs[] = {W.srhs, W.ssol, W.strace, W.vtmp, W.bd_in, W.bd_out, W.cr_y};
    for (void* p : ptrs) cudaFree(p);
    W.srhs = W.ssol = W.strace = W.vtmp = W.cr_y = nullptr;
    W.bd_in = W.bd_out = nullptr;
    W.nb_cap = 0;
    LS_CUDA(cudaMalloc(&W.srhs, es * cnt));
    LS_CUDA(cudaMalloc(&W.ssol, es * cnt));
    LS_CUDA(cudaMalloc(&W.strace, es * (size_t)h->L * h->n * nb));
    LS_CUDA(cudaMalloc(&W.vtmp, sizeof(double2) * N * 4 * nb));
    LS_CUDA(cudaMalloc(&W.bd_in, sizeof(double2) * N * nb));
    LS_CUDA(cudaMalloc(&W.bd_out, sizeof(double2) * N * nb));
    LS_CUDA(cudaMalloc(&W.cr_y, es * (size_t)h->n * h->q * nb));
    W.nb_cap = nb;
    return LS_OK;
}

void ls_lanes_free(ls_handle* h) {
    for (auto& W : h->lanes) {
        lane_graphs_free(W);
        void* ptrs[] = {W.srhs, W.ssol, W.strace, W.vtmp, W.bd_in, W.bd_out, W.cr_y, W.dense_part};
        for (void* p : ptrs) cudaFree(p);
        if (W.stream) cudaStreamDestroy(W.stream);
        if (W.done) cudaEventDestroy(W.done);
        W = ls_handle::SweepLane{};
    }
    if (h->ev_fork) cudaEventDestroy(h->ev_fork);
    h->ev_fork = nullptr;
}

// The inverse of the reduced system of level c (the first level >= 2 with at most kInverseMax
// unknowns; level K - 1 has two blocks, so there is one) of every strip of a direction: the
// steps of the levels from c on, in FP64, applied to the identity's columns in place -- every
// strip and column in the same launches.  Stored in the solves' precision.  Called by
// ls_factor once the factors in pool64 are complete (and the stream idle: the steps read
// factors ahead of their turn).
int ls_cr_inverse_build(ls_handle* h, int dir) {
    DirFactors& F = h->fac[dir];
    const int q = h->q, L = h->L;
    int c = 2;
    while (c < F.K - 1 && F.lev[c].nk * q > kInverseMax) ++c;
    const int nc = F.lev[c].nk * q;
    const size_t per = (size_t)nc * nc, total = per * L;
    double2 *A = nullptr, *y = nullptr;
    LS_CUDA(cudaMalloc(&A, sizeof(double2) * total));
    int rc = LS_OK;
    do {
        if (cudaMalloc(&y, sizeof(double2) * total) != cudaSuccess) { rc = ls_no_memory(); break; }
        k_identity<<<1216, 256, 0, h->stream>>>(total, nc, A);
        h->launches++;
        CrStep<double> a{};
        a.q = q;
        a.pool = F.pool64;
        a.pool_strip = F.mats_per_strip * (size_t)q * q;
        a.x = A;
        a.y = y;
        a.SB = a.YB = nc;
        a.x_strip = per;
        a.nb = nc;
        a.S = 1;
        a.R = q;
        const unsigned groups = (unsigned)((nc + 7) / 8);
        for (int k = c; k < F.K && rc == LS_OK; ++k) {
            const CrLevel& lv = F.lev[k];
            a.k = k - c;
            a.nk = lv.nk;
            a.off_a = lv.off_dinv;
            a.off_b = lv.off_f;
            a.off_c = lv.off_g;
            a.nlead = lv.neven;
            rc = cr_launch<double, 1, 8>(h, a, (unsigned)lv.nk, (unsigned)L, groups);
        }
        if (rc != LS_OK) break;
        a.k = 0;
        a.nk = 1;
        a.off_a = F.off_top;
        if ((rc = cr_launch<double, 3, 8>(h, a, 1, (unsigned)L, groups)) != LS_OK) break;
        for (int k = F.K - 1; k >= c && rc == LS_OK; --k) {
            const CrLevel& lv = F.lev[k];
            a.k = k - c;
            a.nk = lv.nk;
            a.off_b = lv.off_p;
            a.off_c = lv.off_q;
            if (lv.nodd) rc = cr_launch<double, 2, 8>(h, a, (unsigned)lv.nodd, (unsigned)L, groups);
        }
        if (rc != LS_OK) break;
        if (h->prec == LS_MIXED) {
            if (cudaMalloc(&F.inv, sizeof(float2) * total) != cudaSuccess) { rc = ls_no_memory(); break; }
            k_inverse32<<<1216, 256, 0, h->stream>>>(total, A, static_cast<float2*>(F.inv));
            h->launches++;
        } else {
            F.inv = A;
            A = nullptr;
        }
        F.inv_c = c;
        F.inv_nc = nc;
        cudaError_t e = cudaPeekAtLastError();
        if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
        if (e != cudaSuccess) rc = ls_cuda_fail(e);
    } while (0);
    cudaFree(A);
    cudaFree(y);
    return rc;
}

int ls_sweep_alloc(ls_handle* h) {
    LS_TRY(smem_optin(h->prec == LS_MIXED));
    for (int k = 1; k < ls_handle::kLanes; ++k) {
        LS_CUDA(cudaStreamCreateWithFlags(&h->lanes[k].stream, cudaStreamNonBlocking));
        LS_CUDA(cudaEventCreateWithFlags(&h->lanes[k].done, cudaEventDisableTiming));
    }
    LS_CUDA(cudaEventCreateWithFlags(&h->ev_fork, cudaEventDisableTiming));
    h->lane = 0;
    return ls_sweep_reserve(h, 1);
}

// Algorithm 1 on direction dir (0: horizontal layers; 1: vertical layers) for nb
// right-hand sides g (nb x N, contiguous) into v.
int ls_sweep_dir_b(ls_handle* h, int dir, const double2* g, double2* v, int nb) {
    if (nb < 1 || nb > ls_bd_cap(h)) return LS_EINVAL;
    LS_TRY(ls_sweep_reserve(h, nb));  // no-op when called inside a capture (reserved beforehand)
    const size_t N = (size_t)h->n * h->n;
    double2* t0 = static_cast<double2*>(h->lanes[h->lane].vtmp);
    double2* t1 = t0 + N * nb;
    if (dir == 0) {
        if (h->prec == LS_MIXED) return sweep_impl<float>(h, 0, g, v, nb);
        return sweep_impl<double>(h, 0, g, v, nb);
    }
    LS_TRY(ls_transpose64_b(h, g, t0, nb));
    if (h->prec == LS_MIXED) LS_TRY(sweep_impl<float>(h, 1, t0, t1, nb));
    else LS_TRY(sweep_impl<double>(h, 1, t0, t1, nb));
    return ls_transpose64_b(h, t1, v, nb);
}

int ls_sweep_dir(ls_handle* h, int dir, const double2* g, double2* v) { return ls_sweep_dir_b(h, dir, g, v, 1); }

// Algorithm 2 for nb right-hand sides: v = u1 + u2, u1 = Alg. 1 horizontal (g),
// u2 = Alg. 1 vertical (g - C u1).
// Mixed precision: the fields g, v and the intermediate u1, e are FP32 (the values the FP32
// sweeps read and produce), half the traffic of FP64 fields.
static int bd_direct_mixed(ls_handle* h, const float2* g, float2* v, int nb) {
    const size_t N = (size_t)h->n * h->n;
    float2* u1f = reinterpret_cast<float2*>(static_cast<double2*>(h->lanes[h->lane].vtmp) + 2 * N * nb);
    float2* ef = u1f + N * nb;
    LS_TRY((sweep_impl<float, float2, float2, float2>(h, 0, g, u1f, nb)));
    LS_TRY(ls_stencil_refine_f32(h, u1f, g, ef, nb));   // e = g - C u1
    // vertical layers on e as it is stored (their grid is its transpose): the gather reads
    // it transposed, and the scatter writes v = u1 + the result, transposed back
    return sweep_impl<float, float2, float2, float2>(h, 1, ef, v, nb, true, u1f);
}

static int bd_direct(ls_handle* h, const double2* g, double2* v, int nb) {
    const size_t N = (size_t)h->n * h->n;
    double2* u1 = static_cast<double2*>(h->lanes[h->lane].vtmp) + 2 * N * nb;
    double2* e = u1 + N * nb;
    LS_TRY(ls_sweep_dir_b(h, 0, g, u1, nb));
    LS_TRY(ls_stencil_apply_b(h, 0, 2, u1, g, e, nb));   // e = g - C u1
    // vertical layers on e as it is stored (their grid is its transpose): the gather reads
    // it transposed, and the scatter writes v = u1 + the result, transposed back
    return sweep_impl<double>(h, 1, e, v, nb, true, u1);
}

void ls_bd_graph_free(ls_handle* h) {
    for (auto& W : h->lanes) lane_graphs_free(W);
}

// A graph per share of the chip (the CUDA-core steps' row chunks depend on it).
static ls_handle::SweepLane::Graph& lane_graph(ls_handle* h, int nb) {
    const int share = cr_on_tensor_cores<float>(h, nb) ? 0 : cr_share(h) / 2;   // 1, 2, 4 -> 0, 1, 2
    return h->lanes[h->lane].graphs[nb][share];
}

// Capture Algorithm 2 for nb right-hand sides on the staging buffers once (the
// sequence of launches and all pointers are fixed after ls_factor), then replay it.
static int bd_capture(ls_handle* h, int nb) {
    cudaStream_t cap = nullptr;
    LS_CUDA(cudaStreamCreateWithFlags(&cap, cudaStreamNonBlocking));
    cudaStream_t saved = h->stream;
    const long long l0 = h->launches;
    h->stream = cap;
    int rc = LS_OK;
    cudaGraph_t graph = nullptr;
    cudaError_t e = cudaStreamBeginCapture(cap, cudaStreamCaptureModeThreadLocal);
    if (e == cudaSuccess) {
        if (h->prec == LS_MIXED)
            rc = bd_direct_mixed(h, reinterpret_cast<const float2*>(h->lanes[h->lane].bd_in),
                                 reinterpret_cast<float2*>(h->lanes[h->lane].bd_out), nb);
        else
            rc = bd_direct(h, h->lanes[h->lane].bd_in, h->lanes[h->lane].bd_out, nb);
        e = cudaStreamEndCapture(cap, &graph);
    }
    h->stream = saved;
    const long long nodes = h->launches - l0;
    h->launches = l0;
    cudaStreamDestroy(cap);
    if (rc != LS_OK) {
        if (graph) cudaGraphDestroy(graph);
        return rc;
    }
    if (e != cudaSuccess) return ls_cuda_fail(e);
    cudaGraphExec_t exec = nullptr;
    e = cudaGraphInstantiate(&exec, graph, 0);
    if (e != cudaSuccess) {
        cudaGraphDestroy(graph);
        return ls_cuda_fail(e);
    }
    lane_graph(h, nb) = {graph, exec, nodes};
    return LS_OK;
}

// Algorithm 2 on FP32 fields (mixed precision): the captured graph reads and writes the
// lane's staging buffers as FP32.
int ls_bd_b(ls_handle* h, const float2* g, float2* v, int nb) {
    if (h->prec != LS_MIXED) return LS_ESTATE;
    if (nb < 1 || nb > ls_bd_cap(h)) return LS_EINVAL;
    LS_TRY(ls_sweep_reserve(h, nb));
    if (!h->opts.use_graphs) return bd_direct_mixed(h, g, v, nb);
    ls_handle::SweepLane& W = h->lanes[h->lane];
    ls_handle::SweepLane::Graph& G = lane_graph(h, nb);
    if (!G.exec) LS_TRY(bd_capture(h, nb));
    const size_t N = (size_t)h->n * h->n;
    LS_CUDA(cudaMemcpyAsync(W.bd_in, g, sizeof(float2) * N * nb, cudaMemcpyDeviceToDevice, h->stream));
    LS_CUDA(cudaGraphLaunch(G.exec, h->stream));
    h->launches += G.nodes;
    LS_CUDA(cudaMemcpyAsync(v, W.bd_out, sizeof(float2) * N * nb, cudaMemcpyDeviceToDevice, h->stream));
    return LS_OK;
}

int ls_bd_b(ls_handle* h, const double2* g, double2* v, int nb) {
    if (nb < 1 || nb > ls_bd_cap(h)) return LS_EINVAL;
    LS_TRY(ls_sweep_reserve(h, nb));
    ls_handle::SweepLane& W = h->lanes[h->lane];
    ls_handle::SweepLane::Graph& G = lane_graph(h, nb);
    const size_t N = (size_t)h->n * h->n;
    if (h->prec == LS_MIXED) {   // through FP32 copies in the lane's staging buffers
        float2* in = reinterpret_cast<float2*>(W.bd_in);
        float2* out = reinterpret_cast<float2*>(W.bd_out);
        for (int b = 0; b < nb; ++b) LS_TRY(ls_vec_copy(h, g + b * N, in + b * N));
        if (!h->opts.use_graphs) {
            LS_TRY(bd_direct_mixed(h, in, out, nb));
        } else {
            if (!G.exec) LS_TRY(bd_capture(h, nb));
            LS_CUDA(cudaGraphLaunch(G.exec, h->stream));
            h->launches += G.nodes;
        }
        for (int b = 0; b < nb; ++b) LS_TRY(ls_vec_copy(h, out + b * N, v + b * N));
        return LS_OK;
    }
    if (!h->opts.use_graphs) return bd_direct(h, g, v, nb);
    if (!G.exec) LS_TRY(bd_capture(h, nb));
    LS_CUDA(cudaMemcpyAsync(W.bd_in, g, sizeof(double2) * N * nb, cudaMemcpyDeviceToDevice, h->stream));
    LS_CUDA(cudaGraphLaunch(G.exec, h->stream));
    h->launches += G.nodes;
    LS_CUDA(cudaMemcpyAsync(v, W.bd_out, sizeof(double2) * N * nb, cudaMemcpyDeviceToDevice, h->stream));
    return LS_OK;
}

template <typename FT>
static int bd_lanes(ls_handle* h, const FT* g, FT* v, int nb, int chunk, const unsigned char* on) {
    if (chunk < 1) return LS_EINVAL;
    const size_t N = (size_t)h->n * h->n;
    const int nchunks = (nb + chunk - 1) / chunk;
    std::vector<int> run;
    for (int c = 0; c < nchunks; ++c) {
        bool any = !on;
        for (int b = c * chunk; b < nb && b < (c + 1) * chunk && !any; ++b) any = on[b] != 0;
        if (any) run.push_back(c);
    }
    if (run.empty()) return LS_OK;
    if (run.size() == 1) {
        const int b0 = run[0] * chunk, cnt = nb - b0 < chunk ? nb - b0 : chunk;
        return ls_bd_b(h, g + b0 * N, v + b0 * N, cnt);
    }
    cudaStream_t main = h->stream;
    LS_CUDA(cudaEventRecord(h->ev_fork, main));
    h->chains = run.size() < ls_handle::kLanes ? (int)run.size() : ls_handle::kLanes;
    bool used[ls_handle::kLanes] = {};
    int rc = LS_OK;
    for (size_t ci = 0; ci < run.size() && rc == LS_OK; ++ci) {
        const int c = run[ci];
        const int k = (int)(ci % ls_handle::kLanes);
        const int b0 = c * chunk, cnt = nb - b0 < chunk ? nb - b0 : chunk;
        ls_handle::SweepLane& W = h->lanes[k];
        if (k > 0 && !used[k]) {
            const cudaError_t e = cudaStreamWaitEvent(W.stream, h->ev_fork, 0);
            if (e != cudaSuccess) {
                rc = ls_cuda_fail(e);
                break;
            }
        }
        used[k] = true;
        h->stream = k > 0 ? W.stream : main;
        h->lane = k;
        rc = ls_bd_b(h, g + b0 * N, v + b0 * N, cnt);
        h->stream = main;
        h->lane = 0;
    }
    h->chains = 1;
    for (int k = 1; k < ls_handle::kLanes; ++k) {  // join, also after a failure
        if (!used[k]) continue;
        cudaEventRecord(h->lanes[k].done, h->lanes[k].stream);
        cudaStreamWaitEvent(main, h->lanes[k].done, 0);
    }
    return rc;
}

int ls_bd_lanes(ls_handle* h, const double2* g, double2* v, int nb, int chunk, const unsigned char* on) {
    return bd_lanes(h, g, v, nb, chunk, on);
}
int ls_bd_lanes(ls_handle* h, const float2* g, float2* v, int nb, int chunk, const unsigned char* on) {
    return bd_lanes(h, g, v, nb, chunk, on);
}

int ls_bd(ls_handle* h, const double2* g, double2* v) { return ls_bd_b(h, g, v, 1); }

int ls_bd_cap(const ls_handle* h) {
    if (h->prec != LS_MIXED) return 4;
    return h->tc_ready && h->cr_tc ? ls_cr_tc_max_nb(h) : 8;
}

template <typename T>
static int strip_solve(ls_handle* h, int dir, int layer, const double2* b, double2* x, unsigned nblk, size_t SB) {
    using C = cpx_t<T>;
    const int n = h->n, q = h->q;
    C* sol = static_cast<C*>(h->lanes[0].ssol);
    C* rhs = static_cast<C*>(h->lanes[0].srhs);
    if (cr_on_tensor_cores<T>(h, 1)) {   // in place
        LS_LAUNCH(h, k_strip_in<T>, nblk, 256, 0, n, q, b, sol);
        if constexpr (sizeof(T) == 4) LS_TRY(cr_solve_tc(h, dir, layer, sol, SB, 1));
    } else {
        LS_LAUNCH(h, k_strip_in<T>, nblk, 256, 0, n, q, b, rhs);
        RhsSrc<T> src{};
        src.rhs = rhs;
        src.SB = SB;
        src.n = n;
        src.q = q;
        LS_TRY(cr_solve<T>(h, dir, layer, sol, SB, 1, src));
    }
    LS_LAUNCH(h, k_strip_out<T>, nblk, 256, 0, n, q, sol, x);
    return LS_OK;
}

int ls_strip_solve(ls_handle* h, int dir, int layer, const double2* b, double2* x) {
    const int n = h->n, q = h->q;
    const size_t cnt = (size_t)n * q;
    const unsigned nblk = (unsigned)((cnt + 255) / 256);
    const size_t SB = (size_t)h->L * cnt;
    return h->prec == LS_MIXED ? strip_solve<float>(h, dir, layer, b, x, nblk, SB)
                               : strip_solve<double>(h, dir, layer, b, x, nblk, SB);
}
