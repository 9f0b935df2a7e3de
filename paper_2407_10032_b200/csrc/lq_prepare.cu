// Stage 2 -- Algorithm 1 line 4: dampen H, invert, and take the upper Cholesky factor of the
// inverse ("Scaling to Billion-Parameter LLMs Using Cholesky and Dampening").
//
// Route: with H_d = H + damp*I, factor H_d = R R^T with R upper triangular (a Cholesky
// factorisation run from the last column backwards).  Then H_d^-1 = R^-T R^-1 and, by
// uniqueness of the Cholesky factor, U = R^-1 is exactly the upper factor with
// H_d^-1 = U^T U that the column loop needs; diag(H_d^-1)_j = sum_k U[k][j]^2.
// That is one factorisation plus one triangular inversion (2/3 c^3 flops) instead of
// factor + invert + factor again.
//
// The two are run as ONE sweep over 128-wide block columns k = last .. 0.  R is inverted in
// place by block Gauss-Jordan elimination with the pivots taken in the same descending order,
// so that step k needs exactly what the factorisation has produced by then:
//   diag   : A[k][k] (symmetric positive definite) -> V_k = R_kk^-1            (one CTA)
//   panel  : P_i = A[i][k] V_k^T = R[i][k]  (i < k);   A[k][j] <- V_k A[k][j]  (j > k, final U)
//   update : A[i][j] -= P_i P_j^T   (i <= j < k, the Cholesky trailing update)
//            A[i][j] -= P_i A[k][j] (i < k < j, the Gauss-Jordan update)
//            A[i][k]  = -P_i V_k    (i < k)
// Every product has inner dimension 128 and all of a step's updates form one launch over the
// whole width, so the grid stays large from the first step to the last.
//
// The matrix and the diagonal blocks are fp64 (fp32 factors of an ill-conditioned H move too many quantisation decisions).
// Matrices below 48 blocks (6144 columns) are bound by the serial chain of diagonal blocks and stay on the FP64 tensor-core
// MMA (mma.sync m8n8k4 f64, fed by a cp.async ring) throughout.  Wider ones are swept in outer blocks of OBB = 8 block columns
// (1024 columns): only an outer block's own 1024 x 1024 diagonal part goes through the steps above; its panels, the final rows
// of U beside it and the updates of all other tiles are products of inner dimension 1024 on the integer tensor cores
// (tcgen05 kind::i8, lq_tc_gemm), see wide_sweep().  The fp64 operands are cut into balanced 8-bit integer digits below a
// per-row power of two; the digit products of one level sum exactly in int32.
//   far tiles : 5 digits, 15 products; the leading pair (s = t = 1) is a result of its own, the levels s + t = 3 .. 6 are
//               combined, least significant first, in fp32, and the two are added in fp64.  Worth ~39 bits relative to the
//               largest entry of a row; entries of one row of a panel differ by several bits, which is why four slices are
//               not enough (U then comes out 1e-7 to 5e-7 of its largest entry off, measured here and in the CPU emulation
//               alike; five hold it to 1e-8).
//   panels, rows of U : 6 digits, 21 products, two exact leading levels (they are products with the inverse factor V, whose
//               entries are up to sqrt(cond) larger than the results').
// An fp32 accumulation of split floating-point operands keeps ~20 bits whatever the number of terms and moves 0.1 - 0.2 % of the
// codes.  The older form with the outer block's rows and columns updated step by step on the FP64 MMA and the far tiles' slices as
// bf16 values remains selectable for tests.
#include "lq_common.cuh"
#include "lq_digits.cuh"

namespace {

constexpr int NB = 128;          // block width

// ------------------------------------------------------------------ set-up kernels --
// scal[0] = damp = damp_frac * mean(diag H), dead (zero) diagonal entries counted as 1.
__global__ void diag_mean_kernel(const float* __restrict__ H, int64_t c, int64_t ldh, double damp_frac,
                                 double* __restrict__ scal) {
    __shared__ double red[1024];
    double s = 0.0;
    for (int64_t i = threadIdx.x; i < c; i += blockDim.x) {
        float d = LQ_AT(H + i * ldh + i);
        s += (d == 0.0f) ? 1.0 : static_cast<double>(d);
    }
    red[threadIdx.x] = s;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) scal[0] = damp_frac * red[0] / static_cast<double>(c);
}

// Zero the weight columns of dead input channels.
template <typename T>
__global__ void zero_dead_columns_kernel(const float* __restrict__ H, int64_t c, int64_t ldh, T* __restrict__ W,
                                         int64_t r, int64_t ldw) {
    const int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (j >= c) return;
    if (LQ_AT(H + j * ldh + j) != 0.0f) return;
    for (int64_t i = blockIdx.y; i < r; i += gridDim.y) LQ_AT(W + i * ldw + j) = T(0.0f);
}

// A[cp x cp] (fp64): upper triangle of H plus damping; identity on the padding; the strictly
// lower part is zeroed.  Non-finite inputs are reported.
__global__ void load_damped_kernel(const float* __restrict__ H, int64_t c, int64_t ldh, const double* __restrict__ scal,
                                   double* __restrict__ A, int64_t cp, lq_dev_status* st) {
    const int64_t i = blockIdx.y;
    const double damp = scal[0];
    // four entries per thread: one 16-byte read where the row of H allows it, two 16-byte writes
    const bool vec = (ldh % 4 == 0) && ((reinterpret_cast<uintptr_t>(H) & 15) == 0);
    for (int64_t j0 = 4 * (blockIdx.x * (int64_t)blockDim.x + threadIdx.x); j0 < cp; j0 += 4 * (int64_t)gridDim.x * blockDim.x) {
        double v[4] = {0.0, 0.0, 0.0, 0.0};
        if (i < c && j0 + 3 >= i && j0 < c) {
            float hv[4] = {0.0f, 0.0f, 0.0f, 0.0f};
            if (vec && j0 + 3 < c) {
                const float4 x = LQ_AT(reinterpret_cast<const float4*>(H + i * ldh + j0));
                hv[0] = x.x; hv[1] = x.y; hv[2] = x.z; hv[3] = x.w;
            } else {
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    if (j0 + e < c) hv[e] = LQ_AT(H + i * ldh + j0 + e);
            }
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int64_t j = j0 + e;
                if (j < c && j >= i) {
                    if (!isfinite(hv[e])) lq_report(st, LQ_ERR_NONFINITE, i * c + j);
                    v[e] = static_cast<double>(hv[e]);
                    if (i == j) v[e] = (hv[e] == 0.0f ? 1.0 : v[e]) + damp;
                }
            }
        }
        if (i >= c && i >= j0 && i < j0 + 4) v[i - j0] = 1.0;        // identity on the padding
        double2* out = reinterpret_cast<double2*>(A + i * cp + j0);  // cp is a multiple of 128
        LQ_AT(out) = make_double2(v[0], v[1]);
        LQ_AT(out + 1) = make_double2(v[2], v[3]);
    }
}

// ------------------------------------------------------------------ FP64 MMA -------
__device__ __forceinline__ void dmma(double& c0, double& c1, double a, double b) {
    asm volatile("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0, %1}, {%2}, {%3}, {%0, %1};"
                 : "+d"(c0), "+d"(c1) : "d"(a), "d"(b));
}
__device__ __forceinline__ void cp_async16(void* smem_dst, const void* gsrc) {
    const uint32_t d = static_cast<uint32_t>(__cvta_generic_to_shared(smem_dst));
    if (!LQ_DBG_OK(gsrc, 16) || !LQ_DBG_OK(smem_dst, 16)) return;       // debug build: a copy outside the registered buffers is skipped
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(gsrc) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// Programmatic dependent launch along the serial chain: a kernel launched with launch_chained() may be placed on the
// SMs while its predecessor in the stream still runs; it calls chain_wait() before it touches anything the predecessor
// wrote (the wait returns when the predecessor has completed and its writes are visible).  chain_release() in the
// predecessor says that the successor's CTAs may be placed from now on; without it they are placed when the
// predecessor ends.  In a kernel launched the plain way both are no-ops.
__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void chain_release() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// ------------------------------------------------------------ tile product, K = 128 --
// C[TM x TN] = beta * C + alpha * A[TM x 128] * op(B), all fp64 row-major, by 256 threads = 8 warps
// arranged WMW x (8 / WMW); each warp owns an (8 MI) x 32 patch as MI x 4 MMA tiles, so
// TM = 8 MI WMW and TN = 32 (8 / WMW).  NT: B is given as TN rows of K (C = A B^T), otherwise as
// K rows of TN.  K is streamed 16 at a time through a 3-stage cp.async ring; the shared-memory
// pitches make every fragment load conflict-free.  The output may alias B when the tile spans
// all of B's rows and columns that it reads (all of B has been read before the first store).
// Optional extra outputs: a plain copy (C2) and a transposed copy (Ct).
//   <4, 4, *>  128 x 64   the bulk of the updates (two CTAs per SM)
//   <2, 4, *>   64 x 64   panel and "next" tiles: short launches that sit on the critical path
//   <2, 8, *>  128 x 32   row scaling in place (a CTA owns whole columns)
constexpr int TK = 16, NST = 3;
constexpr int AP = 20;                       // pitch (doubles) of a K-major chunk row: 16 + 4
constexpr int GEMM_THREADS = 256;
constexpr int GEMM_SMEM = NST * (128 * AP + TK * (64 + 4)) * 8;     // the largest instantiation

struct TileOut {
    double* C;  int64_t ldc;
    double* C2; int64_t ldc2;     // optional copy of the result
    double* Ct; int64_t ldct;     // optional transposed copy: Ct[col * ldct + row]
};

template <int MI, int WMW, bool NT>
__device__ __forceinline__ void gemm_tile(const double* __restrict__ A, int64_t lda, const double* B, int64_t ldb,
                                          double alpha, double beta, const TileOut& o, double* smem) {
    constexpr int WNW = 8 / WMW;
    constexpr int TMR = 8 * MI * WMW, TNC = 32 * WNW;
    constexpr int BP = TNC + 4;                               // pitch of an N-major chunk row (NN form)
    constexpr int STAGE = TMR * AP + (NT ? TNC * AP : TK * BP);
    static_assert(NST * STAGE * 8 <= GEMM_SMEM, "shared memory");
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int wm = warp / WNW, wn = warp % WNW;
    const int fr = lane >> 2, fk = lane & 3;

    auto issue = [&](int kc) {
        double* as = smem + (kc % NST) * STAGE;
        double* bs = as + TMR * AP;
#pragma unroll
        for (int u = 0; u < TMR * 8 / GEMM_THREADS; ++u) {
            const int idx = tid + GEMM_THREADS * u, row = idx >> 3, seg = idx & 7;
            cp_async16(as + row * AP + seg * 2, A + (int64_t)row * lda + kc * TK + seg * 2);
        }
        if (NT) {
#pragma unroll
            for (int u = 0; u < TNC * 8 / GEMM_THREADS; ++u) {
                const int idx = tid + GEMM_THREADS * u, row = idx >> 3, seg = idx & 7;
                cp_async16(bs + row * AP + seg * 2, B + (int64_t)row * ldb + kc * TK + seg * 2);
            }
        } else {
            constexpr int SEGS = TNC / 2;                     // 16-byte pieces per row
#pragma unroll
            for (int u = 0; u < TK * SEGS / GEMM_THREADS; ++u) {
                const int idx = tid + GEMM_THREADS * u, row = idx / SEGS, seg = idx % SEGS;
                cp_async16(bs + row * BP + seg * 2, B + (int64_t)(kc * TK + row) * ldb + seg * 2);
            }
        }
    };

    double acc[MI][4][2];
#pragma unroll
    for (int i = 0; i < MI; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j][0] = acc[i][j][1] = 0.0;

    constexpr int NCHUNK = NB / TK;
    issue(0); cp_async_commit();
    issue(1); cp_async_commit();
#pragma unroll 1
    for (int kc = 0; kc < NCHUNK; ++kc) {
        cp_async_wait<NST - 2>();
        __syncthreads();
        if (kc + NST - 1 < NCHUNK) issue(kc + NST - 1);
        cp_async_commit();
        const double* as = smem + (kc % NST) * STAGE + (wm * 8 * MI + fr) * AP + fk;
        const double* bs = smem + (kc % NST) * STAGE + TMR * AP + (NT ? (wn * 32 + fr) * AP + fk : fk * BP + wn * 32 + fr);
#pragma unroll
        for (int kk = 0; kk < TK / 4; ++kk) {
            double a[MI], b[4];
#pragma unroll
            for (int i = 0; i < MI; ++i) a[i] = as[8 * i * AP + kk * 4];
#pragma unroll
            for (int j = 0; j < 4; ++j) b[j] = NT ? bs[8 * j * AP + kk * 4] : bs[kk * 4 * BP + 8 * j];
#pragma unroll
            for (int i = 0; i < MI; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) dmma(acc[i][j][0], acc[i][j][1], a[i], b[j]);
        }
    }
    cp_async_wait<0>();
    __syncthreads();      // every thread's copies have landed: B may now be overwritten

#pragma unroll
    for (int i = 0; i < MI; ++i) {
        const int row = wm * 8 * MI + 8 * i + fr;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int col = wn * 32 + 8 * j + 2 * fk;
            double2 v;
            v.x = alpha * acc[i][j][0];
            v.y = alpha * acc[i][j][1];
            double* cp = o.C + (int64_t)row * o.ldc + col;
            if (beta != 0.0) {
                const double2 old = LQ_AT(reinterpret_cast<const double2*>(cp));
                v.x += beta * old.x;
                v.y += beta * old.y;
            }
            LQ_AT(reinterpret_cast<double2*>(cp)) = v;
            if (o.C2) LQ_AT(reinterpret_cast<double2*>(o.C2 + (int64_t)row * o.ldc2 + col)) = v;
            if (o.Ct) {
                LQ_AT(o.Ct + (int64_t)col * o.ldct + row) = v.x;
                LQ_AT(o.Ct + (int64_t)(col + 1) * o.ldct + row) = v.y;
            }
        }
    }
}

// Step k, panel.  Blocks [0, 4k): 64 x 64 tiles of P_i = A[i][k] V_k^T (to Pbuf: this step's 128 columns of the
// outer block's panel buffer, row stride ldp; and transposed into Q's columns of block i).  Blocks [4k, 4(nblk-1)): 128 x 32 tiles of the row scaling
// A[k][j] <- V_k A[k][j] for j > k (in place: these are final entries of U) with a copy in Q's
// columns of block j.  Q is 128 x cp: the right-hand operand of the step's update for every
// block column.
__global__ void __launch_bounds__(GEMM_THREADS, 2)
panel_kernel(double* __restrict__ A, int64_t cp, int k, double* __restrict__ Pbuf, int64_t ldp, double* __restrict__ Q) {
    extern __shared__ double smem[];
    const int t = blockIdx.x >> 2, q = blockIdx.x & 3;
    chain_wait();                                       // launched behind the diagonal kernel of this step
    const double* Vk = A + (int64_t)k * NB * cp + (int64_t)k * NB;
    TileOut o = {};
    if (t < k) {
        const int i = t, mh = q >> 1, h = q & 1;
        o.C = Pbuf + ((int64_t)i * NB + mh * 64) * ldp + h * 64; o.ldc = ldp;
        o.Ct = Q + (int64_t)(h * 64) * cp + (int64_t)i * NB + mh * 64; o.ldct = cp;
        gemm_tile<2, 4, true>(A + ((int64_t)i * NB + mh * 64) * cp + (int64_t)k * NB, cp, Vk + (int64_t)(h * 64) * cp, cp, 1.0,
                              0.0, o, smem);
    } else {
        const int j = t + 1;
        double* row = A + (int64_t)k * NB * cp + (int64_t)j * NB + q * 32;
        o.C = row; o.ldc = cp;
        o.C2 = Q + (int64_t)j * NB + q * 32; o.ldc2 = cp;
        gemm_tile<2, 8, false>(Vk, cp, row, cp, 1.0, 0.0, o, smem);
    }
}

// Step k, eager update of tiles (i, j), i < k: A[i][j] -= P_i Q[:, j] (A[i][k] = -P_i V_k).  A launch covers the
// block rows i_base + blockIdx.y and the block columns j_base + (blockIdx.x >> 1) (128 x 64 tiles).  The tiles of
// block column k-1 and of block row k-1 are all that step k-1's diagonal and panel kernels read, so they can be
// updated first ("next") and the remainder ("rest") left to run beside step k-1.  With a look-ahead of two steps the
// tiles of block row and column k-2 ("next2") leave the rest as well, so that step k-1's "next" update waits for a
// short launch only and the rest of step k has two chain steps to finish:
//   part 0: every tile of the launch;  part 2: all but block row and block column k-1;
//   part 4: all but block rows and block columns k-1 and k-2;
//   part 1: next only, grid 4 nblk x 1, 64 x 64 tiles -- block tile t < k is (t, k-1), t >= k is (k-1, t);
//   part 3: next2 only, same grid -- block tile t < k-1 is (t, k-2), t >= k is (k-2, t) (tile (k-2, k-1) belongs to next);
//   part 5: next without the diagonal tile (k-1, k-1), which crit_kernel has updated already.
__global__ void __launch_bounds__(GEMM_THREADS, 2)
update_kernel(double* __restrict__ A, int64_t cp, int k, int part, int i_base, int j_base, const double* __restrict__ Pbuf,
              int64_t ldp, const double* __restrict__ Q) {
    extern __shared__ double smem[];
    int i, j, r0, c0;
    if (part == 1 || part == 3 || part == 5) {
        const int t = blockIdx.x >> 2;
        const int nx = part == 3 ? k - 2 : k - 1;         // the block row and column this launch brings up to date
        if (part == 3 && t == k - 1) return;
        if (part == 5 && t == k - 1) return;              // the diagonal tile was updated by crit_kernel
        if (t <= nx) { i = t; j = nx; } else { i = nx; j = t; }
        r0 = ((blockIdx.x >> 1) & 1) * 64;
        c0 = (blockIdx.x & 1) * 64;
    } else if (part >= 10) {
        // parts 0 and 2 of the deferred sweep in one launch (part - 10): first the block rows [i_base, k) (part 2:
        // [i_base, k-1)) over the whole width, one grid row each; then the block rows [0, i_base) over the j_base block
        // columns of the outer block, packed into grid rows of the same width
        const int o_lo = i_base, obw = j_base;
        const int nA = k - o_lo - (part == 12 ? 1 : 0);
        if (static_cast<int>(blockIdx.y) < nA) {
            i = o_lo + blockIdx.y;
            j = blockIdx.x >> 1;
            c0 = (blockIdx.x & 1) * 64;
        } else {
            const int64_t lin = static_cast<int64_t>(blockIdx.y - nA) * gridDim.x + blockIdx.x;
            i = static_cast<int>(lin / (2 * obw));
            if (i >= o_lo) return;
            const int xx = static_cast<int>(lin - static_cast<int64_t>(i) * (2 * obw));
            j = o_lo + (xx >> 1);
            c0 = (xx & 1) * 64;
        }
        if (part == 12 && (j == k - 1 || i == k - 1)) return;
        r0 = 0;
    } else {
        j = j_base + (blockIdx.x >> 1);
        i = i_base + blockIdx.y;
        if (part >= 2 && (j == k - 1 || i == k - 1)) return;
        if (part == 4 && (j == k - 2 || i == k - 2)) return;
        r0 = 0;
        c0 = (blockIdx.x & 1) * 64;
    }
    if (j < i) return;                                  // strictly lower tiles of the symmetric part
    if (part == 1) chain_release();                     // the next step's diagonal kernel may take its SM now; it waits for this launch to end
    const double* Pi = Pbuf + ((int64_t)i * NB + r0) * ldp;
    TileOut o = {};
    o.C = A + ((int64_t)i * NB + r0) * cp + (int64_t)j * NB + c0; o.ldc = cp;
    // A[i][k] = -P_i V_k;  A[i][j] -= P_i Q[:, j] otherwise
    const double* Bsrc = (j == k) ? A + (int64_t)k * NB * cp + (int64_t)k * NB + c0 : Q + (int64_t)j * NB + c0;
    const double beta = (j == k) ? 0.0 : 1.0;
    if (part == 1 || part == 3 || part == 5) gemm_tile<2, 4, false>(Pi, ldp, Bsrc, cp, -1.0, beta, o, smem);
    else gemm_tile<4, 4, false>(Pi, ldp, Bsrc, cp, -1.0, beta, o, smem);
}

// Step k, the one tile the next diagonal block waits for.  phase 0: P' = A[k-1][k] V_k^T (the panel tile of block row
// k-1, into the scratch Pc, 128 x 128); phase 1: A[k-1][k-1] -= P' P'^T.  Four CTAs of 64 x 64 each: they find free
// places on the SMs at once, where the panel and "next" launches (over a hundred CTAs) queue behind the bulk update.
// The panel launch computes the same P' again for everybody else.
__global__ void __launch_bounds__(GEMM_THREADS, 2)
crit_kernel(double* __restrict__ A, int64_t cp, int k, int phase, double* __restrict__ Pc) {
    extern __shared__ double smem[];
    chain_wait();
    const int mh = blockIdx.x >> 1, hh = blockIdx.x & 1;
    TileOut o = {};
    if (phase == 0) {
        const double* Vk = A + (int64_t)k * NB * cp + (int64_t)k * NB;
        o.C = Pc + (int64_t)(mh * 64) * NB + hh * 64; o.ldc = NB;
        gemm_tile<2, 4, true>(A + ((int64_t)(k - 1) * NB + mh * 64) * cp + (int64_t)k * NB, cp, Vk + (int64_t)(hh * 64) * cp, cp, 1.0, 0.0, o, smem);
    } else {
        o.C = A + ((int64_t)(k - 1) * NB + mh * 64) * cp + (int64_t)(k - 1) * NB + hh * 64; o.ldc = cp;
        gemm_tile<2, 4, true>(Pc + (int64_t)(mh * 64) * NB, NB, Pc + (int64_t)(hh * 64) * NB, NB, -1.0, 1.0, o, smem);
    }
}

// ------------------------------------------------ deferred update: operands as digit slices ----
// x = 2^e (d_1 2^-8 + d_2 2^-16 + ... + d_S 2^-8S) + remainder, with integer digits |d_s| <= 128 and e such that
// |x| 2^-e <= 1/2 for every entry of the row: slice s holds d_s 2^-8s as bf16 (exact).
constexpr int OBB = 8;                   // block columns per outer block
constexpr int LDP = LQ_DIGIT_LD;         // row stride of the panel buffer and of the slices
static_assert(LDP == OBB * NB, "an outer block is one row of digits");
constexpr int NSL = 5;                   // slices
constexpr int64_t BAND = 8192;           // rows of the deferred region handled per product

__device__ __forceinline__ int exp_for(double mx) { return mx > 0.0 ? ilogb(mx) + 2 : 0; }

__device__ __forceinline__ void digits_of(double x, int e, __nv_bfloat16 (&d)[NSL]) {
    double rest = scalbn(x, 8 - e);                     // |rest| <= 128
    double w = 0.00390625;                              // 2^-8
#pragma unroll
    for (int s = 0; s < NSL; ++s) {
        const double q = rint(rest);
        d[s] = __float2bfloat16_rn(static_cast<float>(q * w));     // an integer of at most 8 bits times a power of two
        rest = (rest - q) * 256.0;
        w *= 0.00390625;
    }
}
// Rows [0, rows) of the panel buffer (K columns each): exponent and slices.  One CTA per row.
__global__ void __launch_bounds__(256)
slice_rows_kernel(const double* __restrict__ P, int64_t ldp, int K, int* __restrict__ ex, __nv_bfloat16* __restrict__ SL,
                  int64_t slice_rows) {
    __shared__ double red[8];
    const int64_t row = blockIdx.x;
    const double* p = P + row * ldp;
    double v[4];
    double mx = 0.0;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const int kx = threadIdx.x + 256 * u;
        v[u] = kx < K ? LQ_AT(p + kx) : 0.0;
        mx = fmax(mx, fabs(v[u]));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = mx;
    __syncthreads();
    mx = red[0];
#pragma unroll
    for (int w = 1; w < 8; ++w) mx = fmax(mx, red[w]);
    const int e = isfinite(mx) ? exp_for(mx) : 0;
    if (threadIdx.x == 0) LQ_AT(ex + row) = e;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const int kx = threadIdx.x + 256 * u;
        if (kx >= K) continue;
        __nv_bfloat16 d[NSL];
        digits_of(isfinite(v[u]) ? v[u] : 0.0, e, d);
#pragma unroll
        for (int s = 0; s < NSL; ++s) LQ_AT(SL + (s * slice_rows + row) * LDP + kx) = d[s];
    }
}

// Exponents of the columns j >= col0 of the K rows of A that start at row0 (the final rows of U of an outer block).
__global__ void __launch_bounds__(256)
col_exp_kernel(const double* __restrict__ A, int64_t cp, int64_t row0, int K, int64_t col0, int* __restrict__ ex) {
    // 32 columns per CTA, eight threads per column (each takes every eighth row), so that a column's K loads do not queue
    // behind one another in one thread
    __shared__ double part[8][32];
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const int64_t j = col0 + blockIdx.x * 32LL + tx;
    double mx = 0.0;
    if (j < cp)
        for (int kx = ty; kx < K; kx += 8) mx = fmax(mx, fabs(LQ_AT(A + (row0 + kx) * cp + j)));
    part[ty][tx] = mx;
    __syncthreads();
    if (ty == 0 && j < cp) {
#pragma unroll
        for (int q = 1; q < 8; ++q) mx = fmax(mx, part[q][tx]);
        LQ_AT(ex + j) = isfinite(mx) ? exp_for(mx) : 0;
    }
}

// Slices of those columns, transposed: SL[s][j][kx] = digit s of A[row0 + kx][j].  64 x 64 tiles through shared memory.
__global__ void __launch_bounds__(256)
slice_cols_kernel(const double* __restrict__ A, int64_t cp, int64_t row0, int K, int64_t col0, const int* __restrict__ ex,
                  __nv_bfloat16* __restrict__ SL, int64_t slice_rows) {
    __shared__ double tile[64][65];
    const int64_t j0 = col0 + (int64_t)blockIdx.x * 64;
    const int k0 = blockIdx.y * 64;
    for (int idx = threadIdx.x; idx < 64 * 64; idx += 256) {
        const int a = idx >> 6, b = idx & 63;            // row k0 + a, column j0 + b
        const int64_t j = j0 + b;
        tile[a][b] = (k0 + a < K && j < cp) ? LQ_AT(A + (row0 + k0 + a) * cp + j) : 0.0;
    }
    __syncthreads();
    for (int idx = threadIdx.x; idx < 64 * 64; idx += 256) {
        const int b = idx >> 6, a = idx & 63;            // output row j0 + b, position k0 + a
        const int64_t j = j0 + b;
        if (j >= cp || k0 + a >= K) continue;
        const double x = tile[a][b];
        __nv_bfloat16 d[NSL];
        digits_of(isfinite(x) ? x : 0.0, LQ_AT(ex + j), d);
#pragma unroll
        for (int s = 0; s < NSL; ++s) LQ_AT(SL + (s * slice_rows + j) * LDP + k0 + a) = d[s];
    }
}

// A[row0 + i][col0 + j] -= 2^(ex[row0 + i] + ex[col0 + j]) (Ta[i][col0 + j] + Tb[i][col0 + j]) over nrows x ncols entries;
// with `upper`, only the 128 x 128 blocks on or above the diagonal; columns [hole0, hole1) are left out.  Two columns per thread.
__global__ void __launch_bounds__(256)
apply_kernel(double* __restrict__ A, int64_t cp, const float* __restrict__ Ta, const float* __restrict__ Tb, int64_t ldt,
             const int* __restrict__ ex, int64_t row0, int64_t nrows, int64_t col0, int64_t ncols, int upper, int64_t hole0, int64_t hole1) {
    const int64_t i = blockIdx.y;
    const int64_t row = row0 + i;
    const int er = LQ_AT(ex + row);
    for (int64_t j2 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; 2 * j2 < ncols; j2 += (int64_t)gridDim.x * blockDim.x) {
        const int64_t col = col0 + 2 * j2;
        if ((upper && col / NB < row / NB) || (col >= hole0 && col < hole1)) continue;
        const float2 a = LQ_AT(reinterpret_cast<const float2*>(Ta + i * ldt + col));
        const float2 b = LQ_AT(reinterpret_cast<const float2*>(Tb + i * ldt + col));
        double2* ap = reinterpret_cast<double2*>(A + row * cp + col);
        double2 v = LQ_AT(ap);
        v.x -= scalbn(static_cast<double>(a.x) + static_cast<double>(b.x), er + LQ_AT(ex + col));
        v.y -= scalbn(static_cast<double>(a.y) + static_cast<double>(b.y), er + LQ_AT(ex + col + 1));
        LQ_AT(ap) = v;
    }
}

// --------------------------------------------------------- diagonal block kernel ----
// In place on the 128 x 128 diagonal block k of A: reads its upper triangle (symmetric positive
// definite), computes the upper R with block = R R^T and writes V = R^-1 (upper, zeros below)
// back.  One CTA of 256 threads.  The block is handled as 4 x 4 sub-blocks of
// 32 with the same sweep as the outer algorithm: warp 0 factorises and inverts a 32 x 32
// diagonal sub-block in registers (one row per lane), then all warps do the panel, update and
// scaling products with the FP64 MMA out of shared memory.
constexpr int SB = 32;
constexpr int DP = 132;          // pitch of the block in shared memory (conflict-free fragments)
constexpr int PP = 36;           // pitch of the panel buffer
constexpr int DIAG_THREADS = 256;
constexpr int DIAG_SMEM = (NB * DP + (NB - SB) * PP + 2 * SB + SB) * 8;

// 32 x 32 sub-block at S (pitch DP): upper triangle in, V = R^-1 out (upper, zeros below).
__device__ __forceinline__ void warp_factor_invert(double* S, double* colbuf, double* rinvb, int lane,
                                                   long long col_global, long long c_real, lq_dev_status* st) {
    double a[SB];
#pragma unroll
    for (int t = 0; t < SB; ++t) a[t] = (t >= lane) ? S[lane * DP + t] : 0.0;
    // R R^T factorisation, last column first; lane i holds row i.  The pivots form the one serial chain of the whole
    // stage: the entry that becomes the next pivot is updated and broadcast first, the other columns' updates follow
    // and fill the latency of that broadcast and of the next reciprocal square root.
    double d = __shfl_sync(0xffffffffu, a[SB - 1], SB - 1);
#pragma unroll
    for (int j = SB - 1; j >= 0; --j) {
        if (!(d > 0.0) || !isfinite(d)) {
            if (lane == 0 && col_global + j < c_real) lq_report(st, LQ_ERR_NOT_POSITIVE_DEFINITE, col_global + j);
            d = 1.0;
        }
        const double rinv = rsqrt(d);
        const double l = (lane < j) ? a[j] * rinv : ((lane == j) ? d * rinv : 0.0);   // R[i][j]; sqrt(d) on the diagonal
        a[j] = l;
        if (lane == j) rinvb[j] = rinv;
        double* cb = colbuf + (j & 1) * SB;
        cb[lane] = (lane < j) ? l : 0.0;
        __syncwarp();
        if (j > 0) {
            a[j - 1] = fma(-l, cb[j - 1], a[j - 1]);
            d = __shfl_sync(0xffffffffu, a[j - 1], j - 1);
        }
#pragma unroll
        for (int t = 0; t < j - 1; ++t) a[t] -= l * cb[t];            // meaningful for lane <= t
    }
    // R to shared memory (rows), then V = R^-1, lane i forming row i column by column.  Every finished entry V[i][t] is
    // pushed at once into the right-hand sides of all later columns (independent multiply-adds), so between one entry
    // and the next there is one multiply-add and the scaling -- fp64 operations take ~23 cycles each here, and summing
    // a column's terms only when its turn comes puts several of them in series.
#pragma unroll
    for (int t = 0; t < SB; ++t) S[lane * DP + t] = (t >= lane) ? a[t] : 0.0;
    __syncwarp();
    double v[SB];
#pragma unroll
    for (int j = 0; j < SB; ++j) v[j] = (lane == j) ? 1.0 : 0.0;          // right-hand sides, turned into V in place
#pragma unroll
    for (int t = 0; t < SB; ++t) {
        const double vt = (lane <= t) ? v[t] * rinvb[t] : 0.0;
        v[t] = vt;
#pragma unroll
        for (int j = t + 1; j < SB; ++j) v[j] = fma(-vt, S[t * DP + j], v[j]);
    }
    __syncwarp();
#pragma unroll
    for (int t = 0; t < SB; ++t) S[lane * DP + t] = v[t];
}

// 16 x 16 output patch, K = 32, out of shared memory.  a(r, t): left operand, row r of the patch;
// B is given either as rows of K (NT: Bt[n * ldb + t]) or as K rows (NN: Bn[t * ldb + n]).
template <bool NT>
__device__ __forceinline__ void patch16(const double* Ap, int lda, const double* Bp, int ldb, int lane, double (&acc)[2][2][2]) {
    const int fr = lane >> 2, fk = lane & 3;
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 2; ++j) acc[i][j][0] = acc[i][j][1] = 0.0;
#pragma unroll
    for (int kk = 0; kk < SB / 4; ++kk) {
        double a[2], b[2];
#pragma unroll
        for (int i = 0; i < 2; ++i) a[i] = Ap[(8 * i + fr) * lda + kk * 4 + fk];
#pragma unroll
        for (int j = 0; j < 2; ++j) b[j] = NT ? Bp[(8 * j + fr) * ldb + kk * 4 + fk] : Bp[(kk * 4 + fk) * ldb + 8 * j + fr];
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int j = 0; j < 2; ++j) dmma(acc[i][j][0], acc[i][j][1], a[i], b[j]);
    }
}

__global__ void __launch_bounds__(DIAG_THREADS, 1)
diag_block_kernel(double* __restrict__ A, int64_t cp, int64_t blk, int64_t c_real, lq_dev_status* st) {
    extern __shared__ double sm[];
    double* S = sm;                       // NB x DP
    double* Pb = S + NB * DP;             // (NB - SB) x PP
    double* colbuf = Pb + (NB - SB) * PP; // 2 x SB
    double* rinvb = colbuf + 2 * SB;      // SB
    double* base = A + blk * NB * cp + blk * NB;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int fr = lane >> 2, fk = lane & 3;
    constexpr int NW = DIAG_THREADS / 32;

    chain_wait();                                       // launched behind the previous step's "next" update
    for (int idx = tid; idx < NB * (NB / 2); idx += DIAG_THREADS) {
        const int row = idx >> 6, c2 = (idx & 63) * 2;
        cp_async16(S + row * DP + c2, base + (int64_t)row * cp + c2);
    }
    cp_async_commit();
    cp_async_wait<0>();
    __syncthreads();

#pragma unroll 1
    for (int kb = NB / SB - 1; kb >= 0; --kb) {
        const int c0 = kb * SB;
        const int right = NB - c0 - SB;               // columns to the right of this sub-block
        double* D = S + c0 * DP + c0;                 // diagonal sub-block
        if (warp == 0) warp_factor_invert(D, colbuf, rinvb, lane, blk * NB + c0, c_real, st);
        __syncthreads();
        // panel: Pb[m][q] = sum_t S[m][c0 + t] V[q][t]   (m < c0); row scaling: S[c0 + q][j] <- sum_t V[q][t] S[c0 + t][j]  (j > c0 + 32)
        {
            const int nP = (c0 / 16) * 2;
            const int nR = right / 8;
            for (int item = warp; item < nP + nR; item += NW) {
                if (item < nP) {
                    const int m0 = (item >> 1) * 16, q0 = (item & 1) * 16;
                    double acc[2][2][2];
                    patch16<true>(S + m0 * DP + c0, DP, D + q0 * DP, DP, lane, acc);
#pragma unroll
                    for (int i = 0; i < 2; ++i)
#pragma unroll
                        for (int j = 0; j < 2; ++j) {
                            double* p = Pb + (m0 + 8 * i + fr) * PP + q0 + 8 * j + 2 * fk;
                            p[0] = acc[i][j][0];
                            p[1] = acc[i][j][1];
                        }
                } else {
                    // one warp owns an 8-column strip over all 32 rows, so the in-place update is safe
                    const int j0 = c0 + SB + (item - nP) * 8;
                    double acc[4][2];
#pragma unroll
                    for (int i = 0; i < 4; ++i) acc[i][0] = acc[i][1] = 0.0;
#pragma unroll
                    for (int kk = 0; kk < SB / 4; ++kk) {
                        const double b = S[(c0 + kk * 4 + fk) * DP + j0 + fr];
#pragma unroll
                        for (int i = 0; i < 4; ++i) dmma(acc[i][0], acc[i][1], D[(8 * i + fr) * DP + kk * 4 + fk], b);
                    }
                    __syncwarp();
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        double* p = S + (c0 + 8 * i + fr) * DP + j0 + 2 * fk;
                        p[0] = acc[i][0];
                        p[1] = acc[i][1];
                    }
                }
            }
        }
        __syncthreads();
        // update of the rows above: 16 x 16 patches over the whole width
        {
            const int nRow = c0 / 16;
            for (int item = warp; item < nRow * 8; item += NW) {
                const int rg = item >> 3, cg = item & 7;
                const int m0 = rg * 16, n0 = cg * 16;
                double acc[2][2][2];
                double sign_old;
                if (n0 < c0) {
                    if (cg < rg) continue;                                   // symmetric part: upper patches only
                    patch16<true>(Pb + m0 * PP, PP, Pb + n0 * PP, PP, lane, acc);          // P_m P_n^T
                    sign_old = 1.0;
                } else if (n0 < c0 + SB) {
                    patch16<false>(Pb + m0 * PP, PP, D + (n0 - c0), DP, lane, acc);        // P_m V
                    sign_old = 0.0;
                } else {
                    patch16<false>(Pb + m0 * PP, PP, S + c0 * DP + n0, DP, lane, acc);     // P_m (scaled row)
                    sign_old = 1.0;
                }
#pragma unroll
                for (int i = 0; i < 2; ++i)
#pragma unroll
                    for (int j = 0; j < 2; ++j) {
                        double* p = S + (m0 + 8 * i + fr) * DP + n0 + 8 * j + 2 * fk;
                        p[0] = sign_old * p[0] - acc[i][j][0];
                        p[1] = sign_old * p[1] - acc[i][j][1];
                    }
            }
        }
        __syncthreads();
    }

    chain_release();                                    // the panel kernel's CTAs may be placed while the block is written back
    for (int idx = tid; idx < NB * (NB / 2); idx += DIAG_THREADS) {
        const int row = idx >> 6, c2 = (idx & 63) * 2;
        double2 v;
        v.x = (c2 >= row) ? S[row * DP + c2] : 0.0;
        v.y = (c2 + 1 >= row) ? S[row * DP + c2 + 1] : 0.0;
        LQ_AT(reinterpret_cast<double2*>(base + (int64_t)row * cp + c2)) = v;
    }
}

// U (fp32, c x c, upper, zeros below) and dinv[j] = sum_k U64[k][j]^2.  A CTA converts 256 rows of 32
// columns and leaves the sum of squares of its piece of every column in part[row chunk][column];
// dinv_kernel adds the pieces of a column in row order (a fixed order: the result is reproducible).
constexpr int FIN_ROWS = 256;
__global__ void __launch_bounds__(256)
finalize_kernel(const double* __restrict__ A, int64_t cp, int64_t c, float* __restrict__ U, int64_t ldu,
                double* __restrict__ part) {
    __shared__ double red[8][33];
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const int64_t j = (int64_t)blockIdx.x * 32 + tx;
    const int64_t i0 = (int64_t)blockIdx.y * FIN_ROWS;
    const int64_t i1 = i0 + FIN_ROWS < c ? i0 + FIN_ROWS : c;
    double s = 0.0;
    if (j < c) {
        // eight rows' reads in flight (one at a time, a column of 32 rows was 32 trips to the L2: 18 us at c = 512)
        for (int64_t ib = i0 + ty; ib < i1; ib += 64) {
            double u[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const int64_t i = ib + 8 * e;
                u[e] = (i < i1 && i <= j) ? LQ_AT(A + i * cp + j) : 0.0;
            }
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const int64_t i = ib + 8 * e;
                s = fma(u[e], u[e], s);
                if (i < i1) LQ_AT(U + i * ldu + j) = static_cast<float>(u[e]);
            }
        }
    }
    red[ty][tx] = s;
    __syncthreads();
    if (ty == 0 && j < c) {
        double t = 0.0;
#pragma unroll
        for (int w = 0; w < 8; ++w) t += red[w][tx];
        LQ_AT(part + (int64_t)blockIdx.y * c + j) = t;
    }
}
__global__ void dinv_kernel(const double* __restrict__ part, int64_t c, int n_chunks, float* __restrict__ dinv) {
    const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= c) return;
    double t = 0.0;
    for (int q = 0; q * (int64_t)FIN_ROWS <= j && q < n_chunks; ++q) t += LQ_AT(part + (int64_t)q * c + j);
    LQ_AT(dinv + j) = static_cast<float>(t);
}

// ------------------------------------------- outer blocks as digit products (wide matrices) ----
// Inside an outer block only its own 1024 x 1024 diagonal part goes through the steps diag / panel / update; everything else
// the block's steps do is three products with its inverse factor V, of inner dimension 1024, on the integer tensor cores:
//   P = A[above][block] V^T,   A[above][block] = -P V,   A[block][right] = V A[block][right]   (final rows of U).
// Six digits per operand (47 bits below the largest entry), 21 digit products; the two leading levels leave the tensor core as
// their exact int32 sums T1, T2, the rest as one fp32 sum T3, and x = 2^(ea + eb) (2^-16 T1 + 2^-24 T2 + T3).  One digit more than
// the far tiles get, because P is not a sum of terms of its own size: entries of V are up to sqrt(cond) times larger.  The
// columns of A and of V meet at an index t that carries the scale of feature t (A[i][t] ~ s_t, V[q][t] ~ 1 / s_t): both are
// balanced by a power of two 2^f(t) near sqrt(A[t][t]) before the digits are taken.
constexpr int NSW = 6;

// f(t) = floor(log2(A[t][t]) / 2) of the block's diagonal, before its steps overwrite it.
__global__ void shift_kernel(const double* __restrict__ D, int64_t cp, int K, int* __restrict__ f) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= K) return;
    const double x = LQ_AT(D + t * cp + t);
    LQ_AT(f + t) = x > 0.0 && isfinite(x) ? ilogb(x) >> 1 : 0;
}

// Rows src[row][0..K) (fp64, row stride ld), entry t times 2^(sign f(t)): exponent ex[row] and NSW digits.  One CTA per row.
__global__ void __launch_bounds__(256)
slice_rows_wide_kernel(const double* __restrict__ src, int64_t ld, int K, const int* __restrict__ f, int sign, int* __restrict__ ex,
                       uint8_t* __restrict__ SL, int64_t slice_bytes) {
    __shared__ double red[8];
    const int64_t row = blockIdx.x;
    const int t = 4 * threadIdx.x;
    double v[4] = {0.0, 0.0, 0.0, 0.0}, mx = 0.0;
    if (t < K) {
        const double2* p = reinterpret_cast<const double2*>(src + row * ld + t);
        const double2 a = LQ_AT(p), b = LQ_AT(p + 1);
        v[0] = a.x; v[1] = a.y; v[2] = b.x; v[3] = b.y;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            v[u] = scalbn(v[u], sign * LQ_AT(f + t + u));
            mx = fmax(mx, digit_mag(v[u]));
        }
    }
    mx = cta_max256(mx, red);
    const int e = isfinite(mx) ? exp_for8(mx) : 0;
    if (threadIdx.x == 0) LQ_AT(ex + row) = e;
    if (t < K) store_digits<NSW>(v, e, SL + row * LDP + t, slice_bytes);
}

__device__ __forceinline__ double wide_sum(int t1, int t2, float t3, int e) {
    return scalbn(fma(static_cast<double>(t1), 1.0 / 65536.0, fma(static_cast<double>(t2), 1.0 / 16777216.0, static_cast<double>(t3))), e);
}

// Rows of P out of their three sums (row stride LDP), straight into digits; ex[row] holds the exponent of the row's left operand
// and becomes that of P.  One CTA per row.
__global__ void __launch_bounds__(256)
slice_sums_kernel(const int* __restrict__ T1, const int* __restrict__ T2, const float* __restrict__ T3, int K, int* __restrict__ ex,
                  const int* __restrict__ eb, uint8_t* __restrict__ SL, int64_t slice_bytes) {
    __shared__ double red[8];
    const int64_t row = blockIdx.x;
    const int t = 4 * threadIdx.x;
    const int ea = LQ_AT(ex + row);
    double v[4] = {0.0, 0.0, 0.0, 0.0}, mx = 0.0;
    if (t < K) {
        const int4 a = LQ_AT(reinterpret_cast<const int4*>(T1 + row * LDP + t)), b = LQ_AT(reinterpret_cast<const int4*>(T2 + row * LDP + t));
        const float4 c = LQ_AT(reinterpret_cast<const float4*>(T3 + row * LDP + t));
        v[0] = wide_sum(a.x, b.x, c.x, ea + LQ_AT(eb + t));
        v[1] = wide_sum(a.y, b.y, c.y, ea + LQ_AT(eb + t + 1));
        v[2] = wide_sum(a.z, b.z, c.z, ea + LQ_AT(eb + t + 2));
        v[3] = wide_sum(a.w, b.w, c.w, ea + LQ_AT(eb + t + 3));
#pragma unroll
        for (int u = 0; u < 4; ++u) mx = fmax(mx, digit_mag(v[u]));
    }
    mx = cta_max256(mx, red);                         // its barrier also puts every thread's read of ex[row] before the write
    const int e = isfinite(mx) ? exp_for8(mx) : 0;
    if (threadIdx.x == 0) LQ_AT(ex + row) = e;
    if (t < K) store_digits<NSW>(v, e, SL + row * LDP + t, slice_bytes);
}

// dst[row][j] = sign * the sum of T1, T2, T3 at (row, j); ea by row, eb by column.  cols is a multiple of 128.
__global__ void __launch_bounds__(256)
store_sums_kernel(const int* __restrict__ T1, const int* __restrict__ T2, const float* __restrict__ T3, int64_t ldt, int64_t cols, double sign,
                  const int* __restrict__ ea, const int* __restrict__ eb, double* __restrict__ dst, int64_t ld) {
    const int64_t row = blockIdx.y;
    const int e = LQ_AT(ea + row);
    for (int64_t j = 4 * (blockIdx.x * (int64_t)blockDim.x + threadIdx.x); j < cols; j += 4 * (int64_t)gridDim.x * blockDim.x) {
        const int4 a = LQ_AT(reinterpret_cast<const int4*>(T1 + row * ldt + j)), b = LQ_AT(reinterpret_cast<const int4*>(T2 + row * ldt + j));
        const float4 c = LQ_AT(reinterpret_cast<const float4*>(T3 + row * ldt + j));
        double2 lo, hi;
        lo.x = sign * wide_sum(a.x, b.x, c.x, e + LQ_AT(eb + j));
        lo.y = sign * wide_sum(a.y, b.y, c.y, e + LQ_AT(eb + j + 1));
        hi.x = sign * wide_sum(a.z, b.z, c.z, e + LQ_AT(eb + j + 2));
        hi.y = sign * wide_sum(a.w, b.w, c.w, e + LQ_AT(eb + j + 3));
        double2* out = reinterpret_cast<double2*>(dst + row * ld + j);
        LQ_AT(out) = lo;
        LQ_AT(out + 1) = hi;
    }
}

// Launches a kernel of the chain so that it may be placed before its predecessor in the stream has ended (the kernel
// itself waits with chain_wait()).
template <typename... KArgs, typename... Args>
cudaError_t launch_chained(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr; cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

struct PrepLayout {
    int64_t nblk, cp, band;
    size_t scal, a, pbuf, q, ex, sl, ta, tb, total, panel_bytes;
};
PrepLayout prep_layout(int64_t c) {
    PrepLayout L;
    L.nblk = lq_ceil_div(c, NB);
    L.cp = L.nblk * NB;
    L.band = L.cp < BAND ? L.cp : BAND;
    size_t off = 0;
    L.scal = off; off += 256;
    L.a = off;    off += lq_align_up(static_cast<size_t>(L.cp) * L.cp * sizeof(double), 256);
    L.panel_bytes = lq_align_up(static_cast<size_t>(L.cp) * NB * sizeof(double), 256);
    L.pbuf = off; off += lq_align_up(static_cast<size_t>(L.cp) * LDP * sizeof(double), 256);   // the panels of one outer block
    L.q = off;    off += 4 * L.panel_bytes;            // Q of the last four steps: with a look-ahead of two steps the rest of step k+2's update may still read its Q while step k's is written
    L.ex = off;   off += lq_align_up(static_cast<size_t>(L.cp) * sizeof(int), 256);
    L.sl = off;   off += lq_align_up(static_cast<size_t>(NSL) * L.cp * LDP * sizeof(__nv_bfloat16), 256);
    L.ta = off;   off += lq_align_up(static_cast<size_t>(L.band) * L.cp * sizeof(float), 256);
    L.tb = off;   off += lq_align_up(static_cast<size_t>(L.band) * L.cp * sizeof(float), 256);
    L.total = off;
    return L;
}

int launch_apply(cudaStream_t st, double* A, int64_t cp, const float* Ta, const float* Tb, const int* ex, int64_t row0, int64_t nrows,
                 int64_t col0, int64_t ncols, int upper, int64_t hole0 = 0, int64_t hole1 = 0) {
    const unsigned gx = static_cast<unsigned>(lq_ceil_div(ncols / 2, 256) < 256 ? lq_ceil_div(ncols / 2, 256) : 256);
    apply_kernel<<<dim3(gx, static_cast<unsigned>(nrows)), 256, 0, st>>>(A, cp, Ta, Tb, cp, ex, row0, nrows, col0, ncols, upper, hole0, hole1);
    LQ_LAUNCH_CHECK();
    return LQ_OK;
}

// The updates that the steps of outer block [o_lo, o_hi] owe to the tiles outside its rows and columns:
//   A[i][j] -= sum_k P_i^(k) Q_j^(k)    for block rows i < o_lo and block columns j outside the outer block, j >= i,
// with Q_j^(k) = P_j^(k)^T left of the outer block (the Cholesky part) and the final row k of U right of it (the
// Gauss-Jordan part).  Both operands go through the digit slices; row bands of at most `band` rows at a time.
int deferred_update_bf16(lq_handle* h, cudaStream_t st, double* A, int64_t cp, int64_t o_lo, int64_t o_hi, const double* Pob, int* ex,
                         void* SL, float* Ta, float* Tb, int64_t band) {
    const int K = static_cast<int>((o_hi - o_lo + 1) * NB);
    const int64_t top = o_lo * NB;                     // rows [0, top) are updated
    const int64_t right0 = (o_hi + 1) * NB;            // columns [right0, cp) on the right of the outer block
    const int64_t n_right = cp - right0;
    __nv_bfloat16* sl = static_cast<__nv_bfloat16*>(SL);
    slice_rows_kernel<<<static_cast<unsigned>(top), 256, 0, st>>>(Pob, LDP, K, ex, sl, cp);
    LQ_LAUNCH_CHECK();
    if (n_right > 0) {
        col_exp_kernel<<<static_cast<unsigned>(lq_ceil_div(n_right, 32)), 256, 0, st>>>(A, cp, top, K, right0, ex);
        LQ_LAUNCH_CHECK();
        dim3 g(static_cast<unsigned>(lq_ceil_div(n_right, 64)), static_cast<unsigned>(lq_ceil_div(K, 64)));
        slice_cols_kernel<<<g, 256, 0, st>>>(A, cp, top, K, right0, ex, sl, cp);
        LQ_LAUNCH_CHECK();
    }
    // passes: the leading pair alone (exact), then the pairs of levels s + t = NSL + 1 down to 3, least significant first
    lq_tc_gemm_args lead = {};
    lead.A_all = lead.B_all = SL;
    lead.a_rows = lead.b_rows = static_cast<int64_t>(NSL) * cp;
    lead.lda = lead.ldb = LDP;
    lead.ldd = cp;
    lead.K = K;
    lead.alpha = 1.0f;
    lead.n_pass = 1;
    lead.seg_iters = 4;                                // 256 digit products per partial sum, far below 2^24
    lq_tc_gemm_args tail = lead;
    tail.seg_iters = 0;
    tail.n_pass = 0;
    tail.n_lvl = 0;
    tail.chunk_kb = 2;             // 128 of the inner dimension per segment: 5 x 128 x 2^14 < 2^24 per partial sum, exact in fp32
    int pair_s[LQ_TC_MAX_PASS], pair_t[LQ_TC_MAX_PASS];
    for (int lvl = NSL + 1; lvl >= 3; --lvl) {
        int cnt = 0;
        for (int sdig = 1; sdig <= NSL; ++sdig) {
            const int tdig = lvl - sdig;
            if (tdig < 1 || tdig > NSL) continue;
            pair_s[tail.n_pass] = sdig - 1;
            pair_t[tail.n_pass] = tdig - 1;
            ++tail.n_pass;
            ++cnt;
        }
        tail.lvl_npass[tail.n_lvl++] = cnt;
    }
    for (int64_t b0 = 0; b0 < top; b0 += band) {
        const int64_t b1 = b0 + band < top ? b0 + band : top;
        for (int side = 0; side < 2; ++side) {
            // side 0: columns [b0, top) with the tiles below the diagonal left out; side 1: columns [right0, cp)
            const int64_t col0 = side == 0 ? b0 : right0;
            const int64_t ncols = side == 0 ? top - b0 : n_right;
            if (ncols <= 0) continue;
            for (int which = 0; which < 2; ++which) {
                lq_tc_gemm_args g = which == 0 ? lead : tail;
                g.D = (which == 0 ? Ta : Tb) + col0;
                g.M = b1 - b0;
                g.N = ncols;
                g.upper_only = side == 0 ? 1 : 0;
                for (int ps = 0; ps < g.n_pass; ++ps) {
                    const int sd = which == 0 ? 0 : pair_s[ps], td = which == 0 ? 0 : pair_t[ps];
                    g.a_row_off[ps] = sd * cp + b0;
                    g.b_row_off[ps] = td * cp + col0;
                }
                int rc = lq_tc_gemm(h, st, g);
                if (rc) return rc;
            }
            int rc = launch_apply(st, A, cp, Ta, Tb, ex, b0, b1 - b0, col0, ncols, side == 0 ? 1 : 0);
            if (rc) return rc;
        }
    }
    return LQ_OK;
}

// ------------------------------------------------------------------ the sweep on wide matrices --
// The products of NS digits per operand, integer digits: levels s + t = 2 .. NS + 1.  The leading level, exact, has an output of
// its own (raw: the two leading ones, as int32), then the others, least significant first.
lq_tc_gemm_args digit_product(int ns, bool raw, const uint8_t* Aall, int64_t a_rows, int64_t a_slice, int64_t a0, const uint8_t* Ball,
                              int64_t b_rows, int64_t b_slice, int64_t b0, int64_t M, int64_t N, int K) {
    lq_tc_gemm_args g = {};
    g.A_all = Aall; g.a_rows = a_rows; g.lda = LDP;
    g.B_all = Ball; g.b_rows = b_rows; g.ldb = LDP;
    g.M = M; g.N = N; g.K = K;
    g.alpha = 1.0f;
    g.int8_ops = 1;
    g.chunk_kb = LDP / 128;        // a level is one segment: its int32 sums over the whole inner dimension are exact
    g.raw_out = raw ? 1 : 0;
    const int lead = raw ? 2 : 1;
    for (int i = 0; i < ns; ++i) {
        const int lvl = i < lead ? 2 + i : ns + 1 - (i - lead);
        int cnt = 0;
        for (int sd = 1; sd <= ns; ++sd) {
            const int td = lvl - sd;
            if (td < 1 || td > ns) continue;
            g.a_signed[g.n_pass] = g.b_signed[g.n_pass] = 1;
            g.a_row_off[g.n_pass] = (sd - 1) * a_slice + a0;
            g.b_row_off[g.n_pass] = (td - 1) * b_slice + b0;
            ++g.n_pass;
            ++cnt;
        }
        g.lvl_scale[g.n_lvl] = static_cast<float>(ldexp(1.0, -8 * lvl));
        g.lvl_npass[g.n_lvl++] = cnt;
    }
    return g;
}

// Block columns are taken in outer blocks of 8, last first.  Per outer block:
//   chain : its diagonal part D (1024 x 1024) through diag / panel / update -- 8 serial steps of a few tiles -> V
//   bulk  : digits of V, of the columns of A above D and of the rows right of it; P; then first the update of the next outer
//           block's diagonal part, after which the chain goes on with it; then A[above][block] = -P V, the final rows of U
//           right of D, and the update of all other tiles:  A[i][j] -= P_i Q_j,  Q = P^T left of the block, U right of it.
// The chain (0.55 ms per outer block, a dozen SMs for a few microseconds at a time) runs on the high-priority stream beside the
// bulk of the outer block before it; the persistent products of that time leave it SPARE_SMS SMs.
constexpr int SPARE_SMS = 16;
constexpr double CHAIN_SECONDS = 0.7e-3;      // so long the products leave SMs free
constexpr double DIGIT_OPS_RATE = 2.2e15;     // integer operations per second of those products (2.2 - 2.6 measured)

int wide_sweep(lq_handle* h, cudaStream_t st, double* A, int64_t cp, int64_t c, char* wsp, const PrepLayout& L) {
    const bool fork = h->aux != nullptr && h->chain != nullptr;
    cudaStream_t cs = fork ? h->chain : st, gs = fork ? h->aux : st;
    const int64_t n_ob = lq_ceil_div(L.nblk, OBB);
    double* Ql = reinterpret_cast<double*>(wsp + L.q);                         // step products of D: right operand ...
    double* Pl = reinterpret_cast<double*>(wsp + L.q + L.panel_bytes);         // ... and panel
    int* fsh = reinterpret_cast<int*>(wsp + L.q + 2 * L.panel_bytes);          // f(t), two outer blocks alternating
    int* evt = fsh + 2 * LDP;                                                  // exponents of the columns of V
    uint8_t* SL = reinterpret_cast<uint8_t*>(wsp + L.sl);                      // slice s of row i of the matrix: s cp + i
    uint8_t* VT = reinterpret_cast<uint8_t*>(wsp + L.pbuf);                    // slices of the columns of V: s 1024 + q
    const int64_t sl_bytes = cp * LDP, vt_bytes = static_cast<int64_t>(LDP) * LDP;
    int* ex = reinterpret_cast<int*>(wsp + L.ex);
    float* Ta = reinterpret_cast<float*>(wsp + L.ta);
    float* Tb = reinterpret_cast<float*>(wsp + L.tb);
    const int64_t t_elems = 2 * L.band * cp;                                   // Ta and Tb lie side by side
    static_assert(NSW <= 2 * NSL, "the slices' space is laid out for NSL slices of 16-bit digits");
    if (fork) {
        LQ_CUDA_TRY(cudaEventRecord(h->ev_fork, st));
        LQ_CUDA_TRY(cudaStreamWaitEvent(cs, h->ev_fork, 0));
        LQ_CUDA_TRY(cudaStreamWaitEvent(gs, h->ev_fork, 0));
    }
    double busy = 0.0;             // estimated time of the products issued since the chain was let go
    auto product = [&](lq_tc_gemm_args& g) {
        g.spare_sms = fork && busy < CHAIN_SECONDS ? SPARE_SMS : 0;
        busy += 2.0 * g.M * g.N * g.K * g.n_pass * (g.upper_only ? 0.5 : 1.0) * (g.tri ? 0.6 : 1.0) / DIGIT_OPS_RATE;
        return lq_tc_gemm(h, gs, g);
    };
    // the far tiles of rows [r0, r0 + nr) x columns [c0, c1) but [hole0, hole1), those below the diagonal left out
    auto far_tiles = [&](int64_t r0, int64_t nr, int64_t c0, int64_t c1, int64_t hole0, int64_t hole1, int K) {
        lq_tc_gemm_args g = digit_product(NSL, false, SL, NSW * cp, cp, r0, SL, NSW * cp, cp, c0, nr, c1 - c0 - (hole1 - hole0), K);
        g.D_first = Ta + c0;
        g.D = Tb + c0;
        g.ldd = cp;
        g.upper_only = c0 == r0 ? 1 : 0;
        g.hole_at = hole0 - c0;
        g.hole = hole1 - hole0;
        int rc = product(g);
        return rc ? rc : launch_apply(gs, A, cp, Ta, Tb, ex, r0, nr, c0, c1 - c0, g.upper_only, hole0, hole1);
    };
    for (int64_t m = n_ob - 1; m >= 0; --m) {
        const int64_t o_lo = m * OBB, o_hi = (o_lo + OBB < L.nblk ? o_lo + OBB : L.nblk) - 1;
        const int obw = static_cast<int>(o_hi - o_lo + 1), K = obw * NB;
        const int64_t top = o_lo * NB, right0 = top + K, n_right = cp - right0;
        double* D = A + top * cp + top;
        int* f = fsh + (m & 1) * LDP;
        // ---- chain
        if (m < n_ob - 1 && fork) LQ_CUDA_TRY(cudaStreamWaitEvent(cs, h->ev_next, 0));
        shift_kernel<<<static_cast<unsigned>(lq_ceil_div(K, 256)), 256, 0, cs>>>(D, cp, K, f);
        LQ_LAUNCH_CHECK();
        for (int k = obw - 1; k >= 0; --k) {
            LQ_CUDA_TRY(launch_chained(diag_block_kernel, dim3(1), dim3(DIAG_THREADS), DIAG_SMEM, cs, A, cp, o_lo + k, c, h->dstatus));
            if (obw == 1) break;
            LQ_CUDA_TRY(launch_chained(panel_kernel, dim3(static_cast<unsigned>(4 * (obw - 1))), dim3(GEMM_THREADS), GEMM_SMEM, cs, D, cp, k,
                                       Pl, static_cast<int64_t>(NB), Ql));
            if (k == 0) break;
            update_kernel<<<dim3(static_cast<unsigned>(2 * obw), static_cast<unsigned>(k)), GEMM_THREADS, GEMM_SMEM, cs>>>(
                D, cp, k, 0, 0, 0, Pl, static_cast<int64_t>(NB), Ql);
            LQ_LAUNCH_CHECK();
        }
        if (fork) {
            LQ_CUDA_TRY(cudaEventRecord(h->ev_rest, cs));
            LQ_CUDA_TRY(cudaStreamWaitEvent(gs, h->ev_rest, 0));
        }
        // ---- bulk: digits of V and of the columns above it
        busy = CHAIN_SECONDS;                                  // nothing runs beside these
        if (top + n_right > 0) {
            slice_rows_wide_kernel<<<static_cast<unsigned>(K), 256, 0, gs>>>(D, cp, K, f, 1, ex + top, SL + top * LDP, sl_bytes);
            LQ_LAUNCH_CHECK();
        }
        if (top > 0) {
            slice_rows_wide_kernel<<<static_cast<unsigned>(top), 256, 0, gs>>>(A + top, cp, K, f, -1, ex, SL, sl_bytes);
            LQ_LAUNCH_CHECK();
            // P, straight into digits
            const int64_t most = t_elems / (3 * LDP) / 256 * 256;
            for (int64_t r0 = 0; r0 < top; r0 += most) {
                const int64_t nr = top - r0 < most ? top - r0 : most;
                lq_tc_gemm_args g = digit_product(NSW, true, SL, NSW * cp, cp, r0, SL, NSW * cp, cp, top, nr, K, K);
                g.D_first = Ta; g.D_second = Ta + nr * LDP; g.D = Ta + 2 * nr * LDP;
                g.ldd = LDP;
                g.tri = 1;
                int rc = product(g);
                if (rc) return rc;
                slice_sums_kernel<<<static_cast<unsigned>(nr), 256, 0, gs>>>(
                    reinterpret_cast<const int*>(g.D_first), reinterpret_cast<const int*>(g.D_second), g.D, K, ex + r0, ex + top,
                    SL + r0 * LDP, sl_bytes);
                LQ_LAUNCH_CHECK();
            }
            // the next outer block's diagonal part first: the chain goes on with it
            const int64_t next = top - LDP;
            int rc = far_tiles(next, LDP, next, top, top, top, K);
            if (rc) return rc;
            if (fork) LQ_CUDA_TRY(cudaEventRecord(h->ev_next, gs));
            busy = 0.0;
            slice_cols_wide_kernel<NSW><<<static_cast<unsigned>(K / 32), SC_THREADS, 0, gs>>>(A + top * cp, cp, K, top, right0, nullptr, evt, nullptr, VT,
                                                                                             vt_bytes);
            LQ_LAUNCH_CHECK();
        }
        if (n_right > 0) {
            slice_cols_wide_kernel<NSW><<<static_cast<unsigned>(lq_ceil_div(n_right, 32)), SC_THREADS, 0, gs>>>(
                A + top * cp, cp, K, right0, cp, f, ex + right0, nullptr, SL + right0 * LDP, sl_bytes);
            LQ_LAUNCH_CHECK();
            // final rows of U right of D, and their digits for the far tiles
            const int64_t most = t_elems / (3 * LDP) / 256 * 256;
            for (int64_t j0 = 0; j0 < n_right; j0 += most) {
                const int64_t nc = n_right - j0 < most ? n_right - j0 : most;
                lq_tc_gemm_args g = digit_product(NSW, true, SL, NSW * cp, cp, top, SL, NSW * cp, cp, right0 + j0, K, nc, K);
                g.D_first = Ta; g.D_second = Ta + K * nc; g.D = Ta + 2 * K * nc;
                g.ldd = nc;
                g.tri = 3;
                int rc = product(g);
                if (rc) return rc;
                const unsigned gx = static_cast<unsigned>(lq_ceil_div(nc, 1024));
                store_sums_kernel<<<dim3(gx, static_cast<unsigned>(K)), 256, 0, gs>>>(
                    reinterpret_cast<const int*>(g.D_first), reinterpret_cast<const int*>(g.D_second), g.D, nc, nc, 1.0, ex + top,
                    ex + right0 + j0, A + top * cp + right0 + j0, cp);
                LQ_LAUNCH_CHECK();
            }
            if (top > 0) {
                slice_cols_wide_kernel<NSL><<<static_cast<unsigned>(lq_ceil_div(n_right, 32)), SC_THREADS, 0, gs>>>(
                    A + top * cp, cp, K, right0, cp, nullptr, ex + right0, nullptr, SL + right0 * LDP, sl_bytes);
                LQ_LAUNCH_CHECK();
            }
        }
        if (top > 0) {
            const int64_t most = t_elems / (3 * LDP) / 256 * 256;
            for (int64_t r0 = 0; r0 < top; r0 += most) {
                const int64_t nr = top - r0 < most ? top - r0 : most;
                lq_tc_gemm_args g = digit_product(NSW, true, SL, NSW * cp, cp, r0, VT, NSW * LDP, LDP, 0, nr, K, K);
                g.D_first = Ta; g.D_second = Ta + nr * LDP; g.D = Ta + 2 * nr * LDP;
                g.ldd = LDP;
                g.tri = 2;
                int rc = product(g);
                if (rc) return rc;
                store_sums_kernel<<<dim3(1, static_cast<unsigned>(nr)), 256, 0, gs>>>(
                    reinterpret_cast<const int*>(g.D_first), reinterpret_cast<const int*>(g.D_second), g.D, LDP, K, -1.0, ex + r0, evt,
                    A + r0 * cp + top, cp);
                LQ_LAUNCH_CHECK();
            }
            const int64_t left = top - LDP;                    // the rows of the next outer block have their square already
            for (int64_t r0 = 0; r0 < top;) {
                // while the chain runs, a band that ends about when it does: the next one gets the whole chip
                int64_t nr = L.band;
                if (fork && busy < CHAIN_SECONDS) {
                    const double per_row = 2.0 * (cp - K - r0) * K * 15 / DIGIT_OPS_RATE;
                    const int64_t fit = (static_cast<int64_t>((CHAIN_SECONDS - busy) / per_row) + 255) / 256 * 256;
                    if (fit < 1024) busy = CHAIN_SECONDS;      // too little to be a launch of its own
                    else if (fit < nr) nr = fit;
                }
                if (r0 < left && r0 + nr > left) nr = left - r0;
                if (r0 + nr > top) nr = top - r0;
                const int64_t c0 = r0 < left ? r0 : right0;
                int rc = c0 < cp ? far_tiles(r0, nr, c0, cp, r0 < left ? top : cp, r0 < left ? right0 : cp, K) : static_cast<int>(LQ_OK);
                if (rc) return rc;
                r0 += nr;
            }
        }
    }
    if (fork) {
        LQ_CUDA_TRY(cudaEventRecord(h->ev_join, gs));          // the last outer block's products followed the chain
        LQ_CUDA_TRY(cudaStreamWaitEvent(st, h->ev_join, 0));
    }
    return LQ_OK;
}

}  // namespace

extern "C" int lq_prepare_hinv_workspace(int64_t c, size_t* bytes) {
    if (!bytes || c <= 0) return LQ_ERR_INVALID_ARG;
    *bytes = prep_layout(c).total;
    return LQ_OK;
}

extern "C" int lq_prepare_hinv(lq_handle* h, void* stream, const float* H, int64_t c, int64_t ldh, float damp_frac,
                               float* U, int64_t ldu, float* dinv, void* W, int32_t w_dtype, int64_t r, int64_t ldw,
                               void* ws, size_t ws_bytes) {
    if (!h || !H || !U || !dinv || c <= 0 || ldh < c || ldu < c || !(damp_frac >= 0.0f)) return LQ_ERR_INVALID_ARG;
    if (W && (r <= 0 || ldw < c || (w_dtype != LQ_F32 && w_dtype != LQ_BF16))) return LQ_ERR_INVALID_ARG;
    const PrepLayout L = prep_layout(c);
    if (!ws || ws_bytes < L.total) return LQ_ERR_WORKSPACE_TOO_SMALL;
    if (reinterpret_cast<uintptr_t>(ws) & 255) return LQ_ERR_INVALID_ARG;
    if (L.nblk > 32767 || L.cp > 65535) return LQ_ERR_UNSUPPORTED;   // grid.y of the set-up and update launches; room for the column sums
    cudaStream_t st = static_cast<cudaStream_t>(stream);

    const int64_t nblk = L.nblk, cp = L.cp;
    char* wsp = static_cast<char*>(ws);
    double* scal = reinterpret_cast<double*>(wsp + L.scal);
    double* A = reinterpret_cast<double*>(wsp + L.a);

    {
        LQ_DBG_SCOPE(h, st);
        LQ_DBG_REG(H, (static_cast<size_t>(c - 1) * ldh + c) * sizeof(float));
        LQ_DBG_REG(U, (static_cast<size_t>(c - 1) * ldu + c) * sizeof(float));
        LQ_DBG_REG(dinv, static_cast<size_t>(c) * sizeof(float));
        if (W) LQ_DBG_REG(W, (static_cast<size_t>(r - 1) * ldw + c) * (w_dtype == LQ_F32 ? 4 : 2));
        LQ_DBG_REG(ws, L.total);
        LQ_DBG_COMMIT();
    }
    static lq_once_per_device attr_set;
    if (attr_set.first()) {
        LQ_CUDA_TRY(cudaFuncSetAttribute(diag_block_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, DIAG_SMEM));
        LQ_CUDA_TRY(cudaFuncSetAttribute(panel_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, GEMM_SMEM));
        LQ_CUDA_TRY(cudaFuncSetAttribute(update_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, GEMM_SMEM));
        LQ_CUDA_TRY(cudaFuncSetAttribute(crit_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, GEMM_SMEM));
    }

    diag_mean_kernel<<<1, 1024, 0, st>>>(H, c, ldh, static_cast<double>(damp_frac), scal);
    LQ_LAUNCH_CHECK();
    if (W) {
        dim3 g(static_cast<unsigned>(lq_ceil_div(c, 256)), static_cast<unsigned>(r < 64 ? r : 64));
        if (w_dtype == LQ_F32)
            zero_dead_columns_kernel<float><<<g, 256, 0, st>>>(H, c, ldh, static_cast<float*>(W), r, ldw);
        else
            zero_dead_columns_kernel<__nv_bfloat16><<<g, 256, 0, st>>>(H, c, ldh, static_cast<__nv_bfloat16*>(W), r, ldw);
        LQ_LAUNCH_CHECK();
    }
    {
        dim3 g(static_cast<unsigned>(lq_ceil_div(cp, 1024) < 32 ? lq_ceil_div(cp, 1024) : 32), static_cast<unsigned>(cp));
        load_damped_kernel<<<g, 256, 0, st>>>(H, c, ldh, scal, A, cp, h->dstatus);
        LQ_LAUNCH_CHECK();
    }

    // The sweep, outer block by outer block (last first).  Inside an outer block every step updates the rows and the
    // columns of the outer block at once (the "eager" tiles).  With an auxiliary stream, step k's diagonal and panel
    // kernels and the "next" part of its update stay on the caller's stream; the rest of the eager update goes to
    // the auxiliary stream and overlaps step k-1's diagonal and panel kernels.  When the outer block is complete,
    // all other tiles get its steps' updates in one product on the bf16 tensor cores (deferred_update).
    const bool defer = nblk > OBB && nblk >= h->prep_defer_min_blocks;
    const bool wide = defer && h->prep_slices_int8 != 0;
    if (wide) {
        int rc = wide_sweep(h, st, A, cp, c, wsp, L);
        if (rc) return rc;
    }
    cudaStream_t aux = h->aux;
    const bool fork = !wide && aux != nullptr && nblk > 2;
    // With the fork the sweep leaves the caller's stream: the chain goes to the handle's high-priority stream `cs`, the
    // bulk of the eager updates to the low-priority `aux`; the caller's stream joins again after the last step.
    cudaStream_t cs = fork ? h->chain : st;
    if (fork) {
        LQ_CUDA_TRY(cudaEventRecord(h->ev_fork, st));
        LQ_CUDA_TRY(cudaStreamWaitEvent(aux, h->ev_fork, 0));
        LQ_CUDA_TRY(cudaStreamWaitEvent(cs, h->ev_fork, 0));
    }
    double* Pob = reinterpret_cast<double*>(wsp + L.pbuf);
    // Small matrices are bound by the serial chain of diagonal blocks, not by the updates: they stay on the FP64 MMA
    // throughout (one outer block as wide as the matrix).
    const int64_t obb = defer ? OBB : nblk;
    if (defer && !wide) LQ_CUDA_TRY(cudaMemsetAsync(wsp + L.sl, 0, static_cast<size_t>(NSL) * cp * LDP * sizeof(__nv_bfloat16), cs));
    bool rest_pending = false, next2_pending = false;
    const bool deep = fork && !defer && h->mid != nullptr;
    const int64_t n_ob = wide ? 0 : lq_ceil_div(nblk, obb);
    if (deep) {
        // Nothing deferred (o_lo = 0): look-ahead of two steps, and only what the next diagonal block waits for on the chain.
        //   chain (highest priority): diagonal kernel of step k, then crit_kernel: the panel tile of block row k-1 and the
        //                             update of tile (k-1, k-1) -- the next diagonal block;
        //   middle stream           : panel of step k (after the diagonal kernel), "next" (block row and column k-1 but for
        //                             its diagonal tile; after crit_kernel, which read the tile (k-1, k) that "next"
        //                             overwrites), "next2" (block row and column k-2; after the rest of step k+1);
        //   low-priority stream     : the rest of step k (after the panel of step k and, in stream order, the rest of step k+1).
        // crit_kernel of step k waits for "next2" of step k+1 (and with it for "next" of step k+1 and the rest of step
        // k+2), which wrote the tiles it reads and updates.
        cudaStream_t mid = h->mid;
        LQ_CUDA_TRY(cudaStreamWaitEvent(mid, h->ev_fork, 0));
        double* Pc = reinterpret_cast<double*>(wsp + L.sl);          // 128 x 128 scratch of crit_kernel (the slices' space is free here)
        for (int64_t k = nblk - 1; k >= 0; --k) {
            double* Pk = Pob + (k & 3) * NB;
            double* Qk = reinterpret_cast<double*>(wsp + L.q + (k & 3) * L.panel_bytes);
            const int ki = static_cast<int>(k);
            LQ_CUDA_TRY(launch_chained(diag_block_kernel, dim3(1), dim3(DIAG_THREADS), DIAG_SMEM, cs, A, cp, k, c, h->dstatus));
            LQ_CUDA_TRY(cudaEventRecord(h->ev_diag, cs));
            if (k > 0) {
                if (next2_pending) LQ_CUDA_TRY(cudaStreamWaitEvent(cs, h->ev_next2, 0));
                next2_pending = false;
                crit_kernel<<<4, GEMM_THREADS, GEMM_SMEM, cs>>>(A, cp, ki, 0, Pc);
                LQ_LAUNCH_CHECK();
                LQ_CUDA_TRY(launch_chained(crit_kernel, dim3(4), dim3(GEMM_THREADS), GEMM_SMEM, cs, A, cp, ki, 1, Pc));
                LQ_CUDA_TRY(cudaEventRecord(h->ev_crit, cs));
            }
            LQ_CUDA_TRY(cudaStreamWaitEvent(mid, h->ev_diag, 0));
            panel_kernel<<<static_cast<unsigned>(4 * (nblk - 1)), GEMM_THREADS, GEMM_SMEM, mid>>>(A, cp, ki, Pk, LDP, Qk);
            LQ_LAUNCH_CHECK();
            if (k == 0) {
                LQ_CUDA_TRY(cudaEventRecord(h->ev_next2, mid));
                next2_pending = true;
                break;
            }
            if (k >= 3) LQ_CUDA_TRY(cudaEventRecord(h->ev_next, mid));       // the panel of step k is complete
            LQ_CUDA_TRY(cudaStreamWaitEvent(mid, h->ev_crit, 0));
            update_kernel<<<static_cast<unsigned>(4 * nblk), GEMM_THREADS, GEMM_SMEM, mid>>>(A, cp, ki, 5, 0, 0, Pk, LDP, Qk);
            LQ_LAUNCH_CHECK();
            if (k >= 2) {
                if (rest_pending) LQ_CUDA_TRY(cudaStreamWaitEvent(mid, h->ev_rest, 0));
                update_kernel<<<static_cast<unsigned>(4 * nblk), GEMM_THREADS, GEMM_SMEM, mid>>>(A, cp, ki, 3, 0, 0, Pk, LDP, Qk);
                LQ_LAUNCH_CHECK();
            }
            LQ_CUDA_TRY(cudaEventRecord(h->ev_next2, mid));
            next2_pending = true;
            if (k >= 3) {
                LQ_CUDA_TRY(cudaStreamWaitEvent(aux, h->ev_next, 0));
                dim3 g(static_cast<unsigned>(2 * nblk), static_cast<unsigned>(k - 2));
                update_kernel<<<g, GEMM_THREADS, GEMM_SMEM, aux>>>(A, cp, ki, 4, 0, 0, Pk, LDP, Qk);
                LQ_LAUNCH_CHECK();
                LQ_CUDA_TRY(cudaEventRecord(h->ev_rest, aux));
                rest_pending = true;
            }
        }
    } else
    for (int64_t m = n_ob - 1; m >= 0; --m) {
        const int64_t o_lo = m * obb;
        const int64_t o_hi = (o_lo + obb < nblk ? o_lo + obb : nblk) - 1;
        const int obw = static_cast<int>(o_hi - o_lo + 1);
        for (int64_t k = o_hi; k >= o_lo; --k) {
            // this step's 128 columns of the panel buffer: its place in the outer block, or one of four alternating
            // slots when nothing is deferred (the updates of the two steps before may still be reading theirs)
            double* Pk = Pob + (defer ? k - o_lo : (k & 3)) * NB;
            double* Qk = reinterpret_cast<double*>(wsp + L.q + (k & 3) * L.panel_bytes);
            const int ki = static_cast<int>(k);
            LQ_CUDA_TRY(launch_chained(diag_block_kernel, dim3(1), dim3(DIAG_THREADS), DIAG_SMEM, cs, A, cp, k, c, h->dstatus));
            if (nblk > 1) {
                LQ_CUDA_TRY(launch_chained(panel_kernel, dim3(static_cast<unsigned>(4 * (nblk - 1))), dim3(GEMM_THREADS), GEMM_SMEM, cs,
                                           A, cp, ki, Pk, LDP, Qk));
            }
            if (k == 0) break;
            // eager tiles of step k: block rows [o_lo, k) over the whole width, block rows [0, o_lo) over the
            // outer block's columns
            const int rows_in = static_cast<int>(k - o_lo);
            if (!fork || k == o_lo) {
                if (rest_pending) LQ_CUDA_TRY(cudaStreamWaitEvent(cs, h->ev_rest, 0));
                rest_pending = false;
                if (rows_in > 0 || o_lo > 0) {      // both regions in one launch: one partial round of CTAs instead of two
                    const int64_t rows_b = lq_ceil_div(o_lo * 2 * obw, 2 * nblk);
                    dim3 g(static_cast<unsigned>(2 * nblk), static_cast<unsigned>(rows_in + rows_b));
                    update_kernel<<<g, GEMM_THREADS, GEMM_SMEM, cs>>>(A, cp, ki, 10, static_cast<int>(o_lo), obw, Pk, LDP, Qk);
                    LQ_LAUNCH_CHECK();
                }
                continue;
            }
            if (rest_pending) LQ_CUDA_TRY(cudaStreamWaitEvent(cs, h->ev_rest, 0));     // step k+1's rest touched the same tiles
            update_kernel<<<static_cast<unsigned>(4 * nblk), GEMM_THREADS, GEMM_SMEM, cs>>>(A, cp, ki, 1, 0, 0, Pk, LDP, Qk);
            LQ_LAUNCH_CHECK();
            rest_pending = false;
            if (rows_in > 1 || o_lo > 0) {
                LQ_CUDA_TRY(cudaEventRecord(h->ev_next, cs));
                LQ_CUDA_TRY(cudaStreamWaitEvent(aux, h->ev_next, 0));
                {                              // block row k-1 is part of "next"; both regions in one launch
                    const int64_t rows_b = lq_ceil_div(o_lo * 2 * obw, 2 * nblk);
                    dim3 g(static_cast<unsigned>(2 * nblk), static_cast<unsigned>(rows_in - 1 + rows_b));
                    update_kernel<<<g, GEMM_THREADS, GEMM_SMEM, aux>>>(A, cp, ki, 12, static_cast<int>(o_lo), obw, Pk, LDP, Qk);
                    LQ_LAUNCH_CHECK();
                }
                LQ_CUDA_TRY(cudaEventRecord(h->ev_rest, aux));
                rest_pending = true;
            }
        }
        if (o_lo > 0) {
            if (rest_pending) LQ_CUDA_TRY(cudaStreamWaitEvent(cs, h->ev_rest, 0));
            rest_pending = false;
            int rc = deferred_update_bf16(h, cs, A, cp, o_lo, o_hi, Pob, reinterpret_cast<int*>(wsp + L.ex),
                                     wsp + L.sl, reinterpret_cast<float*>(wsp + L.ta),
                                     reinterpret_cast<float*>(wsp + L.tb), L.band);
            if (rc) return rc;
        }
    }
    if (rest_pending) LQ_CUDA_TRY(cudaStreamWaitEvent(cs, h->ev_rest, 0));
    if (next2_pending) LQ_CUDA_TRY(cudaStreamWaitEvent(cs, h->ev_next2, 0));
    if (fork) {
        LQ_CUDA_TRY(cudaEventRecord(h->ev_join, cs));
        LQ_CUDA_TRY(cudaStreamWaitEvent(st, h->ev_join, 0));
    }
    {
        // the panel buffers are free now: they hold the per-chunk column sums (c / 256 x c doubles <= 2 panels for c <= 65536)
        double* part = reinterpret_cast<double*>(wsp + L.pbuf);
        const int n_chunks = static_cast<int>(lq_ceil_div(c, FIN_ROWS));
        dim3 g(static_cast<unsigned>(lq_ceil_div(c, 32)), static_cast<unsigned>(n_chunks));
        finalize_kernel<<<g, 256, 0, st>>>(A, cp, c, U, ldu, part);
        LQ_LAUNCH_CHECK();
        dinv_kernel<<<static_cast<unsigned>(lq_ceil_div(c, 256)), 256, 0, st>>>(part, c, n_chunks, dinv);
        LQ_LAUNCH_CHECK();
    }
    return LQ_OK;
}

// ------------------------------------------------------------ diagonal of the factor --
namespace {
__global__ void chol_diag_kernel(const float* __restrict__ U, int64_t c, int64_t ldu, float* __restrict__ d) {
    const int64_t j = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (j < c) LQ_AT(d + j) = LQ_AT(U + j * ldu + j);
}
}  // namespace

extern "C" int lq_chol_diag(lq_handle* h, void* stream, const float* U, int64_t c, int64_t ldu, float* d) {
    if (!h || !U || !d || c <= 0 || ldu < c) return LQ_ERR_INVALID_ARG;
    {
        LQ_DBG_SCOPE(h, static_cast<cudaStream_t>(stream));
        LQ_DBG_REG(U, (static_cast<size_t>(c - 1) * ldu + c) * sizeof(float));
        LQ_DBG_REG(d, static_cast<size_t>(c) * sizeof(float));
        LQ_DBG_COMMIT();
    }
    chol_diag_kernel<<<static_cast<unsigned>(lq_ceil_div(c, 256)), 256, 0, static_cast<cudaStream_t>(stream)>>>(U, c, ldu, d);
    LQ_LAUNCH_CHECK();
    return LQ_OK;
}
