// Algorithm 2 (Appendix, "LeanQuant-Exact"): every row is quantised in its own greedy order with a
// full downdate of its own copy of the inverse Hessian (Eq. 3 for the weights, Eq. 9 for the inverse).
//
// One CTA per row, fp64 throughout (the decisions -- which weight next, which grid point -- must be
// those of a float64 evaluation).  The O(c^2) downdate of Eq. 9 is not applied after every step but every
// `nb` steps: the columns v_m taken out by the steps of the current batch stay in shared memory, the column
// that a step needs is
//     Hinv_now[:, i] = Hinv_batch_start[:, i] - sum_m v_m (v_m[i] / pivot_m),
// and a batch ends with one rank-nb update of the matrix, which cuts its memory traffic by nb.
// The diagonal, which the greedy choice reads at every step, is kept up to date separately.
//
// The rows' matrices do not fit the L2 (296 CTAs x 4.7 MB at c = 768), so their traffic is what bounds the kernel, and the
// layout is made for it.  The weights still to do are kept compact: a batch's update reads the upper triangle of the n
// weights that the batch started with and writes the one of the n - nb that are left, packed, into the other half of
// the row's slot (two packed triangles of c - 1 and fewer fill no more than c x c).  The shared memory for the batch's columns holds
// more of them as n falls: nb grows.  Together n^2 / 2 entries per batch instead of n c / 2 at a fixed nb: c^3 / 7 bytes
// per row and weight where the loop over all columns moved 2 c^3 / 7.  The first batch reads U^T U itself, which all rows share.
// The update itself runs on the FP64 MMA (a column of the batch is a step of K): an eighth of the instructions of the same
// multiply-adds, which were six tenths of the kernel's issue slots.  A step needs one barrier, and what it can do before its
// column has arrived it does: the pivot is the maintained diagonal, the batch's downdates are summed on their own.
// 768 x 768, 4 bits: 37.2 -> 19.8 ms (compaction 27.4, MMA and the shorter step 21.7, asking for strips ahead 20.5, bisection and
// one quantisation per offer 19.8); 23 GB of DRAM traffic per 296 rows where it was 50.  What is left is the latency of a
// step's column and three rounds of 296 rows for 768.
#include <cstdint>

#include "lq_common.cuh"

namespace {

constexpr int EX_THREADS = 256;
constexpr int EX_WARPS = EX_THREADS / 32;
constexpr int EX_MAX_NB = 32;

// Hinv = U^T U in fp64 from the fp32 upper factor (Hinv[i][j] = sum_{k <= min(i,j)} U[k][i] U[k][j])
__global__ void __launch_bounds__(1024) utu_kernel(const float* __restrict__ U, int64_t ldu, int64_t c, double* __restrict__ Hinv) {
    __shared__ double a[32][33], b[32][33];
    const int tx = threadIdx.x, ty = threadIdx.y;
    const int64_t i0 = static_cast<int64_t>(blockIdx.y) * 32, j0 = static_cast<int64_t>(blockIdx.x) * 32;
    const int64_t kend = min(min(i0, j0) + 32, c);
    double acc = 0.0;
    for (int64_t k0 = 0; k0 < kend; k0 += 32) {
        const int64_t k = k0 + ty;
        a[ty][tx] = (k < c && i0 + tx < c) ? static_cast<double>(U[k * ldu + i0 + tx]) : 0.0;
        b[ty][tx] = (k < c && j0 + tx < c) ? static_cast<double>(U[k * ldu + j0 + tx]) : 0.0;
        __syncthreads();
#pragma unroll 8
        for (int kk = 0; kk < 32; ++kk) acc = fma(a[kk][ty], b[kk][tx], acc);
        __syncthreads();
    }
    if (i0 + ty < c && j0 + tx < c) Hinv[(i0 + ty) * c + j0 + tx] = acc;
}

template <typename T>
__device__ __forceinline__ double ex_load(const T* p);
template <>
__device__ __forceinline__ double ex_load<float>(const float* p) { return static_cast<double>(*p); }
template <>
__device__ __forceinline__ double ex_load<__nv_bfloat16>(const __nv_bfloat16* p) { return static_cast<double>(__bfloat162float(*p)); }

struct ExactArgs {
    const void* W; int64_t ldw;
    const double* Hinv0;          // c x c
    double* slots;                // gridDim.x copies of c x c
    const float* grid;            // r x K (non-uniform)
    const float* scale; const int32_t* zero; int group, n_groups;       // affine
    uint8_t* codes;
    void* what; int what_bf16; int64_t ldwh;
    double* loss_rows;            // r
    lq_dev_status* dstatus;
    size_t slot_stride;           // doubles between two copies
    int64_t r; int c; int K;
    int vcap;                     // doubles of shared memory for the columns of a batch
};

// Nearest grid point by the midpoint rule (the number of midpoints strictly below w: found by bisection where they ascend,
// as fitted grids do), or quant_aff.
template <bool AFFINE>
__device__ __forceinline__ void ex_quant(double w, const double* __restrict__ gpts, const double* __restrict__ mids, bool ascending, int K,
                                         double S, double Z, int& code, double& q) {
    if (AFFINE) {
        double t = rint(w / S) + Z;
        t = fmin(fmax(t, 0.0), static_cast<double>(K - 1));
        code = static_cast<int>(t);
        q = (t - Z) * S;
    } else {
        int a = 0;
        if (ascending) {
            for (int h = K >> 1; h > 0; h >>= 1) a += (w > mids[a + h - 1]) ? h : 0;
        } else {
            for (int k = 0; k + 1 < K; ++k) a += (w > mids[k]) ? 1 : 0;
        }
        code = a;
        q = gpts[a];
    }
}

constexpr int EX_MAX_PER = 32;      // weights per thread at most
constexpr int EX_MAX_C = 7465;      // widest row: its values, diagonals and one column of a batch fill the shared memory
constexpr int EX_DONE = 0x8000;     // flag beside the name of a weight
static_assert(EX_MAX_C <= EX_THREADS * EX_MAX_PER && EX_MAX_C < EX_DONE, "positions");

// Distance of the batch's columns: 2 modulo 4, so that the 4 x 8 operand tiles of the MMA meet 32 different banks.
__host__ __device__ __forceinline__ int ex_pitch(int n) { return ((n + 1) & ~3) + 2; }
// Entries of the space that the list of old positions shares with the warps' coefficients.
__host__ __device__ __forceinline__ int ex_names(int c) {
    constexpr int least = EX_WARPS * EX_MAX_NB * 4;
    return c > least ? (c + 3) & ~3 : least;
}
__device__ __forceinline__ void ex_dmma(double& c0, double& c1, double a, double b) {
    asm volatile("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0, %1}, {%2}, {%3}, {%0, %1};"
                 : "+d"(c0), "+d"(c1) : "d"(a), "d"(b));
}

// Start of row p of the packed upper triangle of an n x n matrix, less p: entry (p, q) is at ex_row(p, n) + q.
__device__ __forceinline__ uint32_t ex_row(int p, int n) {
    return static_cast<uint32_t>(p) * static_cast<uint32_t>(n - 1) - static_cast<uint32_t>(p) * static_cast<uint32_t>(p - 1) / 2;
}

// Minimum over the warp of (score, position), smaller positions first among equal scores; a thread without a weight left
// has (INFINITY, 0x7fffffff).  On the order-preserving integer images: three 32-bit reductions.
struct ExBest { uint32_t hi, lo; int pos; };
__device__ __forceinline__ ExBest ex_key(double score, int pos) {
    const long long b = __double_as_longlong(score);
    const unsigned long long k = static_cast<unsigned long long>(b) ^ (b < 0 ? ~0ull : 0x8000000000000000ull);
    return {static_cast<uint32_t>(k >> 32), static_cast<uint32_t>(k), pos};
}
__device__ __forceinline__ ExBest ex_warp_min(ExBest x) {
    ExBest r;
    r.hi = __reduce_min_sync(0xffffffffu, x.hi);
    r.lo = __reduce_min_sync(0xffffffffu, x.hi == r.hi ? x.lo : 0xffffffffu);
    r.pos = __reduce_min_sync(0xffffffffu, x.hi == r.hi && x.lo == r.lo ? x.pos : 0x7fffffff);
    return r;
}

// PER: weights per thread (4 up to c = 1024: the column stays in registers; else EX_MAX_PER).
template <typename T, bool AFFINE, int PER>
__global__ void __launch_bounds__(EX_THREADS, 2) exact_row_kernel(ExactArgs A) {
    constexpr int UN = PER <= 4 ? PER : 4;
    extern __shared__ __align__(16) unsigned char ex_smem[];
    const int c = A.c, K = A.K;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    double* w = reinterpret_cast<double*>(ex_smem);          // c: the row, error-compensated as it goes (by position)
    double* d = w + c;                                       // c: diagonal of the current inverse
    double* V = d + c;                                       // A.vcap: the columns taken out in the current batch, vs apart
    double* rpiv = V + A.vcap;                               // EX_MAX_NB: reciprocals of their pivots
    double* gpts = rpiv + EX_MAX_NB;                         // 16, and the 15 midpoints between them
    double* mids = gpts + 16;
    double* coef = mids + 16 + warp * EX_MAX_NB;             // a step's  -v_m[i] / pivot_m, by every warp for itself
    uint16_t* old = reinterpret_cast<uint16_t*>(mids + 16);  // c, in the same place: position before the compaction
    uint16_t* id = old + ex_names(c);                        // c: the weight at a position, with EX_DONE once it is quantised
    __shared__ ExBest red[2][EX_WARPS];
    __shared__ double red_q[2][EX_WARPS];
    __shared__ int red_c[2][EX_WARPS];
    __shared__ int sh_cnt[EX_WARPS];

    double* slot = A.slots + static_cast<size_t>(blockIdx.x) * A.slot_stride;
    double* half[2] = {slot, slot + static_cast<size_t>(c) * (c - 1) / 2};
    // columns of a batch for n weights: what the space holds, whole steps of the MMA where it holds two or more
    auto batch = [&](int n) {
        const int most = min(EX_MAX_NB, A.vcap / ex_pitch(n));
        return most >= 8 ? most & ~3 : most;
    };

    for (int64_t row = blockIdx.x; row < A.r; row += gridDim.x) {
        const T* wp = static_cast<const T*>(A.W) + row * A.ldw;
        for (int j = tid; j < c; j += EX_THREADS) {
            w[j] = ex_load<T>(wp + j);
            d[j] = A.Hinv0[static_cast<size_t>(j) * c + j];
            id[j] = static_cast<uint16_t>(j);
        }
        if (!AFFINE && tid < K) {
            gpts[tid] = static_cast<double>(A.grid[row * K + tid]);
            if (tid + 1 < K) mids[tid] = 0.5 * (gpts[tid] + static_cast<double>(A.grid[row * K + tid + 1]));
        }
        __syncthreads();
        const bool ascending = __syncthreads_and(AFFINE || tid + 2 >= K || mids[tid] <= mids[tid + 1]) != 0;

        auto quant = [&](double x, int weight, int& code, double& q) {
            double S = 1.0, Z = 0.0;
            if (AFFINE) {
                const int64_t gi = row * A.n_groups + weight / A.group;
                S = static_cast<double>(A.scale[gi]);
                Z = static_cast<double>(A.zero[gi]);
            }
            ex_quant<AFFINE>(x, gpts, mids, ascending, K, S, Z, code, q);
        };

        int n = c;                                  // weights the current batch started with
        int vs = ex_pitch(n), nb = batch(n), kb = 0;
        const double* M = A.Hinv0;                  // their matrix: U^T U (square) in the first batch, a packed triangle later
        bool square = true;
        int to = 0;                                 // half of the slot that the next update writes
        double loss = 0.0;                          // kept by the first warp
        // a thread's best weight: loss error (q - w)^2 / (2 Hinv_ii), position, grid point and code.  j ascends within a thread:
        // first minimum.  A thread whose scores are all infinite or NaN offers its first weight, behind every finite score of
        // the others.
        double best = INFINITY, bq = 0.0;
        int bp = 0x7fffffff, bc = 0;
        auto offer = [&](int j, int weight, double wj, double dj) {
            int code;
            double q;
            quant(wj, weight, code, q);
            const double e = q - wj;
            const double sc = __ddiv_rn(__dmul_rn(e, e), 2.0 * dj);
            if (sc < best || bp == 0x7fffffff) { bp = j; bq = q; bc = code; }
            best = sc < best ? sc : best;
        };
        for (int j = tid; j < n; j += EX_THREADS) offer(j, j, w[j], d[j]);
        for (int step = 0; step < c; ++step) {
            const int par = step & 1;
            // (a) the weight with the least loss error among those still to do
            const ExBest mine = ex_warp_min(ex_key(best, bp));
            if (lane == 0) red[par][warp] = mine;
            if (bp == mine.pos) { red_q[par][warp] = bq; red_c[par][warp] = bc; }       // one lane: positions have one owner
            __syncthreads();
            const ExBest theirs = red[par][lane & (EX_WARPS - 1)];
            const int i = ex_warp_min(theirs).pos;
            const int from = __ffs(__ballot_sync(0xffffffffu, theirs.pos == i)) - 1;
            const double qi = red_q[par][from];
            const int code_i = red_c[par][from];
            // (b) column i of the current inverse: the stored matrix as of the start of the batch, minus the
            //     batch's downdates  sum_m v_m[j] v_m[i] / pivot_m, which are summed while the column is on its way
            const uint32_t row_i = square ? static_cast<uint32_t>(i) * c : ex_row(i, n);
            double vj[PER];
#pragma unroll UN
            for (int t = 0; t < PER; ++t) {
                const int j = tid + t * EX_THREADS;
                if (j >= n) break;
                vj[t] = 0.0;
                if (id[j] < EX_DONE) vj[t] = (square || j >= i) ? M[row_i + j] : M[ex_row(j, n) + i];      // U^T U is symmetric to the bit
            }
            const double dii = d[i], wi = w[i], rd = 1.0 / dii;
            if (lane < kb) coef[lane] = -(V[lane * vs + i] * rpiv[lane]);
            __syncwarp();
            const double err = wi - qi;
            if (warp == 0) loss += __ddiv_rn(__dmul_rn(err, err), 2.0 * dii);
            best = INFINITY;
            bp = 0x7fffffff;
            double acc[UN];
            if (PER <= 4) {
#pragma unroll
                for (int t = 0; t < UN; ++t) acc[t] = 0.0;
#pragma unroll 4
                for (int m = 0; m < kb; ++m) {
                    const double cm = coef[m];
#pragma unroll
                    for (int t = 0; t < UN; ++t) {
                        const int j = tid + t * EX_THREADS;
                        if (j < n) acc[t] = fma(cm, V[m * vs + j], acc[t]);
                    }
                }
            }
            // (c) quantise weight i, spread its error (Eq. 3), downdate the diagonal (Eq. 9), score what is left
#pragma unroll UN
            for (int t = 0; t < PER; ++t) {
                const int j = tid + t * EX_THREADS;
                if (j >= n) break;
                const int nj = id[j];
                double x = 0.0;
                if (j == i) {
                    x = dii;
                    id[i] = static_cast<uint16_t>(nj | EX_DONE);
                    rpiv[kb] = rd;
                    A.codes[row * c + nj] = static_cast<uint8_t>(code_i);
                    if (A.what) {
                        if (A.what_bf16) static_cast<__nv_bfloat16*>(A.what)[row * A.ldwh + nj] = __float2bfloat16_rn(static_cast<float>(qi));
                        else static_cast<float*>(A.what)[row * A.ldwh + nj] = static_cast<float>(qi);
                    }
                    if (!(dii > 0.0)) lq_report(A.dstatus, LQ_ERR_NOT_POSITIVE_DEFINITE, row * c + nj);
                } else if (nj < EX_DONE) {
                    double a = 0.0;
                    if (PER <= 4) a = acc[t % UN];
                    else for (int m = 0; m < kb; ++m) a = fma(coef[m], V[m * vs + j], a);
                    x = vj[t] + a;
                    const double g = x * rd;
                    const double wj = __dsub_rn(w[j], __dmul_rn(g, err));
                    const double dj = __dsub_rn(d[j], __dmul_rn(x, g));
                    w[j] = wj;
                    d[j] = dj;
                    offer(j, nj, wj, dj);
                }
                V[kb * vs + j] = x;
            }
            ++kb;
            // (d) end of a batch: Hinv[j][l] -= sum_m v_m[j] v_m[l] / pivot_m for the weights j <= l still to do, which move up
            if (kb < nb || step + 1 == c) continue;
            __syncthreads();
            {   // ascending list of the positions still to do
                const int per = (n + EX_THREADS - 1) / EX_THREADS;
                const int j_lo = min(tid * per, n), j_hi = min(j_lo + per, n);
                int cnt = 0;
                for (int j = j_lo; j < j_hi; ++j) cnt += id[j] < EX_DONE ? 1 : 0;
                int incl = cnt;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int y = __shfl_up_sync(0xffffffffu, incl, o);
                    if (lane >= o) incl += y;
                }
                if (lane == 31) sh_cnt[warp] = incl;
                __syncthreads();
                int base = incl - cnt;
                for (int x = 0; x < warp; ++x) base += sh_cnt[x];
                for (int j = j_lo; j < j_hi; ++j)
                    if (id[j] < EX_DONE) old[base++] = static_cast<uint16_t>(j);
                __syncthreads();
            }
            const int n2 = n - kb;
            double* out = half[to];
            // Each warp takes eight rows at a time and walks them in strips of 64 columns from the diagonal on.  Of the two
            // 8 x 8 tiles u of 16 columns, entry e of lane (fr, fk) is column fk + 4 u + 8 e of row fr: four lanes then read
            // and write a whole 32-byte sector.
            const int fr = lane >> 2, fk = lane & 3;
            for (int p = warp * 8; p < n2; p += EX_WARPS * 8) {
                const int pr = p + fr, o = old[min(pr, n2 - 1)];
                const double* hr = M + (square ? static_cast<uint32_t>(o) * c : ex_row(o, n));
                double* hw = out + ex_row(pr, n2);
                double a[EX_MAX_NB / 4];
#pragma unroll
                for (int s4 = 0; s4 < EX_MAX_NB / 4; ++s4) {
                    const int m = 4 * s4 + fk;
                    a[s4] = m < kb ? -(V[m * vs + o] * rpiv[m]) : 0.0;
                }
                // the strips are asked for ahead of their use (a line of 16 columns per lane): two strips ahead along the
                // rows, and the first two strips of the rows this warp takes next
                auto ask = [&](const double* base, int l) {
                    if (l < n2) asm volatile("prefetch.global.L2 [%0];" ::"l"(base + old[l]));
                };
                ask(hr, p + 64 + 16 * fk);
                {
                    const int pn = pr + EX_WARPS * 8;
                    if (pn < n2) {
                        const int on = old[pn];
                        const double* hn = M + (square ? static_cast<uint32_t>(on) * c : ex_row(on, n));
                        ask(hn, max(pn, pn - fr + 16 * fk));
                        ask(hn, pn - fr + 64 + 16 * fk);
                    }
                }
                for (int l0 = p; l0 < n2; l0 += 64) {
                    ask(hr, l0 + 128 + 16 * fk);
                    double x[8][2];
#pragma unroll
                    for (int u = 0; u < 8; ++u)
#pragma unroll
                        for (int e = 0; e < 2; ++e) {
                            const int l = l0 + 16 * (u >> 1) + fk + 4 * (u & 1) + 8 * e;
                            x[u][e] = (l < n2 && l >= pr) ? hr[old[l]] : 0.0;
                        }
                    const double* vb[8];
#pragma unroll
                    for (int u = 0; u < 8; ++u) {
                        const int l = l0 + 16 * (u >> 1) + (fr >> 1) + 4 * (u & 1) + 8 * (fr & 1);
                        vb[u] = V + (l < n2 ? old[l] : 0);
                    }
#pragma unroll
                    for (int s4 = 0; s4 < EX_MAX_NB / 4; ++s4) {
                        if (4 * s4 >= kb) break;
                        const int m = min(4 * s4 + fk, kb - 1);           // beyond the batch: a is zero, any entry will do
#pragma unroll
                        for (int u = 0; u < 8; ++u) ex_dmma(x[u][0], x[u][1], a[s4], vb[u][m * vs]);
                    }
#pragma unroll
                    for (int u = 0; u < 8; ++u)
#pragma unroll
                        for (int e = 0; e < 2; ++e) {
                            const int l = l0 + 16 * (u >> 1) + fk + 4 * (u & 1) + 8 * e;
                            if (l < n2 && l >= pr) hw[l] = x[u][e];
                        }
                }
            }
            // the weights left move up: their values, diagonals and names (a thread reads before any thread writes)
            for (int j0 = 0; j0 < n2; j0 += EX_THREADS) {
                const int j = j0 + tid;
                double wj = 0.0, dj = 0.0;
                uint16_t ij = 0;
                if (j < n2) { const int o = old[j]; wj = w[o]; dj = d[o]; ij = id[o]; }
                __syncthreads();                    // also: every warp is done with V and the matrix
                if (j < n2) { w[j] = wj; d[j] = dj; id[j] = ij; }
            }
            __syncthreads();
            M = out;
            square = false;
            to ^= 1;
            n = n2;
            vs = ex_pitch(n);
            nb = batch(n);
            kb = 0;
            best = INFINITY;
            bp = 0x7fffffff;
            for (int j = tid; j < n; j += EX_THREADS) offer(j, id[j], w[j], d[j]);
        }
        if (tid == 0) A.loss_rows[row] = loss;
        __syncthreads();
    }
}

__global__ void exact_loss_reduce_kernel(const double* __restrict__ rows, int64_t r, double* __restrict__ out) {
    __shared__ double part[256];
    double s = 0.0;
    for (int64_t k = threadIdx.x; k < r; k += 256) s += rows[k];      // fixed order per thread, fixed tree below
    part[threadIdx.x] = s;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if (threadIdx.x < o) part[threadIdx.x] += part[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) *out = part[0];
}

struct ExactPlan {
    int vcap;
    int slots;
    size_t smem;
    size_t off_hinv, off_slots, off_loss, total;
};

size_t exact_smem(int c, int vcap) {
    return (static_cast<size_t>(2) * c + vcap + EX_MAX_NB + 32) * sizeof(double) + static_cast<size_t>(ex_names(c) + c) * sizeof(uint16_t);
}

// Two CTAs per SM if that leaves at least 8 columns per batch, else one.  An SM has 228 KB of shared memory, of which each
// CTA takes 1 KB for the system and 416 bytes for the static arrays above.
int exact_plan(int64_t r, int64_t c, int sm_count, ExactPlan* P) {
    if (c > EX_MAX_C) return LQ_ERR_UNSUPPORTED;
    const int ci = static_cast<int>(c), vs = ex_pitch(ci);
    auto room = [&](size_t bytes) {
        const size_t rest = exact_smem(ci, 0);
        const int64_t most = static_cast<int64_t>(EX_MAX_NB) * vs, have = rest < bytes ? static_cast<int64_t>((bytes - rest) / sizeof(double)) : 0;
        return static_cast<int>(have < most ? have : most);
    };
    int per_sm = 2;
    P->vcap = room(114 * 1024 - 1440);
    if (P->vcap < 8 * vs) {
        per_sm = 1;
        P->vcap = room(220 * 1024);
        if (P->vcap < vs) return LQ_ERR_UNSUPPORTED;
    }
    P->smem = exact_smem(ci, P->vcap);
    const size_t mat = lq_align_up(static_cast<size_t>(c) * c * sizeof(double), 256);
    int64_t slots = static_cast<int64_t>(sm_count) * per_sm;
    if (slots > r) slots = r;
    const int64_t fit = static_cast<int64_t>((static_cast<size_t>(16) << 30) / mat);     // copies of the inverse: at most 16 GiB
    if (slots > fit) slots = fit < 1 ? 1 : fit;
    P->slots = static_cast<int>(slots);
    P->off_hinv = 0;
    P->off_slots = mat;
    P->off_loss = mat + static_cast<size_t>(P->slots) * mat;
    P->total = P->off_loss + lq_align_up(static_cast<size_t>(r) * sizeof(double), 256);
    return LQ_OK;
}

int check_cfg_exact(const lq_config* cfg) {
    if (!cfg) return LQ_ERR_INVALID_ARG;
    if (cfg->bits < 2 || cfg->bits > 4) return LQ_ERR_INVALID_ARG;
    if (cfg->grid_type != LQ_GRID_NONUNIFORM && cfg->grid_type != LQ_GRID_AFFINE) return LQ_ERR_INVALID_ARG;
    if (cfg->grid_type == LQ_GRID_AFFINE && cfg->group_size < 0) return LQ_ERR_INVALID_ARG;
    return LQ_OK;
}

}  // namespace

extern "C" int lq_quantize_exact_workspace(const lq_config* cfg, int64_t r, int64_t c, size_t* bytes) {
    int e = check_cfg_exact(cfg);
    if (e) return e;
    if (!bytes || r <= 0 || c <= 0) return LQ_ERR_INVALID_ARG;
    int dev = 0, sms = 0;
    LQ_CUDA_TRY(cudaGetDevice(&dev));
    LQ_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    ExactPlan P;
    e = exact_plan(r, c, sms, &P);
    if (e) return e;
    *bytes = P.total;
    return LQ_OK;
}

extern "C" int lq_quantize_exact(lq_handle* h, void* stream, const lq_config* cfg, const void* W, int32_t w_dtype, int64_t r,
                                 int64_t c, int64_t ldw, const float* U, int64_t ldu, const float* grid, const float* scale,
                                 const int32_t* zero, uint8_t* codes, void* W_hat, int32_t what_dtype, int64_t ldwh,
                                 double* loss_out, void* ws, size_t ws_bytes) {
    int e = check_cfg_exact(cfg);
    if (e) return e;
    if (!h || !W || !U || !codes || r <= 0 || c <= 0 || ldw < c || ldu < c) return LQ_ERR_INVALID_ARG;
    if (w_dtype != LQ_F32 && w_dtype != LQ_BF16) return LQ_ERR_INVALID_ARG;
    if (W_hat && (ldwh < c || (what_dtype != LQ_F32 && what_dtype != LQ_BF16))) return LQ_ERR_INVALID_ARG;
    const bool affine = cfg->grid_type == LQ_GRID_AFFINE;
    int group = 0, n_groups = 1;
    if (affine) {
        if (!scale || !zero) return LQ_ERR_INVALID_ARG;
        const int64_t g = cfg->group_size == 0 ? c : cfg->group_size;
        if (c % g) return LQ_ERR_INVALID_ARG;
        group = static_cast<int>(g);
        n_groups = static_cast<int>(c / g);
    } else if (!grid) {
        return LQ_ERR_INVALID_ARG;
    }
    ExactPlan P;
    e = exact_plan(r, c, h->sm_count, &P);
    if (e) return e;
    if (!ws || ws_bytes < P.total) return LQ_ERR_WORKSPACE_TOO_SMALL;
    if (reinterpret_cast<uintptr_t>(ws) & 255) return LQ_ERR_INVALID_ARG;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    char* wsp = static_cast<char*>(ws);
    double* Hinv0 = reinterpret_cast<double*>(wsp + P.off_hinv);

    {
        dim3 g(static_cast<unsigned>(lq_ceil_div(c, 32)), static_cast<unsigned>(lq_ceil_div(c, 32)));
        utu_kernel<<<g, dim3(32, 32), 0, st>>>(U, ldu, c, Hinv0);
        LQ_LAUNCH_CHECK();
    }
    ExactArgs A;
    A.W = W; A.ldw = ldw;
    A.Hinv0 = Hinv0;
    A.slots = reinterpret_cast<double*>(wsp + P.off_slots);
    A.grid = grid; A.scale = scale; A.zero = zero; A.group = group > 0 ? group : 1; A.n_groups = n_groups;
    A.codes = codes;
    A.what = W_hat; A.what_bf16 = (what_dtype == LQ_BF16); A.ldwh = ldwh;
    A.loss_rows = reinterpret_cast<double*>(wsp + P.off_loss);
    A.dstatus = h->dstatus;
    A.slot_stride = lq_align_up(static_cast<size_t>(c) * c * sizeof(double), 256) / sizeof(double);
    A.r = r; A.c = static_cast<int>(c); A.K = 1 << cfg->bits; A.vcap = P.vcap;

#define LQ_EXACT_LAUNCH_PER(TT, AFF, PER)                                                                                       \
    do {                                                                                                                      \
        LQ_CUDA_TRY(cudaFuncSetAttribute(exact_row_kernel<TT, AFF, PER>, cudaFuncAttributeMaxDynamicSharedMemorySize, 222 * 1024)); \
        exact_row_kernel<TT, AFF, PER><<<P.slots, EX_THREADS, P.smem, st>>>(A);                                               \
    } while (0)
#define LQ_EXACT_LAUNCH(TT, AFF)                                                                                              \
    do {                                                                                                                      \
        if (c <= 4 * EX_THREADS) LQ_EXACT_LAUNCH_PER(TT, AFF, 4);                                                             \
        else LQ_EXACT_LAUNCH_PER(TT, AFF, EX_MAX_PER);                                                                        \
    } while (0)
    if (w_dtype == LQ_F32) {
        if (affine) LQ_EXACT_LAUNCH(float, true); else LQ_EXACT_LAUNCH(float, false);
    } else {
        if (affine) LQ_EXACT_LAUNCH(__nv_bfloat16, true); else LQ_EXACT_LAUNCH(__nv_bfloat16, false);
    }
#undef LQ_EXACT_LAUNCH
#undef LQ_EXACT_LAUNCH_PER
    LQ_LAUNCH_CHECK();
    if (loss_out) {
        exact_loss_reduce_kernel<<<1, 256, 0, st>>>(A.loss_rows, r, loss_out);
        LQ_LAUNCH_CHECK();
    }
    return LQ_OK;
}
