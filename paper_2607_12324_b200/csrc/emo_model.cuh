// Pack modelling (Sec. 4.5): Eq. 6, a non-negative least-squares fit of every pack's feature vector by the
// micro-benchmarks' metric vectors, and Eq. 7, the pack's tables as the weighted sums of the micro-benchmarks'
// tables.  Included only by emo_lib.cu.
#pragma once
#include <cuda_runtime.h>

#include <cstdint>

constexpr int kModelMaxM = 16;       // micro-benchmarks (the paper uses 12)
constexpr size_t kModelMaxSmem = 48 * 1024;      // most bytes of metrics, tables and Gram matrix that a call may bring

struct ModelParams {
    int n_packs, n, m, L;
    const double *B;        // [n][m] metric matrix
    const double *feat;     // [n_packs][n]
    const double *Tb, *Eb;  // [m][L]
    double *x;              // [n_packs][m]
    double *T_out, *E_out;  // [n_packs][L]
    int32_t *status;
};

// Half a warp per pack, lane i for unknown i (m <= 16).  The Gram matrix G = B^T B is the same for all packs; every block builds
// it once in shared memory and then takes packs in turn.
//
// Active-set method of Lawson and Hanson on the normal equations: start from x = 0 with every variable held at
// zero; move the variable with the largest positive gradient component w = c - G x into the free set; solve
// the free set's equations G_PP z = c_P; while z has non-positive entries step from x towards z as
// far as feasibility allows and return the variables that reach zero to the held set; accept z; repeat until no
// gradient component is positive.  Every accepted x lowers the objective, so the loop ends; it is also bounded
// by 3 m outer and 3 m inner rounds (status -9 otherwise: never seen).
//
// The equations are never solved anew: the lanes keep the rows of the dictionary
//     basic_i = b_i - sum_j a_ij nonbasic_j        (x_i is basic where i is free, the residual r_i = (c - G x)_i where it is held)
// in registers, and a variable that changes sides is one principal pivot, m fused multiply-adds per lane with the pivot's row
// broadcast through shared memory.  b then holds z on the free set and w on the held one.  A dictionary of a symmetric matrix is
// symmetric up to the sign between free and held, which gives every lane its entry of the pivot column from the pivot's row.
// One step of iterative refinement against G at the end takes out what the pivots' roundings left (a_PP is the inverse of G_PP).
//
// Measured, 14 694 packs of 16 metrics, 12 unknowns and 32 levels: one thread per pack with a factorisation in local memory per
// step 500 us (115 blocks of four warps, every operand through L1); this one 48 us; 200 000 packs 0.42 ms (0.46 with a case for the pivot's row and
// column in every update: the selects were a third of its instructions).
constexpr int kModelThreads = 256, kModelRow = 18;      // scratch row of a pack: 16 entries and b, padded to keep two rows off each other's banks

__device__ __forceinline__ double emo_model_half_max(double v)
{
#pragma unroll
    for (int o = 8; o; o >>= 1) v = fmax(v, __shfl_xor_sync(0xFFFFFFFFu, v, o));
    return v;
}

__global__ void __launch_bounds__(kModelThreads, 3) emo_pack_model_kernel(ModelParams p)
{
    extern __shared__ __align__(16) double emo_model_smem[];
    __shared__ __align__(16) double G[kModelMaxM * kModelMaxM];
    __shared__ double unit[kModelMaxM];
    __shared__ __align__(16) double rows[kModelThreads / 16 * kModelRow];
    const int m = p.m, n = p.n, L = p.L;
    double *Bs = emo_model_smem;                   // [n][m]
    double *Ts = Bs + n * m;                       // [m][L]
    double *Es = Ts + m * L;                       // [m][L]
    for (int i = threadIdx.x; i < n * m; i += blockDim.x) Bs[i] = p.B[i];
    for (int i = threadIdx.x; i < m * L; i += blockDim.x) {
        Ts[i] = p.Tb[i];
        Es[i] = p.Eb[i];
    }
    __syncthreads();
    for (int i = threadIdx.x; i < kModelMaxM * kModelMaxM; i += blockDim.x) {
        const int a = i / kModelMaxM, b = i % kModelMaxM;
        double s = 0.0;
        if (a < m && b < m)
            for (int r = 0; r < n; ++r) s += Bs[r * m + a] * Bs[r * m + b];
        G[i] = s;
    }
    __syncthreads();
    // every unknown in units of a power of two that brings its diagonal entry to [1/2, 2): exact, and no pivot of an entering
    // variable is above 2
    if (threadIdx.x < kModelMaxM) {
        const double g = G[threadIdx.x * (kModelMaxM + 1)];
        // (half the exponent, odd ones rounded up: a shift, a division would round towards zero and leave [2, 4) as it is)
        unit[threadIdx.x] = (g > 0.0 && g < 1e300) ? ldexp(1.0, -((ilogb(g) + 1) >> 1)) : 1.0;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < kModelMaxM * kModelMaxM; i += blockDim.x) G[i] *= unit[i / kModelMaxM] * unit[i % kModelMaxM];
    __syncthreads();
    constexpr unsigned kFull = 0xFFFFFFFFu;
    const int me = threadIdx.x & 15, half = (threadIdx.x & 31) >> 4;
    const double scale = unit[me], unscale = 1.0 / scale;
    const int mc = min(me, m - 1);                 // lanes beyond the unknowns shadow the last one and are never chosen
    double *row = rows + (threadIdx.x / 16) * kModelRow;
    const unsigned stride = gridDim.x * (blockDim.x / 16), n_packs = (unsigned)p.n_packs;
    // both halves of a warp go round together
    for (unsigned base = (blockIdx.x * blockDim.x + (threadIdx.x & ~31u)) / 16; base < n_packs; base += stride) {
        const bool live = base + (unsigned)half < n_packs;
        const size_t pk = (size_t)(live ? base + half : base);
        double c = 0.0;
        for (int r = 0; r < n; ++r) c += Bs[r * m + mc] * p.feat[pk * n + r];
        if (me >= m) c = 0.0;
        const double cmax = emo_model_half_max(fabs(c));
        const double tol = 1e-13 * (cmax > 0.0 ? cmax : 1.0);
        c *= scale;
        double a[kModelMaxM], b = c, x = 0.0;
#pragma unroll
        for (int j = 0; j < kModelMaxM; ++j) a[j] = G[j * kModelMaxM + me];
        bool is_free = false, done = !live, failed = false;
        unsigned leaving = 0;                      // variables of this pack still to be returned to the held set
        int outer = 0, inner = 0;
        while (__any_sync(kFull, !done)) {
            // the next pivot: a variable that leaves, else the held one with the largest gradient component, the first among equals
            const double grad = b * unscale, w = (!is_free && me < m && grad > tol) ? grad : 0.0;
            const double best = emo_model_half_max(w);
            const unsigned who = (__ballot_sync(kFull, w > 0.0 && w == best) >> (16 * half)) & 0xFFFFu;
            const unsigned free_set = (__ballot_sync(kFull, is_free) >> (16 * half)) & 0xFFFFu;
            int k = 0;
            if (leaving) {
                k = __ffs(leaving) - 1;
                leaving &= leaving - 1u;
            } else if (!done) {
                if (who == 0u || outer == 3 * m) done = true;
                else {
                    k = __ffs(who) - 1;
                    ++outer;
                    inner = 0;
                }
            }
            const bool k_free = (free_set >> k) & 1u;
            if (!done && me == k) {
                double2 *o = reinterpret_cast<double2 *>(row);
#pragma unroll
                for (int j = 0; j < kModelMaxM; j += 2) o[j / 2] = make_double2(a[j], a[j + 1]);
                row[kModelMaxM] = b;
            }
            __syncwarp();
            const double d = row[k];
            double f = row[me];
            // a column that depends on the free ones cannot improve the fit, and no other one has a larger component
            if (!done && !k_free && d <= 1e-14 * G[k * (kModelMaxM + 1)]) done = true;
            __syncwarp();
            const bool go = !done;
            const double inv = 1.0 / d;
            const double2 *o = reinterpret_cast<const double2 *>(row);
            if (!__any_sync(kFull, go && k_free)) {
                // a variable enters: with d + 1 in the pivot's place every entry is one fused multiply-add, without a case for the
                // pivot's row (a - (1 - inv) a = inv a) or column (f - f inv (d + 1) = -f inv); nothing cancels, d being at most 2
                if (go && me == k) row[k] = d + 1.0;
                __syncwarp();
                if (go) {
                    f = me == k ? 1.0 - inv : (is_free ? -(f * inv) : f * inv);
#pragma unroll
                    for (int j = 0; j < kModelMaxM; j += 2) {
                        const double2 q = o[j / 2];
                        a[j] -= f * q.x;
                        a[j + 1] -= f * q.y;
                    }
                    b -= f * row[kModelMaxM];
                }
            } else {
                if (go && me == k) row[k] = 1.0;
                __syncwarp();
                if (go) {
                    f = me == k ? -inv : (is_free == k_free ? f * inv : -(f * inv));
                    const unsigned clear = me == k ? 0xFFFFu : 1u << k;
#pragma unroll
                    for (int j = 0; j < kModelMaxM; j += 2) {
                        const double2 q = o[j / 2];
                        a[j] = ((clear >> j) & 1u ? 0.0 : a[j]) - f * q.x;
                        a[j + 1] = ((clear >> (j + 1)) & 1u ? 0.0 : a[j + 1]) - f * q.y;
                    }
                    b = (me == k ? 0.0 : b) - f * row[kModelMaxM];
                }
            }
            if (go && me == k) is_free = !is_free;
            __syncwarp();
            // feasible?  otherwise the longest step towards z that keeps x >= 0
            const bool solved = !done && leaving == 0u, bad = solved && is_free && b <= 0.0;
            double alpha = 2.0;
            if (__any_sync(kFull, bad)) alpha = -emo_model_half_max(bad ? -(x / (x - b)) : -2.0);
            const bool step = solved && alpha <= 1.0;
            if (solved && !step && is_free) x = b;
            bool out = false;
            if (step && is_free) {
                const bool bound = bad && x / (x - b) == alpha;      // exactly at zero up to rounding: it leaves
                x += alpha * (b - x);
                out = bound || x <= 0.0 || (b <= 0.0 && (x <= 1e-300 || x <= 1e-15 * fabs(b)));
                if (out) x = 0.0;
            }
            const unsigned outs = (__ballot_sync(kFull, out) >> (16 * half)) & 0xFFFFu;
            if (step) {
                leaving = outs;
                if (++inner == 3 * m) failed = done = true;
            }
        }
        if (failed && live && me == 0 && p.status) atomicMin(p.status, -9);
        row[me] = x;
        __syncwarp();
        double r = c;
#pragma unroll
        for (int j = 0; j < kModelMaxM; ++j) r -= G[j * kModelMaxM + me] * row[j];
        __syncwarp();
        row[me] = is_free ? r : 0.0;
        __syncwarp();
        if (is_free && !failed) {
            double dx = 0.0;
#pragma unroll
            for (int j = 0; j < kModelMaxM; ++j) dx += a[j] * row[j];
            x = fmax(x + dx, 0.0);
        }
        x *= scale;
        __syncwarp();
        row[me] = x;
        __syncwarp();
        if (live) {
            if (me < m) p.x[pk * m + me] = x;
            // Eq. 7
            for (int l = me; l < L; l += 16) {
                double t = 0.0, e = 0.0;
                for (int i = 0; i < m; ++i) {
                    t += row[i] * Ts[i * L + l];
                    e += row[i] * Es[i * L + l];
                }
                p.T_out[pk * L + l] = t;
                p.E_out[pk * L + l] = e;
            }
        }
        __syncwarp();
    }
}
