// Skeletonization of large boxes (sm_103a): boxes whose column count is too
// large for one CTA are spread over the whole GPU.
//
//  * big_ygen        materializes the proxy matrices Y_c of Eq. (3.3) of all
//                    large boxes of a sublevel in HBM (kernel and SCI parts
//                    apart when rho_g is needed, Sec. 4.4);
//  * big_pow_*       rho_g = min(1, |Y^K_g| / |Y^S_g|) by 8 power iterations
//                    from the all-ones vector, directly on Y_g;
//  * big_step /      column-pivoted Householder QR (Lemma 2.2), one pair of
//    big_update      launches per pivot step for all large groups at once: one
//                    CTA per group picks the pivot and forms the reflector, a
//                    warp per remaining column applies it and brings the
//                    column norm up to date in FP64 (see kNormKeep);
//  * big_T           T = R1^{-1} R2 and the skeleton / redundant order;
//  * be_*            the batched elimination of medium and large boxes: Lemma
//                    2.4 blocks, Lemma 2.1 LU or LDL, inverses and the Schur
//                    update, one launch per stage for all of them.
#include <algorithm>

#include "hif_common.cuh"
#include "launch.h"

namespace hif {

// --------------------------------------------------------------- Y gen ----

template <typename T>
__global__ void big_ygen_kernel(BigArgs a) {
    const BigBox bb = a.bigboxes[blockIdx.y];
    const BoxDesc bx = a.boxes[bb.box];
    const int n = bx.n, npairs = bx.m_near + a.P;
    const int dim = a.g.dim;
    const bool scival = bx.has_sci && a.sci.nsub > 0;
    const bool split = scival && a.second_kind;
    const bool sym = bx.sym != 0;        // Y'_c: outgoing rows only (Sec. 5)
    T* YK = static_cast<T*>(a.YK) + bb.y_off;
    T* YS = split ? static_cast<T*>(a.YS) + bb.y_off : nullptr;
    const int64_t m = bb.m;
    const int* cols = a.cols + bx.col_off;
    const int* near = a.near + bx.near_off;
    const double c0 = bx.ctr[0], c1 = bx.ctr[1], c2 = dim == 3 ? bx.ctr[2] : 0.0;
    const int64_t tot = (int64_t)npairs * n;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < tot; e += (int64_t)gridDim.x * blockDim.x) {
        const int p = (int)(e % npairs), l = (int)(e / npairs);
        const int j = cols[l];
        const T cx0 = (T)(a.g.x[(int64_t)dim * j] - c0), cx1 = (T)(a.g.x[(int64_t)dim * j + 1] - c1);
        const T cx2 = dim == 3 ? (T)(a.g.x[(int64_t)dim * j + 2] - c2) : T(0);
        int rid, rcomp = 0;
        T rx0, rx1, rx2, rb, rwc;
        if (p < bx.m_near) {
            rid = near[p];
            if (a.g.ncomp == 2) rcomp = rid & 1;
            rx0 = (T)(a.g.x[(int64_t)dim * rid] - c0);
            rx1 = (T)(a.g.x[(int64_t)dim * rid + 1] - c1);
            rx2 = dim == 3 ? (T)(a.g.x[(int64_t)dim * rid + 2] - c2) : T(0);
            rb = (T)a.g.b[rid];
            rwc = (T)(a.g.w[rid] * a.g.c[rid]);
        } else {
            const int kx = p - bx.m_near;
            rid = -1;
            if (a.g.ncomp == 2) rcomp = kx & 1;
            rx0 = (T)(bx.radius * a.proxy[dim * kx]);
            rx1 = (T)(bx.radius * a.proxy[dim * kx + 1]);
            rx2 = dim == 3 ? (T)(bx.radius * a.proxy[dim * kx + 2]) : T(0);
            rb = T(1);
            rwc = T(1);
        }
        T k1, k2, s1, s2;
        y_pair<T>(a.g.kernel_id, rid, rx0, rx1, rx2, rb, rwc, j, cx0, cx1, cx2, (T)(a.g.w[j] * a.g.c[j]),
                  (T)a.g.b[j], (T)(a.g.b[j] * a.g.w[j]), scival, a.sci, k1, k2, s1, s2, rcomp,
                  (T)a.g.wavenumber);
        T* col = YK + m * l;
        if (sym) {
            col[p] = split ? k1 : k1 + s1;
            if (split) YS[m * l + p] = s1;
        } else if (split) {
            col[2 * p] = k1;
            col[2 * p + 1] = k2;
            YS[m * l + 2 * p] = s1;
            YS[m * l + 2 * p + 1] = s2;
        } else {
            col[2 * p] = k1 + s1;
            col[2 * p + 1] = k2 + s2;
        }
    }
}

// ------------------------------------------------------- rho_g (Sec 4.4) --

// t = Y_g v   (which: 0 = Y^K, 1 = Y^S), one thread per row
template <typename T>
__global__ void big_pow_tv_kernel(BigArgs a) {
    const BigGroup G = a.groups[blockIdx.y];
    if (!G.need_rho) return;
    const int which = blockIdx.z;
    const T* Y = static_cast<const T*>(which == 0 ? a.YK : a.YS) + G.y_off;
    const double* v = a.vec_v + 2 * G.vec_off + which * (int64_t)G.n;
    double* t = a.vec_t + 2 * G.row_off + which * (int64_t)G.m;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < G.m; i += gridDim.x * blockDim.x) {
        // rho_g needs only a rough norm ratio: FP32 data accumulate in FP32
        // (an FP64 FMA per entry binds the pass to the FP64 pipe)
        if constexpr (sizeof(T) == 4) {
            float acc = 0.f;
            for (int l = 0; l < G.n; ++l) acc = fmaf(Y[i + (int64_t)G.m * l], (float)v[l], acc);
            t[i] = acc;
        } else {
            double acc = 0.0;
            for (int l = 0; l < G.n; ++l) acc += (double)Y[i + (int64_t)G.m * l] * v[l];
            t[i] = acc;
        }
    }
}

// w = Y_g^T t, one warp per column
template <typename T>
__global__ void big_pow_w_kernel(BigArgs a) {
    const BigGroup G = a.groups[blockIdx.y];
    if (!G.need_rho) return;
    const int which = blockIdx.z;
    const T* Y = static_cast<const T*>(which == 0 ? a.YK : a.YS) + G.y_off;
    const double* t = a.vec_t + 2 * G.row_off + which * (int64_t)G.m;
    double* w = a.vec_w + 2 * G.vec_off + which * (int64_t)G.n;
    const int lane = threadIdx.x & 31;
    const int l = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (l >= G.n) return;
    double acc = 0.0;
    if constexpr (sizeof(T) == 4) {
        float af = 0.f;
        for (int i = lane; i < G.m; i += 32) af = fmaf(Y[i + (int64_t)G.m * l], (float)t[i], af);
        acc = (double)af;
    } else {
        for (int i = lane; i < G.m; i += 32) acc += (double)Y[i + (int64_t)G.m * l] * t[i];
    }
    acc = warp_sum(acc);
    if (lane == 0) w[l] = acc;
}

// mode 0: v = w / |w| (v = 0 when w = 0); mode 1: est = |t|; mode 2: v = 1/sqrt(n)
__global__ void big_pow_norm_kernel(BigArgs a, int mode) {
    const BigGroup G = a.groups[blockIdx.x];
    if (!G.need_rho) return;
    const int which = blockIdx.y;
    double* v = a.vec_v + 2 * G.vec_off + which * (int64_t)G.n;
    const double* w = a.vec_w + 2 * G.vec_off + which * (int64_t)G.n;
    const double* t = a.vec_t + 2 * G.row_off + which * (int64_t)G.m;
    __shared__ double red[256];
    if (mode == 2) {
        for (int l = threadIdx.x; l < G.n; l += blockDim.x) v[l] = 1.0 / sqrt((double)G.n);
        return;
    }
    const double* src = mode == 0 ? w : t;
    const int len = mode == 0 ? G.n : G.m;
    double s = 0.0;
    for (int i = threadIdx.x; i < len; i += blockDim.x) s += src[i] * src[i];
    red[threadIdx.x] = s;
    __syncthreads();
    for (int k = blockDim.x / 2; k > 0; k >>= 1) {
        if (threadIdx.x < k) red[threadIdx.x] += red[threadIdx.x + k];
        __syncthreads();
    }
    const double tot = red[0];
    if (mode == 1) {
        if (threadIdx.x == 0) a.est[2 * blockIdx.x + which] = sqrt(tot);
        return;
    }
    const double inv = tot > 0.0 ? 1.0 / sqrt(tot) : 0.0;
    for (int l = threadIdx.x; l < G.n; l += blockDim.x) v[l] = w[l] * inv;
}

// tolerance per group and Y = Y^K + Y^S
__global__ void big_tol_kernel(BigArgs a, int ngroups) {
    const int gi = blockIdx.x * blockDim.x + threadIdx.x;
    if (gi >= ngroups) return;
    BigGroup& G = a.groups[gi];
    double rho = 1.0;
    if (G.need_rho) {
        const double eK = a.est[2 * gi], eS = a.est[2 * gi + 1];
        if (eS > 0.0) rho = fmin(1.0, eK / eS);
    }
    double tol = rho * a.eps;
    if (tol < a.tol_floor) tol = a.tol_floor;
    G.tol = tol;
}

template <typename T>
__global__ void big_add_kernel(T* YK, const T* YS, int64_t n) {
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x)
        YK[e] += YS[e];
}

// --------------------------------------------------- pivoted QR steps ----

template <typename T>
__global__ void big_norm_init_kernel(BigArgs a) {
    const BigGroup G = a.groups[blockIdx.y];
    const T* Y = static_cast<const T*>(a.YK) + G.y_off;
    const int lane = threadIdx.x & 31;
    const int l = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        BigState& S = a.state[blockIdx.y];
        S.k = 0;
        S.stop = 0;
        S.nu0 = 0.0;
        S.tau = 0.0;
        S.j0 = 0;
        S.pend = 0;
        S.last_step = -1;
    }
    if (l >= G.n) return;
    double s = 0.0;
    for (int i = lane; i < G.m; i += 32) {
        const double v = (double)Y[i + (int64_t)G.ld * l];
        s += v * v;
    }
    s = warp_sum(s);
    if (lane == 0) {
        a.nrm[G.vec_off + l] = s;
        a.nrm0[G.vec_off + l] = s;
        a.perm[G.vec_off + l] = l;
    }
}

constexpr int BST = 256;   // threads of the step kernel: one CTA walks the pivot column of m rows

// Squared column norms of the pivot steps (Lemma 2.2).  In 64 bits the square
// after a step is the previous one less that of the new pivot row's entry, until
// it falls below kNormKeep of the last sum over the column and is summed anew
// (summed at every step, a third of the 64-bit work of a step were these sums).
// What a step decides, the pivot and the rank, it decides on sums: of the
// columns whose carried square lies within kNormTie of the largest (several
// of them, or one that close to the threshold) those not fresh are summed
// first.  A carried square is off by at most 2^-53 of the last sum per
// subtraction and by the rounding of the reflections, a few times m 2^-53 of
// the square at worst: 1,000 steps on 10,000 rows cost at most 2e-7 of it at
// the kNormKeep line, so no column outside that margin can be the largest.
// A square is fresh while nrm0 > 0; a carried one has its last sum negated.
// 32-bit columns, whose stored entries move by far more, are always summed.
// Pivot steps of n = 200, b != c, 203.5 ms, n = 64 8.2, Helmholtz n = 64, where
// the two columns of an unknown tie at every step, 36.1; deciding on the carried
// squares alone 202.1, 7.8 and 32.9; sums at every step cost n = 200 40 ms more.
constexpr double kNormKeep = 1e-2;
constexpr double kNormTie = 1e-6;

template <typename T>
__global__ void __launch_bounds__(BST) big_step_kernel(BigArgs a, int j) {
    const BigGroup G = a.groups[blockIdx.x];
    BigState* S = a.state + blockIdx.x;
    if (S->stop) return;
    T* W = static_cast<T*>(a.YK) + G.y_off;
    const int64_t ld = G.ld;
    double* nrm = a.nrm + G.vec_off;
    double* nrm0 = a.nrm0 + G.vec_off;
    int* perm = a.perm + G.vec_off;
    __shared__ double redv[BST];
    __shared__ int redi[BST];
    __shared__ T hs[BST];
    const int kmax = min(G.m, G.n);
    if (j >= kmax) {
        if (threadIdx.x == 0) S->stop = 1;
        return;
    }
    // largest square, ties to the lowest original column, in redv[0] and redi[0]
    auto find_pivot = [&]() {
        double best = -1.0;
        int bl = -1, bo = 1 << 30;
        for (int l = j + threadIdx.x; l < G.n; l += BST) {
            const double v = nrm[l];
            if (v > best || (v == best && perm[l] < bo)) { best = v; bo = perm[l]; bl = l; }
        }
        redv[threadIdx.x] = best;
        redi[threadIdx.x] = bl;
        __syncthreads();
        for (int s = BST / 2; s > 0; s >>= 1) {
            if (threadIdx.x < s) {
                const double v2 = redv[threadIdx.x + s], v1 = redv[threadIdx.x];
                const int l2 = redi[threadIdx.x + s], l1 = redi[threadIdx.x];
                if (l2 >= 0 && (l1 < 0 || v2 > v1 || (v2 == v1 && perm[l2] < perm[l1]))) {
                    redv[threadIdx.x] = v2;
                    redi[threadIdx.x] = l2;
                }
            }
            __syncthreads();
        }
    };
    find_pivot();
    if constexpr (sizeof(T) == 8) {
        // columns that could be the largest, and those of them not fresh
        const double top = redv[0], line = (1.0 - kNormTie) * top;
        int close = 0, carried = 0;
        for (int l = j + threadIdx.x; l < G.n; l += BST)
            if (nrm[l] >= line) {
                ++close;
                carried |= nrm0[l] < 0.0;
            }
        const bool several = __syncthreads_count(close > 0) > 1 || __syncthreads_or(close > 1);
        const double th = j == 0 ? 0.0 : G.tol * S->nu0, th2 = th * th;
        if (__syncthreads_or(carried) && (several || fabs(top - th2) <= kNormTie * th2)) {
            // (neighbours on different warps: the two columns of a complex
            // unknown tie at every step)
            const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
            constexpr int NW = BST / 32;
            for (int l0 = j + wid; l0 < G.n; l0 += BST) {
                const int l = l0 + NW * lane;
                unsigned todo = __ballot_sync(0xffffffffu, l < G.n && nrm[l] >= line && nrm0[l] < 0.0);
                for (; todo; todo &= todo - 1) {
                    const int q = l0 + NW * (__ffs(todo) - 1);
                    double sum = 0.0;
#pragma unroll 16
                    for (int i = j + lane; i < G.m; i += 32) {
                        const double c = (double)W[i + ld * q];
                        sum += c * c;
                    }
                    sum = warp_sum(sum);
                    if (lane == 0) nrm[q] = nrm0[q] = sum;
                }
            }
            __syncthreads();
            find_pivot();
        }
    }
    const double bnorm = sqrt(fmax(redv[0], 0.0));
    const int p = redi[0];
    const double nu0 = j == 0 ? bnorm : S->nu0;
    __syncthreads();
    if (bnorm <= G.tol * nu0 || bnorm == 0.0 || p < j) {
        if (threadIdx.x == 0) {
            S->stop = 1;
            if (j == 0) S->nu0 = bnorm;
        }
        return;
    }
    // columns j and p swapped, and the sum of squares below row j of the new
    // column j; SU rows per thread in flight (one CTA walks the m rows)
    constexpr int SU = 8;
    T s = T(0);
    for (int i0 = threadIdx.x; i0 < G.m; i0 += BST * SU) {
        T xj[SU], xp[SU];
#pragma unroll
        for (int u = 0; u < SU; ++u) {
            const int i = i0 + BST * u;
            xj[u] = i < G.m ? W[i + ld * j] : T(0);
            xp[u] = i < G.m && p != j ? W[i + ld * p] : xj[u];
        }
#pragma unroll
        for (int u = 0; u < SU; ++u) {
            const int i = i0 + BST * u;
            if (i < G.m && p != j) {
                W[i + ld * j] = xp[u];
                W[i + ld * p] = xj[u];
            }
            if (i > j && i < G.m) s += xp[u] * xp[u];
        }
    }
    __syncthreads();
    if (threadIdx.x == 0 && p != j) {
        const int t = perm[j]; perm[j] = perm[p]; perm[p] = t;
        double tn = nrm[j]; nrm[j] = nrm[p]; nrm[p] = tn;
        tn = nrm0[j]; nrm0[j] = nrm0[p]; nrm0[p] = tn;
    }
    hs[threadIdx.x] = s;
    __syncthreads();
    for (int k = blockDim.x / 2; k > 0; k >>= 1) {
        if (threadIdx.x < k) hs[threadIdx.x] += hs[threadIdx.x + k];
        __syncthreads();
    }
    const T ss = hs[0];
    const T alpha = W[j + ld * j];
    T tau = T(0), scal = T(0);
    if (ss != T(0)) {
        const T beta = -copysign(sqrt(alpha * alpha + ss), alpha);
        tau = (beta - alpha) / beta;
        scal = T(1) / (alpha - beta);
    }
    __syncthreads();
    if (tau != T(0)) {
        for (int i0 = j + 1 + threadIdx.x; i0 < G.m; i0 += BST * SU) {
            T x[SU];
#pragma unroll
            for (int u = 0; u < SU; ++u) x[u] = i0 + BST * u < G.m ? W[i0 + BST * u + ld * j] : T(0);
#pragma unroll
            for (int u = 0; u < SU; ++u)
                if (i0 + BST * u < G.m) W[i0 + BST * u + ld * j] = x[u] * scal;
        }
        if (threadIdx.x == 0) W[j + ld * j] = -copysign(sqrt(alpha * alpha + ss), alpha);
    }
    if (threadIdx.x == 0) {
        if (j == 0) S->nu0 = bnorm;
        S->tau = (double)tau;
        S->k = j + 1;
    }
}

// (U rows per lane are loaded before their FMAs: bytes in flight bound the
// step.  n = 200, b != c, 64-bit: 234 -> 175 ms of updates, 128 of them FP64.)
template <typename T>
__global__ void __launch_bounds__(256, 4) big_update_kernel(BigArgs a, int j) {
    const BigGroup G = a.groups[blockIdx.y];
    const BigState S = a.state[blockIdx.y];
    if (S.k != j + 1 || S.stop) return;
    const int lane = threadIdx.x & 31;
    const int l = j + 1 + blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (l >= G.n) return;
    T* W = static_cast<T*>(a.YK) + G.y_off;
    const int64_t ld = G.ld;
    T* col = W + ld * l;
    const T* v = W + ld * j;
    const T tau = (T)S.tau;
    constexpr int U = 8;                 // rows in flight per lane
    T w = T(0);
    if (tau != T(0)) {
        int i = j + 1 + lane;
        for (; i + 32 * (U - 1) < G.m; i += 32 * U) {
            T x[U], y[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                x[u] = col[i + 32 * u];
                y[u] = v[i + 32 * u];
            }
#pragma unroll
            for (int u = 0; u < U; ++u) w += y[u] * x[u];
        }
        for (; i < G.m; i += 32) w += v[i] * col[i];
        w = warp_sum(w);
        w = (w + col[j]) * tau;
        __syncwarp();
        if (lane == 0) col[j] -= w;
    }
    if (tau != T(0)) {
        int i = j + 1 + lane;
        for (; i + 32 * (U - 1) < G.m; i += 32 * U) {
            T x[U], y[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                x[u] = col[i + 32 * u];
                y[u] = v[i + 32 * u];
            }
#pragma unroll
            for (int u = 0; u < U; ++u) col[i + 32 * u] = x[u] - w * y[u];
        }
        for (; i < G.m; i += 32) col[i] -= w * v[i];
    }
    // the square of the new norm (see kNormKeep)
    double* nrm = a.nrm + G.vec_off + l;
    double* nrm0 = a.nrm0 + G.vec_off + l;
    __syncwarp();
    const double rj = (double)col[j], last = fabs(*nrm0);
    double s = fmax(*nrm - rj * rj, 0.0), sum = -last;
    __syncwarp();
    if (sizeof(T) == 4 || !(s >= kNormKeep * last)) {
        s = 0.0;
        for (int i = j + 1 + lane; i < G.m; i += 32) {
            const double c = (double)col[i];
            s += c * c;
        }
        sum = s = warp_sum(s);
    }
    if (lane == 0) *nrm0 = sum;
    if (lane == 0) *nrm = s;
}

// ---------------------------------------- blocked pivoted QR (panels) ----
//
// The pivoted QR of Lemma 2.2 with delayed trailing updates: within a panel
// of nb pivots only the pivot column and the pivot row are brought up to
// date; every trailing column l keeps F[l, q] = tau_q (W^T v_q)_l minus the
// earlier reflectors' share, so that W_updated = W - V F^T, and the panel
// ends with one product W[rows below the panel, trailing] -= V F^T.  The
// pivot choice and the rank test use the squared column norms downdated by
// the new pivot row's entries (in FP64); when a norm falls below
// sqrt(eps_T) of its value at the last exact computation the group ends its
// panel early, and every panel ends with the norms recomputed from the
// updated columns.  Per pivot the trailing columns are read once (for F),
// instead of read twice and written once.

constexpr int QPB = 32;   // maximum panel width

// start of a panel for every group still pivoting
__global__ void bqp_start_kernel(BigArgs a, int ngroups) {
    const int gi = blockIdx.x * blockDim.x + threadIdx.x;
    if (gi >= ngroups) return;
    BigState& S = a.state[gi];
    if (S.stop) return;
    S.j0 = S.k;
    S.pend = 0;
}

// distributed shared memory of a cluster
__device__ __forceinline__ uint32_t cl_peer(const void* p, int rank) {
    uint32_t out;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(out) : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
    return out;
}
__device__ __forceinline__ void cl_store(uint32_t a, double v) {
    asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(a), "d"(v) : "memory");
}
__device__ __forceinline__ void cl_store(uint32_t a, float v) {
    asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory");
}
__device__ __forceinline__ void cl_store(uint32_t a, int v) {
    asm volatile("st.shared::cluster.s32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ void cl_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// one pivot of the panel: argmax of the downdated norms, column swap, the pivot
// column brought up to date, its reflector, and g = V_panel^T v.  The rows of a
// group are dealt to a cluster of `cl` CTAs (as many as leave two per SM): the
// steps of a pivot are passes over the m rows of up to 32 columns, and between
// two bqp_f launches nothing else runs.  Every CTA finds the pivot itself;
// the cluster's barriers (the reflector's norm, g) follow, and rank 0 keeps the
// group's state.  Measured on a GB300, 3D n = 32 (eight boxes of up to 1,968
// columns and 28,000 rows): 55 us a pivot with one CTA per group, 35 with up to
// eight; with clusters for four times as many groups (three waves) 47.
constexpr int QPT = 512;   // threads of the pivot kernel

template <typename T>
__global__ void __launch_bounds__(QPT) bqp_pivot_kernel(BigArgs a, int step, int cl) {
    const int gi = blockIdx.x / cl, rank = blockIdx.x % cl;
    const BigGroup G = a.groups[gi];
    BigState* S = a.state + gi;
    if (S->stop || S->pend) return;
    const int j = S->k, j0 = S->j0, jj = j - j0;
    const int nb = a.nb;
    if (jj >= nb) return;
    const int kmax = min(G.m, G.n);
    const bool lead = rank == 0 && threadIdx.x == 0;
    if (j >= kmax) {
        if (lead) S->stop = 1;
        return;
    }
    T* W = static_cast<T*>(a.YK) + G.y_off;
    const int64_t ld = G.ld;
    const int n = G.n;
    double* nrm = a.nrm + G.vec_off;
    double* nrm0 = a.nrm0 + G.vec_off;
    int* perm = a.perm + G.vec_off;
    T* F = static_cast<T*>(a.F) + G.vec_off * nb;
    T* gq = static_cast<T*>(a.gv) + (int64_t)gi * QPB;
    constexpr int NW = QPT / 32;
    __shared__ double redv[NW];
    __shared__ int redi[NW], redo[NW];
    __shared__ T hs[NW], fj[QPB], part[NW][QPB];
    __shared__ T cs[8], calpha, cg[8][QPB];             // sent by the CTAs of the cluster
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    // pivot: largest downdated norm, ties to the lowest original column
    auto better = [](double v2, int o2, int l2, double v, int o, int l) {
        return l2 >= 0 && (l < 0 || v2 > v || (v2 == v && o2 < o));
    };
    double best = -1.0;
    int bl = -1, bo = 1 << 30;
    for (int l = j + threadIdx.x; l < n; l += QPT) {
        const double v = nrm[l];
        if (v > best || (v == best && perm[l] < bo)) { best = v; bo = perm[l]; bl = l; }
    }
    for (int q = 0; q < 2; ++q) {
        for (int off = 16; off; off >>= 1) {
            const double v2 = __shfl_xor_sync(0xffffffffu, best, off);
            const int o2 = __shfl_xor_sync(0xffffffffu, bo, off), l2 = __shfl_xor_sync(0xffffffffu, bl, off);
            if (better(v2, o2, l2, best, bo, bl)) { best = v2; bo = o2; bl = l2; }
        }
        if (q == 0) {
            if (lane == 0) { redv[wid] = best; redo[wid] = bo; redi[wid] = bl; }
            __syncthreads();
            best = lane < NW ? redv[lane] : -1.0;
            bo = lane < NW ? redo[lane] : 1 << 30;
            bl = lane < NW ? redi[lane] : -1;
        }
    }
    const double bnorm = sqrt(fmax(best, 0.0));
    const int p = bl;
    const double nu0 = j == 0 ? bnorm : S->nu0;
    // the rank test decides on exact norms: within a panel (downdated norms,
    // relative error up to ~sqrt(eps_T) in the square) a maximum near the
    // threshold ends the panel instead, and the next panel's first pivot,
    // on the recomputed norms, decides
    const double margin = sizeof(T) == 4 ? 1e-3 : 1e-7;
    if (jj > 0 && bnorm <= G.tol * nu0 * (1.0 + margin) && p >= j) {
        if (lead) S->pend = 1;
        return;
    }
    if (bnorm <= G.tol * nu0 || bnorm == 0.0 || p < j) {
        if (lead) {
            S->stop = 1;
            if (j == 0) S->nu0 = bnorm;
        }
        return;
    }
    // this CTA's rows [i0, i1) of j .. m - 1 (rank 0: also the finished rows
    // above, which only swap)
    const int per = (G.m - j + cl - 1) / cl;
    const int i0 = min(G.m, j + rank * per), i1 = min(G.m, i0 + per);
    if (cl > 1) cl_sync();                              // every CTA is there before the first remote store
    if (threadIdx.x < jj) fj[threadIdx.x] = F[p + (int64_t)n * threadIdx.x];
    if (rank == 0 && p != j)
        for (int i = threadIdx.x; i < j; i += QPT) {
            const T t = W[i + ld * j];
            W[i + ld * j] = W[i + ld * p];
            W[i + ld * p] = t;
        }
    __syncthreads();
    // the pivot column up to date, W[i, j] = W[i, p] - sum_q W[i, j0 + q] F[p, q],
    // and the sum of its squares below row j
    T ssum = T(0);
    for (int i = i0 + threadIdx.x; i < i1; i += QPT) {
        T acc = W[i + ld * p];
        if (p != j) W[i + ld * p] = W[i + ld * j];
#pragma unroll 8
        for (int q = 0; q < jj; ++q) acc -= W[i + ld * (j0 + q)] * fj[q];
        W[i + ld * j] = acc;
        if (i > j) ssum += acc * acc;
        else for (int q = 0; q < cl; ++q) cl_store(cl_peer(&calpha, q), acc);
    }
    ssum = warp_sum(ssum);
    if (lane == 0) hs[wid] = ssum;
    __syncthreads();
    if (wid == 0) {
        ssum = warp_sum(lane < NW ? hs[lane] : T(0));
        if (lane < cl) cl_store(cl_peer(&cs[rank], lane), ssum);
    }
    if (cl > 1) cl_sync();
    else __syncthreads();
    T ss = T(0);
    for (int q = 0; q < cl; ++q) ss += cs[q];
    const T alpha = calpha;
    T tau = T(0), scal = T(0), beta = alpha;
    if (ss != T(0)) {
        beta = -copysign(sqrt(alpha * alpha + ss), alpha);
        tau = (beta - alpha) / beta;
        scal = T(1) / (alpha - beta);
    }
    // v, and g[q] = sum_{i >= j} W[i, j0 + q] v_i, v_j = 1
    T acc[QPB];
#pragma unroll
    for (int q = 0; q < QPB; ++q) acc[q] = T(0);
    for (int i = i0 + threadIdx.x; i < i1; i += QPT) {
        T vi = T(1);
        if (i > j) {
            vi = W[i + ld * j];
            if (tau != T(0)) {
                vi *= scal;
                W[i + ld * j] = vi;
            }
        }
#pragma unroll
        for (int q = 0; q < QPB; ++q)
            if (q < jj) acc[q] += W[i + ld * (j0 + q)] * vi;
    }
    if (jj > 0) {
#pragma unroll
        for (int q = 0; q < QPB; ++q) {
            if (q >= jj) break;
            const T v = warp_sum(acc[q]);
            if (lane == 0) part[wid][q] = v;
        }
        __syncthreads();
        if (threadIdx.x < jj) {
            T v = T(0);
            for (int w = 0; w < NW; ++w) v += part[w][threadIdx.x];
            cl_store(cl_peer(&cg[rank][threadIdx.x], 0), v);
        }
    }
    if (cl > 1) cl_sync();
    else __syncthreads();
    if (rank != 0) return;
    if (threadIdx.x < jj) {
        T v = T(0);
        for (int q = 0; q < cl; ++q) v += cg[q][threadIdx.x];
        gq[threadIdx.x] = v;
        if (p != j) F[p + (int64_t)n * threadIdx.x] = F[j + (int64_t)n * threadIdx.x];
        F[j + (int64_t)n * threadIdx.x] = fj[threadIdx.x];
    }
    if (threadIdx.x == 0) {
        if (p != j) {
            const int t = perm[j]; perm[j] = perm[p]; perm[p] = t;
            double tn = nrm[j]; nrm[j] = nrm[p]; nrm[p] = tn;
            tn = nrm0[j]; nrm0[j] = nrm0[p]; nrm0[p] = tn;
        }
        if (tau != T(0)) W[j + ld * j] = beta;
        if (j == 0) S->nu0 = bnorm;
        S->tau = (double)tau;
        S->k = j + 1;
        S->last_step = step;
    }
}

// F[l, jj] for the trailing columns (a warp per two columns, which share the
// reads of v), the pivot row's entry brought up to date, and the norm downdated.
// Bound by the bytes in flight: with 16 rows of the columns per lane loaded
// before their FMAs the 3D n = 32 launches went from 107 to 73 ms (4.8 TB/s).
template <typename T>
__global__ void __launch_bounds__(256, 4) bqp_f_kernel(BigArgs a, int step) {
    const BigGroup G = a.groups[blockIdx.y];
    const BigState S = a.state[blockIdx.y];
    if (S.stop || S.last_step != step) return;
    const int j = S.k - 1, j0 = S.j0, jj = j - j0;
    const int nb = a.nb;
    const int lane = threadIdx.x & 31;
    const int l0 = j + 1 + 2 * (blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5));
    if (l0 >= G.n) return;
    T* W = static_cast<T*>(a.YK) + G.y_off;
    const int64_t ld = G.ld;
    const int n = G.n;
    T* F = static_cast<T*>(a.F) + G.vec_off * nb;
    const T* gq = static_cast<const T*>(a.gv) + (int64_t)blockIdx.y * QPB;
    const T tau = (T)S.tau;
    const bool two = l0 + 1 < n;
    const T* c0 = W + ld * l0;
    const T* c1 = two ? c0 + ld : c0;
    const T* v = W + ld * j;
    T d0 = T(0), d1 = T(0);
    int i = j + 1 + lane;
    constexpr int U = sizeof(T) == 4 ? 8 : 4;       // rows in flight per lane and column
    for (; i + 32 * (U - 1) < G.m; i += 32 * U) {
        T vv[U], x0[U], x1[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            x0[u] = c0[i + 32 * u];
            x1[u] = c1[i + 32 * u];
            vv[u] = v[i + 32 * u];
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            d0 += vv[u] * x0[u];
            d1 += vv[u] * x1[u];
        }
    }
    for (; i < G.m; i += 32) {
        d0 += v[i] * c0[i];
        d1 += v[i] * c1[i];
    }
    d0 = warp_sum(d0);
    d1 = warp_sum(d1);
    if (lane < (two ? 2 : 1)) {
        const int l = l0 + lane;
        T* col = W + ld * l;
        const T dot = (lane == 0 ? d0 : d1) + col[j];
        T corr = T(0);
#pragma unroll 4
        for (int q = 0; q < jj; ++q) corr += F[l + (int64_t)n * q] * gq[q];
        const T f = tau * (dot - corr);
        F[l + (int64_t)n * jj] = f;
        // pivot row: W[j, l] -= sum_{q < jj} W[j, j0 + q] F[l, q] + F[l, jj]
        T r = col[j] - f;
#pragma unroll 4
        for (int q = 0; q < jj; ++q) r -= W[j + ld * (j0 + q)] * F[l + (int64_t)n * q];
        col[j] = r;
        double* nrm = a.nrm + G.vec_off;
        const double* nrm0 = a.nrm0 + G.vec_off;
        const double nn = fmax(nrm[l] - (double)r * (double)r, 0.0);
        nrm[l] = nn;
        // the downdated norm keeps ~sqrt(eps_T) relative accuracy only while
        // it stays above sqrt(eps_T) of the last exact value
        const double tol3z = sizeof(T) == 4 ? 3.4526698e-4 : 1.4901161e-8;
        if (nn <= tol3z * nrm0[l]) atomicExch(&a.state[blockIdx.y].pend, 1);
    }
}

// end of a panel: rows below the panel of the trailing columns, W -= V F^T
// (64 x 64 tiles, K = the panel's pivots)
template <typename T>
__global__ void __launch_bounds__(256) bqp_update_kernel(BigArgs a) {
    const BigGroup G = a.groups[blockIdx.z];
    const BigState S = a.state[blockIdx.z];
    if (S.stop) return;
    const int j0 = S.j0, kb = S.k - S.j0, r0 = S.k;
    if (kb <= 0) return;
    const int i0 = r0 + blockIdx.x * 64, c0 = r0 + blockIdx.y * 64;
    if (i0 >= G.m || c0 >= G.n) return;
    T* W = static_cast<T*>(a.YK) + G.y_off;
    const int64_t ld = G.ld;
    const int n = G.n;
    const T* F = static_cast<const T*>(a.F) + G.vec_off * a.nb;
    __shared__ T Vs[QPB][64 + 1];
    __shared__ T Fs[QPB][64 + 1];
    for (int q = threadIdx.x; q < 64 * QPB; q += 256) {
        const int rr = q % 64, c = q / 64;
        const int i = i0 + rr, l = c0 + rr;
        Vs[c][rr] = (c < kb && i < G.m) ? W[i + ld * (j0 + c)] : T(0);
        Fs[c][rr] = (c < kb && l < n) ? F[l + (int64_t)n * c] : T(0);
    }
    __syncthreads();
    const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
    T acc[4][4] = {};
    for (int c = 0; c < kb; ++c) {
        T av[4], bv[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) av[q] = Vs[c][tx + 16 * q];
#pragma unroll
        for (int q = 0; q < 4; ++q) bv[q] = Fs[c][ty + 16 * q];
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
            for (int w = 0; w < 4; ++w) acc[u][w] += av[u] * bv[w];
    }
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int w = 0; w < 4; ++w) {
            const int i = i0 + tx + 16 * u, l = c0 + ty + 16 * w;
            if (i < G.m && l < n) W[i + ld * l] -= acc[u][w];
        }
}

// exact norms of rows k.. of the trailing columns (a warp per column)
template <typename T>
__global__ void __launch_bounds__(256) bqp_norm_kernel(BigArgs a) {
    const BigGroup G = a.groups[blockIdx.y];
    const BigState S = a.state[blockIdx.y];
    if (S.stop) return;
    const int r0 = S.k;
    const int lane = threadIdx.x & 31;
    const int l = r0 + blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (l >= G.n) return;
    const T* col = static_cast<const T*>(a.YK) + G.y_off + G.ld * l;
    double s = 0.0;
    if constexpr (sizeof(T) == 4) {
        float sf = 0.f;
        for (int i = r0 + lane; i < G.m; i += 32) sf = fmaf(col[i], col[i], sf);
        s = (double)sf;
    } else {
        for (int i = r0 + lane; i < G.m; i += 32) s += (double)col[i] * (double)col[i];
    }
    s = warp_sum(s);
    if (lane == 0) {
        a.nrm[G.vec_off + l] = s;
        a.nrm0[G.vec_off + l] = s;
    }
}

template <typename T>
cudaError_t big_qp_panel(const BigArgs& a, int ngroups, int max_n, int max_m, int& step, cudaStream_t st) {
    if (ngroups == 0) return cudaSuccess;
    if (a.nb < 1 || a.nb > QPB) return cudaErrorInvalidValue;
    note_launch();
    bqp_start_kernel<<<(ngroups + 127) / 128, 128, 0, st>>>(a, ngroups);
    int cl = 1;
    while (cl < 8 && 2 * cl * ngroups <= 2 * a.num_sms && max_m > 1024 * cl) cl *= 2;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)(ngroups * cl));
    cfg.blockDim = dim3(QPT);
    cfg.stream = st;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = (unsigned)cl;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = cl > 1 ? 1 : 0;
    for (int jj = 0; jj < a.nb; ++jj, ++step) {
        note_launch();
        const cudaError_t e = cudaLaunchKernelEx(&cfg, bqp_pivot_kernel<T>, a, step, cl);
        if (e != cudaSuccess) return e;
        note_launch();
        bqp_f_kernel<T><<<dim3((max_n + 15) / 16, ngroups), 256, 0, st>>>(a, step);
    }
    note_launch();
    bqp_update_kernel<T><<<dim3((max_m + 63) / 64, (max_n + 63) / 64, ngroups), 256, 0, st>>>(a);
    note_launch();
    bqp_norm_kernel<T><<<dim3((max_n + 7) / 8, ngroups), 256, 0, st>>>(a);
    return cudaGetLastError();
}

// T = R1^{-1} R2 (redundant columns in ascending original order), outputs.
// One CTA per TW redundant columns, by blocks of 32 rows from the last: the
// products with the rows already solved, then the triangular block itself, a
// column per lane.  (One thread per column read R1 row by row from global
// memory: 3D n = 32, k ~ 900, 32-bit, 27.6 ms for the sublevels' large groups,
// 0.8 now; n = 200, 64-bit, 14.6 and 3.4.)
constexpr int TW = 8;

template <typename T>
__global__ void __launch_bounds__(256) big_T_kernel(BigArgs a) {
    const BigGroup G = a.groups[blockIdx.y];
    const GroupDesc gd = a.gdesc[G.group];
    const int k = a.state[blockIdx.y].k;
    const int n = G.n, r = n - k;
    const T* W = static_cast<const T*>(a.YK) + G.y_off;
    const int64_t ld = G.ld;
    const int* perm = a.perm + G.vec_off;
    T* Tout = static_cast<T*>(a.Tws) + gd.T_off;
    int* pout = a.perm_out + gd.perm_off;
    const int t = threadIdx.x, l0 = blockIdx.x * TW;
    if (l0 == 0 && t == 0) a.k_out[G.group] = k;
    for (int l = l0 + t; l < min(l0 + TW, k); l += 256) pout[l] = perm[l];
    if (l0 >= r) return;
    __shared__ T Rs[32][33];
    __shared__ T Xs[32][TW + 1];
    __shared__ int pos[TW];
    const int ti = t % 32, tj = t / 32, l = l0 + tj;          // one warp per column
    {
        const int o = l < r ? perm[k + l] : 0;
        int c = 0;
        for (int q = ti; l < r && q < r; q += 32) c += perm[k + q] < o;
        for (int off = 16; off; off >>= 1) c += __shfl_xor_sync(0xffffffffu, c, off);
        if (ti == 0 && l < r) {
            pos[tj] = c;
            pout[k + c] = o;
        }
    }
    __syncthreads();
    T* tcol = l < r ? Tout + (int64_t)k * pos[tj] : nullptr;
    const int nb = (k + 31) / 32;
    for (int I = nb - 1; I >= 0; --I) {
        const int gi = 32 * I + ti;
        T acc = gi < k && l < r ? W[gi + ld * (k + l)] : T(0);
        for (int K = nb - 1; K >= I; --K) {
            __syncthreads();
            for (int q = t; q < 1024; q += 256) {
                const int i = q % 32, c = q / 32, ri = 32 * I + i, rc = 32 * K + c;
                Rs[i][c] = ri < k && rc < k ? W[ri + ld * rc] : T(0);
            }
            const int gk = 32 * K + ti;
            if (K > I) Xs[ti][tj] = gk < k && l < r ? tcol[gk] : T(0);
            __syncthreads();
            if (K == I) break;
#pragma unroll
            for (int c = 0; c < 32; ++c) acc -= Rs[ti][c] * Xs[c][tj];
        }
        // the triangular block: the column's warp, from the last row up
        const int last = min(31, k - 1 - 32 * I);
        T x = T(0);
        const T di = ti <= last ? Rs[ti][ti] : T(1), ri = T(1) / di;
        for (int i = last; i >= 0; --i) {
            // acc / di: the reciprocal and one correction step
            T v = acc * ri;
            v = fma(fma(-v, di, acc), ri, v);
            v = __shfl_sync(0xffffffffu, v, i);
            if (ti == i) x = v;
            if (ti < i) acc -= Rs[ti][i] * v;
        }
        if (gi < k && l < r) tcol[gi] = x;
    }
}

// ---------------------------------------------------------- launchers ----

template <typename T>
cudaError_t big_ygen(const BigArgs& a, int nbig, int64_t max_entries, cudaStream_t st) {
    if (nbig == 0) return cudaSuccess;
    dim3 grid((unsigned)std::min<int64_t>((max_entries + 255) / 256, 4096), nbig);
    note_launch();
    big_ygen_kernel<T><<<grid, 256, 0, st>>>(a);
    return cudaGetLastError();
}

template <typename T>
cudaError_t big_rho(const BigArgs& a, int ngroups, int max_m, int max_n, cudaStream_t st) {
    if (ngroups == 0) return cudaSuccess;
    dim3 gn(ngroups, 2);
    dim3 gtv((max_m + 255) / 256, ngroups, 2);
    dim3 gw((max_n + 7) / 8, ngroups, 2);
    note_launch();
    big_pow_norm_kernel<<<gn, 256, 0, st>>>(a, 2);
    for (int it = 0; it < 8; ++it) {
        note_launch();
        big_pow_tv_kernel<T><<<gtv, 256, 0, st>>>(a);
        note_launch();
        big_pow_w_kernel<T><<<gw, 256, 0, st>>>(a);
        note_launch();
        big_pow_norm_kernel<<<gn, 256, 0, st>>>(a, 0);
    }
    note_launch();
    big_pow_tv_kernel<T><<<gtv, 256, 0, st>>>(a);
    note_launch();
    big_pow_norm_kernel<<<gn, 256, 0, st>>>(a, 1);
    note_launch();
    big_tol_kernel<<<(ngroups + 127) / 128, 128, 0, st>>>(a, ngroups);
    return cudaGetLastError();
}

template <typename T>
cudaError_t big_add(void* YK, const void* YS, int64_t n, cudaStream_t st) {
    if (n == 0) return cudaSuccess;
    note_launch();
    big_add_kernel<T><<<(unsigned)std::min<int64_t>((n + 255) / 256, 152 * 32), 256, 0, st>>>(
        static_cast<T*>(YK), static_cast<const T*>(YS), n);
    return cudaGetLastError();
}

template <typename T>
cudaError_t big_qr_init(const BigArgs& a, int ngroups, int max_n, cudaStream_t st) {
    if (ngroups == 0) return cudaSuccess;
    dim3 g((max_n + 7) / 8, ngroups);
    note_launch();
    big_norm_init_kernel<T><<<g, 256, 0, st>>>(a);
    return cudaGetLastError();
}

template <typename T>
cudaError_t big_qr_step(const BigArgs& a, int ngroups, int max_n, int j, cudaStream_t st) {
    note_launch();
    big_step_kernel<T><<<ngroups, BST, 0, st>>>(a, j);
    const int cols = max_n - j - 1;
    if (cols > 0) {
        dim3 g((cols + 7) / 8, ngroups);
        note_launch();
        big_update_kernel<T><<<g, 256, 0, st>>>(a, j);
    }
    return cudaGetLastError();
}

template <typename T>
cudaError_t big_finish(const BigArgs& a, int ngroups, int max_n, cudaStream_t st) {
    if (ngroups == 0) return cudaSuccess;
    dim3 g((max_n + TW - 1) / TW, ngroups);
    note_launch();
    big_T_kernel<T><<<g, 256, 0, st>>>(a);
    return cudaGetLastError();
}

// ---------------------------------------------- batched elimination ----
//
// All large boxes of a sublevel are eliminated together: every stage below is
// one launch whose last grid dimension runs over the boxes.  Box e works on
// its own workspace A_e (n x n, order (rd, sk)) and T_e (k x r).

template <typename T>
struct EBox {
    int k, r, n;
    T* A;
    T* Tm;
    __device__ EBox(const BatchElimArgs& a, int e) {
        const ElimDesc& d = a.ed[e];
        k = d.k;
        r = d.r;
        n = k + r;
        A = static_cast<T*>(a.ws) + d.ws_off;
        Tm = A + (int64_t)n * n;
    }
};

template <typename T>
__global__ void be_gather_kernel(BatchElimArgs a) {
    const int e = blockIdx.y;
    const ElimDesc d = a.ed[e];
    const EBox<T> B(a, e);
    const int* sk = a.sk + d.sk_off;
    const int* rd = a.rd + d.rd_off;
    const int ref = B.r > 0 ? rd[0] : sk[0];
    const int dm = a.g.dim;
    const double r0 = a.g.x[(int64_t)dm * ref], r1 = a.g.x[(int64_t)dm * ref + 1];
    const double r2 = dm == 3 ? a.g.x[(int64_t)dm * ref + 2] : 0.0;
    const int64_t tot = (int64_t)B.n * B.n;
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < tot; q += (int64_t)gridDim.x * blockDim.x) {
        const int p = (int)(q % B.n), c = (int)(q / B.n);
        const int i = p < B.r ? rd[p] : sk[p - B.r];
        const int j = c < B.r ? rd[c] : sk[c - B.r];
        B.A[q] = entry<T>(a.g, a.sci, i, j, r0, r1, r2);
    }
}

template <typename T>
__global__ void be_T_kernel(BatchElimArgs a) {
    const int e = blockIdx.x;
    const ElimDesc d = a.ed[e];
    const EBox<T> B(a, e);
    for (int q = threadIdx.x; q < B.k * B.r; q += blockDim.x) B.Tm[q] = T(0);
    __syncthreads();
    const T* Tws = static_cast<const T*>(a.Tws);
    for (int gi = 0; gi < d.ngroups; ++gi) {
        const ElimGroup G = a.groups[d.grp_off + gi];
        for (int q = threadIdx.x; q < G.kg * G.rg; q += blockDim.x) {
            const int i = q % G.kg, jj = q / G.kg;
            B.Tm[(G.ko + i) + (int64_t)B.k * (G.ro + jj)] = Tws[G.T_off + q];
        }
    }
}

// the GEMMs of Lemma 2.4, one op per launch:
// 0: B_sr = A_sr - A_ss T     1: B_rr -= T^T B_sr     2: B_rr -= A_rs T
// 3: B_rs = A_rs - T^T A_ss
// TS x TS tiles: 64, or 32 where the boxes give few of them.
template <typename T, int TS>
__global__ void __launch_bounds__(256) be_gemm_kernel(BatchElimArgs a, int op) {
    constexpr int Q = TS / 16;
    __shared__ T As[16][TS + 1];
    __shared__ T Bs[16][TS + 1];
    const int e = blockIdx.z;
    const ElimDesc d = a.ed[e];
    const EBox<T> Bx(a, e);
    const int k = Bx.k, r = Bx.r;
    const int64_t ld = Bx.n;
    T* Arr = Bx.A;
    T* Asr = Bx.A + r;
    T* Ars = Bx.A + ld * r;
    T* Ass = Bx.A + ld * r + r;
    int m, n, kk;
    const T* A;
    const T* Bm;
    T* C;
    int64_t lda, ldb, ldc;
    bool tA = false;
    switch (op) {
        case 0: m = k; n = r; kk = k; A = Ass; lda = ld; Bm = Bx.Tm; ldb = k; C = Asr; ldc = ld; break;
        case 1: m = r; n = r; kk = k; A = Bx.Tm; lda = k; tA = true; Bm = Asr; ldb = ld; C = Arr; ldc = ld; break;
        case 2: m = r; n = r; kk = k; A = Ars; lda = ld; Bm = Bx.Tm; ldb = k; C = Arr; ldc = ld; break;
        default: if (d.ldl) return; m = r; n = k; kk = k; A = Bx.Tm; lda = k; tA = true; Bm = Ass; ldb = ld; C = Ars; ldc = ld; break;
    }
    const int i0 = blockIdx.x * TS, j0 = blockIdx.y * TS;
    if (i0 >= m || j0 >= n || kk == 0) return;
    const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
    T acc[Q][Q] = {};
    for (int l0 = 0; l0 < kk; l0 += 16) {
        for (int q = threadIdx.x; q < TS * 16; q += 256) {
            const int rr = q % TS, l = q / TS;
            const int i = i0 + rr, kx = l0 + l;
            T v = T(0);
            if (i < m && kx < kk) v = tA ? A[kx + lda * i] : A[i + lda * kx];
            As[l][rr] = v;
            const int jj = j0 + rr;
            T u = T(0);
            if (jj < n && kx < kk) u = Bm[kx + ldb * jj];
            Bs[l][rr] = u;
        }
        __syncthreads();
#pragma unroll
        for (int l = 0; l < 16; ++l) {
            T av[Q], bv[Q];
#pragma unroll
            for (int q = 0; q < Q; ++q) av[q] = As[l][tx + 16 * q];
#pragma unroll
            for (int q = 0; q < Q; ++q) bv[q] = Bs[l][ty + 16 * q];
#pragma unroll
            for (int p = 0; p < Q; ++p)
#pragma unroll
                for (int q = 0; q < Q; ++q) acc[p][q] += av[p] * bv[q];
        }
        __syncthreads();
    }
    for (int p = 0; p < Q; ++p)
        for (int q = 0; q < Q; ++q) {
            const int i = i0 + tx + 16 * p, jj = j0 + ty + 16 * q;
            if (i < m && jj < n) C[i + ldc * jj] -= acc[p][q];
        }
}

// The same products as tensor-core problems (FP32): one TcGemmProb per box
// for op, C -= op(A) op(B) (op 4: C = -X Z); a box without work gets m = 0.
__global__ void be_probs_kernel(BatchElimArgs a, int op, TcGemmProb* out) {
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= a.nbox) return;
    const ElimDesc d = a.ed[e];
    const EBox<float> Bx(a, e);
    const int k = Bx.k, r = Bx.r;
    const int64_t ld = Bx.n;
    float* Arr = Bx.A;
    float* Asr = Bx.A + r;
    float* Ars = Bx.A + ld * r;
    float* Ass = Bx.A + ld * r + r;
    TcGemmProb p{};
    p.alpha = -1.f;
    p.beta = 1;
    switch (op) {
        case 0: p = TcGemmProb{Ass, Bx.Tm, Asr, ld, k, ld, k, r, k, 0, 0, -1.f, 1}; break;
        case 1: p = TcGemmProb{Bx.Tm, Asr, Arr, k, ld, ld, r, r, k, 1, 0, -1.f, 1}; break;
        case 2: p = TcGemmProb{Ars, Bx.Tm, Arr, ld, k, ld, r, r, k, 0, 0, -1.f, 1}; break;
        case 3: p = TcGemmProb{Bx.Tm, Ass, Ars, k, ld, ld, r, k, k, 1, 0, -1.f, 1}; break;
        default: {
            const float* pool = static_cast<const float*>(a.pool);
            p = TcGemmProb{pool + d.X_out, pool + d.Y_out,
                           static_cast<float*>(a.sci_pool) + (d.sci_out < 0 ? 0 : d.sci_out), k, r, k, k, k, r, 0,
                           0, -1.f, 0};
            }
            if (k == 0 || d.sci_out < 0) p.m = 0;
            break;
    }
    if (k == 0 && op < 4) p.m = 0;
    out[e] = p;
}

// ---- factorization of B_rr in shared memory, one cluster of CTAs per box ----
//
// One pivot step is a search, a column that every CTA needs and a rank-1
// update: for r of a few hundred the chain of steps, not the arithmetic, sets
// the time, and from global memory a step costs several dependent round trips.
// Here the block lives in the shared memory of a cluster (columns dealt out
// in turn), a step's column goes to every CTA by distributed shared memory,
// and the steps are separated by one (LU) or two (LDL) cluster barriers.
// Pivots are not moved: `at` maps positions to rows (and columns, LDL), with
// the interchanges of the textbook scheme applied to it alone, so ties go to
// the lowest position as they do there.  Output in position order: LU (L
// strictly below the diagonal), or for LDL boxes L below, D, and D L^T above.
// Measured on a GB300 against the one-CTA and panel kernels this replaces: a
// 64-bit LDL block of 388 rows 60 -> 8 ms with all its stages; all eliminations of
// n = 64 (it and four blocks of 348) 12 ms, with the searches on integers and one
// reciprocal per step 8.7 (7.2 with the unsymmetric update below).
constexpr int FT = 512;
constexpr int FCL = 8;                       // largest cluster
constexpr size_t kFactorSmemMax = 224 * 1024;

template <typename T>
size_t be_factor_smem(int r, int cl) {
    return (size_t)((r + cl - 1) / cl) * r * sizeof(T) + 2 * (size_t)r * sizeof(T) + 2 * (size_t)r * sizeof(int) + 64;
}

// largest v, then lowest pos, over the warp; id follows (-1: no candidate)
template <typename T>
__device__ __forceinline__ void warp_best(T& v, int& pos, int& id) {
    for (int o = 16; o; o >>= 1) {
        const T v2 = __shfl_xor_sync(0xffffffffu, v, o);
        const int p2 = __shfl_xor_sync(0xffffffffu, pos, o), i2 = __shfl_xor_sync(0xffffffffu, id, o);
        if (i2 >= 0 && (id < 0 || v2 > v || (v2 == v && p2 < pos))) { v = v2; pos = p2; id = i2; }
    }
}

// |v| as an integer of the same order: comparing these costs no FP64 operation
// (64 cycles of a scheduler each; the searches were half of a 64-bit step)
__device__ __forceinline__ long long abs_key(double v) { return __double_as_longlong(v) & 0x7fffffffffffffffLL; }
__device__ __forceinline__ long long abs_key(float v) { return __float_as_int(v) & 0x7fffffff; }
template <typename T> constexpr long long kInfKey = sizeof(T) == 8 ? 0x7ff0000000000000LL : 0x7f800000LL;
// largest key, then lowest pos, over the warp; id follows (-1: no candidate)
__device__ __forceinline__ void warp_best_key(long long& v, int& pos, int& id) {
    for (int o = 16; o; o >>= 1) {
        const long long v2 = __shfl_xor_sync(0xffffffffu, v, o);
        const int p2 = __shfl_xor_sync(0xffffffffu, pos, o), i2 = __shfl_xor_sync(0xffffffffu, id, o);
        if (i2 >= 0 && (id < 0 || v2 > v || (v2 == v && p2 < pos))) { v = v2; pos = p2; id = i2; }
    }
}
__device__ __forceinline__ void cl_store(uint32_t a, long long v) {
    asm volatile("st.shared::cluster.s64 [%0], %1;" ::"r"(a), "l"(v) : "memory");
}

template <typename T>
__global__ void __launch_bounds__(FT) be_factor_kernel(BatchElimArgs a, int cl) {
    const int e = blockIdx.x / cl, rank = blockIdx.x % cl;
    const ElimDesc d = a.ed[e];
    const int r = d.r;
    if (r > a.factor_max_r) return;                   // panel path (the whole cluster leaves)
    const int64_t ld = d.k + r;
    T* Ag = static_cast<T*>(a.ws) + d.ws_off;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ long long cval[2][FCL];
    __shared__ int cid[2][FCL], cpos[2][FCL], cstat[2], spiv;
    __shared__ T cinv[2], sinv;
    const int own = (r - rank + cl - 1) / cl;         // columns rank, rank + cl, ...
    T* A = reinterpret_cast<T*>(smem_raw);            // A[i + r * s]: column rank + cl * s
    T* col = A + (size_t)((r + cl - 1) / cl) * r;     // col[r * parity + i]
    int* at = reinterpret_cast<int*>(col + 2 * r);
    int* pos = at + r;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    constexpr int NW = FT / 32;
    for (int q = threadIdx.x; q < own * r; q += FT) A[q] = Ag[q % r + ld * (rank + cl * (q / r))];
    for (int i = threadIdx.x; i < r; i += FT) at[i] = pos[i] = i;
    __syncthreads();
    if (cl > 1) cl_sync();                            // every CTA is there before the first remote store
    for (int j = 0; j < r; ++j) {
        T* c = col + r * (j & 1);
        int p;
        if (d.ldl) {
            // remaining diagonal entry of largest magnitude
            if (warp == 0) {
                long long v = -1;
                int ps = 0, id = -1;
                for (int s = lane; s < own; s += 32) {
                    const int q = rank + cl * s, pq = pos[q];
                    const long long x = abs_key(A[q + r * s]);
                    if (pq >= j && x <= kInfKey<T> && (id < 0 || x > v || (x == v && pq < ps))) { v = x; ps = pq; id = q; }
                }
                warp_best_key(v, ps, id);
                if (lane < cl) {
                    cl_store(cl_peer(&cval[j & 1][rank], lane), v);
                    cl_store(cl_peer(&cpos[j & 1][rank], lane), ps);
                    cl_store(cl_peer(&cid[j & 1][rank], lane), id);
                }
            }
            if (cl > 1) cl_sync();
            else __syncthreads();
            long long v = -1;
            int ps = 0;
            p = -1;
            for (int q = 0; q < cl; ++q) {
                const long long x = cval[j & 1][q];
                const int pq = cpos[j & 1][q], id = cid[j & 1][q];
                if (id >= 0 && (p < 0 || x > v || (x == v && pq < ps))) { v = x; ps = pq; p = id; }
            }
            if (p < 0) p = at[j];                     // no comparable entry: the test below fails
            if (p % cl == rank) {
                const T* src = A + (size_t)r * (p / cl);
                for (int i = threadIdx.x; i < r; i += FT) {
                    const T x = pos[i] >= j ? src[i] : T(0);
                    for (int q = 0; q < cl; ++q) cl_store(cl_peer(c + i, q), x);
                }
                if (warp == 0) {                      // the pivot's test and reciprocal, for all
                    long long cm = 0;
                    for (int i = lane; i < r; i += 32)
                        if (i != p && pos[i] >= j) cm = max(cm, abs_key(src[i]));
                    for (int o = 16; o; o >>= 1) cm = max(cm, __shfl_xor_sync(0xffffffffu, cm, o));
                    const T dp = src[p], m = sizeof(T) == 8 ? (T)__longlong_as_double(cm) : (T)__int_as_float((int)cm);
                    const long long kd = abs_key(dp);
                    const int st = kd == 0 || kd >= kInfKey<T> ? 2 : fabs(dp) >= (T)a.ldl_alpha * m ? 0 : 1;
                    const T iv = T(1) / dp;
                    if (lane < cl) {
                        cl_store(cl_peer(&cstat[j & 1], lane), st);
                        cl_store(cl_peer(&cinv[j & 1], lane), iv);
                    }
                }
            }
            if (cl > 1) cl_sync();
            else __syncthreads();
            const int st = cstat[j & 1];
            if (st != 0) {
                if (rank == 0 && threadIdx.x == 0) {
                    atomicOr(a.status, st == 2 ? (int)DEV_SINGULAR : (int)DEV_LDL_FALLBACK);
                    if (st == 1) a.ldl_fail[a.fail_idx[e]] = 1;
                }
                break;
            }
            const T inv = cinv[j & 1];
            for (int s = warp; s < own; s += NW) {
                const int q = rank + cl * s;
                if (pos[q] < j || q == p) continue;
                // (c_i c_q) inv, which is the same for (i, q) and (q, i): the
                // remaining block stays symmetric to the bit.  c_i (c_q inv)
                // would save an operation (1.5 ms at n = 64, 64 bits), but its
                // rounding of c_q inv is common to the column
                const T f = c[q];
                T* x = A + (size_t)r * s;
                for (int i = lane; i < r; i += 32)
                    if (i != p) x[i] -= c[i] * f * inv;
            }
            if (p % cl == rank) {
                T* x = A + (size_t)r * (p / cl);
                for (int i = threadIdx.x; i < r; i += FT)
                    if (pos[i] >= j && i != p) x[i] = c[i] * inv;
            }
        } else {
            // largest remaining entry of column j
            if (j % cl == rank) {
                T* x = A + (size_t)r * (j / cl);
                if (warp == 0) {
                    long long v = -1;
                    int ps = 0, id = -1;
                    for (int i = lane; i < r; i += 32) {
                        const long long y = abs_key(x[i]);
                        const int pi = pos[i];
                        if (pi >= j && y <= kInfKey<T> && (id < 0 || y > v || (y == v && pi < ps))) { v = y; ps = pi; id = i; }
                    }
                    warp_best_key(v, ps, id);
                    if (id < 0) id = at[j];           // (all NaN: the pivot test below fails)
                    const long long kd = abs_key(x[id]);
                    if (lane < cl) {
                        cl_store(cl_peer(&cid[j & 1][0], lane), id);
                        cl_store(cl_peer(&cstat[j & 1], lane), kd == 0 || kd >= kInfKey<T> ? 2 : 0);
                    }
                    const T iv = T(1) / x[id];
                    if (lane == 0) {
                        spiv = id;
                        sinv = iv;
                    }
                }
                __syncthreads();
                const int pp = spiv;
                const T pinv = sinv;
                for (int i = threadIdx.x; i < r; i += FT) {
                    const bool on = pos[i] >= j && i != pp;
                    const T l = on ? x[i] * pinv : T(0);
                    if (on) x[i] = l;
                    for (int q = 0; q < cl; ++q) cl_store(cl_peer(c + i, q), l);
                }
            }
            if (cl > 1) cl_sync();
            else __syncthreads();
            p = cid[j & 1][0];
            if (cstat[j & 1] != 0) {
                if (rank == 0 && threadIdx.x == 0) atomicOr(a.status, (int)DEV_SINGULAR);
                break;
            }
            for (int s = warp; s < own; s += NW) {
                if (rank + cl * s <= j) continue;
                T* x = A + (size_t)r * s;
                const T u = x[p];
                for (int i = lane; i < r; i += 32) x[i] -= c[i] * u;
            }
        }
        __syncthreads();                              // updates done, pos and at read
        if (threadIdx.x == 0) {
            const int t = at[j], pp = pos[p];
            at[j] = p;
            at[pp] = t;
            pos[t] = pp;
            pos[p] = j;
        }
        __syncthreads();
    }
    if (cl > 1) cl_sync();                            // no CTA leaves while a peer may store to it
    else __syncthreads();
    for (int q = threadIdx.x; q < own * r; q += FT) {
        const int i = q % r, s = q / r, o = rank + cl * s, j = d.ldl ? pos[o] : o;
        const T* x = A + (size_t)r * s;
        const T v = x[at[i]];
        if (!d.ldl || i >= j) Ag[i + ld * j] = v;
        if (d.ldl && i > j) Ag[j + ld * i] = v * x[o];
    }
    if (rank == 0)
        for (int i = threadIdx.x; i < r; i += FT) a.perm[d.piv_out + i] = at[i];
}

// the largest block that fits into a cluster's shared memory
template <typename T>
int be_factor_max_r() {
    int r = 1;
    while (be_factor_smem<T>(r + 1, FCL) <= kFactorSmemMax) ++r;
    return r;
}

template <typename T>
cudaError_t launch_be_factor(const BatchElimArgs& a, int max_r, cudaStream_t st) {
    // CTAs per box: as many as the largest block needs, more while the
    // sublevel's boxes leave SMs idle and each CTA keeps 16 columns
    int cl = 1;
    while (cl < FCL && be_factor_smem<T>(max_r, cl) > kFactorSmemMax) cl *= 2;
    while (cl < FCL && 2 * cl * a.nbox <= a.num_sms && max_r >= 32 * cl) cl *= 2;
    const size_t smem = be_factor_smem<T>(max_r, cl);
    cudaError_t e = cudaFuncSetAttribute(be_factor_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)kFactorSmemMax);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)(a.nbox * cl));
    cfg.blockDim = dim3(FT);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = (unsigned)cl;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = cl > 1 ? 1 : 0;
    note_launch();
    return cudaLaunchKernelEx(&cfg, be_factor_kernel<T>, a, cl);
}

// blocked LU of B_rr (Lemma 2.1) of blocks too large for that, panel /
// interchange+TRSM / update stages
constexpr int PNT = 512;   // threads of the LU panel kernel (the pivot search spans all rows)

template <typename T>
__global__ void __launch_bounds__(PNT) be_panel_kernel(BatchElimArgs a, int j0) {
    const int e = blockIdx.x;
    const ElimDesc d = a.ed[e];
    const EBox<T> Bx(a, e);
    const int n = Bx.r;
    if (j0 >= n || n <= a.factor_max_r) return;
    const int nb = min(32, n - j0);
    const int64_t ld = Bx.n;
    T* A = Bx.A;
    int* piv = a.piv + d.piv_out;
    __shared__ T redv[PNT];
    __shared__ int redi[PNT];
    for (int j = j0 + threadIdx.x; j < j0 + nb; j += blockDim.x) piv[j] = j;
    __syncthreads();
    for (int j = j0; j < j0 + nb; ++j) {
        T best = T(-1);
        int bi = j;
        for (int i = j + threadIdx.x; i < n; i += blockDim.x) {
            const T v = fabs(A[i + ld * j]);
            if (v > best) { best = v; bi = i; }
        }
        redv[threadIdx.x] = best;
        redi[threadIdx.x] = bi;
        __syncthreads();
        for (int s = blockDim.x / 2; s > 0; s >>= 1) {
            if (threadIdx.x < s) {
                const T v2 = redv[threadIdx.x + s];
                const int i2 = redi[threadIdx.x + s];
                if (v2 > redv[threadIdx.x] || (v2 == redv[threadIdx.x] && i2 < redi[threadIdx.x])) {
                    redv[threadIdx.x] = v2;
                    redi[threadIdx.x] = i2;
                }
            }
            __syncthreads();
        }
        int p = redi[0];
        if (p < j || p >= n) p = j;
        __syncthreads();
        if (threadIdx.x == 0) piv[j] = p;
        if (p != j)
            for (int c = j0 + threadIdx.x; c < j0 + nb; c += blockDim.x) {
                const T t = A[j + ld * c];
                A[j + ld * c] = A[p + ld * c];
                A[p + ld * c] = t;
            }
        __syncthreads();
        const T dg = A[j + ld * j];
        if (dg == T(0) || !isfinite((double)dg)) {
            if (threadIdx.x == 0) atomicOr(a.status, (int)DEV_SINGULAR);
            return;
        }
        const T inv = T(1) / dg;
        for (int i = j + 1 + threadIdx.x; i < n; i += blockDim.x) {
            const T l = A[i + ld * j] * inv;
            A[i + ld * j] = l;
            for (int c = j + 1; c < j0 + nb; ++c) A[i + ld * c] -= l * A[j + ld * c];
        }
        __syncthreads();
    }
}

// The same panel with its rows dealt to a cluster of PCL CTAs, in shared memory:
// every CTA sends its best candidate of the column with its row, and the CTA
// that holds row j that row too, to all the others, so that a column costs one
// cluster barrier.  (The one-CTA panel in global memory took ~12 us a column:
// 61 ms of the 3D n = 32 elimination.)
constexpr int PCL = 8;

template <typename T>
size_t be_panel_smem(int rows) {
    return (size_t)((rows + PCL - 1) / PCL) * 33 * sizeof(T);
}

template <typename T>
__global__ void __launch_bounds__(256) be_panel_cluster_kernel(BatchElimArgs a, int j0) {
    const int e = blockIdx.x / PCL, rank = blockIdx.x % PCL;
    const ElimDesc d = a.ed[e];
    const EBox<T> Bx(a, e);
    const int n = Bx.r;
    if (j0 >= n || n <= a.factor_max_r) return;           // the whole cluster
    const int nb = min(32, n - j0), rows = n - j0, per = (rows + PCL - 1) / PCL;
    const int i0 = j0 + rank * per, own = max(0, min(per, n - i0));
    const int64_t ld = Bx.n;
    T* A = Bx.A;
    int* piv = a.piv + d.piv_out;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T* P = reinterpret_cast<T*>(smem_raw);                // P[33 i + c]: row i0 + i, column j0 + c
    __shared__ T crow[2][PCL][32], jrow[2][32], cval[2][PCL], wv[8];
    __shared__ int cid[2][PCL], wi[8];
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    for (int q = t; q < own * nb; q += 256) P[33 * (q % own) + q / own] = A[i0 + q % own + ld * (j0 + q / own)];
    __syncthreads();
    cl_sync();
    bool bad = false;
    for (int c = 0; c < nb; ++c) {
        const int j = j0 + c, buf = c & 1;
        T best = T(-1);
        int bi = -1, dummy = 0;
        for (int i = t; i < own; i += 256) {
            const T v = fabs(P[33 * i + c]);
            if (i0 + i >= j && (bi < 0 ? v == v : v > best)) { best = v; bi = i0 + i; }
        }
        dummy = bi;                                       // ties: lowest row
        warp_best(best, dummy, bi);
        if (lane == 0) { wv[warp] = best; wi[warp] = bi; }
        __syncthreads();
        // warp q sends this CTA's candidate (and row j) to CTA q
        best = lane < 8 ? wv[lane] : T(-1);
        bi = dummy = lane < 8 ? wi[lane] : -1;
        warp_best(best, dummy, bi);
        if (bi >= 0) cl_store(cl_peer(&crow[buf][rank][lane], warp), lane < nb ? P[33 * (bi - i0) + lane] : T(0));
        if (lane == 0) {
            cl_store(cl_peer(&cval[buf][rank], warp), best);
            cl_store(cl_peer(&cid[buf][rank], warp), bi);
        }
        if (j >= i0 && j < i0 + own && lane < nb) cl_store(cl_peer(&jrow[buf][lane], warp), P[33 * (j - i0) + lane]);
        cl_sync();
        int p = -1, pr = 0;
        best = T(-1);
        for (int q = 0; q < PCL; ++q) {
            const int id = cid[buf][q];
            const T v = cval[buf][q];
            if (id >= 0 && (p < 0 || v > best || (v == best && id < p))) { best = v; p = id; pr = q; }
        }
        if (p < 0) p = j;                                 // all NaN: the test below fails
        const T* prow = best >= T(0) ? crow[buf][pr] : jrow[buf];
        if (rank == 0 && t == 0) piv[j] = p;
        const T dg = prow[c];
        if (dg == T(0) || !isfinite((double)dg)) {
            if (rank == 0 && t == 0) atomicOr(a.status, (int)DEV_SINGULAR);
            bad = true;
            break;
        }
        const T inv = T(1) / dg;
        for (int i = t; i < own; i += 256) {
            const int g = i0 + i;
            T* x = P + 33 * i;
            if (g == p && p != j)
                for (int q = 0; q < nb; ++q) x[q] = jrow[buf][q];
            if (g == j)
                for (int q = 0; q < nb; ++q) x[q] = prow[q];
            if (g <= j) continue;
            const T l = x[c] * inv;
            x[c] = l;
            for (int q = c + 1; q < nb; ++q) x[q] -= l * prow[q];
        }
        __syncthreads();
    }
    cl_sync();                                            // no CTA leaves while a peer may store to it
    if (bad) {
        for (int j = j0 + t; rank == 0 && j < j0 + nb; j += 256)
            if (j > j0) piv[j] = j;
        return;
    }
    for (int q = t; q < own * nb; q += 256) A[i0 + q % own + ld * (j0 + q / own)] = P[33 * (q % own) + q / own];
}

template <typename T>
__global__ void be_swap_trsm_kernel(BatchElimArgs a, int j0) {
    const int e = blockIdx.y;
    const ElimDesc d = a.ed[e];
    const EBox<T> Bx(a, e);
    const int n = Bx.r;
    if (j0 >= n || n <= a.factor_max_r) return;
    const int nb = min(32, n - j0);
    const int64_t ld = Bx.n;
    T* A = Bx.A;
    const int* piv = a.piv + d.piv_out;
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= n || (c >= j0 && c < j0 + nb)) return;
    for (int j = j0; j < j0 + nb; ++j) {
        const int p = piv[j];
        if (p != j) {
            const T t = A[j + ld * c];
            A[j + ld * c] = A[p + ld * c];
            A[p + ld * c] = t;
        }
    }
    if (c >= j0 + nb)
        for (int i = j0; i < j0 + nb; ++i) {
            T v = A[i + ld * c];
            for (int l = j0; l < i; ++l) v -= A[i + ld * l] * A[l + ld * c];
            A[i + ld * c] = v;
        }
}

template <typename T>
__global__ void __launch_bounds__(256) be_update_kernel(BatchElimArgs a, int j0) {
    const int e = blockIdx.z;
    const EBox<T> Bx(a, e);
    const int n = Bx.r;
    if (j0 >= n || n <= a.factor_max_r) return;
    const int nb = min(32, n - j0);
    const int s = j0 + nb;
    const int i0 = s + blockIdx.x * 64, c0 = s + blockIdx.y * 64;
    if (i0 >= n || c0 >= n) return;
    const int64_t ld = Bx.n;
    T* A = Bx.A;
    __shared__ T Ls[64][33];
    __shared__ T Us[32][65];
    for (int q = threadIdx.x; q < 64 * nb; q += blockDim.x) {
        const int i = q % 64, l = q / 64;
        Ls[i][l] = (i0 + i < n) ? A[(i0 + i) + ld * (j0 + l)] : T(0);
    }
    for (int q = threadIdx.x; q < 64 * nb; q += blockDim.x) {
        const int l = q % nb, c = q / nb;
        Us[l][c] = (c0 + c < n) ? A[(j0 + l) + ld * (c0 + c)] : T(0);
    }
    __syncthreads();
    const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
    T acc[4][4] = {};
    for (int l = 0; l < nb; ++l) {
        T av[4], bv[4];
        for (int q = 0; q < 4; ++q) av[q] = Ls[tx + 16 * q][l];
        for (int q = 0; q < 4; ++q) bv[q] = Us[l][ty + 16 * q];
        for (int p = 0; p < 4; ++p)
            for (int q = 0; q < 4; ++q) acc[p][q] += av[p] * bv[q];
    }
    for (int p = 0; p < 4; ++p)
        for (int q = 0; q < 4; ++q) {
            const int i = i0 + tx + 16 * p, c = c0 + ty + 16 * q;
            if (i < n && c < n) A[i + ld * c] -= acc[p][q];
        }
}

// ---- after the LU of B_rr: the factor outputs by blocked products --------
//
// With P B_rr = L U = L D U' (L, U' unit triangular), Lemma 2.4's blocks
// are X = B_sr U^{-1}, Z = L^{-1} P B_rs, the Schur update S = -X Z, and the
// sweeps keep Y = D^{-1} Z and the unit triangular inverses L^{-1}, U'^{-1}.
// The inverses are formed from the diagonal IB x IB blocks up, by substitution
// and then by doubling (be_inv_level_kernel; F = L, or U'^T for the upper
// factor).  X and Z are blocked substitutions (only the IB x IB diagonal
// blocks enter through their inverses: multiplying by the whole explicit
// inverse measured a less accurate FP32 factor), S a tiled product.

// D, the unit factors (LU_out: L strictly below, U' strictly above, zero
// diagonal) and the row permutation P of the pivots
template <typename T>
__global__ void be_lu_out_kernel(BatchElimArgs a) {
    const int e = blockIdx.y;
    const ElimDesc d = a.ed[e];
    const EBox<T> Bx(a, e);
    const int r = Bx.r;
    const int64_t ld = Bx.n;
    const T* Arr = Bx.A;
    T* pool = static_cast<T*>(a.pool);
    T* Dv = pool + d.D_out;
    T* LUo = pool + d.LU_out;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const int64_t t0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    for (int64_t q = t0; q < r; q += stride) Dv[q] = Arr[q + ld * q];
    for (int64_t q = t0; q < (int64_t)r * r; q += stride) {
        const int i = (int)(q % r), j = (int)(q / r);
        LUo[q] = i == j || (d.ldl && i < j) ? T(0) : (i < j ? Arr[i + ld * j] / Arr[i + ld * i] : Arr[i + ld * j]);
    }
    if (t0 == 0 && r > a.factor_max_r) {
        int* pm = a.perm + d.piv_out;
        const int* piv = a.piv + d.piv_out;
        for (int i = 0; i < r; ++i) pm[i] = i;
        for (int j = 0; j < r; ++j) {
            const int p = piv[j];
            const int t = pm[j]; pm[j] = pm[p]; pm[p] = t;
        }
    }
}

constexpr int IB = 32;   // block size of the triangular inverses

// Unit lower factor F(i, l), i > l: L itself (UP false) or U'^T (UP true);
// its inverse's entries (i > j) go to LUi_out at (i, j) or, transposed, (j, i)
// (U'^T, and L of an LDL box, whose inverse shares L's array).
template <typename T, bool UP>
__device__ __forceinline__ T tri_f(const T* F, int64_t r, int i, int l) {
    return UP ? F[l + r * i] : F[i + r * l];
}
template <typename T>
__device__ __forceinline__ T* tri_x(T* X, int64_t r, bool xt, int i, int j) {
    return xt ? X + j + r * i : X + i + r * j;
}

// inverses of the IB x IB diagonal blocks (one warp per block and box)
template <typename T, bool UP>
__global__ void be_dinv_kernel(BatchElimArgs a) {
    const int e = blockIdx.y;
    const ElimDesc d = a.ed[e];
    const int r = d.r;
    const int b0 = blockIdx.x * IB;
    if (b0 >= r || (UP && d.ldl)) return;
    const bool xt = UP || d.ldl;
    const int nbk = min(IB, r - b0);
    const T* F = static_cast<const T*>(a.pool) + d.LU_out;
    T* X = static_cast<T*>(a.pool) + d.LUi_out;
    __shared__ T Fs[IB][IB + 1];
    __shared__ T Xs[IB][IB + 1];
    const int t = threadIdx.x;
    for (int q = t; q < IB * IB; q += 32) {
        const int i = UP ? q / IB : q % IB, l = UP ? q % IB : q / IB;   // coalesced either way
        Fs[i][l] = (i < nbk && l < nbk && i > l) ? tri_f<T, UP>(F, r, b0 + i, b0 + l) : T(0);
    }
    __syncthreads();
    if (t < nbk) {
        for (int i = 0; i < IB; ++i) Xs[i][t] = T(0);
        for (int i = t + 1; i < nbk; ++i) {
            T v = -Fs[i][t];
            for (int l = t + 1; l < i; ++l) v -= Fs[i][l] * Xs[l][t];
            Xs[i][t] = v;
        }
    }
    __syncthreads();
    for (int q = t; q < IB * IB; q += 32) {
        const int i = UP ? q / IB : q % IB, j = UP ? q % IB : q / IB;
        if (i < nbk && j < nbk && i > j) *tri_x(X, r, xt, b0 + i, b0 + j) = Xs[i][j];
    }
    if (t < nbk) X[(b0 + t) + (int64_t)r * (b0 + t)] = T(0);
}

// From the inverses of the diagonal blocks of size s to those of size 2 s:
// with F = [F11 0; F21 F22] the block below is -inv(F22) (F21 inv(F11)).
// PH 1: T = F21 inv(F11), into B_rr's work space (no longer needed); PH 2:
// X21 = -inv(F22) T.  An error of T reaches X21 times inv(F22), which block
// substitution does not do, so one correction follows: PH 3: T += F22 X21, the
// block of F X - I; PH 4: X21 -= inv(F22) T.  (32 bits, eps = 1e-6, solve then
// apply, geometric mean of the relative error over 20 problems of n = 512: 9.3e-7
// with block substitution, 1.0e-6 by doubling alone, 5.6e-7 with the correction;
// 8 of n = 1024: 1.8e-6, 2.5e-6, 1.2e-6, for 1-5% of the factorization.)  One CTA per 32 x 32 tile, pair of blocks and box, so a
// level fills the GPU.  (Block column by block column, each one a chain over
// its blocks, the 3D n = 32 inverses took 39 ms, the n = 200 64-bit ones 21;
// with the cluster panels the eliminations went from 123 to 46 and from 92 to
// 70 ms.)
template <typename T, bool UP, int PH>
__global__ void __launch_bounds__(256) be_inv_level_kernel(BatchElimArgs a, int s) {
    const int e = blockIdx.z;
    const ElimDesc d = a.ed[e];
    const int r = d.r, nt = s / IB;
    const int ti0 = blockIdx.x % nt, tj0 = blockIdx.x / nt;
    const int b = 2 * s * blockIdx.y, i0 = b + s + IB * ti0, j0 = b + IB * tj0;
    if (i0 >= r || (UP && d.ldl)) return;
    const bool xt = UP || d.ldl;
    const T* F = static_cast<const T*>(a.pool) + d.LU_out;
    T* X = static_cast<T*>(a.pool) + d.LUi_out;
    const EBox<T> Bx(a, e);
    T* Tm = Bx.A;
    const int64_t ld = Bx.n;
    __shared__ T Ls[IB][IB + 1];
    __shared__ T Rs[IB][IB + 1];
    const int t = threadIdx.x, ti = t % IB, tj = t / IB;          // entries (ti, tj + 8 q)
    T acc[4] = {T(0), T(0), T(0), T(0)};
    // entry (i, j) of the unit lower inverse inside a diagonal block of size s
    auto inv_at = [&](int i, int j) -> T {
        return i < r && j < r ? (i == j ? T(1) : i > j ? *tri_x(X, r, xt, i, j) : T(0)) : T(0);
    };
    // left operand F (PH 1, 3) or inv(F22); right operand X (PH 1, 3) or T
    constexpr bool LF = PH == 1 || PH == 3;
    const int k0 = PH == 1 ? tj0 : 0, k1 = PH == 1 ? nt : ti0 + 1;
    for (int K = k0; K < k1; ++K) {
        const int g0 = (PH == 1 ? b : b + s) + IB * K;            // rows of the right operand
        __syncthreads();
        for (int q = t; q < IB * IB; q += 256) {
            const int u = q % IB, v = q / IB;
            {
                // coalesced along the stored rows
                const int i = (LF ? UP : xt) ? v : u, l = (LF ? UP : xt) ? u : v;
                const int gi = i0 + i, gl = g0 + l;
                if (LF) Ls[i][l] = gi < r && gl < gi ? tri_f<T, UP>(F, r, gi, gl) : T(gi < r && gl == gi);
                else Ls[i][l] = inv_at(gi, gl);
            }
            {
                const bool tr = LF && xt;
                const int l = tr ? v : u, c = tr ? u : v;
                const int gl = g0 + l, gc = j0 + c;
                Rs[l][c] = LF ? inv_at(gl, gc) : gl < r ? Tm[gl + ld * gc] : T(0);
            }
        }
        __syncthreads();
#pragma unroll 8
        for (int l = 0; l < IB; ++l) {
            const T f = Ls[ti][l];
#pragma unroll
            for (int q = 0; q < 4; ++q) acc[q] += f * Rs[l][tj + 8 * q];
        }
    }
    const int gi = i0 + ti;
    if (gi >= r) return;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int gj = j0 + tj + 8 * q;
        if (PH == 1) Tm[gi + ld * gj] = acc[q];
        if (PH == 2) *tri_x(X, r, xt, gi, gj) = -acc[q];
        if (PH == 3) Tm[gi + ld * gj] += acc[q];
        if (PH == 4) *tri_x(X, r, xt, gi, gj) -= acc[q];
    }
}

// X = B_sr U^{-1} by block columns: X_J = (B_J - sum_{K<J} X_K U_KJ) inv(U_JJ),
// inv(U_JJ) = (I + S_JJ) D_J^{-1} with S_JJ the stored strict upper part of
// the diagonal block of U'^{-1}.  LDL box: B_sr P^T (D L^T)^{-1}.  One CTA per
// RT rows of X and box (64, or 16 where the boxes give few CTAs); thread
// (tx, ty) holds entries (tx, ty + CT q) of the RT x 32 block.
template <typename T, int RT>
__global__ void __launch_bounds__(256) be_trsm_x_kernel(BatchElimArgs a) {
    const int e = blockIdx.y;
    const ElimDesc d = a.ed[e];
    const EBox<T> Bx(a, e);
    const int k = Bx.k, r = Bx.r;
    constexpr int CT = 256 / RT, NQ = IB / CT;
    const int i0 = blockIdx.x * RT;
    if (i0 >= k) return;
    const int64_t ld = Bx.n;
    const T* Arr = Bx.A;
    const T* Asr = Bx.A + r;
    T* X = static_cast<T*>(a.pool) + d.X_out;
    const T* Si = static_cast<const T*>(a.pool) + d.LUi_out;
    const T* Dv = static_cast<const T*>(a.pool) + d.D_out;
    __shared__ T Xs[RT][IB + 1];
    __shared__ T Us[IB][IB + 1];
    const int tx = threadIdx.x % RT, ty = threadIdx.x / RT;
    const int i = i0 + tx;
    const int* pm = a.perm + d.piv_out;
    const int rb = (r + IB - 1) / IB;
    for (int J = 0; J < rb; ++J) {
        T acc[NQ];
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
            const int c = J * IB + ty + CT * q;
            acc[q] = (i < k && c < r) ? Asr[i + ld * (d.ldl ? pm[c] : c)] : T(0);
        }
        for (int K = 0; K < J; ++K) {
            __syncthreads();
            for (int q = threadIdx.x; q < RT * IB; q += 256) {
                const int rr = q % RT, l = q / RT, gl = K * IB + l;
                Xs[rr][l] = (i0 + rr < k && gl < r) ? X[(i0 + rr) + (int64_t)k * gl] : T(0);
            }
            for (int q = threadIdx.x; q < IB * IB; q += 256) {
                const int l = q % IB, c = q / IB, gl = K * IB + l, gc = J * IB + c;
                Us[l][c] = (gl < r && gc < r) ? Arr[gl + ld * gc] : T(0);
            }
            __syncthreads();
#pragma unroll 8
            for (int l = 0; l < IB; ++l) {
                const T xv = Xs[tx][l];
#pragma unroll
                for (int q = 0; q < NQ; ++q) acc[q] -= xv * Us[l][ty + CT * q];
            }
        }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < NQ; ++q) Xs[tx][ty + CT * q] = acc[q];
        for (int q = threadIdx.x; q < IB * IB; q += 256) {
            const int l = q % IB, c = q / IB, gl = J * IB + l, gc = J * IB + c;
            Us[l][c] = (l < c && gc < r) ? Si[gl + (int64_t)r * gc] : T(0);
        }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
            const int c = ty + CT * q, gc = J * IB + c;
            T v = Xs[tx][c];
            for (int l = 0; l < c; ++l) v += Xs[tx][l] * Us[l][c];
            if (i < k && gc < r) X[i + (int64_t)k * gc] = v / Dv[gc];
        }
    }
}

// Z = L^{-1} P B_rs by block rows: Z_I = (I + S_II) (PB_I - sum_{K<I} L_IK Z_K),
// S_II the stored strict lower part of the diagonal block of L^{-1}.  Z goes
// to Y_out (scaled by D^{-1} later); LDL boxes need none.  One CTA per RT
// columns of Z and box; thread (tr, tc) holds entries (tr, tc + 8 q) of the
// 32 x RT block.
template <typename T, int RT>
__global__ void __launch_bounds__(256) be_trsm_z_kernel(BatchElimArgs a) {
    const int e = blockIdx.y;
    const ElimDesc d = a.ed[e];
    const EBox<T> Bx(a, e);
    const int k = Bx.k, r = Bx.r;
    constexpr int NQ = RT / 8;
    const int j0 = blockIdx.x * RT;
    if (j0 >= k || d.ldl) return;
    const int64_t ld = Bx.n;
    const T* Arr = Bx.A;
    const T* Ars = Bx.A + ld * r;
    T* Z = static_cast<T*>(a.pool) + d.Y_out;
    const T* Si = static_cast<const T*>(a.pool) + d.LUi_out;
    const int* pm = a.perm + d.piv_out;
    __shared__ T Ls[IB][IB + 1];
    __shared__ T Zs[IB][RT + 1];
    const int tr = threadIdx.x % IB, tc = threadIdx.x / IB;
    const int rb = (r + IB - 1) / IB;
    for (int I = 0; I < rb; ++I) {
        const int gi = I * IB + tr;
        T acc[NQ];
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
            const int j = j0 + tc + 8 * q;
            acc[q] = (gi < r && j < k) ? Ars[pm[gi] + ld * j] : T(0);
        }
        for (int K = 0; K < I; ++K) {
            __syncthreads();
            for (int q = threadIdx.x; q < IB * IB; q += 256) {
                const int rr = q % IB, l = q / IB, g1 = I * IB + rr, g2 = K * IB + l;
                Ls[rr][l] = (g1 < r && g2 < r) ? Arr[g1 + ld * g2] : T(0);
            }
            for (int q = threadIdx.x; q < IB * RT; q += 256) {
                const int l = q % IB, c = q / IB, gl = K * IB + l;
                Zs[l][c] = (gl < r && j0 + c < k) ? Z[gl + (int64_t)r * (j0 + c)] : T(0);
            }
            __syncthreads();
#pragma unroll 8
            for (int l = 0; l < IB; ++l) {
                const T lv = Ls[tr][l];
#pragma unroll
                for (int q = 0; q < NQ; ++q) acc[q] -= lv * Zs[l][tc + 8 * q];
            }
        }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < NQ; ++q) Zs[tr][tc + 8 * q] = acc[q];
        for (int q = threadIdx.x; q < IB * IB; q += 256) {
            const int rr = q % IB, l = q / IB, g1 = I * IB + rr, g2 = I * IB + l;
            Ls[rr][l] = (rr > l && g1 < r) ? Si[g1 + (int64_t)r * g2] : T(0);
        }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
            const int c = tc + 8 * q;
            T v = Zs[tr][c];
            for (int l = 0; l < tr; ++l) v += Ls[tr][l] * Zs[l][c];
            if (gi < r && j0 + c < k) Z[gi + (int64_t)r * (j0 + c)] = v;
        }
    }
}

// S = -X Z into the SCI pool, -X D X^T of an LDL box (TS x TS tiles, K = r by 16)
template <typename T, int TS>
__global__ void __launch_bounds__(256) be_schur_kernel(BatchElimArgs a) {
    constexpr int Q = TS / 16;
    __shared__ T As[16][TS + 1];
    __shared__ T Bs[16][TS + 1];
    const int e = blockIdx.z;
    const ElimDesc d = a.ed[e];
    const int k = d.k, r = d.r;
    if (k == 0 || d.sci_out < 0) return;
    const int i0 = blockIdx.x * TS, j0 = blockIdx.y * TS;
    if (i0 >= k || j0 >= k) return;
    const T* X = static_cast<const T*>(a.pool) + d.X_out;
    const T* Z = static_cast<const T*>(a.pool) + d.Y_out;
    const T* Dv = static_cast<const T*>(a.pool) + d.D_out;
    const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
    T acc[Q][Q] = {};
    for (int l0 = 0; l0 < r; l0 += 16) {
        for (int q = threadIdx.x; q < TS * 16; q += 256) {
            const int rr = q % TS, l = q / TS;
            const int i = i0 + rr, kx = l0 + l, jj = j0 + rr;
            As[l][rr] = (i < k && kx < r) ? X[i + (int64_t)k * kx] : T(0);
            Bs[l][rr] = (jj < k && kx < r) ? (d.ldl ? X[jj + (int64_t)k * kx] * Dv[kx] : Z[kx + (int64_t)r * jj]) : T(0);
        }
        __syncthreads();
#pragma unroll
        for (int l = 0; l < 16; ++l) {
            T av[Q], bv[Q];
#pragma unroll
            for (int q = 0; q < Q; ++q) av[q] = As[l][tx + 16 * q];
#pragma unroll
            for (int q = 0; q < Q; ++q) bv[q] = Bs[l][ty + 16 * q];
#pragma unroll
            for (int p = 0; p < Q; ++p)
#pragma unroll
                for (int q = 0; q < Q; ++q) acc[p][q] += av[p] * bv[q];
        }
        __syncthreads();
    }
    T* S = static_cast<T*>(a.sci_pool) + d.sci_out;
    for (int p = 0; p < Q; ++p)
        for (int q = 0; q < Q; ++q) {
            const int i = i0 + tx + 16 * p, jj = j0 + ty + 16 * q;
            if (i < k && jj < k) S[i + (int64_t)k * jj] = -acc[p][q];
        }
}

// Y = D^{-1} Z in place, and T
template <typename T>
__global__ void be_finish_kernel(BatchElimArgs a) {
    const int e = blockIdx.y;
    const ElimDesc d = a.ed[e];
    const EBox<T> Bx(a, e);
    const int k = Bx.k, r = Bx.r;
    T* pool = static_cast<T*>(a.pool);
    const T* Dv = pool + d.D_out;
    T* Yo = pool + d.Y_out;
    T* To = pool + d.T_out;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const int64_t t0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (!d.ldl)
        for (int64_t q = t0; q < (int64_t)r * k; q += stride) Yo[q] /= Dv[q % r];
    for (int64_t q = t0; q < (int64_t)k * r; q += stride) To[q] = Bx.Tm[q];
}

template <typename T>
cudaError_t big_elim_batch(const BatchElimArgs& a, int max_n, int max_k, int max_r, int small_r, cudaStream_t st) {
    const int nb = a.nbox;
    if (nb == 0) return cudaSuccess;
    note_launch();
    be_gather_kernel<T><<<dim3((unsigned)std::min<int64_t>(((int64_t)max_n * max_n + 255) / 256, 1024), nb), 256, 0, st>>>(a);
    note_launch();
    be_T_kernel<T><<<nb, 256, 0, st>>>(a);
    // small tiles while 64 x 64 ones would leave SMs idle (n = 64, 64-bit: 4
    // boxes of 348 give 36 tiles of 64, 484 of 32)
    const int tm = std::max(max_k, max_r);
    const bool small = (int64_t)((tm + 63) / 64) * ((tm + 63) / 64) * nb < 2 * a.num_sms;
    const int ts = small ? 32 : 64, tk = (max_k + ts - 1) / ts, tr = (max_r + ts - 1) / ts;
    auto gemm_op = [&](int op, int mt, int nt) {
        note_launch();
        if (small) be_gemm_kernel<T, 32><<<dim3(mt, nt, nb), 256, 0, st>>>(a, op);
        else be_gemm_kernel<T, 64><<<dim3(mt, nt, nb), 256, 0, st>>>(a, op);
    };
    // FP32: the products of Lemma 2.4 and the Schur update on the tensor cores
    TcGemmProb* probs = static_cast<TcGemmProb*>(a.gemm_probs);
    const bool tcg = sizeof(T) == 4 && probs != nullptr;
    auto tc_op = [&](int op, int mm, int nn) -> cudaError_t {
        note_launch();
        be_probs_kernel<<<(nb + 127) / 128, 128, 0, st>>>(a, op, probs + (int64_t)op * nb);
        return launch_tc_gemm(probs + (int64_t)op * nb, nb, mm, nn, a.status, DEV_TIMEOUT, st);
    };
    if (max_k > 0 && tcg) {
        cudaError_t e;
        if ((e = tc_op(0, max_k, max_r)) != cudaSuccess) return e;
        if ((e = tc_op(1, max_r, max_r)) != cudaSuccess) return e;
        if ((e = tc_op(2, max_r, max_r)) != cudaSuccess) return e;
        if ((e = tc_op(3, max_r, max_k)) != cudaSuccess) return e;
    } else if (max_k > 0) {
        gemm_op(0, tk, tr);
        gemm_op(1, tr, tr);
        gemm_op(2, tr, tr);
        gemm_op(3, tr, tk);
    }
    if (small_r > 0) {
        const cudaError_t e = launch_be_factor<T>(a, small_r, st);
        if (e != cudaSuccess) return e;
    }
    for (int j0 = 0; max_r > a.factor_max_r && j0 < max_r; j0 += 32) {
        const size_t ps = be_panel_smem<T>(max_r - j0);
        note_launch();
        if (ps <= 200 * 1024) {
            cudaError_t e = cudaFuncSetAttribute(be_panel_cluster_kernel<T>,
                                                 cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
            if (e != cudaSuccess) return e;
            cudaLaunchConfig_t cfg{};
            cfg.gridDim = dim3((unsigned)(nb * PCL));
            cfg.blockDim = dim3(256);
            cfg.dynamicSmemBytes = ps;
            cfg.stream = st;
            cudaLaunchAttribute at{};
            at.id = cudaLaunchAttributeClusterDimension;
            at.val.clusterDim.x = PCL;
            at.val.clusterDim.y = at.val.clusterDim.z = 1;
            cfg.attrs = &at;
            cfg.numAttrs = 1;
            if ((e = cudaLaunchKernelEx(&cfg, be_panel_cluster_kernel<T>, a, j0)) != cudaSuccess) return e;
        } else {
            be_panel_kernel<T><<<nb, PNT, 0, st>>>(a, j0);
        }
        note_launch();
        be_swap_trsm_kernel<T><<<dim3((max_r + 127) / 128, nb), 128, 0, st>>>(a, j0);
        const int rest = max_r - j0 - 32;
        if (rest > 0) {
            note_launch();
            be_update_kernel<T><<<dim3((rest + 63) / 64, (rest + 63) / 64, nb), 256, 0, st>>>(a, j0);
        }
    }
    note_launch();
    be_lu_out_kernel<T><<<dim3((unsigned)std::min<int64_t>(((int64_t)max_r * max_r + 255) / 256, 512), nb), 256, 0, st>>>(a);
    const int rb = (max_r + IB - 1) / IB;
    note_launch();
    be_dinv_kernel<T, false><<<dim3(rb, nb), 32, 0, st>>>(a);
    note_launch();
    be_dinv_kernel<T, true><<<dim3(rb, nb), 32, 0, st>>>(a);
    if (max_k > 0) {
        // rows (columns) of a substitution's CTA: 64, or 16 while 64 would
        // leave SMs without one (n = 200, 64-bit: 16 boxes of k ~ 500)
        const int rt = (int64_t)((max_k + 63) / 64) * nb < 2 * a.num_sms ? 16 : 64;
        const dim3 gt((max_k + rt - 1) / rt, nb);
        note_launch();
        if (rt == 16) be_trsm_x_kernel<T, 16><<<gt, 256, 0, st>>>(a);
        else be_trsm_x_kernel<T, 64><<<gt, 256, 0, st>>>(a);
        note_launch();
        if (rt == 16) be_trsm_z_kernel<T, 16><<<gt, 256, 0, st>>>(a);
        else be_trsm_z_kernel<T, 64><<<gt, 256, 0, st>>>(a);
        if (tcg) {
            const cudaError_t e = tc_op(4, max_k, max_k);
            if (e != cudaSuccess) return e;
        } else {
            note_launch();
            if (small) be_schur_kernel<T, 32><<<dim3(tk, tk, nb), 256, 0, st>>>(a);
            else be_schur_kernel<T, 64><<<dim3(tk, tk, nb), 256, 0, st>>>(a);
        }
    }
    // inverses of the unit triangular factors, by doubling the inverted blocks
    for (int s = IB; s < max_r; s *= 2) {
        const int nt = s / IB;
        const dim3 g(nt * nt, (max_r + 2 * s - 1) / (2 * s), nb);
        note_launch();
        be_inv_level_kernel<T, false, 1><<<g, 256, 0, st>>>(a, s);
        note_launch();
        be_inv_level_kernel<T, false, 2><<<g, 256, 0, st>>>(a, s);
        note_launch();
        be_inv_level_kernel<T, false, 3><<<g, 256, 0, st>>>(a, s);
        note_launch();
        be_inv_level_kernel<T, false, 4><<<g, 256, 0, st>>>(a, s);
        note_launch();
        be_inv_level_kernel<T, true, 1><<<g, 256, 0, st>>>(a, s);
        note_launch();
        be_inv_level_kernel<T, true, 2><<<g, 256, 0, st>>>(a, s);
        note_launch();
        be_inv_level_kernel<T, true, 3><<<g, 256, 0, st>>>(a, s);
        note_launch();
        be_inv_level_kernel<T, true, 4><<<g, 256, 0, st>>>(a, s);
    }
    note_launch();
    be_finish_kernel<T><<<dim3((unsigned)std::clamp<int64_t>(((int64_t)max_k * max_r + 255) / 256, 1, 512), nb), 256,
                           0, st>>>(a);
    return cudaGetLastError();
}

#define HIF_INST(T)                                                                                            \
    template cudaError_t big_ygen<T>(const BigArgs&, int, int64_t, cudaStream_t);                              \
    template cudaError_t big_rho<T>(const BigArgs&, int, int, int, cudaStream_t);                              \
    template cudaError_t big_add<T>(void*, const void*, int64_t, cudaStream_t);                                \
    template cudaError_t big_qr_init<T>(const BigArgs&, int, int, cudaStream_t);                               \
    template cudaError_t big_qr_step<T>(const BigArgs&, int, int, int, cudaStream_t);                          \
    template cudaError_t big_qp_panel<T>(const BigArgs&, int, int, int, int&, cudaStream_t);                   \
    template cudaError_t big_finish<T>(const BigArgs&, int, int, cudaStream_t);                                \
    template cudaError_t big_elim_batch<T>(const BatchElimArgs&, int, int, int, int, cudaStream_t);               \
    template int be_factor_max_r<T>();
HIF_INST(double)
HIF_INST(float)

}  // namespace hif
