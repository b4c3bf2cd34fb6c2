// Apply / solve sweeps of the factorization in factored form (sm_103a).
//
// F^{-1} = V_0 ... V_last D^{-1} U_last^T ... U_0^T and F = U_0^{-T} ... D ...
// V_0^{-1} (Eqs. (3.2), (4.1), (4.2)).  One launch per sublevel and direction:
// a box's skeleton and redundant entries of the working vectors are gathered
// into shared memory, the box's small factors (T, L, U, X, Y, D of Lemmas 2.1
// and 2.3) are streamed once from HBM, and the result is scattered back.
// Boxes of one sublevel touch disjoint DOFs.  The diagonal D^{-1} (or D) is
// fused into the sweep that last touches a box's redundant DOFs.
#include <algorithm>

#include "hif_common.cuh"
#include "launch.h"

namespace hif {

enum SweepMode {
    SOLVE_UP = 0, SOLVE_DOWN = 1, APPLY_UP = 2, APPLY_DOWN = 3,
    SOLVET_UP = 4, SOLVET_DOWN = 5, APPLYT_UP = 6, APPLYT_DOWN = 7
};

// For an LDL box (symmetric A, Sec. 5: P B_rr P^T = L D L^T, U = L^T P,
// Y = X^T) the box's factors are symmetric, so the transposed operation of a
// pass is the pass itself: solve_down = solve^T_down, solve^T_up = solve_up,
// apply_up = apply^T_up, apply^T_down = apply_down.  Those four bodies read
// only T, X, D, the permutation and L or L^{-1} (packed in one array: L in the
// strict lower triangle, L^{-1} transposed in the strict upper one).
__host__ __device__ constexpr int ldl_mode(int m) {
    return m == SOLVE_DOWN ? SOLVET_DOWN : m == SOLVET_UP ? SOLVE_UP : m == APPLY_UP ? APPLYT_UP
         : m == APPLYT_DOWN ? APPLY_DOWN : m;
}

// ---- a box on a cluster of CTAs ------------------------------------------------
//
// What bounds a pass: with one right-hand side the factors are read once for
// one FMA per element, so it is the latency of those reads and the number of
// bytes in flight; with eight 64-bit ones it is the FP64 pipe (2 FMA per clock
// and SM).  The three products of a pass depend on one another, and the upper
// sublevels have few boxes.  So
//  - a box is spread over a cluster of up to 8 CTAs that exchange the vectors
//    between the products through distributed shared memory (one launch per
//    pass, two cluster barriers in a solve pass, one in an apply pass),
//  - the vectors sit in shared memory one DOF after the other with the NC
//    right-hand sides adjacent, and a factor element is read once for all of
//    them (blockIdx.y takes the next NC),
//  - products with M as stored give a lane a row and the warps of a tile of 32
//    rows equal parts of the columns; products with M^T give a warp R columns
//    of M, the lanes along them, and add R x NC sums over the lanes by halving
//    exchanges.
// Measured on a GB300 (one F^{-1}, before with one CTA and one right-hand side
// at a time per box, and now): n = 512, 64-bit factors, 8 right-hand sides
// 15.2 -> 7.2 ms (3.1 ms of it FP64 pipe), one 10.0 -> 1.5 ms; n = 256 at
// eps = 1e-9, one, 5.0 -> 0.7 ms; n = 1024, 32-bit, 8: 12 -> 2.1 ms; n = 64, 64-bit,
// one: 0.50 -> 0.16 ms.
// Row tiles of 32 go to the CTAs of a cluster in turn.  The order of every sum
// depends on the box and the launch shape of its sublevel only, not on the
// number of right-hand sides: R and with it the first column that the lanes
// take of a transposed triangular product do depend on it, but that only turns
// the columns round the lanes, and the tree of exchanges (distances 16, 8, 4, 2,
// 1) pairs the same sums however they are turned.

namespace {

template <typename T, int NC> struct alignas(sizeof(T) * NC > 16 ? 16 : sizeof(T) * NC) Row { T v[NC]; };

struct Team {                   // the CTAs of one box
    int rank, size;
};

__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }

__device__ __forceinline__ void team_sync(const Team& tm) {
    if (tm.size == 1) {
        __syncthreads();
    } else {
        cluster_arrive();
        cluster_wait();
    }
}

__device__ __forceinline__ uint32_t peer_addr(const void* p, int rank) {
    uint32_t out;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(out) : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
    return out;
}
__device__ __forceinline__ void st_peer(uint32_t a, double v) {
    asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(a), "d"(v) : "memory");
}
__device__ __forceinline__ void st_peer(uint32_t a, float v) {
    asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory");
}
// *p = v in every CTA of the team (p: this CTA's shared memory)
template <typename T>
__device__ __forceinline__ void put_all(const Team& tm, T* p, T v) {
    if (tm.size == 1) {
        *p = v;
        return;
    }
    for (int q = 0; q < tm.size; ++q) st_peer(peer_addr(p, q), v);
}

// v[0 .. CNT) summed over the lanes: while more than one sum is left, a lane
// keeps half of them and gives the others to its partner, so lane L ends with
// sum L / (32 / CNT) in v[0].
template <typename T, int CNT, int OFF, int V>
__device__ __forceinline__ void lane_sums(T (&v)[V], int lane) {
    if constexpr (OFF > 0) {
        if constexpr (CNT > 1) {
            constexpr int H = CNT / 2;
            const bool hi = lane & OFF;
#pragma unroll
            for (int e = 0; e < H; ++e) {
                const T give = hi ? v[e] : v[e + H], keep = hi ? v[e + H] : v[e];
                v[e] = keep + __shfl_xor_sync(0xffffffffu, give, OFF);
            }
            lane_sums<T, H, OFF / 2>(v, lane);
        } else {
            v[0] += __shfl_xor_sync(0xffffffffu, v[0], OFF);
            lane_sums<T, 1, OFF / 2>(v, lane);
        }
    }
}

// How op(M) is read: element (i, l) at M[i + ld l], or M[l + ld i] when
// trans; tri: +1 / -1 keep only l < i / l > i.
template <typename T>
struct Op {
    const T* M;
    int64_t ld;
    bool trans;
    int tri;
};

// f(i, c, sum_l op(M)[i, l] in[pidx ? pidx[l] : l][c]) for this CTA's rows i of
// [0, p); op(M) is p x q.  With `rows` the operator's row is rows[i].  red: 32
// NC values per warp.  All threads of the CTA; ends with a CTA barrier.
template <typename T, int NC, int U, typename F>
__device__ __forceinline__ void product(const Team& tm, const Op<T>& A, int p, int q, const Row<T, NC>* in,
                                        const int* pidx, const int* rows, T* red, F f) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int tiles = (p + 31) / 32, mine = tiles > tm.rank ? (tiles - tm.rank + tm.size - 1) / tm.size : 0;
    if (!A.trans) {
        const int ks = mine > 0 && mine < nw ? nw / mine : 1;      // parts of the columns per tile
        for (int it = warp; it < mine * ks; it += nw) {
            const int b = 32 * (tm.rank + tm.size * (it / ks)), i = b + lane, ic = i < p ? i : p - 1;
            const int lo = A.tri < 0 ? b + 1 : 0, hi = A.tri > 0 ? min(q, b + 31) : q;
            const int len = hi > lo ? (hi - lo + ks - 1) / ks : 0;
            int l = lo + (it % ks) * len;
            const int le = min(hi, l + len);
            T acc[NC];
#pragma unroll
            for (int c = 0; c < NC; ++c) acc[c] = T(0);
            const T* col = A.M + ic + A.ld * l;
            for (; l < le; l += U, col += A.ld * U) {
                T m[U];
#pragma unroll
                for (int u = 0; u < U; ++u) m[u] = l + u < le ? __ldg(col + A.ld * u) : T(0);
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    // (terms are left out, not multiplied by zero: Inf and NaN stay in their rows)
                    if (l + u >= le) break;
                    const Row<T, NC> x = in[pidx ? pidx[l + u] : l + u];
                    if (A.tri > 0 ? l + u >= ic : A.tri < 0 && l + u <= ic) continue;
#pragma unroll
                    for (int c = 0; c < NC; ++c) acc[c] += m[u] * x.v[c];
                }
            }
            if (ks == 1) {
                if (i < p)
#pragma unroll
                    for (int c = 0; c < NC; ++c) f(i, c, acc[c]);
            } else {
#pragma unroll
                for (int c = 0; c < NC; ++c) red[(it * NC + c) * 32 + lane] = acc[c];
            }
        }
        if (ks > 1) {
            __syncthreads();
            for (int e = threadIdx.x; e < mine * NC * 32; e += blockDim.x) {
                const int t = e / (NC * 32), c = e / 32 % NC, i = 32 * (tm.rank + tm.size * t) + e % 32;
                if (i >= p) continue;
                T s = T(0);
                for (int z = 0; z < ks; ++z) s += red[((t * ks + z) * NC + c) * 32 + e % 32];
                f(i, c, s);
            }
        }
    } else {
        constexpr int R = NC == 1 ? 8 : NC == 2 && sizeof(T) == 8 ? 4 : 16 / NC, V = R * NC, G = 32 / R;   // columns of M and sums per warp
        for (int it = warp; it < mine * G; it += nw) {
            const int i0 = 32 * (tm.rank + tm.size * (it / G)) + R * (it % G);
            if (i0 >= p) continue;
            const int lo = A.tri < 0 ? i0 + 1 : 0, hi = A.tri > 0 ? min(q, i0 + R - 1) : q;
            const T* col[R];
#pragma unroll
            for (int u = 0; u < R; ++u) {
                const int i = min(i0 + u, p - 1);
                col[u] = A.M + A.ld * (rows ? rows[i] : i);
            }
            T v[V];
#pragma unroll
            for (int e = 0; e < V; ++e) v[e] = T(0);
#pragma unroll (NC == 8 ? 4 : 2)
            for (int l = lo + lane; l < hi; l += 32) {
                T m[R];
#pragma unroll
                for (int u = 0; u < R; ++u) m[u] = __ldg(col[u] + l);
                const Row<T, NC> x = in[pidx ? pidx[l] : l];
#pragma unroll
                for (int u = 0; u < R; ++u) {
                    if (A.tri > 0 ? l >= i0 + u : A.tri < 0 && l <= i0 + u) continue;
#pragma unroll
                    for (int c = 0; c < NC; ++c) v[u * NC + c] += m[u] * x.v[c];
                }
            }
            lane_sums<T, V, 16>(v, lane);
            const int e = lane / (32 / V), i = i0 + e / NC;
            if (lane % (32 / V) == 0 && i < p) f(i, e % NC, v[0]);
        }
    }
    __syncthreads();
}

}  // namespace

// U: columns in flight per lane of a product with M as stored.  The big variant
// (512 threads, U = 16) is for the few wide boxes of the upper sublevels,
// where a CTA streams its rows alone and only loads in flight help; elsewhere
// fewer registers and more CTAs per SM do (n = 512, one right-hand side, 1024
// boxes of ~190 rows: 141 us at 162 registers, 100 us at 80).
template <typename T, int NC, bool BIG>
__global__ void __launch_bounds__(BIG ? 512 : 256, BIG ? 1 : sizeof(T) == 8 ? (NC == 8 ? 2 : 3) : 4)
sweep_kernel(SweepArgs a) {
    constexpr int U = BIG ? 16 : 8;
    const Team tm{(int)(blockIdx.x % a.cluster), a.cluster};
    if (tm.size > 1) cluster_arrive();               // waited for before the first store to a peer
    const BoxFac bf = a.boxes[blockIdx.x / a.cluster];
    const int k = bf.k, r = bf.r, c0 = blockIdx.y * NC, nr = min(NC, a.nrhs - c0);
    extern __shared__ __align__(16) unsigned char smem_raw[];
    using V = Row<T, NC>;
    T* red = reinterpret_cast<T*>(smem_raw);
    V* xs = reinterpret_cast<V*>(red + (blockDim.x / 32) * 32 * NC);
    V* xr = xs + k;
    V* tmp = xr + r;
    T* x = static_cast<T*>(a.x) + c0;
    const int64_t stride = a.ldx;                    // x: one DOF after the other, right-hand sides adjacent
    const int* sk = a.sk_ids + bf.sk_off;
    const int* rd = a.rd_ids + bf.rd_off;
    const int* perm = a.perm + bf.piv_off;
    const T* pool = static_cast<const T*>(a.pool);
    const T* D = pool + bf.D_off;
    const int mode = bf.ldl ? ldl_mode(a.mode) : a.mode;
    const bool ldl = bf.ldl != 0;
    const Op<T> Tn{pool + bf.T_off, k, false, 0}, Tt{pool + bf.T_off, k, true, 0};       // T: k x r
    const Op<T> Xn{pool + bf.X_off, k, false, 0}, Xt{pool + bf.X_off, k, true, 0};       // X: k x r
    const Op<T> Yn{pool + bf.Y_off, r, false, 0}, Yt{pool + bf.Y_off, r, true, 0};       // Y: r x k
    const T* LU = pool + bf.LU_off;
    const T* LUi = pool + bf.LUi_off;
    auto gather = [&](V* dst, const int* ids, int cnt) {
        for (int e = threadIdx.x; e < cnt * NC; e += blockDim.x) {
            const int i = e / NC, c = e % NC;
            dst[i].v[c] = c < nr ? x[ids[i] * stride + c] : T(0);
        }
        __syncthreads();
    };

    if (mode == SOLVE_UP || mode == SOLVE_DOWN || mode == SOLVET_UP || mode == SOLVET_DOWN) {
        // xr <- (D^{-1}) xr - op(M1) xs; xr <- op(unit factor)^{-1} xr; xs -= op(M2) xr
        //   SOLVE_UP    U^T = Q^T then R^T:   M1 = T^T, L^{-1} P,   M2 = X
        //   SOLVE_DOWN  D^{-1}, V = Q S:      M1 = Y,   U^{-1},     M2 = T
        //   SOLVET_UP   V^T = S^T Q^T:        M1 = T^T, U^{-T},     M2 = Y^T
        //   SOLVET_DOWN D^{-T}, U = Q R:      M1 = X^T, P^T L^{-T}, M2 = T
        const bool down = mode == SOLVE_DOWN || mode == SOLVET_DOWN;
        const Op<T> M1 = mode == SOLVE_DOWN ? Yn : mode == SOLVET_DOWN ? Xt : Tt;
        const Op<T> M2 = mode == SOLVE_UP ? Xn : mode == SOLVET_UP ? Yt : Tn;
        // L^{-1}: strict lower of LUi (LU box) or transposed in its upper (LDL box)
        const Op<T> B = mode == SOLVE_UP     ? Op<T>{LUi, r, ldl, 1}
                        : mode == SOLVE_DOWN ? Op<T>{LUi, r, false, -1}
                        : mode == SOLVET_UP  ? Op<T>{LUi, r, true, 1}
                                             : Op<T>{LUi, r, !ldl, -1};
        gather(xs, sk, k);
        if (tm.size > 1) cluster_wait();
        product<T, NC, U>(tm, M1, r, k, xs, nullptr, nullptr, red, [&](int i, int c, T s) {
            T v = c < nr ? x[rd[i] * stride + c] : T(0);
            if (down) v /= D[i];
            put_all(tm, &xr[i].v[c], v - s);
        });
        team_sync(tm);
        const int* pin = mode == SOLVE_UP ? perm : nullptr;
        product<T, NC, U>(tm, B, r, r, xr, pin, nullptr, red, [&](int i, int c, T s) {
            const T v = xr[pin ? pin[i] : i].v[c] + s;
            const int j = mode == SOLVET_DOWN ? perm[i] : i;
            put_all(tm, &tmp[j].v[c], v);
            if (c < nr) x[rd[j] * stride + c] = v;
        });
        team_sync(tm);
        product<T, NC, U>(tm, M2, k, r, tmp, nullptr, nullptr, red, [&](int i, int c, T s) {
            if (c < nr) x[sk[i] * stride + c] = xs[i].v[c] - s;
        });
    } else {
        // xs += op(M2) xr; xr <- op(unit factor) xr; xr += op(M1) xs (times D)
        //   APPLY_UP    V^{-1} = S^{-1} Q^{-1}, D:  M2 = T,   U,     M1 = Y
        //   APPLY_DOWN  U^{-T} = Q^{-T} R^{-T}:     M2 = X,   P^T L, M1 = T^T
        //   APPLYT_UP   U^{-1} = R^{-1} Q^{-1}, D:  M2 = T,   L^T P, M1 = X^T
        //   APPLYT_DOWN V^{-T} = Q^{-T} S^{-T}:     M2 = Y^T, U^T,   M1 = T^T
        const bool up = mode == APPLY_UP || mode == APPLYT_UP;
        const Op<T> M2 = mode == APPLY_DOWN ? Xn : mode == APPLYT_DOWN ? Yt : Tn;
        const Op<T> M1 = mode == APPLY_UP ? Yn : mode == APPLYT_UP ? Xt : Tt;
        const Op<T> B = mode == APPLY_UP     ? Op<T>{LU, r, false, -1}
                        : mode == APPLY_DOWN ? Op<T>{LU, r, false, 1}
                        : mode == APPLYT_UP  ? Op<T>{LU, r, true, -1}
                                             : Op<T>{LU, r, true, 1};
        gather(xr, rd, r);
        if (tm.size > 1) cluster_wait();
        product<T, NC, U>(tm, M2, k, r, xr, nullptr, nullptr, red, [&](int i, int c, T s) {
            const T v = (c < nr ? x[sk[i] * stride + c] : T(0)) + s;
            put_all(tm, &xs[i].v[c], v);
            if (c < nr) x[sk[i] * stride + c] = v;
        });
        // a row of the unit factor's product stays with its CTA
        const int* pin = mode == APPLYT_UP ? perm : nullptr;
        product<T, NC, U>(tm, B, r, r, xr, pin, nullptr, red, [&](int i, int c, T s) {
            tmp[i].v[c] = xr[pin ? pin[i] : i].v[c] + s;
        });
        team_sync(tm);
        const int* pout = mode == APPLY_DOWN ? perm : nullptr;
        product<T, NC, U>(tm, M1, r, k, xs, nullptr, pout, red, [&](int i, int c, T s) {
            const int j = pout ? pout[i] : i;
            T v = tmp[i].v[c] + s;
            if (up) v *= D[j];
            if (c < nr) x[rd[j] * stride + c] = v;
        });
    }
}

size_t sweep_smem_bytes(int k2r, int nc, int threads, int elem) {
    return ((size_t)threads + k2r) * nc * elem + 64;
}

namespace {
template <typename T, int NC, bool BIG>
cudaError_t launch_nc(const SweepArgs& a, int nbox, int threads, size_t smem, cudaStream_t st) {
    // The kernel's dynamic shared-memory limit is only ever raised, to the
    // one fixed ceiling: launches captured in a CUDA graph keep their own
    // sizes, and no later launch may lower the limit below what a captured
    // node needs.
    if (smem > kSweepSmemMax) return cudaErrorInvalidValue;
    if (smem > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(sweep_kernel<T, NC, BIG>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)kSweepSmemMax);
        if (e != cudaSuccess) return e;
    }
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)(nbox * a.cluster), (unsigned)((a.nrhs + NC - 1) / NC));
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = (unsigned)a.cluster;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = a.cluster > 1 ? 1 : 0;
    note_launch();
    return cudaLaunchKernelEx(&cfg, sweep_kernel<T, NC, BIG>, a);
}
}  // namespace

template <typename T>
cudaError_t launch_sweep(const SweepArgs& a, int nbox, int nc, int threads, size_t smem, cudaStream_t st) {
    if (nbox == 0) return cudaSuccess;
    if (threads < 32 || threads > 512 || threads % 32 || a.cluster < 1 || a.cluster > 8)
        return cudaErrorInvalidValue;
    const bool big = threads > 256;
    switch (nc) {
        case 1: return big ? launch_nc<T, 1, true>(a, nbox, threads, smem, st) : launch_nc<T, 1, false>(a, nbox, threads, smem, st);
        case 2: return big ? launch_nc<T, 2, true>(a, nbox, threads, smem, st) : launch_nc<T, 2, false>(a, nbox, threads, smem, st);
        case 4: return big ? launch_nc<T, 4, true>(a, nbox, threads, smem, st) : launch_nc<T, 4, false>(a, nbox, threads, smem, st);
        case 8: return big ? launch_nc<T, 8, true>(a, nbox, threads, smem, st) : launch_nc<T, 8, false>(a, nbox, threads, smem, st);
        default: return cudaErrorInvalidValue;
    }
}

template cudaError_t launch_sweep<double>(const SweepArgs&, int, int, int, size_t, cudaStream_t);
template cudaError_t launch_sweep<float>(const SweepArgs&, int, int, int, size_t, cudaStream_t);

// ---- wide boxes: the same passes spread over the GPU ------------------------
//
// A box with k + r in the thousands keeps one CTA busy for its whole pass
// while the other SMs idle, so the wide boxes of a sublevel take their pass as
// a sequence of stage launches over (box, 64-row tile): gather, matrix-vector
// products with T, X, Y, the triangular products (I + strict op(M)) with the
// unit factors or their inverses, permutations, scatter.  Each box keeps its
// three vectors in a global work space: B0 = skeleton part (k x nr), B1 =
// redundant part (r x nr), B2 = a second redundant vector.  Right-hand sides
// go 16 at a time.  The stage order of every mode is that of sweep_kernel.

namespace {

constexpr int WR = 16;      // right-hand sides per stage launch

template <typename T>
struct WideView {
    int k, r;
    T* B[3];
    int len[3];
    __device__ WideView(const WideArgs& a, int e, const BoxFac& bf) {
        k = bf.k;
        r = bf.r;
        T* base = static_cast<T*>(a.ws) + a.ws_off[e] * (int64_t)a.nr;
        B[0] = base;
        B[1] = base + (int64_t)k * a.nr;
        B[2] = B[1] + (int64_t)r * a.nr;
        len[0] = k;
        len[1] = r;
        len[2] = r;
    }
};

template <typename T>
__device__ __forceinline__ const T* wide_mat(const WideArgs& a, const BoxFac& bf, int mat, int64_t& ld) {
    const T* pool = static_cast<const T*>(a.pool);
    switch (mat) {
        case 0: ld = bf.k; return pool + bf.T_off;       // T: k x r
        case 1: ld = bf.k; return pool + bf.X_off;       // X: k x r
        case 2: ld = bf.r; return pool + bf.Y_off;       // Y: r x k
        case 3: ld = bf.r; return pool + bf.LU_off;      // unit factors, r x r
        default: ld = bf.r; return pool + bf.LUi_off;    // their inverses, r x r
    }
}

}  // namespace

template <typename T>
__global__ void wide_gather_kernel(WideArgs a, int div_d) {
    const int e = blockIdx.y;
    const BoxFac bf = a.boxes[e];
    WideView<T> v(a, e, bf);
    const T* x = static_cast<const T*>(a.x);
    const int* sk = a.sk_ids + bf.sk_off;
    const int* rd = a.rd_ids + bf.rd_off;
    const T* D = static_cast<const T*>(a.pool) + bf.D_off;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < (int64_t)(v.k + v.r) * a.nr; q += stride) {
        const int c = (int)(q / (v.k + v.r)), i = (int)(q % (v.k + v.r));
        if (i < v.k) v.B[0][i + (int64_t)v.k * c] = x[sk[i] * a.ldx + c];
        else {
            const int j = i - v.k;
            const T val = x[rd[j] * a.ldx + c];
            v.B[1][j + (int64_t)v.r * c] = div_d ? val / D[j] : val;
        }
    }
}

template <typename T>
__global__ void wide_scatter_kernel(WideArgs a, int xr_buf, int mul_d) {
    const int e = blockIdx.y;
    const BoxFac bf = a.boxes[e];
    WideView<T> v(a, e, bf);
    T* x = static_cast<T*>(a.x);
    const int* sk = a.sk_ids + bf.sk_off;
    const int* rd = a.rd_ids + bf.rd_off;
    const T* D = static_cast<const T*>(a.pool) + bf.D_off;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < (int64_t)(v.k + v.r) * a.nr; q += stride) {
        const int c = (int)(q / (v.k + v.r)), i = (int)(q % (v.k + v.r));
        if (i < v.k) x[sk[i] * a.ldx + c] = v.B[0][i + (int64_t)v.k * c];
        else {
            const int j = i - v.k;
            const T val = v.B[xr_buf][j + (int64_t)v.r * c];
            x[rd[j] * a.ldx + c] = mul_d ? val * D[j] : val;
        }
    }
}

// out = P in (inverse 0: out[i] = in[perm[i]]) or P^T in (out[perm[i]] = in[i])
template <typename T>
__global__ void wide_perm_kernel(WideArgs a, int out_buf, int in_buf, int inverse) {
    const int e = blockIdx.y;
    const BoxFac bf = a.boxes[e];
    WideView<T> v(a, e, bf);
    const int* perm = a.perm + bf.piv_off;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < (int64_t)v.r * a.nr; q += stride) {
        const int c = (int)(q / v.r), i = (int)(q % v.r);
        const int64_t o = (int64_t)v.r * c;
        if (!inverse) v.B[out_buf][i + o] = v.B[in_buf][perm[i] + o];
        else v.B[out_buf][perm[i] + o] = v.B[in_buf][i + o];
    }
}

// One product stage on rows [64 blockIdx.x, +64) of `out` for every wide box:
//   tri 0: out += s op(M) in                      (M = T, X or Y)
//   tri 1: out  = in' + strict op(M) in'          (M = LU or LUi; in' = P in
//          with perm_in, else in), opLower = lower_store != trans
// op(M)[i, l] = trans ? M[l + ld i] : M[i + ld l].  Not transposed: a thread
// per output row (coalesced column reads of M), the input staged in shared
// memory 64 rows at a time; transposed: a warp per output row (coalesced
// reads of column i of M) with warp reductions.
template <typename T, bool TRANS>
__global__ void __launch_bounds__(256) wide_mv_kernel(WideArgs a, int out_buf, int in_buf, int mat, T s, int tri,
                                                      int lower_store, int perm_in) {
    const int e = blockIdx.y;
    const BoxFac bf = a.boxes[e];
    WideView<T> v(a, e, bf);
    const int p = v.len[out_buf], q = v.len[in_buf];
    const int i0 = blockIdx.x * 64;
    if (i0 >= p) return;
    int64_t ld;
    const T* M = wide_mat<T>(a, bf, mat, ld);
    const int* perm = a.perm + bf.piv_off;
    T* out = v.B[out_buf];
    const T* in = v.B[in_buf];
    const int nr = a.nr;
    const bool opLower = (lower_store != 0) != TRANS;
    auto inval = [&](int l, int c) -> T { return in[(perm_in ? perm[l] : l) + (int64_t)q * c]; };
    if (!TRANS) {
        __shared__ T ins[64][WR + 1];
        const int tx = threadIdx.x % 64, tc = threadIdx.x / 64;      // rhs tc, tc + 4, ...
        const int i = i0 + tx;
        T acc[WR / 4];
#pragma unroll
        for (int u = 0; u < WR / 4; ++u) acc[u] = T(0);
        // tri: only l < i (opLower) or l > i contribute
        const int lbeg = tri && !opLower ? i0 + 1 : 0;
        const int lend = tri && opLower ? min(q, i0 + 64) : q;
        for (int l0 = lbeg; l0 < lend; l0 += 64) {
            __syncthreads();
            for (int z = threadIdx.x; z < 64 * WR; z += 256) {
                const int ll = z % 64, c = z / 64;
                ins[ll][c] = (l0 + ll < lend && c < nr) ? inval(l0 + ll, c) : T(0);
            }
            __syncthreads();
            if (i < p) {
                const int cnt = min(64, lend - l0);
                for (int ll = 0; ll < cnt; ++ll) {
                    const int l = l0 + ll;
                    if (tri && (opLower ? l >= i : l <= i)) continue;
                    const T m = M[i + ld * l];
#pragma unroll
                    for (int u = 0; u < WR / 4; ++u) acc[u] += m * ins[ll][tc + 4 * u];
                }
            }
        }
        if (i < p)
#pragma unroll
            for (int u = 0; u < WR / 4; ++u) {
                const int c = tc + 4 * u;
                if (c >= nr) continue;
                T* o = out + i + (int64_t)p * c;
                if (tri) *o = inval(i, c) + acc[u];
                else *o += s * acc[u];
            }
    } else {
        const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
        for (int ii = w; ii < 64; ii += 8) {
            const int i = i0 + ii;
            if (i >= p) break;
            const T* col = M + ld * i;
            T acc[WR];
#pragma unroll
            for (int c = 0; c < WR; ++c) acc[c] = T(0);
            const int lbeg = tri && !opLower ? i + 1 : 0;
            const int lend = tri && opLower ? i : q;
            for (int l = lbeg + lane; l < lend; l += 32) {
                const T m = col[l];
#pragma unroll
                for (int c = 0; c < WR; ++c)
                    if (c < nr) acc[c] += m * inval(l, c);
            }
#pragma unroll
            for (int c = 0; c < WR; ++c) acc[c] = warp_sum(acc[c]);
            if (lane < nr) {
                T val = T(0);
#pragma unroll
                for (int c = 0; c < WR; ++c)
                    if (c == lane) val = acc[c];
                T* o = out + i + (int64_t)p * lane;
                if (tri) *o = inval(i, lane) + val;
                else *o += s * val;
            }
        }
    }
}

template <typename T>
static cudaError_t wide_mv(const WideArgs& a, int nwide, int rows, int out_buf, int in_buf, int mat, bool trans,
                           T s, int tri, int lower_store, int perm_in, cudaStream_t st) {
    if (rows <= 0) return cudaSuccess;
    const dim3 g((rows + 63) / 64, nwide);
    note_launch();
    if (trans) wide_mv_kernel<T, true><<<g, 256, 0, st>>>(a, out_buf, in_buf, mat, s, tri, lower_store, perm_in);
    else wide_mv_kernel<T, false><<<g, 256, 0, st>>>(a, out_buf, in_buf, mat, s, tri, lower_store, perm_in);
    return cudaGetLastError();
}

// The pass of `mode` for the wide boxes; a.nr <= 16 right-hand sides.
template <typename T>
cudaError_t launch_wide_sweep(const WideArgs& a, int nwide, int max_k, int max_r, int mode, cudaStream_t st) {
    if (nwide == 0) return cudaSuccess;
    if (a.nr < 1 || a.nr > WR) return cudaErrorInvalidValue;
    const dim3 ge((unsigned)std::min<int64_t>(((int64_t)(max_k + max_r) * a.nr + 255) / 256, 256), nwide);
    const dim3 gp((unsigned)std::min<int64_t>(((int64_t)max_r * a.nr + 255) / 256, 256), nwide);
    cudaError_t err = cudaSuccess;
    auto chk = [&](cudaError_t x) { if (err == cudaSuccess) err = x; };
    auto mv = [&](int rows, int ob, int ib, int mat, bool tr, T sg) { chk(wide_mv<T>(a, nwide, rows, ob, ib, mat, tr, sg, 0, 0, 0, st)); };
    auto tri = [&](int ob, int ib, int mat, bool lower_store, bool tr, bool pin) {
        chk(wide_mv<T>(a, nwide, max_r, ob, ib, mat, tr, T(1), 1, lower_store ? 1 : 0, pin ? 1 : 0, st));
    };
    auto perm = [&](int ob, int ib, bool inv) {
        note_launch();
        wide_perm_kernel<T><<<gp, 256, 0, st>>>(a, ob, ib, inv ? 1 : 0);
        chk(cudaGetLastError());
    };
    auto gather = [&](bool divd) {
        note_launch();
        wide_gather_kernel<T><<<ge, 256, 0, st>>>(a, divd ? 1 : 0);
        chk(cudaGetLastError());
    };
    auto scatter = [&](int xr_buf, bool muld) {
        note_launch();
        wide_scatter_kernel<T><<<ge, 256, 0, st>>>(a, xr_buf, muld ? 1 : 0);
        chk(cudaGetLastError());
    };
    enum { MT = 0, MX = 1, MY = 2, MLU = 3, MLUI = 4 };
    switch (mode) {
        case SOLVE_UP:        // xr -= T^T xs; xr <- L^{-1} P xr; xs -= X xr
            gather(false);
            mv(max_r, 1, 0, MT, true, T(-1));
            tri(2, 1, MLUI, true, false, true);
            mv(max_k, 0, 2, MX, false, T(-1));
            scatter(2, false);
            break;
        case SOLVE_DOWN:      // xr /= D; xr -= Y xs; xr <- U'^{-1} xr; xs -= T xr
            gather(true);
            mv(max_r, 1, 0, MY, false, T(-1));
            tri(2, 1, MLUI, false, false, false);
            mv(max_k, 0, 2, MT, false, T(-1));
            scatter(2, false);
            break;
        case APPLY_UP:        // xs += T xr; xr <- U' xr; xr += Y xs; xr *= D
            gather(false);
            mv(max_k, 0, 1, MT, false, T(1));
            tri(2, 1, MLU, false, false, false);
            mv(max_r, 2, 0, MY, false, T(1));
            scatter(2, true);
            break;
        case APPLY_DOWN:      // xs += X xr; xr <- P^T L xr; xr += T^T xs
            gather(false);
            mv(max_k, 0, 1, MX, false, T(1));
            tri(2, 1, MLU, true, false, false);
            perm(1, 2, true);
            mv(max_r, 1, 0, MT, true, T(1));
            scatter(1, false);
            break;
        case SOLVET_UP:       // xr -= T^T xs; xr <- U'^{-T} xr; xs -= Y^T xr
            gather(false);
            mv(max_r, 1, 0, MT, true, T(-1));
            tri(2, 1, MLUI, false, true, false);
            mv(max_k, 0, 2, MY, true, T(-1));
            scatter(2, false);
            break;
        case SOLVET_DOWN:     // xr /= D; xr -= X^T xs; xr <- P^T L^{-T} xr; xs -= T xr
            gather(true);
            mv(max_r, 1, 0, MX, true, T(-1));
            tri(2, 1, MLUI, true, true, false);
            perm(1, 2, true);
            mv(max_k, 0, 1, MT, false, T(-1));
            scatter(1, false);
            break;
        case APPLYT_UP:       // xs += T xr; xr <- L^T P xr; xr += X^T xs; xr *= D
            gather(false);
            mv(max_k, 0, 1, MT, false, T(1));
            tri(2, 1, MLU, true, true, true);
            mv(max_r, 2, 0, MX, true, T(1));
            scatter(2, true);
            break;
        case APPLYT_DOWN:     // xs += Y^T xr; xr <- U'^T xr; xr += T^T xs
            gather(false);
            mv(max_k, 0, 1, MY, true, T(1));
            tri(2, 1, MLU, false, true, false);
            mv(max_r, 2, 0, MT, true, T(1));
            scatter(2, false);
            break;
        default: return cudaErrorInvalidValue;
    }
    return err;
}

template cudaError_t launch_wide_sweep<double>(const WideArgs&, int, int, int, int, cudaStream_t);
template cudaError_t launch_wide_sweep<float>(const WideArgs&, int, int, int, int, cudaStream_t);

// ---------------------------------------------------- precision moves ----

// Working vectors hold the right-hand sides of a DOF side by side, so a box's
// gather reads whole sectors (column by column it read 8 bytes of each).
template <typename T>
__global__ void to_work_kernel(const double* src, int64_t lds, T* dst, int64_t N, int nrhs) {
    const int64_t tot = N * nrhs;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < tot; e += (int64_t)gridDim.x * blockDim.x)
        dst[e] = (T)src[e / nrhs + lds * (e % nrhs)];
}

template <typename T>
__global__ void from_work_kernel(const T* src, double* dst, int64_t ldd, int64_t N, int nrhs) {
    const int64_t tot = N * nrhs;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < tot; e += (int64_t)gridDim.x * blockDim.x)
        dst[e / nrhs + ldd * (e % nrhs)] = (double)src[e];
}

template <typename T>
cudaError_t launch_to_work(const double* src, int64_t lds, T* dst, int64_t N, int nrhs, cudaStream_t st) {
    const int64_t tot = N * nrhs;
    if (tot == 0) return cudaSuccess;
    const int blocks = (int)((tot + 255) / 256 < 152 * 16 ? (tot + 255) / 256 : 152 * 16);
    note_launch();
    to_work_kernel<T><<<blocks, 256, 0, st>>>(src, lds, dst, N, nrhs);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_from_work(const T* src, double* dst, int64_t ldd, int64_t N, int nrhs, cudaStream_t st) {
    const int64_t tot = N * nrhs;
    if (tot == 0) return cudaSuccess;
    const int blocks = (int)((tot + 255) / 256 < 152 * 16 ? (tot + 255) / 256 : 152 * 16);
    note_launch();
    from_work_kernel<T><<<blocks, 256, 0, st>>>(src, dst, ldd, N, nrhs);
    return cudaGetLastError();
}

template cudaError_t launch_to_work<double>(const double*, int64_t, double*, int64_t, int, cudaStream_t);
template cudaError_t launch_to_work<float>(const double*, int64_t, float*, int64_t, int, cudaStream_t);
template cudaError_t launch_from_work<double>(const double*, double*, int64_t, int64_t, int, cudaStream_t);
template cudaError_t launch_from_work<float>(const float*, double*, int64_t, int64_t, int, cudaStream_t);

}  // namespace hif
