// Patch kernels: FV matrices of eq. ulbe, the refill procedure of Sec. 4,
// the outer-node feed of eq. postcollision2_u, the n FV sub-steps of one
// lattice step (one persistent cooperative kernel), the force on the lamina
// and the reductions of the hydrodynamic-function fit (Sec. 2.1).
//
// Patch state: one record of kRec values per node, f'[0..8] (deviation from
// w_i rho0) followed by the quadratic equilibrium terms z[0..2] (z_of).
#include <cooperative_groups.h>

#include <algorithm>
#include <utility>
#include <vector>

#include "adj_node.cuh"
#include "fv_node.cuh"
#include "hlbm_dev.cuh"

namespace hk {

constexpr int kMaxRow = 64;

template <typename T>
__device__ __forceinline__ void load_f(const T* rec, T (&f)[9]) {
#pragma unroll
    for (int i = 0; i < 9; ++i) f[i] = rec[i];
}

template <typename T>
__device__ __forceinline__ void store_rec(T* rec, const T (&f)[9], T rho0) {
    T z[3];
    z_of(f, rho0, z);
#pragma unroll
    for (int i = 0; i < 9; ++i) rec[i] = f[i];
#pragma unroll
    for (int j = 0; j < 3; ++j) rec[9 + j] = z[j];
#pragma unroll
    for (int j = 12; j < kRec; ++j) rec[j] = T(0);
}

// ------------------------------------------------------ FV matrices
// Cell-vertex FV on median-dual control volumes with f linear on each
// triangle.  Per node P (V_P = sum_T |T|/3):
//   g_Pk = -(1/V_P) sum_{T ni P,k} (|T|/3) grad phi_k|_T   (the boundary flux
//          of CV(P), by the gradient theorem), S_ik = c_i . g_Pk;
//   C_Pk = (1/V_P) sum_{T ni P,k} |T| (11/54 if k = P else 7/108)
//          (integral of phi_k over CV(P)), or the identity when lumped.
template <typename T>
__global__ void k_fv_coeffs(Dev<T> d, int lumped, Coef<T>* coef) {
    int P = blockIdx.x * blockDim.x + threadIdx.x;
    if (P >= d.n) return;
    int r0 = d.row_ptr[P], r1 = d.row_ptr[P + 1];
    double gx[kMaxRow], gy[kMaxRow], cc[kMaxRow];
    for (int e = 0; e < r1 - r0; ++e) gx[e] = gy[e] = cc[e] = 0.0;
    double V = 0.0;
    for (int e = d.tstart[P]; e < d.tstart[P + 1]; ++e) {
        const int32_t* v = d.tri + 3 * d.tlist[e];
        double X[3], Y[3];
        for (int j = 0; j < 3; ++j) {
            X[j] = d.xy[2 * v[j]];
            Y[j] = d.xy[2 * v[j] + 1];
        }
        double A2 = (X[1] - X[0]) * (Y[2] - Y[0]) - (X[2] - X[0]) * (Y[1] - Y[0]);
        double area = 0.5 * fabs(A2);
        V += area / 3.0;
        for (int a = 0; a < 3; ++a) {
            int b = (a + 1) % 3, c = (a + 2) % 3;
            double grx = (Y[b] - Y[c]) / A2, gry = (X[c] - X[b]) / A2;
            int pos = -1;
            for (int q = r0; q < r1; ++q)
                if (d.col[q] == v[a]) pos = q - r0;
            if (pos < 0) continue;
            gx[pos] -= area / 3.0 * grx;
            gy[pos] -= area / 3.0 * gry;
            cc[pos] += area * (v[a] == P ? 11.0 / 54.0 : 7.0 / 108.0);
        }
    }
    for (int e = 0; e < r1 - r0; ++e) {
        Coef<T> c;
        c.col = d.col[r0 + e];
        c.gx = T(gx[e] / V);
        c.gy = T(gy[e] / V);
        c.c = lumped ? T(c.col == P ? 1 : 0) : T(cc[e] / V);
        coef[r0 + e] = c;
    }
}

template <typename T>
void launch_fv_coeffs(const Dev<T>& d, int lumped, Coef<T>* coef, cudaStream_t s) {
    k_fv_coeffs<T><<<(d.n + 127) / 128, 128, 0, s>>>(d, lumped, coef);
}

// ------------------------------------------------ bilinear from lattice
// Sec. 4 (type 1): bilinear Lagrange interpolation of rho, u and f^neq over
// the four lattice nodes of the cell enclosing (wx, wy).  The lattice state
// is read from a window (origin ox, oy) of pre-collision populations; with
// cls given, the four donors must be discretization nodes.
// st = (drho, ux, uy, f^neq[9]).
//
// Four lanes (aligned, all calling) share a point: lane q takes corner q, and
// every lane returns the sums.  One thread per point took the corners one
// after another, 36 dependent loads and in FP64 some 600 instructions.
template <typename T>
__device__ __forceinline__ void bilinear_quad(const Dev<T>& d, const T* box, int ox, int oy, const int8_t* cls,
                                              double wx, double wy, bool live, int q, T (&st)[12], int& cell) {
    const double fx0 = floor(wx), fy0 = floor(wy);
    const int ix = (int)fx0, iy = (int)fy0;
    const double ax = __dsub_rn(wx, fx0), ay = __dsub_rn(wy, fy0);
    const T w = T(((q & 1) ? ax : 1.0 - ax) * ((q >> 1) ? ay : 1.0 - ay));
    cell = iy * d.nx + ix;
    const int bx = ix + (q & 1) - ox, by = iy + (q >> 1) - oy;
    bool have = live;
    if (live && ((unsigned)bx >= (unsigned)d.bw || (unsigned)by >= (unsigned)d.bh)) {
        atomicOr(d.status, HLBM_ST_DONOR_NOT_COMPUTED);
        have = false;
    }
    const int64_t b = have ? (int64_t)by * d.bw + bx : 0;
    if (have && cls && cls[b] != CLS_DISC) atomicOr(d.status, HLBM_ST_DONOR_NOT_COMPUTED);
    T f[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) f[i] = have ? box[i * d.bplane + b] : T(0);
    state_of(f, d.rho0, st);
    // the sum in corner order
    const T wq = have ? w : T(0);
    T w4[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) w4[c] = __shfl_sync(0xffffffffu, wq, c, 4);
#pragma unroll
    for (int j = 0; j < 12; ++j) {
        T v[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) v[c] = __shfl_sync(0xffffffffu, st[j], c, 4);
        st[j] = fma_rn(w4[3], v[3], fma_rn(w4[2], v[2], fma_rn(w4[1], v[1], mul_rn(w4[0], v[0]))));
    }
}

// eq. continuity_stresses: f = f^eq(rho, u) + (1 - 1/(2 tau_s)) f^neq,s
template <typename T>
__device__ __forceinline__ void f_from_state(const Dev<T>& d, const T (&st)[12], T (&f)[9]) {
    const T dr = st[0], r = add_rn(d.rho0, dr), ux = st[1], uy = st[2];
    if constexpr (sizeof(T) == 4) {
        T x[9];
        pops_to(feq_x(dr, r, ux, uy), x);
#pragma unroll
        for (int i = 0; i < 9; ++i) f[i] = fma_rn(d.kneq, st[3 + i], mul_rn(w_of<T>(i), x[i]));
        return;
    }
    const T q = mul_rn(T(-1.5), fma_rn(ux, ux, mul_rn(uy, uy)));
    f[0] = fma_rn(d.kneq, st[3], mul_rn(w_of<T>(0), fma_rn(r, q, dr)));
#pragma unroll
    for (int i = 1; i < 9; ++i) {
        if (opp_of(i) < i) continue;
        T a, b;
        feq_pair(i, dr, r, ux, uy, q, a, b);
        f[i] = fma_rn(d.kneq, st[3 + i], a);
        f[opp_of(i)] = fma_rn(d.kneq, st[3 + opp_of(i)], b);
    }
}

// The type-1 state of the lanes of a warp that ask for it (all lanes call):
// eight at a time, four lanes each.
template <typename T>
__device__ __forceinline__ void bilinear_warp(const Dev<T>& d, const T* box, int ox, int oy, const int8_t* cls,
                                              double wx, double wy, bool want, T (&st)[12], int& cell) {
    const int lane = threadIdx.x & 31;
    for (unsigned left = __ballot_sync(0xffffffffu, want); left;) {
        // quad g serves the g-th lane left
        const int g = lane >> 2, n = min(8, __popc(left));
        unsigned rest = left;
        int src = 0;
        for (int k = 0; k < n; ++k) {
            const int l = __ffs(rest) - 1;
            rest &= rest - 1;
            if (k == g) src = l;
        }
        const double px = __shfl_sync(0xffffffffu, wx, src), py = __shfl_sync(0xffffffffu, wy, src);
        T s[12];
        int c;
        bilinear_quad(d, box, ox, oy, cls, px, py, g < n, lane & 3, s, c);
        // back to the lane: its quad is its rank among those left
        const int rank = __popc(left & ((1u << lane) - 1u));
        const bool mine = ((left >> lane) & 1u) && rank < 8;
#pragma unroll
        for (int j = 0; j < 12; ++j) {
            const T v = __shfl_sync(0xffffffffu, s[j], 4 * (mine ? rank : 0));
            if (mine) st[j] = v;
        }
        c = __shfl_sync(0xffffffffu, c, 4 * (mine ? rank : 0));
        if (mine) cell = c;
        left = rest;
    }
}

// initial patch: every node by the type-1 rule from the initial lattice state
template <typename T>
__global__ void k_patch_init(Dev<T> d, StepArgs a) {
    const int P = blockIdx.x * blockDim.x + threadIdx.x;
    const bool live = P < d.n;
    const double x = live ? d.xy[2 * P] : 0.0, y = live ? d.xy[2 * P + 1] : 0.0;
    T st[12], f[9];
    int cell;
    bilinear_warp(d, d.sbox_old, a.pbx0, a.pby0, (const int8_t*)nullptr, __dadd_rn(a.cx, x), __dadd_rn(a.cy, y), live, st,
                  cell);
    if (!live) return;
    f_from_state(d, st, f);
    store_rec(d.fu_out + (int64_t)kRec * P, f, d.rho0);
}

template <typename T>
void launch_patch_init(const Dev<T>& d, const StepArgs& a, cudaStream_t s) {
    k_patch_init<T><<<(d.n + 127) / 128, 128, 0, s>>>(d, a);
}

// ------------------------------------------------------------ refill
// Sec. 4 at the start of step t: each non-wall node, moved by (dX, dY), is
// located in the previous configuration: type 3 (inside a triangle:
// barycentric f), type 2 (inside the body: keep f), type 1 (outside the
// patch: bilinear from the lattice state at t).  Wall nodes keep f and rho.
//
// The blocks from refill_blocks on classify the lattice nodes of the window
// (Sec. 4): geometry only, independent of the refill, and read next by the eq.
// 178 fill; a launch of its own beside this one cost two events and a second
// stream's latency.  Move phase (refill, classification, fill): 38 -> 28 us on a
// 1788-node FP32 patch, 62 -> 44 on 3008 FP64 nodes, 79 -> 70 on 200k.
template <typename T>
__global__ void __launch_bounds__(128) k_refill(Dev<T> d, StepArgs a, int refill_blocks) {
    if ((int)blockIdx.x >= refill_blocks) {
        const int64_t b = ((int64_t)blockIdx.x - refill_blocks) * blockDim.x + threadIdx.x;
        if (b < d.bplane) classify_node(d, a, b);
        return;
    }
    const int P = blockIdx.x * blockDim.x + threadIdx.x;
    const bool live = P < d.n;
    const T* in = d.fu_in;
    const bool wall = live && d.kind[P] == HLBM_NODE_WALL;
    const double x = live ? d.xy[2 * P] : 0.0, y = live ? d.xy[2 * P + 1] : 0.0;
    T f[9];
    int type = 0, donor = -1;
    if (live && !wall) {
        const double qx = __dadd_rn(x, a.dX), qy = __dadd_rn(y, a.dY);
        double lam[3];
        const int k = locate_from_node(d, P, qx, qy, lam);
        if (k >= 0) {
            const int32_t* v = d.tri + 3 * k;
            const T l0 = T(lam[0]), l1 = T(lam[1]), l2 = T(lam[2]);
            const T *a0 = in + (int64_t)kRec * v[0], *a1 = in + (int64_t)kRec * v[1], *a2 = in + (int64_t)kRec * v[2];
#pragma unroll
            for (int i = 0; i < 9; ++i) f[i] = fma_rn(l2, a2[i], fma_rn(l0, a0[i], mul_rn(l1, a1[i])));
            type = 3;
            donor = k;
        } else if (fabs(qx) <= d.half_L && fabs(qy) <= d.half_T) {
            load_f(in + (int64_t)kRec * P, f);
            type = 2;
        } else {
            type = 1;
        }
    }
    __syncwarp();
    {
        T st[12];
        int cell = -1;
        bilinear_warp(d, d.sbox_old, a.pbx0, a.pby0, d.cls_prev, __dadd_rn(a.cx, x), __dadd_rn(a.cy, y), type == 1, st, cell);
        if (type == 1) {
            f_from_state(d, st, f);
            donor = cell;
        }
    }
    if (!live) return;
    T* out = d.fu_out + (int64_t)kRec * P;
    d.rtype[P] = type;
    d.rdonor[P] = donor;
    if (wall) {
#pragma unroll
        for (int j = 0; j < kRec; ++j) out[j] = in[(int64_t)kRec * P + j];
        return;
    }
    store_rec(out, f, d.rho0);
}

template <typename T>
void launch_refill(const Dev<T>& d, const StepArgs& a, cudaStream_t s) {
    const int rb = (d.n + 127) / 128, cb = (int)((d.bplane + 127) / 128);
    k_refill<T><<<rb + cb, 128, 0, s>>>(d, a, rb);
}

// ------------------------------------------------- outer-node feed
// Lattice state at t (previous window) and t+1 (this step's window),
// bilinear at the outer nodes: snap[0] and snap[1], 12 values each.  Eight
// lanes per node: four corners at each time.
template <typename T>
__global__ void __launch_bounds__(128) k_feed(Dev<T> d, StepArgs a) {
    const int g = blockIdx.x * blockDim.x + threadIdx.x, o = g >> 3, side = (g >> 2) & 1, q = g & 3;
    const bool live = o < d.n_outer;
    const int P = d.outer[live ? o : 0];
    const double wx = __dadd_rn(a.cx, d.xy[2 * P]), wy = __dadd_rn(a.cy, d.xy[2 * P + 1]);
    T s[12];
    int cell;
    bilinear_quad(d, side ? (const T*)d.sbox_new : d.sbox_old, side ? a.bx0 : a.pbx0, side ? a.by0 : a.pby0,
                  side ? (const int8_t*)d.cls_cur : d.cls_prev, wx, wy, live, q, s, cell);
    if (!live) return;
    const int64_t no = d.n_outer;
#pragma unroll
    for (int j = 0; j < 12; ++j)
        if ((j & 3) == q) d.snap[(12 * side + j) * no + o] = s[j];
}

template <typename T>
void launch_feed(const Dev<T>& d, const StepArgs& a, cudaStream_t s) {
    if (d.n_outer) k_feed<T><<<(8 * d.n_outer + 127) / 128, 128, 0, s>>>(d, a);
}

// ----------------------------------------------------------- FV steps
// n explicit steps of eq. ulbe on interior and wall nodes,
//   f_P += dt_u sum_k [ (c_i . g_Pk) f_k - (C_Pk / tau_u) (f_k - f_k^eq) ],
// evaluated as dt_u [ S_i - (Cf_i - f^eq_i(Q)) / tau_u ]
// with S_i = sum_{k != P} (c_i . g_Pk) (f'_k,i - f'_P,i),
// Cf_i = sum_k C_Pk f'_k,i, Q = sum_k C_Pk q_k (the deviations drop out of
// the streaming sum because sum_k g_Pk = 0).
// Wall nodes then take the lamina velocity: f += f^eq(rho, U) - f^eq(rho, u).
// Outer nodes take the lattice state, linear in time at theta = (m+1)/n:
//   f = f^eq(rho, u) + (1 - 1/(2 tau_s)) f^neq   (eq. postcollision2_u).
// The arithmetic of a node is in fv_node.cuh, shared by every FV kernel.
template <typename T>
__device__ __forceinline__ void fv_outer(const Dev<T>& d, int P, int m, T (&fn)[9]) {
    fv_outer_from(d, d.snap + d.outer_of[P], (int64_t)d.n_outer, m, fn);
}

template <typename T>
__device__ __forceinline__ void fv_node(const Dev<T>& d, const T* __restrict__ in, T* __restrict__ out, int P,
                                        int m, T U, T V) {
    const int8_t kind = d.kind[P];
    T fn[9];
    if (kind == HLBM_NODE_OUTER) {
        fv_outer(d, P, m, fn);
        if (d.outer_fv) {
            // eq. postcollision2_u with its FV sums: interpolated values at
            // interpolation nodes (this one included), patch values elsewhere
            FvAcc<T> acc;
            fv_acc_init(acc);
            const int r0 = d.row_ptr[P], r1 = d.row_ptr[P + 1];
            for (int e = r0 + 1; e < r1; ++e) {
                const Coef<T> c = d.coef[e];
                T f[9], z[3];
                if (d.kind[c.col] == HLBM_NODE_OUTER) {
                    fv_outer(d, c.col, m, f);
                    z_of(f, d.rho0, z);
                } else {
                    const T* rec = in + (int64_t)kRec * c.col;
#pragma unroll
                    for (int i = 0; i < 9; ++i) f[i] = rec[i];
#pragma unroll
                    for (int j = 0; j < 3; ++j) z[j] = rec[9 + j];
                }
                fv_acc_entry(acc, c.gx, c.gy, c.c, f, z, fn);
            }
            T fP[9], zP[3];
#pragma unroll
            for (int i = 0; i < 9; ++i) fP[i] = fn[i];
            z_of(fP, d.rho0, zP);
            fv_acc_finish(d, acc, d.coef[r0].c, fP, zP, fn);
        }
        store_rec(out + (int64_t)kRec * P, fn, d.rho0);
        return;
    }
    T fP[9], zP[3];
    const T* own = in + (int64_t)kRec * P;
#pragma unroll
    for (int i = 0; i < 9; ++i) fP[i] = own[i];
#pragma unroll
    for (int j = 0; j < 3; ++j) zP[j] = own[9 + j];
    FvAcc<T> acc;
    fv_acc_init(acc);
    const int r0 = d.row_ptr[P], r1 = d.row_ptr[P + 1];
    for (int e = r0 + 1; e < r1; ++e) {
        const Coef<T> c = d.coef[e];
        T f[9], z[3];
        const T* rec = in + (int64_t)kRec * c.col;
#pragma unroll
        for (int i = 0; i < 9; ++i) f[i] = rec[i];
#pragma unroll
        for (int j = 0; j < 3; ++j) z[j] = rec[9 + j];
        fv_acc_entry(acc, c.gx, c.gy, c.c, f, z, fP);
    }
    fv_acc_finish(d, acc, d.coef[r0].c, fP, zP, fn);
    if (kind == HLBM_NODE_WALL) fv_wall(d, U, V, fn);
    store_rec(out + (int64_t)kRec * P, fn, d.rho0);
}

__device__ __forceinline__ unsigned long long ld_acquire(const unsigned long long* p) {
    unsigned long long v;
    asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ void st_release(unsigned long long* p, unsigned long long v) {
    asm volatile("st.release.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

// 16-byte global -> shared copy that bypasses L1; completed by cp_async_wait_all
__device__ __forceinline__ void cp_async16(void* smem_dst, const void* gmem_src) {
    const unsigned dst = (unsigned)__cvta_generic_to_shared(smem_dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(gmem_src) : "memory");
}

__device__ __forceinline__ void cp_async_wait_all() {
    asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;" ::: "memory");
}

constexpr int kFvThreads = 256;

// Lamina velocity at the end of sub-step m, t + (m+1)/n (the wall nodes'
// Dirichlet value, eq. 182); INDUCED motion interpolates v(t) -> v(t+1).
template <typename T>
__device__ __forceinline__ void wall_velocity(const Dev<T>& d, const StepArgs& a, int m, T& U, T& V) {
    const double time = double(a.t) + double(m + 1) / double(d.n_sub);
    U = T(0);
    V = T(0);
    if (d.motion == HLBM_MOTION_HARMONIC) {
        V = T(d.A * d.omega * cos(d.omega * time));
    } else if (d.motion == HLBM_MOTION_UNIFORM) {
        U = T(d.vx);
        V = T(d.vy);
    } else if (d.motion == HLBM_MOTION_INDUCED) {
        V = T(a.v0 + double(m + 1) / double(d.n_sub) * (a.v1 - a.v0));
    }
}

// All n sub-steps of one lattice step in one cooperative launch.  Block b
// owns the node tile [tile_start[b], tile_start[b+1]) (nodes are numbered
// along a Morton curve, so tiles are compact).  Before sub-step m a block
// waits only for the tiles that own columns of its rows to finish sub-step
// m-1 (monotone progress counters, acquire/release); that also guarantees
// they are done reading the buffer it is about to overwrite.  Sub-step m
// reads record buffer m%2 and writes buffer (m+1)%2.  Every wait is
// bounded: on timeout the block raises HLBM_ST_SYNC_TIMEOUT and the abort
// flag, and every block returns.
template <typename T>
__global__ void __launch_bounds__(kFvThreads) k_fv_steps(Dev<T> d, StepArgs a, const T* buf0, T* buf1) {
    __shared__ int abort_sh;
    const int tile = blockIdx.x;
    const int p0 = d.tile_start[tile], p1 = d.tile_start[tile + 1];
    if (threadIdx.x == 0) abort_sh = 0;
    const unsigned long long base = (unsigned long long)a.t * (unsigned long long)d.n_sub;
    const int nb0 = d.tile_nb_ptr[tile], nb1 = d.tile_nb_ptr[tile + 1];
    __syncthreads();
    for (int m = 0; m < d.n_sub; ++m) {
        if (m > 0 && threadIdx.x < 32) {
            bool ok = true;
            for (int e = nb0 + (int)threadIdx.x; e < nb1 && ok; e += 32) {
                const unsigned long long* pc = d.progress + d.tile_nb[e];
                long spins = 0;
                while (ld_acquire(pc) < base + m) {
                    if (*(volatile unsigned*)d.abort_flag) {
                        ok = false;
                        break;
                    }
                    if (++spins > d.spin_limit) {
                        atomicOr(d.status, HLBM_ST_SYNC_TIMEOUT);
                        atomicExch(d.abort_flag, 1u);
                        ok = false;
                        break;
                    }
                    __nanosleep(128);
                }
            }
            __threadfence();
            ok = __all_sync(0xffffffffu, ok);
            if (threadIdx.x == 0 && !ok) abort_sh = 1;
        }
        __syncthreads();
        if (abort_sh) return;
        const T* in = (m & 1) ? (const T*)buf1 : buf0;
        T* out = (m & 1) ? (T*)buf0 : buf1;
        T U, V;
        wall_velocity(d, a, m, U, V);
        for (int P = p0 + threadIdx.x; P < p1; P += blockDim.x) fv_node(d, in, out, P, m, U, V);
        __syncthreads();
        if (threadIdx.x == 0 && tile != d.stall_tile) {
            __threadfence();
            st_release(d.progress + tile, base + m + 1);
        }
    }
}

template <typename T>
int fv_tile_capacity() {
    int dev = 0, sms = 0, per = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_fv_steps<T>, kFvThreads, 0);
    return sms * per;
}

template <typename T>
cudaError_t launch_fv_persistent(const Dev<T>& d, const StepArgs& a, cudaStream_t s) {
    Dev<T> dd = d;
    StepArgs aa = a;
    const T* b0 = d.fu_in;
    T* b1 = d.fu_out;
    void* args[] = {&dd, &aa, &b0, &b1};
    return cudaLaunchCooperativeKernel((const void*)k_fv_steps<T>, dim3(d.n_tiles), dim3(kFvThreads), args, 0, s);
}

// Shared-memory variant of k_fv_steps: one block per SM and everything its
// inner loop reads in shared memory.  Block b holds, for its tile of nodes:
//   - the records (f', z; 12 values) of its own nodes, updated in place:
//     the new values of a thread's nodes wait in registers until every read
//     of the old ones is done,
//   - the records of its halo (the nodes of other tiles its rows read),
//     reloaded each sub-step,
//   - the off-diagonal FV entries in ELL form (tile-local column, g_Pk,
//     C_Pk) and per node C_PP; the pivot g_PP is minus the sum of the
//     off-diagonal g_Pk (the rows of g sum to zero),
//   - node kinds, which nodes other tiles read, and a node order with the
//     nodes that read no halo first.
// A sub-step first updates the nodes that read no halo, then waits for the
// neighbour tiles, loads the halo and updates the rest, so the exchange
// overlaps the first part.  Only nodes read by other tiles are written to
// global memory each sub-step, into record buffer (m+1)%2; the final state
// of every node goes to buffer n%2.
// threads per block and own nodes per thread (tile_n <= kSlots * threads):
// FP32 1024 x 2 fits 64 registers per thread; FP64 512 x 1
template <typename T>
constexpr int kSmemThreads = sizeof(T) == 4 ? 1024 : 512;
template <typename T>
constexpr int kSlots = sizeof(T) == 4 ? 2 : 1;
constexpr int kSR = 12;  // values per record in shared memory
constexpr int kSnap = 24;  // outer-node feed values (12 at t, 12 at t + 1)

template <typename T>
int fv_tile_max() {
    return kSlots<T> * kSmemThreads<T>;
}

struct TileSmem {
    size_t own, halo, ecol, ecoef, cpp, order, kind, send, hid, uv, omap, osnap, cnt, total;
};

template <typename T>
__host__ __device__ inline TileSmem tile_smem_layout(int cap, int hcap, int roff, int n_sub, int ocap) {
    auto up = [](size_t x) { return (x + 15) / 16 * 16; };
    TileSmem L;
    size_t o = 0;
    L.own = o;
    o = up(o + sizeof(T) * kSR * (size_t)cap);
    L.halo = o;
    o = up(o + sizeof(T) * kSR * (size_t)hcap);
    L.ecoef = o;
    o = up(o + sizeof(T) * 3 * (size_t)roff * cap);
    L.cpp = o;
    o = up(o + sizeof(T) * (size_t)cap);
    L.uv = o;
    o = up(o + sizeof(T) * 2 * (size_t)n_sub);
    L.osnap = o;
    o = up(o + sizeof(T) * kSnap * (size_t)ocap);
    L.hid = o;
    o = up(o + sizeof(int32_t) * (size_t)hcap);
    L.ecol = o;
    o = up(o + sizeof(uint16_t) * (size_t)roff * cap);
    L.order = o;
    o = up(o + sizeof(uint16_t) * (size_t)cap);
    L.kind = o;
    o = up(o + (size_t)cap);
    L.send = o;
    o = up(o + (size_t)cap);
    L.omap = o;
    o = up(o + sizeof(int16_t) * (size_t)cap);
    L.cnt = o;
    o = up(o + (size_t)cap);
    L.total = o;
    return L;
}

template <typename T>
size_t fv_smem_bytes(int tile_cap, int halo_cap, int roff, int n_sub, int ocap) {
    return tile_smem_layout<T>(tile_cap, halo_cap, roff, n_sub, ocap).total;
}

// 16-byte (float) or 2 x 16-byte (double) vector load and store
template <typename T>
struct Vec4 {
    T x, y, z, w;
};
template <typename T>
__device__ __forceinline__ Vec4<T> ld4(const T* p) {
    Vec4<T> v;
    if constexpr (sizeof(T) == 4) {
        const float4 a4 = *reinterpret_cast<const float4*>(p);
        v.x = a4.x, v.y = a4.y, v.z = a4.z, v.w = a4.w;
    } else {
        const double2 a2 = *reinterpret_cast<const double2*>(p);
        const double2 b2 = *reinterpret_cast<const double2*>(p + 2);
        v.x = a2.x, v.y = a2.y, v.z = b2.x, v.w = b2.y;
    }
    return v;
}
template <typename T>
__device__ __forceinline__ void st4(T* p, T x, T y, T z, T w) {
    if constexpr (sizeof(T) == 4) {
        *reinterpret_cast<float4*>(p) = make_float4(x, y, z, w);
    } else {
        *reinterpret_cast<double2*>(p) = make_double2(x, y);
        *reinterpret_cast<double2*>(p + 2) = make_double2(z, w);
    }
}

template <typename T>
__device__ __forceinline__ void read_rec12(const T* r, T (&f)[9], T (&z)[3]) {
    const Vec4<T> a = ld4(r), b = ld4(r + 4), c = ld4(r + 8);
    f[0] = a.x, f[1] = a.y, f[2] = a.z, f[3] = a.w;
    f[4] = b.x, f[5] = b.y, f[6] = b.z, f[7] = b.w;
    f[8] = c.x, z[0] = c.y, z[1] = c.z, z[2] = c.w;
}

// f'[0..8] of a record, and its z terms on their own (the pivot of a row is
// read before its entries for the gradient differences, its z only at the end)
template <typename T>
__device__ __forceinline__ void read_rec9(const T* r, T (&f)[9]) {
    const Vec4<T> a = ld4(r), b = ld4(r + 4);
    f[0] = a.x, f[1] = a.y, f[2] = a.z, f[3] = a.w;
    f[4] = b.x, f[5] = b.y, f[6] = b.z, f[7] = b.w;
    f[8] = r[8];
}
template <typename T>
__device__ __forceinline__ void read_z3(const T* r, T (&z)[3]) {
    z[0] = r[9], z[1] = r[10], z[2] = r[11];
}

template <typename T>
__device__ __forceinline__ void fv_node_tile(const Dev<T>& d, const unsigned char* sm, const TileSmem& L, int r,
                                             T (&fn)[9]) {
    const int cap = d.tile_cap, roff = d.ell_width - 1;
    const T* own = reinterpret_cast<const T*>(sm + L.own);
    const T* halo = reinterpret_cast<const T*>(sm + L.halo) - (size_t)kSR * cap;
    const T* ec = reinterpret_cast<const T*>(sm + L.ecoef);
    const uint16_t* ecol = reinterpret_cast<const uint16_t*>(sm + L.ecol);
    T fP[9], zP[3];
    read_rec9(own + (size_t)kSR * r, fP);
    FvAcc<T> acc;
    fv_acc_init(acc);
    const int ne = reinterpret_cast<const uint8_t*>(sm + L.cnt)[r];  // off-diagonal entries of the row
    for (int j = 0; j < ne; ++j) {
        const int e = j * cap + r;
        const int col = ecol[e];
        T f[9], z[3];
        read_rec12((col < cap ? own : halo) + (size_t)kSR * col, f, z);
        fv_acc_entry(acc, ec[e], ec[(roff + j) * cap + r], ec[(2 * roff + j) * cap + r], f, z, fP);
    }
    read_z3(own + (size_t)kSR * r, zP);
    fv_acc_finish(d, acc, reinterpret_cast<const T*>(sm + L.cpp)[r], fP, zP, fn);
}

// eq. postcollision2_u with its FV sums at the outer node in slot r, whose
// interpolated value fn holds on entry: the starred values are the
// interpolated ones at interpolation nodes (own ones from the staged feed,
// halo ones from global memory) and the patch records elsewhere
template <typename T>
__device__ __noinline__ void fv_outer_sums_tile(const Dev<T>& d, const unsigned char* sm, const TileSmem& L, int r,
                                                int m, T (&fn)[9]) {
    const int cap = d.tile_cap, roff = d.ell_width - 1;
    const T* own = reinterpret_cast<const T*>(sm + L.own);
    const T* halo = reinterpret_cast<const T*>(sm + L.halo);
    const T* ec = reinterpret_cast<const T*>(sm + L.ecoef);
    const uint16_t* ecol = reinterpret_cast<const uint16_t*>(sm + L.ecol);
    const int8_t* kd = reinterpret_cast<const int8_t*>(sm + L.kind);
    const int16_t* om = reinterpret_cast<const int16_t*>(sm + L.omap);
    const T* osn = reinterpret_cast<const T*>(sm + L.osnap);
    const int32_t* hid = reinterpret_cast<const int32_t*>(sm + L.hid);
    FvAcc<T> acc;
    fv_acc_init(acc);
    const int ne = reinterpret_cast<const uint8_t*>(sm + L.cnt)[r];
    for (int j = 0; j < ne; ++j) {
        const int e = j * cap + r;
        const int col = ecol[e];
        T f[9], z[3];
        if (col < cap) {
            if (kd[col] == HLBM_NODE_OUTER) {
                fv_outer_from(d, osn + kSnap * om[col], 1, m, f);
                z_of(f, d.rho0, z);
            } else {
                read_rec12(own + (size_t)kSR * col, f, z);
            }
        } else {
            const int g = hid[col - cap];
            if (d.kind[g] == HLBM_NODE_OUTER) {
                fv_outer(d, g, m, f);
                z_of(f, d.rho0, z);
            } else {
                read_rec12(halo + (size_t)kSR * (col - cap), f, z);
            }
        }
        fv_acc_entry(acc, ec[e], ec[(roff + j) * cap + r], ec[(2 * roff + j) * cap + r], f, z, fn);
    }
    T fP[9], zP[3];
#pragma unroll
    for (int i = 0; i < 9; ++i) fP[i] = fn[i];
    z_of(fP, d.rho0, zP);
    fv_acc_finish(d, acc, reinterpret_cast<const T*>(sm + L.cpp)[r], fP, zP, fn);
}

template <typename T, bool kOuterFv>
__device__ __forceinline__ void fv_update_slot(const Dev<T>& d, const unsigned char* sm, const TileSmem& L, int r, int m,
                                               T (&fn)[9]) {
    const int8_t kind = reinterpret_cast<const int8_t*>(sm + L.kind)[r];
    if (kind == HLBM_NODE_OUTER) {
        const int q = reinterpret_cast<const int16_t*>(sm + L.omap)[r];
        fv_outer_from(d, reinterpret_cast<const T*>(sm + L.osnap) + kSnap * q, 1, m, fn);
        if constexpr (kOuterFv) fv_outer_sums_tile(d, sm, L, r, m, fn);
        return;
    }
    fv_node_tile(d, sm, L, r, fn);
    if (kind == HLBM_NODE_WALL) {
        const T* uv = reinterpret_cast<const T*>(sm + L.uv);
        fv_wall(d, uv[m], uv[d.n_sub + m], fn);
    }
}

template <typename T, bool kOuterFv>
__global__ void __launch_bounds__(kSmemThreads<T>, 1) k_fv_tiles(Dev<T> d, StepArgs a, T* g0, T* g1) {
    extern __shared__ __align__(16) unsigned char sm[];
    __shared__ int abort_sh;
    const int cap = d.tile_cap, hcap = d.halo_cap, roff = d.ell_width - 1;
    const TileSmem L = tile_smem_layout<T>(cap, hcap, roff, d.n_sub, d.tile_ocap);
    T* own = reinterpret_cast<T*>(sm + L.own);
    T* halo = reinterpret_cast<T*>(sm + L.halo);
    T* uv = reinterpret_cast<T*>(sm + L.uv);
    int32_t* hid = reinterpret_cast<int32_t*>(sm + L.hid);
    const uint16_t* order = reinterpret_cast<const uint16_t*>(sm + L.order);
    const int8_t* send = reinterpret_cast<const int8_t*>(sm + L.send);
    const int tile = blockIdx.x;
    const int p0 = d.tile_start[tile], p1 = d.tile_start[tile + 1], tile_n = p1 - p0;
    const int h0 = d.halo_ptr[tile], halo_n = d.halo_ptr[tile + 1] - h0;
    const int tid = threadIdx.x, nt = blockDim.x;
    // nodes updated before the halo arrives: the interior ones, but only as
    // many as fill whole rounds of the block, so that the rest (boundary
    // nodes and the remainder) take exactly one more round
    const int rounds = (tile_n + nt - 1) / nt;
    const int n_int = min(d.tile_interior[tile], (rounds - 1) * nt);
    // ---- tile set-up: wall velocity per sub-step, own records (buffer 0),
    // matrices, kinds, send flags, node order, halo ids
    for (int m = tid; m < d.n_sub; m += nt) wall_velocity(d, a, m, uv[m], uv[d.n_sub + m]);
    for (int x = tid; x < 3 * tile_n; x += nt) {
        const int sl = x / 3, c = x - 3 * sl;
        const Vec4<T> v = ld4(g0 + (int64_t)kRec * (p0 + d.tile_order[p0 + sl]) + 4 * c);
        st4(own + (size_t)kSR * sl + 4 * c, v.x, v.y, v.z, v.w);
    }
    {
        const Coef<T>* ell = d.ell + (int64_t)d.ell_width * p0;
        T* ec = reinterpret_cast<T*>(sm + L.ecoef);
        uint16_t* ecol = reinterpret_cast<uint16_t*>(sm + L.ecol);
        T* cpp = reinterpret_cast<T*>(sm + L.cpp);
        for (int x = tid; x < d.ell_width * tile_n; x += nt) {
            const int j = x / tile_n, r = x - j * tile_n;
            const Coef<T> c = ell[x];
            if (j == 0) {
                cpp[r] = c.c;
            } else {
                const int e = (j - 1) * cap + r;
                ecol[e] = (uint16_t)c.col;
                ec[e] = c.gx;
                ec[(roff + j - 1) * cap + r] = c.gy;
                ec[(2 * roff + j - 1) * cap + r] = c.c;
            }
        }
        int8_t* kd = reinterpret_cast<int8_t*>(sm + L.kind);
        int8_t* sd = reinterpret_cast<int8_t*>(sm + L.send);
        uint16_t* od = reinterpret_cast<uint16_t*>(sm + L.order);
        uint8_t* cn = reinterpret_cast<uint8_t*>(sm + L.cnt);
        for (int sl = tid; sl < tile_n; sl += nt) {
            const int r = d.tile_order[p0 + sl];
            kd[sl] = d.kind[p0 + r];
            sd[sl] = d.send[p0 + r];
            od[sl] = (uint16_t)r;
            cn[sl] = (uint8_t)(d.row_ptr[p0 + r + 1] - d.row_ptr[p0 + r] - 1);
        }
        for (int h = tid; h < halo_n; h += nt) hid[h] = d.halo_ids[h0 + h];
        // the outer nodes' feed (written by k_feed before this launch)
        const int o0 = d.tile_outer_ptr[tile], on = d.tile_outer_ptr[tile + 1] - o0;
        int16_t* om = reinterpret_cast<int16_t*>(sm + L.omap);
        T* osn = reinterpret_cast<T*>(sm + L.osnap);
        for (int q = tid; q < on; q += nt) om[d.tile_outer_r[o0 + q]] = (int16_t)q;
        const int64_t no = d.n_outer;
        for (int x = tid; x < kSnap * on; x += nt) {
            const int q = x / kSnap, j = x - kSnap * q;
            osn[x] = d.snap[j * no + d.outer_of[p0 + d.tile_order[p0 + d.tile_outer_r[o0 + q]]]];
        }
    }
    if (tid == 0) abort_sh = 0;
    __syncthreads();
    const unsigned long long base = (unsigned long long)a.t * (unsigned long long)d.n_sub;
    const int nb0 = d.tile_nb_ptr[tile], nb1 = d.tile_nb_ptr[tile + 1];
    for (int m = 0; m < d.n_sub; ++m) {
        T fn[kSlots<T>][9];
        // nodes that read no halo
#pragma unroll
        for (int s = 0; s < kSlots<T>; ++s) {
            const int x = tid + s * nt;
            if (x < n_int) fv_update_slot<T, kOuterFv>(d, sm, L, x, m, fn[s]);
        }
        // warp 0: wait for the neighbour tiles to publish state m (lane l
        // acquires the counters l, l + 32, ...; the warp barrier then orders
        // every lane's later reads after all of them), then copy the halo
        // records into shared memory asynchronously while the other warps
        // still update their nodes
        if (tid < 32) {
            bool ok = true;
            if (m > 0) {
                for (int e = nb0 + tid; e < nb1 && ok; e += 32) {
                    const unsigned long long* pc = d.progress + d.tile_nb[e];
                    long spins = 0;
                    while (ld_acquire(pc) < base + m) {
                        if (*(volatile unsigned*)d.abort_flag) {
                            ok = false;
                            break;
                        }
                        if (++spins > d.spin_limit) {
                            atomicOr(d.status, HLBM_ST_SYNC_TIMEOUT);
                            atomicExch(d.abort_flag, 1u);
                            ok = false;
                            break;
                        }
                        __nanosleep(32);
                    }
                }
            }
            __syncwarp();
            ok = __all_sync(0xffffffffu, ok);
            if (ok) {
                const T* gin = (m & 1) ? g1 : g0;
                constexpr int kChunks = kSR * (int)sizeof(T) / 16;  // 16-byte pieces of a record
                for (int x = tid; x < kChunks * halo_n; x += 32) {
                    const int h = x / kChunks, c = x - kChunks * h;
                    cp_async16(reinterpret_cast<unsigned char*>(halo) + (size_t)h * kSR * sizeof(T) + 16 * c,
                               reinterpret_cast<const unsigned char*>(gin + (int64_t)kRec * hid[h]) + 16 * c);
                }
            }
            cp_async_wait_all();
            if (tid == 0 && !ok) abort_sh = 1;
        }
        __syncthreads();
        if (abort_sh) return;
        // nodes that read the halo
#pragma unroll
        for (int s = 0; s < kSlots<T>; ++s) {
            const int x = tid + s * nt;
            if (x >= n_int && x < tile_n) fv_update_slot<T, kOuterFv>(d, sm, L, x, m, fn[s]);
        }
        __syncthreads();
        // publish state m+1
        T* gout = (m & 1) ? g0 : g1;
        const bool last = (m == d.n_sub - 1);
#pragma unroll
        for (int s = 0; s < kSlots<T>; ++s) {
            const int x = tid + s * nt;
            if (x < tile_n) {
                T z[3];
                z_of(fn[s], d.rho0, z);
                T* o = own + (size_t)kSR * x;
                st4(o, fn[s][0], fn[s][1], fn[s][2], fn[s][3]);
                st4(o + 4, fn[s][4], fn[s][5], fn[s][6], fn[s][7]);
                st4(o + 8, fn[s][8], z[0], z[1], z[2]);
                if (last || send[x]) {
                    T* rec = gout + (int64_t)kRec * (p0 + order[x]);
                    st4(rec, fn[s][0], fn[s][1], fn[s][2], fn[s][3]);
                    st4(rec + 4, fn[s][4], fn[s][5], fn[s][6], fn[s][7]);
                    st4(rec + 8, fn[s][8], z[0], z[1], z[2]);
                }
            }
        }
        __syncthreads();
        if (tid == 0 && tile != d.stall_tile) {
            __threadfence();
            st_release(d.progress + tile, base + m + 1);
        }
    }
}

// ---------------------------------------------------------------------------
// Tensor-memory variant of k_fv_tiles.  Each thread's own FV rows (per
// off-diagonal entry g_Pk, C_Pk and the tile-local column; C_PP and the
// entry count) live in tensor memory (TMEM), which a thread reads from its
// own lane with tcgen05.ld.  That frees the shared memory the coefficients
// took, so the records are double-buffered: sub-step m reads buffer m%2 and
// each thread writes its nodes' new records into the other buffer as soon
// as they are computed.  A sub-step then needs two block barriers (halo in,
// sub-step done) and no separate publish pass.
//
// TMEM: the block allocates all 512 columns.  Warp w reads lanes
// 32 (w % 4) .. 32 (w % 4) + 31 (one per thread) and its own column range
// kTmemCols<T> * (w / 4) .. + kTmemCols<T>: one slot of kTmemSlotWords<T>
// words per node the thread updates.
template <typename T>
constexpr int kTmemEntryWords = sizeof(T) == 4 ? 4 : 8;  // gx, gy, c, col (FP64: 2 words each, col, pad)
template <typename T>
constexpr int kTmemSlotWords = sizeof(T) == 4 ? 32 : 64;
template <typename T>
constexpr int kTmemCols = kSlots<T> * kTmemSlotWords<T>;
static_assert(1024 / 32 / 4 * kTmemCols<float> == 512, "TMEM columns (FP32)");
static_assert(512 / 32 / 4 * kTmemCols<double> <= 512, "TMEM columns (FP64)");

__device__ __forceinline__ void tmem_alloc_512(uint32_t* smem_dst) {
    const unsigned dst = (unsigned)__cvta_generic_to_shared(smem_dst);
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(dst) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc_512(uint32_t taddr) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(taddr) : "memory");
}
__device__ __forceinline__ void tmem_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tmem_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
// 4 words from this thread's lane, columns taddr .. taddr + 3; complete on return
__device__ __forceinline__ void tmem_ld4(uint32_t taddr, uint32_t (&v)[4]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3])
        : "r"(taddr)
        : "memory");
}
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t (&v)[8]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
        : "r"(taddr)
        : "memory");
}
__device__ __forceinline__ void tmem_st4(uint32_t taddr, uint32_t a, uint32_t b, uint32_t c, uint32_t e) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1, %2, %3, %4};" ::"r"(taddr), "r"(a), "r"(b),
                 "r"(c), "r"(e)
                 : "memory");
}
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

template <typename T>
__device__ __forceinline__ uint32_t lo_word(T v) {
    if constexpr (sizeof(T) == 4)
        return __float_as_uint(v);
    else
        return (uint32_t)__double2loint(v);
}
template <typename T>
__device__ __forceinline__ uint32_t hi_word(T v) {
    if constexpr (sizeof(T) == 4)
        return 0u;
    else
        return (uint32_t)__double2hiint(v);
}
template <typename T>
__device__ __forceinline__ T from_words(uint32_t lo, uint32_t hi) {
    if constexpr (sizeof(T) == 4)
        return __uint_as_float(lo);
    else
        return __hiloint2double((int)hi, (int)lo);
}

// one FV entry of the thread's slot: (g_x, g_y, C, column)
template <typename T>
__device__ __forceinline__ void tmem_entry(uint32_t taddr, T& gx, T& gy, T& c, int& col) {
    if constexpr (sizeof(T) == 4) {
        uint32_t v[4];
        tmem_ld4(taddr, v);
        gx = from_words<T>(v[0], 0);
        gy = from_words<T>(v[1], 0);
        c = from_words<T>(v[2], 0);
        col = (int)v[3];
    } else {
        uint32_t v[8];
        tmem_ld8(taddr, v);
        gx = from_words<T>(v[0], v[1]);
        gy = from_words<T>(v[2], v[3]);
        c = from_words<T>(v[4], v[5]);
        col = (int)v[6];
    }
}

struct TmemSmem {
    size_t own0, own1, halo, uv, osnap, hid, order, kind, send, omap, total;
};

template <typename T>
__host__ __device__ inline TmemSmem tmem_smem_layout(int cap, int hcap, int n_sub, int ocap) {
    auto up = [](size_t x) { return (x + 15) / 16 * 16; };
    TmemSmem L;
    size_t o = 0;
    L.own0 = o;
    o = up(o + sizeof(T) * kSR * (size_t)cap);
    L.own1 = o;
    o = up(o + sizeof(T) * kSR * (size_t)cap);
    L.halo = o;
    o = up(o + sizeof(T) * kSR * (size_t)hcap);
    L.uv = o;
    o = up(o + sizeof(T) * 2 * (size_t)n_sub);
    L.osnap = o;
    o = up(o + sizeof(T) * kSnap * (size_t)ocap);
    L.hid = o;
    o = up(o + sizeof(int32_t) * (size_t)hcap);
    L.order = o;
    o = up(o + sizeof(uint16_t) * (size_t)cap);
    L.kind = o;
    o = up(o + (size_t)cap);
    L.send = o;
    o = up(o + (size_t)cap);
    L.omap = o;
    o = up(o + sizeof(int16_t) * (size_t)cap);
    L.total = o;
    return L;
}

template <typename T>
size_t fv_tmem_smem_bytes(int tile_cap, int halo_cap, int n_sub, int ocap) {
    return tmem_smem_layout<T>(tile_cap, halo_cap, n_sub, ocap).total;
}

// The update of the node in slot r of a warp-uniform call (lanes with
// valid = false take part in the TMEM loads only) and its write into the
// next record buffer and, when other tiles read it or on the last
// sub-step, into global buffer gout.
template <typename T>
__device__ __forceinline__ void fv_tmem_node(const Dev<T>& d, const unsigned char* sm, const TmemSmem& L,
                                             const T* cur, T* nxt, uint32_t tslot, bool valid, int r, int m, T* gout,
                                             bool last, int p0) {
    const int cap = d.tile_cap;
    const int8_t kind = valid ? reinterpret_cast<const int8_t*>(sm + L.kind)[r] : (int8_t)HLBM_NODE_OUTER;
    uint32_t hdr[4];
    tmem_ld4(tslot + kTmemMaxEntries * kTmemEntryWords<T>, hdr);
    const T cP = from_words<T>(hdr[0], hdr[1]);
    const int ne = (valid && kind != HLBM_NODE_OUTER) ? (int)hdr[2] : 0;
    const int nem = __reduce_max_sync(0xffffffffu, (unsigned)ne);
    T fn[9];
    T fP[9] = {};
    if (valid && kind != HLBM_NODE_OUTER) read_rec9(cur + (size_t)kSR * r, fP);
    FvAcc<T> acc;
    fv_acc_init(acc);
    const T* halo = reinterpret_cast<const T*>(sm + L.halo) - (size_t)kSR * cap;
#pragma unroll
    for (int j = 0; j < kTmemMaxEntries; ++j) {
        if (j >= nem) break;
        T gx, gy, c;
        int col;
        tmem_entry<T>(tslot + j * kTmemEntryWords<T>, gx, gy, c, col);
        if (j < ne) {
            T f[9], z[3];
            read_rec12((col < cap ? cur : halo) + (size_t)kSR * col, f, z);
            fv_acc_entry(acc, gx, gy, c, f, z, fP);
        }
    }
    if (!valid) return;
    if (kind == HLBM_NODE_OUTER) {
        const int q = reinterpret_cast<const int16_t*>(sm + L.omap)[r];
        fv_outer_from(d, reinterpret_cast<const T*>(sm + L.osnap) + kSnap * q, 1, m, fn);
    } else {
        T zP[3];
        read_z3(cur + (size_t)kSR * r, zP);
        fv_acc_finish(d, acc, cP, fP, zP, fn);
        if (kind == HLBM_NODE_WALL) {
            const T* uv = reinterpret_cast<const T*>(sm + L.uv);
            fv_wall(d, uv[m], uv[d.n_sub + m], fn);
        }
    }
    T z[3];
    z_of(fn, d.rho0, z);
    T* o = nxt + (size_t)kSR * r;
    st4(o, fn[0], fn[1], fn[2], fn[3]);
    st4(o + 4, fn[4], fn[5], fn[6], fn[7]);
    st4(o + 8, fn[8], z[0], z[1], z[2]);
    if (last || reinterpret_cast<const int8_t*>(sm + L.send)[r]) {
        T* rec = gout + (int64_t)kRec * (p0 + reinterpret_cast<const uint16_t*>(sm + L.order)[r]);
        st4(rec, fn[0], fn[1], fn[2], fn[3]);
        st4(rec + 4, fn[4], fn[5], fn[6], fn[7]);
        st4(rec + 8, fn[8], z[0], z[1], z[2]);
    }
}

// The body of the tensor-memory FV kernel for tile `tile` of the solver d
// (one block); k_fv_tmem runs one solver, k_fv_tmem_pack several.
template <typename T>
__device__ __forceinline__ void fv_tmem_body(const Dev<T>& d, const StepArgs& a, T* g0, T* g1, const int tile,
                                             unsigned char* sm, int& abort_sh, uint32_t& tmem_base_sh) {
    const int cap = d.tile_cap, hcap = d.halo_cap;
    const TmemSmem L = tmem_smem_layout<T>(cap, hcap, d.n_sub, d.tile_ocap);
    T* own0 = reinterpret_cast<T*>(sm + L.own0);
    T* own1 = reinterpret_cast<T*>(sm + L.own1);
    T* halo = reinterpret_cast<T*>(sm + L.halo);
    T* uv = reinterpret_cast<T*>(sm + L.uv);
    int32_t* hid = reinterpret_cast<int32_t*>(sm + L.hid);
    const int p0 = d.tile_start[tile], p1 = d.tile_start[tile + 1], tile_n = p1 - p0;
    const int h0 = d.halo_ptr[tile], halo_n = d.halo_ptr[tile + 1] - h0;
    const int tid = threadIdx.x, nt = blockDim.x, warp = tid >> 5;
    const int rounds = (tile_n + nt - 1) / nt;
    const int n_int = min(d.tile_interior[tile], (rounds - 1) * nt);
    // ---- TMEM for the block
    if (warp == 0) tmem_alloc_512(&tmem_base_sh);
    tmem_fence_before();
    __syncthreads();
    tmem_fence_after();
    const uint32_t tbase = tmem_base_sh;
    const uint32_t twarp = tbase + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)(kTmemCols<T> * (warp >> 2));
    // ---- set-up: wall velocity, records (buffer 0), kinds, flags, order, halo ids, outer feed
    for (int m = tid; m < d.n_sub; m += nt) wall_velocity(d, a, m, uv[m], uv[d.n_sub + m]);
    for (int x = tid; x < 3 * tile_n; x += nt) {
        const int sl = x / 3, c = x - 3 * sl;
        const Vec4<T> v = ld4(g0 + (int64_t)kRec * (p0 + d.tile_order[p0 + sl]) + 4 * c);
        st4(own0 + (size_t)kSR * sl + 4 * c, v.x, v.y, v.z, v.w);
    }
    {
        int8_t* kd = reinterpret_cast<int8_t*>(sm + L.kind);
        int8_t* sd = reinterpret_cast<int8_t*>(sm + L.send);
        uint16_t* od = reinterpret_cast<uint16_t*>(sm + L.order);
        for (int sl = tid; sl < tile_n; sl += nt) {
            const int r = d.tile_order[p0 + sl];
            kd[sl] = d.kind[p0 + r];
            sd[sl] = d.send[p0 + r];
            od[sl] = (uint16_t)r;
        }
        for (int h = tid; h < halo_n; h += nt) hid[h] = d.halo_ids[h0 + h];
        const int o0 = d.tile_outer_ptr[tile], on = d.tile_outer_ptr[tile + 1] - o0;
        int16_t* om = reinterpret_cast<int16_t*>(sm + L.omap);
        T* osn = reinterpret_cast<T*>(sm + L.osnap);
        for (int q = tid; q < on; q += nt) om[d.tile_outer_r[o0 + q]] = (int16_t)q;
        const int64_t no = d.n_outer;
        for (int x = tid; x < kSnap * on; x += nt) {
            const int q = x / kSnap, j = x - kSnap * q;
            osn[x] = d.snap[j * no + d.outer_of[p0 + d.tile_order[p0 + d.tile_outer_r[o0 + q]]]];
        }
        // this thread's rows into its TMEM slots (every lane stores; lanes
        // without a node store zeros)
        const Coef<T>* ell = d.ell + (int64_t)d.ell_width * p0;
#pragma unroll
        for (int s = 0; s < kSlots<T>; ++s) {
            const int x = tid + s * nt;
            const bool have = x < tile_n;
            const uint32_t tslot = twarp + (uint32_t)(s * kTmemSlotWords<T>);
            const int q = have ? p0 + d.tile_order[p0 + x] : 0;
            const int ne = have ? d.row_ptr[q + 1] - d.row_ptr[q] - 1 : 0;
            for (int j = 0; j < kTmemMaxEntries; ++j) {
                Coef<T> c{};
                c.col = x;
                c.gx = c.gy = c.c = T(0);
                if (have && j < ne) c = ell[(int64_t)(j + 1) * tile_n + x];
                const uint32_t t = tslot + (uint32_t)(j * kTmemEntryWords<T>);
                if constexpr (sizeof(T) == 4) {
                    tmem_st4(t, lo_word(c.gx), lo_word(c.gy), lo_word(c.c), (uint32_t)c.col);
                } else {
                    tmem_st4(t, lo_word(c.gx), hi_word(c.gx), lo_word(c.gy), hi_word(c.gy));
                    tmem_st4(t + 4, lo_word(c.c), hi_word(c.c), (uint32_t)c.col, 0u);
                }
            }
            const T cP = have ? ell[x].c : T(0);
            tmem_st4(tslot + kTmemMaxEntries * kTmemEntryWords<T>, lo_word(cP), hi_word(cP), (uint32_t)ne, 0u);
        }
        tmem_wait_st();
    }
    if (tid == 0) abort_sh = 0;
    tmem_fence_before();
    __syncthreads();
    tmem_fence_after();
    const unsigned long long base = (unsigned long long)a.t * (unsigned long long)d.n_sub;
    const int nb0 = d.tile_nb_ptr[tile], nb1 = d.tile_nb_ptr[tile + 1];
    for (int m = 0; m < d.n_sub; ++m) {
        const T* cur = (m & 1) ? own1 : own0;
        T* nxt = (m & 1) ? own0 : own1;
        T* gout = (m & 1) ? g0 : g1;
        const bool last = (m == d.n_sub - 1);
        // nodes that read no halo (warp-uniform calls)
#pragma unroll
        for (int s = 0; s < kSlots<T>; ++s) {
            const int x = tid + s * nt;
            const bool v = x < n_int;
            if (__any_sync(0xffffffffu, v))
                fv_tmem_node(d, sm, L, cur, nxt, twarp + (uint32_t)(s * kTmemSlotWords<T>), v, x, m, gout, last,
                             p0);
        }
        // warp 0: neighbour wait and halo copy, as in k_fv_tiles
        if (warp == 0) {
            bool ok = true;
            if (m > 0) {
                for (int e = nb0 + tid; e < nb1 && ok; e += 32) {
                    const unsigned long long* pc = d.progress + d.tile_nb[e];
                    long spins = 0;
                    while (ld_acquire(pc) < base + m) {
                        if (*(volatile unsigned*)d.abort_flag) {
                            ok = false;
                            break;
                        }
                        if (++spins > d.spin_limit) {
                            atomicOr(d.status, HLBM_ST_SYNC_TIMEOUT);
                            atomicExch(d.abort_flag, 1u);
                            ok = false;
                            break;
                        }
                        __nanosleep(32);
                    }
                }
            }
            __syncwarp();
            ok = __all_sync(0xffffffffu, ok);
            if (ok) {
                const T* gin = (m & 1) ? g1 : g0;
                constexpr int kChunks = kSR * (int)sizeof(T) / 16;
                for (int x = tid; x < kChunks * halo_n; x += 32) {
                    const int h = x / kChunks, c = x - kChunks * h;
                    cp_async16(reinterpret_cast<unsigned char*>(halo) + (size_t)h * kSR * sizeof(T) + 16 * c,
                               reinterpret_cast<const unsigned char*>(gin + (int64_t)kRec * hid[h]) + 16 * c);
                }
            }
            cp_async_wait_all();
            if (tid == 0 && !ok) abort_sh = 1;
        }
        __syncthreads();
        if (abort_sh) break;
        // nodes that read the halo
#pragma unroll
        for (int s = 0; s < kSlots<T>; ++s) {
            const int x = tid + s * nt;
            const bool v = x >= n_int && x < tile_n;
            if (__any_sync(0xffffffffu, v))
                fv_tmem_node(d, sm, L, cur, nxt, twarp + (uint32_t)(s * kTmemSlotWords<T>), v, x, m, gout, last,
                             p0);
        }
        __syncthreads();
        if (tid == 0 && tile != d.stall_tile) {
            __threadfence();
            st_release(d.progress + tile, base + m + 1);
        }
    }
    // ---- release TMEM (also after an abort: every warp is past its last tcgen05.ld)
    tmem_fence_before();
    __syncthreads();
    tmem_fence_after();
    if (warp == 0) tmem_dealloc_512(tbase);
}

template <typename T>
__global__ void __launch_bounds__(kSmemThreads<T>, 1) k_fv_tmem(Dev<T> d, StepArgs a, T* g0, T* g1) {
    extern __shared__ __align__(16) unsigned char sm[];
    __shared__ int abort_sh;
    __shared__ uint32_t tmem_base_sh;
    fv_tmem_body<T>(d, a, g0, g1, blockIdx.x, sm, abort_sh, tmem_base_sh);
}

// Several solvers' FV sub-steps in one cooperative launch: block b runs
// tile b - block0 of the item whose range [block0, next block0) holds b.
// Each item keeps its own tables, counters, sub-step count and buffers;
// items only share the GPU.
template <typename T>
__global__ void __launch_bounds__(kSmemThreads<T>, 1) k_fv_tmem_pack(const __grid_constant__ FvPack<T> pk) {
    extern __shared__ __align__(16) unsigned char sm[];
    __shared__ int abort_sh;
    __shared__ uint32_t tmem_base_sh;
    int i = 0;
    while (i + 1 < pk.n && pk.block0[i + 1] <= (int)blockIdx.x) ++i;
    fv_tmem_body<T>(pk.d[i], pk.a[i], pk.g0[i], pk.g1[i], (int)blockIdx.x - pk.block0[i], sm, abort_sh,
                    tmem_base_sh);
}

template <typename T>
cudaError_t launch_fv_tmem_pack(const FvPack<T>& pk, int blocks, size_t smem, cudaStream_t s) {
    FvPack<T> p = pk;
    void* args[] = {&p};
    return cudaLaunchCooperativeKernel((const void*)k_fv_tmem_pack<T>, dim3(blocks), dim3(kSmemThreads<T>), args,
                                       smem, s);
}

template <typename T>
int fv_tmem_tile_capacity(size_t smem) {
    if (smem == 0) return 0;
    int dev = 0, sms = 0, per = 0, maxsm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaDeviceGetAttribute(&maxsm, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    // each block allocates all 512 TMEM columns of its SM, so a second block
    // on the same SM would wait for the first: only run where one fits
    for (const void* fn : {(const void*)k_fv_tmem<T>, (const void*)k_fv_tmem_pack<T>}) {
        cudaFuncAttributes fa{};
        if (cudaFuncGetAttributes(&fa, fn) != cudaSuccess) {
            cudaGetLastError();
            return 0;
        }
        const int limit = maxsm - (int)fa.sharedSizeBytes;
        if (smem > (size_t)limit) return 0;
        if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, limit) != cudaSuccess) {
            cudaGetLastError();
            return 0;
        }
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, fn, kSmemThreads<T>, smem);
        if (per != 1) return 0;
    }
    return sms;
}

template <typename T>
cudaError_t launch_fv_tmem(const Dev<T>& d, const StepArgs& a, cudaStream_t s) {
    Dev<T> dd = d;
    StepArgs aa = a;
    T* b0 = (T*)d.fu_in;
    T* b1 = d.fu_out;
    void* args[] = {&dd, &aa, &b0, &b1};
    size_t smem = fv_tmem_smem_bytes<T>(d.tile_cap, d.halo_cap, d.n_sub, d.tile_ocap);
    return cudaLaunchCooperativeKernel((const void*)k_fv_tmem<T>, dim3(d.n_tiles), dim3(kSmemThreads<T>), args, smem,
                                       s);
}

// ---------------------------------------------------------------------------
// Deep tiles: the FV sub-steps with one exchange between tiles every K
// sub-steps (temporal blocking).  A tile holds, as local "slots", its own
// nodes and K layers of ghost nodes around them: layer j holds the nodes
// that the updates of layer j-1 read and that are not in earlier layers
// (outer nodes read nothing, except with outer_fv).  Sub-step s of a block of K recomputes the
// own nodes and ghost layers 1 .. K-1-s from the tile's own data, so the
// tile needs its neighbours' records only once per block.  The arithmetic of
// a node is that of the other FV kernels (fv_node.cuh, same entry order), so
// the results are the same bit for bit.
//
// Exchange.  An own node that other tiles hold as a ghost is sent at the end
// of a block as packets of 16 bytes, three FP32 values (one FP64 value) and
// a tag, each stored and loaded as one 128-bit access: a reader polls the
// packet itself, so that neither a fence, nor a flag, nor a second round
// trip for the data stands between the sender's store and the reader's copy
// (with the counters and cp.async copies of the other kernels, 3.8 us per
// sub-step on a 2588-node FP32 patch at K = 2, 3.7 on 45 304 nodes and 28 on
// 3008 FP64 nodes; with the packets and the pair arithmetic 2.4, 2.6 and
// 17.7, and with several lanes per node, below, 1.6, 2.4 and 7.1).  Tags are unique over the solver's life
// (StepArgs::xtag), so a packet left by an earlier launch is never taken for
// a new one.  Packets alternate between two buffers; a tile overwrites the
// packets of exchange e when it sends exchange e + 2, after having received
// exchange e + 1 of every tile it reads, which that tile sent after its reads
// of exchange e.  A tile read by one that it does not itself read (outer
// nodes read nothing) waits for that tile's progress counter instead.
//
// Slots: own nodes (those reading only own nodes first), then the ghost
// layers in order.  Records of all slots are double-buffered in shared
// memory (pair order: f1 .. f8, f0, z0 .. z2); the FV rows of the computed
// slots live in tensor memory, one row image per slot (header cP, ne, then
// per off-diagonal entry gx, gy, C and the local slot of the column; FP64
// values take two words).  Slot x is updated by thread x % kDeepFv, which
// reads its row image from its own TMEM lane: FP32 runs 768 FV threads of
// two slots and loads a row two entries at a time (64 registers), FP64 512
// threads of two slots that load a row in two halves.  The FP32 block has
// 256 more threads (8 warps) that run the next lattice step's stream-collide
// away from the patch (FarArgs) while the FV warps step the patch.
template <typename T, bool kFar>
constexpr int kDeepThreads = sizeof(T) == 4 ? (kFar ? 1024 : 768) : 512;  // block size
template <typename T>
constexpr int kDeepFv = sizeof(T) == 4 ? 768 : 512;  // FV threads: warps 0 .. kDeepFv / 32 - 1
template <typename T>
constexpr int kDeepSlotWords = sizeof(T) == 4 ? 32 : 64;  // TMEM columns of one slot
template <typename T>
constexpr int kDeepGroups = 2;  // slots per FV thread
template <typename T>
constexpr int kDeepHalf = kDeepSlotWords<T> / 2;  // words per tcgen05.ld of a row
template <typename T>
constexpr int kDeepEntryWords = sizeof(T) == 4 ? 4 : 8;
static_assert(kDeepSlotWords<float> * (kDeepGroups<float> * kDeepFv<float> / 128) <= 512 &&
                  kDeepSlotWords<double> * (kDeepGroups<double> * kDeepFv<double> / 128) <= 512,
              "row images of all slots within the 512 TMEM columns");
static_assert(1 + kTmemMaxEntries <= 8, "row image: header and 7 entries");
template <typename T>
constexpr int kPktValues = sizeof(T) == 4 ? 3 : 1;  // values of a 16-byte packet
template <typename T>
constexpr int kPkts = kSR / kPktValues<T>;  // packets of a record

template <typename T>
int fv_deep_tmem_slots() {
    return kDeepGroups<T> * kDeepFv<T>;
}
// own nodes reading only own nodes from which a tile updates them ahead of the
// others, while the ghosts are on their way: when they fill the FV warps; fewer
// are left for after the wait, since one pass over all slots then takes no
// longer than over a part.  (FP64 from 64 nodes on: the FP64 pipe is busy
// either way; 25.5 instead of 22.6 us per sub-step on 24 380 nodes, K = 2.)
template <typename T>
int fv_deep_early() {
    return kDeepFv<T>;
}
template <typename T>
int fv_deep_row_words() {
    return kDeepSlotWords<T>;
}
template <typename T>
size_t fv_deep_packet_bytes(int n) {
    return (size_t)2 * n * kPkts<T> * 16;
}

// Quads (FP64, small tiles): rows in shared memory, one is 7 entries (g.c of the
// four axes, C, column) and a header.  They are a branch of the kernel that keeps
// a node per lane's rows in tensor memory, which is allocated all the same.
struct alignas(16) QuadEntry {
    double k[4];  // gx, gy, gx + gy, gx - gy
    double c;
    int32_t col, pad;
};
struct alignas(16) QuadRow {
    QuadEntry e[kTmemMaxEntries];
    double cP;
    int32_t ne, pad;
};

struct DeepSmem {
    size_t buf0, buf1, uv, osnap, star, rows, gid, kind, send, omap, total;
};

// quad_rows: computed slots whose rows are kept in shared memory (0: none);
// stars: outer slots whose interpolated records are kept, twice (outer_fv)
template <typename T>
__host__ __device__ inline DeepSmem deep_smem_layout(int cap, int n_sub, int ocap, int quad_rows, int stars) {
    auto up = [](size_t x) { return (x + 15) / 16 * 16; };
    DeepSmem L;
    size_t o = 0;
    L.buf0 = o;
    o = up(o + sizeof(T) * kSR * (size_t)cap);
    L.buf1 = o;
    o = up(o + sizeof(T) * kSR * (size_t)cap);
    L.uv = o;
    o = up(o + sizeof(T) * 2 * (size_t)n_sub);
    L.osnap = o;
    o = up(o + sizeof(T) * kSnap * (size_t)ocap);
    L.star = o;
    o = up(o + 2 * sizeof(T) * kSR * (size_t)stars);
    L.rows = o;
    o = up(o + sizeof(QuadRow) * (size_t)quad_rows);
    L.gid = o;
    o = up(o + sizeof(int32_t) * (size_t)cap);
    L.kind = o;
    o = up(o + (size_t)cap);
    L.send = o;
    o = up(o + (size_t)cap);
    L.omap = o;
    o = up(o + sizeof(int16_t) * (size_t)cap);
    L.total = o;
    return L;
}

template <typename T>
size_t fv_deep_smem_bytes(int slot_cap, int n_sub, int ocap, int quad_rows, int stars) {
    return deep_smem_layout<T>(slot_cap, n_sub, ocap, quad_rows, stars).total;
}

// ---- packets: one relaxed 128-bit access each (value bits low, tag on top)
struct Packet {
    unsigned long long lo, hi;
};
__device__ __forceinline__ void st_packet(void* p, unsigned long long lo, unsigned long long hi) {
    asm volatile(
        "{\n\t.reg .b128 q;\n\tmov.b128 q, {%1, %2};\n\tst.relaxed.gpu.global.b128 [%0], q;\n\t}" ::"l"(p), "l"(lo),
        "l"(hi)
        : "memory");
}
__device__ __forceinline__ Packet ld_packet(const void* p) {
    Packet k;
    asm volatile("{\n\t.reg .b128 q;\n\tld.relaxed.gpu.global.b128 q, [%2];\n\tmov.b128 {%0, %1}, q;\n\t}"
                 : "=l"(k.lo), "=l"(k.hi)
                 : "l"(p)
                 : "memory");
    return k;
}
__device__ __forceinline__ unsigned packet_tag(const Packet& k) { return (unsigned)(k.hi >> 32); }

// the packets of a record of pairs (order of the shared-memory records)
__device__ __forceinline__ void send_record(unsigned char* p, const RecP<float>& r, unsigned tag) {
    const unsigned long long t = (unsigned long long)tag << 32;
    auto w = [](float v) { return (unsigned long long)__float_as_uint(v); };
    st_packet(p, r.A.v, t | w(px(r.B)));
    st_packet(p + 16, w(py(r.B)) | (w(px(r.C)) << 32), t | w(py(r.C)));
    st_packet(p + 32, r.D.v, t | w(px(r.E)));
    st_packet(p + 48, w(py(r.E)) | (w(px(r.F)) << 32), t | w(py(r.F)));
}
__device__ __forceinline__ void send_record(unsigned char* p, const RecP<double>& r, unsigned tag) {
    const unsigned long long t = (unsigned long long)tag << 32;
    const double v[12] = {r.A.a, r.A.b, r.B.a, r.B.b, r.C.a, r.C.b, r.D.a, r.D.b, r.E.a, r.E.b, r.F.a, r.F.b};
#pragma unroll
    for (int k = 0; k < 12; ++k) st_packet(p + 16 * k, (unsigned long long)__double_as_longlong(v[k]), t);
}
// a packet's values into the record at dst (packet c of it)
__device__ __forceinline__ void take_packet(float* dst, int c, const Packet& k) {
    dst[3 * c] = __uint_as_float((unsigned)k.lo);
    dst[3 * c + 1] = __uint_as_float((unsigned)(k.lo >> 32));
    dst[3 * c + 2] = __uint_as_float((unsigned)k.hi);
}
__device__ __forceinline__ void take_packet(double* dst, int c, const Packet& k) {
    dst[c] = __longlong_as_double((long long)k.lo);
}

// ---- records of pairs in shared memory (16-byte accesses)
__device__ __forceinline__ RecP<float> ld_rec(const float* p) {
    RecP<float> r;
    const ulonglong2 a = *reinterpret_cast<const ulonglong2*>(p), b = *reinterpret_cast<const ulonglong2*>(p + 4),
                     c = *reinterpret_cast<const ulonglong2*>(p + 8);
    r.A.v = a.x, r.B.v = a.y, r.C.v = b.x, r.D.v = b.y, r.E.v = c.x, r.F.v = c.y;
    return r;
}
__device__ __forceinline__ RecP<double> ld_rec(const double* p) {
    const double2* q = reinterpret_cast<const double2*>(p);
    RecP<double> r;
    auto get = [&](int k) {
        const double2 v = q[k];
        return pk(v.x, v.y);
    };
    r.A = get(0), r.B = get(1), r.C = get(2), r.D = get(3), r.E = get(4), r.F = get(5);
    return r;
}
__device__ __forceinline__ void st_rec(float* p, const RecP<float>& r) {
    *reinterpret_cast<ulonglong2*>(p) = make_ulonglong2(r.A.v, r.B.v);
    *reinterpret_cast<ulonglong2*>(p + 4) = make_ulonglong2(r.C.v, r.D.v);
    *reinterpret_cast<ulonglong2*>(p + 8) = make_ulonglong2(r.E.v, r.F.v);
}
__device__ __forceinline__ void st_rec(double* p, const RecP<double>& r) {
    double2* q = reinterpret_cast<double2*>(p);
    auto put = [&](int k, const Pr<double>& v) { q[k] = make_double2(v.a, v.b); };
    put(0, r.A), put(1, r.B), put(2, r.C), put(3, r.D), put(4, r.E), put(5, r.F);
}
template <typename T>
__device__ __forceinline__ RecP<T> rec_of(const Pops<T>& p, const T (&z)[3]) {
    return RecP<T>{p.A, p.B, p.C, p.D, pk(p.f0, z[0]), pk(z[1], z[2])};
}

// 16 or 32 words of this thread's TMEM lane, complete on return
template <int N>
__device__ __forceinline__ void tmem_ldn(uint32_t taddr, uint32_t (&v)[N]) {
    static_assert(N == 32, "x32");
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, "
        "%14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
          "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]),
          "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]),
          "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
        : "r"(taddr)
        : "memory");
}

// entry (gx, gy, C, column) at word w of a row image half
template <typename T, int N>
__device__ __forceinline__ void deep_entry(const uint32_t (&v)[N], int w, T& gx, T& gy, T& c, int& col) {
    gx = from_words<T>(v[w], v[w + 1]);
    gy = from_words<T>(v[w + 2], v[w + 3]);
    c = from_words<T>(v[w + 4], v[w + 5]);
    col = (int)v[w + 6];
}

// Record of one node's sub-step for the reverse mode (StepArgs-wide buffer
// Dev::fv_rec, [n_sub][n][kAdjRec]): the collision sums n_1 .. n_8, n_0, the
// velocity of the state before the sub-step, and at wall nodes rho and u of
// the update before the wall rule.
constexpr int kAdjRec = 16;
enum { kAdjN0 = 8, kAdjU = 9, kAdjWall = 11 };

template <typename T>
__device__ __forceinline__ void adj_record(const Dev<T>& d, int m, int g, bool row, const Pops<T>& n, bool wall,
                                           const T (&mo)[3], T ux, T uy) {
    T* r = d.fv_rec + ((int64_t)m * d.n + g) * kAdjRec;
    if (row) {
        const T v[9] = {px(n.A), py(n.A), px(n.B), py(n.B), px(n.C), py(n.C), px(n.D), py(n.D), n.f0};
#pragma unroll
        for (int i = 0; i < 9; ++i) r[i] = v[i];
        if (wall) {
#pragma unroll
            for (int j = 0; j < 3; ++j) r[kAdjWall + j] = mo[j];
        }
    }
    if (m + 1 < d.n_sub) {  // the velocity of the next sub-step's state
        r[(int64_t)d.n * kAdjRec + kAdjU] = ux;
        r[(int64_t)d.n * kAdjRec + kAdjU + 1] = uy;
    }
}

// The update of slot x (warp-uniform call: lanes with valid = false take
// part in the TMEM loads only), written into the next record buffer and,
// when pkt is set, sent to the tiles that hold the node as a ghost.  The row
// image is loaded by every lane of the warp at points where the warp is
// converged (tcgen05.ld is .sync.aligned); only the arithmetic between the
// loads is predicated.
// kOuterFv: outer nodes take eq. postcollision2_u with its FV sums (outer_fv):
// their row is summed like any other, over the starred values -- star, the
// interpolated records of this sub-step at outer slots, own one included, and
// the patch records elsewhere.
template <typename T, bool kRecord, bool kOuterFv>
__device__ __forceinline__ void deep_node(const Dev<T>& d, const unsigned char* sm, const DeepSmem& L, const T* cur,
                                          T* nxt, uint32_t tslot, bool valid, int x, int m, unsigned char* pkt,
                                          unsigned tag, bool own_slot, const T* star) {
    constexpr int EW = kDeepEntryWords<T>;
    const int8_t* kd = reinterpret_cast<const int8_t*>(sm + L.kind);
    const int16_t* om = reinterpret_cast<const int16_t*>(sm + L.omap);
    const int8_t kind = valid ? kd[x] : (int8_t)HLBM_NODE_OUTER;
    const bool outer = kind == HLBM_NODE_OUTER;
    const bool row = kOuterFv ? valid : !outer;  // the slot's row is summed
    const T* own_rec = cur + (size_t)kSR * x;
    if (kOuterFv && outer && valid) own_rec = star + (size_t)kSR * om[x];
    auto rec_at = [&](int col) {
        const T* r = cur + (size_t)kSR * col;
        if (kOuterFv && outer && kd[col] == HLBM_NODE_OUTER) r = star + (size_t)kSR * om[col];
        return ld_rec(r);
    };
    Pops<T> P{};
    if (row) {
        const RecP<T> own = ld_rec(own_rec);
        P.A = own.A, P.B = own.B, P.C = own.C, P.D = own.D;
    }
    FvSums<T> acc;
    fv_sums_init(acc);
    T cP;
    if constexpr (sizeof(T) == 4) {
        // header, then the entries two by two up to the warp's longest row
        uint32_t hdr[4];
        tmem_ld4(tslot, hdr);
        cP = __uint_as_float(hdr[0]);
        const int ne = row ? (int)hdr[1] : 0;
        const int nem = (int)__reduce_max_sync(0xffffffffu, (unsigned)ne);
        // two entries per tensor-memory load (one wait for both; entry 7 of
        // the last pair reads the next columns, which no row uses)
#pragma unroll
        for (int j = 0; j < kTmemMaxEntries; j += 2) {
            if (j >= nem) break;
            uint32_t e[8];
            tmem_ld8(tslot + EW * (j + 1), e);
            if (j < ne)
                fv_sums_entry(acc, __uint_as_float(e[0]), __uint_as_float(e[1]), __uint_as_float(e[2]),
                              rec_at((int)e[3]), P);
            if (j + 1 < ne)
                fv_sums_entry(acc, __uint_as_float(e[4]), __uint_as_float(e[5]), __uint_as_float(e[6]),
                              rec_at((int)e[7]), P);
        }
    } else {
        constexpr int H = kDeepHalf<T>;
        constexpr int E0 = H / EW - 1;  // entries in the first half (after the header)
        uint32_t v[H];
        tmem_ldn<H>(tslot, v);
        cP = from_words<T>(v[0], v[1]);
        const int ne = row ? (int)v[2] : 0;
#pragma unroll
        for (int j = 0; j < E0; ++j) {
            if (j < ne) {
                T gx, gy, c;
                int col;
                deep_entry<T, H>(v, EW * (j + 1), gx, gy, c, col);
                fv_sums_entry(acc, gx, gy, c, rec_at(col), P);
            }
        }
        __syncwarp();
        tmem_ldn<H>(tslot + H, v);  // entries E0 .. 6
#pragma unroll
        for (int j = E0; j < kTmemMaxEntries; ++j) {
            if (j < ne) {
                T gx, gy, c;
                int col;
                deep_entry<T, H>(v, EW * (j - E0), gx, gy, c, col);
                fv_sums_entry(acc, gx, gy, c, rec_at(col), P);
            }
        }
    }
    if (!valid) return;
    Pops<T> fn, nq{};
    T mo[3] = {};
    if (!row) {
        fn = fv_outer_from(d, reinterpret_cast<const T*>(sm + L.osnap) + kSnap * om[x], 1, m);
    } else {
        fn = fv_sums_finish(d, acc, cP, ld_rec(own_rec), nq);
        if (kind == HLBM_NODE_WALL) {
            const T* uv = reinterpret_cast<const T*>(sm + L.uv);
            fv_wall(d, uv[m], uv[d.n_sub + m], fn, mo);
        }
    }
    T z[3], ux, uy;
    z_of(fn, d.rho0, z, ux, uy);
    if constexpr (kRecord) {
        if (own_slot)
            adj_record(d, m, reinterpret_cast<const int32_t*>(sm + L.gid)[x], kind != HLBM_NODE_OUTER, nq,
                       kind == HLBM_NODE_WALL, mo, ux, uy);
    }
    const RecP<T> r = rec_of(fn, z);
    st_rec(nxt + (size_t)kSR * x, r);
    if (pkt) send_record(pkt, r, tag);
}

// ---- FP64 quads.  FP64 instructions issue at one per 64 cycles from a warp
// and one per 19 from an SM (measured; however many lanes are active), so a
// warp that updates a node per lane (some 400 FP64 instructions) takes 12 us
// even when it is alone on its SM, while the other three partitions idle.
// On small tiles four lanes share a node: lane q of a quad holds the pair of
// opposite directions q (x, y, (1,1), (-1,1)) and one of f0, z0, z1, z2,
// some 110 instructions, and the sums over directions go through shuffles
// within the quad: 7.2 us per sub-step against 17.7 on a 3008-node patch
// (with tiles of at least 16 nodes instead of 64).  Every value is formed by the expression of fv_node.cuh,
// so the bits are those of a node per lane.
struct Quad {
    int q;              // lane in the quad
    double w;           // weight of the lane's directions
    double sgn;         // +1 on odd lanes, -1 on even ones
};
__device__ __forceinline__ double qshfl(double v, int src) { return __shfl_sync(0xffffffffu, v, src, 4); }

// moments of the set whose pair (a, b) each lane holds, f0 in lane 0's e
__device__ __forceinline__ void quad_moments(const Quad& Q, double a, double b, double e, double& m0, double& mx,
                                             double& my) {
    const double s = __dadd_rn(a, b), dd = __dsub_rn(a, b);
    const double s2 = __dadd_rn(s, __shfl_xor_sync(0xffffffffu, s, 1));
    const double s4 = __dadd_rn(s2, __shfl_xor_sync(0xffffffffu, s2, 2));
    m0 = __dadd_rn(qshfl(e, 0), s4);
    const double v = __dadd_rn(dd, __fma_rn(Q.sgn, qshfl(dd, 3), qshfl(dd, 2)));
    mx = qshfl(v, 0);
    my = qshfl(v, 1);
}
// c . (x, y) of the lane's first direction
__device__ __forceinline__ double quad_dot(const Quad& Q, double x, double y) {
    const double v = __fma_rn(Q.q == 3 ? -1.0 : 1.0, x, y);
    return Q.q == 0 ? x : Q.q == 1 ? y : v;
}

// the update of the quad's slot x (every lane of the warp takes part)
template <bool kRecord>
__device__ __forceinline__ void quad_node(const Dev<double>& d, const unsigned char* sm, const DeepSmem& L,
                                          const double* cur, double* nxt, const Quad& Q, bool valid, int x, int m,
                                          unsigned char* pkt, unsigned tag, bool own_slot) {
    double* rec = nullptr;  // this sub-step's record of the node
    if constexpr (kRecord) {
        if (valid && own_slot)
            rec = d.fv_rec + ((int64_t)m * d.n + reinterpret_cast<const int32_t*>(sm + L.gid)[x]) * kAdjRec;
    }
    const int q = Q.q, ia = q < 2 ? q : q + 2, ib = ia + 2, ie = 8 + q;
    const int8_t kind = valid ? reinterpret_cast<const int8_t*>(sm + L.kind)[x] : (int8_t)HLBM_NODE_OUTER;
    const bool row = kind != HLBM_NODE_OUTER;
    double a = 0.0, b = 0.0, e = 0.0;
    if (__any_sync(0xffffffffu, row)) {
        const QuadRow* R = reinterpret_cast<const QuadRow*>(sm + L.rows) + (row ? x : 0);
        const double* own = cur + (size_t)kSR * (row ? x : 0);
        const double Pa = own[ia], Pb = own[ib], Pe = own[ie];
        const int ne = row ? R->ne : 0;
        double Sa = 0.0, Sb = 0.0, Ca = 0.0, Cb = 0.0, Ce = 0.0;
#pragma unroll 2
        for (int j = 0; j < ne; ++j) {
            const double k = R->e[j].k[q], c = R->e[j].c;
            const double* o = cur + (size_t)kSR * R->e[j].col;
            const double fa = o[ia], fb = o[ib], fe = o[ie];
            Sa = __fma_rn(k, __dsub_rn(fa, Pa), Sa);
            Sb = __fma_rn(k, __dsub_rn(fb, Pb), Sb);
            Ca = __fma_rn(c, fa, Ca);
            Cb = __fma_rn(c, fb, Cb);
            Ce = __fma_rn(c, fe, Ce);
        }
        __syncwarp();
        Ca = __fma_rn(R->cP, Pa, Ca);
        Cb = __fma_rn(R->cP, Pb, Cb);
        Ce = __fma_rn(R->cP, Pe, Ce);
        double dr, jx, jy;
        quad_moments(Q, Ca, Cb, Ce, dr, jx, jy);
        const double Z0 = qshfl(Ce, 1), Z1 = qshfl(Ce, 2), Z2 = qshfl(Ce, 3);
        const double zs = __dadd_rn(Z0, Z2), q0 = __fma_rn(-1.5, zs, dr);
        const double zd = __fma_rn(q == 3 ? -2.0 : 2.0, Z1, zs);
        const double G = __fma_rn(4.5, q == 0 ? Z0 : q == 1 ? Z2 : zd, q0), H = __dmul_rn(3.0, quad_dot(Q, jx, jy));
        Ca = __fma_rn(-Q.w, __dadd_rn(G, H), Ca);
        Cb = __fma_rn(-Q.w, __dsub_rn(G, H), Cb);
        Ce = __fma_rn(-w_of<double>(0), q0, Ce);
        double m0, mx, my;
        quad_moments(Q, Ca, Cb, Ce, m0, mx, my);
        const double H2 = __dmul_rn(3.0, quad_dot(Q, mx, my));
        Ca = __fma_rn(-Q.w, __dadd_rn(m0, H2), Ca);
        Cb = __fma_rn(-Q.w, __dsub_rn(m0, H2), Cb);
        Ce = __fma_rn(-w_of<double>(0), m0, Ce);
        const double iv = q == 3 ? -d.inv_tau_u : d.inv_tau_u, dt = q == 3 ? -d.dt_u : d.dt_u;
        a = __fma_rn(dt, __fma_rn(-iv, Ca, Sa), Pa);
        b = __fma_rn(-dt, __fma_rn(iv, Cb, Sb), Pb);
        e = __fma_rn(d.dt_u, __dmul_rn(-d.inv_tau_u, Ce), Pe);
        const bool wall = kind == HLBM_NODE_WALL;
        if constexpr (kRecord) {
            if (rec && row) {
                rec[ia] = Ca;
                rec[ib] = Cb;
                if (q == 0) rec[kAdjN0] = Ce;
            }
        }
        if (__any_sync(0xffffffffu, wall)) {
            const double* uv = reinterpret_cast<const double*>(sm + L.uv);
            const double U = uv[m], V = uv[d.n_sub + m];
            quad_moments(Q, a, b, e, dr, jx, jy);
            const double rho = __dadd_rn(d.rho0, dr), inv = 1.0 / rho;
            const double ux = __dmul_rn(jx, inv), uy = __dmul_rn(jy, inv);
            const double dx = __dsub_rn(U, ux), dy = __dsub_rn(V, uy), sx = __dadd_rn(U, ux), sy = __dadd_rn(V, uy);
            const double bb = __dmul_rn(-1.5, __fma_rn(dx, sx, __dmul_rn(dy, sy)));
            const double cd = quad_dot(Q, dx, dy);
            const double Gw = __fma_rn(__dmul_rn(4.5, cd), quad_dot(Q, sx, sy), bb), Hw = __dmul_rn(3.0, cd);
            const double wr = __dmul_rn(Q.w, rho);
            if constexpr (kRecord) {
                if (rec && wall && q < 3) rec[kAdjWall + q] = q == 0 ? rho : q == 1 ? ux : uy;
            }
            if (wall) {
                a = __fma_rn(wr, __dadd_rn(Gw, Hw), a);
                b = __fma_rn(wr, __dsub_rn(Gw, Hw), b);
                e = __fma_rn(__dmul_rn(w_of<double>(0), rho), bb, e);
            }
        }
    }
    if (valid && !row) {
        const double* sn = reinterpret_cast<const double*>(sm + L.osnap) +
                           kSnap * reinterpret_cast<const int16_t*>(sm + L.omap)[x];
        const double th = double(m + 1) / double(d.n_sub), t0 = __dsub_rn(1.0, th);
        auto at = [&](int j) { return __fma_rn(t0, sn[j], __dmul_rn(th, sn[12 + j])); };
        const double dr = at(0), ux = at(1), uy = at(2), rho = __dadd_rn(d.rho0, dr);
        const double qq = __dmul_rn(-1.5, __fma_rn(ux, ux, __dmul_rn(uy, uy))), c = quad_dot(Q, ux, uy);
        const double G = __fma_rn(rho, __fma_rn(__dmul_rn(4.5, c), c, qq), dr), H = __dmul_rn(rho, __dmul_rn(3.0, c));
        a = __fma_rn(d.kneq, at(4 + ia), __dmul_rn(Q.w, __dadd_rn(G, H)));
        b = __fma_rn(d.kneq, at(4 + ib), __dmul_rn(Q.w, __dsub_rn(G, H)));
        e = __fma_rn(d.kneq, at(3), __dmul_rn(w_of<double>(0), __fma_rn(rho, qq, dr)));
    }
    __syncwarp();
    double dr, jx, jy;
    quad_moments(Q, a, b, e, dr, jx, jy);
    const double inv = 1.0 / __dadd_rn(d.rho0, dr), ux = __dmul_rn(jx, inv), uy = __dmul_rn(jy, inv);
    if (q != 0) e = __dmul_rn(q == 3 ? jy : jx, q == 1 ? ux : uy);
    if constexpr (kRecord) {
        if (rec && m + 1 < d.n_sub && q < 2) rec[(int64_t)d.n * kAdjRec + kAdjU + q] = q == 0 ? ux : uy;
    }
    if (!valid) return;
    double* o = nxt + (size_t)kSR * x;
    o[ia] = a;
    o[ib] = b;
    o[ie] = e;
    if (pkt) {
        const unsigned long long t = (unsigned long long)tag << 32;
        st_packet(pkt + 16 * ia, (unsigned long long)__double_as_longlong(a), t);
        st_packet(pkt + 16 * ib, (unsigned long long)__double_as_longlong(b), t);
        st_packet(pkt + 16 * ie, (unsigned long long)__double_as_longlong(e), t);
    }
}

// ---- FP32 pairs of lanes.  With one node per thread the few warps of a small
// tile have nothing to overlap the update's chain of some 500 instructions
// with: 1.85 us of a sub-step's 2.3 on a 2588-node patch (63 own nodes per
// tile), 1.0 / K more for the exchange.  Where a tile's computed slots fit, two
// lanes share a node: lane 0 holds the pairs A, B (axes) and E, lane 1 C, D
// (diagonals) and F, each with its share of the row in registers; the sums
// over directions take one shuffle: 1.6 us per sub-step on that patch, 2.4 on
// 45 304 nodes.  Every value is formed by the expression of fv_node.cuh, so the
// bits are those of a node per lane.
constexpr int kDuoThreads = 768;  // 80 registers a thread
constexpr int kDuoSlots = kDuoThreads / 2;
struct Duo {
    int q;                             // lane of the pair
    Pr<float> w, dt1, iv1, dt2, iv2;  // minus the weights; the update's signed factors
};
struct DuoRow {
    Pr<float> k[kTmemMaxEntries];  // (gx, gy) on lane 0, (gx + gy, gx - gy) on lane 1; 0 past the row's end
    float c[kTmemMaxEntries];
    int col[kTmemMaxEntries];      // 4 times the slot
    float cP;
};
// Records of cap slots: the pairs A, B of every slot, then C, D, then E, F (cap
// is 4 modulo 8, so that the two lanes of four neighbouring slots read eight
// different bank quads; records of 48 bytes gave two-way conflicts: 52 % of the
// shared-memory cycles of the 45k-node patch's sub-steps)
__host__ __device__ constexpr int duo_cap(int n) { return (n + 3) / 8 * 8 + 4; }
__device__ __forceinline__ int duo_ab(int cap, int q) { return 4 * q * cap; }
__device__ __forceinline__ int duo_ef(int cap, int q) { return 8 * cap + 2 * q; }
__device__ __forceinline__ void duo_put(float* buf, int cap, int x, const RecP<float>& r) {
    *reinterpret_cast<ulonglong2*>(buf + 4 * x) = make_ulonglong2(r.A.v, r.B.v);
    *reinterpret_cast<ulonglong2*>(buf + 4 * cap + 4 * x) = make_ulonglong2(r.C.v, r.D.v);
    *reinterpret_cast<ulonglong2*>(buf + 8 * cap + 4 * x) = make_ulonglong2(r.E.v, r.F.v);
}
__device__ __forceinline__ Pr<float> duo_zero() { return pk(0.0f, 0.0f); }
__device__ __forceinline__ float duo_other(float v) { return __shfl_xor_sync(0xffffffffu, v, 1); }
// (x, y) on lane 0, (x + y, y - x) on lane 1
__device__ __forceinline__ Pr<float> duo_axes(const Duo& Q, float x, float y) {
    return pk(Q.q ? add_rn(x, y) : x, Q.q ? sub_rn(y, x) : y);
}
// moments of the set whose pairs (a, b) each lane holds, f0 in lane 0's e: the
// sums run over directions 0 .. 4 on lane 0, then 5 .. 8 on lane 1
__device__ __forceinline__ void duo_moments(Pr<float> a, Pr<float> b, float e, float& m0, float& mx, float& my) {
    auto from = [](float v, int lane) { return __shfl_sync(0xffffffffu, v, lane, 2); };
    const float f1 = px(a), f2 = py(a), f3 = px(b), f4 = py(b);
    m0 = from(add_rn(add_rn(add_rn(add_rn(e, f1), f2), f3), f4), 0);
    mx = from(sub_rn(f1, f3), 0);
    my = from(sub_rn(f2, f4), 0);
    m0 = from(add_rn(add_rn(add_rn(add_rn(m0, f1), f2), f3), f4), 1);
    mx = from(add_rn(sub_rn(sub_rn(add_rn(mx, f1), f2), f3), f4), 1);
    my = from(sub_rn(sub_rn(add_rn(add_rn(my, f1), f2), f3), f4), 1);
}
// the pairs minus w (g + 3 c . (x, y) + 4.5 Q)
template <bool kQuad>
__device__ __forceinline__ void duo_sub_lin(const Duo& Q, float g, float x, float y, Pr<float> quad, Pr<float>& a,
                                            Pr<float>& b) {
    const Pr<float> c = duo_axes(Q, x, y), gg = pk(g, g), h = pk(4.5f, 4.5f);
    Pr<float> A = pfma(pk(3.0f, 3.0f), c, gg), B = pfma(pk(-3.0f, -3.0f), c, gg);
    if (kQuad) A = pfma(h, quad, A), B = pfma(h, quad, B);
    a = pfma(Q.w, A, a);
    b = pfma(Q.w, B, b);
}

template <bool kRecord, bool kOuterFv>
__device__ __forceinline__ void duo_node(const Dev<float>& d, const unsigned char* sm, const DeepSmem& L,
                                         const float* cur, float* nxt, const Duo& Q, const DuoRow& R, bool valid, int x,
                                         int m, unsigned char* pkt, unsigned tag, bool own_slot, const float* star) {
    const int q = Q.q, ia = 4 * q;
    const int8_t* kd = reinterpret_cast<const int8_t*>(sm + L.kind);
    const int16_t* om = reinterpret_cast<const int16_t*>(sm + L.omap);
    const int8_t kind = valid ? kd[x] : (int8_t)HLBM_NODE_OUTER;
    const bool outer = kind == HLBM_NODE_OUTER;
    const bool row = kOuterFv ? valid : !outer;
    const int cap = d.deep_slot_cap;
    auto pairs = [&](const float* ab, const float* ef, Pr<float>& a, Pr<float>& b, Pr<float>& e) {
        const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(ab);
        a.v = v.x;
        b.v = v.y;
        e.v = *reinterpret_cast<const unsigned long long*>(ef);
    };
    float* rec = nullptr;
    if constexpr (kRecord) {
        if (valid && own_slot) rec = d.fv_rec + ((int64_t)m * d.n + reinterpret_cast<const int32_t*>(sm + L.gid)[x]) * kAdjRec;
    }
    Pr<float> a = duo_zero(), b = a, e = a;
    if (__any_sync(0xffffffffu, row)) {
        const float *ab = cur + duo_ab(cap, q), *ef = cur + duo_ef(cap, q);
        const float *sab = nullptr, *sef = nullptr;  // interpolated records (outer_fv)
        const int own = 4 * (valid ? x : 0);
        Pr<float> Pa, Pb, Pe, Sa = a, Sb = a, Ca = a, Cb = a, Ce = a;
        if (kOuterFv && outer && valid) {
            sab = star + duo_ab(d.deep_ocap, q), sef = star + duo_ef(d.deep_ocap, q);
            pairs(sab + 4 * om[x], sef + 4 * om[x], Pa, Pb, Pe);
        } else {
            pairs(ab + own, ef + own, Pa, Pb, Pe);
        }
#pragma unroll
        for (int j = 0; j < kTmemMaxEntries; ++j) {
            Pr<float> fa, fb, fe;
            if (kOuterFv && outer && valid && kd[R.col[j] >> 2] == HLBM_NODE_OUTER) {
                const int o = 4 * om[R.col[j] >> 2];
                pairs(sab + o, sef + o, fa, fb, fe);
            } else {
                pairs(ab + R.col[j], ef + R.col[j], fa, fb, fe);
            }
            const Pr<float> cc = pk(R.c[j], R.c[j]);
            Sa = pfma(R.k[j], psub(fa, Pa), Sa);
            Sb = pfma(R.k[j], psub(fb, Pb), Sb);
            Ca = pfma(cc, fa, Ca);
            Cb = pfma(cc, fb, Cb);
            Ce = pfma(cc, fe, Ce);
        }
        const Pr<float> cP = pk(R.cP, R.cP);
        Ca = pfma(cP, Pa, Ca);
        Cb = pfma(cP, Pb, Cb);
        Ce = pfma(cP, Pe, Ce);
        // collision sums: lane 0 has (Cf_0, Z0), lane 1 (Z1, Z2)
        float dr, jx, jy, n0 = px(Ce);
        duo_moments(Ca, Cb, n0, dr, jx, jy);
        const float zo = py(Ce), zx = duo_other(zo), Z0 = q ? zx : zo, Z2 = q ? zo : zx;
        const float zs = add_rn(Z0, Z2), q0 = fma_rn(-1.5f, zs, dr);
        const Pr<float> u = pk(q ? add_rn(fma_rn(2.0f, px(Ce), Z0), Z2) : Z0, q ? add_rn(fma_rn(-2.0f, px(Ce), Z0), Z2) : Z2);
        duo_sub_lin<true>(Q, q0, jx, jy, u, Ca, Cb);
        n0 = fma_rn(-w_of<float>(0), q0, n0);
        float m0, mx, my;
        duo_moments(Ca, Cb, n0, m0, mx, my);
        duo_sub_lin<false>(Q, m0, mx, my, Ca, Ca, Cb);
        n0 = fma_rn(-w_of<float>(0), m0, n0);
        a = pfma(Q.dt1, pfma(Q.iv1, Ca, Sa), Pa);
        b = pfma(Q.dt2, pfma(Q.iv2, Cb, Sb), Pb);
        float f0 = fma_rn(d.dt_u, mul_rn(-d.inv_tau_u, n0), px(Pe));
        const bool wall = kind == HLBM_NODE_WALL;
        if constexpr (kRecord) {
            if (rec && row) {
                *reinterpret_cast<ulonglong2*>(rec + ia) = make_ulonglong2(Ca.v, Cb.v);
                if (q == 0) rec[kAdjN0] = n0;
            }
        }
        if (__any_sync(0xffffffffu, wall)) {
            const float* uv = reinterpret_cast<const float*>(sm + L.uv);
            const float U = uv[m], V = uv[d.n_sub + m];
            duo_moments(a, b, f0, dr, jx, jy);
            const float rho = add_rn(d.rho0, dr), inv = 1.0f / rho;
            const float ux = mul_rn(jx, inv), uy = mul_rn(jy, inv);
            const float usq = fma_rn(ux, ux, mul_rn(uy, uy)), Usq = fma_rn(U, U, mul_rn(V, V));
            const float wl = q ? w_of<float>(5) : w_of<float>(1), w0 = w_of<float>(0);
            Pr<float> Xa, Xb, Ya, Yb;
            feq_x(duo_axes(Q, U, V), dr, rho, Usq, Xa, Xb);
            feq_x(duo_axes(Q, ux, uy), dr, rho, usq, Ya, Yb);
            const float X0 = fma_rn(rho, mul_rn(-1.5f, Usq), dr), Y0 = fma_rn(rho, mul_rn(-1.5f, usq), dr);
            if constexpr (kRecord) {
                if (rec && wall) {
                    if (q == 0) rec[kAdjWall] = rho;
                    rec[kAdjWall + 1 + q] = q ? uy : ux;
                }
            }
            if (wall) {
                a = padd(a, pfma(pk(wl, wl), Xa, pmul(pk(-wl, -wl), Ya)));
                b = padd(b, pfma(pk(wl, wl), Xb, pmul(pk(-wl, -wl), Yb)));
                f0 = add_rn(f0, fma_rn(w0, X0, mul_rn(-w0, Y0)));
            }
        }
        e = pk(f0, 0.0f);
    }
    if (valid && !row) {
        const float* sn = reinterpret_cast<const float*>(sm + L.osnap) + kSnap * om[x];
        const float th = float(m + 1) / float(d.n_sub), t0 = sub_rn(1.0f, th);
        auto at = [&](int j) { return fma_rn(t0, sn[j], mul_rn(th, sn[12 + j])); };
        const float dr = at(0), ux = at(1), uy = at(2), rho = add_rn(d.rho0, dr);
        const float usq = fma_rn(ux, ux, mul_rn(uy, uy)), wl = q ? w_of<float>(5) : w_of<float>(1);
        const Pr<float> w = pk(wl, wl), kk = pk(d.kneq, d.kneq);
        Pr<float> Xa, Xb;
        feq_x(duo_axes(Q, ux, uy), dr, rho, usq, Xa, Xb);
        a = pfma(kk, pk(at(4 + ia), at(5 + ia)), pmul(w, Xa));
        b = pfma(kk, pk(at(6 + ia), at(7 + ia)), pmul(w, Xb));
        e = pk(fma_rn(d.kneq, at(3), mul_rn(w_of<float>(0), fma_rn(rho, mul_rn(-1.5f, usq), dr))), 0.0f);
    }
    __syncwarp();
    float dr, jx, jy;
    duo_moments(a, b, px(e), dr, jx, jy);
    const float inv = 1.0f / add_rn(d.rho0, dr), ux = mul_rn(jx, inv), uy = mul_rn(jy, inv);
    e = q ? pk(mul_rn(mul_rn(jx, jy), inv), mul_rn(mul_rn(jy, jy), inv)) : pk(px(e), mul_rn(mul_rn(jx, jx), inv));
    if constexpr (kRecord) {
        if (rec && m + 1 < d.n_sub) rec[(int64_t)d.n * kAdjRec + kAdjU + q] = q ? uy : ux;
    }
    if (!valid) return;
    *reinterpret_cast<ulonglong2*>(nxt + duo_ab(cap, q) + 4 * x) = make_ulonglong2(a.v, b.v);
    *reinterpret_cast<unsigned long long*>(nxt + duo_ef(cap, q) + 4 * x) = e.v;
    if (pkt) {  // packets 2 q, 2 q + 1: (a, b.x), (b.y, e)
        const unsigned long long t = (unsigned long long)tag << 32;
        auto w = [](float v) { return (unsigned long long)__float_as_uint(v); };
        st_packet(pkt + 32 * q, a.v, t | w(px(b)));
        st_packet(pkt + 32 * q + 16, w(py(b)) | (w(px(e)) << 32), t | w(py(e)));
    }
}
__device__ __forceinline__ void take_packet_duo(float* buf, int cap, int x, int c, const Packet& k) {
    const int q = c >> 1;
    float *ab = buf + duo_ab(cap, q) + 4 * x, *ef = buf + duo_ef(cap, q) + 4 * x;
    const float v0 = __uint_as_float((unsigned)k.lo), v1 = __uint_as_float((unsigned)(k.lo >> 32)),
                v2 = __uint_as_float((unsigned)k.hi);
    if (c & 1) {
        ab[3] = v0;
        ef[0] = v1;
        ef[1] = v2;
    } else {
        ab[0] = v0;
        ab[1] = v1;
        ab[2] = v2;
    }
}

// One chunk of the next lattice step's stream-collide (FarArgs, FP32
// storage) on the lattice warps: row y = c / n_seg, nodes [64 seg,
// 64 seg + 64), two per lane.  The pull and BGK arithmetic of a node is that
// of k_stream_collide (the same pulled values through bgk_dev; edge nodes
// through pull_edge), so the results are the same bits.  Every lane of the
// warp takes part in the loads and shuffles; only lanes whose nodes lie
// outside the rectangle store.  (Staging the rows in shared memory with
// cp.async, two chunks per warp, measured slower: the FV tile leaves about
// 50 KB of shared memory, too little to keep more loads in flight.)
__device__ __forceinline__ void far_chunk(const Dev<float>& d, const FarArgs<float>& far, int c, int lane) {
    const int y = c / far.n_seg, seg = c - y * far.n_seg;
    const int x0 = 64 * seg + 2 * lane;
    const bool rows_out = y < far.ey0 || y >= far.ey1;
    if (!rows_out && 64 * seg >= far.ex0 && 64 * seg + 64 <= far.ex1) return;  // the whole chunk inside
    const bool mine = x0 < d.nx && (rows_out || x0 < far.ex0 || x0 >= far.ex1);
    const bool interior = x0 >= 1 && x0 + 2 <= d.nx - 1 && y >= 1 && y <= d.ny - 2;
    const float* __restrict__ A = far.src;
    float* __restrict__ B = far.dst;
    const float omega = 1.0f / d.tau_s;
    float2 p[9];
    float edge[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        int sy = y - cy_of(i);
        sy = sy < 0 ? 0 : (sy >= d.ny ? d.ny - 1 : sy);
        const int64_t row = i * d.plane + (int64_t)sy * d.pitch;
        const int xv = x0 < d.pitch ? x0 : d.pitch - 2;
        p[i] = *reinterpret_cast<const float2*>(A + row + xv);
        if (cx_of(i) == 1) {
            edge[i] = __shfl_up_sync(0xffffffffu, p[i].y, 1);
            if (lane == 0) edge[i] = A[row + (xv > 0 ? xv - 1 : 0)];
        } else if (cx_of(i) == -1) {
            edge[i] = __shfl_down_sync(0xffffffffu, p[i].x, 1);
            if (lane == 31) edge[i] = A[row + (xv + 2 < d.pitch ? xv + 2 : d.pitch - 1)];
        }
    }
    if (!mine) return;
    if (interior) {
        float f[9], o0[9], o1[9];
#pragma unroll
        for (int i = 0; i < 9; ++i) f[i] = cx_of(i) == 0 ? p[i].x : (cx_of(i) == 1 ? edge[i] : p[i].y);
        bgk_dev(f, d.rho0, omega, o0);
#pragma unroll
        for (int i = 0; i < 9; ++i) f[i] = cx_of(i) == 0 ? p[i].y : (cx_of(i) == 1 ? p[i].x : edge[i]);
        bgk_dev(f, d.rho0, omega, o1);
        const int64_t s0 = (int64_t)y * d.pitch + x0;
#pragma unroll
        for (int i = 0; i < 9; ++i) *reinterpret_cast<float2*>(B + i * d.plane + s0) = make_float2(o0[i], o1[i]);
    } else {
        for (int k = 0; k < 2; ++k) {
            const int x = x0 + k;
            if (x >= d.nx) break;
            float g[9], o[9];
#pragma unroll
            for (int i = 0; i < 9; ++i) g[i] = pull_edge<float, float>(d, A, x, y, i);
            bgk_dev(g, d.rho0, omega, o);
#pragma unroll
            for (int i = 0; i < 9; ++i) B[i * d.plane + (int64_t)y * d.pitch + x] = o[i];
        }
    }
}

// lattice warps: chunks of the next step's stream-collide until none is left
__device__ __forceinline__ void far_chunks(const Dev<float>& d, const FarArgs<float>& far) {
    const int lane = threadIdx.x & 31;
    for (; far.n_chunks > 0;) {
        int c = 0;
        if (lane == 0) c = (int)atomicAdd(far.next, 1u);
        c = __shfl_sync(0xffffffffu, c, 0);
        if (c >= far.n_chunks) break;
        far_chunk(d, far, c, lane);
    }
}

// the FV warps' barrier (named barrier 1; the lattice warps never join it)
template <int N>
__device__ __forceinline__ void fv_bar() {
    asm volatile("bar.sync 1, %0;" ::"n"(N) : "memory");
}

// the same, and whether any of them calls it with bad
template <int N>
__device__ __forceinline__ bool fv_bar_or(bool bad) {
    int r;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\tsetp.ne.s32 p, %1, 0;\n\tbar.red.or.pred q, 1, %2, p;\n\tselp.s32 %0, 1, 0, q;\n\t}"
        : "=r"(r)
        : "r"((int)bad), "n"(N)
        : "memory");
    return r != 0;
}
// a barrier of the last n FV threads (named barrier 2)
__device__ __forceinline__ void late_bar(int n) { asm volatile("bar.sync 2, %0;" ::"r"(n) : "memory"); }

// Receives the ghost records of one exchange into the ghost slots of buffer
// cur: thread k of N (counted from the last FV thread, whose warps have the
// fewest nodes) takes packets k, k + N, ...  Each is polled until its tag is
// the exchange's, a bounded number of times; false when a wait ran out or
// another tile gave up.
template <typename T, bool kDuo>
__device__ __forceinline__ bool deep_receive(const Dev<T>& d, const unsigned char* xb, const int32_t* gid, T* cur,
                                             int n_own, int n_slot, unsigned tag, int k, int N) {
    constexpr int PK = kPkts<T>;
    const int np = (n_slot - n_own) * PK;
    bool ok = true;
    for (int p = k; p < np && ok; p += N) {
        const int g = p / PK, c = p - g * PK;
        const int sl = n_own + g;
        const unsigned char* src = xb + ((int64_t)gid[sl] * PK + c) * 16;
        Packet v = ld_packet(src);
        long spins = 0;
        while (packet_tag(v) != tag) {
            if ((spins & 63) == 63 && *(volatile unsigned*)d.abort_flag) {
                ok = false;
                break;
            }
            if (++spins > d.spin_limit) {
                atomicOr(d.status, HLBM_ST_SYNC_TIMEOUT);
                atomicExch(d.abort_flag, 1u);
                ok = false;
                break;
            }
            v = ld_packet(src);
        }
        if constexpr (kDuo)
            take_packet_duo(cur, d.deep_slot_cap, sl, c, v);
        else
            take_packet(cur + (size_t)kSR * sl, c, v);
    }
    return ok;
}

// The FV sub-steps of tile `tile` of the solver d (one block); k_fv_deep runs
// one solver, k_fv_deep_pack several.  kRecord: also writes what the reverse
// mode needs of every sub-step (Dev::fv_rec).
// kDuo (FP32): two lanes per node, no tensor memory, no lattice warps.
template <typename T, bool kRecord, bool kOuterFv, bool kDuo, bool kFar>
__device__ __forceinline__ void fv_deep_body(const Dev<T>& d, const StepArgs& a, T* g0, T* g1, const FarArgs<T>& far,
                                             const int tile, unsigned char* sm, int& abort_sh,
                                             uint32_t& tmem_base_sh) {
    constexpr int NT = kDuo ? kDuoThreads : kDeepFv<T>, BT = kDuo ? kDuoThreads : kDeepThreads<T, kFar>;
    constexpr int G = kDeepGroups<T>, SW = kDeepSlotWords<T>;
    const int tid = threadIdx.x, warp = tid >> 5;
    const int s0 = d.deep_ptr[tile];
    const int32_t* cnt = d.deep_cnt + kDeepCnt * tile;
    const int n_a = cnt[0], n_own = cnt[1], n_slot = cnt[2];
    const int K = d.deep_k;
    const bool quads = sizeof(T) == 8 && !kOuterFv && d.deep_quads > 0;
    const DeepSmem L =
        deep_smem_layout<T>(d.deep_slot_cap, d.n_sub, d.deep_ocap, quads ? d.deep_quads : 0, kOuterFv ? d.deep_ocap : 0);
    T* buf0 = reinterpret_cast<T*>(sm + L.buf0);
    T* buf1 = reinterpret_cast<T*>(sm + L.buf1);
    T* uv = reinterpret_cast<T*>(sm + L.uv);
    int32_t* gid = reinterpret_cast<int32_t*>(sm + L.gid);
    int8_t* kd = reinterpret_cast<int8_t*>(sm + L.kind);
    int8_t* sd = reinterpret_cast<int8_t*>(sm + L.send);
    int16_t* om = reinterpret_cast<int16_t*>(sm + L.omap);
    // ---- tensor memory: all 512 columns; warp w reads lanes 32 (w % 4) ..
    // and, for its slot group j, the columns SW (j NT / 128 + w / 4) ..
    uint32_t tbase = 0;
    if constexpr (!kDuo) {
        if (warp == 0) tmem_alloc_512(&tmem_base_sh);
        tmem_fence_before();
        __syncthreads();
        tmem_fence_after();
        tbase = tmem_base_sh;
    }
    auto tslot_of = [&](int j) {
        return tbase + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)(SW * (j * (NT / 128) + (warp >> 2)));
    };
    // ---- set-up: wall velocity per sub-step, slot tables, records of every
    // slot at sub-step 0, the outer nodes' feed, the row images
    [[maybe_unused]] DuoRow R;
    [[maybe_unused]] Duo Q2;
    if constexpr (kDuo) {
        Q2.q = tid & 1;
        const float w = Q2.q ? -w_of<float>(5) : -w_of<float>(1), dt = d.dt_u, iv = d.inv_tau_u;
        Q2.w = pk(w, w);
        Q2.dt1 = pk(dt, Q2.q ? -dt : dt);
        Q2.iv1 = pk(-iv, Q2.q ? iv : -iv);
        Q2.dt2 = pk(-dt, Q2.q ? dt : -dt);
        Q2.iv2 = pk(iv, Q2.q ? -iv : iv);
    }
    for (int m = tid; m < d.n_sub; m += BT) wall_velocity(d, a, m, uv[m], uv[d.n_sub + m]);
    for (int x = tid; x < n_slot; x += BT) {
        const int g = d.deep_gid[s0 + x];
        gid[x] = g;
        kd[x] = d.kind[g];
        sd[x] = d.deep_send[s0 + x];
        om[x] = -1;
        const T* r = g0 + (int64_t)kRec * g;
        T* o = buf0 + (size_t)kSR * x;
        const Vec4<T> v0 = ld4(r), v1 = ld4(r + 4), v2 = ld4(r + 8);
        T *o1 = o + 4, *o2 = o + 8;
        if constexpr (kDuo) {
            o = buf0 + 4 * x;
            o1 = o + 4 * d.deep_slot_cap;
            o2 = o1 + 4 * d.deep_slot_cap;
        }
        st4(o, v0.y, v0.z, v0.w, v1.x);
        st4(o1, v1.y, v1.z, v1.w, v2.x);
        st4(o2, v0.x, v2.y, v2.z, v2.w);
    }
    __syncthreads();
    {
        const int o0 = d.deep_optr[tile], on = d.deep_optr[tile + 1] - o0;
        T* osn = reinterpret_cast<T*>(sm + L.osnap);
        for (int q = tid; q < on; q += BT) om[d.deep_oslot[o0 + q]] = (int16_t)q;
        const int64_t no = d.n_outer;
        for (int x = tid; x < kSnap * on; x += BT) {
            const int q = x / kSnap, j = x - kSnap * q;
            osn[x] = d.snap[j * no + d.outer_of[gid[d.deep_oslot[o0 + q]]]];
        }
        // row images of the computed slots (lanes without one store zeros;
        // FV warps only)
        const int n_comp = cnt[3];
        const uint4* rows = reinterpret_cast<const uint4*>(d.deep_rows) + (int64_t)(SW / 4) * d.deep_rptr[tile];
        if constexpr (sizeof(T) == 8) {
            // quads: rows into shared memory, an entry per thread
            const uint32_t* img = d.deep_rows + (int64_t)SW * d.deep_rptr[tile];
            for (int x = tid; x < 8 * n_comp && quads; x += BT) {
                const int sl = x >> 3, j = (x & 7) - 1;
                QuadRow& R = reinterpret_cast<QuadRow*>(sm + L.rows)[sl];
                const uint32_t* w = img + (int64_t)SW * sl + kDeepEntryWords<T> * (j + 1);
                if (j < 0) {
                    R.cP = from_words<double>(w[0], w[1]);
                    R.ne = (int)w[2];
                } else {
                    const double gx = from_words<double>(w[0], w[1]), gy = from_words<double>(w[2], w[3]);
                    QuadEntry& E = R.e[j];
                    E.k[0] = gx;
                    E.k[1] = gy;
                    E.k[2] = __dadd_rn(gx, gy);
                    E.k[3] = __dsub_rn(gx, gy);
                    E.c = from_words<double>(w[4], w[5]);
                    E.col = (int)w[6];
                }
            }
        }
        if constexpr (kDuo) {
            // pairs of lanes: this lane's share of its row, in registers
            const int x = tid >> 1;
            const bool have = x < n_comp;
            const uint4 h = have ? rows[(int64_t)(SW / 4) * x] : make_uint4(0u, 0u, 0u, 0u);
            R.cP = __uint_as_float(h.x);
#pragma unroll
            for (int j = 0; j < kTmemMaxEntries; ++j) {
                const bool in_row = have && j < (int)h.y;
                const uint4 u = in_row ? rows[(int64_t)(SW / 4) * x + 1 + j] : make_uint4(0u, 0u, 0u, 0u);
                const float gx = __uint_as_float(u.x), gy = __uint_as_float(u.y);
                R.k[j] = Q2.q ? pk(add_rn(gx, gy), sub_rn(gx, gy)) : pk(gx, gy);
                R.c[j] = __uint_as_float(u.z);
                R.col[j] = 4 * (in_row ? (int)u.w : (have ? x : 0));
            }
        }
#pragma unroll 1
        for (int j = 0; j < G && tid < NT && !quads && !kDuo; ++j) {
            const int x = j * NT + tid;
            const bool have = x < n_comp;
            const uint32_t ts = tslot_of(j);
#pragma unroll 1
            for (int w4 = 0; w4 < SW / 4; ++w4) {
                uint4 u = make_uint4(0u, 0u, 0u, 0u);
                if (have) u = rows[(int64_t)(SW / 4) * x + w4];
                tmem_st4(ts + 4 * w4, u.x, u.y, u.z, u.w);
            }
        }
        if constexpr (!kDuo) tmem_wait_st();
    }
    // interpolated records of the outer slots for sub-step m (outer_fv), thread k of n
    const int n_star = kOuterFv ? d.deep_optr[tile + 1] - d.deep_optr[tile] : 0;
    auto star_at = [&](int m) { return reinterpret_cast<T*>(sm + L.star) + (m & 1) * (size_t)kSR * d.deep_ocap; };
    auto make_stars = [&](int m, int k, int n) {
        for (int q = k; q < n_star; q += n) {
            const Pops<T> f = fv_outer_from(d, reinterpret_cast<const T*>(sm + L.osnap) + kSnap * q, 1, m);
            T z[3], ux, uy;
            z_of(f, d.rho0, z, ux, uy);
            if constexpr (kDuo)
                duo_put(star_at(m), d.deep_ocap, q, rec_of(f, z));
            else
                st_rec(star_at(m) + (size_t)kSR * q, rec_of(f, z));
        }
    };
    if constexpr (kOuterFv) {
        __syncthreads();  // the staged feed
        make_stars(0, tid, BT);
    }
    if (tid == 0) abort_sh = 0;
    if constexpr (!kDuo) tmem_fence_before();
    __syncthreads();
    if constexpr (!kDuo) tmem_fence_after();
    const unsigned long long base = (unsigned long long)a.t * (unsigned long long)d.n_sub;
    if (tid < NT) {
        const int nb0 = d.tile_nb_ptr[tile], nb1 = d.tile_nb_ptr[tile + 1];
        const int64_t xhalf = (int64_t)d.n * kPkts<T> * 16;
        // own nodes that read only own nodes, updated while the ghosts are on
        // their way (0 where that does not pay: fv_deep_early)
        const int n_early = quads || kDuo ? 0 : n_a;
        // first thread of the warps that have slots left after the early part
        // (they lie in the second group: n_a fills the first)
        constexpr bool kSplit = !kDuo && sizeof(T) == 4;
        const int late0 = kSplit && n_early > 0 ? min(NT - 32, (n_early - NT) / 32 * 32) : 0;
        Quad Q;
        Q.q = tid & 3;
        Q.w = w_of<double>(Q.q < 2 ? 1 : 5);
        Q.sgn = (Q.q & 1) ? 1.0 : -1.0;
        int m = 0;
        bool aborted = false;
        for (int b = 0; m < d.n_sub && !aborted; ++b) {
            const int kb = min(K, d.n_sub - m);
            const bool final_block = (m + kb == d.n_sub);
            // block b receives exchange b (b > 0) and sends exchange b + 1
            unsigned char* xout = d.deep_x + ((b + 1) & 1) * xhalf;
            const unsigned tag_out = a.xtag + (unsigned)(b + 1);
            for (int s = 0; s < kb; ++s, ++m) {
                T* cur = (m & 1) ? buf1 : buf0;
                T* nxt = (m & 1) ? buf0 : buf1;
                const bool send = (s == kb - 1) && !final_block && tile != d.stall_tile;
                const int cs = cnt[3 + s];
                int lo = 0;
                bool ok = true;
                // the next sub-step's interpolated records (from the last FV thread down)
                if (kOuterFv && m + 1 < d.n_sub) make_stars(m + 1, NT - 1 - tid, NT);
                if (s == 0 && b > 0) {
#pragma unroll
                    for (int j = 0; j < G && !kDuo; ++j) {
                        const int x = j * NT + tid;
                        const bool v = x < n_early;
                        if constexpr (!kDuo) {
                            if (__any_sync(0xffffffffu, v))
                                deep_node<T, kRecord, kOuterFv>(d, sm, L, cur, nxt, tslot_of(j), v, x, m, nullptr, 0u,
                                                                true, star_at(m));
                        }
                    }
                    // FP32, after an early part: the warps with slots left receive and go
                    // on while the others still update, with a barrier of their own
                    if (tid >= late0) {
                        const int nr = kSplit ? NT - late0 : NT;
                        ok = deep_receive<T, kDuo>(d, d.deep_x + (b & 1) * xhalf, gid, cur, n_own, n_slot,
                                                   a.xtag + (unsigned)b, NT - 1 - tid, nr);
                        // tiles that read this one but are not read by it: their reads of
                        // the packets about to be overwritten are behind their counter
                        for (int e = nb0 + tid - late0; e < nb1 && ok; e += nr) {
                            const unsigned long long* pc = d.progress + d.tile_nb[e];
                            long spins = 0;
                            while (ld_acquire(pc) < base + m) {
                                if (*(volatile unsigned*)d.abort_flag) {
                                    ok = false;
                                    break;
                                }
                                if (++spins > d.spin_limit) {
                                    atomicOr(d.status, HLBM_ST_SYNC_TIMEOUT);
                                    atomicExch(d.abort_flag, 1u);
                                    ok = false;
                                    break;
                                }
                            }
                        }
                        if constexpr (kSplit) {
                            late_bar(nr);
                        } else {
                            if (!ok) abort_sh = 1;
                            fv_bar<NT>();
                            if (abort_sh) {
                                aborted = true;
                                break;
                            }
                        }
                    }
                    // a block of one sub-step ends here: the nodes updated early are sent
                    // only after the receive (which frees the packets they overwrite)
                    if (send && n_early > 0) {
                        bool bad = false;
                        if constexpr (kSplit) bad = fv_bar_or<NT>(!ok);
                        for (int x = tid; x < n_early && !bad; x += NT)
                            if (sd[x])
                                send_record(xout + (int64_t)gid[x] * kPkts<T> * 16, ld_rec(nxt + (size_t)kSR * x), tag_out);
                    }
                    lo = n_early;
                }
                if constexpr (sizeof(T) == 8) {
                    for (int x0 = 8 * warp; x0 < cs && quads; x0 += NT / 4) {
                        const int x = x0 + ((tid & 31) >> 2);
                        const bool v = x < cs;
                        quad_node<kRecord>(
                            d, sm, L, cur, nxt, Q, v, x, m,
                            send && v && x < n_own && sd[x] ? xout + (int64_t)gid[x] * kPkts<T> * 16 : nullptr, tag_out,
                            x < n_own);
                    }
                }
                if constexpr (kDuo) {
                    const int x = tid >> 1;
                    const bool v = x < cs;
                    if (__any_sync(0xffffffffu, v))
                        duo_node<kRecord, kOuterFv>(
                            d, sm, L, cur, nxt, Q2, R, v, x, m,
                            send && v && x < n_own && sd[x] ? xout + (int64_t)gid[x] * kPkts<T> * 16 : nullptr, tag_out,
                            x < n_own, star_at(m));
                }
#pragma unroll
                for (int j = 0; j < G && !quads && !kDuo; ++j) {
                    const int x = j * NT + tid;
                    const bool v = x >= lo && x < cs;
                    if constexpr (!kDuo) {
                        if (__any_sync(0xffffffffu, v))
                            deep_node<T, kRecord, kOuterFv>(
                                d, sm, L, cur, nxt, tslot_of(j), v, x, m,
                                send && v && x < n_own && sd[x] ? xout + (int64_t)gid[x] * kPkts<T> * 16 : nullptr, tag_out,
                                x < n_own, star_at(m));
                    }
                }
                if (kSplit && s == 0 && b > 0) {
                    aborted = fv_bar_or<NT>(!ok);  // a wait ran out: the sub-step's results are dropped
                    if (aborted) break;
                } else {
                    fv_bar<NT>();
                }
            }
            if (!aborted && !final_block && d.deep_pub[tile] && tid == NT - 1 && tile != d.stall_tile)
                st_release(d.progress + tile, base + m);
        }
        // the state after the last completed sub-step, in index order
        const T* fin = (m & 1) ? buf1 : buf0;
        for (int x = tid; x < n_own; x += NT) {
            const T *r = fin + (size_t)kSR * x, *r1 = r + 4, *r2 = r + 8;
            if constexpr (kDuo) {
                r = fin + 4 * x;
                r1 = r + 4 * d.deep_slot_cap;
                r2 = r1 + 4 * d.deep_slot_cap;
            }
            T* o = g1 + (int64_t)kRec * gid[x];
            const Vec4<T> v0 = ld4(r), v1 = ld4(r1), v2 = ld4(r2);
            st4(o, v2.x, v0.x, v0.y, v0.z);
            st4(o + 4, v0.w, v1.x, v1.y, v1.z);
            st4(o + 8, v1.w, v2.y, v2.z, v2.w);
        }
    } else if constexpr (kFar) {
        far_chunks(d, far);
    }
    // ---- release TMEM (also after an abort: every warp is past its last tcgen05.ld)
    if constexpr (!kDuo) {
        tmem_fence_before();
        __syncthreads();
        tmem_fence_after();
        if (warp == 0) tmem_dealloc_512(tbase);
    }
}

template <typename T, bool kRecord, bool kOuterFv, bool kFar>
__global__ void __launch_bounds__(kDeepThreads<T, kFar>, 1) k_fv_deep(Dev<T> d, StepArgs a, T* g0, T* g1, FarArgs<T> far) {
    extern __shared__ __align__(16) unsigned char sm[];
    __shared__ int abort_sh;
    __shared__ uint32_t tmem_base_sh;
    fv_deep_body<T, kRecord, kOuterFv, false, kFar>(d, a, g0, g1, far, blockIdx.x, sm, abort_sh, tmem_base_sh);
}

// Several solvers' FV sub-steps in one cooperative launch: block b runs tile
// b - block0 of the item whose range [block0, next block0) holds b.  Each item
// keeps its own tables, packets, tags, sub-step count and buffers; items only
// share the GPU.
template <typename T>
__global__ void __launch_bounds__(kDeepThreads<T, false>, 1) k_fv_deep_pack(const __grid_constant__ FvPack<T> pk) {
    extern __shared__ __align__(16) unsigned char sm[];
    __shared__ int abort_sh;
    __shared__ uint32_t tmem_base_sh;
    int i = 0;
    while (i + 1 < pk.n && pk.block0[i + 1] <= (int)blockIdx.x) ++i;
    fv_deep_body<T, false, false, false, false>(pk.d[i], pk.a[i], pk.g0[i], pk.g1[i], FarArgs<T>{}, (int)blockIdx.x - pk.block0[i], sm,
                                                abort_sh, tmem_base_sh);
}

// FP32 patches whose tiles' computed slots fit pairs of lanes.  Blocks past
// the tiles run the next step's stream-collide away from the patch (FarArgs) on
// all their warps.
template <bool kRecord, bool kOuterFv>
__global__ void __launch_bounds__(kDuoThreads, 1) k_fv_duo(Dev<float> d, StepArgs a, float* g0, float* g1,
                                                           FarArgs<float> far) {
    extern __shared__ __align__(16) unsigned char sm[];
    __shared__ int abort_sh;
    uint32_t none = 0;
    if ((int)blockIdx.x >= d.n_tiles)
        far_chunks(d, far);
    else
        fv_deep_body<float, kRecord, kOuterFv, true, false>(d, a, g0, g1, far, blockIdx.x, sm, abort_sh, none);
}
__global__ void __launch_bounds__(kDuoThreads, 1) k_fv_duo_pack(const __grid_constant__ FvPack<float> pk) {
    extern __shared__ __align__(16) unsigned char sm[];
    __shared__ int abort_sh;
    uint32_t none = 0;
    int i = 0;
    while (i + 1 < pk.n && pk.block0[i + 1] <= (int)blockIdx.x) ++i;
    fv_deep_body<float, false, false, true, false>(pk.d[i], pk.a[i], pk.g0[i], pk.g1[i], FarArgs<float>{},
                                            (int)blockIdx.x - pk.block0[i], sm, abort_sh, none);
}

template <typename T>
cudaError_t launch_fv_deep_pack(const FvPack<T>& pk, int blocks, size_t smem, cudaStream_t s) {
    FvPack<T> p = pk;
    void* args[] = {&p};
    const void* fn = (const void*)k_fv_deep_pack<T>;
    int threads = kDeepThreads<T, false>;
    if constexpr (sizeof(T) == 4) {
        bool duo = true;
        for (int k = 0; k < pk.n; ++k) duo = duo && pk.d[k].deep_duo;
        if (duo) {
            fn = (const void*)k_fv_duo_pack;
            threads = kDuoThreads;
        }
    }
    return cudaLaunchCooperativeKernel(fn, dim3(blocks), dim3(threads), args, smem, s);
}
template <typename T>
int fv_deep_cap(int n) {
    return sizeof(T) == 4 ? duo_cap(n) : n;
}
template <typename T>
int fv_deep_duo_slots() {
    return sizeof(T) == 4 ? kDuoSlots : 0;
}

template <typename T>
int fv_deep_tile_capacity(size_t smem) {
    if (smem == 0) return 0;
    int dev = 0, sms = 0, per = 0, maxsm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaDeviceGetAttribute(&maxsm, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    // each block allocates all 512 TMEM columns: only one block per SM
    std::vector<std::pair<const void*, int>> fns;
    for (const void* fn : {(const void*)k_fv_deep<T, false, false, false>, (const void*)k_fv_deep<T, true, false, false>,
                           (const void*)k_fv_deep<T, false, true, false>, (const void*)k_fv_deep_pack<T>})
        fns.push_back({fn, kDeepThreads<T, false>});
    if constexpr (sizeof(T) == 4)
        for (const void* fn : {(const void*)k_fv_deep<T, false, false, true>, (const void*)k_fv_deep<T, false, true, true>})
            fns.push_back({fn, kDeepThreads<T, true>});
    if constexpr (sizeof(T) == 4)
        for (const void* fn : {(const void*)k_fv_duo<false, false>, (const void*)k_fv_duo<true, false>,
                               (const void*)k_fv_duo<false, true>, (const void*)k_fv_duo_pack})
            fns.push_back({fn, kDuoThreads});
    for (const auto& [fn, threads] : fns) {
        cudaFuncAttributes fa{};
        if (cudaFuncGetAttributes(&fa, fn) != cudaSuccess) {
            cudaGetLastError();
            return 0;
        }
        const int limit = maxsm - (int)fa.sharedSizeBytes;
        if (smem > (size_t)limit) return 0;
        if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, limit) != cudaSuccess) {
            cudaGetLastError();
            return 0;
        }
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, fn, threads, smem);
        if (per != 1) return 0;
    }
    return sms;
}

template <typename T>
cudaError_t launch_fv_deep(const Dev<T>& d, const StepArgs& a, const FarArgs<T>* far, cudaStream_t s) {
    Dev<T> dd = d;
    StepArgs aa = a;
    T* b0 = (T*)d.fu_in;
    T* b1 = d.fu_out;
    FarArgs<T> fa{};
    if (far && sizeof(T) == 4) fa = *far;
    void* args[] = {&dd, &aa, &b0, &b1, &fa};
    const size_t smem = fv_deep_smem_bytes<T>(d.deep_slot_cap, d.n_sub, d.deep_ocap, d.deep_quads,
                                               d.outer_fv ? d.deep_ocap : 0);
    const void* fn = d.outer_fv ? (const void*)k_fv_deep<T, false, true, false>
                     : d.fv_rec ? (const void*)k_fv_deep<T, true, false, false>
                                : (const void*)k_fv_deep<T, false, false, false>;
    int threads = kDeepThreads<T, false>, blocks = d.n_tiles;
    if constexpr (sizeof(T) == 4) {
        if (fa.n_chunks > 0 && !d.fv_rec) {
            fn = d.outer_fv ? (const void*)k_fv_deep<T, false, true, true> : (const void*)k_fv_deep<T, false, false, true>;
            threads = kDeepThreads<T, true>;
        }
        if (d.deep_duo) {
            fn = d.outer_fv ? (const void*)k_fv_duo<false, true>
                 : d.fv_rec ? (const void*)k_fv_duo<true, false>
                            : (const void*)k_fv_duo<false, false>;
            threads = kDuoThreads;
            if (fa.n_chunks > 0) blocks += fa.blocks;  // on SMs without a tile
        }
    }
    return cudaLaunchCooperativeKernel(fn, dim3(blocks), dim3(threads), args, smem, s);
}

// Row image of computed slot i: header (C_PP, entry count), then the
// off-diagonal entries of row gid[i] in row order with their local columns.
template <typename T>
__global__ void k_build_deep_rows(Dev<T> d, const int32_t* gid, const int32_t* lcol, int64_t count,
                                  uint32_t* rows) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= count) return;
    constexpr int SW = kDeepSlotWords<T>, EW = kDeepEntryWords<T>;
    uint32_t* r = rows + (int64_t)SW * i;
    for (int w = 0; w < SW; ++w) r[w] = 0u;
    const int P = gid[i];
    const int r0 = d.row_ptr[P], ne = d.row_ptr[P + 1] - r0 - 1;
    const T cP = d.coef[r0].c;
    r[0] = lo_word(cP);
    if constexpr (sizeof(T) == 4) {
        r[1] = (uint32_t)ne;
    } else {
        r[1] = hi_word(cP);
        r[2] = (uint32_t)ne;
    }
    for (int j = 0; j < ne && j < kTmemMaxEntries; ++j) {
        const Coef<T> c = d.coef[r0 + 1 + j];
        uint32_t* e = r + EW * (j + 1);
        e[0] = lo_word(c.gx);
        if constexpr (sizeof(T) == 4) {
            e[1] = lo_word(c.gy);
            e[2] = lo_word(c.c);
            e[3] = (uint32_t)lcol[(int64_t)kTmemMaxEntries * i + j];
        } else {
            e[1] = hi_word(c.gx);
            e[2] = lo_word(c.gy);
            e[3] = hi_word(c.gy);
            e[4] = lo_word(c.c);
            e[5] = hi_word(c.c);
            e[6] = (uint32_t)lcol[(int64_t)kTmemMaxEntries * i + j];
        }
    }
}

template <typename T>
void launch_build_deep_rows(const Dev<T>& d, const int32_t* gid, const int32_t* lcol, int64_t count, uint32_t* rows,
                            cudaStream_t s) {
    if (count > 0) k_build_deep_rows<T><<<(unsigned)((count + 127) / 128), 128, 0, s>>>(d, gid, lcol, count, rows);
}

// ELL copy of the FV matrices for the shared-memory kernel: entry i takes
// CSR entry src[i] with tile-local column col[i] (src -1: padding, zero)
template <typename T>
__global__ void k_build_ell(const Coef<T>* coef, const int32_t* src, const int32_t* col, Coef<T>* ell, int64_t count) {
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= count) return;
    Coef<T> c;
    c.col = col[i];
    c.gx = c.gy = c.c = T(0);
    if (src[i] >= 0) {
        const Coef<T> s = coef[src[i]];
        c.gx = s.gx;
        c.gy = s.gy;
        c.c = s.c;
    }
    ell[i] = c;
}

template <typename T>
void launch_build_ell(const Coef<T>* coef, const int32_t* src, const int32_t* col, Coef<T>* ell, int64_t count,
                      cudaStream_t s) {
    k_build_ell<T><<<(unsigned)((count + 255) / 256), 256, 0, s>>>(coef, src, col, ell, count);
}

template <typename T>
int fv_smem_tile_capacity(size_t smem) {
    if (smem == 0) return 0;
    int dev = 0, sms = 0, per = 0, maxsm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaDeviceGetAttribute(&maxsm, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    // the opt-in maximum less the kernel's static shared memory, so that
    // solvers with different tile sizes can all launch; residency follows
    // from the bytes each launch asks for
    int cap = 1 << 30;
    for (const void* fn : {(const void*)k_fv_tiles<T, false>, (const void*)k_fv_tiles<T, true>}) {
        cudaFuncAttributes fa{};
        if (cudaFuncGetAttributes(&fa, fn) != cudaSuccess) {
            cudaGetLastError();
            return 0;
        }
        const int limit = maxsm - (int)fa.sharedSizeBytes;
        if (smem > (size_t)limit) return 0;
        if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, limit) != cudaSuccess) {
            cudaGetLastError();
            return 0;
        }
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, fn, kSmemThreads<T>, smem);
        cap = std::min(cap, sms * per);
    }
    return cap;
}

template <typename T>
cudaError_t launch_fv_smem(const Dev<T>& d, const StepArgs& a, cudaStream_t s) {
    Dev<T> dd = d;
    StepArgs aa = a;
    T* b0 = (T*)d.fu_in;
    T* b1 = d.fu_out;
    void* args[] = {&dd, &aa, &b0, &b1};
    size_t smem = fv_smem_bytes<T>(d.tile_cap, d.halo_cap, d.ell_width - 1, d.n_sub, d.tile_ocap);
    const void* fn = d.outer_fv ? (const void*)k_fv_tiles<T, true> : (const void*)k_fv_tiles<T, false>;
    return cudaLaunchCooperativeKernel(fn, dim3(d.n_tiles), dim3(kSmemThreads<T>), args, smem, s);
}

// ------------------------------------------------------------- force
// Stress at wall nodes, sigma = -(rho - rho0) c_s^2 I - sum_i f^neq_i c_i c_i,
// integrated by the trapezoid rule over the wall segments with the body's
// outward normal (force of the fluid on the lamina, per unit length).
template <typename T>
__device__ void wall_stress(const Dev<T>& d, int P, double s[3]) {
    T f[9];
    load_f(d.fu_in + (int64_t)kRec * P, f);
    T dr, r, ux, uy;
    moments_dev(f, d.rho0, dr, r, ux, uy);
    double pxx = 0, pxy = 0, pyy = 0;
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        double fneq = double(f[i] - feq_dev<T>(i, dr, r, ux, uy));
        pxx += fneq * (cx_of(i) * cx_of(i));
        pxy += fneq * (cx_of(i) * cy_of(i));
        pyy += fneq * (cy_of(i) * cy_of(i));
    }
    double p = double(dr) / 3.0;
    s[0] = -p - pxx;
    s[1] = -pxy;
    s[2] = -p - pyy;
}

template <typename T>
__global__ void __launch_bounds__(128) k_force_segments(Dev<T> d) {
    int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= d.nseg) return;
    double sa[3], sb[3];
    wall_stress(d, d.seg_a[k], sa);
    wall_stress(d, d.seg_b[k], sb);
    double nx = d.seg_n[2 * k], ny = d.seg_n[2 * k + 1];
    d.fcontrib[2 * k] = 0.5 * ((sa[0] + sb[0]) * nx + (sa[1] + sb[1]) * ny);
    d.fcontrib[2 * k + 1] = 0.5 * ((sa[1] + sb[1]) * nx + (sa[2] + sb[2]) * ny);
}

// fixed-order sum of the segment contributions (independent of scheduling)
__global__ void __launch_bounds__(512) k_force_sum(const double* contrib, int nseg, double* force, int64_t t_out,
                                                  unsigned* status) {
    __shared__ double sx[512], sy[512];
    double fx = 0.0, fy = 0.0;
    for (int k = threadIdx.x; k < nseg; k += blockDim.x) {
        fx += contrib[2 * k];
        fy += contrib[2 * k + 1];
    }
    sx[threadIdx.x] = fx;
    sy[threadIdx.x] = fy;
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
        if (threadIdx.x < w) {
            sx[threadIdx.x] += sx[threadIdx.x + w];
            sy[threadIdx.x] += sy[threadIdx.x + w];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        force[2 * t_out] = sx[0];
        force[2 * t_out + 1] = sy[0];
        if (!isfinite(sx[0]) || !isfinite(sy[0])) atomicOr(status, HLBM_ST_NONFINITE);
    }
}

template <typename T>
void launch_force(const Dev<T>& d, int64_t t_out, cudaStream_t s) {
    if (d.nseg > 0) k_force_segments<T><<<(d.nseg + 127) / 128, 128, 0, s>>>(d);
    k_force_sum<<<1, 512, 0, s>>>(d.fcontrib, d.nseg, d.force, t_out, d.status);
}

// ---------------------------------------------------------- readback
template <typename T>
__global__ void k_patch_macro(Dev<T> d, double* rho, double* ux, double* uy, double* f9) {
    int P = blockIdx.x * blockDim.x + threadIdx.x;
    if (P >= d.n) return;
    T f[9];
    load_f(d.fu_in + (int64_t)kRec * P, f);
    T dr, r, vx, vy;
    moments_dev(f, d.rho0, dr, r, vx, vy);
    if (rho) rho[P] = double(d.rho0) + double(dr);
    if (ux) ux[P] = double(vx);
    if (uy) uy[P] = double(vy);
    if (f9) {
#pragma unroll
        for (int i = 0; i < 9; ++i) f9[9 * (int64_t)P + i] = double(f[i]) + double(w_of<T>(i)) * double(d.rho0);
    }
}

template <typename T>
void launch_patch_macro(const Dev<T>& d, double* rho, double* ux, double* uy, double* f9, cudaStream_t s) {
    k_patch_macro<T><<<(d.n + 127) / 128, 128, 0, s>>>(d, rho, ux, uy, f9);
}

// ------------------------------------------- hydrodynamic function fit
// Sums of the normal equations of F_y(t) = a sin(w t) + b cos(w t).
__global__ void __launch_bounds__(512) k_gamma_sums(const double* force, int64_t t0, int64_t t1, double omega,
                                                    double* out) {
    __shared__ double sh[5][512];
    double acc[5] = {0, 0, 0, 0, 0};
    for (int64_t t = t0 + threadIdx.x; t <= t1; t += blockDim.x) {
        double s, c;
        sincos(omega * (double)t, &s, &c);
        double F = force[2 * t + 1];
        acc[0] += s * s;
        acc[1] += s * c;
        acc[2] += c * c;
        acc[3] += F * s;
        acc[4] += F * c;
    }
    for (int j = 0; j < 5; ++j) sh[j][threadIdx.x] = acc[j];
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
        if (threadIdx.x < w)
            for (int j = 0; j < 5; ++j) sh[j][threadIdx.x] += sh[j][threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x < 5) out[threadIdx.x] = sh[threadIdx.x][0];
}

__global__ void __launch_bounds__(512) k_gamma_resid(const double* force, int64_t t0, int64_t t1, double omega,
                                                     double a, double b, double* out) {
    __shared__ double sh[512];
    double acc = 0.0;
    for (int64_t t = t0 + threadIdx.x; t <= t1; t += blockDim.x) {
        double s, c;
        sincos(omega * (double)t, &s, &c);
        double e = force[2 * t + 1] - (a * s + b * c);
        acc += e * e;
    }
    sh[threadIdx.x] = acc;
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
        if (threadIdx.x < w) sh[threadIdx.x] += sh[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) out[0] = sh[0];
}

void launch_gamma_sums(const double* force, int64_t t0, int64_t t1, double omega, double* out, cudaStream_t s) {
    k_gamma_sums<<<1, 512, 0, s>>>(force, t0, t1, omega, out);
}

void launch_gamma_resid(const double* force, int64_t t0, int64_t t1, double omega, double a, double b,
                        double* out, cudaStream_t s) {
    k_gamma_resid<<<1, 512, 0, s>>>(force, t0, t1, omega, a, b, out);
}

// ------------------------------------------------------------ adjoint
template <typename T>
__device__ __forceinline__ void load_d(const T* p, T (&f)[9]) {
#pragma unroll
    for (int i = 0; i < 9; ++i) f[i] = p[i];
}

// sum over the warp, one atomic per warp (every lane of the warp must call)
__device__ __forceinline__ void warp_atomic_add(double* dst, double v) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    if ((threadIdx.x & 31) == 0 && v != 0.0) atomicAdd(dst, v);
}

template <typename R>
__device__ __forceinline__ void atomic_add9(R* dst, const R (&v)[9]) {
#pragma unroll
    for (int i = 0; i < 9; ++i)
        if (v[i] != R(0)) atomicAdd(dst + i, v[i]);
}

// the window node of lattice cell corner q (0..3) for the bilinear stencil
// at (wx, wy), its weight and the weight's derivative in wy; false when the
// corner is outside the window (the forward skipped it)
template <typename T>
__device__ __forceinline__ bool bilinear_corner(const Dev<T>& d, int ox, int oy, double wx, double wy, int q,
                                                int64_t& b, double& w, double& dwy) {
    const double fx0 = floor(wx), fy0 = floor(wy);
    const int ix = (int)fx0, iy = (int)fy0;
    const double ax = __dsub_rn(wx, fx0), ay = __dsub_rn(wy, fy0);
    const double wxq = (q & 1) ? ax : 1.0 - ax, wyq = (q >> 1) ? ay : 1.0 - ay;
    w = wxq * wyq;
    dwy = (q >> 1) ? wxq : -wxq;
    const int bx = ix + (q & 1) - ox, by = iy + (q >> 1) - oy;
    if ((unsigned)bx >= (unsigned)d.bw || (unsigned)by >= (unsigned)d.bh) return false;
    b = (int64_t)by * d.bw + bx;
    return true;
}

// derivatives of the barycentric coordinates of triangle k in q_y
__device__ __forceinline__ void bary_dqy(const double* g, double (&dl)[3]) {  // FP64 geometry
    const double x1 = g[2], x2 = g[4], det = g[6];
    dl[1] = -x2 / det;
    dl[2] = x1 / det;
    dl[0] = -dl[1] - dl[2];
}

// Adjoint of F_y at t+1 (lamF = dJ/dF_y(t+1)) into the patch state that the
// force was computed from (d.fu_in): sigma_xy = -sum f^neq c_x c_y,
// sigma_yy = -dr/3 - sum f^neq c_y^2, F_y = sum_seg (sigma_xy n_x + sigma_yy n_y)
// at the mean of its two nodes.
template <typename T>
__global__ void k_adj_force(Dev<T> d, double lamF, T* lP) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= d.nseg) return;
    const T nx = T(d.seg_n[2 * k]), ny = T(d.seg_n[2 * k + 1]);
    const T lxy = 0.5 * nx * lamF, lyy = 0.5 * ny * lamF;
    for (int e = 0; e < 2; ++e) {
        const int P = e == 0 ? d.seg_a[k] : d.seg_b[k];
        T f[9], dr, rho, ux, uy;
        load_d(d.fu_in + (int64_t)kRec * P, f);
        mom_d(f, T(d.rho0), dr, rho, ux, uy);
        T ln[9], out[9];
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            ln[i] = -(lxy * cx_of(i) * cy_of(i) + lyy * cy_of(i) * cy_of(i));
            out[i] = -lyy / 3.0 + ln[i];
        }
        jfeqT_add(ux, uy, ln, T(-1), out);
        atomic_add9(lP + 9 * (int64_t)P, out);
    }
}

// ---- reverse of the FV sub-steps.  With psi_P the adjoint of node P's update
// (through the wall rule at wall nodes, zero at outer nodes), the adjoint of
// state k before the sub-step is
//   psi_k + sum_P [ dt (c_j . g_Pk) psi_P,j - dt / tau_u C_Pk psi_P,j ]
//         + dt / tau_u (J_feq(k)^T sum_P C_Pk psi_P)_j
// over the rows P that read k.  psi of the sub-step before it is formed from
// that at the node itself, so a sub-step is one pass and one exchange.
// It needs only what the forward sub-step recorded (adj_record): its collision
// sums, velocities and the wall moments; J_feq needs u alone, since its B
// terms carry the rho they are divided by.  Four lanes share a node as in the
// FP64 quads of the forward kernel: lane q holds the pair of opposite
// directions q, f0 rides on lane 0.  Bound by the FP64 issue rate of a warp
// (64 cycles an instruction) in FP64, by the exchange between SMs in FP32.
// Reverse sweep of 48 steps on the 3008-node FP64 patch (n = 50): 404 ms with
// a node per thread on 24 SMs, three grid barriers per sub-step and the sums
// formed again, 62 ms so; 160 steps of the 2588-node FP32 patch (n = 96):
// 664 ms and 94 ms.
template <typename T>
__device__ __forceinline__ ANode<T> adj_node(const Dev<T>& d, const AQuad<T>& Q, int k, bool valid) {
    ANode<T> N;
    N.valid = valid;
    N.k = valid ? k : 0;
    N.kind = valid ? d.kind[N.k] : (int8_t)HLBM_NODE_INTERIOR;
#pragma unroll
    for (int j = 0; j < 6; ++j) N.s0[j] = N.s1[j] = T(0);
#pragma unroll
    for (int j = 0; j < 4; ++j) N.g0[j] = N.g1[j] = T(0);
#pragma unroll
    for (int j = 0; j < 3; ++j) N.kq[j] = T(0);
    if (N.kind == HLBM_NODE_OUTER) {
        const int64_t no = d.n_outer;
        const T* p = d.snap + d.outer_of[N.k];
        const int at[6] = {0, 1, 2, 4 + Q.ia, 4 + Q.ib, 3};
#pragma unroll
        for (int j = 0; j < 6; ++j) {
            N.s0[j] = p[at[j] * no];
            N.s1[j] = p[(12 + at[j]) * no];
        }
    }
    return N;
}
// the outer node's sums into the feed adjoint
template <typename T>
__device__ __forceinline__ void adj_node_out(const Dev<T>& d, const AQuad<T>& Q, const ANode<T>& N, T* lsnap) {
    if (N.kind != HLBM_NODE_OUTER) return;
    const int64_t no = d.n_outer;
    T* p = lsnap + d.outer_of[N.k];
    auto put = [&](int j, T v0, T v1) {
        p[j * no] += v0;
        p[(12 + j) * no] += v1;
    };
    put(4 + Q.ia, N.g0[0], N.g1[0]);
    put(4 + Q.ib, N.g0[1], N.g1[1]);
    if (Q.q == 0) put(3, N.g0[2], N.g1[2]);
    if (Q.q < 3) put(Q.q, N.g0[3], N.g1[3]);
}
template <typename T>
__device__ __forceinline__ ARec<T> adj_rec(const Dev<T>& d, const AQuad<T>& Q, const ANode<T>& N, const T* rec, int m) {
    const T* r = rec + ((int64_t)m * d.n + N.k) * kAdjRec;
    ARec<T> v;
    const bool row = N.kind != HLBM_NODE_OUTER, wall = N.kind == HLBM_NODE_WALL;
    v.na = row ? r[Q.ia] : T(0);
    v.nb = row ? r[Q.ib] : T(0);
    v.n0 = row && Q.q == 0 ? r[kAdjN0] : T(0);
    v.rho = wall ? r[kAdjWall] : T(1);
    v.wx = wall ? r[kAdjWall + 1] : T(0);
    v.wy = wall ? r[kAdjWall + 2] : T(0);
    return v;
}

template <typename T>
__device__ __forceinline__ void adj_put(const AQuad<T>& Q, const ANode<T>& N, T* psi, T pa, T pb, T p0) {
    if (!N.valid) return;
    T* o = psi + kAdjPsi * (int64_t)N.k;
    o[Q.ia] = pa;
    o[Q.ib] = pb;
    if (Q.q == 0) o[kAdjN0] = p0;
}

// psi as packets (see k_fv_deep): one per lane of the quad in FP32 (its pair,
// f0 and the tag), three in FP64 (a value each; the third on lane 0 only)
template <typename T>
constexpr int kAdjPkts = sizeof(T) == 4 ? 1 : 3;
__device__ __forceinline__ void adj_send(unsigned char* p, int, float a, float b, float c, unsigned tag) {
    auto w = [](float v) { return (unsigned long long)__float_as_uint(v); };
    st_packet(p, w(a) | (w(b) << 32), w(c) | ((unsigned long long)tag << 32));
}
__device__ __forceinline__ void adj_send(unsigned char* p, int q, double a, double b, double c, unsigned tag) {
    const unsigned long long t = (unsigned long long)tag << 32;
    st_packet(p, (unsigned long long)__double_as_longlong(a), t);
    st_packet(p + 16, (unsigned long long)__double_as_longlong(b), t);
    if (q == 0) st_packet(p + 32, (unsigned long long)__double_as_longlong(c), t);
}
__device__ __forceinline__ bool adj_recv(const unsigned char* p, int, float& a, float& b, float& c, unsigned tag) {
    const Packet k = ld_packet(p);
    a = __uint_as_float((unsigned)k.lo);
    b = __uint_as_float((unsigned)(k.lo >> 32));
    c = __uint_as_float((unsigned)k.hi);
    return packet_tag(k) == tag;
}
__device__ __forceinline__ bool adj_recv(const unsigned char* p, int q, double& a, double& b, double& c, unsigned tag) {
    const Packet k = ld_packet(p), l = ld_packet(p + 16);
    a = __longlong_as_double((long long)k.lo);
    b = __longlong_as_double((long long)l.lo);
    bool ok = packet_tag(k) == tag && packet_tag(l) == tag;
    c = 0.0;
    if (q == 0) {
        const Packet e = ld_packet(p + 32);
        c = __longlong_as_double((long long)e.lo);
        ok = ok && packet_tag(e) == tag;
    }
    return ok;
}

// kEntries > 0: every quad has at most one node, of at most that many row
// entries, and keeps them, its outer state and its sums in registers over the
// sub-steps; psi travels as tagged packets from node to node, without a
// barrier.  A node overwrites its packets of sub-step m at sub-step m - 2,
// after receiving psi of sub-step m - 1 from every node that reads its own (the
// rows are symmetric), each of which read the packets of sub-step m before
// sending it.  Quads take the nodes in `order` (by kind), so that a warp runs
// the wall rule or the outer rule only where its nodes need it.  Tags (tag0 + the sub-step's distance from the last) grow over
// the solver's life.  0: any patch, with grid barriers.
template <typename T, int kEntries>
__global__ void __launch_bounds__(128) k_adj_fv_rev(Dev<T> d, StepArgs a, const T* rec, const T* P0, const T* lPn, T* x0,
                                                    T* x1, const Coef<T>* tco, T* lsnap, double* par, double* lV,
                                                    T* lPm, int use_tab, unsigned char* px, unsigned tag0,
                                                    const int32_t* order) {
    namespace cg = cooperative_groups;
    cg::grid_group grid = cg::this_grid();
    const int n = d.n, ns = d.n_sub;
    const AQuad<T> Q = aquad<T>();
    const int nq = gridDim.x * blockDim.x / 4, gq = (blockIdx.x * blockDim.x + threadIdx.x) / 4;
    // time fraction and wall velocity of every sub-step (an FP64 cosine and
    // divisions each), when they fit
    extern __shared__ __align__(16) unsigned char sm[];
    T* tab = reinterpret_cast<T*>(sm);
    for (int m = threadIdx.x; m < ns && use_tab; m += blockDim.x) {
        tab[3 * m] = T(m + 1) / T(ns);
        wall_velocity(d, a, m, tab[3 * m + 1], tab[3 * m + 2]);
    }
    __syncthreads();
    auto at_substep = [&](int m, T& th, T& U, T& V) {
        if (use_tab) {
            th = tab[3 * m], U = tab[3 * m + 1], V = tab[3 * m + 2];
        } else {
            th = T(m + 1) / T(ns);
            wall_velocity(d, a, m, U, V);
        }
    };
    // velocity of node k's state before sub-step m
    auto velocity = [&](int k, int m, T& ux, T& uy) {
        if (m > 0) {
            const T* r = rec + ((int64_t)m * n + k) * kAdjRec + kAdjU;
            ux = r[0];
            uy = r[1];
        } else {
            T f[9], dr, rho;
            load_d(P0 + (int64_t)kRec * k, f);
            mom_d(f, T(d.rho0), dr, rho, ux, uy);
        }
    };
    // the adjoint of state m at the node from the row sums
    const T dt = d.dt_u, di = d.dt_u * d.inv_tau_u;
    auto close = [&](T pa, T pb, T p0, T ux, T uy, T Sa, T Sb, T La, T Lb, T L0, T& la, T& lb, T& l0) {
        T fa, fx, fy;
        aq_feq(Q, ux, uy, La, Lb, L0, fa, fx, fy);
        const T g = fa - fx * ux - fy * uy, c = aq_dot(Q, fx, fy);
        la = pa + dt * Q.sgn * Sa - di * La + di * (g + c);
        lb = pb - dt * Q.sgn * Sb - di * Lb + di * (g - c);
        l0 = Q.q == 0 ? p0 - di * L0 + di * g : T(0);
    };
    auto put_out = [&](int k, T la, T lb, T l0) {
        T* o = lPm + 9 * (int64_t)k;
        o[1 + Q.ia] = la;
        o[1 + Q.ib] = lb;
        if (Q.q == 0) o[0] = l0;
    };
    T l_inv = T(0), th, U, V;
    double l_kneq = 0.0;
    auto add_v = [&](int m, T l_v) {
        if (__any_sync(0xffffffffu, l_v != T(0))) warp_atomic_add(lV + (int64_t)a.t * ns + m, double(l_v));
    };
    if constexpr (kEntries > 0) {
        constexpr int E = kEntries;
        ANode<T> N = adj_node(d, Q, gq < n ? order[gq] : 0, gq < n);
        T eg[E], ec[E];
        int ecol[E];
        const int r0 = d.row_ptr[N.k], r1 = d.row_ptr[N.k + 1];
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const bool have = r0 + e < r1;
            const Coef<T> c = tco[have ? r0 + e : r0];
            eg[e] = have ? aq_dot(Q, Q.sgn * c.gx, Q.sgn * c.gy) : T(0);  // lane 3: gx - gy
            ec[e] = have ? c.c : T(0);
            ecol[e] = have ? c.col : N.k;
        }
        // the packets of node g for the sub-step i steps from the last
        auto at = [&](int g, int i) {
            return px + (((int64_t)(i & 1) * n + g) * 4 + Q.q) * (kAdjPkts<T> * 16);
        };
        ARec<T> r = adj_rec(d, Q, N, rec, ns - 1);
        T pa, pb, p0;
        {
            T l_v = T(0);
            at_substep(ns - 1, th, U, V);
            const T* l = lPn + 9 * (int64_t)N.k;
            adj_psi(d, Q, N, r, th, U, V, l[1 + Q.ia], l[1 + Q.ib], Q.q == 0 ? l[0] : T(0), pa, pb, p0, l_inv, l_kneq, l_v);
            if (N.valid) adj_send(at(N.k, 0), Q.q, pa, pb, p0, tag0);
            adj_kneq(N, l_kneq);
            add_v(ns - 1, l_v);
        }
        bool ok = true;
        for (int m = ns - 1; m >= 0 && ok; --m) {
            const int i = ns - 1 - m;
            T ux, uy, l_v = T(0);
            velocity(N.k, m, ux, uy);
            if (m > 0) {
                r = adj_rec(d, Q, N, rec, m - 1);
                at_substep(m - 1, th, U, V);
            }
            T fa[E], fb[E], f0[E], Sa = T(0), Sb = T(0), La = T(0), Lb = T(0), L0 = T(0), la, lb, l0;
            for (long spins = 0; ok; ++spins) {
                bool have = true;
#pragma unroll
                for (int e = 0; e < E; ++e) have = adj_recv(at(ecol[e], i), Q.q, fa[e], fb[e], f0[e], tag0 + i) && have;
                if (__all_sync(0xffffffffu, have || !N.valid)) break;
                if ((spins & 63) == 63) ok = !*(volatile unsigned*)d.abort_flag;
                if (spins > d.spin_limit / E) {  // E packets a turn
                    atomicOr(d.status, HLBM_ST_SYNC_TIMEOUT);
                    atomicExch(d.abort_flag, 1u);
                    ok = false;
                }
                ok = __all_sync(0xffffffffu, ok);
            }
#pragma unroll
            for (int e = 0; e < E; ++e) {
                Sa += eg[e] * fa[e];
                Sb += eg[e] * fb[e];
                La += ec[e] * fa[e];
                Lb += ec[e] * fb[e];
                L0 += ec[e] * f0[e];
            }
            close(pa, pb, p0, ux, uy, Sa, Sb, La, Lb, L0, la, lb, l0);
            if (m > 0) {
                adj_psi(d, Q, N, r, th, U, V, la, lb, l0, pa, pb, p0, l_inv, l_kneq, l_v);
                if (N.valid && ok) adj_send(at(N.k, i + 1), Q.q, pa, pb, p0, tag0 + i + 1);
                adj_kneq(N, l_kneq);
                add_v(m - 1, l_v);
            } else if (N.valid) {
                put_out(N.k, la, lb, l0);
            }
        }
        adj_node_out(d, Q, N, lsnap);
    } else {
        T l_v = T(0);
        at_substep(ns - 1, th, U, V);
        for (int base = 0; base < n; base += nq) {  // the same number of turns on every thread
            ANode<T> N = adj_node(d, Q, base + gq, base + gq < n);
            const T* l = lPn + 9 * (int64_t)N.k;
            T pa, pb, p0;
            adj_psi(d, Q, N, adj_rec(d, Q, N, rec, ns - 1), th, U, V, l[1 + Q.ia], l[1 + Q.ib], Q.q == 0 ? l[0] : T(0), pa,
                    pb, p0, l_inv, l_kneq, l_v);
            adj_put(Q, N, x0, pa, pb, p0);
            adj_kneq(N, l_kneq);
            adj_node_out(d, Q, N, lsnap);
        }
        add_v(ns - 1, l_v);
        for (int m = ns - 1; m >= 0; --m) {
            const T* psi = ((ns - 1 - m) & 1) ? x1 : x0;
            T* nxt = ((ns - 1 - m) & 1) ? x0 : x1;
            l_v = T(0);
            if (m > 0) at_substep(m - 1, th, U, V);
            grid.sync();
            for (int base = 0; base < n; base += nq) {
                ANode<T> N = adj_node(d, Q, base + gq, base + gq < n);
                T Sa = T(0), Sb = T(0), La = T(0), Lb = T(0), L0 = T(0), la, lb, l0, ux, uy;
                const int r0 = d.row_ptr[N.k], r1 = N.valid ? d.row_ptr[N.k + 1] : r0;
#pragma unroll 2
                for (int e = r0; e < r1; ++e) {
                    const Coef<T> c = tco[e];
                    const T* p = psi + kAdjPsi * (int64_t)c.col;
                    const T g = aq_dot(Q, Q.sgn * c.gx, Q.sgn * c.gy);
                    const T pa = p[Q.ia], pb = p[Q.ib];
                    Sa += g * pa;
                    Sb += g * pb;
                    La += c.c * pa;
                    Lb += c.c * pb;
                    L0 += c.c * p[kAdjN0];
                }
                __syncwarp();
                velocity(N.k, m, ux, uy);
                const T* p = psi + kAdjPsi * (int64_t)N.k;
                close(p[Q.ia], p[Q.ib], p[kAdjN0], ux, uy, Sa, Sb, La, Lb, L0, la, lb, l0);
                if (m > 0) {
                    T pa, pb, p0;
                    adj_psi(d, Q, N, adj_rec(d, Q, N, rec, m - 1), th, U, V, la, lb, l0, pa, pb, p0, l_inv, l_kneq, l_v);
                    adj_put(Q, N, nxt, pa, pb, p0);
                    adj_kneq(N, l_kneq);
                    adj_node_out(d, Q, N, lsnap);
                } else if (N.valid) {
                    put_out(N.k, la, lb, l0);
                }
            }
            if (m > 0) add_v(m - 1, l_v);
        }
    }
    warp_atomic_add(par + 1, double(l_inv));
    warp_atomic_add(par + 3, l_kneq);
}

// The transposed rows: entry e of row k (pivot first) holds g and C of row
// col's entry of column k; the pivot's g is minus the sum of the row's own.
template <typename T>
__global__ void k_adj_rows(Dev<T> d, const int32_t* tpos, Coef<T>* tco) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= d.n) return;
    const int r0 = d.row_ptr[k], r1 = d.row_ptr[k + 1];
    Coef<T> pv = d.coef[r0];
    pv.gx = pv.gy = T(0);
    for (int e = r0 + 1; e < r1; ++e) {
        pv.gx -= d.coef[e].gx;
        pv.gy -= d.coef[e].gy;
        Coef<T> c = d.coef[tpos[e]];
        c.col = d.coef[e].col;
        tco[e] = c;
    }
    pv.col = k;
    tco[r0] = pv;
}

// The FV sub-steps of a step from patch state P0 with their records, in
// global memory with grid barriers: for the patches and kernels whose forward
// step does not record.
template <typename T>
__global__ void __launch_bounds__(128) k_adj_fv_record(Dev<T> d, StepArgs a, const T* P0, T* b0, T* b1) {
    namespace cg = cooperative_groups;
    cg::grid_group grid = cg::this_grid();
    const int nth = gridDim.x * blockDim.x, gtid = blockIdx.x * blockDim.x + threadIdx.x;
    for (int m = 0; m < d.n_sub; ++m) {
        const T* in = m == 0 ? P0 : ((m & 1) ? b1 : b0);
        T* out = (m & 1) ? b0 : b1;
        T U, V;
        wall_velocity(d, a, m, U, V);
        for (int P = gtid; P < d.n; P += nth) {
            const int8_t kind = d.kind[P];
            Pops<T> fn, nq{};
            T mo[3] = {};
            if (kind == HLBM_NODE_OUTER) {
                fn = fv_outer_from(d, d.snap + d.outer_of[P], (int64_t)d.n_outer, m);
            } else {
                auto get = [&](int g) {
                    const T* r = in + (int64_t)kRec * g;
                    return RecP<T>{pk(r[1], r[2]), pk(r[3], r[4]), pk(r[5], r[6]),
                                   pk(r[7], r[8]), pk(r[0], r[9]), pk(r[10], r[11])};
                };
                const RecP<T> own = get(P);
                const Pops<T> Q{own.A, own.B, own.C, own.D, px(own.E)};
                FvSums<T> acc;
                fv_sums_init(acc);
                const int r0 = d.row_ptr[P], r1 = d.row_ptr[P + 1];
                for (int e = r0 + 1; e < r1; ++e) {
                    const Coef<T> c = d.coef[e];
                    fv_sums_entry(acc, c.gx, c.gy, c.c, get(c.col), Q);
                }
                fn = fv_sums_finish(d, acc, d.coef[r0].c, own, nq);
                if (kind == HLBM_NODE_WALL) fv_wall(d, U, V, fn, mo);
            }
            T z[3], ux, uy;
            z_of(fn, d.rho0, z, ux, uy);
            adj_record(d, m, P, kind != HLBM_NODE_OUTER, nq, kind == HLBM_NODE_WALL, mo, ux, uy);
            T f[9];
            pops_to(fn, f);
            T* r = out + (int64_t)kRec * P;
#pragma unroll
            for (int i = 0; i < 9; ++i) r[i] = f[i];
#pragma unroll
            for (int j = 0; j < 3; ++j) r[9 + j] = z[j];
        }
        grid.sync();
    }
}

// Reverse of the outer nodes' feed: snap[0] bilinear from the window state
// at t (previous window), snap[1] from the one at t+1; positions at y(t).
template <typename T>
__global__ void k_adj_feed(Dev<T> d, StepArgs a, const T* lsnap, T* lSo, T* lSn, double* lY) {
    const int o = blockIdx.x * blockDim.x + threadIdx.x;
    double gy = 0.0;
    if (o < d.n_outer) {
        const int P = d.outer[o];
        const double wx = __dadd_rn(a.cx, d.xy[2 * P]), wy = __dadd_rn(a.cy, d.xy[2 * P + 1]);
        const int64_t no = d.n_outer;
        for (int side = 0; side < 2; ++side) {
            const T* box = side == 0 ? d.sbox_old : (const T*)d.sbox_new;
            const int ox = side == 0 ? a.pbx0 : a.bx0, oy = side == 0 ? a.pby0 : a.by0;
            T* lS = side == 0 ? lSo : lSn;
            T ls[12];
#pragma unroll
            for (int j = 0; j < 12; ++j) ls[j] = lsnap[(12 * side + j) * no + o];
            for (int q = 0; q < 4; ++q) {
                int64_t b;
                double w, dw;
                if (!bilinear_corner(d, ox, oy, wx, wy, q, b, w, dw)) continue;
                T f[9], st[12], out[9];
#pragma unroll
                for (int i = 0; i < 9; ++i) {
                    f[i] = T(box[i * d.bplane + b]);
                    out[i] = 0.0;
                }
                state_d(f, T(d.rho0), st);
                stateT_add(st, T(d.rho0), ls, T(w), out);
#pragma unroll
                for (int i = 0; i < 9; ++i)
                    if (out[i] != 0.0) atomicAdd(lS + i * d.bplane + b, out[i]);
                T dot = 0.0;
#pragma unroll
                for (int j = 0; j < 12; ++j) dot += ls[j] * st[j];
                gy += dw * double(dot);
            }
        }
    }
    warp_atomic_add(lY + a.t, gy);
}

// source element of population i pulled by node (x, y) (the boundary rules
// of the stream-collide: bounce-back walls, zero-gradient outflow, periodic)
template <typename T>
__device__ __forceinline__ int64_t pull_src(const Dev<T>& d, int x, int y, int i) {
    int sx = x - cx_of(i), sy = y - cy_of(i);
    if (sx < 0 || sx >= d.nx) {
        if (d.bc_x == HLBM_BC_PERIODIC)
            sx = (sx + d.nx) % d.nx;
        else if (d.bc_x == HLBM_BC_WALL)
            return opp_of(i) * d.plane + (int64_t)y * d.pitch + x;
        else
            sx = x;
    }
    if (sy < 0 || sy >= d.ny) {
        if (d.bc_y == HLBM_BC_PERIODIC)
            sy = (sy + d.ny) % d.ny;
        else if (d.bc_y == HLBM_BC_WALL)
            return opp_of(i) * d.plane + (int64_t)y * d.pitch + x;
        else
            sy = y;
    }
    return i * d.plane + (int64_t)sy * d.pitch + sx;
}

// Reverse of the stream-collide (pull, BGK with 1/tau_s) at every node it
// wrote (discretization nodes), plus the window state it wrote (lSn).
template <typename T>
__global__ void k_adj_stream(Dev<T> d, StepArgs a, const T* lfB, const T* lSn, T* lfA, double* par) {
    const int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y;
    T l_om = 0;
    bool active = x < d.nx;
    int64_t b = -1;
    if (active) {
        const unsigned rx = (unsigned)(x - a.bx0), ry = (unsigned)(y - a.by0);
        if (rx < (unsigned)d.bw && ry < (unsigned)d.bh) {
            b = (int64_t)ry * d.bw + rx;
            active = d.cls_cur[b] == CLS_DISC;
        }
    }
    if (active) {
        const T* A = d.fA;
        T f[9];
        int64_t src[9];
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            src[i] = pull_src(d, x, y, i);
            f[i] = T(A[src[i]]);
        }
        T dr, rho, ux, uy;
        mom_d(f, T(d.rho0), dr, rho, ux, uy);
        const T om = 1.0 / T(d.tau_s);
        const T k0 = T(1.0 - double(om)), k1 = T(1.0 - double(om) - double(k0));  // 1 - omega
        const int64_t s = (int64_t)y * d.pitch + x;
        T lam[9], mu[9], eq[9];
        feq_all(dr, rho, ux, uy, eq);
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            lam[i] = lfB[i * d.plane + s];
            mu[i] = sizeof(T) == 8 ? k0 * lam[i] : fma_rn(lam[i], k0, lam[i] * k1);
            l_om -= lam[i] * (f[i] - eq[i]);
        }
        jfeqT_add(ux, uy, lam, om, mu);
        if (b >= 0) {
#pragma unroll
            for (int i = 0; i < 9; ++i) mu[i] += lSn[i * d.bplane + b];
        }
#pragma unroll
        for (int i = 0; i < 9; ++i)
            if (mu[i] != 0.0) atomicAdd(lfA + src[i], mu[i]);
    }
    warp_atomic_add(par + 0, l_om);
}

// Reverse of the eq. postcollision2_s fill: the adjoint of the populations
// it wrote goes to the patch state it interpolated (and is consumed).
template <typename T>
__global__ void k_adj_fill(Dev<T> d, StepArgs a, T* lfA, T* lP, double* par, double* lY) {
    const int64_t b = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    double l_k = 0.0, gy = 0.0;
    bool fill = false;
    int x = 0, y = 0;
    if (b < d.bplane) {
        const int8_t c = d.cls_cur[b];
        x = a.bx0 + (int)(b % d.bw);
        y = a.by0 + (int)(b / d.bw);
        if (c == CLS_INTERP) {
            fill = true;
        } else if (c == CLS_DISC && !a.first) {
            const unsigned px = (unsigned)(x - a.pbx0), py = (unsigned)(y - a.pby0);
            const int8_t prev = (px < (unsigned)d.bw && py < (unsigned)d.bh) ? d.cls_prev[(int64_t)py * d.bw + px]
                                                                             : (int8_t)CLS_DISC;
            fill = prev != CLS_DISC;
        }
    }
    if (fill) {
        const int64_t s = (int64_t)y * d.pitch + x;
        T lp[9];
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            lp[i] = lfA[i * d.plane + s];
            lfA[i * d.plane + s] = 0.0;
        }
        double lam[3];
        const double qx = __dsub_rn((double)x, a.cx), qy = __dsub_rn((double)y, a.cy);
        const int k = locate_dev(d, qx, qy, lam);
        if (k >= 0) {
            const T rho0 = T(d.rho0);
            T fv[3][9], sv[3][12], st[12];
#pragma unroll
            for (int j = 0; j < 12; ++j) st[j] = 0.0;
            for (int q = 0; q < 3; ++q) {
                load_d(d.fu_in + (int64_t)kRec * d.tri[3 * k + q], fv[q]);
                state_d(fv[q], rho0, sv[q]);
#pragma unroll
                for (int j = 0; j < 12; ++j) st[j] += T(lam[q]) * sv[q][j];
            }
            T ls[12];
            ffsT(st, rho0, T(d.k178), lp, ls, l_k);
            double dl[3];
            bary_dqy(d.trigeo + 8 * (int64_t)k, dl);
            for (int q = 0; q < 3; ++q) {
                T out[9];
#pragma unroll
                for (int i = 0; i < 9; ++i) out[i] = 0.0;
                stateT_add(sv[q], rho0, ls, T(lam[q]), out);
                atomic_add9(lP + 9 * (int64_t)d.tri[3 * k + q], out);
                T dot = 0.0;
#pragma unroll
                for (int j = 0; j < 12; ++j) dot += ls[j] * sv[q][j];
                gy -= dl[q] * double(dot);  // q_y = y - c_y
            }
        }
    }
    warp_atomic_add(par + 2, l_k);
    warp_atomic_add(lY + a.t, gy);
}

// Reverse of the refill of Sec. 4 (types 1, 2, 3 and wall nodes) from the
// adjoint lPm of the refilled state into the state before it (lP0) and the
// window state at t (lSo).
template <typename T>
__global__ void k_adj_refill(Dev<T> d, StepArgs a, const T* lPm, T* lP0, T* lSo, double* par,
                             double* lY) {
    const int P = blockIdx.x * blockDim.x + threadIdx.x;
    double l_k = 0.0, gy = 0.0, gdy = 0.0;
    if (P < d.n) {
        T lam[9];
#pragma unroll
        for (int i = 0; i < 9; ++i) lam[i] = lPm[9 * (int64_t)P + i];
        const int type = d.rtype[P];
        const T rho0 = T(d.rho0);
        if (type == 0 || type == 2) {
            atomic_add9(lP0 + 9 * (int64_t)P, lam);
        } else if (type == 3) {
            const int k = d.rdonor[P];
            const double qx = __dadd_rn(d.xy[2 * P], a.dX), qy = __dadd_rn(d.xy[2 * P + 1], a.dY);
            double l0, l1, l2, dl[3];
            bary_rn(d.trigeo + 8 * (int64_t)k, qx, qy, l0, l1, l2);
            bary_dqy(d.trigeo + 8 * (int64_t)k, dl);
            const T lb[3] = {T(l0), T(l1), T(l2)};
            for (int q = 0; q < 3; ++q) {
                const int v = d.tri[3 * k + q];
                T out[9], f[9];
                load_d(d.fu_in + (int64_t)kRec * v, f);
                T dot = 0.0;
#pragma unroll
                for (int i = 0; i < 9; ++i) {
                    out[i] = lb[q] * lam[i];
                    dot += lam[i] * f[i];
                }
                atomic_add9(lP0 + 9 * (int64_t)v, out);
                gdy += dl[q] * double(dot);
            }
        } else if (type == 1) {
            const double wx = __dadd_rn(a.cx, d.xy[2 * P]), wy = __dadd_rn(a.cy, d.xy[2 * P + 1]);
            T st[12], fq[4][9], sq[4][12];
            double wq[4], dwq[4];
            int64_t bq[4];
            bool ok[4];
#pragma unroll
            for (int j = 0; j < 12; ++j) st[j] = 0.0;
            for (int q = 0; q < 4; ++q) {
                ok[q] = bilinear_corner(d, a.pbx0, a.pby0, wx, wy, q, bq[q], wq[q], dwq[q]);
                if (!ok[q]) continue;
#pragma unroll
                for (int i = 0; i < 9; ++i) fq[q][i] = T(d.sbox_old[i * d.bplane + bq[q]]);
                state_d(fq[q], rho0, sq[q]);
#pragma unroll
                for (int j = 0; j < 12; ++j) st[j] += T(wq[q]) * sq[q][j];
            }
            T ls[12];
            ffsT(st, rho0, T(d.kneq), lam, ls, l_k);
            for (int q = 0; q < 4; ++q) {
                if (!ok[q]) continue;
                T out[9];
#pragma unroll
                for (int i = 0; i < 9; ++i) out[i] = 0.0;
                stateT_add(sq[q], rho0, ls, T(wq[q]), out);
#pragma unroll
                for (int i = 0; i < 9; ++i)
                    if (out[i] != 0.0) atomicAdd(lSo + i * d.bplane + bq[q], out[i]);
                T dot = 0.0;
#pragma unroll
                for (int j = 0; j < 12; ++j) dot += ls[j] * sq[q][j];
                gy += dwq[q] * double(dot);
            }
        }
    }
    warp_atomic_add(par + 3, l_k);
    warp_atomic_add(lY + a.t, gy + gdy);
    warp_atomic_add(lY + a.t - 1, -gdy);
}

template <typename T>
void launch_adj_force(const Dev<T>& d, double lamF, T* lP, cudaStream_t s) {
    if (d.nseg > 0) k_adj_force<T><<<(d.nseg + 127) / 128, 128, 0, s>>>(d, lamF, lP);
}
size_t adj_packet_bytes(int n) { return (size_t)2 * n * 4 * 3 * 16; }
size_t adj_record_values(int n, int n_sub) { return (size_t)n_sub * n * kAdjRec; }
template <typename T>
void launch_adj_rows(const Dev<T>& d, const int32_t* tpos, Coef<T>* tco, cudaStream_t s) {
    k_adj_rows<T><<<(d.n + 127) / 128, 128, 0, s>>>(d, tpos, tco);
}
// as many blocks of `block` threads as `threads` needs, all resident
static int resident_blocks(const void* fn, int64_t threads, size_t smem = 0, int block = 128) {
    int dev = 0, sms = 0, per = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, fn, block, smem);
    return (int)std::max<int64_t>(1, std::min<int64_t>((threads + block - 1) / block, (int64_t)std::max(per, 1) * sms));
}
template <typename T>
cudaError_t launch_adj_fv_record(const Dev<T>& d, const StepArgs& a, const T* P0, T* b0, T* b1, cudaStream_t s) {
    const void* fn = (const void*)k_adj_fv_record<T>;
    Dev<T> dd = d;
    StepArgs aa = a;
    void* args[] = {&dd, &aa, &P0, &b0, &b1};
    return cudaLaunchCooperativeKernel(fn, dim3(resident_blocks(fn, d.n)), dim3(128), args, 0, s);
}
template <typename T>
cudaError_t launch_adj_fv(const Dev<T>& d, const StepArgs& a, const T* rec, const T* P0, const T* lPn, T* x0, T* x1,
                          const Coef<T>* tco, T* lsnap, double* par, double* lV, T* lPm, int max_row,
                          unsigned char* px, unsigned tag0, const int32_t* order,
                          cudaStream_t s) {
    // one node per quad over resident blocks (at most 7 off-diagonal entries), else any
    const void* fn = (const void*)k_adj_fv_rev<T, kTmemMaxEntries + 1>;
    // FP64: three warps issue at the full rate of a warp on its own, four do not
    const int block = sizeof(T) == 8 ? 96 : 128;
    const size_t tab = 3 * (size_t)d.n_sub * sizeof(T), smem = tab <= 48 * 1024 ? tab : 0;
    if (max_row > kTmemMaxEntries + 1 || (int64_t)resident_blocks(fn, 4 * (int64_t)d.n, smem, block) * (block / 4) < d.n)
        fn = (const void*)k_adj_fv_rev<T, 0>;
    int use_tab = smem > 0;
    Dev<T> dd = d;
    StepArgs aa = a;
    void* args[] = {&dd, &aa, &rec, &P0, &lPn, &x0, &x1, &tco, &lsnap, &par, &lV, &lPm, &use_tab, &px, &tag0, &order};
    return cudaLaunchCooperativeKernel(fn, dim3(resident_blocks(fn, 4 * (int64_t)d.n, smem, block)), dim3(block), args, smem,
                                       s);
}
template <typename T>
void launch_adj_feed(const Dev<T>& d, const StepArgs& a, const T* lsnap, T* lSo, T* lSn, double* lY,
                     cudaStream_t s) {
    if (d.n_outer) k_adj_feed<T><<<(d.n_outer + 127) / 128, 128, 0, s>>>(d, a, lsnap, lSo, lSn, lY);
}
template <typename T>
void launch_adj_stream(const Dev<T>& d, const StepArgs& a, const T* lfB, const T* lSn, T* lfA,
                       double* par, cudaStream_t s) {
    dim3 grid((d.nx + 127) / 128, d.ny);
    k_adj_stream<T><<<grid, 128, 0, s>>>(d, a, lfB, lSn, lfA, par);
}
template <typename T>
void launch_adj_fill(const Dev<T>& d, const StepArgs& a, T* lfA, T* lP, double* par, double* lY,
                     cudaStream_t s) {
    k_adj_fill<T><<<(unsigned)((d.bplane + 127) / 128), 128, 0, s>>>(d, a, lfA, lP, par, lY);
}
template <typename T>
void launch_adj_refill(const Dev<T>& d, const StepArgs& a, const T* lPm, T* lP0, T* lSo, double* par,
                       double* lY, cudaStream_t s) {
    k_adj_refill<T><<<(d.n + 127) / 128, 128, 0, s>>>(d, a, lPm, lP0, lSo, par, lY);
}

#define HLBM_INST(T)                                                                                        \
    template void launch_fv_coeffs<T>(const Dev<T>&, int, Coef<T>*, cudaStream_t);                          \
    template void launch_patch_init<T>(const Dev<T>&, const StepArgs&, cudaStream_t);                         \
    template void launch_refill<T>(const Dev<T>&, const StepArgs&, cudaStream_t);                             \
    template void launch_feed<T>(const Dev<T>&, const StepArgs&, cudaStream_t);                               \
    template int fv_tile_capacity<T>();                                                                       \
    template cudaError_t launch_fv_persistent<T>(const Dev<T>&, const StepArgs&, cudaStream_t);               \
    template size_t fv_smem_bytes<T>(int, int, int, int, int);                                                     \
    template int fv_tile_max<T>();                                                                            \
    template void launch_build_ell<T>(const Coef<T>*, const int32_t*, const int32_t*, Coef<T>*, int64_t,       \
                                      cudaStream_t);                                                          \
    template int fv_smem_tile_capacity<T>(size_t);                                                            \
    template cudaError_t launch_fv_smem<T>(const Dev<T>&, const StepArgs&, cudaStream_t);                     \
    template size_t fv_tmem_smem_bytes<T>(int, int, int, int);                                                \
    template int fv_tmem_tile_capacity<T>(size_t);                                                            \
    template cudaError_t launch_fv_tmem<T>(const Dev<T>&, const StepArgs&, cudaStream_t);                     \
    template cudaError_t launch_fv_tmem_pack<T>(const FvPack<T>&, int, size_t, cudaStream_t);                 \
    template int fv_deep_tmem_slots<T>();                                                                     \
    template int fv_deep_cap<T>(int);                                                                         \
    template int fv_deep_duo_slots<T>();                                                                      \
    template int fv_deep_early<T>();                                                                          \
    template int fv_deep_row_words<T>();                                                                      \
    template size_t fv_deep_packet_bytes<T>(int);                                                             \
    template size_t fv_deep_smem_bytes<T>(int, int, int, int, int);                                                \
    template int fv_deep_tile_capacity<T>(size_t);                                                            \
    template cudaError_t launch_fv_deep_pack<T>(const FvPack<T>&, int, size_t, cudaStream_t);                 \
    template cudaError_t launch_fv_deep<T>(const Dev<T>&, const StepArgs&, const FarArgs<T>*, cudaStream_t);  \
    template void launch_build_deep_rows<T>(const Dev<T>&, const int32_t*, const int32_t*, int64_t, uint32_t*, \
                                            cudaStream_t);                                                    \
    template void launch_force<T>(const Dev<T>&, int64_t, cudaStream_t);                                      \
    template void launch_patch_macro<T>(const Dev<T>&, double*, double*, double*, double*, cudaStream_t);    \
    template void launch_adj_force<T>(const Dev<T>&, double, T*, cudaStream_t);                               \
    template void launch_adj_rows<T>(const Dev<T>&, const int32_t*, Coef<T>*, cudaStream_t);                  \
    template cudaError_t launch_adj_fv_record<T>(const Dev<T>&, const StepArgs&, const T*, T*, T*, cudaStream_t); \
    template cudaError_t launch_adj_fv<T>(const Dev<T>&, const StepArgs&, const T*, const T*, const T*, T*, T*, \
                                          const Coef<T>*, T*, double*, double*, T*, int, unsigned char*, unsigned,             \
                                          const int32_t*, cudaStream_t);                                      \
    template void launch_adj_feed<T>(const Dev<T>&, const StepArgs&, const T*, T*, T*, double*, cudaStream_t); \
    template void launch_adj_stream<T>(const Dev<T>&, const StepArgs&, const T*, const T*, T*, double*,        \
                                       cudaStream_t);                                                         \
    template void launch_adj_fill<T>(const Dev<T>&, const StepArgs&, T*, T*, double*, double*, cudaStream_t);  \
    template void launch_adj_refill<T>(const Dev<T>&, const StepArgs&, const T*, T*, T*, double*, double*,     \
                                       cudaStream_t);
HLBM_INST(float)
HLBM_INST(double)

}  // namespace hk
