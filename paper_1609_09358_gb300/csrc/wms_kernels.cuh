// wms_kernels.cuh -- training kernels of the learned weighted min-sum BP: forward with stored
// messages and the hand-written reverse sweep that returns the gradient of the per-edge,
// per-iteration scale factors.
//
// Forward (T iterations, no early stop): the BP of Sec. II-B with every g term scaled,
//   R sweep, PE stage s:  R[s+1][j]   = clip(w[t][0][s-1][j]   g(R[s][j], L'[s+1][j+d] + R[s][j+d]))
//                         R[s+1][j+d] = clip(w[t][0][s-1][j+d] g(R[s][j], L'[s+1][j]) + R[s][j+d])
//   L sweep, PE stage s:  L[s][j]     = clip(w[t][1][s-1][j]   g(L[s+1][j], L[s+1][j+d] + R[s][j+d]))
//                         L[s][j+d]   = clip(w[t][1][s-1][j+d] g(R[s][j], L[s+1][j]) + L[s+1][j+d])
// (L' = previous iteration), output LLR(u) = L[1] + R[1] of the last iteration, or of every
// iteration (`all`: a per-iteration training loss).  Same arithmetic, operation by operation,
// as the inference kernel with weights, so both agree bit for bit.  R[n+1] is read by nothing, so
// stage n of the R sweep is left out (its scales have gradient 0).
//
// Backward: reverse-mode through the unrolled iterations.  Message versions: R^t[s+1] depends on
// R^t[s] and L^{t-1}[s+1]; L^t[s] on L^t[s+1] and R^t[s].  Reverse order: for t = T-1..0 the L
// sweep is undone for s = 1..n, then the R sweep for s = n-1..1; by then every consumer of a message
// has been undone, so its adjoint is complete.  Within a stage each input node feeds exactly one PE,
// so adjoints accumulate without atomics; the weight gradients of all frames are summed with
// atomicAdd.  Subgradients: g(a, b) = sign(a) sign(b) min(|a|, |b|) passes the adjoint times
// sign(b) to a when |a| <= |b| and times sign(a) to b otherwise; clip passes it where |x| < M.
//
// Layout: the decoders' register-blocked plan (bp_kernel.cuh): a frame on N / 2^b threads, 2^b nodes
// of every column per thread, b stages between column exchanges.  Forward messages and backward
// adjoints stay in registers.  The adjoints have the same shape as the messages: undoing the L sweep
// consumes the columns aL[s+1] left by the later iteration and produces aR[s], undoing the R sweep
// the other way round, so about n columns are live and they cross groups where the messages do.
// Memory sees the messages once per sweep: per frame and iteration columns 2..n of R and of L,
// [T][2][n-1][N] floats, each column in the order of the thread that uses it (16 bytes per thread and
// access).  What bounds both kernels is that stream (2 (n-1) N floats per frame and iteration written
// once, read twice, the second time from L2) and, for the backward one, a float reduction in L2 per
// weight, frame and iteration.
// Measured (N = 1024, T = 20, 4096 frames): forward 1.21 ms, backward 2.45 ms, against 2.98 and 8.71
// for kernels with one PE per thread, every message (backward: every adjoint too) in memory and a
// barrier after every stage.  Without the reductions the backward one took 2.16 ms; with two frames
// per thread (half the scale loads and reductions, 600 bytes of spills) it took 3.7.
#pragma once

#include "bp_kernel.cuh"
#include "polar_common.cuh"

namespace polar {

struct WMSArgs {
    const float* llr;
    int B, T;
    float M;
    const float* w;        // [T][2][n][N]
    int all;               // outputs / their adjoints for every iteration ([T][B][N]) or the last ([B][N])
    float* llr_u;          // forward output
    const float* grad_u;   // backward input, same shape as llr_u
    float* grad_w;         // backward output [T][2][n][N], accumulated
    float* store;          // [B][T][2][n-1][N], 16-byte aligned
    const DevCode* code;
    // 16-byte accesses of llr_u / grad_u, w and grad_w where a thread's nodes are consecutive
    int out16, w16, gw16;
};

cudaError_t wms_forward_launch(int logn, const WMSArgs& a, cudaStream_t st);
cudaError_t wms_backward_launch(int logn, const WMSArgs& a, cudaStream_t st);

#ifdef POLAR_WMS_KERNELS

// Frames per CTA: a frame of at most 32 threads shares its CTA, wider ones own it.
template <class P>
constexpr int wms_frames_per_cta() { return P::T <= 32 ? 128 / P::T : 1; }

template <class P>
struct WMSThread {
    static constexpr int N = P::N, R = P::R, T = P::T, n = P::LOGN, NG = P::NG;
    int t;
    int xbase[NG];
    float* xbuf;  // [2][XW]
    __device__ __forceinline__ void init(int t_, float* xb)
    {
        t = t_;
        xbuf = xb;
        static_for<0, NG>([&](auto G) { xbase[G.value] = P::addr(P::tpart(G.value, t)); });
    }
    // one column from the mapping of group A to that of group B through exchange buffer x
    template <int A, int B>
    __device__ __forceinline__ void exchange(float (&v)[R], int x) const
    {
        float* xb = xbuf + (x & 1) * P::XW;
#pragma unroll
        for (int k = 0; k < R; ++k) xput<P, A>(xb, xbase, t, k, v[k]);
        group_sync<T, false>(0);
#pragma unroll
        for (int k = 0; k < R; ++k) v[k] = xget<P, B>(xb, xbase, t, k);
    }
    // this thread's values of a row of N floats in node order, mapping of group G; consecutive
    // nodes (group 0) as 16-byte loads if the row is aligned
    template <int G>
    __device__ __forceinline__ void row(const float* p, bool v16, float (&v)[R]) const
    {
        if (P::win(G) == 0 && v16) {
#pragma unroll
            for (int k = 0; k < R; k += 4) {
                const float4 x = __ldg(reinterpret_cast<const float4*>(p + P::node(G, t, k)));
                v[k] = x.x;
                v[k + 1] = x.y;
                v[k + 2] = x.z;
                v[k + 3] = x.w;
            }
        } else {
#pragma unroll
            for (int k = 0; k < R; ++k) v[k] = __ldg(p + P::node(G, t, k));
        }
    }
    // stored column: [R / 4][T][4]
    __device__ __forceinline__ void put(float* col, const float (&v)[R]) const
    {
#pragma unroll
        for (int k = 0; k < R; k += 4)
            reinterpret_cast<float4*>(col)[(k >> 2) * T + t] = make_float4(v[k], v[k + 1], v[k + 2], v[k + 3]);
    }
};

// Offset of stored column c (2..n) of R (dir 0) or L (dir 1) of iteration t in a frame's store.
template <class P>
__device__ __forceinline__ size_t wms_col(int t, int dir, int c)
{
    return ((size_t)(t * 2 + dir) * (P::LOGN - 1) + (c - 2)) * P::N;
}

template <class P, int THREADS, int CTAS>
__global__ void __launch_bounds__(THREADS, CTAS) wms_forward_kernel(const WMSArgs a)
{
    constexpr int N = P::N, R = P::R, n = P::LOGN, NG = P::NG, F = wms_frames_per_cta<P>();
    extern __shared__ __align__(16) float wms_smem[];
    const int slot = threadIdx.x / P::T, b = blockIdx.x * F + slot;
    if (b >= a.B) return;  // whole groups: a CTA shared by several frames only synchronises warps
    WMSThread<P> th;
    th.init(threadIdx.x % P::T, wms_smem + slot * 2 * P::XW);
    const int t = th.t;
    const DevCode& C = *a.code;
    const float M = a.M;
    const float* y = a.llr + (size_t)b * N;
    float* store = a.store + (size_t)b * a.T * 2 * (n - 1) * N;
    float Lc[n + 2][R], Rc[n + 2][R];
#pragma unroll
    for (int k = 0; k < R; ++k) {
        Lc[n + 1][k] = stage_clip(__ldg(y + P::node(NG - 1, t, k)), M);
        Rc[1][k] = frozen_at(C.frozen_bits, P::node(0, t, k)) ? M : 0.0f;
    }
#pragma unroll
    for (int c = 2; c <= n; ++c)
#pragma unroll
        for (int k = 0; k < R; ++k) Lc[c][k] = 0.0f;
    // scales of the stage being computed and of the next one (loaded a stage ahead: with loads at
    // their use the forward kernel took the same, the backward one 3.5 ms)
    float wv[R], wn[R];
    th.template row<0>(a.w, a.w16, wn);
    for (int it = 0; it < a.T; ++it) {
        const float* w = a.w + (size_t)it * 2 * n * N;
        static_for<1, n>([&](auto S) {
            constexpr int s = S.value, q = s - 1, g = P::grp(q), dd = 1 << (q - P::win(g));
#pragma unroll
            for (int k = 0; k < R; ++k) wv[k] = wn[k];
            if constexpr (s < n - 1)
                th.template row<P::grp(s)>(w + s * N, a.w16, wn);
            else
                th.template row<P::grp(n - 1)>(w + (2 * n - 1) * N, a.w16, wn);
#pragma unroll
            for (int k = 0; k < R; ++k) {
                if (k & dd) continue;
                const int k2 = k | dd;
                const float a1 = Rc[s][k], a2 = Rc[s][k2];
                Rc[s + 1][k] = clipm(fmul(wv[k], xmin(a1, fadd(Lc[s + 1][k2], a2))), M);
                Rc[s + 1][k2] = clipm(fadd(fmul(wv[k2], xmin(a1, Lc[s + 1][k])), a2), M);
            }
            if constexpr (P::rcross(s)) th.template exchange<g, P::grp(s)>(Rc[s + 1], P::xidx_r(s));
            th.put(store + wms_col<P>(it, 0, s + 1), Rc[s + 1]);
        });
        static_for_down<n, 1>([&](auto S) {
            constexpr int s = S.value, q = s - 1, g = P::grp(q), dd = 1 << (q - P::win(g));
#pragma unroll
            for (int k = 0; k < R; ++k) wv[k] = wn[k];
            if constexpr (s > 1)
                th.template row<P::grp(s - 2 < 0 ? 0 : s - 2)>(w + (n + s - 2) * N, a.w16, wn);
            else if (it + 1 < a.T)
                th.template row<0>(w + 2 * n * N, a.w16, wn);
#pragma unroll
            for (int k = 0; k < R; ++k) {
                if (k & dd) continue;
                const int k2 = k | dd;
                const float l1 = Lc[s + 1][k], l2 = Lc[s + 1][k2];
                Lc[s][k] = clipm(fmul(wv[k], xmin(l1, fadd(l2, Rc[s][k2]))), M);
                Lc[s][k2] = clipm(fadd(fmul(wv[k2], xmin(Rc[s][k], l1)), l2), M);
            }
            if constexpr (P::lcross(s)) th.template exchange<g, P::grp(s - 2 < 0 ? 0 : s - 2)>(Lc[s], P::xidx_l(s));
            if constexpr (s > 1) th.put(store + wms_col<P>(it, 1, s), Lc[s]);
        });
        if (a.all || it == a.T - 1) {
            float* out = a.llr_u + ((size_t)(a.all ? it : 0) * a.B + b) * N + P::node(0, t, 0);
            float u[R];
#pragma unroll
            for (int k = 0; k < R; ++k) u[k] = fadd(Lc[1][k], Rc[1][k]);
#pragma unroll
            for (int k = 0; k < R; k += 4) {
                if (a.out16) {
                    *reinterpret_cast<float4*>(out + k) = make_float4(u[k], u[k + 1], u[k + 2], u[k + 3]);
                } else {
                    out[k] = u[k];
                    out[k + 1] = u[k + 1];
                    out[k + 2] = u[k + 2];
                    out[k + 3] = u[k + 3];
                }
            }
        }
    }
}

// Reverse of one PE: forward o1 = clip(w1 g(u, v + q)), o2 = clip(w2 g(r, u) + q2) in the
// generic form shared by both sweeps; returns adjoints of the inputs and the weight gradients.
// (d/dv = d/dq: both enter through their sum.)
struct PEGrad {
    float du, dv, dr, dq2, dw1, dw2;
};
__device__ __forceinline__ float wms_signed(float x, float s) { return s < 0.0f ? -x : x; }
__device__ __forceinline__ PEGrad pe_backward(float u, float v, float q, float r, float q2, float w1, float w2, float M,
                                              float go1, float go2)
{
    PEGrad G;
    const float s1 = fadd(v, q);
    const float g1 = xmin(u, s1);
    const float g2 = xmin(r, u);
    const float c1 = fabsf(fmul(w1, g1)) < M ? go1 : 0.0f;
    const float c2 = fabsf(fadd(fmul(w2, g2), q2)) < M ? go2 : 0.0f;
    G.dw1 = c1 * g1;
    G.dw2 = c2 * g2;
    G.dq2 = c2;
    const float gg1 = c1 * w1, gg2 = c2 * w2;
    const bool first = fabsf(u) <= fabsf(s1);  // u is the smaller of (u, s1)
    const float d1 = wms_signed(gg1, first ? s1 : u);
    const bool rfirst = fabsf(r) <= fabsf(u);  // r is the smaller of (r, u)
    const float d2 = wms_signed(gg2, rfirst ? u : r);
    G.dv = first ? 0.0f : d1;
    G.dr = rfirst ? d2 : 0.0f;
    G.du = (first ? d1 : 0.0f) + (rfirst ? 0.0f : d2);
    return G;
}

// Adds a thread's R weight gradients (mapping of group G) to a row of N floats in node order.
template <class P, int G>
__device__ __forceinline__ void wms_add_row(float* p, bool v16, int t, const float (&v)[P::R])
{
    if (P::win(G) == 0 && v16) {
#pragma unroll
        for (int k = 0; k < P::R; k += 4)
            asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(p + P::node(G, t, k)), "f"(v[k]),
                         "f"(v[k + 1]), "f"(v[k + 2]), "f"(v[k + 3])
                         : "memory");
    } else {
#pragma unroll
        for (int k = 0; k < P::R; ++k) atomicAdd(p + P::node(G, t, k), v[k]);
    }
}

// The steps of one iteration's reverse sweep: m = 0..n-1 undo the L sweep's stages 1..n, m = n..2n-2
// the R sweep's stages n-1..1.
template <class P>
__host__ __device__ constexpr int wms_step_stage(int m) { return m < P::LOGN ? m + 1 : 2 * P::LOGN - 1 - m; }

template <class P>
__host__ __device__ constexpr int wms_slot_floats() { return 2 * P::XW + 2 * 2 * P::N; }  // exchange, staged columns

// Staging of the stored columns: [2 steps][R, L][R / 4][T][4] floats.
template <class P>
struct WMSStage {
    float* rows;
    uint32_t at;         // shared address of this thread's first value
    const float* store;  // the frame's store, at this thread's first value
    int t;
    __device__ __forceinline__ void copy(uint32_t to, const float* col) const
    {
#pragma unroll
        for (int k = 0; k < P::R / 4; ++k)
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(to + 16 * P::T * k), "l"(col + 4 * P::T * k)
                         : "memory");
    }
    // queue the columns of step m of iteration `it` into half `par` (one group per step, empty past
    // the end)
    template <int m>
    __device__ __forceinline__ void issue(int it, uint32_t par) const
    {
        constexpr int n = P::LOGN, N = P::N, s = wms_step_stage<P>(m);
        const uint32_t to = at + par * (2 * N * 4);
        if (it >= 0) {
            if (s > 1) copy(to, store + wms_col<P>(it, 0, s));
            if (m < n) {
                if (s < n) copy(to + N * 4, store + wms_col<P>(it, 1, s + 1));
            } else if (it > 0) {
                copy(to + N * 4, store + wms_col<P>(it - 1, 1, s + 1));
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    }
    __device__ __forceinline__ void take(uint32_t par, int which, float (&v)[P::R]) const
    {
        const float4* p = reinterpret_cast<const float4*>(rows + (par * 2 + which) * P::N) + t;
#pragma unroll
        for (int k = 0; k < P::R; k += 4) {
            const float4 x = p[(k >> 2) * P::T];
            v[k] = x.x;
            v[k + 1] = x.y;
            v[k + 2] = x.z;
            v[k + 3] = x.w;
        }
    }
};

// Scales of step m of an iteration whose scales start at w, mapping of its stage's group.
template <class P, int m>
__device__ __forceinline__ void wms_scales(const WMSThread<P>& th, const float* w, bool v16, float (&v)[P::R])
{
    constexpr int s = wms_step_stage<P>(m);
    th.template row<P::grp(s - 1)>(w + (m < P::LOGN ? P::LOGN + s - 1 : s - 1) * P::N, v16, v);
}

// The stored columns come through thread-private shared memory (each thread reads back only what it
// copied: no barrier), copied asynchronously two steps ahead, the scales one step ahead in registers:
// the sweep is one long dependent chain with few warps per SM, so loads at their use leave it waiting.
template <class P, int THREADS, int CTAS>
__global__ void __launch_bounds__(THREADS, CTAS) wms_backward_kernel(const WMSArgs a)
{
    constexpr int N = P::N, R = P::R, n = P::LOGN, NG = P::NG, F = wms_frames_per_cta<P>(), STEPS = 2 * n - 1;
    extern __shared__ __align__(16) float wms_smem[];
    const int slot = threadIdx.x / P::T, b = blockIdx.x * F + slot;
    if (b >= a.B) return;
    WMSThread<P> th;
    th.init(threadIdx.x % P::T, wms_smem + slot * wms_slot_floats<P>());
    const int t = th.t;
    WMSStage<P> stg;
    stg.rows = th.xbuf + 2 * P::XW;
    stg.at = (uint32_t)__cvta_generic_to_shared(stg.rows) + 16 * t;
    stg.store = a.store + (size_t)b * a.T * 2 * (n - 1) * N + 4 * t;
    stg.t = t;
    const DevCode& C = *a.code;
    const float M = a.M;
    const float* y = a.llr + (size_t)b * N;
    float aL[n + 2][R], aR[n + 2][R];  // aL[c]: of the later iteration until undone, then of this one
#pragma unroll
    for (int c = 1; c <= n; ++c)
#pragma unroll
        for (int k = 0; k < R; ++k) aL[c][k] = 0.0f;
    uint32_t par = 0;
    stg.template issue<0>(a.T - 1, 0);
    stg.template issue<1>(a.T - 1, 1);
    float wv[R], wn[R];
    wms_scales<P, 0>(th, a.w + (size_t)(a.T - 1) * 2 * n * N, a.w16, wn);
    for (int it = a.T - 1; it >= 0; --it) {
        const float* w = a.w + (size_t)it * 2 * n * N;
        float* gw = a.grad_w + (size_t)it * 2 * n * N;
        // LLR(u) of iteration t is L^t[1] + R[1]: its adjoint enters at column 1 (nothing else
        // reads L[1], so the column holds no other contribution)
        float cur[R];
        if (a.all || it == a.T - 1) {
            th.template row<0>(a.grad_u + ((size_t)(a.all ? it : 0) * a.B + b) * N, a.out16, cur);
        } else {
#pragma unroll
            for (int k = 0; k < R; ++k) cur[k] = 0.0f;
        }
        static_for<0, STEPS>([&](auto MC) {
            constexpr int m = MC.value, s = wms_step_stage<P>(m), g = P::grp(s - 1);
            constexpr int dd = 1 << (s - 1 - P::win(g));
            constexpr bool undo_l = m < n;
            if constexpr (m == n) {
                // R[n+1] has no consumer: the R sweep's stage n passes nothing
#pragma unroll
                for (int k = 0; k < R; ++k) cur[k] = aR[n][k];
            }
            if constexpr (!undo_l && P::lcross(s + 1)) th.template exchange<P::grp(s), g>(cur, P::xidx_l(s + 1));
            float l[R], r[R], dw[R];
#pragma unroll
            for (int k = 0; k < R; ++k) wv[k] = wn[k];
            if constexpr (m + 1 < STEPS)
                wms_scales<P, m + 1>(th, w, a.w16, wn);
            else if (it > 0)
                wms_scales<P, 0>(th, w - 2 * n * N, a.w16, wn);
            asm volatile("cp.async.wait_group 1;" ::: "memory");
            if constexpr (s == 1) {
#pragma unroll
                for (int k = 0; k < R; ++k) r[k] = frozen_at(C.frozen_bits, P::node(0, t, k)) ? M : 0.0f;
            } else {
                stg.take(par, 0, r);
            }
            if constexpr (undo_l && s == n) {
#pragma unroll
                for (int k = 0; k < R; ++k) l[k] = stage_clip(__ldg(y + P::node(NG - 1, t, k)), M);
            } else {
                if (undo_l || it > 0) {
                    stg.take(par, 1, l);
                } else {
#pragma unroll
                    for (int k = 0; k < R; ++k) l[k] = 0.0f;
                }
            }
#pragma unroll
            for (int k = 0; k < R; ++k) {
                if (k & dd) continue;
                const int k2 = k | dd;
                PEGrad G;
                if constexpr (undo_l) {
                    // o1 = clip(w1 g(l1, l2 + a2)), o2 = clip(w2 g(a1, l1) + l2)
                    G = pe_backward(l[k], l[k2], r[k2], r[k], l[k2], wv[k], wv[k2], M, cur[k], cur[k2]);
                    if constexpr (s < n) {
                        cur[k] = aL[s + 1][k] + G.du;
                        cur[k2] = aL[s + 1][k2] + (G.dv + G.dq2);
                    }
                    if constexpr (s > 1) {
                        aR[s][k] = G.dr;
                        aR[s][k2] = G.dv;
                    }
                } else {
                    // o1 = clip(w1 g(a1, l2 + a2)), o2 = clip(w2 g(a1, l1) + a2): generic form with
                    // u = a1, v = l2, q = a2, r = l1 (g(r, u) = g(l1, a1) = g(a1, l1)), q2 = a2
                    G = pe_backward(r[k], l[k2], r[k2], l[k], r[k2], wv[k], wv[k2], M, cur[k], cur[k2]);
                    if constexpr (s > 1) {
                        cur[k] = aR[s][k] + G.du;
                        cur[k2] = aR[s][k2] + (G.dv + G.dq2);
                    }
                    aL[s + 1][k] = G.dr;
                    aL[s + 1][k2] = G.dv;
                }
                dw[k] = G.dw1;
                dw[k2] = G.dw2;
            }
            // the step's staged columns are consumed: refill their half
            if constexpr (m + 2 < STEPS)
                stg.template issue<m + 2>(it, par);
            else
                stg.template issue<m + 2 - STEPS>(it - 1, par);
            par ^= 1;
            wms_add_row<P, g>(gw + (undo_l ? n + s - 1 : s - 1) * N, a.gw16, t, dw);
            if constexpr (undo_l && P::rcross(s)) th.template exchange<g, P::grp(s)>(cur, P::xidx_r(s));
        });
    }
}

#endif  // POLAR_WMS_KERNELS

}  // namespace polar
