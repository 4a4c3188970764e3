// Weighted product-sum BP with a hand-written adjoint (differentiable
// decoding; not part of the paper).  For iterations t = 0..T-1 over the edges
// e = (i, j) of H in CSR order, with weights W[0][t][e] (check -> variable,
// wc) and W[1][t][e] (variable -> check, wv):
//
//   q_e(t) = clip(wv[t][e] * (lambda_j + sum_{e' in M(j), e' != e} r_e'(t-1)), -Q, Q),   r(-1) = 0
//   r_e(t) = wc[t][e] * (-1)^{s_i} prod_{e' in N(i), e' != e} sgn(q_e'(t))
//                     * phi(sum_{e' in N(i), e' != e} phi(max(|q_e'(t)|, qmin)))
//   L_j(t) = lambda_j + sum_{e in M(j)} r_e(t)
//
// phi(x) = -log tanh(x/2) (Sec. II.C.1's product-sum rule in log form).  With
// unit weights and no clipping this is the decoder's flooding product-sum BP.
//
// Bound by instruction issue: phi (log1p of a quotient by expm1) and 1 / sinh take
// some 60 instructions each and are evaluated twice per edge and iteration in the
// forward, three times in the adjoint.  So those run with one lane per edge (432
// edges: 14 passes of a warp, 96 % of the lanes; a lane per check would keep 72 of
// 96), and only the short sums over a check or a variable run with a lane per
// check or variable, in place over one value per edge in shared memory.
//
// A team of G threads decodes a shot: 64 when there are enough shots, else 256.
// The forward saves S of every iteration (with the outgoing sign) in the
// workspace: r(t) = wc phi(S) and then q(t+1) follow from it, so the adjoint
// neither keeps a segment of q and r in shared memory (which left 8 warps on an
// SM) nor evaluates phi(|q|) again.  Every operation is the one the definition
// gives, in one fixed order, so gradients of long unrolled runs, which amplify
// rounding, do not depend on the launch.
//
// Gradients are summed over shots in a fixed order: the shots of a block (4 to 8)
// in shared memory at each iteration (sum64), the blocks' sums by a second kernel,
// both in FP64: partial sums of gradients that cancel may lie far above the total, up
// to beyond the float range.  A store of every shot's gradients was 283 MB a call.
//
// BB[[144,12,12]], T = 20, 4096 shots: forward 545 -> 299 us (issue 79 %), adjoint
// with the sum of the gradients 3310 -> 567 us a call (11 900 -> about 5050 warp
// instructions per shot and iteration).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>

#include "bpdc_internal.h"

namespace bpdc {
namespace {

constexpr float kQmin = 1e-6f;
constexpr int kNoEdge16 = 0xFFFF;

__device__ __forceinline__ float wphi(float x) { return log1pf(2.0f / expm1f(x)); }

// 1 / sinh(x) for x > 0 without overflow: 2 e^-x / (1 - e^-2x)
__device__ __forceinline__ float inv_sinh(float x) { return 2.0f * expf(-x) / -expm1f(-2.0f * x); }

__device__ __forceinline__ uint32_t syn_bit(const uint32_t *sy, int i) { return (__ldg(sy + (i >> 5)) >> (i & 31)) & 1u; }

__device__ __forceinline__ float with_sign(float mag, bool neg)
{
    return __uint_as_float(__float_as_uint(mag) | (neg ? 0x80000000u : 0u));
}
__device__ __forceinline__ bool sign_of(float x) { return (__float_as_uint(x) >> 31) != 0u; }

// Most shots of a block.
constexpr int most_shots(int G) { return 1024 / G < 8 ? 1024 / G : 8; }

// The G threads that work on a shot; named barrier 1 + index of the shot in the block.
template <int G>
__device__ __forceinline__ void team_sync(int team)
{
    asm volatile("bar.sync %0, %1;" ::"r"(1 + team), "n"(G) : "memory");
}

// The sum of n <= MOST floats x[0], x[stride], ... to more than FP64's 53 bits: a
// float that collects the sum, one that collects its exact rounding errors (two-sum)
// and one for theirs, added up in FP64 at the end.  FP64 runs at a 64th of the FP32
// rate here: with an FP64 add for each of the 71 million terms of 4096 BB[[144,12,12]]
// shots, T = 20, a backward call takes 599 us, with this form 567 (533 with two floats,
// some 48 bits and the range of one).  Sums that leave the float range on the way, or
// hold an infinity or a NaN, are taken again term by term in FP64.
__device__ __forceinline__ void two_sum(float &s, float x, float &err)
{
    const float t = s + x, b = t - s;
    err = (s - (t - b)) + (x - b);
    s = t;
}
// Conversions to FP64 run at that rate too, so the three floats are widened by integer
// operations: 3000 phenomenological BB[[72,12,6]] shots, T = 6, 761 -> 678 us (610 with
// two floats), 1023 BB[[144,12,12]] shots, T = 20, 225 -> 208, but 4096 shots 562 -> 567.
// Small values are scaled by 2^64 first, which makes denormals normal (the last float
// of a training step's small gradients often is one; a path of their own for them cost
// a step 10 us).
__device__ __forceinline__ double widen(float x)
{
    const bool small = fabsf(x) < 0x1p-62f;
    const uint32_t u = __float_as_uint(x * (small ? 0x1p64f : 1.0f)), m = u & 0x7FFFFFFFu;
    const uint32_t hi = m ? (m >> 3) + (small ? (1023u - 127u - 64u) << 20 : (1023u - 127u) << 20) : 0u;
    return __hiloint2double((int)((u & 0x80000000u) | hi), (int)(u << 29));
}
template <int MOST>
__device__ __forceinline__ double sum64(const float *x, int n, size_t stride)
{
    float v[MOST];
#pragma unroll
    for (int w = 0; w < MOST; ++w) v[w] = w < n ? x[w * stride] : 0.0f;
    float a = v[0], b, c = 0.0f;
    two_sum(a, v[1], b);
#pragma unroll
    for (int w = 2; w < MOST; ++w) {
        if (w >= n) break;
        float e, f;
        two_sum(a, v[w], e);
        two_sum(b, e, f);
        c += f;
    }
    // where a is not finite, neither is its error b
    if (isfinite(b + c)) return widen(a) + (widen(b) + widen(c));
    double s = 0.0;
    for (int w = 0; w < n; ++w) s += (double)x[w * stride];
    return s;
}

// In place over the edges of every variable (lanes over variables; m-th edge of
// variable j in c_edget[m * N + j]): out(j, base, pre_m + suf_m) with pre_m / suf_m
// the sums of the values before / after edge m, and total(j, values) per variable.
template <int G, int CM, typename Base, typename Total>
__device__ __forceinline__ void var_phase(const DevGraph &g, float *x, int u, int cm, bool write, Base base, Total total)
{
    for (int j = u; j < g.N; j += G) {
        int ee[CM];
        float v[CM], pre[CM];
        float sum = 0.0f;
#pragma unroll
        for (int m = 0; m < CM; ++m) {
            ee[m] = kNoEdge16;
            v[m] = 0.0f;
            if (m < cm) {
                ee[m] = __ldg(g.c_edget + m * g.N + j);
                if (ee[m] != kNoEdge16) v[m] = x[ee[m]];
            }
            pre[m] = sum;
            sum += v[m];
        }
        const float b = base(j);
        total(j, b, v);
        if (!write) continue;
        float suf = 0.0f;
#pragma unroll
        for (int m = CM - 1; m >= 0; --m) {
            if (ee[m] != kNoEdge16) x[ee[m]] = b + (pre[m] + suf);
            suf += v[m];
        }
    }
}

template <int G, int CM, int RM>
__global__ void __launch_bounds__(G == 64 ? 512 : 1024, G == 64 ? 4 : 2) wbp_forward_kernel(DevGraph g, WbpArgs a)
{
    extern __shared__ float sm[];
    const int team = threadIdx.x / G, u = threadIdx.x % G, W = blockDim.x / G;
    const int E = a.E, T = a.T;
    float *x = sm + (size_t)team * E;   // per edge: r, then lambda + sum r, phi(|q|), S, r again
    const float clip = a.clip;
    for (int64_t b = (int64_t)blockIdx.x * W + team; b < a.B; b += (int64_t)gridDim.x * W) {
        const uint32_t *sy = a.syn + b * g.MW;
        float *post = a.post ? a.post + (size_t)b * T * g.N : nullptr;
        float *save = a.S + (size_t)b * T * E;
        for (int e = u; e < E; e += G) x[e] = 0.0f;
        team_sync<G>(team);
        for (int t = 0; t <= T; ++t) {
            // posteriors of iteration t-1 and lambda + the other r of iteration t
            var_phase<G, CM>(
                g, x, u, a.cm, t < T, [&](int j) { return __ldg(g.lam_col + j); },
                [&](int j, float lam, const float (&r)[CM]) {
                    if (!post || t == 0) return;
                    float L = lam;
#pragma unroll
                    for (int m = 0; m < CM; ++m) L += r[m];
                    post[(size_t)(t - 1) * g.N + j] = L;
                });
            if (t == T) break;
            team_sync<G>(team);
            const float *wv = a.W + (size_t)(T + t) * E, *wc = a.W + (size_t)t * E;
            for (int e = u; e < E; e += G) {
                const float q = fminf(fmaxf(__ldg(wv + e) * x[e], -clip), clip);
                x[e] = with_sign(wphi(fmaxf(fabsf(q), kQmin)), q < 0.0f);
            }
            team_sync<G>(team);
            for (int i = u; i < g.M; i += G) {
                const int e0 = __ldg(g.h_ptr + i), d = __ldg(g.h_ptr + i + 1) - e0;
                float f[RM], suf[RM + 1];
                uint32_t negs = 0, par = syn_bit(sy, i);
#pragma unroll
                for (int k = 0; k < RM; ++k) {
                    f[k] = 0.0f;
                    if (k < d) {
                        const float v = x[e0 + k];
                        f[k] = fabsf(v);
                        const uint32_t ng = sign_of(v) ? 1u : 0u;
                        negs |= ng << k;
                        par ^= ng;
                    }
                }
                suf[RM] = 0.0f;
#pragma unroll
                for (int k = RM - 1; k >= 0; --k) suf[k] = suf[k + 1] + f[k];
                float pre = 0.0f;
#pragma unroll
                for (int k = 0; k < RM; ++k) {
                    if (k < d) {
                        x[e0 + k] = with_sign(pre + suf[k + 1], ((par ^ (negs >> k)) & 1u) != 0);
                        pre += f[k];
                    }
                }
            }
            team_sync<G>(team);
            for (int e = u; e < E; e += G) {
                const float sv = x[e], c = wphi(fabsf(sv));
                save[(size_t)t * E + e] = sv;
                x[e] = __ldg(wc + e) * (sign_of(sv) ? -c : c);
            }
            team_sync<G>(team);
        }
        team_sync<G>(team);
    }
}

template <int G, int CM, int RM>
__global__ void __launch_bounds__(G == 64 ? 512 : 1024, G == 64 ? 4 : 2) wbp_backward_kernel(DevGraph g, WbpArgs a, float *grad_w)
{
    extern __shared__ float sm[];
    const int team = threadIdx.x / G, u = threadIdx.x % G, W = blockDim.x / G;
    const int E = a.E, T = a.T;
    const size_t nw = (size_t)2 * T * E;
    // per shot and edge: adjoint chain, r(t-1) then lambda + the others then the wv
    // gradient, c(t) = phi(S(t)), the wc gradient
    float *x = sm + (size_t)team * 4 * E, *r = x + E, *cc = r + E, *pc = cc + E;
    const float clip = a.clip;
    float *part = a.part + (size_t)blockIdx.x * 2 * nw;
    const bool direct = (int64_t)W >= a.B;   // one block, one round: the sum is the result
    for (int64_t base = (int64_t)blockIdx.x * W; base < a.B; base += (int64_t)gridDim.x * W) {
        const int64_t b = base + team;
        const bool on = b < a.B;
        const int shots = (int)(a.B - base < W ? a.B - base : W);
        const float *gp = a.gpost + (size_t)b * T * g.N, *S = a.S + (size_t)b * T * E;
        if (on) {
            for (int e = u; e < E; e += G) {
                x[e] = 0.0f;
                cc[e] = wphi(fabsf(__ldg(S + (size_t)(T - 1) * E + e)));
            }
            team_sync<G>(team);
        }
        for (int t = T - 1; t >= 0; --t) {
            // adjoint of r(t): the posterior L(t) and, through q(t+1), the other edges
            if (on)
                var_phase<G, CM>(
                    g, x, u, a.cm, true, [&](int j) { return __ldg(gp + (size_t)t * g.N + j); },
                    [](int, float, const float (&)[CM]) {});
            __syncthreads();   // and the previous iteration's sums have been taken
            if (on) {
                const float *wc = a.W + (size_t)t * E, *St = S + (size_t)t * E;
                for (int e = u; e < E; e += G) {
                    const float rb = x[e], sv = __ldg(St + e);
                    const float s = sign_of(sv) ? -1.0f : 1.0f;
                    pc[e] = rb * s * cc[e];
                    x[e] = rb * __ldg(wc + e) * s * inv_sinh(fabsf(sv));
                    if (t > 0) {
                        const float s1 = __ldg(St - E + e), c1 = wphi(fabsf(s1));
                        cc[e] = c1;
                        r[e] = __ldg(wc - E + e) * (sign_of(s1) ? -c1 : c1);
                    } else {
                        r[e] = 0.0f;   // r(-1)
                    }
                }
                team_sync<G>(team);
                // the sum over the other edges of every check
                for (int i = u; i < g.M; i += G) {
                    const int e0 = __ldg(g.h_ptr + i), d = __ldg(g.h_ptr + i + 1) - e0;
                    float gk[RM], pre[RM];
                    float sum = 0.0f;
#pragma unroll
                    for (int k = 0; k < RM; ++k) {
                        gk[k] = k < d ? x[e0 + k] : 0.0f;
                        pre[k] = sum;
                        sum += gk[k];
                    }
                    float suf = 0.0f;
#pragma unroll
                    for (int k = RM - 1; k >= 0; --k) {
                        if (k < d) x[e0 + k] = pre[k] + suf;
                        suf += gk[k];
                    }
                }
                // lambda + the other r(t-1) of every edge
                var_phase<G, CM>(g, r, u, a.cm, true, [&](int j) { return __ldg(g.lam_col + j); },
                                 [](int, float, const float (&)[CM]) {});
                team_sync<G>(team);
                const float *wv = a.W + (size_t)(T + t) * E;
                for (int e = u; e < E; e += G) {
                    const float av = r[e], w = __ldg(wv + e);
                    const float q = fminf(fmaxf(w * av, -clip), clip), ax = fabsf(q);
                    const float is = inv_sinh(ax);
                    const float dq = ax >= kQmin ? (q < 0.0f ? -is : is) : 0.0f;
                    const float qb = dq * x[e];
                    const bool in = fabsf(w * av) <= clip;
                    x[e] = in ? qb * w : 0.0f;
                    r[e] = in ? qb * av : 0.0f;
                }
            }
            __syncthreads();
            // the block's sums over its shots, in shot order
            for (int n = threadIdx.x; n < 2 * E; n += blockDim.x) {
                const bool second = n >= E;
                const int e = second ? n - E : n;
                const float *src = sm + (second ? E : 3 * E) + e;
                const size_t at = (size_t)((second ? T : 0) + t) * E + e;
                double s = sum64<most_shots(G)>(src, shots, (size_t)4 * E);
                if (base != (int64_t)blockIdx.x * W)
                    s += __hiloint2double(__float_as_int(part[at]), __float_as_int(part[nw + at]));
                if (direct) {
                    grad_w[at] = (float)s;
                } else {
                    part[at] = __int_as_float(__double2hiint(s));
                    part[nw + at] = __int_as_float(__double2loint(s));
                }
            }
        }
        __syncthreads();
    }
}

// Sum of the blocks' partial sums in block order: 32 weights x 8 runs of blocks.
__global__ void __launch_bounds__(256) wbp_reduce_kernel(const float *part, int blocks, int64_t nw, float *out)
{
    __shared__ double sums[8][32];
    const int lane = threadIdx.x & 31, run = threadIdx.x >> 5;
    const int64_t w = (int64_t)blockIdx.x * 32 + lane;
    const int per = (blocks + 7) / 8, b1 = min(blocks, (run + 1) * per);
    double s = 0.0;
    if (w < nw)
        for (int b = run * per; b < b1; ++b) {
            const float *p = part + (size_t)b * 2 * nw + w;
            s += __hiloint2double(__float_as_int(p[0]), __float_as_int(p[nw]));
        }
    sums[run][lane] = s;
    __syncthreads();
    if (run == 0 && w < nw) {
        for (int k = 1; k < 8; ++k) s += sums[k][lane];
        out[w] = (float)s;
    }
}

// Threads per shot: 64 where that gives every SM 16 warps (of the shots an SM gets
// and has memory for in the adjoint), else 256.  BB[[144,12,12]], T = 20, forward /
// backward call: 2000 shots 220 / 315 us with 64 threads, 288 / 380 with 256; 1023
// shots 188 / 243 against 177 / 204; 300 shots 170 / 227 against 123 / 172.
// Phenomenological BB[[72,12,6]] (1944 edges, 7 shots fit an SM), 3000 shots, T = 6:
// 367 / 1428 against 348 / 679.
int team_size(int64_t B, int E, int sms)
{
    const int64_t per_sm = std::min<int64_t>((B + sms - 1) / sms, (int64_t)(kMaxWbpSmem / ((size_t)16 * E)));
    return per_sm * 2 >= 16 ? 64 : 256;
}

// Shots of a block (at most `most`) for an even load: the SM with the most blocks
// gets as few shots as possible, then the most shots a block.  4096 shots take 4
// blocks of 7 on an SM instead of 4 of 8 (backward call 599 -> 567 us).  More than
// 4 blocks do not fit an SM: the teams' named barriers take all 16 of a block, and
// an SM has 64 (blocks of 3 shots, 27 on an SM, ran 12 at a time: forward 406 us
// against 328).
int shots_per_block(int64_t B, int least, int most, int sms)
{
    int best = most;
    int64_t load = INT64_MAX;
    for (int w = most; w >= least; --w) {
        const int64_t n = ((B + w - 1) / w + sms - 1) / sms;
        if (n > 4 && w < most) break;
        if (n * w < load) { best = w; load = n * w; }
    }
    return best;
}

// Shots of a backward block and number of blocks.  Their partial sums (2 x 2 x T x E
// floats a block) lie before the saved S in the workspace, which leaves at least
// B (T + 1) E floats: at least four shots a block, and blocks take several rounds of
// shots where that is short.
void backward_plan(int64_t B, int E, int T, int G, int sms, int *shots, int64_t *blocks)
{
    const int most = (int)std::min<size_t>(most_shots(G), kMaxWbpSmem / ((size_t)16 * E));
    const int64_t room = std::max<int64_t>(1, B * (T + 1) / ((int64_t)4 * T));
    int w = shots_per_block(B, std::min(4, most), most, sms);
    while (w < most && (B + w - 1) / w > room) ++w;
    *shots = (int)std::min<int64_t>(w, B);
    *blocks = std::min((B + *shots - 1) / *shots, room);
}

template <typename K>
cudaError_t allow_smem(K kernel, size_t smem)
{
    if (smem <= 48 * 1024) return cudaSuccess;
    return cudaFuncSetAttribute((const void *)kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
}

}  // namespace

cudaError_t launch_wbp_forward(const DevGraph &g, const WbpArgs &a, cudaStream_t s)
{
    if (a.B <= 0) return cudaSuccess;
    if (a.E > kWbpMaxEdges) return cudaErrorInvalidValue;
    const int G = team_size(a.B, a.E, a.sms);
    const int w = shots_per_block(a.B, 1, most_shots(G), a.sms);
    const size_t smem = (size_t)w * a.E * sizeof(float);
    const int grid = (int)std::min<int64_t>((a.B + w - 1) / w, (int64_t)a.sms * 32);
    auto go = [&](auto kernel) {
        const cudaError_t e = allow_smem(kernel, smem);
        if (e != cudaSuccess) return e;
        kernel<<<grid, w * G, smem, s>>>(g, a);
        return cudaGetLastError();
    };
    const bool small = a.cm <= 4 && a.rm <= 8;
    if (G == 64) return small ? go(wbp_forward_kernel<64, 4, 8>) : go(wbp_forward_kernel<64, kWbpMaxCol, kWbpMaxRow>);
    return small ? go(wbp_forward_kernel<256, 4, 8>) : go(wbp_forward_kernel<256, kWbpMaxCol, kWbpMaxRow>);
}

cudaError_t launch_wbp_backward(const DevGraph &g, const WbpArgs &a, float *grad_w, cudaStream_t s)
{
    const int64_t n = (int64_t)2 * a.T * a.E;
    if (a.B <= 0) return cudaMemsetAsync(grad_w, 0, sizeof(float) * n, s);
    if (a.E > kWbpMaxEdges) return cudaErrorInvalidValue;
    const int G = team_size(a.B, a.E, a.sms);
    int w;
    int64_t blocks;
    backward_plan(a.B, a.E, a.T, G, a.sms, &w, &blocks);
    const size_t smem = (size_t)w * 4 * a.E * sizeof(float);
    auto go = [&](auto kernel) {
        const cudaError_t e = allow_smem(kernel, smem);
        if (e != cudaSuccess) return e;
        kernel<<<(int)blocks, w * G, smem, s>>>(g, a, grad_w);
        return cudaGetLastError();
    };
    const bool small = a.cm <= 4 && a.rm <= 8;
    const cudaError_t e =
        G == 64 ? (small ? go(wbp_backward_kernel<64, 4, 8>) : go(wbp_backward_kernel<64, kWbpMaxCol, kWbpMaxRow>))
                : (small ? go(wbp_backward_kernel<256, 4, 8>) : go(wbp_backward_kernel<256, kWbpMaxCol, kWbpMaxRow>));
    if (e != cudaSuccess || w >= a.B) return e;   // one block in one round has written the gradient
    wbp_reduce_kernel<<<(int)((n + 31) / 32), 256, 0, s>>>(a.part, (int)blocks, n, grad_w);
    return cudaGetLastError();
}

}  // namespace bpdc
