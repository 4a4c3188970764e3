// Seeded shot sampler: errors, syndromes e H^T and observables e L^T.
//
// Bound by the integer pipes: one SplitMix64 output per (shot, column), about 24
// instructions of which six are multiplies; the outputs are a few words per
// shot.  Lane = column, so that a warp vote is the packed error word.
//   - narrow (up to 256 columns, 1024 checks and logicals): one warp per shot,
//     everything in registers.  Lane = check for the syndrome: the parity of a
//     check is the parity of (error words AND its row mask), the vote over the
//     lanes the packed syndrome word; logical operators are further such rows.
//   - wide: a warp (to 1024 columns) or the block's eight (above: one warp would
//     take over 32 passes, and short batches of large graphs would leave the chip
//     idle) draw a shot.  Each warp lists the columns it drew in shared memory;
//     then lane = error: the column's checks are flipped by shared atomics and
//     its logical words XORed in registers.  Errors are few (p <= 0.1 in use), so
//     this costs a few passes where visiting the rows of H would cost an access
//     per edge (at p = 1/2 the two cost the same).
// Before, a block of 256 threads drew each shot with five block barriers, a
// shared atomic per set bit and a visit of every row: 1.34 ms per 10^6 shots of
// 144 columns and 1.36 ms per 10^5 of 2500 columns; now 0.30 ms (259 instead of
// 1145 warp instructions per shot, ALU pipe 74 %) and 0.60 ms.
#include <cstdint>
#include <type_traits>
#include <cuda_runtime.h>

#include "bpdc_internal.h"

namespace bpdc {
namespace {

constexpr int kSampleThreads = 256;
constexpr int kTeamColumns = 1024;   // wide form: more columns than this take a block per shot
constexpr uint64_t kGolden = 0x9E3779B97F4A7C15ull;

// Whether the high word of the SplitMix64 output of state z (Steele, Lea &
// Flood 2014) is below thr <= 2^31 (priors are at most 1/2).  The output's last
// step, z ^ (z >> 31), flips the lowest bit of the high word where its highest
// is set; such a word is at least 2^31 with or without it, so the step is left
// out.
__device__ __forceinline__ bool drawn(uint64_t z, uint32_t thr)
{
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return (uint32_t)(z >> 32) < thr;
}

// NW: error words (ceil(N / 32)); the row masks hold 4 or 8 words a row.
template <int NW>
__global__ void __launch_bounds__(kSampleThreads) sample_narrow_kernel(DevGraph g, int64_t B, uint64_t seed,
                                                                       uint64_t shot_offset, uint32_t *syn,
                                                                       uint32_t *obs, uint32_t *err)
{
    const int lane = threadIdx.x & 31, wpb = kSampleThreads / 32;
    const int rows = g.MW + (obs ? g.KW : 0);
    uint32_t thr[NW];
#pragma unroll
    for (int c = 0; c < NW; ++c) thr[c] = __ldg(g.thr + c * 32 + lane);
    for (int64_t b = (int64_t)blockIdx.x * wpb + (threadIdx.x >> 5); b < B; b += (int64_t)gridDim.x * wpb) {
        const uint64_t z = seed + ((shot_offset + (uint64_t)b) * (uint64_t)g.N + (uint64_t)lane + 1ull) * kGolden;
        uint32_t w[NW], mine = 0;
#pragma unroll
        for (int c = 0; c < NW; ++c) {
            w[c] = __ballot_sync(0xFFFFFFFFu, drawn(z + (uint64_t)c * (32ull * kGolden), thr[c]));
            if (lane == c) mine = w[c];
        }
        if (err && lane < NW) err[(size_t)b * NW + lane] = mine;
        // word c of the syndrome (c < MW) and of the observables stays on lane c
        const uint4 *m = g.row_mask + lane * ((NW + 3) / 4);
        for (int c = 0; c < rows; ++c, m += 32 * ((NW + 3) / 4)) {
            uint32_t x = 0;
#pragma unroll
            for (int k = 0; k < NW; k += 4) {
                const uint4 v = __ldg(m + k / 4);
                x ^= w[k] & v.x;
                if (k + 1 < NW) x ^= w[k + 1] & v.y;
                if (k + 2 < NW) x ^= w[k + 2] & v.z;
                if (k + 3 < NW) x ^= w[k + 3] & v.w;
            }
            const uint32_t word = __ballot_sync(0xFFFFFFFFu, (__popc(x) & 1) != 0);
            if (lane == c) mine = word;
        }
        if (lane < g.MW) syn[(size_t)b * g.MW + lane] = mine;
        else if (lane < rows) obs[(size_t)b * g.KW + lane - g.MW] = mine;
    }
}

// WARPS: warps per shot (1 or the block's 8).  KWR > 0: at most KWR logical words,
// XORed in registers; 0: by shared atomics.
template <int WARPS, int KWR>
__global__ void __launch_bounds__(kSampleThreads) sample_wide_kernel(DevGraph g, int64_t B, uint64_t seed,
                                                                     uint64_t shot_offset, uint32_t *syn,
                                                                     uint32_t *obs, uint32_t *err)
{
    constexpr int TPB = kSampleThreads / 32 / WARPS;   // shots a block draws at a time
    extern __shared__ uint32_t sm[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int team = warp / WARPS, tw = warp % WARPS, tl = tw * 32 + lane;
    const int wpw = (g.NW + WARPS - 1) / WARPS;        // error words a warp draws at most
    uint32_t *sb = sm + team * (g.MW + g.KW), *ob = sb + g.MW;
    uint16_t *list = reinterpret_cast<uint16_t *>(sm + TPB * (g.MW + g.KW)) + (size_t)warp * wpw * 32;
    auto sync = [] {
        if constexpr (WARPS == 1) __syncwarp();
        else __syncthreads();
    };
    const uint32_t below = (1u << lane) - 1u;
    for (int x = tl; x < g.MW + g.KW; x += WARPS * 32) sb[x] = 0;
    sync();
    for (int64_t b0 = (int64_t)blockIdx.x * TPB; b0 < B; b0 += (int64_t)gridDim.x * TPB) {
        const int64_t b = b0 + team;
        if (WARPS == 1 && b >= B) break;
        uint64_t z = seed + ((shot_offset + (uint64_t)b) * (uint64_t)g.N + (uint64_t)tl + 1ull) * kGolden;
        int n = 0;
        uint32_t *const erow = err + (size_t)b * g.NW;
#pragma unroll 2
        for (int j = tl; j < g.NW * 32; j += WARPS * 32) {
            const bool hit = drawn(z, __ldg(g.thr + j));
            z += (uint64_t)(WARPS * 32) * kGolden;
            const uint32_t word = __ballot_sync(0xFFFFFFFFu, hit);
            if (hit) list[n + __popc(word & below)] = (uint16_t)j;
            n += __popc(word);
            if (err && lane == 0) erow[j >> 5] = word;
        }
        __syncwarp();
        uint32_t acc[KWR > 0 ? KWR : 1];
#pragma unroll
        for (int x = 0; x < (KWR > 0 ? KWR : 1); ++x) acc[x] = 0;
        for (int i = lane; i < n; i += 32) {
            const int j = list[i];
            const int a1 = __ldg(g.c_ptr + j + 1);
            for (int a = __ldg(g.c_ptr + j); a < a1; ++a) {
                const int r = __ldg(g.c_chk + a);
                atomicXor(sb + (r >> 5), 1u << (r & 31));
            }
            if (!obs) continue;
            const uint32_t *lc = g.l_col + (size_t)j * g.KW;
            if constexpr (KWR > 0) {
#pragma unroll
                for (int x = 0; x < KWR; ++x)
                    if (x < g.KW) acc[x] ^= __ldg(lc + x);
            } else {
                for (int x = 0; x < g.KW; ++x) {
                    const uint32_t v = __ldg(lc + x);
                    if (v) atomicXor(ob + x, v);
                }
            }
        }
        if (KWR > 0 && obs) {
            __syncwarp();
#pragma unroll
            for (int x = 0; x < KWR; ++x) {
                if (x >= g.KW) break;
                const uint32_t v = __reduce_xor_sync(0xFFFFFFFFu, acc[x]);
                if (v && lane == 0) atomicXor(ob + x, v);
            }
        }
        sync();
        for (int x = tl; x < g.MW + g.KW; x += WARPS * 32) {   // out, and cleared for the next shot
            const uint32_t v = sb[x];
            sb[x] = 0;
            if (x < g.MW) syn[(size_t)b * g.MW + x] = v;
            else if (obs) obs[(size_t)b * g.KW + x - g.MW] = v;
        }
        sync();
    }
}

int grid_size(int64_t B, int per_block, int sms)
{
    const int64_t need = (B + per_block - 1) / per_block;
    return (int)(need < sms * 8 ? need : sms * 8);   // 2048 threads on each SM
}

template <int WARPS, int KWR>
cudaError_t launch_wide(const DevGraph &g, int64_t B, uint64_t seed, uint64_t shot_offset, uint32_t *syn,
                        uint32_t *obs, uint32_t *err, int sms, cudaStream_t s)
{
    constexpr int TPB = kSampleThreads / 32 / WARPS;
    const size_t smem = (size_t)TPB * (g.MW + g.KW) * 4 + (size_t)8 * ((g.NW + WARPS - 1) / WARPS) * 32 * 2;
    if (smem > 48 * 1024) {
        const cudaError_t e = cudaFuncSetAttribute((const void *)sample_wide_kernel<WARPS, KWR>,
                                                   cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    sample_wide_kernel<WARPS, KWR>
        <<<grid_size(B, TPB, sms), kSampleThreads, smem, s>>>(g, B, seed, shot_offset, syn, obs, err);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_sample(const DevGraph &g, int64_t B, uint64_t seed, uint64_t shot_offset, uint32_t *syn,
                          uint32_t *obs, uint32_t *err, int sms, cudaStream_t s)
{
    if (B <= 0) return cudaSuccess;
    if (g.NW <= kSampleMaskWords && g.MW + g.KW <= 32) {
        static_assert(kSampleMaskWords == 8, "one instance per word count");
        decltype(&sample_narrow_kernel<1>) const fn[] = {
            sample_narrow_kernel<1>, sample_narrow_kernel<2>, sample_narrow_kernel<3>, sample_narrow_kernel<4>,
            sample_narrow_kernel<5>, sample_narrow_kernel<6>, sample_narrow_kernel<7>, sample_narrow_kernel<8>};
        fn[g.NW - 1]<<<grid_size(B, 8, sms), kSampleThreads, 0, s>>>(g, B, seed, shot_offset, syn, obs, err);
        return cudaGetLastError();
    }
    auto go = [&](auto w, auto k) {
        return launch_wide<decltype(w)::value, decltype(k)::value>(g, B, seed, shot_offset, syn, obs, err, sms, s);
    };
    using std::integral_constant;
    // a block per shot also where eight shots' logical words would not fit its memory
    if (g.N > kTeamColumns || (size_t)8 * (g.MW + g.KW + g.NW * 16) * 4 > 48 * 1024) {
        const integral_constant<int, 8> w{};
        return g.KW <= 1 ? go(w, integral_constant<int, 1>{}) : g.KW <= 8 ? go(w, integral_constant<int, 8>{})
                                                                          : go(w, integral_constant<int, 0>{});
    }
    const integral_constant<int, 1> w{};
    return g.KW <= 1 ? go(w, integral_constant<int, 1>{}) : g.KW <= 8 ? go(w, integral_constant<int, 8>{})
                                                                      : go(w, integral_constant<int, 0>{});
}

}  // namespace bpdc
