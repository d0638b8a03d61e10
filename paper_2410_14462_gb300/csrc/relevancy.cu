// Relevancy of uplifted CLIP features to text queries (appendix, "Relevancy
// scores", after LERF): with s_iq = f^_i . phi^_q and s_ik = f^_i . phi^_k
// (l2-normalised feature, query and canonical-phrase embeddings),
//   r_iq = min_k exp(T s_iq) / (exp(T s_iq) + exp(T s_ik))
//        = min_k 1 / (1 + exp(T (s_ik - s_iq))).
//
// The work streams the feature rows once and does m = queries + phrases dot
// products of length d per row: a skinny product S = F Phi^T (n x d times
// d x m) with its epilogue, on CUDA cores (float32 accuracy).  A lane owns one
// or two rows and keeps all their m dots in registers: per channel it multiplies its
// rows' features (16-byte loads of its own rows from a staged chunk) with the
// normalised embeddings (16-byte loads, the same for the whole warp) in packed
// float32 pairs of embeddings.  Every warp streams its own rows, in chunks of 12
// channels by cp.async, the next one in flight while one is used; the blocks
// are persistent, so the embeddings are normalised once per block.  Each dot
// product is one fmaf chain over the channels in order, the row's squared norm
// two, over the even and the odd ones.
//
// Bound: the FMA pipe with the embeddings' shared-memory reads close behind (n d m
// multiply-adds, m rounded up to a multiple of 4).  500k x 512 features, 21 queries
// and 4 phrases: 874 -> 465 us against tiles of 4 rows x 4 embeddings per thread, padded
// to 32, 412 with the norm's products in packed pairs behind a step's dots (before
// them, or one by one between them, the accumulators spill: 478), and 403 with the rows'
// shares dealt over all SMs.  Four rows per lane at 8
// warps per SM, and scalar instead of packed multiply-adds, measured 460 and 520 us
// where this form took 465.
#include <algorithm>

#include "common.cuh"
#include "spec.cuh"

namespace ludvig {

namespace {

constexpr int kRelMaxM = 64;                   // queries + phrases
constexpr int kRelMaxSmemFloats = 40 * 1024;   // normalised embeddings in shared memory (160 KB)
constexpr int kRelWarps = 16;                  // at most, per block
constexpr int kRelChunk = 12;                  // channels staged at a time; a row's pitch too: the 16-byte
                                               // reads of 8 consecutive rows (48 bytes apart) hit all 32 banks

__device__ __forceinline__ void rel_copy(float* dst, const float* src, int bytes, bool in) {
    const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
    const int n = in ? bytes : 0;   // (nothing read, zeros written)
    if (bytes == 16)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(n) : "memory");
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(d), "l"(src), "r"(n) : "memory");
}

struct RelArgs {
    const float* f;
    int64_t n;
    int d, nq, m, vec;   // vec: rows start on 16-byte boundaries (d % 4 == 0 and f aligned)
    float T;
    float* r;
};

// Rows base .. base + 32 R of a warp (lane l: rows base + 32 a + l).
template <int M, int R>
__device__ __forceinline__ void relevancy_rows(const RelArgs& g, const float* sphi, float* stage, int64_t base) {
    const int lane = threadIdx.x & 31;
    const int d = g.d, d4 = (d + 3) & ~3, nq = g.nq;
    const int64_t n = g.n;
    const int nchunks = (d + kRelChunk - 1) / kRelChunk;
    constexpr int kRows = 32 * R;
    auto load_chunk = [&](int k) {
        float* dst = stage + (k & 1) * (kRows * kRelChunk);
        const int c0 = k * kRelChunk;
        if (g.vec) {
#pragma unroll
            for (int t = 0; t < kRows * 3 / 32; ++t) {
                const int e = lane + 32 * t, row = e / 3, c = 4 * (e - 3 * row);
                const bool in = base + row < n && c0 + c < d;
                rel_copy(dst + 4 * e, in ? g.f + (base + row) * d + c0 + c : g.f, 16, in);
            }
        } else {
            for (int e = lane; e < kRows * kRelChunk; e += 32) {
                const int row = e / kRelChunk, c = e - row * kRelChunk;
                const bool in = base + row < n && c0 + c < d;
                rel_copy(dst + e, in ? g.f + (base + row) * d + c0 + c : g.f, 4, in);
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    __syncwarp();
    load_chunk(0);
    F2 acc[R][M / 2];
    F2 norm[R];
#pragma unroll
    for (int a = 0; a < R; ++a) {
        norm[a] = f2(0.f, 0.f);
#pragma unroll
        for (int e = 0; e < M / 2; ++e) acc[a][e] = f2(0.f, 0.f);
    }
    for (int k = 0; k < nchunks; ++k) {
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncwarp();   // chunk k has landed for all lanes, chunk k - 1 is used up
        if (k + 1 < nchunks) load_chunk(k + 1);
        const float* st = stage + (k & 1) * (kRows * kRelChunk) + lane * kRelChunk;
        const int c0 = k * kRelChunk, cw = min(kRelChunk, d4 - c0);
#pragma unroll 1
        for (int c = 0; c < cw; c += 4) {
            float4 x[R];
#pragma unroll
            for (int a = 0; a < R; ++a) {
                x[a] = *reinterpret_cast<const float4*>(st + a * (32 * kRelChunk) + c);
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const float* pr = sphi + (size_t)(c0 + c + q) * M;
                F2 xx[R];
#pragma unroll
                for (int a = 0; a < R; ++a) {
                    const float v = q == 0 ? x[a].x : q == 1 ? x[a].y : q == 2 ? x[a].z : x[a].w;
                    xx[a] = f2(v, v);
                }
#pragma unroll
                for (int e = 0; e < M / 4; ++e) {
                    const ulonglong2 p = *reinterpret_cast<const ulonglong2*>(pr + 4 * e);
#pragma unroll
                    for (int a = 0; a < R; ++a) {
                        acc[a][2 * e] = f2_fma(xx[a], F2{p.x}, acc[a][2 * e]);
                        acc[a][2 * e + 1] = f2_fma(xx[a], F2{p.y}, acc[a][2 * e + 1]);
                    }
                }
            }
#pragma unroll
            for (int a = 0; a < R; ++a) {
                const F2 lo = f2(x[a].x, x[a].y), hi = f2(x[a].z, x[a].w);
                norm[a] = f2_fma(hi, hi, f2_fma(lo, lo, norm[a]));
            }
        }
    }
    // the minimum over the phrases for every (row, query), 32 rows at a time
    // through shared memory (the output of consecutive rows is contiguous)
#pragma unroll
    for (int a = 0; a < R; ++a) {
        __syncwarp();
        float s[M];
#pragma unroll
        for (int e = 0; e < M / 2; ++e) {
            const float2 v = f2_get(acc[a][e]);
            s[2 * e] = v.x;
            s[2 * e + 1] = v.y;
        }
        const float2 halves = f2_get(norm[a]);
        const float nn = halves.x + halves.y;
        const float inv = nn > 0.f ? 1.0f / sqrtf(nn) : 0.f;
        if (isfinite(nn)) {
            // 1 / (1 + exp(T inv (s_k - s_q))) falls with s_k: the largest phrase decides
            float top = -INFINITY;
#pragma unroll
            for (int e = 0; e < M; ++e)
                if (e >= nq && e < g.m) top = fmaxf(top, s[e]);
#pragma unroll
            for (int q = 0; q < M; ++q)
                if (q < nq) stage[lane * nq + q] = fminf(1.f, 1.0f / (1.0f + expf(g.T * inv * (top - s[q]))));
        } else {
#pragma unroll 1
            for (int q = 0; q < nq; ++q) {
                float sq = 0.f, best = 1.f;
#pragma unroll
                for (int e = 0; e < M; ++e)
                    if (e == q) sq = s[e];
#pragma unroll
                for (int e = 0; e < M; ++e)
                    if (e >= nq && e < g.m) best = fminf(best, 1.0f / (1.0f + expf(g.T * inv * (s[e] - sq))));
                stage[lane * nq + q] = best;
            }
        }
        __syncwarp();
        const int64_t row0 = base + 32 * a;
        const int rows = (int)max((int64_t)0, min((int64_t)32, n - row0));
        for (int o = lane; o < rows * nq; o += 32) g.r[row0 * nq + o] = stage[o];
    }
}

// Rows per lane, so that the dots (M R registers) fit at 16 warps per SM.
constexpr int rel_rows(int M) { return M <= 32 ? 2 : 1; }

// Floats of a warp's stage: two chunks of its rows, or 32 rows of output.
template <int M>
constexpr int rel_stage() {
    return 2 * 32 * rel_rows(M) * kRelChunk > 32 * (M - 1) ? 2 * 32 * rel_rows(M) * kRelChunk : 32 * (M - 1);
}

template <int M>
__global__ void __launch_bounds__(32 * kRelWarps, 1) k_relevancy(const RelArgs g, const float* __restrict__ phi,
                                                                int64_t rows_per_warp) {
    extern __shared__ __align__(16) float smem[];
    const int d = g.d, d4 = (d + 3) & ~3, m = g.m;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    float* sphi = smem;                            // [d4][M], normalised, zero past d and m
    float* stage = sphi + (size_t)d4 * M + warp * rel_stage<M>();
    for (int e = warp; e < M; e += nwarps) {
        float s = 0.f;
        if (e < m)
            for (int c = lane; c < d; c += 32) {
                const float v = phi[(int64_t)e * d + c];
                s = fmaf(v, v, s);
            }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        const float inv = s > 0.f ? 1.0f / sqrtf(s) : 0.f;
        for (int c = lane; c < d4; c += 32) sphi[c * M + e] = e < m && c < d ? phi[(int64_t)e * d + c] * inv : 0.f;
    }
    __syncthreads();
    // this warp's rows, 32 R at a time and what is left in halves (equal shares:
    // whole groups alone would leave most warps idle in the last round), the shares
    // dealt to the blocks in turn, so that few rows spread over all SMs: 5000 x 512, 25
    // embeddings 125 -> 74 us (87 with blocks of 128 rows)
    int64_t r0 = ((int64_t)warp * gridDim.x + blockIdx.x) * rows_per_warp;
    const int64_t r1 = min(g.n, r0 + rows_per_warp);
    constexpr int R = rel_rows(M);
    for (; r1 - r0 > 32 * (R - 1); r0 += 32 * R) relevancy_rows<M, R>(g, sphi, stage, r0);
    if constexpr (R > 1)
        if (r1 > r0) relevancy_rows<M, 1>(g, sphi, stage, r0);
}

template <int M>
ludvig_status launch_relevancy(const float* f, int64_t n, int d, const float* phi, int nq, int m, float T, float* r,
                               cudaStream_t st) {
    // set once per process; a function-local static is initialised by one thread
    static const cudaError_t configured =
        cudaFuncSetAttribute(k_relevancy<M>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
    LV_CUDA(configured);
    int dev = 0, sms = 0;
    LV_CUDA(cudaGetDevice(&dev));
    LV_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    // one block per SM, of as many warps as have room for their stage (at least
    // 8: the embeddings take at most 160 KB, a stage 8 KB)
    const size_t stage = sizeof(float) * rel_stage<M>(), embed = sizeof(float) * (size_t)((d + 3) & ~3) * M;
    const int nwarps = (int)std::min<size_t>(kRelWarps, (227 * 1024 - embed) / stage);
    const size_t smem = embed + nwarps * stage;
    const int64_t rpw = std::max<int64_t>(32, round_up(ceil_div(n, (int64_t)sms * nwarps), 32));
    RelArgs g{f, n, d, nq, m, d % 4 == 0 && (reinterpret_cast<uintptr_t>(f) & 15) == 0, T, r};
    k_relevancy<M><<<(unsigned)std::min<int64_t>(sms, ceil_div(n, rpw)), 32 * nwarps, smem, st>>>(g, phi, rpw);
    LV_LAUNCH();
    return LUDVIG_OK;
}

int relevancy_bucket(int m) { return m <= 8 ? 8 : m <= 16 ? 16 : m <= 32 ? 32 : 64; }

}  // namespace

}  // namespace ludvig

using namespace ludvig;

extern "C" ludvig_status ludvig_relevancy(const float* feats, int64_t n, int32_t d, const float* phi, int32_t n_queries,
                                          int32_t n_canon, float temperature, float* r, void* stream) {
    LV_ARG(n >= 0 && d >= 1, "bad sizes");
    LV_ARG(n_queries >= 1 && n_canon >= 1 && n_queries + n_canon <= kRelMaxM,
           "need 1 <= queries, 1 <= phrases, queries + phrases <= %d", kRelMaxM);
    LV_ARG((int64_t)relevancy_bucket(n_queries + n_canon) * d <= kRelMaxSmemFloats,
           "(queries + phrases, rounded up to 8, 16, 32 or 64) x d must be <= %d", kRelMaxSmemFloats);
    LV_ARG(temperature > 0.f, "temperature must be positive");
    if (n == 0) return LUDVIG_OK;
    LV_ARG(feats != nullptr && phi != nullptr && r != nullptr, "NULL buffer");
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    StageScope scope(LUDVIG_STAGE_RELEVANCY, st);
    const int m = n_queries + n_canon;
    switch ((m + 3) / 4) {
#define LV_REL(M) return launch_relevancy<M>(feats, n, d, phi, n_queries, m, temperature, r, st)
        case 1: LV_REL(4);
        case 2: LV_REL(8);
        case 3: LV_REL(12);
        case 4: LV_REL(16);
        case 5: LV_REL(20);
        case 6: LV_REL(24);
        case 7: LV_REL(28);
        case 8: LV_REL(32);
        case 9:
        case 10: LV_REL(40);
        case 11:
        case 12: LV_REL(48);
        case 13:
        case 14: LV_REL(56);
        default: LV_REL(64);
#undef LV_REL
    }
}
