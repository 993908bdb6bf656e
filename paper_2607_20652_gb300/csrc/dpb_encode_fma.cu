// dpb_encode_fma.cu -- the §2.2 encoder with the child scoring of Eq. 6 on the
// FP32 pipe, for the rows the tensor-core encoder does not take (fp32 storage;
// bf16 with d not a multiple of 32 or above 1024): global selection, 16
// children per parent, beams up to 16. One warp per token.
//
// Scoring. Lane l owns coordinates l, l + 32, ...: for each of them it flips
// its x by the signs of 4 parents and adds the product with the level's 16
// generator signs, fp32 +-1 read from the plan's table GF (through L1), into
// 64 register sums, two per packed multiply-add: the product with +-1 is
// exact, so each sum rounds like a plain add. A halving butterfly then adds
// the lanes' sums: at step o a lane keeps half of its sums and hands the other
// half to lane ^ o, so 64 sums take 62 shuffles and end 2 to a lane (flat
// index 2 lane + e = 16 slot + j). Every sum is taken in the order of a
// per-child lane sum followed by an xor butterfly (o = 16, 8, ..., 1).
//
// What bounds it: the latency of the table loads and of a token's own chain at 12
// warps per SM (168 registers): about 70 instructions and 18 L1 wavefronts per 32
// coordinates and 4 parents, 41% of the cycles issue, L1 a third of its
// wavefronts. Measured, encode and decode of 3,001 fp32 rows (d = 768, 4 levels,
// beam 8, k = 32): 97 us, where a popcount per (child, coordinate), a warp sum
// per child and selection by bisection took 552 us; 256 rows of d = 64 (3
// levels, beam 4, k = 8): 71 to 15 us.
//
// Selection is that of the tensor-core encoder (dpb_encode_mma.cuh): the union
// threshold on 64-bit words at level 0, sorted code lists kept by rank merges.
#include "dpb_encode_mma.cuh"

namespace dpb {

namespace {

using mmaenc::cword;
using mmaenc::cword_idx;
using mmaenc::cword_z;
using mmaenc::kBeam;

// Blocks of two warps: a token is a long chain, and small blocks leave the
// spreading of a ragged batch over the SMs to the block scheduler.
// 6 blocks per SM (168 registers, both trips' generator signs in registers)
// took 96.7 us at 3,001 rows and 340 us at 12,000; 8 blocks (one trip's) 119
// and 340 us, 10 blocks (96 registers, some spilled) 97 and 374 us.
constexpr int kWarps = 2;
constexpr int kBlocks = 6;
constexpr int PT = 4;       // parents per scoring tile: 8 take 232 registers, 123 us at 3,001 rows against 97

struct FmaArgs {
    const void *x;
    int64_t T;
    const float *mu, *sigma;
    int32_t *idx;
    float *val, *xnorm;
    int32_t *status;
    const uint32_t *M, *G, *DD;
    const float4 *GF;  // [(L-1)][nq][4][32]
    int d, nq, levels, k, beam, ecap;
    float inv_sqrt_d;
};

// Words of a warp's shared memory: the row, the code list [k] and the scratch
// [ecap] (64-bit), the beam [16] and the repeat bits [8].
__host__ __device__ inline int fma_warp_words(int d, int k, int ecap) {
    return 4 * ((d + 3) / 4) + 2 * k + 2 * ecap + 16 + 8;
}

// z = (s - mu_c) / sigma_c.
__device__ __forceinline__ float z_of(float s, uint32_t c, const FmaArgs &a, int32_t *status) {
    if (!a.mu) return s;
    const float sd = a.sigma[c];
    if (!(sd > 0.f)) set_status(status, DPB_DEV_BAD_SIGMA);
    return (s - a.mu[c]) / sd;
}

// Halving butterfly over the lanes: v[0..N) summed across lanes, N / 32 sums
// left to a lane, flat index lane (N / 32) + e.
template <int N, int O>
__device__ __forceinline__ void halve_sums(float *v) {
    if constexpr (O > 0) {
        const bool up = (threadIdx.x & O) != 0;
#pragma unroll
        for (int i = 0; i < N / 2; ++i) {
            const float keep = up ? v[i + N / 2] : v[i], send = up ? v[i] : v[i + N / 2];
            v[i] = keep + __shfl_xor_sync(kFull, send, O);
        }
        halve_sums<N / 2, O / 2>(v);
    }
}

// Marks in dup (bit 16 S + j) every child p_S ^ g_j that a smaller slot's
// parent shares: p_S ^ p_S' == g_j ^ g_j' for some j'.
__device__ __forceinline__ void mark_repeats(const uint32_t *beams, int nb, const uint32_t *ddl, uint32_t *dup) {
    const int lane = threadIdx.x & 31;
    if (lane < 8) dup[lane] = 0u;
    __syncwarp();
#pragma unroll 1
    for (int q = lane; q < nb * (nb - 1) / 2; q += 32) {
        int S = 1;  // q = S (S - 1) / 2 + S'
        while ((S + 1) * S / 2 <= q) ++S;
        const uint32_t delta = beams[S] ^ beams[q - S * (S - 1) / 2];
        uint32_t h = dedup_hash(delta);
        for (int probe = 0; probe < kDedupSlots; ++probe) {
            const uint32_t ent = ddl[h];
            if (ent == 0u) break;
            if ((ent >> 4) == delta + 1u) {
                const uint32_t bit = (uint32_t)S * 16u + (ent & 15u);
                atomicOr(&dup[bit >> 5], 1u << (bit & 31u));
            }
            h = (h + 1u) & (kDedupSlots - 1);
        }
    }
    __syncwarp();
}

template <typename Tin, int KPL>
__global__ void __launch_bounds__(kWarps * 32, kBlocks) encode_fma_kernel(FmaArgs a) {
    extern __shared__ __align__(16) uint32_t smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int d = a.d, k = a.k, nq = a.nq;
    float *xs = reinterpret_cast<float *>(smem + warp * fma_warp_words(d, k, a.ecap));
    uint64_t *L = reinterpret_cast<uint64_t *>(xs + 4 * ((d + 3) / 4));
    uint64_t *E = L + k;
    uint32_t *beams = reinterpret_cast<uint32_t *>(E + a.ecap);
    uint32_t *dup = beams + 16;
    const int slot = lane >> 3, j0 = (2 * lane) & 15;  // this lane's children of a tile: slot, j0 and j0 + 1

    for (int64_t t = (int64_t)blockIdx.x * kWarps + warp; t < a.T; t += (int64_t)gridDim.x * kWarps) {
        const Tin *row = static_cast<const Tin *>(a.x) + t * d;
        float ss = 0.f;
#pragma unroll 4  // the row's loads in flight together
        for (int i = lane; i < d; i += 32) {
            const float v = ld_elem(row, i);
            xs[i] = v;
            ss += v * v;
        }
        ss = warp_sum(ss);
        if (a.xnorm && lane == 0) a.xnorm[t] = sqrtf(ss);
        __syncwarp();

        // ---- level 0: every coordinate is a candidate ----
        auto z0 = [&](int i) { return z_of(xs[i], (uint32_t)i, a, a.status); };
        auto z0q = [&](int i) { return z_of(xs[i], (uint32_t)i, a, nullptr); };
        bool done = false;
        if constexpr (KPL <= 4) {
            if (KPL <= 2 && d <= 64)  // two coordinates a lane at most: a union of 64 holds them all
                done = mmaenc::level0_union64<2, KPL>(z0, z0q, d, k, E, a.ecap, L, beams);
            else
                done = mmaenc::level0_union64<(KPL <= 2 ? 4 : 8), KPL>(z0, z0q, d, k, E, a.ecap, L, beams);
        }
        if (!done)
            mmaenc::level0_bisect(z0, z0q, 0, d, k, reinterpret_cast<float *>(E),
                                  reinterpret_cast<uint32_t *>(E) + a.ecap, a.ecap, L, beams);
        if (a.beam > kBeam) {
            if (lane < a.beam) beams[lane] = cword_idx(L[lane]);  // k >= beam
            __syncwarp();
        }

        for (int l = 1; l < a.levels; ++l) {
            const bool next = l + 1 < a.levels;
            const uint32_t *gl = a.G + l * DPB_MAX_CHILDREN;
            const float4 *gf = a.GF + (size_t)(l - 1) * nq * 128 + lane;
            mark_repeats(beams, a.beam, a.DD + (l - 1) * kDedupSlots, dup);
            uint64_t cw0[4] = {0ull, 0ull, 0ull, 0ull};  // the words of slots 0..7 (beams above 8)
            uint64_t c[4] = {0ull, 0ull, 0ull, 0ull};    // this lane's children of a group of 8 slots
            for (int h = 0; h * PT < a.beam; ++h) {
                const int S = PT * h + slot;
                float2 acc2[PT * 8];  // pairs of generators
#pragma unroll
                for (int i = 0; i < PT * 8; ++i) acc2[i] = make_float2(0.f, 0.f);
                uint32_t par[PT];
#pragma unroll
                for (int b = 0; b < PT; ++b) par[b] = PT * h + b < a.beam ? beams[PT * h + b] : 0u;
#pragma unroll 2  // two blocks' loads in flight
                for (int q = 0; q < nq; ++q) {
                    const int i = 32 * q + lane;
                    const float xv = i < d ? xs[i] : 0.f;
                    const uint32_t m = i < d ? __ldg(a.M + i) : 0u;
                    float4 s[4];
#pragma unroll
                    for (int w = 0; w < 4; ++w) s[w] = __ldg(gf + (q * 4 + w) * 32);
#pragma unroll
                    for (int b = 0; b < PT; ++b) {
                        const float xp = flip(xv, sign31(m, par[b]));
                        const float2 x2 = make_float2(xp, xp);
#pragma unroll
                        for (int w = 0; w < 4; ++w) {
                            float2 &lo = acc2[b * 8 + 2 * w], &hi = acc2[b * 8 + 2 * w + 1];
                            lo = __ffma2_rn(x2, make_float2(s[w].x, s[w].y), lo);
                            hi = __ffma2_rn(x2, make_float2(s[w].z, s[w].w), hi);
                        }
                    }
                }
                float acc[PT * 16];
#pragma unroll
                for (int i = 0; i < PT * 8; ++i) {
                    acc[2 * i] = acc2[i].x;
                    acc[2 * i + 1] = acc2[i].y;
                }
                halve_sums<PT * 16, 16>(acc);
                // ---- this lane's two children of the tile as candidate words ----
                uint64_t cw[2] = {0ull, 0ull};
                if (S < a.beam) {
                    const uint32_t p = beams[S];
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        const uint32_t ci = p ^ gl[j0 + e], bit = (uint32_t)S * 16u + (uint32_t)(j0 + e);
                        if (!((dup[bit >> 5] >> (bit & 31u)) & 1u))
                            cw[e] = cword(z_of(__fmul_rn(acc[e], a.inv_sqrt_d), ci, a, a.status), ci);
                    }
                }
                c[2] = h & 1 ? cw[0] : 0ull;
                c[3] = h & 1 ? cw[1] : 0ull;
                if (!(h & 1)) {
                    c[0] = cw[0];
                    c[1] = cw[1];
                    if ((h + 1) * PT < a.beam) continue;
                }
                // ---- a group's children into the code list; the next beam ----
                const bool one = a.beam <= kBeam;  // a single group
                const int nent = mmaenc::merge_entrants<KPL>(L, k, E, c, next && one ? beams : nullptr);
                if (one) {
                    if (next && (nent < kBeam || nent > 32)) mmaenc::beam_tournament(c, beams);
                } else if (h < 2) {
#pragma unroll
                    for (int e = 0; e < 4; ++e) cw0[e] = c[e];
                } else if (next) {
                    mmaenc::beam_tournament16(cw0, c, beams, a.beam);
                }
                __syncwarp();
            }
        }
        for (int e = lane; e < k; e += 32) {
            const uint64_t w = L[e];
            a.idx[t * k + e] = (int32_t)cword_idx(w);
            a.val[t * k + e] = cword_z(w);
        }
        __syncwarp();
    }
}

template <typename Tin, int KPL>
cudaError_t run(const FmaArgs &a, cudaStream_t stream) {
    const void *fn = (const void *)encode_fma_kernel<Tin, KPL>;
    const size_t smem = sizeof(uint32_t) * kWarps * (size_t)fma_warp_words(a.d, a.k, a.ecap);
    const cudaError_t e = allow_smem(fn, smem);
    if (e != cudaSuccess) return e;
    const int64_t want = (a.T + kWarps - 1) / kWarps;
    encode_fma_kernel<Tin, KPL><<<(unsigned)std::min<int64_t>(want, 1 << 20), kWarps * 32, smem, stream>>>(a);
    return cudaGetLastError();
}

template <typename Tin>
cudaError_t dispatch(const FmaArgs &a, cudaStream_t stream) {
    if (a.k <= 32) return run<Tin, 1>(a, stream);
    if (a.k <= 64) return run<Tin, 2>(a, stream);
    if (a.k <= 128) return run<Tin, 4>(a, stream);
    return run<Tin, 8>(a, stream);
}

}  // namespace

cudaError_t launch_encode_fma(const dpb_plan *p, const void *x, int64_t T, const float *mu, const float *sigma,
                              int32_t *idx, float *val, float *xnorm, int32_t *status, cudaStream_t stream) {
    const dpb_config &c = p->cfg;
    FmaArgs a{};
    a.x = x;
    a.T = T;
    a.mu = mu;
    a.sigma = sigma;
    a.idx = idx;
    a.val = val;
    a.xnorm = xnorm;
    a.status = status;
    a.M = p->dM;
    a.G = p->dG;
    a.DD = p->dDD;
    a.GF = reinterpret_cast<const float4 *>(p->dGF);
    a.d = c.d;
    a.nq = (c.d + 31) / 32;
    a.levels = c.levels;
    a.k = c.k;
    a.beam = c.beam;
    a.ecap = mmaenc::entrant_cap(c.k, 0);
    a.inv_sqrt_d = p->inv_sqrt_d;
    return c.dtype == DPB_BF16 ? dispatch<__nv_bfloat16>(a, stream) : dispatch<float>(a, stream);
}

}  // namespace dpb
