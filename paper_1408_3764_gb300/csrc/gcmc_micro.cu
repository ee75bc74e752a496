// gcmc_micro.cu -- the microcell list of Sec. 3.3.
//
//   k_mc_count / k_mc_place / k_mc_sort   build (Sec. 3.3.1): every particle
//       goes to the microcell of its grid position, the slot array is stored
//       slot-major (slot k of every cell contiguous), and each cell lists its
//       particles species by species, index by index;
// The chain evaluated over the microcells is the chain kernel's microcell form
// (gcmc_chain.cu).
//
// Microcells have equal edges L / M, M = ceil(L / edge); the cube of cells
// around a point spans D cells each way, D = 1 + floor((rcg - 1) M / 2^32):
// a partner within the cutoff lies less than rcg grid steps away along each
// axis, and a cell d steps away starts more than (d - 1) 2^32 / M grid steps
// from any point of the centre cell.  When 2D + 1 > M every cell of the axis
// is visited once.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <string>

#include "gcmc_ctx.h"

namespace gcmc {

// ------------------------------------------------------------------ build
// Particles are enumerated species-major: flat index f = first[s] + i.
struct SpeciesPrefix {
    int64_t first[kMaxSpecies + 1];
};

__device__ __forceinline__ void species_of(const SpeciesPrefix &p, int S, int64_t f, int &s, int64_t &i)
{
    s = 0;
    while (s + 1 < S && f >= p.first[s + 1]) ++s;
    i = f - p.first[s];
}

__device__ __forceinline__ int64_t micro_of(uint4 r, uint32_t M)
{
    return ((int64_t)cell_coord(r.z, M) * M + cell_coord(r.y, M)) * M + cell_coord(r.x, M);
}

__global__ void k_mc_count(const uint4 *__restrict__ pos_by_id, int64_t maxN, SpeciesPrefix p, int S,
                           int64_t N, uint32_t M, int32_t *__restrict__ cnt)
{
    for (int64_t f = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; f < N; f += (int64_t)gridDim.x * blockDim.x) {
        int s;
        int64_t i;
        species_of(p, S, f, s, i);
        atomicAdd(&cnt[micro_of(pos_by_id[s * maxN + i], M)], 1);
    }
}

__global__ void k_mc_max(const int32_t *__restrict__ cnt, int64_t ncm, int32_t *__restrict__ out)
{
    int m = 0;
    for (int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; c < ncm; c += (int64_t)gridDim.x * blockDim.x)
        m = max(m, cnt[c]);
    for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0) atomicMax(out, m);
}

__global__ void k_mc_place(const uint4 *__restrict__ pos_by_id, int64_t maxN, SpeciesPrefix p, int S, int64_t N,
                           uint32_t M, int64_t ncm, int32_t *__restrict__ fill, uint4 *__restrict__ slots)
{
    for (int64_t f = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; f < N; f += (int64_t)gridDim.x * blockDim.x) {
        int s;
        int64_t i;
        species_of(p, S, f, s, i);
        const uint4 r = pos_by_id[s * maxN + i];
        const int64_t c = micro_of(r, M);
        const int k = atomicAdd(&fill[c], 1);
        slots[(int64_t)k * ncm + c] = r;
    }
}

// Orders each cell's entries by (species, index) -- the order of the ids --
// and writes the byte counts.  One thread per cell, at most 15 entries.
__global__ void k_mc_sort(const int32_t *__restrict__ fill, int64_t ncm, uint4 *__restrict__ slots,
                          uint8_t *__restrict__ count)
{
    for (int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; c < ncm; c += (int64_t)gridDim.x * blockDim.x) {
        const int n = fill[c];
        uint4 v[kMicroMaxCap];
        for (int k = 0; k < n; ++k) v[k] = slots[(int64_t)k * ncm + c];
        for (int k = 1; k < n; ++k) {  // insertion sort on (species, index)
            const uint4 x = v[k];
            const uint64_t kx = ((uint64_t)tag_species(x.w) << 32) | tag_index(x.w);
            int j = k - 1;
            while (j >= 0 && (((uint64_t)tag_species(v[j].w) << 32) | tag_index(v[j].w)) > kx) {
                v[j + 1] = v[j];
                --j;
            }
            v[j + 1] = x;
        }
        for (int k = 0; k < n; ++k) slots[(int64_t)k * ncm + c] = v[k];
        count[c] = (uint8_t)n;
    }
}

void micro_free(gcmc_ctx *ctx)
{
    if (ctx->mc_count) cudaFree(ctx->mc_count);
    if (ctx->mc_pos) cudaFree(ctx->mc_pos);
    ctx->mc_count = nullptr;
    ctx->mc_pos = nullptr;
    ctx->mc_valid = false;
}

// The library's limit on the microcells: 4 bits per microcell and 4 bytes per
// cell of the cube around a point, with 1,480 bytes more, are at most what a CTA
// may have of shared memory.  The chain keeps neither there; the limit is the
// one that callers know.
static size_t micro_bytes(int64_t ncm, int nax)
{
    return (size_t)nax * nax * nax * 4 + (size_t)((ncm + 1) / 2 + 15) / 16 * 16 + 1480;
}

gcmc_status micro_build(gcmc_ctx *ctx, double edge, int cap_req)
{
    const double md = std::ceil(ctx->L / edge);
    if (!(md >= 1.0) || md > 1023.0)
        return fail(ctx, GCMC_ERR_INVALID_ARG, "gcmc_build_microcells: more than 1023 microcells per side");
    const int M = (int)md;
    const int64_t ncm = (int64_t)M * M * M;
    const int D = 1 + (int)(((uint64_t)(ctx->rcg - 1) * (uint64_t)M) >> 32);
    if (micro_bytes(ncm, std::min(2 * D + 1, M)) > ctx->smem_optin)
        return fail(ctx, GCMC_ERR_INVALID_ARG,
                    "gcmc_build_microcells: too many microcells (the limit counts 4 bits each and 4 bytes per cell of the cube)");
    SpeciesPrefix p{};
    for (int s = 0; s < ctx->S; ++s) p.first[s + 1] = p.first[s] + ctx->n_host[s];
    for (int s = ctx->S; s < kMaxSpecies; ++s) p.first[s + 1] = p.first[s];
    const int64_t N = p.first[ctx->S];
    gcmc_status st = ensure_scratch(ctx, (size_t)(ncm + 4) * sizeof(int32_t));
    if (st != GCMC_OK) return st;
    int32_t *tmp = (int32_t *)ctx->scratch;
    int32_t *d_max = tmp + ncm;
    GCMC_CUDA(ctx, cudaMemsetAsync(tmp, 0, (size_t)(ncm + 4) * sizeof(int32_t), ctx->stream));
    const int nb = (int)std::max<int64_t>(1, std::min<int64_t>((N + 255) / 256, (int64_t)ctx->num_sms * 8));
    const int nbc = (int)std::max<int64_t>(1, std::min<int64_t>((ncm + 255) / 256, (int64_t)ctx->num_sms * 8));
    if (N > 0)
        k_mc_count<<<nb, 256, 0, ctx->stream>>>(ctx->pos_by_id, ctx->maxN, p, ctx->S, N, (uint32_t)M, tmp);
    k_mc_max<<<nbc, 256, 0, ctx->stream>>>(tmp, ncm, d_max);
    ctx->launches += N > 0 ? 2 : 1;
    GCMC_CUDA(ctx, cudaGetLastError());
    int32_t fullest = 0;
    GCMC_CUDA(ctx, cudaMemcpyAsync(&fullest, d_max, sizeof(int32_t), cudaMemcpyDeviceToHost, ctx->stream));
    GCMC_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
    const int cap = cap_req > 0 ? cap_req : std::max(5, (int)fullest);
    if (fullest > cap || cap > kMicroMaxCap)
        return fail(ctx, GCMC_ERR_CELL_OVERFLOW,
                    "gcmc_build_microcells: a microcell holds " + std::to_string(fullest) + " particles");
    micro_free(ctx);
    GCMC_CUDA(ctx, cudaMalloc(&ctx->mc_count, (size_t)ncm));
    GCMC_CUDA(ctx, cudaMalloc(&ctx->mc_pos, (size_t)cap * ncm * sizeof(uint4)));
    GCMC_CUDA(ctx, cudaMemsetAsync(tmp, 0, (size_t)ncm * sizeof(int32_t), ctx->stream));
    if (N > 0)
        k_mc_place<<<nb, 256, 0, ctx->stream>>>(ctx->pos_by_id, ctx->maxN, p, ctx->S, N, (uint32_t)M, ncm, tmp,
                                                ctx->mc_pos);
    k_mc_sort<<<nbc, 256, 0, ctx->stream>>>(tmp, ncm, ctx->mc_pos, ctx->mc_count);
    ctx->launches += N > 0 ? 2 : 1;
    GCMC_CUDA(ctx, cudaGetLastError());
    GCMC_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
    ctx->mc_edge = edge;
    ctx->mc_cap_req = cap_req;
    ctx->mc_M = M;
    ctx->mc_ncell = ncm;
    ctx->mc_cap = cap;
    ctx->mc_D = D;
    ctx->mc_valid = true;
    return GCMC_OK;
}

// Grows the slots per microcell; the slot-major layout keeps every entry
// at its index, so the old array is the new array's prefix.
gcmc_status micro_grow(gcmc_ctx *ctx, int ncap)
{
    uint4 *np = nullptr;
    GCMC_CUDA(ctx, cudaMalloc(&np, (size_t)ncap * ctx->mc_ncell * sizeof(uint4)));
    GCMC_CUDA(ctx, cudaMemcpyAsync(np, ctx->mc_pos, (size_t)ctx->mc_cap * ctx->mc_ncell * sizeof(uint4),
                                   cudaMemcpyDeviceToDevice, ctx->stream));
    GCMC_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
    cudaFree(ctx->mc_pos);
    ctx->mc_pos = np;
    ctx->mc_cap = ncap;
    return GCMC_OK;
}

}  // namespace gcmc

