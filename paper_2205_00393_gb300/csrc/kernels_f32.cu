// FP32 CUDA-core kernels of libtnc: the permute-fused complex64 contraction
// GEMM, the FP64 final reduction and the FP64 slice sum.
//
// Pairwise contraction (Sec. 2.1.1) in the TTGT arrangement of Sec. 5.3.1
// (free modes of A first, contracted modes last; contracted modes of B first):
// the permutation is folded into the operand load. Each binary mode of an
// operand has an element stride; the address of A(m, k) is the sum of the
// strides of the set bits of m and k. As in the paper's recursion formula
// (Sec. 5.3.1, map[i+k] = map[i] + k*offset) only the tile-local low bits go
// through a table; the high bits of a tile origin contribute one offset.
#include "f32_device.cuh"
#include "kernels.h"

namespace tnc {

namespace {

using namespace f32dev;

template <int NTH, int RM, int WN, int MINB>
__global__ void __launch_bounds__(NTH, MINB) k_gemm_f32(const __grid_constant__ GemmParams p) {
    dep_trigger();
    extern __shared__ __align__(16) uint8_t gemm_dyn[];
    gemm_tile<0, NTH, RM, WN>(p, blockIdx.x, blockIdx.z, p.slice0, *reinterpret_cast<GemmSmemT<NTH, RM, WN>*>(gemm_dyn));
}

template <int NTH, int WN, int CL>
__global__ void __launch_bounds__(NTH, 3) k_gemm_f32_cluster(const __grid_constant__ GemmParams p) {
    dep_trigger();
    extern __shared__ __align__(16) uint8_t gemm_dyn[];
    gemm_tile_cluster<NTH, WN, CL>(p, blockIdx.x / CL, blockIdx.x % CL, blockIdx.z, p.slice0,
                                   *reinterpret_cast<GemmClusterSmem<NTH, WN>*>(gemm_dyn));
}

// Grouped contractions run on 32 x 64 tiles by 128 threads, three CTAs per SM: most
// nodes of a level have a few tiles at most, and the smaller tile shortens the chain
// of each (K = 512, M = 2^8, N = 2^6: 58 us against 74 us on the 64 x 64 tile of 256
// threads). A fourth CTA would take the registers of a tile whose parameters are
// in shared memory below what it needs: a 20-qubit call 162 us instead of 157.
constexpr int GT = 128;
using GroupSmem = GemmSmemT<GT, 4, 2>;

// Parameters of a CTA's contraction, copied to shared memory by the whole CTA: a
// small tile is a chain of dependent loads (its map entry, its parameters, its
// operands), and reading the stride tables from global memory one entry after
// another was the longest part of it, after the binary search over tile
// offsets that the map replaces. The 20-qubit call of 18 such levels went from
// 275 to 237 us, a level of 1 to 100 small contractions from 9.4 to 7.9 us (cold
// caches).
struct GroupCta {
    GroupSmem tile;
    GemmParams p;
};
__device__ __forceinline__ const GemmParams& stage_params(const GemmParams* src, GroupCta& cta) {
    static_assert(sizeof(GemmParams) % 8 == 0, "copied in 8-byte words");
    const uint64_t* from = reinterpret_cast<const uint64_t*>(src);
    uint64_t* to = reinterpret_cast<uint64_t*>(&cta.p);
    for (int i = threadIdx.x; i < (int)(sizeof(GemmParams) / 8); i += GT) to[i] = from[i];
    __syncthreads();
    return cta.p;
}

// Many independent contractions in one launch (nodes of one tree level): CTA
// b serves tile map[b].y of node map[b].x.
__global__ void __launch_bounds__(GT, 3) k_gemm_f32_group(const GemmParams* __restrict__ params,
                                                       const int2* __restrict__ map, int64_t slice0) {
    dep_trigger();
    extern __shared__ __align__(16) uint8_t gemm_dyn[];
    GroupCta& cta = *reinterpret_cast<GroupCta*>(gemm_dyn);
    const int2 nt = map[blockIdx.x];
    gemm_tile<0, GT, 4, 2, true>(stage_params(params + nt.x, cta), nt.y, blockIdx.z, slice0, cta.tile);
}

// FP64 partial sums of a contraction with R = M*N <= 64 outputs.
__global__ void __launch_bounds__(256) k_root_partials(const __grid_constant__ RootParams rp,
                                                       double2* partials) {
    dep_trigger();
    dep_wait();
    __shared__ double2 red[256];
    __shared__ int64_t root_ta[5][256], root_tb[5][256];  // offsets of 8-bit groups of j (K <= 2^40)
    const int R = 1 << (rp.g.mb + rp.g.nb);
    const int z = blockIdx.y;
    root_chunk<0>(rp, blockIdx.x, z, rp.g.slice0, partials + ((int64_t)z * rp.chunks + blockIdx.x) * R, red, root_ta,
                  root_tb);
}

// out[y][r] += sum_i partials[y][i][perm(r)], y = blockIdx.y (a fixed order: accumulate_items)
__global__ void __launch_bounds__(256) k_accumulate_partials(const double2* partials, int count,
                                                             const __grid_constant__ PermParams pp, double2* out) {
    dep_trigger();
    dep_wait();
    __shared__ double2 red[256];
    const int64_t R = 1ll << pp.obits;
    accumulate_items<0>(partials + blockIdx.y * (count * R), count, pp, (int64_t)blockIdx.x * 256, out + blockIdx.y * R, red);
}

// out[y][r] += sum_z src_(y batch + z)[perm(r)] in FP64, z ascending, y = blockIdx.y
__global__ void k_slice_sum_f32(const __grid_constant__ SumParams p, int batch, double2* out) {
    dep_trigger();
    dep_wait();
    const int64_t R = 1ll << p.obits;
    const int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= R) return;
    const int64_t off = bits_offset(r, p.ostride, p.obits, 0);
    double2 acc = make_double2(0.0, 0.0);
    const int64_t z0 = (int64_t)blockIdx.y * batch;
    for (int64_t z = z0; z < z0 + batch; ++z) {
        const float2* src = p.src.ptr + z * p.src.batch_stride + slice_offset(p.src, p.slice0 + z);
        float2 v = src[off];
        acc.x += v.x;
        acc.y += v.y;
    }
    double2* const o = out + blockIdx.y * R + r;
    o->x += acc.x;
    o->y += acc.y;
}

}  // namespace

__global__ void __launch_bounds__(GT, 3) k_gemm_f32_group_multi(const GemmParams* __restrict__ params,
                                                             const int2* __restrict__ map, const int* __restrict__ net,
                                                             const int64_t* __restrict__ rs0,
                                                             const int* __restrict__ rb);

// The grouped FP32 kernels take GroupCta (over 48 KB) as dynamic shared memory;
// the limit is raised once per process (a host-side setting, not a stream
// operation, so it is safe before or during graph capture).
cudaError_t gemm_smem_attr() {
    static cudaError_t done = [] {
        cudaError_t e = cudaFuncSetAttribute(k_gemm_f32_group, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(GroupCta));
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(k_gemm_f32_group_multi, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)sizeof(GroupCta));
        return e;
    }();
    return done;
}

template <int NTH, int RM, int WN, int MINB>
static cudaError_t launch_gemm_f32_tiles(const GemmParams& p, int batch, cudaStream_t s) {
    using Cfg = TileCfg<NTH, RM, WN>;
    using Smem = GemmSmemT<NTH, RM, WN>;
    static const cudaError_t attr = cudaFuncSetAttribute(k_gemm_f32<NTH, RM, WN, MINB>,
                                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(Smem));
    if (attr != cudaSuccess) return attr;
    const int64_t M = 1ll << p.mb, N = 1ll << p.nb;
    const int64_t tiles = ((M + Cfg::BM - 1) / Cfg::BM) * ((N + Cfg::BN - 1) / Cfg::BN);
    if (tiles > 0x7fffffffll || batch < 1 || batch > 65535) return cudaErrorInvalidConfiguration;
    return launch_dependent(k_gemm_f32<NTH, RM, WN, MINB>, dim3((unsigned)tiles, 1, batch), dim3(NTH), sizeof(Smem), s, 1, p);
}

template <int NTH, int WN, int CL>
static cudaError_t launch_gemm_f32_cluster(const GemmParams& p, int batch, cudaStream_t s) {
    using Cfg = TileCfg<NTH, 4, WN>;
    using Smem = GemmClusterSmem<NTH, WN>;
    static const cudaError_t attr = cudaFuncSetAttribute(k_gemm_f32_cluster<NTH, WN, CL>,
                                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(Smem));
    if (attr != cudaSuccess) return attr;
    const int64_t M = 1ll << p.mb, N = 1ll << p.nb;
    const int64_t tiles = ((M + Cfg::BM - 1) / Cfg::BM) * ((N + Cfg::BN - 1) / Cfg::BN);
    if (tiles > 0x7fffffffll / CL || batch < 1 || batch > 65535) return cudaErrorInvalidConfiguration;
    return launch_dependent(k_gemm_f32_cluster<NTH, WN, CL>, dim3((unsigned)(tiles * CL), 1, batch), dim3(NTH), sizeof(Smem),
                            s, CL, p);
}

// Choice of the tile, by the number T of CTAs that 32 x 64 tiles (64 x 32 where
// N <= 32: half of a 64-wide tile would be padding) give, all slices of the
// batch together. Every choice gives the same bits.
//  - few tiles and K >= 128: clusters, whose CTAs share the k groups of one
//    tile. 152 SMs hold 456 such CTAs, and while T is below an SM each, eight
//    per tile fill the chip: (M, N, K) = (2^10, 2^6, 2^14) 285 us against 1217
//    on one CTA per tile, (2^6, 2^6, 2^12) 56 against 313, (2^9, 2^9, 2^9)
//    54 against 60; at T = 256, four: (2^10, 2^9, 2^10) 130 us, against 137 with
//    eight and 140 without. Beyond that clusters lose ((2^10, 2^10, 2^10),
//    T = 512: 237 against 224).
//  - two SMs' worth of tiles or more: 64 x 64 tiles with 8 x 4 outputs per thread,
//    which load fewer bytes per product from shared memory: (2^11, 2^11, 2^11)
//    1364 us (50.4 TFLOP/s, 0.69 of the FFMA rate) against 1480.
//  - otherwise 32 x 64 tiles (K < 128, or narrow outputs): (2^9, 2^9, 2^7) 30 us
//    against 35.
cudaError_t launch_gemm_f32(const GemmParams& p, int batch, cudaStream_t s) {
    const bool narrow = p.nb <= 5;
    const int64_t T = narrow ? (int64_t)batch << (p.mb > 6 ? p.mb - 6 : 0)
                             : (int64_t)batch << ((p.mb > 5 ? p.mb - 5 : 0) + p.nb - 6);
    const int cl = T <= 152 ? (p.kb >= 9 ? 8 : p.kb == 8 ? 4 : p.kb == 7 ? 2 : 1)
                            : T <= 304 ? (p.kb >= 8 ? 4 : p.kb == 7 ? 2 : 1) : 1;
    if (narrow) {
        switch (cl) {
            case 8: return launch_gemm_f32_cluster<128, 1, 8>(p, batch, s);
            case 4: return launch_gemm_f32_cluster<128, 1, 4>(p, batch, s);
            case 2: return launch_gemm_f32_cluster<128, 1, 2>(p, batch, s);
            default: return launch_gemm_f32_tiles<128, 4, 1, 4>(p, batch, s);
        }
    }
    switch (cl) {
        case 8: return launch_gemm_f32_cluster<128, 2, 8>(p, batch, s);
        case 4: return launch_gemm_f32_cluster<128, 2, 4>(p, batch, s);
        case 2: return launch_gemm_f32_cluster<128, 2, 2>(p, batch, s);
        default: break;
    }
    return T > 304 ? launch_gemm_f32_tiles<128, 8, 2, 2>(p, batch, s) : launch_gemm_f32_tiles<128, 4, 2, 4>(p, batch, s);
}

// Grouped contractions of several networks: node i belongs to network
// net[i]; slice z of the launch maps to slice rs0[net] + z of that network and
// exists only for z < rb[net] (networks batch different numbers of slices).
__global__ void __launch_bounds__(GT, 3) k_gemm_f32_group_multi(const GemmParams* __restrict__ params,
                                                             const int2* __restrict__ map, const int* __restrict__ net,
                                                             const int64_t* __restrict__ rs0,
                                                             const int* __restrict__ rb) {
    dep_trigger();
    extern __shared__ __align__(16) uint8_t gemm_dyn[];
    GroupCta& cta = *reinterpret_cast<GroupCta*>(gemm_dyn);
    const int2 nt = map[blockIdx.x];
    const int w = net[nt.x];
    if ((int)blockIdx.z >= rb[w]) {
        dep_wait();
        return;
    }
    gemm_tile<0, GT, 4, 2, true>(stage_params(params + nt.x, cta), nt.y, blockIdx.z, rs0[w], cta.tile);
}

// Root reductions of several networks in one launch: block x serves chunk
// x - blk_off[i] of network i; partial sums go to that network's buffer.
__global__ void __launch_bounds__(256) k_root_partials_multi(const RootParams* __restrict__ roots,
                                                             double2* const* __restrict__ partials,
                                                             const int64_t* __restrict__ blk_off, int n,
                                                             const int64_t* __restrict__ rs0,
                                                             const int* __restrict__ rb) {
    dep_trigger();
    dep_wait();
    __shared__ double2 red[256];
    __shared__ int64_t root_ta[5][256], root_tb[5][256];
    const int64_t x = blockIdx.x;
    int lo = 0, hi = n - 1;
    while (lo < hi) {
        int mid = (lo + hi + 1) >> 1;
        if (blk_off[mid] <= x) lo = mid;
        else hi = mid - 1;
    }
    const int z = blockIdx.z;
    if (z >= rb[lo]) return;
    const RootParams& rp = roots[lo];
    const int chunk = (int)(x - blk_off[lo]);
    const int R = 1 << (rp.g.mb + rp.g.nb);
    root_chunk<0>(rp, chunk, z, rs0[lo], partials[lo] + ((int64_t)z * rp.chunks + chunk) * R, red, root_ta, root_tb);
}

// out_i[r] += sum over network i's partial sums (slices in order, then chunks; as
// accumulate_items adds them), one block per network.
__global__ void __launch_bounds__(256) k_accumulate_multi(const RootParams* __restrict__ roots,
                                                          double2* const* __restrict__ partials,
                                                          const PermParams* __restrict__ perms,
                                                          double2* const* __restrict__ outs, const int* __restrict__ rb) {
    dep_trigger();
    dep_wait();
    __shared__ double2 red[256];
    const int i = blockIdx.x;
    const PermParams& pp = perms[i];
    const int count = rb[i] * roots[i].chunks;
    const int64_t items = (int64_t)acc_lanes(count) << pp.obits;
    for (int64_t it = 0; it < items; it += 256) accumulate_items<0>(partials[i], count, pp, it, outs[i], red);
}

bool gemm_f32_long(int kb) { return kb >= 8; }

int64_t gemm_f32_group_tiles(int mb, int nb) {
    using Cfg = TileCfg<GT, 4, 2>;
    return (((1ll << mb) + Cfg::BM - 1) / Cfg::BM) * (((1ll << nb) + Cfg::BN - 1) / Cfg::BN);
}

int64_t gemm_f32_tiles(int mb, int nb) {
    int64_t M = 1ll << mb, N = 1ll << nb;
    return ((M + 63) / 64) * ((N + 63) / 64);
}

cudaError_t launch_gemm_f32_group(const GemmParams* d_params, const int2* d_map, int64_t total_tiles, int64_t slice0,
                                  int batch, cudaStream_t s) {
    if (total_tiles < 1 || total_tiles > 0x7fffffffll || batch < 1 || batch > 65535) return cudaErrorInvalidConfiguration;
    cudaError_t e = gemm_smem_attr();
    if (e != cudaSuccess) return e;
    return launch_dependent(k_gemm_f32_group, dim3((unsigned)total_tiles, 1, batch), dim3(GT), sizeof(GroupCta), s, 1, d_params,
                            d_map, slice0);
}

cudaError_t launch_gemm_f32_group_multi(const GemmParams* d_params, const int2* d_map, int64_t total_tiles,
                                        const int* d_net, const int64_t* d_rs0, const int* d_rb, int max_batch,
                                        cudaStream_t s) {
    if (total_tiles < 1 || total_tiles > 0x7fffffffll || max_batch < 1 || max_batch > 65535)
        return cudaErrorInvalidConfiguration;
    cudaError_t e = gemm_smem_attr();
    if (e != cudaSuccess) return e;
    return launch_dependent(k_gemm_f32_group_multi, dim3((unsigned)total_tiles, 1, max_batch), dim3(GT), sizeof(GroupCta), s, 1,
                            d_params, d_map, d_net, d_rs0, d_rb);
}

cudaError_t launch_root_multi(const RootParams* d_roots, double2* const* d_partials, const int64_t* d_blk_off,
                              int n, int64_t total_blocks, const PermParams* d_perms, double2* const* d_outs,
                              const int64_t* d_rs0, const int* d_rb, int max_batch, cudaStream_t s) {
    if (n < 1 || total_blocks < 1 || total_blocks > 0x7fffffffll || max_batch < 1 || max_batch > 65535)
        return cudaErrorInvalidConfiguration;
    cudaError_t e = launch_dependent(k_root_partials_multi, dim3((unsigned)total_blocks, 1, max_batch), dim3(256), 0, s, 1, d_roots,
                                     d_partials, d_blk_off, n, d_rs0, d_rb);
    if (e != cudaSuccess) return e;
    return launch_dependent(k_accumulate_multi, dim3(n), dim3(256), 0, s, 1, d_roots, d_partials, d_perms, d_outs, d_rb);
}

cudaError_t launch_root_partials(const RootParams& p, int batch, double2* partials, cudaStream_t s) {
    if (p.g.mb + p.g.nb > 6 || batch < 1 || batch > 65535) return cudaErrorInvalidConfiguration;
    return launch_dependent(k_root_partials, dim3(p.chunks, batch), dim3(256), 0, s, 1, p, partials);
}

cudaError_t launch_accumulate_partials(const double2* partials, int count, const PermParams& pp,
                                       double2* out, cudaStream_t s, int groups) {
    const int64_t items = (int64_t)acc_lanes(count) << pp.obits;
    return launch_dependent(k_accumulate_partials, dim3((unsigned)((items + 255) / 256), groups), dim3(256), 0, s, 1, partials,
                            count, pp, out);
}

cudaError_t launch_slice_sum_f32(const SumParams& p, int batch, double2* out, cudaStream_t s, int groups) {
    int64_t R = 1ll << p.obits;
    return launch_dependent(k_slice_sum_f32, dim3((unsigned)((R + 255) / 256), groups), dim3(256), 0, s, 1, p, batch, out);
}

}  // namespace tnc
