// A whole slice in one CTA, for networks whose tensors all fit in shared memory.
//
// A call of tiny contractions is bound by dependencies: 20 tree levels of a few
// hundred multiply-accumulates each. As launches a level costs several
// microseconds, as tasks of the persistent executor about four (ticket,
// descriptor, counters, parameters and operands are dependent trips to L2). Here
// the leaves, every intermediate and the tables of the plan sit in shared
// memory, a CTA computes the slice-invariant contractions and then its slices,
// and a level costs one barrier. Every output is the same sum in the same order
// as in the FP32 tile and in the final contraction's chunk.
// Measured (12-qubit call, 16 slices, 2^13.4 multiply-accumulates each): 76 us
// persistent, 64 as launches, 19 this way; 13 bitstrings of a 12-qubit circuit 28 us
// instead of 534. What is left is the host's part of a call (two launches), the copy
// of the tables and about 0.5 us a level.
#include "f32_device.cuh"
#include "kernels.h"
#include "launch.cuh"

namespace tnc {

namespace {

using namespace f32dev;

constexpr int TT = kTinyThreads;

// One output element of one contraction: 64-term FP32 partials added with TwoSum
// (gemm_tile's arithmetic).
__device__ __forceinline__ float2 tiny_element(const float2* A, const float2* B, const uint32_t* kt, int K) {
    float2 acc = make_float2(0.f, 0.f), comp = make_float2(0.f, 0.f);
    for (int k0 = 0; k0 < K; k0 += 64) {
        const int ke = k0 + 64 < K ? k0 + 64 : K;
        float2 part = make_float2(0.f, 0.f);
#pragma unroll 4
        for (int k = k0; k < ke; ++k) {
            const uint32_t o = kt[k];
            const float2 a = A[o & 0xFFFFu], b = B[o >> 16];
            part.x = fmaf(a.x, b.x, part.x);
            part.x = fmaf(-a.y, b.y, part.x);
            part.y = fmaf(a.x, b.y, part.y);
            part.y = fmaf(a.y, b.x, part.y);
        }
        float s = acc.x + part.x, v = s - acc.x;
        comp.x += (acc.x - (s - v)) + (part.x - v);
        acc.x = s;
        s = acc.y + part.y;
        v = s - acc.y;
        comp.y += (acc.y - (s - v)) + (part.y - v);
        acc.y = s;
    }
    return make_float2(acc.x + comp.x, acc.y + comp.y);
}

__global__ void __launch_bounds__(TT) k_tiny(const __grid_constant__ TinyParams p) {
    extern __shared__ __align__(16) uint8_t tiny_smem[];
    double2* const red = reinterpret_cast<double2*>(tiny_smem);
    float2* const data = reinterpret_cast<float2*>(red + 256);
    uint32_t* const W = reinterpret_cast<uint32_t*>(data + p.data_elems);
    const int tid = threadIdx.x;
    for (int i = tid; i < p.words / 4; i += TT) reinterpret_cast<uint4*>(W)[i] = reinterpret_cast<const uint4*>(p.tables)[i];
    for (int i = tid; i < p.leaf_elems; i += TT) data[i] = p.leaves[i];
    if (p.clear)
        for (int64_t i = (int64_t)blockIdx.x * TT + tid; i < p.groups << p.obits; i += (int64_t)gridDim.x * TT)
            p.out[i] = make_double2(0.0, 0.0);  // k_tiny_sum adds into it
    if (blockIdx.x == 0 && tid == 0) *p.err = 0;
    __syncthreads();
    uint32_t* const base = W + p.o_base;  // element offset of every tensor in data
    auto level = [&](int l) {
        const uint32_t* L = W + p.o_levels + 2 * l;  // items, first word of its map
        const uint32_t items = L[0];
        const uint16_t* map = reinterpret_cast<const uint16_t*>(W + L[1]);
        for (uint32_t it = tid; it < items; it += TT) {
            const uint32_t* op = W + p.o_ops + kTinyOpWords * map[it >> 2];
            const uint32_t bits = op[3], e = it - op[7];
            const int mb = bits & 0xFF, nb = (bits >> 8) & 0xFF, kb = bits >> 16;
            if (e >> (mb + nb)) continue;  // padding to four items
            const float2* A = data + base[op[0]] + W[op[4] + (e >> nb)];
            const float2* B = data + base[op[1]] + W[op[5] + (e & ((1u << nb) - 1u))];
            data[op[2] + e] = tiny_element(A, B, W + op[6], 1 << kb);
        }
        __syncthreads();
    };
    for (int l = 0; l < p.inv_levels; ++l) level(l);
    for (int64_t i = blockIdx.x; i < p.per * p.groups; i += gridDim.x) {
        const int64_t id = p.first + (i / p.per) * p.stride + i % p.per;  // slice id: variant, then slice
        const int64_t v = p.sbits < 62 ? id >> p.sbits : 0;
        if (tid < p.n_sliced) {  // leaves with sliced modes: where this slice's values begin
            const uint32_t* sl = W + p.o_sliced + 3 * tid;  // leaf, first entry, entries
            uint32_t off = W[p.o_static + sl[0]];
            for (uint32_t q = 0; q < sl[2]; ++q) {
                const uint32_t* en = W + sl[1] + 2 * q;  // slice bit, stride
                if ((id >> en[0]) & 1) off += en[1];
            }
            base[sl[0]] = off;
        }
        for (int q = tid; q < p.n_var; q += TT) {  // elements of variant leaves
            const uint32_t* en = W + p.o_var + 3 * q;  // place in the variant buffer, place in data, leaf elements
            data[en[1]] = p.variants[(int64_t)en[0] + v * en[2]];
        }
        __syncthreads();
        for (int l = p.inv_levels; l < p.levels; ++l) level(l);
        // final contraction: root_chunk's sums (one chunk)
        const uint32_t* op = W + p.o_root;
        const uint32_t bits = op[3];
        const int mb = bits & 0xFF, nb = (bits >> 8) & 0xFF, K = 1 << (bits >> 16);
        const int R = 1 << (mb + nb), lanes = 256 / R, r = tid / lanes, lane = tid % lanes;
        if (tid < 256) {
            const float2* A = data + base[op[0]] + W[op[4] + (r >> nb)];
            const float2* B = data + base[op[1]] + W[op[5] + (r & ((1 << nb) - 1))];
            const uint32_t* kt = W + op[6];
            double re = 0.0, im = 0.0;
            if (K >= lanes) {
                const int nj = K / lanes;
                for (int j0 = 0; j0 < nj; j0 += 16) {
                    float sr = 0.f, si = 0.f;
                    for (int j = j0; j < j0 + 16 && j < nj; ++j) {
                        const uint32_t o = kt[lanes * j + lane];
                        const float2 a = A[o & 0xFFFFu], b = B[o >> 16];
                        sr = fmaf(a.x, b.x, sr);
                        sr = fmaf(-a.y, b.y, sr);
                        si = fmaf(a.x, b.y, si);
                        si = fmaf(a.y, b.x, si);
                    }
                    re += sr;
                    im += si;
                }
            } else {
                for (int k = lane; k < K; k += lanes) {
                    const uint32_t o = kt[k];
                    const float2 a = A[o & 0xFFFFu], b = B[o >> 16];
                    re += (double)a.x * b.x - (double)a.y * b.y;
                    im += (double)a.x * b.y + (double)a.y * b.x;
                }
            }
            red[tid] = make_double2(re, im);
        }
        __syncthreads();
        for (int st = lanes / 2; st > 0; st >>= 1) {
            if (tid < 256 && lane < st) {
                const double2 o = red[tid + st];
                red[tid].x += o.x;
                red[tid].y += o.y;
            }
            __syncthreads();
        }
        if (tid < 256 && lane == 0) p.partials[i * R + r] = red[tid];
        __syncthreads();
    }
}

// (after k_tiny) out[g][r] += the ordered FP64 sum of group g's partials
__global__ void __launch_bounds__(256) k_tiny_sum(const double2* partials, int count, const __grid_constant__ PermParams pp,
                                                  double2* out) {
    __shared__ double2 red[256];
    dep_wait();
    const int64_t R = 1ll << pp.obits;
    accumulate_items<0>(partials + blockIdx.x * (count * R), count, pp, 256ll * blockIdx.y, out + blockIdx.x * R, red);
}

}  // namespace

size_t tiny_smem_bytes(int64_t data_elems, int64_t words) { return 256 * sizeof(double2) + data_elems * 8 + words * 4; }

cudaError_t launch_tiny(const TinyParams& p, const PermParams& pp, cudaStream_t s) {
    const size_t smem = tiny_smem_bytes(p.data_elems, p.words);
    if (p.per < 1 || p.groups < 1 || p.groups > 0x7fffffffll || p.per > 0x7fffffffll || smem > kTinySmem || p.words % 4 ||
        p.data_elems % 2)
        return cudaErrorInvalidValue;
    static const cudaError_t attr = cudaFuncSetAttribute(k_tiny, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTinySmem);
    if (attr != cudaSuccess) return attr;
    // a CTA of its own per slice while they fit at once, then several slices per CTA (the
    // slice-invariant contractions are computed once per CTA)
    const int64_t per_sm = std::max<int64_t>(1, std::min<int64_t>(2048 / TT, (int64_t)(220 * 1024 / (smem + 1024))));
    const int64_t ctas = std::min<int64_t>(p.per * p.groups, 152 * per_sm);
    k_tiny<<<(unsigned)ctas, TT, smem, s>>>(p);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const int64_t sum_blocks = (((int64_t)acc_lanes((int)p.per) << pp.obits) + 255) / 256;
    return launch_dependent(k_tiny_sum, dim3((unsigned)p.groups, (unsigned)sum_blocks), dim3(256), 0, s, 1, p.partials, (int)p.per, pp, p.out);
}

}  // namespace tnc
