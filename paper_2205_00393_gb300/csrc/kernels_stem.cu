// Fused multi-step stem kernel: the GPU form of the paper's secondary slicing
// (Sec. 5.2, Fig. 8-9). A stem tensor that absorbs small branch tensors in n
// consecutive narrow contractions is read from HBM once and written once:
// the modes that live through all n steps (the paper slices exactly these,
// picking them by lifetime) index independent sub-tensors, one per CTA; each
// CTA keeps its sub-tensor in shared memory across the n absorptions. Every
// contraction is the same complex product as on the FP32 path (products and
// sums in FP32), so a fused group gives what its n separate launches give up
// to the order of the additions within one output element.
#include <type_traits>

#include "kernels.h"
#include "launch.cuh"

namespace tnc {

namespace {

constexpr int NT = 256;

__device__ __forceinline__ int64_t slice_offset(const Operand& op, int64_t s) {
    int64_t off = 0;
    for (int j = 0; j < op.n_sl; ++j) off += ((s >> op.sl_bit[j]) & 1) * op.sl_stride[j];
    return off;
}

template <typename T>
__device__ __forceinline__ T bits_dec(uint32_t x, const T* str, int nbits) {
    T off = 0;
    for (int b = 0; b < nbits; ++b)
        if ((x >> b) & 1u) off += str[b];
    return off;
}

__device__ __forceinline__ void cmac(float2& acc, float2 a, float2 b) {
    acc.x = fmaf(a.x, b.x, acc.x);
    acc.x = fmaf(-a.y, b.y, acc.x);
    acc.y = fmaf(a.x, b.y, acc.y);
    acc.y = fmaf(a.y, b.x, acc.y);
}

// x with a zero bit inserted at each of the first nk positions of ins (ascending)
__device__ __forceinline__ uint32_t deposit(uint32_t x, const int* ins, int nk) {
#pragma unroll
    for (int t = 0; t < 4; ++t)
        if (t < nk) x = ((x >> ins[t]) << (ins[t] + 1)) | (x & ((1u << ins[t]) - 1u));
    return x;
}

// In-place step with K = N = 2^NK: every thread takes two rows per iteration
// (two independent FMA chains), loads their K elements, and writes the K
// results back to the same positions.
template <int NK>
__device__ __forceinline__ void inplace_step(float2* cur, const float2* bd, const int* ins, const int* kx, int rows,
                                             int tid) {
    constexpr int K = 1 << NK;
    // rows r0 + tid and r0 + NT + tid: consecutive lanes take consecutive rows
    for (int r0 = 0; r0 < rows; r0 += 2 * NT) {
        const bool two = r0 + NT + tid < rows;
        if (r0 + tid >= rows) break;
        uint32_t base[2];
        float2 x[2][K];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            base[h] = deposit((uint32_t)(r0 + h * NT + tid), ins, NK);
#pragma unroll
            for (int k = 0; k < K; ++k) x[h][k] = (h == 0 || two) ? cur[base[h] + kx[k]] : make_float2(0.f, 0.f);
        }
#pragma unroll
        for (int n = 0; n < K; ++n) {
            float2 acc[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
#pragma unroll
            for (int k = 0; k < K; ++k) {
                const float2 b = bd[k * K + n];
                cmac(acc[0], x[0][k], b);
                cmac(acc[1], x[1][k], b);
            }
            cur[base[0] + kx[n]] = acc[0];
            if (two) cur[base[1] + kx[n]] = acc[1];
        }
    }
}

// One CTA per outer assignment (blockIdx.x) and slice of the batch (blockIdx.z).
// Shared memory: one or two buffers of 2^cap_log2 complex elements (X_{i-1},
// X_i) and the dense [K][N] copies of every step's branch.
__global__ void __launch_bounds__(NT, 4) k_stem_fused(const StemParams* __restrict__ P, int cap_log2,
                                                   int64_t slice0) {
    dep_wait();
    extern __shared__ float2 stem_smem[];
    const StemParams& p = *P;
    float2* cur = stem_smem;
    float2* nxt = stem_smem + (1 << cap_log2);
    float2* bsm = stem_smem + ((p.two_buffers ? 2 : 1) << cap_log2);
    const int z = blockIdx.z, tid = threadIdx.x;
    const int64_t s = slice0 + z;
    const uint32_t u = blockIdx.x;
    // dense [k][n] copies of the branches of this slice
    for (int i = 0; i < p.nsteps; ++i) {
        const StemStep& st = p.steps[i];
        const int N = 1 << st.nn, KN = 1 << (st.nk + st.nn);
        const float2* bp = st.br.ptr + z * st.br.batch_stride + slice_offset(st.br, s);
        for (int e = tid; e < KN; e += NT)
            bsm[st.b_off + e] = bp[bits_dec((uint32_t)(e >> st.nn), st.kstr_b, st.nk) +
                                   bits_dec((uint32_t)(e & (N - 1)), st.nstr_b, st.nn)];
    }
    // the sub-tensor X_0 of T_0 at this outer assignment
    int64_t ib = 0, ob = 0;
    for (int b = 0; b < p.nu; ++b)
        if ((u >> b) & 1u) {
            ib += p.ustr_in[b];
            ob += p.ustr_out[b];
        }
    const float2* src = p.in.ptr + z * p.in.batch_stride + slice_offset(p.in, s) + ib;
    {
        // element e = tid + NT * j: the low 8 bits are this thread's, decoded
        // once; every element goes straight to shared memory as an 8-byte
        // asynchronous copy, all of them in flight before the wait
        const int n_in = p.n_in, lo_bits = n_in < 8 ? n_in : 8;
        const int64_t lo = bits_dec((uint32_t)tid, p.istr, lo_bits);
        const int cnt = (1 << n_in) > NT ? (1 << n_in) / NT : 1;
        if (tid < (1 << n_in))
            for (int j = 0; j < cnt; ++j) {
                const uint32_t dst = static_cast<uint32_t>(__cvta_generic_to_shared(cur + tid + NT * j));
                const float2* g = src + lo + bits_dec((uint32_t)j, p.istr + 8, n_in - lo_bits);
                asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(dst), "l"(g) : "memory");
            }
        asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;" ::: "memory");
    }
    __syncthreads();
    for (int i = 0; i < p.nsteps; ++i) {
        const StemStep& st = p.steps[i];
        const int nk = st.nk, K = 1 << nk, N = 1 << st.nn, rows = 1 << st.nr;
        int kx[16];
#pragma unroll
        for (int k = 0; k < 16; ++k) kx[k] = k < K ? bits_dec((uint32_t)k, st.kstr_x, nk) : 0;
        const float2* bd = bsm + st.b_off;
        if (st.inplace && (nk == 1 || nk == 2) && rows >= 2) {
            int ins[4];
#pragma unroll
            for (int t = 0; t < 4; ++t) ins[t] = t < nk ? st.ins[t] : 0;
            if (nk == 1) inplace_step<1>(cur, bd, ins, kx, rows, tid);
            else inplace_step<2>(cur, bd, ins, kx, rows, tid);
            __syncthreads();
        } else if (st.inplace) {
            // rows r: the bits of X outside the contracted positions; a zero
            // is inserted at each contracted position, ascending
            int ins[4];
#pragma unroll
            for (int t = 0; t < 4; ++t) ins[t] = t < nk ? st.ins[t] : 0;
            for (int r = tid; r < rows; r += NT) {
                uint32_t base = (uint32_t)r;
#pragma unroll
                for (int t = 0; t < 4; ++t)
                    if (t < nk) base = ((base >> ins[t]) << (ins[t] + 1)) | (base & ((1u << ins[t]) - 1u));
                float2 xk[16];
#pragma unroll
                for (int k = 0; k < 16; ++k) xk[k] = k < K ? cur[base + kx[k]] : make_float2(0.f, 0.f);
#pragma unroll
                for (int n = 0; n < 16; ++n) {
                    if (n >= K) break;
                    float2 acc = make_float2(0.f, 0.f);
#pragma unroll
                    for (int k = 0; k < 16; ++k)
                        if (k < K) cmac(acc, xk[k], bd[k * K + n]);
                    cur[base + kx[n]] = acc;
                }
            }
            __syncthreads();
        } else {
            int rstr[kStemMaxInner];
#pragma unroll
            for (int b = 0; b < kStemMaxInner; ++b) rstr[b] = b < st.nr ? st.rstr[b] : 0;
            for (int r = tid; r < rows; r += NT) {
                int xo = 0;
#pragma unroll
                for (int b = 0; b < kStemMaxInner; ++b)
                    if ((r >> b) & 1) xo += rstr[b];
                float2 xk[16];
#pragma unroll
                for (int k = 0; k < 16; ++k) xk[k] = k < K ? cur[xo + kx[k]] : make_float2(0.f, 0.f);
                for (int n = 0; n < N; ++n) {
                    float2 acc = make_float2(0.f, 0.f);
#pragma unroll
                    for (int k = 0; k < 16; ++k)
                        if (k < K) cmac(acc, xk[k], bd[k * N + n]);
                    nxt[r * N + n] = acc;
                }
            }
            __syncthreads();
            float2* t = cur;
            cur = nxt;
            nxt = t;
        }
    }
    float2* dst = p.out + z * p.out_batch_stride + ob;
    {
        const int n_out = p.n_out, lo_bits = n_out < 8 ? n_out : 8;
        const int64_t lo = bits_dec((uint32_t)tid, p.ostr, lo_bits);
        const int cnt = (1 << n_out) > NT ? (1 << n_out) / NT : 1;
        if (tid < (1 << n_out))
            for (int j = 0; j < cnt; ++j)
                dst[lo + bits_dec((uint32_t)j, p.ostr + 8, n_out - lo_bits)] = cur[tid + NT * j];
    }
}

// ------------------------------------------------------ groups in registers
//
// What bounds a group of gates: per element and one-mode gate 8 FMAs (two-mode:
// 16), in all about as long as reading and writing the stem once. k_stem_fused
// spends most of its time elsewhere: every step moves the sub-tensor through
// shared memory and loads the gate's matrix once per row. Here a thread keeps
// 32 elements in registers for all steps of a pass (the five register positions
// cover the modes of typically four to seven steps, so a group takes two or
// three passes) and the matrix in registers for a whole step. The first pass
// loads from global memory and the last stores to it; shared memory carries the
// sub-tensor between passes only, XOR-swizzled so that whichever positions a
// pass holds in registers, its lanes' positions fall into distinct banks.
// Every output is the same sum in the same order as in k_stem_fused.
// Measured on the 28-qubit stem path (2 GiB stem, FP32): 220 ms per call with
// k_stem_fused alone, 75 ms with this kernel, 2.7-3.1 TB/s per launch of 7 to 9
// gates; the FMA pipe is then busy 32-36% of the time and the issue slots 53%.

// bank columns: bit p of a position index adds kBankCol[p] to the low four bits of
// the shared-memory slot (identity below 16). Any 8 of the 13 columns span all
// 16 banks (each linear functional is nonzero on at least six of them).
constexpr int kBankCol[kStemRegMaxN] = {1, 2, 4, 8, 13, 11, 7, 14, 5, 3, 6, 10, 12};
constexpr uint32_t slot_bit(int p) { return p < 4 ? 1u << p : (1u << p) | (uint32_t)kBankCol[p]; }
constexpr int RE = 1 << kStemRegBits;  // elements a thread holds

// (x0, x1) <- one-mode gate of (x0, x1): each output is the FMA chain of cmac, x0's
// products first. The last FMA of every output comes after the other inputs'
// last use, so the results can take the inputs' registers.
__device__ __forceinline__ void butterfly1(float2& x0, float2& x1, const float2 (&b)[4]) {
    asm volatile(
        "{\n.reg .f32 t0, t1, t2, t3, n0, n1;\n"
        "neg.f32 n0, %1;\nneg.f32 n1, %3;\n"
        "mul.rn.f32 t0, %0, %4;\nmul.rn.f32 t1, %0, %5;\nmul.rn.f32 t2, %0, %6;\nmul.rn.f32 t3, %0, %7;\n"
        "fma.rn.f32 t0, n0, %5, t0;\nfma.rn.f32 t1, %1, %4, t1;\nfma.rn.f32 t2, n0, %7, t2;\nfma.rn.f32 t3, %1, %6, t3;\n"
        "fma.rn.f32 t0, %2, %8, t0;\nfma.rn.f32 t1, %2, %9, t1;\nfma.rn.f32 t2, %2, %10, t2;\nfma.rn.f32 t3, %2, %11, t3;\n"
        "fma.rn.f32 %0, n1, %9, t0;\nfma.rn.f32 %1, %3, %8, t1;\nfma.rn.f32 %2, n1, %11, t2;\nfma.rn.f32 %3, %3, %10, t3;\n}\n"
        : "+f"(x0.x), "+f"(x0.y), "+f"(x1.x), "+f"(x1.y)
        : "f"(b[0].x), "f"(b[0].y), "f"(b[1].x), "f"(b[1].y), "f"(b[2].x), "f"(b[2].y), "f"(b[3].x), "f"(b[3].y));
}

// one-mode gate on register bit A: b[k * 2 + n]
template <int A>
__device__ __forceinline__ void reg_gate1(float2 (&x)[RE], const float2* bd) {
    float2 b[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) b[e] = bd[e];
#pragma unroll
    for (int r = 0; r < RE; ++r)
        if (!(r >> A & 1)) butterfly1(x[r], x[r | 1 << A], b);
}

// projection of register bit A: b[k]; the result keeps the places where the bit is 0
template <int A>
__device__ __forceinline__ void reg_project(float2 (&x)[RE], const float2* bd) {
    const float2 b0 = bd[0], b1 = bd[1];
#pragma unroll
    for (int r = 0; r < RE; ++r) {
        if (r >> A & 1) continue;
        float2 acc = make_float2(0.f, 0.f);
        cmac(acc, x[r], b0);
        cmac(acc, x[r | 1 << A], b1);
        x[r] = acc;
    }
}

// two-mode gate on register bits A, A + 1 (k, n bit 0 at A): b[k * 4 + n]
template <int A>
__device__ __forceinline__ void reg_gate2(float2 (&x)[RE], const float2* bd) {
    float2 b[16];
#pragma unroll
    for (int e = 0; e < 16; ++e) b[e] = bd[e];
#pragma unroll
    for (int r = 0; r < RE; ++r) {
        if (r >> A & 3) continue;
        float2 xk[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) xk[k] = x[r | k << A];
#pragma unroll
        for (int n = 0; n < 4; ++n) {
            float2 acc = make_float2(0.f, 0.f);
#pragma unroll
            for (int k = 0; k < 4; ++k) cmac(acc, xk[k], b[k * 4 + n]);
            x[r | n << A] = acc;
        }
    }
}

// one mode becomes two: register bits A (contracted, then n bit 0) and A + 1 (n bit 1): b[k * 4 + n]
template <int A>
__device__ __forceinline__ void reg_grow1(float2 (&x)[RE], const float2* bd) {
    float2 b[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) b[e] = bd[e];
#pragma unroll
    for (int r = 0; r < RE; ++r) {
        if (r >> A & 3) continue;
        const float2 x0 = x[r], x1 = x[r | 1 << A];
#pragma unroll
        for (int n = 0; n < 4; ++n) {
            float2 acc = make_float2(0.f, 0.f);
            cmac(acc, x0, b[n]);
            cmac(acc, x1, b[4 + n]);
            x[r | n << A] = acc;
        }
    }
}

// two modes are added at register bits A, A + 1: b[n]
template <int A>
__device__ __forceinline__ void reg_grow0(float2 (&x)[RE], const float2* bd) {
    float2 b[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) b[e] = bd[e];
#pragma unroll
    for (int r = 0; r < RE; ++r) {
        if (r >> A & 3) continue;
        const float2 x0 = x[r];
#pragma unroll
        for (int n = 0; n < 4; ++n) {
            float2 acc = make_float2(0.f, 0.f);
            cmac(acc, x0, b[n]);
            x[r | n << A] = acc;
        }
    }
}

// f(r, address of the thread's element r) for all r without a bit of `skip`:
// the addresses follow a Gray code, one addition (op +-, or ^ for slots) each.
template <typename Addr, typename F>
__device__ __forceinline__ void reg_walk(Addr at, const Addr (&st)[kStemRegBits], int skip, F f) {
    auto walk = [&](auto masked) {
        Addr a = at;
#pragma unroll
        for (int i = 0; i < RE; ++i) {
            const int r = i ^ (i >> 1);
            if (i > 0) {
                int bit = 0;
#pragma unroll
                for (int t = kStemRegBits - 1; t >= 0; --t)
                    if (i >> t & 1) bit = t;
                if constexpr (sizeof(Addr) == 4) a ^= st[bit];
                else a = (r >> bit & 1) ? a + st[bit] : a - st[bit];
            }
            if (!decltype(masked)::value || !(r & skip)) f(r, a);
        }
    };
    if (skip) walk(std::true_type{});
    else walk(std::false_type{});
}

// One CTA of 2^(n - 5) threads (at least a warp) per outer assignment
// (blockIdx.x) and slice of the batch (blockIdx.z).
template <int NTH>
__global__ void __launch_bounds__(NTH, 512 / NTH) k_stem_reg(const __grid_constant__ StemRegParams p,
                                                                  const StemRegBranches* __restrict__ branches,
                                                                  int64_t slice0) {
    extern __shared__ float2 stem_smem[];
    float2* const bsm = stem_smem + (1 << p.n);
    const int z = blockIdx.z, tid = threadIdx.x;
    const int64_t s = slice0 + z;
    const uint32_t u = blockIdx.x;
    int64_t ib = 0, ob = 0;
    for (int b = 0; b < p.nu; ++b)
        if ((u >> b) & 1u) {
            ib += p.ustr_in[b];
            ob += p.ustr_out[b];
        }
    dep_wait();
    float2 x[RE];
    for (int q = 0; q < p.npass; ++q) {
        const StemRegPass& ps = p.pass[q];
        const bool active = tid < (1 << ps.nt);
        uint32_t slot = 0, sr[kStemRegBits];  // in bytes
#pragma unroll
        for (int t = 0; t < kStemRegMaxN - kStemRegBits; ++t) slot ^= (tid >> t & 1) ? ps.tslot[t] : 0;
        char* const sb = reinterpret_cast<char*>(stem_smem);
#pragma unroll
        for (int a = 0; a < kStemRegBits; ++a) sr[a] = ps.rslot[a];
        if (q == 0) {
            if (active) {
                uint64_t g = reinterpret_cast<uint64_t>(p.in.ptr + z * p.in.batch_stride + slice_offset(p.in, s) + ib);
                uint64_t st[kStemRegBits];
#pragma unroll
                for (int t = 0; t < kStemRegMaxN - kStemRegBits; ++t) g += (tid >> t & 1) ? p.tstr_in[t] : 0;
#pragma unroll
                for (int a = 0; a < kStemRegBits; ++a) st[a] = p.rstr_in[a];
                reg_walk(g, st, ps.unborn,
                         [&](int r, uint64_t a) { x[r] = *reinterpret_cast<const float2*>(a); });
            }
            // dense copies of this slice's branches, while the loads are in flight
            for (int e = tid; e < p.nentries; e += NTH) {
                const int2 en = branches->entry[e];
                const Operand& op = branches->br[en.x];
                bsm[e] = op.ptr[z * op.batch_stride + slice_offset(op, s) + en.y];
            }
            __syncthreads();
        } else if (active) {
            reg_walk(slot, sr, ps.unborn, [&](int r, uint32_t a) { x[r] = *reinterpret_cast<const float2*>(sb + a); });
        }
        if (active)
            for (int i = ps.step0; i < ps.step1; ++i) {
                const StemRegStep st = p.step[i];
                const float2* bd = bsm + st.b_off;
                switch (st.kind * 8 + st.reg) {
                    case SR_GATE1 * 8 + 0: reg_gate1<0>(x, bd); break;
                    case SR_GATE1 * 8 + 1: reg_gate1<1>(x, bd); break;
                    case SR_GATE1 * 8 + 2: reg_gate1<2>(x, bd); break;
                    case SR_GATE1 * 8 + 3: reg_gate1<3>(x, bd); break;
                    case SR_GATE1 * 8 + 4: reg_gate1<4>(x, bd); break;
                    case SR_PROJECT * 8 + 0: reg_project<0>(x, bd); break;
                    case SR_PROJECT * 8 + 1: reg_project<1>(x, bd); break;
                    case SR_PROJECT * 8 + 2: reg_project<2>(x, bd); break;
                    case SR_PROJECT * 8 + 3: reg_project<3>(x, bd); break;
                    case SR_PROJECT * 8 + 4: reg_project<4>(x, bd); break;
                    case SR_GROW1 * 8 + 0: reg_grow1<0>(x, bd); break;
                    case SR_GROW1 * 8 + 1: reg_grow1<2>(x, bd); break;
                    case SR_GROW0 * 8 + 0: reg_grow0<0>(x, bd); break;
                    case SR_GROW0 * 8 + 1: reg_grow0<2>(x, bd); break;
                    case SR_GATE2 * 8 + 0: reg_gate2<0>(x, bd); break;
                    default: reg_gate2<2>(x, bd); break;
                }
            }
        if (q + 1 < p.npass) {
            if (active) reg_walk(slot, sr, ps.dead, [&](int r, uint32_t a) { *reinterpret_cast<float2*>(sb + a) = x[r]; });
            __syncthreads();
        } else if (active) {
            uint64_t g = reinterpret_cast<uint64_t>(p.out + z * p.out_batch_stride + ob);
            uint64_t st[kStemRegBits];
#pragma unroll
            for (int t = 0; t < kStemRegMaxN - kStemRegBits; ++t) g += (tid >> t & 1) ? p.tstr_out[t] : 0;
#pragma unroll
            for (int a = 0; a < kStemRegBits; ++a) st[a] = p.rstr_out[a];
            reg_walk(g, st, ps.dead,
                     [&](int r, uint64_t a) { *reinterpret_cast<float2*>(a) = x[r]; });
        }
    }
}

template <int NTH>
cudaError_t launch_stem_reg_impl(const StemRegParams& p, const StemRegBranches* br, int64_t slice0, int batch,
                                 cudaStream_t s) {
    const size_t smem = ((size_t)(1u << p.n) + p.nentries) * sizeof(float2);
    static const cudaError_t attr = cudaFuncSetAttribute(
        k_stem_reg<NTH>, cudaFuncAttributeMaxDynamicSharedMemorySize,
        (int)(((NTH * RE > (1 << kStemRegMinN) ? NTH * RE : (1 << kStemRegMinN)) + kStemRegMaxEntries) * sizeof(float2)));
    if (attr != cudaSuccess) return attr;
    return launch_dependent(k_stem_reg<NTH>, dim3(1u << p.nu, 1, batch), dim3(NTH), smem, s, 1, p, br, slice0);
}

}  // namespace

cudaError_t launch_stem_fused(const StemParams* d_params, const StemParams& hp, int cap_log2, int64_t slice0,
                              int batch, cudaStream_t s) {
    if (!d_params || cap_log2 < 1 || cap_log2 > kStemMaxInner || hp.nu < 0 || hp.nu > 30 || hp.nsteps < 1 ||
        hp.nsteps > kStemMaxSteps || hp.n_in > cap_log2 || hp.n_out > cap_log2 || batch < 1 || batch > 65535)
        return cudaErrorInvalidValue;
    // every step reads exactly the sub-tensor the previous one wrote, and an
    // in-place step's positions lie inside it, ascending
    int bits = hp.n_in;
    bool two = false;
    for (int i = 0; i < hp.nsteps; ++i) {
        const StemStep& st = hp.steps[i];
        if (st.nk < 0 || st.nk > 4 || st.nn < 0 || st.nn > 4 || st.nr < 0 || st.nr + st.nk != bits ||
            st.nr + st.nn > cap_log2 || st.b_off < 0 || st.b_off + (1 << (st.nk + st.nn)) > hp.b_total)
            return cudaErrorInvalidValue;
        if (st.inplace) {
            if (st.nk != st.nn) return cudaErrorInvalidValue;
            for (int t = 0; t < st.nk; ++t)
                if (st.ins[t] < 0 || st.ins[t] >= bits || (t > 0 && st.ins[t] <= st.ins[t - 1]))
                    return cudaErrorInvalidValue;
        } else {
            two = true;
        }
        bits = st.nr + st.nn;
    }
    if (bits != hp.n_out || (two && !hp.two_buffers)) return cudaErrorInvalidValue;
    const size_t smem = ((size_t)((hp.two_buffers ? 2u : 1u) << cap_log2) + (size_t)hp.b_total) * sizeof(float2);
    if (smem > 227 * 1024) return cudaErrorInvalidValue;
    static int set_for = 0;
    if ((int)smem > set_for) {
        cudaError_t e = cudaFuncSetAttribute(k_stem_fused, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        set_for = (int)smem;
    }
    return launch_dependent(k_stem_fused, dim3(1u << hp.nu, 1, batch), dim3(NT), smem, s, 1, d_params, cap_log2, slice0);
}

namespace {
// a pass's positions while the passes are planned
struct PassPlan {
    StemRegPass ps{};
    int8_t rp[kStemRegBits], tp[kStemRegMaxN - kStemRegBits];
};
}  // namespace

bool stem_reg_params(const StemParams& sp, StemRegParams& r, StemRegBranches& rb) {
    r = StemRegParams{};
    rb = StemRegBranches{};
    int64_t istr[kStemRegMaxN] = {}, ostr[kStemRegMaxN] = {};  // by position
    PassPlan plan[kStemMaxSteps + 2];
    auto log2_of = [](int64_t v) {
        int b = 0;
        while ((1ll << b) < v) ++b;
        return b;
    };
    int n = sp.n_in;  // positions
    for (int i = 0; i < sp.nsteps; ++i)
        if (sp.steps[i].nn == 2 && sp.steps[i].nk < 2) n += 2 - sp.steps[i].nk;
    if (n < kStemRegMinN || n > kStemRegMaxN || sp.n_in < kStemRegBits || sp.nu < 0 || sp.nu > 30 || sp.nsteps < 1 ||
        sp.nsteps > kStemMaxSteps || sp.b_total > kStemRegMaxEntries)
        return false;
    r.in = sp.in;
    r.out = sp.out;
    r.out_batch_stride = sp.out_batch_stride;
    r.n = n;
    r.nu = sp.nu;
    r.nentries = sp.b_total;
    // outer modes by their stride in T_0: consecutive CTAs then read neighbouring runs, whose
    // 128-byte lines they share (in the plan's order, the stem was read twice from DRAM)
    for (int b = 0; b < sp.nu; ++b) {
        int j = b;
        for (; j > 0 && r.ustr_in[j - 1] > sp.ustr_in[b]; --j) {
            r.ustr_in[j] = r.ustr_in[j - 1];
            r.ustr_out[j] = r.ustr_out[j - 1];
        }
        r.ustr_in[j] = sp.ustr_in[b];
        r.ustr_out[j] = sp.ustr_out[b];
    }
    for (int b = 0; b < sp.n_in; ++b) istr[b] = sp.istr[b];
    // positions of the steps' modes: pos[b] is the position of bit b of the current X
    int pos[kStemMaxInner];
    for (int b = 0; b < sp.n_in; ++b) pos[b] = b;
    int bits = sp.n_in, next = sp.n_in, spos[kStemMaxSteps][2];
    for (int i = 0; i < sp.nsteps; ++i) {
        const StemStep& st = sp.steps[i];
        const bool gate = st.inplace && st.nk == st.nn && (st.nk == 1 || st.nk == 2);
        const bool project = !st.inplace && st.nk == 1 && st.nn == 0;
        const bool grow = !st.inplace && st.nk < 2 && st.nn == 2;
        if ((!gate && !project && !grow) || st.nr + st.nk != bits) return false;
        rb.br[i] = st.br;
        r.step[i].kind = project ? SR_PROJECT : grow ? (st.nk ? SR_GROW1 : SR_GROW0) : st.nk == 1 ? SR_GATE1 : SR_GATE2;
        r.step[i].b_off = (int16_t)st.b_off;
        for (int e = 0; e < 1 << (st.nk + st.nn); ++e) {  // dense [k][n]
            int off = 0;
            for (int b = 0; b < st.nk; ++b)
                if ((e >> st.nn) >> b & 1) off += st.kstr_b[b];
            for (int b = 0; b < st.nn; ++b)
                if (e >> b & 1) off += st.nstr_b[b];
            rb.entry[st.b_off + e] = make_int2(i, off);
        }
        for (int b = 0; b < st.nk; ++b) spos[i][b] = pos[log2_of(st.kstr_x[b])];
        for (int b = st.nk; b < st.nn; ++b) spos[i][b] = next++;  // a mode that is born
        if (!gate) {  // X becomes [kept bits | new bits]
            int now[kStemMaxInner];
            for (int b = 0; b < st.nr; ++b) now[st.nn + b] = pos[log2_of(st.rstr[b])];
            for (int b = 0; b < st.nn; ++b) now[b] = spos[i][b];
            bits = st.nr + st.nn;
            for (int b = 0; b < bits; ++b) pos[b] = now[b];
        }
    }
    if (bits != sp.n_out || next != n) return false;
    for (int b = 0; b < bits; ++b) ostr[pos[b]] = sp.ostr[b];
    uint32_t alive = (1u << sp.n_in) - 1;  // positions that hold data
    const uint32_t last_alive = [&] {
        uint32_t m = 0;
        for (int b = 0; b < bits; ++b) m |= 1u << pos[b];
        return m;
    }();
    auto count = [](uint32_t m) {
        int c = 0;
        for (; m; m &= m - 1) ++c;
        return c;
    };
    // positions of `from` in ascending stride
    auto by_stride = [&](uint32_t from, const int64_t* str) {
        int c = 0;
        int8_t v[kStemRegMaxN] = {};
        for (int p = 0; p < n; ++p)
            if (from >> p & 1) {
                int j = c++;
                for (; j > 0 && str[v[j - 1]] > str[p]; --j) v[j] = v[j - 1];
                v[j] = (int8_t)p;
            }
        struct { int8_t v[kStemRegMaxN]; int n; } o;
        for (int j = 0; j < kStemRegMaxN; ++j) o.v[j] = v[j];
        o.n = c;
        return o;
    };
    // Register positions of a pass holding `used` (slots given, -1 free): free slots
    // take the alive positions of the largest stride, threads the others, lanes
    // the smallest strides first (coalesced access), or, for a pass that only
    // touches shared memory, four positions of independent bank columns.
    auto fill = [&](PassPlan& ps, const int64_t* str) {
        uint32_t used = 0;
        for (int a = 0; a < kStemRegBits; ++a)
            if (ps.rp[a] >= 0) used |= 1u << ps.rp[a];
        auto o = by_stride(alive & ~used, str);
        for (int a = kStemRegBits - 1; a >= 0; --a)
            if (ps.rp[a] < 0) {
                ps.rp[a] = o.v[--o.n];
                used |= 1u << ps.rp[a];
            }
        ps.ps.nt = (int8_t)o.n;
        for (int t = 0; t < o.n; ++t) ps.tp[t] = o.v[t];
    };
    auto spread_lanes = [&](PassPlan& ps) {
        int span[4], ns = 0, front = 0;
        for (int t = 0; t < ps.ps.nt && ns < 4; ++t) {
            int c = kBankCol[ps.tp[t]];
            for (int j = 0; j < ns; ++j) c = (c ^ span[j]) < c ? c ^ span[j] : c;
            if (!c) continue;
            span[ns++] = c;
            const int8_t v = ps.tp[t];
            for (int j = t; j > front; --j) ps.tp[j] = ps.tp[j - 1];
            ps.tp[front++] = v;
        }
    };
    // whether a pass that reads (writes) global memory leaves at least two of the
    // three smallest strides to its lanes
    auto coalesced = [&](const PassPlan& ps, uint32_t live, const int64_t* str) {
        const auto o = by_stride(live, str);
        int c = 0;
        for (int j = 0; j < 3 && j < o.n; ++j)
            for (int a = 0; a < kStemRegBits; ++a) c += ps.rp[a] == o.v[j];
        return c <= 1;
    };
    auto empty_pass = [&](int at) {
        PassPlan ps;
        for (int a = 0; a < kStemRegBits; ++a) ps.rp[a] = -1;
        ps.ps.step0 = ps.ps.step1 = (int8_t)at;
        return ps;
    };
    int i = 0;
    while (i < sp.nsteps) {
        if (count(alive) < kStemRegBits || r.npass > kStemMaxSteps) return false;
        PassPlan ps = empty_pass(i);
        int pair[2][2], np = 0, single[kStemRegBits], nsg = 0;
        auto pair_of = [&](int p) {
            for (int q = 0; q < np; ++q)
                if (pair[q][0] == p || pair[q][1] == p) return q;
            return -1;
        };
        auto single_of = [&](int p) {
            for (int q = 0; q < nsg; ++q)
                if (single[q] == p) return q;
            return -1;
        };
        int j = i;
        for (; j < sp.nsteps; ++j) {
            if (r.step[j].kind >= SR_GATE2) {  // two positions in one pair of register bits
                const int a = spos[j][0], b = spos[j][1], qa = pair_of(a), qb = pair_of(b);
                if (qa >= 0 || qb >= 0) {
                    if (qa == qb && pair[qa][0] == a && pair[qa][1] == b) continue;
                    break;  // its modes sit in other pairs (or in the other order)
                }
                const int freed = (single_of(a) >= 0) + (single_of(b) >= 0);
                if (np == 2 || 2 * np + nsg - freed + 2 > kStemRegBits) break;
                for (int v : {a, b}) {
                    const int q = single_of(v);
                    if (q >= 0) single[q] = single[--nsg];
                }
                pair[np][0] = a;
                pair[np][1] = b;
                ++np;
            } else {
                const int a = spos[j][0];
                if (pair_of(a) >= 0 || single_of(a) >= 0) continue;
                if (2 * np + nsg + 1 > kStemRegBits) break;
                single[nsg++] = a;
            }
        }
        for (int q = 0; q < np; ++q) {
            ps.rp[2 * q] = (int8_t)pair[q][0];
            ps.rp[2 * q + 1] = (int8_t)pair[q][1];
        }
        for (int q = 0; q < nsg; ++q) ps.rp[2 * np + q] = (int8_t)single[q];
        ps.ps.step1 = (int8_t)j;
        const bool first = r.npass == 0;
        fill(ps, first ? istr : ostr);
        for (int a = 0; a < kStemRegBits; ++a)
            if (!(alive >> ps.rp[a] & 1)) ps.ps.unborn |= (int8_t)(1 << a);
        if (first && !coalesced(ps, alive, istr)) {  // load with coalesced lanes first
            PassPlan in = empty_pass(0);
            fill(in, istr);
            plan[r.npass++] = in;
        }
        for (int t = i; t < j; ++t) {
            for (int a = 0; a < kStemRegBits; ++a)
                if (ps.rp[a] == spos[t][0]) r.step[t].reg = (int8_t)(r.step[t].kind >= SR_GATE2 ? a / 2 : a);
            if (r.step[t].kind == SR_GROW1) alive |= 1u << spos[t][1];
            if (r.step[t].kind == SR_GROW0) alive |= 1u << spos[t][0] | 1u << spos[t][1];
            if (r.step[t].kind == SR_PROJECT) {
                ps.ps.dead |= (int8_t)(1 << r.step[t].reg);
                alive &= ~(1u << spos[t][0]);
            }
        }
        plan[r.npass++] = ps;
        i = j;
    }
    if (alive != last_alive) return false;
    if (!coalesced(plan[r.npass - 1], alive, ostr) && count(alive) >= kStemRegBits) {
        PassPlan out = empty_pass(sp.nsteps);
        fill(out, ostr);
        plan[r.npass++] = out;
    }
    for (int q = 1; q + 1 < r.npass; ++q) spread_lanes(plan[q]);
    for (int q = 0; q < r.npass; ++q) {
        r.pass[q] = plan[q].ps;
        for (int a = 0; a < kStemRegBits; ++a) r.pass[q].rslot[a] = (uint16_t)(8 * slot_bit(plan[q].rp[a]));
        for (int t = 0; t < r.pass[q].nt; ++t) r.pass[q].tslot[t] = (uint16_t)(8 * slot_bit(plan[q].tp[t]));
    }
    const PassPlan &pf = plan[0], &pl = plan[r.npass - 1];
    for (int a = 0; a < kStemRegBits; ++a) {
        r.rstr_in[a] = 8 * istr[pf.rp[a]];
        r.rstr_out[a] = 8 * ostr[pl.rp[a]];
    }
    for (int t = 0; t < pf.ps.nt; ++t) r.tstr_in[t] = 8 * istr[pf.tp[t]];
    for (int t = 0; t < pl.ps.nt; ++t) r.tstr_out[t] = 8 * ostr[pl.tp[t]];
    return true;
}

cudaError_t launch_stem_reg(const StemRegParams& p, const StemRegBranches* br, int64_t slice0, int batch, cudaStream_t s) {
    if (!br || p.n < kStemRegMinN || p.n > kStemRegMaxN || p.nu < 0 || p.nu > 30 || p.npass < 1 || p.nentries < 1 ||
        p.nentries > kStemRegMaxEntries || batch < 1 || batch > 65535)
        return cudaErrorInvalidValue;
    switch (p.n) {
        case 13: return launch_stem_reg_impl<256>(p, br, slice0, batch, s);
        case 12: return launch_stem_reg_impl<128>(p, br, slice0, batch, s);
        case 11: return launch_stem_reg_impl<64>(p, br, slice0, batch, s);
        default: return launch_stem_reg_impl<32>(p, br, slice0, batch, s);
    }
}

}  // namespace tnc
