// Device code shared by the FP32 CUDA-core kernels and the persistent
// executor: the permute-fused complex64 contraction tile and the FP64 final
// reduction. BAR selects the barrier among the threads that run a routine:
// 0 = the whole CTA (__syncthreads), 1 = named barrier 1 over threads 0-255 of
// a larger CTA (the persistent executor's other warps do not take part).
#pragma once

#include <type_traits>

#include "kernels.h"
#include "launch.cuh"

namespace tnc {
namespace f32dev {

template <int BAR>
__device__ __forceinline__ void bar_sync() {
    if constexpr (BAR == 0) __syncthreads();
    else asm volatile("bar.sync 1, 256;" ::: "memory");
}

constexpr int BK = 16, NT = 256;
constexpr int LOG_BK = 4;

__device__ __forceinline__ int64_t slice_offset(const Operand& op, int64_t s) {
    int64_t off = 0;
    for (int j = 0; j < op.n_sl; ++j) off += ((s >> op.sl_bit[j]) & 1) * op.sl_stride[j];
    return off;
}

// sum of str[j] over the set bits j in [from, nbits) of x
__device__ __forceinline__ int64_t bits_offset(int64_t x, const int64_t* str, int nbits, int from) {
    int64_t off = 0;
    for (int j = from; j < nbits; ++j)
        if ((x >> j) & 1) off += str[j];
    return off;
}

// Packed pairs of FP32 values in one 64-bit register: fma.rn.f32x2 rounds each
// half like fmaf, with one instruction (two cycles of the FMA pipe) for both.
using f32x2 = unsigned long long;

__device__ __forceinline__ f32x2 pack2(float lo, float hi) {
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ float2 unpack2(f32x2 v) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
    f32x2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
    f32x2 d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f32x2 sub2(f32x2 a, f32x2 b) {
    f32x2 d;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
    f32x2 d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}

// C[m][n] = sum_k A(m,k) B(k,n), one BM x 64 tile per CTA of 256 threads, RM x 4
// complex per thread (BM = 16 RM).
//
// What bounds it: the FMA pipe and the 128 bytes per clock that shared memory
// returns to registers (a broadcast does not make a load cheaper). Real and
// imaginary parts are accumulated for pairs of rows by packed FMAs,
//     Cr += Ar (br, br);  Cr += Ai (-bi, -bi);  Ci += Ar (bi, bi);  Ci += Ai (br, br),
// with Ar, Ai the parts of rows m, m + 1: for every element the four roundings
// of four scalar FMAs, in the same order. A is staged as two planes (parts), so
// its pairs are loaded as they are; the doubled factors of B's four columns are
// made in registers. Per k and thread the 8 x 4 tile issues 64 packed FMAs (128
// pipe cycles), 6 16-byte loads (24 cycles of shared memory) and 20 moves.
//
// Shared-memory stages are double buffered: the gather of tile t+1 goes to
// registers while tile t is multiplied, then to the other stage (one barrier
// per tile). Accumulation is two-level: each group of GROUP_TILES k-tiles is
// summed in a fresh partial that is then added to the result with TwoSum
// (Knuth's error-free addition), whose rounding errors are collected in a
// per-thread compensation kept in shared memory and added once at the end.
// The FP32 rounding error thus grows like the 64-term partial sums alone
// instead of also with the K / 64 additions of partials.
constexpr int GROUP_TILES = 4;   // 64 k-terms per partial sum

// Tile shape: NTH threads, WN warps along n (the others along m), RM x 4
// complex per thread.
template <int NTH, int RM, int WN> struct TileCfg {
    static constexpr int BM = NTH / 32 / WN * 4 * RM, BN = 32 * WN;
};

__host__ __device__ constexpr int log2_of(int v) { return v <= 1 ? 0 : 1 + log2_of(v / 2); }

// Staged operands of one tile.
template <int NTH, int RM, int WN> struct GemmStage {
    static constexpr int BM = TileCfg<NTH, RM, WN>::BM, BN = TileCfg<NTH, RM, WN>::BN;
    float Ar[2][BK][BM + 4], Ai[2][BK][BM + 4];  // 16-byte aligned rows
    float2 Bs[2][BK][BN + 2];
    // kstep[b]: offset of k-tile t + 1 minus that of k-tile t when b bits of t
    // carry (bit b of t + 1 is its lowest set bit)
    int64_t kstepA[kMaxBits], kstepB[kMaxBits];
    int64_t sa[4], sb[4];  // TileWork::sa, sb where registers are short
};
template <int NTH, int RM, int WN> struct GemmSmemT : GemmStage<NTH, RM, WN> {
    f32x2 comp[4 * RM][NTH];       // TwoSum compensation of each thread's outputs
};
using GemmSmem = GemmSmemT<256, 4, 2>;

// a += b with the rounding error of the addition added to c (TwoSum: the
// error term is exact whatever the magnitudes of a and b)
__device__ __forceinline__ void two_sum_into(f32x2& a, f32x2 b, f32x2& c) {
    const f32x2 s = add2(a, b);
    const f32x2 bv = sub2(s, a);
    const f32x2 e = add2(sub2(a, sub2(s, bv)), sub2(b, bv));
    a = s;
    c = add2(c, e);
}

// The gather, staging and products of one output tile (slice z, slice id
// slice0 + z) of the contraction described by p.
// LEAN: registers are short (grouped contractions with their parameters in shared
// memory, the persistent executor).
template <int NTH, int RM, int WN, bool LEAN = false> struct TileWork {
    using Cfg = TileCfg<NTH, RM, WN>;
    static constexpr int EA = Cfg::BM * BK / NTH, EB = Cfg::BN * BK / NTH;  // elements a thread gathers per k-tile
    static constexpr int RP = RM / 2;                                      // row pairs of a thread
    GemmStage<NTH, RM, WN>& sm;
    int64_t M, N, K, m0, n0;
    // plain pointers: the predecessor launch, or another CTA of the persistent executor,
    // may write the operands while this CTA decodes its parameters (launch.cuh)
    const float2 *A, *B;
    bool a_kfast, b_nfast;
    bool full;  // no element of the tile lies past M, N or K
    int64_t sa[LEAN ? 1 : log2_of(EA)], sb[LEAN ? 1 : log2_of(EB)];  // offsets of the bits of an element's number (the same in every thread)
    int tm, tn;
    int64_t khA = 0, khB = 0;  // offsets of the k-tile to gather
    float2 ra[EA], rb[EB];

    // Fills kstepA, kstepB (and sm.sa, sm.sb); the wait for the predecessor and a
    // barrier must follow before the first gather.
    __device__ __forceinline__ TileWork(const GemmParams& p, int64_t tile, int z, int64_t slice0,
                                        GemmStage<NTH, RM, WN>& stage)
        : sm(stage) {
        const int tid = threadIdx.x;
        M = 1ll << p.mb;
        N = 1ll << p.nb;
        K = 1ll << p.kb;
        const int64_t tiles_n = (N + Cfg::BN - 1) / Cfg::BN;
        m0 = (tile / tiles_n) * Cfg::BM;
        n0 = (tile % tiles_n) * Cfg::BN;
        A = p.A.ptr + z * p.A.batch_stride + slice_offset(p.A, slice0 + z);
        B = p.B.ptr + z * p.B.batch_stride + slice_offset(p.B, slice0 + z);
        if (tid < p.kb - LOG_BK) {
            int64_t da = p.ak[LOG_BK + tid], db = p.bk[LOG_BK + tid];
            for (int j = 0; j < tid; ++j) {
                da -= p.ak[LOG_BK + j];
                db -= p.bk[LOG_BK + j];
            }
            sm.kstepA[tid] = da;
            sm.kstepB[tid] = db;
        }
        // load mapping: walk the operand's unit-stride mode with consecutive threads
        a_kfast = p.kb > 0 && p.ak[0] == 1;
        b_nfast = p.nb > 0 && p.bn[0] == 1;
        int m, k, n, kb;
        a_mk(0, m, k);
        b_nk(0, n, kb);
        A += bits_offset(m0 + m, p.am, p.mb, 0) + bits_offset(k, p.ak, p.kb, 0);
        B += bits_offset(n0 + n, p.bn, p.nb, 0) + bits_offset(kb, p.bk, p.kb, 0);
        // bit t of an element's number is bit lo + t of its k (or m, n)
        constexpr int LT = log2_of(NTH) - LOG_BK, LA = log2_of(NTH / Cfg::BM), LB = log2_of(NTH / Cfg::BN);
        auto step_a = [&](int t) {
            return a_kfast ? (LT + t < p.mb ? p.am[LT + t] : 0) : LA + t < p.kb ? p.ak[LA + t] : 0;
        };
        auto step_b = [&](int t) {
            return b_nfast ? (LB + t < p.kb ? p.bk[LB + t] : 0) : LT + t < p.nb ? p.bn[LT + t] : 0;
        };
        static_assert(log2_of(EA) <= 4 && log2_of(EB) <= 4, "size of the shared copies");
        if constexpr (LEAN) {
            if (tid < log2_of(EA)) sm.sa[tid] = step_a(tid);
            if (tid < log2_of(EB)) sm.sb[tid] = step_b(tid);
        } else {
#pragma unroll
            for (int t = 0; t < log2_of(EA); ++t) sa[t] = step_a(t);
#pragma unroll
            for (int t = 0; t < log2_of(EB); ++t) sb[t] = step_b(t);
        }
        full = m0 + Cfg::BM <= M && n0 + Cfg::BN <= N && K >= BK;
        // lanes 4 (m) x 8 (n): thread rows tm .. tm + 3 (and, for RM = 8, tm + 16 ..
        // tm + 19), columns tn, tn + 1, tn + 16, tn + 17
        const int lane = tid & 31, warp = tid >> 5;
        tm = (warp / WN) * (4 * RM) + 4 * (lane >> 3);
        tn = (warp % WN) * 32 + 2 * (lane & 7);
    }
    __device__ __forceinline__ void a_mk(int i, int& m, int& k) const {
        const int e = threadIdx.x + i * NTH;
        m = a_kfast ? e / BK : e % Cfg::BM;
        k = a_kfast ? e % BK : e / Cfg::BM;
    }
    __device__ __forceinline__ void b_nk(int i, int& n, int& k) const {
        const int e = threadIdx.x + i * NTH;
        n = b_nfast ? e % Cfg::BN : e / BK;
        k = b_nfast ? e / Cfg::BN : e % BK;
    }
    // moves khA, khB from k-tile t to k-tile t + 1
    __device__ __forceinline__ void next_tile(int64_t t) {
        const int carry = __ffsll(t + 1) - 1;
        khA += sm.kstepA[carry];
        khB += sm.kstepB[carry];
    }
    // The elements of a thread differ in three bits or so of k (or of m, n), and the
    // offsets of these bits are the same in every thread: one pointer per operand, an
    // addition per element, and no predicates where the tile has no edge. (Rows and
    // columns from tables in shared memory were two loads and two 64-bit additions
    // per element, in a loop that shared memory bounds as much as the FMAs:
    // (2^11, 2^10, 2^12) 1731 us against 1510, (2^13, 2^6, 2^11) 281 against 229, a
    // 24-qubit call 2.32 ms against 2.11.) LEAN keeps the one path with predicates:
    // a level of small contractions waits for its instructions (20 qubits: 162 us
    // against 166).
    __device__ __forceinline__ void gather() {
        auto load = [&](auto masked) {
#pragma unroll
            for (int i = 0; i < EA; ++i) {
                int64_t o = 0;
#pragma unroll
                for (int t = 0; t < log2_of(EA); ++t)
                    if (i >> t & 1) o += LEAN ? sm.sa[t] : sa[t];
                if constexpr (decltype(masked)::value) {
                    int m, k;
                    a_mk(i, m, k);
                    ra[i] = make_float2(0.f, 0.f);
                    if (m0 + m < M && k < K) ra[i] = A[khA + o];
                } else {
                    ra[i] = A[khA + o];
                }
            }
#pragma unroll
            for (int i = 0; i < EB; ++i) {
                int64_t o = 0;
#pragma unroll
                for (int t = 0; t < log2_of(EB); ++t)
                    if (i >> t & 1) o += LEAN ? sm.sb[t] : sb[t];
                if constexpr (decltype(masked)::value) {
                    int n, k;
                    b_nk(i, n, k);
                    rb[i] = make_float2(0.f, 0.f);
                    if (n0 + n < N && k < K) rb[i] = B[khB + o];
                } else {
                    rb[i] = B[khB + o];
                }
            }
        };
        if (!LEAN && full) load(std::false_type{});
        else load(std::true_type{});
    }
    __device__ __forceinline__ void stage_store(int st) {
#pragma unroll
        for (int i = 0; i < EA; ++i) {
            int m, k;
            a_mk(i, m, k);
            sm.Ar[st][k][m] = ra[i].x;
            sm.Ai[st][k][m] = ra[i].y;
        }
#pragma unroll
        for (int i = 0; i < EB; ++i) {
            int n, k;
            b_nk(i, n, k);
            sm.Bs[st][k][n] = rb[i];
        }
    }
    // part[h][row pair][column] += the products of row kk of stage st (h: 0 Re, 1 Im)
    __device__ __forceinline__ void step(int st, int kk, f32x2 (&part)[2][RP][4]) const {
        f32x2 ar[RP], ai[RP];
#pragma unroll
        for (int q = 0; q < RM / 4; ++q) {
            const ulonglong2 r = *reinterpret_cast<const ulonglong2*>(&sm.Ar[st][kk][tm + 16 * q]);
            const ulonglong2 i = *reinterpret_cast<const ulonglong2*>(&sm.Ai[st][kk][tm + 16 * q]);
            ar[2 * q] = r.x;
            ar[2 * q + 1] = r.y;
            ai[2 * q] = i.x;
            ai[2 * q + 1] = i.y;
        }
        const float4 b01 = *reinterpret_cast<const float4*>(&sm.Bs[st][kk][tn]);
        const float4 b23 = *reinterpret_cast<const float4*>(&sm.Bs[st][kk][tn + 16]);
        const float br[4] = {b01.x, b01.z, b23.x, b23.z}, bi[4] = {b01.y, b01.w, b23.y, b23.w};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const f32x2 brr = pack2(br[j], br[j]), bii = pack2(bi[j], bi[j]), bin = pack2(-bi[j], -bi[j]);
#pragma unroll
            for (int i = 0; i < RP; ++i) {
                part[0][i][j] = fma2(ar[i], brr, part[0][i][j]);
                part[1][i][j] = fma2(ar[i], bii, part[1][i][j]);
            }
#pragma unroll
            for (int i = 0; i < RP; ++i) {
                part[0][i][j] = fma2(ai[i], bin, part[0][i][j]);
                part[1][i][j] = fma2(ai[i], brr, part[1][i][j]);
            }
        }
    }
    // every row of stage st (K is a power of two: below BK, the one k-tile's
    // zero-padded rows are skipped)
    __device__ __forceinline__ void multiply(int st, f32x2 (&part)[2][RP][4]) const {
        if (K >= BK) {
#pragma unroll
            for (int kk = 0; kk < BK; ++kk) step(st, kk, part);
        } else {
            for (int kk = 0; kk < (int)K; kk += 2) {  // (K = 1: a zero row of both operands)
                step(st, kk, part);
                step(st, kk + 1, part);
            }
        }
    }
    // row of the tile of row pair i, half h
    __device__ __forceinline__ int64_t row(int i, int h) const { return m0 + tm + 16 * (i / 2) + 2 * (i % 2) + h; }
};

// One output tile `tile` of slice z (slice id slice0 + z) of the contraction
// described by p.
template <int BAR = 0, int NTH = 256, int RM = 4, int WN = 2, bool LEAN = BAR == 1>
__device__ __forceinline__ void gemm_tile(const GemmParams& p, int64_t tile, int z, int64_t slice0,
                                          GemmSmemT<NTH, RM, WN>& sm) {
    using W = TileWork<NTH, RM, WN, LEAN>;
    constexpr int RP = W::RP;
    const int tid = threadIdx.x;
    W w(p, tile, z, slice0, sm);
    if constexpr (BAR == 0) dep_wait();
    bar_sync<BAR>();
    f32x2 acc[2][RP][4], part[2][RP][4];
#pragma unroll
    for (int i = 0; i < RP; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                acc[h][i][j] = 0;
                part[h][i][j] = 0;
            }
    const int64_t ntiles = (w.K + BK - 1) / BK;
    w.gather();
    w.stage_store(0);
    bar_sync<BAR>();
    for (int64_t t = 0; t < ntiles; ++t) {
        const int st = (int)(t & 1);
        if (t + 1 < ntiles) {
            w.next_tile(t);
            w.gather();
        }
        w.multiply(st, part);
        if (t + 1 == ntiles) break;
        if ((t + 1) % GROUP_TILES == 0) {  // comp: this thread's own slots, written by its first group
#pragma unroll
            for (int i = 0; i < RP; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j)
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        f32x2 c = t < GROUP_TILES ? 0 : sm.comp[8 * i + 2 * j + h][tid];
                        two_sum_into(acc[h][i][j], part[h][i][j], c);
                        sm.comp[8 * i + 2 * j + h][tid] = c;
                        part[h][i][j] = 0;
                    }
        }
        w.stage_store(st ^ 1);
        bar_sync<BAR>();
    }
    // the last group, then the compensation
#pragma unroll
    for (int i = 0; i < RP; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                f32x2 c = ntiles <= GROUP_TILES ? 0 : sm.comp[8 * i + 2 * j + h][tid];
                two_sum_into(acc[h][i][j], part[h][i][j], c);
                acc[h][i][j] = add2(acc[h][i][j], c);
            }
    float2* C = p.C + z * p.c_batch_stride;
#pragma unroll
    for (int i = 0; i < RP; ++i)
#pragma unroll
        for (int q = 0; q < 2; ++q) {  // columns tn + 16 q, + 1
            float2 re[2], im[2];  // of the two columns, both rows
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                re[j] = unpack2(acc[0][i][2 * q + j]);
                im[j] = unpack2(acc[1][i][2 * q + j]);
            }
            const int64_t n = w.n0 + w.tn + 16 * q;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int64_t m = w.row(i, h);
                if (m >= w.M) continue;
                const float4 v = h ? make_float4(re[0].y, im[0].y, re[1].y, im[1].y)
                                   : make_float4(re[0].x, im[0].x, re[1].x, im[1].x);
                if (n + 1 < w.N) *reinterpret_cast<float4*>(C + m * w.N + n) = v;
                else if (n < w.N) C[m * w.N + n] = make_float2(v.x, v.y);
            }
        }
}

// The same tile by a cluster of CL CTAs, for contractions of few output tiles
// and a long K. CTA r of the cluster forms the 64-term partials of the k groups
// r, r + CL, ...; after each round of CL groups the partials are exchanged
// through distributed shared memory, and the CTA that owns an output adds the
// CL partials in group order with TwoSum: the sums, and so the bits, of
// gemm_tile. Thread t's partials live at xch[.][e][t], e = 8 * row pair +
// 2 * column + h; CTA r owns e in [r E, (r + 1) E), E = 4 RM / CL. Two exchange
// buffers, so one cluster barrier per round is enough: a CTA refills a buffer
// after the next round's barrier, which follows every read of it.
template <int NTH, int WN> struct GemmClusterSmem : GemmStage<NTH, 4, WN> {
    f32x2 xch[2][16][NTH];
};

__device__ __forceinline__ f32x2 ld_cluster(const f32x2* p, uint32_t rank) {
    uint32_t a = static_cast<uint32_t>(__cvta_generic_to_shared(p)), ra;
    f32x2 v;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(a), "r"(rank));
    asm volatile("ld.shared::cluster.b64 %0, [%1];" : "=l"(v) : "r"(ra) : "memory");
    return v;
}
__device__ __forceinline__ void cluster_barrier() {
    __syncwarp();  // .aligned: the whole warp executes it together, also after a predicated store
    asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

template <int NTH, int WN, int CL>
__device__ __forceinline__ void gemm_tile_cluster(const GemmParams& p, int64_t tile, uint32_t rank, int z, int64_t slice0,
                                                  GemmClusterSmem<NTH, WN>& sm) {
    static_assert(CL == 2 || CL == 4 || CL == 8, "a CTA owns whole complex outputs");
    using W = TileWork<NTH, 4, WN>;
    constexpr int E = 16 / CL;
    const int tid = threadIdx.x;
    W w(p, tile, z, slice0, sm);
    f32x2 part[2][2][4], acc[E], comp[E];
#pragma unroll
    for (int e = 0; e < E; ++e) acc[e] = comp[e] = 0;
    const int64_t rounds = w.K / (BK * GROUP_TILES) / CL;  // K is a multiple of 64 CL
    auto seek = [&](int64_t round) {  // the first k-tile of this CTA's group of the round
        const int64_t k = (round * CL + rank) * (BK * GROUP_TILES);
        w.khA = bits_offset(k, p.ak, p.kb, LOG_BK);
        w.khB = bits_offset(k, p.bk, p.kb, LOG_BK);
    };
    dep_wait();
    __syncthreads();
    seek(0);
    w.gather();
    w.stage_store(0);
    __syncthreads();
    for (int64_t r = 0; r < rounds; ++r) {
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) part[0][i][j] = part[1][i][j] = 0;
#pragma unroll 1
        for (int t = 0; t < GROUP_TILES; ++t) {
            const bool more = t + 1 < GROUP_TILES || r + 1 < rounds;
            if (more) {
                if (t + 1 < GROUP_TILES) w.next_tile(t);
                else seek(r + 1);
                w.gather();
            }
            w.multiply(t & 1, part);
            if (more) w.stage_store((t & 1) ^ 1);
            __syncthreads();
        }
        f32x2(*x)[NTH] = sm.xch[r & 1];
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                x[8 * i + 2 * j][tid] = part[0][i][j];
                x[8 * i + 2 * j + 1][tid] = part[1][i][j];
            }
        cluster_barrier();
#pragma unroll
        for (int q = 0; q < CL; ++q)
#pragma unroll
            for (int e = 0; e < E; ++e) two_sum_into(acc[e], ld_cluster(&x[rank * E + e][tid], q), comp[e]);
    }
    float2* C = p.C + z * p.c_batch_stride;
#pragma unroll
    for (int e = 0; e < E; e += 2) {
        const int i = (rank * E + e) / 8, j = (rank * E + e) / 2 % 4;
        const int64_t n = w.n0 + w.tn + 16 * (j / 2) + j % 2;
        const float2 re = unpack2(add2(acc[e], comp[e])), im = unpack2(add2(acc[e + 1], comp[e + 1]));
        if (n < w.N) {
            if (w.row(i, 0) < w.M) C[w.row(i, 0) * w.N + n] = make_float2(re.x, im.x);
            if (w.row(i, 1) < w.M) C[w.row(i, 1) * w.N + n] = make_float2(re.y, im.y);
        }
    }
    cluster_barrier();  // this CTA's exchange buffers are read until every CTA is here
}

// Sum over this thread's k in [k_lo, k_hi) (k = k_lo + lane, + lanes, ...) of
// A[k] B[k] for the final contraction. When the block's K range holds whole
// rows of lanes, k = lanes * j + lane: the low bits are the lane (one offset
// per thread) and the offsets of j's bits come from shared-memory tables ta,
// tb, one per 8-bit group (K <= 2^40); products are summed in FP32 over runs
// of 16 j and the runs in FP64. Called by every thread of the block.
template <int BAR = 0>
__device__ void root_dot(const GemmParams& p, const float2* A, const float2* B, int64_t k_lo, int64_t k_hi,
                         int lane, int lanes, int64_t (*root_ta)[256], int64_t (*root_tb)[256], double& re,
                         double& im) {
    const int64_t kc = k_hi - k_lo;
    int lb = 0;
    while ((1 << lb) < lanes) ++lb;
    if (kc >= lanes) {
        // k = lanes * j + lane: the low lb bits are the lane (one offset per
        // thread); the offsets of j's bits come from shared-memory tables, one
        // per 8-bit group. Products are summed in FP32 over runs of 16 j and
        // the runs in FP64.
        const int jb = p.kb - lb, ng = jb > 0 ? (jb + 7) / 8 : 1;  // (K = lanes: one table of zeros)
        for (int idx = threadIdx.x; idx < ng * 256; idx += 256) {
            const int g = idx >> 8, e = idx & 255;
            int64_t oa = 0, ob = 0;
            for (int t = 0; t < 8; ++t) {
                const int bit = lb + 8 * g + t;
                if (bit < p.kb && ((e >> t) & 1)) {
                    oa += p.ak[bit];
                    ob += p.bk[bit];
                }
            }
            root_ta[g][e] = oa;
            root_tb[g][e] = ob;
        }
        bar_sync<BAR>();
        const float2* Al = A + bits_offset(lane, p.ak, lb, 0);
        const float2* Bl = B + bits_offset(lane, p.bk, lb, 0);
        const int64_t j_lo = k_lo >> lb, j_hi = k_hi >> lb;
        // eight j at a time (j_hi - j_lo is a power of two), all their loads in flight
        // before the first product: one at a time, a chunk of 64 j waited 64 times. (One
        // at a time inside the persistent executor, where the registers are short.)
        constexpr int RB = BAR == 0 ? 8 : 1;
        for (int64_t j0 = j_lo; j0 < j_hi; j0 += 16) {
            float sr = 0.f, si = 0.f;
            for (int64_t jb = j0; jb < j0 + 16 && jb < j_hi; jb += RB) {
                const int nj = j_hi - jb < RB ? (int)(j_hi - jb) : RB;
                int64_t oa = 0, ob = 0;
                for (int g = 1; g < ng; ++g) {
                    const int e = (int)((jb >> (8 * g)) & 255);
                    oa += root_ta[g][e];
                    ob += root_tb[g][e];
                }
                const int e0 = (int)(jb & 255);
                float2 a[RB], b[RB];
#pragma unroll
                for (int t = 0; t < RB; ++t)
                    if (t < nj) {
                        a[t] = Al[oa + root_ta[0][e0 + t]];
                        b[t] = Bl[ob + root_tb[0][e0 + t]];
                    }
#pragma unroll
                for (int t = 0; t < RB; ++t)
                    if (t < nj) {
                        sr = fmaf(a[t].x, b[t].x, sr);
                        sr = fmaf(-a[t].y, b[t].y, sr);
                        si = fmaf(a[t].x, b[t].y, si);
                        si = fmaf(a[t].y, b[t].x, si);
                    }
            }
            re += sr;
            im += si;
        }
    } else {
        for (int64_t k = k_lo + lane; k < k_hi; k += lanes) {
            float2 a = A[bits_offset(k, p.ak, p.kb, 0)];
            float2 b = B[bits_offset(k, p.bk, p.kb, 0)];
            re += (double)a.x * b.x - (double)a.y * b.y;
            im += (double)a.x * b.y + (double)a.y * b.x;
        }
    }
}


// FP64 partial sums of chunk `chunk` of a final contraction with R = M*N <= 64
// outputs, slice z (slice id slice0 + z), written to out[r] (r < R). Run by
// threads 0-255; red, ta, tb are shared-memory scratch.
template <int BAR = 0>
__device__ __forceinline__ void root_chunk(const RootParams& rp, int chunk, int z, int64_t slice0, double2* out,
                                           double2* red, int64_t (*ta)[256], int64_t (*tb)[256]) {
    const GemmParams& p = rp.g;
    const int R = 1 << (p.mb + p.nb);
    const int lanes = 256 / R;
    const int r = threadIdx.x / lanes, lane = threadIdx.x % lanes;
    const int64_t m = r >> p.nb, n = r & ((1 << p.nb) - 1);
    const int64_t s = slice0 + z;
    const float2* A = p.A.ptr + z * p.A.batch_stride + slice_offset(p.A, s) + bits_offset(m, p.am, p.mb, 0);
    const float2* B = p.B.ptr + z * p.B.batch_stride + slice_offset(p.B, s) + bits_offset(n, p.bn, p.nb, 0);
    const int64_t K = 1ll << p.kb;
    const int64_t kc = K / rp.chunks;
    const int64_t k_lo = chunk * kc, k_hi = k_lo + kc;
    double re = 0.0, im = 0.0;
    root_dot<BAR>(p, A, B, k_lo, k_hi, lane, lanes, ta, tb, re, im);
    red[threadIdx.x] = make_double2(re, im);
    bar_sync<BAR>();
    for (int st = lanes / 2; st > 0; st >>= 1) {
        if (lane < st) {
            double2 o = red[threadIdx.x + st];
            red[threadIdx.x].x += o.x;
            red[threadIdx.x].y += o.y;
        }
        bar_sync<BAR>();
    }
    if (lane == 0) out[r] = red[threadIdx.x];
}

// Ordered FP64 sum of a final contraction's `count` partial sums per output,
// added to out: output r's are shared by L lanes (a power of two of at most 128, at
// least 8 values each), lane l adding values l, l + L, ... and the lanes' sums
// being added as a tree. L depends on count alone, so every caller adds in the
// same order. (One lane per output read count values one after another: 67 us for
// 8 slices of 64 chunks and 16 outputs.) Items are (r, l) pairs; threads 0-255 serve
// items [item0, item0 + 256); red is shared-memory scratch of 256 entries.
__host__ __device__ inline int acc_lanes(int count) {
    int L = 1;
    while (L < 128 && 16 * L <= count) L *= 2;
    return L;
}
template <int BAR = 0>
__device__ __forceinline__ void accumulate_items(const double2* partials, int count, const PermParams& pp, int64_t item0,
                                                 double2* out, double2* red) {
    const int L = acc_lanes(count), tid = threadIdx.x;
    const int64_t R = 1ll << pp.obits, item = item0 + tid, r = item / L;
    const int l = (int)(item % L);
    const bool on = r < R;
    double2 acc = make_double2(0.0, 0.0);
    if (on) {
        const double2* src = partials + bits_offset(r, pp.ostride, pp.obits, 0);
#pragma unroll(BAR == 0 ? 8 : 2)
        for (int i = l; i < count; i += L) {
            const double2 v = src[(int64_t)i * R];
            acc.x += v.x;
            acc.y += v.y;
        }
    }
    for (int st = L / 2; st > 0; st >>= 1) {
        red[tid] = acc;
        bar_sync<BAR>();
        if (l < st) {
            const double2 o = red[tid + st];
            acc.x += o.x;
            acc.y += o.y;
        }
        bar_sync<BAR>();
    }
    if (on && l == 0) {
        out[r].x += acc.x;
        out[r].y += acc.y;
    }
}

}  // namespace f32dev
}  // namespace tnc
