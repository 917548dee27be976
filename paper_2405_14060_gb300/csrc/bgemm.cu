// Batched strided GEMM kernels (CUDA cores): contractions whose row, column
// or summed group is too small for the tensor-core tiles and whose operands
// are both too large to stream against a small one (bgemm.cuh).
//
//   k_bgemm      FP32: persistent blocks (two per SM), each walking its share of
//                the output tiles (item, g, m tile, n tile, K split).  The A and
//                B tiles are gathered through the offset tables straight into
//                shared memory by asynchronous copies (of 4, 2 or 1 floats, as
//                the operand's contiguous runs allow), kStages - 1 K steps ahead
//                of the multiply-adds; the pipeline runs across tile boundaries,
//                so short summed spaces (K of 8 to 32, common in evidence-batched
//                trees) still keep the memory system busy.  Shapes of the
//                batched workload (us before, with scalar shared loads and
//                copies, and now; entries 2^27 + 2^10): rows 2^20, 128 columns,
//                8 summed 291 / 171; 2^17, 1024, 32 463 / 297; 2^17, 32, 1024
//                400 / 290; 2^20, 8, 128 327 / 170; 2^18 x 4 rows, 36, 24 271 /
//                186.
//   k_bgemm_direct  FP64: a warp computes a strip of
//                rows times 1, 2 or 4 columns straight from the operands (L1),
//                without tiles in shared memory.
//   k_bgemm_fin  when K is split: sums the split partials in split order
//                (deterministic), applies the operands' power-of-two scales,
//                stores C and records its per-item maximum.
//
// Sum-product rescaling as in every other kernel: A and B enter multiplied by
// 2^-e (e the binary exponent of their recorded maxima; applied to the
// accumulated product, which is exact in binary floating point) and the
// kernel records the maximum of C.
#include <algorithm>
#include <cmath>
#include <utility>

#include "bgemm.cuh"
#include "devutil.cuh"

namespace tn {

namespace {

constexpr int kThreads = 256;
constexpr int kBK = 16;       // summed indices per pipeline stage
constexpr int kStages = 4;    // stages in flight (kStages - 1 ahead of the math)

struct TilePos {
    int64_t m0, n0, g, beta;
    int split;
};

__device__ __forceinline__ TilePos tile_pos(const BDesc &d, int64_t t, int BM, int BN) {
    const int64_t tiles_m = (d.M + BM - 1) / BM, tiles_n = (d.N + BN - 1) / BN;
    TilePos p;
    int64_t r, q = t;
    if (d.c_gfast) {
        q = div_tile(q, d.G, log2_if_pow2(d.G), r);
        p.g = r;
    }
    q = div_tile(q, tiles_m, log2_if_pow2(tiles_m), r);
    p.m0 = r * BM;
    q = div_tile(q, tiles_n, log2_if_pow2(tiles_n), r);
    p.n0 = r * BN;
    if (!d.c_gfast) {
        q = div_tile(q, d.G, log2_if_pow2(d.G), r);
        p.g = r;
    }
    q = div_tile(q, d.nbeta, log2_if_pow2(d.nbeta), r);
    p.beta = r;
    p.split = (int)q;
    return p;
}

// Task t of the direct kernel: columns fastest, then rows, G, items, splits.
__device__ __forceinline__ TilePos direct_pos(const BDesc &d, int64_t t, int MW, int TN) {
    const int64_t tm = (d.M + MW - 1) / MW, tn = (d.N + TN - 1) / TN;
    TilePos p;
    int64_t r, q = div_tile(t, tn, -1, r);
    p.n0 = r * TN;
    q = div_tile(q, tm, -1, r);
    p.m0 = r * MW;
    q = div_tile(q, d.G, -1, r);
    p.g = r;
    q = div_tile(q, d.nbeta, -1, r);
    p.beta = r;
    p.split = (int)q;
    return p;
}

// Asynchronous copy of V floats (1, 2 or 4); zeros when !ok.
template <int V>
__device__ __forceinline__ void cp_vec(uint32_t dst, const float *src, bool ok) {
    const int n = ok ? 4 * V : 0;
    if constexpr (V == 4)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(n)
                     : "memory");
    else if constexpr (V == 2)
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(dst), "l"(src), "r"(n)
                     : "memory");
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(n)
                     : "memory");
}
// Packed pairs of floats: d += a * b in both halves (one instruction).
__device__ __forceinline__ void fma2(uint64_t &d, uint64_t a, uint64_t b) {
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(a), "l"(b));
}
__device__ __forceinline__ uint64_t dup2(float v) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %1};" : "=l"(r) : "f"(v));
    return r;
}
__device__ __forceinline__ float half_of(uint64_t v, int h) {
    float lo, hi;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
    return h ? hi : lo;
}

// One operand tile of ROWS rows (of M or N) x kBK summed indices, gathered into
// one stage of kBK rows of ROWS + 4 floats.  A thread keeps either its rows or
// its summed index fixed over a step, whichever its operand's fastest label is
// in, so that neighbouring threads read neighbouring addresses; copies of V
// floats where the operand's rows run contiguously.
template <int ROWS, bool REG = true>
struct Gather {
    static constexpr int N = (ROWS * kBK + kThreads - 1) / kThreads;   // floats a thread
    static constexpr int LD = ROWS + 4, SIZE = kBK * LD;
    // REG: offsets of this thread's rows (one unless summed fastest; -1: none);
    // else (64 outputs a thread leave no registers) they are looked up every step
    int32_t off[REG ? N : 1];
    const int32_t *trow;
    int left;

    // rows of this thread's copies for a tile starting at row r0
    __device__ __forceinline__ void rows(const int32_t *t, int64_t nrow, int r0, bool kfast, int v) {
        if constexpr (!REG) {
            trow = t + r0;
            left = (int)min(nrow - r0, (int64_t)ROWS);
        } else if (kfast) {
#pragma unroll
            for (int i = 0; i < N; ++i) {
                const int r = (int)threadIdx.x / kBK + i * (kThreads / kBK);
                off[i] = r < ROWS && r0 + r < nrow ? __ldg(t + r0 + r) : -1;
            }
        } else {
            const int r = r0 + (int)threadIdx.x % (ROWS / v) * v;
            off[0] = r < nrow ? __ldg(t + r) : -1;
        }
    }
    // offset of row r of the tile, this thread's i-th (-1: past the end)
    __device__ __forceinline__ int32_t row_off(int r, int i) const {
        if constexpr (REG) return off[i];
        return r < left ? __ldg(trow + r) : -1;
    }
    __device__ __forceinline__ void issue(uint32_t s, const float *base, const int32_t *tk, int k0,
                                          int kend, int klen, bool kfast, int v) const {
        if (kfast) {
            const int kk = (int)threadIdx.x % kBK, k = k0 + kk;
            if (kk >= klen) return;
            const bool kok = k < kend;
            const int32_t ko = kok ? __ldg(tk + k) : 0;
#pragma unroll
            for (int i = 0; i < N; ++i) {
                const int r = (int)threadIdx.x / kBK + i * (kThreads / kBK);
                if (r >= ROWS) break;
                const int32_t ro = row_off(r, i);
                const bool ok = kok && ro >= 0;
                cp_vec<1>(s + 4u * (uint32_t)(kk * LD + r), ok ? base + (ro + ko) : base, ok);
            }
        } else if (v == 4) {
            along<4>(s, base, tk, k0, kend, klen);
        } else if (v == 2) {
            along<2>(s, base, tk, k0, kend, klen);
        } else {
            along<1>(s, base, tk, k0, kend, klen);
        }
    }
    template <int V>
    __device__ __forceinline__ void along(uint32_t s, const float *base, const int32_t *tk, int k0,
                                          int kend, int klen) const {
        constexpr int per = ROWS / V, step = kThreads / per;
        static_assert(step * per == kThreads, "copy grid");
        const int r = ((int)threadIdx.x % per) * V;
        const int32_t ro = row_off(r, 0);
#pragma unroll
        for (int i = 0; i < (kBK + step - 1) / step; ++i) {
            const int kk = (int)threadIdx.x / per + i * step;
            if (kk >= klen) break;
            const bool ok = ro >= 0 && k0 + kk < kend;
            cp_vec<V>(s + 4u * (uint32_t)(kk * LD + r),
                      ok ? base + (ro + __ldg(tk + k0 + kk)) : base, ok);
        }
    }
};

// FP32 kernel: a thread holds TM x TN outputs as pairs of rows (fma.rn.f32x2),
// rows RQ side by side (4 where C stores quads of rows, else 2, so that a warp's
// stores of shorter runs still fill sectors together), columns up to 4.  A
// word of shared memory per lane costs a clock of its pipe, a multiply-add a
// quarter: 8 x 8 outputs balance the two, 8 x 4 are bound by the loads at 2/3.
// NFAST: lanes run along C's columns.
template <int BM, int BN, int TM, int TN, bool NFAST, int RQ>
__global__ void __launch_bounds__(kThreads, 2)
    k_bgemm(const __grid_constant__ BDesc d, float *part, int ntiles) {
    constexpr int MT = BM / TM, NT = BN / TN;   // thread grid
    static_assert(MT * NT == kThreads, "thread grid");
    using GA = Gather<BM, (TM * TN < 64)>;
    using GB = Gather<BN, (TM * TN < 64)>;
    constexpr int SA = GA::SIZE, SB = GB::SIZE;
    extern __shared__ __align__(16) float smf[];
    float *As = smf, *Bs = smf + kStages * SA;
    const int tid = threadIdx.x;
    const int nks = (int)((d.kchunk + kBK - 1) / kBK);   // K steps per tile
    const int mine =
        ntiles > (int)blockIdx.x ? (ntiles - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;
    // a last step with at most half of its summed indices: the other half is
    // neither copied nor multiplied (64 outputs a thread: only where it is also
    // the first step, for want of registers)
    constexpr bool TAIL = TM * TN < 64;
    const int klast = d.nsplit == 1 && d.K - (TAIL ? (int64_t)(nks - 1) * kBK : 0) <= kBK / 2
                          ? kBK / 2 : kBK;
    const uint32_t sA0 = (uint32_t)__cvta_generic_to_shared(As);
    const uint32_t sB0 = (uint32_t)__cvta_generic_to_shared(Bs);
    // producer state: the tile (local index) and K step being loaded next
    int p_li = 0, p_ks = 0, p_stage = 0, p_kbeg = 0, p_kend = 0;
    const float *pA = (const float *)d.A, *pB = (const float *)d.B;
    GA ga;
    GB gb;
    auto issue = [&]() {
        if (p_li < mine) {
            if (p_ks == 0) {
                const TilePos tp =
                    tile_pos(d, (int64_t)blockIdx.x + (int64_t)p_li * gridDim.x, BM, BN);
                pA = (const float *)d.A + tp.beta * d.bsa + __ldg(d.tag + tp.g);
                pB = (const float *)d.B + tp.beta * d.bsb + __ldg(d.tbg + tp.g);
                p_kbeg = (int)(tp.split * d.kchunk);
                p_kend = (int)min(d.K, (int64_t)p_kbeg + d.kchunk);
                ga.rows(d.tam, d.M, (int)tp.m0, d.a_kfast, d.va);
                gb.rows(d.tbn, d.N, (int)tp.n0, d.b_kfast, d.vb);
            }
            const int k0 = p_kbeg + p_ks * kBK, klen = !TAIL || p_ks == nks - 1 ? klast : kBK;
            ga.issue(sA0 + (uint32_t)(p_stage * SA * 4), pA, d.tak, k0, p_kend, klen, d.a_kfast, d.va);
            gb.issue(sB0 + (uint32_t)(p_stage * SB * 4), pB, d.tbk, k0, p_kend, klen, d.b_kfast, d.vb);
            if (++p_ks == nks) {
                p_ks = 0;
                ++p_li;
            }
            p_stage = p_stage == kStages - 1 ? 0 : p_stage + 1;
        }
        cp_async_commit();
    };
    // thread grid: im of MT, in of NT
    constexpr int LN = NFAST ? (NT < 8 ? NT : 8) : (NT < 4 ? NT : 4);   // lanes along N
    constexpr int LM = 32 / LN, WM = MT / LM;                           // warps along M
    static_assert(WM >= 1 && WM * LM == MT, "warp grid");
    const int lane = tid & 31, warp = tid >> 5;
    const int ln = NFAST ? lane % LN : lane / LM, lm = NFAST ? lane / LN : lane % LM;
    const int im = (warp % WM) * LM + lm, in = (warp / WM) * LN + ln;
    // rows and columns of this thread (i-th row, j-th column)
    auto row = [&](int i) { return im * RQ + i % RQ + (i / RQ) * (RQ * MT); };
    constexpr int CQ = TN < 4 ? TN : 4;   // columns side by side
    auto col = [&](int j) { return in * CQ + j % CQ + (j / CQ) * (CQ * NT); };
    uint64_t acc[TM / 2][TN];
#pragma unroll
    for (int i = 0; i < TM / 2; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) acc[i][j] = 0ull;
    auto value = [&](int i, int j) { return half_of(acc[i >> 1][j], i & 1); };
    auto kstep = [&](const float *ra, const float *rb) {
        uint64_t a[TM / 2];
#pragma unroll
        for (int i = 0; i < TM / 2; i += RQ / 2) {
            if (RQ == 4) *(ulonglong2 *)(a + i) = *(const ulonglong2 *)(ra + row(2 * i));
            else a[i] = *(const uint64_t *)(ra + row(2 * i));
        }
        float b[TN];
#pragma unroll
        for (int j = 0; j < TN; j += CQ) {
            if (CQ == 4) *(float4 *)(b + j) = *(const float4 *)(rb + col(j));
            else if (CQ == 2) *(float2 *)(b + j) = *(const float2 *)(rb + col(j));
            else b[j] = rb[col(j)];
        }
#pragma unroll
        for (int j = 0; j < TN; ++j) {
            const uint64_t bb = dup2(b[j]);
#pragma unroll
            for (int i = 0; i < TM / 2; ++i) fma2(acc[i][j], a[i], bb);
        }
    };
#pragma unroll
    for (int s = 0; s < kStages - 1; ++s) issue();
    int c_li = 0, c_ks = 0, c_stage = 0;
    while (c_li < mine) {
        cp_async_wait<kStages - 2>();
        __syncthreads();
        issue();
        const float *sa = As + c_stage * SA, *sb = Bs + c_stage * SB;
#pragma unroll(TM * TN < 64 ? 8 : 2)
        for (int kk = 0; kk < kBK / 2; ++kk) kstep(sa + kk * GA::LD, sb + kk * GB::LD);
        if (klast == kBK || (TAIL && c_ks < nks - 1)) {
#pragma unroll(TM * TN < 64 ? 8 : 2)
            for (int kk = kBK / 2; kk < kBK; ++kk) kstep(sa + kk * GA::LD, sb + kk * GB::LD);
        }
        c_stage = c_stage == kStages - 1 ? 0 : c_stage + 1;
        if (++c_ks < nks) continue;
        c_ks = 0;
        // last K step of a tile: store it and start the next one
        const TilePos tp = tile_pos(d, (int64_t)blockIdx.x + (int64_t)c_li * gridDim.x, BM, BN);
        ++c_li;
        const int m0 = (int)tp.m0, n0 = (int)tp.n0;
        if (d.nsplit > 1) {
            // unscaled partials, dense [split][item][g][n][m]
            float *P = part + (((int64_t)tp.split * d.nbeta + tp.beta) * d.G + tp.g) * d.M * d.N;
#pragma unroll
            for (int i = 0; i < TM; ++i)
#pragma unroll
                for (int j = 0; j < TN; ++j) {
                    const int m = m0 + row(i), n = n0 + col(j);
                    if (m < d.M && n < d.N) P[(int64_t)n * d.M + m] = value(i, j);
                }
        } else {
            const float sca = d.mxa ? pow2neg<float>(exp_of_bits(d.mxa[tp.beta * d.mxa_bs])) : 1.f;
            const float scb = d.mxb ? pow2neg<float>(exp_of_bits(d.mxb[tp.beta * d.mxb_bs])) : 1.f;
            const float sc = sca * scb;
            float *Cb = (float *)d.C + tp.beta * d.bsc + __ldg(d.tcg + tp.g);
            float mx = 0.f;
            if (!NFAST && RQ == 4) {
                // quads of rows are contiguous in C
#pragma unroll
                for (int i = 0; i < TM; i += 4) {
                    const int m = m0 + row(i);
                    if (m >= d.M) continue;
                    float *Cm = Cb + __ldg(d.tcm + m);
#pragma unroll
                    for (int j = 0; j < TN; ++j) {
                        const int n = n0 + col(j);
                        if (n >= d.N) continue;
                        const float4 v = make_float4(value(i, j) * sc, value(i + 1, j) * sc,
                                                     value(i + 2, j) * sc, value(i + 3, j) * sc);
                        *(float4 *)(Cm + __ldg(d.tcn + n)) = v;
                        mx = fmaxf(mx, fmaxf(fmaxf(v.x, v.y), fmaxf(v.z, v.w)));
                    }
                }
            } else if (!NFAST && d.vc == 2) {
                // pairs of rows are contiguous in C
#pragma unroll
                for (int i = 0; i < TM; i += 2) {
                    const int m = m0 + row(i);
                    if (m >= d.M) continue;
                    float *Cm = Cb + __ldg(d.tcm + m);
#pragma unroll
                    for (int j = 0; j < TN; ++j) {
                        const int n = n0 + col(j);
                        if (n >= d.N) continue;
                        const float2 v = make_float2(value(i, j) * sc, value(i + 1, j) * sc);
                        *(float2 *)(Cm + __ldg(d.tcn + n)) = v;
                        mx = fmaxf(mx, fmaxf(v.x, v.y));
                    }
                }
            } else if (NFAST && TN >= 4 && d.vc == 4) {
                // quads of columns are contiguous in C
#pragma unroll
                for (int i = 0; i < TM; ++i) {
                    const int m = m0 + row(i);
                    if (m >= d.M) continue;
                    float *Cm = Cb + __ldg(d.tcm + m);
#pragma unroll
                    for (int j = 0; j + 3 < TN; j += 4) {
                        const int n = n0 + col(j);
                        if (n >= d.N) continue;
                        const float4 v = make_float4(value(i, j) * sc, value(i, j + 1) * sc,
                                                     value(i, j + 2) * sc, value(i, j + 3) * sc);
                        *(float4 *)(Cm + __ldg(d.tcn + n)) = v;
                        mx = fmaxf(mx, fmaxf(fmaxf(v.x, v.y), fmaxf(v.z, v.w)));
                    }
                }
            } else {
                int32_t cn[TN];
#pragma unroll
                for (int j = 0; j < TN; ++j) {
                    const int n = n0 + col(j);
                    cn[j] = n < d.N ? __ldg(d.tcn + n) : -1;
                }
#pragma unroll
                for (int i = 0; i < TM; ++i) {
                    const int m = m0 + row(i);
                    const int32_t cm = m < d.M ? __ldg(d.tcm + m) : -1;
#pragma unroll
                    for (int j = 0; j < TN; ++j)
                        if (cm >= 0 && cn[j] >= 0) {
                            const float v = value(i, j) * sc;
                            Cb[cm + cn[j]] = v;
                            mx = fmaxf(mx, v);
                        }
                }
            }
            record_max(d.mxc, tp.beta, true, (double)mx);
        }
#pragma unroll
        for (int i = 0; i < TM / 2; ++i)
#pragma unroll
            for (int j = 0; j < TN; ++j) acc[i][j] = 0ull;
    }
    cp_async_wait<0>();
}

// One warp per task: 32 / KL rows (lanes) times TN columns of one (item, g),
// over one split of the summed space, KL = 1 << klog lanes sharing an output's
// summed indices.  Tasks run columns fastest, so the warps of a block read the
// same rows of A.
//
// FP64: an SM does two multiply-adds a clock, a warp's multiply-add takes 16,
// its two or three loads (L1 hits) 2 to 32, so nothing but the count of
// multiply-adds matters: no padding (a 64 x 64 x 16 tile costs 16 us whatever
// part of it is used) and an even spread over the SMs.  The small nodes of a
// 12 x 12 grid with 16 evidence sets took 29 us each on tiles and take 7.4 us;
// 10 x 10 grid PR + MAR 520 -> 253 us, the batched 12 x 12 step 1112 -> 381 us.
template <typename T, int TN>
__global__ void __launch_bounds__(kThreads) k_bgemm_direct(const __grid_constant__ BDesc d, T *part,
                                                           int64_t ntask) {
    __shared__ double smax[kThreads / 32];
    __shared__ int64_t sbeta[kThreads / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int KL = 1 << d.klog, ks = lane & (KL - 1), MW = 32 >> d.klog;
    const int64_t t = (int64_t)blockIdx.x * (kThreads / 32) + warp;
    int64_t beta = -1;
    T mx = 0;
    if (t < ntask) {
        const TilePos tp = direct_pos(d, t, MW, TN);
        beta = tp.beta;
        const int64_t m = tp.m0 + (lane >> d.klog);
        const bool om = m < d.M;
        const T *A = (const T *)d.A + tp.beta * d.bsa + __ldg(d.tag + tp.g) +
                     __ldg(d.tam + (om ? m : d.M - 1));
        const T *B = (const T *)d.B + tp.beta * d.bsb + __ldg(d.tbg + tp.g);
        int32_t bo[TN];
#pragma unroll
        for (int j = 0; j < TN; ++j)
            bo[j] = __ldg(d.tbn + (tp.n0 + j < d.N ? tp.n0 + j : d.N - 1));
        // what the stores need is on its way beside the operands
        int32_t cn[TN];
#pragma unroll
        for (int j = 0; j < TN; ++j) cn[j] = __ldg(d.tcn + (tp.n0 + j < d.N ? tp.n0 + j : d.N - 1));
        T *Cb = (T *)d.C + tp.beta * d.bsc + __ldg(d.tcg + tp.g) + __ldg(d.tcm + (om ? m : 0));
        const unsigned long long ma = d.mxa ? d.mxa[tp.beta * d.mxa_bs] : 0ull;
        const unsigned long long mb = d.mxb ? d.mxb[tp.beta * d.mxb_bs] : 0ull;
        T acc[TN];
#pragma unroll
        for (int j = 0; j < TN; ++j) acc[j] = T(0);
        const int k0 = (int)(tp.split * d.kchunk);
        const int k1 = (int)min(d.K, (int64_t)k0 + d.kchunk);
        constexpr int U = TN == 1 ? 8 : TN == 2 ? 6 : 4;   // summed indices loaded together
        int k = k0 + ks;
        for (; k + (U - 1) * KL < k1; k += U * KL) {
            T a[U], b[U][TN];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int32_t ka = __ldg(d.tak + k + u * KL), kb = __ldg(d.tbk + k + u * KL);
                a[u] = __ldg(A + ka);
#pragma unroll
                for (int j = 0; j < TN; ++j) b[u][j] = __ldg(B + (bo[j] + kb));
            }
#pragma unroll
            for (int u = 0; u < U; ++u)
#pragma unroll
                for (int j = 0; j < TN; ++j) acc[j] += a[u] * b[u][j];
        }
#pragma unroll 2
        for (; k < k1; k += KL) {
            const int32_t ka = __ldg(d.tak + k), kb = __ldg(d.tbk + k);
            const T a = __ldg(A + ka);
#pragma unroll
            for (int j = 0; j < TN; ++j) acc[j] += a * __ldg(B + (bo[j] + kb));
        }
        for (int s = KL >> 1; s > 0; s >>= 1)
#pragma unroll
            for (int j = 0; j < TN; ++j) acc[j] += __shfl_xor_sync(0xffffffffu, acc[j], s);
        const bool st = om && ks == 0;
        if (d.nsplit > 1) {
            // unscaled partials, dense [split][item][g][n][m]
            T *P = part + (((int64_t)tp.split * d.nbeta + tp.beta) * d.G + tp.g) * d.M * d.N;
#pragma unroll
            for (int j = 0; j < TN; ++j)
                if (st && tp.n0 + j < d.N) P[(tp.n0 + j) * d.M + m] = acc[j];
        } else {
            const T sca = d.mxa ? pow2neg<T>(exp_of_bits(ma)) : T(1);
            const T scb = d.mxb ? pow2neg<T>(exp_of_bits(mb)) : T(1);
            const T sc = sca * scb;
#pragma unroll
            for (int j = 0; j < TN; ++j)
                if (st && tp.n0 + j < d.N) {
                    const T v = acc[j] * sc;
                    Cb[cn[j]] = v;
                    mx = mx > v ? mx : v;
                }
        }
    }
    if (!d.mxc || d.nsplit > 1) return;   // uniform
    // one recorded maximum per run of equal items in the block
#pragma unroll
    for (int s = 16; s > 0; s >>= 1) {
        const T o = __shfl_xor_sync(0xffffffffu, mx, s);
        mx = mx > o ? mx : o;
    }
    if (lane == 0) {
        smax[warp] = (double)mx;
        sbeta[warp] = beta;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 0; w < kThreads / 32;) {
            const int64_t b = sbeta[w];
            unsigned long long m = 0ull;
            for (; w < kThreads / 32 && sbeta[w] == b; ++w) {
                const unsigned long long o = dbits(smax[w]);
                m = o > m ? o : m;
            }
            if (b >= 0 && m) atomicMax(d.mxc + b, m);
        }
    }
}

template <typename T>
__global__ void __launch_bounds__(kThreads) k_bgemm_fin(const __grid_constant__ BDesc d,
                                                        const T *part) {
    const int64_t per = d.G * d.M * d.N, total = per * d.nbeta;
    const int64_t o = (int64_t)blockIdx.x * kThreads + threadIdx.x;
    const bool active = o < total;
    int64_t beta = 0;
    T v = 0;
    if (active) {
        beta = o / per;
        int64_t r = o - beta * per;
        const int64_t g = r / (d.M * d.N);
        r -= g * d.M * d.N;
        const int64_t n = r / d.M, m = r - n * d.M;
        T acc = 0;
        for (int sp = 0; sp < d.nsplit; ++sp) acc += part[(int64_t)sp * total + o];
        T sa = d.mxa ? pow2neg<T>(exp_of_bits(d.mxa[beta * d.mxa_bs])) : T(1);
        T sb = d.mxb ? pow2neg<T>(exp_of_bits(d.mxb[beta * d.mxb_bs])) : T(1);
        v = acc * (sa * sb);
        ((T *)d.C)[beta * d.bsc + d.tcg[g] + d.tcm[m] + d.tcn[n]] = v;
    }
    record_max(d.mxc, beta, active, (double)v);
}

// FP32 tile shapes (BM x BN, thread tiles TM x TN): 0 for n > 48, 1 for
// 16 < n <= 48, 2 for 8 < n <= 16, 3 for n <= 8 and few rows (128 x 8: the wider
// tiles would leave half of every row and, for short rows, half of every column
// idle), 4 for n > 64 and 5 for n <= 8 where there are rows enough.
constexpr int kBM[6] = {128, 256, 256, 128, 128, 256}, kBN[6] = {64, 32, 16, 8, 128, 8};
constexpr int kTM[6] = {8, 8, 8, 4, 8, 4}, kTN[6] = {4, 4, 2, 1, 8, 2};

// Launch one instantiation as a persistent grid: resident blocks per SM from
// the occupancy calculator (queried once), at most one block per tile.
template <int TILE, bool NFAST, int RQ>
void go(const BDesc &d, float *part, int64_t ntiles, cudaStream_t st) {
    // tile counts are checked on the host to fit 31 bits
    constexpr int BM = kBM[TILE], BN = kBN[TILE];
    constexpr size_t smem =
        (size_t)kStages * (Gather<BM>::SIZE + Gather<BN>::SIZE) * sizeof(float);
    auto kern = k_bgemm<BM, BN, kTM[TILE], kTN[TILE], NFAST, RQ>;
    static PerDevice once;
    static std::atomic<int> per_sm{1};   // the same on every sm_103a device
    const int dev = current_device();
    once.once(dev, [&] {
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        int b = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, kern, kThreads, smem) ==
                cudaSuccess &&
            b > 0)
            per_sm = b;
    });
    const int64_t grid = std::min<int64_t>(ntiles, (int64_t)sm_count(dev) * per_sm);
    kern<<<(unsigned)grid, kThreads, smem, st>>>(d, part, (int)ntiles);
}

template <int TILE>
void go_rows(const BDesc &d, float *part, int64_t ntiles, cudaStream_t st) {
    if (d.c_nfast) go<TILE, true, 4>(d, part, ntiles, st);
    else if (d.vc == 4) go<TILE, false, 4>(d, part, ntiles, st);
    else go<TILE, false, 2>(d, part, ntiles, st);
}

}  // namespace

// Direct form: warps wanted (eight an SM keep the FP64 pipe and the load
// latency covered), then the most columns per thread (loads of A shared), lanes
// per output and splits of the summed space that give them.
static int64_t direct_tasks(const BDesc &d) {
    const int64_t mw = 32 >> d.klog;
    return ((d.M + mw - 1) / mw) * ((d.N + d.direct - 1) / d.direct) * d.G * d.nbeta;
}
static void configure_direct(BDesc &d) {
    const int64_t want = 152LL * 8;
    // lanes run along rows: C's fastest group goes there when the columns fill
    // a warp's store
    if (d.c_nfast && d.N >= 16) {
        std::swap(d.M, d.N);
        std::swap(d.A, d.B);
        std::swap(d.bsa, d.bsb);
        std::swap(d.mxa, d.mxb);
        std::swap(d.mxa_bs, d.mxb_bs);
        std::swap(d.tag, d.tbg);
        std::swap(d.tam, d.tbn);
        std::swap(d.tcm, d.tcn);
        std::swap(d.tak, d.tbk);
        std::swap(d.a_kfast, d.b_kfast);
        d.c_nfast = 0;
    }
    d.klog = 0;
    while (d.klog < 5 && (16 >> d.klog) >= d.M && d.K >= (8LL << d.klog)) ++d.klog;
    d.direct = d.N >= 4 ? 4 : d.N >= 2 ? 2 : 1;
    // a long summed space is split over blocks (their loads of A still serve
    // four columns), a shorter one over the columns and lanes of a warp, which
    // needs no second kernel
    if (d.K < 4096) {
        while (d.direct > 1 && direct_tasks(d) < want) d.direct /= 2;
        while (d.klog < 5 && direct_tasks(d) < want && d.K >= (8LL << d.klog)) ++d.klog;
    }
    int64_t ns = 1;
    const int64_t tasks = direct_tasks(d);
    if (tasks < want && d.K >= 1024)
        ns = std::max<int64_t>(1, std::min<int64_t>((want + tasks - 1) / tasks, d.K / 512));
    d.kchunk = (d.K + ns - 1) / ns;
    d.kchunk = std::max<int64_t>((d.kchunk + 31) / 32 * 32, 32);
    d.nsplit = (int)std::max<int64_t>(1, (d.K + d.kchunk - 1) / d.kchunk);
}

// Tile shape and K split; d.tile = -1 when the contraction does not fit the
// kernels' 31-bit tile and group indices.
void bgemm_configure(BDesc &d, int elem_bytes) {
    d.direct = 0;
    d.klog = 0;
    d.tc = 0;
    d.tile = d.N > 48 ? 0 : d.N > 16 ? 1 : d.N > 8 ? 2 : 3;
    if (d.M >= (1LL << 31) || d.N >= (1LL << 31) || d.K >= (1LL << 31)) {
        d.tile = -1;
        return;
    }
    // FP64 always direct (the pipe's two multiply-adds a clock and SM leave
    // nothing for tiles to save); FP32 never: tiles and direct form measured the
    // same on the 24 x 24 grid's small nodes (3026 us a call against 3046)
    if (elem_bytes == 8) {
        configure_direct(d);
        if ((double)direct_tasks(d) * d.nsplit >= 1e10) d.tile = -1;
        return;
    }
    // 128 x 128 where that pads the columns no more than 128 x 64 and leaves
    // every SM two blocks
    if (d.N > 64 && (d.N + 127) / 128 * 128 <= (d.N + 63) / 64 * 64 * 9 / 8 &&
        ((d.M + 127) / 128) * ((d.N + 127) / 128) * d.G * d.nbeta >= 152 * 2)
        d.tile = 4;
    if (d.N <= 8 && ((d.M + 255) / 256) * d.G * d.nbeta >= 152 * 2) d.tile = 5;
    const int bm = kBM[d.tile], bn = kBN[d.tile];
    const int64_t tiles = ((d.M + bm - 1) / bm) * ((d.N + bn - 1) / bn) * d.G * d.nbeta;
    // split the summed space when the output tiles alone leave most SMs idle
    // and every split still runs several K steps; partials stay under 1 GiB
    int64_t ns = 1;
    // (then about four waves of two resident blocks per SM, so that the last
    // wave's idle SMs weigh little)
    const int64_t want = 152LL * 3;
    if (tiles < want && d.K >= 8 * kBK) {
        ns = std::min<int64_t>((152LL * 8 + tiles - 1) / tiles, d.K / (4 * kBK));
        const int64_t outs = d.G * d.M * d.N * d.nbeta;
        while (ns > 1 && (double)ns * outs * elem_bytes > (double)(1LL << 30)) ns /= 2;
        ns = std::max<int64_t>(1, ns);
    }
    int64_t chunk = (d.K + ns - 1) / ns;
    chunk = (chunk + kBK - 1) / kBK * kBK;
    d.kchunk = std::max<int64_t>(chunk, kBK);
    d.nsplit = (int)((d.K + d.kchunk - 1) / d.kchunk);
    if (d.nsplit < 1) d.nsplit = 1;
    // the kernels count tiles and index groups in 31 bits
    if ((double)tiles * d.nsplit >= 2147483647.0) d.tile = -1;
    // float data with whole K per tile and wide tiles: the tensor-core gather
    // kernel (with 32-column tiles its per-tile handoffs cost more than the
    // CUDA-core multiply-adds; measured on the 3-regular batched workload)
    d.tc = d.tile >= 0 && d.nsplit == 1 && d.N > 64 && d.M >= 128 &&
           (double)tc_gather_tiles(d) < 2147483647.0;
}

// One thread per table entry.  A single contraction builds its tables here (a
// 2^18-row node's 525 000 offsets: 1.3 ms of host loops and a 2 MB copy, now
// about 5 us on the device); programs build theirs once, on the host.
__global__ void __launch_bounds__(256) k_group_tables(const __grid_constant__ GroupTabs g,
                                                      int32_t *out) {
    for (int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x; i < g.total;
         i += (int64_t)gridDim.x * 256) {
        int t = 0;
        while (t < 8 && i >= g.start[t + 1]) ++t;
        uint32_t r = (uint32_t)(i - g.start[t]);   // groups hold fewer than 2^31 indices
        int64_t off = 0;
        for (int k = g.nd[t] - 1; k >= 0; --k) {
            const uint32_t q = r / (uint32_t)g.sz[t][k];
            off += (int64_t)(r - q * (uint32_t)g.sz[t][k]) * g.st[t][k];
            r = q;
        }
        out[i] = (int32_t)off;
    }
}

void launch_group_tables(const GroupTabs &g, int32_t *out, cudaStream_t st) {
    const int64_t blocks = std::min<int64_t>((g.total + 255) / 256, 152 * 8);
    k_group_tables<<<(unsigned)std::max<int64_t>(1, blocks), 256, 0, st>>>(g, out);
}

size_t bgemm_scratch_bytes(const BDesc &d, int elem_bytes) {
    if (d.nsplit <= 1) return 0;
    return (size_t)d.nsplit * (size_t)(d.G * d.M * d.N * d.nbeta) * (size_t)elem_bytes;
}

int bgemm_launches(const BDesc &d) { return d.nsplit > 1 && !d.tc ? 2 : 1; }

template <>
void launch_bgemm<double>(const BDesc &d, void *scratch, cudaStream_t st) {
    const int64_t outs = d.G * d.M * d.N * d.nbeta;
    if (outs == 0) return;
    const int64_t ntask = direct_tasks(d) * d.nsplit;
    const unsigned grid = (unsigned)((ntask + kThreads / 32 - 1) / (kThreads / 32));
    double *p = (double *)scratch;
    if (d.direct == 1) k_bgemm_direct<double, 1><<<grid, kThreads, 0, st>>>(d, p, ntask);
    else if (d.direct == 2) k_bgemm_direct<double, 2><<<grid, kThreads, 0, st>>>(d, p, ntask);
    else k_bgemm_direct<double, 4><<<grid, kThreads, 0, st>>>(d, p, ntask);
    if (d.nsplit > 1)
        k_bgemm_fin<double>
            <<<(unsigned)((outs + kThreads - 1) / kThreads), kThreads, 0, st>>>(d, p);
}

template <>
void launch_bgemm<float>(const BDesc &d, void *scratch, cudaStream_t st) {
    const int64_t outs = d.G * d.M * d.N * d.nbeta;
    if (outs == 0) return;
    if (d.tc) {
        launch_tc_gather(d, st);
        return;
    }
    const int bm = kBM[d.tile], bn = kBN[d.tile];
    const int64_t ntiles =
        ((d.M + bm - 1) / bm) * ((d.N + bn - 1) / bn) * d.G * d.nbeta * d.nsplit;
    float *part = (float *)scratch;
    switch (d.tile) {
        case 0: go_rows<0>(d, part, ntiles, st); break;
        case 1: go_rows<1>(d, part, ntiles, st); break;
        case 2: go_rows<2>(d, part, ntiles, st); break;
        case 3: go_rows<3>(d, part, ntiles, st); break;
        case 4: go_rows<4>(d, part, ntiles, st); break;
        default: go_rows<5>(d, part, ntiles, st); break;
    }
    if (d.nsplit > 1)
        k_bgemm_fin<float>
            <<<(unsigned)((outs + kThreads - 1) / kThreads), kThreads, 0, st>>>(d, part);
}

}  // namespace tn
