// Micro-subtree kernel: one CTA evaluates every pairwise contraction of one
// small subtree of the contraction tree (forward), or the adjoint contractions
// of its nodes (backward).  Subtrees are independent, so one launch covers all
// of them; this replaces thousands of launches of microsecond-size kernels near
// the leaves of a tree (factor tensors absorbing unity vectors, fields and
// couplings) by one.
//
// Latency-bound: a node waits for its operands, and reading a record, two
// maxima and the operands from L2 costs about 3 us.  So the nodes go level by
// level (the nodes of a level are independent; 64-node subtrees have 8 to 30
// levels), a level's outputs are cut into warp tasks that the CTA's warps take
// in turn, and records, maxima and values lie in shared memory as far as they
// fit (inputs gathered at the start in one pass, results also written to the
// arena): a level costs shared-memory latencies and a barrier.  Outputs with a
// long summed space share it among up to 32 lanes.  10 x 10 grid, PR + MAR in
// FP64: 333 us for 63-node subtrees one node after another, 69 us now (and 33
// launches a call instead of 92); 300-variable network, max-plus: 144 us, 83 us
// when the whole tree of 599 nodes is one subtree.
#include <algorithm>
#include <cmath>

#include "devutil.cuh"
#include "kernels.cuh"
#include "micro.cuh"

namespace tn {

// Order-preserving integer keys: of non-negative values (their bits), and of
// any value (sign-folded bits; 0 sorts below all).
__device__ __forceinline__ unsigned long long key_of(float v) { return __float_as_uint(v); }
__device__ __forceinline__ unsigned long long key_of(double v) { return dbits(v); }
template <typename T> __device__ __forceinline__ T key_val(unsigned long long k);
template <> __device__ __forceinline__ float key_val<float>(unsigned long long k) {
    return __uint_as_float((uint32_t)k);
}
template <> __device__ __forceinline__ double key_val<double>(unsigned long long k) {
    return __longlong_as_double((long long)k);
}
__device__ __forceinline__ unsigned long long skey_of(float v) {
    const uint32_t b = __float_as_uint(v);
    return (b >> 31) ? ~b : b | 0x80000000u;
}
__device__ __forceinline__ unsigned long long skey_of(double v) { return okey(v); }
template <typename T> __device__ __forceinline__ T skey_val(unsigned long long k);
template <> __device__ __forceinline__ float skey_val<float>(unsigned long long k) {
    const uint32_t b = (uint32_t)k;
    return __uint_as_float((b >> 31) ? b & 0x7fffffffu : ~b);
}
template <> __device__ __forceinline__ double skey_val<double>(unsigned long long k) {
    return __longlong_as_double((long long)((k >> 63) ? k & 0x7fffffffffffffffull : ~k));
}
// Largest key among the lanes of a segment (seg = 32, a smaller power of two,
// or 0: the lane's own).
__device__ __forceinline__ unsigned long long warp_max(unsigned long long m, int seg) {
    if (seg == 32) {
        const uint32_t hi = __reduce_max_sync(0xffffffffu, (uint32_t)(m >> 32));
        const uint32_t lo =
            __reduce_max_sync(0xffffffffu, (uint32_t)(m >> 32) == hi ? (uint32_t)m : 0u);
        return ((unsigned long long)hi << 32) | lo;
    }
    for (int s = seg >> 1; s > 0; s >>= 1) {
        const unsigned long long o = __shfl_xor_sync(0xffffffffu, m, s);
        m = o > m ? o : m;
    }
    return m;
}

template <typename T, int SEMI>
__global__ void __launch_bounds__(MICRO_THREADS)
    k_micro(const unsigned char *__restrict__ blob, const MicroSub *__restrict__ subs, T *arena,
            unsigned long long *mx, int32_t *am) {
    extern __shared__ __align__(16) unsigned char sm[];
    const MicroSub sub = subs[blockIdx.x];
    const int nthr = blockDim.x;
    const uint32_t *src = (const uint32_t *)(blob + sub.off + sub.bytes);
    unsigned long long *smx = (unsigned long long *)(sm + sub.bytes);
    T *sv = (T *)(smx + ((sub.nmx + 1) & ~1));
    // the indices of the first gathers are on their way while the records come
    const uint32_t i0 = threadIdx.x < sub.nin ? __ldg(src + threadIdx.x) : 0u;
    const uint32_t q0 = threadIdx.x < sub.nmx ? __ldg(src + sub.nin + threadIdx.x) : 0u;
    for (int i = threadIdx.x; i < sub.bytes / 16; i += nthr)
        ((uint4 *)sm)[i] = __ldg((const uint4 *)(blob + sub.off) + i);
    if (threadIdx.x < sub.nin) sv[threadIdx.x] = arena[i0];
    if (threadIdx.x < sub.nmx) smx[threadIdx.x] = (q0 >> 31) ? 0ull : mx[q0];
#pragma unroll 4
    for (int i = threadIdx.x + nthr; i < sub.nin; i += nthr) sv[i] = arena[__ldg(src + i)];
    for (int i = threadIdx.x + nthr; i < sub.nmx; i += nthr) {
        const uint32_t q = __ldg(src + sub.nin + i);
        smx[i] = (q >> 31) ? 0ull : mx[q];
    }
    __syncthreads();
    const int32_t *lev = (const int32_t *)sm;
    const uint32_t *tasks = (const uint32_t *)(sm + sub.tasks);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int l = 0; l < sub.nlevels; ++l) {
        const int t1 = lev[l + 1];
        for (int t = lev[l] + warp; t < t1; t += nthr / 32) {
            const uint32_t task = tasks[t];
            const MicroHead &d = *(const MicroHead *)(sm + (task >> 16) * 16);
            const int4 *od = (const int4 *)(&d + 1), *kd = od + d.nout;
            const int kl = 1 << d.klog, ks = lane & (kl - 1);
            const int idx = (int)(task & 0xffffu) * (32 >> d.klog) + (lane >> d.klog);
            const bool on = idx < d.elems;
            const int at = on ? idx : 0;
            int beta = 0, o = at;
            if (d.nbeta > 1) {
                beta = at / d.nout_total;
                o = at - beta * d.nout_total;
            }
            unsigned long long ma = 0ull, mb = 0ull;
            if (d.smxa >= 0) ma = smx[d.smxa + beta * d.mxa_bs];
            else if (d.mxa >= 0) ma = __ldcg(mx + d.mxa + beta * d.mxa_bs);
            if (d.smxb >= 0) mb = smx[d.smxb + beta * d.mxb_bs];
            else if (d.mxb >= 0) mb = __ldcg(mx + d.mxb + beta * d.mxb_bs);
            unsigned long long *mc = d.smxc >= 0 ? smx + d.smxc : mx + d.mxc;
            int oa = beta * d.bsa, ob = beta * d.bsb;
            const bool pow2 = d.flags & 1;
            if (d.otab >= 0) {
                const uint32_t q = *(const uint32_t *)(sm + d.otab + 4 * o);
                oa += q & 0xffff;
                ob += q >> 16;
            } else if (pow2) {
                for (int q = 0; q < d.nout; ++q) {
                    const int4 g = od[q];
                    const int dg = (o >> g.y) & (g.x - 1);
                    oa += dg * g.z;
                    ob += dg * g.w;
                }
            } else {
                for (int q = d.nout - 1; q >= 0; --q) {
                    const int4 g = od[q];
                    const int r = o / g.x, dg = o - r * g.x;
                    o = r;
                    oa += dg * g.z;
                    ob += dg * g.w;
                }
            }
            const T *A = (d.sA >= 0 ? sv + d.sA : arena + d.offA) + oa;
            const T *B = (d.sB >= 0 ? sv + d.sB : arena + d.offB) + ob;
            const uint32_t *kt = (const uint32_t *)(sm + d.ktab);
            // offsets of summed index k without a table
            auto koff = [&](int k, int &ka, int &kb) {
                ka = kb = 0;
                if (pow2) {
                    for (int q = 0; q < d.nk; ++q) {
                        const int4 g = kd[q];
                        const int dg = (k >> g.y) & (g.x - 1);
                        ka += dg * g.z;
                        kb += dg * g.w;
                    }
                } else {
                    for (int q = d.nk - 1; q >= 0; --q) {
                        const int4 g = kd[q];
                        const int r = k / g.x, dg = k - r * g.x;
                        k = r;
                        ka += dg * g.z;
                        kb += dg * g.w;
                    }
                }
            };
            // lanes of one item within the warp (0: neighbours may differ)
            int seg = 32;
            if (d.nbeta > 1) {
                const int nout = d.nout_total;
                seg = (nout & (nout - 1)) ? 0 : min(32, nout << d.klog);
                if (seg == 0 &&
                    __all_sync(0xffffffffu, beta == __shfl_sync(0xffffffffu, beta, 0) || !on))
                    seg = 32;
            }
            if (SEMI == SUM) {
                T acc = 0;
                if (d.ktab >= 0) {
#pragma unroll 4
                    for (int k = ks; k < d.ktotal; k += kl) {
                        const uint32_t q = kt[k];
                        acc += A[q & 0xffff] * B[q >> 16];
                    }
                } else {
#pragma unroll 2
                    for (int k = ks; k < d.ktotal; k += kl) {
                        int ka, kb;
                        koff(k, ka, kb);
                        acc += A[ka] * B[kb];
                    }
                }
                for (int s = kl >> 1; s > 0; s >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, s);
                const T sa = d.mxa >= 0 ? pow2neg<T>(exp_of_bits(ma)) : T(1);
                const T sb = d.mxb >= 0 ? pow2neg<T>(exp_of_bits(mb)) : T(1);
                acc *= sa * sb;   // exact: both are powers of two
                if (on && ks == 0) {
                    arena[d.offC + idx] = acc;
                    if (d.sC >= 0) sv[d.sC + idx] = acc;
                }
                // the recorded maximum: non-negative values order like their bits
                if (d.mxc >= 0) {
                    const unsigned long long m = warp_max(key_of(on && acc > T(0) ? acc : T(0)), seg);
                    const bool first = seg ? (lane & (seg - 1)) == 0 : ks == 0;
                    if (on && first && m) {
                        const unsigned long long v = dbits((double)key_val<T>(m));
                        if (d.flags & 2) *mc = v;
                        else atomicMax(mc + beta, v);
                    }
                }
            } else {
                // operands max-normalised by their recorded maxima
                const T xa = d.mxa >= 0 ? okey_off<T>(ma) : T(0);
                const T xb = d.mxb >= 0 ? okey_off<T>(mb) : T(0);
                T best = -INFINITY;
                int bk = INT32_MAX;
                if (d.ktab >= 0) {
#pragma unroll 4
                    for (int k = ks; k < d.ktotal; k += kl) {
                        const uint32_t q = kt[k];
                        const T v = (A[q & 0xffff] - xa) + (B[q >> 16] - xb);
                        if (v > best) {
                            best = v;
                            bk = k;
                        }
                    }
                } else {
                    for (int k = ks; k < d.ktotal; k += kl) {
                        int ka, kb;
                        koff(k, ka, kb);
                        const T v = (A[ka] - xa) + (B[kb] - xb);
                        if (v > best) {
                            best = v;
                            bk = k;
                        }
                    }
                }
                // the largest value, ties to the lowest summed index
                for (int s = kl >> 1; s > 0; s >>= 1) {
                    const T v = __shfl_xor_sync(0xffffffffu, best, s);
                    const int k = __shfl_xor_sync(0xffffffffu, bk, s);
                    if (v > best || (v == best && k < bk)) {
                        best = v;
                        bk = k;
                    }
                }
                if (bk == INT32_MAX) bk = 0;
                if (on && ks == 0) {
                    arena[d.offC + idx] = best;
                    if (d.sC >= 0) sv[d.sC + idx] = best;
                    if (d.amoff >= 0) am[d.amoff + idx] = bk;
                }
                if (d.mxc >= 0) {
                    const unsigned long long m =
                        warp_max(on && best > T(-INFINITY) ? skey_of(best) : 0ull, seg);
                    const bool first = seg ? (lane & (seg - 1)) == 0 : ks == 0;
                    if (on && first && m) {
                        const double v = (double)skey_val<T>(m);
                        if (isfinite(v)) {
                            if (d.flags & 2) *mc = okey(v);
                            else atomicMax(mc + beta, okey(v));
                        }
                    }
                }
            }
        }
        __syncthreads();
    }
    for (int i = threadIdx.x; i < sub.nmx; i += nthr) {
        const uint32_t q = __ldg(src + sub.nin + i);
        if (q >> 31) mx[q & 0x7fffffffu] = smx[i];
    }
}

template <typename T>
void launch_micro(const unsigned char *blob, const MicroSub *subs, int nsub, int smem, int semiring,
                  int threads, T *arena, unsigned long long *mx, int32_t *am, cudaStream_t st) {
    if (nsub <= 0) return;
    static PerDevice once;
    once.once(current_device(), [] {
        cudaFuncSetAttribute(k_micro<T, SUM>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             MICRO_SMEM);
        cudaFuncSetAttribute(k_micro<T, MAXPLUS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             MICRO_SMEM);
    });
    if (semiring == SUM)
        k_micro<T, SUM><<<nsub, threads, smem, st>>>(blob, subs, arena, mx, am);
    else k_micro<T, MAXPLUS><<<nsub, threads, smem, st>>>(blob, subs, arena, mx, am);
}

template void launch_micro<float>(const unsigned char *, const MicroSub *, int, int, int, int, float *,
                                  unsigned long long *, int32_t *, cudaStream_t);
template void launch_micro<double>(const unsigned char *, const MicroSub *, int, int, int, int, double *,
                                   unsigned long long *, int32_t *, cudaStream_t);

}  // namespace tn
