// Dense pairwise contractions as batched GEMMs (the paper's "each pairwise
// contraction can be decomposed into BLAS operations", Sec. Tensor networks),
// written for sm_103a:
//
//   k_permute    operand preparation: a strided tensor to GEMM form
//                [batch][rows][K] (K contiguous), with the per-item exact
//                power-of-two rescale and the conversion to the GEMM input
//                type; also used to scatter a GEMM result into a tensor's
//                layout while recording its per-item maximum.
//   k_tc_gemm    tcgen05 tensor-core GEMM: D = X Y^T per batch, X and Y
//                K-major, TF32 (kind::tf32) or BF16 (kind::f16) inputs staged
//                by TMA (128-byte swizzle) through an mbarrier ring, FP32
//                accumulators in TMEM, epilogue through tcgen05.ld and shared
//                memory.  One thread issues TMA, one issues MMAs, four warps
//                drain TMEM.  128 x 256 tiles (ring of four slabs, two TMEM
//                buffers), persistent for short K, so that a tile's epilogue
//                overlaps the next tile's MMAs; 256 x 256 tiles (ring of
//                three, one buffer of two accumulators) for long K.
//   k_sgemm      FP32 GEMM on CUDA cores: four tile shapes, packed pairs.
//   k_simt_gemm  FP64 GEMM on CUDA cores, for contractions past the index
//                ranges of the direct kernel (bgemm.cu).
//
// Every mbarrier wait is bounded in time: a wait that exceeds ~2 s sets the
// error flag and the CTA skips the rest of its work.  Before it frees its
// TMEM and exits it waits (bounded again) for the asynchronous work it has
// already started: the TMA transfers of the last stages it issued and, via a
// final commit, every MMA it issued.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <mutex>
#include <vector>

#include "devutil.cuh"
#include "gemm.cuh"
#include "tcutil.cuh"

namespace tn {

// ------------------------------------------------------------- permute

template <typename TI, int OT>
__device__ __forceinline__ void store_conv(void *out, int64_t i, TI x);

// Element-wise form: one element per thread and step, in the input type (the
// scale is an exact power of two).
template <typename TI, int OT>
__global__ void __launch_bounds__(256) k_permute(const __grid_constant__ PDesc p, int64_t per) {
    // blockIdx.y = batch item when the outermost dimension is the batch label
    // and maxima are recorded (per = entries per item); else blockIdx.y = 0
    // and per = total.
    const int64_t item = blockIdx.y;
    TI mxv = 0;
    constexpr int U = 8;
    const TI *in = (const TI *)p.in;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i0 < per; i0 += stride * U) {
        int64_t oi[U], oo[U], beta[U];
        TI v[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            int64_t i = i0 + u * stride;
            const int64_t idx = item * per + (i < per ? i : 0);
            oi[u] = 0;
            oo[u] = 0;
            beta[u] = 0;
            if (p.pow2) {
                for (int d = 0; d < p.nd; ++d) {
                    int64_t dg = (idx >> p.sh[d]) & (int64_t)(p.sz[d] - 1);
                    oi[u] += dg * p.sin[d];
                    oo[u] += dg * p.sout[d];
                    if (d == p.beta_dim) beta[u] = dg;
                }
            } else {
                int64_t r = idx;
                for (int d = p.nd - 1; d >= 0; --d) {
                    int64_t dg = r % p.sz[d];
                    r /= p.sz[d];
                    oi[u] += dg * p.sin[d];
                    oo[u] += dg * p.sout[d];
                    if (d == p.beta_dim) beta[u] = dg;
                }
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) v[u] = in[oi[u]];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (i0 + u * stride >= per) continue;
            TI x = v[u];
            if (p.mxi) x *= pow2neg<TI>(exp_of_bits(p.mxi[beta[u] * p.mxi_bs]));
            store_conv<TI, OT>(p.out, oo[u], x);
            mxv = mxv > x ? mxv : x;
        }
    }
    if (p.mxo) block_max_atomic(p.mxo + item, (double)mxv);
}

template <typename TI, int OT>
__device__ __forceinline__ void store_conv(void *out, int64_t i, TI x) {
    if (OT == E_F64) ((double *)out)[i] = (double)x;
    else if (OT == E_F32) ((float *)out)[i] = (float)x;
    else ((__nv_bfloat16 *)out)[i] = __float2bfloat16_rn((float)x);
}

// Tiled form: each block walks a contiguous range of tiles (up to PT_MAXN
// entries each, input and output runs of at least 32 entries) through three
// shared-memory buffers: while tile q is written out, the asynchronous copies
// of tiles q + 1 and q + 2 are in flight, and one barrier per tile both
// publishes a landed tile and frees the buffer of the previous one.  Thread 0
// advances the tiles' base offsets digit by digit, three tiles ahead, and
// publishes them in shared memory.  Loads follow the input order (t.vin
// inputs per 16-byte copy when the plan allows), stores the output order
// (t.vec outputs per 16-byte store, their shared-memory slots read as one
// vector of 16-bit integers).
//
// One launch takes one or two permutations (blockIdx.z; the row and the column
// operand of a GEMM): their reads and writes overlap, and the last blocks of one
// do not leave the SMs idle before the other (1000 x 1155 and 777 x 1155, three
// items, to TF32: 27 us one after the other, 25 us together).
struct PPair {
    PDesc p[2];
    int64_t per[2];       // tiles per item
    int blocks[2], items[2];
};
template <typename TI, int OT>
__global__ void __launch_bounds__(256, 4) k_permute_tiled(const __grid_constant__ PPair a) {
    const PDesc &p = a.p[blockIdx.z];
    const int64_t per_item = a.per[blockIdx.z];
    const int nblocks = a.blocks[blockIdx.z];
    if ((int)blockIdx.x >= nblocks || (int)blockIdx.y >= a.items[blockIdx.z]) return;
    extern __shared__ __align__(16) unsigned char smraw[];
    __shared__ int64_t sbase[4][3];   // per tile (mod 4): input base, output base, item
    const PTile &t = p.tl;
    const int n = t.tn;
    const int nbuf = t.nbuf, swz = t.swz;
    TI *sm0 = (TI *)smraw;
    const int64_t item = blockIdx.y;
    const int32_t *tin = t.ttab, *tout = t.ttab + n;
    const uint16_t *slot = (const uint16_t *)(t.ttab + 2 * n);
    const TI *in = (const TI *)p.in;
    TI mxv = 0;
    // this block's tiles [q0, q1)
    const int64_t q0 = per_item * blockIdx.x / nblocks;
    const int64_t q1 = per_item * (blockIdx.x + 1) / nblocks;
    // digits of the last published tile (thread 0 only)
    int32_t dg[MAXD];
    int64_t cbi = 0, cbo = 0;
    if (threadIdx.x == 0) {
        uint32_t g = (uint32_t)(item * per_item + q0);
        for (int k = t.nrest - 1; k >= 0; --k) {
            uint32_t v;
            if (t.rsh[k] >= 0) {
                v = g & (uint32_t)(t.rsz[k] - 1);
                g >>= t.rsh[k];
            } else {
                v = g % (uint32_t)t.rsz[k];
                g /= (uint32_t)t.rsz[k];
            }
            dg[k] = (int32_t)v;
            cbi += (int64_t)v * t.rin[k];
            cbo += (int64_t)v * t.rout[k];
        }
    }
    // thread 0: publish the bases of tile q (called for q0, q0 + 1, ... in order)
    auto publish = [&](int64_t q) {
        if (threadIdx.x != 0 || q >= q1) return;
        if (q > q0) {
            for (int k = t.nrest - 1; k >= 0; --k) {
                cbi += t.rin[k];
                cbo += t.rout[k];
                if (++dg[k] < t.rsz[k]) break;
                cbi -= t.rin[k] * t.rsz[k];
                cbo -= t.rout[k] * t.rsz[k];
                dg[k] = 0;
            }
        }
        const int s = (int)(q & 3);
        sbase[s][0] = cbi;
        sbase[s][1] = cbo;
        sbase[s][2] = t.rest_beta >= 0 ? dg[t.rest_beta] : 0;
    };
    const bool vin = t.vin > 0 && ((uintptr_t)p.in & 15) == 0;
    // copies of tile q into buffer buf (an empty group past the range)
    auto issue = [&](int64_t q, int buf) {
        if (q < q1) {
            const int64_t bi = sbase[q & 3][0];
            const uint32_t s0 = (uint32_t)__cvta_generic_to_shared(sm0 + buf * nbuf);
            if (vin) {
                constexpr int GI = 16 / (int)sizeof(TI);
                for (int e = threadIdx.x * GI; e < n; e += 256 * GI)
                    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                                     s0 + (uint32_t)(pt_slot<sizeof(TI)>(e, swz) * sizeof(TI))),
                                 "l"(in + bi + __ldg(tin + e))
                                 : "memory");
            } else {
                for (int e = threadIdx.x; e < n; e += 256)
                    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(
                                     s0 + (uint32_t)(pt_slot<sizeof(TI)>(e, swz) * sizeof(TI))),
                                 "l"(in + bi + __ldg(tin + e)), "n"(sizeof(TI))
                                 : "memory");
            }
        }
        cp_async_commit();
    };
    const bool vec = t.vec > 0 && ((uintptr_t)p.out & 15) == 0;
    publish(q0);
    publish(q0 + 1);
    publish(q0 + 2);
    __syncthreads();
    issue(q0, 0);
    issue(q0 + 1, 1);
    int buf = 0;
    for (int64_t q = q0; q < q1; ++q) {
        cp_async_wait<1>();
        // every thread's copies of tile q landed, every thread is done with
        // tile q - 1 (its buffer is free), and the bases of q + 2 are visible
        __syncthreads();
        issue(q + 2, buf == 0 ? 2 : buf - 1);
        publish(q + 3);
        const int64_t bo = sbase[q & 3][1], beta = sbase[q & 3][2];
        const TI sc = p.mxi ? pow2neg<TI>(exp_of_bits(p.mxi[beta * p.mxi_bs])) : TI(1);
        const TI *sm = sm0 + buf * nbuf;
        if (vec) {
            constexpr int G = OT == E_F64 ? 2 : OT == E_F32 ? 4 : 8;
            for (int e0 = threadIdx.x * G; e0 < n; e0 += 256 * G) {
                uint16_t sl[G];
                if (G == 8) *(uint4 *)sl = __ldg((const uint4 *)(slot + e0));
                else if (G == 4) *(uint2 *)sl = __ldg((const uint2 *)(slot + e0));
                else *(uint32_t *)sl = __ldg((const uint32_t *)(slot + e0));
                TI x[G];
#pragma unroll
                for (int j = 0; j < G; ++j) {
                    x[j] = sm[sl[j]] * sc;
                    mxv = mxv > x[j] ? mxv : x[j];
                }
                const int64_t o = bo + __ldg(tout + e0);
                if (OT == E_BF16) {
                    uint4 v;
                    uint32_t *w = (uint32_t *)&v;
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        __nv_bfloat162 h = __floats2bfloat162_rn((float)x[2 * j], (float)x[2 * j + 1]);
                        w[j] = *(uint32_t *)&h;
                    }
                    *(uint4 *)((__nv_bfloat16 *)p.out + o) = v;
                } else if (OT == E_F32) {
                    *(float4 *)((float *)p.out + o) =
                        make_float4((float)x[0], (float)x[1], (float)x[2], (float)x[3]);
                } else {
                    *(double2 *)((double *)p.out + o) = make_double2((double)x[0], (double)x[1]);
                }
            }
        } else {
            for (int e = threadIdx.x; e < n; e += 256) {
                TI x = sm[__ldg(slot + e)] * sc;
                store_conv<TI, OT>(p.out, bo + __ldg(tout + e), x);
                mxv = mxv > x ? mxv : x;
            }
        }
        buf = buf == 2 ? 0 : buf + 1;
    }
    cp_async_wait<0>();
    if (p.mxo) block_max_atomic(p.mxo + item, (double)mxv);
}

void plan_permute_tiles(PDesc &p, PTabs &pt) {
    p.tl.tn = 0;
    pt.n = 0;
    if (p.nd < 2 || p.total < 8192 || p.total / 64 >= (1LL << 31)) return;
    struct D { int64_t sz, sin, sout; bool beta; };
    std::vector<D> d;
    for (int i = 0; i < p.nd; ++i) d.push_back({p.sz[i], p.sin[i], p.sout[i], i == p.beta_dim});
    constexpr int64_t RUN = 32;
    std::vector<char> in_u(d.size(), 0);
    int64_t n = 1;
    bool full = false;
    // dims below `lim` on one side (lim < 0: the next input-fastest dims
    // until the tile holds 2048 entries), up to `cap` entries in the tile (a
    // dim that would pass it is split; at PT_MAXN the tile is full)
    auto add_below = [&](bool by_in, int64_t lim, int64_t cap) {
        while (!full && (lim > 0 || n < 2048)) {
            int best = -1;
            for (int i = 0; i < (int)d.size(); ++i) {
                if (in_u[i] || d[i].beta || d[i].sz < 2) continue;
                int64_t st = by_in ? d[i].sin : d[i].sout;
                if (lim > 0 && st >= lim) continue;
                if (best < 0 || st < (by_in ? d[best].sin : d[best].sout)) best = i;
            }
            if (best < 0) return;
            if (n * d[best].sz <= cap) {
                in_u[best] = 1;
                n *= d[best].sz;
                continue;
            }
            int64_t lo = cap / n;
            while (lo >= 2 && d[best].sz % lo) --lo;
            if (lo >= 2) {
                D hi{d[best].sz / lo, d[best].sin * lo, d[best].sout * lo, false};
                D lw{lo, d[best].sin, d[best].sout, false};
                d[best] = hi;
                d.insert(d.begin() + best + 1, lw);
                in_u.insert(in_u.begin() + best + 1, 1);
                n *= lo;
            }
            if (cap >= PT_MAXN) full = true;
            return;
        }
    };
    // the input's contiguous side first, but at most 128 entries of it, so
    // that a long contiguous input run (a plain transpose) still leaves room
    // for at least 32 contiguous outputs; then the output's; then more of
    // the input's
    add_below(true, RUN, 4 * RUN);
    add_below(false, RUN, PT_MAXN);
    add_below(true, -1, PT_MAXN);
    if (n < 256) return;
    std::vector<int> U;
    for (int i = 0; i < (int)d.size(); ++i)
        if (in_u[i]) U.push_back(i);
    auto order_by = [&](bool by_in) {
        std::vector<int> o = U;
        std::sort(o.begin(), o.end(), [&](int a, int b) {
            return by_in ? d[a].sin < d[b].sin : d[a].sout < d[b].sout;
        });
        return o;   // fastest digit first
    };
    std::vector<int> oi = order_by(true), oo = order_by(false);
    // digit vector -> index in the input order
    std::vector<int64_t> wi(d.size(), 0);
    {
        int64_t w = 1;
        for (int i : oi) {
            wi[i] = w;
            w *= d[i].sz;
        }
    }
    {
        int64_t mi = 0, mo = 0;
        for (int i : U) {
            mi += (d[i].sz - 1) * d[i].sin;
            mo += (d[i].sz - 1) * d[i].sout;
        }
        if (mi >= (1LL << 31) || mo >= (1LL << 31) || U.size() > (size_t)MAXD) return;
    }
    PTile &t = p.tl;
    t.nrest = 0;
    t.rest_beta = -1;
    t.ntiles = 1;
    for (int i = 0; i < (int)d.size(); ++i) {
        if (in_u[i]) continue;
        if (t.nrest >= MAXD) return;
        if (d[i].beta) t.rest_beta = t.nrest;
        t.rsz[t.nrest] = (int32_t)d[i].sz;
        t.rsh[t.nrest] = (d[i].sz & (d[i].sz - 1)) ? -1 : __builtin_ctzll((unsigned long long)d[i].sz);
        t.rin[t.nrest] = d[i].sin;
        t.rout[t.nrest] = d[i].sout;
        t.ntiles *= d[i].sz;
        ++t.nrest;
    }
    // per-item maxima need the batch dim outermost (one item per grid row)
    if ((p.mxo && t.rest_beta > 0) || t.ntiles >= (1LL << 31)) return;
    t.tn = (int)n;
    t.ttab = nullptr;   // device table, set by the caller
    pt.n = (int)n;
    pt.esz = p.in_type == E_F64 ? 8 : 4;
    pt.ni = pt.no = (int)U.size();
    for (int q = 0; q < pt.ni; ++q) {
        pt.isz[q] = (int32_t)d[oi[q]].sz;
        pt.ioff[q] = (int32_t)d[oi[q]].sin;
        pt.osz[q] = (int32_t)d[oo[q]].sz;
        pt.ooff[q] = (int32_t)d[oo[q]].sout;
        pt.oin[q] = (int32_t)wi[oo[q]];
    }
    // 16-byte stores / input copies of G entries: every aligned group of G
    // entries (in output / input order) is contiguous and starts on a multiple
    // of G elements in every tile, that is, the contiguous run of the fastest
    // digits holds a multiple of G entries and every other stride is one
    auto groups = [&](int G, const int32_t *sz, const int32_t *off, int nd, const int64_t *rest) {
        if (n % G) return 0;
        int64_t run = 1;
        int q = 0;
        while (q < nd && off[q] == run) run *= sz[q++];
        if (run % G) return 0;
        for (; q < nd; ++q)
            if (off[q] % G) return 0;
        for (int k = 0; k < t.nrest; ++k)
            if (rest[k] % G) return 0;
        return G;
    };
    t.vec = groups(p.out_type == E_F64 ? 2 : p.out_type == E_F32 ? 4 : 8, pt.osz, pt.ooff, pt.no,
                   t.rout);
    t.vin = groups(p.in_type == E_F64 ? 2 : 4, pt.isz, pt.ioff, pt.ni, t.rin);
    // shared-memory layout: the one whose reads of a tile (output order, t.vec
    // entries per thread, or one) take the fewest wavefronts, counted on 16
    // warp-wide loads spread over the tile (all of a full tile's 128 cost 100 us
    // a permutation, more than it takes to run)
    {
        const int G = t.vec > 0 ? t.vec : 1;
        const int nload = ((int)n + 31) / 32, step = std::max(1, nload / 16);
        int ein[32][32], lanes[32], ns = 0;   // input index of every sampled lane
        for (int w = 0; w < nload && ns < 32; w += step, ++ns) {
            // load w: the 32 lanes of warp w / G, entry w % G of each
            int l = 0;
            for (; l < 32; ++l) {
                int r = ((w / G) * 32 + l) * G + w % G, x = 0;
                if (r >= (int)n) break;
                for (int q = 0; q < pt.no; ++q) {
                    const int y = r / pt.osz[q];
                    x += (r - y * pt.osz[q]) * pt.oin[q];
                    r = y;
                }
                ein[ns][l] = x;
            }
            lanes[ns] = l;
        }
        int best = -1;
        for (int swz = 0; swz < PT_NSWZ; ++swz) {
            int waves = 0;
            for (int w = 0; w < ns; ++w) {
                int8_t cnt[32] = {0};
                int32_t seen[32][32];
                int mx = 0;
                for (int l = 0; l < lanes[w]; ++l) {
                    const int slot = pt.esz == 8 ? pt_slot<8>(ein[w][l], swz)
                                                 : pt_slot<4>(ein[w][l], swz);
                    const int32_t word = slot * (pt.esz / 4);
                    const int bank = word & 31;
                    bool dup = false;   // per bank, the distinct words
                    for (int k = 0; k < cnt[bank]; ++k) dup = dup || seen[bank][k] == word;
                    if (!dup) seen[bank][cnt[bank]++] = word;
                    mx = std::max(mx, (int)cnt[bank]);
                }
                waves += mx;
            }
            if (best < 0 || waves < best) {
                best = waves;
                t.swz = swz;
            }
            if (best <= ns * (pt.esz / 4)) break;   // no conflict anywhere
        }
        t.nbuf = pt_nbuf((int)n, t.swz);
        pt.swz = t.swz;
    }
}

// Table entry e: input offset, output offset, shared-memory slot of the e-th
// output.
__host__ __device__ inline void permute_entry(const PTabs &t, int e, int32_t &in, int32_t &out,
                                              uint16_t &slot) {
    int r = e;
    in = 0;
    for (int q = 0; q < t.ni; ++q) {
        const int x = r / t.isz[q];
        in += (r - x * t.isz[q]) * t.ioff[q];
        r = x;
    }
    r = e;
    out = 0;
    int ein = 0;
    for (int q = 0; q < t.no; ++q) {
        const int x = r / t.osz[q], dg = r - x * t.osz[q];
        out += dg * t.ooff[q];
        ein += dg * t.oin[q];
        r = x;
    }
    slot = (uint16_t)(t.esz == 8 ? pt_slot<8>(ein, t.swz) : pt_slot<4>(ein, t.swz));
}

void fill_permute_table(const PTabs &t, int32_t *out) {
    uint16_t *slot = (uint16_t *)(out + 2 * t.n);
    for (int e = 0; e < t.n; ++e) permute_entry(t, e, out[e], out[t.n + e], slot[e]);
}

__global__ void __launch_bounds__(256) k_permute_tables(const __grid_constant__ PTabs3 a) {
    const PTabs &t = a.t[blockIdx.y];
    const int e = blockIdx.x * 256 + threadIdx.x;
    if (e >= t.n) return;
    int32_t *out = a.out[blockIdx.y];
    permute_entry(t, e, out[e], out[t.n + e], ((uint16_t *)(out + 2 * t.n))[e]);
}

void launch_permute_tables(const PTabs3 &a, cudaStream_t st) {
    int n = 0;
    for (auto &t : a.t) n = std::max(n, t.n);
    if (n > 0) k_permute_tables<<<dim3((unsigned)((n + 255) / 256), 3), 256, 0, st>>>(a);
}

// One or two (n) tiled permutations of the same types in one launch.
static void launch_tiled(const PDesc *const *ps, int n, cudaStream_t st) {
    PPair a;
    size_t sm = 0;
    int gx = 1, gy = 1;
    for (int i = 0; i < n; ++i)   // three tile buffers
        sm = std::max(sm, 3 * (size_t)ps[i]->tl.nbuf * (ps[i]->in_type == E_F64 ? 8 : 4));
    // as many blocks per SM as shared memory holds
    const int64_t bps = std::max<int64_t>(1, std::min<int64_t>(8, (227 * 1024) / (sm + 1024)));
    for (int i = 0; i < n; ++i) {
        const PDesc &p = *ps[i];
        a.p[i] = p;
        a.items[i] = (p.mxo && p.tl.rest_beta == 0) ? p.tl.rsz[0] : 1;
        a.per[i] = p.tl.ntiles / a.items[i];
        const int64_t cap = std::max<int64_t>(1, (152LL * bps) / a.items[i]);
        a.blocks[i] = (int)std::max<int64_t>(1, std::min(a.per[i], cap));
        gx = std::max(gx, a.blocks[i]);
        gy = std::max(gy, a.items[i]);
    }
    static PerDevice once;
    once.once(current_device(), [] {
        const int mx = 3 * pt_nbuf(PT_MAXN, 0) * 8;
        cudaFuncSetAttribute(k_permute_tiled<double, E_F64>,
                             cudaFuncAttributeMaxDynamicSharedMemorySize, mx);
        cudaFuncSetAttribute(k_permute_tiled<float, E_F32>,
                             cudaFuncAttributeMaxDynamicSharedMemorySize, mx);
        cudaFuncSetAttribute(k_permute_tiled<float, E_BF16>,
                             cudaFuncAttributeMaxDynamicSharedMemorySize, mx);
    });
    const dim3 grid((unsigned)gx, (unsigned)gy, (unsigned)n);
    const PDesc &p = *ps[0];
    if (p.in_type == E_F64) k_permute_tiled<double, E_F64><<<grid, 256, sm, st>>>(a);
    else if (p.out_type == E_F32) k_permute_tiled<float, E_F32><<<grid, 256, sm, st>>>(a);
    else k_permute_tiled<float, E_BF16><<<grid, 256, sm, st>>>(a);
}

int launch_permutes(const PDesc *x, const PDesc *y, cudaStream_t st) {
    auto tiled = [](const PDesc *p) { return p && p->total > 0 && p->tl.tn > 0 && p->tl.ttab; };
    // up to 2^25 entries each, where a launch's ramp and tail weigh: three
    // 1000 x 777 x 1155 products in TF32 133.5 -> 130.6 us a call, 4096^3 BF16 284 -> 276 (beyond, the
    // larger shared-memory tile of the two sets the blocks of both: 1.7 GB and
    // 5.5 GB operands took 2.36 ms together, 1.70 one after the other)
    if (tiled(x) && tiled(y) && x->in_type == y->in_type && x->out_type == y->out_type &&
        std::max(x->total, y->total) <= (1LL << 25)) {
        const PDesc *ps[2] = {x, y};
        launch_tiled(ps, 2, st);
        return 1;
    }
    if (x) launch_permute(*x, st);
    if (y) launch_permute(*y, st);
    return (x ? 1 : 0) + (y ? 1 : 0);
}

void launch_permute(const PDesc &p, cudaStream_t st) {
    if (p.total <= 0) return;
    if (p.tl.tn > 0 && p.tl.ttab) {
        const PDesc *ps[1] = {&p};
        launch_tiled(ps, 1, st);
        return;
    }
    int nitems = 1;
    if (p.mxo && p.beta_dim == 0) nitems = p.sz[0];
    int64_t per = p.total / nitems;
    dim3 grid = item_grid((per + 3) / 4, nitems);
    if (p.in_type == E_F64) k_permute<double, E_F64><<<grid, 256, 0, st>>>(p, per);
    else if (p.out_type == E_F32) k_permute<float, E_F32><<<grid, 256, 0, st>>>(p, per);
    else k_permute<float, E_BF16><<<grid, 256, 0, st>>>(p, per);
}

// ------------------------------------------------------------ tcgen05 GEMM

constexpr int TC_BM = 128, TC_BN = 256;
constexpr int TC_XBYTES = TC_BM * 128, TC_YBYTES = TC_BN * 128;    // one 128-byte K slab
// epilogue staging: per warp, 32 rows of 32 columns (rows of 36 floats, so that
// 16-byte accesses along and across rows meet no bank conflict)
constexpr int TC_EROW = 36, TC_EPI = 4 * 32 * TC_EROW * 4;
// MT blocks of 128 rows a tile: K slabs in the ring, shared memory
constexpr int tc_stages(int mt) { return mt == 2 ? 3 : 4; }
constexpr int tc_smem(int mt) {
    return tc_stages(mt) * (mt * TC_XBYTES + TC_YBYTES) + TC_EPI + 1024 + 256;
}
constexpr int TC_THREADS = 192;   // warps 0-3 epilogue, warp 4 MMA issuer, warp 5 TMA producer

struct TCParams {
    int64_t R, C, ldd, bsd;
    int64_t ntn, ntm;           // column / row tiles; tiles = batch x rows x columns
    int64_t ntiles;
    const unsigned long long *mxsx;   // scale of X applied to D (NULL: none)
    int kt;                     // number of 128-byte K slabs
    float *D;
    unsigned long long *mxd;
    int64_t beta_div_batch, beta_div_row;
    int *err;
    unsigned long long wait_ns;   // limit of the producer's and the MMA issuer's waits
};

// Tile t: batch item, first row, first column.  Within a batch item the
// row tiles go in groups of TC_GROUP, and a group's tiles run rows fastest,
// so that the tiles processed together read a few row panels of X and a few
// column panels of Y (which then stay in L2) rather than all of Y.
constexpr int TC_GROUP = 8;
template <int MT>
__device__ __forceinline__ void tc_tile(const TCParams &p, int64_t t, int &bz, int64_t &m0,
                                        int64_t &n0) {
    const int64_t per_b = p.ntn * p.ntm;
    bz = (int)(t / per_b);
    const int64_t rem = t - (int64_t)bz * per_b;
    const int64_t per_g = (int64_t)TC_GROUP * p.ntn;
    const int64_t grp = rem / per_g, loc = rem - grp * per_g;
    const int64_t rows = min((int64_t)TC_GROUP, p.ntm - grp * TC_GROUP);
    m0 = (grp * TC_GROUP + loc % rows) * (TC_BM * MT);
    n0 = (loc / rows) * TC_BN;
}

// Persistent: CTA b takes tiles b, b + grid, ...  The TMA warp fills a ring
// of three or four K slabs (X and Y tiles, 128-byte swizzle) across tile
// boundaries; the MMA warp accumulates tile i into one of two 256-column TMEM
// buffers (i & 1) while the four epilogue warps drain the other one, so a
// tile's TMEM -> global epilogue overlaps the next tile's MMAs.  Every wait
// is bounded: on a timeout the error flag is set, the producer waits for the
// copies it issued, the MMA warp for the MMAs it issued, and TMEM is freed.
template <int BF16, int MT>
__global__ void __launch_bounds__(TC_THREADS, 1)
    k_tc_gemm(const __grid_constant__ CUtensorMap tx, const __grid_constant__ CUtensorMap ty,
              const __grid_constant__ TCParams p) {
    constexpr int S = tc_stages(MT), XB = MT * TC_XBYTES;
    constexpr int NB = MT == 2 ? 1 : 2;   // accumulators of a tile that TMEM holds
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint8_t *sX = smem;
    uint8_t *sY = smem + S * XB;
    // barriers: full[S], empty[S], tfull[2], tempty[2], fin; then the TMEM slot
    float *sE = (float *)(sY + S * TC_YBYTES);
    uint64_t *bars = (uint64_t *)((uint8_t *)sE + TC_EPI);
    uint32_t *tslot = (uint32_t *)(bars + 2 * S + 5);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t full0 = smem_u32(bars), empty0 = smem_u32(bars + S),
                   tfull0 = smem_u32(bars + 2 * S),
                   tempty0 = smem_u32(bars + 2 * S + 2),
                   fin = smem_u32(bars + 2 * S + 4);
    const int mine = p.ntiles > (int64_t)blockIdx.x
                         ? (int)((p.ntiles - 1 - (int64_t)blockIdx.x) / gridDim.x) + 1
                         : 0;
    if (threadIdx.x == 0) {
        for (int s = 0; s < S; ++s) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(full0 + 8 * s));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(empty0 + 8 * s));
        }
        for (int a = 0; a < 2; ++a) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(tfull0 + 8 * a));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(tempty0 + 8 * a),
                         "r"(TC_BM));
        }
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(fin));
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(&tx) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(&ty) : "memory");
    }
    if (warp == 4) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         smem_u32(tslot)),
                     "r"(2 * TC_BN));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tslot;
    const int KT = p.kt;
    if (warp == 5) {
        if (lane == 0) {
            // ------------------------------------------------ TMA producer
            int q = 0;   // K slabs issued so far (all tiles)
            bool ok = true;
            for (int li = 0; li < mine && ok; ++li) {
                int bz;
                int64_t m0, n0;
                tc_tile<MT>(p, (int64_t)blockIdx.x + (int64_t)li * gridDim.x, bz, m0, n0);
                for (int kt = 0; kt < KT; ++kt, ++q) {
                    const int s = q % S;
                    if (q >= S &&
                        !mbar_wait(empty0 + 8 * s, ((q / S) - 1) & 1, p.err, p.wait_ns)) {
                        ok = false;
                        break;
                    }
                    const uint32_t fb = full0 + 8 * s;
                    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(fb),
                                 "r"(XB + TC_YBYTES)
                                 : "memory");
                    const int kx = kt * (BF16 ? 64 : 32);
#pragma unroll
                    for (int h = 0; h < MT; ++h)   // rows past the end are filled with zeros
                        asm volatile(
                            "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes"
                            " [%0], [%1, {%3, %4, %5}], [%2];" ::"r"(
                                smem_u32(sX + s * XB + h * TC_XBYTES)),
                            "l"(&tx), "r"(fb), "r"(kx), "r"((int)m0 + h * TC_BM), "r"(bz)
                            : "memory");
                    asm volatile(
                        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes"
                        " [%0], [%1, {%3, %4, %5}], [%2];" ::"r"(smem_u32(sY + s * TC_YBYTES)),
                        "l"(&ty), "r"(fb), "r"(kx), "r"((int)n0), "r"(bz)
                        : "memory");
                }
            }
            // the last transfers issued land before the CTA exits (already
            // the case when the MMA warp consumed them; it may have given up)
            for (int r = q > S ? q - S : 0; r < q; ++r)
                mbar_drain(full0 + 8 * (r % S), (r / S) & 1, p.err);
        }
        __syncwarp();
    } else if (warp == 4) {
        if (lane == 0) {
            // ------------------------------------------------- MMA issuer
            // D[128 x 256] (+)= X[128 x K] * Y[256 x K]^T, 4 MMAs of 32 bytes of K per slab
            const uint32_t idesc = (1u << 4) |                               // D: F32
                                   ((BF16 ? 1u : 2u) << 7) |                 // A: BF16 / TF32
                                   ((BF16 ? 1u : 2u) << 10) |                // B: BF16 / TF32
                                   ((uint32_t)(TC_BN >> 3) << 17) |          // N
                                   ((uint32_t)(TC_BM >> 4) << 24);           // M
            int q = 0;
            bool ok = true;
            for (int li = 0; li < mine && ok; ++li) {
                const int a = li % NB;
                // the epilogue has drained this TMEM buffer (tile li - NB)
                if (li >= NB && !mbar_wait(tempty0 + 8 * a, (li / NB - 1) & 1, p.err, p.wait_ns)) {
                    ok = false;
                    break;
                }
                tc_fence_after();
                const uint32_t acc_0 = tmem + (uint32_t)(a * TC_BN);
                for (int kt = 0; kt < KT; ++kt, ++q) {
                    const int s = q % S;
                    if (!mbar_wait(full0 + 8 * s, (q / S) & 1, p.err, p.wait_ns)) {
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    const uint64_t bd = sdesc_sw128(smem_u32(sY + s * TC_YBYTES));
#pragma unroll
                    for (int hk = 0; hk < 4 * MT; ++hk) {
                        const int kk = hk & 3, h = hk >> 2;   // K step, block of rows
                        const uint64_t ad = sdesc_sw128(smem_u32(sX + s * XB + h * TC_XBYTES));
                        const uint32_t acc_t = acc_0 + (uint32_t)(h * TC_BN);
                        const uint32_t accum = (kt | kk) ? 1u : 0u;
                        if (BF16)
                            asm volatile(
                                "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
                                " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(
                                    acc_t),
                                "l"(ad + 2 * kk), "l"(bd + 2 * kk), "r"(idesc), "r"(accum));
                        else
                            asm volatile(
                                "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
                                " tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n}\n" ::"r"(
                                    acc_t),
                                "l"(ad + 2 * kk), "l"(bd + 2 * kk), "r"(idesc), "r"(accum));
                    }
                    asm volatile(
                        "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                            empty0 + 8 * s)
                        : "memory");
                }
                if (ok)
                    asm volatile(
                        "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                            tfull0 + 8 * a)
                        : "memory");
            }
            // completes once every MMA issued above has finished (also after
            // a give-up), so that TMEM is idle when it is released
            (void)ok;
            asm volatile(
                "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(fin)
                : "memory");
            mbar_drain(fin, 0, p.err);
        }
        __syncwarp();
    } else {
        // ----------------------------------------------------- epilogue
        // warp w drains TMEM lanes 32w..32w+31 (rows of the tile)
        const float sxs = p.mxsx ? pow2neg<float>(exp_of_bits(*p.mxsx)) : 1.f;
        for (int li = 0; li < mine; ++li) {
            const int a = li % NB;
            bool have = mbar_wait(tfull0 + 8 * a, (li / NB) & 1, p.err, p.wait_ns);
            have = __all_sync(0xffffffffu, have);
            if (!have) break;
            tc_fence_after();
            int bz;
            int64_t m0, n0;
            tc_tile<MT>(p, (int64_t)blockIdx.x + (int64_t)li * gridDim.x, bz, m0, n0);
#pragma unroll 1
            for (int h = 0; h < MT; ++h) {
                const int64_t row = m0 + h * TC_BM + warp * 32 + lane;
                float mx = 0;
                float *D = p.D + (int64_t)bz * p.bsd;
                float *we = sE + warp * 32 * TC_EROW;
                const bool dvec = (p.ldd & 3) == 0 && (p.bsd & 3) == 0 && ((uintptr_t)p.D & 15) == 0;
                for (int ch = 0; ch < TC_BN / 32; ++ch) {
                    if (n0 + ch * 32 >= p.C) break;   // warp-uniform: no columns left
                    uint32_t r[32];
                    const uint32_t ta =
                        tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)((a + h) * TC_BN + ch * 32);
                    asm volatile(
                        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, "
                        "%10, %11, %12, %13, %14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, "
                        "%26, %27, %28, %29, %30, %31}, [%32];"
                        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]),
                          "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]),
                          "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]),
                          "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
                          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]),
                          "=r"(r[30]), "=r"(r[31])
                        : "r"(ta));
                    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                    // lanes hold rows: through shared memory, so that a warp stores
                    // 128 contiguous bytes of a row at a time (a lane writing its own
                    // row touched 32 half-used sectors per instruction: rows 3000, 777
                    // columns, TF32 38 us, 24 us now; 4.3 GB of results of the batched
                    // workload 2.06 ms, 1.60 ms now)
                    const int64_t c0 = n0 + ch * 32;
                    const bool in = row < p.R;
                    __syncwarp();   // the previous chunk has been read
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        float4 v;
                        v.x = __uint_as_float(r[4 * j + 0]) * sxs;
                        v.y = __uint_as_float(r[4 * j + 1]) * sxs;
                        v.z = __uint_as_float(r[4 * j + 2]) * sxs;
                        v.w = __uint_as_float(r[4 * j + 3]) * sxs;
                        *(float4 *)(we + lane * TC_EROW + 4 * j) = v;
                        // columns past C are products of zero-filled rows of Y
                        if (in) mx = fmaxf(mx, fmaxf(fmaxf(v.x, v.y), fmaxf(v.z, v.w)));
                    }
                    __syncwarp();
                    const int64_t rw = m0 + h * TC_BM + warp * 32;   // the warp's first row
                    if (dvec && c0 + 32 <= p.C) {
                        const int rl = lane >> 3, cq = (lane & 7) * 4;
                        float *d = D + (rw + rl) * p.ldd + c0 + cq;
#pragma unroll
                        for (int q = 0; q < 8; ++q)
                            if (rw + 4 * q + rl < p.R)
                                *(float4 *)(d + (int64_t)(4 * q) * p.ldd) =
                                    *(const float4 *)(we + (4 * q + rl) * TC_EROW + cq);
                    } else if (c0 + lane < p.C) {
                        const int nr = (int)min((int64_t)32, p.R - rw);
                        for (int q = 0; q < nr; ++q)
                            D[(rw + q) * p.ldd + c0 + lane] = we[q * TC_EROW + lane];
                    }
                }
                if (h == MT - 1) {
                    // this TMEM buffer may take the MMAs of tile li + NB
                    tc_fence_before();
                    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(tempty0 + 8 * a)
                                 : "memory");
                }
                const int64_t beta = p.beta_div_batch > 0 ? (int64_t)bz / p.beta_div_batch
                                     : p.beta_div_row > 0 ? (row < p.R ? row : p.R - 1) / p.beta_div_row
                                                          : 0;
                record_max(p.mxd, beta, row < p.R, (double)mx);
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 4)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                     "r"(2 * TC_BN));
}

static PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault,
                                             &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = (PFN_cuTensorMapEncodeTiled_v12000)p;
    });
    return fn;
}

bool tc_gemm_supported(const GDesc &g) {
    int es = g.xtype == E_BF16 ? 2 : 4;
    if (g.xtype == E_F64) return false;
    if (((uintptr_t)g.X | (uintptr_t)g.Y) & 15) return false;
    if ((g.ldx * es) % 16 || (g.ldy * es) % 16) return false;
    if (g.batch > 1 && ((g.bsx * es) % 16 || (g.bsy * es) % 16)) return false;
    if (g.R > (1LL << 31) - TC_BM || g.C > (1LL << 31) - TC_BN) return false;
    if (((g.C + TC_BN - 1) / TC_BN) * ((g.R + TC_BM - 1) / TC_BM) * g.batch >= (1LL << 31)) return false;
    if (g.K < 1) return false;
    return encode_fn() != nullptr;
}

static bool make_map(CUtensorMap *m, const void *base, int64_t K, int64_t rows, int64_t batch,
                     int64_t ld, int64_t bs, int es, bool bf16, int box_rows) {
    cuuint64_t dims[3] = {(cuuint64_t)K, (cuuint64_t)rows, (cuuint64_t)batch};
    cuuint64_t strides[2] = {(cuuint64_t)(ld * es), (cuuint64_t)((batch > 1 ? bs : rows * ld) * es)};
    cuuint32_t box[3] = {(cuuint32_t)(128 / es), (cuuint32_t)box_rows, 1};
    cuuint32_t estr[3] = {1, 1, 1};
    CUresult r = encode_fn()(m, bf16 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32,
                             3, (void *)base, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                             CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS;
}

cudaError_t launch_tc_gemm(const GDesc &g, int *err_flag, cudaStream_t st) {
    static PerDevice once;
    const int dev = current_device();
    once.once(dev, [] {
        cudaFuncSetAttribute(k_tc_gemm<0, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, tc_smem(1));
        cudaFuncSetAttribute(k_tc_gemm<1, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, tc_smem(1));
        cudaFuncSetAttribute(k_tc_gemm<0, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, tc_smem(2));
        cudaFuncSetAttribute(k_tc_gemm<1, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, tc_smem(2));
    });
    bool bf16 = g.xtype == E_BF16;
    int es = bf16 ? 2 : 4;
    CUtensorMap mx, my;
    if (!make_map(&mx, g.X, g.K, g.R, g.batch, g.ldx, g.bsx, es, bf16, TC_BM) ||
        !make_map(&my, g.Y, g.K, g.C, g.batch, g.ldy, g.bsy, es, bf16, TC_BN))
        return cudaErrorInvalidValue;
    TCParams p;
    p.R = g.R;
    p.C = g.C;
    p.ldd = g.ldd;
    p.bsd = g.bsd;
    int kel = 128 / es;
    p.kt = (int)((g.K + kel - 1) / kel);
    p.D = (float *)g.D;
    p.mxd = g.mxd;
    p.mxsx = g.mxsx;
    p.beta_div_batch = g.beta_div_batch;
    p.beta_div_row = g.beta_div_row;
    p.err = err_flag;
    // test hook: a shorter limit for the pipeline's waits (nanoseconds), so
    // that tests can make them give up without any fault
    p.wait_ns = TC_WAIT_NS;
    if (const char *w = getenv("TN_TEST_TC_WAIT_NS")) p.wait_ns = strtoull(w, nullptr, 10);
    p.ntn = (g.C + TC_BN - 1) / TC_BN;
    p.ntm = (g.R + TC_BM - 1) / TC_BM;
    p.ntiles = p.ntn * p.ntm * g.batch;
    if (p.ntiles >= (1LL << 31)) return cudaErrorInvalidConfiguration;
    // short K (at most 64 slabs): persistent, one CTA per SM (its shared
    // memory and the whole TMEM), each tile's epilogue overlapping the next
    // tile's MMAs; long K: one tile per CTA (the epilogue is a small part of
    // the tile, and CTAs started in tile order keep the concurrently read
    // operand panels close together in L2, where persistent CTAs drift apart
    // over hundreds of K slabs; measured on the batched workload's nodes)
    const int nsm = sm_count(dev);
    // long K: 256 x 256 tiles, whose accumulators fill TMEM, when that costs no
    // extra round of tiles.  128 x 256 tiles need 43 (TF32) or 85 (BF16)
    // multiply-adds a byte from L2, 23 to 26 TB/s at the tensor peak; these need
    // three quarters of that.  16384-long BF16 nodes of the batched workload 2.70 ->
    // 2.29 ms (1.92 PFLOP/s), 4096^3 TF32 nodes of the 24 x 24 grid 219 -> 175 us.
    // At 64 slabs and fewer the epilogue, which then overlaps nothing, costs as
    // much as it gains (4096^3 BF16 97 us either way) or more (K = 1024: 1.61 ms
    // against 2.26).
    const int64_t ntm2 = (g.R + 2 * TC_BM - 1) / (2 * TC_BM), t2 = p.ntn * ntm2 * g.batch;
    const bool wide = p.kt > 64 && g.R < (1LL << 30) &&
                      20 * ((t2 + nsm - 1) / nsm) <= 11 * ((p.ntiles + nsm - 1) / nsm);
    if (wide) {
        p.ntm = ntm2;
        p.ntiles = t2;
        if (bf16) k_tc_gemm<1, 2><<<(unsigned)t2, TC_THREADS, tc_smem(2), st>>>(mx, my, p);
        else k_tc_gemm<0, 2><<<(unsigned)t2, TC_THREADS, tc_smem(2), st>>>(mx, my, p);
        return cudaGetLastError();
    }
    dim3 grid((unsigned)(p.kt <= 64 ? std::min<int64_t>(p.ntiles, nsm) : p.ntiles), 1, 1);
    if (bf16) k_tc_gemm<1, 1><<<grid, TC_THREADS, tc_smem(1), st>>>(mx, my, p);
    else k_tc_gemm<0, 1><<<grid, TC_THREADS, tc_smem(1), st>>>(mx, my, p);
    return cudaGetLastError();
}

// ------------------------------------------------------- CUDA-core GEMMs

__global__ void __launch_bounds__(256) k_simt_gemm(const __grid_constant__ GDesc g) {
    using T = double;
    constexpr int BM = 64, BN = 64, BK = 16;
    __shared__ T sx[BK][BM + 1];
    __shared__ T sy[BK][BN + 1];
    const int t = threadIdx.x, ty = t / 16, tx = t % 16;
    // one flat tile index (columns fastest) keeps every grid extent in range
    const int64_t ntn = (g.C + BN - 1) / BN, ntm = (g.R + BM - 1) / BM;
    const int64_t b = (int64_t)blockIdx.x / (ntn * ntm), rem = (int64_t)blockIdx.x - b * ntn * ntm;
    const int64_t r0 = (rem / ntn) * BM, c0 = (rem % ntn) * BN;
    const T *X = (const T *)g.X + b * g.bsx;
    const T *Y = (const T *)g.Y + b * g.bsy;
    T acc[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = 0;
    for (int64_t k0 = 0; k0 < g.K; k0 += BK) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            int e = t + i * 256, rr = e / BK, kk = e % BK;
            int64_t gr = r0 + rr, gc = c0 + rr, gk = k0 + kk;
            sx[kk][rr] = (gr < g.R && gk < g.K) ? X[gr * g.ldx + gk] : T(0);
            sy[kk][rr] = (gc < g.C && gk < g.K) ? Y[gc * g.ldy + gk] : T(0);
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < BK; ++kk) {
            T a[4], c[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) a[i] = sx[kk][ty * 4 + i];
#pragma unroll
            for (int j = 0; j < 4; ++j) c[j] = sy[kk][tx * 4 + j];
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] += a[i] * c[j];
        }
        __syncthreads();
    }
    T mx = 0;
    T *D = (T *)g.D + b * g.bsd;
    const T sxs = g.mxsx ? pow2neg<T>(exp_of_bits(*g.mxsx)) : T(1);
    int64_t rowlast = r0 + ty * 4;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        int64_t r = r0 + ty * 4 + i;
        if (r >= g.R) continue;
        rowlast = r;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            int64_t c = c0 + tx * 4 + j;
            if (c < g.C) {
                const T v = acc[i][j] * sxs;
                D[r * g.ldd + c] = v;
                mx = mx > v ? mx : v;
            }
        }
    }
    bool any = r0 + ty * 4 < g.R;
    int64_t beta = g.beta_div_batch > 0 ? b / g.beta_div_batch
                   : g.beta_div_row > 0 ? (any ? rowlast : g.R - 1) / g.beta_div_row
                                        : 0;
    // rows ty*4..ty*4+3 of one thread may straddle items only if an item has
    // fewer than 4 rows; record per row in that case
    if (g.beta_div_row > 0 && g.beta_div_row < 4 && g.beta_div_batch <= 0) {
        for (int i = 0; i < 4; ++i) {
            int64_t r = r0 + ty * 4 + i;
            double m1 = 0;
            for (int j = 0; j < 4; ++j) {
                int64_t c = c0 + tx * 4 + j;
                if (r < g.R && c < g.C) m1 = fmax(m1, (double)acc[i][j]);
            }
            if (g.mxd && r < g.R && m1 > 0) atomicMax(g.mxd + r / g.beta_div_row, dbits(m1));
        }
        return;
    }
    record_max(g.mxd, beta, any, (double)mx);
}

// FP32 form: BM x BN tiles, eight warps, K steps of 16 through two shared
// buffers (global loads of the next step in registers while the current one is
// multiplied), TM x TN outputs a thread as pairs of rows (fma.rn.f32x2: two
// multiply-adds an instruction, so that shared loads and address work issue
// beside them).  A warp covers 4 x 8 lanes of quads without bank conflicts.
// Bound by the shared-memory pipe for small thread tiles (a word per lane and
// clock: 8 x 4 outputs take 12 clocks of loads for 8 of multiply-adds, 8 x 8 take
// 16 for 16, 12 x 8 take 20 for 24), else by the FP32 pipe.  2048 x 1536 x 1024:
// 316 us with 4 x 4 outputs a thread and scalar shared loads, 150 us
// now (192 x 128 tiles; 163 with 128 x 64, 192 with 128 x 128, 219 with 64 x 64).
__device__ __forceinline__ void unpack2(uint64_t v, float &lo, float &hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ uint64_t dup2(float v) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %1};" : "=l"(r) : "f"(v));
    return r;
}
__device__ __forceinline__ void fma2(uint64_t &d, uint64_t a, uint64_t b) {
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(a), "l"(b));
}

template <int BM, int BN, int TM, int TN>
__global__ void __launch_bounds__(256, TM * TN > 64 ? 1 : 2) k_sgemm(const __grid_constant__ GDesc g) {
    constexpr int BK = 16, LX = BM + 4, LY = BN + 4;
    constexpr int QM = TM / 4, QN = TN / 4;          // quads a thread holds each way
    constexpr int WM = BM / 4, WN = BN / 2;          // a warp's rows and columns
    static_assert(QM * 16 == WM && QN * 32 == WN, "warp tile");
    constexpr int LXN = BM / 64, LYN = BN / 64;      // 16-byte loads a thread and step
    __shared__ __align__(16) float sx[2][BK][LX];
    __shared__ __align__(16) float sy[2][BK][LY];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t ntn = (g.C + BN - 1) / BN, ntm = (g.R + BM - 1) / BM;
    const int64_t b = (int64_t)blockIdx.x / (ntn * ntm), rem = (int64_t)blockIdx.x - b * ntn * ntm;
    const int64_t r0 = (rem / ntn) * BM, c0 = (rem % ntn) * BN;
    const int q = tid & 3, lr = tid >> 2;            // K quad and row of this thread's loads
    const float *xp[LXN], *yp[LYN];
#pragma unroll
    for (int i = 0; i < LXN; ++i)
        xp[i] = (const float *)g.X + b * g.bsx + min(r0 + lr + 64 * i, g.R - 1) * g.ldx + 4 * q;
#pragma unroll
    for (int i = 0; i < LYN; ++i)
        yp[i] = (const float *)g.Y + b * g.bsy + min(c0 + lr + 64 * i, g.C - 1) * g.ldy + 4 * q;
    const int K = (int)g.K, nk = (K + BK - 1) / BK;
    float4 vx[LXN], vy[LYN];
    // entries past K are zero (the padding of a row is not written); K is
    // padded to a multiple of 8 in memory, so quads never leave the row
    auto load = [&](int ks) {
        const int k = ks * BK + 4 * q;
#pragma unroll
        for (int i = 0; i < LXN + LYN; ++i) {
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
            if (k < K) {
                v = __ldg((const float4 *)((i < LXN ? xp[i < LXN ? i : 0] : yp[i < LXN ? 0 : i - LXN]) +
                                           ks * BK));
                if (k + 1 >= K) v.y = 0.f;
                if (k + 2 >= K) v.z = 0.f;
                if (k + 3 >= K) v.w = 0.f;
            }
            if (i < LXN) vx[i < LXN ? i : 0] = v;
            else vy[i < LXN ? 0 : i - LXN] = v;
        }
    };
    auto store = [&](int s) {
#pragma unroll
        for (int i = 0; i < LXN; ++i) {
            const float *v = (const float *)&vx[i];
#pragma unroll
            for (int j = 0; j < 4; ++j) sx[s][4 * q + j][lr + 64 * i] = v[j];
        }
#pragma unroll
        for (int i = 0; i < LYN; ++i) {
            const float *v = (const float *)&vy[i];
#pragma unroll
            for (int j = 0; j < 4; ++j) sy[s][4 * q + j][lr + 64 * i] = v[j];
        }
    };
    const int tm = (warp >> 1) * WM + (lane >> 3) * 4;   // first row quad; the others 16 rows on
    const int tn = (warp & 1) * WN + (lane & 7) * 4;     // first column quad; the others 32 on
    uint64_t acc[TM / 2][TN];   // rows 2i, 2i + 1
#pragma unroll
    for (int i = 0; i < TM / 2; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) acc[i][j] = 0ull;
    load(0);
    store(0);
    __syncthreads();
    for (int ks = 0; ks < nk; ++ks) {
        const int s = ks & 1;
        if (ks + 1 < nk) load(ks + 1);
#pragma unroll
        for (int k = 0; k < BK; ++k) {
            uint64_t a[TM / 2];
            float y[TN];
#pragma unroll
            for (int i = 0; i < QM; ++i)
                *(ulonglong2 *)(a + 2 * i) = *(const ulonglong2 *)&sx[s][k][tm + 16 * i];
#pragma unroll
            for (int j = 0; j < QN; ++j)
                *(float4 *)(y + 4 * j) = *(const float4 *)&sy[s][k][tn + 32 * j];
#pragma unroll
            for (int j = 0; j < TN; ++j) {
                const uint64_t yy = dup2(y[j]);
#pragma unroll
                for (int i = 0; i < TM / 2; ++i) fma2(acc[i][j], a[i], yy);
            }
        }
        if (ks + 1 < nk) store(s ^ 1);
        __syncthreads();
    }
    float *D = (float *)g.D + b * g.bsd;
    const float sxs = g.mxsx ? pow2neg<float>(exp_of_bits(*g.mxsx)) : 1.f;
    const bool vec = (g.ldd & 3) == 0 && (g.bsd & 3) == 0 && ((uintptr_t)g.D & 15) == 0;
    float mxall = 0.f;
#pragma unroll
    for (int i = 0; i < TM; ++i) {
        const int64_t r = r0 + tm + (i >> 2) * 16 + (i & 3);
        float mx = 0.f;
#pragma unroll
        for (int j = 0; j < QN; ++j) {
            const int64_t c = c0 + tn + 32 * j;
            float v[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                float lo, hi;
                unpack2(acc[i >> 1][4 * j + e], lo, hi);
                v[e] = ((i & 1) ? hi : lo) * sxs;
            }
            if (r >= g.R) continue;
            if (vec && c + 4 <= g.C) {
                *(float4 *)(D + r * g.ldd + c) = make_float4(v[0], v[1], v[2], v[3]);
                mx = fmaxf(mx, fmaxf(fmaxf(v[0], v[1]), fmaxf(v[2], v[3])));
            } else {
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    if (c + e < g.C) {
                        D[r * g.ldd + c + e] = v[e];
                        mx = fmaxf(mx, v[e]);
                    }
            }
        }
        // rows of one tile may belong to different items
        if (g.mxd && g.beta_div_batch <= 0 && g.beta_div_row > 0)
            record_max(g.mxd, min(r, g.R - 1) / g.beta_div_row, r < g.R, (double)mx);
        else
            mxall = fmaxf(mxall, mx);
    }
    if (g.mxd && (g.beta_div_batch > 0 || g.beta_div_row <= 0))
        record_max(g.mxd, g.beta_div_batch > 0 ? b / g.beta_div_batch : 0, true, (double)mxall);
}

template <int BM, int BN>
static int64_t sgemm_tiles(const GDesc &g) {
    return ((g.C + BN - 1) / BN) * ((g.R + BM - 1) / BM) * g.batch;
}
void launch_simt_gemm(const GDesc &g, cudaStream_t st) {
    if (g.xtype == E_F64) {
        dim3 grid((unsigned)(((g.C + 63) / 64) * ((g.R + 63) / 64) * g.batch), 1, 1);
        k_simt_gemm<<<grid, 256, 0, st>>>(g);
        return;
    }
    // the tile whose busiest SM has the least work: tiles per SM, rounded up,
    // times a tile's outputs, over the share of the FP32 rate it reaches
    const int64_t t0 = sgemm_tiles<192, 128>(g), t1 = sgemm_tiles<128, 128>(g),
                  t2 = sgemm_tiles<128, 64>(g), t3 = sgemm_tiles<64, 64>(g);
    auto cost = [](int64_t t, int out, double rate) { return (double)((t + 151) / 152) * out / rate; };
    const double c0 = cost(t0, 192 * 128, 0.73), c1 = cost(t1, 128 * 128, 0.76),
                 c2 = cost(t2, 128 * 64, 0.67), c3 = cost(t3, 64 * 64, 0.5);
    const double c = std::min(std::min(c0, c1), std::min(c2, c3));
    if (c == c0) k_sgemm<192, 128, 12, 8><<<(unsigned)t0, 256, 0, st>>>(g);
    else if (c == c1) k_sgemm<128, 128, 8, 8><<<(unsigned)t1, 256, 0, st>>>(g);
    else if (c == c2) k_sgemm<128, 64, 8, 4><<<(unsigned)t2, 256, 0, st>>>(g);
    else k_sgemm<64, 64, 4, 4><<<(unsigned)t3, 256, 0, st>>>(g);
}

}  // namespace tn
