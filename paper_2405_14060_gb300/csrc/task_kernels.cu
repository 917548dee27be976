// Task kernels around the pairwise contractions: leaf construction (factors,
// unity / evidence vectors), log Z from the root and the rescaling exponents,
// marginals from the adjoints of the unity vectors, factor marginals, MPE
// backtracking and backward sampling.
#include <algorithm>
#include <cfloat>
#include <cmath>

#include "devutil.cuh"
#include "task_kernels.cuh"

namespace tn {

__device__ __forceinline__ int exp_bits(unsigned long long b) {
    if (b == 0ull) return 0;
    return (int)((b >> 52) & 0x7ffull) - 1023;
}

// ------------------------------------------------------------------ leaves
//
// Factor leaf: the model's table (optionally its logarithm, for max-plus).
// Unity leaf of variable v (Sec. MAR step 1; Sec. MPE step 1): all ones for a
// free variable; for an observed variable the indicator of its value, which
// multiplies in the slicing T_{V|E=e} of Eq. pr.  In the log domain ones are
// 0 and zeros are -inf.  Each leaf records its maximum for rescaling.  One block
// per 256 entries of a table (a logarithm is some 50 FP64 operations, at two a
// clock and SM: an 18432-entry external leaf took 190 us in one block, 19 us now).
template <typename T>
__global__ void k_leaves(const LeafRec *recs, const double *tables, const int *card, int nvars,
                         const int32_t *evid, int nbeta, int log_mode, T *base,
                         unsigned long long *mx, const int *flags, const int32_t *slice_val) {
    const LeafRec &r = recs[blockIdx.x];
    T *dst = base + r.dst;
    __shared__ double smax[32];
    if (r.kind == LEAF_FACTOR || r.kind == LEAF_EXTERNAL) {
        if ((int64_t)blockIdx.y * blockDim.x >= r.size) return;
        double m = log_mode ? -INFINITY : 0.0;
        for (int64_t i = (int64_t)blockIdx.y * blockDim.x + threadIdx.x; i < r.size;
             i += (int64_t)gridDim.y * blockDim.x) {
            double x;
            if (r.kind == LEAF_FACTOR) {
                int64_t off = r.src + i;
                if (r.nkd >= 0) {
                    off = r.src;
                    int64_t q = i;
                    for (int j = r.nkd - 1; j >= 0; --j) {
                        off += (q % r.ksz[j]) * r.kst[j];
                        q /= r.ksz[j];
                    }
                    for (int j = 0; j < r.nsd; ++j) off += (int64_t)slice_val[r.sidx[j]] * r.sst[j];
                }
                x = tables[off] + 0.0;   // -0.0 (a valid entry) to 0.0: tensors order like their bits
                bool in_log = flags && flags[0];
                if (log_mode && !in_log) x = log(x);
                else if (!log_mode && in_log) x = exp(x);
            } else {
                // external: log of a sum-product result times 2^sigma
                const T *s = (const T *)(uintptr_t)r.src;
                double sig = r.sigma ? *r.sigma : 0.0;
                double v = (double)s[i];
                x = v > 0 ? log(v) + sig * 0.69314718055994530942 : -INFINITY;
            }
            dst[i] = (T)x;
            m = fmax(m, log_mode ? (double)(T)x : x);
        }
        // the maximum: a power-of-two scale source for sum-product, the
        // max-normalisation offset (order-preserving key) for max-plus
#pragma unroll
        for (int s = 16; s > 0; s >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, s));
        if ((threadIdx.x & 31) == 0) smax[threadIdx.x >> 5] = m;
        __syncthreads();
        if (threadIdx.x == 0) {
            double t = log_mode ? -INFINITY : 0.0;
            for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t = fmax(t, smax[w]);
            const unsigned long long k = log_mode ? (isfinite(t) ? okey(t) : 0ull)
                                                  : (unsigned long long)__double_as_longlong(t);
            if (r.size <= blockDim.x) mx[r.mx] = k;
            else if (k) atomicMax(mx + r.mx, k);   // zeroed at the start of every run
        }
    } else {
        if (blockIdx.y) return;
        int v = r.var, c = card[v];
        int nb = r.beta ? nbeta : 1;
        if (r.slice_of_var >= 0) {
            // a sliced variable's vector is the scalar u_v[slice value]
            int xs = slice_val[r.slice_of_var];
            for (int b = threadIdx.x; b < nb; b += blockDim.x) {
                int e = evid ? evid[(int64_t)b * nvars + v] : -1;
                bool one = e < 0 || e == xs;
                dst[b] = log_mode ? (one ? T(0) : T(-INFINITY)) : (one ? T(1) : T(0));
            }
            c = 1;
        } else
        for (int64_t t = threadIdx.x; t < (int64_t)nb * c; t += blockDim.x) {
            int b = (int)(t / c), x = (int)(t % c);
            int e = evid ? evid[(int64_t)b * nvars + v] : -1;
            bool one = e < 0 || e == x;
            dst[t] = log_mode ? (one ? T(0) : T(-INFINITY)) : (one ? T(1) : T(0));
        }
        if (!log_mode)
            for (int b = threadIdx.x; b < nb; b += blockDim.x)
                mx[r.mx + b] = (unsigned long long)__double_as_longlong(1.0);
    }
}

template <typename T>
void launch_leaves(const LeafRec *recs, int nrec, int64_t largest, const double *tables,
                   const int *card, int nvars, const int32_t *evid, int nbeta, int log_mode,
                   T *base, unsigned long long *mx, const int *flags, const int32_t *slice_val,
                   cudaStream_t st) {
    if (nrec <= 0) return;
    const int64_t parts = std::max<int64_t>(1, std::min<int64_t>((largest + 255) / 256, 256));
    k_leaves<T><<<dim3((unsigned)nrec, (unsigned)parts), 256, 0, st>>>(
        recs, tables, card, nvars, evid, nbeta, log_mode, base, mx, flags, slice_val);
}

// ------------------------------------------------------------ slicing

__global__ void k_slice_init(int nbeta, int64_t nm, double *M, double *S, double *A) {
    int b = blockIdx.x;
    if (threadIdx.x == 0) {
        M[b] = -INFINITY;
        S[b] = 0.0;
    }
    for (int64_t i = threadIdx.x; i < nm; i += blockDim.x) A[(int64_t)b * nm + i] = 0.0;
}

void launch_slice_init(int nbeta, int64_t nm, double *M, double *S, double *A, cudaStream_t st) {
    k_slice_init<<<nbeta, 256, 0, st>>>(nbeta, nm, M, S, A);
}

__global__ void k_slice_acc(int nbeta, const double *logz, const double *marg, int64_t nm,
                            const int32_t *slice_val, int nsl, const int32_t *sl_var,
                            const int64_t *sl_moff, const int32_t *sl_card, double *M, double *S,
                            double *A) {
    const int b = blockIdx.x;
    __shared__ double sh_scale, sh_w;
    __shared__ int sh_skip;
    if (threadIdx.x == 0) {
        double lz = logz[b];
        sh_skip = !(lz > -INFINITY);
        if (!sh_skip) {
            double m = M[b], scale = 1.0;
            if (!(m > -INFINITY) || lz > m) {
                scale = m > -INFINITY ? exp(m - lz) : 0.0;
                M[b] = lz;
                m = lz;
            }
            sh_scale = scale;
            sh_w = exp(lz - m);
            S[b] = S[b] * scale + sh_w;
        }
    }
    __syncthreads();
    if (sh_skip) return;
    const double scale = sh_scale, w = sh_w;
    double *a = A + (int64_t)b * nm;
    if (marg) {
        const double *p = marg + (int64_t)b * nm;
        for (int64_t i = threadIdx.x; i < nm; i += blockDim.x) a[i] = a[i] * scale + w * p[i];
        __syncthreads();
        for (int j = threadIdx.x; j < nsl; j += blockDim.x)
            a[sl_moff[j] + slice_val[j]] += w;
    }
    (void)sl_var;
    (void)sl_card;
}

void launch_slice_acc(int nbeta, const double *logz, const double *marg, int64_t nm,
                      const int32_t *slice_val, int nsl, const int32_t *sl_var,
                      const int64_t *sl_moff, const int32_t *sl_card, double *M, double *S,
                      double *A, cudaStream_t st) {
    k_slice_acc<<<nbeta, 256, 0, st>>>(nbeta, logz, marg, nm, slice_val, nsl, sl_var, sl_moff,
                                       sl_card, M, S, A);
}

__global__ void k_slice_fin(int nbeta, int64_t nm, const double *M, const double *S,
                            const double *A, double *logz, double *marg) {
    const int b = blockIdx.x;
    double s = S[b];
    if (threadIdx.x == 0) logz[b] = s > 0 ? M[b] + log(s) : -INFINITY;
    if (marg)
        for (int64_t i = threadIdx.x; i < nm; i += blockDim.x)
            marg[(int64_t)b * nm + i] = s > 0 ? A[(int64_t)b * nm + i] / s : NAN;
}

void launch_slice_fin(int nbeta, int64_t nm, const double *M, const double *S, const double *A,
                      double *logz, double *marg, cudaStream_t st) {
    k_slice_fin<<<nbeta, 256, 0, st>>>(nbeta, nm, M, S, A, logz, marg);
}

// ------------------------------------------------------------------- log Z
//
// log p(e_b) = ln(root_b) + ln2 * sum over every non-root tensor t of e_t(b),
// where e_t is the binary exponent removed when t was consumed.  sigma_out
// (optional) receives the log2 scale sum itself.
// One block per batch item; the exponents are integers, so the block-wide
// sum is exact in any order.
template <typename T>
__global__ void __launch_bounds__(256) k_logz(int nbeta, const T *root, int root_beta,
                                              const unsigned long long *mx, const int64_t *exps,
                                              int nexp, double *logz, double *sigma_out,
                                              int maxplus) {
    const int b = blockIdx.x;
    const double r = (double)root[root_beta ? b : 0];
    if (maxplus) {
        // log p = root + the offsets every consumer subtracted (FP64 sum in a
        // fixed order: per-thread strided sums, then a fixed tree)
        double s = 0.0;
        for (int i = threadIdx.x; i < nexp; i += blockDim.x) {
            int64_t idx = exps[2 * i], bs = exps[2 * i + 1];
            s += okey_off<double>(mx[idx + (bs ? b : 0)]);
        }
        __shared__ double dpart[8];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if ((threadIdx.x & 31) == 0) dpart[threadIdx.x >> 5] = s;
        __syncthreads();
        if (threadIdx.x == 0) {
            double t = 0.0;
            for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += dpart[w];
            logz[b] = r + t;
            if (sigma_out) sigma_out[b] = t;
        }
        return;
    }
    long long s = 0;
    for (int i = threadIdx.x; i < nexp; i += blockDim.x) {
        int64_t idx = exps[2 * i], bs = exps[2 * i + 1];
        s += exp_bits(mx[idx + (bs ? b : 0)]);
    }
    __shared__ long long part[8];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        long long t = 0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += part[w];
        if (sigma_out) sigma_out[b] = (double)t;
        logz[b] = r > 0 ? log(r) + (double)t * 0.69314718055994530942 : -INFINITY;
    }
}

template <typename T>
void launch_logz(int nbeta, const T *root, int root_beta, const unsigned long long *mx,
                 const int64_t *exps, int nexp, double *logz, double *sigma_out, int maxplus,
                 cudaStream_t st) {
    k_logz<T><<<nbeta, 256, 0, st>>>(nbeta, root, root_beta, mx, exps, nexp, logz, sigma_out,
                                     maxplus);
}

// --------------------------------------------------------------- adjoints

template <typename T>
__global__ void k_fill_one(T *p, int64_t n, unsigned long long *mx) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) {
        p[i] = T(1);
        if (mx) mx[i] = (unsigned long long)__double_as_longlong(1.0);
    }
}

template <typename T>
void launch_fill_one(T *p, int64_t n, unsigned long long *mx, cudaStream_t st) {
    k_fill_one<T><<<(unsigned)((n + 255) / 256), 256, 0, st>>>(p, n, mx);
}

// p(v = x | e_b) = u[x] * ubar[x] / sum_y u[y] * ubar[y]: the gradient of
// p(e) with respect to the unity vector of v is p(v, e) (Sec. MAR step 3),
// and the common scale of the stored adjoint cancels in the ratio.
template <typename T>
__global__ void k_marginals(const MargRec *recs, int nvars, int nbeta, const T *fbase,
                            const T *abase, double *marg, int64_t mstride) {
    int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= (int64_t)nvars * nbeta) return;
    int b = (int)(t / nvars), v = (int)(t % nvars);
    const MargRec r = recs[v];
    if (r.sliced) {
        double *o = marg + (int64_t)b * mstride + r.moff;
        for (int x = 0; x < r.card; ++x) o[x] = 0.0;
        return;
    }
    const T *u = fbase + r.fwd + (r.fbeta ? (int64_t)b * r.card : 0);
    const T *ub = abase + r.adj + (r.abeta ? (int64_t)b * r.card : 0);
    double s = 0;
    for (int x = 0; x < r.card; ++x) s += (double)u[x] * (double)ub[x];
    double *out = marg + (int64_t)b * mstride + r.moff;
    for (int x = 0; x < r.card; ++x)
        out[x] = s > 0 ? (double)u[x] * (double)ub[x] / s : NAN;
}

template <typename T>
void launch_marginals(const MargRec *recs, int nvars, int nbeta, const T *fbase, const T *abase,
                      double *marg, int64_t mstride, cudaStream_t st) {
    int64_t n = (int64_t)nvars * nbeta;
    k_marginals<T><<<(unsigned)((n + 127) / 128), 128, 0, st>>>(recs, nvars, nbeta, fbase, abase,
                                                               marg, mstride);
}

// Factor marginals p(scope_f = x | e_b) = T_f[x] * Tbar_f[x] / sum, which is
// d log p(e_b) / d log T_f[x] (Thm. "Tensor network differentiation").
template <typename T>
__global__ void k_factor_grads(const GradRec *recs, int nbeta, const T *fbase, const T *abase,
                               double *grad, int64_t gstride) {
    const GradRec r = recs[blockIdx.x];
    int b = blockIdx.y;
    const T *f = fbase + r.fwd;
    const T *fb = abase + r.adj + (r.abeta ? (int64_t)b * r.size : 0);
    __shared__ double ssum[32];
    double s = 0;
    for (int64_t i = threadIdx.x; i < r.size; i += blockDim.x) s += (double)f[i] * (double)fb[i];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) ssum[threadIdx.x >> 5] = s;
    __syncthreads();
    double tot = 0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) tot += ssum[w];
    double *out = grad + (int64_t)b * gstride + r.goff;
    for (int64_t i = threadIdx.x; i < r.size; i += blockDim.x)
        out[i] = tot > 0 ? (double)f[i] * (double)fb[i] / tot : NAN;
}

template <typename T>
void launch_factor_grads(const GradRec *recs, int nrec, int nbeta, const T *fbase,
                         const T *abase, double *grad, int64_t gstride, cudaStream_t st) {
    if (nrec <= 0) return;
    dim3 grid((unsigned)nrec, (unsigned)nbeta);
    k_factor_grads<T><<<grid, 128, 0, st>>>(recs, nbeta, fbase, abase, grad, gstride);
}

// ---------------------------------------------------------- MPE backtrack
//
// Top-down over the internal nodes: once the output labels of a node are
// assigned (root: none), the stored argmax at that position gives the values
// of the labels maximised at the node.  This is the Boolean mask rule of
// Eq. tropical-back with the mask of each node reduced to the single selected
// entry (ties resolved to the lowest flat index when the maximiser was
// recorded).
//
// Latency-bound: a node waits for its ancestors only, so the records come
// grouped by the number of maximising ancestors and one block per item takes a
// level at a time, one thread per node, with the records and the assignment in
// shared memory (a level then costs one dependent L2 load and a barrier).
// 300-variable network (290 maximising nodes of 599, 31 levels): 436 us with
// one thread walking all nodes, 31 us now.
template <bool SM>
__global__ void __launch_bounds__(256) k_backtrack(const BackHead h, const uint4 *blob,
                                                   const int32_t *argmax, int nvars,
                                                   int32_t *assign) {
    extern __shared__ __align__(16) unsigned char bsm[];
    const int b = blockIdx.x;
    int32_t *row = assign + (int64_t)b * nvars, *x = row;
    const unsigned char *rec = (const unsigned char *)blob;
    if (SM) {
        for (int i = threadIdx.x; i < h.bytes / 16; i += 256) ((uint4 *)bsm)[i] = __ldg(blob + i);
        x = (int32_t *)(bsm + h.bytes);
        rec = bsm;
    }
    // a variable of one value is maximised by no record: free, it takes that value
    for (int v = threadIdx.x; v < nvars; v += 256) x[v] = max(row[v], 0);
    __syncthreads();
    const BackNode *nodes = (const BackNode *)rec;
    const BackLab *labs = (const BackLab *)(rec + h.labs);
    const int2 *digs = (const int2 *)(rec + h.digs);
    const int32_t *lev = (const int32_t *)(rec + h.levels);
    for (int l = 0; l < h.nlevels; ++l) {
        for (int n = lev[l] + threadIdx.x; n < lev[l + 1]; n += 256) {
            const BackNode &d = nodes[n];
            int64_t o = d.aoff + b * d.per;
            for (int i = 0; i < d.nC; ++i) {
                const BackLab q = labs[d.lab0 + i];
                o += x[q.var] * q.stride;
            }
            int k = argmax[o];
            for (int i = d.nK - 1; i >= 0; --i) {
                const int2 g = digs[d.dig0 + i];
                const int q = k / g.y;
                x[g.x] = k - q * g.y;
                k = q;
            }
        }
        __syncthreads();
    }
    if (SM)
        for (int v = threadIdx.x; v < nvars; v += 256) row[v] = x[v];
}

void launch_backtrack(const BackHead &h, const uint4 *blob, const int32_t *argmax, int nbeta,
                      int nvars, int32_t *assign, cudaStream_t st) {
    constexpr size_t kCap = 200 * 1024;
    const size_t smem = (size_t)h.bytes + (size_t)nvars * 4;
    if (smem > kCap) {
        k_backtrack<false><<<nbeta, 256, 0, st>>>(h, blob, argmax, nvars, assign);
        return;
    }
    static PerDevice once;
    once.once(current_device(), [] {
        cudaFuncSetAttribute(k_backtrack<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)kCap);
    });
    k_backtrack<true><<<nbeta, 256, smem, st>>>(h, blob, argmax, nvars, assign);
}

// ------------------------------------------------------- backward sampling
//
// Philox4x32-10 (Salmon, Moraes, Dror, Shaw, "Parallel random numbers: as
// easy as 1, 2, 3", SC 2011): ten rounds of the Philox S-box with the
// multipliers 0xD2511F53, 0xCD9E8D57 and the Weyl key increments 0x9E3779B9,
// 0xBB67AE85 given in that paper.
struct P4 { uint32_t v[4]; };

__device__ __forceinline__ P4 philox4x32_10(P4 c, uint32_t k0, uint32_t k1) {
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        uint64_t p0 = (uint64_t)0xD2511F53u * c.v[0];
        uint64_t p1 = (uint64_t)0xCD9E8D57u * c.v[2];
        uint32_t hi0 = (uint32_t)(p0 >> 32), lo0 = (uint32_t)p0;
        uint32_t hi1 = (uint32_t)(p1 >> 32), lo1 = (uint32_t)p1;
        P4 n;
        n.v[0] = hi1 ^ c.v[1] ^ k0;
        n.v[1] = lo1;
        n.v[2] = hi0 ^ c.v[3] ^ k1;
        n.v[3] = lo0;
        c = n;
        k0 += 0x9E3779B9u;
        k1 += 0xBB67AE85u;
    }
    return c;
}

__device__ __forceinline__ double uniform01(uint64_t sample, uint32_t node, uint64_t seed) {
    P4 c;
    c.v[0] = (uint32_t)sample;
    c.v[1] = (uint32_t)(sample >> 32);
    c.v[2] = node;
    c.v[3] = 0;
    P4 r = philox4x32_10(c, (uint32_t)seed, (uint32_t)(seed >> 32));
    uint64_t m = ((uint64_t)(r.v[0] >> 5) << 26) | (uint64_t)(r.v[1] >> 6);   // 53 bits
    return (double)m * (1.0 / 9007199254740992.0);
}

// At a node C_Z = con({A_X, B_Y}, Z) with the sample's values s_Z already
// drawn, the eliminated labels M are drawn from A[s_Z, m] B[s_Z, m] / C[s_Z]
// (Eq. condition-prob); the stored tensors' common scales cancel.  Records
// (SampNode) hold only the nodes that draw something (K > 1), root first.
//
// One thread per sample.  What bounds it is the chain of draws, each a few
// dependent L2 loads, so everything beside that chain is kept short: the
// sample's values sit in shared memory ([variable][thread], consecutive lanes
// in consecutive bytes; rows of BT + 4 bytes so that the final transposed read
// meets no bank conflict), records, label lists and summed-offset tables are
// read at warp-uniform addresses in 16-byte pieces, and a summed space is
// scanned once: the running sum is kept at 16 block ends and only the block of
// the draw is read again (the same sums in the same order as a second full
// scan).  Summed spaces of 512 and more entries search the block sums of
// k_cdf_blocks where the executor planned them.  16 x 16 grid, FP64, 100000
// samples (166 drawing nodes of 991, one with 4096 entries): 26.2 ms with
// values in global memory, every node visited and two full scans; a whole call
// (forward pass and copy to the host included) went from 27.7 to 3.0 ms; with the
// draws of up to eight entries on integer comparisons the kernel went from 870 to
// 715 us.

// Draw among N or fewer summed assignments held in registers.
template <typename T, int N>
__device__ __forceinline__ int64_t samp_small(const T *A, const T *B,
                                              const longlong2 *__restrict__ kt, int K, double u) {
    // running sums: the last is the total, and the draw compares with each.
    // Sums of values without a sign order like their bits (the leaves turn -0.0
    // into 0.0), and integer comparisons leave the FP64 pipe (two operations a
    // clock and SM, what bounds the kernel) to the products and sums
    double c[N];
    unsigned long long w[N];
#pragma unroll
    for (int k = 0; k < N; ++k) {
        double v = 0;
        if (k < K) {
            const longlong2 o = __ldg(kt + k);
            v = (double)A[o.x] * (double)B[o.y];
        }
        w[k] = dbits(v);
        c[k] = k == 0 ? v : c[k - 1] + v;
    }
    const unsigned long long r0 = dbits(u * c[N - 1]);
    int pick = K - 1;
    bool done = false;
#pragma unroll
    for (int k = 0; k < N; ++k)
        if (!done && r0 < dbits(c[k]) && w[k] != 0ull) {
            pick = k;
            done = true;
        }
    return pick;
}

template <typename T, bool SM>
__global__ void __launch_bounds__(128) k_sample(const SampNode *__restrict__ nodes, int nnodes,
                                                const SampLab *__restrict__ labs,
                                                const int2 *__restrict__ digs,
                                                const longlong2 *__restrict__ ktab,
                                                const T *__restrict__ base,
                                                const double *__restrict__ cdf,
                                                const int32_t *__restrict__ evid, int nvars,
                                                int64_t nsamp, uint64_t seed, int8_t *out) {
    extern __shared__ __align__(16) int8_t xs[];
    const int BT = blockDim.x, tid = threadIdx.x;
    const int64_t s0 = (int64_t)blockIdx.x * BT, s = s0 + tid;
    // variable v of this thread's sample: x[v * xstep]
    int8_t *x = SM ? xs + tid : out + (s < nsamp ? s : nsamp - 1) * nvars;
    const int64_t xstep = SM ? BT + 4 : 1;
    if (s < nsamp) {
        for (int v = 0; v < nvars; ++v) {
            const int e = evid ? __ldg(evid + v) : -1;
            x[v * xstep] = (int8_t)(e >= 0 ? e : 0);
        }
        for (int n = 0; n < nnodes; ++n) {
            const SampNode nd = nodes[n];
            int64_t oa = nd.offA, ob = nd.offB, oc = 0;
#pragma unroll 4
            for (int i = 0; i < nd.nC; ++i) {
                const SampLab l = labs[nd.lab0 + i];
                const int64_t xv = x[l.var * xstep];
                oa += xv * l.sA;
                ob += xv * l.sB;
                oc += xv * l.sC;
            }
            const T *A = base + oa, *B = base + ob;
            const int64_t K = nd.K;
            const longlong2 *kt = ktab + nd.tab0;
            // product of the summed assignment k
            auto weight = [&](int64_t k) {
                if (nd.tab0 >= 0) {
                    const longlong2 o = __ldg(kt + k);
                    return (double)A[o.x] * (double)B[o.y];
                }
                int64_t ka = 0, kb = 0, r = k;
                for (int i = nd.nK - 1; i >= 0; --i) {
                    const int2 dg = digs[nd.dig0 + i];
                    const SampLab l = labs[nd.lab0 + nd.nC + i];
                    const int64_t d = r % dg.y;
                    r /= dg.y;
                    ka += d * l.sA;
                    kb += d * l.sB;
                }
                return (double)A[ka] * (double)B[kb];
            };
            const double u = uniform01((uint64_t)s, (uint32_t)nd.node, seed);
            int64_t pick = K - 1;
            if (K <= 2) {
                pick = samp_small<T, 2>(A, B, kt, (int)K, u);
            } else if (K <= 8) {
                pick = samp_small<T, 8>(A, B, kt, (int)K, u);
            } else if (nd.cdf >= 0) {
                const int64_t nblk = (K + nd.bs - 1) / nd.bs;
                const double *row = cdf + nd.cdf + oc * nblk;
                const double r = u * row[nblk - 1];
                int64_t lo = 0, hi = nblk - 1;
                while (lo < hi) {
                    const int64_t mid = (lo + hi) >> 1;
                    if (row[mid] > r) hi = mid;
                    else lo = mid + 1;
                }
                const int64_t k0 = lo * nd.bs, k1 = min(K, k0 + nd.bs);
                double c = lo ? row[lo - 1] : 0.0;
                pick = k1 - 1;
#pragma unroll 1
                for (int64_t k = k0; k < k1; ++k) {
                    const double w = weight(k);
                    c += w;
                    if (w > 0) {
                        pick = k;   // the block's last possible value if rounding hides the draw
                        if (r < c) break;
                    }
                }
            } else {
                double end[16];   // running sum at the end of each block
                double tot = 0;
                const int64_t bs = (K + 15) >> 4;
#pragma unroll 1
                for (int j = 0; j < 16; ++j) {
                    const int64_t k1 = min(K, (j + 1) * bs);
                    int64_t k = j * bs;
                    if (nd.tab0 >= 0)
                        for (; k + 4 <= k1; k += 4) {
                            double w[4];   // four loads in flight
#pragma unroll
                            for (int q = 0; q < 4; ++q) {
                                const longlong2 o = __ldg(kt + k + q);
                                w[q] = (double)A[o.x] * (double)B[o.y];
                            }
#pragma unroll
                            for (int q = 0; q < 4; ++q) tot += w[q];
                        }
#pragma unroll 1
                    for (; k < k1; ++k) tot += weight(k);
                    end[j] = tot;
                }
                const double r0 = u * tot;
                double c = 0;
                int64_t k0 = K;
#pragma unroll 1
                for (int j = 0; j < 16; ++j)
                    if (r0 < end[j]) {
                        k0 = j * bs;
                        c = j ? end[j - 1] : 0.0;
                        break;
                    }
#pragma unroll 1
                for (int64_t k = k0; k < K; ++k) {
                    const double w = weight(k);
                    c += w;
                    if (r0 < c && w > 0) { pick = k; break; }
                }
            }
            for (int i = nd.nK - 1; i >= 0; --i) {
                const int2 dg = digs[nd.dig0 + i];
                int d = (int)pick;
                if (nd.nK > 1) {
                    d = (int)(pick % dg.y);
                    pick /= dg.y;
                }
                x[dg.x * xstep] = (int8_t)d;
            }
        }
    }
    if (!SM) return;
    // the block's rows: BT samples x nvars bytes, contiguous in the output
    __syncthreads();
    const int rows = (int)min((int64_t)BT, nsamp - s0);
    int8_t *o = out + s0 * nvars;
    const int total = rows * nvars;
    if (((uintptr_t)o & 3) == 0) {
        for (int i = 4 * tid; i < total; i += 4 * BT) {
            int r = i / nvars, v = i - r * nvars;
            uint32_t w = 0;
            int j = 0;
            for (; j < 4 && i + j < total; ++j) {
                w |= (uint32_t)(uint8_t)xs[v * (BT + 4) + r] << (8 * j);
                if (++v == nvars) {
                    v = 0;
                    ++r;
                }
            }
            if (j == 4) *(uint32_t *)(o + i) = w;
            else
                for (int q = 0; q < j; ++q) o[i + q] = (int8_t)(w >> (8 * q));
        }
    } else {
        for (int i = tid; i < total; i += BT) o[i] = xs[(i % nvars) * (BT + 4) + i / nvars];
    }
}

template <typename T>
void launch_sample(const SampNode *nodes, int nnodes, const SampLab *labs, const int2 *digs,
                   const longlong2 *ktab, const T *base, const double *cdf, const int32_t *evid,
                   int nvars, int64_t nsamp, uint64_t seed, int8_t *out, cudaStream_t st) {
    // samples per block: as many as keep the values in 100 KB of shared
    // memory (two blocks an SM); beyond 100 KB at 32, the values stay in `out`
    constexpr size_t kCap = 100 * 1024;
    int bt = 128;
    while (bt > 32 && (size_t)nvars * (bt + 4) > kCap) bt /= 2;
    const size_t smem = (size_t)nvars * (bt + 4);
    if (smem > kCap) {
        k_sample<T, false><<<(unsigned)((nsamp + 127) / 128), 128, 0, st>>>(
            nodes, nnodes, labs, digs, ktab, base, cdf, evid, nvars, nsamp, seed, out);
        return;
    }
    static PerDevice once;
    once.once(current_device(), [] {
        cudaFuncSetAttribute(k_sample<T, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)kCap);
    });
    k_sample<T, true><<<(unsigned)((nsamp + bt - 1) / bt), bt, smem, st>>>(
        nodes, nnodes, labs, digs, ktab, base, cdf, evid, nvars, nsamp, seed, out);
}

// Block sums of a node's conditional weights: cdf[o][j] = sum of A[o, k] B[o, k]
// over summed indices k in [j bs, (j + 1) bs), one warp per (output entry o,
// block j), then running sums over j, one block of threads per output entry.
// A draw searches the nblk sums and scans one block, so the table is 1 / bs of
// a full cumulative table.
template <typename T>
__global__ void __launch_bounds__(256) k_cdf_blocks(const __grid_constant__ CDesc d, int bs,
                                                    int64_t nblk, int64_t total, double *cdf) {
    const int64_t w = ((int64_t)blockIdx.x * 256 + threadIdx.x) >> 5;
    if (w >= total) return;
    const int lane = threadIdx.x & 31;
    const int64_t o = w / nblk, j = w - o * nblk;
    int64_t oa = 0, ob = 0;
    {
        int64_t r = o;
        for (int i = d.nout - 1; i >= 0; --i) {
            const int64_t dg = r % d.osz[i];
            r /= d.osz[i];
            oa += dg * d.osa[i];
            ob += dg * d.osb[i];
        }
    }
    const T *A = (const T *)d.A + oa;
    const T *B = (const T *)d.B + ob;
    const int64_t k1 = min(d.ktotal, (j + 1) * bs);
    double s = 0;
    for (int64_t k = j * bs + lane; k < k1; k += 32) {
        int64_t ka = 0, kb = 0;
        if (d.pow2) {
            for (int i = 0; i < d.nk; ++i) {
                const int64_t dg = (k >> d.ksh[i]) & (int64_t)(d.ksz[i] - 1);
                ka += dg * d.ksa[i];
                kb += dg * d.ksb[i];
            }
        } else {
            int64_t r = k;
            for (int i = d.nk - 1; i >= 0; --i) {
                const int64_t dg = r % d.ksz[i];
                r /= d.ksz[i];
                ka += dg * d.ksa[i];
                kb += dg * d.ksb[i];
            }
        }
        s += (double)A[ka] * (double)B[kb];
    }
#pragma unroll
    for (int q = 16; q > 0; q >>= 1) s += __shfl_xor_sync(0xffffffffu, s, q);
    if (lane == 0) cdf[w] = s;
}

__global__ void __launch_bounds__(256) k_cdf_prefix(int64_t nblk, double *cdf) {
    double *row = cdf + (int64_t)blockIdx.x * nblk;
    const int64_t per = (nblk + 255) / 256;
    const int64_t j0 = threadIdx.x * per, j1 = min(nblk, j0 + per);
    double s = 0;
    for (int64_t j = j0; j < j1; ++j) s += row[j];
    __shared__ double pre[256];
    pre[threadIdx.x] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        double run = 0;
        for (int i = 0; i < 256; ++i) {
            const double t = pre[i];
            pre[i] = run;
            run += t;
        }
    }
    __syncthreads();
    double run = pre[threadIdx.x];
    for (int64_t j = j0; j < j1; ++j) {
        run += row[j];
        row[j] = run;
    }
}

template <typename T>
void launch_cdf_blocks(const CDesc &d, int64_t rows, int bs, double *cdf, cudaStream_t st) {
    const int64_t nblk = (d.ktotal + bs - 1) / bs, total = rows * nblk;
    k_cdf_blocks<T><<<(unsigned)((total + 7) / 8), 256, 0, st>>>(d, bs, nblk, total, cdf);
    k_cdf_prefix<<<(unsigned)rows, 256, 0, st>>>(nblk, cdf);
}

#define INST(T)                                                                                  \
    template void launch_leaves<T>(const LeafRec *, int, int64_t, const double *, const int *,  \
                                   int,                                                         \
                                   const int32_t *, int, int, T *, unsigned long long *,        \
                                   const int *, const int32_t *, cudaStream_t);                 \
    template void launch_logz<T>(int, const T *, int, const unsigned long long *,              \
                                 const int64_t *, int, double *, double *, int, cudaStream_t);  \
    template void launch_fill_one<T>(T *, int64_t, unsigned long long *, cudaStream_t);         \
    template void launch_marginals<T>(const MargRec *, int, int, const T *, const T *,          \
                                      double *, int64_t, cudaStream_t);                         \
    template void launch_factor_grads<T>(const GradRec *, int, int, const T *, const T *,       \
                                         double *, int64_t, cudaStream_t);                      \
    template void launch_sample<T>(const SampNode *, int, const SampLab *, const int2 *,        \
                                   const longlong2 *, const T *, const double *,                \
                                   const int32_t *, int, int64_t, uint64_t, int8_t *,           \
                                   cudaStream_t);                                               \
    template void launch_cdf_blocks<T>(const CDesc &, int64_t, int, double *, cudaStream_t);
INST(float)
INST(double)

}  // namespace tn
