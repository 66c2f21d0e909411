// gen_dispatch.cu -- variant dispatch for occupancy / shared-memory queries and
// the on-demand FP64 evaluation of gBest rows.
#include <climits>

#include "bat_rows.cuh"
#include "sso_kernel.cuh"

namespace psso {

// One entry per (variant, width), each in its own object built from gen_variant.cu.
using GenFn = cudaError_t (*)(int, const KParams*, int, int, size_t, cudaStream_t, int*);
#define PSSO_DECL(v, m) \
    cudaError_t gen_variant_##v##_##m(int, const KParams*, int, int, size_t, cudaStream_t, int*);
PSSO_DECL(0, 1) PSSO_DECL(0, 2) PSSO_DECL(0, 4) PSSO_DECL(0, 8)
PSSO_DECL(1, 1) PSSO_DECL(1, 2) PSSO_DECL(1, 4) PSSO_DECL(1, 8)
PSSO_DECL(2, 1) PSSO_DECL(2, 2) PSSO_DECL(2, 4) PSSO_DECL(2, 8)
#undef PSSO_DECL

cudaError_t gen_call(int variant, int op, int mc_index, const KParams* p, int grid, int block,
                     size_t smem, cudaStream_t s, int* out)
{
    static const GenFn table[3][4] = {
        {gen_variant_0_1, gen_variant_0_2, gen_variant_0_4, gen_variant_0_8},
        {gen_variant_1_1, gen_variant_1_2, gen_variant_1_4, gen_variant_1_8},
        {gen_variant_2_1, gen_variant_2_2, gen_variant_2_4, gen_variant_2_8}};
    if (variant < 0 || variant > 2 || mc_index < 0 || mc_index > 3) return cudaErrorInvalidValue;
    return table[variant][mc_index](op, p, grid, block, smem, s, out);
}

// ---------------------------------------------------------------------------
// Batched throughput pipeline.
using BatFn = cudaError_t (*)(int, const BatParams*, int, int, cudaStream_t, int*);
#define PSSO_BDECL(v, m) \
    cudaError_t bat_variant_##v##_##m(int, const BatParams*, int, int, cudaStream_t, int*);
PSSO_BDECL(0, 1) PSSO_BDECL(0, 2) PSSO_BDECL(0, 4) PSSO_BDECL(0, 8)
PSSO_BDECL(1, 1) PSSO_BDECL(1, 2) PSSO_BDECL(1, 4) PSSO_BDECL(1, 8)
PSSO_BDECL(2, 1) PSSO_BDECL(2, 2) PSSO_BDECL(2, 4) PSSO_BDECL(2, 8)
#undef PSSO_BDECL

cudaError_t bat_call(int variant, int mc_index, int op, const BatParams* p, int grid, int block, cudaStream_t s,
                     int* out)
{
    static const BatFn table[3][4] = {
        {bat_variant_0_1, bat_variant_0_2, bat_variant_0_4, bat_variant_0_8},
        {bat_variant_1_1, bat_variant_1_2, bat_variant_1_4, bat_variant_1_8},
        {bat_variant_2_1, bat_variant_2_2, bat_variant_2_4, bat_variant_2_8}};
    if (variant < 0 || variant > 2 || mc_index < 0 || mc_index > 3) return cudaErrorInvalidValue;
    return table[variant][mc_index](op, p, grid, block, s, out);
}

using RowsFn = cudaError_t (*)(int, bool, int, const BatRowsParams*, int, cudaStream_t, int*);
#define PSSO_RDECL(v) cudaError_t rows_variant_##v(int, bool, int, const BatRowsParams*, int, cudaStream_t, int*);
PSSO_RDECL(0) PSSO_RDECL(1) PSSO_RDECL(2)
#undef PSSO_RDECL

cudaError_t bat_rows_call(int variant, int fn, bool wide, int op, const BatRowsParams* p, int grid, cudaStream_t s,
                          int* out)
{
    static const RowsFn table[3] = {rows_variant_0, rows_variant_1, rows_variant_2};
    if (variant < 0 || variant > 2) return cudaErrorInvalidValue;
    return table[variant](fn, wide, op, p, grid, s, out);
}

// gBest of one instance per block: the lowest-index arg-min of the pBests, then
// the record, log and gBest row.  FP32 bounds that leave more than one candidate
// queue the candidates without an FP64 value for bat_exact, which evaluates those
// of every swarm and finishes the swarm with its last one.  The last kernel's
// last block advances the generation.
//
// Bound: latency (a few loads and block reductions per swarm).  Only the keys
// are read and reduced -- FP32: the smallest and second-smallest lower bound,
// the first's index, the smallest upper bound; FP64: the value as an integer
// key and the index -- and the winner's other fields afterwards: 40 swarms,
// FP64, 17 -> 10 us per launch.  A swarm's candidates evaluated by its own block
// kept one SM's FP64 unit busy (6 us a row of 1000 variables) and most others
// idle: 512 swarms, FP32, generations 20-60: 111-188 -> 45-48 us for both
// kernels, 118.8 -> 101.5 ms per 150 generations (1 to 2 candidates a swarm).
struct BatKey {
    long long v;      // FP64: order_key of the value
    float l1, l2, mh; // FP32
    int i;
};
template <bool F32R>
__device__ __forceinline__ BatKey key_merge(const BatKey& a, const BatKey& b)
{
    BatKey r;
    if constexpr (F32R) {
        const bool bf = b.l1 < a.l1 || (b.l1 == a.l1 && b.i < a.i);
        r.v = 0;
        r.l1 = bf ? b.l1 : a.l1;
        r.i = bf ? b.i : a.i;
        r.l2 = fminf(fminf(a.l2, b.l2), bf ? a.l1 : b.l1);
        r.mh = fminf(a.mh, b.mh);
    } else {
        const bool bf = b.v < a.v || (b.v == a.v && b.i < a.i);
        r.v = bf ? b.v : a.v;
        r.i = bf ? b.i : a.i;
        r.l1 = r.l2 = r.mh = 0.f;
    }
    return r;
}
template <bool F32R>
__device__ __forceinline__ BatKey key_warp(BatKey k)
{
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        BatKey o;
        o.i = __shfl_xor_sync(0xffffffffu, k.i, off);
        o.v = F32R ? 0 : __shfl_xor_sync(0xffffffffu, k.v, off);
        o.l1 = F32R ? __shfl_xor_sync(0xffffffffu, k.l1, off) : 0.f;
        o.l2 = F32R ? __shfl_xor_sync(0xffffffffu, k.l2, off) : 0.f;
        o.mh = F32R ? __shfl_xor_sync(0xffffffffu, k.mh, off) : 0.f;
        k = key_merge<F32R>(k, o);
    }
    return k;
}
// Every thread gets the block's result (256 threads).
template <bool F32R>
__device__ __forceinline__ BatKey key_block(BatKey k, BatKey* sh)
{
    k = key_warp<F32R>(k);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = k;
    __syncthreads();
    k = sh[0];
#pragma unroll
    for (int w = 1; w < 8; ++w) k = key_merge<F32R>(k, sh[w]);
    return k;
}

// The rotated functions' rows, out of line (the whole-row code needs 255
// registers, which left an SM one block of the arg-min).
template <class Pos>
__device__ __noinline__ double exact_row_general(const Hot& in, const Pos* row)
{
    return fit64_row<Pos>(in, row, false);
}

// FP64 fitness of a row by one warp; the plain functions in rolled code (the
// unrolled whole-row code takes longer to fetch than to run once).
template <class Pos>
__device__ double exact_row(const Hot& in, const Pos* row)
{
    const int lane = threadIdx.x & 31, nq = (in.nchunks + 31) >> 5;
    switch (in.fn) {
#define PSSO_ROW_FN(F) \
    case F: return row_f64<F, Pos>(row + 4 * lane, true, lane, 32, in.nchunks, nq, in.D, in.o64, in.w64)
    PSSO_ROW_FN(FN_SPHERE);
    PSSO_ROW_FN(FN_ELLIPSOID);
    PSSO_ROW_FN(FN_RASTRIGIN);
    PSSO_ROW_FN(FN_ROSENBROCK);
    PSSO_ROW_FN(FN_ACKLEY);
#undef PSSO_ROW_FN
    default: return exact_row_general<Pos>(in, row);
    }
}

// Copies the winner's row to the gBest row and writes the record and the log
// (threads tid of nt); value: the winner's FP64 value when `exact`.
template <class Pos, bool F32R>
__device__ __forceinline__ void finish_swarm(const InstDev& d, BatCounters& cnt, long long g, int wi, bool exact,
                                             double value, unsigned extra, int tid, int nt)
{
    const Pos* src = static_cast<const Pos*>(d.P) + (int64_t)wi * d.Dp;
    Pos* dst = static_cast<Pos*>(d.gbrow);
    for (int q = tid; q < d.nchunks; q += nt) {
        Pos v[4];
        ld4(src + 4 * q, v);
        st4(dst + 4 * q, v);
    }
    if (tid != 0) return;
    Winner w;
    w.idx = wi;
    w.ver = d.pver[wi];
    w.acc = cnt.acc;
    w.rck = cnt.rck + extra;
    const bool has = exact || (F32R && (d.pflag[wi] & 1u));
    w.has64 = has ? 1 : 0;
    w.f64 = exact ? value : has ? d.pf64[wi] : 0.0;
    w.lo = exact ? f64_to_f32_rd(w.f64) : d.plo[wi];
    w.hi = exact ? f64_to_f32_ru(w.f64) : d.phi[wi];
    write_gbest(d, w, g);
    cnt.acc = 0;
    cnt.rck = 0;
}

template <class Pos, bool F32R>
__global__ void __launch_bounds__(256) bat_argmin(const InstDev* inst, const int32_t* ids, BatCtl* ctl, BatCounters* cnt)
{
    __shared__ BatKey sh[8];
    __shared__ unsigned n_list, n_placed, first;
    const int k = ids[blockIdx.x];
    const InstDev& d = inst[k];
    const long long g = ctl->gen;
    const int N = (int)d.N;
    const BatKey none = {LLONG_MAX, FLT_MAX, FLT_MAX, FLT_MAX, INT_MAX};
    BatKey c = none;
    for (int i = threadIdx.x; i < N; i += 256) {
        BatKey q = none;
        q.i = i;
        if constexpr (F32R) {
            q.l1 = d.plo[i];
            q.mh = d.phi[i];
        } else {
            q.v = order_key(d.pf64[i]);
        }
        c = key_merge<F32R>(c, q);
    }
    BatKey b = key_block<F32R>(c, sh);
    bool exact = !F32R;
    unsigned todo = 0;
    if constexpr (F32R) {
        if (b.l2 <= b.mh) {
            // the best of the FP64 values that are known, and the pBests without one
            // that can be the minimum
            const float m = b.mh;
            if (threadIdx.x == 0) n_list = n_placed = 0;
            __syncthreads();
            BatKey e = none;
            unsigned mine = 0;
            for (int i = threadIdx.x; i < N; i += 256) {
                if (d.pflag[i] & 1u) {
                    BatKey q = none;
                    q.i = i;
                    q.v = order_key(d.pf64[i]);
                    e = key_merge<false>(e, q);
                } else if (d.plo[i] <= m) {
                    ++mine;
                }
            }
            if (mine) atomicAdd(&n_list, mine);
            b = key_block<false>(e, sh);
            exact = true;
            todo = n_list;
            if (todo > 0) {
                if (threadIdx.x == 0) {
                    first = atomicAdd(&ctl->n_queue, todo);
                    BatPend& pd = ctl->pend[blockIdx.x];
                    pd.inst = k;
                    pd.first = first;
                    pd.n = todo;
                    pd.left = todo;
                    pd.key = b.v;
                    pd.i = b.i;
                }
                __syncthreads();
                for (int i = threadIdx.x; i < N; i += 256)
                    if (!(d.pflag[i] & 1u) && d.plo[i] <= m)
                        ctl->queue[first + atomicAdd(&n_placed, 1u)] = make_int2((int)blockIdx.x, i);
            }
        }
    }
    if (todo == 0) {
        const int wi = b.i < N ? b.i : 0;    // no finite value at all: the first particle
        finish_swarm<Pos, F32R>(d, cnt[k], g, wi, exact, exact ? d.pf64[wi] : 0.0, 0u, (int)threadIdx.x, 256);
    }
    if constexpr (!F32R) {
        // every block has read the generation before it takes a ticket
        if (threadIdx.x == 0) {
            __threadfence();
            if (atomicInc(&ctl->ticket, gridDim.x - 1) == gridDim.x - 1) ctl->gen = g + 1;
        }
    }
}

// The queued candidates' FP64 values, a warp per candidate; neighbours in the
// queue (one swarm's) go to different SMs.  The warp that completes a swarm's
// last candidate takes the exact arg-min.
template <class Pos>
__global__ void __launch_bounds__(256, 4) bat_exact(const InstDev* inst, BatCtl* ctl, BatCounters* cnt)
{
    const int lane = threadIdx.x & 31;
    const long long g = ctl->gen;
    const unsigned n = ctl->n_queue;
    for (unsigned e = (threadIdx.x >> 5) * gridDim.x + blockIdx.x; e < n; e += 8 * gridDim.x) {
        const int2 entry = ctl->queue[e];
        BatPend& pd = ctl->pend[entry.x];
        const int k = pd.inst, i = entry.y;
        const InstDev& d = inst[k];
        if (!PSSO_CHK(i >= 0 && i < d.N, CHK_BAT_ROW, i)) continue;
        const Pos* const row = static_cast<const Pos*>(d.P) + (int64_t)i * d.Dp;
        // (a converged swarm's candidates are mostly copies of the gBest row, whose
        // value is known: they take it; a gBest put there by psso_set_gbest has a
        // value of the caller's)
        bool copy = g > 0 && d.gb->has64 && d.gb->ver != 0xffffffffu;
        const double gf = d.gb->f64;
        const Pos* const gr = static_cast<const Pos*>(d.gbrow);
        for (int q = lane; q < d.nchunks && copy; q += 32) {
            Pos u[4], v[4];
            ld4(row + 4 * q, u);
            ld4(gr + 4 * q, v);
#pragma unroll
            for (int t = 0; t < 4; ++t) copy = copy && same_bits(u[t], v[t]);
        }
        copy = __all_sync(0xffffffffu, copy);
        const double f = copy ? gf : exact_row<Pos>(hot_of(d), row);
        unsigned left = 0;
        if (lane == 0) {
            d.pf64[i] = f;
            d.pflag[i] = 1u;
            d.plo[i] = f64_to_f32_rd(f);
            d.phi[i] = f64_to_f32_ru(f);
            __threadfence();
            left = atomicSub(&pd.left, 1u);
        }
        left = __shfl_sync(0xffffffffu, left, 0);
        if (left != 1u) continue;
        __threadfence();                     // the swarm's other values are visible
        BatKey w = {pd.key, 0.f, 0.f, 0.f, pd.i};
        for (unsigned q = lane; q < pd.n; q += 32) {
            BatKey o = w;
            o.i = ctl->queue[pd.first + q].y;
            o.v = order_key(__ldcg(d.pf64 + o.i));
            w = key_merge<false>(w, o);
        }
        w = key_warp<false>(w);
        const int wi = w.i < (int)d.N ? w.i : 0;
        finish_swarm<Pos, true>(d, cnt[k], g, wi, true, __ldcg(d.pf64 + wi), pd.n, lane, 32);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        if (atomicInc(&ctl->ticket, gridDim.x - 1) == gridDim.x - 1) {
            ctl->n_queue = 0;
            ctl->gen = g + 1;
        }
    }
}

__global__ void bat_set(long long* gen, long long g) { *gen = g; }

cudaError_t launch_bat_argmin(int variant, const InstDev* inst, const int32_t* ids, int n_ids, BatCtl* ctl,
                              BatCounters* cnt, int exact_grid, cudaStream_t s)
{
    if (variant == 0) bat_argmin<double, false><<<n_ids, 256, 0, s>>>(inst, ids, ctl, cnt);
    else if (variant == 1) bat_argmin<float, false><<<n_ids, 256, 0, s>>>(inst, ids, ctl, cnt);
    else {
        bat_argmin<float, true><<<n_ids, 256, 0, s>>>(inst, ids, ctl, cnt);
        bat_exact<float><<<exact_grid, 256, 0, s>>>(inst, ctl, cnt);
    }
    return cudaGetLastError();
}

cudaError_t launch_bat_set_gen(long long* gen, long long g, cudaStream_t s)
{
    bat_set<<<1, 1, 0, s>>>(gen, g);
    return cudaGetLastError();
}

// One block: psso_best's answer in one buffer.  Reading the status, the record
// and the row one by one, after a kernel and a synchronisation of its own for
// the FP64 value, took 43 us a call; one kernel and one copy take 32 us.
// (Written to pinned host memory by the kernel it is 24 us, but the memory costs
// 150-400 us at psso_create.)
template <class Pos>
__global__ void __launch_bounds__(128) best_pack(const InstDev* inst, int k, const StatusDev* status, BestPack* out)
{
    const InstDev& in = inst[k];
    const Pos* row = static_cast<const Pos*>(in.gbrow);
    Pos* dst = reinterpret_cast<Pos*>(out + 1);
    for (int j = threadIdx.x; j < in.Dp; j += blockDim.x) dst[j] = row[j];
    if (threadIdx.x >= 32) return;
    if (!in.gb->has64) {
        const double f = fit64_row<Pos>(hot_of(in), row, true);
        __syncwarp();
        if (threadIdx.x == 0) {
            in.gb->f64 = f;
            in.gb->has64 = 1;
        }
    }
    if (threadIdx.x == 0) {
        out->gb = *in.gb;
        out->status = *status;
    }
}

cudaError_t launch_best(const InstDev* inst, int k, int lattice, const StatusDev* status, BestPack* out, cudaStream_t s)
{
    if (lattice == 1) best_pack<float><<<1, 128, 0, s>>>(inst, k, status, out);
    else best_pack<double><<<1, 128, 0, s>>>(inst, k, status, out);
    return cudaGetLastError();
}

// One block per instance (three fills per instance took 2.3 us each on the host).
__global__ void reset_instances(const InstDev* inst)
{
    const InstDev& in = inst[blockIdx.x];
    const int n = SLOTS * in.R * REC_WORDS;
    for (int q = threadIdx.x; q < n; q += blockDim.x) in.rec[q] = in.rec2[q] = ~0ull;
    if (threadIdx.x == 0) *in.gb = GBestDev{};
}

cudaError_t launch_reset(const InstDev* inst, int n_inst, cudaStream_t s)
{
    reset_instances<<<n_inst, 128, 0, s>>>(inst);
    return cudaGetLastError();
}

}  // namespace psso
