// tc_pair.cuh -- persistent tensor-core GEMM over operand planes by CTA pairs
// (tcgen05 cta_group::2): C tiles of 256 x 128, D_ij = sum over products q of
// sum_k A[pa(q)]_ik B[pb(q)]_jk, each product into its accumulator.
//
// Why pairs.  With one CTA per 128 x 64 tile an MMA read 6 KiB of shared
// memory for 32 clocks of math and a K block of all planes (96 KiB) came from
// L2 for every 128 x 64 x 64 of output: the tensor pipe was busy 48 % of the
// time.  A pair multiplies 256 x 128: each CTA stages its own 128 rows of A and
// half of the tile's B rows (the other half is read from the peer's shared
// memory by the tensor core), so the same 96 KiB per CTA and K block carries
// twice the math, and an MMA reads 6 KiB per 64 clocks.
//
// Tensor memory: four accumulators of 128 columns fill all 512 columns, so
// there is one accumulator set.  Eight epilogue warps (two per lane quarter, 64
// columns each) first join the accumulators into registers, release the set to
// the next tile's MMAs, and then compute on the registers: only the join (about
// 1500 clocks against 10000 to 41000 of a tile's MMAs) is exposed.
//
// Tiles: numbered with the column tile fastest (pairs working at the same time
// share A through L2), dealt round robin to the pairs.  When the tiles of the
// last round are at most half as many as the pairs, each is cut into two 64
// columns wide, so the last round takes 0.6 instead of 1 of a tile's time.  A
// tile whose second half lies beyond the columns is 64 columns wide as well.
//
// Roles (320 threads): warp 0 issues the CTA's TMA copies (all CTAs of the pair
// signal the leader's full barriers), warp 1 issues the MMAs (leader only) and
// owns the tensor memory, warps 2..9 run the epilogue.  Barriers: full[s]
// (leader: one arrival and both CTAs' bytes), empty[s] (both CTAs: committed by
// the leader's MMAs), tfull (both CTAs: a tile's MMAs are complete), tempty
// (leader: the 16 epilogue warps of the pair).  Every wait on them is bounded;
// the barriers without a limit (the two warps of a lane quarter, the block, the
// cluster) are reached by all their threads whether a wait ran out or not.
#pragma once
#include "pdl.cuh"
#include "tc_gemm.cuh"

namespace psso {
namespace tc {

constexpr int PBM = 256, PBN = 128;             // pair tile
constexpr int P_THREADS = 320;
constexpr int P_EPI_WARPS = 8;
constexpr int P_A_BYTES = 128 * BK * 2;         // 16 KiB: one A plane's K block of one CTA
constexpr int P_B_BYTES = 64 * BK * 2;          // 8 KiB: its half of the B rows

template <int PLANES, int STG>
constexpr int pair_smem() { return STG * PLANES * (P_A_BYTES + P_B_BYTES) + 1024; }

__device__ __forceinline__ uint32_t cluster_rank()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cluster_sync()
{
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// The address of this CTA's shared-memory location in CTA `rank` of the cluster.
__device__ __forceinline__ uint32_t map_rank(uint32_t addr, uint32_t rank)
{
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
// Copies a box into this CTA's shared memory; the bytes are counted on a
// barrier of either CTA of the pair.
__device__ __forceinline__ void tma_load_2d_pair(uint32_t dst, const CUtensorMap* map, int x, int y, uint32_t bar)
{
    asm volatile(
        "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%2, %3}], [%4];" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(bar)
        : "memory");
}
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t bar)
{
    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mma_bf16_pair(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                              uint32_t accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}
// Arrives once on the barrier at this offset in both CTAs when every MMA issued
// so far by this thread has completed.
__device__ __forceinline__ void mma_commit_pair(uint32_t bar)
{
    asm volatile(
        "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(
            bar),
        "h"((uint16_t)3)
        : "memory");
}

// Hands the second warp's sums to the first of the two warps that share a
// 64-column group (xch: one slot per row; barrier 1 + lane quarter).
__device__ __forceinline__ float4 pair_exchange(float4 v, int c0, float4* xch)
{
    const int id = 1 + ((threadIdx.x >> 5) & 3);
    if (c0 == 1) *xch = v;
    asm volatile("bar.sync %0, 64;" ::"r"(id) : "memory");
    float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
    if (c0 == 0) o = *xch;
    asm volatile("bar.sync %0, 64;" ::"r"(id) : "memory");
    return o;
}

// Whether ok holds in all threads of the two warps of a lane quarter (the same
// barrier; both warps come here for every tile, after a wait with a limit).
__device__ __forceinline__ bool quarter_all(bool ok)
{
    const int id = 1 + ((threadIdx.x >> 5) & 3);
    uint32_t r;
    __syncwarp();
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.u32 q, %1, 0;\n\t"
        "bar.red.and.pred p, %2, 64, q;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(r)
        : "r"((uint32_t)ok), "r"(id)
        : "memory");
    return r != 0;
}

// The tile walk of one pair.
struct PairTiles {
    int nm, nn, pairs;          // tiles down / across (128 columns), pairs
    int full;                   // tiles dealt whole; the rest as halves
    int count;                  // work items in all
    int n64;                    // 64-column groups of the output
    __host__ __device__ PairTiles(int Np, int Jp, int pairs_) : pairs(pairs_)
    {
        nm = (Np + PBM - 1) / PBM;
        n64 = Jp / 64;
        nn = (n64 + 1) / 2;
        const int t = nm * nn, rest = t % pairs;
        full = 2 * rest <= pairs ? t - rest : t;
        count = full + 2 * (t - full);
    }
    // item -> row tile, first 64-column group, groups (1 or 2; 0: nothing there)
    __host__ __device__ void item(int k, int& tm, int& g0, int& ng) const
    {
        const int t = k < full ? k : full + (k - full) / 2;
        tm = t / nn;
        g0 = 2 * (t % nn);
        ng = n64 - g0 < 2 ? 1 : 2;
        if (k >= full) {
            if ((k - full) & 1) { ng -= 1; g0 += 1; }
            else ng = 1;
        }
    }
};

// Cfg: PLANES, STG (stages), PRODUCTS, pa(q), pb(q), acc(q, kb) (accumulator),
// first(q, kb, ks) (this MMA starts its accumulator).  Epi: tile(tm, g, row)
// (64-column group g, row within the pair's 256), load(taddr, n) (joins the
// accumulators of n x 32 columns from tensor memory: accumulator a at taddr +
// 128 a), compute(c0, n, xch): the same columns, from the group's 32 c0-th on.
// In a 64-column item the two warps of a lane quarter take 32 columns each
// (n = 1) and join what they need in xch (pair_exchange); in a 128-column item
// each takes a group (c0 = 0, n = 2).  tmA / tmB: boxes of 64 x 128 and 64 x 64.
// Returns false (all threads) if a wait ran out.
template <class Cfg, class Epi>
__device__ __forceinline__ bool gemm_pair(const CUtensorMap* tmA, const CUtensorMap* tmB, const GemmArgs& a, Epi& epi)
{
    constexpr int STG = Cfg::STG, PLANES = Cfg::PLANES;
    constexpr int STAGE = PLANES * (P_A_BYTES + P_B_BYTES);
    extern __shared__ __align__(1024) unsigned char tc_smem_raw[];
    // full[STG] | empty[STG] | tfull | tempty | done
    __shared__ __align__(8) uint64_t bars[2 * STG + 3];
    __shared__ uint32_t tmem_slot;
    __shared__ int failed;
    __shared__ float4 xch[128];
    unsigned char* smem = reinterpret_cast<unsigned char*>(
        (reinterpret_cast<uintptr_t>(tc_smem_raw) + 1023) & ~(uintptr_t)1023);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = cluster_rank();
    const int nkb = a.Kp / BK;
    const uint32_t sbase = smem_u32(smem);
    auto full = [&](int s) { return smem_u32(&bars[s]); };
    auto empty = [&](int s) { return smem_u32(&bars[STG + s]); };
    const uint32_t tfull = smem_u32(&bars[2 * STG]), tempty = smem_u32(&bars[2 * STG + 1]),
                   done = smem_u32(&bars[2 * STG + 2]);
    const PairTiles tiles(a.Np, a.Jp, (int)gridDim.x / 2);
    if (threadIdx.x == 32) {
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(tmA)) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(tmB)) : "memory");
    }
    const int first_item = (int)blockIdx.x / 2;

    if (threadIdx.x == 0) {
        for (int s = 0; s < STG; ++s) {
            mbar_init(full(s), 1);
            mbar_init(empty(s), 1);
        }
        mbar_init(tfull, 1);
        mbar_init(tempty, 2 * P_EPI_WARPS);
        mbar_init(done, 1);
        fence_mbar_init();
        failed = 0;
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)),
                     "r"(512)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync();               // the peer's barriers exist
    tc_fence_after();
    pdl_entry();                  // the operands are the previous kernel's
    const uint32_t tmem = tmem_slot;

    if (warp == 0) {
        if (lane == 0) {
            // TMA producer of this CTA; `it` counts K blocks over all items
            int it = 0;
            bool ok = true;
            for (int k = first_item; k < tiles.count && ok && !vload(failed); k += tiles.pairs) {
                int tm, g0, ng;
                tiles.item(k, tm, g0, ng);
                if (ng == 0) continue;
                const int m0 = tm * PBM + (int)rank * 128, n0 = g0 * 64 + (int)rank * 32 * ng;
                for (int kb = 0; kb < nkb; ++kb, ++it) {
                    const int s = it % STG;
                    if (it >= STG && !mbar_wait(empty(s), (uint32_t)((it / STG - 1) & 1))) {
                        failed = 1;
                        ok = false;
                        break;
                    }
                    const uint32_t bar = map_rank(full(s), 0);
                    if (rank == 0) mbar_expect_tx(full(s), 2 * STAGE);
                    const uint32_t st = sbase + (uint32_t)(s * STAGE);
                    for (int p = 0; p < PLANES; ++p) {
                        tma_load_2d_pair(st + (uint32_t)(p * P_A_BYTES), tmA, kb * BK, p * a.Np + m0, bar);
                        tma_load_2d_pair(st + (uint32_t)(PLANES * P_A_BYTES + p * P_B_BYTES), tmB, kb * BK,
                                         p * a.Jp + n0, bar);
                    }
                }
            }
        }
    } else if (warp == 1) {
        if (rank == 0 && lane == 0) {
            int it = 0, tl = 0;
            bool ok = true;
            for (int k = first_item; k < tiles.count && ok && !vload(failed); k += tiles.pairs) {
                int tm, g0, ng;
                tiles.item(k, tm, g0, ng);
                if (ng == 0) continue;
                if (tl >= 1 && !mbar_wait(tempty, (uint32_t)((tl - 1) & 1))) {
                    failed = 1;
                    break;
                }
                tc_fence_after();
                const uint32_t idesc = ng == 2 ? idesc_bf16(PBM, 128) : idesc_bf16(PBM, 64);
                for (int kb = 0; kb < nkb; ++kb, ++it) {
                    const int s = it % STG;
                    if (!mbar_wait(full(s), (uint32_t)((it / STG) & 1))) {
                        failed = 1;
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    const uint32_t st = sbase + (uint32_t)(s * STAGE);
#pragma unroll
                    for (int ks = 0; ks < BK / 16; ++ks) {
                        const uint32_t off = (uint32_t)(ks * 32);   // 16 bf16 along K
                        uint64_t ad[PLANES], bd[PLANES];
#pragma unroll
                        for (int p = 0; p < PLANES; ++p) {
                            ad[p] = sdesc_sw128(st + (uint32_t)(p * P_A_BYTES) + off);
                            bd[p] = sdesc_sw128(st + (uint32_t)(PLANES * P_A_BYTES + p * P_B_BYTES) + off);
                        }
#pragma unroll
                        for (int q = 0; q < Cfg::PRODUCTS; ++q)
                            mma_bf16_pair(tmem + (uint32_t)(Cfg::acc(q, kb) * 128), ad[Cfg::pa(q)], bd[Cfg::pb(q)],
                                          idesc, Cfg::first(q, kb, ks) ? 0u : 1u);
                    }
                    mma_commit_pair(empty(s));     // the stage is free in both CTAs once these MMAs are done
                }
                if (!ok) break;
                mma_commit_pair(tfull);            // the tile's accumulators are complete
                ++tl;
            }
            // every MMA issued by this thread has completed once `done` fires
            mma_commit_pair(done);
        }
    } else {
        // epilogue: warp w reads tensor-memory lanes 32 (w % 4) .. + 31 (one row
        // per lane), the 64-column group (w - 2) / 4 of the tile
        const int qtr = warp & 3, half = (warp - 2) >> 2;
        const uint32_t lane_base = (uint32_t)(32 * qtr) << 16;
        const uint32_t tempty0 = map_rank(tempty, 0);
        int tl = 0;
        for (int k = first_item; k < tiles.count; k += tiles.pairs) {
            int tm, g0, ng;
            tiles.item(k, tm, g0, ng);
            if (ng == 0) continue;
            epi.tile(tm, ng == 2 ? g0 + half : g0, (int)rank * 128 + 32 * qtr + lane);   // its loads travel now
            // the two warps of a lane quarter go on or leave together: each times its
            // own wait, and pair_exchange waits for the other warp without a limit
            const bool ok = mbar_wait(tfull, (uint32_t)(tl & 1));
            ++tl;
            if (!quarter_all(ok)) {
                failed = 1;
                break;
            }
            tc_fence_after();
            epi.load(tmem + lane_base + (uint32_t)((ng == 2 ? 64 : 32) * half), ng);
            // the accumulators may be overwritten once all warps of the pair have read them
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive_cluster(tempty0);
            epi.compute(ng == 2 ? 0 : half, ng, &xch[32 * qtr + lane]);
        }
    }
    __syncwarp();
    __syncthreads();              // the CTA's roles have ended: each has waited for one step at a time
    // both CTAs: the leader's commits have all arrived here.  Waited for from here on
    // only: from the start of the kernel, the limit of this one wait would bound the
    // peer CTA's whole GEMM.
    if (warp == 1 && lane == 0 && !mbar_wait(done, 0u)) failed = 1;
    __syncwarp();
    if (vload(failed)) {          // let this CTA's copies in flight land before it gives up its memory
        const long long t0 = clock64();
        while (clock64() - t0 < 4000000) {}
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync();               // no more remote arrivals, copies or reads between the CTAs
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
    }
    const bool good = !vload(failed);
    if (!good && threadIdx.x == 0 && a.status) atomicExch(a.status, 1);
    return good;
}

// The six split products: the main part in three accumulators (K blocks dealt
// round robin), the corrections in a fourth.
struct SplitCfg {
    static constexpr int PLANES = 3, STG = 3, PRODUCTS = 6;
    __device__ static constexpr int pa(int q) { constexpr int T[6] = {0, 0, 1, 0, 2, 1}; return T[q]; }
    __device__ static constexpr int pb(int q) { constexpr int T[6] = {0, 1, 0, 2, 0, 1}; return T[q]; }
    __device__ static constexpr int acc(int q, int kb) { return q == 0 ? kb % 3 : 3; }
    __device__ static constexpr bool first(int q, int kb, int ks)
    {
        return ks == 0 && (q == 0 ? kb < 3 : q == 1 && kb == 0);
    }
};

// 64 joined columns of one row: z = ((main 0 + main 1) + main 2) + corrections.
struct JoinEpi {
    int N, D, chains;             // chains: main accumulators that received products
    int i, g;                     // row, 64-column group
    float z[2][32];
    __device__ __forceinline__ void tile(int tm, int g_, int row)
    {
        i = tm * PBM + row;
        g = g_;
    }
    __device__ __forceinline__ void load(uint32_t taddr, int n)
    {
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            if (c >= n) break;
            float v[32];
            tmem_ld32(taddr + (uint32_t)(32 * c), z[c]);
            if (chains > 1) {
                tmem_ld32(taddr + (uint32_t)(128 + 32 * c), v);
#pragma unroll
                for (int q = 0; q < 32; ++q) z[c][q] = __fadd_rn(z[c][q], v[q]);
            }
            if (chains > 2) {
                tmem_ld32(taddr + (uint32_t)(256 + 32 * c), v);
#pragma unroll
                for (int q = 0; q < 32; ++q) z[c][q] = __fadd_rn(z[c][q], v[q]);
            }
            tmem_ld32(taddr + (uint32_t)(384 + 32 * c), v);
#pragma unroll
            for (int q = 0; q < 32; ++q) z[c][q] = __fadd_rn(z[c][q], v[q]);
        }
    }
};

// C -> out[i * D + j] (rows < N, columns < D).  vec: 8 (32-byte stores, the
// row pitch and base are multiples of 32 bytes), 4 (16-byte) or 1.
struct StoreEpi : JoinEpi {
    float* out;
    int vec;
    __device__ __forceinline__ void compute(int c0, int nb, float4*)
    {
        if (i >= N) return;
        float* row = out + (size_t)i * D + 64 * g + 32 * c0;
        const int n = D - 64 * g - 32 * c0;   // columns left in the row
#pragma unroll
        for (int c = 0; c < 2; ++c)
#pragma unroll
            for (int q = 0; q < 32; q += 8) {
                if (c >= nb) break;
                const int j = 32 * c + q;
                if (vec == 8 && j + 8 <= n) {
                    asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(row + j),
                                 "f"(z[c][q]), "f"(z[c][q + 1]), "f"(z[c][q + 2]), "f"(z[c][q + 3]), "f"(z[c][q + 4]),
                                 "f"(z[c][q + 5]), "f"(z[c][q + 6]), "f"(z[c][q + 7])
                                 : "memory");
                } else {
#pragma unroll
                    for (int h = 0; h < 8; h += 4) {
                        if (vec >= 4 && j + h + 4 <= n) {
                            *reinterpret_cast<float4*>(row + j + h) =
                                make_float4(z[c][q + h], z[c][q + h + 1], z[c][q + h + 2], z[c][q + h + 3]);
                        } else {
#pragma unroll
                            for (int m = 0; m < 4; ++m)
                                if (j + h + m < n) row[j + h + m] = z[c][q + h + m];
                        }
                    }
                }
            }
    }
};

inline bool aligned(const void* p, size_t a) { return (reinterpret_cast<uintptr_t>(p) & (a - 1)) == 0; }

// StoreEpi's store width for rows of D floats at out.
inline int store_width(const float* out, int64_t D)
{
    return D % 8 == 0 && aligned(out, 32) ? 8 : D % 4 == 0 && aligned(out, 16) ? 4 : 1;
}

// CTAs of a pair GEMM's grid: one pair per two SMs, no more than work items.
inline int pair_grid(int Np, int Jp, int sms)
{
    const int pairs = sms / 2;
    const PairTiles t(Np, Jp, pairs);
    return 2 * (t.count < pairs ? t.count : pairs);
}

}  // namespace tc
}  // namespace psso
