// Dense same-spin products on tcgen05 tensor cores.
//
// The same-spin part of H acts on the vector C[I_a][I_b] as
//   sigma_bb[I_a][I_b] = sum_J F_b[I_b][J] C[I_a][J]      (beta string Hamiltonian)
//   sigma_aa[I_a][I_b] = sum_J F_a[I_a][J] C[J][I_b]      (alpha string Hamiltonian)
// F_s is the Slater-Condon matrix of one spin's strings (tables.cu), symmetric,
// with about 6.6 % nonzeros at 16 orbitals spread over most tiles (83 % of the
// 128 x 128 tiles hold a nonzero), so both products run as dense GEMMs that skip
// only the all-zero k-blocks of the matrix operand's tile (17 % of the 256 x 32
// blocks of F_b and of F_a at 16 orbitals; tiles are taken in pairs, below):
// out[m][n] = sum_k A[m][k] B[n][k] with both operands K-major,
//   beta:  A = F_b (m = I_b, k = J),      B = C (n = I_a, k = J)
//   alpha: A = C^T (m = I_b, k = J),      B = F_a (n = I_a, k = J)
// Both add into y[n * ldy + m] of the same tile, so one launch accumulates the k-blocks
// of the first and then of the second, and its epilogue reads and writes y once; the
// 32 lanes of a warp (consecutive m) write consecutive addresses.  Against one launch
// per product with an epilogue of one column at a time: sigma at 16 orbitals 48.7 ->
// 45.4 ms, at 14 orbitals (3 columns) 7.59 -> 6.47 ms, at 10 orbitals 371 -> 203 us.
//
// Operands are split into two FP16 pieces with power-of-two scales (x = hi + lo);
// three MMAs per k-step (A_hi B_hi + A_lo B_hi + A_hi B_lo) accumulate in FP32
// in tensor memory.  The diagonals of F_a, F_b are kept out of the split matrices;
// the epilogue adds the whole diagonal of H (same-spin
// diagonals and the opposite-spin Coulomb sums, evaluated in FP64 and stored as
// float hi + lo per determinant) times x, hi and lo multiplied separately.
//
// Kernel: pairs of CTAs on tiles of 256 x 256 (or narrower, see tile_columns), each CTA
// 128 of the rows, k-block 32 (64 bytes per row: one SWIZZLE_64B atom row), TMA pipeline of
// six stages (eight for narrower tiles; full/empty mbarriers), one warp issues TMA,
// one issues MMAs for the pair, eight warps drain accumulator chunks (see k_gemm) and run
// the epilogue.  All waits are bounded.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_fp16.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <array>
#include <map>
#include <mutex>
#include <vector>

#include "gemm_tc.cuh"

namespace kpm {
namespace {

// k-block 32 (64-byte rows, SWIZZLE_64B) six stages deep, or 64 (128-byte rows,
// SWIZZLE_128B) three stages deep: the same 192 KB of shared memory.  Chunks of 64 of K
// either way (one-k-block chunks of 32 make the epilogue drain one every 800 cycles of MMA:
// 22.0 ms for both products at 16 orbitals where two-k-block chunks took 18.0, on the kernels
// with a tile per CTA).
#ifndef GM_BK_N
#define GM_BK_N 32
#endif
constexpr int GM_BM = 128, GM_BK = GM_BK_N;
static_assert(GM_BK == 32 || GM_BK == 64, "k-block of 32 or 64");
// Column tiles of 256, 128 or 64 (tile_columns() picks).  Eight epilogue warps, half a
// tile's columns each, drained 32 columns per tensor-memory load; narrower tiles have
// deeper pipelines in the same shared memory.
constexpr int GM_LIST_N = 256;               // rows of F_a per k-block list, for every tile
constexpr int GM_EPI_WARPS = 8;
template <int BN>
struct Tile {
    static constexpr int EPI_COLS = BN / 2;
    static constexpr int STAGES = (BN == 256 ? 6 : 8) * 32 / GM_BK;
    static constexpr uint32_t B_BYTES = BN / 2 * GM_BK * 2;   // per piece, a CTA's half
    static_assert(GM_LIST_N % BN == 0 && EPI_COLS % 32 == 0, "tile geometry");
};
constexpr int GM_TMA_WARP = GM_EPI_WARPS;       // producer (one thread)
constexpr int GM_MMA_WARP = GM_EPI_WARPS + 1;   // MMA issue (one thread)
constexpr int GM_THREADS = 32 * (GM_EPI_WARPS + 2);
// Accumulation chunks over K.  The tensor cores' FP32 accumulation rounds each
// addition into the accumulator toward zero (it shrinks every running sum by up
// to one unit in the last place), a bias that grows with the number of MMAs
// accumulated and would act as a fixed scaling of H; restarting the accumulator
// every 64 of K (12 MMAs; in each k-block the small correction products first,
// so that most of their additions truncate at their own small scale) and adding
// the chunks into FP32 running sums in registers (round to nearest) keeps it to
// a few units of 2^-24.
constexpr int GM_CK = 64 / GM_BK;               // k-blocks per accumulation chunk
// poll interval of the epilogue warps' waits (14 orbitals, three columns: 4.696 ms with 256,
// 4.690 with 32, 4.693 with none)
#ifndef GM_BACKOFF_NS
#define GM_BACKOFF_NS 32
#endif
constexpr uint32_t A_BYTES = GM_BM * GM_BK * 2;  // per piece
// Pairs of CTAs (clusters of two) on vertically adjacent tiles
constexpr int GM_PAIR = 2;
template <int BN>
constexpr uint32_t stage_bytes() { return 2 * A_BYTES + 2 * Tile<BN>::B_BYTES; }
template <int BN>
constexpr size_t gemm_smem() { return Tile<BN>::STAGES * stage_bytes<BN>() + 1024 + 256; }
constexpr long long GM_WAIT = 4000000000LL;
constexpr long long GM_DRAIN = 20000000LL;   // after an abort, per stage: ~10 ms

__device__ __forceinline__ uint32_t su32(const void* p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void mbar_init_(uint64_t* b, uint32_t c) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(su32(b)), "r"(c) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* b, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(su32(b)), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ bool mbar_test(uint64_t* b, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok) : "r"(su32(b)), "r"(parity) : "memory");
    return ok != 0;
}
// the same for a phase that threads of the other CTA arrive on (mbar_arrive_cluster)
__device__ __forceinline__ bool mbar_test_cluster(uint64_t* b, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.relaxed.cluster.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok) : "r"(su32(b)), "r"(parity) : "memory");
    return ok != 0;
}
// bounded wait; returns false (and flags the error) if it ran out
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t* b, uint32_t parity, int* err,
                                                  long long limit) {
    long long t0 = clock64();
    while (!mbar_test(b, parity)) {
        if (clock64() - t0 > limit) {
            atomicExch(err, 1);
            return false;
        }
    }
    return true;
}
// into this CTA's shared memory; the bytes are counted on `bar`, a shared::cluster address
// in either CTA of the pair
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, int x, int y,
                                            uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes.cta_group::2"
        " [%0], [%1, {%2, %3}], [%4];"
        ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(bar)
        : "memory");
}
__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
// shared::cluster address of the same variable in CTA `rank` of the cluster
__device__ __forceinline__ uint32_t mapa(uint32_t addr, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
// all threads of both CTAs of the cluster
__device__ __forceinline__ void cluster_sync_() {
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}
__device__ __forceinline__ void prefetch_map(const CUtensorMap* map) {
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(map)) : "memory");
}
__device__ __forceinline__ void tc_before() {
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_after() {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void mma_ss(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc,
                                       uint32_t acc) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(d), "l"(a), "l"(b), "r"(idesc), "r"(acc) : "memory");
}
// arrive, once the MMAs issued so far have completed, on the mbarrier at this offset in both
// CTAs of the pair
__device__ __forceinline__ void mma_commit_pair(uint64_t* b) {
    asm volatile(
        "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64"
        " [%0], %1;"
        ::"r"(su32(b)), "h"((uint16_t)0x3) : "memory");
}
__device__ __forceinline__ void ld32(uint32_t taddr, uint32_t (&r)[32]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,"
        "%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
          "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
          "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]),
          "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]),
          "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr)
        : "memory");
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// K-major swizzled descriptor: atoms of 8 rows x (2 GM_BK) bytes (one k-block
// row each), SBO = 8 rows between atoms along M/N; the leading offset is unused
// for these layouts.  Layout type 2: SWIZZLE_128B, 4: SWIZZLE_64B.
__device__ __forceinline__ uint64_t sw_desc(uint32_t saddr) {
    constexpr uint32_t row_bytes = GM_BK * 2;
    uint64_t d = 0;
    d |= (uint64_t)((saddr >> 4) & 0x3FFFu);
    d |= (uint64_t)1 << 16;                           // LBO (ignored)
    d |= (uint64_t)((8 * row_bytes) >> 4) << 32;      // SBO
    d |= (uint64_t)1 << 46;                           // version
    d |= (uint64_t)(GM_BK == 64 ? 2 : 4) << 61;       // swizzle mode
    return d;
}

template <int BN>
__host__ __device__ constexpr uint32_t gemm_idesc() {
    // D F32, A/B F16, K-major, N = BN, M = 256 over the pair
    return (1u << 4) | ((uint32_t)(BN >> 3) << 17) | ((uint32_t)(GM_PAIR * GM_BM >> 4) << 24);
}

struct GemmArgs {
    int M, N;                  // M = N_b (m = I_b), N = N_a (n = I_a); sums over N_b, then N_a
    int ncol;                  // columns of the block: operand rows, x and y follow one another
    float* y;                  // y[n * ldy + m] += sums / (wscale sa) + diagonal
    int64_t ldy;
    const float* amax;         // [ncol] max |x| of the split vector operand (operand scale sa)
    // The sums are kept at the smaller of the two matrices' scales w (powers of two): to_w_b
    // = w / wscale_b and to_w_a = w / wscale_a, both at most 1, so that however far apart the
    // magnitudes of F_a and F_b are, no sum (below 2^45) leaves the range of a float.
    float to_w_b, to_w_a, inv_w;
    // exact diagonal term (if x != nullptr): y[n*ldy+m] += d[n*ldy+m] * x[n*ldy+m], the
    // diagonal H_II evaluated in FP64 and stored as float (hi, lo)
    const float* x;
    const float2* dfull;
    int* err;
    int group_m;               // row tiles per rasterisation group (tuned; see DenseSS::autotune)
    // k-blocks holding a nonzero of the matrix operand, per tile of that operand (CSR:
    // kbl[kbs[t] .. kbs[t + 1]) ascending): F_b by pairs of row tiles, F_a by column
    // tile.  A skipped k-block only adds zero products, so the sums are unchanged.
    const int* kbs_b;
    const int* kbl_b;
    const int* kbs_a;
    const int* kbl_a;
};

// operand pieces (hi, lo) of the two products: F_b and the rows of x, the rows of x^T
// and F_a
struct GemmMaps {
    CUtensorMap fb[2], x[2], t[2], fa[2];
};

// bounded wait that also gives up when another role has aborted; roles off the
// critical path sleep backoff_ns between polls so that they leave the issue
// slots to the MMA and TMA threads
template <bool CLUSTER = false>
__device__ __forceinline__ bool wait_or_abort(uint64_t* b, uint32_t parity, volatile int* abort_flag,
                                              int* err, unsigned backoff_ns = 0) {
    long long t0 = clock64();
    while (!(CLUSTER ? mbar_test_cluster(b, parity) : mbar_test(b, parity))) {
        if (backoff_ns) __nanosleep(backoff_ns);
        if (*abort_flag) return false;
        if (clock64() - t0 > GM_WAIT) {
            *abort_flag = 1;
            atomicExch(err, 1);
            return false;
        }
    }
    return true;
}
// On a shared::cluster address.  Relaxed: what it orders are reads of tensor memory, by the
// tcgen05 fences on either side; no other memory is handed over.  (With release and acquire
// at cluster scope a chunk's turn took 5,300 cycles: sigma at 16 orbitals 39.1 ms, 32.1 so.)
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t b) {
    asm volatile("mbarrier.arrive.relaxed.cluster.shared::cluster.b64 _, [%0];" ::"r"(b) : "memory");
}

// Pairs: CTAs 2 p and 2 p + 1 (a cluster) compute row tiles 2 p and 2 p + 1 of the same
// column tile with MMAs over both SMs (cta_group::2, M = 256): each CTA loads its own 128 rows
// of A and half of the rows of B by plain TMA into its own shared memory, and the tensor
// cores of both read both halves of B.  The even CTA's MMA thread issues for the pair: both
// CTAs' loads count their bytes on its "full" barriers, its commits arrive on the "empty" and
// "accumulated" barriers of both, and the epilogue warps of both arrive on its "drained"
// ones.  Each CTA keeps its own rows of the accumulator in its tensor memory.  The pair
// syncs once its barriers are initialised and again before it gives up the tensor memory,
// so nothing is in flight towards a CTA that has ended.
// Why pairs: an MMA of one CTA alone (128 x 256 x 16, 128 cycles) reads 12 KB of shared
// memory, and its k-block's loads write 48 KB per 768 cycles: 160 bytes a cycle, more than
// the 128 there are.  With half of B in each SM it is 64 + 43.  sigma with a tile per CTA and
// with pairs, same bits: 16 orbitals 36.5 and 32.2 ms, 14 (three columns) 4.95 and 4.69,
// (13o, 7 + 6, BF16) 422 and 405 us; where the grid is one wave the pair's syncs cost what it
// gains (10 orbitals, three columns, 53.8 and 54.3 us).
//
// Accumulation in chunks: the MMA thread restarts the accumulator every ck
// k-blocks, alternating two tensor-memory accumulators of BN columns; the
// epilogue warps add each finished chunk into FP32 running sums held in
// registers while the next chunk accumulates.  An FP32 accumulator that takes
// one rounding per k-step over all of K (12870 at 16 orbitals) carries an error
// growing like sqrt(K); in chunks, each accumulator sums a short run and the
// running sum takes one rounding per chunk.
template <int BN>
__global__ void __cluster_dims__(GM_PAIR, 1, 1) __launch_bounds__(GM_THREADS, 1)
k_gemm(const __grid_constant__ GemmMaps maps, const GemmArgs g) {
    constexpr int STAGES = Tile<BN>::STAGES, EPI_COLS = Tile<BN>::EPI_COLS;
    constexpr uint32_t B_BYTES = Tile<BN>::B_BYTES;
    constexpr uint32_t STAGE_BYTES = stage_bytes<BN>();
    static_assert(STAGES * STAGE_BYTES >= GM_EPI_WARPS * EPI_COLS * 32 * 4, "epilogue staging");
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char* smem = reinterpret_cast<unsigned char*>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint64_t* full = reinterpret_cast<uint64_t*>(smem + STAGES * STAGE_BYTES);
    uint64_t* empty = full + STAGES;
    uint64_t* accf = empty + STAGES;   // [2] accumulator chunk finished
    uint64_t* acce = accf + 2;            // [2] accumulator drained (epilogue warps)
    uint32_t* holder = reinterpret_cast<uint32_t*>(acce + 2);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(holder + 1);
    int* consumed = const_cast<int*>(abort_flag) + 1;   // stages the MMA thread passed

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t crank = cluster_rank();   // blockIdx.x % GM_PAIR; 0: issues the MMAs
    // grouped rasterisation over pairs of row tiles: groups of GROUP_M pairs walk
    // all column tiles, so the group's A panels and the current B panels stay in L2
    const int GROUP_M = g.group_m;
    const int nM = (g.M + GM_BM - 1) / GM_BM, nN = (g.N + BN - 1) / BN;
    const int nMP = (nM + GM_PAIR - 1) / GM_PAIR;
    const int per_col = nMP * nN;              // tile pairs of a column
    const int col = blockIdx.x / GM_PAIR / per_col;
    const int b = blockIdx.x / GM_PAIR - col * per_col;
    const int64_t dim = (int64_t)g.N * g.ldy;
    // rows of this column's x (n) and x^T (m) in the operands; a tile past its last row
    // reads the next column's, which only reach sums that are not stored
    const int xrow = col * g.N, trow_ = col * g.M;
    const int gsize = GROUP_M * nN;
    const int first_m = (b / gsize) * GROUP_M;
    const int gm = min(nMP - first_m, GROUP_M);
    const int mp = first_m + (b % gsize) % gm;
    // (with an odd number of row tiles the last pair's second tile lies past M:
    // its A loads read the zero fill and its epilogue writes nothing)
    const int m0 = (mp * GM_PAIR + (int)crank) * GM_BM;
    const int n0 = ((b % gsize) / gm) * BN;
    // k-blocks the pair visits: those of F_b where the pair's 256 rows have a nonzero, then
    // those of F_a where the 256-row list tile of F_a around the B tile has one;
    // accumulation chunks do not cross from one to the other
    const int* kl1 = g.kbl_b + g.kbs_b[mp];
    const int nk1 = g.kbs_b[mp + 1] - g.kbs_b[mp];
    const int* kl2 = g.kbl_a + g.kbs_a[n0 / GM_LIST_N];
    const int nk = nk1 + g.kbs_a[n0 / GM_LIST_N + 1] - g.kbs_a[n0 / GM_LIST_N];
    constexpr int ck = GM_CK;                                  // k-blocks per chunk
    const int nchunk1 = (nk1 + ck - 1) / ck, nchunk = nchunk1 + (nk - nk1 + ck - 1) / ck;

    if (tid == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init_(&full[s], 1);
            mbar_init_(&empty[s], 1);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init_(&accf[i], 1);
            mbar_init_(&acce[i], GM_PAIR * GM_EPI_WARPS);
        }
        *abort_flag = 0;
        *consumed = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        for (int i = 0; i < 2; ++i) {
            prefetch_map(&maps.fb[i]);
            prefetch_map(&maps.x[i]);
            prefetch_map(&maps.t[i]);
            prefetch_map(&maps.fa[i]);
        }
    }
    // (before the allocation: a waiting CTA holds no tensor memory)
    grid_wait();
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], 512;"
                     ::"r"(su32(holder)) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    tc_before();
    cluster_sync_();   // both CTAs' barriers initialised, both halves of the tensor memory held
    tc_after();
    const uint32_t tmem = *holder;

    if (warp == GM_TMA_WARP) {
        if (lane == 0) {
            // TMA producer
            for (int kb = 0; kb < nk; ++kb) {
                const int s = kb % STAGES;
                if (kb >= STAGES &&
                    !wait_or_abort(&empty[s], ((kb / STAGES) - 1) & 1, abort_flag, g.err))
                    break;
                unsigned char* st = smem + s * STAGE_BYTES;
                // the pair's bytes, counted in the even CTA (the odd one's may land first)
                if (crank == 0) mbar_expect_tx(&full[s], GM_PAIR * STAGE_BYTES);
                const uint32_t bar = mapa(su32(&full[s]), 0);
                const bool beta = kb < nk1;
                const int kx = (beta ? kl1[kb] : kl2[kb - nk1]) * GM_BK;
                const CUtensorMap* mA = beta ? maps.fb : maps.t;
                const CUtensorMap* mB = beta ? maps.x : maps.fa;
                const int ma = beta ? m0 : trow_ + m0;
                tma_load_2d(su32(st), mA, kx, ma, bar);
                tma_load_2d(su32(st + A_BYTES), mA + 1, kx, ma, bar);
                // this CTA's half of the B rows
                const int nh = (beta ? xrow : 0) + n0 + (int)crank * (BN / GM_PAIR);
                tma_load_2d(su32(st + 2 * A_BYTES), mB, kx, nh, bar);
                tma_load_2d(su32(st + 2 * A_BYTES + B_BYTES), mB + 1, kx, nh, bar);
            }
            // (the last stages' commits have arrived before this CTA may end)
            for (int kb = max(0, nk - STAGES); kb < nk; ++kb)
                if (!wait_or_abort(&empty[kb % STAGES], (kb / STAGES) & 1, abort_flag, g.err)) break;
        }
    } else if (warp == GM_MMA_WARP) {
        if (lane == 0 && crank == 0) {
            // MMA issuer of the pair: chunk c accumulates its k-blocks (at most ck) into buffer c & 1
            constexpr uint32_t idesc = gemm_idesc<BN>();
            for (int c = 0; c < nchunk; ++c) {
                const uint32_t d = tmem + (uint32_t)((c & 1) * BN);
                if (c >= 2 && !wait_or_abort<true>(&acce[c & 1], ((c >> 1) - 1) & 1, abort_flag, g.err))
                    break;
                tc_after();
                const bool beta = c < nchunk1;
                const int kb0 = beta ? c * ck : nk1 + (c - nchunk1) * ck;
                const int kb1 = min(beta ? nk1 : nk, kb0 + ck);
                bool ok = true;
                for (int kb = kb0; kb < kb1; ++kb) {
                    const int s = kb % STAGES;
                    if (!wait_or_abort(&full[s], (kb / STAGES) & 1, abort_flag, g.err)) {
                        ok = false;
                        break;
                    }
                    *(volatile int*)consumed = kb + 1;
                    tc_after();
                    const uint32_t st = su32(smem + s * STAGE_BYTES);
                    const uint32_t a0 = st, a1 = st + A_BYTES, b0 = st + 2 * A_BYTES,
                                   b1 = st + 2 * A_BYTES + B_BYTES;
                    // correction products (lo x hi, hi x lo) first, while the running
                    // sum is small, then the main products (hi x hi)
#pragma unroll
                    for (int j = 0; j < GM_BK / 16; ++j) {
                        const uint32_t off = j * 32;  // 16 FP16 = 32 bytes along K in the row
                        const uint32_t acc0 = (kb != kb0 || j != 0) ? 1u : 0u;
                        mma_ss(d, sw_desc(a1 + off), sw_desc(b0 + off), idesc, acc0);
                        mma_ss(d, sw_desc(a0 + off), sw_desc(b1 + off), idesc, 1);
                    }
#pragma unroll
                    for (int j = 0; j < GM_BK / 16; ++j) {
                        const uint32_t off = j * 32;
                        mma_ss(d, sw_desc(a0 + off), sw_desc(b0 + off), idesc, 1);
                    }
                    mma_commit_pair(&empty[s]);   // stage s released in both CTAs
                }
                if (!ok) break;
                mma_commit_pair(&accf[c & 1]);
            }
        }
    } else {
        // epilogue warps: running sums of columns [EPI_COLS h, EPI_COLS (h + 1)) for row m
        const int quad = warp & 3, h = warp >> 2;
        const uint32_t trow = tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)(h * EPI_COLS);
        float rs[EPI_COLS];
#pragma unroll
        for (int u = 0; u < EPI_COLS; ++u) rs[u] = 0.f;
        bool ok = true;
        for (int c = 0; c < nchunk && ok; ++c) {
            if (lane == 0)
                ok = wait_or_abort(&accf[c & 1], (c >> 1) & 1, abort_flag, g.err, GM_BACKOFF_NS);
            ok = __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0;
            if (!ok) break;
            // from the scale of F_b's product to the common one, and from F_a's (exact)
            if (c == nchunk1 && g.to_w_b != 1.f) {
#pragma unroll
                for (int u = 0; u < EPI_COLS; ++u) rs[u] *= g.to_w_b;
            }
            const float f = c < nchunk1 ? 1.f : g.to_w_a;
            tc_after();
            const uint32_t src = trow + (uint32_t)((c & 1) * BN);
#pragma unroll
            for (int q = 0; q < EPI_COLS / 32; ++q) {
                uint32_t r[32];
                ld32(src + (uint32_t)(q * 32), r);
#pragma unroll
                for (int u = 0; u < 32; ++u)
                    rs[q * 32 + u] = fmaf(__uint_as_float(r[u]), f, rs[q * 32 + u]);
            }
            tc_before();
            __syncwarp();
            if (lane == 0) mbar_arrive_cluster(mapa(su32(&acce[c & 1]), 0));
        }
        if (ok && !*abort_flag) {
            float scale = (nchunk == nchunk1 ? g.to_w_b : 1.f) * g.inv_w;
            {
                const float mx = g.amax[col];
                if (mx > 0.f && isfinite(mx)) {
                    int e;
                    frexpf(mx, &e);
                    scale = scale / ldexpf(1.f, 14 - max(e, -90));
                }
            }
            // The sums move to the shared memory of the (now idle) stages, which frees
            // their registers for 16 columns' loads in flight at a time: one column at a
            // time waits for memory 128 times, 45 us a tile, most of the product's time
            // at small sizes.  (Every stage's loads have been consumed by the MMAs whose
            // accumulators were drained, so none is in flight into this memory.)
            float* mine = reinterpret_cast<float*>(smem) + warp * (EPI_COLS * 32) + lane;
#pragma unroll
            for (int u = 0; u < EPI_COLS; ++u) mine[u * 32] = rs[u];
            const int m = m0 + quad * 32 + lane;
            const int nb = n0 + h * EPI_COLS;
            constexpr int EG = 16;
            const int ncols = m < g.M ? min(EPI_COLS, g.N - nb) : 0;
            float* y = g.y + col * dim;
            // (x and the diagonal were final before this kernel could start; y was not)
            const float* x = g.x + col * dim;
#pragma unroll 1
            for (int u0 = 0; u0 < ncols; u0 += EG) {
                const int64_t o0 = (int64_t)(nb + u0) * g.ldy + m;
                float yv[EG], xv[EG];
                float2 dv[EG];
#pragma unroll
                for (int u = 0; u < EG; ++u) {
                    if (u0 + u < ncols) {
                        const int64_t o = o0 + u * g.ldy;
                        yv[u] = y[o];
                        if (g.x) {
                            xv[u] = __ldg(x + o);
                            dv[u] = __ldg(g.dfull + o);
                        }
                    }
                }
#pragma unroll
                for (int u = 0; u < EG; ++u) {
                    if (u0 + u < ncols) {
                        float v = yv[u] + mine[(u0 + u) * 32] * scale;
                        // hi and lo multiply separately: the diagonal keeps its FP64 value
                        if (g.x) v = fmaf(dv[u].x, xv[u], fmaf(dv[u].y, xv[u], v));
                        y[o0 + u * g.ldy] = v;
                    }
                }
            }
        }
    }
    tc_before();
    __syncthreads();
    if (tid == 0 && crank == 0 && *abort_flag) {
        // after an abort, wait (bounded) for the pair's copies that may still be in flight: the
        // other CTA has long issued those of the stages that were free
        for (int kb = *consumed; kb < min(nk, *consumed + STAGES); ++kb)
            mbar_wait_bounded(&full[kb % STAGES], (kb / STAGES) & 1, g.err, GM_DRAIN);
    }
    cluster_sync_();   // the other CTA's waits are over too, and its arrivals here done
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, 512;" ::"r"(tmem)
                     : "memory");
}

// max |F[t][r]| over off-diagonal entries t >= 1 (bits of a non-negative double)
__global__ void k_absmax_offdiag(const double* __restrict__ fval, int64_t ns, int nnbr,
                                 unsigned long long* out) {
    double mx = 0.0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < ns * (nnbr - 1);
         i += (int64_t)gridDim.x * blockDim.x)
        mx = fmax(mx, fabs(fval[ns + i]));
    for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_down_sync(0xffffffffu, mx, o));
    if ((threadIdx.x & 31) == 0) atomicMax(out, (unsigned long long)__double_as_longlong(mx));
}

// Dense off-diagonal string Hamiltonian, split into two scaled FP16 pieces.
// The matrix is first zeroed (k_zero_half), then every off-diagonal neighbour
// entry (t >= 1 of the [nnbr][ns] lists) is written.
__global__ void k_dense_offdiag(const int32_t* __restrict__ fcol, const double* __restrict__ fval,
                                int64_t ns, int nnbr, double wscale, __half* __restrict__ hi,
                                __half* __restrict__ lo, int64_t pitch) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= ns * (nnbr - 1)) return;
    const int64_t t = 1 + i / ns, r = i % ns;
    const int64_t c = fcol[t * ns + r];
    const double v = fval[t * ns + r] * wscale;
    const __half h = __double2half(v);
    hi[r * pitch + c] = h;
    lo[r * pitch + c] = __double2half(v - (double)__half2float(h));
}

__global__ void k_zero_half(__half* p, int64_t n) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x)
        p[i] = __float2half(0.f);
}

// mark[(r / rows) * nkb + c / GM_BK] = 1 for every off-diagonal neighbour entry
// (r, c): the k-blocks of each `rows`-row tile of the split matrix that hold a nonzero.
__global__ void k_mark_blocks(const int32_t* __restrict__ fcol, int64_t ns, int nnbr, int rows,
                              int64_t nkb, unsigned char* __restrict__ mark) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= ns * (nnbr - 1)) return;
    const int64_t t = 1 + i / ns, r = i % ns;
    const int64_t c = fcol[t * ns + r];
    mark[(r / rows) * nkb + c / GM_BK] = 1;
}

PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000,
                                             cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
        else
            cudaGetLastError();
    });
    return fn;
}

// 2-D FP16 tensor map: rows x cols (cols innermost, row pitch in elements),
// box = GM_BK columns x box_rows rows, swizzled rows of GM_BK elements (the
// layout sw_desc describes), zero fill out of bounds.
CUtensorMap make_map(const __half* base, int64_t rows, int64_t cols, int64_t pitch, int box_rows) {
    auto fn = encode_fn();
    if (!fn) KPM_THROW(KPM_ECUDA, "cuTensorMapEncodeTiled is not available");
    if (((uintptr_t)base & 15) || ((pitch * 2) & 15))
        KPM_THROW(KPM_EINVAL, "tensor map base/pitch not 16-byte aligned");
    CUtensorMap m;
    cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
    cuuint64_t strides[1] = {(cuuint64_t)(pitch * 2)};
    cuuint32_t box[2] = {(cuuint32_t)GM_BK, (cuuint32_t)box_rows};
    cuuint32_t es[2] = {1, 1};
    CUresult r = fn(&m, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, (void*)base, dims, strides, box, es,
                    CU_TENSOR_MAP_INTERLEAVE_NONE,
                    GM_BK == 64 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B,
                    CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) KPM_THROW(KPM_ECUDA, "cuTensorMapEncodeTiled failed (%d)", (int)r);
    return m;
}

}  // namespace

int64_t half_pitch(int64_t cols) { return (cols + 7) / 8 * 8; }

// CTAs of an M x N product: pairs of row tiles x column tiles, two CTAs each
static unsigned gemm_grid(int64_t M, int64_t N, int bn) {
    const int64_t nM = (M + GM_BM - 1) / GM_BM, nN = (N + bn - 1) / bn;
    return (unsigned)(GM_PAIR * ((nM + GM_PAIR - 1) / GM_PAIR) * nN);
}

static double offdiag_scale(const SpinTables& T, DevBuf& scratch, cudaStream_t st) {
    scratch.ensure(sizeof(unsigned long long));
    KPM_CUDA(cudaMemsetAsync(scratch.p, 0, sizeof(unsigned long long), st));
    if (T.nnbr > 1) {
        k_absmax_offdiag<<<1024, 256, 0, st>>>(T.fval64.as<double>(), T.ns, T.nnbr,
                                               scratch.as<unsigned long long>());
        KPM_LAUNCHED();
    }
    unsigned long long bits = 0;
    KPM_CUDA(cudaMemcpyAsync(&bits, scratch.p, sizeof(bits), cudaMemcpyDeviceToHost, st));
    KPM_CUDA(cudaStreamSynchronize(st));
    double mx;
    std::memcpy(&mx, &bits, sizeof(mx));
    if (!(mx > 0.0)) return 1.0;
    int e;
    std::frexp(mx, &e);  // mx < 2^e
    // (at most 2^300: entries below 2^-324 times a float vanish in a float)
    return std::ldexp(1.0, 14 - std::max(e, -286));
}

static void build_f(const SpinTables& T, double ws, DevBuf& hi, DevBuf& lo, int64_t pitch,
                    cudaStream_t st) {
    const int64_t n = T.ns * pitch;
    hi.alloc(n * 2);
    lo.alloc(n * 2);
    k_zero_half<<<1024, 256, 0, st>>>(hi.as<__half>(), n);
    KPM_LAUNCHED();
    k_zero_half<<<1024, 256, 0, st>>>(lo.as<__half>(), n);
    KPM_LAUNCHED();
    const int64_t ne = T.ns * (int64_t)(T.nnbr - 1);
    if (ne > 0) {
        k_dense_offdiag<<<(unsigned)((ne + 255) / 256), 256, 0, st>>>(
            T.fcol.as<int32_t>(), T.fval64.as<double>(), T.ns, T.nnbr, ws, hi.as<__half>(),
            lo.as<__half>(), pitch);
        KPM_LAUNCHED();
    }
}

// Lists, per tile of `rows` rows of the split matrix of T, the k-blocks holding a
// nonzero (CSR start[ntiles + 1] and list, both int32 on the device).
static void block_lists(const SpinTables& T, int rows, DevBuf& start, DevBuf& list,
                        int64_t* nonzero, int64_t* total, cudaStream_t st) {
    const int64_t ntile = (T.ns + rows - 1) / rows, nkb = (T.ns + GM_BK - 1) / GM_BK;
    DevBuf mark;
    mark.alloc((size_t)(ntile * nkb));
    KPM_CUDA(cudaMemsetAsync(mark.p, 0, mark.bytes, st));
    const int64_t ne = T.ns * (int64_t)(T.nnbr - 1);
    if (ne > 0) {
        k_mark_blocks<<<(unsigned)((ne + 255) / 256), 256, 0, st>>>(
            T.fcol.as<int32_t>(), T.ns, T.nnbr, rows, nkb, mark.as<unsigned char>());
        KPM_LAUNCHED();
    }
    std::vector<unsigned char> h((size_t)(ntile * nkb));
    KPM_CUDA(cudaMemcpyAsync(h.data(), mark.p, h.size(), cudaMemcpyDeviceToHost, st));
    KPM_CUDA(cudaStreamSynchronize(st));
    std::vector<int> hs((size_t)ntile + 1, 0), hl;
    for (int64_t t = 0; t < ntile; ++t) {
        for (int64_t k = 0; k < nkb; ++k)
            if (h[(size_t)(t * nkb + k)]) hl.push_back((int)k);
        hs[(size_t)t + 1] = (int)hl.size();
    }
    if (hl.empty()) hl.push_back(0);  // keeps the list buffer non-empty
    start.alloc(hs.size() * sizeof(int));
    list.alloc(hl.size() * sizeof(int));
    KPM_CUDA(cudaMemcpyAsync(start.p, hs.data(), start.bytes, cudaMemcpyHostToDevice, st));
    KPM_CUDA(cudaMemcpyAsync(list.p, hl.data(), list.bytes, cudaMemcpyHostToDevice, st));
    KPM_CUDA(cudaStreamSynchronize(st));
    *nonzero = hs.back();
    *total = ntile * nkb;
}

void DenseSS::init(const SpinTables& A, const SpinTables& B, bool same, int* err_flag,
                   cudaStream_t st) {
    na = A.ns;
    nb = B.ns;
    pa = half_pitch(na);
    pb = half_pitch(nb);
    xpitch = (nb + 127) / 128 * 128;
    err = err_flag;
    int dev = 0;
    KPM_CUDA(cudaGetDevice(&dev));
    KPM_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
    KPM_CUDA(cudaFuncSetAttribute(k_gemm<256>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)gemm_smem<256>()));
    KPM_CUDA(cudaFuncSetAttribute(k_gemm<128>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)gemm_smem<128>()));
    KPM_CUDA(cudaFuncSetAttribute(k_gemm<64>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)gemm_smem<64>()));
    wscale_b = offdiag_scale(B, fmax, st);
    build_f(B, wscale_b, fb_hi, fb_lo, pb, st);
    if (same) {
        wscale_a = wscale_b;
        fa_hi = &fb_hi;
        fa_lo = &fb_lo;
    } else {
        wscale_a = offdiag_scale(A, fmax, st);
        build_f(A, wscale_a, fa_hi_own, fa_lo_own, pa, st);
        fa_hi = &fa_hi_own;
        fa_lo = &fa_lo_own;
    }
    // beta: F_b is the A operand (pairs of GM_BM-row tiles); alpha: F_a is the B
    // operand (lists by GM_LIST_N rows)
    block_lists(B, GM_PAIR * GM_BM, kbs_b, kbl_b, &kb_nonzero[0], &kb_total[0], st);
    block_lists(A, GM_LIST_N, kbs_a, kbl_a, &kb_nonzero[1], &kb_total[1], st);
}

// The narrowest tile whose grid is one wave: a tile's time is its k-blocks' MMAs and its
// epilogue, both by its width, so below one wave narrower tiles give the same work to more
// SMs (and a shorter epilogue).  Beyond one wave 256 is best: every CTA reads its A tile
// whole, 24 KB a k-block at 128 columns for half the MMAs of the 32 KB at 256.  Measured,
// whole sigma with 256 / 128 / 64 columns: 10 orbitals 51.9 / 44.0 / 40.1 us (three
// columns of x 65.4 / 58.1 / 53.9), 12 orbitals 167 / 158 / 153 (three, where 64
// takes 2.4 waves: 349 / 378 / 401), (13o, 5 + 5) 263 / 252 / 290 (64: 1.7 waves),
// (13o, 7 + 6) 403 / 449 / 493.  Every width adds the same chunks in the same order, so
// the results are the same bits.
int DenseSS::tile_columns(int nc) const {
    for (int bn : {64, 128})
        if (nc * (int64_t)gemm_grid(nb, na, bn) <= nsm) return bn;
    return 256;
}

// y[I_a][I_b] += sum_J Fb[I_b][J] x[I_a][J] (split copies of x in xh/xl, th/tl)
//             + sum_J x^T[I_b][J] Fa[I_a][J] + H_II x[I_a][I_b]
void DenseSS::launch(const float* x, float* y, const float* amax, int nc, int group,
                     cudaStream_t st) {
    const float* diag = diag_full ? x : nullptr;
    const int bn = tile_columns(nc);
    GemmMaps maps;
    maps.fb[0] = make_map(fb_hi.as<__half>(), nb, nb, pb, GM_BM);
    maps.fb[1] = make_map(fb_lo.as<__half>(), nb, nb, pb, GM_BM);
    maps.x[0] = make_map(xh.as<__half>(), nc * na, nb, xpitch, bn / GM_PAIR);
    maps.x[1] = make_map(xl.as<__half>(), nc * na, nb, xpitch, bn / GM_PAIR);
    maps.t[0] = make_map(th.as<__half>(), nc * nb, na, pa, GM_BM);
    maps.t[1] = make_map(tl.as<__half>(), nc * nb, na, pa, GM_BM);
    maps.fa[0] = make_map(fa_hi->as<__half>(), na, na, pa, bn / GM_PAIR);
    maps.fa[1] = make_map(fa_lo->as<__half>(), na, na, pa, bn / GM_PAIR);
    const double w = std::min(wscale_a, wscale_b);
    GemmArgs g{(int)nb, (int)na, nc, y, nb, amax, (float)(w / wscale_b), (float)(w / wscale_a),
               (float)(1.0 / w), diag, diag ? diag_full : nullptr, err, group, kbs_b.as<int>(), kbl_b.as<int>(),
               kbs_a.as<int>(), kbl_a.as<int>()};
    const unsigned grid = nc * gemm_grid(nb, na, bn);
    if (bn == 256) launch_chained(k_gemm<256>, grid, GM_THREADS, gemm_smem<256>(), st, maps, g);
    else if (bn == 128) launch_chained(k_gemm<128>, grid, GM_THREADS, gemm_smem<128>(), st, maps, g);
    else launch_chained(k_gemm<64>, grid, GM_THREADS, gemm_smem<64>(), st, maps, g);
    KPM_LAUNCHED();
}

void DenseSS::apply(const float* x, float* y, const float* amax, int nc, cudaStream_t st) {
    launch(x, y, amax, nc, group_m, st);
}

// Picks the rasterisation group of the GEMM by timing the candidates once per
// device and shape (process-wide cache).  The group only decides which CTA
// computes which output tile, never how a tile is computed, so results do not
// depend on the choice.  Small shapes, where the whole problem sits in L2, keep
// the default.
void DenseSS::autotune(cudaStream_t st) {
    if (na * nb < ((int64_t)1 << 22)) return;
    int dev = 0;
    KPM_CUDA(cudaGetDevice(&dev));
    static std::mutex mu;
    static std::map<std::array<int64_t, 3>, int> cache;
    const std::array<int64_t, 3> key{dev, na, nb};
    {
        std::lock_guard<std::mutex> lk(mu);
        auto it = cache.find(key);
        if (it != cache.end()) {
            group_m = it->second;
            return;
        }
    }
    // scratch operands (zeros: the timing does not depend on the values)
    xh.ensure(x_bytes(1));
    xl.ensure(x_bytes(1));
    th.ensure(t_bytes(1));
    tl.ensure(t_bytes(1));
    KPM_CUDA(cudaMemsetAsync(xh.p, 0, xh.bytes, st));
    KPM_CUDA(cudaMemsetAsync(xl.p, 0, xl.bytes, st));
    KPM_CUDA(cudaMemsetAsync(th.p, 0, th.bytes, st));
    KPM_CUDA(cudaMemsetAsync(tl.p, 0, tl.bytes, st));
    DevBuf ys, one;
    ys.alloc((size_t)na * nb * sizeof(float));
    KPM_CUDA(cudaMemsetAsync(ys.p, 0, ys.bytes, st));
    static const float kOne = 1.0f;
    one.alloc(sizeof(float));
    KPM_CUDA(cudaMemcpyAsync(one.p, &kOne, sizeof(float), cudaMemcpyHostToDevice, st));
    cudaEvent_t e0, e1;
    KPM_CUDA(cudaEventCreate(&e0));
    KPM_CUDA(cudaEventCreate(&e1));
    const int cand[4] = {4, 8, 16, 32};
    auto run = [&](int gsz) { launch(ys.as<float>(), ys.as<float>(), one.as<float>(), 1, gsz, st); };
    run(group_m);  // warm-up
    float best = 0.f;
    for (int c : cand) {
        KPM_CUDA(cudaEventRecord(e0, st));
        run(c);
        KPM_CUDA(cudaEventRecord(e1, st));
        KPM_CUDA(cudaEventSynchronize(e1));
        float ms = 0.f;
        KPM_CUDA(cudaEventElapsedTime(&ms, e0, e1));
        if (best == 0.f || ms < best) {
            best = ms;
            group_m = c;
        }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    std::lock_guard<std::mutex> lk(mu);
    cache[key] = group_m;
}

}  // namespace kpm
