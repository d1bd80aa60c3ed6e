// The grouped Chebyshev expansion (k_poly.cu) on the tensor cores: products
// of symmetric polynomials of H_N in the split 16-bit form
//   A B ~ A_hi B_hi + A_hi B_lo + A_lo B_hi   (hi = round(x), lo = round(x - hi))
// on tcgen05 with FP32 accumulation, for one or many systems per launch.
//
// Storage.  Every matrix is symmetric, so a buffer ("slot") keeps the 256 x
// 256 blocks (a, b), a <= b, only (diagonal blocks whole), each transposed
// (rows of b, columns of a), folded into a rectangle of R = nb / 2 + 1 block
// rows (nb = Kp / 256 blocks per side): block row a < R lies in place, block
// row a >= R, which has nb - a blocks, fills the free left end of block row
// nb - a.  Half the bytes of full storage: twice as many babies fit the
// workspace, more operand tiles stay in L2, and no mirror is written.  A slot
// holds the hi plane and then the lo plane; the same two planes can hold FP32
// values as their upper and lower 16 bits.  An operand tile whose k block lies
// on or right of the diagonal is read as rows of k (MN-major operand, 128-byte
// swizzle, one 3-D TMA box), the others K-major (64-byte swizzle); both run
// at the same speed.  The transposition makes a warp's 32 rows of one output
// column contiguous, so the epilogue needs no staging.
//
// Kernel k_pst_prod: persistent, one CTA per SM, one 128 x 256 output tile
// at a time: warp 0 lane 0 drives the TMA loads of the four operand tiles of
// each 32-wide k-block into a 4-stage ring of 48 KB, warp 1 owns the 512
// tensor-memory columns and lane 0 issues the MMAs, eight epilogue warps add
// each finished unit of one or two k-blocks from one of two accumulators into FP32
// registers (round to nearest; the tensor core's own FP32 accumulation leans
// towards zero with every addition, so its chains are kept short) and then
// write x = alpha A B - prev + add straight from registers: neighbouring lanes
// swap one of two columns, so that a lane moves two rows of one column per
// 32-bit access and a warp whole sectors (with one row per lane and 16-byte
// accesses along the row the epilogue took 60 of 100 us per tile at K =
// 2000).  The ring stays with the producer, and the next tile's loads and
// first two units run under the epilogue.  Every wait is bounded; on expiry the
// CTA sets FLAG_TIMEOUT of the system and of the launch's leader, drains what it
// issued and returns, and the call's later launches find the leader's flag and
// return at once.  hold (a test, DFT_TEST_EXPIRE_WAITS) makes one epilogue warp
// withhold the release of its first accumulator, so that the waits run out.
//
// Density matrix at K = 1230, tail 1e-5 (N_C ~ 1410, direct plan): 118.9 ms
// with the recurrence of k_cheb_tc.cu, 6.1 ms with this (error of P against
// an exact eigensolve 3.6e-5 -> 1.7e-5); SCF step at K = 4650 (Clenshaw plan,
// s = 34, 112 products) 668 -> 87 ms.
#include "ps_plan.cuh"
#include "tc_ptx.cuh"

#include <algorithm>
#include <cmath>
#include <cstdlib>

namespace dft {
namespace {

using namespace tc;

// FP16 pairs in every mixed precision: the operands are bounded, and 16 bits of a
// BF16 pair for the C_q left P 9% further from FP64 than the three-term recurrence
// does on BF16 pairs (its sum is FP32; K = 80 to 1230, four geometries each: 9.9e-5,
// 1.1e-4, 1.3e-4 against 9.0e-5, 1.0e-4, 1.2e-4)
using P16 = H16<false>;

constexpr int BM = 128, BN = 256, BK = 32, STAGES = 4;
// k-blocks per accumulator promotion (PstItem::sub).  Longer chains lean
// further towards zero; the babies' bias acts as a scale of H_N on every term,
// so they take 1.  Giants and weighted products with 1 / 2, density matrix in ms
// (tail 1e-5, without the set-up of H_N): K = 1230 4.35 / 4.17, 2100 9.01 / 8.49,
// 3000 26.8 / 24.4, 4650 60.1 / 54.1; the error of P against FP64 is the same to
// 1% at all of them (relative 1.7e-5, 2.0e-5, 2.4e-5, 2.9e-5; the three-term
// recurrence 3.1e-5, 3.6e-5, -, 4.8e-5).  Up to SUB_FINE_K, where a chain of two
// saves 4% at most, the chains stay at one.
constexpr int SUB_FINE = 1, SUB = 2, SUB_FINE_K = 2048;
constexpr int A_BYTES = BM * BK * 2, B_BYTES = BN * BK * 2;
constexpr int STAGE_BYTES = 2 * A_BYTES + 2 * B_BYTES;
// warps 0 .. 3: producer, MMA issuer and two idle ones, so that the eight
// epilogue warps are whole warpgroups and can take the registers these do not
// need (384 x 168 at launch = 128 x 40 + 256 x 232)
constexpr int NEPI = 256, NTHREADS = 128 + NEPI, CPT = 128;
// behind the ring: barriers, the launch's item table (the first ITEM_SMEM
// items; reading it from global memory at each tile cost 4 us per tile) and
// one 16 x 32 transposition buffer per epilogue warp
constexpr int ITEM_SMEM = 384;
constexpr int TR_WORDS = 16 * 33;
constexpr int SMEM_BYTES = STAGES * STAGE_BYTES + 1024 + 256 + ITEM_SMEM * (int)sizeof(PstItem) + 8 * TR_WORDS * 4;
static_assert(SMEM_BYTES <= 232448, "shared memory of one CTA");
constexpr int TMEM_COLS = 2 * BN;
constexpr int SMS = 152;
// pairs hold x * SC: the low half of an FP16 pair of x itself would be a
// subnormal number for the elements of order K^-1/2 that most of a T_l
// consists of (2^-25 absolute); scaled, the pair keeps 22 bits down to
// 2^-27.  |T_l| <= 4; the b_q of Clenshaw's recurrence grow to Q / 6 for a step
// at a multiple of pi / s (64-bit evaluation, s = 14 to 128, N_C to 65536; 1 at
// the benchmark's Q = 41, 100 at N_C = 65536 with s = 24 and a converged tail),
// so that beyond Q = B_Q all C_q but C_0 carry a power of two that keeps Q / 6
// below 60 of the 64 that a pair holds.
constexpr float SC = 1024.0f, ISC = 1.0f / SC;
constexpr int B_Q = 360;
float clenshaw_down(int Q) {
    float d = 1.0f;
    for (int q = Q; q > B_Q; q = (q + 1) / 2) d *= 0.5f;
    return d;
}

// folded place of block (a, b), a <= b
__device__ __forceinline__ void fold(int a, int b, int nb, int& row, int& col) {
    const bool in_place = a <= nb / 2;
    row = in_place ? a : nb - a;
    col = in_place ? b : b - a;
}

// tile u of a system: blocks (p, q) row by row, both 128-row tiles of a block
// together; row tiles beyond K are left out
__device__ __forceinline__ void tile_at(int u, int nb, int mt, int& i, int& j) {
    int p = 0;
    for (;; ++p) {
        const int rows = min(2, mt - 2 * p), n = (nb - p) * rows;
        if (u < n) {
            j = p + u / rows;
            i = 2 * p + u % rows;
            return;
        }
        u -= n;
    }
}

__device__ __forceinline__ void tma_load_3d(void* dst, const CUtensorMap* map, int x, int y, int z, uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
        ::"r"(smem_u32(dst)), "l"(map), "r"(x), "r"(y), "r"(z), "r"(smem_u32(bar))
        : "memory");
}

// descriptor of an MN-major operand in 128-byte swizzle: 64-element groups of
// the M (N) index 32 k-rows x 128 bytes = 4096 bytes apart (leading offset),
// groups of 8 k-rows 1024 bytes apart (stride offset)
__device__ __forceinline__ uint64_t smem_desc_mn(const void* p) {
    const uint64_t addr = (uint64_t)(smem_u32(p) & 0x3FFFF) >> 4;
    return addr | ((uint64_t)(BK * 128 >> 4) << 16) | ((uint64_t)(1024 >> 4) << 32) | (1ull << 46) | (2ull << 61);
}

// mbar_wait that also gives up when the CTA is leaving (the producer's; in the
// MMA issuer's and the epilogue's waits the extra read cost 0.3% of a density matrix)
__device__ __forceinline__ bool wait_or_leave(uint64_t* bar, uint32_t parity, const volatile int* leave) {
    if (mbar_try_wait(bar, parity)) return true;
    const unsigned long long t0 = globaltimer();
    while (!mbar_try_wait(bar, parity)) {
        if (*leave || globaltimer() - t0 > WAIT_NS) return false;
    }
    return true;
}

// one product of a launch as the roles walk it
struct Work {
    PstItem it;
    const PstSys* S;
    int i, j, p, nk;   // row tile, column block, row block, k-blocks per operand pair
};
__device__ __forceinline__ Work work_at(int t, const PstItem* items, int nitems, const PstSys* __restrict__ sys) {
    int a = 0, b = nitems;   // last item with tile0 <= t
    while (b - a > 1) {
        const int m = (a + b) >> 1;
        if (items[m].tile0 <= t) a = m;
        else b = m;
    }
    Work w;
    w.it = items[a];
    w.S = sys + w.it.sys;
    tile_at(t - w.it.tile0, w.S->nb, (w.S->K + BM - 1) / BM, w.i, w.j);
    w.p = w.i >> 1;
    w.nk = (w.S->K + BK - 1) / BK;
    return w;
}

__global__ void __launch_bounds__(NTHREADS, 1) k_pst_prod(const PstSys* __restrict__ sys,
                                                          const PstItem* __restrict__ items_g, int nitems,
                                                          const int2* __restrict__ pairs, int ntiles,
                                                          int* lead_flags, int hold) {
    using T = P16::T;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint64_t* full = (uint64_t*)(smem + STAGES * STAGE_BYTES);
    uint64_t* empty = full + STAGES;
    uint64_t* accfull = empty + STAGES;
    uint64_t* accempty = accfull + 2;
    uint64_t* drain = accempty + 2;
    uint32_t* tmem_slot = (uint32_t*)(drain + 1);
    volatile int* abort_flag = (volatile int*)(tmem_slot + 1);
    static_assert((2 * STAGES + 5) * 8 + 8 <= 256, "barriers exceed their area");
    PstItem* items_s = (PstItem*)(smem + STAGES * STAGE_BYTES + 256);
    uint32_t* tr_all = (uint32_t*)(items_s + ITEM_SMEM);
    const PstItem* items = nitems <= ITEM_SMEM ? items_s : items_g;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (nitems <= ITEM_SMEM)
        for (int e = threadIdx.x; e < nitems * (int)(sizeof(PstItem) / 4); e += NTHREADS)
            ((int*)items_s)[e] = ((const int*)items_g)[e];
    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int a = 0; a < 2; ++a) {
            mbar_init(&accfull[a], 1);
            mbar_init(&accempty[a], NEPI / 32);   // one arrival per warp: 256 arrivals took longer than a unit's MMAs
        }
        mbar_init(drain, 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "r"(TMEM_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    auto sAh = [&](int s) { return smem + s * STAGE_BYTES; };
    auto sAl = [&](int s) { return smem + s * STAGE_BYTES + A_BYTES; };
    auto sBh = [&](int s) { return smem + s * STAGE_BYTES + 2 * A_BYTES; };
    auto sBl = [&](int s) { return smem + s * STAGE_BYTES + 2 * A_BYTES + B_BYTES; };

    if (warp < 4) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 40;");
    if (warp == 0) {
        if (lane == 0) {
            long long g = 0;   // k-blocks issued by this CTA
            for (int t = blockIdx.x; t < ntiles && !*abort_flag; t += gridDim.x) {
                const Work w = work_at(t, items, nitems, sys);
                const int nb = w.S->nb, lo_row = (nb / 2 + 1) * 256;
                for (int q = w.it.first; q < w.it.last && !*abort_flag; ++q) {
                    const int2 ab = pairs[q];
                    const CUtensorMap* ma = w.S->maps + 4 * ab.x;
                    const CUtensorMap* mb = w.S->maps + 4 * ab.y;
                    for (int kb = 0; kb < w.nk; ++kb, ++g) {
                        const int s = (int)(g % STAGES);
                        const int kq = kb >> 3, kx = (kb & 7) * BK;   // 256-block of k, offset inside
                        int ar, ac, br, bc;
                        fold(min(w.p, kq), max(w.p, kq), nb, ar, ac);
                        fold(min(w.j, kq), max(w.j, kq), nb, br, bc);
                        if (!wait_or_leave(&empty[s], (uint32_t)((g / STAGES) & 1) ^ 1u, abort_flag)) {
                            *abort_flag = 1;
                            break;
                        }
                        mbar_expect_tx(&full[s], STAGE_BYTES);
                        if (kq < w.p) {
                            const int y = ar * 256 + (w.i & 1) * BM, x = ac * 256 + kx;
                            tma_load_2d(sAh(s), ma + 0, x, y, &full[s]);
                            tma_load_2d(sAl(s), ma + 0, x, y + lo_row, &full[s]);
                        } else {
                            const int y = ar * 256 + kx, z = ac * 4 + (w.i & 1) * 2;
                            tma_load_3d(sAh(s), ma + 2, 0, y, z, &full[s]);
                            tma_load_3d(sAl(s), ma + 2, 0, y + lo_row, z, &full[s]);
                        }
                        if (kq < w.j) {
                            const int y = br * 256, x = bc * 256 + kx;
                            tma_load_2d(sBh(s), mb + 1, x, y, &full[s]);
                            tma_load_2d(sBl(s), mb + 1, x, y + lo_row, &full[s]);
                        } else {
                            const int y = br * 256 + kx, z = bc * 4;
                            tma_load_3d(sBh(s), mb + 3, 0, y, z, &full[s]);
                            tma_load_3d(sBl(s), mb + 3, 0, y + lo_row, z, &full[s]);
                        }
                    }
                }
            }
            // the last load issued into each stage must land before exit (whoever leaves
            // the launch early, and at what point: this thread has nothing else to do)
            for (long long q = (g > STAGES ? g - STAGES : 0); q < g; ++q)
                mbar_wait(&full[q % STAGES], (uint32_t)((q / STAGES) & 1));
            // wake the MMA issuer if it waits for the load that does not come (it issues one
            // block on stale operands, whose sums nobody reads)
            if (*abort_flag) mbar_arrive(&full[g % STAGES]);
        }
        __syncwarp();
    } else if (warp == 1) {
        if (lane == 0) {
            const uint32_t idesc0 = (1u << 4) |
                                    ((uint32_t)(BN >> 3) << 17) | ((uint32_t)(BM >> 4) << 24);
            long long g = 0, u = 0;   // k-blocks and units of this CTA
            for (int t = blockIdx.x; t < ntiles && !*abort_flag; t += gridDim.x) {
                const Work w = work_at(t, items, nitems, sys);
                const int nkt = w.nk * (w.it.last - w.it.first);
                int kb = 0;   // within the operand pair
                for (int k0 = 0; k0 < nkt && !*abort_flag; k0 += w.it.sub, ++u) {
                    const int a = (int)(u & 1);
                    if (!mbar_wait(&accempty[a], (uint32_t)(((u >> 1) & 1) ^ 1))) {
                        *abort_flag = 1;
                        break;
                    }
                    tc_fence_after();
                    const uint32_t d = tmem + (uint32_t)(a * BN);
                    bool first = true;
                    for (int k = k0; k < min(nkt, k0 + w.it.sub); ++k, ++g) {
                        const int s = (int)(g % STAGES);
                        if (*abort_flag || !mbar_wait(&full[s], (uint32_t)((g / STAGES) & 1))) {
                            *abort_flag = 1;
                            break;
                        }
                        tc_fence_after();
                        const int kq = kb >> 3;
                        if (++kb == w.nk) kb = 0;
                        const bool at = kq >= w.p, bt = kq >= w.j;   // MN-major operand
                        const uint32_t idesc = idesc0 | ((at ? 1u : 0u) << 15) | ((bt ? 1u : 0u) << 16);
                        const uint64_t ah = at ? smem_desc_mn(sAh(s)) : smem_desc<BK * 2>(sAh(s));
                        const uint64_t al = at ? smem_desc_mn(sAl(s)) : smem_desc<BK * 2>(sAl(s));
                        const uint64_t bh = bt ? smem_desc_mn(sBh(s)) : smem_desc<BK * 2>(sBh(s));
                        const uint64_t bl = bt ? smem_desc_mn(sBl(s)) : smem_desc<BK * 2>(sBl(s));
                        // 16 k: 32 bytes along a K-major row, 16 rows of 128 bytes MN-major
                        const uint64_t as = at ? 128 : 2, bs = bt ? 128 : 2;
                        // the small cross products first: additions to the accumulator lose bits
                        // in proportion to what it holds already
#pragma unroll
                        for (int kk = 0; kk < BK / 16; ++kk) {
                            umma_f16(d, ah + kk * as, bl + kk * bs, idesc, first ? 0u : 1u);
                            umma_f16(d, al + kk * as, bh + kk * bs, idesc, 1u);
                            first = false;
                        }
#pragma unroll
                        for (int kk = 0; kk < BK / 16; ++kk) umma_f16(d, ah + kk * as, bh + kk * bs, idesc, 1u);
                        umma_commit(&empty[s]);
                    }
                    umma_commit(&accfull[a]);
                }
            }
            // every MMA this thread issued must finish before tensor memory is freed
            umma_commit(drain);
            mbar_wait(drain, 0);
            if (*abort_flag) {   // wake the epilogue, which sees the abort
                mbar_arrive(&accfull[0]);
                mbar_arrive(&accfull[1]);
            }
        }
        __syncwarp();
    } else if (warp == 2) {
        // an earlier launch of this call gave up: so does this one (read by an idle
        // warp: in front of the first loads it cost 0.6 us per launch)
        if (lane == 0 && *(volatile int*)&lead_flags[FLAG_TIMEOUT]) *abort_flag = 1;
    }
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 232;");
        const int quad = warp & 3, half = (warp - 4) >> 2;
        const int r_loc = 32 * quad + lane;
        uint32_t* tr = tr_all + (warp - 4) * TR_WORDS;
        long long u = 0;
        bool ok = true;
        for (int t = blockIdx.x; t < ntiles && ok; t += gridDim.x) {
            const Work w = work_at(t, items, nitems, sys);
            const PstSys& S = *w.S;
            const int nunit = (w.nk * (w.it.last - w.it.first) + w.it.sub - 1) / w.it.sub, K = S.K, nb = S.nb;
            int fr, fc;
            fold(w.p, w.j, nb, fr, fc);
            const int ld = nb * 256;
            const size_t plane = (size_t)(nb / 2 + 1) * 256 * ld;
            // this lane's 32-bit words: rows r & ~1, r | 1 (stored columns) of output
            // column c + (lane & 1) (stored row)
            const bool odd = lane & 1;
            const size_t e0 = (size_t)(fr * 256 + half * CPT + odd) * ld + fc * 256 + (w.i & 1) * BM + (r_loc & ~1);
            const int r = w.i * BM + r_loc, c0 = w.j * BN + half * CPT;   // global row, first column
            const bool diag = w.p == w.j, f32_out = (w.it.mode & PST_OUT_F32) != 0, ident = (w.it.mode & PST_IDENT) != 0 && r < K;
            const float alpha = ((w.it.mode & PST_ALPHA2) ? 2.0f : 1.0f) * (ISC * ISC);
            const uint16_t* pv = w.it.prev >= 0 ? (const uint16_t*)S.slot[w.it.prev] + e0 : nullptr;
            const uint16_t* ad = w.it.add >= 0 ? (const uint16_t*)S.slot[w.it.add] + e0 : nullptr;
            uint16_t* out = (uint16_t*)S.slot[w.it.out] + e0;
            const float limit = w.it.limit;
            const bool edge = w.i * BM + BM > K || w.j * BN + BN > K;   // rows or columns beyond K
            bool bad = false;
            constexpr int EB = 16;   // columns per batch, the next one's loads in flight
            uint32_t nh[EB / 2], nl[EB / 2], mh[EB / 2], ml[EB / 2];
            auto fetch = [&](int cb) {
#pragma unroll
                for (int k = 0; k < EB / 2; ++k) {
                    const size_t o = (size_t)(cb + 2 * k) * ld;
                    nh[k] = pv ? *(const uint32_t*)(pv + o) : 0u;
                    nl[k] = pv ? *(const uint32_t*)(pv + plane + o) : 0u;
                    mh[k] = ad ? *(const uint32_t*)(ad + o) : 0u;
                    ml[k] = ad ? *(const uint32_t*)(ad + plane + o) : 0u;
                }
            };
            fetch(0);   // arrives under the products
            float R[CPT];
#pragma unroll
            for (int i = 0; i < CPT; ++i) R[i] = 0.0f;
            for (int q = 0; q < nunit; ++q, ++u) {
                const int a = (int)(u & 1);
                const bool got = mbar_wait(&accfull[a], (uint32_t)((u >> 1) & 1));
                ok = __all_sync(0xffffffffu, got && !*abort_flag);
                if (!ok) break;
                tc_fence_after();
                tmem_add_groups<CPT / 16>(tmem + ((uint32_t)(32 * quad) << 16) + (uint32_t)(a * BN + half * CPT), R);
                tc_fence_before();
                __syncwarp();
                if (lane == 0 && q + 1 < nunit && !(hold && warp == 4 && u == 0)) mbar_arrive(&accempty[a]);
            }
            if (!ok) {
                *abort_flag = 1;
                if (lane == 0) {
                    atomicExch(&S.flags[FLAG_TIMEOUT], 1);
                    atomicExch(&lead_flags[FLAG_TIMEOUT], 1);
                }
                break;
            }
            // the sums go back to the last unit's accumulator, which stays with the
            // epilogue until they are used up, so that the update is a short loop
            // (unrolled over 128 registers it was 90 KB of code per tile, and
            // fetching it took 30 us)
            const int a_last = (int)((u - 1) & 1);
            const uint32_t tacc = tmem + ((uint32_t)(32 * quad) << 16) + (uint32_t)(a_last * BN + half * CPT);
            tc_fence_after();
#pragma unroll
            for (int q = 0; q < CPT / 16; ++q) tmem_st16(tacc + 16 * q, &R[16 * q]);
            tmem_wait_st();
#pragma unroll 1
            for (int cb = 0; cb < CPT; cb += EB) {
                static_assert(EB == 16, "one tensor-memory load per batch");
                uint32_t av[16];
                tmem_ld16(tacc + cb, av);
                uint32_t ph[EB / 2], pl[EB / 2], gh[EB / 2], gl[EB / 2];
#pragma unroll
                for (int k = 0; k < EB / 2; ++k) {
                    ph[k] = nh[k];
                    pl[k] = nl[k];
                    gh[k] = mh[k];
                    gl[k] = ml[k];
                }
                if (cb + EB < CPT) fetch(cb + EB);
                // Step by step over the whole batch, the uniform branches outside: inside
                // the loop over columns they kept the columns' chains of shuffles and
                // conversions from overlapping.  Conversions go in pairs and neighbours exchange
                // sums (one shuffle instead of two).  Clocks of a tile's update, without and with
                // prev: 25,400 and 29,500 before, 14,500 and 15,900 now (the products of a tile
                // take 57,400 at K = 1230).
                // x[2 k], x[2 k + 1]: columns c, c + 1 of this lane's row, one from its own
                // words, one from the neighbour's
                float x[EB];
#pragma unroll
                for (int u = 0; u < EB; ++u) x[u] = alpha * __uint_as_float(av[u]);
                if (pv) {
#pragma unroll
                    for (int k = 0; k < EB / 2; ++k) {
                        const float2 h = P16::to_f2(ph[k]), l = P16::to_f2(pl[k]);
                        const float f0 = h.x + l.x, f1 = h.y + l.y;   // rows r & ~1, r | 1
                        const float got = __shfl_xor_sync(0xffffffffu, odd ? f0 : f1, 1);
                        x[2 * k] = fmaf(-ISC, odd ? got : f0, x[2 * k]);
                        x[2 * k + 1] = fmaf(-ISC, odd ? f1 : got, x[2 * k + 1]);
                    }
                }
                if (ad) {
#pragma unroll
                    for (int k = 0; k < EB / 2; ++k) {
                        const uint32_t f0 = __byte_perm(gl[k], gh[k], 0x5410), f1 = __byte_perm(gl[k], gh[k], 0x7632);
                        const uint32_t got = __shfl_xor_sync(0xffffffffu, odd ? f0 : f1, 1);
                        x[2 * k] += __uint_as_float(odd ? got : f0);
                        x[2 * k + 1] += __uint_as_float(odd ? f1 : got);
                    }
                }
                if (diag && ident) {
#pragma unroll
                    for (int u = 0; u < EB; ++u)
                        if (c0 + cb + u == r) x[u] -= 1.0f;
                }
                if (diag || edge) {
#pragma unroll
                    for (int u = 0; u < EB; ++u) {
                        const int c = c0 + cb + u;
                        bad |= !(fabsf(x[u]) <= limit) && r < K && c < K && (!diag || c >= r);
                    }
                } else {
#pragma unroll
                    for (int u = 0; u < EB; ++u) bad |= !(fabsf(x[u]) <= limit);
                }
                uint32_t own[EB];
                if (f32_out) {
#pragma unroll
                    for (int u = 0; u < EB; ++u) own[u] = __byte_perm(__float_as_uint(x[u]), 0, 0x1032);   // upper half first
                } else {
#pragma unroll
                    for (int k = 0; k < EB / 2; ++k) {
                        const float y0 = x[2 * k] * SC, y1 = x[2 * k + 1] * SC;
                        const uint32_t h = P16::from_f2(y0, y1);
                        const float2 f = P16::to_f2(h);
                        const uint32_t l = P16::from_f2(y0 - f.x, y1 - f.y);
                        own[2 * k] = __byte_perm(h, l, 0x5410);
                        own[2 * k + 1] = __byte_perm(h, l, 0x7632);
                    }
                }
                uint32_t eh[EB / 2], el[EB / 2];   // rows r & ~1, r | 1 of column c + (lane & 1)
#pragma unroll
                for (int k = 0; k < EB / 2; ++k) {
                    const uint32_t mine = odd ? own[2 * k + 1] : own[2 * k];
                    const uint32_t got = __shfl_xor_sync(0xffffffffu, odd ? own[2 * k] : own[2 * k + 1], 1);
                    const uint32_t e = odd ? got : mine, o = odd ? mine : got;
                    eh[k] = __byte_perm(e, o, 0x5410);
                    el[k] = __byte_perm(e, o, 0x7632);
                }
                if (!diag) {
#pragma unroll
                    for (int k = 0; k < EB / 2; ++k) {
                        const size_t at = (size_t)(cb + 2 * k) * ld;
                        *(uint32_t*)(out + at) = eh[k];
                        *(uint32_t*)(out + plane + at) = el[k];
                    }
                } else {
#pragma unroll
                    for (int k = 0; k < EB / 2; ++k) {
                        const size_t at = (size_t)(cb + 2 * k) * ld;
                        const int c = c0 + cb + 2 * k + odd;
                        if (c >= (r | 1)) {
                            *(uint32_t*)(out + at) = eh[k];
                            *(uint32_t*)(out + plane + at) = el[k];
                        } else if (c == (r & ~1)) {
                            out[at] = (uint16_t)eh[k];
                            out[plane + at] = (uint16_t)el[k];
                        }
                        tr[(2 * k) * 33 + lane] = own[2 * k];
                        tr[(2 * k + 1) * 33 + lane] = own[2 * k + 1];
                    }
                }
                if (diag) {
                    // the lower triangle of a diagonal block mirrors the upper one (left to
                    // their own rounding errors the two triangles drift apart, and the
                    // antisymmetric part grows exponentially along a recurrence): 2 rows x 16
                    // columns per access
                    __syncwarp();
                    uint16_t* row = (uint16_t*)S.slot[w.it.out] + (size_t)(fr * 256 + (w.i & 1) * BM + 32 * quad) * ld +
                                    fc * 256 + half * CPT + cb + (lane & 15);
#pragma unroll 4
                    for (int q = 0; q < 16; ++q) {
                        const int rr = 2 * q + (lane >> 4);
                        const uint32_t v = tr[(lane & 15) * 33 + rr];
                        if (c0 + cb + (lane & 15) > w.i * BM + 32 * quad + rr) {
                            row[(size_t)rr * ld] = (uint16_t)v;
                            row[plane + (size_t)rr * ld] = (uint16_t)(v >> 16);
                        }
                    }
                    __syncwarp();
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&accempty[a_last]);
            if (bad && limit > 0.0f) atomicExch(&S.flags[FLAG_SPECTRUM], 1);
        }
        if (!ok && lane == 0) {   // wake the MMA issuer, which sees the abort
            mbar_arrive(&accempty[0]);
            mbar_arrive(&accempty[1]);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS) : "memory");
    }
}

// FP64 symmetric matrix -> pair in a slot, zero beyond K
__global__ void __launch_bounds__(256) k_pst_split(int K, int nb, const double* __restrict__ A, uint16_t* slot) {
    using T = P16::T;
    int a = 0, t = blockIdx.x;   // block (a, b)
    while (t >= nb - a) {
        t -= nb - a;
        ++a;
    }
    const int b = a + t;
    int fr, fc;
    fold(a, b, nb, fr, fc);
    const size_t ld = (size_t)nb * 256, plane = (size_t)(nb / 2 + 1) * 256 * ld;
    const int c = threadIdx.x, gc = a * 256 + c;
    for (int r = blockIdx.y * 16; r < (int)blockIdx.y * 16 + 16; ++r) {
        const int gr = b * 256 + r;
        const double x = gr < K && gc < K ? A[(long long)gr * K + gc] * (double)SC : 0.0;
        const T h = P16::from_d(x);
        const T l = P16::from_d(x - (double)P16::to_f(h));
        uint16_t* o = slot + (size_t)(fr * 256 + r) * ld + fc * 256 + c;
        o[0] = (uint16_t)bits16(h);
        o[plane] = (uint16_t)bits16(l);
    }
}

// four consecutive elements of a pair, as stored and scaled back
__device__ __forceinline__ float4 pair4_raw(uint2 h, uint2 l) {
    using T = P16::T;
    auto f = [](uint32_t a, uint32_t b) { return P16::to_f(from_bits16<T>(a)) + P16::to_f(from_bits16<T>(b)); };
    return make_float4(f(h.x, l.x), f(h.x >> 16, l.x >> 16), f(h.y, l.y), f(h.y >> 16, l.y >> 16));
}
__device__ __forceinline__ float4 pair4(const uint16_t* p, size_t plane) {
    const float4 x = pair4_raw(*(const uint2*)p, *(const uint2*)(p + plane));
    return make_float4(ISC * x.x, ISC * x.y, ISC * x.z, ISC * x.w);
}

// block blockIdx.x of the upper block triangle
__device__ __forceinline__ void block_at(int t, int nb, int& a, int& b) {
    a = 0;
    while (t >= nb - a) {
        t -= nb - a;
        ++a;
    }
    b = a + t;
}

// C_q = sum_{r<s} c_qr T_r (T_0 = I) for up to 8 q at once, each to a slot, as
// a pair (operand) or as FP32 planes.  HBM-bound at large K (K = 4650: 1.74 GB in
// 324 us, 0.79 of the measured copy rate; K = 1230: 160 MB in 46 us, 0.52, where the
// launch has 12 blocks of 256 threads per SM): the babies are read once
// per 8 q; 4 consecutive elements per thread, FP32 FMA chains of s terms.
__global__ void __launch_bounds__(256) k_pst_combine(int K, int nb, int s, PstList T, PstOut out, int q0, int nq,
                                                     const double* __restrict__ c, int f32) {
    using H = P16::T;
    __shared__ float4 cf[PS_MAX_S][2];
    const int qb = blockIdx.z * 8, n = min(8, nq - qb);
    for (int e = threadIdx.x; e < s * 8; e += 256) {
        const int r = e >> 3, q = e & 7;
        ((float*)cf)[e] = q < n ? (float)c[(long long)(q0 + qb + q) * s + r] : 0.0f;
    }
    __syncthreads();
    int a, b, fr, fc;
    block_at(blockIdx.x, nb, a, b);
    fold(a, b, nb, fr, fc);
    const size_t ld = (size_t)nb * 256, plane = (size_t)(nb / 2 + 1) * 256 * ld;
    const int lr = blockIdx.y * 4 + (threadIdx.x >> 6), lc = (threadIdx.x & 63) * 4;
    if (b * 256 + (int)blockIdx.y * 4 >= (K + 31) / 32 * 32) return;   // beyond every operand's k range
    const size_t e0 = (size_t)(fr * 256 + lr) * ld + fc * 256 + lc;
    float acc[8][4];
    const int gr = b * 256 + lr, gc = a * 256 + lc;
#pragma unroll
    for (int q = 0; q < 8; ++q)
#pragma unroll
        for (int k = 0; k < 4; ++k) acc[q][k] = (gr == gc + k && gr < K) ? ((const float*)cf)[q] : 0.0f;
#pragma unroll 4
    for (int r = 1; r < s; ++r) {
        const float4 x = pair4((const uint16_t*)T.p[r] + e0, plane);
        const float4 c0 = cf[r][0], c1 = cf[r][1];
        const float w[8] = {c0.x, c0.y, c0.z, c0.w, c1.x, c1.y, c1.z, c1.w};
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            acc[q][0] = fmaf(w[q], x.x, acc[q][0]);
            acc[q][1] = fmaf(w[q], x.y, acc[q][1]);
            acc[q][2] = fmaf(w[q], x.z, acc[q][2]);
            acc[q][3] = fmaf(w[q], x.w, acc[q][3]);
        }
    }
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        if (q >= n) break;
        uint32_t h[4], l[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const float x = acc[q][k];
            if (f32) {
                h[k] = __float_as_uint(x) >> 16;
                l[k] = __float_as_uint(x) & 0xffffu;
            } else {
                const H th = P16::from_f(x * SC);
                h[k] = bits16(th);
                l[k] = bits16(P16::from_f(x * SC - P16::to_f(th)));
            }
        }
        uint16_t* o = (uint16_t*)out.p[qb + q] + e0;
        *(uint2*)o = make_uint2(h[0] | (h[1] << 16), h[2] | (h[3] << 16));
        *(uint2*)(o + plane) = make_uint2(l[0] | (l[1] << 16), l[2] | (l[3] << 16));
    }
}

// partial Gram sums <G_q, T_r>, 8 x 8 pairs per CTA (blockIdx.x: 8 babies,
// blockIdx.z: 8 giants) over the 4-element groups of CTA column blockIdx.y;
// off-diagonal blocks count twice.  Each baby is read once per 8 giants; the
// CTAs of one column, adjacent in launch order, share the giants' elements in
// L2, so nothing is staged: every thread keeps its 64 FP32 FMA chains
// (GRAM_GROUPS x 4 products long, the buffer of the partial sums is sized for
// that) and the chains meet in FP64.  Bound by the latency of a group's loads
// with one block of 8 warps per SM (164 registers): K = 4650, 4 giants, 1.73 GB
// in 838 us, 0.30 of the measured copy rate and 34% of the issue slots; K = 1230,
// all 58 giants, 0.62 GB in 332 us.
constexpr int GRAM_GROUPS = 32;   // 4-element groups per thread
__global__ void __launch_bounds__(256) k_pst_gram(int K, int nb, PstList G, int nq, PstList T, int s,
                                                  double* __restrict__ part) {
    __shared__ double red[8][64];
    const int rb = blockIdx.x * 8, qb = blockIdx.z * 8;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const size_t ld = (size_t)nb * 256, plane = (size_t)(nb / 2 + 1) * 256 * ld;
    const long long ngroup = (long long)(nb * (nb + 1) / 2) * 16384;   // per block 256 rows of 64 groups
    float f[8][8];
#pragma unroll
    for (int q = 0; q < 8; ++q)
#pragma unroll
        for (int r = 0; r < 8; ++r) f[q][r] = 0.0f;
    // the block of a CTA's groups is one: 256 x GRAM_GROUPS divides 16384
    static_assert(16384 % (256 * GRAM_GROUPS) == 0, "a CTA's groups must lie in one block");
    for (long long base = (long long)blockIdx.y * 256 * GRAM_GROUPS; base < ngroup;
         base += (long long)gridDim.y * 256 * GRAM_GROUPS) {
        int a, b, fr, fc;
        block_at((int)(base >> 14), nb, a, b);
        fold(a, b, nb, fr, fc);
        const float wt = a == b ? 1.0f : 2.0f;   // the pairs' scale is taken out at the end
#pragma unroll 1
        for (int g = 0; g < GRAM_GROUPS; ++g) {
            const int e = (int)(base & 16383) + g * 256 + threadIdx.x;
            const int lr = e >> 6, lc = (e & 63) * 4, gc = a * 256 + lc;
            if (b * 256 + lr >= K || gc >= K) continue;
            const size_t at = (size_t)(fr * 256 + lr) * ld + fc * 256 + lc;
            const int live = min(4, K - gc);
            // every list entry is a valid slot (the host pads them), so all loads of a
            // group are issued before the first is used
            float4 x[8];
            uint2 hx[8], lx[8], hy[4], ly[4];
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const uint16_t* g_ = (const uint16_t*)G.p[qb + q] + at;
                hx[q] = *(const uint2*)g_;
                lx[q] = *(const uint2*)(g_ + plane);
            }
            auto fetch = [&](int r0) {
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    const uint16_t* t_ = (const uint16_t*)T.p[rb + r0 + r] + at;
                    hy[r] = *(const uint2*)t_;
                    ly[r] = *(const uint2*)(t_ + plane);
                }
            };
            fetch(0);
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                x[q] = pair4_raw(hx[q], lx[q]);
                x[q].x *= wt;
                x[q].y *= wt;
                x[q].z *= wt;
                x[q].w *= wt;
                if (live < 4) {   // beyond K the slots may hold anything
                    if (live < 2) x[q].y = 0.f;
                    if (live < 3) x[q].z = 0.f;
                    x[q].w = 0.f;
                }
            }
#pragma unroll
            for (int r0 = 0; r0 < 8; r0 += 4) {
                float4 y[4];
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    y[r] = pair4_raw(hy[r], ly[r]);
                    if (live < 4) {
                        if (live < 2) y[r].y = 0.f;
                        if (live < 3) y[r].z = 0.f;
                        y[r].w = 0.f;
                    }
                }
                if (r0 == 0) fetch(4);
#pragma unroll
                for (int r = 0; r < 4; ++r)
#pragma unroll
                    for (int q = 0; q < 8; ++q)
                        f[q][r0 + r] = fmaf(x[q].x, y[r].x, fmaf(x[q].y, y[r].y, fmaf(x[q].z, y[r].z, fmaf(x[q].w, y[r].w, f[q][r0 + r]))));
            }
        }
    }
    // sums over the warp's lanes: chains of four lanes in FP32, then FP64
#pragma unroll
    for (int q = 0; q < 8; ++q)
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            float v = f[q][r];
            v += __shfl_xor_sync(0xffffffffu, v, 16);
            v += __shfl_xor_sync(0xffffffffu, v, 8);
            double d = (double)v;
            for (int o = 4; o > 0; o >>= 1) d += __shfl_xor_sync(0xffffffffu, d, o);
            if (lane == 0) red[warp][q * 8 + r] = d;
        }
    __syncthreads();
    if (threadIdx.x < 64) {
        const int q = qb + (threadIdx.x >> 3), r = rb + (threadIdx.x & 7);
        double d = 0.0;
        for (int w = 0; w < 8; ++w) d += red[w][threadIdx.x];
        if (q < nq && r < s) part[((long long)blockIdx.y * nq + q) * s + r] = d * ((double)ISC * ISC);
    }
}

// out[y * stride] = Tr of matrix y of the list
__global__ void __launch_bounds__(128) k_pst_trace(int K, int nb, PstList L, double* __restrict__ out, int stride) {
    using H = P16::T;
    __shared__ double red[4];
    const size_t ld = (size_t)nb * 256, plane = (size_t)(nb / 2 + 1) * 256 * ld;
    const uint16_t* X = (const uint16_t*)L.p[blockIdx.x];
    double x = 0.0;
    for (int i = threadIdx.x; i < K; i += 128) {
        int fr, fc;
        fold(i >> 8, i >> 8, nb, fr, fc);
        const size_t e = (size_t)(fr * 256 + (i & 255)) * ld + fc * 256 + (i & 255);
        x += (double)P16::to_f(from_bits16<H>(X[e])) + (double)P16::to_f(from_bits16<H>(X[e + plane]));
    }
    for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = x;
    __syncthreads();
    if (threadIdx.x == 0) out[(long long)blockIdx.x * stride] = (double)ISC * (red[0] + red[1] + red[2] + red[3]);
}

// rho (K x K, FP64, both triangles) = [C_0 or rho] + sum of np FP32 partial
// products - b2, these two times up: C_0 = sum_r c_0r T_r in FP32 FMA chains of
// 8 terms added in FP64
__global__ void __launch_bounds__(256) k_pst_finish(int K, int nb, int s, PstList T, const double* __restrict__ c,
                                                    PstOut part, int np, const uint16_t* b2, double up, int first,
                                                    double* __restrict__ rho) {
    using H = P16::T;
    __shared__ double sh[32][33];
    __shared__ float cf[PS_MAX_S];
    const int nt = (K + 31) / 32;
    int ti, tj;
    block_at(blockIdx.x, nt, ti, tj);
    for (int r = threadIdx.x; r < s; r += 256) cf[r] = (float)c[r];
    __syncthreads();
    int fr, fc;
    fold(ti >> 3, tj >> 3, nb, fr, fc);
    const size_t ld = (size_t)nb * 256, plane = (size_t)(nb / 2 + 1) * 256 * ld;
    const int lc = threadIdx.x & 31;
    auto pr = [](const uint16_t* p, size_t pl) {
        return ISC * (P16::to_f(from_bits16<H>(*p)) + P16::to_f(from_bits16<H>(p[pl])));
    };
    // lanes along the row index gr (contiguous in the slots), element (gr, gc), gc >= gr
    for (int lr = threadIdx.x >> 5; lr < 32; lr += 8) {
        const int gr = ti * 32 + lc, gc = tj * 32 + lr;
        double x = 0.0;
        if (gr < K && gc < K) {
            const size_t e = (size_t)(fr * 256 + (gc & 255)) * ld + fc * 256 + (gr & 255);
            if (first) {
                if (gr == gc) x = c[0];
                for (int r0 = 1; r0 < s; r0 += 8) {
                    float y[8];
#pragma unroll
                    for (int r = 0; r < 8; ++r) y[r] = r0 + r < s ? pr((const uint16_t*)T.p[r0 + r] + e, plane) : 0.0f;
                    float f = 0.0f;
#pragma unroll
                    for (int r = 0; r < 8; ++r) f = r0 + r < s ? fmaf(cf[r0 + r], y[r], f) : f;
                    x += (double)f;
                }
            } else {
                x = rho[(long long)gc * K + gr];
            }
            for (int p = 0; p < np; ++p) {
                const uint16_t* q = (const uint16_t*)part.p[p] + e;
                x = fma(up, (double)__uint_as_float(((uint32_t)q[0] << 16) | q[plane]), x);
            }
            if (b2) x = fma(-up, (double)pr(b2 + e, plane), x);
            if (gc >= gr) rho[(long long)gc * K + gr] = x;
        }
        sh[lc][lr] = x;
    }
    __syncthreads();
    for (int lr = threadIdx.x >> 5; lr < 32; lr += 8) {
        const int gr = ti * 32 + lr, gc = tj * 32 + lc;
        if (gr < K && gc < K && gc > gr) rho[(long long)gr * K + gc] = sh[lr][lc];
    }
}

// D[e] = sum of the partials, one warp per entry, in a fixed order
__global__ void __launch_bounds__(256) k_pst_gram_sum(int nsplit, int n, const double* __restrict__ part,
                                                      double* __restrict__ D) {
    const int e = (blockIdx.x * 256 + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (e >= n) return;
    double x = 0.0;
    for (int p = lane; p < nsplit; p += 32) x += part[(long long)p * n + e];
    for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
    if (lane == 0) D[e] = x;
}

int row_tiles(int K) { return (K + BM - 1) / BM; }
int sys_tiles(const Ctx& c) {
    const int nb = c.Kp / 256, mt = row_tiles(c.K);
    int n = 0;
    for (int p = 0; p < nb; ++p) n += (nb - p) * std::max(0, std::min(2, mt - 2 * p));
    return n;
}

// One call's product launches: items are queued level by level (all systems
// of the batch together) and uploaded once per flush.
struct Queue {
    Ctx& lead;
    cudaStream_t st;
    std::vector<PstItem> items;
    std::vector<int2> pairs;
    struct Launch { int first, n, tiles; };
    std::vector<Launch> launches;
    int open = 0;
    int hold;

    Queue(Ctx& l, cudaStream_t s)
        : lead(l), st(s), hold(std::getenv("DFT_TEST_EXPIRE_WAITS") ? 1 : 0) {}
    void add(int sys, const Ctx& c, std::initializer_list<int2> ab, int prev, int add_, int out, int mode, double limit) {
        PstItem it{};
        it.sys = sys;
        it.first = (int)pairs.size();
        for (const int2& x : ab) pairs.push_back(x);
        finish_item(it, c, prev, add_, out, mode, limit);
    }
    void finish_item(PstItem& it, const Ctx& c, int prev, int add_, int out, int mode, double limit) {
        it.last = (int)pairs.size();
        it.prev = prev;
        it.add = add_;
        it.out = out;
        it.mode = mode & ~PST_FINE;
        it.sub = (mode & PST_FINE) || c.K <= SUB_FINE_K ? SUB_FINE : SUB;
        it.limit = (float)limit;
        if (launches.empty() || !open) {
            launches.push_back({(int)items.size(), 0, 0});
            open = 1;
        }
        it.tile0 = launches.back().tiles;
        launches.back().tiles += sys_tiles(c);
        launches.back().n++;
        items.push_back(it);
    }
    void close() { open = 0; }   // the next item starts a new launch
    void upload() {
        if (items.empty()) return;
        if ((long long)items.size() > PST_ITEM_CAP || (long long)pairs.size() > PST_ITEM_CAP)
            throw Error(DFT_EINTERNAL, "expansion items exceed their buffer");
        DFT_CUDA_CHECK(cudaMemcpyAsync(lead.d_pst_items, items.data(), sizeof(PstItem) * items.size(),
                                       cudaMemcpyHostToDevice, st));
        DFT_CUDA_CHECK(cudaMemcpyAsync(lead.d_pst_pairs, pairs.data(), sizeof(int2) * pairs.size(),
                                       cudaMemcpyHostToDevice, st));
    }
    void launch(size_t k) {
        const Launch& l = launches[k];
        const int grid = std::min(l.tiles, SMS);
        k_pst_prod<<<grid, NTHREADS, SMEM_BYTES, st>>>(lead.d_pst_sys, lead.d_pst_items + l.first, l.n, lead.d_pst_pairs,
                                                       l.tiles, lead.d_flags, hold);
        check_launch("pst_prod");
    }
    void run() {
        upload();
        for (size_t k = 0; k < launches.size(); ++k) launch(k);
        items.clear();
        pairs.clear();
        launches.clear();
        open = 0;
    }
};

// slots of one system: babies T_1 .. T_s at 0 .. s - 1; direct plan: giants
// G_2 .. G_Q at s .. s + Q - 2, then C_q and partial sums; Clenshaw plan: two
// rolling buffers, then C_q (and giants on their way to the Gram sums)
struct View {
    Ctx& c;
    const PsPlan& p;
    explicit View(Ctx& x) : c(x), p(x.ps) {}
    int baby(int r) const { return r - 1; }
    int giant(int q) const { return q == 1 ? p.s - 1 : p.s + q - 2; }
    int extra(int i) const { return p.s + (p.direct ? std::max(0, p.Q - 1) : 0) + i; }
    int nextra() const { return (int)c.pst_slot.size() - extra(0); }
    // T_0 = I is not stored: its entry, and those behind the last, hold T_1's slot
    PstList babies() const {
        PstList T;
        for (int r = 0; r < PS_MAX_S; ++r) T.p[r] = c.pst_slot[baby(r > 0 && r < p.s ? r : 1)];
        return T;
    }
};

void gram(Ctx& c, int q0, const std::vector<int>& slots, cudaStream_t st) {
    const View v(c);
    const int s = v.p.s, nb = c.Kp / 256;
    double* D = c.d_wk;
    const PstList T = v.babies();
    for (size_t k = 0; k < slots.size(); k += PS_MAX_S) {
        const int nq = (int)std::min<size_t>(PS_MAX_S, slots.size() - k);
        PstList G;
        for (int q = 0; q < PS_MAX_S; ++q) G.p[q] = c.pst_slot[slots[k + std::min(q, nq - 1)]];
        if ((long long)nq * s > c.gram_cap) throw Error(DFT_EINTERNAL, "Gram partials exceed their buffer");
        // chains of GRAM_GROUPS groups (longer only if the partial sums did not fit their buffer)
        const int nsplit = (int)std::max<long long>(
            1, std::min<long long>({(long long)nb * (nb + 1) / 2 * (16384 / (256 * GRAM_GROUPS)),
                                    c.gram_cap / ((long long)nq * s), 65535LL}));
        const dim3 grid((s + 7) / 8, nsplit, (nq + 7) / 8);
        double* Dq = D + (long long)(q0 + k) * s;
        if (s > 1) {
            k_pst_gram<<<grid, 256, 0, st>>>(c.K, nb, G, nq, T, s, c.d_gram);
            k_pst_gram_sum<<<(nq * s + 7) / 8, 256, 0, st>>>(nsplit, nq * s, c.d_gram, Dq);
        }
        k_pst_trace<<<nq, 128, 0, st>>>(c.K, nb, G, Dq, s);
        check_launch("pst_gram", 3);
    }
}

void combine(Ctx& c, const double* cf, int q0, int nq, const std::vector<int>& out, bool f32, cudaStream_t st) {
    const View v(c);
    const int nb = c.Kp / 256;
    PstOut o{};
    for (int q = 0; q < nq; ++q) o.p[q] = c.pst_slot[out[q]];
    const PstList T = v.babies();
    const dim3 grid(nb * (nb + 1) / 2, 64, (nq + 7) / 8);
    k_pst_combine<<<grid, 256, 0, st>>>(c.K, nb, v.p.s, T, o, q0, nq, cf, f32 ? 1 : 0);
    check_launch("pst_combine");
}

void finish(Ctx& c, const double* cf, const std::vector<int>& part, int b2, bool first, cudaStream_t st) {
    const View v(c);
    const int nt = (c.K + 31) / 32;
    PstOut o{};
    for (size_t q = 0; q < part.size(); ++q) o.p[q] = c.pst_slot[part[q]];
    const PstList T = v.babies();
    const uint16_t* b = b2 >= 0 ? (const uint16_t*)c.pst_slot[b2] : nullptr;
    const int np = (int)part.size();
    k_pst_finish<<<nt * (nt + 1) / 2, 256, 0, st>>>(c.K, c.Kp / 256, v.p.s, T, cf, o, np, b, 1.0 / v.p.down, first, c.d_rho);
    check_launch("pst_finish");
}

double* coef_ps(Ctx& c) { return c.d_coef + c.n_c_cur; }

}  // namespace

size_t pst_slot_bytes(int Kp) {
    const size_t nb = Kp / 256;
    return (nb / 2 + 1) * 256 * (size_t)Kp * 4;
}

// tensor maps of every slot (K-major boxes of 128 and 256 rows, transposed
// boxes of 128 and 256 columns; both planes are rows of one map) and the slot
// table, uploaded once
void pst_setup(Ctx& c, cudaStream_t st) {
    const int n = (int)c.pst_slot.size(), nb = c.Kp / 256;
    std::vector<CUtensorMap> maps(4 * (size_t)n);
    const cuuint64_t rows = (cuuint64_t)(nb / 2 + 1) * 256 * 2, ld = (cuuint64_t)c.Kp;
    for (int k = 0; k < n; ++k) {
        for (int v = 0; v < 2; ++v) {
            cuuint64_t dims[2] = {ld, rows}, strides[1] = {ld * 2};
            cuuint32_t box[2] = {(cuuint32_t)BK, (cuuint32_t)(v ? BN : BM)}, es[2] = {1, 1};
            CUresult r = encode_fn()(&maps[4 * k + v], CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, c.pst_slot[k], dims, strides,
                                     box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B,
                                     CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
            if (r != CUDA_SUCCESS) throw Error(DFT_ECUDA, "cuTensorMapEncodeTiled (slot) failed");
        }
        for (int v = 0; v < 2; ++v) {
            cuuint64_t dims[3] = {64, rows, ld / 64}, strides[2] = {ld * 2, 128};
            cuuint32_t box[3] = {64, (cuuint32_t)BK, (cuuint32_t)((v ? BN : BM) / 64)}, es[3] = {1, 1, 1};
            CUresult r = encode_fn()(&maps[4 * k + 2 + v], CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 3, c.pst_slot[k], dims,
                                     strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                                     CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
            if (r != CUDA_SUCCESS) throw Error(DFT_ECUDA, "cuTensorMapEncodeTiled (transposed slot) failed");
        }
    }
    DFT_CUDA_CHECK(cudaMemcpyAsync(c.d_pst_maps, maps.data(), sizeof(CUtensorMap) * maps.size(), cudaMemcpyHostToDevice, st));
    DFT_CUDA_CHECK(cudaMemcpyAsync(c.d_pst_slots, c.pst_slot.data(), sizeof(void*) * n, cudaMemcpyHostToDevice, st));
    DFT_CUDA_CHECK(cudaStreamSynchronize(st));   // the host staging goes out of scope
    DFT_CUDA_CHECK(cudaFuncSetAttribute(k_pst_prod, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_BYTES));
}

// T_1 = H_N (from c.d_H, which is free afterwards)
void pst_split_h(Ctx& c, cudaStream_t st) {
    const int nb = c.Kp / 256;
    const dim3 grid(nb * (nb + 1) / 2, 16);
    uint16_t* t1 = (uint16_t*)c.pst_slot[0];
    k_pst_split<<<grid, 256, 0, st>>>(c.K, nb, c.d_H, t1);
    check_launch("pst_split");
}

// Babies, giants and moments of every system (T_1 in place).  moments[q] = 0:
// the coefficients of system q are already fixed, so a Clenshaw plan forms no
// giants and only the spectrum check is left of them.
void pst_pass1(Ctx* const* cs, int n, const int* moments, cudaStream_t st) {
    Ctx& lead = *cs[0];
    std::vector<PstSys> tab(n);
    for (int k = 0; k < n; ++k) {
        Ctx& c = *cs[k];
        const int nslot = (int)c.pst_slot.size();
        // T_1 takes a slot here
        const double waves = sys_tiles(c) / (double)SMS;
        c.ps = ps_plan(c.n_c_cur, nslot - 1, std::ceil(waves), waves, 6);
        c.ps.down = c.ps.direct ? 1.0f : clenshaw_down(c.ps.Q);
        tab[k] = PstSys{c.K, c.Kp / 256, c.d_pst_maps, c.d_pst_slots, c.d_flags};
    }
    DFT_CUDA_CHECK(cudaMemcpyAsync(lead.d_pst_sys, tab.data(), sizeof(PstSys) * n, cudaMemcpyHostToDevice, st));
    Queue Q(lead, st);
    // doubling of every system's X_1 .. X_top, level by level together
    auto doubling = [&](auto&& top_of, auto&& slot_of, auto&& limit_of) {
        for (int m = 1;; m *= 2) {
            bool any = false;
            for (int k = 0; k < n; ++k) {
                const int top = top_of(k);
                for (int j = 1; j <= std::min(m, top - m); ++j) {
                    Q.add(k, *cs[k], {make_int2(slot_of(k, m), slot_of(k, j))}, m > j ? slot_of(k, m - j) : -1, -1,
                          slot_of(k, m + j), PST_ALPHA2 | (m == j ? PST_IDENT : 0), limit_of(k, m + j));
                    any = true;
                }
            }
            Q.close();
            if (!any) break;
        }
    };
    for (int r = 1;; ++r) {
        bool any = false;
        for (int k = 0; k < n; ++k) {
            const PsPlan& p = cs[k]->ps;
            if (r >= (p.Q > 0 ? p.s : p.s - 1)) continue;
            const View v(*cs[k]);
            Q.add(k, *cs[k], {make_int2(v.baby(1), v.baby(r))}, r > 1 ? v.baby(r - 1) : -1, -1, v.baby(r + 1),
                  PST_FINE | PST_ALPHA2 | (r == 1 ? PST_IDENT : 0), r + 1 == p.s && p.Q == 1 ? growth_limit(p.s, p.n_c) : 4.0);
            any = true;
        }
        Q.close();
        if (!any) break;
    }
    doubling([&](int k) { const PsPlan& p = cs[k]->ps; return p.direct ? p.Q : 0; },
             [&](int k, int q) { return View(*cs[k]).giant(q); },
             [&](int k, int q) { const PsPlan& p = cs[k]->ps; return q == p.Q ? growth_limit(p.Q * p.s, p.n_c) : 4.0; });
    Q.run();
    for (int k = 0; k < n; ++k) {
        Ctx& c = *cs[k];
        const PsPlan& p = c.ps;
        const View v(c);
        const int s = p.s, nb = c.Kp / 256;
        if (moments[k] && s > 1) {
            PstList L{};
            for (int r = 1; r < s; ++r) L.p[r - 1] = c.pst_slot[v.baby(r)];
            k_pst_trace<<<s - 1, 128, 0, st>>>(c.K, nb, L, c.d_wk + 1, 1);
            check_launch("pst_trace");
        }
        if (p.direct && moments[k] && p.Q > 0) {
            std::vector<int> g;
            for (int q = 1; q <= p.Q; ++q) g.push_back(v.giant(q));
            gram(c, 1, g, st);
        }
        if (!p.direct && moments[k] && p.Q > 0) {
            const int r0 = v.extra(0), nring = v.nextra(), ts = v.baby(s);
            // giants G_2 .. G_Q (none where Q = 1, whose G_1 = T_s has its Gram sums all
            // the same) in a ring of nring buffers; the Gram sums take up to nring - 2
            // at a time, so that the babies are read less often
            std::vector<int> at(p.Q + 1, ts);
            for (int q = 2; q <= p.Q; ++q) at[q] = r0 + (q - 2) % nring;
            for (int q = 1; q < p.Q; ++q) {
                Q.add(k, c, {make_int2(ts, at[q])}, q > 1 ? at[q - 1] : -1, -1, at[q + 1],
                      PST_ALPHA2 | (q == 1 ? PST_IDENT : 0), q + 1 == p.Q ? growth_limit(p.Q * s, p.n_c) : 4.0);
                Q.close();
            }
            Q.upload();
            int done = 1;   // giants 1 .. done - 1 are in the Gram sums
            for (int q = 1; q <= p.Q; ++q) {
                const int have = q - done + 1;
                if (q == p.Q || have >= std::max(1, nring - 2)) {
                    gram(c, done, std::vector<int>(at.begin() + done, at.begin() + q + 1), st);
                    done = q + 1;
                }
                if (q < p.Q) Q.launch(q - 1);
            }
            Q.items.clear();
            Q.pairs.clear();
            Q.launches.clear();
            Q.open = 0;
        }
        // the spectrum check beyond the last giant (the giants' buffers, or those behind them, are free)
        const PsCheck ck = ps_check(p, p.direct || moments[k]);
        int cur = v.baby(std::max(1, ck.baby));
        for (int i = 0, l = ck.baby; i < ck.doublings; ++i) {
            // T_{2l} = 2 T_l^2 - I or T_{2l+1} = 2 T_l T_{l+1} - T_1
            const int out = v.extra(i & 1);
            l *= 2;
            Q.add(k, c, {make_int2(cur, ck.odd ? cur + 1 : cur)}, ck.odd ? v.baby(1) : -1, -1, out,
                  PST_ALPHA2 | (ck.odd ? 0 : PST_IDENT), i + 1 == ck.doublings ? growth_limit(l + ck.odd, p.n_c) : 4.0);
            Q.close();
            cur = out;
        }
        Q.run();
        if (moments[k]) launch_ps_moments(c.K, p, c.d_wk, c.d_mom, st);
    }
}

// rho = sum_l a_l T_l of every system (coefficients in its d_coef) into d_rho
void pst_pass2(Ctx* const* cs, int n, cudaStream_t st) {
    Ctx& lead = *cs[0];
    Queue Q(lead, st);
    for (int k = 0; k < n; ++k) {
        Ctx& c = *cs[k];
        launch_ps_coefs(c.ps, c.d_coef, coef_ps(c), coef_ps(c) + (long long)(c.ps.Q + 1) * c.ps.s, st);
    }
    // direct plans: chunks of giants, all systems' products of a chunk together
    std::vector<int> at(n, 1);
    for (bool any = true; any;) {
        any = false;
        std::vector<std::vector<int>> part(n);
        int total = 0;
        for (int k = 0; k < n; ++k)
            if (cs[k]->ps.direct) total += sys_tiles(*cs[k]);
        for (int k = 0; k < n; ++k) {
            Ctx& c = *cs[k];
            const PsPlan& p = c.ps;
            const View v(c);
            if (!p.direct || at[k] > p.Q) continue;
            any = true;
            const int left = p.Q - at[k] + 1, spare = v.nextra();
            // about four waves of tiles over the batch; fewer giants per FP32 sum also
            // mean less rounding
            const int want = std::max(1, std::min(left, 4 * SMS / std::max(1, total) + 1));
            const int np = std::max(1, std::min({want, spare / 2, PS_MAX_ITEMS}));
            const int nq = std::min({left, spare - np, PS_MAX_ITEMS});
            std::vector<int> cq;
            for (int q = 0; q < nq; ++q) cq.push_back(v.extra(q));
            combine(c, coef_ps(c), at[k], nq, cq, false, st);
            const int npu = std::min(np, nq);
            for (int y = 0; y < npu; ++y) {
                PstItem it{};
                it.sys = k;
                it.first = (int)Q.pairs.size();
                for (int q = (int)((long long)nq * y / npu); q < (int)((long long)nq * (y + 1) / npu); ++q)
                    Q.pairs.push_back(make_int2(v.giant(at[k] + q), cq[q]));
                part[k].push_back(v.extra(nq + y));
                Q.finish_item(it, c, -1, -1, part[k].back(), PST_OUT_F32, 0.0);
            }
        }
        if (!any) break;
        Q.run();
        for (int k = 0; k < n; ++k) {
            Ctx& c = *cs[k];
            if (part[k].empty()) continue;
            const bool first = at[k] == 1;
            const int left = c.ps.Q - at[k] + 1, spare = View(c).nextra();
            const int want = std::max(1, std::min(left, 4 * SMS / std::max(1, total) + 1));
            const int np = std::max(1, std::min({want, spare / 2, PS_MAX_ITEMS}));
            at[k] += std::min({left, spare - np, PS_MAX_ITEMS});
            finish(c, coef_ps(c), part[k], -1, first, st);
        }
    }
    for (int k = 0; k < n; ++k) {
        Ctx& c = *cs[k];
        const PsPlan& p = c.ps;
        const View v(c);
        if (p.Q == 0) {
            finish(c, coef_ps(c), {}, -1, true, st);
            continue;
        }
        if (p.direct) continue;
        // Clenshaw in T_s: b_q = C_q + 2 T_s b_{q+1} - b_{q+2}, C_q formed W at a time
        const int W = std::min(8, v.nextra() - 2), ts = v.baby(p.s);
        int b1 = v.extra(0), b2 = v.extra(1);
        combine(c, coef_ps(c), p.Q, 1, {b1}, false, st);
        std::vector<int> add_at(p.Q + 1);
        bool have2 = false;
        for (int q = p.Q - 1; q >= 1; --q) {
            add_at[q] = v.extra(2 + (p.Q - 1 - q) % W);
            Q.add(k, c, {make_int2(ts, b1)}, have2 ? b2 : -1, add_at[q], b2, PST_ALPHA2, 0.0);
            Q.close();
            std::swap(b1, b2);
            have2 = true;
        }
        const int tail = v.extra(2);
        Q.add(k, c, {make_int2(ts, b1)}, -1, -1, tail, PST_OUT_F32, 0.0);
        Q.upload();
        int l = 0;
        for (int q = p.Q - 1; q >= 1; --q, ++l) {
            if ((p.Q - 1 - q) % W == 0) {
                // C_{q - m + 1} .. C_q, lowest first
                const int m = std::min(W, q);
                std::vector<int> o;
                for (int i = 0; i < m; ++i) o.push_back(add_at[q - m + 1 + i]);
                combine(c, coef_ps(c), q - m + 1, m, o, true, st);
            }
            Q.launch(l);
        }
        Q.launch(l);
        finish(c, coef_ps(c), {tail}, have2 ? b2 : -1, true, st);
        Q.items.clear();
        Q.pairs.clear();
        Q.launches.clear();
        Q.open = 0;
    }
}

}  // namespace dft
