// Tensor-core adjoint of the SH bake (sm_103a): see the comment at the top of namespace bwd.
#include "shm_tc.cuh"

namespace shm {
namespace tc {
// ------------------------------------------------------------------------------------------
// Adjoint of the bake on the tensor cores.  The bake is linear in the coefficients (Algorithm 1:
// table = sum_k c_k basis_k), so its reverse mode is the transposed contraction
//     dcoeffs[g][k] = sum_c dlut[g][c] basis[k][c]                     (c over the 4T table scalars)
// with a CTA's group of up to 128 glyphs on the MMA M side (rows beyond the group hold stale data and
// are never stored; see plan() for the group size) and the coefficients on N (K padded to
// Kp <= 128).  Operands:
//   A = dlut tiles [R glyphs x 32 c], loaded raw by TMA (128-byte swizzle) and split by four warps,
//       one glyph row per thread, into tf32 hi = x truncated and lo = tf32_rna(x - hi), which go to
//       TMEM: the MMAs read A from there;
//   B = the transposed tf32 split of the basis, hiS / loS (part of shm_sh_basis's buffer), stored as
//       one contiguous [Kp][16 c] slab per 16 columns with its rows already in the 64-byte swizzled
//       order that a tensor load would produce, so each B tile is one plain bulk copy (a tensor load
//       of [Kp][16] from a [Kp][4T] array would be Kp separate 64-byte pieces).
// D = A_hi B_hi + A_hi B_lo + A_lo B_hi (3xTF32, as the forward bake), in two MMAs per K step: B_hi
// and B_lo lie back to back in a stage, so A_hi [B_hi; B_lo] is one MMA of N = 2 Kp whose columns
// [0, Kp) take A_hi B_hi and [Kp, 2 Kp) A_hi B_lo, and A_lo B_hi adds into [0, Kp); the drain warps
// add both halves.
// What bounds it: HBM reads of dlut (455 MB in 67 us at 4,096 glyphs, N = 32) and, with hi and lo in
// shared memory, that memory's port (78 KB of traffic per 8 KB of A: raw in, out, hi and lo in, and
// out again for the MMAs; 46 KB with A in TMEM) and the per-stage work of the roles, which are serial
// chains of waits.  A training step (query, its reverse, this kernel, the bake; 4,096 glyphs, N = 32,
// L = 8) took 867 us with 16-column stages split in shared memory by six warps; 837 with two slabs a
// stage; 834 with A in TMEM, 802 when the drain's sums stopped taking registers from the other roles
// and ring positions were counted instead of divided, 797 without an L2 prefetch of dlut (160 KB of
// loads in flight need none).  At 16,384 glyphs this kernel went from 852 us to 597 (floor 267).
// Tried: 1 / 4 slabs a stage 852 / 935 (the serial chain; too few TMEM slots); one accumulator and more
// slots 802; stores to TMEM waited for a stage later 800-811.
// Accuracy: the error of the tensor cores' float32 accumulation grew with the length of the sum
// kept in one TMEM accumulator (measured: 4.6e-5 of the largest entry after 434 stages, against
// 7.9e-6 for a plain float32 sum).  So the MMAs accumulate CH stages at a time into one of two
// TMEM buffers, and four drain warps add each finished chunk into float32 registers (one glyph row
// per thread, Kp values) while the MMAs fill the other buffer.
// TMEM (512 columns): two accumulators of 2 Kp columns, then as many split stages of 64 columns as
// fit; at Kp = 128 one accumulator, else no column were left (each chunk's drain then holds up the MMAs).
// The c range may be split over the S CTAs of a thread-block cluster (small glyph counts); at the
// end every CTA writes its register sums to shared memory and each CTA sums a slice of them over
// the cluster's ranks in rank order through distributed shared memory, so the result does not
// depend on timing (deterministic, no atomics, no workspace).
//   warp 0 lane 0: TMA producer   warp 1: TMEM allocation, lane 0 issues the MMAs
//   warps 4-7: drain and its partial sums   warps 8-11: tf32 split   (TMEM lane quadrant = warp % 4)
// Every mbarrier wait is bounded (1 s) and raises SHM_DEV_TIMEOUT on expiry; the cluster barriers
// are reached by every thread of every CTA the same number of times, aborted or not.
namespace bwd {

constexpr int MG = 128;                       // glyph rows (MMA M)
constexpr int KPMAX = 128;                    // register sums per drain thread
constexpr int SUB = 2;                        // 16-column slabs per stage (a row of A: 128 bytes)
constexpr uint32_t A_BYTES = MG * SUB * KC * 4;  // 16 KB
constexpr int CH = 16 / SUB;                  // stages per TMEM chunk (256 columns)
constexpr int THREADS = 384;
constexpr int SPLIT_T = 128;                  // tf32-split threads: warps 8-11, one glyph row each
constexpr uint32_t STAGE_CAP = 196 * 1024;    // shared memory for the stages (and the partials after them)
constexpr uint32_t BAR_BYTES = 1024;
constexpr int MAXSTAGE = 8;

struct Args {
    const float* hiS;  // basis slabs, [NC][Kp][16] each, rows pre-swizzled
    const float* loS;
    int M4;        // table scalars per glyph (4T), the reduction length
    int G, K, Kp;
    int R;         // glyph rows per group (<= MG; the MMA's rows beyond R are never stored)
    int groups;
    int S;         // CTAs per cluster (splits of the c range)
    int NC;        // slabs over the whole c range
    int nstage;    // pipeline depth
    int nacc;      // accumulators in TMEM
    int nslot;     // split A stages in TMEM
    uint32_t b_bytes, stage_bytes;  // one B tile; a stage: A, then B hi and B lo of each slab
    float* dcoeffs;
    int32_t* dev_status;
};

// Plain bulk copy of `bytes` (a multiple of 16, both addresses 16-byte aligned) into shared memory,
// completing on `bar`.
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(dst), "l"(src), "r"(bytes), "r"(bar)
                 : "memory");
}

// tf32 by truncation (the low 13 mantissa bits cleared): one logic operation where the rounding
// conversion is a slower instruction; the remainder x - hi is exact and carries what was cut off.
__device__ __forceinline__ float tf32_trunc(float x) { return __uint_as_float(__float_as_uint(x) & 0xFFFFE000u); }

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

__device__ __forceinline__ float ld_dsmem(uint32_t local_addr, uint32_t rank)
{
    uint32_t remote;
    float v;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(local_addr), "r"(rank));
    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(remote) : "memory");
    return v;
}

__device__ __forceinline__ uint32_t idesc(int NB)
{
    return (1u << 4) | (2u << 7) | (2u << 10) | ((uint32_t)(NB >> 3) << 17) | ((uint32_t)(MG >> 4) << 24);
}

// D += A B with A in TMEM (lane = row, one column per k) and B in shared memory.
__device__ __forceinline__ void mma_tf32_n(uint32_t d, uint32_t a, uint64_t b, uint32_t id, uint32_t acc)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::tf32 [%0], [%1], %2, %3, p;\n\t}\n"
        ::"r"(d), "r"(a), "l"(b), "r"(id), "r"(acc)
        : "memory");
}

// 32 columns of this warp's 32 TMEM lanes
__device__ __forceinline__ void tmem_st32(uint32_t taddr, const uint32_t (&r)[32])
{
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x32.b32 [%32], "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31};"
        ::"r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
          "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]),
          "r"(r[16]), "r"(r[17]), "r"(r[18]), "r"(r[19]), "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]),
          "r"(r[24]), "r"(r[25]), "r"(r[26]), "r"(r[27]), "r"(r[28]), "r"(r[29]), "r"(r[30]), "r"(r[31]),
          "r"(taddr)
        : "memory");
}

// Position in a ring of n buffers and the parity of its current pass.
struct Ring {
    int i, n;
    uint32_t ph;
    __device__ __forceinline__ explicit Ring(int n_) : i(0), n(n_), ph(0) {}
    __device__ __forceinline__ void next()
    {
        if (++i == n) { i = 0; ph ^= 1; }
    }
};

__global__ void __launch_bounds__(THREADS, 1)
    k_sh_gemm_bwd_tc(const __grid_constant__ CUtensorMap mA, Args a)
{
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint8_t* bars = smem;
    uint8_t* stages = smem + BAR_BYTES;
    // barriers: full / conv / empty per stage (MAXSTAGE each at most), chunk full / empty per TMEM
    // buffer, the drain barrier
    const uint32_t full0 = smem_u32(bars), conv0 = full0 + 8 * MAXSTAGE, empty0 = conv0 + 8 * MAXSTAGE,
                   cfull0 = empty0 + 8 * MAXSTAGE, cempty0 = cfull0 + 16, drain = cempty0 + 16;
    uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(bars + 512);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(bars + 520);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = cluster_rank();
    const int g_base = (blockIdx.x / a.S) * a.R;
    const int c0 = (int)(((int64_t)a.NC * rank) / a.S), c1 = (int)(((int64_t)a.NC * (rank + 1)) / a.S);
    const int nsl = c1 - c0;                     // slabs of this CTA
    const int nst = (nsl + SUB - 1) / SUB;       // stages, the last one with fewer slabs perhaps
    const int nchunk = (nst + CH - 1) / CH;
    const uint32_t ID = idesc(a.Kp), ID2 = idesc(2 * a.Kp);

    const auto slabs_of = [&](int it) { return min(SUB, nsl - it * SUB); };
    // stage st: A raw, then B hi and B lo of slab u back to back
    const auto stA = [&](int st) { return stages + (size_t)st * a.stage_bytes; };
    const auto stB = [&](int st, int u) { return smem_u32(stA(st)) + A_BYTES + (uint32_t)u * 2 * a.b_bytes; };

    if (threadIdx.x == 0) {
        for (int st = 0; st < a.nstage; ++st) {
            mbar_init(full0 + 8 * st, 1);
            mbar_init(conv0 + 8 * st, SPLIT_T);
            mbar_init(empty0 + 8 * st, 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(cfull0 + 8 * b, 1);
            mbar_init(cempty0 + 8 * b, 128);
        }
        mbar_init(drain, 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_holder)),
                     "r"(512u)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = *tmem_holder;
    const uint32_t tmem_a = tmem + (uint32_t)(a.nacc * 2 * a.Kp);  // then nslot split stages of 32 SUB columns
    float* P = reinterpret_cast<float*>(stages);  // [128][Kp + 1] partial sums of this CTA, after the last MMA
    const int PS = a.Kp + 1;

    if (warp == 0 && lane == 0) {
        // ---------------------------------------------------------------- TMA producer
        int it = 0;
        Ring r(a.nstage);
        for (; it < nst; ++it, r.next()) {
            const int st = r.i;
            const uint32_t ph = r.ph;
            if (!mbar_wait(empty0 + 8 * st, ph ^ 1, abort_flag, WAIT_LIMIT_NS)) break;
            const uint32_t fb = full0 + 8 * st;
            const int m = slabs_of(it);
            // the box is SUB slabs wide also where the range ends with fewer (columns past it are not used)
            mbar_expect_tx(fb, (uint32_t)a.R * SUB * KC * 4 + (uint32_t)m * 2 * a.b_bytes);
            tma_load_2d(smem_u32(stA(st)), &mA, (c0 + it * SUB) * KC, g_base, fb);
            for (int u = 0; u < m; ++u) {
                const size_t slab = (size_t)(c0 + it * SUB + u) * a.Kp * KC;
                bulk_load(stB(st, u), a.hiS + slab, a.b_bytes, fb);
                bulk_load(stB(st, u) + a.b_bytes, a.loS + slab, a.b_bytes, fb);
            }
        }
        if (it < nst) {
            // aborted: the last load issued into each stage must land before the shared memory is reused
            for (int k = 1; k <= a.nstage && k <= it; ++k) {
                const int last = it - k;
                const uint64_t t0 = globaltimer();
                while (!mbar_try_wait(full0 + 8 * (last % a.nstage), (uint32_t)(last / a.nstage) & 1) &&
                       globaltimer() - t0 < DRAIN_LIMIT_NS) {
                }
            }
        }
    } else if (warp == 1 && lane == 0) {
        // ---------------------------------------------------------------- MMA issuer
        bool ok = true, any = false;
        int it = 0;
        Ring rs(a.nstage), ra(a.nslot);
        for (int j = 0; j < nchunk && ok; ++j) {
            const int b = j % a.nacc;
            if (!mbar_wait(cempty0 + 8 * b, ((uint32_t)(j / a.nacc) & 1) ^ 1, abort_flag, WAIT_LIMIT_NS)) { ok = false; break; }
            fence_after();
            const uint32_t d = tmem + (uint32_t)(b * 2 * a.Kp);
            const int jend = min(nst, (j + 1) * CH);
            for (; it < jend; ++it, rs.next(), ra.next()) {
                const int st = rs.i;
                const uint32_t ph = rs.ph;
                if (!mbar_wait(conv0 + 8 * st, ph, abort_flag, WAIT_LIMIT_NS)) { ok = false; break; }
                fence_after();
                const int m = slabs_of(it);
                for (int u = 0; u < m; ++u) {
                    const uint32_t ah = tmem_a + (uint32_t)((ra.i * SUB + u) * 32), al = ah + 16;
                    const uint32_t bh = stB(st, u);
#pragma unroll
                    for (int kk = 0; kk < KC / 8; ++kk) {
                        const uint32_t o = kk * 32;  // bytes of 8 k in B; A: 8 columns
                        // columns [0, Kp): A_hi B_hi (+ A_lo B_hi below); [Kp, 2 Kp): A_hi B_lo, one MMA of
                        // N = 2 Kp over the slab's B_hi and B_lo, which lie back to back
                        mma_tf32_n(d, ah + kk * 8, sdesc(bh + o), ID2, (it != j * CH || u != 0 || kk != 0) ? 1u : 0u);
                        mma_tf32_n(d, al + kk * 8, sdesc(bh + o), ID, 1);
                    }
                }
                any = true;
                mma_commit(empty0 + 8 * st);
            }
            if (ok) mma_commit(cfull0 + 8 * b);
        }
        if (!ok && any) {
            mma_commit(drain);
            const uint64_t t0 = globaltimer();
            while (!mbar_try_wait(drain, 0) && globaltimer() - t0 < DRAIN_LIMIT_NS) {
            }
        }
    } else if (warp >= 8) {
        // ---------------------------------------------------------------- tf32 split of each stage
        // thread = glyph row = TMEM lane; a stage's hi and lo go to 32 columns of TMEM per slab
        const int wq = warp & 3, row = 32 * wq + lane;
        const uint32_t lanes = (uint32_t)(32 * wq) << 16;
        Ring rs(a.nstage), ra(a.nslot), rp(a.nstage);
        for (int it = 0; it < nst; ++it, rs.next(), ra.next()) {
            float4 v[SUB][4];
            bool ok = mbar_wait(full0 + 8 * rs.i, rs.ph, abort_flag, WAIT_LIMIT_NS);
            const uint8_t* src = stA(rs.i) + row * (SUB * KC * 4);
#pragma unroll
            for (int u = 0; u < SUB; ++u)
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    v[u][q] = *reinterpret_cast<const float4*>(src + 16 * ((4 * u + q) ^ (row & 7)));
            if (it >= a.nslot) {  // the MMAs that read this TMEM slot before
                ok = ok && mbar_wait(empty0 + 8 * rp.i, rp.ph, abort_flag, WAIT_LIMIT_NS);
                rp.next();
            }
            if (!__all_sync(0xFFFFFFFFu, ok)) break;
            fence_after();
#pragma unroll
            for (int u = 0; u < SUB; ++u) {
                uint32_t r[32];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const float x[4] = {v[u][q].x, v[u][q].y, v[u][q].z, v[u][q].w};
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const float h = tf32_trunc(x[e]);
                        r[4 * q + e] = __float_as_uint(h);
                        r[16 + 4 * q + e] = __float_as_uint(tf32_rna(x[e] - h));
                    }
                }
                tmem_st32(tmem_a + lanes + (uint32_t)((ra.i * SUB + u) * 32), r);
            }
            asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
            fence_before();
            mbar_arrive(conv0 + 8 * rs.i);
        }
    } else if (warp >= 4) {
        // ---------------------------------------------------------------- drain: chunk sums -> registers
        const int wq = warp & 3;
        float acc[KPMAX];  // the glyph row's running sums
#pragma unroll
        for (int i = 0; i < KPMAX; ++i) acc[i] = 0.0f;
        int j = 0;
        for (; j < nchunk; ++j) {
            const int b = j % a.nacc;
            if (!mbar_wait(cfull0 + 8 * b, (uint32_t)(j / a.nacc) & 1, abort_flag, WAIT_LIMIT_NS)) break;
            fence_after();
#pragma unroll
            for (int cc = 0; cc < KPMAX; cc += 32) {
                if (cc < a.Kp) {
                    uint32_t r[32];
                    const uint32_t t0 = tmem + ((uint32_t)(32 * wq) << 16) + (uint32_t)(b * 2 * a.Kp + cc);
                    tmem_ld32(t0, r);  // A_hi B_hi + A_lo B_hi
#pragma unroll
                    for (int i = 0; i < 32; ++i) acc[cc + i] += __uint_as_float(r[i]);
                    tmem_ld32(t0 + (uint32_t)a.Kp, r);  // A_hi B_lo
#pragma unroll
                    for (int i = 0; i < 32; ++i) acc[cc + i] += __uint_as_float(r[i]);
                }
            }
            fence_before();
            mbar_arrive(cempty0 + 8 * b);
        }
        // all MMAs of this CTA are done, so every stage has been loaded, split and read
        if (j == nchunk) {
            const int row = 32 * wq + lane;
#pragma unroll
            for (int i = 0; i < KPMAX; ++i)
                if (i < a.Kp) P[row * PS + i] = acc[i];
        }
    }
    __syncthreads();
    // ---------------------------------------------------------------- epilogue: cluster reduction
    const bool aborted = *abort_flag != 0;
    cluster_sync();
    const uint32_t P_s = smem_u32(P);
    const int E = a.R * a.K;
    const int e0 = (int)(((int64_t)E * rank) / a.S), e1 = (int)(((int64_t)E * (rank + 1)) / a.S);
    for (int e = e0 + threadIdx.x; e < e1; e += blockDim.x) {
        const int row = e / a.K, k = e - row * a.K;
        const int g = g_base + row;
        float sum = 0.0f;
        for (int rr = 0; rr < a.S; ++rr) sum += ld_dsmem(P_s + 4u * (uint32_t)(row * PS + k), (uint32_t)rr);
        if (g < a.G && !aborted) a.dcoeffs[(int64_t)g * a.K + k] = sum;
    }
    cluster_sync();
    if (threadIdx.x == 0 && aborted && a.dev_status) atomicOr(a.dev_status, SHM_DEV_TIMEOUT);
    if (warp == 1) {
        fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u) : "memory");
    }
}

// tf32 split of the basis into the adjoint's slabs: entry (k, c) of slab s = c / 16 at
// s*16*Kp + 16k + 4((c%16)/4 XOR (k/2)%4) + c%4 (16-byte chunks swizzled within each 64-byte row as
// the 64-byte swizzle places them); hi = tf32(full[k][c]), lo = tf32(full - hi); rows k >= K and
// columns c >= M4 of the last slab zero.
__global__ void k_split_basis_t(const float* __restrict__ full, int K, int Kp, int64_t M4, float* __restrict__ hiS,
                                float* __restrict__ loS)
{
    const int64_t NC = (M4 + KC - 1) / KC;
    const int64_t n = NC * Kp * KC;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t slab = e / ((int64_t)Kp * KC);
        const int r = (int)(e - slab * Kp * KC);
        const int k = r / KC, q = r % KC;            // row and position within the stored row
        const int cc = (((q >> 2) ^ ((k >> 1) & 3)) << 2) | (q & 3);  // logical column within the slab
        const int64_t c = slab * KC + cc;
        const float v = (k < K && c < M4) ? __ldg(full + (int64_t)k * M4 + c) : 0.0f;
        const float h = tf32_rna(v);
        hiS[e] = h;
        loS[e] = tf32_rna(v - h);
    }
}

// 2-D map over a row-major [rows][M4] f32 array, boxes of [box_rows][32] in the 128-byte swizzle (row
// reads without bank conflicts).
static bool make_map_c(CUtensorMap* m, const float* base, int rows, int M4, int box_rows)
{
    return encode_map_2d(m, base, M4, rows, SUB * KC, box_rows, CU_TENSOR_MAP_SWIZZLE_128B,
                         CU_TENSOR_MAP_L2_PROMOTION_L2_256B);
}

// Plan of the tensor-core adjoint for (G, K, Kp, M4) on `sms` SMs; false when it does not apply
// (the CUDA-core kernel is used then).  Glyph groups of R <= 128 rows: with at least 64 glyphs per
// SM, R is chosen so that the groups fill whole waves of the SMs (16,384 glyphs on 152 SMs: 108
// rows, 152 CTAs, where 128-row groups would leave 24 SMs idle); below that, 128-row groups whose c
// range is split over the CTAs of a cluster.
static bool plan(int G, int K, int Kp, int M4, int sms, int max_cluster, Args* out)
{
    Args a{};
    a.M4 = M4; a.G = G; a.K = K; a.Kp = Kp;
    if (Kp > KPMAX || Kp % 16 != 0) return false;
    a.R = MG;
    if ((int64_t)G >= 64LL * sms) {
        const int64_t waves = ((int64_t)G + (int64_t)MG * sms - 1) / ((int64_t)MG * sms);
        a.R = (int)(((int64_t)G + waves * sms - 1) / (waves * sms));
    }
    const int groups = (G + a.R - 1) / a.R;
    a.groups = groups;
    a.S = sms / groups;
    if (a.S > max_cluster) a.S = max_cluster;
    if (a.S < 1) a.S = 1;
    a.NC = (M4 + KC - 1) / KC;
    if (a.S > a.NC) a.S = a.NC;
    a.b_bytes = (uint32_t)Kp * KC * 4;
    a.stage_bytes = A_BYTES + SUB * 2 * a.b_bytes;
    a.nstage = (int)(STAGE_CAP / a.stage_bytes);
    if (a.nstage > MAXSTAGE) a.nstage = MAXSTAGE;
    if (a.nstage < 2) return false;
    a.nacc = 4 * a.Kp + 2 * 32 * SUB <= 512 ? 2 : 1;
    a.nslot = (512 - a.nacc * 2 * a.Kp) / (32 * SUB);
    if (a.nslot > a.nstage) a.nslot = a.nstage;
    if ((uint64_t)MG * (Kp + 1) * 4 > (uint64_t)a.nstage * a.stage_bytes) return false;  // partials fit
    *out = a;
    return true;
}

}  // namespace bwd
}  // namespace tc

// basis: [K][M] full, hi [M][Kp], lo [M][Kp], then the adjoint's slabs hiS and loS [NC][Kp][16]
cudaError_t launch_basis_split_t(int N, int L, float* basis, cudaStream_t s)
{
    const int K = (L + 1) * (L + 1), Kp = sh_kpad(L);
    const int64_t M = 4LL * 6 * (N + 2) * (N + 2);
    const int64_t slabs = (M + tc::KC - 1) / tc::KC * tc::KC * Kp;
    float* hiS = basis + (int64_t)K * M + 2 * M * Kp;
    float* loS = hiS + slabs;
    tc::bwd::k_split_basis_t<<<(unsigned)((slabs + 255) / 256 < 65535 * 8 ? (slabs + 255) / 256 : 65535 * 8), 256, 0,
                               s>>>(basis, K, Kp, M, hiS, loS);
    return cudaGetLastError();
}

// Tensor-core adjoint of the SH bake; returns cudaErrorNotSupported when its plan does not apply
// (the caller then runs the CUDA-core kernel).
cudaError_t launch_sh_build_bwd_tc(int N, int G, int L, const float* dlut, const float* basis, float* dcoeffs,
                                   int32_t* dev_status, cudaStream_t s)
{
    using namespace tc::bwd;
    const int K = (L + 1) * (L + 1), Kp = sh_kpad(L);
    const int M4 = 4 * 6 * (N + 2) * (N + 2);
    const float* hiS = basis + (int64_t)K * M4 + 2LL * M4 * Kp;
    const float* loS = hiS + ((int64_t)M4 + tc::KC - 1) / tc::KC * tc::KC * Kp;
    cudaError_t e = ensure_dynamic_smem((const void*)k_sh_gemm_bwd_tc, (int)(1024 + BAR_BYTES + STAGE_CAP));
    if (e != cudaSuccess) return e;
    // clusters of up to 16 CTAs where the device allows them, else the portable 8
    static int max_cluster = 0;
    if (max_cluster == 0) {
        max_cluster = 8;
        if (cudaFuncSetAttribute((const void*)k_sh_gemm_bwd_tc, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) ==
            cudaSuccess) {
            cudaLaunchConfig_t q = {};
            q.gridDim = dim3(16, 1, 1);
            q.blockDim = dim3(THREADS, 1, 1);
            q.dynamicSmemBytes = 1024 + BAR_BYTES + STAGE_CAP;
            cudaLaunchAttribute at;
            at.id = cudaLaunchAttributeClusterDimension;
            at.val.clusterDim.x = 16;
            at.val.clusterDim.y = 1;
            at.val.clusterDim.z = 1;
            q.attrs = &at;
            q.numAttrs = 1;
            int n = 0;
            if (cudaOccupancyMaxActiveClusters(&n, (const void*)k_sh_gemm_bwd_tc, &q) == cudaSuccess && n > 0)
                max_cluster = 16;
        }
        (void)cudaGetLastError();
    }
    Args a;
    if (!plan(G, K, Kp, M4, sm_count(), max_cluster, &a)) return cudaErrorNotSupported;
    CUtensorMap mA;
    if (((uintptr_t)hiS & 15u) != 0 || !make_map_c(&mA, dlut, G, M4, a.R))
        return cudaErrorNotSupported;
    a.hiS = hiS;
    a.loS = loS;
    a.dcoeffs = dcoeffs;
    a.dev_status = dev_status;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(a.groups * a.S), 1, 1);
    cfg.blockDim = dim3(THREADS, 1, 1);
    cfg.dynamicSmemBytes = 1024 + BAR_BYTES + (size_t)a.nstage * a.stage_bytes;
    cfg.stream = s;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = (unsigned)a.S;
    attr.val.clusterDim.y = 1;
    attr.val.clusterDim.z = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_sh_gemm_bwd_tc, mA, a);
}
}  // namespace shm
