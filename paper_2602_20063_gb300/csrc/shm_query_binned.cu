// Binned query (§3.2-§3.4) for one table larger than L2 queried in random order (the procedural
// planet of §4.10: N = 2048, 403 MB f32).
//
// Unsorted, every query's 2x2 footprint lands in a different part of the table, so each query
// pulls two or three 32 B sectors from DRAM (random sector rate, not streaming bandwidth, sets
// the pace).  Here the batch is first partitioned by the table region its footprint reads: bin =
// (face, band of cell rows), a band holding tens of MB of records.  The query kernel then walks the
// bins in order, so the few bands in flight at any moment stay resident in L2 and the table is read
// from DRAM about once per pass; everything else is coalesced streaming.
//
// The partition is local to blocks of PQ consecutive queries, which fit in shared memory: a bin is then
// one run per block (228 queries, 2.7 KB at 18 bins) instead of one contiguous range, which costs the query
// kernel nothing, and needs no global counts, no scan over the blocks and no second reading of the
// directions.
//
//   1. k_bin_partition  a block's directions in by one bulk copy, bin and slot of each, directions out
//                       in slot order by one bulk copy, and per query its slot     (12 B/q in, 14 B/q out)
//   2. k_bin_query      the query's chart, cell, footprint and Hermite steps on the runs, bin by bin, R, R_u,
//                       R_v written over the direction                              (12 B/q in, 12 B/q out)
//   3. k_bin_finish     a block's results in by one bulk copy; each query, in original order, takes
//                       (R, R_u, R_v) from its slot; the S^2 gradient and normal (§3.4) are
//                       recomputed from the original direction                      (26 B/q in, 28 B/q out)
//
// Blocks are double-buffered and CTAs persistent, so a block's copy runs under the previous block's work.
// Per query the arithmetic is that of shm_query: the chart, cell, footprint and Hermite sums run in
// step 2, the S^2 gradient and normal in step 3 on the same float32 values, so the outputs equal
// shm_query's.
//
// 2^26 random queries of the N = 2048 f32 planet: 2,112 -> 1,750 us; 2^24: partition 83 us (counting, scanning
// and scattering into globally contiguous bins 160 before) and finish 132 (192).
#include "shm_stage.cuh"
#include "shm_tc.cuh"

namespace shm {

namespace {

constexpr int PT = 512;            // threads of the partition and finish kernels
constexpr int PW = PT / 32;        // warps
constexpr int PK = 8;              // queries per thread and block; a warp takes 32 PK consecutive ones
constexpr int PQ = PT * PK;        // queries per block
constexpr uint32_t PBYTES = PQ * 12;
constexpr int MAXB = 256;          // bins at most

struct BinParams {
    int N;          // interior resolution of glyph 0
    int band_rows;  // cell rows per band
    int nb;         // bands per face
    int B;          // bins = 6 nb
    int64_t nblk;   // blocks
    int64_t Q;
    int bulk;       // directions in device memory, 16-byte aligned: blocks arrive by bulk copies
};

// Bin of a direction: face and band of the chart coordinate v (§3.2).  Only the partition uses it,
// so it may be approximate: one fast reciprocal, no exact cell arithmetic; a query near a band edge
// may land in the neighbouring band, which costs nothing but locality.  Zero / non-finite directions go to bin 0; the query kernel flags them.
__device__ __forceinline__ int bin_of(const BinParams& p, float d0, float d1, float d2)
{
    const float a0 = fabsf(d0), a1 = fabsf(d1), a2 = fabsf(d2);
    int k = 0;
    float m = a0;
    if (a1 > m) { k = 1; m = a1; }
    if (a2 > m) { k = 2; m = a2; }
    if (!(m > 0.0f) || !(m <= 3.402823466e38f)) return 0;
    const float dk = pick3(k, d0, d1, d2);
    const float dv = pick3(k == 0 ? 2 : k - 1, d0, d1, d2);  // the chart's second axis c_f
    const int f = 2 * k + (dk < 0.0f ? 1 : 0);
    const float x = fmaf(__fdividef(dv, m), 0.5f * (float)p.N, 0.5f * (float)(p.N + 1));  // v N + 1/2
    int j = (int)x;  // x >= 0 up to rounding; the clamp covers the rest
    j = min(max(j, 0), p.N);
    if (!(x == x)) j = 0;
    return f * p.nb + j / p.band_rows;
}

__device__ __forceinline__ int block_size(const BinParams& p, int64_t blk) { return (int)min((int64_t)PQ, p.Q - blk * PQ); }

// Two block buffers [PQ][3] f32 in shared memory, filled by bulk copies (full blocks, source readable by
// them) or plain loads.
struct Blocks {
    float* buf;          // 2 x [PQ][3]
    uint32_t buf_s, bar; // their shared-memory addresses; one mbarrier per buffer
    const float* src;
    bool bulk;

    __device__ __forceinline__ float* at(int b) const { return buf + b * (PQ * 3); }
    __device__ __forceinline__ bool is_bulk(const BinParams& p, int64_t blk) const { return bulk && block_size(p, blk) == PQ; }
    // thread 0
    __device__ __forceinline__ void issue(const BinParams& p, int64_t blk, int b) const
    {
        if (is_bulk(p, blk))
            stage::issue(bar + 8 * b, buf_s + b * PBYTES, reinterpret_cast<const unsigned char*>(src + blk * (PQ * 3)), PBYTES);
    }
    // every thread; then a barrier.  False if the copy did not land within the limit.
    __device__ __forceinline__ bool wait(const BinParams& p, int64_t blk, int b, uint32_t parity) const
    {
        if (is_bulk(p, blk)) return stage::bar_wait(bar + 8 * b, parity, stage::WAIT_NS);
        const int n = 3 * block_size(p, blk);
        float* dst = at(b);
        for (int i = threadIdx.x; i < n; i += PT) dst[i] = __ldcs(src + blk * (PQ * 3) + i);
        return true;
    }
};

// Thread 0's next block: after the CTA's first one, blocks are handed out by a counter, asked one block
// ahead so that its latency is hidden.  (SMs differ by up to 20 % in speed here: with a fixed share per
// CTA the slow ones set the time, and the query kernel's units in flight spread over five bins.)
struct NextBlock {
    uint32_t* taken;
    uint32_t raw = 0;
    __device__ __forceinline__ void prefetch() { raw = atomicAdd(taken, 1u); }
    __device__ __forceinline__ int64_t get() const { return (int64_t)gridDim.x + raw; }
};

// Exclusive prefix over the 512 threads' values, in thread order.
__device__ __forceinline__ int prefix_512(int v, int* wtot)
{
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    int x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) wtot[w] = x;
    __syncthreads();
    int before = 0;
    for (int k = 0; k < w; ++k) before += wtot[k];
    return before + x - v;
}

struct PartSmem {
    unsigned long long bar[2];
    int64_t next[2];
    int abort_flag;
    int wtot[PW];
    int start[MAXB];
    int cnt[PW / 2][MAXB];  // per pair of warps: queries per bin, then the pair's prefix within the bin
};
constexpr int PART_SMEM = 2 * (int)PBYTES;

// ---------------------------------------------------------------------------------- 1. partition
__global__ void __launch_bounds__(PT, 2) k_bin_partition(BinParams p, const float* __restrict__ dirs, float* sorted,
                                                         unsigned short* __restrict__ slots,
                                                         unsigned short* __restrict__ starts, uint32_t* taken, int32_t* dev_status)
{
    extern __shared__ __align__(128) unsigned char dsm[];
    __shared__ PartSmem sm;
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const Blocks in{reinterpret_cast<float*>(dsm), (uint32_t)__cvta_generic_to_shared(dsm),
                    (uint32_t)__cvta_generic_to_shared(&sm.bar[0]), dirs, p.bulk != 0};
    if (tid == 0) {
        stage::init(in.bar);
        stage::init(in.bar + 8);
        sm.abort_flag = 0;
    }
    for (int i = tid; i < PW / 2 * MAXB; i += PT) (&sm.cnt[0][0])[i] = 0;
    __syncthreads();
    uint32_t phase = 0;
    int b = 0;
    NextBlock take{taken};
    if (tid == 0) {
        in.issue(p, blockIdx.x, 0);
        take.prefetch();
    }
    for (int64_t blk = blockIdx.x, next; blk < p.nblk; blk = next, b ^= 1) {
        const int n = block_size(p, blk);
        if (tid == 0) {
            next = take.get();
            sm.next[b] = next;
            if (next < p.nblk) {
                tc::bulk_wait_read_all();  // the store that used the other buffer has read it
                in.issue(p, next, b ^ 1);
                take.prefetch();
            }
        }
        const bool bulk = in.is_bulk(p, blk);
        if (!in.wait(p, blk, b, (phase >> b) & 1)) sm.abort_flag = 1;
        __syncthreads();
        next = sm.next[b];
        if (sm.abort_flag) {
            if (tid == 0) {
                if (dev_status) atomicOr(dev_status, SHM_DEV_TIMEOUT);
                if (bulk) stage::bar_wait(in.bar + 8 * b, (phase >> b) & 1, stage::DRAIN_NS);
                if (next < p.nblk && in.is_bulk(p, next))
                    stage::bar_wait(in.bar + 8 * (b ^ 1), (phase >> (b ^ 1)) & 1, stage::DRAIN_NS);
            }
            break;
        }
        if (bulk) phase ^= 1u << b;
        float* buf = in.at(b);
        float d[PK][3];
        int br[PK];  // bin and rank within (warp, bin)
#pragma unroll
        for (int k = 0; k < PK; ++k) {
            const int i = w * (32 * PK) + k * 32 + lane;
            int bin = -1;
            if (i < n) {
                d[k][0] = buf[3 * i]; d[k][1] = buf[3 * i + 1]; d[k][2] = buf[3 * i + 2];
                bin = bin_of(p, d[k][0], d[k][1], d[k][2]);
            }
            const int r = bin >= 0 ? atomicAdd(&sm.cnt[w / 2][bin], 1) : 0;
            br[k] = bin < 0 ? -1 : (bin << 16 | r);
        }
        __syncthreads();
        int total = 0;
        if (tid < p.B)
            for (int ww = 0; ww < PW / 2; ++ww) {
                const int x = sm.cnt[ww][tid];
                sm.cnt[ww][tid] = total;
                total += x;
            }
        const int at = prefix_512(total, sm.wtot);
        if (tid < p.B) {
            sm.start[tid] = at;
            starts[blk * p.B + tid] = (unsigned short)at;
        }
        __syncthreads();  // also: every direction of the block is in registers
#pragma unroll
        for (int k = 0; k < PK; ++k) {
            if (br[k] < 0) continue;
            const int i = w * (32 * PK) + k * 32 + lane, bin = br[k] >> 16;
            const int e = sm.start[bin] + sm.cnt[w / 2][bin] + (br[k] & 0xffff);
            buf[3 * e] = d[k][0]; buf[3 * e + 1] = d[k][1]; buf[3 * e + 2] = d[k][2];
            __stcs(slots + blk * PQ + i, (unsigned short)e);
        }
        if (n == PQ) asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncthreads();
        if (n == PQ) {
            if (tid == 0) {
                asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(sorted + blk * (PQ * 3)),
                             "r"(in.buf_s + b * PBYTES), "r"(PBYTES)
                             : "memory");
                tc::bulk_commit();
            }
        } else {
            for (int i = tid; i < 3 * n; i += PT) sorted[blk * (PQ * 3) + i] = buf[i];
        }
        for (int i = tid; i < PW / 2 * MAXB; i += PT) (&sm.cnt[0][0])[i] = 0;
        // the next iteration's barrier orders these writes before the next ranking
    }
    if (tid == 0) tc::bulk_wait_all();
}

// ---------------------------------------------------------------------------------- 2. query
// The query of §3.2-§3.3 on the runs, keeping R, R_u, R_v only (the S^2 gradient and normal follow in
// step 3).  Same device functions as shm_query, hence the same values.  Work unit = (bin, block, piece): a
// warp's units follow each other bin by bin, so the bands in flight at any time are the few that the
// resident warps' units cover; `pieces` cuts runs so that small batches still fill the SMs.  Units are
// handed out by a counter: with a fixed share per warp, SMs of different speed drifted apart until five
// bins were in flight and the table came from DRAM eight times instead of 2.5 (2^26 queries, 1,998 us).
// A warp keeps 64 queries in flight and loads the next 64 directions under their footprints; directions and
// results cross a 96-float buffer so that every global access is 128 contiguous bytes.  Bound: requests
// from L1 to L2, about three per footprint; three CTAs per SM keep the bins in flight fewer than four.
constexpr int QB = 256, QILP = 2;
constexpr int SHORT_RUN = 100;  // queries of a block's mean run

template <int DT, int LAYOUT>
__global__ void __launch_bounds__(QB, 3) k_bin_query(BinParams p, LutView L, const unsigned short* __restrict__ starts,
                                                     int pieces, int grab, float* sorted, uint32_t* taken,
                                                     int32_t* __restrict__ dev_status)
{
    __shared__ float tr[QB / 32][QILP][96];
    const GlyphRef G = glyph_ref(L, 0);
    const float qnan = __int_as_float(0x7fc00000);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    uint32_t status = 0;
    const uint32_t units = (uint32_t)(p.nblk * p.B * pieces), nblk = (uint32_t)p.nblk;
    // first slot and end of a unit's queries (clamped: an aborted partition leaves them undefined)
    const auto bounds = [&](uint32_t u, int64_t& base, int& s0, int& s1) {
        base = 0;
        s0 = s1 = 0;
        if (u >= units) return;
        const uint32_t v = u / (uint32_t)pieces;
        const int piece = (int)(u - v * pieces), bin = (int)(v / nblk);
        const int64_t blk = v - bin * nblk;
        const int n = block_size(p, blk);
        const int a = min((int)__ldg(starts + blk * p.B + bin), n);
        const int e = bin + 1 < p.B ? min(max((int)__ldg(starts + blk * p.B + bin + 1), a), n) : n;
        base = blk * PQ;
        s0 = a + (e - a) * piece / pieces;
        s1 = a + (e - a) * (piece + 1) / pieces;
    };
    // the iteration at hand: queries [r, s1) of the run at `run`, at most 64; the next one's directions load
    // under its footprints
    // units u .. and their successors nu .. (bounds loaded a unit ahead), taken `grab` at a time from the counter
    // (asked a batch ahead), so that the units in flight stay within a fraction of a bin
    uint32_t u = (blockIdx.x * (QB / 32) + w) * grab, nu = u, left = grab - 1, raw = 0;  // left: rest of nu's batch
    const uint32_t first = gridDim.x * (QB / 32) * grab;
    if (lane == 0) raw = atomicAdd(taken, (uint32_t)grab);
    const auto advance = [&] {
        if (left > 0) {
            ++nu;
            --left;
        } else {
            nu = first + __shfl_sync(0xffffffffu, raw, 0);
            left = grab - 1;
            if (lane == 0 && nu < units) raw = atomicAdd(taken, (uint32_t)grab);
        }
    };
    int64_t base, nbase;
    int r, s1, n0, n1;
    float* run = sorted;
    const auto settle = [&] {  // (base, r, s1) of unit u or of the next one that holds queries
        while (r >= s1 && u < units) {
            u = nu;
            base = nbase; r = n0; s1 = n1;
            advance();
            bounds(nu, nbase, n0, n1);
        }
        run = sorted + 3 * base;
    };
    float f[QILP][3];
    const auto load = [&] {
#pragma unroll
        for (int v = 0; v < QILP; ++v)
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const int i = v * 96 + c * 32 + lane;
                f[v][c] = i < 3 * (s1 - r) ? __ldcs(run + 3 * r + i) : 0.0f;
            }
    };
    bounds(u, base, r, s1);
    advance();
    bounds(nu, nbase, n0, n1);
    settle();
    load();
    while (r < s1) {
        float* const out = run + 3 * r;
        const int n = s1 - r;
#pragma unroll
        for (int v = 0; v < QILP; ++v)
#pragma unroll
            for (int c = 0; c < 3; ++c) tr[w][v][c * 32 + lane] = f[v][c];
        __syncwarp();
        float d[QILP][3];
#pragma unroll
        for (int v = 0; v < QILP; ++v)
#pragma unroll
            for (int c = 0; c < 3; ++c) d[v][c] = tr[w][v][3 * lane + c];
        __syncwarp();
        r += 32 * QILP;
        settle();
        load();
#pragma unroll
        for (int v = 0; v < QILP; ++v) {
            QueryResult o;
            Chart c;
            o.R = o.Ru = o.Rv = qnan;
            if (v * 32 + lane < n && !query_one<DT, LAYOUT>(L, G, d[v][0], d[v][1], d[v][2], o, c)) {
                o.R = o.Ru = o.Rv = qnan;
                status |= SHM_DEV_NONFINITE;
            }
            tr[w][v][3 * lane] = o.R; tr[w][v][3 * lane + 1] = o.Ru; tr[w][v][3 * lane + 2] = o.Rv;
        }
        __syncwarp();
#pragma unroll
        for (int v = 0; v < QILP; ++v)
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const int i = v * 96 + c * 32 + lane;
                if (i < 3 * n) __stcs(out + i, tr[w][v][c * 32 + lane]);
            }
        __syncwarp();
    }
    report_status(dev_status, status);
}

// ---------------------------------------------------------------------------------- 3. finish
// Results, directions and slots of a block arrive together (104 KB) while the block before it is finished;
// one CTA of 1,024 threads per SM, four queries per thread and block.
constexpr int FT = 1024, FW = FT / 32, FK = PQ / FT;
constexpr uint32_t FBYTES = 2 * PBYTES + 2 * PQ;  // results, directions, slots
constexpr int FINISH_SMEM = 2 * (int)FBYTES;

// VEC: grad and normal 16-byte aligned: a warp's 384 B of gradients and normals cross a per-warp buffer as
// 24 16-byte stores.
template <bool VEC>
__global__ void __launch_bounds__(FT, 1) k_bin_finish(BinParams p, const float* __restrict__ dirs, const float* sorted,
                                                      const unsigned short* slots, float* __restrict__ R,
                                                      float* __restrict__ grad, float* __restrict__ normal,
                                                      float* __restrict__ chart, uint32_t* taken, int32_t* __restrict__ dev_status)
{
    extern __shared__ __align__(128) unsigned char dsm[];
    __shared__ unsigned long long s_bar[2];
    __shared__ int64_t s_next[2];
    __shared__ int s_abort;
    __shared__ __align__(16) float s_tr[FW][96];
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const float qnan = __int_as_float(0x7fc00000);
    const uint32_t bar = (uint32_t)__cvta_generic_to_shared(&s_bar[0]), dsm_s = (uint32_t)__cvta_generic_to_shared(dsm);
    if (tid == 0) {
        stage::init(bar);
        stage::init(bar + 8);
        s_abort = 0;
    }
    __syncthreads();
    float* tr = s_tr[w];
    const auto store3 = [&](float* out, int64_t q0, bool full, bool live, const Vec3& v) {
        if (VEC && full) {
            tr[3 * lane] = v.x; tr[3 * lane + 1] = v.y; tr[3 * lane + 2] = v.z;
            __syncwarp();
            if (lane < 24) __stcs(reinterpret_cast<float4*>(out + 3 * q0) + lane, reinterpret_cast<const float4*>(tr)[lane]);
            __syncwarp();
        } else if (live) {
            const int64_t q = q0 + lane;
            __stcs(out + 3 * q, v.x); __stcs(out + 3 * q + 1, v.y); __stcs(out + 3 * q + 2, v.z);
        }
    };
    const auto is_bulk = [&](int64_t blk) { return p.bulk && block_size(p, blk) == PQ; };
    const auto issue = [&](int64_t blk, int b) {  // thread 0
        if (!is_bulk(blk)) return;
        const uint32_t dst = dsm_s + b * FBYTES;
        stage::expect(bar + 8 * b, FBYTES);
        stage::copy(bar + 8 * b, dst, sorted + blk * (PQ * 3), PBYTES);
        stage::copy(bar + 8 * b, dst + PBYTES, dirs + blk * (PQ * 3), PBYTES);
        stage::copy(bar + 8 * b, dst + 2 * PBYTES, slots + blk * PQ, 2 * PQ);
    };
    uint32_t phase = 0;
    int b = 0;
    NextBlock take{taken};
    if (tid == 0) {
        issue(blockIdx.x, 0);
        take.prefetch();
    }
    for (int64_t blk = blockIdx.x, next; blk < p.nblk; blk = next, b ^= 1) {
        const int n = block_size(p, blk);
        if (tid == 0) {
            next = take.get();
            s_next[b] = next;
            // every read of the other buffer ended before the last iteration's final barrier
            if (next < p.nblk) {
                issue(next, b ^ 1);
                take.prefetch();
            }
        }
        const bool bulk = is_bulk(blk);
        float* res = reinterpret_cast<float*>(dsm + b * FBYTES);
        float* dir = res + 3 * PQ;
        unsigned short* slot = reinterpret_cast<unsigned short*>(dir + 3 * PQ);
        if (bulk) {
            if (!stage::bar_wait(bar + 8 * b, (phase >> b) & 1, stage::WAIT_NS)) s_abort = 1;
        } else {
            for (int i = tid; i < 3 * n; i += FT) {
                res[i] = __ldcs(sorted + blk * (PQ * 3) + i);
                dir[i] = __ldcs(dirs + blk * (PQ * 3) + i);
            }
            for (int i = tid; i < n; i += FT) slot[i] = __ldcs(slots + blk * PQ + i);
        }
        __syncthreads();
        next = s_next[b];
        if (s_abort) {
            if (tid == 0) {
                if (dev_status) atomicOr(dev_status, SHM_DEV_TIMEOUT);
                if (bulk) stage::bar_wait(bar + 8 * b, (phase >> b) & 1, stage::DRAIN_NS);
                if (next < p.nblk && is_bulk(next)) stage::bar_wait(bar + 8 * (b ^ 1), (phase >> (b ^ 1)) & 1, stage::DRAIN_NS);
            }
            break;
        }
        if (bulk) phase ^= 1u << b;
#pragma unroll
        for (int k = 0; k < FK; ++k) {
            const int i0 = (w * FK + k) * 32, i = i0 + lane;
            const int64_t q0 = blk * PQ + i0, q = q0 + lane;
            const bool full = i0 + 32 <= n, live = i < n;
            if (i0 >= n) break;  // warp-uniform
            float d0 = 0.0f, d1 = 0.0f, d2 = 0.0f, v0 = qnan, v1 = qnan, v2 = qnan;
            if (live) {
                const int e = min((int)slot[i], n - 1);
                v0 = res[3 * e]; v1 = res[3 * e + 1]; v2 = res[3 * e + 2];
                d0 = dir[3 * i]; d1 = dir[3 * i + 1]; d2 = dir[3 * i + 2];
            }
            Chart c;
            Vec3 g{qnan, qnan, qnan}, nn{qnan, qnan, qnan};
            if (chart_of(d0, d1, d2, c)) {
                g = s2_gradient(c, v1, v2);
                nn = surface_normal(d0, d1, d2, v0, g);
            }
            if (R && live) __stcs(R + q, v0);
            if (grad) store3(grad, q0, full, live, g);
            if (normal) store3(normal, q0, full, live, nn);
            if (chart && live) { __stcs(chart + 2 * q, v1); __stcs(chart + 2 * q + 1, v2); }
        }
        __syncthreads();  // every read of this buffer is done before the copy after next lands in it
    }
}

template <int DT, int LAYOUT>
cudaError_t launch_bin_query(const BinParams& p, const LutView& L, const unsigned short* starts, float* sorted,
                             uint32_t* taken, int32_t* dev_status, cudaStream_t s)
{
    static int resident = 0;
    if (resident == 0) {
        int r = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&r, k_bin_query<DT, LAYOUT>, QB, 0) != cudaSuccess || r < 1)
            r = 1;
        resident = r;
    }
    const int64_t cap = (int64_t)sm_count() * resident, warps = cap * (QB / 32), runs = p.nblk * p.B;
    if (runs > 0x40000000) return cudaErrorInvalidConfiguration;  // Q > 10^10 at 252 bins
    // at least four units per resident warp, pieces of at least 32 queries of a block's mean run
    int64_t pieces = (4 * warps + runs - 1) / runs;
    const int64_t most = PQ / (32 * (int64_t)p.B);
    if (pieces > most) pieces = most;
    if (pieces < 1) pieces = 1;
    // One unit at a time keeps the units in flight within the fewest bins; two halve the counter's load.  They pay
    // where they still cover less than half a bin (2^26 queries: 1,751 against 1,788 us; 2^24: 548 against 486), and where
    // runs are short: one address takes about 500 additions per microsecond, which bound 54 bins of 76 queries a block
    // (f32 cells of N = 2048, 2^22 / 2^24 / 2^25 queries: 221 / 727 / 1,055 us one at a time, 171 / 538 / 986 two).
    const int grab = 4 * warps <= p.nblk * pieces || PQ / p.B < SHORT_RUN ? 2 : 1;
    int64_t blocks = (runs * pieces + QB / 32 - 1) / (QB / 32);
    if (blocks > cap) blocks = cap;
    k_bin_query<DT, LAYOUT><<<(unsigned)blocks, QB, 0, s>>>(p, L, starts, (int)pieces, grab, sorted, taken, dev_status);
    return cudaGetLastError();
}

cudaError_t launch_bin_query_any(const BinParams& p, const LutView& L, const unsigned short* starts, float* sorted,
                                 uint32_t* taken, int32_t* dev_status, cudaStream_t s)
{
    if (L.layout == SHM_LAYOUT_TEXEL) {
        if (L.dtype == SHM_F32) return launch_bin_query<SHM_F32, SHM_LAYOUT_TEXEL>(p, L, starts, sorted, taken, dev_status, s);
        if (L.dtype == SHM_F16) return launch_bin_query<SHM_F16, SHM_LAYOUT_TEXEL>(p, L, starts, sorted, taken, dev_status, s);
        return launch_bin_query<SHM_BF16, SHM_LAYOUT_TEXEL>(p, L, starts, sorted, taken, dev_status, s);
    }
    if (L.dtype == SHM_F32) return launch_bin_query<SHM_F32, SHM_LAYOUT_CELL>(p, L, starts, sorted, taken, dev_status, s);
    if (L.dtype == SHM_F16) return launch_bin_query<SHM_F16, SHM_LAYOUT_CELL>(p, L, starts, sorted, taken, dev_status, s);
    return launch_bin_query<SHM_BF16, SHM_LAYOUT_CELL>(p, L, starts, sorted, taken, dev_status, s);
}

constexpr int64_t align256(int64_t x) { return (x + 255) & ~(int64_t)255; }

struct BinLayout {
    BinParams p;
    int64_t o_sorted, o_slot, o_start, o_taken, bytes;
};

// Bands of cell rows holding about band_bytes of records each (at least one row, at most 42 bands
// per face so that the 6 faces' bins fit in a byte).
bool binned_plan(const LutView& L, int64_t Q, int64_t band_bytes, BinLayout* out)
{
    if (L.N_uniform <= 0 || Q < 0) return false;
    const int N = L.N_uniform;
    const int64_t rec = (L.layout == SHM_LAYOUT_CELL ? 4 : 1) * (L.dtype == SHM_F32 ? 16 : 8);
    const int64_t row = (int64_t)(L.layout == SHM_LAYOUT_CELL ? N + 1 : N + 2) * rec;
    if (band_bytes <= 0) band_bytes = BINNED_DEFAULT_BAND_BYTES;
    int64_t rows = band_bytes / row;
    if (rows < 1) rows = 1;
    if (rows > N + 1) rows = N + 1;
    int64_t nb = (N + 1 + rows - 1) / rows;
    if (nb > MAXB / 6) {
        nb = MAXB / 6;
        rows = (N + 1 + nb - 1) / nb;
        nb = (N + 1 + rows - 1) / rows;
    }
    BinLayout z;
    z.p.N = N;
    z.p.band_rows = (int)rows;
    z.p.nb = (int)nb;
    z.p.B = (int)(6 * nb);
    z.p.nblk = (Q + PQ - 1) / PQ;
    z.p.Q = Q;
    z.p.bulk = 0;
    // partitioned directions (then results), slots, run starts: 14 B per query
    int64_t o = 0;
    z.o_sorted = o; o = align256(o + 12 * Q);
    z.o_slot = o;   o = align256(o + 2 * Q);
    z.o_start = o;  o = align256(o + 2 * z.p.B * z.p.nblk);
    z.o_taken = o;  // three counters
    z.bytes = align256(o + 3 * (int64_t)sizeof(uint32_t));
    *out = z;
    return true;
}

}  // namespace

int64_t binned_workspace_bytes(const LutView& L, int64_t Q, int64_t band_bytes)
{
    BinLayout z;
    if (!binned_plan(L, Q, band_bytes, &z)) return -1;
    return z.bytes;
}

int binned_bins(const LutView& L, int64_t band_bytes, int* band_rows)
{
    BinLayout z;
    if (!binned_plan(L, 0, band_bytes, &z)) return -1;
    if (band_rows) *band_rows = z.p.band_rows;
    return z.p.B;
}

cudaError_t launch_query_binned(const QueryArgs& a, int64_t band_bytes, void* ws, size_t ws_bytes, cudaStream_t s)
{
    BinLayout z;
    if (!binned_plan(a.L, a.Q, band_bytes, &z) || (int64_t)ws_bytes < z.bytes || !ws) return cudaErrorInvalidValue;
    if (a.Q == 0) return cudaSuccess;
    // bulk copies read device memory at 16-byte aligned addresses; other directions use plain loads
    cudaPointerAttributes at;
    z.p.bulk = 0;
    const auto al16 = [](const void* q) { return ((uintptr_t)q & 15u) == 0; };
    if (al16(a.dirs) && cudaPointerGetAttributes(&at, a.dirs) == cudaSuccess && at.type == cudaMemoryTypeDevice)
        z.p.bulk = 1;
    (void)cudaGetLastError();
    unsigned char* w = static_cast<unsigned char*>(ws);
    float* sorted = reinterpret_cast<float*>(w + z.o_sorted);
    unsigned short* slots = reinterpret_cast<unsigned short*>(w + z.o_slot);
    unsigned short* starts = reinterpret_cast<unsigned short*>(w + z.o_start);
    uint32_t* taken = reinterpret_cast<uint32_t*>(w + z.o_taken);  // blocks / units handed out by each kernel
    const bool vec = al16(a.grad) && al16(a.normal);
    const void* fin = vec ? (const void*)k_bin_finish<true> : (const void*)k_bin_finish<false>;
    cudaError_t e = ensure_dynamic_smem((const void*)k_bin_partition, PART_SMEM);
    if (e == cudaSuccess) e = ensure_dynamic_smem(fin, FINISH_SMEM);
    if (e != cudaSuccess) return e;
    const int64_t sms = sm_count();
    const unsigned grid = (unsigned)(z.p.nblk < 2 * sms ? z.p.nblk : 2 * sms);
    const unsigned fgrid = (unsigned)(z.p.nblk < sms ? z.p.nblk : sms);
    e = cudaMemsetAsync(taken, 0, 3 * sizeof(uint32_t), s);
    if (e != cudaSuccess) return e;
    k_bin_partition<<<grid, PT, PART_SMEM, s>>>(z.p, a.dirs, sorted, slots, starts, taken, a.dev_status);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    e = launch_bin_query_any(z.p, a.L, starts, sorted, taken + 1, a.dev_status, s);
    if (e != cudaSuccess) return e;
    if (vec)
        k_bin_finish<true><<<fgrid, FT, FINISH_SMEM, s>>>(z.p, a.dirs, sorted, slots, a.R, a.grad, a.normal, a.chart, taken + 2,
                                                           a.dev_status);
    else
        k_bin_finish<false><<<fgrid, FT, FINISH_SMEM, s>>>(z.p, a.dirs, sorted, slots, a.R, a.grad, a.normal, a.chart, taken + 2,
                                                           a.dev_status);
    return cudaGetLastError();
}

}  // namespace shm
