// Reverse pass of the query with atomic accumulation (the per-query math is in shm_bwd.cuh): every
// corner record's float4 of gradients is added with one vector reduction (red.global.add.v4.f32),
// two lanes of a warp adding the two adjacent records of a footprint row in the same instruction,
// so the summation order, hence the last bits of dL/dtable, depends on scheduling.
// Per-glyph segments on small uniform tables take k_query_bwd_staged: the table is staged in shared
// memory as in the forward.  (Accumulating each glyph's gradients in a shared-memory slab with
// shared float atomics instead measured 4.8 ms against 3.3 ms for the global vector atomics on the
// 2^26-query glyph field: sixteen scattered 4-byte shared atomics per query cost more than four
// 16-byte L2 ones.)
#include "shm_bwd.cuh"
#include "shm_stage.cuh"

namespace shm {

// One query's cell and upstream values, kept for the paired reductions after its reverse pass.
struct CaptureEmit {
    int64_t base = 0;  // the glyph's first record in the gradient table
    int P = 0;         // the glyph's padded table width
    int64_t rec = -1;  // record of corner (0,0) in the gradient table; -1: no contribution
    float s = 0.0f, t = 0.0f, g_r = 0.0f, g_rs = 0.0f, g_rt = 0.0f;
    __device__ __forceinline__ void operator()(int64_t r, float s_, float t_, float gr, float grs, float grt)
    {
        rec = base + r;
        s = s_;
        t = t_;
        g_r = gr;
        g_rs = grs;
        g_rt = grt;
    }
};

__device__ __forceinline__ float4 shfl_xor_f4(float4 v, int m)
{
    return make_float4(__shfl_xor_sync(0xffffffffu, v.x, m), __shfl_xor_sync(0xffffffffu, v.y, m),
                       __shfl_xor_sync(0xffffffffu, v.z, m), __shfl_xor_sync(0xffffffffu, v.w, m));
}

// The corner reductions of a warp's queries (every lane calls it), in pairs of lanes: lanes 2k and
// 2k + 1 add the two adjacent records (i, j), (i+1, j) of one query's footprint row in the same
// instruction, 32 contiguous bytes, so each vector-reduction instruction reaches the L2 as about 16
// requests instead of 32 scattered ones (glyph field: reverse pass 2.23 -> 2.01 ms).  Four
// instructions per lane as before; the partner's weights and cell come by shuffles.
__device__ __forceinline__ void paired_reds(float4* dl, const CaptureEmit& e, int lane)
{
    float4 w[4];
    if (e.rec >= 0) {
        corner_weights(e.s, e.t, e.g_r, e.g_rs, e.g_rt, w);
    } else {
#pragma unroll
        for (int m = 0; m < 4; ++m) w[m] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    const bool even = (lane & 1) == 0;
    const int64_t prec = ((int64_t)__shfl_xor_sync(0xffffffffu, (int)(e.rec >> 32), 1) << 32) |
                         (uint32_t)__shfl_xor_sync(0xffffffffu, (int)(uint32_t)e.rec, 1);
    const int pP = __shfl_xor_sync(0xffffffffu, e.P, 1);
    // each lane passes the partner the weights the partner writes: even lanes their (i+1) records,
    // odd lanes their (i) records, for rows j and j + 1
    const float4 r0 = shfl_xor_f4(even ? w[1] : w[0], 1);
    const float4 r1 = shfl_xor_f4(even ? w[3] : w[2], 1);
    const int64_t qa = even ? e.rec : prec, qb = even ? prec : e.rec;  // the even and the odd lane's cells
    const int Pa = even ? e.P : pP, Pb = even ? pP : e.P;
    const int da = even ? 0 : 1;
    if (qa >= 0) {
        atomicAdd(dl + qa + da, even ? w[0] : r0);
        atomicAdd(dl + qa + Pa + da, even ? w[2] : r1);
    }
    if (qb >= 0) {
        atomicAdd(dl + qb + da, even ? r0 : w[1]);
        atomicAdd(dl + qb + Pb + da, even ? r1 : w[3]);
    }
}

// Sum of a CTA's per-thread losses, added once: with an addition per warp (9,728 on the fit workload) the
// rounding of the growing float32 sum alone reached 1e-6 of it and varied from run to run; with one per
// CTA (152) it stays near 2e-7.
__device__ __forceinline__ void add_loss(float* loss, float v)
{
    __shared__ float s_loss[32];
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) s_loss[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x < 32) {
        v = threadIdx.x < blockDim.x / 32 ? s_loss[threadIdx.x] : 0.0f;
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (threadIdx.x == 0) atomicAdd(loss, v);
    }
}

// CTA of the per-query pass, and the most consecutive rounds of 32 queries per warp.  The fused fit takes CTAs of
// 1,024 threads, whose warps' queries lie side by side (4,096 of them), so a glyph's records are reused in L1, while
// all CTAs together still work on few glyphs, whose tables and gradients (836 KB each at N = 64) must stay in L2:
// fit workload 502 -> 470 us; CTAs of 256 threads 488; a contiguous range of glyphs per CTA 770 to 1,800 (L2
// thrashes).  Upstream gradients bring 28 B more per query, and there the large CTAs' common pace loses: 256 threads
// (four CTAs per SM) against 1,024 take 38.8 / 42.7 us for 10^6 queries of one glyph of N = 64, 233.8 / 239.8 for 4,096
// each of 1,000, 68.4 / 73.7 for 2 M queries of 100 glyphs of N = 32 by ids.
template <bool FIT>
struct BwdCta {
    static constexpr int threads = FIT ? 1024 : 256;
    static constexpr int resident = FIT ? 1 : 4;
    static constexpr int per_sm = FIT ? 1 : 8;  // CTAs launched per SM at most
};
constexpr int BROUNDS = 4;

template <int DT, int LAYOUT, bool FIT>
__global__ void __launch_bounds__(BwdCta<FIT>::threads, BwdCta<FIT>::resident) k_query_bwd(BackwardArgs a, int rounds)
{
    constexpr int BBLOCK = BwdCta<FIT>::threads;
    float loss_acc = 0.0f;
    const int lane = threadIdx.x & 31;
    const int64_t chunk = 32 * rounds;
    const int64_t warp0 = ((int64_t)blockIdx.x * BBLOCK + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * BBLOCK) >> 5;
    const int G = a.L.n_glyphs;
    uint32_t status = 0;
    const float qnan = __int_as_float(0x7fc00000);

    for (int64_t c0 = warp0 * chunk; c0 < a.Q; c0 += nwarps * chunk) {
        int g = 0;
        if (a.seg) {
            g = (c0 < __ldg(a.seg)) ? -1 : seg_find_warp(a.seg, G, c0);
        }
#pragma unroll 1
        for (int it = 0; it < rounds; ++it) {
            const int64_t q = c0 + it * 32 + lane;
            if (c0 + it * 32 >= a.Q) break;  // warp-uniform: the paired reductions need every lane
            CaptureEmit sink;
            if (q < a.Q) {
                int gq = 0;
                if (a.glyph) {
                    gq = __ldg(a.glyph + q);
                } else if (a.seg) {
                    if (g < 0 && q >= __ldg(a.seg)) g = 0;
                    while (g >= 0 && g < G && q >= __ldg(a.seg + g + 1)) ++g;
                    gq = g;
                }
                float3 dd = make_float3(qnan, qnan, qnan);
                const float d0 = __ldcs(a.dirs + 3 * q), d1 = __ldcs(a.dirs + 3 * q + 1), d2 = __ldcs(a.dirs + 3 * q + 2);
                Chart c;
                bool ok = (gq >= 0 && gq < G);
                if (!ok) status |= SHM_DEV_BOUNDS;
                if (ok && !chart_of(d0, d1, d2, c)) { ok = false; status |= SHM_DEV_NONFINITE; }
                if (ok) {
                    const GlyphRef Gr = glyph_ref(a.L, gq);
                    sink.base = glyph_ref(a.D, gq).base;
                    sink.P = Gr.N + 2;
                    auto fetch = [&a, &Gr](int f, int i, int j) { return fetch_corners<DT, LAYOUT>(a.L.data, Gr, f, i, j); };
                    if constexpr (FIT) bwd_query<FIT>(a, PreFit(a, q), Gr, c, d0, d1, d2, fetch, sink, dd, loss_acc);
                    else bwd_query<FIT>(a, GlobalUp{a, q}, Gr, c, d0, d1, d2, fetch, sink, dd, loss_acc);
                }
                if (a.ddirs) {
                    __stcs(a.ddirs + 3 * q, dd.x);
                    __stcs(a.ddirs + 3 * q + 1, dd.y);
                    __stcs(a.ddirs + 3 * q + 2, dd.z);
                }
            }
            paired_reds(reinterpret_cast<float4*>(a.dlut), sink, lane);
        }
    }
    if (FIT && a.loss) add_loss(a.loss, loss_acc);
    report_status(a.dev_status, status);
}

// Per-glyph segments on tables that fit in shared memory: a CTA takes one unit of the path through
// glyphs and queries (shm_stage.cuh), stages each glyph's table (as the forward does) and answers the
// footprint reads from it; the gradient atomics of a glyph then come from one SM, or the few that share
// it, within a short window, so its dL/dtable slab stays in L2 while it is hit.
//
// SET: the gradient table is written instead of accumulated into.  A glyph that lies wholly inside a unit
// has its slab zeroed by that CTA while its table copy is in flight, so the zeros and the sums meet in L2
// and DRAM sees one write of the slab instead of a fill, a read and a write; the glyphs that a unit
// boundary cuts are zeroed first by k_zero_cut.
constexpr int SBB = 512;
constexpr int WINDOWS_PER_SM = 2;
constexpr uint32_t WHOLE_BYTES = 80000;
constexpr int BWD_PATH_BYTES = 64;  // table bytes per unit of path cost: the copy and the slab's traffic in queries

__device__ __forceinline__ void zero_slab(float4* slab, int records, int tid, int threads)
{
    for (int r = tid; r < records; r += threads) slab[r] = make_float4(0.f, 0.f, 0.f, 0.f);
}

// Block b zeroes the slab of the glyph that the boundary between units b and b + 1 cuts, unless an
// earlier boundary cuts it too.
__global__ void __launch_bounds__(1024) k_zero_cut(const __grid_constant__ stage::Path path, float4* dlut, int records)
{
    __shared__ stage::Pos s_cut[2];
    const int warp = threadIdx.x >> 5;
    if (warp < 2) {
        const stage::Pos p = path.at(blockIdx.x + warp);
        if ((threadIdx.x & 31) == 0) s_cut[warp] = p;
    }
    __syncthreads();
    const stage::Pos before = s_cut[0], cut = s_cut[1];
    if (cut.g >= path.G) return;
    const int64_t s0 = stage::seg_at(path.seg, path.Q, cut.g);
    if (cut.q <= s0 || (before.g == cut.g && before.q > s0)) return;
    zero_slab(dlut + (int64_t)cut.g * records, records, threadIdx.x, 1024);
}

// One CTA per glyph, with a bound on a CTA's share of a long segment: the queries are covered by windows of
// `size` of them, each with a CTA of its own after the glyphs'.  A glyph's CTA takes its segment through the end
// of the window after the one it starts in; what lies beyond goes window by window to the windows' CTAs.  A segment
// of at most `size` queries is never cut, and none holds a CTA for more than two windows.
struct Windows {
    int64_t size;
    int n;
    uint64_t inv;  // 2^64 / size, rounded up: s / size = umulhi(s, inv) for s size < 2^64
    Windows(int64_t Q, int n_) : size(n_ > 0 ? (Q + n_ - 1) / n_ + 1 : 2), n(n_), inv(UINT64_MAX / (uint64_t)size + 1) {}
    __device__ __forceinline__ int64_t own_end(int64_t s0) const { return (int64_t)(__umul64hi((uint64_t)s0, inv) + 2) * size; }
    // The long segment that goes on in window b (a whole warp calls it); G: none.
    __device__ __forceinline__ int glyph(const int64_t* seg, int G, int64_t Q, int b) const
    {
        const int64_t lo = b * size;
        if (lo >= Q || lo < __ldg(seg)) return G;
        const int g = seg_find_warp(seg, G, lo);
        return g < G && own_end(stage::seg_at(seg, Q, g)) <= lo ? g : G;
    }
};

// Block b zeroes the slab of the glyph whose first part beyond its own CTA's share is in window b.
__global__ void __launch_bounds__(256) k_zero_long(const int64_t* seg, int G, int64_t Q, Windows win, float4* dlut, int records)
{
    __shared__ int s_g;
    if (threadIdx.x < 32) {
        const int g = win.glyph(seg, G, Q, blockIdx.x);
        const bool first = g < G && win.own_end(stage::seg_at(seg, Q, g)) == blockIdx.x * win.size;
        if (threadIdx.x == 0) s_g = first ? g : -1;
    }
    __syncthreads();
    if (s_g >= 0) zero_slab(dlut + (int64_t)s_g * records, records, threadIdx.x, 256);
}

template <int DT, bool FIT, bool SET>
__global__ void __launch_bounds__(SBB, 2) k_query_bwd_staged(BackwardArgs a, uint32_t table_bytes, int nbuf,
                                                             const __grid_constant__ stage::Path path, Windows win)
{
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ int s_abort;
    __shared__ stage::Pos s_unit[2];
    const uint32_t bar = (uint32_t)__cvta_generic_to_shared(smem);
    const unsigned char* tables = smem + stage::TABLE_OFFSET;
    const uint32_t table_s = bar + stage::TABLE_OFFSET;
    const int tid = threadIdx.x;
    const int G = a.L.n_glyphs, N = a.L.N_uniform, P = N + 2;
    const int records = 6 * P * P;
    using Up = std::conditional_t<FIT, PreFit, PreUp>;
    uint32_t status = 0;
    float loss_acc = 0.0f;
    const float qnan = __int_as_float(0x7fc00000);
    if (tid == 0) {
        stage::init(bar);
        stage::init(bar + 8);
        s_abort = 0;
    }
    stage::Pos start, end;
    if (win.n > 0) {
        // the windows' CTAs come last: few have work, and where one does it is not long (ahead of the glyphs' their
        // searches delayed every SM, 1.4 % on 5,000 glyphs of 4,000 queries, N = 24)
        const int g = (int)blockIdx.x, k = g - G;
        if (k >= 0) {
            if (tid < 32) {
                const int on = win.glyph(a.seg, G, a.Q, k);
                if (tid == 0) s_unit[0].g = on;
            }
            __syncthreads();  // also publishes the mbarriers
            start = stage::Pos{s_unit[0].g, k * win.size};
            end = stage::Pos{start.g, (k + 1) * win.size};
        } else {
            start = stage::Pos{g, 0};
            end = stage::Pos{g, win.own_end(stage::seg_at(a.seg, a.Q, g))};
            __syncthreads();  // publishes the mbarriers
        }
    } else {
        path.unit(s_unit, start, end);  // its barrier also publishes the mbarriers
    }

    // SET: glyphs z .. are still to be zeroed: those wholly inside this unit, through glyph `last`
    int z = start.g;
    const auto zero_through = [&](int last) {
        for (; z <= last && z < G; ++z)
            if ((z > start.g || start.q <= stage::seg_at(a.seg, a.Q, z)) && (z < end.g || end.q >= stage::seg_at(a.seg, a.Q, z + 1)))
                zero_slab(reinterpret_cast<float4*>(a.dlut) + (int64_t)z * records, records, tid, SBB);
    };
    const auto copy = [&](int g, int buf) {
        stage::issue(bar + 8 * buf, table_s + buf * table_bytes,
                     reinterpret_cast<const unsigned char*>(a.L.data) + (size_t)g * table_bytes, table_bytes);
    };
    uint32_t phase = 0;  // bit buf: parity of the buffer's next completion
    int buf = 0;
    stage::Part part = stage::next_part(a.seg, G, a.Q, start.g, start, end);
    if (tid == 0 && part.a < part.b) copy(part.g, 0);
    // queries outside every segment, under the first copy
    {
        const int64_t lo = min(max(__ldg(a.seg), (int64_t)0), a.Q);
        const int64_t hi = min(max(__ldg(a.seg + G), lo), a.Q);
        const int64_t stride = (int64_t)gridDim.x * SBB;
        for (int side = 0; side < 2; ++side) {
            const int64_t b = side ? hi : 0, e = side ? a.Q : lo;
            for (int64_t q = b + (int64_t)blockIdx.x * SBB + tid; q < e; q += stride) {
                status |= SHM_DEV_BOUNDS;
                if (a.ddirs) { a.ddirs[3 * q] = qnan; a.ddirs[3 * q + 1] = qnan; a.ddirs[3 * q + 2] = qnan; }
            }
        }
    }
    while (part.a < part.b) {
        const int g = part.g;
        const int64_t s1 = part.b;
        const stage::Part next = stage::next_part(a.seg, G, a.Q, g + 1, start, end);
        const bool more = next.a < next.b;
        if (tid == 0 && more && nbuf == 2) copy(next.g, buf ^ 1);
        // this thread's first inputs load while the table copy runs, each later round's under the
        // reductions of the round before
        float d0 = 0.f, d1 = 0.f, d2 = 0.f;
        Up up;
        const auto load = [&](int64_t q) {
            if (q >= s1) return;
            d0 = __ldcs(a.dirs + 3 * q); d1 = __ldcs(a.dirs + 3 * q + 1); d2 = __ldcs(a.dirs + 3 * q + 2);
            up.load(a, q);
        };
        load(part.a + tid);
        if (SET) zero_through(g);
        if (!stage::bar_wait(bar + 8 * buf, (phase >> buf) & 1, stage::WAIT_NS)) s_abort = 1;
        __syncthreads();
        if (s_abort) {
            status |= SHM_DEV_TIMEOUT;
            if (tid == 0) {
                stage::bar_wait(bar + 8 * buf, (phase >> buf) & 1, stage::DRAIN_NS);
                if (more && nbuf == 2) stage::bar_wait(bar + 8 * (buf ^ 1), (phase >> (buf ^ 1)) & 1, stage::DRAIN_NS);
            }
            break;
        }
        phase ^= 1u << buf;
        const unsigned char* table = tables + buf * table_bytes;
        auto fetch = [table, P](int f, int i, int j) { return stage::corners<DT>(table, P, f, i, j); };
        const GlyphRef Gr = glyph_ref(a.L, g);
        const int64_t dbase = glyph_ref(a.D, g).base;
        // warp-uniform trip count: the paired reductions need every lane of the warp
        for (int64_t qw = part.a + (tid & ~31); qw < s1; qw += SBB) {
            const int64_t q = qw + (tid & 31);
            CaptureEmit sink;
            sink.base = dbase;
            sink.P = P;
            if (q < s1) {
                float3 dd = make_float3(qnan, qnan, qnan);
                Chart c;
                if (chart_of(d0, d1, d2, c)) bwd_query<FIT>(a, up, Gr, c, d0, d1, d2, fetch, sink, dd, loss_acc);
                else status |= SHM_DEV_NONFINITE;
                if (a.ddirs) { __stcs(a.ddirs + 3 * q, dd.x); __stcs(a.ddirs + 3 * q + 1, dd.y); __stcs(a.ddirs + 3 * q + 2, dd.z); }
            }
            load(q + SBB);
            paired_reds(reinterpret_cast<float4*>(a.dlut), sink, tid & 31);
        }
        __syncthreads();  // every read of this table is done before the next copy lands
        if (nbuf == 2) buf ^= 1;
        else if (tid == 0 && more) copy(next.g, 0);
        part = next;
    }
    if (SET) zero_through(end.g);
    if (FIT && a.loss) add_loss(a.loss, loss_acc);
    report_status(a.dev_status, status);
}

template <int DT, bool FIT, bool SET>
static cudaError_t launch_bwd_staged_ft(const BackwardArgs& a, uint32_t table_bytes, cudaStream_t s)
{
    const int nbuf = 2 * (int64_t)table_bytes <= STAGED_TABLE_MAX_BYTES ? 2 : 1;
    const int smem = stage::TABLE_OFFSET + nbuf * (int)table_bytes;
    cudaError_t e = ensure_dynamic_smem((const void*)k_query_bwd_staged<DT, FIT, SET>, smem);
    if (e != cudaSuccess) return e;
    const int64_t w = table_bytes / BWD_PATH_BYTES;
    const int G = a.L.n_glyphs, records = 6 * (a.L.N_uniform + 2) * (a.L.N_uniform + 2);
    float4* const dlut = reinterpret_cast<float4*>(a.dlut);
    // Many glyphs, one table buffer: a CTA per glyph, which nothing cuts but a very long segment and which the
    // hardware hands out as SMs come free.  Neighbouring glyphs are then in flight together (16,384 x 4,096 queries,
    // even, N = 32: 2,055 us in cut units, 1,962 for strided glyphs, 1,727 so).  From 24 glyphs an SM always; from 10
    // where tables of at least WHOLE_BYTES have fewer queries than their own traffic is worth: 2,000 / 3,000 even
    // glyphs of 1,500 queries, N = 32, 145 / 212 us in units and 124 / 181 so, uneven ones 147 / 211 and 144 / 196.
    // Elsewhere the last uneven glyph shows: 3,000 of 4,000 queries, N = 24, 312 us in units and 365 so; 1,400 of 1,500,
    // N = 32, 107 and 110; and with two buffers the unit hides the next table's copy (1,000 uneven glyphs of
    // N = 20, in a training step: 376 us and 582).
    const bool whole = nbuf == 1 && (G >= 24 * sm_count() || (G >= 10 * sm_count() && table_bytes >= WHOLE_BYTES && a.Q <= w * G));
    const int64_t units = stage::units_for(a.Q, G, w, (int64_t)sm_count() * 2);
    const stage::Path path(a.seg, G, a.Q, w, units);
    const Windows win(a.Q, whole ? WINDOWS_PER_SM * sm_count() : 0);
    if (SET && whole) k_zero_long<<<(unsigned)win.n, 256, 0, s>>>(a.seg, G, a.Q, win, dlut, records);
    if (SET && !whole && units > 1) k_zero_cut<<<(unsigned)(units - 1), 1024, 0, s>>>(path, dlut, records);
    k_query_bwd_staged<DT, FIT, SET><<<(unsigned)(whole ? win.n + G : units), SBB, smem, s>>>(a, table_bytes, nbuf, path, win);
    return cudaGetLastError();
}

template <int DT>
static cudaError_t launch_bwd_staged(const BackwardArgs& a, uint32_t table_bytes, cudaStream_t s)
{
    if (a.fit) return launch_bwd_staged_ft<DT, true, false>(a, table_bytes, s);
    return a.set ? launch_bwd_staged_ft<DT, false, true>(a, table_bytes, s)
                 : launch_bwd_staged_ft<DT, false, false>(a, table_bytes, s);
}

template <int DT, int LAYOUT, bool FIT>
static cudaError_t launch_bwd_f(const BackwardArgs& a, cudaStream_t s)
{
    using Cta = BwdCta<FIT>;
    const int64_t at_once = (int64_t)sm_count() * Cta::resident * Cta::threads, cap = (int64_t)sm_count() * Cta::per_sm;
    int64_t rounds = (a.Q + at_once - 1) / at_once;  // small batches: every SM first
    if (rounds > BROUNDS) rounds = BROUNDS;
    int64_t blocks = (a.Q + Cta::threads * rounds - 1) / (Cta::threads * rounds);
    if (blocks > cap) blocks = cap;
    k_query_bwd<DT, LAYOUT, FIT><<<(unsigned)blocks, Cta::threads, 0, s>>>(a, (int)rounds);
    return cudaGetLastError();
}

template <int DT, int LAYOUT>
static cudaError_t launch_bwd_t(const BackwardArgs& a, cudaStream_t s)
{
    return a.fit ? launch_bwd_f<DT, LAYOUT, true>(a, s) : launch_bwd_f<DT, LAYOUT, false>(a, s);
}

cudaError_t launch_query_bwd(const BackwardArgs& a, cudaStream_t s)
{
    if (a.Q == 0 && !a.set) return cudaSuccess;
    const int dt = a.L.dtype, ly = a.L.layout;
    // per-glyph segments on small uniform tables: stage each glyph's table in shared memory
    if (a.Q > 0 && a.seg && !a.glyph && a.L.N_uniform > 0 && a.D.N_uniform == a.L.N_uniform && ly == SHM_LAYOUT_TEXEL) {
        const int64_t P = (int64_t)a.L.N_uniform + 2;
        const int64_t bytes = 6 * P * P * (dt == SHM_F32 ? 16 : 8);
        // Pays from fewer queries than in the forward (query_is_staged), since the staged pass's reductions also
        // meet in L2: 3,000 even glyphs of 400 / 500 queries, N = 32, 104 / 112 us staged and 118 / 131 not; of 200 / 256,
        // N = 23, 62 / 64 and 59 / 76; on small tables the copy's latency dominates (10,000 of 200, N = 8: 109 and 91), and below
        // ten glyphs an SM uneven ones lose (300 of 600, N = 32: 20 staged and 14 not).
        const int64_t least = bytes / (a.L.n_glyphs >= 10 * sm_count() ? 256 : 128), per = least > 256 ? least : 256;
        if (bytes <= STAGED_TABLE_MAX_BYTES && a.Q >= a.L.n_glyphs * per) {
            if (dt == SHM_F32) return launch_bwd_staged<SHM_F32>(a, (uint32_t)bytes, s);
            if (dt == SHM_F16) return launch_bwd_staged<SHM_F16>(a, (uint32_t)bytes, s);
            return launch_bwd_staged<SHM_BF16>(a, (uint32_t)bytes, s);
        }
    }
    if (a.set) {
        const int64_t P = (int64_t)a.D.N_uniform + 2;
        const cudaError_t e = cudaMemsetAsync(a.dlut, 0, (size_t)(6 * P * P * 16) * a.D.n_glyphs, s);
        if (e != cudaSuccess) return e;
        if (a.Q == 0) return cudaSuccess;
    }
    if (ly == SHM_LAYOUT_TEXEL) {
        if (dt == SHM_F32) return launch_bwd_t<SHM_F32, SHM_LAYOUT_TEXEL>(a, s);
        if (dt == SHM_F16) return launch_bwd_t<SHM_F16, SHM_LAYOUT_TEXEL>(a, s);
        return launch_bwd_t<SHM_BF16, SHM_LAYOUT_TEXEL>(a, s);
    }
    if (dt == SHM_F32) return launch_bwd_t<SHM_F32, SHM_LAYOUT_CELL>(a, s);
    if (dt == SHM_F16) return launch_bwd_t<SHM_F16, SHM_LAYOUT_CELL>(a, s);
    return launch_bwd_t<SHM_BF16, SHM_LAYOUT_CELL>(a, s);
}

}  // namespace shm

namespace shm {

// Adam (Kingma & Ba, 2015) with bias correction; optionally zeroes the gradient for the next step.
__device__ __forceinline__ void adam_one(float& p, float& g, float& m, float& v, float lr, float b1, float b2,
                                         float eps, float c1, float c2, int zero_grad)
{
    const float gi = g;
    const float mi = b1 * m + (1.0f - b1) * gi;
    const float vi = b2 * v + (1.0f - b2) * gi * gi;
    m = mi;
    v = vi;
    p -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    if (zero_grad) g = 0.0f;
}

// VEC4: all four arrays 16-byte aligned; 128-bit loads and stores over n/4 quadruples, then the tail.
template <bool VEC4>
__global__ void __launch_bounds__(256) k_adam(float* __restrict__ p, float* __restrict__ g, float* __restrict__ m,
                                              float* __restrict__ v, int64_t n, float lr, float b1, float b2, float eps,
                                              float c1, float c2, int zero_grad)
{
    const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, stride = (int64_t)gridDim.x * blockDim.x;
    int64_t done = 0;
    if (VEC4) {
        const int64_t n4 = n / 4;
        float4 *p4 = reinterpret_cast<float4*>(p), *g4 = reinterpret_cast<float4*>(g);
        float4 *m4 = reinterpret_cast<float4*>(m), *v4 = reinterpret_cast<float4*>(v);
        for (int64_t i = tid; i < n4; i += stride) {
            float4 P = p4[i], Gq = g4[i], M = m4[i], V = v4[i];
            adam_one(P.x, Gq.x, M.x, V.x, lr, b1, b2, eps, c1, c2, zero_grad);
            adam_one(P.y, Gq.y, M.y, V.y, lr, b1, b2, eps, c1, c2, zero_grad);
            adam_one(P.z, Gq.z, M.z, V.z, lr, b1, b2, eps, c1, c2, zero_grad);
            adam_one(P.w, Gq.w, M.w, V.w, lr, b1, b2, eps, c1, c2, zero_grad);
            p4[i] = P;
            m4[i] = M;
            v4[i] = V;
            if (zero_grad) g4[i] = Gq;
        }
        done = n4 * 4;
    }
    for (int64_t i = done + tid; i < n; i += stride) adam_one(p[i], g[i], m[i], v[i], lr, b1, b2, eps, c1, c2, zero_grad);
}

cudaError_t launch_adam(float* param, float* grad, float* m, float* v, int64_t n, float lr, float beta1, float beta2,
                        float eps, int step, int zero_grad, cudaStream_t s)
{
    if (n == 0) return cudaSuccess;
    const float c1 = 1.0f - (float)pow((double)beta1, (double)step);
    const float c2 = 1.0f - (float)pow((double)beta2, (double)step);
    const bool vec = (((uintptr_t)param | (uintptr_t)grad | (uintptr_t)m | (uintptr_t)v) & 15u) == 0;
    int64_t blocks = (n / (vec ? 4 : 1) + 255) / 256;
    const int64_t cap = (int64_t)sm_count() * 8;
    if (blocks > cap) blocks = cap;
    if (blocks < 1) blocks = 1;
    if (vec) k_adam<true><<<(unsigned)blocks, 256, 0, s>>>(param, grad, m, v, n, lr, beta1, beta2, eps, c1, c2, zero_grad);
    else k_adam<false><<<(unsigned)blocks, 256, 0, s>>>(param, grad, m, v, n, lr, beta1, beta2, eps, c1, c2, zero_grad);
    return cudaGetLastError();
}

}  // namespace shm
