// Value-only reconstruction baselines (§4.2 Table psnr_value, §4.5 Table cost_extended):
// nearest, bilinear + finite-difference gradient, 16-tap Catmull-Rom with analytic gradient and
// the cubic B-spline of the 4-bilinear-fetch "fast bicubic", on a SHM_LAYOUT_VALUE table, run
// through the same query kernel skeletons as the Hermite query: per query, or staged for per-glyph
// segments on small tables.
//
// Staged (k_recon_staged): as k_query_staged, a CTA takes one unit of the path through glyphs and
// queries, the glyph's value table (31 KB at N = 32 f32) comes into shared memory by one bulk copy
// while the previous glyph's queries run, and the 4 to 32 taps are shared-memory reads.  A value table
// need not be a multiple of 16 bytes, so the copy starts at the 16-byte boundary before it (within the
// pool: the first glyph is aligned) and its last bytes, up to 15, come by plain loads.  The work common to
// all methods (chart, gradient, normal, 40 B of I/O) bounds the small ones, the taps the B-spline.  2,048
// glyphs N = 32 f32, 2^23 queries, per query before -> staged: nearest 135 -> 86 us, bilinear 175 -> 94,
// Catmull-Rom 265 -> 107, B-spline 750 -> 199 (its five shifted lookups share 32 taps instead of 80).
#include "shm_query_kernel.cuh"
#include "shm_stage.cuh"

namespace shm {

namespace {

constexpr int RS_BLOCK = 512;

template <int DT>
struct StagedFace {
    const unsigned char* face;  // entry (0, 0) = texel (-1, -1)
    int S;
    __device__ __forceinline__ float operator()(int i, int j) const
    {
        const int e = (j + 1) * S + (i + 1);
        if (DT == SHM_F32) return reinterpret_cast<const float*>(face)[e];
        if (DT == SHM_F16) return __half2float(reinterpret_cast<const __half*>(face)[e]);
        return __bfloat162float(reinterpret_cast<const __nv_bfloat16*>(face)[e]);
    }
};

template <int DT, int METHOD>
__global__ void __launch_bounds__(RS_BLOCK, 2) k_recon_staged(QueryArgs a, uint32_t table_bytes, uint32_t slot, int nbuf,
                                                              const __grid_constant__ stage::Path path)
{
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ int s_abort;
    __shared__ stage::Pos s_unit[2];
    constexpr int ELEM = DT == SHM_F32 ? 4 : 2;
    const uint32_t bar = (uint32_t)__cvta_generic_to_shared(smem);
    unsigned char* tables = smem + stage::TABLE_OFFSET;
    const uint32_t table_s = bar + stage::TABLE_OFFSET;
    const int tid = threadIdx.x;
    const int G = a.L.n_glyphs, N = a.L.N_uniform, S = N + 4;
    const unsigned char* pool = reinterpret_cast<const unsigned char*>(a.L.data);
    const float qnan = __int_as_float(0x7fc00000);
    uint32_t status = 0;

    const auto store = [&](int64_t q, float R, const Vec3& g, const Vec3& n, float Ru, float Rv, int f, int i, int j) {
        if (a.R) __stcs(a.R + q, R);
        if (a.grad) { __stcs(a.grad + 3 * q, g.x); __stcs(a.grad + 3 * q + 1, g.y); __stcs(a.grad + 3 * q + 2, g.z); }
        if (a.normal) { __stcs(a.normal + 3 * q, n.x); __stcs(a.normal + 3 * q + 1, n.y); __stcs(a.normal + 3 * q + 2, n.z); }
        if (a.chart) { a.chart[2 * q] = Ru; a.chart[2 * q + 1] = Rv; }
        if (a.fij) { a.fij[3 * q] = f; a.fij[3 * q + 1] = i; a.fij[3 * q + 2] = j; }
    };
    const Vec3 nan3{qnan, qnan, qnan};
    if (tid == 0) {
        stage::init(bar);
        stage::init(bar + 8);
        s_abort = 0;
    }
    stage::Pos start, end;
    path.unit(s_unit, start, end);

    // bytes [lo, lo + table_bytes) of the pool: whole 16-byte blocks from the boundary before lo, and the
    // remainder
    const auto copy = [&](int g, int buf) {
        const size_t lo = (size_t)g * table_bytes, from = lo & ~(size_t)15, to = (lo + table_bytes) & ~(size_t)15;
        stage::issue(bar + 8 * buf, table_s + buf * slot, pool + from, (uint32_t)(to - from));
    };
    const auto copy_rest = [&](int g, int buf) {
        const size_t lo = (size_t)g * table_bytes, from = lo & ~(size_t)15, to = (lo + table_bytes) & ~(size_t)15;
        const int rest = (int)(lo + table_bytes - to);
        if (tid * 2 < rest)
            *reinterpret_cast<uint16_t*>(tables + buf * slot + (to - from) + tid * 2) =
                __ldg(reinterpret_cast<const uint16_t*>(pool + to) + tid);
    };
    uint32_t phase = 0;
    int buf = 0;
    stage::Part part = stage::next_part(a.seg, G, a.Q, start.g, start, end);
    if (tid == 0 && part.a < part.b) copy(part.g, 0);
    // queries outside every segment, under the first copy
    {
        const int64_t lo = stage::seg_at(a.seg, a.Q, 0), hi = max(stage::seg_at(a.seg, a.Q, G), lo);
        const int64_t stride = (int64_t)gridDim.x * RS_BLOCK;
        for (int side = 0; side < 2; ++side) {
            const int64_t b = side ? hi : 0, e = side ? a.Q : lo;
            for (int64_t q = b + (int64_t)blockIdx.x * RS_BLOCK + tid; q < e; q += stride) {
                status |= SHM_DEV_BOUNDS;
                store(q, qnan, nan3, nan3, qnan, qnan, -1, -1, -1);
            }
        }
    }
    while (part.a < part.b) {
        const int g = part.g;
        int64_t q = part.a + tid;
        float d0 = 0.f, d1 = 0.f, d2 = 0.f;
        if (q < part.b) { d0 = __ldcs(a.dirs + 3 * q); d1 = __ldcs(a.dirs + 3 * q + 1); d2 = __ldcs(a.dirs + 3 * q + 2); }
        const stage::Part next = stage::next_part(a.seg, G, a.Q, g + 1, start, end);
        const bool more = next.a < next.b;
        if (tid == 0 && more && nbuf == 2) copy(next.g, buf ^ 1);
        copy_rest(g, buf);
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
        const float r0 = a.L.r0 ? __ldg(a.L.r0 + g) : 0.0f;
        const unsigned char* table = tables + buf * slot + (((size_t)g * table_bytes) & 15);
        const auto face = [&](int f) { return StagedFace<DT>{table + f * S * S * ELEM, S}; };
        for (; q < part.b; q += RS_BLOCK) {
            const int64_t qn = q + RS_BLOCK;
            float n0 = 0.f, n1 = 0.f, n2 = 0.f;
            if (qn < part.b) { n0 = __ldcs(a.dirs + 3 * qn); n1 = __ldcs(a.dirs + 3 * qn + 1); n2 = __ldcs(a.dirs + 3 * qn + 2); }
            QueryResult r;
            Chart c;
            if (recon_eval<METHOD>(face, N, r0, d0, d1, d2, r, c)) {
                store(q, r.R, r.grad, a.normal ? surface_normal(d0, d1, d2, r.R, r.grad) : nan3, r.Ru, r.Rv, r.f, r.i, r.j);
            } else {
                status |= SHM_DEV_NONFINITE;
                store(q, qnan, nan3, nan3, qnan, qnan, -1, -1, -1);
            }
            d0 = n0; d1 = n1; d2 = n2;
        }
        __syncthreads();  // every read of this table is done before the next copy lands
        if (nbuf == 2) buf ^= 1;
        else if (tid == 0 && more) copy(next.g, 0);
        part = next;
    }
    report_status(a.dev_status, status);
}

template <int DT, int METHOD>
cudaError_t launch_recon_staged(const QueryArgs& a, uint32_t table_bytes, cudaStream_t s)
{
    const uint32_t slot = (table_bytes + 31) & ~15u;  // up to 15 bytes before the table, rounded to 16
    const int nbuf = 2 * (int64_t)slot <= STAGED_TABLE_MAX_BYTES ? 2 : 1;
    const int smem = stage::TABLE_OFFSET + nbuf * (int)slot;
    const cudaError_t e = ensure_dynamic_smem((const void*)k_recon_staged<DT, METHOD>, smem);
    if (e != cudaSuccess) return e;
    const int64_t w = table_bytes / stage::QUERY_BYTES;
    const int64_t units = stage::units_for(a.Q, a.L.n_glyphs, w, (int64_t)sm_count() * 2);
    k_recon_staged<DT, METHOD><<<(unsigned)units, RS_BLOCK, smem, s>>>(a, table_bytes, slot, nbuf,
                                                                     stage::Path(a.seg, a.L.n_glyphs, a.Q, stage::path_weight(w, a.L.n_glyphs, units), units));
    return cudaGetLastError();
}

template <int DT, int METHOD>
cudaError_t launch_recon_t(const QueryArgs& a, cudaStream_t s)
{
    // The rule of query_is_staged, with the value table's bytes; the nearest baseline's single tap needs
    // more queries to pay for the copy (3,000 glyphs N = 32 f32, 256 / 512 queries each: staged 30.8 / 35.1
    // us against 28.8 / 48.9; Catmull-Rom 32.4 / 38.7 against 55.8 / 77.7).
    if (a.seg && !a.glyph && a.L.N_uniform > 0) {
        const int64_t S = (int64_t)a.L.N_uniform + 4;
        const int64_t bytes = 6 * S * S * (DT == SHM_F32 ? 4 : 2);
        const int64_t least = METHOD == SHM_RECON_NEAREST ? 512 : 256;
        const int64_t per = bytes / 128 > least ? bytes / 128 : least;
        if (bytes + 31 <= STAGED_TABLE_MAX_BYTES && a.Q >= a.L.n_glyphs * per)
            return launch_recon_staged<DT, METHOD>(a, (uint32_t)bytes, s);
    }
    return launch_fwd_t<DT, SHM_LAYOUT_VALUE, METHOD>(a, s);
}

template <int METHOD>
cudaError_t launch_recon_m(const QueryArgs& a, cudaStream_t s)
{
    if (a.L.dtype == SHM_F32) return launch_recon_t<SHM_F32, METHOD>(a, s);
    if (a.L.dtype == SHM_F16) return launch_recon_t<SHM_F16, METHOD>(a, s);
    return launch_recon_t<SHM_BF16, METHOD>(a, s);
}

}  // namespace

cudaError_t launch_query_recon(const QueryArgs& a, int method, cudaStream_t s)
{
    if (a.Q == 0) return cudaSuccess;
    switch (method) {
    case SHM_RECON_NEAREST: return launch_recon_m<SHM_RECON_NEAREST>(a, s);
    case SHM_RECON_BILINEAR: return launch_recon_m<SHM_RECON_BILINEAR>(a, s);
    case SHM_RECON_BICUBIC: return launch_recon_m<SHM_RECON_BICUBIC>(a, s);
    default: return launch_recon_m<SHM_RECON_FAST_BICUBIC>(a, s);
    }
}

}  // namespace shm
