// Host side of the fused sparse pass (paper Sec. 7 steps 2-4): shared-memory sizing, the choice of the block size and
// of the kernel.  sparse_step.cuh holds the step and the iterative solves, sparse_kernel.cuh the routing certificate
// and the two-level front end; each family is instantiated in a translation unit of its own so that they compile in
// parallel.
#include "sparse_kernel.cuh"
#include "sparse_step.cuh"

namespace vsa {


namespace {

// the routing variants (sparse_kernel.cuh)
size_t sparse_smem_bytes(const Geometry& g, int P, int K_c, int threads, int P_super)
{
    const int PT = P << g.tile_shift;   // routed tiles of 16 tokens
    if (P_super > 0)   // two-level front end
        return (size_t)two_level_smem_words(g.max_pages, P, PT, K_c, P_super) * 4 + 16;
    // the register variants keep a copy of the block-table row
    size_t words = (size_t)bt_stage_offset_words(g.max_pages, P, PT, K_c);
    if (g.max_pages <= 32 * threads) words += (size_t)g.max_pages;
    return words * 4 + 16;
}

int sm_count() { return device_sm_count(); }

// The closed-form family (sparse_step.cuh).  Thread-block size: one block of 512 threads per SM while there are
// no more units than SMs, two of 256 up to two units per SM, four of 128 beyond.  More than 64 pages stay with 256: each of
// four warps vouches for P / 4 of its 32 lanes, which for P near 128 lets so many pages through that the list overflows
// and the exact selection runs.  Microseconds per layer, 256 / 128 threads, bf16 cache: P = 128 384 units of 32k tokens
// 83 / 96, 1024 173 / 193, 2048 305 / 352; P = 112 1024 160 / 179; P = 96 within 5 % either way (1024 units of 8k 123 / 117,
// of 32k 148 / 149); P = 64 384 57.5 / 55.4, 1024 122 / 118.  (On the e4m3 cache 128 threads win up to P = 128, 2048
// units 303 / 274, which the rule leaves.)
int step_threads(const Geometry& g, int P)
{
    const long long units = (long long)g.batch * g.n_q_heads;
    if (units <= sm_count()) return 512;
    return units > 2 * sm_count() && P <= 64 ? 128 : 256;
}

size_t step_smem_bytes(const Geometry& g, int P, int K_c, bool fused, bool solve)
{
    return (size_t)step_layout(solve ? 256 : step_threads(g, P), g.head_dim, g.max_pages, P, P << g.tile_shift, K_c, fused,
                               false, solve).total * 4;
}

// Query heads of a cluster: those of a KV head, eight at most (the portable cluster size).
int scan_heads(const Geometry& g) { return g.group < 8 ? g.group : 8; }

// The clusters of a sparse pass that scans the pages itself, or none where a scan ahead of it is faster.  The kernel boundary
// and the scores' way through memory are 1.5 us of a step, but the scan then runs on the SMs of the units only.
//
// Few pages, fixed-order scores: two or more (tile of 16 pages, head) items to a group of lanes cost what that saves, and with 256
// threads two units share an SM.  Up to `half`: one item for every other group of lanes.  Blocks that only help with the scan
// double this where that many SMs are free anyway.  Microseconds per layer, scan ahead / here, by items of the largest context per
// block: one sequence, 8 KV heads of 4 heads, 4k 12.6 / 11.1 (16), 8k 12.6 / 12.2 (32), with helpers 11.8 (16), 16k 12.6 / 12.8 (32, with
// helpers); two of 4k 12.8 / 11.7, four 13.1 / 12.1; eight of 4k (256 threads) 16.1 / 16.1.  One head a group 4k 12.9 / 11.6 (16), 16k
// 14.1 / 14.7 (32); two heads 4k 12.8 / 11.4.  Eight heads, whose scan ahead is slower: 4k 14.9 / 12.9 (16), 16k 14.2 / 13.7 (64).
//
// Many pages, scores by MMAs (0.6 us slower than the fixed order where every warp has a tile at most: 4k 11.2 / 11.8): four tiles to a
// warp at least, on most of the SMs; two blocks of 256 threads share one.  Ahead / here: 8 of 32k (4 tiles) 22.3 / 21.2, 8 of
// 64k 29.2 / 27.7, 4 of 64k 20.5 / 19.4, 4 of 128k (8) 27.1 / 26.8, D = 64 8 of 32k 22.0 / 18.7, D = 256 34.1 / 33.0, four entropic
// iterations 4 of 32k 33.1 / 28.0, 8 of 32k 36.9 / 36.6; with two tiles 8 of 16k 19.1 / 19.3, 4 of 32k 17.4 / 17.4, on 32 SMs one of 128k
// 17.9 / 22.5, and with helpers on 64 19.4.  Eight heads, whose scan ahead is slower: any number, 4 of 20k (2 KV heads) 14.6 / 13.8, 16
// heads of one KV head 2 of 64k 15.4 / 14.8, but no more than one on few SMs, one of 32k 14.9 / 14.6.
//
// A cluster needs its SMs in one GPC: of 148 one block each, 132 are within reach of clusters of four and 120 of eight.  128 units
// of one head a group, which share no rows: 15.4 / 15.7.
struct ScanCluster {
    int blocks;   // 0: a scan ahead
    int per_sm;   // blocks that share an SM
    bool mma;     // scores by MMAs
};

ScanCluster scan_cluster(const Geometry& g, int threads)
{
    const int heads = scan_heads(g), groups = threads / step_lanes_per_row(g.head_dim), half = groups / 2, sms = sm_count();
    const long long clusters = (long long)g.batch * g.n_q_heads / heads, tiles = (g.max_pages + 15) / 16;
    if (threads < 256) return {0, 0, false};
    auto fits = [&](int c, int per_sm) { return clusters * c * 16 <= (long long)per_sm * (c == 8 ? 13 : c == 1 ? 7 : 14) * sms; };
    auto items = [&](int c) { return (tiles + c - 1) / c * heads; };
    int c = heads;
    while (items(c) > half && 2 * c <= 8 && 2 * c * clusters * 16 <= 7 * sms) c *= 2;
    if (items(c) <= (heads == 8 ? 4 * half : half) && fits(c, 1)) return {c, 1, false};
    const long long blocks = clusters * heads, warps = (long long)heads * (threads / 32);
    if (3 * blocks >= 2 * sms ? heads < 8 && tiles < 4 * warps : heads < 8 || tiles > warps) return {0, 0, false};
    if (fits(heads, 1)) return {heads, 1, true};
    return threads == 256 && fits(heads, 2) ? ScanCluster{heads, 2, true} : ScanCluster{0, 0, false};
}

// Order of a unit's tiles, see BY_POSITION (sparse_step.cuh); not a matter of the stream, so that the sums are not.
bool step_by_position(const Geometry& g, int P, int threads, bool fp8, StepScan rule)
{
    if (!step_order_open(threads, g.head_dim, fp8) || rule == StepScan::AheadMma || rule == StepScan::InsideMma) return true;
    const bool rounds = (P << g.tile_shift) > threads / step_lanes_per_row(g.head_dim);
    return threads == 512 && rule == StepScan::Ahead && rounds && g.group > 1 && 2LL * g.batch * g.n_q_heads > sm_count();
}

// thread-block size of the routing variants for a launch
int sparse_block_threads(const Geometry& g, int P, bool listed, bool two_level, int P_super)
{
    const long long units = (long long)g.batch * g.n_q_heads;
    const bool many = units > 2 * sm_count() && (P << g.tile_shift) <= 64;
    const int threads = units <= sm_count() ? 512 : 256;
    // two-level front end: every thread holds 8 representative scores and 8 of the 16 * P_super exact scores
    if (two_level) return many && (g.max_pages + 15) / 16 <= 8 * 128 && P_super <= 64 ? 128 : threads;
    return many && !listed && g.max_pages <= 32 * 128 ? 128 : threads;
}

}  // namespace

// What a launch of the closed-form family depends on beside its arrays.  selects: the pages are selected from scores, by MMAs with near
static StepParams step_params(const Geometry& g, int P, int K_c, int threads, bool selects, bool near, bool fp8, bool solve, const ScanCluster& scan)
{
    StepParams p = {};
    p.geo = g;
    p.P = P;
    p.K_c = K_c;
    p.lay = step_layout(threads, g.head_dim, g.max_pages, P, P << g.tile_shift, K_c, selects, fp8, solve, scan.blocks, scan_heads(g), near);
    p.scan_per_sm = scan.per_sm;
    p.scan_mma = scan.mma;
    while ((1 << p.cluster_shift) < scan.blocks) ++p.cluster_shift;
    while ((1 << p.heads_shift) < scan_heads(g)) ++p.heads_shift;
    while ((1 << p.group_shift) < g.group) ++p.group_shift;
    return p;
}

static cudaError_t launch_step_of(const StepParams& p, int threads, bool fp8, int solver, cudaStream_t stream)
{
    if (solver) return launch_step_solve(p, solver, stream);
    if (fp8) return launch_step_fp8(p, threads, stream);
    if (p.geo.head_dim == 64) return launch_step_d64(p, threads, stream);
    if (p.geo.head_dim == 256) return launch_step_d256(p, threads, stream);
    return launch_step(p, threads, stream);
}

// Where the step of a shape scores its pages when it has the whole device, and its parameters if that is inside
struct ScanRule {
    StepScan scan;
    StepParams inside;
};

static ScanRule scan_rule(const Geometry& g, int P, int K_c, int threads, bool fp8, int solver)
{
    const ScanCluster c = scan_cluster(g, threads);
    if (c.blocks) {
        const StepParams p = step_params(g, P, K_c, threads, true, c.mma, fp8, solver != 0, c);
        if ((size_t)p.lay.total * 4 <= (size_t)(c.per_sm == 2 ? 113 : 227) * 1024) return {c.mma ? StepScan::InsideMma : StepScan::Inside, p};
    }
    const bool mma = threads == 128 && route_mma_wins(g) && route_bound_bytes(g) <= dense_partials_bytes(g) &&
                     (size_t)step_params(g, P, K_c, threads, true, true, fp8, false, {0, 0, false}).lay.total * 4 <= (size_t)227 * 1024;
    return {mma ? StepScan::AheadMma : StepScan::Ahead, {}};
}

StepScan step_scan(const Geometry& g, int P, int K_c, bool fp8, int solver, cudaStream_t stream)
{
    const int threads = solver ? 256 : step_threads(g, P);
    ScanRule rule = scan_rule(g, P, K_c, threads, fp8, solver);
    if (rule.scan == StepScan::Ahead || rule.scan == StepScan::AheadMma) return rule.scan;
    // The rule counts the SMs of one chip.  What a stream really has (another chip's GPCs, a green context, a share of the SMs
    // under MPS) may hold fewer clusters at once, or none, and then there would be no launch: the scan ahead.
    int n = 0;
    const uint16_t any = 0;
    rule.inside.summaries = &any;   // (of the kernels that scan)
    rule.inside.active_clusters = &n;
    if (launch_step_of(rule.inside, threads, fp8, solver, stream) != cudaSuccess) {
        (void)cudaGetLastError();
        return StepScan::Ahead;
    }
    return (long long)n * scan_heads(g) >= (long long)g.batch * g.n_q_heads ? rule.scan : StepScan::Ahead;
}

bool sparse_shared_memory_fits(const Geometry& g, int P, int K_c, bool fused, bool solve, bool cert, int P_super)
{
    if (!cert && P_super == 0) return step_smem_bytes(g, P, K_c, fused, solve) <= (size_t)227 * 1024;
    return sparse_smem_bytes(g, P, K_c, sparse_block_threads(g, P, false, P_super > 0, P_super), P_super) <= (size_t)227 * 1024;
}

int sparse_register_select_max_pages(long long units) { return 32 * (units <= sm_count() ? 512 : 256); }

cudaError_t launch_sparse(const Geometry& g, const void* q, const void* k_cache, const void* v_cache,
                          const int32_t* block_table, const int32_t* seq_lens, int32_t* routed_pages,
                          const float* page_scores, int P, int K_c, float epsilon, float gap_threshold, float* out,
                          vsa_diag_t* diag, int32_t* fallback_list, int32_t* fallback_count, cudaStream_t stream,
                          int solver_iters, vsa_solve_t* solve, const float* rad_logical, vsa_cert_t* cert,
                          int solver_kind, const int32_t* unit_list, const int32_t* unit_count, int routed_stride,
                          const void* tl_summaries, int P_super, const float* k_scale, const float* v_scale,
                          const void* scan_summaries, int32_t* flags, int32_t* tickets, const uint32_t* bounds)
{
    if ((k_scale || v_scale) && (!k_scale || !v_scale || solve || cert || tl_summaries || g.head_dim != kHeadDim))
        return cudaErrorInvalidValue;
    if (g.head_dim != kHeadDim && (solve || cert || tl_summaries)) return cudaErrorInvalidValue;   // (refused by the entry points)
    if (!cert && !tl_summaries) {
        const int threads = solve ? 256 : step_threads(g, P), solver = solve ? solver_kind : 0;
        const bool fp8 = k_scale != nullptr;
        const ScanRule rule = scan_rule(g, P, K_c, threads, fp8, solver);
        const bool inside = !page_scores && scan_summaries;
        StepParams p = inside ? rule.inside
                              : step_params(g, P, K_c, threads, page_scores != nullptr, bounds != nullptr, fp8, solve != nullptr, {0, 0, false});
        p.q = (const uint16_t*)q;
        p.k = (const uint16_t*)k_cache;
        p.v = (const uint16_t*)v_cache;
        p.block_table = block_table;
        p.seq_lens = seq_lens;
        p.routed_pages = routed_pages;
        p.page_scores = page_scores;
        p.summaries = (const uint16_t*)scan_summaries;
        p.bounds = bounds;
        p.flags = flags;
        p.tickets = tickets;
        p.n_tickets = tickets ? dense_ticket_count(g) : 0;
        p.by_position = step_by_position(g, P, threads, fp8, rule.scan);
        p.epsilon = epsilon;
        p.gap_threshold = gap_threshold;
        p.out = out;
        p.diag = diag;
        p.fallback_list = fallback_list;
        p.fallback_count = fallback_count;
        p.solver_iters = solver_iters;
        p.solve = solve;
        p.k_scale = k_scale;
        p.v_scale = v_scale;
        return launch_step_of(p, threads, fp8, solver, stream);
    }
    SparseArgs a;
    a.g = g;
    const int threads = sparse_block_threads(g, P, unit_list != nullptr, tl_summaries != nullptr, P_super);
    a.smem = sparse_smem_bytes(g, P, K_c, threads, tl_summaries ? P_super : 0);
    a.tl_summaries = (const uint16_t*)tl_summaries;
    a.P_super = P_super;
    a.rad_logical = rad_logical;
    a.cert = cert;
    a.unit_list = unit_list;
    a.unit_count = unit_count;
    a.routed_stride = routed_stride > 0 ? routed_stride : P;
    a.q = (const uint16_t*)q;
    a.k = (const uint16_t*)k_cache;
    a.v = (const uint16_t*)v_cache;
    a.block_table = block_table;
    a.seq_lens = seq_lens;
    a.routed_pages = routed_pages;
    a.page_scores = page_scores;
    a.P = P;
    a.K_c = K_c;
    a.epsilon = epsilon;
    a.gap_threshold = gap_threshold;
    a.out = out;
    a.diag = diag;
    a.fallback_list = fallback_list;
    a.fallback_count = fallback_count;
    a.stream = stream;
    if (solve || !page_scores) return cudaErrorInvalidValue;
    if (tl_summaries) return cert ? cudaErrorInvalidValue : launch_sparse_two_level(a, threads);
    return launch_sparse_cert(a, threads);
}

}  // namespace vsa
