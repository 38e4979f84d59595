// lbmp_internal.h -- host-side handle of the C ABI and the kernel launchers
// shared between the translation units of the library.
#pragma once

#include <cuda_runtime.h>

#include <string.h>

#include <cmath>

#include "../../include/lbmp.h"
#include "lbmp_common.cuh"

struct lbmp_handle {
    lbmp_grid grid;
    int D, Q;
    int Qg;            // phase-field populations: Q, or 2D+1 on the reduced phase lattice
    bool reduced;      // LBMP_FLAG_PHASE_REDUCED
    lbmp_params params;
    lbmp_derived der;
    lbmp::DevParams dp;
    cudaStream_t stream;
    int device;
    long long N;
    // ping-pong population sets; buffers hold post-collision values of the
    // previous step (pull streaming reads them upstream)
    float* f[2];
    float* g[2];
    // z-slab (lbmp_create_slab): global planes [slab_z0, slab_z1) held with
    // slab_ghost[0] / [1] ghost planes below / above; slab = false otherwise
    bool slab;
    int slab_z0, slab_z1, slab_ghost[2];
    // in-place AA storage (LBMP_FLAG_AA): f[1] == f[0], g[1] == g[0], and
    // parity is the phase (0 natural, 1 swapped; dp.aa = 1 + parity)
    bool aa;
    float* phi;        // reference pair only: phi = sum g as hi [0, N) + lo [N, 2N), refreshed by the phi pass
    lbmp_allocator alloc;  // caller's device allocator (alloc == null: cudaMalloc / cudaFree)
    float* phiu;       // reduced phase lattice: phi u of the previous step, [k < D][cell]; else null
    bool divu;         // LBMP_FLAG_DIVU
    float* uvel[2];    // LBMP_FLAG_DIVU: stored velocity [k < D][cell], uvel[parity] the previous step's; else null
    int parity;        // f[parity], g[parity] hold the current state
    long step;
    int kernel;        // LBMP_OPT_KERNEL: 0 default, 1 reference pair, 2 bulk-copy staging
    int opt_chunk;     // LBMP_OPT_CHUNK: planes (rows) per work item, 0 = automatic
    int opt_ctas;      // LBMP_OPT_CTAS_PER_SM: resident CTAs per SM of the grid, 0 = occupancy maximum
    int opt_tile;      // LBMP_OPT_TILE: tile shape of the FP32 D3Q27 fused kernel (0 32x4, 1 16x8, 2 8x16)
    int probe[3];
    // planes per work item and kernel last chosen for the step, and what for
    int shape[2], shape_for[6];
    // step graphs (lbmp_step): kStepGraph steps captured from each starting
    // parity, for the launch options in graph_key; warm once a plain step
    // ran with those options (the kernels' one-time set-up is not captured)
    cudaGraphExec_t step_graph[2];
    long long graph_key[6];
    bool graph_warm, graph_off;
    // observables scratch (partial sums per block) and result slot
    double* red;
    int red_blocks;
    double* red_out;
};

namespace lbmp {

// one member of a batch, as the batch kernels see it (device memory)
struct BatchDomain {
    DevParams p;
    float* f[2];
    float* g[2];
    float* phiu;  // reduced phase lattice: stored previous phi u; else null
    int parity, steps_left;
    int tiles_x, tiles_y, chunk, item_begin, items;
};

// Estimated time of a launch of `tiles` tiles marching through `nmarch` planes
// (rows in 2-D) in items of `chunk` planes, on per_sm CTAs of each of `sms` SMs,
// in units of its own kernel: a plane takes `plane` + the CTAs that share the
// SM, an item `extra` planes more than it updates, a grid that is not launched
// early (launch_after) `gap`.  In the first rounds the slots run in step, so the
// time is that of the rounds, the last one with the CTAs that are left; later
// the slots have drifted apart and the time tends to the mean load.
struct MarchCost {
    double plane, extra, gap;
};
inline double march_time(const MarchCost& m, int tiles, int nmarch, int chunk, int per_sm, int sms)
{
    const int per_tile = (nmarch + chunk - 1) / chunk;
    const long long slots = (long long)per_sm * sms, items = (long long)tiles * per_tile;
    const long long rounds = (items + slots - 1) / slots;
    const double full = m.plane + per_sm, last = m.plane + (double)(items - (rounds - 1) * slots) / sms;
    const double in_step = (chunk + m.extra) * ((double)(rounds - 1) * full + last);
    const double mean = (double)tiles * (nmarch + m.extra * per_tile) / (double)slots * full;
    const double least = (chunk + m.extra) * (rounds == 1 ? last : full);
    const double w = std::exp(-0.4 * (double)(rounds - 1));
    return w * in_step + (1.0 - w) * (mean > least ? mean : least) + (2 * items > slots ? m.gap : 0.0);
}
constexpr int kLongestItem = 64;  // planes (items of up to 72 were measured)

// Launch shape of a persistent fused kernel over `tiles` tiles marching
// through `nmarch` planes (rows in 2-D): planes per work item and grid size,
// from the handle's options or the shape with the least estimated time.
struct LaunchShape {
    int chunk, nitems, grid;
    bool half_empty;  // the grid takes at most half of the GPU's slots
};
inline LaunchShape shape_of(const lbmp_handle* h, int tiles, int nmarch, int chunk, int per_sm, int sms)
{
    const long long cap = (long long)((h->opt_ctas > 0 && h->opt_ctas < per_sm) ? h->opt_ctas : per_sm) * sms;
    LaunchShape L;
    L.chunk = chunk < nmarch ? chunk : nmarch;
    L.nitems = tiles * ((nmarch + L.chunk - 1) / L.chunk);
    L.grid = (int)(L.nitems < cap ? L.nitems : cap);
    L.half_empty = 2LL * L.grid <= (long long)per_sm * sms;
    return L;
}

// n kernels that compute the same step: cost[k] in units that compare, per_sm[k]
// the CTAs each reaches.  The choice is kept in the handle until the options it
// was made for change (64 estimates, 2 us of host time).  The constants of each
// kernel are the best of a grid over 64 (FP32 D3Q27: 238) domains of 2e4 to 1e7
// (2e7) cells, each measured with every chunk of a dense set.  On 50 other
// domains of that range, time against the rule before (the longest axis halved
// until 2.5 rounds of the grid are full, else the best of a simpler estimate),
// on average and at worst: D3Q27 FP16 0.949 and 1.04, BF16 0.947 and 1.01, FP32
// in place 0.984 and 1.01, reduced phase lattice 0.989 and 1.01, D2Q9 FP32 0.978
// and 1.05, reduced 0.988 and 1.08, FP16 and BF16 0.930 and 1.01.  The best
// measured chunks of the first set: 0.955, 0.981, 0.987, 0.972 and 0.946 for
// 16-bit, in place, reduced and the two D2Q9 forms.
inline int best_shape(lbmp_handle* h, int tiles, int nmarch, const MarchCost* cost, const double* scale,
                      const int* per_sm, int n, int sms, int& chunk)
{
    const int key[6] = {tiles, nmarch, h->opt_chunk, h->opt_ctas, per_sm[0], n};
    if (h->shape[0] == 0 || memcmp(key, h->shape_for, sizeof key) != 0) {
        double best = 0.0;
        const int c0 = h->opt_chunk > 0 ? (h->opt_chunk < nmarch ? h->opt_chunk : nmarch)
                                        : (nmarch < kLongestItem ? nmarch : kLongestItem);
        const int c1 = h->opt_chunk > 0 ? c0 : 1;
        for (int k = 0; k < n; ++k) {
            const int per = (h->opt_ctas > 0 && h->opt_ctas < per_sm[k]) ? h->opt_ctas : per_sm[k];
            for (int c = c0; c >= c1; --c) {
                const double t = scale[k] * march_time(cost[k], tiles, nmarch, c, per, sms);
                if ((k == 0 && c == c0) || t < best) {
                    best = t;
                    h->shape[0] = c;
                    h->shape[1] = k;
                }
            }
        }
        memcpy(h->shape_for, key, sizeof key);
    }
    chunk = h->shape[0];
    return h->shape[1];
}
inline LaunchShape launch_shape(lbmp_handle* h, const MarchCost& cost, int tiles, int nmarch, int per_sm, int sms)
{
    if (per_sm < 1) per_sm = 1;
    const double one = 1.0;
    int chunk;
    best_shape(h, tiles, nmarch, &cost, &one, &per_sm, 1, sms, chunk);
    return shape_of(h, tiles, nmarch, chunk, per_sm, sms);
}

// The FP32 D3Q27 step, and which of its two kernels: with f' loaded one plane
// ahead at per_sm[1] CTAs per SM, or without at per_sm[0].  Loading ahead takes
// 0.9 of the time per plane and CTA but starts an item with half a plane more,
// so it wins where the items are long and its smaller grid does not add a
// round.  Against the rule before and no loading ahead: 2.1 % less time on
// average (the best measured choices: 3.6 %) and at most 2 % more for all but
// 7 of 238 domains.  With the default items, without loading ahead and now: 72^3
// 51.2 and 46.1 us, 112^3 144 and 134, 128^3 199 and 187; but 160^3 363 and 401.
constexpr MarchCost kCostFp32[2] = {{1.25, 0.4, 0.0}, {1.25, 0.9, 0.0}};
constexpr double kScaleFp32[2] = {1.0, 0.9};
inline LaunchShape launch_shape_ahead(lbmp_handle* h, int tiles, int nmarch, const int per_sm[2], int sms,
                                      bool& ahead)
{
    int chunk;
    ahead = best_shape(h, tiles, nmarch, kCostFp32, kScaleFp32, per_sm, 2, sms, chunk) != 0;
    return shape_of(h, tiles, nmarch, chunk, per_sm[ahead], sms);
}

// Planes (rows) per work item of `n` domains stepped by one batch launch, domain
// k with tiles[k] tiles marching through nmarch[k] planes, on `slots` resident
// CTAs (and of the observables' march).  Where 8 or more planes per item leave
// 2.5 rounds of the full grid, the largest power-of-two part of the longest
// domain that does: each item stages two planes more than it updates, so longer
// items win until the rounds get coarse.  Smaller work cannot fill 2.5 rounds;
// there the time is about rounds x (planes + 1.5) x (0.7 + occupancy), the stages
// of one item times a stage's latency, which grows with the number of CTAs that
// share an SM, and the rule takes the planes that make it smallest.
inline int planes_per_item(const int* tiles, const int* nmarch, int n, long long slots)
{
    int longest = 1;
    for (int k = 0; k < n; ++k) longest = nmarch[k] > longest ? nmarch[k] : longest;
    const auto items = [&](int c) {
        long long t = 0;
        for (int k = 0; k < n; ++k) t += (long long)tiles[k] * ((nmarch[k] + c - 1) / c);
        return t;
    };
    int chunk = longest;
    while (chunk > 8 && 2 * items(chunk) < 5 * slots) chunk /= 2;
    if (2 * items(chunk) >= 5 * slots) return chunk;
    const int top = longest < 64 ? longest : 64;
    double best = 0.0;
    for (int c = top; c >= 1; --c) {
        const long long it = items(c), rounds = (it + slots - 1) / slots;
        const double cost = (double)rounds * (c + 1.5) * (0.7 + (double)it / (double)(rounds * slots));
        if (c == top || cost < best) {
            best = cost;
            chunk = c;
        }
    }
    return chunk;
}

// Priority of a batch's second branch (its D2Q9 members): one level above the
// batch's stream, so that its few short items go before the D3Q27 kernels of the
// same step, which fill every slot of the GPU (they would otherwise start when
// those end), and no further before the caller's other work.  (Smaller numbers are
// greater priorities.)
inline int branch_priority(int stream_priority, int greatest)
{
    return stream_priority > greatest ? stream_priority - 1 : greatest;
}

// Launch of a step kernel that begins with after_previous().  A grid that
// leaves at least half of the GPU's slots empty is launched while the kernel
// before it in the stream still runs (also as an edge of a captured graph): on
// the legacy default stream a step of 64x256 D2Q9 cells takes 3.7 us instead
// of 6.2, one of the 400x250 impact 8.4 instead of 10.2.  Fuller grids are not:
// their early CTAs wait in the slots that the running step drains, which made
// 1024x512 D2Q9 3 %, 64^3 D3Q27 3 % and 128x128x512 11 % slower.
template <class... P, class... A>
inline cudaError_t launch_after(void (*kernel)(P...), const LaunchShape& L, unsigned block, size_t smem,
                                cudaStream_t stream, const A&... args)
{
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)L.grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cfg.attrs = &attr;
    cfg.numAttrs = L.half_empty ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}

// bytes of one population set (f' or g) in the handle's storage form
inline size_t set_bytes(const lbmp_handle* h)
{
    const size_t N = (size_t)h->N, Q = (size_t)h->Q;
    if (h->params.storage == LBMP_FP32) return sizeof(float) * Q * N;
    return sizeof(float) * N + sizeof(unsigned short) * (Q - 1) * N;  // reference + 16-bit codes
}
// bytes of one phase-field population set (equals set_bytes but on the reduced phase lattice)
inline size_t gset_bytes(const lbmp_handle* h)
{
    if (h->reduced) return sizeof(float) * (size_t)h->Qg * (size_t)h->N;
    return set_bytes(h);
}
// bytes of the stored previous phi u (reduced phase lattice)
inline size_t phiu_bytes(const lbmp_handle* h) { return h->reduced ? sizeof(float) * h->D * (size_t)h->N : 0; }
// bytes of one stored velocity field (LBMP_FLAG_DIVU)
inline size_t uvel_bytes(const lbmp_handle* h) { return h->divu ? sizeof(float) * h->D * (size_t)h->N : 0; }

// The autotuners time real step kernels.  On the reduced phase lattice a
// step replaces the stored previous phi u in place, so a trial launch would
// leave this step's phi u where the next step expects the previous one (its
// d/dt(phi u) would read zero).  phiu_save copies the stored phi u of h into
// a fresh device buffer (*copy, null when h keeps none) on `stream`;
// phiu_restore copies it back on `stream`, waits for the copy and frees the
// buffer.
cudaError_t phiu_save(lbmp_handle* h, cudaStream_t stream, float** copy);
cudaError_t phiu_restore(lbmp_handle* h, cudaStream_t stream, float* copy);

// device memory of a handle: the caller's allocator, or cudaMalloc
cudaError_t dev_alloc(lbmp_handle* h, void** p, size_t bytes);
void dev_free(lbmp_handle* h, void* p, size_t bytes);
// where the phi pass writes phi (hi, lo; 2N floats): the handle's phi array
// when it keeps one (the reference pair reads it while writing the other
// population set), else the f' population set the next step overwrites,
// whose contents are dead between steps
inline float* phi_buf(const lbmp_handle* h) { return h->phi ? h->phi : h->f[1 - h->parity]; }
// allocate the phi array the reference pair needs (not during a capture)
cudaError_t ensure_phi(lbmp_handle* h);

// kernel launchers (return cudaError_t of the launch)
cudaError_t launch_phi_pass(lbmp_handle* h);
cudaError_t launch_phiu_reset(lbmp_handle* h);  // reduced phase lattice: previous phi u := current
cudaError_t launch_step_simple(lbmp_handle* h);
cudaError_t launch_step_fused3(lbmp_handle* h);        // FP32 D3Q27, 32 x 4 tiles
cudaError_t launch_step_fused3_t16x8(lbmp_handle* h);  // FP32 D3Q27, 16 x 8 tiles
cudaError_t launch_step_fused3_t8x16(lbmp_handle* h);  // FP32 D3Q27, 8 x 16 tiles
cudaError_t launch_step_fused3_red(lbmp_handle* h);    // FP32 D3Q27 flow, D3Q7 phase field, 32 x 4 tiles
// the observables' partial sums of an FP32 D3Q27 domain (full / reduced phase
// lattice) in one march: [4 k] of *nparts <= max_parts CTAs, and phi on the
// spike and bubble columns into cols (or null)
cudaError_t launch_obs_fused3(lbmp_handle* h, double* part, int max_parts, int* nparts, double* cols);
cudaError_t launch_obs_fused3_red(lbmp_handle* h, double* part, int max_parts, int* nparts, double* cols);
cudaError_t launch_init(lbmp_handle* h, int case_id, const double* args, int nargs, unsigned long long seed);
cudaError_t launch_set_state(lbmp_handle* h, const double* dev_f, const double* dev_g);
cudaError_t launch_get_state(lbmp_handle* h, double* dev_f, double* dev_g);
// dev_out: [0..3] mass, kinetic energy, max|u|, non-finite count; [4..5] probe
// pressures; [16..16+2nv) phi on the spike and bubble columns
cudaError_t launch_observables(lbmp_handle* h, double* dev_out);
cudaError_t launch_mass(lbmp_handle* h, double* dev_out4);  // writes 4 doubles, [0] = mass
bool fused_supported(const lbmp_handle* h);
// batch kernel of one tile shape of the FP32 D3Q27 fused step
struct Batch3Ops {
    int tile_x, tile_y;
    // attributes, and the resident CTAs per SM of the kernel (not capturable)
    cudaError_t (*prepare)(int device, int& per_sm);
    // persistent form (null where a kind has the member-grid form): the
    // members' work items walked by one grid, members read from the device table
    cudaError_t (*launch)(const BatchDomain* table, int ndom, int nitems, int device, cudaStream_t stream);
    // member-grid form (null where a kind has none): members [0, n) of the
    // host table `host` passed as kernel parameters, each with its population
    // sets for the parity host[k].parity ^ flip; blockIdx.y selects the member,
    // whose steps_left the kernel reads from the device table `dev`.  At most
    // grid_members members per launch.
    cudaError_t (*launch_grid)(const BatchDomain* host, const BatchDomain* dev, int n, int flip, int device,
                               cudaStream_t stream);
    int grid_members;
};
extern const Batch3Ops batch3_ops_32x4, batch3_ops_16x8, batch3_ops_8x16;
extern const Batch3Ops batch3_ops_f16, batch3_ops_bf16;  // shifted 16-bit members (32 x 4 tiles)
extern const Batch3Ops batch3_ops_red;                    // FP32 members with the D3Q7 phase field
extern const Batch3Ops batch2_ops_f16, batch2_ops_bf16;  // shifted 16-bit D2Q9 members (128-cell rows)
cudaError_t launch_step_fused2s(lbmp_handle* h);         // shifted 16-bit storage, D2Q9
inline const Batch3Ops& batch3_ops(int tile)
{
    return tile == 1 ? batch3_ops_16x8 : (tile == 2 ? batch3_ops_8x16 : batch3_ops_32x4);
}
cudaError_t launch_step_fused2(lbmp_handle* h);
cudaError_t launch_step_aa(lbmp_handle* h);  // in-place AA storage: phi pass, then the AA step of the phase
// keep dp.aa in step with the phase after every change of parity
inline void sync_aa(lbmp_handle* h)
{
    if (h->aa) h->dp.aa = 1 + h->parity;
}
cudaError_t launch_step_fused16(lbmp_handle* h);  // shifted 16-bit storage, D3Q27
bool bulk_supported(const lbmp_handle* h);         // FP32 D3Q27 with nx % 4 == 0
cudaError_t launch_step_fused_bulk(lbmp_handle* h);
// the step kernel(s) selected by LBMP_OPT_KERNEL for this handle (no parity flip)
cudaError_t launch_step(lbmp_handle* h);
int batch2_tile_x();
cudaError_t prepare_batch2(int device, bool reduced, bool sym, int& per_sm);  // reduced: D2Q5 phase field; sym: x symmetry axis
cudaError_t launch_batch2(const BatchDomain* table, int ndom, int nitems, int device, cudaStream_t stream,
                          bool reduced, bool sym);
cudaError_t launch_batch_epilogue(BatchDomain* table, int ndom, cudaStream_t stream);
// record a message for lbmp_last_error() and return code
int set_error(int code, const char* msg);

}  // namespace lbmp
