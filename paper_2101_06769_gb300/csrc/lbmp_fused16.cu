// lbmp_fused16.cu -- the fused D3Q27 step for the shifted 16-bit storage
// forms (FP16 or BF16 codes plus one FP32 reference per cell, layout in
// lbmp_common.cuh).
//
// Work decomposition, summation orders and per-cell arithmetic are those of
// the FP32 fused kernel (lbmp_fused.cu); what differs is the decoding of the
// pulled values and the encoding of the outputs:
//   * a pulled value needs its 16-bit code and the reference R of the cell
//     that wrote it.  The references of the planes around the marching plane
//     are staged in shared memory, four planes per population set in
//     rotation, one new plane per step: g over the tile plus two rings (a ring
//     cell's phi pulls from one cell further out), f' over the tile plus one
//     ring.  Offsets of the staged plane cells are computed once per segment.
//   * the 16-bit codes of the own and ring cells' g(z+1) and of f'(z) are loaded
//     to registers (2-byte loads) and decoded when the reference planes are in
//     place; the own cells' decoded g is kept in shared memory for the collision
//     one plane later.
//   * the ghost plane beyond a wall (mirrored phi, reading A17) is a copy of
//     the wall plane's phi instead of a second staging of that plane.
// What bounds it: instruction issue (58 % of the slots; every value is decoded
// and encoded; DRAM stands at a quarter of its rate) and the instruction cache,
// the first of its stalls.  128^3 FP16 issues 2741 instructions per cell (3553
// when g codes were staged as 32-bit words, the two population sets were emitted
// in two passes, divisions were the compiler's and items had 8 planes).
// 128x128x512 RT workload, FP16 / BF16: 1.00 / 0.99 ms per step; 1.05 / 1.03
// with a second barrier per plane (three phi planes in rotation); 1.21 / 1.18
// before all of these.  The ring's codes loaded beside the others spill (480 B)
// wherever their decoding is put: 1.09-1.14; one decoding loop run over the own
// and the ring cell, 500 instructions of code less, 1.02; four CTAs per SM (500 B
// of spills) 1.12.
#define LBMP_TILE_NS tile16
#ifndef LBMP_FUSED_BYTEOFF
#define LBMP_FUSED_BYTEOFF 2
#endif
#include <stdint.h>

#include "lbmp_repro.cuh"
#include "lbmp_internal.h"
#include "lbmp_tile.cuh"

namespace lbmp {

namespace {

using namespace LBMP_TILE_NS;

// the encoder of one cell's outputs at a cell offset of the tile geometry: the
// codes at base + offset, the reference at its 4-byte slot
template <class St>
struct EncCell {
    static constexpr bool kTotal = true;
    unsigned short* const* qb;
    float* R;
    cell_off self;
    float off;
    mutable float sq;
    unsigned seed;  // code_seed of the writer cell (stochastic rounding)
    __device__ __forceinline__ void pair(int a, float2 v) const
    {
        unsigned short ca, cb;
        encode_pair<3, St>(a, v, off, seed, sq, ca, cb);
        *at_cell(qb[a], self) = ca;
        *at_cell(qb[26 - a], self) = cb;
    }
    __device__ __forceinline__ void finish(float th, float tl) const
    {
        R[elem_index(self)] = ref_from_total<3>(th, tl, sq);
    }
};

constexpr int C3 = 13;
constexpr int GX = TX + 4, GY = TY + 4, GPLANE = GX * GY;  // g reference plane: tile + two rings
constexpr size_t kSmem16 = sizeof(float2) * 4 * PLANE + sizeof(float) * (2 * Q3 * NT + 4 * GPLANE + 4 * PLANE) +
                           sizeof(int) * (GPLANE + PLANE);

struct DirPtrs16 {
    const unsigned short* fin[Q3];  // per-direction code arrays; entry C3 unused
    const unsigned short* gin[Q3];
    unsigned short* fout[Q3];
    unsigned short* gout[Q3];
    const float* rfin;  // references
    const float* rgin;
    float* rfout;
    float* rgout;
};

constexpr MarchCost kCost = {6.0, 1.25, 0.0};

struct FusedArgs16 {
    int tiles_x, tiles_y, chunk, nitems;
};

__device__ __forceinline__ bool ghost_plane(const DevParams& p, int zz)
{
    return !p.vert_periodic && (zz < 0 || zz >= p.nz);
}

// reference plane k (logical index; periodic wrap) into rotation slot k & 3;
// planes beyond a wall are never read (their populations bounce) and are skipped
__device__ __forceinline__ void load_ref_plane(const DevParams& p, const float* src, int k, float* planes, int size,
                                               const int* off, int tid)
{
    int zk = k;
    if (k < 0 || k >= p.nz) {
        if (!p.vert_periodic) return;
        zk = pmod(k, p.nz);
    }
    const float* base = src + zk * (p.nx * p.ny);
    float* d = planes + ((k + 8) & 3) * size;
    for (int e = tid; e < size; e += NT) cp_async4(d + e, base + off[e]);
}

template <bool Walls>
struct CodeLoad {
    const unsigned short* const* base;
    const Column& C;
    const Plane& P;
    unsigned short* q;
    template <int a>
    __device__ __forceinline__ void step() const
    {
        if constexpr (a != C3) q[a] = *pulled<Walls, a>(base, C, P);
    }
};

// pulled codes of one cell to registers
__device__ __forceinline__ void load_codes(const unsigned short* const* base, const Column& C, const Plane& P_,
                                           unsigned short* q)
{
    if (P_.lo || P_.hi)  // uniform across the CTA
        Unroll<Q3>::run(CodeLoad<true>{base, C, P_, q});
    else
        Unroll<Q3>::run(CodeLoad<false>{base, C, P_, q});
}

// references of the writers of the pulled pair (a, opp(a)): slot is the cell's
// index in the reference-plane layout of row length RL, Rm / R0 / Rp the
// planes below, at and above the cell
template <bool Walls>
__device__ __forceinline__ float2 pair_refs(int a, const float* Rm, const float* R0, const float* Rp, int slot, int RL,
                                            bool lo, bool hi)
{
    const int cx = Lat<3>::cx(a), cy = Lat<3>::cy(a), cz = Lat<3>::cz(a);
    const auto ref = [&](int sx, int sy, int sz) {  // writer x - (sx, sy, sz)
        if (Walls && ((sz == 1 && lo) || (sz == -1 && hi))) return R0[slot];
        return (sz == 1 ? Rm : (sz == -1 ? Rp : R0))[slot - sx - sy * RL];
    };
    return f2(ref(cx, cy, cz), ref(-cx, -cy, -cz));
}

// Decode the codes q of one cell's g and sum phi (hi, lo) from the exact
// parts of the values (phi_sum_shifted); Keep: also store the decoded values
// at buf[a * stride] (the tile's own cells, whose values the collision reads;
// ring cells need phi only).
template <bool Walls, class St, bool Keep>
__device__ __forceinline__ float2 decode_g(const unsigned short* q, const float* Rm, const float* R0, const float* Rp,
                                           int slot, bool lo, bool hi, float* buf, int stride)
{
    float2 phi;
    phi_sum_shifted<3>(
        [&]() {
            const float v = wint<3>(C3) * R0[slot];
            if (Keep) buf[C3 * stride] = v;
            return v;
        },
        [&](int a, float2& wr, float2& wq) {
            const int b = Q3 - 1 - a;
            const float2 R = pair_refs<Walls>(a, Rm, R0, Rp, slot, GX, lo, hi);
            const float2 qv = f2(St::dec(q[a]), St::dec(q[b]));
            decode_pair<3, St>(a, R, qv, wr, wq);
            if (Keep) {
                const float2 v = decode_pair<3, St>(a, R, qv);  // = wr + wq, rounded once
                buf[a * stride] = v.x;
                buf[b * stride] = v.y;
            }
        },
        phi.x, phi.y);
    return phi;
}

template <class St>
struct Seg16 {
    const DevParams& p;
    const DirPtrs16& D;
    const ThreadGeo& T;
    const Column& own;
    const Column& ring;
    float* RG;
    float* RF;
    const int* offG;
    const int* offF;

    // reference planes zz+2 (g) and zz+1 (f') into their rotation slots
    __device__ __forceinline__ void issue_refs(int zz) const
    {
        load_ref_plane(p, D.rgin, zz + 2, RG, GPLANE, offG, T.tid);
        load_ref_plane(p, D.rfin, zz + 1, RF, PLANE, offF, T.tid);
        cp_async_commit();
    }

    // codes of plane zz of the own cell
    __device__ __forceinline__ void load_g(int zz, unsigned short* qo) const
    {
        if (ghost_plane(p, zz)) return;
        Plane P;
        set_plane(P, p, plane_src(p, zz));
        load_codes(D.gin, own, P, qo);
    }

    // decode plane zz (unless a ghost) and write its phi; the ring cells' codes
    // are loaded here (with the own and f' codes they would spill)
    template <bool Walls>
    __device__ __forceinline__ void phi_of(int zz, bool lo, bool hi, const unsigned short* qo, float* gbuf,
                                           float2* phi_plane) const
    {
        const float* Rm = RG + ((zz + 7) & 3) * GPLANE;
        const float* R0 = RG + ((zz + 8) & 3) * GPLANE;
        const float* Rp = RG + ((zz + 9) & 3) * GPLANE;
        if (T.tid < NRING) {
            Plane P;
            set_plane(P, p, plane_src(p, zz));
            unsigned short qr[Q3];
            load_codes(D.gin, ring, P, qr);
            phi_plane[T.rslot] =
                decode_g<Walls, St, false>(qr, Rm, R0, Rp, (T.ly + 2) * GX + T.lx + 2, lo, hi, nullptr, 0);
        }
        phi_plane[T.oslot] =
            decode_g<Walls, St, true>(qo, Rm, R0, Rp, (T.ty + 2) * GX + T.tx + 2, lo, hi, gbuf + T.tid, NT);
    }
    __device__ __forceinline__ void finish(int zz, const unsigned short* qo, float* gbuf, float2* phi_plane) const
    {
        if (ghost_plane(p, zz)) return;
        const int pz = plane_src(p, zz);
        const bool lo = !p.vert_periodic && pz == 0, hi = !p.vert_periodic && pz == p.nz - 1;
        if (lo || hi)
            phi_of<true>(zz, lo, hi, qo, gbuf, phi_plane);
        else
            phi_of<false>(zz, false, false, qo, gbuf, phi_plane);
    }

    // phi of the ghost plane = phi of the wall plane (each thread copies the
    // slots it wrote itself)
    __device__ __forceinline__ void copy_phi(const float2* from, float2* to) const
    {
        if (T.tid < NRING) to[T.rslot] = from[T.rslot];
        to[T.oslot] = from[T.oslot];
    }

    // decoded f' of plane z from its codes and the reference planes
    template <bool Walls>
    __device__ __forceinline__ void decode_f(int z, bool lo, bool hi, const unsigned short* q, float* fr) const
    {
        const float* Rm = RF + ((z + 7) & 3) * PLANE;
        const float* R0 = RF + ((z + 8) & 3) * PLANE;
        const float* Rp = RF + ((z + 9) & 3) * PLANE;
        fr[C3] = wint<3>(C3) * R0[T.oslot];
#pragma unroll
        for (int a = 0; a < C3; ++a) {
            const int b = Q3 - 1 - a;
            const float2 R = pair_refs<Walls>(a, Rm, R0, Rp, T.oslot, RX, lo, hi);
            const float2 v = decode_pair<3, St>(a, R, f2(St::dec(q[a]), St::dec(q[b])));
            fr[a] = v.x;
            fr[b] = v.y;
        }
    }
};

template <class St>
__device__ __forceinline__ void fused_segment16(const DevParams& p, const DirPtrs16& Dp, const ThreadGeo& T,
                                                float* smem, int x0, int y0, int z0, int z1)
{
    float2* phiS = (float2*)smem;                // (hi, lo) [4][PLANE]
    float* gS = (float*)(phiS + 4 * PLANE);      // [2][27][NT] decoded own g
    float* RG = gS + 2 * Q3 * NT;                // [4][GPLANE] g references
    float* RF = RG + 4 * GPLANE;                 // [4][PLANE] f' references
    int* offG = (int*)(RF + 4 * PLANE);
    int* offF = offG + GPLANE;
    const int tid = T.tid;
    Column own, ring;
    set_column(own, p, pmod(x0 + T.tx, p.nx), pmod(y0 + T.ty, p.ny));
    set_column(ring, p, pmod(x0 + T.lx, p.nx), pmod(y0 + T.ly, p.ny));
    const bool valid = (x0 + T.tx < p.nx) && (y0 + T.ty < p.ny);
    for (int e = tid; e < GPLANE; e += NT)
        offG[e] = pmod(y0 + e / GX - 2, p.ny) * p.nx + pmod(x0 + e % GX - 2, p.nx);
    for (int e = tid; e < PLANE; e += NT) offF[e] = pmod(y0 + e / RX - 1, p.ny) * p.nx + pmod(x0 + e % RX - 1, p.nx);
    __syncthreads();
    const Seg16<St> S{p, Dp, T, own, ring, RG, RF, offG, offF};
    unsigned short qo[Q3];
    // reference planes needed before the first two stagings
    load_ref_plane(p, Dp.rgin, z0 - 2, RG, GPLANE, offG, tid);
    load_ref_plane(p, Dp.rgin, z0 - 1, RG, GPLANE, offG, tid);
    load_ref_plane(p, Dp.rgin, z0, RG, GPLANE, offG, tid);
    load_ref_plane(p, Dp.rfin, z0 - 1, RF, PLANE, offF, tid);
    // One barrier per plane: phi and the references have four planes in rotation,
    // so what a thread that has passed the barrier of plane z writes for plane
    // z+2 is what no thread reads any more after that barrier.
    const auto phi_at = [&](int zz) { return phiS + ((zz - z0 + 1) & 3) * PLANE; };
#pragma unroll 1
    for (int k = 0; k < 2; ++k) {  // planes z0 - 1 and z0
        S.load_g(z0 - 1 + k, qo);
        cp_async_commit();
        cp_async_wait_all();
        __syncthreads();
        S.finish(z0 - 1 + k, qo, gS + (k ^ 1) * Q3 * NT, phi_at(z0 - 1 + k));
        S.issue_refs(z0 - 1 + k);
    }
    cp_async_wait_all();
    if (ghost_plane(p, z0 - 1)) S.copy_phi(phi_at(z0), phi_at(z0 - 1));
    __syncthreads();
    for (int z = z0; z < z1; ++z) {
        const int cur = (z - z0) & 1;
        // the codes of g(z+1) and f'(z) and the next reference planes in flight together
        S.issue_refs(z + 1);
        S.load_g(z + 1, qo);
        Plane P;
        set_plane(P, p, z);
        repro::FlowMoments m;
        {
            unsigned short q[Q3];
            load_codes(Dp.fin, own, P, q);
            S.finish(z + 1, qo, gS + (cur ^ 1) * Q3 * NT, phi_at(z + 1));
            if (ghost_plane(p, z + 1)) S.copy_phi(phi_at(z), phi_at(z + 1));
            float fr[Q3];
            if (P.lo || P.hi)
                S.template decode_f<true>(z, P.lo, P.hi, q, fr);
            else
                S.template decode_f<false>(z, false, false, q, fr);
            repro::flow_moments<3>(m, fr);
        }
        cp_async_wait_all();
        __syncthreads();
        if (valid) {
            const float2* pm = phi_at(z - 1) + T.oslot;
            const float2* pc = phi_at(z) + T.oslot;
            const float2* pn = phi_at(z + 1) + T.oslot;
            const float2 centre = pc[0];
            float grad[3], lap, inv_rho, nu, dh[27];
            repro::stencil_from<3>(
                [&](int a) {
                    const int cz = Lat<3>::cz(a);
                    return (cz < 0 ? pm : (cz == 0 ? pc : pn))[Lat<3>::cy(a) * RX + Lat<3>::cx(a)];
                },
                centre, grad, lap);
            repro::CellState s;
            repro::flow_closure<3>(p, centre.x, grad, lap, m, s, inv_rho, nu);
            repro::flow_relax<3>(m, s, inv_rho, nu, dh);
            const cell_off self = P.zs[1] + own.ys[1] + own.xs[1];
            const GFromStrided gin{gS + cur * Q3 * NT + tid, NT};  // this cell's decoded pre-collision g
            float off_f, off_g;
            repro::rest_offsets<3, St>(p, s, dh, gin, off_f, off_g);
            repro::collide_outputs<3>(
                p, s, repro::DhArray{dh}, m, gin, centre.x, centre.y,
                EncCell<St>{Dp.fout, Dp.rfout, self, off_f, 0.f, code_seed(p, elem_index(self), 0)},
                EncCell<St>{Dp.gout, Dp.rgout, self, off_g, 0.f, code_seed(p, elem_index(self), 1)});
        }
    }
    __syncthreads();  // the caller may reuse shared memory
}

template <class St>
__global__ void __launch_bounds__(NT, LBMP_FUSED_MINB) step_fused3s_kernel(DevParams p, FusedArgs16 A, DirPtrs16 Dp)
{
    extern __shared__ __align__(16) float smem16[];
    const ThreadGeo T = thread_geo();
    for (int item = blockIdx.x + after_previous(); item < A.nitems; item += gridDim.x) {
        const int tile = item % (A.tiles_x * A.tiles_y);
        const int chunk = item / (A.tiles_x * A.tiles_y);
        const int z0 = chunk * A.chunk;
        fused_segment16<St>(p, Dp, T, smem16, (tile % A.tiles_x) * TX, (tile / A.tiles_x) * TY, z0,
                            min(z0 + A.chunk, p.nz));
    }
}

// Batch form (FP16 / BF16 members of a batch): as the FP32 batch kernel, a
// CTA looks up the member of each work item in the device table and stages
// its parameters and direction bases in shared memory.
template <class St>
__global__ void __launch_bounds__(NT, LBMP_FUSED_MINB) step_batch3s_kernel(const BatchDomain* __restrict__ table,
                                                                           int ndom, int nitems)
{
    extern __shared__ __align__(16) float smem16[];
    __shared__ DevParams sp;
    __shared__ DirPtrs16 sd;
    __shared__ int s_dom, s_tx, s_ty, s_chunk, s_begin, s_active;
    const ThreadGeo T = thread_geo();
    int cur = -1;
    for (int item = blockIdx.x; item < nitems; item += gridDim.x) {
        __syncthreads();  // every thread has read the previous item's shared values
        if (threadIdx.x == 0) {
            int lo = 0, hi = ndom - 1;  // last member with item_begin <= item
            while (lo < hi) {
                const int mid = (lo + hi + 1) >> 1;
                if (table[mid].item_begin <= item)
                    lo = mid;
                else
                    hi = mid - 1;
            }
            s_dom = lo;
        }
        __syncthreads();
        const int d = s_dom;
        if (d != cur) {
            const BatchDomain& B = table[d];
            const int par = B.parity;
            const size_t N = (size_t)B.p.N;
            if (threadIdx.x == 0) {
                sp = B.p;
                s_tx = B.tiles_x;
                s_ty = B.tiles_y;
                s_chunk = B.chunk;
                s_begin = B.item_begin;
                s_active = B.steps_left > 0;
                sd.rfin = B.f[par];
                sd.rgin = B.g[par];
                sd.rfout = B.f[par ^ 1];
                sd.rgout = B.g[par ^ 1];
            }
            for (int k = threadIdx.x; k < 4 * Q3; k += blockDim.x) {
                const int set = k / Q3, a = k % Q3;
                const size_t off = (size_t)(a - (a > C3)) * N;
                unsigned short* base = (unsigned short*)((set == 0 || set == 2 ? B.f : B.g)[set < 2 ? par : par ^ 1] + N);
                unsigned short* q = a != C3 ? base + off : nullptr;
                if (set == 0) sd.fin[a] = q;
                if (set == 1) sd.gin[a] = q;
                if (set == 2) sd.fout[a] = q;
                if (set == 3) sd.gout[a] = q;
            }
            cur = d;
            __syncthreads();
        }
        if (!s_active) continue;  // uniform
        const int local = item - s_begin;
        const int tiles = s_tx * s_ty;
        const int tile = local % tiles;
        const int z0 = (local / tiles) * s_chunk;
        fused_segment16<St>(sp, sd, T, smem16, (tile % s_tx) * TX, (tile / s_tx) * TY, z0, min(z0 + s_chunk, sp.nz));
    }
}

template <class St>
struct BatchCfg16 {
    static int dev, cap, ctas;
    static cudaError_t prepare(int device, int& per_sm_out)
    {
        if (dev != device) {
            cudaError_t e = cudaFuncSetAttribute(step_batch3s_kernel<St>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                 (int)kSmem16);
            if (e != cudaSuccess) return e;
            int per_sm = 0, sms = 0;
            e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, step_batch3s_kernel<St>, NT, kSmem16);
            if (e != cudaSuccess) return e;
            e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device);
            if (e != cudaSuccess) return e;
            ctas = per_sm > 0 ? per_sm : 1;
            cap = ctas * sms;
            dev = device;
        }
        per_sm_out = ctas;
        return cudaSuccess;
    }
    static cudaError_t launch(const BatchDomain* table, int ndom, int nitems, int device, cudaStream_t stream)
    {
        if (dev != device) return cudaErrorNotReady;  // prepare first
        if (nitems <= 0) return cudaSuccess;
        const int grid = nitems < cap ? nitems : cap;
        step_batch3s_kernel<St><<<grid, NT, kSmem16, stream>>>(table, ndom, nitems);
        return cudaGetLastError();
    }
};
template <class St>
int BatchCfg16<St>::dev = -1;
template <class St>
int BatchCfg16<St>::cap = 0;
template <class St>
int BatchCfg16<St>::ctas = 0;

struct Cfg16 {
    int device = -1;
    int per_sm = 0, sms = 0;
};

template <class St>
cudaError_t launch16(lbmp_handle* h, Cfg16& cfg)
{
    if (cfg.device != h->device) {
        cudaError_t e = cudaFuncSetAttribute(step_fused3s_kernel<St>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)kSmem16);
        if (e != cudaSuccess) return e;
        int per_sm = 0, sms = 0;
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, step_fused3s_kernel<St>, NT, kSmem16);
        if (e != cudaSuccess) return e;
        e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, h->device);
        if (e != cudaSuccess) return e;
        cfg.per_sm = per_sm > 0 ? per_sm : 1;
        cfg.sms = sms;
        cfg.device = h->device;
    }
    DirPtrs16 D;
    const int s = h->parity, d = 1 - h->parity;
    const size_t N = (size_t)h->N;
    const unsigned short* cf = (const unsigned short*)(h->f[s] + N);
    const unsigned short* cg = (const unsigned short*)(h->g[s] + N);
    unsigned short* of = (unsigned short*)(h->f[d] + N);
    unsigned short* og = (unsigned short*)(h->g[d] + N);
    for (int a = 0; a < Q3; ++a) {
        const size_t off = (size_t)(a - (a > C3)) * N;
        const bool mv = a != C3;
        D.fin[a] = mv ? cf + off : nullptr;
        D.gin[a] = mv ? cg + off : nullptr;
        D.fout[a] = mv ? of + off : nullptr;
        D.gout[a] = mv ? og + off : nullptr;
    }
    D.rfin = h->f[s];
    D.rgin = h->g[s];
    D.rfout = h->f[d];
    D.rgout = h->g[d];
    FusedArgs16 A;
    A.tiles_x = (h->grid.nx + TX - 1) / TX;
    A.tiles_y = (h->grid.ny + TY - 1) / TY;
    const LaunchShape L = launch_shape(h, kCost, A.tiles_x * A.tiles_y, h->grid.nz, cfg.per_sm, cfg.sms);
    A.chunk = L.chunk;
    A.nitems = L.nitems;
    return launch_after(step_fused3s_kernel<St>, L, NT, kSmem16, h->stream, h->dp, A, D);
}

Cfg16 g_cfg_f16, g_cfg_bf16;

}  // namespace

const Batch3Ops batch3_ops_f16 = {TX, TY, BatchCfg16<StoreF16>::prepare, BatchCfg16<StoreF16>::launch, nullptr, 0};
const Batch3Ops batch3_ops_bf16 = {TX, TY, BatchCfg16<StoreBF16>::prepare, BatchCfg16<StoreBF16>::launch, nullptr, 0};

cudaError_t launch_step_fused16(lbmp_handle* h)
{
    if (h->D != 3 || (h->grid.nx & 1)) return cudaErrorInvalidValue;
    if (h->params.storage == LBMP_FP16_SHIFTED) return launch16<StoreF16>(h, g_cfg_f16);
    if (h->params.storage == LBMP_BF16_SHIFTED) return launch16<StoreBF16>(h, g_cfg_bf16);
    return cudaErrorInvalidValue;
}

}  // namespace lbmp
