// lb_tma.cu -- the FP32 one-pass time step with each tile's populations and
// reference densities, halo included, brought into shared memory by the
// tensor memory accelerator (cp.async.bulk.tensor, completion on an mbarrier)
// instead of per-thread loads.  The explicit FP32 arithmetic of lb_vops.cuh,
// in the same order as fused_tile, so the results are the same bit for bit:
// the densities of the staged nodes are the sums of Eq. (6) over the boxed
// populations, then the forces of Eqs. (8), (9), the collision of Eqs. (1),
// (2), (5) and the push streaming of collide_site.
//
// Box of a tile (x0, y0) of 32 x TY nodes: columns x0 - 4 .. x0 + 35 (the
// D2Q25 halo needs 2; 4 keep the x offset a multiple of 16 bytes), rows
// y0 - 2 .. y0 + TY + 1, all 18 population planes; a second box holds the 2
// reference-density planes.  Parts of the box beyond the lattice are filled
// with zeros by the copy and not used: the halo slots there (across a
// periodic edge, or wall ghost rows) are formed as in fused_tile.  The
// tiles that tma_box_tile rejects (lattices smaller than the box) run as plain
// one-pass tiles: of the same launch where a list holds both kinds, of k_fused
// where it holds no other.
#include "lb_kernels.cuh"
#include "lb_launch.h"

namespace lbk {

namespace {

template <int TYv>
struct TmaBox {
    static constexpr int H = TYv + 2 * HALO;
    static constexpr int kPop = kTmaBoxW * H * 18;   // floats
    static constexpr int kRef = kTmaBoxW * H * 2;
    static constexpr int kStage = kPop + kRef;
    static constexpr unsigned kBytes = (unsigned)kStage * 4u;
    static_assert((kPop * 4) % 128 == 0 && (kStage * 4) % 128 == 0, "stage buffers stay 128-byte aligned");
};

// Resident blocks per SM the kernel is compiled for: as the plain one-pass
// kernel, unless the staging buffer leaves room for fewer.
template <int TYv>
constexpr int kTmaMinBlocks = (225 * 1024) / (TmaBox<TYv>::kBytes + 8 * 1024) < kCollideMinBlocks<float, TYv>
                                  ? (225 * 1024) / (TmaBox<TYv>::kBytes + 8 * 1024)
                                  : kCollideMinBlocks<float, TYv>;

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t *bar, unsigned count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t *bar, unsigned bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, unsigned phase)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(phase)
        : "memory");
    return ok != 0;
}

// Bounded wait for the completion of phase `phase` of *bar.
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, unsigned phase, long long limit)
{
    const long long start = clock64();
    while (!mbar_try_wait(bar, phase))
        if (clock64() - start > limit) return false;
    return true;
}

// Bring the box at (x, y, z) of the tensor into L2 (no shared memory, no
// completion to wait for).
__device__ __forceinline__ void tma_prefetch_3d(const CUtensorMap *map, int x, int y, int z)
{
    asm volatile("cp.async.bulk.prefetch.tensor.3d.L2.global.tile [%0, {%1, %2, %3}];" ::"l"(map), "r"(x), "r"(y), "r"(z)
                 : "memory");
}

__device__ __forceinline__ void tma_load_3d(void *dst, const CUtensorMap *map, int x, int y, int z, uint64_t *bar)
{
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
        ::"r"(smem_u32(dst)), "l"(map), "r"(x), "r"(y), "r"(z), "r"(smem_u32(bar))
        : "memory");
}

// The slot's node lies beyond the lattice (across a periodic edge, or a wall
// ghost row): not in the box's lattice part.
__device__ __forceinline__ bool slot_outside(const Lat<float> &G, int4 t, int sx, int sy)
{
    const int gx = t.y + sx - HALO, gy = t.z + sy - HALO;
    return gx < 0 || gx >= G.nx || gy < 0 || gy >= G.ny;
}

// fused_tile with the tile's and the halo's populations and reference
// densities read from the box (pop: [18][H][40], ref: [2][H][40]).  Slots beyond
// the lattice (of the halo, and of a ragged tile's missing nodes) were staged
// by the caller.
template <int TYv>
__device__ __forceinline__ void fused_tile_box(const Lat<float> *__restrict__ lats, int4 t, int parity,
                                               CollideSmem<TYv> &sm, const float *__restrict__ pop,
                                               const float *__restrict__ ref)
{
    constexpr int SHv = TYv + 2 * HALO, H = SHv, W = kTmaBoxW;
    const Lat<float> &G = lats[t.x];
    const int tid = threadIdx.y * TX + threadIdx.x;
    for (int i = tid; i < (int)(sizeof(Lat<float>) / 4); i += TX * TYv)
        reinterpret_cast<uint32_t *>(&sm.L)[i] = reinterpret_cast<const uint32_t *>(&G)[i];
    // staged slot (sx, sy) is box column sx + 2, row sy; its densities are
    // the sums of node_density.  The node's own density and force-free moments from one read of its
    // populations, then the densities of the halo ring
    const int x = t.y + threadIdx.x, y = t.z + threadIdx.y;
    const int cx = threadIdx.x + HALO, cy = threadIdx.y + HALO;
    const size_t c = (size_t)y * G.pitch + x;
    // the node's own populations stay in the box: collide_site reads them there
    const float *own = pop + cy * W + cx + 2;
    float fk[2][9], Rn[2];
    NodeMoments nm;
    const bool valid = x < G.nx && y < G.ny;
    if (valid) {
        float2 v[9];
#pragma unroll
        for (int i = 0; i < 9; ++i) v[i] = make_float2(own[i * H * W], own[(9 + i) * H * W]);
        const float2 R2 = make_float2(ref[cy * W + cx + 2], ref[(H + cy) * W + cx + 2]);
        const float2 rn = vadd(R2, vzeroth<float2>(v));
        Rn[0] = R2.x;
        Rn[1] = R2.y;
        G.rho[parity ^ 1][c] = rn.x;
        G.rho[parity ^ 1][G.plane + c] = rn.y;
        sm.sr[cy][cx] = rn;
        sm.sp[cy][cx] = make_float2(psi_of<float>(rn.x), psi_of<float>(rn.y));
        node_moments(v, rn, R2, nm);
    }
    // both species' densities of a ring slot
    auto slot_density = [&](int sx, int sy) {
        float2 v[9];
#pragma unroll
        for (int i = 0; i < 9; ++i)
            v[i] = make_float2(pop[(i * H + sy) * W + sx + 2], pop[((9 + i) * H + sy) * W + sx + 2]);
        return vadd(make_float2(ref[sy * W + sx + 2], ref[(H + sy) * W + sx + 2]), vzeroth<float2>(v));
    };
    for (int h = tid; h < kRing<TYv>; h += TX * TYv) {
        int sx, sy;
        ring_slot<TYv>(h, sx, sy);
        if (slot_outside(G, t, sx, sy)) continue;
        const float2 r = slot_density(sx, sy);
        sm.sr[sy][sx] = r;
        sm.sp[sy][sx] = make_float2(psi_of<float>(r.x), psi_of<float>(r.y));
    }
    __syncthreads();
    if (!valid) return;
    const bool inner = t.y >= 1 && t.y + TX + 1 <= sm.L.nx && t.z >= 1 && t.z + TYv + 1 <= sm.L.ny;
    const PairStage<SHv> sg{sm.sr, sm.sp};
    if (inner) collide_site<true, true>(sm.L, G.f[parity ^ 1], sg, fk, Rn, x, y, cx, cy, own, H * W, &nm);
    else collide_site<false, true>(sm.L, G.f[parity ^ 1], sg, fk, Rn, x, y, cx, cy, own, H * W, &nm);
}

// A tile of a lattice smaller than the box: the plain one-pass tile, staged in the box's shared memory.  Out of line, so
// that it does not shape the box tiles' registers.
template <int TYv>
__device__ __noinline__ void plain_tile(const Lat<float> *__restrict__ lats, int4 t, int parity, float *box)
{
    static_assert(sizeof(CollideSmem<TYv>) <= TmaBox<TYv>::kBytes, "staged in the box");
    fused_tile<TYv, false>(lats, t, parity, *reinterpret_cast<CollideSmem<TYv> *>(box));
}

// One block per tile: thread 0 starts the two copies, every thread waits
// (bounded) on the mbarrier, then the tile is computed from the box.  (With
// ragged tiles in a second launch 28 lattices of 220^2 took 70 us a step, 1000^2
// 48.4, 333 x 97 11.6; as plain tiles of the one launch 64, 42.9, 7.1; boxed 57,
// 41.5, 6.6.)  kMixed: tiles without the mark run as plain_tile.  The call costs
// registers (height 2: 94 a thread against 72, 4: 78 against 72, 8: 64 both), so
// at heights 2 and 4 a list of boxes alone takes the form without it (512^2 in
// tiles of 4: 14.8 and 14.0 us a step; 1000^2 in tiles of 8: 40.2 with, 41.3
// without).
template <int TYv, bool kMixed>
__global__ void __launch_bounds__(TX *TYv, kTmaMinBlocks<TYv>)
    k_fused_tma(const Lat<float> *__restrict__ lats, const int4 *__restrict__ tiles, int tile_offset, int parity,
                const TmaMaps *__restrict__ maps, int *err, long long wait_cycles, int drop_tile, int n_tiles,
                int ahead, int wave)
{
    using B = TmaBox<TYv>;
    constexpr int ti = TYv == 2 ? 0 : (TYv == 4 ? 1 : 2);
    extern __shared__ __align__(128) float box[];
    __shared__ __align__(8) uint64_t bar;
    __shared__ CollideSmem<TYv> sm;
    // the mark: the tile's lattice holds a whole box (so its maps exist), as the host found when it sorted the list (tma_box_tile),
    // which keeps the lattice's descriptor off the way to the copy
    const int4 t = tiles[tile_offset + blockIdx.x];
    if constexpr (kMixed)
        if (t.w != kTmaBoxMark) {
            plain_tile<TYv>(lats, t, parity, box);
            return;
        }
    const int tid = threadIdx.y * TX + threadIdx.x;
    // the boxes of the tile `ahead` blocks later (about one wave of resident
    // blocks) into L2, so that its copies find them there; a block of the
    // first wave issues it once its own box has landed, so that it does not
    // compete with the first wave's own copies
    const bool first_wave = (int)blockIdx.x < wave;
    auto prefetch_ahead = [&]() {
        if (ahead > 0 && (int)blockIdx.x + ahead < n_tiles) {
            const int4 tn = tiles[tile_offset + blockIdx.x + ahead];
            if (!kMixed || tn.w == kTmaBoxMark) {
                tma_prefetch_3d(&maps[tn.x].pop[ti][parity], tn.y - 4, tn.z - HALO, 0);
                tma_prefetch_3d(&maps[tn.x].ref[ti][parity], tn.y - 4, tn.z - HALO, 0);
            }
        }
    };
    // the copy of drop_tile (a test hook) is never started: its wait runs out
    const bool issued = tile_offset + (int)blockIdx.x != drop_tile;
    if (tid == 0) {
        mbar_init(&bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        if (issued) {
            mbar_expect_tx(&bar, B::kBytes);
            tma_load_3d(box, &maps[t.x].pop[ti][parity], t.y - 4, t.z - HALO, 0, &bar);
            tma_load_3d(box + B::kPop, &maps[t.x].ref[ti][parity], t.y - 4, t.z - HALO, 0, &bar);
        }
        if (!first_wave) prefetch_ahead();
    }
    // slots beyond the lattice load their nodes directly (wrapped, or wall
    // ghost rows): done while the copy is in flight.  They lie in the halo ring,
    // and in a ragged tile also among its own, up to two beyond its last node
    {
        const Lat<float> &G = lats[t.x];
        if ((t.y == 0 || t.y + TX + HALO > G.nx || t.z < HALO || t.z + TYv + HALO > G.ny)) {
            const int w = G.nx - t.y, hh = G.ny - t.z;
            const bool ragged = w < TX || hh < TYv;
            const int slots = ragged ? SW * (TYv + 2 * HALO) : kRing<TYv>;
            for (int h = tid; h < slots; h += TX * TYv) {
                int sx = h % SW, sy = h / SW;
                if (!ragged) ring_slot<TYv>(h, sx, sy);
                if (sx < w + 2 * HALO && sy < hh + 2 * HALO && slot_outside(G, t, sx, sy)) {
                    float rA, rB;
                    slot_densities<float, false>(G, t, parity, sx, sy, rA, rB);
                    sm.sr[sy][sx] = make_float2(rA, rB);
                    sm.sp[sy][sx] = make_float2(psi_of<float>(rA), psi_of<float>(rB));
                }
            }
        }
    }
    __syncthreads();   // the barrier is initialised before anyone waits on it
    const bool ok = mbar_wait(&bar, 0, wait_cycles);
    if (!__syncthreads_and(ok)) {
        if (tid == 0) {
            atomicExch(err, 1);
            // let a copy still in flight land before the block ends (bounded
            // too, by at least 2^31 clocks, ~1 s)
            if (issued) mbar_wait(&bar, 0, wait_cycles > (1ll << 31) ? wait_cycles : (1ll << 31));
        }
        return;
    }
    if (tid == 0 && first_wave) prefetch_ahead();
    fused_tile_box<TYv>(lats, t, parity, sm, box, box + B::kPop);
}

// Distance, in quarters of a wave of resident blocks, between a tile and the
// tile whose boxes it prefetches into L2 (0: none).  Half a wave to a wave
// measured alike (a 4096^2 step 3 % shorter than without the prefetch);
// beyond it the boxes are prefetched too early.
constexpr int kPrefetchQuarterWaves = 3;

template <int TYv, bool kMixed>
struct TmaKernel {
    static constexpr size_t kSmem = TmaBox<TYv>::kBytes;
    static int grid_wave;   // resident blocks on the device
    static cudaError_t prepare()
    {
        cudaError_t e = cudaFuncSetAttribute(k_fused_tma<TYv, kMixed>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmem);
        int dev = 0, sms = 0, occ = 0;
        if (e == cudaSuccess) e = cudaGetDevice(&dev);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (e == cudaSuccess)
            e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_fused_tma<TYv, kMixed>, TX * TYv, kSmem);
        if (e == cudaSuccess) grid_wave = sms * occ;
        return e;
    }
    static cudaError_t launch(const Lat<float> *lats, const int4 *tiles, int tile_offset, int n_tiles, int parity,
                              const TmaMaps *maps, int *err, long long wait_cycles, int drop_tile, cudaStream_t s)
    {
        k_fused_tma<TYv, kMixed><<<n_tiles, dim3(TX, TYv), kSmem, s>>>(lats, tiles, tile_offset, parity, maps, err, wait_cycles,
                                                               drop_tile, n_tiles,
                                                               kPrefetchQuarterWaves * grid_wave / 4, grid_wave);
        return cudaGetLastError();
    }
};
template <int TYv, bool kMixed>
int TmaKernel<TYv, kMixed>::grid_wave = 0;

template <int TYv>
cudaError_t prepare_height_tma(bool mixed)
{
    if constexpr (TYv < 8) {
        const cudaError_t e = TmaKernel<TYv, false>::prepare();
        if (e != cudaSuccess || !mixed) return e;
    }
    return TmaKernel<TYv, true>::prepare();
}

template <int TYv>
cudaError_t launch_height_tma(const Lat<float> *lats, const int4 *tiles, int tile_offset, int n_tiles, int n_box, int parity,
                              const TmaMaps *maps, int *err, long long wait_cycles, int drop_tile, cudaStream_t s)
{
    if constexpr (TYv < 8)
        if (n_box == n_tiles)
            return TmaKernel<TYv, false>::launch(lats, tiles, tile_offset, n_tiles, parity, maps, err, wait_cycles, drop_tile, s);
    return TmaKernel<TYv, true>::launch(lats, tiles, tile_offset, n_tiles, parity, maps, err, wait_cycles, drop_tile, s);
}

}  // namespace

cudaError_t prepare_fused_tma(bool mixed)
{
    cudaError_t e = prepare_height_tma<2>(mixed);
    if (e == cudaSuccess) e = prepare_height_tma<4>(mixed);
    if (e == cudaSuccess) e = prepare_height_tma<8>(mixed);
    return e;
}

cudaError_t launch_fused_tma(const Lat<float> *lats, const int4 *tiles, int tile_offset, int n_tiles, int n_box, int parity,
                             const TmaMaps *maps, int *err, long long wait_cycles, int drop_tile, int ty, cudaStream_t s)
{
    if (n_tiles <= 0) return cudaSuccess;
    if (n_box <= 0) return Launch<float>::fused(lats, tiles, tile_offset, n_tiles, parity, ty, s);
    switch (ty) {
    case 2: return launch_height_tma<2>(lats, tiles, tile_offset, n_tiles, n_box, parity, maps, err, wait_cycles, drop_tile, s);
    case 4: return launch_height_tma<4>(lats, tiles, tile_offset, n_tiles, n_box, parity, maps, err, wait_cycles, drop_tile, s);
    case 8: return launch_height_tma<8>(lats, tiles, tile_offset, n_tiles, n_box, parity, maps, err, wait_cycles, drop_tile, s);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace lbk
