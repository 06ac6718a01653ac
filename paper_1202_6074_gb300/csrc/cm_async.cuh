// Step kernel of 16-bit storage with the pull staged ahead in shared memory.
//
// The two-cells-per-thread step at 16-bit storage is bound by its FP32 arithmetic as long as warps
// are there to issue it: k_step_pair has 20 to 24 warps an SM, each of which waits for its 45 loads,
// computes, and stores. Here a warp works off a run of tiles of 64 cells of a row, and while it
// computes one tile the asynchronous copies of its next one are under way (two stages in shared
// memory). A tile is nine groups (e_y, e_z) of three 128-byte rows (e_x = +1, 0, -1) and the 16 bytes
// beside them that the e_x = +-1 rows are read into: 26 copies of 16 bytes, one instruction of the
// warp. The collision then reads its populations at constant offsets from one shared-memory
// address, without the address arithmetic of 45 global loads (warp instructions per 32 cells of the
// unforced step: 400 -> 366).
// Measured per step against k_step_pair (same collision): Taylor-Green 256^3 BF16 304 -> 275 us
// (6.6 TB/s of 108 B a cell), channel LES 1024 x 256 x 256 BF16 1430 -> 1250 us, force-field LES 512^3 BF16
// 3180 -> 3100 us. A copy ahead into L2 instead (cp.async.bulk.prefetch) was 15 % slower: what is
// bound is the arithmetic beside the loads, not DRAM latency.
#pragma once

#include "cm_pair.cuh"

namespace cm {

constexpr int kTileCells = 64;                         // cells of a warp's tile (two per lane)
constexpr int kGroupBytes = 16 + 3 * 128 + 16;         // [left halo | e_x = +1 | 0 | -1 | right halo]
constexpr int kPullBytes = 9 * kGroupBytes;
constexpr int kFieldBytes = 3 * kTileCells * 4;        // the tile's FP32 force field
template <class FT> __host__ __device__ constexpr int async_stage_bytes() { return kPullBytes + (FT::FIELD ? kFieldBytes : 0); }
template <class FT> __host__ __device__ constexpr int async_smem_bytes() { return 2 * (kBlock / 32) * async_stage_bytes<FT>(); }

__device__ __forceinline__ void copy_async16(unsigned dst, const void* src) {
    asm volatile("cp.async.cg.shared.global.L2::256B [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void copies_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void copies_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// Resident blocks per SM the registers are sized for, and tiles a warp works off. The stages hide the
// memory latency, so fewer warps do than in k_step_pair: 5 blocks (96 registers) for the unforced
// collision (4: +1.8 % time, 6: +3 %), 4 (128) where the force keeps more values alive (FX at 5: +21 %,
// spilling; the force field at 5: +7 %). A run of tiles pays its first copies' latency once, and
// the hardware's block scheduler evens the load out over runs: one run per resident warp (a static
// share of the grid each) lost 10 %, because the scheduler favours old warps and the last ones
// then run alone. 8 tiles against 16: unforced -2 %, FX +1 %, force field +1 % time. The last eighth
// of the tiles (eight a warp at most) goes out in runs of two, so that the blocks of the last wave end together: a channel
// 256 x 192 x 192 179.8 -> 172.9 us a step, the unforced step at 256^3 278.6 -> 275.4.
template <class FT> __host__ __device__ constexpr int async_blocks() { return FT::SIMPLE ? 5 : 4; }
template <class FT> constexpr int async_run() { return FT::SIMPLE ? 8 : 16; }

struct Tile { int x, y, z; };     // tile index in its row, row, plane
// the launch's tiles are numbered along x, y, z from plane z0; a block takes `run` tiles per warp,
// one after another in the numbering, its warps side by side
struct TileWalk {
    int nt;                // tiles per row
    int tiles;             // tiles of the launch
    int run, tail;         // tiles per warp of the first `runs` blocks, and of the blocks after them
    int runs;
    Tile step;             // the block's warps as a tile difference
    int z0;
};

// one 16-bit entry / two adjacent ones from shared memory
template <class S> __device__ __forceinline__ float2 lds2(const unsigned char* q) {
    const unsigned v = *reinterpret_cast<const unsigned*>(q);
    if constexpr (std::is_same_v<S, __nv_bfloat16>) return make_float2(__uint_as_float(v << 16), __uint_as_float(v & 0xffff0000u));
    else return __half22float2(*reinterpret_cast<const __half2*>(&v));
}

template <class S, class FT>
__global__ void __launch_bounds__(kBlock, async_blocks<FT>()) k_step_async(const S* __restrict__ src, S* __restrict__ dst,
                                                                            const float* __restrict__ Ff, PR<float> p,
                                                                            TileWalk w) {
    static_assert(sizeof(S) == 2, "the stages hold 16-bit entries");
    extern __shared__ __align__(16) unsigned char smem[];
    constexpr int STAGE = async_stage_bytes<FT>();
    chain_begin();
    const int lane = threadIdx.x & 31;
    constexpr int WPB = kBlock / 32;
    const bool first = (int)blockIdx.x < w.runs;
    const int len = WPB * (first ? w.run : w.tail);
    const int base = first ? blockIdx.x * len : w.runs * (WPB * w.run) + ((int)blockIdx.x - w.runs) * len;
    int t = base + (threadIdx.x >> 5);
    const int end = min(w.tiles, base + len);
    if (t >= end) return;
    unsigned char* const buf = smem + (threadIdx.x >> 5) * (2 * STAGE);
    const size_t PS = p.S64;
    // this lane's copy in every group: 16 bytes of the e_x row a at column 8 (lane & 7) of the tile,
    // or (lanes 24, 25) the 16 bytes left of the e_x = +1 row and right of the e_x = -1 row
    const int a = lane < 24 ? 2 - (lane >> 3) : lane == 24 ? 2 : 0;
    const unsigned cdst = (unsigned)__cvta_generic_to_shared(buf) + (lane < 24 ? 16 + 16 * lane : lane == 24 ? 0 : kGroupBytes - 16);
    const S* const csrc = src + (size_t)a * PS;

    auto near = [&](const Tile& q) -> bool {      // next to a y or z wall: pulled directly
        if constexpr (FT::WALLS)
            return (p.bc[1] == 1 && (q.y == 0 || q.y == p.ny - 1)) || (p.bc[2] == 1 && (q.z == 0 || q.z == p.nz - 1));
        else return false;
    };
    auto stage = [&](const Tile& q, unsigned at) {
        if constexpr (FT::FIELD) {
            const size_t cell = ((size_t)q.z * p.ny + q.y) * p.nx + q.x * kTileCells;
            const unsigned fd = (unsigned)__cvta_generic_to_shared(buf) + at + kPullBytes + 16 * lane;
            const float* f = Ff + cell + 4 * (lane & 15);
            copy_async16(fd, f + (lane >> 4) * p.N64);
            if (lane < 16) copy_async16(fd + 512, f + 2 * p.N64);
        }
        if (near(q)) return;
        int col = q.x * kTileCells;
        if (lane < 24) col += 8 * (lane & 7);
        else if (lane == 24) col = col == 0 ? p.nx - 8 : col - 8;
        else col = col + kTileCells == p.nx ? 0 : col + kTileCells;
        int ys[3], zs[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            int sy = q.y + 1 - k, sz = q.z + 1 - k;
            if (sy < 0) sy += p.ny;
            else if (sy >= p.ny) sy -= p.ny;
            if (sz < 0) sz += p.wz;
            else if (sz >= p.nz) sz -= p.wz;
            ys[k] = sy * p.nx;
            zs[k] = sz * p.ny * p.nx;
        }
        if (lane < 26) {
            const S* const c0 = csrc + col;
            sfor<9>([&](auto G) {
                constexpr int g = decltype(G)::value;
                copy_async16(cdst + at + g * kGroupBytes, c0 + (zs[g / 3] + ys[g % 3]) + (size_t)(3 * g) * PS);
            });
        }
    };

    Tile q{t % w.nt, (t / w.nt) % p.ny, t / w.nt / p.ny + w.z0};
    unsigned at = 0;
    chain_wait();
    stage(q, 0);
    copies_commit();
    for (;;) {
        Tile n{q.x + w.step.x, q.y + w.step.y, q.z + w.step.z};
        if (n.x >= w.nt) { n.x -= w.nt; ++n.y; }
        if (n.y >= p.ny) { n.y -= p.ny; ++n.z; }
        t += WPB;
        const bool more = t < end;
        if (more) stage(n, STAGE - at);
        copies_commit();
        copies_wait<1>();
        __syncwarp();
        const unsigned char* const b = buf + at;
        const int x0 = q.x * kTileCells + 2 * lane;
        const unsigned cell = (unsigned)((q.z * p.ny + q.y) * p.nx + x0);
        F2 h[27];
        if (near(q)) {
            if constexpr (FT::WALLS) gather_adj<S, true, FT::BIG>(src, x0, q.y, q.z, p, h);
        } else {
            const unsigned char* const c = b + 16 + 4 * lane;
            sfor<9>([&](auto G) {
                constexpr int g = decltype(G)::value;
                const unsigned char* const r = c + g * kGroupBytes;
                const S* const rp = reinterpret_cast<const S*>(r);                 // e_x = +1
                const S* const rm = reinterpret_cast<const S*>(r + 256);           // e_x = -1
                const float2 d = lds2<S>(r + 128);
                h[3 * g + 2] = F2(Codec<S>::ld_shared(rp - 1), Codec<S>::ld_shared(rp));
                h[3 * g + 1] = F2(d.x, d.y);
                h[3 * g + 0] = F2(Codec<S>::ld_shared(rm + 1), Codec<S>::ld_shared(rm + 2));
            });
        }
        F2 F[3];
        if constexpr (FT::FIELD) {
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                const float2 f = *reinterpret_cast<const float2*>(b + kPullBytes + 256 * d + 8 * lane);
                F[d] = F2(f.x, f.y);
            }
        } else {
#pragma unroll
            for (int d = 0; d < 3; ++d) F[d] = F2(p.F[d]);
        }
        __syncwarp();      // every lane has read the stage before the next iteration writes into it
        constexpr bool DEV = pair_dev<S, FT>();
        collide<3, F2, FT, DEV>(h, F, p, smagorinsky_constant<float, FT::LES>(p, q.y));
        sfor<27>([&](auto I) {
            constexpr int i = decltype(I)::value;
            Codec<S>::st2(dst + cell + PS * i, h[slot<3>(i)].v.x, h[slot<3>(i)].v.y);
        });
        if (!more) break;
        q = n;
        at = STAGE - at;
    }
}

template <class S, class FT>
void launch_async(const void* src, void* dst, const void* Ff, const Params& p, cudaStream_t st) {
    constexpr int bytes = async_smem_bytes<FT>();
    cudaFuncSetAttribute(k_step_async<S, FT>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    cudaFuncSetAttribute(k_step_async<S, FT>, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
    TileWalk w;
    w.nt = p.nx / kTileCells;
    w.tiles = w.nt * p.ny * step_planes(p);
    const int wpb = kBlock / 32, resident = async_resident_warps<FT>(p), share = w.tiles / (3 * resident);
    w.run = share < 1 ? 1 : share < async_run<FT>() ? share : async_run<FT>();
    w.tail = w.run < 2 ? 1 : 2;
    const int tail = w.tiles / 8 < 8 * resident ? w.tiles / 8 : 8 * resident;
    w.runs = (w.tiles - tail) / (wpb * w.run);
    const int blocks = w.runs + (w.tiles - w.runs * wpb * w.run + wpb * w.tail - 1) / (wpb * w.tail);
    w.step = Tile{wpb % w.nt, (wpb / w.nt) % p.ny, wpb / w.nt / p.ny};
    w.z0 = p.z0;
    launch_chained_smem(p, k_step_async<S, FT>, blocks, kBlock, bytes, st, (const S*)src, (S*)dst, (const float*)Ff,
                        typed<float>(p), w);
}

}  // namespace cm
