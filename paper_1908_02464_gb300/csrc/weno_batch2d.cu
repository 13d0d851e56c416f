// Batched 2D solver: the 2D instantiations of the persistent batch kernel
// (weno_batch.cuh).  Each stage is the grid solver's pair of sweeps: the y
// tiles write their flux divergence (Eq. goveq5) to an accumulator, then the
// x tiles add their own and apply the RK3 combination.
#include <cuda_runtime.h>

#include "weno_batch.cuh"

namespace wis {

// Tile shapes (LINES x SEG, LINES (SEG + 1) faces = CTA size) of the x and y
// sweeps.  Batched instances have short lines (tens of cells), so the tiles
// hold several lines; the y tiles hold 8 or 4 x-adjacent columns, so that
// their loads are row pieces.  1024 explosions in FP64: 59, 57 and 60 ms (one
// CTA per instance: 103, 106 and 150 ms); with the primitives shared between
// the sweeps the first takes 55 ms.  4096 boxes of 16 to 64 cells a side in
// FP32: 70, 72 and 94 ms with 32 warps per SM (64 registers a thread; 112 to 124
// registers and half as many warps took half as long again).  2000 boxes of 8
// to 20 cells, one or two tiles a sweep, are the other way round: 2.9 ms, 2.2 ms
// with one CTA per instance and the larger number of registers.
template <int V> struct Batch2Shape;
template <> struct Batch2Shape<0> { static constexpr int NT = 128, XL = 4, XS = 31, YL = 8, YS = 15; };
template <> struct Batch2Shape<1> { static constexpr int NT = 128, XL = 2, XS = 63, YL = 4, YS = 31; };
template <> struct Batch2Shape<2> { static constexpr int NT = 64, XL = 2, XS = 31, YL = 4, YS = 15; };

template <int V>
struct Batch2Cfg : Batch2Shape<V> {
    using S = Batch2Shape<V>;
    template <typename T> static constexpr size_t smem_bytes()
    {
        constexpr size_t x = SweepSmem<T, 2, S::XL, S::XS>::bytes, y = SweepSmem<T, 2, S::YL, S::YS>::bytes;
        return x > y ? x : y;
    }
    template <typename T> static constexpr int min_blocks() { return (sizeof(T) == 8 ? 512 : 1024) / S::NT; }
};

cudaError_t batch2d_config(int prec, bool fx, int v, int* blocks_per_sm, size_t* smem)
{
    return batch_config_p<2, Batch2Cfg>(prec, fx, v, blocks_per_sm, smem);
}
cudaError_t batch2d_launch(int prec, bool fx, int v, const BatchArgs& b, int blocks, cudaStream_t s)
{
    return batch_launch_p<2, Batch2Cfg>(prec, fx, v, b, blocks, s);
}
int batch2d_tiles(int v, int nx, int ny, int d)
{
    if (v == 1) return batch_tiles<Batch2Cfg<1>>(2, nx, ny, d);
    if (v == 2) return batch_tiles<Batch2Cfg<2>>(2, nx, ny, d);
    return batch_tiles<Batch2Cfg<0>>(2, nx, ny, d);
}

}  // namespace wis
