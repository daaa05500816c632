// Pressure residual and norms without any device allocation.
//
// Some callers cannot allocate device memory: a host program whose memory is
// owned by a pooling allocator that forbids raw cudaMalloc, a control loop
// that must not pay the latency (and implicit synchronisation) of an
// allocation, or a plug-in that has to keep the process's device footprint
// fixed.  This file gives them r = b - A p and the squared norms ||r||^2,
// ||b||^2 on their own device buffers.  The only scratch the kernel needs
// (one pair of partial sums per block and a block counter) lives in the
// file-scope array below, which every GPU that loads the library holds until
// the process exits.
#include <mutex>
#include <string>

#include "fvm_internal.cuh"

namespace {

// the largest grids taken, counted in blocks of 32 x 4 x 2 cells
constexpr int SX = 32, SY = 4, SZ = 2;
constexpr int kMaxBlocks = 1 << 16;                     // 65,536 blocks = 16,777,216 cells at most
constexpr int kScratchDoubles = 2 * kMaxBlocks + 32;    // partial sums, then the block counter

static __device__ __align__(256) double g_residual_scratch[kScratchDoubles];

// The kernel is bound by the FP64 pipe (two lanes a clock and SM here): one thread per cell with
// a warp reduction of r^2 and b^2 took about 37 FP64 operations a cell, 194 us at 201 x 130 x 97
// cells.  Now each difference across a face is formed once and used by both cells: along x by the
// lane of the upper cell (a shuffle hands it down; 31 cells a warp), along y by a thread that owns
// kRows (4) rows, along z by the march, and the squares are summed in registers: 13 FP64 instructions a
// row of 31 cells, 81 us a call for 194 (58 us at the pipe's rate).
// A warp's item is 31 x kRows x zc cells; the items go round the warps of at most kBlocks blocks, or one to
// a block first where there are few.
constexpr int kWarps = 8, kLanes = 31;
constexpr int kBlocks = 304;                            // two blocks on each of 152 SMs

struct Tiles {
    int x, y, z, zc;
};

// r = b - A p on a box without obstacles: a face of the domain is
// zero-gradient (dirichlet[face] = 0) or zero-value (1) for p.
template <int kRows>
__global__ void __launch_bounds__(32 * kWarps) k_residual_static(const double* __restrict__ p,
                                                                 const double* __restrict__ b, double* __restrict__ r,
                                                                 double* __restrict__ norms, double* scratch, int nx,
                                                                 int ny, int nz, double ih2x, double ih2y, double ih2z,
                                                                 unsigned dir_mask, Tiles tiles, int few) {
    __shared__ double red[2][kWarps];
    __shared__ bool last;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int sy = nx, sz = nx * ny;
    // (the sign by an integer operation: as a negation it took FP64 instructions, six of 18 a cell)
    auto ghost = [&](int face, double v) {
        return __hiloint2double(__double2hiint(v) ^ (int)(((dir_mask >> face) & 1u) << 31), __double2loint(v));
    };
    double r2 = 0.0, b2 = 0.0;
    const int total = tiles.x * tiles.y * tiles.z;
    for (int t = few ? warp * gridDim.x + blockIdx.x : blockIdx.x * kWarps + warp; t < total; t += gridDim.x * kWarps) {
        const int tx = t % tiles.x, ty = (t / tiles.x) % tiles.y, tz = t / (tiles.x * tiles.y);
        // lane l holds cell i: the warp's cells and the one after them (at the top face its ghost)
        const int i = tx * kLanes + lane, j0 = ty * kRows;
        const int k0 = tz * tiles.zc, k1 = min(nz, k0 + tiles.zc);
        const int ic = min(i, nx - 1), rows = min(kRows, ny - j0);
        const bool own = lane < kLanes && i < nx;
        // the cell's value in row j (clamped into the grid) of plane k; beyond x+ the ghost
        auto at = [&](int j, int k) {
            const double v = __ldg(p + ic + sy * min(max(j, 0), ny - 1) + sz * k);
            return i >= nx ? ghost(1, v) : v;
        };
        // what plane k needs beside plane k itself, asked for a plane ahead (the item's first plane
        // together with planes k0 and k0 - 1: a small grid's call is one round trip to memory; 33 x 33 x 33
        // cells 14.0 -> 12.4 us, 201 x 130 x 97 83 -> 81)
        double pn[kRows], bv[kRows], edge[kRows], below, above;
        auto fetch = [&](int k) {
#pragma unroll
            for (int q = 0; q < kRows; ++q) {
                const int c = ic + sy * min(j0 + q, ny - 1) + sz * k;
                pn[q] = at(j0 + q, min(k + 1, nz - 1));
                bv[q] = __ldg(b + c);
                edge[q] = lane == 0 && i > 0 ? __ldg(p + c - 1) : 0.0;
            }
            below = at(j0 - 1, k);            // (clamped: at the faces not used)
            above = at(j0 + kRows, k);
        };
        double pc[kRows], dz[kRows];   // plane k, and its difference to plane k - 1
#pragma unroll
        for (int q = 0; q < kRows; ++q) {
            pc[q] = at(j0 + q, k0);
            dz[q] = at(j0 + q, max(k0 - 1, 0));
        }
        fetch(k0);
#pragma unroll
        for (int q = 0; q < kRows; ++q) dz[q] = pc[q] - (k0 > 0 ? dz[q] : ghost(4, pc[q]));
        for (int k = k0; k < k1; ++k) {
            double xm[kRows], up[kRows], bk[kRows];
#pragma unroll
            for (int q = 0; q < kRows; ++q) {
                up[q] = k + 1 < nz ? pn[q] : ghost(5, pc[q]);
                bk[q] = bv[q];
                xm[q] = __shfl_up_sync(0xffffffffu, pc[q], 1);
                if (lane == 0) xm[q] = i > 0 ? edge[q] : ghost(0, pc[q]);
            }
            const double lo = j0 > 0 ? below : ghost(2, pc[0]), hi4 = above;
            if (k + 1 < k1) fetch(k + 1);
            double dy = pc[0] - lo;
#pragma unroll
            for (int q = 0; q < kRows; ++q) {
                const double dx = pc[q] - xm[q];                          // i > 0 .. nx: to the cell below
                const double dxu = __shfl_down_sync(0xffffffffu, dx, 1);  // its other face
                const double hi = j0 + q + 1 >= ny ? ghost(3, pc[q]) : (q + 1 < kRows ? pc[q + 1 < kRows ? q + 1 : q] : hi4);
                const double dyu = hi - pc[q], dzu = up[q] - pc[q];
                double Ap = 0.0;
                if (nx > 1) Ap += (dx - dxu) * ih2x;
                if (ny > 1) Ap += (dy - dyu) * ih2y;
                if (nz > 1) Ap += (dz[q] - dzu) * ih2z;
                const double rv = bk[q] - Ap;
                if (own && q < rows) {
                    r[i + sy * (j0 + q) + sz * k] = rv;
                    r2 = fma(rv, rv, r2);
                    b2 = fma(bk[q], bk[q], b2);
                }
                dy = dyu;
                dz[q] = dzu;
                pc[q] = up[q];
            }
        }
    }
    for (int off = 16; off > 0; off >>= 1) {
        r2 += __shfl_xor_sync(0xffffffffu, r2, off);
        b2 += __shfl_xor_sync(0xffffffffu, b2, off);
    }
    if (lane == 0) {
        red[0][warp] = r2;
        red[1][warp] = b2;
    }
    __syncthreads();
    const int nblk = gridDim.x, bid = blockIdx.x;
    unsigned* counter = (unsigned*)(scratch + 2 * kMaxBlocks);
    if (tid == 0) {
        double s0 = 0.0, s1 = 0.0;
        for (int w = 0; w < kWarps; ++w) {
            s0 += red[0][w];
            s1 += red[1][w];
        }
        scratch[2 * bid] = s0;
        scratch[2 * bid + 1] = s1;
        __threadfence();
        last = atomicAdd(counter, 1u) == (unsigned)nblk - 1u;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    // the last block sums the partials in a fixed order
    double a0 = 0.0, a1 = 0.0;
    for (int x = tid; x < nblk; x += 32 * kWarps) {
        a0 += __ldcg(scratch + 2 * x);
        a1 += __ldcg(scratch + 2 * x + 1);
    }
    for (int off = 16; off > 0; off >>= 1) {
        a0 += __shfl_xor_sync(0xffffffffu, a0, off);
        a1 += __shfl_xor_sync(0xffffffffu, a1, off);
    }
    __syncthreads();
    if ((tid & 31) == 0) {
        red[0][tid >> 5] = a0;
        red[1][tid >> 5] = a1;
    }
    __syncthreads();
    if (tid == 0) {
        double s0 = 0.0, s1 = 0.0;
        for (int w = 0; w < kWarps; ++w) {
            s0 += red[0][w];
            s1 += red[1][w];
        }
        norms[0] = s0;
        norms[1] = s1;
        *counter = 0u;
    }
}

// Device address of the scratch array, looked up once per device.
std::mutex g_mu;
double* g_scratch_ptr[256] = {};

fvm_status scratch_for_current_device(double** out, std::string& err) {
    // first use on a device: look up the array's device address with that device current
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess || dev < 0 || dev >= 256) {
        err = std::string("cudaGetDevice: ") + cudaGetErrorString(e);
        return FVM_ERR_CUDA;
    }
    std::lock_guard<std::mutex> lock(g_mu);
    if (!g_scratch_ptr[dev]) {
        void* ptr = nullptr;
        e = cudaGetSymbolAddress(&ptr, g_residual_scratch);
        if (e != cudaSuccess || !ptr) {
            err = std::string("cudaGetSymbolAddress: ") + cudaGetErrorString(e);
            return FVM_ERR_CUDA;
        }
        g_scratch_ptr[dev] = (double*)ptr;
    }
    *out = g_scratch_ptr[dev];
    return FVM_OK;
}

}  // namespace

extern "C" fvm_status fvm_poisson_residual_static(const double* p, const double* b, int32_t nx, int32_t ny,
                                                  int32_t nz, const double h[3], const int32_t dirichlet[6],
                                                  double* r, double* norms, void* stream) {
    if (!p || !b || !r || !norms || !h || !dirichlet) {
        set_last_error("null argument");
        return FVM_ERR_INVALID;
    }
    if (nx < 1 || ny < 1 || nz < 1 || !(h[0] > 0.0) || !(h[1] > 0.0) || !(h[2] > 0.0)) {
        set_last_error("grid dimensions must be >= 1 and spacings > 0");
        return FVM_ERR_INVALID;
    }
    // block counts in 64-bit arithmetic (nx near INT32_MAX must not wrap), each factor checked
    // before the product: y and z are also bounded by the launch limit of 65,535 blocks
    const int64_t gx = ((int64_t)nx + SX - 1) / SX, gy = ((int64_t)ny + SY - 1) / SY, gz = ((int64_t)nz + SZ - 1) / SZ;
    if (gx > kMaxBlocks || gy > 65535 || gz > 65535 || gx * gy > kMaxBlocks || gx * gy * gz > kMaxBlocks) {
        set_last_error("grid larger than the static scratch holds (65,536 blocks of 32 x 4 x 2 cells, at most "
                       "65,535 along y and z)");
        return FVM_ERR_INVALID;
    }
    // the axes with more than one cell, in their order (a collapsed one changes no index): rows and planes
    // of a warp's item are then there (200 x 1 x 200 cells: 26 us with three of four rows missing, 12.4 so)
    int n[3] = {1, 1, 1}, axes = 0;
    double ih2[3] = {0.0, 0.0, 0.0};
    unsigned mask = 0;
    const int given[3] = {nx, ny, nz};
    for (int a = 0; a < 3; ++a) {
        if (given[a] == 1) continue;
        n[axes] = given[a];
        ih2[axes] = 1.0 / (h[a] * h[a]);
        for (int side = 0; side < 2; ++side)
            if (dirichlet[2 * a + side]) mask |= 1u << (2 * axes + side);
        ++axes;
    }
    // rows per item: four, or one where items of four rows and one plane are fewer than blocks (a chain of
    // four rows takes longer than the launch: 31 x 31 x 31 cells 27.5 us at four rows and planes, 10.7 so,
    // as one cell a thread)
    Tiles tiles;
    tiles.x = (int)(((int64_t)n[0] + kLanes - 1) / kLanes);
    const int rows = (int64_t)tiles.x * (((int64_t)n[1] + 3) / 4) * n[2] <= kBlocks ? 1 : 4;
    tiles.y = (int)(((int64_t)n[1] + rows - 1) / rows);
    // planes per item: the fewest rounds of items over the 608 warp schedulers times the planes of a
    // round (one more for the difference an item starts with), and three rounds or more where the
    // grid has them (two warps a scheduler kept the FP64 pipe only two thirds busy)
    int64_t best = 0, tiles_rounds = 0;
    for (int zc = 32; zc >= 1; --zc) {
        const int64_t z = ((int64_t)n[2] + zc - 1) / zc, rounds = ((int64_t)tiles.x * tiles.y * z + 607) / 608;
        const int64_t cost = rounds * ((n[2] < zc ? n[2] : zc) + 1);
        if (best == 0 || tiles_rounds < 3 || (cost < best && rounds >= 3)) {
            best = cost;
            tiles_rounds = rounds;
            tiles.z = (int)z;
            tiles.zc = zc;
        }
    }
    // few: up to four warps' items a block, dealt out over the blocks first
    const int64_t total = (int64_t)tiles.x * tiles.y * tiles.z;   // (below 2^20)
    const bool few = total <= 4 * kBlocks;
    const int64_t blocks = few ? total : (total + kWarps - 1) / kWarps;
    const dim3 block(32 * kWarps);
    const dim3 grid((unsigned)(blocks < kBlocks ? blocks : kBlocks));
    double* scratch = nullptr;
    std::string err;
    fvm_status st = scratch_for_current_device(&scratch, err);
    if (st != FVM_OK) {
        set_last_error(err);
        return st;
    }
    cudaStream_t s = (cudaStream_t)stream;
    // the block counter must start at zero (a memset, not an allocation)
    cudaError_t e = cudaMemsetAsync(scratch + 2 * kMaxBlocks, 0, sizeof(unsigned), s);
    if (e == cudaSuccess) {
        const auto kernel = rows == 1 ? k_residual_static<1> : k_residual_static<4>;
        kernel<<<grid, block, 0, s>>>(p, b, r, norms, scratch, n[0], n[1], n[2], ih2[0], ih2[1], ih2[2], mask, tiles, few);
        e = cudaGetLastError();
    }
    if (e != cudaSuccess) {
        set_last_error(std::string("launch: ") + cudaGetErrorString(e));
        return FVM_ERR_CUDA;
    }
    set_last_error("");
    return FVM_OK;
}
