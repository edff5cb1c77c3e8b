// Learned warm start: a 3-D convolutional net that maps the coarse-only solution, upsampled onto a
// refined block (plus a halo), to the refined solution there.  The net's output initialises the
// refined levels with f = f^eq(rho, u) (Eq. fequ); the LBM then runs unmodified.
//
// Net: L layers of 3x3x3 convolutions (zero padding, stride 1), width 16, ReLU between layers,
// none after the last.  Tensors are channels-last volumes of 16 BF16 channels (32 bytes per
// voxel), `nvol` volumes of D x H x W voxels stored one after another, x fastest.  Products
// run on the tensor cores (BF16 operands, FP32 accumulate): the convolutions with tcgen05.mma, or with
// mma.sync m16n8k16 where the caller asks for it, the weight gradient with mma.sync.  Weights are kept
// in FP32 (master copy, Adam moments) and rounded to BF16 for the products.
//
//   forward   Z_l = b_l + sum_o W_l[o] X_l[v + o]          X_{l+1} = relu(Z_l)
//   backward  dW_l[o] += sum_v dZ_l[v] (x) X_l[v + o]      db_l = sum_v dZ_l[v]
//             dX_l[v] = sum_o W_l[o]^T dZ_l[v - o]         dZ_{l-1} = dX_l * [X_l > 0]
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstddef>
#include <cstdio>
#include <cstring>
#include <string>
#include <vector>

#include "devmem.h"
#include "lbm_internal.h"

namespace {

constexpr int CH = 16;       // channels of every tensor (unused channels are zero)
constexpr int TAPS = 27;     // 3x3x3 offsets, o = (dz + 1) * 9 + (dy + 1) * 3 + (dx + 1)

struct Dims {
    int D, H, W;   // voxels per volume along z, y, x
    int nvol;      // volumes
    long long V;   // voxels per volume
    long long N;   // all voxels
};

__device__ __forceinline__ void mma16816(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};\n"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// Linear index of voxel v shifted by tap o, or -1 outside its volume (zero padding).
__device__ __forceinline__ long long shifted(const Dims& d, long long v, int o) {
    if (v >= d.N) return -1;
    const long long vol = v / d.V;
    long long r = v - vol * d.V;
    const int x = int(r % d.W);
    r /= d.W;
    const int y = int(r % d.H), z = int(r / d.H);
    const int dx = o % 3 - 1, dy = (o / 3) % 3 - 1, dz = o / 9 - 1;
    const int sx = x + dx, sy = y + dy, sz = z + dz;
    if (sx < 0 || sx >= d.W || sy < 0 || sy >= d.H || sz < 0 || sz >= d.D) return -1;
    return vol * d.V + ((long long)(sz) * d.H + sy) * d.W + sx;
}

// Z[v][n] = bias[n] + sum_o sum_k Wt[o][n][k] X[v + o][k] over 16 voxels per warp; then
// optionally relu (act = 1) or multiplication by [mask > 0] (act = 2, the ReLU derivative of the
// layer whose output `mask` is).  Wt is BF16 [27][16 out][16 in].
__global__ void __launch_bounds__(256) conv_kernel(const __nv_bfloat16* __restrict__ X, const __nv_bfloat16* __restrict__ Wt,
                                                   const float* __restrict__ bias, __nv_bfloat16* __restrict__ Z, Dims d,
                                                   int act, const __nv_bfloat16* __restrict__ mask) {
    __shared__ uint32_t sw[TAPS * CH * CH / 2];
    for (int i = threadIdx.x; i < TAPS * CH * CH / 2; i += blockDim.x) sw[i] = reinterpret_cast<const uint32_t*>(Wt)[i];
    __syncthreads();
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const long long v0 = ((long long)(blockIdx.x) * 8 + (threadIdx.x >> 5)) * 16;
    if (v0 >= d.N) return;
    float acc[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
    const uint32_t* X32 = reinterpret_cast<const uint32_t*>(X);
    for (int o = 0; o < TAPS; o++) {
        const long long r0 = shifted(d, v0 + g, o), r1 = shifted(d, v0 + g + 8, o);
        uint32_t a[4];
        a[0] = r0 >= 0 ? __ldg(X32 + r0 * (CH / 2) + t) : 0u;
        a[1] = r1 >= 0 ? __ldg(X32 + r1 * (CH / 2) + t) : 0u;
        a[2] = r0 >= 0 ? __ldg(X32 + r0 * (CH / 2) + t + 4) : 0u;
        a[3] = r1 >= 0 ? __ldg(X32 + r1 * (CH / 2) + t + 4) : 0u;
#pragma unroll
        for (int nt = 0; nt < 2; nt++) {
            const int n = nt * 8 + g;
            const uint32_t b0 = sw[(o * CH + n) * (CH / 2) + t], b1 = sw[(o * CH + n) * (CH / 2) + t + 4];
            mma16816(acc[nt], a, b0, b1);
        }
    }
#pragma unroll
    for (int nt = 0; nt < 2; nt++)
#pragma unroll
        for (int h = 0; h < 2; h++) {
            const long long v = v0 + g + 8 * h;
            if (v >= d.N) continue;
            const int n = nt * 8 + 2 * t;
            float z0 = acc[nt][2 * h] + (bias ? bias[n] : 0.f), z1 = acc[nt][2 * h + 1] + (bias ? bias[n + 1] : 0.f);
            if (act == 1) {
                z0 = fmaxf(z0, 0.f);
                z1 = fmaxf(z1, 0.f);
            } else if (act == 2) {
                const __nv_bfloat162 m = reinterpret_cast<const __nv_bfloat162*>(mask)[v * (CH / 2) + n / 2];
                if (!(__bfloat162float(m.x) > 0.f)) z0 = 0.f;
                if (!(__bfloat162float(m.y) > 0.f)) z1 = 0.f;
            }
            reinterpret_cast<__nv_bfloat162*>(Z)[v * (CH / 2) + n / 2] = __floats2bfloat162_rn(z0, z1);
        }
}

// ---------------------------------------------------------------- tcgen05 convolution
// The same product as conv_kernel on the 5th-generation tensor cores.  A unit is a part of HC x WC voxels of a
// plane and a run of ZC planes of a volume.  The planes of X pass through a ring of four in shared memory: a plane is
// (HC + 2) rows of P slots (P = WC + 2 rounded up to 4; zero outside the volume), kept as two halves of 8 channels and
// four residues of the slot number, so that four consecutive voxels of a row make one row of the MMA's M: half c of
// slot s at byte 16 ((4 c + s % 4) NG + s / 4) of its plane.  With 128 rows of four voxels an input voxel (residue j of
// the row, or the last of the row before, or the first of the row after) is one M128 K16 operand and feeds up to
// three outputs, taps dx = 1, 0, -1, which are adjacent column blocks of 16: N = 48 in one MMA (32 or 16 at the ends of the
// four).  A tap row (dz, dy) is six MMAs for 512 slots in place of twelve of N = 16: an MMA this narrow is
// bound by reading its 4 KB of A from shared memory (32 clocks), so the reads per voxel halve.  Each output's 27 products
// are added in the order of the taps, as with one MMA per tap.
// While plane z multiplies (one thread of a warp of its own issues, about as long as the products take; FP32
// accumulators in one of two TMEM buffers, a commit to an mbarrier), four warps read plane z - 1 from the other buffer (tcgen05.ld 32x32b.x16: a voxel's 16 channels), apply bias and
// activation as conv_kernel does and store 128 bytes per lane, and the copies of plane z + 2 are in flight.
// 512 volumes of 18^3, one layer: 150 us with one MMA per tap and whole planes staged three times, now 107.  Bound:
// the shared-memory pipe, 88 % of the elapsed time (65 % the MMAs' operand reads, 23 % the copies and the bias reads,
// two thirds of them bank conflicts), and the wait for a plane's copies with a CTA barrier: with a third of the MMAs a
// layer still takes 85 us.
constexpr int TC_W_BYTES = TAPS * 2 * CH * 8 * 2;   // weights [dz, dy][half][dx = 1, 0, -1][n][8] BF16
constexpr int TC_BAR_OFF = TC_W_BYTES;              // two mbarriers, the TMEM address, two flags, the bias
constexpr int TC_TM_OFF = TC_W_BYTES + 16;
constexpr int TC_FAIL_OFF = TC_W_BYTES + 20;
constexpr int TC_BIAS_OFF = TC_W_BYTES + 32;
constexpr int TC_A_OFF = 14336;                     // then the ring
constexpr int TC_RING = 4, TC_COLS = 64;            // planes, TMEM columns of a buffer
constexpr int TC_THREADS = 160;                     // four warps that copy and write Z, one that issues the products
constexpr int TC_COPIES = 10;                       // 16-byte copies per thread and plane

struct TcGeom {
    int HC, WC, ZC;       // voxels of a unit
    int nx, ny, nz;       // units along each axis
    int P, NG;            // slots per row, groups of four slots per plane
    int grid;
    size_t smem;
};

__device__ __forceinline__ uint64_t smem_desc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
    // start address, leading byte offset (K direction), stride byte offset (M/N direction), all in
    // 16-byte units; bit 46: descriptor version of tcgen05; no swizzle, base offset 0
    return uint64_t((addr >> 4) & 0x3FFF) | (uint64_t((lbo >> 4) & 0x3FFF) << 16) |
           (uint64_t((sbo >> 4) & 0x3FFF) << 32) | (uint64_t(1) << 46);
}
__device__ __forceinline__ void tc_mma(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d), "l"(a), "l"(b), "r"(idesc), "r"(acc));
}
__device__ __forceinline__ void tc_ld16(uint32_t (&r)[16], uint32_t addr) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(addr));
}

__global__ void __launch_bounds__(TC_THREADS, 3) conv_tc_kernel(const __nv_bfloat16* __restrict__ X, const __nv_bfloat16* __restrict__ Wt,
                                                      const float* __restrict__ bias, __nv_bfloat16* __restrict__ Z, Dims d,
                                                      int act, const __nv_bfloat16* __restrict__ mask, TcGeom g,
                                                      int* __restrict__ err, int wait_test) {
    extern __shared__ __align__(1024) unsigned char sm[];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t base = static_cast<uint32_t>(__cvta_generic_to_shared(sm));
    const uint32_t bar = base + TC_BAR_OFF, abase = base + TC_A_OFF;
    const uint32_t plane_bytes = uint32_t(8 * g.NG * 16);
    // weights Wt[o][n][k] -> [dz, dy][k / 8][1 - dx][n][k % 8], 16 bytes at a time
    for (int i = tid; i < TAPS * 2 * CH; i += blockDim.x) {
        const int n = i % CH, blk = (i / CH) % 3, c = (i / (3 * CH)) & 1, zy = i / (6 * CH);
        const int o = zy * 3 + 2 - blk;
        reinterpret_cast<uint4*>(sm)[i] = *reinterpret_cast<const uint4*>(Wt + (o * CH + n) * CH + c * 8);
    }
    if (tid < CH) reinterpret_cast<float*>(sm + TC_BIAS_OFF)[tid] = bias ? bias[tid] : 0.f;
    volatile int* fail = reinterpret_cast<volatile int*>(sm + TC_FAIL_OFF);
    if (tid == 0) {
        fail[0] = fail[1] = 0;
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar) : "memory");
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar + 8) : "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(base + TC_TM_OFF), "r"(2 * TC_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = *reinterpret_cast<volatile uint32_t*>(sm + TC_TM_OFF);
    const uint32_t id16 = (1u << 4) | (1u << 7) | (1u << 10) | ((16u >> 3) << 17) | ((128u >> 4) << 24);
    const uint32_t id32 = id16 + ((16u >> 3) << 17), id48 = id16 + ((32u >> 3) << 17);
    const float* sbias = reinterpret_cast<const float*>(sm + TC_BIAS_OFF);
    const int slots = (g.HC + 2) * g.P;
    const long long units = (long long)d.nvol * g.nz * g.ny * g.nx;
    uint32_t phase[2] = {0u, 0u};
    bool failed = false;
    for (long long unit = blockIdx.x; unit < units && !failed; unit += gridDim.x) {
        long long r = unit;
        const int cx = int(r % g.nx);
        r /= g.nx;
        const int cy = int(r % g.ny);
        r /= g.ny;
        const int z0 = int(r % g.nz) * g.ZC, z1 = min(z0 + g.ZC, d.D);
        const long long vol = r / g.nz;
        const int x0 = cx * g.WC, y0 = cy * g.HC;
        const int wc = min(g.WC, d.W - x0), hc = min(g.HC, d.H - y0);   // voxels of this unit
        // this thread's copies of a plane: 16-byte halves i = tid + 128 k of the slots; where they come from within
        // the volume's plane (or -1: zero) and where they go within the ring's
        int from[TC_COPIES], to[TC_COPIES];
#pragma unroll
        for (int k = 0; k < TC_COPIES; k++) {
            const int i = tid + 128 * k, c = i & 1, s = i >> 1;
            const int sy = s / g.P, sx = s - sy * g.P;
            const int y = y0 + sy - 1, x = x0 + sx - 1;
            from[k] = (y >= 0 && y < d.H && x >= 0 && x < d.W) ? (y * d.W + x) * 2 + c : -1;
            to[k] = s < slots && warp < 4 ? ((4 * c + (s & 3)) * g.NG + (s >> 2)) * 16 : -1;
        }
        auto load = [&](int z) {   // plane z into ring slot (z + 1) % TC_RING
            const bool pv = z >= 0 && z < d.D;
            const uint4* plane = reinterpret_cast<const uint4*>(X) + (vol * d.D + (pv ? z : 0)) * d.H * d.W * 2;
            const uint32_t ring = abase + uint32_t((z + 1) & (TC_RING - 1)) * plane_bytes;
#pragma unroll
            for (int k = 0; k < TC_COPIES; k++) {
                if (to[k] < 0) continue;
                const bool ok = pv && from[k] >= 0;
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(ring + uint32_t(to[k])),
                             "l"(plane + (ok ? from[k] : 0)), "r"(ok ? 16 : 0)
                             : "memory");
            }
        };
        // this lane's four output voxels: slots P + 4 group .. + 3, one row
        const int os = g.P + 4 * tid, oy = os / g.P, ox = os - oy * g.P;
        const bool orow = oy <= hc;
        // Z of plane z from TMEM buffer z & 1
        auto drain = [&](int z) {
            const int h = z & 1;
            // bounded wait (the wait test issues no products and gives up after a short wait: nothing
            // asynchronous but its own copies is outstanding when the CTA then releases its TMEM)
            uint32_t done = 0;
            const int limit = wait_test ? (1 << 10) : (1 << 24);
            for (int it = 0; it < limit && !done; it++)
                asm volatile(
                    "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
                    : "=r"(done) : "r"(bar + 8 * h), "r"(phase[h]) : "memory");
            phase[h] ^= 1u;
            // A flag per buffer: the last two drains of a unit follow one another without a barrier of the CTA between
            // them, and a warp that reads the first one's flag late must not see what the second one set, leave, and
            // keep the others at their barrier.
            if (!done) {
                fail[h] = 1;
                atomicExch(err, 1);
            }
            asm volatile("bar.sync 1, 128;" ::: "memory");   // the four warps agree
            if (fail[h]) {
                failed = true;
                return;
            }
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const long long row = ((vol * d.D + z) * d.H + (y0 + oy - 1)) * d.W + (x0 - 1);
#pragma unroll
            for (int jj = 0; jj < 4; jj += 2) {   // two voxels at a time: 32 registers
                uint32_t v[2][16];
#pragma unroll
                for (int j = 0; j < 2; j++)
                    tc_ld16(v[j], tmem + (uint32_t(warp * 32) << 16) + uint32_t(h * TC_COLS + (jj + j) * 16));
                asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                if (!orow) continue;
#pragma unroll
                for (int j = 0; j < 2; j++) {
                    const int x = ox + jj + j;
                    if (x < 1 || x > wc) continue;
                    const long long at = row + x;
                    uint4 m[2];
                    if (act == 2) {
                        m[0] = reinterpret_cast<const uint4*>(mask + at * CH)[0];
                        m[1] = reinterpret_cast<const uint4*>(mask + at * CH)[1];
                    }
                    uint4 out[2];
                    uint32_t* o32 = reinterpret_cast<uint32_t*>(out);
                    const __nv_bfloat162* mk = reinterpret_cast<const __nv_bfloat162*>(m);
#pragma unroll
                    for (int c = 0; c < 8; c++) {
                        float a0 = __uint_as_float(v[j][2 * c]) + sbias[2 * c];
                        float a1 = __uint_as_float(v[j][2 * c + 1]) + sbias[2 * c + 1];
                        if (act == 1) {
                            a0 = fmaxf(a0, 0.f);
                            a1 = fmaxf(a1, 0.f);
                        } else if (act == 2) {
                            if (!(__bfloat162float(mk[c].x) > 0.f)) a0 = 0.f;
                            if (!(__bfloat162float(mk[c].y) > 0.f)) a1 = 0.f;
                        }
                        const __nv_bfloat162 t = __floats2bfloat162_rn(a0, a1);
                        o32[c] = *reinterpret_cast<const uint32_t*>(&t);
                    }
                    uint4* dst = reinterpret_cast<uint4*>(Z + at * CH);
                    dst[0] = out[0];
                    dst[1] = out[1];
                }
            }
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        };
        load(z0 - 1);
        load(z0);
        load(z0 + 1);
        for (int z = z0; z < z1; z++) {
            asm volatile("cp.async.wait_all;\n" ::: "memory");   // planes up to z + 1 have landed
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            failed = __syncthreads_or(failed);   // the same for every thread
            if (failed) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            if (tid == 128 && !wait_test) {
                const uint32_t D = tmem + uint32_t((z & 1) * TC_COLS);
                const uint64_t b0 = smem_desc(base, uint32_t(3 * CH * 16), 128u);
                const int G0 = g.P >> 2;
                for (int zy = 0; zy < 9; zy++) {
                    const int dz = zy / 3 - 1, dy = zy % 3 - 1;
                    const uint32_t ring = abase + uint32_t((z + dz + 1) & (TC_RING - 1)) * plane_bytes;
                    // residue 0 of the first group, row moved by dy; residues are NG groups apart
                    const uint64_t a = smem_desc(ring + uint32_t((G0 + dy * G0) * 16), uint32_t(4 * g.NG * 16), 128u);
                    const uint64_t b = b0 + uint64_t(zy * 6 * CH);
                    const uint64_t NG = uint64_t(g.NG);
                    if (zy == 0) {   // the first product of each column block does not accumulate
                        tc_mma(D, a + 3 * NG - 1, b + 2 * CH, id16, 0);
                        tc_mma(D, a, b + CH, id16, 1);
                        tc_mma(D + 16, a, b + 2 * CH, id16, 0);
                        tc_mma(D, a + NG, b, id32, 1);
                        tc_mma(D + 32, a + NG, b + 2 * CH, id16, 0);
                        tc_mma(D + 16, a + 2 * NG, b, id32, 1);
                        tc_mma(D + 48, a + 2 * NG, b + 2 * CH, id16, 0);
                    } else {
                        tc_mma(D, a + 3 * NG - 1, b + 2 * CH, id16, 1);
                        tc_mma(D, a, b + CH, id32, 1);
                        tc_mma(D, a + NG, b, id48, 1);
                        tc_mma(D + 16, a + 2 * NG, b, id48, 1);
                    }
                    tc_mma(D + 32, a + 3 * NG, b, id32, 1);
                    tc_mma(D + 48, a + 1, b, id16, 1);
                }
                asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar + 8 * (z & 1))
                             : "memory");
            }
            if (warp < 4) {
                if (z > z0) drain(z - 1);
                if (!failed && z + 1 < z1) load(z + 2);   // in the place of plane z - 2, whose products are done
            }
        }
        if (warp < 4 && !failed) drain(z1 - 1);
        failed = __syncthreads_or(failed);   // the next unit's copies follow this unit's products and reads
    }
    asm volatile("cp.async.wait_all;\n" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(2 * TC_COLS) : "memory");
}

// ---------------------------------------------------------------- weight gradient
// dW[o][m][n] += sum_v dZ[v][m] X[v + o][n] and db[m] += sum_v dZ[v][m]: a contraction over voxels with 16 x 16
// results per tap.  A unit is a (volume, z-plane) part of HC x WC voxels.  Its dZ (zero border) and the three
// planes of X around it (with their own border voxels, zero outside the volume) are staged as slots of (WC + 2)-wide
// rows, in two halves of 8 channels, 16 bytes per slot, so that every tap's operand is the same run of slots moved by
// dy P + dx, read by ldmatrix from any slot.  Warp (split, dz) takes every second run of 16 slots, loads dZ once and
// the nine taps of its plane, and keeps their 72 sums in registers; they are added up in shared memory after at
// most kWgradUnits units (so that no FP32 chain grows with the batch) and leave the CTA as 16-byte reductions.
// Bound: ldmatrix and mma.sync issue.  (tcgen05 has 64 rows at least: 48 of them would be padding for the 16
// output channels, which costs as much tensor time.)  Read straight from global memory, tap by tap with 2-byte loads,
// the gradient of one layer over 32 x 18^3 voxels took 430 us, now 19.
constexpr int kWgradThreads = 192;
constexpr int kWgradUnits = 4;

struct WgradGeom {
    int HC, WC;        // voxels of a unit along y and x
    int ny, nx;        // units per plane
    int P, NSL, nt;    // slots per row and per plane (a multiple of 8), runs of 16 slots
    long long units;
    size_t smem;
};

__device__ __forceinline__ void ldsm4t(uint32_t (&r)[4], uint32_t addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}

__global__ void __launch_bounds__(kWgradThreads, 2) wgrad_kernel(const __nv_bfloat16* __restrict__ X,
                                                                 const __nv_bfloat16* __restrict__ dZ,
                                                                 float* __restrict__ dW, Dims d, WgradGeom g) {
    extern __shared__ __align__(128) unsigned char wsm[];
    float* sums = reinterpret_cast<float*>(wsm);                    // [27][16][16], then [16] for db
    constexpr int kSums = TAPS * CH * CH + CH;
    unsigned char* planes = wsm + kSums * 4;                        // dZ, then X of z - 1, z, z + 1
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int dz = warp % 3, split = warp / 3;
    const int plane_bytes = 2 * g.NSL * 16;
    const uint32_t base = static_cast<uint32_t>(__cvta_generic_to_shared(planes));
    for (int i = tid; i < kSums; i += kWgradThreads) sums[i] = 0.f;
    // slots that no unit writes (borders of dZ, the tail of every plane) stay zero
    for (int i = tid; i < 8 * g.NSL; i += kWgradThreads) *reinterpret_cast<uint4*>(planes + i * 16) = make_uint4(0u, 0u, 0u, 0u);
    // row addresses of the ldmatrix operands: lane l gives row l % 8 of matrix l / 8.  A (dZ, m x k): matrices
    // (k 0-7, m 0-7), (k 0-7, m 8-15), (k 8-15, m 0-7), (k 8-15, m 8-15); B (X, k x n): the middle two exchanged.
    const uint32_t a_lane = base + uint32_t((((lane >> 3) & 1) * g.NSL + (lane & 7) + ((lane >> 4) & 1) * 8) * 16);
    const uint32_t b_lane = base + uint32_t((1 + dz) * plane_bytes) +
                            uint32_t(((lane >> 4) * g.NSL + (lane & 7) + ((lane >> 3) & 1) * 8) * 16);
    float acc[9][2][4], bacc[4];
    auto clear = [&]() {
#pragma unroll
        for (int o = 0; o < 9; o++)
#pragma unroll
            for (int k = 0; k < 8; k++) acc[o][k >> 2][k & 3] = 0.f;
#pragma unroll
        for (int k = 0; k < 4; k++) bacc[k] = 0.f;
    };
    // adds the warps' sums up in shared memory, one split after the other
    auto flush = [&]() {
        for (int s = 0; s < 2; s++) {
            __syncthreads();
            if (split != s) continue;
            const int r = lane >> 2, t = lane & 3;
#pragma unroll
            for (int o = 0; o < 9; o++)
#pragma unroll
                for (int n = 0; n < 2; n++)
#pragma unroll
                    for (int h = 0; h < 2; h++) {
                        float2* p = reinterpret_cast<float2*>(sums + ((dz * 9 + o) * CH + r + 8 * h) * CH + n * 8 + 2 * t);
                        float2 v = *p;
                        v.x += acc[o][n][2 * h];
                        v.y += acc[o][n][2 * h + 1];
                        *p = v;
                    }
            if (dz == 1 && t == 0) {
                sums[TAPS * CH * CH + r] += bacc[0];
                sums[TAPS * CH * CH + r + 8] += bacc[2];
            }
        }
    };
    clear();
    int held = 0;
    for (long long unit = blockIdx.x; unit < g.units; unit += gridDim.x) {
        long long r = unit;
        const int cx = int(r % g.nx);
        r /= g.nx;
        const int cy = int(r % g.ny);
        r /= g.ny;
        const int z = int(r % d.D);
        const long long vol = r / d.D;
        const int x0 = cx * g.WC, y0 = cy * g.HC;
        __syncthreads();   // the previous unit's operands are read
        for (int i = tid; i < 2 * (g.HC + 2) * g.P; i += kWgradThreads) {
            const int c = i & 1, slot = i >> 1;
            const int sy = slot / g.P, sx = slot - sy * g.P;
            const int y = y0 + sy - 1, x = x0 + sx - 1;
            const bool in = y >= 0 && y < d.H && x >= 0 && x < d.W;
            const bool own = in && sy >= 1 && sy <= g.HC && sx >= 1 && sx <= g.WC;
            const long long v = ((vol * d.D + z) * d.H + (in ? y : 0)) * d.W + (in ? x : 0);
            const uint32_t to = base + uint32_t((c * g.NSL + slot) * 16);
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(to), "l"(dZ + v * CH + c * 8), "r"(own ? 16 : 0) : "memory");
#pragma unroll
            for (int p = 0; p < 3; p++) {
                const int zz = z + p - 1;
                const bool ok = in && zz >= 0 && zz < d.D;
                const long long vx = ok ? v + (long long)(p - 1) * d.H * d.W : v;
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(to + uint32_t((1 + p) * plane_bytes)),
                             "l"(X + vx * CH + c * 8), "r"(ok ? 16 : 0) : "memory");
            }
        }
        asm volatile("cp.async.wait_all;\n" ::: "memory");
        __syncthreads();
        for (int t = split; t < g.nt; t += 2) {
            const int s0 = g.P + 1 + 16 * t;
            uint32_t a[4];
            ldsm4t(a, a_lane + uint32_t(s0 * 16));
#pragma unroll
            for (int o = 0; o < 9; o++) {
                uint32_t b[4];
                ldsm4t(b, b_lane + uint32_t((s0 + (o / 3 - 1) * g.P + (o % 3 - 1)) * 16));
                mma16816(acc[o][0], a, b[0], b[1]);
                mma16816(acc[o][1], a, b[2], b[3]);
            }
            if (dz == 1) mma16816(bacc, a, 0x3F803F80u, 0x3F803F80u);   // times one: the sum over the voxels
        }
        if (++held == kWgradUnits) {
            flush();
            clear();
            held = 0;
        }
    }
    flush();
    __syncthreads();
    for (int i = tid; i < kSums / 4; i += kWgradThreads) {
        const float4 v = reinterpret_cast<const float4*>(sums)[i];
        asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(dW + 4 * i), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w) : "memory");
    }
}

// Rounds weight i of layer `layer` (FP32 [27][16 out][16 in]) to its BF16 copies for the forward product and, flipped
// and transposed, for the backward data product: Wb[o'][k][m] = W[26 - o'][m][k].
constexpr int PER_LAYER = TAPS * CH * CH + CH;   // weights, then biases
__device__ __forceinline__ void round_weight(int layer, int i, float w, __nv_bfloat16* __restrict__ Wf, __nv_bfloat16* __restrict__ Wb) {
    const int o = i / (CH * CH), m = (i / CH) % CH, k = i % CH;
    const __nv_bfloat16 b = __float2bfloat16_rn(w);
    Wf[size_t(layer) * TAPS * CH * CH + i] = b;
    Wb[size_t(layer) * TAPS * CH * CH + ((TAPS - 1 - o) * CH + k) * CH + m] = b;
}
__global__ void weights_kernel(const float* __restrict__ p, int n, __nv_bfloat16* __restrict__ Wf, __nv_bfloat16* __restrict__ Wb) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int layer = i / PER_LAYER, j = i - layer * PER_LAYER;
    if (j < TAPS * CH * CH) round_weight(layer, j, p[i], Wf, Wb);
}

// Adam (Kingma & Ba 2015) with bias correction, on n parameters, and the BF16 copies of the new weights.
__global__ void adam_kernel(float* __restrict__ p, const float* __restrict__ grad, float* __restrict__ m, float* __restrict__ v,
                            int n, float lr, float b1, float b2, float eps, float c1, float c2, __nv_bfloat16* __restrict__ Wf,
                            __nv_bfloat16* __restrict__ Wb) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float gr = grad[i];
    const float mi = b1 * m[i] + (1.f - b1) * gr, vi = b2 * v[i] + (1.f - b2) * gr * gr;
    m[i] = mi;
    v[i] = vi;
    const float w = p[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    p[i] = w;
    const int layer = i / PER_LAYER, j = i - layer * PER_LAYER;
    if (j < TAPS * CH * CH) round_weight(layer, j, w, Wf, Wb);
}

// What a gradient call leaves for the host: the weighted squared error, the sum of the weights, and the flag of a
// tcgen05 wait that ran out.
struct Status {
    double loss, weights;
    int err;
};

// Sum of a value per thread over the CTA (256 threads), at thread 0.
__device__ __forceinline__ double cta_sum(double s) {
    __shared__ double red[8];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
    __syncthreads();
    double t = 0.0;
    if (threadIdx.x == 0)
        for (int k = 0; k < 8; k++) t += red[k];
    return t;
}

// Sum of the loss weights (their count is the denominator of the mean), in FP64.
__global__ void __launch_bounds__(256) weight_sum_kernel(const float* __restrict__ weight, long long N, Status* st) {
    double s = 0.0;
    for (long long v = (long long)(blockIdx.x) * blockDim.x + threadIdx.x; v < N; v += (long long)(gridDim.x) * blockDim.x) {
        const float w = weight[v];
        if (w != 0.f) s += double(w);
    }
    s = cta_sum(s);
    if (threadIdx.x == 0 && s != 0.0) atomicAdd(&st->weights, s);
}

// Prediction = skip + Z (first `nout` channels), FP32 [N][nout].
__global__ void __launch_bounds__(256) predict_kernel(const __nv_bfloat16* __restrict__ Z, const float* __restrict__ skip,
                                                      long long N, int nout, float* __restrict__ pred) {
    const long long v = (long long)(blockIdx.x) * blockDim.x + threadIdx.x;
    if (v >= N) return;
    if (nout == 4 && ((reinterpret_cast<uintptr_t>(skip) | reinterpret_cast<uintptr_t>(pred)) & 15) == 0) {
        const uint2 z = *reinterpret_cast<const uint2*>(Z + v * CH);
        const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&z.x));
        const float2 b = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&z.y));
        float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
        if (skip) s = reinterpret_cast<const float4*>(skip)[v];
        reinterpret_cast<float4*>(pred)[v] = make_float4(a.x + s.x, a.y + s.y, b.x + s.z, b.y + s.w);
        return;
    }
    for (int c = 0; c < nout; c++) pred[v * nout + c] = __bfloat162float(Z[v * CH + c]) + (skip ? skip[v * nout + c] : 0.f);
}

// Squared error of skip + Z against the target over the voxels `weight` marks, summed in FP64; dZ = 2 weight
// (pred - target) / count as BF16 (other channels 0), count = nout times the sum of the weights.  WIDE: four channels
// and 16-byte aligned inputs, one load each.  Bound: latency.  With four 2- and 4-byte loads per input, and the FP64
// sum in every lane for all 16 channels (predicated off, which the FP64 pipe takes as long for: 80 % busy), 32 volumes
// of 18^3 took 22.7 us; 6.6 now that warps without a weighted voxel branch past the sum.
template <bool WIDE>
__global__ void __launch_bounds__(256) loss_kernel(const __nv_bfloat16* __restrict__ Z, const float* __restrict__ skip,
                                                   const float* __restrict__ target, const float* __restrict__ weight,
                                                   long long N, int nout, __nv_bfloat16* __restrict__ dZ, Status* st) {
    constexpr int NC = WIDE ? 4 : CH;
    const long long v = (long long)(blockIdx.x) * blockDim.x + threadIdx.x;
    double s = 0.0;
    __shared__ float inv_count;   // one FP64 division per CTA
    if (threadIdx.x == 0) inv_count = float(1.0 / (st->weights * double(nout)));
    float e[NC], w = 0.f;
    bool sum = false;
    if (v < N) {
        w = weight ? weight[v] : 1.f;
        if (WIDE) {
            const uint2 z = *reinterpret_cast<const uint2*>(Z + v * CH);
            const float4 t = reinterpret_cast<const float4*>(target)[v];
            const float4 k = skip ? reinterpret_cast<const float4*>(skip)[v] : make_float4(0.f, 0.f, 0.f, 0.f);
            const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&z.x));
            const float2 b = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&z.y));
            e[0] = a.x + k.x - t.x;
            e[1] = a.y + k.y - t.y;
            e[2] = b.x + k.z - t.z;
            e[3] = b.y + k.w - t.w;
        } else {
#pragma unroll
            for (int c = 0; c < NC; c++)
                e[c] = c < nout ? __bfloat162float(Z[v * CH + c]) + (skip ? skip[v * nout + c] : 0.f) - target[v * nout + c] : 0.f;
        }
        sum = w != 0.f;
#pragma unroll
        for (int c = 0; c < NC; c++) sum |= !(fabsf(e[c]) < INFINITY);   // 0 e^2 is NaN for an infinite e
    }
    if (__any_sync(0xFFFFFFFFu, sum)) {
#pragma unroll
        for (int c = 0; c < NC; c++)
            if ((WIDE || c < nout) && sum) s += double(w) * double(e[c]) * double(e[c]);
    }
    if (__syncthreads_or(sum)) {
        s = cta_sum(s);
        if (threadIdx.x == 0 && s != 0.0) atomicAdd(&st->loss, s);
    }
    if (v < N) {
        uint32_t out[CH / 2] = {};
#pragma unroll
        for (int c = 0; c < NC; c++) {
            const float g = WIDE || c < nout ? 2.f * w * e[c] * inv_count : 0.f;
            const uint32_t b = __bfloat16_as_ushort(__float2bfloat16_rn(g));
            out[c >> 1] |= b << (16 * (c & 1));
        }
        uint4* dst = reinterpret_cast<uint4*>(dZ + v * CH);
        dst[0] = make_uint4(out[0], out[1], out[2], out[3]);
        dst[1] = make_uint4(out[4], out[5], out[6], out[7]);
    }
}

// ---------------------------------------------------------------- host side

lbm_status nfail(lbm_status s, const char* msg) {
    lbm::set_last_error(msg);
    return s;
}

#define NCU(call)                                                                      \
    do {                                                                               \
        cudaError_t e_ = (call);                                                       \
        if (e_ != cudaSuccess) {                                                       \
            char b_[256];                                                              \
            snprintf(b_, sizeof b_, "%s failed: %s", #call, cudaGetErrorString(e_));   \
            return nfail(e_ == cudaErrorMemoryAllocation ? LBM_ENOMEM : LBM_ECUDA, b_); \
        }                                                                              \
    } while (0)

// SplitMix64 (Steele, Lea & Flood 2014), for the weight initialisation.
uint64_t splitmix(uint64_t& s) {
    uint64_t z = (s += 0x9E3779B97F4A7C15ULL);
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
    return z ^ (z >> 31);
}

}  // namespace

struct lbm_net {
    int layers = 0, cin = 0, cout = 0;
    cudaStream_t stream = nullptr;
    cudaStream_t side = nullptr;           // the copy of the input beside the layers
    cudaEvent_t ev[2] = {nullptr, nullptr};
    float* params = nullptr;   // per layer: W [27][16][16], b [16]
    float* grads = nullptr;    // of the last gradient call that was accepted
    float* gsum = nullptr;     // sums of the call at work; the two change places when it is accepted
    float* m = nullptr;
    float* v = nullptr;
    __nv_bfloat16* wf = nullptr;   // per layer: forward BF16 weights
    __nv_bfloat16* wb = nullptr;   // per layer: backward-data BF16 weights
    int64_t step = 0;
    // activations of the last forward pass: X_0 .. X_{L-1}, Z_{L-1}; and two gradient buffers
    std::vector<__nv_bfloat16*> act;
    __nv_bfloat16* g0 = nullptr;
    __nv_bfloat16* g1 = nullptr;
    long long cap = 0;       // voxels the activation buffers hold
    Status* d_st = nullptr;  // loss, weight sum and the tcgen05 kernel's timeout flag
    Status* h_st = nullptr;  // pinned
    int backend = 1;         // 1: tcgen05 products where the volume fits, 0: mma.sync only
    int wait_test = 0;       // 1: the tcgen05 kernel issues no products, so its bounded wait runs out
    int sms = 0;
    Dims d{};
    lbm::DevMem mem;         // device memory: the caller's allocator hook or cudaMalloc
};

namespace {

void free_acts(lbm_net* n) {
    for (auto* p : n->act) n->mem.put(p);
    n->act.clear();
    n->mem.put(n->g0);
    n->mem.put(n->g1);
    n->g0 = n->g1 = nullptr;
    n->cap = 0;
}

lbm_status ensure_acts(lbm_net* n, long long N) {
    if (n->cap >= N) return LBM_OK;
    free_acts(n);
    const size_t bytes = size_t(N) * CH * sizeof(__nv_bfloat16);
    for (int l = 0; l <= n->layers; l++) {
        __nv_bfloat16* p = nullptr;
        if (!n->mem.get(&p, bytes)) {
            free_acts(n);
            return nfail(LBM_ENOMEM, "cannot allocate the activations");
        }
        n->act.push_back(p);
    }
    if (!n->mem.get(&n->g0, bytes) || !n->mem.get(&n->g1, bytes)) {
        free_acts(n);
        return nfail(LBM_ENOMEM, "cannot allocate the activation gradients");
    }
    n->cap = N;
    return LBM_OK;
}

// Units of conv_tc_kernel: parts of at most 128 groups of four slots (the MMA's rows), rows of at most 64 slots so that
// the border costs little, and runs of planes that fill the CTAs evenly.
TcGeom tc_geometry(const Dims& d, int sms) {
    TcGeom g{};
    g.nx = (d.W + 61) / 62;
    g.WC = (d.W + g.nx - 1) / g.nx;
    g.nx = (d.W + g.WC - 1) / g.WC;
    g.P = (g.WC + 2 + 3) & ~3;
    const int rows = 512 / g.P;
    g.ny = (d.H + rows - 1) / rows;
    g.HC = (d.H + g.ny - 1) / g.ny;
    g.ny = (d.H + g.HC - 1) / g.HC;
    g.NG = (g.HC + 2) * g.P / 4 + 1;
    // the last plane's operands run to 128 groups from a row's first, which may pass the ring's end
    g.smem = size_t(TC_A_OFF) + (size_t(TC_RING) * 8 * g.NG + 128 + g.P) * 16;
    const int per_sm = int(std::min<size_t>(228 * 1024 / (g.smem + 1024), 512 / (2 * TC_COLS)));
    const long long parts = (long long)d.nvol * g.ny * g.nx, ctas = (long long)sms * per_sm;
    // planes per run: the fewest rounds of (planes + what a run costs besides, about one plane) over the CTAs
    double best = 1e300;
    for (int nz = 1; nz <= d.D && nz <= 64; nz++) {
        const int zc = (d.D + nz - 1) / nz;
        const long long units = parts * ((d.D + zc - 1) / zc);
        const double cost = double((units + ctas - 1) / ctas) * (zc + 1.0);
        if (cost < best * 0.999) {
            best = cost;
            g.ZC = zc;
        }
    }
    g.nz = (d.D + g.ZC - 1) / g.ZC;
    g.grid = int(std::min<long long>(parts * g.nz, ctas));
    return g;
}
constexpr size_t kTcSmem = TC_A_OFF + (size_t(TC_RING) * 8 * (512 / 4 + 2 * 64 / 4 + 1) + 128 + 64) * 16;   // the most

// Z = conv(X) (+ bias, activation) with the tensor-core kernel the net is set to use.
lbm_status conv(lbm_net* n, const __nv_bfloat16* X, const __nv_bfloat16* Wt, const float* bias, __nv_bfloat16* Z,
                const Dims& d, int act, const __nv_bfloat16* mask) {
    if (n->backend == 1 && (long long)d.H * d.W < (1LL << 29)) {
        const TcGeom g = tc_geometry(d, n->sms);
        NCU(cudaFuncSetAttribute(conv_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, int(kTcSmem)));
        conv_tc_kernel<<<g.grid, TC_THREADS, g.smem, n->stream>>>(X, Wt, bias, Z, d, act, mask, g, &n->d_st->err, n->wait_test);
    } else {
        conv_kernel<<<int((d.N + 127) / 128), 256, 0, n->stream>>>(X, Wt, bias, Z, d, act, mask);
    }
    NCU(cudaGetLastError());
    return LBM_OK;
}

// Reads the status back (synchronises the stream); LBM_ETIMEOUT if a tcgen05 wait ran out since the last check.
lbm_status check_err(lbm_net* n) {
    NCU(cudaMemcpyAsync(n->h_st, n->d_st, sizeof(Status), cudaMemcpyDeviceToHost, n->stream));
    NCU(cudaStreamSynchronize(n->stream));
    if (n->h_st->err) {
        NCU(cudaMemset(&n->d_st->err, 0, sizeof(int)));
        return nfail(LBM_ETIMEOUT, "a tensor-core wait ran out; the outputs of this call are incomplete");
    }
    return LBM_OK;
}

// Units of wgrad_kernel: whole planes where their staging fits in kWgradStage (two CTAs per SM with the sums),
// else parts, the longer side halved until they do.
constexpr size_t kWgradStage = 80 * 1024;
WgradGeom wgrad_geometry(const Dims& d) {
    WgradGeom g{};
    auto bytes = [&](int h, int w) {
        g.P = w + 2;
        g.NSL = ((h + 2) * g.P + 18 + 7) & ~7;
        return size_t(4) * 2 * g.NSL * 16;
    };
    g.HC = d.H;
    g.WC = d.W;
    while (bytes(g.HC, g.WC) > kWgradStage) {
        if (g.HC >= g.WC) g.HC = (g.HC + 1) / 2;
        else g.WC = (g.WC + 1) / 2;
    }
    g.ny = (d.H + g.HC - 1) / g.HC;
    g.nx = (d.W + g.WC - 1) / g.WC;
    g.smem = bytes(g.HC, g.WC) + size_t(PER_LAYER) * 4;
    g.nt = (g.HC * g.P + 15) / 16;
    g.units = (long long)d.nvol * d.D * g.ny * g.nx;
    return g;
}

lbm_status refresh_weights(lbm_net* n) {
    const int np = n->layers * PER_LAYER;
    weights_kernel<<<(np + 255) / 256, 256, 0, n->stream>>>(n->params, np, n->wf, n->wb);
    NCU(cudaGetLastError());
    return LBM_OK;
}

lbm_status check_dims(int D, int H, int W, int nvol, Dims& d) {
    if (D < 1 || H < 1 || W < 1 || nvol < 1) return nfail(LBM_EINVAL, "volume dimensions must be positive");
    d.D = D;
    d.H = H;
    d.W = W;
    d.nvol = nvol;
    d.V = (long long)D * H * W;
    d.N = d.V * nvol;
    if (d.N > (1LL << 40)) return nfail(LBM_EINVAL, "too many voxels");
    return LBM_OK;
}

// Forward pass over x (BF16 [N][16]); keeps every layer's input for the backward pass.  n->d stays empty until every
// layer is enqueued, so that no gradient follows a pass that was refused.
lbm_status forward(lbm_net* n, const __nv_bfloat16* x, const Dims& d) {
    n->d = Dims{};
    lbm_status s = ensure_acts(n, d.N);
    if (s) return s;
    // The copy of the input that a later gradient needs runs beside the layers (512 volumes of 18^3: 32 us, the
    // layers are far from the memory rate; a forward pass with features and loss 950 -> 926 us); the first layer reads the
    // input itself where its alignment allows.
    const bool beside = (reinterpret_cast<uintptr_t>(x) & 15) == 0;
    if (beside) {
        NCU(cudaEventRecord(n->ev[0], n->stream));
        NCU(cudaStreamWaitEvent(n->side, n->ev[0], 0));
    }
    NCU(cudaMemcpyAsync(n->act[0], x, size_t(d.N) * CH * sizeof(__nv_bfloat16), cudaMemcpyDeviceToDevice, beside ? n->side : n->stream));
    if (beside) NCU(cudaEventRecord(n->ev[1], n->side));
    lbm_status st = LBM_OK;
    for (int l = 0; l < n->layers; l++) {
        const float* b = n->params + size_t(l) * PER_LAYER + TAPS * CH * CH;
        st = conv(n, l == 0 && beside ? x : n->act[l], n->wf + size_t(l) * TAPS * CH * CH, b, n->act[l + 1], d,
                             l + 1 < n->layers ? 1 : 0, nullptr);
        if (st) break;
    }
    if (beside) NCU(cudaStreamWaitEvent(n->stream, n->ev[1], 0));   // also on failure: the copy still reads x
    if (st) return st;
    n->d = d;
    return LBM_OK;
}

}  // namespace

extern "C" {

lbm_status lbm_net_create(int32_t layers, int32_t in_channels, int32_t out_channels, uint64_t seed, void* stream,
                          const lbm_allocator* alloc, lbm_net** out) {
    if (!out) return nfail(LBM_EINVAL, "out is NULL");
    *out = nullptr;
    if (layers < 1 || layers > 16 || in_channels < 1 || in_channels > CH || out_channels < 1 || out_channels > CH)
        return nfail(LBM_EINVAL, "layers must be 1..16 and channel counts 1..16");
    lbm_net* n = new (std::nothrow) lbm_net;
    if (!n) return nfail(LBM_ENOMEM, "host allocation failed");
    n->layers = layers;
    n->cin = in_channels;
    n->cout = out_channels;
    n->stream = static_cast<cudaStream_t>(stream);
    if (!n->mem.bind(alloc, n->stream)) {
        delete n;
        return nfail(LBM_EINVAL, "an allocator hook with alloc needs release");
    }
    const size_t np = size_t(layers) * PER_LAYER;
    // He-uniform initialisation over the fan-in of each layer (27 taps x its input channels);
    // channels beyond a layer's inputs or outputs keep zero weights
    std::vector<float> h(np, 0.f);
    uint64_t st = seed;
    for (int l = 0; l < layers; l++) {
        const int ci = l == 0 ? in_channels : CH, co = l + 1 == layers ? out_channels : CH;
        const float bound = std::sqrt(6.f / float(TAPS * ci));
        for (int o = 0; o < TAPS; o++)
            for (int m = 0; m < co; m++)
                for (int k = 0; k < ci; k++) {
                    const double u = double(splitmix(st) >> 11) * (1.0 / 9007199254740992.0);
                    h[size_t(l) * PER_LAYER + (o * CH + m) * CH + k] = float((2.0 * u - 1.0) * bound);
                }
    }
    auto bail = [&](lbm_status s) {
        std::string keep = lbm_last_error();
        lbm_net_destroy(n);
        lbm::set_last_error(keep.c_str());
        return s;
    };
    if (!n->mem.get(&n->params, np * 4) || !n->mem.get(&n->grads, np * 4) || !n->mem.get(&n->gsum, np * 4) ||
        !n->mem.get(&n->m, np * 4) ||
        !n->mem.get(&n->v, np * 4) || !n->mem.get(&n->wf, size_t(layers) * TAPS * CH * CH * 2) ||
        !n->mem.get(&n->wb, size_t(layers) * TAPS * CH * CH * 2) || !n->mem.get(&n->d_st, sizeof(Status)) ||
        cudaMallocHost(&n->h_st, sizeof(Status)) != cudaSuccess)
        return bail(nfail(LBM_ENOMEM, "cannot allocate the net"));
    if (cudaStreamCreateWithFlags(&n->side, cudaStreamNonBlocking) != cudaSuccess ||
        cudaEventCreateWithFlags(&n->ev[0], cudaEventDisableTiming) != cudaSuccess ||
        cudaEventCreateWithFlags(&n->ev[1], cudaEventDisableTiming) != cudaSuccess)
        return bail(nfail(LBM_ECUDA, "cannot create the copy stream"));
    if (cudaMemcpy(n->params, h.data(), np * 4, cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemset(n->m, 0, np * 4) != cudaSuccess || cudaMemset(n->v, 0, np * 4) != cudaSuccess ||
        cudaMemset(n->d_st, 0, sizeof(Status)) != cudaSuccess)
        return bail(nfail(LBM_ECUDA, "cannot initialise the net"));
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&n->sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return bail(nfail(LBM_ECUDA, "no CUDA device"));
    lbm_status s = refresh_weights(n);
    if (s) return bail(s);
    *out = n;
    return LBM_OK;
}

lbm_status lbm_net_destroy(lbm_net* n) {
    if (!n) return LBM_OK;
    if (n->stream) cudaStreamSynchronize(n->stream);
    free_acts(n);
    for (const void* p : {static_cast<const void*>(n->params), static_cast<const void*>(n->grads),
                          static_cast<const void*>(n->gsum), static_cast<const void*>(n->m), static_cast<const void*>(n->v),
                          static_cast<const void*>(n->wf), static_cast<const void*>(n->wb),
                          static_cast<const void*>(n->d_st)})
        n->mem.put(p);
    if (n->h_st) cudaFreeHost(n->h_st);
    if (n->side) cudaStreamDestroy(n->side);
    for (cudaEvent_t e : n->ev)
        if (e) cudaEventDestroy(e);
    delete n;
    return LBM_OK;
}

lbm_status lbm_net_num_params(const lbm_net* n, int64_t* count) {
    if (!n || !count) return nfail(LBM_EINVAL, "NULL argument");
    *count = int64_t(n->layers) * PER_LAYER;
    return LBM_OK;
}

lbm_status lbm_net_get_params(const lbm_net* n, float* host) {
    if (!n || !host) return nfail(LBM_EINVAL, "NULL argument");
    NCU(cudaStreamSynchronize(n->stream));
    NCU(cudaMemcpy(host, n->params, size_t(n->layers) * PER_LAYER * 4, cudaMemcpyDeviceToHost));
    return LBM_OK;
}

lbm_status lbm_net_set_params(lbm_net* n, const float* host) {
    if (!n || !host) return nfail(LBM_EINVAL, "NULL argument");
    NCU(cudaStreamSynchronize(n->stream));
    NCU(cudaMemcpy(n->params, host, size_t(n->layers) * PER_LAYER * 4, cudaMemcpyHostToDevice));
    return refresh_weights(n);
}

lbm_status lbm_net_forward(lbm_net* n, const void* x, int32_t D, int32_t H, int32_t W, int32_t nvol, void* z) {
    if (!n || !x || !z) return nfail(LBM_EINVAL, "NULL argument");
    Dims d;
    lbm_status s = check_dims(D, H, W, nvol, d);
    if (s || (s = forward(n, static_cast<const __nv_bfloat16*>(x), d))) return s;
    NCU(cudaMemcpyAsync(z, n->act[n->layers], size_t(d.N) * CH * 2, cudaMemcpyDeviceToDevice, n->stream));
    return check_err(n);
}

lbm_status lbm_net_predict(lbm_net* n, const void* x, const float* skip, int32_t D, int32_t H, int32_t W, int32_t nvol,
                           float* pred) {
    if (!n || !x || !pred) return nfail(LBM_EINVAL, "NULL argument");
    Dims d;
    lbm_status s = check_dims(D, H, W, nvol, d);
    if (s || (s = forward(n, static_cast<const __nv_bfloat16*>(x), d))) return s;
    predict_kernel<<<int((d.N + 255) / 256), 256, 0, n->stream>>>(n->act[n->layers], skip, d.N, n->cout, pred);
    NCU(cudaGetLastError());
    return check_err(n);
}

lbm_status lbm_net_train_step(lbm_net* n, const void* x, const float* skip, const float* target, const float* weight,
                              int32_t D, int32_t H, int32_t W, int32_t nvol, float lr, double* loss) {
    if (!n || !x || !target) return nfail(LBM_EINVAL, "NULL argument");
    Dims d;
    lbm_status s = check_dims(D, H, W, nvol, d);
    if (s || (s = forward(n, static_cast<const __nv_bfloat16*>(x), d))) return s;
    lbm_status r = lbm_net_gradient(n, skip, target, weight, loss);
    if (r) return r;
    n->step++;
    const float b1 = 0.9f, b2 = 0.999f;
    const float c1 = float(1.0 - std::pow(double(b1), double(n->step))), c2 = float(1.0 - std::pow(double(b2), double(n->step)));
    const int np = n->layers * PER_LAYER;
    adam_kernel<<<(np + 255) / 256, 256, 0, n->stream>>>(n->params, n->grads, n->m, n->v, np, lr, b1, b2, 1e-8f, c1, c2, n->wf,
                                                        n->wb);
    NCU(cudaGetLastError());
    return LBM_OK;
}

lbm_status lbm_net_gradient(lbm_net* n, const float* skip, const float* target, const float* weight, double* loss) {
    if (!n || !target) return nfail(LBM_EINVAL, "NULL argument");
    if (n->act.empty() || n->d.N == 0) return nfail(LBM_EINVAL, "run a forward pass first");
    const Dims& d = n->d;
    // the sum of the weights stays on the device until the loss is read (the MSE denominator is nout times it)
    NCU(cudaMemsetAsync(n->d_st, 0, offsetof(Status, err), n->stream));
    NCU(cudaMemsetAsync(n->gsum, 0, size_t(n->layers) * PER_LAYER * 4, n->stream));
    if (weight) {
        weight_sum_kernel<<<int(std::min<long long>((d.N + 255) / 256, 2LL * n->sms)), 256, 0, n->stream>>>(weight, d.N, n->d_st);
    } else {
        n->h_st->weights = double(d.N);
        NCU(cudaMemcpyAsync(&n->d_st->weights, &n->h_st->weights, sizeof(double), cudaMemcpyHostToDevice, n->stream));
    }
    const bool wide = n->cout == 4 && ((reinterpret_cast<uintptr_t>(skip) | reinterpret_cast<uintptr_t>(target)) & 15) == 0;
    (wide ? loss_kernel<true> : loss_kernel<false>)<<<int((d.N + 255) / 256), 256, 0, n->stream>>>(
        n->act[n->layers], skip, target, weight, d.N, n->cout, n->g0, n->d_st);
    const WgradGeom g = wgrad_geometry(d);
    NCU(cudaFuncSetAttribute(wgrad_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, int(kWgradStage + PER_LAYER * 4)));
    const int wgrid = int(std::min<long long>(g.units, 2LL * n->sms));
    __nv_bfloat16* dz = n->g0;
    __nv_bfloat16* dx = n->g1;
    // A layer's weight gradient runs on the side stream beside its data gradient, which reads the same dz; the next
    // layer's data gradient overwrites dz, so the two join before it.  32 volumes of 18^3, where neither fills the SMs
    // for its whole time: a training step 316 -> 297 us.
    lbm_status cs = LBM_OK;
    for (int l = n->layers - 1; l >= 0 && !cs; l--) {
        NCU(cudaEventRecord(n->ev[0], n->stream));
        NCU(cudaStreamWaitEvent(n->side, n->ev[0], 0));
        wgrad_kernel<<<wgrid, kWgradThreads, g.smem, n->side>>>(n->act[l], dz, n->gsum + size_t(l) * PER_LAYER, d, g);
        if (l > 0) {
            cs = conv(n, dz, n->wb + size_t(l) * TAPS * CH * CH, nullptr, dx, d, 2, n->act[l]);
            std::swap(dz, dx);
        }
        NCU(cudaEventRecord(n->ev[1], n->side));
        NCU(cudaStreamWaitEvent(n->stream, n->ev[1], 0));
    }
    if (cs) return cs;
    NCU(cudaGetLastError());
    const lbm_status st = check_err(n);
    const double count = n->h_st->weights * n->cout;
    if (st) return st;
    // known only now, after sums over NaN (the loss divides by the count): they are not published
    if (!(count > 0.0)) return nfail(LBM_EINVAL, "the loss weights are all zero");
    std::swap(n->grads, n->gsum);
    if (loss) *loss = n->h_st->loss / count;
    return LBM_OK;
}

lbm_status lbm_net_set_wait_test(lbm_net* n, int32_t on) {
    if (!n) return nfail(LBM_EINVAL, "net is NULL");
    n->wait_test = on ? 1 : 0;
    return LBM_OK;
}

lbm_status lbm_net_set_backend(lbm_net* n, int32_t backend) {
    if (!n || (backend != 0 && backend != 1)) return nfail(LBM_EINVAL, "backend must be 0 (mma.sync) or 1 (tcgen05)");
    n->backend = backend;
    return LBM_OK;
}

lbm_status lbm_net_get_grads(const lbm_net* n, float* host) {
    if (!n || !host) return nfail(LBM_EINVAL, "NULL argument");
    NCU(cudaStreamSynchronize(n->stream));
    NCU(cudaMemcpy(host, n->grads, size_t(n->layers) * PER_LAYER * 4, cudaMemcpyDeviceToHost));
    return LBM_OK;
}

}  // extern "C"

// ---------------------------------------------------------------- warm-start data movement
namespace {

// Coarse-only solution on a full level-0 grid of nb[3] blocks of B^3 cells, block-major in the
// forest's order (block (bx, by, bz) is block (bz nb1 + by) nb0 + bx).  Value of component `comp`
// of a field [ncomp][n0] at cell (i, j, k), with periodic axes wrapped and walled axes clamped.
struct Coarse {
    const double* rho;
    const double* u;
    long long n0;
    int nb[3], B, per;
    __device__ __forceinline__ int fold(int i, int a) const {
        const int N = nb[a] * B;
        if ((per >> a) & 1) return ((i % N) + N) % N;
        return i < 0 ? 0 : (i >= N ? N - 1 : i);
    }
    __device__ __forceinline__ long long index(int i, int j, int k) const {
        i = fold(i, 0);
        j = fold(j, 1);
        k = fold(k, 2);
        const long long blk = ((long long)(k / B) * nb[1] + j / B) * nb[0] + i / B;
        return blk * B * B * B + ((long long)(k % B) * B + j % B) * B + i % B;
    }
};

// Features of the voxels of z-plane `vz` of the volume around block `blk` of level L: the coarse solution
// sampled trilinearly at each voxel's cell centre (Sec. 2: cell-centred values), the obstacle / outside-domain
// flag and the level.  One CTA per (volume, plane, part of T x T voxels of the plane, T <= kFeatTile).
// A cell centre lies n / 2^(L + 1) coarse cells from the first cell's centre, n = 2 g + 1 - 2^L for the cell's
// level-L coordinate g, so its coarse cell and its weights follow from integers, exactly.  The interpolation runs
// axis by axis over the plane: the coarse cells under it at its z (two values each, in FP64), those at each voxel
// row's y, then the voxels along x.  FP64 operations bound the kernel, at 1.7 a clock and SM: with eight corners and
// all spheres per voxel it took 100 a voxel (512 volumes of 18^3 at level 1: 834 us), axis by axis 20 (279 us).  Now
// the passes along y and x run in integers that keep every bit (see `fixed`), no division is left, and FP32 decides on a
// sphere wherever its error allows, which leaves the z pass: 95 us (85 with 64-bit integers alone, which cut values far
// below the plane's largest).  Spheres whose box distance to the plane exceeds their radius are left out before the
// voxels test them.  128 threads: the passes of a plane of 18^2 are 121, 198 and 324 items long and end in barriers
// (64-bit integers, 256 threads: 114 us, 192 99, 128 and 96 85).
constexpr int kFeatThreads = 128;
constexpr int kFeatSpheres = 64;   // spheres tested per round
constexpr int kFeatTile = 32;

__global__ void __launch_bounds__(kFeatThreads) features_kernel(Coarse c, int level, int B, int halo, const int* __restrict__ blocks,
                                                                const double* __restrict__ spheres, int nspheres, double rho_scale,
                                                                double u_scale, int T, int nt, __nv_bfloat16* __restrict__ x, float* __restrict__ skip) {
    extern __shared__ long long fsm[];
    __shared__ int near_[kFeatSpheres];
    __shared__ float4 rel_[kFeatSpheres];   // a sphere's centre from the plane's first voxel, and its radius squared
    __shared__ float tie_[kFeatSpheres];    // below this difference FP64 decides
    __shared__ int nnear;
    __shared__ int wgt[2][kFeatTile];       // weight of the upper coarse cell along x and y, of 2^(L + 1)
    __shared__ int at[2][kFeatTile];        // the lower coarse cell, from the part's first
    __shared__ int top[4], low[4];          // the largest exponent of each component on the plane, and of its non-zero values the smallest
    __shared__ double wz[4];                // weights along z times the scales: density lower, upper, velocity lower, upper
    const int D = B + 2 * halo;
    const int tile = int(blockIdx.x % unsigned(nt * nt));
    const int unit = int(blockIdx.x / unsigned(nt * nt));
    const int b = unit / D, vz = unit - b * D;
    const int x0 = (tile % nt) * T, y0 = (tile / nt) * T;
    const int TX = min(T, D - x0), TY = min(T, D - y0);
    const int tid = threadIdx.x;
    const int g0[3] = {blocks[3 * b] * B - halo + x0, blocks[3 * b + 1] * B - halo + y0, blocks[3 * b + 2] * B - halo};
    // coarse cell below the level-L cell g along an axis (before wrapping), and the weight of the cell above it
    const double wunit = __hiloint2double((1022 - level) << 20, 0);   // 2^-(L + 1)
    auto cell = [&](int g) { return (2 * g + 1 - (1 << level)) >> (level + 1); };
    auto weight = [&](int g) { return (2 * g + 1 - (1 << level)) & ((2 << level) - 1); };
    const int cx0 = cell(g0[0]), cy0 = cell(g0[1]);
    if (tid < 2 * kFeatTile) {
        const int a = tid / kFeatTile, i = tid - a * kFeatTile;
        wgt[a][i] = weight(g0[a] + i);
        at[a][i] = cell(g0[a] + i) - (a == 0 ? cx0 : cy0);
    }
    const int ncx = cell(g0[0] + TX - 1) - cx0 + 2, ncy = cell(g0[1] + TY - 1) - cy0 + 2;
    // at the plane's z [4][ncy][ncx], and at each voxel row's y [4][TY][ncx]: bits of doubles, or the upper limbs of
    // whole numbers, whose lower limbs lie behind
    const int np = ncx * ncy, nr = TY * ncx;
    long long* const plane = fsm;
    long long* const rows = plane + 4 * np;
    uint32_t* const plane_lo = reinterpret_cast<uint32_t*>(rows + 4 * nr);
    uint32_t* const rows_lo = plane_lo + 4 * np;
    // i / ncx and i / TX for i < 34^2 (i times the reciprocal's error stays below 2^16)
    const unsigned by_ncx = (65535u + unsigned(ncx)) / unsigned(ncx), by_tx = (65535u + unsigned(TX)) / unsigned(TX);
    const int gz = g0[2] + vz, cz = cell(gz);
    if (tid < 4) {
        top[tid] = 0;
        low[tid] = 0x7FF;
        const int w1 = weight(gz);
        wz[tid] = double(tid & 1 ? w1 : (2 << level) - w1) * wunit * (tid < 2 ? rho_scale : u_scale);
    }
    __syncthreads();
    {
        int e[4] = {0, 0, 0, 0}, m[4] = {0x7FF, 0x7FF, 0x7FF, 0x7FF};
        for (int i = tid; i < np; i += kFeatThreads) {
            const int j = int((unsigned(i) * by_ncx) >> 16);
            double v[2][4];
#pragma unroll
            for (int h = 0; h < 2; h++) {
                const long long k = c.index(cx0 + i - j * ncx, cy0 + j, cz + h);
                const double rho = c.rho[k];
                // obstacle cells of the coarse solution hold no (finite) value
                const bool ok = (__double2hiint(rho) & 0x7FF00000) != 0x7FF00000;
                v[h][0] = ok ? rho - 1.0 : 0.0;
#pragma unroll
                for (int a = 0; a < 3; a++) v[h][1 + a] = ok ? c.u[a * c.n0 + k] : 0.0;
            }
#pragma unroll
            for (int a = 0; a < 4; a++) {
                const long long t = __double_as_longlong(wz[a ? 2 : 0] * v[0][a] + wz[a ? 3 : 1] * v[1][a]);
                plane[a * np + i] = t;
                const int x = max(int(t >> 52) & 0x7FF, 1);
                if (t << 1) {   // a component of zeros has no exponent
                    e[a] = max(e[a], x);
                    m[a] = min(m[a], x);
                }
            }
        }
#pragma unroll
        for (int a = 0; a < 4; a++) {
            const int hi = __reduce_max_sync(0xFFFFFFFFu, e[a]), lo = __reduce_min_sync(0xFFFFFFFFu, m[a]);
            if ((tid & 31) == 0 && hi > 0) {
                atomicMax(&top[a], hi);
                atomicMin(&low[a], lo);
            }
        }
    }
    __syncthreads();
    // The weights along y and x are whole numbers of 2^(L + 1)ths, so these two passes run in integers of an upper limb
    // of 64 bits and a lower one of 32: a plane's component is scaled by the power of two that puts its largest value
    // just below 2^(bits + 32), which leaves room for both weights.  Every bit of every value is kept, so that the float
    // is the only rounding (FP64 sums round each term to 2^-53), where the component's smallest value is not too far
    // below its largest (2^-39 of it at level 0, 2^-33 at level 3); other planes take FP64.  back: the power of two to a float,
    // with 2^-32 for the values that the lower limb reaches still in the normal range.
    const int bits = 62 - 2 * (level + 1);
    bool fixed = level <= 3;
    float back[4];
#pragma unroll
    for (int a = 0; a < 4; a++) {
        const int t = top[a] - 1022 - 62;
        // infinities and NaN, scales beyond a float's, values that would lose bits
        if (top[a] != 0 && (t < -118 || t > 127 || top[a] - low[a] > bits + 32 - 53)) fixed = false;
        back[a] = top[a] == 0 || !fixed ? 0.f : __int_as_float((t + 127) << 23);
    }
    if (fixed) {
        for (int i = tid; i < np; i += kFeatThreads)
#pragma unroll
            for (int a = 0; a < 4; a++) {
                const long long v = plane[a * np + i];
                const int e = int(v >> 52) & 0x7FF;
                const unsigned long long m = (unsigned long long)(v & 0xFFFFFFFFFFFFFLL) | (e ? 1ULL << 52 : 0ULL);
                const int sh = m ? bits + 32 - 53 - (top[a] - max(e, 1)) : 0;   // 0 to 39
                long long hi = (long long)(sh < 32 ? m >> (32 - sh) : m << (sh - 32));
                uint32_t lo = sh < 32 ? uint32_t(m) << sh : 0u;
                if (v < 0) {   // the two's complement of both limbs
                    lo = 0u - lo;
                    hi = -hi - (lo != 0u);
                }
                plane[a * np + i] = hi;
                plane_lo[a * np + i] = lo;
            }
        __syncthreads();
    }
    // w0 p + w1 q of two numbers, the lower limb's carry added
    auto mix = [](int w0, int w1, long long ph, uint32_t pl, long long qh, uint32_t ql, uint32_t& lo) {
        const unsigned long long l = (unsigned long long)(pl) * unsigned(w0) + (unsigned long long)(ql) * unsigned(w1);
        lo = uint32_t(l);
        return w0 * ph + w1 * qh + (long long)(l >> 32);
    };
    for (int i = tid; i < nr; i += kFeatThreads) {
        const int y = int((unsigned(i) * by_ncx) >> 16), cx = i - y * ncx;
        const int w1 = wgt[1][y], w0 = (2 << level) - w1, o = at[1][y] * ncx + cx;
        if (fixed) {
#pragma unroll
            for (int a = 0; a < 4; a++) {
                const int p = a * np + o;
                rows[a * nr + i] = mix(w0, w1, plane[p], plane_lo[p], plane[p + ncx], plane_lo[p + ncx], rows_lo[a * nr + i]);
            }
        } else {
#pragma unroll
            for (int a = 0; a < 4; a++)
                rows[a * nr + i] = __double_as_longlong(w0 * wunit * __longlong_as_double(plane[a * np + o]) +
                                                        w1 * wunit * __longlong_as_double(plane[a * np + o + ncx]));
        }
    }
    const float sf = __int_as_float((127 - level) << 23);   // 2^-L
    const long long Nf[3] = {(long long)(c.nb[0] * c.B) << level, (long long)(c.nb[1] * c.B) << level,
                             (long long)(c.nb[2] * c.B) << level};
    auto outside = [&](int g, int a) { return !((c.per >> a) & 1) && (g < 0 || g >= Nf[a]); };
    const long long first = (((long long)(b) * D + vz) * D + y0) * D + x0;
    const bool wide = ((reinterpret_cast<uintptr_t>(x) | reinterpret_cast<uintptr_t>(skip)) & 15) == 0;
    const int rounds = nspheres > 0 ? (nspheres + kFeatSpheres - 1) / kFeatSpheres : 1;
    for (int r = 0; r < rounds; r++) {
        // the spheres of this round that reach the plane's box of cell centres
        __syncthreads();
        if (tid == 0) nnear = 0;
        __syncthreads();
        const int sp = r * kFeatSpheres + tid;
        if (tid < kFeatSpheres && sp < nspheres) {
            // In FP32 from the plane's first voxel: distances squared are off by less than 2^-20 of `size`, the sum of
            // squares of what enters them (offset and extent along each axis, and the radius); FP64 decides below that.
            const double* q = spheres + 4 * sp;
            const float ext[3] = {float(TX - 1) * sf, float(TY - 1) * sf, 0.f};
            float c3[3], d2 = 0.f, size = 0.f;
#pragma unroll
            for (int a = 0; a < 3; a++) {
                c3[a] = float(q[a] - double(2 * (g0[a] + (a == 2 ? vz : 0)) + 1) * wunit);
                const float t = c3[a] < 0.f ? c3[a] : fmaxf(c3[a] - ext[a], 0.f), m = fabsf(c3[a]) + ext[a];
                d2 += t * t;
                size += m * m;
            }
            const float rad = float(q[3]), r2 = rad * rad, tie = (size + r2) * 0x1p-20f + 1e-30f;
            if (!(d2 - r2 > tie)) {
                const int k = atomicAdd(&nnear, 1);
                near_[k] = sp;
                rel_[k] = make_float4(c3[0], c3[1], c3[2], r2);
                tie_[k] = tie;
            }
        }
        __syncthreads();
        const bool last = r == rounds - 1;
        for (int i = tid; i < TX * TY; i += kFeatThreads) {
            const int y = int((unsigned(i) * by_tx) >> 16), vx = i - y * TX;
            const int g[3] = {g0[0] + vx, g0[1] + y, g0[2] + vz};
            const long long id = first + (long long)(y) * D + vx;
            __nv_bfloat16* xo = x + id * CH;
            // the flag of the rounds before this one waits in the output
            bool solid = r > 0 ? __bfloat162float(xo[4]) != 0.f : outside(g[0], 0) || outside(g[1], 1) || outside(g[2], 2);
            if (!solid) {
                const float px = float(vx) * sf, py = float(y) * sf;
                for (int k = 0; k < nnear && !solid; k++) {
                    const float4 c4 = rel_[k];
                    const float fx = px - c4.x, fy = py - c4.y, diff = fx * fx + fy * fy + c4.z * c4.z - c4.w;
                    solid = diff < 0.f;
                    if (fabsf(diff) > tie_[k]) continue;
                    const double* q = spheres + 4 * near_[k];
                    const double dx = double(2 * g[0] + 1) * wunit - q[0], dy = double(2 * g[1] + 1) * wunit - q[1],
                                 dz = double(2 * g[2] + 1) * wunit - q[2];
                    solid = dx * dx + dy * dy + dz * dz < q[3] * q[3];
                }
            }
            if (!last) {
                xo[4] = __float2bfloat16_rn(solid ? 1.f : 0.f);
                continue;
            }
            const int w1 = wgt[0][vx], w0 = (2 << level) - w1, o = y * ncx + at[0][vx];
            float f[4];
            if (fixed) {
#pragma unroll
                for (int a = 0; a < 4; a++) {
                    const int p = a * nr + o;
                    uint32_t lo;
                    const long long hi = mix(w0, w1, rows[p], rows_lo[p], rows[p + 1], rows_lo[p + 1], lo);
                    // one rounding to 24 bits: of both limbs where they fit in 64 bits, else of the upper one with a
                    // last bit for what lies below it
                    const bool both = (unsigned long long)(hi + (1LL << 30)) < (1ULL << 31);
                    const long long t = both ? (long long)((unsigned long long)(hi) << 32 | lo) : hi | (lo != 0u);
                    f[a] = __ll2float_rn(t) * (both ? 0x1p-32f : 1.f) * back[a];
                }
            } else {
#pragma unroll
                for (int a = 0; a < 4; a++)
                    f[a] = float(w0 * wunit * __longlong_as_double(rows[a * nr + o]) +
                                 w1 * wunit * __longlong_as_double(rows[a * nr + o + 1]));
            }
            const float flag = solid ? 1.f : 0.f, lev = float(level) * 0.5f;
            if (wide) {
                auto pack = [](float lo, float hi) {
                    const __nv_bfloat162 t = __floats2bfloat162_rn(lo, hi);
                    return *reinterpret_cast<const uint32_t*>(&t);
                };
                uint4* dst = reinterpret_cast<uint4*>(xo);
                dst[0] = make_uint4(pack(f[0], f[1]), pack(f[2], f[3]), pack(flag, lev), 0u);
                dst[1] = make_uint4(0u, 0u, 0u, 0u);
                if (skip) reinterpret_cast<float4*>(skip)[id] = make_float4(f[0], f[1], f[2], f[3]);
            } else {
                const float vals[6] = {f[0], f[1], f[2], f[3], flag, lev};
#pragma unroll
                for (int ch = 0; ch < CH; ch++) xo[ch] = __float2bfloat16_rn(ch < 6 ? vals[ch] : 0.f);
                if (skip)
                    for (int a = 0; a < 4; a++) skip[id * 4 + a] = f[a];
            }
        }
    }
}

// Refined solution (block-major rho[n], u[3][n] of one level) -> training targets on the interior
// of each volume; weight 1 there on fluid cells, 0 on the halo and on obstacle cells.
__global__ void targets_kernel(const double* __restrict__ rho, const double* __restrict__ u, long long n, int B, int halo,
                               int nblocks, double rho_scale, double u_scale, float* __restrict__ target,
                               float* __restrict__ weight) {
    const int D = B + 2 * halo;
    const long long V = (long long)D * D * D;
    const long long id = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (id >= V * nblocks) return;
    const int b = int(id / V);
    long long r = id - b * V;
    const int vx = int(r % D) - halo;
    r /= D;
    const int vy = int(r % D) - halo, vz = int(r / D) - halo;
    float t[4] = {0.f, 0.f, 0.f, 0.f};
    float w = 0.f;
    if (vx >= 0 && vx < B && vy >= 0 && vy < B && vz >= 0 && vz < B) {
        const long long k = (long long)b * B * B * B + ((long long)vz * B + vy) * B + vx;
        if (isfinite(rho[k])) {
            t[0] = float((rho[k] - 1.0) * rho_scale);
            for (int a = 0; a < 3; a++) t[1 + a] = float(u[a * n + k] * u_scale);
            w = 1.f;
        }
    }
    for (int a = 0; a < 4; a++) target[id * 4 + a] = t[a];
    weight[id] = w;
}

// Prediction on the interior of each volume -> block-major rho[n], u[3][n] of one level.
__global__ void fields_kernel(const float* __restrict__ pred, int B, int halo, int nblocks, double rho_scale,
                              double u_scale, double* __restrict__ rho, double* __restrict__ u) {
    const long long n = (long long)nblocks * B * B * B;
    const long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    const int b = int(k / ((long long)B * B * B));
    long long r = k - (long long)b * B * B * B;
    const int x = int(r % B);
    r /= B;
    const int y = int(r % B), z = int(r / B);
    const int D = B + 2 * halo;
    const long long id = (long long)b * D * D * D + ((long long)(z + halo) * D + (y + halo)) * D + (x + halo);
    rho[k] = 1.0 + double(pred[id * 4]) / rho_scale;
    for (int a = 0; a < 3; a++) u[a * n + k] = double(pred[id * 4 + 1 + a]) / u_scale;
}

}  // namespace

extern "C" {

lbm_status lbm_warmstart_features(const double* coarse_rho, const double* coarse_u, const int32_t coarse_blocks[3],
                                  int32_t B, int32_t periodic_mask, int32_t level, int32_t halo, const int32_t* blocks,
                                  int32_t nblocks, const double* spheres, int32_t nspheres, double rho_scale,
                                  double u_scale, void* x, float* skip, void* stream) {
    if (!coarse_rho || !coarse_u || !coarse_blocks || !blocks || !x || (nspheres > 0 && !spheres))
        return nfail(LBM_EINVAL, "NULL argument");
    if (B < 1 || halo < 0 || level < 0 || level > 20 || nblocks < 0 || nspheres < 0)
        return nfail(LBM_EINVAL, "invalid sizes");
    if (nblocks == 0) return LBM_OK;
    Coarse c{coarse_rho, coarse_u, 0, {coarse_blocks[0], coarse_blocks[1], coarse_blocks[2]}, B, periodic_mask};
    c.n0 = (long long)c.nb[0] * c.nb[1] * c.nb[2] * B * B * B;
    const int D = B + 2 * halo, nt = (D + kFeatTile - 1) / kFeatTile, T = (D + nt - 1) / nt;
    const long long ctas = (long long)D * nblocks * nt * nt;
    if (ctas >= (1LL << 31)) return nfail(LBM_EINVAL, "too many volumes");
    // the coarse cells under T voxels of an axis: at most (T - 1) / 2^level + 1 of them and the upper neighbour, which
    // at kFeatTile and level 0 take 108 KB
    const int nc = (T - 1) / (1 << level) + 3;
    const size_t smem = size_t(4) * (nc * nc + T * nc) * (sizeof(long long) + sizeof(uint32_t));
    NCU(cudaFuncSetAttribute(features_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 112 * 1024));
    features_kernel<<<unsigned(ctas), kFeatThreads, smem, static_cast<cudaStream_t>(stream)>>>(
        c, level, B, halo, blocks, spheres, nspheres, rho_scale, u_scale, T, nt, static_cast<__nv_bfloat16*>(x), skip);
    NCU(cudaGetLastError());
    return LBM_OK;
}

lbm_status lbm_warmstart_targets(const double* rho, const double* u, int32_t B, int32_t halo, int32_t nblocks,
                                 double rho_scale, double u_scale, float* target, float* weight, void* stream) {
    if (!rho || !u || !target || !weight) return nfail(LBM_EINVAL, "NULL argument");
    if (B < 1 || halo < 0 || nblocks < 0) return nfail(LBM_EINVAL, "invalid sizes");
    if (nblocks == 0) return LBM_OK;
    const long long D = B + 2 * halo, total = D * D * D * nblocks, n = (long long)nblocks * B * B * B;
    targets_kernel<<<unsigned((total + 255) / 256), 256, 0, static_cast<cudaStream_t>(stream)>>>(
        rho, u, n, B, halo, nblocks, rho_scale, u_scale, target, weight);
    NCU(cudaGetLastError());
    return LBM_OK;
}

lbm_status lbm_warmstart_fields(const float* pred, int32_t B, int32_t halo, int32_t nblocks, double rho_scale,
                                double u_scale, double* rho, double* u, void* stream) {
    if (!pred || !rho || !u) return nfail(LBM_EINVAL, "NULL argument");
    if (B < 1 || halo < 0 || nblocks < 0) return nfail(LBM_EINVAL, "invalid sizes");
    if (nblocks == 0) return LBM_OK;
    const long long n = (long long)nblocks * B * B * B;
    fields_kernel<<<unsigned((n + 255) / 256), 256, 0, static_cast<cudaStream_t>(stream)>>>(pred, B, halo, nblocks,
                                                                                          rho_scale, u_scale, rho, u);
    NCU(cudaGetLastError());
    return LBM_OK;
}

}  // extern "C"
