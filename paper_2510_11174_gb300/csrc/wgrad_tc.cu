// Weight gradients on the 5th-generation tensor cores, for the 3x3x3
// convolutions of the regime classifier and the field surrogate and for the
// dense layers of SwitchNet (paper, Methodology and Results: the networks are
// trained on data the simulation generates).
//
//   dW[co][ci][t] = sum over cells of dZ[cell][co] X[cell + s(t)][ci]
//
// is a contraction over the cells, and both operands lie channels-last, i.e.
// with the contracted index outermost: the tensor core takes them as they are
// (MN-major operands), so TMA boxes of the layer's own tensors are all the
// staging there is.
//
// Convolution (k_wgrad_conv).  An operand's shared-memory descriptor repeats its
// 16- or 32-channel block along M or N at a stride of its own, and that stride
// may be a shift in space.  M = 128 rows are one operand's channels at 128 / CA
// consecutive y-shifts (stride: a row of cells; three are the taps, the others
// compute sums nobody reads), N = 3 CB columns the other operand's channels at
// three z-shifts (stride: a plane), and the x-tap is the start cell of the
// other operand's run: three MMAs per 16 cells give all 27 taps.  With A(p) the
// first operand and B(p) the second at position p,
//   D_dx[(sy, a)][(sz, b)] = sum_p A[x, y + sy - 1, z][a] B[x + dx - 1, y, z + sz - 1][b],
// where out-of-volume cells are 0 (TMA fill).  A is dZ (taps (sz, 2 - sy, dx)) or
// X (taps (2 - sz, sy, 2 - dx)), whichever has 32 channels.
// A CTA walks columns of 16 (x) x 8 (y) cells along z with rings of planes of
// both operands and 3 x 3 CB accumulator columns in TMEM; the partial sums of a channel block's CTAs are
// added in a fixed order (deterministic).
// Dense layer (k_wgrad_dense): the same with plain 64-cell tiles, M = 128 output
// columns, N = 16, 128 or 256 input columns.
//   warp 0      TMA producer;
//   warp 1      MMA issuer;
//   warps 2..17 epilogue: tcgen05.ld of the accumulators into FP32 register sums
//               (see wg_epilogue), FP32 partials to global memory at the end of
//               the CTA's range.
// What bounds the convolution: fetching the operands from shared memory, 56
// cycles per 128 x 96 x 16 MMA (48 of math), 10.5 cycles a cell.  The former
// kernel wanted [16 positions][channel] transposes of both operands over the
// padded volume, three of them for the x-shifts of dZ, and read nine shifted
// boxes of them for every chunk: 400 us a layer plus 30 us a transpose for
// 1,048,576 cells, whatever the channels.
// Waits are bounded (ST_TIMEOUT on giving up, as in the convolutions).
#include <cuda.h>
#include <cuda_bf16.h>

#include <mutex>

#include "conv_tc.cuh"
#include "hyb_internal.cuh"

namespace hyb {

static constexpr long long WG_MBAR_LIMIT = 1LL << 26;
static constexpr int WX = 16, WY = 8;  // cells of a block: one K = 16 run in x, rows
static constexpr int WROWS = 128;      // accumulator rows

// MN-major operand (channels contiguous, one swizzle-wide row per cell): `mn` bytes between channel blocks along M or N, `k` bytes between groups of 8 cells
__device__ __forceinline__ uint64_t smem_desc_mn(uint32_t addr, uint32_t mn, uint32_t k, uint32_t layout) {
    uint64_t d = 0;
    d |= (uint64_t)((addr >> 4) & 0x3FFFu);
    d |= (uint64_t)((mn >> 4) & 0x3FFFu) << 16;
    d |= (uint64_t)((k >> 4) & 0x3FFFu) << 32;
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)layout << 61;
    return d;
}
static constexpr uint32_t SW128 = 2, SW64 = 4, SW32 = 6;  // layout types
// both operands MN-major (bits 15 and 16)
__host__ __device__ constexpr uint32_t idesc_mn(int N) { return idesc_bf16(128, N) | (1u << 15) | (1u << 16); }

struct WgConvArgs {
    float *part;               // [block][cta][9 CB columns][128 rows]
    int B, D, H, W;
    int nab;                   // channel blocks of A (block = ab + nab * bb)
    int lz;                    // planes per column
    int flush;                 // planes (8 K-steps each) the accumulators hold before they are taken over
    int *status;
};

template <int CA, int CB>
struct WgConv {
    static constexpr int RA = WROWS / CA;                  // y-shifts stacked in M
    static constexpr int AROW = WX * CA * 2;               // bytes of a row of A cells
    static constexpr int ABOX = AROW * (WY + 2);           // rows y - 1 .. y + 8
    static constexpr int BROW = (WX + 2) * CB * 2;
    static constexpr int BBOX = BROW * WY;
    // the MMAs of the last rows read RA - 3 rows past A's box (sums nobody reads)
    static constexpr int NA = 6, NB = CB == 32 ? 14 : 16;  // planes in the rings
    static constexpr int BOFF = ((NA * ABOX + (RA - 3) * AROW) + 1023) / 1024 * 1024;
    static constexpr int SMEM = BOFF + NB * BBOX + 1024;
    static constexpr int COLS = 9 * CB;                    // accumulator columns: [dx][sz][CB]
    static_assert(SMEM <= 226 * 1024 && BBOX % 512 == 0 && ABOX % 1024 == 0, "rings");
};

__device__ __forceinline__ void wg_unit(long long u, const WgConvArgs &a, int nx, int ny, int nzc, int &x, int &y,
                                        int &z0, int &z1, int &b) {
    uint32_t t = (uint32_t)u;
    x = (int)(t % (uint32_t)nx) * WX;
    t /= (uint32_t)nx;
    y = (int)(t % (uint32_t)ny) * WY;
    t /= (uint32_t)ny;
    z0 = (int)(t % (uint32_t)nzc) * a.lz;
    b = (int)(t / (uint32_t)nzc);
    z1 = min(z0 + a.lz, a.D);
}

// The tensor core's FP32 accumulation truncates, so a sum's error grows with the
// number of products added in place (a 64 -> 128 layer over 131,072 cells: 9e-6
// off after 431, 3e-7 after 64).  Where channel blocks share the SMs a CTA has
// more than the 1 / (number of SMs) of the cells it would have alone: the 16
// epilogue warps take the accumulators over after every such share and add
// them, rounded to nearest, to registers; warp w of a lane quarter keeps COLS / 4
// columns.
static constexpr int WG_EPI = 16;
static constexpr int WG_THREADS = 64 + 32 * WG_EPI;

// 32 lanes x 32 bits x G consecutive columns, without a wait
template <int G>
__device__ __forceinline__ void tmem_ld_cols(uint32_t taddr, float (&v)[G]) {
    uint32_t r[G];
    if constexpr (G == 8)
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                     : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                     : "r"(taddr));
    else
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
                     : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                     : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < G; ++i) v[i] = __uint_as_float(r[i]);
}

// `flushes` rounds: wait for the accumulators (columns from taddr; BUF buffers
// of `pitch` columns in turn), add them, hand them back; then the sums as
// partials [column][128 rows].  false: a wait gave up.
template <int COLS, int BUF>
__device__ __forceinline__ bool wg_epilogue(uint32_t taddr, int pitch, uint64_t *full, uint64_t *empty, long long flushes,
                                            int warp, int lane, const int *abort_flag, float *__restrict__ dst) {
    constexpr int CPW = COLS / 4, G = CPW % 8 == 0 ? 8 : 4;
    const int q = warp & 3, w = (warp - 2) >> 2;
    float acc[CPW];
#pragma unroll
    for (int k = 0; k < CPW; ++k) acc[k] = 0.0f;
    for (long long i = 0; i < flushes; ++i) {
        const int b = (int)(i % BUF);
        const bool ok = mbar_wait_abort(smem_u32(&full[b]), (uint32_t)(i / BUF) & 1u, WG_MBAR_LIMIT, abort_flag);
        if (!__all_sync(0xffffffffu, ok)) return false;
        fence_after_sync();
        const uint32_t t = taddr + ((uint32_t)(q * 32) << 16) + (uint32_t)(b * pitch + w * CPW);
#pragma unroll
        for (int c = 0; c < CPW; c += G) {
            float v[G];
            tmem_ld_cols<G>(t + (uint32_t)c, v);
#pragma unroll
            for (int k = 0; k < G; ++k) acc[c + k] += v[k];
        }
        fence_before_sync();
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&empty[b]));
    }
    const int row = q * 32 + lane;
#pragma unroll
    for (int k = 0; k < CPW; ++k) dst[(w * CPW + k) * WROWS + row] = acc[k];
    return true;
}

template <int CA, int CB>
__global__ void __launch_bounds__(WG_THREADS, 1) k_wgrad_conv(const __grid_constant__ CUtensorMap ta,
                                                       const __grid_constant__ CUtensorMap tb,
                                                       const __grid_constant__ WgConvArgs a) {
    using Cfg = WgConv<CA, CB>;
    constexpr int NA = Cfg::NA, NB = Cfg::NB;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    __shared__ __align__(8) uint64_t fa_b[NA], ea_b[NA], fb_b[NB], eb_b[NB], tfull_b, tempty_b, done_b;
    __shared__ uint32_t taddr_s;
    __shared__ int abort_s;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (warp == 1) {
        tmem_alloc(smem_u32(&taddr_s), 512);
        tmem_relinquish();
    }
    if (tid == 0) {
        for (int s = 0; s < NA; ++s) {
            mbar_init(smem_u32(&fa_b[s]), 1);
            mbar_init(smem_u32(&ea_b[s]), 1);
        }
        for (int s = 0; s < NB; ++s) {
            mbar_init(smem_u32(&fb_b[s]), 1);
            mbar_init(smem_u32(&eb_b[s]), 1);
        }
        mbar_init(smem_u32(&tfull_b), 1);
        mbar_init(smem_u32(&tempty_b), WG_EPI);
        mbar_init(smem_u32(&done_b), 1);
        abort_s = 0;
        fence_mbar_init();
        prefetch_tmap(&ta);
        prefetch_tmap(&tb);
    }
    fence_before_sync();
    __syncthreads();
    fence_after_sync();
    const uint32_t taddr = taddr_s, sa = smem_u32(smem), sb = sa + Cfg::BOFF;
    const int nx = (a.W + WX - 1) / WX, ny = (a.H + WY - 1) / WY, nzc = (a.D + a.lz - 1) / a.lz;
    const long long nunits = (long long)a.B * nzc * ny * nx;
    const int ca = (int)(blockIdx.y % (unsigned)a.nab) * CA, cb = (int)(blockIdx.y / (unsigned)a.nab) * CB;
    auto fail = [&]() {
        atomicOr(a.status, ST_TIMEOUT);
        *(volatile int *)&abort_s = 1;
    };

    if (warp == 0) {
        if (lane == 0) {
            int s = 0, t = 0;          // ring positions of A and B
            uint32_t ps = 0, pt = 0;
            long long na = 0, nb = 0;  // copies issued
            bool stop = false;
            for (long long u = blockIdx.x; u < nunits && !stop; u += gridDim.x) {
                int x, y, z0, z1, b;
                wg_unit(u, a, nx, ny, nzc, x, y, z0, z1, b);
                for (int z = z0 - 1; z <= z1 && !stop; ++z) {
                    if (!mbar_wait(smem_u32(&eb_b[t]), pt ^ 1, WG_MBAR_LIMIT) || *(volatile int *)&abort_s) {
                        fail();
                        stop = true;
                        break;
                    }
                    mbar_arrive_expect_tx(smem_u32(&fb_b[t]), Cfg::BBOX);
                    tma_load_5d(sb + (uint32_t)(t * Cfg::BBOX), &tb, cb, x - 1, y, z, b, smem_u32(&fb_b[t]));
                    ++nb;
                    if (++t == NB) {
                        t = 0;
                        pt ^= 1;
                    }
                    if (z < z0 || z >= z1) continue;
                    if (!mbar_wait(smem_u32(&ea_b[s]), ps ^ 1, WG_MBAR_LIMIT) || *(volatile int *)&abort_s) {
                        fail();
                        stop = true;
                        break;
                    }
                    mbar_arrive_expect_tx(smem_u32(&fa_b[s]), Cfg::ABOX);
                    tma_load_5d(sa + (uint32_t)(s * Cfg::ABOX), &ta, ca, x, y - 1, z, b, smem_u32(&fa_b[s]));
                    ++na;
                    if (++s == NA) {
                        s = 0;
                        ps ^= 1;
                    }
                }
            }
            if (*(volatile int *)&abort_s) {
                // copies in flight complete before exit
                for (int k = 0; k < NA && na > 0; ++k, --na) {
                    if (--s < 0) {
                        s = NA - 1;
                        ps ^= 1;
                    }
                    mbar_wait(smem_u32(&fa_b[s]), ps, WG_MBAR_LIMIT);
                }
                for (int k = 0; k < NB && nb > 0; ++k, --nb) {
                    if (--t < 0) {
                        t = NB - 1;
                        pt ^= 1;
                    }
                    mbar_wait(smem_u32(&fb_b[t]), pt, WG_MBAR_LIMIT);
                }
            }
        }
    } else if (warp == 1) {
        // the whole warp runs the loop; an elected lane issues
        constexpr uint32_t LA = CA == 32 ? SW64 : SW32, LB = CB == 32 ? SW64 : SW32;
        // M: channel blocks a row of A cells apart; N: a plane of B apart; K groups: 8 cells
        const uint64_t a0 = smem_desc_mn(0, Cfg::AROW, 8 * CA * 2, LA), b0 = smem_desc_mn(0, Cfg::BBOX, 8 * CB * 2, LB);
        const uint32_t ahi = (uint32_t)(a0 >> 32), bhi = (uint32_t)(b0 >> 32);
        const uint32_t alo = (uint32_t)a0 + (sa >> 4), blo = (uint32_t)b0 + (sb >> 4);  // below 2^14: no carry
        int s = 0, t = 0;        // A plane, next B plane to wait for
        uint32_t ps = 0, pt = 0;
        uint32_t acc = 0;        // 0: the first products overwrite the accumulators
        int planes = 0;          // planes in the accumulators
        uint32_t pf = 0;         // parity of the last hand-over
        LookAhead<NB, NA> look;
        bool stop = false;
        for (long long u = blockIdx.x; u < nunits && !stop; u += gridDim.x) {
            int x, y, z0, z1, b;
            wg_unit(u, a, nx, ny, nzc, x, y, z0, z1, b);
            int first = t;       // ring slot of B plane z - 1
            for (int z = z0 - 1; z <= z1; ++z) {
                // A plane z - 1 with B planes z - 2, z - 1, z
                if (!look.wait(fb_b, t, pt, fa_b, s, ps, z > z0, lane, WG_MBAR_LIMIT, &abort_s)) {
                    if (lane == 0) fail();
                    stop = true;
                    break;
                }
                if (++t == NB) {
                    t = 0;
                    pt ^= 1;
                }
                if (z <= z0) continue;
                if (planes == a.flush) {
                    // hand the accumulators over and begin again
                    umma_commit_warp(smem_u32(&tfull_b));
                    if (!__all_sync(0xffffffffu, mbar_wait_abort(smem_u32(&tempty_b), pf, WG_MBAR_LIMIT, &abort_s))) {
                        if (lane == 0) fail();
                        stop = true;
                        break;
                    }
                    pf ^= 1;
                    planes = 0;
                    acc = 0;
                }
                ++planes;
                fence_after_sync();
                const int n1 = min(3, NB - first);   // planes before the ring wraps
                const uint32_t ap = alo + (uint32_t)(s * (Cfg::ABOX >> 4));
                const uint32_t bp = blo + (uint32_t)(first * (Cfg::BBOX >> 4));
                if (n1 == 3) {
#pragma unroll
                    for (int j = 0; j < WY; ++j)
#pragma unroll
                        for (int dx = 0; dx < 3; ++dx)
                            umma_bf16_warp(taddr + (uint32_t)(dx * 3 * CB), ap + (uint32_t)((j * Cfg::AROW) >> 4), ahi,
                                           bp + (uint32_t)((j * Cfg::BROW + dx * CB * 2) >> 4), bhi, idesc_mn(3 * CB),
                                           acc | (uint32_t)j);
                } else {
#pragma unroll 1
                    for (int j = 0; j < WY; ++j)
#pragma unroll
                        for (int dx = 0; dx < 3; ++dx) {
                            const uint32_t ad = ap + (uint32_t)((j * Cfg::AROW) >> 4);
                            const uint32_t off = (uint32_t)((j * Cfg::BROW + dx * CB * 2) >> 4);
                            const uint32_t d = taddr + (uint32_t)(dx * 3 * CB);
                            umma_bf16_warp(d, ad, ahi, bp + off, bhi, idesc_mn(8) - (1u << 17) + ((uint32_t)(n1 * CB) << 14),
                                           acc | (uint32_t)j);
                            umma_bf16_warp(d + (uint32_t)(n1 * CB), ad, ahi, blo + off, bhi,
                                           idesc_mn(8) - (1u << 17) + ((uint32_t)((3 - n1) * CB) << 14), acc | (uint32_t)j);
                        }
                }
                acc = 1;
                umma_commit_warp(smem_u32(&ea_b[s]));
                umma_commit_warp(smem_u32(&eb_b[first]));
                if (++first == NB) first = 0;
                if (z == z1) {
                    umma_commit_warp(smem_u32(&eb_b[first]));
                    if (++first == NB) first = 0;
                    umma_commit_warp(smem_u32(&eb_b[first]));
                }
                if (++s == NA) {
                    s = 0;
                    ps ^= 1;
                }
            }
        }
        if (planes) umma_commit_warp(smem_u32(&tfull_b));
        umma_commit_warp(smem_u32(&done_b));
        mbar_wait(smem_u32(&done_b), 0, WG_MBAR_LIMIT);
    } else {
        long long total = 0;     // planes of this CTA's columns
        for (long long u = blockIdx.x; u < nunits; u += gridDim.x) {
            int x, y, z0, z1, b;
            wg_unit(u, a, nx, ny, nzc, x, y, z0, z1, b);
            total += z1 - z0;
        }
        if (!wg_epilogue<Cfg::COLS, 1>(taddr, 0, &tfull_b, &tempty_b, (total + a.flush - 1) / a.flush, warp, lane, &abort_s,
                                       a.part + ((long long)blockIdx.y * gridDim.x + blockIdx.x) * Cfg::COLS * WROWS) &&
            lane == 0)
            fail();
    }
    fence_before_sync();
    __syncthreads();
    fence_after_sync();
    if (warp == 1) tmem_dealloc(taddr, 512);
}

// dense layer: K tiles of 64 cells, boxes of 64 channels (128-byte rows), or of
// 16 channels when the layer has 16 inputs
struct WgDenseArgs {
    float *part;      // [co slice][cta][N columns][128 rows]
    long long tiles;  // of 64 cells
    int flush;        // tiles the accumulators hold before they are taken over
    int *status;
};

template <int N>
struct WgDense {
    static constexpr int BW = N < 64 ? N : 64;      // channels of a B box
    static constexpr int ABYTES = 2 * 64 * 128;     // 128 output channels
    static constexpr int BBYTES = N * 128;
    static constexpr int STAGE = ABYTES + BBYTES;
    static constexpr int STAGES = N == 256 ? 4 : 6;
    static constexpr int SMEM = STAGES * STAGE + 1024;
};

__device__ __forceinline__ void tma_load_2d(uint32_t dst, const void *tmap, int c0, int c1, uint32_t mbar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
        ::"r"(dst), "l"(tmap), "r"(c0), "r"(c1), "r"(mbar)
        : "memory");
}

template <int N>
__global__ void __launch_bounds__(WG_THREADS, 1) k_wgrad_dense(const __grid_constant__ CUtensorMap tz,
                                                        const __grid_constant__ CUtensorMap tx,
                                                        const __grid_constant__ WgDenseArgs a) {
    using Cfg = WgDense<N>;
    constexpr int STAGES = Cfg::STAGES;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *ring = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    __shared__ __align__(8) uint64_t full_b[STAGES], empty_b[STAGES], tfull_b[2], tempty_b[2], done_b;
    __shared__ uint32_t taddr_s;
    __shared__ int abort_s;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (warp == 1) {
        tmem_alloc(smem_u32(&taddr_s), 512);
        tmem_relinquish();
    }
    if (tid == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(smem_u32(&full_b[s]), 1);
            mbar_init(smem_u32(&empty_b[s]), 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(smem_u32(&tfull_b[b]), 1);
            mbar_init(smem_u32(&tempty_b[b]), WG_EPI);
        }
        mbar_init(smem_u32(&done_b), 1);
        abort_s = 0;
        fence_mbar_init();
        prefetch_tmap(&tz);
        prefetch_tmap(&tx);
    }
    fence_before_sync();
    __syncthreads();
    fence_after_sync();
    const uint32_t taddr = taddr_s, ring_s = smem_u32(ring);
    const int co0 = (int)blockIdx.y * 128;
    auto fail = [&]() {
        atomicOr(a.status, ST_TIMEOUT);
        *(volatile int *)&abort_s = 1;
    };
    if (warp == 0) {
        if (lane == 0) {
            int s = 0;
            uint32_t ph = 0;
            long long issued = 0;
            for (long long k = blockIdx.x; k < a.tiles; k += gridDim.x) {
                if (!mbar_wait(smem_u32(&empty_b[s]), ph ^ 1, WG_MBAR_LIMIT) || *(volatile int *)&abort_s) {
                    fail();
                    break;
                }
                const uint32_t fb = smem_u32(&full_b[s]), st = ring_s + (uint32_t)(s * Cfg::STAGE);
                mbar_arrive_expect_tx(fb, Cfg::STAGE);
                for (int c = 0; c < 2; ++c) tma_load_2d(st + (uint32_t)(c * 8192), &tz, co0 + 64 * c, (int)(k * 64), fb);
                for (int c = 0; c < N / Cfg::BW; ++c)
                    tma_load_2d(st + (uint32_t)(Cfg::ABYTES + c * Cfg::BW * 128), &tx, c * Cfg::BW, (int)(k * 64), fb);
                ++issued;
                if (++s == STAGES) {
                    s = 0;
                    ph ^= 1;
                }
            }
            if (*(volatile int *)&abort_s) {
                for (int k = 0; k < STAGES && issued > 0; ++k, --issued) {
                    if (--s < 0) {
                        s = STAGES - 1;
                        ph ^= 1;
                    }
                    mbar_wait(smem_u32(&full_b[s]), ph, WG_MBAR_LIMIT);
                }
            }
        }
    } else if (warp == 1) {
        if (lane == 0) {
            // two accumulator buffers in turn, a.flush tiles each
            int s = 0, tiles = 0, buf = 0;
            uint32_t ph = 0, acc = 0, pb = 1;
            for (long long k = blockIdx.x; k < a.tiles; k += gridDim.x) {
                if (tiles == a.flush) {
                    umma_commit(smem_u32(&tfull_b[buf]));
                    buf ^= 1;
                    if (buf == 0) pb ^= 1;
                    tiles = 0;
                    acc = 0;
                }
                if ((tiles == 0 && !mbar_wait_abort(smem_u32(&tempty_b[buf]), pb, WG_MBAR_LIMIT, &abort_s)) ||
                    !mbar_wait_abort(smem_u32(&full_b[s]), ph, WG_MBAR_LIMIT, &abort_s)) {
                    fail();
                    tiles = 0;
                    break;
                }
                ++tiles;
                fence_after_sync();
                const uint32_t st = ring_s + (uint32_t)(s * Cfg::STAGE);
                const uint64_t ad = smem_desc_mn(st, 8192, 1024, SW128);
                const uint64_t bd = N < 64 ? smem_desc_mn(st + Cfg::ABYTES, 2048, 8 * N * 2, SW32)
                                           : smem_desc_mn(st + Cfg::ABYTES, 8192, 1024, SW128);
#pragma unroll
                for (int kk = 0; kk < 4; ++kk) {
                    umma_bf16(taddr + (uint32_t)(buf * 256), ad + (uint64_t)((kk * 16 * 128) >> 4),
                              bd + (uint64_t)((kk * 16 * Cfg::BW * 2) >> 4), idesc_mn(N), acc);
                    acc = 1;
                }
                umma_commit(smem_u32(&empty_b[s]));
                if (++s == STAGES) {
                    s = 0;
                    ph ^= 1;
                }
            }
            if (tiles) umma_commit(smem_u32(&tfull_b[buf]));
            umma_commit(smem_u32(&done_b));
            mbar_wait(smem_u32(&done_b), 0, WG_MBAR_LIMIT);
        }
    } else {
        const long long total = (long long)blockIdx.x < a.tiles ? (a.tiles - blockIdx.x + gridDim.x - 1) / gridDim.x : 0;
        if (!wg_epilogue<N, 2>(taddr, 256, tfull_b, tempty_b, (total + a.flush - 1) / a.flush, warp, lane, &abort_s,
                               a.part + ((long long)blockIdx.y * gridDim.x + blockIdx.x) * N * WROWS) &&
            lane == 0)
            fail();
    }
    fence_before_sync();
    __syncthreads();
    fence_after_sync();
    if (warp == 1) tmem_dealloc(taddr, 512);
}

// The CTAs' partials of one accumulator column added in a fixed order: 128 rows
// x 4 quarters of the CTAs per block, then the quarters; coalesced along the
// rows.  Column (dx, sz, b) and row (sy, a) of a convolution's channel block go
// to the tap they stand for, column ci and row co of a dense slice to gw[co][ci].
struct WgReduceArgs {
    const float *part;
    int ncta, cols;
    int taps, ca, cb, nab, a_is_dz;
    int ci_n, co_n;
    float *gw;
};
__global__ void __launch_bounds__(512) k_wgrad_reduce(const WgReduceArgs r) {
    __shared__ float sh[4][WROWS];
    const int row = threadIdx.x & 127, h = threadIdx.x >> 7;
    const int col = blockIdx.x, blk = blockIdx.y;
    const float *src = r.part + ((long long)blk * r.ncta * r.cols + col) * WROWS + row;
    const int per = (r.ncta + 3) / 4, k1 = min(r.ncta, (h + 1) * per);
    float s = 0.0f;
#pragma unroll 8
    for (int k = h * per; k < k1; ++k) s += src[(long long)k * r.cols * WROWS];
    sh[h][row] = s;
    __syncthreads();
    if (h != 0) return;
    s = ((sh[0][row] + sh[1][row]) + sh[2][row]) + sh[3][row];
    int ci, co, t = 0;
    if (r.taps == 27) {
        const int sy = row / r.ca, ac = (blk % r.nab) * r.ca + row % r.ca;
        const int dx = col / (3 * r.cb), sz = (col / r.cb) % 3, bc = (blk / r.nab) * r.cb + col % r.cb;
        if (sy > 2) return;
        co = r.a_is_dz ? ac : bc;
        ci = r.a_is_dz ? bc : ac;
        t = r.a_is_dz ? (sz * 3 + 2 - sy) * 3 + dx : ((2 - sz) * 3 + sy) * 3 + 2 - dx;
    } else {
        co = blk * 128 + row;
        ci = col;
    }
    if (co < r.co_n && ci < r.ci_n) r.gw[((long long)co * r.ci_n + ci) * r.taps + t] = s;
}

// FP32 [cells] -> BF16 channel 0 of 16 (the last layer's dlogit as an operand)
__global__ void k_f32_to_16(const float *__restrict__ src, long long cells, __nv_bfloat16 *__restrict__ dst) {
    const long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (c >= cells) return;
    uint4 *o = reinterpret_cast<uint4 *>(dst + c * 16);
    o[0] = make_uint4((uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(src[c])), 0u, 0u, 0u);
    o[1] = make_uint4(0u, 0u, 0u, 0u);
}

// bias gradient partials, bpart[blk][c] = sum over the block's cells of dZ[cell][c]:
// 16-byte loads, a thread keeps the sums of one group of eight channels (C = 16 .. 256)
__global__ void __launch_bounds__(256) k_bias_part(const __nv_bfloat16 *__restrict__ dz, int C, long long cells,
                                                   float *__restrict__ bpart) {
    __shared__ float sh[256][9];
    const int ng = C / 8, g = threadIdx.x % ng, r0 = threadIdx.x / ng, R = 256 / ng;
    float s[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) s[j] = 0.0f;
#pragma unroll 4
    for (long long i = blockIdx.x * (long long)R + r0; i < cells; i += (long long)gridDim.x * R) {
        const uint4 u = reinterpret_cast<const uint4 *>(dz + i * C)[g];
        const __nv_bfloat16 *h = reinterpret_cast<const __nv_bfloat16 *>(&u);
#pragma unroll
        for (int j = 0; j < 8; ++j) s[j] += __bfloat162float(h[j]);
    }
#pragma unroll
    for (int j = 0; j < 8; ++j) sh[threadIdx.x][j] = s[j];
    __syncthreads();
    if (threadIdx.x < C) {
        float b = 0.0f;
        for (int k = 0; k < R; ++k) b += sh[k * ng + threadIdx.x / 8][threadIdx.x % 8];
        bpart[(long long)blockIdx.x * C + threadIdx.x] = b;
    }
}

// the same for an FP32 gradient of one channel
__global__ void __launch_bounds__(256) k_bias_part_f32(const float *__restrict__ dz, long long cells,
                                                       float *__restrict__ bpart) {
    __shared__ float sh[256];
    float s = 0.0f;
    for (long long i = blockIdx.x * 256LL + threadIdx.x; i < cells; i += (long long)gridDim.x * 256) s += dz[i];
    sh[threadIdx.x] = s;
    __syncthreads();
    for (int w = 128; w > 0; w >>= 1) {
        if (threadIdx.x < w) sh[threadIdx.x] += sh[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) bpart[blockIdx.x] = sh[0];
}

// out[c] = sum over k of part[k][c] (nk rows of pitch np): one block per column,
// thread i adds rows i, i + 256, ... in order, then a fixed-shape tree
__global__ void __launch_bounds__(256) k_sum_cols(const float *__restrict__ part, int nk, int np,
                                                  float *__restrict__ out) {
    __shared__ float sh[256];
    const int c = blockIdx.x;
    float s = 0.0f;
    for (int k = threadIdx.x; k < nk; k += 256) s += part[(long long)k * np + c];
    sh[threadIdx.x] = s;
    __syncthreads();
    for (int w = 128; w > 0; w >>= 1) {
        if (threadIdx.x < w) sh[threadIdx.x] += sh[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) out[c] = sh[0];
}

typedef CUresult (*EncodeTiledFn3)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                   const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                   CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static EncodeTiledFn3 encode_fn3() {
    static EncodeTiledFn3 fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = (EncodeTiledFn3)p;
    });
    return fn;
}

// channels-last BF16 [B][D][H][W][C], box (c, bx, by, 1, 1)
static hyb_status vol_map(CUtensorMap *tm, const __nv_bfloat16 *base, int C, const WgradJob &j, int c, int bx, int by) {
    EncodeTiledFn3 enc = encode_fn3();
    if (!enc) return set_error(HYB_ECUDA, "cuTensorMapEncodeTiled is not available");
    const cuuint64_t es = 2;
    const cuuint64_t dims[5] = {(cuuint64_t)C, (cuuint64_t)j.W, (cuuint64_t)j.H, (cuuint64_t)j.D, (cuuint64_t)j.B};
    const cuuint64_t st[4] = {es * C, es * C * j.W, es * C * j.W * j.H, es * C * j.W * j.H * j.D};
    const cuuint32_t box[5] = {(cuuint32_t)c, (cuuint32_t)bx, (cuuint32_t)by, 1, 1};
    const cuuint32_t estr[5] = {1, 1, 1, 1, 1};
    const CUresult r = enc(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, (void *)base, dims, st, box, estr,
                           CU_TENSOR_MAP_INTERLEAVE_NONE,
                           c == 32 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_32B,
                           CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return set_error(HYB_ECUDA, "cuTensorMapEncodeTiled failed (" + std::to_string((int)r) + ")");
    return HYB_OK;
}

// rows [cells][C], box (c, 64 cells)
static hyb_status row_map(CUtensorMap *tm, const __nv_bfloat16 *base, int C, long long cells, int c) {
    EncodeTiledFn3 enc = encode_fn3();
    if (!enc) return set_error(HYB_ECUDA, "cuTensorMapEncodeTiled is not available");
    const cuuint64_t dims[2] = {(cuuint64_t)C, (cuuint64_t)cells};
    const cuuint64_t st[1] = {(cuuint64_t)C * 2};
    const cuuint32_t box[2] = {(cuuint32_t)c, 64};
    const cuuint32_t estr[2] = {1, 1};
    const CUresult r = enc(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, (void *)base, dims, st, box, estr,
                           CU_TENSOR_MAP_INTERLEAVE_NONE,
                           c == 64 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_32B,
                           CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return set_error(HYB_ECUDA, "cuTensorMapEncodeTiled failed (" + std::to_string((int)r) + ")");
    return HYB_OK;
}

template <class K, class A>
static hyb_status wg_launch(K kern, int smem, const CUtensorMap &m0, const CUtensorMap &m1, const A &a, dim3 grid,
                            cudaStream_t st) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return set_error(HYB_ECUDA, std::string("wgrad smem attribute: ") + cudaGetErrorString(e));
    kern<<<grid, WG_THREADS, smem, st>>>(m0, m1, a);
    e = cudaGetLastError();
    if (e != cudaSuccess) return set_error(HYB_ECUDA, std::string("wgrad launch: ") + cudaGetErrorString(e));
    return HYB_OK;
}

static int n_sms() {
    static int nsm = 0;
    if (!nsm) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
        if (nsm <= 0) nsm = 1;
    }
    return nsm;
}

static hyb_status wg_reserve(void **p, long long &have, long long want, const char *what) {
    if (have >= want) return HYB_OK;
    if (*p) cudaFree(*p);
    *p = nullptr;
    have = 0;
    if (cudaMalloc(p, (size_t)want) != cudaSuccess) return set_error(HYB_ENOMEM, what);
    have = want;
    return HYB_OK;
}

hyb_status wgrad_tc(const WgradJob &j, WgradScratch &ws, cudaStream_t st) {
    const bool conv = j.taps == 27;
    if (!(j.taps == 27 || j.taps == 1)) return set_error(HYB_EINVAL, "wgrad: 27 or 1 taps");
    const long long cells = (long long)j.B * j.D * j.H * j.W;
    if (cells < 1 || j.co_n < 1 || j.ci_n < 1) return set_error(HYB_EINVAL, "wgrad: empty operand");
    if (cells >= (1LL << 30)) return set_error(HYB_EINVAL, "wgrad: more than 2^30 cells");
    const int xp = j.x_pitch, zp = j.dz_f32 ? 16 : j.dz_pitch;
    if (xp % 16 || zp % 16 || xp > 256 || zp > 256 || xp < j.ci_n || zp < j.co_n || (!conv && (zp % 128 || (xp != 16 && xp != 128 && xp != 256))))
        return set_error(HYB_EINVAL, "wgrad: channel pitch");
    const __nv_bfloat16 *dz = j.dz;
    if (j.dz_f32) {
        const hyb_status rs = wg_reserve(&ws.buf, ws.bytes, cells * 32, "wgrad operand buffer");
        if (rs != HYB_OK) return rs;
        k_f32_to_16<<<(unsigned)((cells + 255) / 256), 256, 0, st>>>(j.dz_f32, cells, (__nv_bfloat16 *)ws.buf);
        dz = (const __nv_bfloat16 *)ws.buf;
    }
    constexpr int BIAS_BLOCKS = 152 * 4;
    const int nsm = n_sms();
    WgReduceArgs r;
    memset(&r, 0, sizeof(r));
    r.taps = j.taps;
    r.ci_n = j.ci_n;
    r.co_n = j.co_n;
    r.gw = j.gw;
    CUtensorMap ta, tb;
    hyb_status s;
    int nblk;
    if (conv) {
        // A is the operand in 32-channel blocks (dZ when both are)
        const int xb = xp % 32 == 0 ? 32 : 16, zb = zp % 32 == 0 ? 32 : 16;
        r.a_is_dz = zb == 32;
        r.ca = r.a_is_dz ? zb : xb;
        r.cb = r.a_is_dz ? xb : zb;
        r.nab = (r.a_is_dz ? zp : xp) / r.ca;
        nblk = r.nab * (r.a_is_dz ? xp : zp) / r.cb;
        r.cols = 9 * r.cb;
    } else {
        nblk = zp / 128;
        r.cols = xp;
    }
    // the channel blocks share the SMs; split over the cells within a block
    r.ncta = std::max(1, nsm / nblk);
    WgConvArgs ca;
    memset(&ca, 0, sizeof(ca));
    long long work;
    if (conv) {
        const long long cols = (long long)j.B * ((j.H + WY - 1) / WY) * ((j.W + WX - 1) / WX);
        ca.lz = 32;  // planes per column: long ones share their halo, short ones balance the CTAs
        while (ca.lz > 4 && cols * ((j.D + ca.lz - 1) / ca.lz) < 6LL * r.ncta) ca.lz /= 2;
        work = cols * ((j.D + ca.lz - 1) / ca.lz);
    } else {
        work = (cells + 63) / 64;
    }
    r.ncta = (int)std::min<long long>(r.ncta, work);
    const long long pneed = std::max<long long>((long long)nblk * r.ncta * r.cols * WROWS, (long long)BIAS_BLOCKS * 256) * 4;
    if ((s = wg_reserve((void **)&ws.part, ws.pbytes, pneed, "wgrad partial buffers")) != HYB_OK) return s;
    r.part = ws.part;
    const dim3 grid((unsigned)r.ncta, (unsigned)nblk);
    if (conv) {
        ca.part = ws.part;
        ca.B = j.B;
        ca.D = j.D;
        ca.H = j.H;
        ca.W = j.W;
        ca.nab = r.nab;
        ca.flush = (int)((cells + 128LL * nsm - 1) / (128LL * nsm));
        ca.status = j.status;
        s = vol_map(&ta, r.a_is_dz ? dz : j.x, r.a_is_dz ? zp : xp, j, r.ca, WX, WY + 2);
        if (s == HYB_OK) s = vol_map(&tb, r.a_is_dz ? j.x : dz, r.a_is_dz ? xp : zp, j, r.cb, WX + 2, WY);
        if (s != HYB_OK) return s;
        if (r.ca == 32 && r.cb == 32) s = wg_launch(k_wgrad_conv<32, 32>, WgConv<32, 32>::SMEM, ta, tb, ca, grid, st);
        else if (r.ca == 32) s = wg_launch(k_wgrad_conv<32, 16>, WgConv<32, 16>::SMEM, ta, tb, ca, grid, st);
        else s = wg_launch(k_wgrad_conv<16, 16>, WgConv<16, 16>::SMEM, ta, tb, ca, grid, st);
    } else {
        WgDenseArgs d;
        d.part = ws.part;
        d.tiles = work;
        d.flush = (int)((work + nsm - 1) / nsm);
        d.status = j.status;
        s = row_map(&ta, dz, zp, cells, 64);
        if (s == HYB_OK) s = row_map(&tb, j.x, xp, cells, xp < 64 ? 16 : 64);
        if (s != HYB_OK) return s;
        if (xp == 16) s = wg_launch(k_wgrad_dense<16>, WgDense<16>::SMEM, ta, tb, d, grid, st);
        else if (xp == 128) s = wg_launch(k_wgrad_dense<128>, WgDense<128>::SMEM, ta, tb, d, grid, st);
        else s = wg_launch(k_wgrad_dense<256>, WgDense<256>::SMEM, ta, tb, d, grid, st);
    }
    if (s != HYB_OK) return s;
    k_wgrad_reduce<<<dim3((unsigned)r.cols, (unsigned)nblk), 512, 0, st>>>(r);
    if (j.gb) {
        // bias: per-block sums over the cells, then the blocks (the partials above
        // are consumed by the reduction first, in stream order)
        if (j.dz_f32) {
            k_bias_part_f32<<<BIAS_BLOCKS, 256, 0, st>>>(j.dz_f32, cells, ws.part);
            k_sum_cols<<<1, 256, 0, st>>>(ws.part, BIAS_BLOCKS, 1, j.gb);
        } else {
            k_bias_part<<<BIAS_BLOCKS, 256, 0, st>>>(dz, zp, cells, ws.part);
            k_sum_cols<<<j.co_n, 256, 0, st>>>(ws.part, BIAS_BLOCKS, zp, j.gb);
        }
    }
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return set_error(HYB_ECUDA, std::string("wgrad: ") + cudaGetErrorString(e));
    return HYB_OK;
}

}  // namespace hyb
