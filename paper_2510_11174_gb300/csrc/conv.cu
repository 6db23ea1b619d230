// 3x3x3 convolutions of the regime classifier (arXiv 2510.11174, Methodology
// and Results: a convolutional network on per-channel normalised fields, with
// Monte Carlo dropout for uncertainty; here the 3D CNN 6->32->32->16->1 with
// BF16 weights and FP32 accumulation).
//
// k_conv3_tc: implicit GEMM on the 5th-generation tensor cores, persistent
// and warp-specialised.  The three x-taps of the stencil go into the N
// dimension: for each of the 9 (dz, dy) taps one tcgen05.mma multiplies the
// 128 input cells of a 16 (x) x 8 (y) x 1 (z) block, shifted by (dz, dy), by
// the weights of all three x-taps side by side (3 C_out columns), so every A
// tile read from shared memory feeds three times the math.  The epilogue adds
// the three partial sums of neighbouring x cells (lanes m - 1, m, m + 1, one
// warp shuffle each way), so a block yields its 14 (x) x 8 (y) interior
// outputs (16 where the volume begins and ends in it); blocks step by 14 cells
// in x.
// A CTA walks a column of blocks along z: each plane of the halo (16 x 10
// cells, all channels) is fetched once by TMA into a ring of planes and used by
// the three output planes it touches.  With 16 outputs the three z-taps go into
// N too (ZN = 3): one MMA of 144 columns adds a plane's share to the
// accumulators of three output planes at once, which lie side by side in a ring
// of TMEM slots.  In every layout an output's sum is formed in the same order
// (per x-tap: dz, dy, 16-channel block; then left + middle + right).
//   warp 0      TMA producer: waits for a free plane, posts the expected bytes
//               on its "full" barrier and issues the copy (zero fill outside
//               the volume comes from the tensor map);
//   warp 1      MMA issuer (M = 128 cells x K = 16 per instruction) into a ring
//               of 5 (32 outputs) or 10 (16 outputs) TMEM accumulators; commits
//               free the plane and hand the accumulator to the epilogue;
//   warps 2..17 epilogue, one warp per TMEM lane quarter and 16-channel output
//               group, in 2 (32 outputs) or 4 (16 outputs) sets that take the
//               output planes in turn: tcgen05.ld of the accumulator rows, the
//               x-tap sum across lanes, bias, ReLU, Philox dropout with inverted
//               scaling, channels-last stores.  What does not depend on the
//               accumulator (dropout bits, bias) is computed before waiting for
//               it.
// What bounds it: an MMA takes max(N / 2, (4 KB + 32 N B) / 128 B) cycles (the
// math, or fetching its operands from shared memory: 56 at N = 96, 44 at N =
// 48, 72 at N = 144, measured in a chain of 1800), and the TMA's writes take
// about a cycle per cell and 64 B on the same shared-memory port.  Walking along
// z with 64-byte rows writes 160 cells per output plane; a halo of three planes
// per block in 32-byte rows wrote 960, as much as the MMAs' own 1008 cycles.
// The operand of tap (dz, dy) is a plane shifted by dy rows: its 128 cells are
// 128 consecutive rows of 64 (32 input channels) or 32 bytes (16), so every tap
// and 16-channel block is a plain K-major swizzled matrix descriptor -- no
// im2col; the TMA and the tensor core both apply the swizzle to the absolute
// shared address, so an operand may start at any row.
// Every wait is bounded: a wait that gives up sets ST_TIMEOUT, the roles stop
// issuing work, copies and MMAs in flight are waited for (bounded) and TMEM
// is released.
#include <cuda.h>
#include <cuda_bf16.h>

#include <mutex>

#include "conv_tc.cuh"
#include "hyb_internal.cuh"
#include "philox.cuh"

namespace hyb {

static constexpr int TX = 16, TY = 8;                 // A block (cells): M = 128 rows
static constexpr int TXO = TX - 2;                     // output cells per block row (the interior)
static constexpr int HY = TY + 2;                      // halo rows of a plane (x needs none: the x-taps live in N)
static constexpr int PCELLS = TX * HY;                 // cells of a plane (160)
static constexpr int EPC = 16;                         // output channels per epilogue warp
static constexpr long long MBAR_LIMIT = 1LL << 26;     // polls before a wait gives up

// dropout keep decision of channel ch at cell (b, lin): Philox counter
// (lin, b, (layer << 16) | (ch >> 3), pass), key (seed, 0xD0); 16-bit field
// ch & 7 of the output (word (ch & 7) >> 1, low half for even ch); kept when
// the field is >= thr = round(p 2^16)
__host__ __device__ inline bool dropout_keep(uint32_t seed, uint32_t pass, uint32_t layer, uint32_t b, uint32_t lin,
                                             int ch, uint32_t thr) {
    const u32x4 r = philox4x32_10(lin, b, (layer << 16) | ((uint32_t)ch >> 3), pass, seed, 0xD0u);
    const uint32_t f = (r.v[(ch & 7) >> 1] >> (16 * (ch & 1))) & 0xFFFFu;
    return f >= thr;
}

// Tile t covers the cells 14 t .. 14 t + 15 of a row and yields the outputs that
// have both x-neighbours in it, plus the volume's first and last cell, whose
// missing neighbour is 0: ceil((W - 2) / 14) tiles, one for 16 cells (a patch
// of the surrogate) instead of two.  A launch covers all tile columns, or those
// whose outputs meet the requested x-range.
__host__ __device__ inline void conv_tiles_x(int W, int x_lo, int x_hi, int &tx0, int &ntx) {
    const int all = W <= TX ? 1 : (W - 2 + TXO - 1) / TXO;
    tx0 = 0;
    ntx = all;
    if (x_hi > x_lo) {
        const int last = x_hi < 2 ? 0 : (x_hi - 2) / TXO;
        tx0 = x_lo < 1 ? 0 : (x_lo - 1) / TXO;
        if (tx0 > all - 1) tx0 = all - 1;
        ntx = (last < all - 1 ? last : all - 1) - tx0 + 1;
        if (ntx < 0) ntx = 0;
    }
}

// a column of blocks: x tile, y tile, output planes z0 .. z1 - 1, batch
struct ConvUnit {
    int tx, ty, z0, z1, b;
};
__device__ __forceinline__ ConvUnit conv_unit(long long u, int tx0, int nx, int ny, int nzc, int lz, int D) {
    ConvUnit c;
    uint32_t t = (uint32_t)u;  // unit counts fit in 32 bits (checked at launch)
    c.tx = (int)(t % (uint32_t)nx) + tx0;
    t /= (uint32_t)nx;
    c.ty = (int)(t % (uint32_t)ny);
    t /= (uint32_t)ny;
    c.z0 = (int)(t % (uint32_t)nzc) * lz;
    c.b = (int)(t / (uint32_t)nzc);
    c.z1 = min(c.z0 + lz, D);
    return c;
}

// index of a ring of S entries and the parity of its current round
template <int S>
struct Ring {
    int s = 0;
    uint32_t ph = 0;
    __device__ __forceinline__ void next() {
        if (++s == S) {
            s = 0;
            ph ^= 1;
        }
    }
};

template <int KC, int N>
struct ConvCfg {
    static constexpr int NP = 3 * N;                   // columns of one accumulator: the three x-taps side by side
    static constexpr int ZN = N == 16 ? 3 : 1;         // output planes one MMA adds to
    static constexpr int ROWB = KC * 16;               // bytes of a cell in shared memory
    static constexpr int WBYTES = 27 * KC * N * 16;    // weights, core layout [9 (dz, dy) or 3 (dy)][KC][ZN 3 N][8]
    static constexpr int RING = (WBYTES + 1023) / 1024 * 1024;  // plane ring offset (swizzle-aligned)
    static constexpr int PLANE = PCELLS * ROWB;        // a multiple of 1024
    static constexpr int SMEM_MAX = 227 * 1024 - 1024; // dynamic share (static barriers take the rest)
    static constexpr int FIT = (SMEM_MAX - 1024 - RING) / PLANE;
    static constexpr int PLANES = FIT > 16 ? 16 : FIT; // the copies in flight must cover the L2 latency of a plane
    static constexpr int SMEM = RING + PLANES * PLANE + 1024;  // + alignment slack
    static constexpr int NACC = 480 / NP;              // TMEM accumulators
    static constexpr int NG = N / EPC;                 // 16-channel output groups
    static constexpr int NSET = 4 / NG;                // epilogue sets (16 warps in all)
    static constexpr int NTHREADS = 64 + 512;          // producer, MMA issuer, epilogue
};

// EXT: the launch sums over input-channel chunks, adds a shortcut or runs
// several MC passes side by side (the epilogue without them has no spills)
template <int KC, int N, bool EXT>
__global__ void __launch_bounds__(ConvCfg<KC, N>::NTHREADS, 1)
    k_conv3_tc(const __grid_constant__ CUtensorMap tmap, ConvArgs a) {
    using Cfg = ConvCfg<KC, N>;
    constexpr int PLANES = Cfg::PLANES, NACC = Cfg::NACC, NP = Cfg::NP, ZN = Cfg::ZN;
    static_assert(PLANES >= 5 && Cfg::PLANE % 1024 == 0, "plane ring");
    extern __shared__ uint8_t smem_raw[];
    // 1024-byte aligned base: weights first, then the plane ring
    uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint8_t *wsm = smem;
    uint8_t *ring = smem + Cfg::RING;
    __shared__ __align__(8) uint64_t full_b[PLANES], empty_b[PLANES], tfull_b[NACC], tempty_b[NACC], wfull_b, done_b;
    __shared__ __align__(16) float bias_s[N];
    __shared__ uint32_t taddr_s;
    __shared__ int abort_s;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

    if (tid >= 64 && tid < 64 + N)
        bias_s[tid - 64] = a.bias ? __ldg(a.bias + a.out_off + (int)(blockIdx.x % (unsigned)a.nslice) * N + tid - 64) : 0.0f;
    if (warp == 1) {
        tmem_alloc(smem_u32(&taddr_s), 512);
        tmem_relinquish();
    }
    if (tid == 0) {
        for (int s = 0; s < PLANES; ++s) {
            mbar_init(smem_u32(&full_b[s]), 1);
            mbar_init(smem_u32(&empty_b[s]), 1);
        }
        for (int k = 0; k < NACC; ++k) {
            mbar_init(smem_u32(&tfull_b[k]), 1);
            mbar_init(smem_u32(&tempty_b[k]), 4 * Cfg::NG);
        }
        mbar_init(smem_u32(&wfull_b), 1);
        mbar_init(smem_u32(&done_b), 1);
        abort_s = 0;
        fence_mbar_init();
        prefetch_tmap(&tmap);
        // weights by bulk copies while TMEM is allocated and the first planes arrive; they
        // are in core layout [9 (dz, dy)][KC][NP] already, with ZN = 3 the rows of the
        // three dz of one dy go side by side, dz = 2 (the plane below) first
        const uint32_t wb = smem_u32(&wfull_b), w0 = smem_u32(wsm);
        const char *wt = reinterpret_cast<const char *>(a.wt) + (blockIdx.x % (unsigned)a.nslice) * Cfg::WBYTES;
        mbar_arrive_expect_tx(wb, Cfg::WBYTES);
        if (ZN == 1) {
            bulk_load(w0, wt, Cfg::WBYTES, wb);
        } else {
            for (int i = 0; i < 9 * KC; ++i) {
                const int z = i % 3, kc = (i / 3) % KC, dy = i / (3 * KC);
                bulk_load(w0 + (uint32_t)(i * NP * 16), wt + (((2 - z) * 3 + dy) * KC + kc) * NP * 16, NP * 16, wb);
            }
        }
    }
    fence_before_sync();
    __syncthreads();
    fence_after_sync();
    const uint32_t taddr = taddr_s;
    int tx0, tiles_x;
    conv_tiles_x(a.W, a.x_lo, a.x_hi, tx0, tiles_x);
    const int tiles_y = a.H / TY, nzc = (a.D + a.lz - 1) / a.lz;
    const long long nunits = (long long)a.B * nzc * tiles_y * tiles_x;
    // the CTAs of a launch share its output slices: slice = blockIdx.x % nslice
    const int slice = (int)(blockIdx.x % (unsigned)a.nslice);
    const long long u0 = blockIdx.x / (unsigned)a.nslice, ustep = gridDim.x / (unsigned)a.nslice;
    const uint32_t ring_s = smem_u32(ring), w_s = smem_u32(wsm);

    if (warp == 0) {
        // ------------------------------------------------------------ producer
        if (lane == 0) {
            Ring<PLANES> r;
            long long issued = 0;
            bool stop = false;
            for (long long u = u0; u < nunits && !stop; u += ustep) {
                const ConvUnit c = conv_unit(u, tx0, tiles_x, tiles_y, nzc, a.lz, a.D);
                for (int p = c.z0 - 1; p <= c.z1; ++p) {
                    if (!mbar_wait_abort(smem_u32(&empty_b[r.s]), r.ph ^ 1, MBAR_LIMIT, &abort_s)) {
                        atomicOr(a.status, ST_TIMEOUT);
                        *(volatile int *)&abort_s = 1;
                        stop = true;
                        break;
                    }
                    const uint32_t fb = smem_u32(&full_b[r.s]);
                    mbar_arrive_expect_tx(fb, Cfg::PLANE);
                    tma_load_5d(ring_s + (uint32_t)(r.s * Cfg::PLANE), &tmap, a.cin_off, c.tx * TXO, c.ty * TY - 1,
                                p, EXT && a.bmod ? c.b % a.bmod : c.b, fb);
                    ++issued;
                    r.next();
                }
            }
            // copies still in flight when the loop stopped early complete before exit
            if (*(volatile int *)&abort_s) {
                for (int k = 0; k < PLANES && issued > 0; ++k, --issued) {
                    if (--r.s < 0) {
                        r.s = PLANES - 1;
                        r.ph ^= 1;
                    }
                    mbar_wait(smem_u32(&full_b[r.s]), r.ph, MBAR_LIMIT);
                }
            }
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------ MMA issuer
        // (the whole warp runs the loop; an elected lane issues)
        const uint64_t a0 = KC == 4 ? smem_desc_sw64(0, 8 * 64) : smem_desc_sw32(0, 8 * 32);
        const uint64_t b0 = smem_desc(0, ZN * NP * 16, 128);
        const uint32_t ahi = (uint32_t)(a0 >> 32), bhi = (uint32_t)(b0 >> 32);
        const uint32_t alo = (uint32_t)a0 + (ring_s >> 4), blo = (uint32_t)b0 + (w_s >> 4);  // below 2^14: no carry
        Ring<PLANES> pr;       // the plane being waited for
        Ring<NACC> ar;         // the accumulator of the next output plane to begin
        LookAhead<PLANES, NACC> look;
        if (!mbar_wait_abort(smem_u32(&wfull_b), 0, MBAR_LIMIT, &abort_s) && lane == 0) {
            atomicOr(a.status, ST_TIMEOUT);
            *(volatile int *)&abort_s = 1;
        }
        int ps[3] = {0, 0, 0}; // ring slots of planes p - 2, p - 1, p
        bool stop = false;
        for (long long u = u0; u < nunits && !stop; u += ustep) {
            const ConvUnit c = conv_unit(u, tx0, tiles_x, tiles_y, nzc, a.lz, a.D);
            int s0 = ar.s;     // accumulator of output plane max(p - 1, z0)
            for (int p = c.z0 - 1; p <= c.z1; ++p) {
                ps[0] = ps[1];
                ps[1] = ps[2];
                ps[2] = pr.s;
                // the output plane that this plane begins
                const bool begins = ZN == 3 ? p + 1 < c.z1 : p - 1 >= c.z0;
                if (!look.wait(full_b, pr.s, pr.ph, tempty_b, ar.s, ar.ph ^ 1, begins, lane, MBAR_LIMIT, &abort_s)) {
                    if (lane == 0) {
                        atomicOr(a.status, ST_TIMEOUT);
                        *(volatile int *)&abort_s = 1;
                    }
                    stop = true;
                    break;
                }
                pr.next();
                fence_after_sync();
                if constexpr (ZN == 1) {
                    if (p - 1 < c.z0) continue;
                    const uint32_t d = taddr + (uint32_t)(ar.s * NP);
                    constexpr uint32_t idesc = idesc_bf16(128, NP);
#pragma unroll
                    for (int dz = 0; dz < 3; ++dz) {
                        const uint32_t ad = alo + (uint32_t)((ps[dz] * Cfg::PLANE) >> 4);
#pragma unroll
                        for (int dy = 0; dy < 3; ++dy)
#pragma unroll
                            for (int kk = 0; kk < KC / 2; ++kk)
                                umma_bf16_warp(d, ad + (uint32_t)((dy * TX * Cfg::ROWB + kk * 32) >> 4), ahi,
                                               blo + (uint32_t)((((dz * 3 + dy) * KC + 2 * kk) * NP * 16) >> 4), bhi, idesc,
                                               (dz | dy | kk) != 0);
                    }
                    umma_commit_warp(smem_u32(&empty_b[ps[0]]));   // the lowest plane may be refilled
                    if (p == c.z1) {
                        umma_commit_warp(smem_u32(&empty_b[ps[1]]));
                        umma_commit_warp(smem_u32(&empty_b[ps[2]]));
                    }
                    umma_commit_warp(smem_u32(&tfull_b[ar.s]));    // the accumulator is ready
                    ar.next();
                } else {
                    const uint32_t ad = alo + (uint32_t)(ps[2] * (Cfg::PLANE >> 4));
                    if (p > c.z0 && begins && s0 + 2 < NACC) {
                        // inside a column: three output planes in accumulators s0 .. s0 + 2, the
                        // last one begun (its first product overwrites it); constants only
                        const uint32_t d = taddr + (uint32_t)(s0 * NP);
                        umma_bf16_warp(d, ad, ahi, blo, bhi, idesc_bf16(128, 2 * NP), 1);
                        umma_bf16_warp(d + 2 * NP, ad, ahi, blo + 2 * NP, bhi, idesc_bf16(128, NP), 0);
#pragma unroll
                        for (int i = 1; i < 3 * KC / 2; ++i)
                            umma_bf16_warp(d, ad + (uint32_t)(((i / (KC / 2)) * TX * Cfg::ROWB + (i % (KC / 2)) * 32) >> 4),
                                           ahi, blo + (uint32_t)(i * 6 * NP), bhi, idesc_bf16(128, 3 * NP), 1);
                    } else {
                        // output planes lo .. hi (dz = p - z + 1), in consecutive accumulators from s0
                        const int lo = max(p - 1, c.z0), hi = min(p + 1, c.z1 - 1), n = hi - lo + 1;
                        const uint32_t bd = blo + (uint32_t)(((lo - p + 1) * NP * 16) >> 4);
                        auto mma = [&](int dy, int kk, int first, int cnt, uint32_t acc) {
                            const int sl = s0 + first;
                            umma_bf16_warp(taddr + (uint32_t)((sl < NACC ? sl : sl - NACC) * NP),
                                           ad + (uint32_t)((dy * TX * Cfg::ROWB + kk * 32) >> 4), ahi,
                                           bd + (uint32_t)(first * NP) + (uint32_t)(((dy * KC + 2 * kk) * 3 * NP * 16) >> 4),
                                           bhi, idesc_bf16(128, 8) - (1u << 17) + ((uint32_t)(cnt * NP) << 14), acc);
                        };
                        // the first product of a new accumulator overwrites it
                        const int old = begins ? n - 1 : n, n1 = min(n, NACC - s0), o1 = min(old, n1);
                        if (o1 > 0) mma(0, 0, 0, o1, 1);
                        if (old > o1) mma(0, 0, o1, old - o1, 1);
                        if (begins) mma(0, 0, n - 1, 1, 0);
                        if (n1 == n) {
#pragma unroll
                            for (int i = 1; i < 3 * KC / 2; ++i) mma(i / (KC / 2), i % (KC / 2), 0, n, 1);
                        } else {
                            // the accumulator ring wraps
#pragma unroll
                            for (int i = 1; i < 3 * KC / 2; ++i) {
                                mma(i / (KC / 2), i % (KC / 2), 0, n1, 1);
                                mma(i / (KC / 2), i % (KC / 2), n1, n - n1, 1);
                            }
                        }
                    }
                    umma_commit_warp(smem_u32(&empty_b[ps[2]]));
                    if (begins) ar.next();
                    if (p - 1 >= c.z0) {
                        umma_commit_warp(smem_u32(&tfull_b[s0]));  // output plane p - 1 is complete
                        if (++s0 == NACC) s0 = 0;
                    }
                }
            }
        }
        // every MMA issued has finished reading shared memory before exit
        umma_commit_warp(smem_u32(&done_b));
        mbar_wait(smem_u32(&done_b), 0, MBAR_LIMIT);
    } else {
        // ------------------------------------------------------------ epilogue
        const int q = warp & 3;                    // TMEM lane quarter this warp may access
        const int grp = ((warp - 2) >> 2) % Cfg::NG;  // its 16 output channels of the slice
        const int set = ((warp - 2) >> 2) / Cfg::NG;  // its share of the output planes
        const int m = q * 32 + lane;               // accumulator row = cell of the block
        const float scale = a.scale_out ? a.drop_scale : 1.0f;
        const uint64_t scale2 = f32x2(scale, scale);
        const int bx = m & (TX - 1);               // cell of the block row (0 and TX - 1 are halo)
        const long long opitch = a.out_pitch ? a.out_pitch : N;
        const long long HW = (long long)a.H * a.W, ostep = HW * opitch;
        // dropout threshold in both halves; its top bits pick the compare below
        const uint32_t thr = a.drop_thr, thr7 = (thr & 0x7FFFu) * 0x10001u, thr_low = thr < 0x8000u ? 0xFFFFFFFFu : 0u;
        const int ch0 = a.out_off + slice * N + grp * EPC;  // first channel of the warp in the output
        const uint32_t bias4 = smem_u32(bias_s + grp * EPC);
        Ring<NACC> ar;
        int turn = 0;
        bool stop = false;
        for (long long u = u0; u < nunits && !stop; u += ustep) {
            const ConvUnit c = conv_unit(u, tx0, tiles_x, tiles_y, nzc, a.lz, a.D);
            const int cx = c.tx * TXO + bx, cy = c.ty * TY + (m >> 4);
            // a block's first and last cell yield an output only where the volume ends there;
            // cells past the volume write nothing
            const bool valid = cx < a.W && (bx != 0 || cx == 0) && (bx != TX - 1 || cx == a.W - 1);
            uint32_t lin = (uint32_t)(((long long)c.z0 * a.H + cy) * a.W + (valid ? cx : 0));
            long long obase = ((((long long)c.b * a.D + c.z0) * a.H + cy) * a.W + (valid ? cx : 0)) * opitch + ch0;
            // where the shortcut of the cell lies
            long long rbase = EXT ? ((((long long)(a.bmod ? c.b % a.bmod : c.b) * a.D + c.z0) * a.H + cy) * a.W +
                                     (valid ? cx : 0)) * a.res_ch + ch0
                                  : 0;
            // several MC passes of one batch run side by side: sample b is pass b / pass_b's
            const uint32_t bdrop = EXT && a.pass_b ? (uint32_t)c.b % (uint32_t)a.pass_b : (uint32_t)c.b;
            const uint32_t pass = a.pass + (EXT && a.pass_b ? (uint32_t)c.b / (uint32_t)a.pass_b : 0u);
            for (int z = c.z0; z < c.z1; ++z, lin += (uint32_t)HW, obase += ostep, ar.next()) {
                const bool mine = turn == set;
                if (++turn == Cfg::NSET) turn = 0;
                if (!mine) continue;
                // first what does not need the accumulator (it overlaps the MMAs): the
                // dropout masks, one half-word per channel (kept where its field >= threshold)
                uint32_t keep[EPC / 2];
#pragma unroll
                for (int w = 0; w < EPC / 2; ++w) keep[w] = 0xFFFFFFFFu;
                if (thr) {
#pragma unroll
                    for (int h = 0; h < EPC / 8; ++h) {
                        const u32x4 r = philox4x32_10(lin, bdrop, (a.layer << 16) | (uint32_t)(ch0 / 8 + h), pass, a.seed, 0xD0u);
#pragma unroll
                        for (int w = 0; w < 4; ++w) {
                            // per half: bit 15 of t is (low 15 bits >= the threshold's)
                            const uint32_t t = (r.v[w] | 0x80008000u) - thr7;
                            const uint32_t ge = (r.v[w] & t) | (thr_low & (r.v[w] | t));
                            asm("prmt.b32 %0, %1, 0, 0xBB99;" : "=r"(keep[h * 4 + w]) : "r"(ge));
                        }
                    }
                }
                const bool ok = mbar_wait_abort(smem_u32(&tfull_b[ar.s]), ar.ph, MBAR_LIMIT, &abort_s);
                if (!__all_sync(0xffffffffu, ok)) {
                    if (lane == 0) {
                        atomicOr(a.status, ST_TIMEOUT);
                        *(volatile int *)&abort_s = 1;
                    }
                    stop = true;
                    break;
                }
                fence_after_sync();
                // row m holds, per x-tap dx, the partial sum of the outputs at cell
                // x - dx + 1; the output at x is D_0[x - 1] + D_1[x] + D_2[x + 1]
                uint64_t v2[EPC / 2];
                {
                    float p[3 * EPC];
                    const uint32_t rowa = taddr + ((uint32_t)(q * 32) << 16) + (uint32_t)(ar.s * NP + grp * EPC);
                    tmem_ld16x3(rowa, rowa + (uint32_t)N, rowa + (uint32_t)(2 * N), p);
                    fence_before_sync();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(smem_u32(&tempty_b[ar.s]));
                    // lanes m - 1 and m + 1 are the x-neighbours; the block row's first and last
                    // cell have none where the volume ends there (elsewhere they write nothing)
#pragma unroll
                    for (int o = 0; o < EPC; o += 2) {
                        const float l0 = __shfl_up_sync(0xffffffffu, p[o], 1);
                        const float l1 = __shfl_up_sync(0xffffffffu, p[o + 1], 1);
                        const float r0 = __shfl_down_sync(0xffffffffu, p[2 * EPC + o], 1);
                        const float r1 = __shfl_down_sync(0xffffffffu, p[2 * EPC + o + 1], 1);
                        const uint64_t left = f32x2(bx == 0 ? 0.0f : l0, bx == 0 ? 0.0f : l1);
                        const uint64_t right = f32x2(bx == TX - 1 ? 0.0f : r0, bx == TX - 1 ? 0.0f : r1);
                        v2[o / 2] = add2(add2(left, f32x2(p[EPC + o], p[EPC + o + 1])), right);
                    }
                }
                if (valid) {
                    if (EXT && a.part_in) {
                        // the sums of the input-channel chunks before this one
                        const float4 *p4 = reinterpret_cast<const float4 *>(a.part_in + obase);
#pragma unroll
                        for (int j = 0; j < EPC / 4; ++j) {
                            const float4 p0 = p4[j];
                            v2[2 * j] = add2(f32x2(p0.x, p0.y), v2[2 * j]);
                            v2[2 * j + 1] = add2(f32x2(p0.z, p0.w), v2[2 * j + 1]);
                        }
                    }
                    if (EXT && a.raw_out) {
                        float4 *o4 = reinterpret_cast<float4 *>(a.raw_out + obase);
#pragma unroll
                        for (int j = 0; j < EPC / 4; ++j) {
                            const float2 s0 = unpack2(v2[2 * j]), s1 = unpack2(v2[2 * j + 1]);
                            o4[j] = make_float4(s0.x, s0.y, s1.x, s1.y);
                        }
                    }
                    float v[EPC];
#pragma unroll
                    for (int j = 0; j < EPC; j += 4) {
                        // the bias stays in shared memory: the loop has no registers for it, and a
                        // spill costs an L2 round trip here (the L1 is all shared memory)
                        uint64_t b2[2];
                        asm volatile("ld.shared.v2.b64 {%0, %1}, [%2];" : "=l"(b2[0]), "=l"(b2[1]) : "r"(bias4 + 4u * j));
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            float2 s2 = unpack2(add2(v2[j / 2 + h], b2[h]));
                            if (a.relu) s2 = make_float2(fmaxf(s2.x, 0.0f), fmaxf(s2.y, 0.0f));
                            s2 = unpack2(mul2(f32x2(s2.x, s2.y), scale2));
                            v[j + 2 * h] = s2.x;
                            v[j + 2 * h + 1] = s2.y;
                        }
                    }
                    if (a.y_f32) {
                        float4 *o4 = reinterpret_cast<float4 *>(a.y_f32 + obase);
#pragma unroll
                        for (int j = 0; j < EPC; ++j)
                            if (!((keep[j >> 1] >> (16 * (j & 1))) & 1u)) v[j] = 0.0f;
#pragma unroll
                        for (int j = 0; j < EPC / 4; ++j)
                            o4[j] = make_float4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
                    } else if (!EXT || a.y) {
                        uint32_t o[EPC / 2];
#pragma unroll
                        for (int j = 0; j < EPC / 2; ++j) {
                            const __nv_bfloat162 h = __floats2bfloat162_rn(v[2 * j], v[2 * j + 1]);
                            o[j] = *reinterpret_cast<const uint32_t *>(&h) & keep[j];
                        }
                        if (EXT && ch0 < a.res_ch) {
                            // identity shortcut: the dropped-out FP32 value plus the layer's input, one rounding
                            const uint4 *r4 = reinterpret_cast<const uint4 *>(a.res + rbase + (z - c.z0) * HW * a.res_ch);
                            const uint4 ra = r4[0], rb = r4[1];
                            const uint32_t rw[EPC / 2] = {ra.x, ra.y, ra.z, ra.w, rb.x, rb.y, rb.z, rb.w};
#pragma unroll
                            for (int j = 0; j < EPC / 2; ++j) {
                                const float x0 = __uint_as_float(rw[j] << 16), x1 = __uint_as_float(rw[j] & 0xFFFF0000u);
                                const __nv_bfloat162 h = __floats2bfloat162_rn((keep[j] & 1u ? v[2 * j] : 0.0f) + x0,
                                                                               (keep[j] >> 16 ? v[2 * j + 1] : 0.0f) + x1);
                                o[j] = *reinterpret_cast<const uint32_t *>(&h);
                            }
                        }
                        uint4 *o4 = reinterpret_cast<uint4 *>(a.y + obase);
                        o4[0] = make_uint4(o[0], o[1], o[2], o[3]);
                        o4[1] = make_uint4(o[4], o[5], o[6], o[7]);
                }
                }
            }
        }
    }
    fence_before_sync();
    __syncthreads();
    fence_after_sync();
    if (warp == 1) tmem_dealloc(taddr, 512);
}

// ---------------------------------------------------------------- host side

typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static EncodeTiledFn encode_fn() {
    static EncodeTiledFn fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = (EncodeTiledFn)p;
    });
    return fn;
}

// tensor map of a channels-last BF16 activation [B][D][H][W][C]: dims
// (C, W, H, D, B), box (16 or 32 channels, halo x, halo y, 1 plane, 1)
static hyb_status make_tmap(CUtensorMap *tm, const ConvArgs &a) {
    EncodeTiledFn enc = encode_fn();
    if (!enc) return set_error(HYB_ECUDA, "cuTensorMapEncodeTiled is not available");
    const cuuint64_t C = (cuuint64_t)(a.cin_total ? a.cin_total : a.cin);
    const cuuint64_t dims[5] = {C, (cuuint64_t)a.W, (cuuint64_t)a.H, (cuuint64_t)a.D, (cuuint64_t)(a.bmod ? a.bmod : a.B)};
    const cuuint64_t es = 2;
    const cuuint64_t strides[4] = {es * C, es * C * a.W, es * C * a.W * a.H, es * C * a.W * a.H * a.D};
    const cuuint32_t box[5] = {(cuuint32_t)a.cin, (cuuint32_t)TX, (cuuint32_t)HY, 1, 1};
    const cuuint32_t estr[5] = {1, 1, 1, 1, 1};
    CUresult r = enc(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, (void *)a.x, dims, strides, box, estr,
                     CU_TENSOR_MAP_INTERLEAVE_NONE, a.cin == 32 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_32B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                     CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return set_error(HYB_ECUDA, "cuTensorMapEncodeTiled failed (" + std::to_string((int)r) + ")");
    return HYB_OK;
}

template <int KC, int N, bool EXT>
static hyb_status launch_cfg(const ConvArgs &a, cudaStream_t st) {
    using Cfg = ConvCfg<KC, N>;
    CUtensorMap tm;
    hyb_status s = make_tmap(&tm, a);
    if (s != HYB_OK) return s;
    // per-device launch set-up, done once (its host cost shows on small grids)
    static std::mutex mu;
    static int ready_dev[64] = {0}, nsm_dev[64] = {0};
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev < 0 || dev >= 64) return set_error(HYB_EINVAL, "device index out of range");
    int nsm;
    {
        std::lock_guard<std::mutex> lock(mu);
        if (!ready_dev[dev]) {
            cudaError_t e = cudaFuncSetAttribute(k_conv3_tc<KC, N, EXT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                 Cfg::SMEM);
            if (e != cudaSuccess)
                return set_error(HYB_ECUDA, std::string("conv smem attribute: ") + cudaGetErrorString(e));
            cudaDeviceGetAttribute(&nsm_dev[dev], cudaDevAttrMultiProcessorCount, dev);
            ready_dev[dev] = 1;
        }
        nsm = nsm_dev[dev];
    }
    cudaError_t e;
    int tx0, ntx;
    conv_tiles_x(a.W, a.x_lo, a.x_hi, tx0, ntx);
    // output planes per column: the length that leaves the busiest SM the fewest
    // planes to compute, a fetched halo plane counted as a fifth of one (its
    // shared-memory writes against an output plane's MMAs).  Columns of one plane
    // suit volumes that leave SMs idle otherwise: a classifier forward of 8 x 16 x 8
    // cells 58.8 us with columns of two or more, 53.1 with one; a surrogate's of 16^3
    // 98.7 -> 92.5 us
    const long long cols = (long long)a.B * (a.H / TY) * ntx;
    if (cols == 0) return HYB_OK;
    ConvArgs b = a;
    if (b.nslice < 1) b.nslice = 1;
    const long long per = std::max(1, nsm / b.nslice);  // CTAs per output slice
    double best = 0.0;
    for (int lz = 1; lz <= 32; ++lz) {
        const long long u = cols * ((a.D + lz - 1) / lz);
        const double t = (double)((u + per - 1) / per) * (std::min(lz, a.D) + 0.4);
        if (lz == 1 || t < best) {
            best = t;
            b.lz = lz;
        }
    }
    const long long units = cols * ((a.D + b.lz - 1) / b.lz);
    const long long grid = std::min<long long>(units, per) * b.nslice;  // one CTA per SM (all of its TMEM)
    k_conv3_tc<KC, N, EXT><<<(unsigned)grid, Cfg::NTHREADS, Cfg::SMEM, st>>>(tm, b);
    e = cudaGetLastError();
    if (e != cudaSuccess) return set_error(HYB_ECUDA, std::string("conv launch: ") + cudaGetErrorString(e));
    return HYB_OK;
}

hyb_status launch_conv3_tc(const ConvArgs &a, cudaStream_t st) {
    if (a.W < 1 || a.H % TY != 0 || a.B < 1 || a.D < 1)
        return set_error(HYB_EINVAL, "conv shape: H % 8 == 0 required");
    if ((long long)a.B * a.D * (a.H / TY) * ((a.W + TXO - 1) / TXO) >= (1LL << 31))
        return set_error(HYB_EINVAL, "conv shape: more than 2^31 tiles");
    if (((uintptr_t)a.x & 15) || ((uintptr_t)a.y & 15) || ((uintptr_t)a.y_f32 & 15) || ((uintptr_t)a.wt & 15) ||
        ((uintptr_t)a.part_in & 15) || ((uintptr_t)a.raw_out & 15) || ((uintptr_t)a.res & 15) ||
        (!a.y && !a.y_f32 && !a.raw_out))
        return set_error(HYB_EINVAL, "conv operands must be present and 16-byte aligned");
    {
        // channel chunks: 16-channel aligned input and output slices (TMA x coordinate in
        // 32-byte steps, 32-byte stores)
        const int ct = a.cin_total ? a.cin_total : a.cin, op = a.out_pitch ? a.out_pitch : a.N;
        const int ns = a.nslice > 1 ? a.nslice : 1;
        if (ct % 16 || a.cin_off < 0 || a.cin_off % 16 || a.cin_off + a.cin > ct || op % 16 || a.out_off < 0 ||
            a.out_off % 16 || a.out_off + ns * a.N > op || a.res_ch % 16 || (a.res_ch && !a.res))
            return set_error(HYB_EINVAL, "conv channel slices out of range or misaligned");
    }
    const bool ext = a.part_in || a.raw_out || a.res_ch || a.bmod || a.pass_b;
    if (a.cin == 16 && a.N == 32) return ext ? launch_cfg<2, 32, true>(a, st) : launch_cfg<2, 32, false>(a, st);
    if (a.cin == 32 && a.N == 32) return ext ? launch_cfg<4, 32, true>(a, st) : launch_cfg<4, 32, false>(a, st);
    if (a.cin == 32 && a.N == 16) return ext ? launch_cfg<4, 16, true>(a, st) : launch_cfg<4, 16, false>(a, st);
    if (a.cin == 16 && a.N == 16) return ext ? launch_cfg<2, 16, true>(a, st) : launch_cfg<2, 16, false>(a, st);
    return set_error(HYB_EINVAL, "conv channels: (C_in, C_out) in {16, 32} x {16, 32}");
}


// ---------------------------------------------------------------- last layer
// k_conv_last_tc: the 16 -> 1 channel layer with all 27 taps in the MMA N
// dimension.  A plane block of 16 (x) x 8 (y) cells (M = 128 rows, K = the 16
// channels) times the weights of the 27 taps (N = 32, padded) gives, per cell
// c and tap t, the partial product P[c][t] = sum_ci x[c][ci] w[t][ci] -- one
// MMA per plane.  The output at cell c is y[c] = b + sum_t P[c + offset(t)][t]:
// the z part of the sum runs in registers (a cell's own partials of three
// consecutive planes), the in-plane 3 x 3 part through shared memory; the
// 14 x 6 interior cells of the block have all their neighbours in it.  A CTA walks a column of such blocks through z
// (chunks of LZC output planes plus one plane of halo on either side), so
// every plane is multiplied once and used by three output planes.
//   warp 0      TMA producer: one 16 x 8 x 1 x 16-channel box per plane
//               (zero fill outside the volume) into a ring of LSTAGES;
//   warp 1      MMA issuer: one tcgen05.mma (128 x 32 x 16) per plane into
//               one of two TMEM accumulators;
//   warps 2..5  epilogue: tcgen05.ld of the 32 columns, the z sums in
//               registers, the 9 in-plane partials of the completed output
//               plane into shared memory, a named barrier of the four warps,
//               the 3 x 3 gather, bias, and the logit or the sigmoid folded
//               into the MC mean / M2 (Welford).
// Waits are bounded; a warp whose wait gives up records ST_TIMEOUT and stops
// waiting, but the epilogue warps keep meeting at their barrier until the
// end, so no warp is left behind at it.
static constexpr int LTX = 16, LTY = 8;            // block (cells) = 128 MMA rows
static constexpr int LOX = LTX - 2, LOY = LTY - 2; // interior outputs per block row / column
static constexpr int LZC = 32;                     // output planes per work unit
static constexpr int LSTAGES = 4;
static constexpr int LCTAS = 4;                    // CTAs per SM (64 TMEM columns each)
static constexpr int LPF = 3;                      // planes of MC statistics read ahead
static constexpr int LSTAGE = LTX * LTY * 32;      // bytes of one plane block (4096)
static constexpr int LSMEM = LSTAGES * LSTAGE + 2 * 9 * 128 * 4 + 1024 + 1024;  // ring, 2 x Q, weights, slack

struct LastTiles {
    int tx0, tx_n, ty_n, zc_n;
    long long units;
};

// work units of the last layer: all block columns, or those whose outputs
// meet x_lo <= x < x_hi when x_hi > x_lo
__host__ __device__ inline LastTiles last_tiles(int B, int D, int H, int W, int x_lo, int x_hi) {
    LastTiles t;
    const int all = (W + LOX - 1) / LOX;
    if (x_hi > x_lo) {
        t.tx0 = x_lo / LOX;
        const int tx1 = (x_hi + LOX - 1) / LOX;
        t.tx_n = (tx1 < all ? tx1 : all) - t.tx0;
        if (t.tx_n < 0) t.tx_n = 0;
    } else {
        t.tx0 = 0;
        t.tx_n = all;
    }
    t.ty_n = (H + LOY - 1) / LOY;
    t.zc_n = (D + LZC - 1) / LZC;
    t.units = (long long)B * t.zc_n * t.ty_n * t.tx_n;
    return t;
}

// unit u -> block position and z range; planes z = zlo - 1 .. zhi
__device__ inline void last_unit(long long u, const LastTiles &t, int D, int &tx, int &ty, int &zlo, int &zhi,
                                 int &b) {
    tx = (int)(u % t.tx_n) + t.tx0;
    u /= t.tx_n;
    ty = (int)(u % t.ty_n);
    u /= t.ty_n;
    const int zc = (int)(u % t.zc_n);
    b = (int)(u / t.zc_n);
    zlo = zc * LZC;
    zhi = min(zlo + LZC, D);
}

__global__ void __launch_bounds__(192, LCTAS) k_conv_last_tc(const __grid_constant__ CUtensorMap tmap,
                                                      const __grid_constant__ LastArgs a) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint8_t *ring = smem;                                          // LSTAGES x 4 KB (1 KB aligned)
    uint8_t *wsm = smem + LSTAGES * LSTAGE;                        // 1 KB of weights
    float *qs = reinterpret_cast<float *>(wsm + 1024);             // [2][9][128] in-plane partials Q
    __shared__ __align__(8) uint64_t full_b[LSTAGES], empty_b[LSTAGES], tfull_b[2], tempty_b[2], done_b;
    __shared__ uint32_t taddr_s;
    __shared__ int abort_s;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

    if (warp == 1) {
        tmem_alloc(smem_u32(&taddr_s), 64);
        tmem_relinquish();
    }
    if (tid == 0) {
        for (int s = 0; s < LSTAGES; ++s) {
            mbar_init(smem_u32(&full_b[s]), 1);
            mbar_init(smem_u32(&empty_b[s]), 1);
        }
        for (int k = 0; k < 2; ++k) {
            mbar_init(smem_u32(&tfull_b[k]), 1);
            mbar_init(smem_u32(&tempty_b[k]), 4);
        }
        mbar_init(smem_u32(&done_b), 1);
        abort_s = 0;
        fence_mbar_init();
        prefetch_tmap(&tmap);
    }
    for (int i = tid; i < 256; i += 192) reinterpret_cast<uint32_t *>(wsm)[i] = a.w[i];
    fence_proxy_async_smem();
    fence_before_sync();
    __syncthreads();
    fence_after_sync();
    const uint32_t taddr = taddr_s;
    const LastTiles lt = last_tiles(a.B, a.D, a.H, a.W, a.x_lo, a.x_hi);
    const uint32_t ring_s = smem_u32(ring), w_s = smem_u32(wsm);

    if (warp == 0) {
        // ------------------------------------------------------------ producer
        if (lane == 0) {
            int s = 0;
            uint32_t ph = 0;
            long long issued = 0;
            bool stop = false;
            for (long long u = blockIdx.x; u < lt.units && !stop; u += gridDim.x) {
                int tx, ty, zlo, zhi, b;
                last_unit(u, lt, a.D, tx, ty, zlo, zhi, b);
                for (int z = zlo - 1; z <= zhi; ++z) {
                    if (!mbar_wait(smem_u32(&empty_b[s]), ph ^ 1, MBAR_LIMIT) || *(volatile int *)&abort_s) {
                        atomicOr(a.status, ST_TIMEOUT);
                        *(volatile int *)&abort_s = 1;
                        stop = true;
                        break;
                    }
                    const uint32_t fb = smem_u32(&full_b[s]);
                    mbar_arrive_expect_tx(fb, LSTAGE);
                    tma_load_5d(ring_s + (uint32_t)(s * LSTAGE), &tmap, 0, tx * LOX - 1, ty * LOY - 1, z, b, fb);
                    ++issued;
                    if (++s == LSTAGES) {
                        s = 0;
                        ph ^= 1;
                    }
                }
            }
            if (*(volatile int *)&abort_s) {
                for (int k = 0; k < LSTAGES && issued > 0; ++k, --issued) {
                    if (--s < 0) {
                        s = LSTAGES - 1;
                        ph ^= 1;
                    }
                    mbar_wait(smem_u32(&full_b[s]), ph, MBAR_LIMIT);
                }
            }
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------ MMA issuer
        if (lane == 0) {
            constexpr uint32_t idesc = idesc_bf16(128, 32);
            const uint64_t a0 = smem_desc_sw32(ring_s, 8 * 32);
            const uint64_t bd = smem_desc(w_s, 32 * 16, 128);
            int s = 0;
            uint32_t ph = 0;
            long long it = 0;
            bool stop = false;
            for (long long u = blockIdx.x; u < lt.units && !stop; u += gridDim.x) {
                int tx, ty, zlo, zhi, b;
                last_unit(u, lt, a.D, tx, ty, zlo, zhi, b);
                for (int z = zlo - 1; z <= zhi; ++z, ++it) {
                    const int acc = (int)(it & 1);
                    const uint32_t aph = (uint32_t)((it >> 1) & 1);
                    if (!mbar_wait(smem_u32(&tempty_b[acc]), aph ^ 1, MBAR_LIMIT) ||
                        !mbar_wait(smem_u32(&full_b[s]), ph, MBAR_LIMIT) || *(volatile int *)&abort_s) {
                        atomicOr(a.status, ST_TIMEOUT);
                        *(volatile int *)&abort_s = 1;
                        stop = true;
                        break;
                    }
                    fence_after_sync();
                    umma_bf16(taddr + (uint32_t)(acc * 32), a0 + (uint64_t)((s * LSTAGE) >> 4), bd, idesc, 0);
                    umma_commit(smem_u32(&empty_b[s]));
                    umma_commit(smem_u32(&tfull_b[acc]));
                    if (++s == LSTAGES) {
                        s = 0;
                        ph ^= 1;
                    }
                }
            }
            umma_commit(smem_u32(&done_b));
            mbar_wait(smem_u32(&done_b), 0, MBAR_LIMIT);
        }
    } else {
        // ------------------------------------------------------------ epilogue
        // With P_z[c][t] the partials of plane z, the output of plane o at
        // cell c is b + sum over (dy, dx) of Q_o[c + (dy - 1, dx - 1)][dy, dx],
        // where Q_o[c][dy, dx] = sum over dz of P_{o + dz - 1}[c][(dz, dy, dx)]
        // needs only the cell's own rows: each thread accumulates it in
        // registers as the planes stream past (r1: plane o + 1's part so far,
        // r2: plane o's), and only the 9 values of Q cross threads, through a
        // double-buffered shared array and one barrier per plane.
        const int q = warp & 3;
        const int m = q * 32 + lane;                 // row = cell of the block
        const int lx = m & (LTX - 1), ly = m >> 4;
        const bool interior = lx >= 1 && lx <= LOX && ly >= 1 && ly <= LOY;
        const float inv_k = a.mc_k > 0 ? 1.0f / (float)a.mc_k : 0.0f;  // the Welford weight of this pass
        bool dead = false;
        const long long V = (long long)a.D * a.H * a.W;
        long long it = 0;
        for (long long u = blockIdx.x; u < lt.units; u += gridDim.x) {
            int tx, ty, zlo, zhi, b;
            last_unit(u, lt, a.D, tx, ty, zlo, zhi, b);
            const int cx = tx * LOX + lx - 1, cy = ty * LOY + ly - 1;
            // with an x-range, the block's cells outside it keep their statistics
            const bool valid = interior && cx < a.W && cy < a.H && (a.x_hi <= a.x_lo || (cx >= a.x_lo && cx < a.x_hi));
            float r1[9], r2[9];
#pragma unroll
            for (int k = 0; k < 9; ++k) r1[k] = r2[k] = 0.0f;
            // MC statistics of output planes zo .. zo + LPF - 1, read LPF planes
            // ahead so that their latency spans several planes
            // (at the top of the iteration for output plane zo, entry k holds plane zo + k)
            const long long HW = (long long)a.H * a.W;
            const long long t0 = (long long)b * V + ((long long)(zlo - 2) * a.H + cy) * a.W + cx;
            float pmq[LPF], m2q[LPF];
#pragma unroll
            for (int k = 0; k < LPF; ++k) {
                pmq[k] = m2q[k] = 0.0f;
                const int zk = zlo - 2 + k;
                if (valid && a.mc_k >= 2 && zk >= zlo && zk < zhi) {
                    pmq[k] = a.pm[t0 + k * HW];
                    m2q[k] = a.m2[t0 + k * HW];
                }
            }
            for (int z = zlo - 1; z <= zhi; ++z, ++it) {
                const int acc = (int)(it & 1);
                const uint32_t aph = (uint32_t)((it >> 1) & 1);
                const int zo = z - 1;                // output plane completed by plane z
                const bool out = valid && zo >= zlo;
                const long long t = (long long)b * V + ((long long)zo * a.H + cy) * a.W + cx;
                const float mo = pmq[0], m2o = m2q[0];
#pragma unroll
                for (int k = 0; k + 1 < LPF; ++k) {
                    pmq[k] = pmq[k + 1];
                    m2q[k] = m2q[k + 1];
                }
                pmq[LPF - 1] = m2q[LPF - 1] = 0.0f;
                if (valid && a.mc_k >= 2 && zo + LPF >= zlo && zo + LPF < zhi) {
                    pmq[LPF - 1] = a.pm[t + LPF * HW];
                    m2q[LPF - 1] = a.m2[t + LPF * HW];
                }
                if (!dead) {
                    const bool ok = mbar_wait(smem_u32(&tfull_b[acc]), aph, MBAR_LIMIT) &&
                                    !*(volatile int *)&abort_s;
                    if (!__all_sync(0xffffffffu, ok)) {
                        if (lane == 0) {
                            atomicOr(a.status, ST_TIMEOUT);
                            *(volatile int *)&abort_s = 1;
                        }
                        dead = true;
                    }
                }
                float p[32];
                if (!dead) {
                    fence_after_sync();
                    tmem_ld32(taddr + ((uint32_t)(q * 32) << 16) + (uint32_t)(acc * 32), p);
                    fence_before_sync();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(smem_u32(&tempty_b[acc]));
                } else {
#pragma unroll
                    for (int k = 0; k < 32; ++k) p[k] = 0.0f;
                }
                // plane z is tap dz = 2 of output zo, dz = 1 of zo + 1, dz = 0 of zo + 2
                float *qb = qs + (int)(it & 1) * (9 * 128);
#pragma unroll
                for (int k = 0; k < 9; ++k) {
                    qb[k * 128 + m] = r2[k] + p[18 + k];
                    r2[k] = r1[k] + p[9 + k];
                    r1[k] = p[k];
                }
                // Q of plane zo is complete (and the buffer written two planes
                // ago is no longer read): the four epilogue warps meet
                asm volatile("bar.sync 1, 128;" ::: "memory");
                if (!dead && out) {
                    float s0 = 0.0f, s1 = 0.0f, s2 = 0.0f;
#pragma unroll
                    for (int dx = 0; dx < 3; ++dx) {
                        s0 += qb[(0 * 3 + dx) * 128 + m - LTX + dx - 1];
                        s1 += qb[(1 * 3 + dx) * 128 + m + dx - 1];
                        s2 += qb[(2 * 3 + dx) * 128 + m + LTX + dx - 1];
                    }
                    const float logit = a.bias + s0 + s1 + s2;
                    if (a.mc_k == 0) {
                        a.logit[t] = logit;
                    } else {
                        const float pv = __frcp_rn(1.0f + __expf(-logit));
                        if (a.mc_k == 1) {
                            a.pm[t] = pv;
                            a.m2[t] = 0.0f;
                        } else {
                            const float d = pv - mo;
                            const float mn = mo + d * inv_k;
                            a.pm[t] = mn;
                            a.m2[t] = m2o + d * (pv - mn);
                        }
                    }
                }
            }
        }
    }
    fence_before_sync();
    __syncthreads();
    fence_after_sync();
    if (warp == 1) tmem_dealloc(taddr, 64);
}

hyb_status launch_conv_last_tc(const LastArgs &a, cudaStream_t st) {
    if (a.B < 1 || a.D < 1 || a.H < 1 || a.W < 1) return set_error(HYB_EINVAL, "last layer: empty volume");
    if (((uintptr_t)a.x & 15) || (a.mc_k == 0 && !a.logit) || (a.mc_k > 0 && (!a.pm || !a.m2)))
        return set_error(HYB_EINVAL, "last layer: operands missing or not 16-byte aligned");
    const LastTiles lt = last_tiles(a.B, a.D, a.H, a.W, a.x_lo, a.x_hi);
    EncodeTiledFn enc = encode_fn();
    if (!enc) return set_error(HYB_ECUDA, "cuTensorMapEncodeTiled is not available");
    CUtensorMap tm;
    const cuuint64_t dims[5] = {16, (cuuint64_t)a.W, (cuuint64_t)a.H, (cuuint64_t)a.D, (cuuint64_t)a.B};
    const cuuint64_t strides[4] = {32ull, 32ull * a.W, 32ull * a.W * a.H, 32ull * a.W * a.H * a.D};
    const cuuint32_t box[5] = {16, (cuuint32_t)LTX, (cuuint32_t)LTY, 1, 1};
    const cuuint32_t estr[5] = {1, 1, 1, 1, 1};
    CUresult r = enc(&tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, (void *)a.x, dims, strides, box, estr,
                     CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_32B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                     CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return set_error(HYB_ECUDA, "last layer: tensor map (" + std::to_string((int)r) + ")");
    static std::mutex mu;
    static int ready_dev[64] = {0}, nsm_dev[64] = {0};
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev < 0 || dev >= 64) return set_error(HYB_EINVAL, "device index out of range");
    int nsm;
    {
        std::lock_guard<std::mutex> lock(mu);
        if (!ready_dev[dev]) {
            cudaError_t e = cudaFuncSetAttribute(k_conv_last_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, LSMEM);
            if (e != cudaSuccess)
                return set_error(HYB_ECUDA, std::string("last layer smem attribute: ") + cudaGetErrorString(e));
            cudaDeviceGetAttribute(&nsm_dev[dev], cudaDevAttrMultiProcessorCount, dev);
            ready_dev[dev] = 1;
        }
        nsm = nsm_dev[dev];
    }
    // LCTAS CTAs per SM by registers and shared memory (the occupancy query
    // answers 1 for kernels that allocate tensor memory); units are
    // independent, so any residency gives the same result
    if (lt.units == 0) return HYB_OK;
    const long long grid = std::min<long long>(lt.units, (long long)nsm * LCTAS);
    k_conv_last_tc<<<(unsigned)grid, 192, LSMEM, st>>>(tm, a);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return set_error(HYB_ECUDA, std::string("last layer launch: ") + cudaGetErrorString(e));
    return HYB_OK;
}

// Self-test of the bounded barrier wait the convolutions use: one thread
// waits on an mbarrier that nothing arrives at, gives up after `polls` polls
// and latches ST_TIMEOUT -- the path a stalled tensor-core pipeline takes.
__global__ void k_wait_selftest(long long polls, int *__restrict__ status) {
    __shared__ __align__(8) uint64_t bar;
    if (threadIdx.x == 0) {
        mbar_init(smem_u32(&bar), 1);
        fence_mbar_init();
        if (!mbar_wait(smem_u32(&bar), 0, polls)) atomicOr(status, ST_TIMEOUT);
    }
}

void launch_wait_selftest(long long polls, int *status, cudaStream_t st) {
    k_wait_selftest<<<1, 32, 0, st>>>(polls, status);
}

}  // namespace hyb
