// Weight gradient of a 3x3x3 convolution (circular padding) on the tcgen05
// tensor cores:
//     dW[co][ci][kz][ky][kx] = sum_p dZ[co, p] X[ci, p + (kx - 1, ky - 1, kz - 1)],
// a GEMM with K = cells.  Both operands come straight from row-planar
// activations (layout in conv_tc.cuh), in which a cell's eight channels are
// one 16-byte row: staged by the TMA, a plane of 136 cells is a column of
// MN-major core matrices (8 channels x 8 cells, 128 contiguous bytes), K
// advancing by 128 bytes per core matrix and the next 8 channels one plane
// (2176 bytes) further.  A shift of the input by one cell (the kx taps) is a
// 16-byte shift of the operand's start.
//
// The sum is split by the input cell q (each tile's 128 cells):
//     dW_kx[ci][co] = sum_q X[ci, q] dZ[co, q + 1 - kx]   (for each (kz, ky) input row),
// so the A operand (the activations, rows of the tile's cells) is the same for
// the three kx taps and the B operand is dZ at three one-cell shifts.  The nine
// input rows (y + ky - 1, z + kz - 1) of a tile lie in three consecutive z-slices
// of three rows each, held in a ring of slices.  GEMM M = 128 rows = 16
// consecutive planes (input row, channel group) x 8 channels: with 32 input
// channels one block per slice (its 12 planes; the 4 planes after it are read
// into discarded rows), with 8 one block over the 9 planes of the three slices,
// kept contiguous by mirroring the ring's first two slots after its last.
// N = (kx, output channel): the TMA lands dZ's tile (with its periodic halo
// cells) beside three copy areas, and the epilogue warps, idle until the end,
// write the copies shifted by 0, 1 and 2 cells, plane after plane, so that one
// descriptor spans all three at a uniform stride (N = 3 x 16 or 3 x 32); rows of
// cells past nx (a ragged tile) are written as zeros, so those cells add nothing.
// Each M block owns an accumulator in TMEM for the CTA's
// whole run, so the sum over all cells a CTA processes stays on chip; at the end
// the epilogue warps write per-CTA partial sums, which a second kernel adds in
// binary64 in a fixed order.
//
// Warp roles: warp 8 (one thread) issues the TMA copies, warp 9 the MMAs; warps 0-7, two
// sets, prepare the dZ tiles' shifted copies in turn and read the accumulators at the end
// (warps 0-3 zero them).  Every wait is bounded; on timeout the role records an error word
// and stops.
#pragma once

#include "conv_tc.cuh"

namespace ac {
namespace tc {

constexpr int WTHREADS = 32 * (4 * 2 + 2);  // two sets of copy warps, TMA, MMA

struct WgradTcArgs {
    float *part;  // [grid][NACC][N3][128] per-CTA partial sums
    int nx, ny, nz;
    int zc;       // tiles per column segment
    unsigned *err;
};

// Shape constants of the weight-gradient kernel for CIN input and COUT output channels.
template <int CIN, int COUT>
struct WgradShape {
    static constexpr int KC = CIN / 8;                       // planes per input row
    static constexpr int NPL = 9 * KC;                       // planes of the nine-row run
    // 32 input channels: one M block per slice (its 12 planes, 4 more rows discarded),
    // so no block crosses a slice and the ring needs no mirror; 8 input channels: one
    // block over the 9 planes of three slices kept contiguous by a mirrored ring
    static constexpr bool MIRROR = KC == 1;
    static constexpr int NMB = MIRROR ? 1 : 3;               // M blocks
    static constexpr int BLK = MIRROR ? 0 : 3 * KC;          // planes per block (stride of P0)
    static constexpr int DKC = COUT < 16 ? 2 : COUT / 8;     // planes of a dZ tile
    static constexpr int NB = 8 * DKC;                       // output channels (padded)
    static constexpr int N3 = 3 * NB;                        // GEMM N = (kx, channel)
    static constexpr int NACC = NMB;                         // accumulators (one per M block)
    static constexpr int TCOLS = NACC * N3 <= 32 ? 32 : NACC * N3 <= 64 ? 64 : NACC * N3 <= 128 ? 128
                                 : NACC * N3 <= 256 ? 256 : 512;
    static constexpr int NSLOT = MIRROR ? 8 : 5;             // slice ring (plus two mirrors)
    static constexpr int ROW = KC * PLANE;
    static constexpr int SLICE = 3 * ROW;
    static constexpr int NL = 2;                             // landed dZ tiles (TMA ring)
    static constexpr int NC = 2;                             // sets of three shifted copies
    static constexpr int COPY = DKC * PLANE;                 // one dZ tile (one copy)
    // bytes the A operand can reach past the start of the last ring slot: 16 planes
    // from its block's start (the mirrored ring: all blocks start in the first slot)
    static constexpr int RING_A = (NSLOT - 1) * SLICE + 16 * PLANE;
    static constexpr int RING_S = (MIRROR ? NSLOT + 2 : NSLOT) * SLICE;
    static constexpr int RING = RING_A > RING_S ? RING_A : RING_S;
    static constexpr size_t SMEM = (size_t)RING + (size_t)(3 * NC + NL) * COPY;
    static_assert(NACC * N3 <= 512 && N3 % 16 == 0 && N3 <= 256 && (CIN == 8 || CIN == 32) &&
                      (COUT == 8 || COUT == 32), "shape");
};



// Instruction descriptor with both operands MN-major (bits 15 and 16).
__host__ __device__ constexpr uint32_t idesc_bf16_mn(int m, int n) {
    return idesc_bf16(m, n) | (1u << 15) | (1u << 16);
}

template <int CIN, int COUT>
__global__ void __launch_bounds__(WTHREADS, 1)
    wgrad_tc_kernel(const __grid_constant__ CUtensorMap xmap, const __grid_constant__ CUtensorMap dmap,
                    const WgradTcArgs a) {
    using S = WgradShape<CIN, COUT>;
    constexpr int KC = S::KC, NMB = S::NMB, N3 = S::N3, NACC = S::NACC, NSLOT = S::NSLOT;
    constexpr int ROW = S::ROW, SLICE = S::SLICE, NL = S::NL, NC = S::NC, DKC = S::DKC;
    constexpr int COPY = S::COPY;
    constexpr uint32_t SLICE_TX = 3 * KC * PLANE;
    constexpr uint32_t DZ_TX = DKC * PLANE;
    extern __shared__ __align__(1024) unsigned char smem[];
    // lfull: a dZ tile landed; lempty: its copies are taken; cready: a copy set is
    // written; cempty: the MMAs reading a copy set are done
    __shared__ uint64_t full[NSLOT], empty[NSLOT], lfull[NL], lempty[NL], cready[NC], cempty[NC], done;
    __shared__ uint32_t tmem_base;
    unsigned char *Ss = smem;
    unsigned char *Cs = smem + S::RING;             // copy sets, 3 COPY each
    unsigned char *Ls = Cs + 3 * NC * COPY;         // landed tiles
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int segs = (a.nx + TM - 1) / TM;
    const long long nseg = (long long)((a.nz + a.zc - 1) / a.zc) * a.ny * segs;
    ConvTcArgs ga;  // the fields segment_of reads
    ga.nx = a.nx;
    ga.ny = a.ny;
    ga.nz = a.nz;
    ga.zc = a.zc;

    if (warp == 0) tmem_alloc(&tmem_base, S::TCOLS);
    if (threadIdx.x == 256) {
        for (int b = 0; b < NSLOT; ++b) {
            mbar_init(&full[b], 1);
            mbar_init(&empty[b], 1);
        }
        for (int b = 0; b < NL; ++b) {
            mbar_init(&lfull[b], 1);
            mbar_init(&lempty[b], 4);
        }
        for (int b = 0; b < NC; ++b) {
            mbar_init(&cready[b], 4);
            mbar_init(&cempty[b], 1);
        }
        mbar_init(&done, 1);
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    // the ring bytes past the slots are only read into discarded rows: keep them finite
    for (int i = S::RING_S + 16 * (int)threadIdx.x; i < S::RING; i += 16 * WTHREADS)
        *reinterpret_cast<uint4 *>(Ss + i) = make_uint4(0, 0, 0, 0);
    fence_proxy_async_smem();
    __syncthreads();  // barriers initialised, TMEM address published
    tc_fence_after_sync();
    const uint32_t tmem = tmem_base;
    if (warp < 4) {
        for (int k = 0; k < NACC * N3 / 16; ++k)
            tmem_zero<16>(tmem + ((uint32_t)(warp * 32) << 16) + k * 16);
        tc_fence_before_sync();
    }
    __syncthreads();
    tc_fence_after_sync();

    if (warp == 8) {
        if (lane == 0) {  // ---- TMA producer: slices 0, 1, then (slice i + 2, dZ tile i)
            int b = 0, l = 0;         // slot of the next slice, buffer of the next dZ tile
            unsigned round = 0, lround = 0;  // completed passes over the slots, the buffers
            bool ok = true;
            auto slice = [&](const Segment &sg, int j) {
                if (round > 0 && !mbar_wait(&empty[b], (round - 1) & 1)) return false;
                const int copies = S::MIRROR && b < 2 ? 2 : 1;
                mbar_expect_tx(&full[b], copies * SLICE_TX);
                const int z = wrapi(sg.z0 + j - 1, a.nz);
                for (int c = 0; c < copies; ++c) {
                    unsigned char *dst = Ss + (b + c * NSLOT) * SLICE;
#pragma unroll
                    for (int r = 0; r < 3; ++r)
                        tma_load_5d(dst + r * ROW, &xmap, &full[b], 0, sg.seg * (TM / 8), 0,
                                    wrapi(sg.y + r - 1, a.ny), z);
                }
                if (++b == NSLOT) {
                    b = 0;
                    ++round;
                }
                return true;
            };
            for (long long g = blockIdx.x; g < nseg && ok; g += gridDim.x) {
                const Segment sg = segment_of(g, ga, segs);
                ok = slice(sg, 0) && slice(sg, 1);
                for (int i = 0; i < sg.len && ok; ++i) {
                    ok = slice(sg, i + 2);
                    if (!ok) break;
                    if (lround > 0 && !mbar_wait(&lempty[l], (lround - 1) & 1)) {
                        ok = false;
                        break;
                    }
                    mbar_expect_tx(&lfull[l], DZ_TX);
                    // landed row r = slot x0 + r, cell x0 + r - 1
                    tma_load_5d(Ls + l * COPY, &dmap, &lfull[l], 0, sg.seg * (TM / 8), 0, sg.y,
                                sg.z0 + i);
                    if (++l == NL) {
                        l = 0;
                        ++lround;
                    }
                }
            }
            if (!ok) atomicExch(a.err, 1u);
            // no copy may be in flight when the CTA exits: wait for each buffer's last fill
            for (int q = 0; q < NSLOT; ++q) {
                const unsigned fills = round + (q < b);
                if (fills) mbar_wait(&full[q], (fills - 1) & 1);
            }
            for (int q = 0; q < NL; ++q) {
                const unsigned fills = lround + (q < l);
                if (fills) mbar_wait(&lfull[q], (fills - 1) & 1);
            }
        }
    } else if (warp == 9) {
        // ---- MMA issuer: the whole warp runs the loop, one elected lane issues
        int b = 0, c = 0;             // slot of the run's first slice, copy set of the tile
        unsigned fill = 0, cfill = 0;  // parities of their fills
        bool ok = true;
        const uint32_t idesc = idesc_bf16_mn(TM, N3);
        for (long long g = blockIdx.x; g < nseg && ok; g += gridDim.x) {
            const Segment sg = segment_of(g, ga, segs);
            const int L = sg.len;
            const int valid = a.nx - sg.seg * TM;
            const int nks = valid >= TM ? TM / 16 : (valid + 15) / 16;  // K-steps with cells < nx
            for (int i = 0; i < L; ++i) {
                // the run's three slices have landed (the first two were waited for by the
                // previous tile of the segment, or are waited now); the tile's copies are ready
                int slot[3];
                bool here = true;
#pragma unroll
                for (int q = 0; q < 3; ++q) {
                    slot[q] = b + q < NSLOT ? b + q : b + q - NSLOT;
                    if (i == 0 || q == 2)
                        here = mbar_wait(&full[slot[q]], b + q < NSLOT ? fill : fill ^ 1u) && here;
                }
                here = mbar_wait(&cready[c], cfill) && here;
                ok = __all_sync(0xffffffffu, here);
                if (!ok) break;
                tc_fence_after_sync();
                // A: the tile's cells x0 + k are staged rows k + 1 of every plane of the run;
                // block mb starts at plane 0 of the run's (mb)-th slice
                uint64_t a0[NMB];
#pragma unroll
                for (int mb = 0; mb < NMB; ++mb)  // block mb: the run's slice mb, in its own slot
                    a0[mb] = smem_desc(smem_u32(Ss + slot[mb] * SLICE) + 16, CORE, PLANE);
                const uint64_t b0 = smem_desc(smem_u32(Cs + c * 3 * COPY), CORE, PLANE);
                for (int ks = 0; ks < nks; ++ks) {
                    const uint64_t step = (uint32_t)(ks * 256) >> 4;
#pragma unroll
                    for (int mb = 0; mb < NMB; ++mb)
                        mma_bf16_elect(tmem + (uint32_t)(mb * N3), a0[mb] + step, b0 + step, idesc);
                }
                mma_commit_elect(&cempty[c]);
                mma_commit_elect(&empty[slot[0]]);  // the run's first slice serves no later tile
                if (i == L - 1) {
                    mma_commit_elect(&empty[slot[1]]);
                    mma_commit_elect(&empty[slot[2]]);
                }
                b += i == L - 1 ? 3 : 1;
                if (b >= NSLOT) {
                    b -= NSLOT;
                    fill ^= 1u;
                }
                if (++c == NC) {
                    c = 0;
                    cfill ^= 1u;
                }
            }
        }
        if (!ok && lane == 0) atomicExch(a.err, 1u);
        mma_commit_elect(&done);  // every MMA of the CTA, before the epilogue reads TMEM
    } else {  // ---- warps 0-7: the dZ tiles' shifted copies, then TMEM lanes 32 quad ..
        // Two sets of four warps, each with its own landed tile and copy set, so that one
        // tile's waits and fence overlap the other's copies (128^3, with 8 input channels:
        // 98 -> 92 us; with 32, where the MMAs' operands bound it: 116 -> 115, 135 -> 134).
        const int tid = threadIdx.x & 127, set = warp >> 2, quad = warp & 3;
        bool ok = true;
        static_assert(NL == 2 && NC == 2, "a landed tile and a copy set for each set of warps");
        const int c = set;
        int turn = 0;        // set whose turn the next tile is
        unsigned round = 0;  // tiles this set has copied
        for (long long g = blockIdx.x; g < nseg && ok; g += gridDim.x) {
            const Segment sg = segment_of(g, ga, segs);
            const int valid = a.nx - sg.seg * TM;  // rows r < valid are cells < nx
            for (int i = 0; i < sg.len; ++i) {
                turn ^= 1;
                if (turn == set) continue;  // (set 0 takes the first)
                bool here = mbar_wait(&lfull[c], round & 1);
                if (round > 0)  // the MMAs that read this copy set last are done
                    here = mbar_wait(&cempty[c], (round - 1) & 1) && here;
                ok = __all_sync(0xffffffffu, here);
                if (!ok) break;
                unsigned char *base = Cs + c * 3 * COPY;  // copy kx at base + kx * COPY
                const unsigned char *landed = Ls + c * COPY;
                // copy kx, row r = landed row r + 2 - kx (cell x0 + r + 1 - kx); rows of
                // cells past nx (r >= valid) zero.  Each landed row is read once: row tid
                // of each plane, then the two rows past the tile.
                auto spread = [&](int pl, int row) {
                    const uint4 v = reinterpret_cast<const uint4 *>(landed + pl * PLANE)[row];
                    const uint4 z = make_uint4(0, 0, 0, 0);
#pragma unroll
                    for (int k = 0; k < 3; ++k) {
                        const int r = row - k;  // copy 2 - k
                        if (r >= 0 && r < TM)
                            reinterpret_cast<uint4 *>(base + (2 - k) * COPY + pl * PLANE)[r] =
                                r < valid ? v : z;
                    }
                };
#pragma unroll
                for (int pl = 0; pl < DKC; ++pl) spread(pl, tid);
                if (tid < 2 * DKC) spread(tid >> 1, TM + (tid & 1));
                // generic reads of the landed tile before the TMA refills it, generic
                // writes of the copies before the tensor core reads them
                fence_proxy_async_smem();
                __syncwarp();
                if (lane == 0) {
                    mbar_arrive(&lempty[c]);
                    mbar_arrive(&cready[c]);
                }
                ++round;
            }
        }
        if (ok) ok = __all_sync(0xffffffffu, mbar_wait(&done, 0));
        tc_fence_after_sync();
        if (ok) {
            const int m = quad * 32 + lane;
            constexpr int CH = N3 % 32 == 0 ? 32 : 16;
#pragma unroll 1
            for (int k = 0; k < NACC; ++k)
#pragma unroll 1
                for (int c0 = set * CH; c0 < N3; c0 += 2 * CH) {
                    const uint32_t taddr =
                        tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)(k * N3 + c0);
                    float v[CH];
                    if constexpr (CH == 32)
                        tmem_ld32(taddr, v);
                    else
                        tmem_ld16(taddr, v);
                    float *dst = a.part + (((long long)blockIdx.x * NACC + k) * N3 + c0) * TM + m;
#pragma unroll
                    for (int n = 0; n < CH; ++n) dst[n * TM] = v[n];
                }
        } else if (lane == 0) {
            atomicExch(a.err, 1u);
        }
    }
    tc_fence_before_sync();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, S::TCOLS);
}

// gW[co][ci][kz][ky][kx] (ci < cin_real) from the per-CTA partials: one thread
// per partial entry (M block mb, column n = kx NB + co, row m), rows fastest so
// that the CTAs' blocks are read coalesced; entries that hold no gradient (padded
// columns, rows past a block's planes) are skipped.  Row m of block mb is plane
// P = mb BLK + m / 8 of the run, channel 8 (P % KC) + m % 8, tap row P / KC = 3 kz + ky.
// Binary64 sums, RSPLIT runs of CTAs at once, added in order: one chain of 152 additions
// took 23 us at any layer's size, eight take 13 us with 128 x 48 and 128 x 96 entries
// and 27 us with 3 x 128 x 96, where the FP64 pipe bounds them.
constexpr int RSPLIT = 8, RENTRIES = 32;

template <int CIN, int COUT>
__global__ void __launch_bounds__(RSPLIT * RENTRIES)
    wgrad_tc_reduce_kernel(const float *__restrict__ part, int ctas, int cin_real, float *__restrict__ gW) {
    using S = WgradShape<CIN, COUT>;
    constexpr int PER_CTA = S::NACC * S::N3 * TM;
    static_assert(PER_CTA % RENTRIES == 0, "whole blocks");
    __shared__ double sh[RSPLIT][RENTRIES];
    const int e = threadIdx.x % RENTRIES, run = threadIdx.x / RENTRIES;
    const int t = blockIdx.x * RENTRIES + e;
    const int m = t % TM, n = (t / TM) % S::N3, mb = t / (TM * S::N3);
    const int kx = n / S::NB, co = n % S::NB;
    const int P = mb * S::BLK + m / 8;
    const int ci = 8 * (P % S::KC) + m % 8;
    const bool live = co < COUT && P < S::NPL && (S::BLK == 0 || m / 8 < S::BLK) && ci < cin_real;
    const int chunk = (ctas + RSPLIT - 1) / RSPLIT;
    double s = 0.0;
    if (live)
        for (int b = run * chunk; b < min(ctas, (run + 1) * chunk); ++b)
            s += part[(long long)b * PER_CTA + t];
    sh[run][e] = s;
    __syncthreads();
    if (run == 0 && live) {
        for (int q = 1; q < RSPLIT; ++q) s += sh[q][e];
        gW[(co * cin_real + ci) * 27 + (P / S::KC) * 3 + kx] = (float)s;
    }
}

}  // namespace tc
}  // namespace ac
