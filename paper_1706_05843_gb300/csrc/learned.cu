// learned.cu -- kernels of the learned preconditioner: 3^4 convolutions as
// implicit GEMMs on the BF16 tensor cores (FP32 accumulate), their two
// backward passes, activation packing and Adam.
//
// Forward and backward-data (the same product with the mirrored, transposed
// weights): k_conv_tc, on the 5th-generation tensor cores (tcgen05.mma, the
// accumulator in tensor memory), described at the kernel.
// Backward-weights: k_conv_wgrad, mma.sync over the same staged segments.
#include "learned.h"

#include <algorithm>
#include <cstdint>

namespace eofa {

namespace {

__device__ __forceinline__ unsigned smem_u32(const void* p) {
    return (unsigned)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void cp_async16(void* sdst, const void* gsrc) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(smem_u32(sdst)), "l"(gsrc));
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;\n" ::); }
template <int N>
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N)); }

__device__ __forceinline__ void ldsm_x4_t(unsigned* r, const void* p) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(smem_u32(p)));
}
__device__ __forceinline__ void mma16816(float* d, const unsigned* a, unsigned b0, unsigned b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};\n"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// element offset of 16-byte chunk c of row r in a [rows][32] BF16 tile
__device__ __forceinline__ int swz(int r, int c) { return r * 32 + ((c ^ ((r >> 1) & 3)) << 3); }

__device__ __forceinline__ int wrapi(int v, int n) { return v < 0 ? v + n : (v >= n ? v - n : v); }
enum Epi { EPI_LEAKY_BF16 = 0, EPI_F32 = 1, EPI_DMASK_BF16 = 2 };

// ---------------------------------------------------------------------------
// The convolution on the 5th-generation tensor cores (tcgen05).
//
// A CTA keeps all 81 weight blocks in shared memory (166 KB) and walks
// columns: 128 rows of one slice's (z, y, x) volume over a range of t.  The
// volume is numbered with a halo, [z][Y + 2][x + 2], so that every spatial
// tap is a constant offset in that numbering: a time slice's rows for one dz
// (a segment: 128 + 2 (line + 1) positions) are loaded once, in the canonical
// no-swizzle K-major layout with 16-byte rows, and the nine (dy, dx) taps
// read it through matrix descriptors that start at other rows.  Rows of the
// halo are computed and dropped.
//
// One input slice t' serves the outputs t' - 1, t', t' + 1 (dt = 1, 0, -1) in
// one M128 x N96 x K16 MMA: the accumulators of consecutive outputs are
// consecutive 32-column slots of tensor memory, a ring of 16.  Walking t'
// upwards keeps every output's sum in the order of the taps (dt, dz, dy, dx),
// K16 halves innermost.  A slot is read out (tcgen05.ld), zeroed and given
// back by the epilogue warps while the MMAs of the next slices run.
//
// Roles: warps 0-3 epilogue (one TMEM lane a thread), warp 4 one thread
// issues the MMAs, warps 5-7 load segments (cp.async) through a ring.  Every
// mbarrier wait is bounded; on expiry the CTA records the event in
// g_tc_fault, every role leaves its loop, the copies and MMAs in flight are
// waited for and the tensor memory is freed.
//
// What bounds it: shared-memory reads of the operands (4 KB of A and 3 KB of B
// an MMA beside the segments' own 10 KB per 18 MMAs): 93 clocks an MMA measured,
// 19% of them spent waiting for a segment, against 48 clocks of tensor work;
// tensor pipe 44%.  Lines without a halo and a copy of each segment per dx, so
// that every A view starts at a 128-byte line, took 1.65 against 1.68 ms for the
// network at 16^3 x 32 and 0.56 against 0.54 ms at 40 x 8 x 8 x 16: the
// alignment of the views is not what costs.  16^3 x 32, 16 slices:
// 0.417 ms a layer, 2.2 ms for the kernel it replaces, which gathered the 128
// neighbour rows of every tap through L1 (97% of its peak, tensor pipe 7%).
// ---------------------------------------------------------------------------
__device__ int g_tc_fault;  // set when a bounded wait of the tcgen05 convolution expired

constexpr int kCvRows = 128;                 // output positions of a tile (MMA M)
constexpr int kCvSlots = 16;                 // accumulator slots of 32 columns
constexpr int kCvWBytes = 81 * 32 * 32 * 2;  // the packed weights
constexpr int kCvTapBytes = 96 * 32 * 2;     // one spatial tap: [q = ci / 8][n = 96][8]
constexpr int kCvThreads = 256;
constexpr int kCvLoaders = 96;
constexpr int kCvMaxSeg = 6;
constexpr int kCvBarBytes = (2 * kCvMaxSeg + 2 * kCvSlots + 2) * 8;
constexpr int kCvSmemMax = 232448;
constexpr long kTcSpin = 1L << 22;           // mbarrier polls before a wait counts as expired

// shared-memory matrix descriptor of a canonical K-major tile without
// swizzle: start and the stride between core matrices along K (lbo) in the
// low word, 128 bytes between 8-row groups and descriptor version 1 in the
// high word.  Adding n to the low word moves the start by 16 n bytes.
__device__ __forceinline__ unsigned tc_desc_lo(unsigned saddr, unsigned lbo) {
    return ((saddr >> 4) & 0x3FFF) | ((lbo >> 4) << 16);
}
__device__ __forceinline__ unsigned long long tc_desc(unsigned lo) {
    return ((unsigned long long)((128u >> 4) | (1u << 14)) << 32) | lo;
}
// instruction descriptor: D FP32, A and B BF16, both K-major, M = 128
__device__ __forceinline__ unsigned tc_idesc(unsigned n) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((n >> 3) << 17) | ((128u >> 4) << 24);
}
__device__ __forceinline__ void tc_mma(unsigned d, unsigned a_lo, unsigned b_lo, unsigned idesc) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, 1, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d),
        "l"(tc_desc(a_lo)), "l"(tc_desc(b_lo)), "r"(idesc)
        : "memory");
}
__device__ __forceinline__ void tc_commit(unsigned bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_init(unsigned a, unsigned n) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(a), "r"(n) : "memory");
}
__device__ __forceinline__ void mbar_arrive(unsigned a) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(a) : "memory");
}
// true when the phase of the given parity has completed; gives up after
// kTcSpin polls (setting *fault) or when another role has
__device__ __forceinline__ bool mbar_wait(unsigned a, unsigned parity, volatile int* fault) {
    for (long i = 0; i < kTcSpin; ++i) {
        unsigned done;
        asm volatile(
            "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(done)
            : "r"(a), "r"(parity)
            : "memory");
        if (done) return true;
        if ((i & 63) == 63 && *fault) return false;
    }
    *fault = 1;
    return false;
}

// how the lattice is cut into columns (host; the same for every layer)
struct ConvPlan {
    int nxb, wb;      // blocks in x and their width
    int line, plane;  // positions of a haloed line (wb + 2) and plane ((Y + 2) line)
    int vol;          // positions of one block's volume
    int tiles;        // 128-position tiles of it
    int nt, nts;      // outputs of a column along t, columns along t
    int np, nseg;     // positions of a segment, ring of segments
    long cols;
};

template <int EPI>
__global__ void __launch_bounds__(kCvThreads, 1)
    k_conv_tc(const bf16* __restrict__ in, const bf16* __restrict__ W, void* __restrict__ out,
              const bf16* __restrict__ mask, ConvGeom g, ConvPlan pl, int ostride) {
    extern __shared__ __align__(128) unsigned char tc_smem[];
    unsigned char* sW = tc_smem;                      // [27][4][96][16 bytes]
    unsigned char* sA = tc_smem + kCvWBytes;          // [nseg][4][np][16 bytes]
    int2* tab = reinterpret_cast<int2*>(sA + (size_t)pl.nseg * pl.np * 64);  // [np]: (y X + x, z) of a position
    unsigned long long* bars = reinterpret_cast<unsigned long long*>(tab + pl.np);
    const unsigned b_full = smem_u32(bars), b_empty = b_full + 8 * kCvMaxSeg;
    const unsigned b_accf = b_empty + 8 * kCvMaxSeg, b_acce = b_accf + 8 * kCvSlots, b_fin = b_acce + 8 * kCvSlots;
    __shared__ unsigned s_tmem;
    __shared__ volatile int s_fault;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

    if (tid == 0) {
        s_fault = 0;
        for (int i = 0; i < pl.nseg; ++i) {
            mbar_init(b_full + 8 * i, kCvLoaders);
            mbar_init(b_empty + 8 * i, 1);
        }
        for (int i = 0; i < kCvSlots; ++i) {
            mbar_init(b_accf + 8 * i, 1);
            mbar_init(b_acce + 8 * i, kCvRows);
        }
        mbar_init(b_fin, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(&s_tmem))
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    for (int i = tid; i < kCvWBytes / 16; i += kCvThreads) cp_async16(sW + 16 * i, W + 8 * i);
    cp_commit();
    cp_wait<0>();
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const unsigned tmem = s_tmem;

    // column -> (slice, x block, tile, first output t, outputs)
    struct Col {
        int sl, xb, p0, t0, nt;
    };
    auto column = [&](long c) {
        Col k;
        k.t0 = (int)(c % pl.nts) * pl.nt;
        c /= pl.nts;
        k.p0 = (int)(c % pl.tiles) * kCvRows;
        c /= pl.tiles;
        k.xb = (int)(c % pl.nxb);
        k.sl = (int)(c / pl.nxb);
        k.nt = min(pl.nt, g.T - k.t0);
        return k;
    };
    auto zero_slot = [&](unsigned taddr) {
        const unsigned z = 0u;
        asm volatile(
            "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, "
            "%1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1};" ::"r"(taddr),
            "r"(z)
            : "memory");
        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
    };

    if (warp < 4) {
        // ------------------------------------------------ epilogue
        const unsigned tlane = tmem + ((unsigned)(warp * 32) << 16);
        for (int i = 0; i < kCvSlots; ++i) {
            zero_slot(tlane + 32 * i);
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            mbar_arrive(b_acce + 8 * i);
        }
        long o = 0;
        bool ok = true;
        for (long cc = blockIdx.x; cc < pl.cols && ok; cc += gridDim.x) {
            const Col k = column(cc);
            const int p = k.p0 + tid;
            const int z = p / pl.plane, r = p - z * pl.plane, yp = r / pl.line, xp = r - yp * pl.line;
            const int x = k.xb * pl.wb + xp - 1;
            const bool valid = p < pl.vol && yp >= 1 && yp <= g.Y && xp >= 1 && xp <= pl.wb && x < g.X;
            const long site0 = (long)k.sl * g.V + ((long)z * g.Y + (yp - 1)) * g.X + x;
            for (int i = 0; i < k.nt; ++i, ++o) {
                const int slot = (int)(o % kCvSlots);
                ok = __all_sync(0xffffffffu, mbar_wait(b_accf + 8 * slot, (unsigned)(o / kCvSlots) & 1, &s_fault));
                if (!ok) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                unsigned r32[32];
                asm volatile(
                    "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, "
                    "%14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
                    : "=r"(r32[0]), "=r"(r32[1]), "=r"(r32[2]), "=r"(r32[3]), "=r"(r32[4]), "=r"(r32[5]),
                      "=r"(r32[6]), "=r"(r32[7]), "=r"(r32[8]), "=r"(r32[9]), "=r"(r32[10]), "=r"(r32[11]),
                      "=r"(r32[12]), "=r"(r32[13]), "=r"(r32[14]), "=r"(r32[15]), "=r"(r32[16]), "=r"(r32[17]),
                      "=r"(r32[18]), "=r"(r32[19]), "=r"(r32[20]), "=r"(r32[21]), "=r"(r32[22]), "=r"(r32[23]),
                      "=r"(r32[24]), "=r"(r32[25]), "=r"(r32[26]), "=r"(r32[27]), "=r"(r32[28]), "=r"(r32[29]),
                      "=r"(r32[30]), "=r"(r32[31])
                    : "r"(tlane + 32 * slot));
                asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                zero_slot(tlane + 32 * slot);
                asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                mbar_arrive(b_acce + 8 * slot);
                if (!valid) continue;
                const long gi = site0 + (long)(k.t0 + i) * g.Z * g.Y * g.X;
                if constexpr (EPI == EPI_F32) {
                    // ostride 24 or 32; negative: rows that are not 16-byte aligned
                    const int os = abs(ostride);
                    float* row = reinterpret_cast<float*>(out) + gi * os;
                    if (ostride < 0) {
#pragma unroll
                        for (int e = 0; e < 32; ++e)
                            if (e < os) row[e] = __uint_as_float(r32[e]);
                        continue;
                    }
                    float4* dst = reinterpret_cast<float4*>(row);
#pragma unroll
                    for (int q = 0; q < 8; ++q)
                        if (4 * q < os)
                            dst[q] = make_float4(__uint_as_float(r32[4 * q]), __uint_as_float(r32[4 * q + 1]),
                                                 __uint_as_float(r32[4 * q + 2]), __uint_as_float(r32[4 * q + 3]));
                } else {
                    uint4* dst = reinterpret_cast<uint4*>(reinterpret_cast<bf16*>(out) + gi * kCP);
                    const uint4* mk = reinterpret_cast<const uint4*>(mask + gi * kCP);
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        uint4 mq = make_uint4(0u, 0u, 0u, 0u);
                        if constexpr (EPI == EPI_DMASK_BF16) mq = mk[q];
                        const unsigned* mw = reinterpret_cast<const unsigned*>(&mq);
                        unsigned w[4];
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            float v0 = __uint_as_float(r32[8 * q + 2 * e]), v1 = __uint_as_float(r32[8 * q + 2 * e + 1]);
                            if constexpr (EPI == EPI_LEAKY_BF16) {
                                v0 = v0 > 0.f ? v0 : kLeaky * v0;
                                v1 = v1 > 0.f ? v1 : kLeaky * v1;
                            } else {
                                const __nv_bfloat162 m = *reinterpret_cast<const __nv_bfloat162*>(&mw[e]);
                                v0 *= __bfloat162float(m.x) > 0.f ? 1.f : kLeaky;
                                v1 *= __bfloat162float(m.y) > 0.f ? 1.f : kLeaky;
                            }
                            const __nv_bfloat162 b = __floats2bfloat162_rn(v0, v1);
                            w[e] = *reinterpret_cast<const unsigned*>(&b);
                        }
                        dst[q] = make_uint4(w[0], w[1], w[2], w[3]);
                    }
                }
            }
        }
    } else if (warp == 4) {
        // ------------------------------------------------ MMA issue
        if (lane == 0) {
            const unsigned hA = 2 * (unsigned)pl.np, hB = 2 * 96;  // 16-byte units between the K16 halves
            const unsigned line = (unsigned)pl.line;
            const unsigned w0 = tc_desc_lo(smem_u32(sW), 96 * 16);
            unsigned o = 0;           // outputs of the columns before this one
            unsigned slot = 0, par = 0;  // segment ring
            bool ok = true;
            for (long cc = blockIdx.x; cc < pl.cols && ok; cc += gridDim.x) {
                const int nt = column(cc).nt;
                for (int i = 0; i < nt + 2 && ok; ++i) {  // input slice t0 - 1 + i serves outputs i - 2, i - 1, i
                    const int lo = max(0, i - 2), hi = min(nt - 1, i);
                    if (i < nt) {
                        const unsigned q = o + (unsigned)i;  // the output this slice starts
                        if (!mbar_wait(b_acce + 8 * (q % kCvSlots), (q / kCvSlots) & 1, &s_fault)) {
                            ok = false;
                            break;
                        }
                        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    }
                    const unsigned s0 = (o + (unsigned)lo) % kCvSlots, n = (unsigned)(hi - lo + 1);
                    const unsigned n1 = min(n, kCvSlots - s0), n2 = n - n1;  // n2: the part that wraps to slot 0
                    const unsigned wlo = w0 + (unsigned)(lo - (i - 2)) * 32;
                    const unsigned d = tmem + 32 * s0, id1 = tc_idesc(32 * n1), id2 = tc_idesc(32 * n2);
                    for (int dz = 0; dz < 3; ++dz) {
                        if (!mbar_wait(b_full + 8 * slot, par, &s_fault)) {
                            ok = false;
                            break;
                        }
                        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                        const unsigned as = tc_desc_lo(smem_u32(sA) + slot * (unsigned)pl.np * 64, (unsigned)pl.np * 16);
                        const unsigned ws = wlo + (unsigned)dz * 9 * (kCvTapBytes / 16);
                        if (n2 == 0) {
#pragma unroll
                            for (unsigned tp = 0; tp < 9; ++tp) {
                                const unsigned at = as + (tp / 3) * line + tp % 3, wt = ws + tp * (kCvTapBytes / 16);
                                tc_mma(d, at, wt, id1);
                                tc_mma(d, at + hA, wt + hB, id1);
                            }
                        } else {
#pragma unroll 1
                            for (unsigned tp = 0; tp < 9; ++tp) {
                                const unsigned at = as + (tp / 3) * line + tp % 3, wt = ws + tp * (kCvTapBytes / 16);
                                tc_mma(d, at, wt, id1);
                                tc_mma(tmem, at, wt + n1 * 32, id2);
                                tc_mma(d, at + hA, wt + hB, id1);
                                tc_mma(tmem, at + hA, wt + hB + n1 * 32, id2);
                            }
                        }
                        tc_commit(b_empty + 8 * slot);
                        if (++slot == (unsigned)pl.nseg) slot = 0, par ^= 1;
                    }
                    if (ok && i >= 2) tc_commit(b_accf + 8 * ((o + (unsigned)i - 2) % kCvSlots));
                }
                o += (unsigned)nt;
            }
            // every MMA issued has completed before the tensor memory is freed
            volatile int none = 0;
            tc_commit(b_fin);
            mbar_wait(b_fin, 0, &none);
        }
        __syncwarp();
    } else {
        // ------------------------------------------------ segment loads
        // a warp loads a third of the positions; four lanes a position
        const int part = (pl.np + 2) / 3, lo = (warp - 5) * part, hi = min(pl.np, lo + part);
        int slot = 0, par = 1;  // the first round finds the ring empty
        int pend = -1;          // slot whose copies have not been published yet
        bool ok = true;
        for (long cc = blockIdx.x; cc < pl.cols && ok; cc += gridDim.x) {
            const Col c = column(cc);
            __syncwarp();
            for (int pos = lo + lane; pos < hi; pos += 32) {
                // positions outside the volume feed dropped rows only
                const int p = min(max(c.p0 - pl.line - 1 + pos, 0), pl.vol - 1);
                const int z = p / pl.plane, r = p - z * pl.plane, yp = r / pl.line;
                const int y = wrapi(yp - 1, g.Y), x = wrapi(c.xb * pl.wb + (r - yp * pl.line) - 1, g.X);
                tab[pos] = make_int2(y * g.X + x, z);
            }
            __syncwarp();
            for (int i = 0; i < c.nt + 2 && ok; ++i) {
                int t = c.t0 - 1 + i;
                t = t < 0 ? t + g.T : (t >= g.T ? t - g.T : t);
                const bf16* base = in + ((long)c.sl * g.V + (long)t * g.Z * g.Y * g.X) * kCP + 8 * (lane & 3);
                for (int dz = -1; dz <= 1; ++dz) {
                    ok = __all_sync(0xffffffffu, mbar_wait(b_empty + 8 * slot, (unsigned)par, &s_fault));
                    if (!ok) break;
                    unsigned char* dst = sA + ((size_t)slot * 4 + (lane & 3)) * pl.np * 16;
                    for (int pos = lo + (lane >> 2); pos < hi; pos += 8) {
                        const int2 e = tab[pos];
                        const long n = (long)wrapi(e.y + dz, g.Z) * g.Y * g.X + e.x;
                        cp_async16(dst + pos * 16, base + n * kCP);
                    }
                    cp_commit();
                    if (pend >= 0) {  // the previous segment has arrived
                        cp_wait<1>();
                        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                        mbar_arrive(b_full + 8 * pend);
                    }
                    pend = slot;
                    if (++slot == pl.nseg) slot = 0, par ^= 1;
                }
            }
        }
        cp_wait<0>();
        if (ok && pend >= 0) {
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            mbar_arrive(b_full + 8 * pend);
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (tid == 0 && s_fault) atomicExch(&g_tc_fault, 1);
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem) : "memory");
}

// ---------------------------------------------------------------------------
// Weight gradient: dW[tap][co][ci] += sum_rows dy[row][co] in[shift(row, tap)][ci],
// the same haloed numbering and segments as the convolution.  A CTA belongs to
// one dt and takes an equal share of the (column, t) steps; a step holds the
// 128 rows of dy (zero in the halo) and the three dz segments of in at t + dt
// in shared memory, and its 18 warps, two per (dz, dy) with 16 input channels
// each, form the three dx taps with mma.sync, rows along K.  Every element loaded serves nine taps
// (before: one, each tap re-reading both fields through L1; 16^3 x 32, 8
// slices: 1.6 -> 0.82 ms a layer).  Sums: 64
// k16 products in the tensor cores, then FP32 registers over the CTA's share,
// one atomic per element and CTA.  Bound by the rate of mma.sync, the
// instruction chosen (math pipe throttle leads the stalls, tensor pipe 46%; nine
// warps of 32 channels: 0.93 ms).
// The zero rows of dy would turn an Inf of in into NaN: a CTA whose sums are
// not all finite leaves them to a second launch for all layers (MASKED), in which
// the halo's rows of in are zero as well and the other CTAs return at once (masked
// in every pass: the network's gradients at 16^3 x 32, 8 slices 4.31 -> 4.81 ms; a
// second walk in the same kernel 4.27 -> 4.37 ms, for its registers; this form
// 4.27 -> 4.22 ms, and 435 -> 440 us at 4^4, one slice).
// ---------------------------------------------------------------------------
constexpr int kWgThreads = 576;
constexpr int kWgStages = 3;
constexpr int kWgFlush = 8;  // steps (of 8 k16 products) between sums into the FP32 registers

struct WgLayer {
    const bf16* in;
    const bf16* dy;
    float* dW;
    int* redo;  // a flag for each CTA
    int cout, cin;
};
struct WgLayers {
    WgLayer l[kNetLayers];
};

// MASKED: blockIdx.y numbers the layers, otherwise layer 0 alone
template <bool MASKED>
__global__ void __launch_bounds__(kWgThreads, 1)
    k_conv_wgrad(const __grid_constant__ WgLayers layers, ConvGeom g, ConvPlan pl) {
    const WgLayer& L = layers.l[MASKED ? blockIdx.y : 0];
    if (MASKED && !L.redo[blockIdx.x]) return;
    const bf16* __restrict__ in = L.in;
    const bf16* __restrict__ dy = L.dy;
    float* __restrict__ dW = L.dW;
    const int cout = L.cout, cin = L.cin;
    extern __shared__ __align__(128) unsigned char wg_smem[];
    const int stage_elems = (kCvRows + 3 * pl.np) * 32;
    bf16* st0 = reinterpret_cast<bf16*>(wg_smem);                                   // [stages][dy | in dz 0..2]
    int2* tab = reinterpret_cast<int2*>(st0 + (size_t)kWgStages * stage_elems);     // [np]: (y X + x, z or -1 - z)
    __shared__ unsigned s_rows[kWgStages][kCvRows / 32];                            // a bit for each row of the lattice
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int dt = blockIdx.x % 3 - 1, rank = blockIdx.x / 3, ranks = gridDim.x / 3;
    const long steps = (long)g.S * pl.nxb * pl.tiles * g.T;
    const long s0 = steps * rank / ranks, s1 = steps * (rank + 1) / ranks;
    const long slice = (long)g.Z * g.Y * g.X;

    long tab_col = -1;
    auto issue = [&](long s, int buf) {
        const long col = s / g.T;
        const int t = (int)(s - col * g.T);
        const int tile = (int)(col % pl.tiles);
        const long c2 = col / pl.tiles;
        const int xb = (int)(c2 % pl.nxb), sl = (int)(c2 / pl.nxb);
        if (col != tab_col) {  // uniform over the CTA
            tab_col = col;
            for (int pos = tid; pos < pl.np; pos += kWgThreads) {
                const int q = tile * kCvRows - pl.line - 1 + pos;
                const int p = min(max(q, 0), pl.vol - 1);
                const int z = p / pl.plane, r = p - z * pl.plane, yp = r / pl.line, xp = r - yp * pl.line;
                const int xr = xb * pl.wb + xp - 1;
                const bool valid = q >= 0 && q < pl.vol && yp >= 1 && yp <= g.Y && xp >= 1 && xp <= pl.wb && xr < g.X;
                tab[pos] = make_int2(wrapi(yp - 1, g.Y) * g.X + wrapi(xr, g.X), valid ? z : -1 - z);
            }
            __syncthreads();
        }
        if (MASKED && tid < kCvRows) {
            const unsigned rows = __ballot_sync(0xffffffffu, tab[tid + pl.line + 1].y >= 0);
            if (lane == 0) s_rows[buf][warp] = rows;
        }
        bf16* sD = st0 + (size_t)buf * stage_elems;
        const int ti = wrapi(t + dt, g.T);
        const bf16* bd = dy + ((long)sl * g.V + t * slice) * kCP;
        const bf16* bi = in + ((long)sl * g.V + ti * slice) * kCP;
        for (int j = tid; j < 4 * kCvRows; j += kWgThreads) {
            const int r = j >> 2, q = j & 3;
            const int2 e = tab[r + pl.line + 1];
            bf16* dst = sD + swz(r, q);
            if (e.y >= 0) cp_async16(dst, bd + ((long)e.y * g.Y * g.X + e.x) * kCP + 8 * q);
            else *reinterpret_cast<uint4*>(dst) = make_uint4(0u, 0u, 0u, 0u);
        }
        for (int dz = 0; dz < 3; ++dz) {
            bf16* sI = sD + (kCvRows + dz * pl.np) * 32;
            for (int j = tid; j < 4 * pl.np; j += kWgThreads) {
                const int r = j >> 2, q = j & 3;
                const int2 e = tab[r];
                const int z = wrapi((e.y >= 0 ? e.y : -1 - e.y) + dz - 1, g.Z);
                cp_async16(sI + swz(r, q), bi + ((long)z * g.Y * g.X + e.x) * kCP + 8 * q);
            }
        }
    };

    float acc[3][2][2][4], sum[3][2][2][4];
#pragma unroll
    for (int i = 0; i < 48; ++i) (&acc[0][0][0][0])[i] = (&sum[0][0][0][0])[i] = 0.f;
    auto flush = [&]() {
#pragma unroll
        for (int i = 0; i < 48; ++i) {
            (&sum[0][0][0][0])[i] += (&acc[0][0][0][0])[i];
            (&acc[0][0][0][0])[i] = 0.f;
        }
    };

    const int dz = warp % 9 / 3, dyy = warp % 3, nh = warp / 9;
    const int i8 = lane >> 3;
    for (int i = 0; i < kWgStages - 1; ++i) {
        if (s0 + i < s1) issue(s0 + i, i);
        cp_commit();
        __syncthreads();  // the table may be rewritten by the next issue
    }
    int buf = 0;
    for (long s = s0; s < s1; ++s) {
        cp_wait<kWgStages - 2>();
        __syncthreads();  // this step's stage has arrived; the oldest stage and the table are free
        const long nx = s + kWgStages - 1;
        if (nx < s1) issue(nx, buf == 0 ? kWgStages - 1 : buf - 1);
        cp_commit();
        const bf16* D = st0 + (size_t)buf * stage_elems;
        const bf16* In = D + (kCvRows + dz * pl.np) * 32;
        const int off = dyy * pl.line;
#pragma unroll 2
        for (int kb = 0; kb < kCvRows / 16; ++kb) {
            unsigned af[2][4], bfr[3][4];
#pragma unroll
            for (int mt = 0; mt < 2; ++mt)   // A = dy^T: (co, k) from rows k, columns co
                ldsm_x4_t(af[mt], D + swz(kb * 16 + (lane & 7) + (i8 >> 1) * 8, mt * 2 + (i8 & 1)));
#pragma unroll
            for (int dx = 0; dx < 3; ++dx)   // B = in_shift: (k, ci) rows k
                ldsm_x4_t(bfr[dx], In + swz(off + dx + kb * 16 + (lane & 7) + (i8 & 1) * 8, nh * 2 + (i8 >> 1)));
            if constexpr (MASKED) {  // this lane's rows k: 2 (lane & 3) + 0, 1 and those + 8
                const unsigned rows = s_rows[buf][kb >> 1] >> ((kb & 1) * 16 + (lane & 3) * 2);
                const unsigned m0 = (rows & 1) * 0xffffu | (rows >> 1 & 1) * 0xffff0000u;
                const unsigned m1 = (rows >> 8 & 1) * 0xffffu | (rows >> 9 & 1) * 0xffff0000u;
#pragma unroll
                for (int i = 0; i < 12; ++i) bfr[i / 4][i % 4] &= i % 2 ? m1 : m0;
            }
#pragma unroll
            for (int dx = 0; dx < 3; ++dx)
#pragma unroll
                for (int mt = 0; mt < 2; ++mt)
#pragma unroll
                    for (int nt = 0; nt < 2; ++nt)
                        mma16816(acc[dx][mt][nt], af[mt], bfr[dx][nt * 2], bfr[dx][nt * 2 + 1]);
        }
        if ((s - s0) % kWgFlush == kWgFlush - 1) flush();
        buf = buf + 1 == kWgStages ? 0 : buf + 1;
    }
    cp_wait<0>();
    flush();
    if constexpr (!MASKED) {
        float nf = 0.f;
#pragma unroll
        for (int i = 0; i < 48; ++i) nf += 0.f * (&sum[0][0][0][0])[i];  // NaN from Inf or NaN
        const int bad = __syncthreads_or(nf != 0.f);
        if (tid == 0) L.redo[blockIdx.x] = bad;
        if (bad) return;
    }
    if (s0 == s1) return;
#pragma unroll
    for (int dx = 0; dx < 3; ++dx) {
        float* dst = dW + (long)((((dt + 1) * 3 + dz) * 3 + dyy) * 3 + dx) * cout * cin;
#pragma unroll
        for (int mt = 0; mt < 2; ++mt)
#pragma unroll
            for (int nt = 0; nt < 2; ++nt)
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const int co = mt * 16 + (lane >> 2) + (e >> 1) * 8;
                    const int ci = (nh * 2 + nt) * 8 + (lane & 3) * 2 + (e & 1);
                    if (co < cout && ci < cin) atomicAdd(dst + (long)co * cin + ci, sum[dx][mt][nt][e]);
                }
    }
}

// place of W[tap][co][ci] in the packed weights: per spatial tap [ci / 8][n][8]
// with n = 32 (1 - dt) + co, dt = -1, 0, 1 (the outputs of an input slice in
// ascending t)
__device__ __forceinline__ int packed_w(int tap, int co, int ci) {
    return (((tap % 27) * 4 + (ci >> 3)) * 96 + 32 * (2 - tap / 27) + co) * 8 + (ci & 7);
}

// public FP32 weights -> padded BF16 forward and mirrored/transposed backward operands
__global__ void k_convert(const float* __restrict__ Wm, bf16* __restrict__ Wf, bf16* __restrict__ Wb, int cout,
                          int cin) {
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= 81 * 32 * 32) return;
    const int tap = e / 1024, co = (e / 32) % 32, ci = e % 32;
    const float v = (co < cout && ci < cin) ? Wm[((long)tap * cout + co) * cin + ci] : 0.f;
    Wf[packed_w(tap, co, ci)] = __float2bfloat16(v);
    Wb[packed_w(80 - tap, ci, co)] = __float2bfloat16(v);
}

// rows of 24 floats -> rows of 32 BF16, zero padded: one thread makes a
// 16-byte piece (0.17 -> 0.05 ms for 2 M rows against one thread an element);
// vec: in24 is 16-byte aligned
__global__ void k_pack(const float* __restrict__ in24, bf16* __restrict__ a32, long rows, bool vec) {
    const long t = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= rows * 4) return;
    const int q = (int)(t & 3);
    uint4 v = make_uint4(0u, 0u, 0u, 0u);
    if (q < 3) {
        const float* src = in24 + (t >> 2) * 24 + 8 * q;
        float f[8];
        if (vec) {
            const float4 a = reinterpret_cast<const float4*>(src)[0], b = reinterpret_cast<const float4*>(src)[1];
            f[0] = a.x; f[1] = a.y; f[2] = a.z; f[3] = a.w;
            f[4] = b.x; f[5] = b.y; f[6] = b.z; f[7] = b.w;
        } else {
#pragma unroll
            for (int i = 0; i < 8; ++i) f[i] = src[i];
        }
        __nv_bfloat162 h[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) h[i] = __floats2bfloat162_rn(f[2 * i], f[2 * i + 1]);
        v = *reinterpret_cast<const uint4*>(h);
    }
    reinterpret_cast<uint4*>(a32)[t] = v;
}

__global__ void k_f32_to_bf16(const float* __restrict__ a, bf16* __restrict__ b, long n) {
    const long e = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (e < n) b[e] = __float2bfloat16(a[e]);
}

__global__ void k_adam(float* __restrict__ w, const float* __restrict__ g, float* __restrict__ m,
                       float* __restrict__ v, long n, float lr, float b1, float b2, float eps, float c1, float c2) {
    const long e = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= n) return;
    const float gg = g[e];
    const float mm = b1 * m[e] + (1.f - b1) * gg;
    const float vv = b2 * v[e] + (1.f - b2) * gg * gg;
    m[e] = mm;
    v[e] = vv;
    w[e] -= lr * (mm / c1) / (sqrtf(vv / c2) + eps);
}

inline int blocks_for(long n, int bt) { return (int)((n + bt - 1) / bt); }

bool aligned16(const void* p) { return ((uintptr_t)p & 15) == 0; }

// The cut of a lattice into columns.  x is split into blocks of at most 64
// (a segment then leaves room for at least three in the ring); t is split so
// that the columns fill the SMs: the cost of a split is its rounds of
// columns times the input slices a column reads (two more than its outputs).
ConvPlan conv_plan(const ConvGeom& g, int sms) {
    ConvPlan p;
    p.nxb = (g.X + 63) / 64;
    p.wb = (g.X + p.nxb - 1) / p.nxb;
    p.line = p.wb + 2;
    p.plane = (g.Y + 2) * p.line;
    p.vol = g.Z * p.plane;
    p.tiles = (p.vol + kCvRows - 1) / kCvRows;
    p.np = kCvRows + 2 * p.line + 2;
    p.nseg = std::min(kCvMaxSeg, (kCvSmemMax - 1024 - kCvWBytes - kCvBarBytes - p.np * 8) / (p.np * 64));
    const long base = (long)g.S * p.nxb * p.tiles;
    double best = 0.0;
    p.nt = g.T;
    for (int n = 1; n <= g.T; ++n) {  // n columns along t
        const int nt = (g.T + n - 1) / n;
        const long cols = base * ((g.T + nt - 1) / nt);
        const double cost = (double)((cols + sms - 1) / sms) * (nt + 2);
        if (n == 1 || cost < best) best = cost, p.nt = nt;
        if (cols > 64L * sms) break;
    }
    p.nts = (g.T + p.nt - 1) / p.nt;
    p.cols = base * p.nts;
    return p;
}

template <int EPI>
cudaError_t conv(const bf16* in, const bf16* W, void* out, const bf16* mask, const ConvGeom& g, cudaStream_t st,
                 int ostride = kCP) {
    if ((long)g.V * g.S == 0) return cudaSuccess;
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_conv_tc<EPI>, cudaFuncAttributeMaxDynamicSharedMemorySize, kCvSmemMax - 1024);
    if (e != cudaSuccess) return e;
    const ConvPlan p = conv_plan(g, sms);
    const size_t smem = kCvWBytes + (size_t)p.np * (p.nseg * 64 + 8) + kCvBarBytes;
    k_conv_tc<EPI><<<(int)std::min<long>(p.cols, sms), kCvThreads, smem, st>>>(in, W, out, mask, g, p,
                                                                               aligned16(out) ? ostride : -ostride);
    return cudaGetLastError();
}

// one layer's weight gradient, or (masked) the sums of all layers' that were
// not finite
template <bool MASKED>
cudaError_t wgrad(const WgLayers& layers, const ConvGeom& g, cudaStream_t st) {
    if ((long)g.V * g.S == 0) return cudaSuccess;
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    const ConvPlan p = conv_plan(g, sms);
    const size_t smem = (size_t)kWgStages * (kCvRows + 3 * p.np) * 64 + (size_t)p.np * 8;
    e = cudaFuncSetAttribute(k_conv_wgrad<MASKED>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    // three CTA classes (dt); a share of fewer than 2 steps is not worth its atomics
    const long steps = (long)g.S * p.nxb * p.tiles * g.T;
    const int ranks = (int)std::max<long>(1, std::min<long>(std::min(sms, kWgMaxCtas) / 3, (steps + 1) / 2));
    k_conv_wgrad<MASKED><<<dim3(3 * ranks, MASKED ? kNetLayers : 1), kWgThreads, smem, st>>>(layers, g, p);
    return cudaGetLastError();
}

}  // namespace

cudaError_t net_convert(const NetDev& n, cudaStream_t st) {
    long off = 0;
    for (int l = 0; l < kNetLayers; ++l) {
        k_convert<<<blocks_for(81 * 32 * 32, 256), 256, 0, st>>>(n.Wm + off, n.Wf[l], n.Wb[l], kNetCout[l],
                                                                 kNetCin[l]);
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        off += kNetLayerW[l];
    }
    return cudaSuccess;
}

cudaError_t net_hidden(const NetDev& n, const ConvGeom& g, const bf16* a0, bf16* a1, bf16* a2, cudaStream_t st) {
    cudaError_t e = conv<EPI_LEAKY_BF16>(a0, n.Wf[0], a1, nullptr, g, st);
    return e != cudaSuccess ? e : conv<EPI_LEAKY_BF16>(a1, n.Wf[1], a2, nullptr, g, st);
}

cudaError_t net_forward(const NetDev& n, const ConvGeom& g, const bf16* a0, bf16* a1, bf16* a2, float* out,
                        cudaStream_t st, int ostride) {
    const cudaError_t e = net_hidden(n, g, a0, a1, a2, st);
    return e != cudaSuccess ? e : conv<EPI_F32>(a2, n.Wf[2], out, nullptr, g, st, ostride);
}

cudaError_t net_backward(const NetDev& n, const ConvGeom& g, const bf16* a0, const bf16* a1, const bf16* a2,
                         const bf16* dob, float* dW, float* din, bf16* d1, bf16* d2, cudaStream_t st, int dstride) {
    cudaError_t e;
    const WgLayer w0 = {a0, d1, dW, n.redo, kNetCout[0], kNetCin[0]};
    const WgLayer w1 = {a1, d2, w0.dW + kNetLayerW[0], n.redo + kWgMaxCtas, kNetCout[1], kNetCin[1]};
    const WgLayer w2 = {a2, dob, w1.dW + kNetLayerW[1], n.redo + 2 * kWgMaxCtas, kNetCout[2], kNetCin[2]};
    if ((e = wgrad<false>({{w2}}, g, st)) != cudaSuccess) return e;
    if ((e = conv<EPI_DMASK_BF16>(dob, n.Wb[2], d2, a2, g, st)) != cudaSuccess) return e;
    if ((e = wgrad<false>({{w1}}, g, st)) != cudaSuccess) return e;
    if ((e = conv<EPI_DMASK_BF16>(d2, n.Wb[1], d1, a1, g, st)) != cudaSuccess) return e;
    if ((e = wgrad<false>({{w0}}, g, st)) != cudaSuccess) return e;
    if ((e = wgrad<true>({{w0, w1, w2}}, g, st)) != cudaSuccess) return e;
    if (din) return conv<EPI_F32>(d1, n.Wb[0], din, nullptr, g, st, dstride);
    return cudaSuccess;
}

cudaError_t to_bf16(const float* a, bf16* b, long n, cudaStream_t st) {
    k_f32_to_bf16<<<blocks_for(n, 256), 256, 0, st>>>(a, b, n);
    return cudaGetLastError();
}

cudaError_t net_fault(int* fault) {
    // read and clear the flag the convolution sets when a bounded wait expired
    cudaError_t e = cudaMemcpyFromSymbol(fault, g_tc_fault, sizeof(int));
    if (e == cudaSuccess && *fault) {
        const int zero = 0;
        e = cudaMemcpyToSymbol(g_tc_fault, &zero, sizeof(int));
    }
    return e;
}

cudaError_t pack_act(const float* in24, bf16* a32, long rows, cudaStream_t st) {
    k_pack<<<blocks_for(rows * 4, 256), 256, 0, st>>>(in24, a32, rows, aligned16(in24));
    return cudaGetLastError();
}

cudaError_t adam_step(float* w, const float* g, float* m, float* v, long n, float lr, float b1, float b2,
                      float eps, int t, cudaStream_t st) {
    const float c1 = 1.f - powf(b1, (float)t), c2 = 1.f - powf(b2, (float)t);
    k_adam<<<blocks_for(n, 256), 256, 0, st>>>(w, g, m, v, n, lr, b1, b2, eps, c1, c2);
    return cudaGetLastError();
}

}  // namespace eofa
