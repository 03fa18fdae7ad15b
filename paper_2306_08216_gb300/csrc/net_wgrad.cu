// net_wgrad.cu -- weight and bias gradients of the warm-start network's
// 3 x 3 convolutions on the fifth-generation tensor cores.
//
// dW[co][tap][ci] = sum over pixels p of dZ[p][co] X[p shifted by tap][ci] is a
// matrix product whose K dimension is the pixel, and both operands are stored
// with the other dimension contiguous (NHWC), so both are fed to tcgen05.mma
// MN-major: a TMA box of 64 (or 32) channels x 256 pixels is a stack of pixel
// rows in the swizzled layout, eight pixels to a swizzle atom, and one MMA
// step takes K = 16 pixels.
//   A  the box of dZ, M = 128 output channels (two 64-channel blocks, or one
//      block of 64 or 32 with the other accumulator rows left unread);
//   B  the box of X started one column left, at, or right of the tile (the
//      tap's dx) and one row above it, two rows taller than the tile: the
//      three taps of a kernel column are the SAME shared-memory rows read one
//      image row apart, that is three N blocks whose stride is the box's row
//      pitch.  One MMA of N = 3 CB therefore serves three taps, and X is read
//      three times per pixel (plus the two halo rows) and not nine;
//   bias gradient: one more MMA of N = 16 against a tile of ones, in the
//      work items of the first input-channel block at dx = 0.
// A persistent CTA walks work items (run of pixel chunks, dx, ci block, co
// block): warp 0 copies, warp 1 issues the MMAs of one chunk (16 K steps) into
// one of two TMEM accumulators, warps 2-5 add the other one to FP32 registers
// and, at the end of the item, the registers to the gradient vector.  The
// tensor cores' FP32 accumulation drops low bits at every K step, so a short
// chain of them with rounded additions in between is the more accurate sum
// (16 steps against the mma.sync kernel's 82), and one atomic per element and
// CTA is the cheaper one.
// Bound: the copies of X and dZ through L2 (three column shifts, each co and
// ci block again) and the smem operand reads of the MMAs.
// Measured, 16 samples of 128 x 128, weight and bias gradients of all 15 layers:
// 342 us (2027 us on the mma.sync kernel and its bias reduction); per chunk of
// 32 x 32 channels 1.6 us of a CTA.  With the accumulator added to memory every
// five chunks, element by element, 755 us.
// Every wait is bounded, as in net_tc.cu.
#include "net_tc.cuh"

namespace mdfnet {

namespace {

constexpr int WG_PIX = 256;             // pixels of a chunk (K of a ring slot)
constexpr int WG_THREADS = 32 * 6;
constexpr int WG_BIAS_N = 16;           // columns of the bias MMA

// MN-major operand in the swizzled layout of TMA: pixel rows of `CH` channels
// (2 CH bytes); lbo: bytes between blocks of CH channels, 8-pixel groups are
// contiguous.
template <int CH>
__device__ __forceinline__ uint64_t mnmajor_desc(uint32_t saddr, uint32_t lbo) {
    constexpr uint64_t sbo = 8 * CH * 2;
    constexpr uint64_t layout = CH == 64 ? 2 : 4;
    return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)(lbo >> 4) << 16) | ((sbo >> 4) << 32) |
           ((uint64_t)1 << 46) | (layout << 61);
}

// kind::f16 instruction descriptor with both operands MN-major (bits 15, 16).
__host__ __device__ constexpr uint32_t idesc_bf16_mn(int M, int N) {
    return idesc_bf16(M, N) | (1u << 15) | (1u << 16);
}

// *p += x where ok, without a branch.
__device__ __forceinline__ void red_add_if(float *p, float x, bool ok) {
    asm volatile(
        "{\n\t.reg .pred q;\n\t"
        "setp.ne.b32 q, %2, 0;\n\t"
        "@q red.global.add.f32 [%0], %1;\n\t}" ::"l"(p),
        "f"(x), "r"((int)ok)
        : "memory");
}

__device__ __forceinline__ void red_add4_if(float *p, const float *x, bool ok) {
    asm volatile(
        "{\n\t.reg .pred q;\n\t"
        "setp.ne.b32 q, %5, 0;\n\t"
        "@q red.global.add.v4.f32 [%0], {%1, %2, %3, %4};\n\t}" ::"l"(p),
        "f"(x[0]), "f"(x[1]), "f"(x[2]), "f"(x[3]), "r"((int)ok)
        : "memory");
}

struct WgTile {
    int Wx, Hy, Bn;  // 256 pixels as columns x rows x images
};

struct WgWork {
    WgTile tile;
    int tx, ty, tb;       // tiles per row, per column, along the batch
    int chunks, group;    // tiles in all, tiles per work item
    int nci, nco;         // channel blocks
    int items;
};

template <int CA, int CB, int MB, int STAGES>
struct WgSmem {
    static constexpr int A_BYTES = MB * WG_PIX * CA * 2;
    static constexpr int B_BYTES = 320 * CB * 2;  // at most 320 pixel rows (tile plus two image rows)
    static constexpr int STAGE = A_BYTES + B_BYTES;
    static constexpr int ONES = STAGES * STAGE;   // 16 pixels x 64 ones
    static constexpr int BARS = ONES + 2048;
    static constexpr int NBAR = 2 * STAGES + 5;
    static constexpr int TOTAL = BARS + NBAR * 8 + 16 + 1024;
};

template <int CA, int CB, int MB, int STAGES>
__global__ void __launch_bounds__(WG_THREADS, 1)
    wgrad_tc_kernel(const __grid_constant__ CUtensorMap zmap, const __grid_constant__ CUtensorMap xmap,
                    const WGradArgs a, const WgWork w, int *err) {
    using S = WgSmem<CA, CB, MB, STAGES>;
    constexpr int N = 3 * CB;       // columns of one accumulator, then the bias
    constexpr int ACC = 256;        // TMEM columns reserved for it
    extern __shared__ unsigned char smem_raw[];
    unsigned char *smem = reinterpret_cast<unsigned char *>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
    uint64_t *full = reinterpret_cast<uint64_t *>(smem + S::BARS);
    uint64_t *empty = full + STAGES;
    uint64_t *tfull = empty + STAGES;
    uint64_t *tempty = tfull + 2;
    uint64_t *drain = tempty + 2;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(drain + 1);
    __shared__ int s_fail;
    __shared__ int s_issued, s_consumed;
    volatile int *fail = &s_fail;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int rows = w.tile.Bn * (w.tile.Hy + 2) * w.tile.Wx;  // pixel rows of a B box

    if (tid == 0) {
        s_fail = 0;
        s_issued = s_consumed = 0;
        for (int s = 0; s < STAGES; ++s) {
            mb_init(&full[s], 1);
            mb_init(&empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mb_init(&tfull[b], 1);
            mb_init(&tempty[b], 4);
        }
        mb_init(drain, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    for (int i = tid; i < 2048 / 4; i += WG_THREADS)
        reinterpret_cast<uint32_t *>(smem + S::ONES)[i] = 0x3f803f80u;  // BF16 ones
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    if (warp == 1) tmem_alloc(tmem_slot, 2 * ACC);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    // item -> pixel group (slowest), then dx, ci block, co block
    auto item_of = [&](int it, int &grp, int &dx, int &cib, int &cob) {
        cob = it % w.nco;
        it /= w.nco;
        cib = it % w.nci;
        it /= w.nci;
        dx = it % 3;
        grp = it / 3;
    };
    auto chunks_of = [&](int grp) {
        const int c0 = grp * w.group;
        return w.chunks - c0 < w.group ? w.chunks - c0 : w.group;
    };

    if (warp == 0) {
        if (lane == 0) {
            // ---- TMA producer
            int k = 0;
            for (int it = blockIdx.x; it < w.items && !*fail; it += gridDim.x) {
                int grp, dx, cib, cob;
                item_of(it, grp, dx, cib, cob);
                const int nc = chunks_of(grp);
                for (int j = 0; j < nc; ++j, ++k) {
                    const int s = k % STAGES;
                    if (k >= STAGES && !mb_wait_f(&empty[s], (uint32_t)(((k / STAGES) - 1) & 1), fail)) {
                        *fail = 1;
                        break;
                    }
                    int c = grp * w.group + j;
                    const int x0 = (c % w.tx) * w.tile.Wx;
                    c /= w.tx;
                    const int y0 = (c % w.ty) * w.tile.Hy;
                    const int b0 = (c / w.ty) * w.tile.Bn;
                    unsigned char *sa = smem + s * S::STAGE;
                    mb_expect_tx(&full[s], (uint32_t)(S::A_BYTES + rows * CB * 2));
                    for (int m = 0; m < MB; ++m)
                        tma_load_4d(&zmap, &full[s], sa + m * WG_PIX * CA * 2, (cob * MB + m) * CA, x0, y0, b0);
                    tma_load_4d(&xmap, &full[s], sa + S::A_BYTES, cib * CB, x0 + dx - 1, y0 - 1, b0);
                    s_issued = k + 1;
                }
            }
        }
    } else if (warp == 1) {
        if (lane == 0) {
            // ---- MMA issuer
            constexpr uint32_t idesc = idesc_bf16_mn(TC_BM, N), idesc_b = idesc_bf16_mn(TC_BM, WG_BIAS_N);
            // a single block of A: the accumulator rows of the blocks after it
            // are not read back, so those may be any rows of the slot (each
            // eight pixels on: the last step reads into the slot's B box)
            constexpr uint32_t lbo_a = MB == 2 ? WG_PIX * CA * 2 : 8 * CA * 2;
            const uint32_t lbo_b = (uint32_t)(w.tile.Wx * CB * 2);
            // descriptor steps of 16 pixels, in 16-byte units; a B box has two
            // halo rows more between images of fewer than 256 pixels
            const int img = w.tile.Wx * w.tile.Hy;
            constexpr uint64_t step_a = 16 * CA * 2 / 16, step_b = 16 * CB * 2 / 16;
            const uint64_t skip_b = (uint64_t)(2 * w.tile.Wx * CB * 2 / 16);
            const uint64_t od = mnmajor_desc<64>(s_u32(smem + S::ONES), 1024);
            int k = 0;
            bool ok = true;
            for (int it = blockIdx.x; it < w.items && ok; it += gridDim.x) {
                int grp, dx, cib, cob;
                item_of(it, grp, dx, cib, cob);
                const bool bias = dx == 0 && cib == 0;
                const int nc = chunks_of(grp);
                for (int j = 0; j < nc; ++j, ++k) {
                    const int s = k % STAGES, acc = k & 1;
                    if (k >= 2 && !mb_wait_f(&tempty[acc], (uint32_t)(((k >> 1) - 1) & 1), fail)) {
                        ok = false;
                        break;
                    }
                    if (!mb_wait_f(&full[s], (uint32_t)((k / STAGES) & 1), fail)) {
                        ok = false;
                        break;
                    }
                    s_consumed = k + 1;
                    tc_fence_after();
                    const uint32_t d = tmem + (uint32_t)(acc * ACC);
                    const uint32_t sa = s_u32(smem + s * S::STAGE);
                    uint64_t ad = mnmajor_desc<CA>(sa, lbo_a), bd = mnmajor_desc<CB>(sa + S::A_BYTES, lbo_b);
#pragma unroll
                    for (int p = 0; p < WG_PIX; p += 16) {
                        umma_f16(d, ad, bd, idesc, p != 0);
                        if (bias) umma_f16(d + N, ad, od, idesc_b, p != 0);
                        ad += step_a;
                        bd += step_b;
                        if (((p + 16) & (img - 1)) == 0) bd += skip_b;
                    }
                    umma_commit(&empty[s]);
                    umma_commit(&tfull[acc]);
                }
            }
            if (!ok) *fail = 1;
            umma_commit(drain);
            mb_wait(drain, 0);
        }
    } else {
        // ---- warps 2-5: add the accumulator to the gradient; TMEM lane =
        // output channel, column = (kernel row, input channel)
        const int q = warp & 3;
        int k = 0;
        for (int it = blockIdx.x; it < w.items; it += gridDim.x) {
            int grp, dx, cib, cob;
            item_of(it, grp, dx, cib, cob);
            const int nc = chunks_of(grp);
            const bool bias = dx == 0 && cib == 0;
            const int row = q * 32 + lane;
            const int co = cob * MB * CA + row;
            const bool mine = row < MB * CA && co < a.cout_real;
            // the warp has an output channel (uniform over its lanes)
            const bool busy = cob * MB * CA + q * 32 < a.cout_real && q * 32 < MB * CA;
            float sum[N], bsum = 0.0f;
#pragma unroll
            for (int c = 0; c < N; ++c) sum[c] = 0.0f;
            bool ready = true;
            for (int j = 0; j < nc; ++j, ++k) {
                const int acc = k & 1;
                if (lane == 0) ready = mb_wait_f(&tfull[acc], (uint32_t)((k >> 1) & 1), fail);
                ready = __shfl_sync(0xffffffffu, ready ? 1 : 0, 0) != 0;
                if (!ready) break;
                tc_fence_after();
                // TMEM loads are warp-collective, so the lanes of a warp never
                // part in here: those without a channel add what nobody reads
                if (busy) {
                    const uint32_t base = tmem + (uint32_t)(acc * ACC) + ((uint32_t)(q * 32) << 16);
                    float v[16];
#pragma unroll
                    for (int c = 0; c < N; c += 16) {
                        tmem_ld16(base + (uint32_t)c, v);
#pragma unroll
                        for (int e = 0; e < 16; ++e) sum[c + e] += v[e];
                    }
                    if (bias) {
                        tmem_ld16(base + (uint32_t)N, v);
                        bsum += v[0];
                    }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbarrier_arrive(&tempty[acc]);
            }
            if (!ready) {
                if (lane == 0) *fail = 1;
                break;
            }
            if (busy) {
                float *g0 = a.g + a.off + (long long)(mine ? co : 0) * 9 * a.cin_real;
                if (((a.off | a.cin_real) & 3) == 0) {  // 16-byte aligned groups of four input channels
#pragma unroll
                    for (int c = 0; c < N; c += 4) {
                        const int ci = cib * CB + c % CB;
                        red_add4_if(g0 + ((c / CB) * 3 + dx) * a.cin_real + ci, sum + c, mine && ci < a.cin_real);
                    }
                } else {
#pragma unroll
                    for (int c = 0; c < N; ++c) {
                        const int ci = cib * CB + c % CB;
                        red_add_if(g0 + ((c / CB) * 3 + dx) * a.cin_real + ci, sum[c], mine && ci < a.cin_real);
                    }
                }
                if (bias)
                    red_add_if(a.g + a.off + (long long)a.cout_real * 9 * a.cin_real + (mine ? co : 0), bsum, mine);
            }
            __syncwarp();
        }
    }
    __syncthreads();
    if (s_fail) {
        if (tid == 0) {
            atomicCAS(err, 0, 1);
            for (int k = s_consumed; k < s_issued; ++k) mb_wait(&full[k % STAGES], (uint32_t)((k / STAGES) & 1));
        }
        __syncthreads();
    }
    tc_fence_after();
    if (warp == 1) tmem_dealloc(tmem, 2 * ACC);
}

// 256 pixels: at most 32 columns (a tall tile has the fewest halo rows), then
// rows of an image, then images.
bool wg_tile(int R, WgTile *t) {
    if (R < 8 || (R & (R - 1))) return false;
    t->Wx = R < 32 ? R : 32;
    t->Hy = R < WG_PIX / t->Wx ? R : WG_PIX / t->Wx;
    t->Bn = WG_PIX / (t->Wx * t->Hy);
    return true;
}

template <int CA, int CB, int MB, int STAGES>
cudaError_t wg_launch(const WGradArgs &a, int num_sms, int *err, cudaStream_t st) {
    using S = WgSmem<CA, CB, MB, STAGES>;
    WgWork w;
    if (!wg_tile(a.R, &w.tile)) return cudaErrorInvalidValue;
    if (w.tile.Bn * (w.tile.Hy + 2) * w.tile.Wx > 320) return cudaErrorInvalidValue;
    w.tx = a.R / w.tile.Wx;
    w.ty = a.R / w.tile.Hy;
    w.tb = (a.B + w.tile.Bn - 1) / w.tile.Bn;
    const long long chunks = (long long)w.tx * w.ty * w.tb;
    w.nci = a.Cin / CB;
    w.nco = a.Cout / (MB * CA);
    const long long tiles = 3ll * w.nci * w.nco;
    if (chunks * tiles > (1ll << 30)) return cudaErrorInvalidValue;
    w.chunks = (int)chunks;
    // chunks per work item: one item per SM where there are that many chunks
    long long splits = num_sms / tiles;
    if (splits < 1) splits = 1;
    if (splits > chunks) splits = chunks;
    w.group = (int)((chunks + splits - 1) / splits);
    w.items = (int)(((chunks + w.group - 1) / w.group) * tiles);
    auto enc = tensor_map_encoder();
    if (!enc) return cudaErrorNotSupported;
    CUtensorMap zmap, xmap;
    for (int k = 0; k < 2; ++k) {
        const int C = k ? a.Cin : a.Cout, ch = k ? CB : CA;
        const cuuint64_t dims[4] = {(cuuint64_t)C, (cuuint64_t)a.R, (cuuint64_t)a.R, (cuuint64_t)a.B};
        const cuuint64_t strides[3] = {(cuuint64_t)C * 2, (cuuint64_t)a.R * C * 2, (cuuint64_t)a.R * a.R * C * 2};
        const cuuint32_t box[4] = {(cuuint32_t)ch, (cuuint32_t)w.tile.Wx, (cuuint32_t)(w.tile.Hy + (k ? 2 : 0)),
                                   (cuuint32_t)w.tile.Bn};
        const cuuint32_t es[4] = {1, 1, 1, 1};
        if (enc(k ? &xmap : &zmap, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<bf16 *>(k ? a.X : a.dZ), dims,
                strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
                ch == 64 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return cudaErrorInvalidValue;
    }
    auto k = wgrad_tc_kernel<CA, CB, MB, STAGES>;
    static std::atomic<unsigned long long> configured{0};  // devices whose attribute is set
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const unsigned long long bit = 1ull << (dev & 63);
    if (!(configured.load() & bit)) {
        e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, S::TOTAL);
        if (e != cudaSuccess) return e;
        configured.fetch_or(bit);
    }
    const int grid = w.items < num_sms ? w.items : num_sms;
    k<<<(unsigned)grid, WG_THREADS, S::TOTAL, st>>>(zmap, xmap, a, w, err);
    return cudaGetLastError();
}

}  // namespace

bool conv_wgrad_tc_applies(const WGradArgs &a) {
    WgTile t;
    return wg_tile(a.R, &t) && (a.Cin == 32 || a.Cin % 64 == 0) &&
           (a.Cout == 32 || a.Cout == 64 || a.Cout % 128 == 0);
}

// Boxes of 32 channels (64-byte pixel rows) where a layer has 32, of 64
// otherwise, two of dZ where it has 128 or more: a box never reaches past a
// tensor's channels.  The ring takes what shared memory holds.
cudaError_t conv_wgrad_tc(const WGradArgs &a, int num_sms, int *err, cudaStream_t st) {
    if (!conv_wgrad_tc_applies(a)) return cudaErrorInvalidValue;
    if (a.Cin == 32) {
        if (a.Cout == 32) return wg_launch<32, 32, 1, 5>(a, num_sms, err, st);
        return a.Cout == 64 ? wg_launch<64, 32, 1, 4>(a, num_sms, err, st)
                            : wg_launch<64, 32, 2, 2>(a, num_sms, err, st);
    }
    if (a.Cout == 32) return wg_launch<32, 64, 1, 3>(a, num_sms, err, st);
    return a.Cout == 64 ? wg_launch<64, 64, 1, 3>(a, num_sms, err, st)
                        : wg_launch<64, 64, 2, 2>(a, num_sms, err, st);
}

}  // namespace mdfnet
