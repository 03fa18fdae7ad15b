// net_wgrad.cu -- weight gradient of the warm-start network's 3 x 3
// convolutions on the fifth-generation tensor cores.
//
// dW[co][tap][ci] = sum over pixels p of dZ[p][co] X[p shifted by tap][ci] is a
// matrix product whose K dimension is the pixel, and both operands are stored
// with the other dimension contiguous (NHWC), so both are fed to tcgen05.mma
// MN-major: a TMA box of 64 (or 32) channels x 128 or 256 pixels is a stack of
// pixel rows in the swizzled layout, eight pixels to a swizzle atom, and one MMA
// step takes K = 16 pixels.
//   A  the box of dZ, M = 128 output channels (two 64-channel blocks, or one
//      block of 64 or 32 with the other accumulator rows left unread);
//   B  the box of X started one column left, at, or right of the tile (the
//      tap's dx) and one row above it, two rows taller than the tile: the
//      three taps of a kernel column are the SAME shared-memory rows read one
//      image row apart, that is three N blocks whose stride is the box's row
//      pitch.  One MMA of N = 3 CB therefore serves three taps, and X is read
//      three times per pixel (plus the halo rows) and not nine.
// The order of the sums is that of the mma.sync kernel (net_kernels.cu): the same
// runs of consecutive pixels (wgrad_split), each run one chain of FP32
// accumulations, 16 pixels at a time, and one atomic addition per element and
// run.  The tensor cores' accumulation drops low bits at every step, so another
// split of the pixels is another rounding of every weight, and the first steps of
// Adam, which move a weight by lr g / |g|, make a visible difference of it; with
// the same runs the partial sums of the two kernels are equal to the bit and only
// the order in which the atomics arrive is left open.  Hence the box covers
// consecutive pixels: whole rows, or a piece of one row.
// A persistent CTA walks work items (run, dx, ci block, co block): warp 0
// copies, warp 1 issues the MMAs of one run into one of two TMEM accumulators,
// warps 2-5 add the other one to the gradient vector.
// Bound: the copies of X and dZ through L2 (three column shifts, the halo rows of
// the flat boxes, each co and ci block again) and the smem operand reads of the
// MMAs.
// Measured, 16 samples of 128 x 128, weight gradients of all 15 layers: 347 us
// (1357 us on the mma.sync kernel).
// Every wait is bounded, as in net_tc.cu.
#include "net_tc.cuh"

namespace mdfnet {

namespace {

constexpr int WG_THREADS = 32 * 6;
constexpr int WG_MAX_STAGES = 8;
constexpr int WG_RING = 200 * 1024;  // shared memory of the ring
constexpr int WG_SMEM = WG_RING + (2 * WG_MAX_STAGES + 5) * 8 + 16 + 1024;

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

// A box: kp consecutive pixels as columns x rows x images.
struct WgTile {
    int kp, Wx, Hy, Bn;
};

struct WgWork {
    WgTile tile;
    int img_shift;        // log2 of the tile's pixels per image
    int rows;             // pixel rows of a B box (two halo rows per image)
    int stage, stages;    // bytes of a ring slot, slots
    int ktiles, chunk;    // 32-pixel pieces in all, and of a run
    int nci, nco;         // channel blocks
    int items;
};

template <int CA, int CB, int MB>
__global__ void __launch_bounds__(WG_THREADS, 1)
    wgrad_tc_kernel(const __grid_constant__ CUtensorMap zmap, const __grid_constant__ CUtensorMap xmap,
                    const WGradArgs a, const WgWork w, int *err) {
    constexpr int N = 3 * CB;                   // columns of one accumulator
    constexpr int ACC = N <= 128 ? 128 : 256;   // TMEM columns reserved for it
    extern __shared__ unsigned char smem_raw[];
    unsigned char *smem = reinterpret_cast<unsigned char *>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
    const int stages = w.stages, a_bytes = MB * w.tile.kp * CA * 2;
    uint64_t *full = reinterpret_cast<uint64_t *>(smem + stages * w.stage);
    uint64_t *empty = full + WG_MAX_STAGES;
    uint64_t *tfull = empty + WG_MAX_STAGES;
    uint64_t *tempty = tfull + 2;
    uint64_t *drain = tempty + 2;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(drain + 1);
    __shared__ int s_fail;
    __shared__ int s_issued, s_consumed;
    volatile int *fail = &s_fail;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

    if (tid == 0) {
        s_fail = 0;
        s_issued = s_consumed = 0;
        for (int s = 0; s < stages; ++s) {
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
    if (warp == 1) tmem_alloc(tmem_slot, 2 * ACC);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    // item -> run of pixels [p0, p1) (slowest), then dx, ci block, co block
    auto item_of = [&](int it, int &p0, int &p1, int &dx, int &cib, int &cob) {
        cob = it % w.nco;
        it /= w.nco;
        cib = it % w.nci;
        it /= w.nci;
        dx = it % 3;
        const int k0 = it / 3 * w.chunk, k1 = k0 + w.chunk < w.ktiles ? k0 + w.chunk : w.ktiles;
        p0 = k0 * 32;
        p1 = k1 * 32;
    };

    if (warp == 0) {
        if (lane == 0) {
            // ---- TMA producer: the boxes that the run touches
            int k = 0, s = 0;
            uint32_t turn = 0;
            for (int it = blockIdx.x; it < w.items && !*fail; it += gridDim.x) {
                int p0, p1, dx, cib, cob;
                item_of(it, p0, p1, dx, cib, cob);
                for (int j = p0 / w.tile.kp; j <= (p1 - 1) / w.tile.kp; ++j) {
                    if (k >= stages && !mb_wait_f(&empty[s], turn ^ 1, fail)) {
                        *fail = 1;
                        break;
                    }
                    int p = j * w.tile.kp;
                    const int x0 = p % a.R;
                    p /= a.R;
                    const int y0 = p % a.R, b0 = p / a.R;
                    unsigned char *sa = smem + s * w.stage;
                    mb_expect_tx(&full[s], (uint32_t)(a_bytes + w.rows * CB * 2));
                    for (int m = 0; m < MB; ++m)
                        tma_load_4d(&zmap, &full[s], sa + m * w.tile.kp * CA * 2, (cob * MB + m) * CA, x0, y0, b0);
                    tma_load_4d(&xmap, &full[s], sa + a_bytes, cib * CB, x0 + dx - 1, y0 - 1, b0);
                    s_issued = ++k;
                    if (++s == stages) {
                        s = 0;
                        turn ^= 1;
                    }
                }
            }
        }
    } else if (warp == 1) {
        if (lane == 0) {
            // ---- MMA issuer
            constexpr uint32_t idesc = idesc_bf16_mn(TC_BM, N);
            // a single block of A: the accumulator rows of the blocks after it
            // are not read back, so those may be any rows of the slot (each
            // eight pixels on: the last step reads into the slot's B box)
            const uint32_t lbo_a = MB == 2 ? (uint32_t)(w.tile.kp * CA * 2) : 8 * CA * 2;
            const uint32_t lbo_b = (uint32_t)(w.tile.Wx * CB * 2);
            int k = 0, s = 0, t = 0;
            uint32_t turn = 0;
            bool ok = true;
            for (int it = blockIdx.x; it < w.items && ok; it += gridDim.x, ++t) {
                int p0, p1, dx, cib, cob;
                item_of(it, p0, p1, dx, cib, cob);
                const int acc = t & 1;
                if (t >= 2 && !mb_wait_f(&tempty[acc], (uint32_t)(((t >> 1) - 1) & 1), fail)) {
                    ok = false;
                    break;
                }
                tc_fence_after();
                const uint32_t d = tmem + (uint32_t)(acc * ACC);
                uint32_t add = 0;
                for (int j = p0 / w.tile.kp; j <= (p1 - 1) / w.tile.kp; ++j) {
                    if (!mb_wait_f(&full[s], turn, fail)) {
                        ok = false;
                        break;
                    }
                    s_consumed = ++k;
                    tc_fence_after();
                    const uint32_t sa = s_u32(smem + s * w.stage);
                    const uint64_t ad = mnmajor_desc<CA>(sa, lbo_a);
                    const uint64_t bd = mnmajor_desc<CB>(sa + (uint32_t)a_bytes, lbo_b);
                    // the part of the run in this box
                    const int base = j * w.tile.kp;
                    const int q0 = p0 > base ? p0 - base : 0;
                    const int q1 = p1 - base < w.tile.kp ? p1 - base : w.tile.kp;
                    for (int q = q0; q < q1; q += 16) {
                        // descriptor steps in 16-byte units; a B box has two halo
                        // rows more between its images
                        const int qb = q + (q >> w.img_shift) * 2 * w.tile.Wx;
                        umma_f16(d, ad + (uint64_t)(q * CA * 2 / 16), bd + (uint64_t)(qb * CB * 2 / 16), idesc, add);
                        add = 1;
                    }
                    umma_commit(&empty[s]);
                    if (++s == stages) {
                        s = 0;
                        turn ^= 1;
                    }
                }
                if (!ok) break;
                umma_commit(&tfull[acc]);
            }
            if (!ok) *fail = 1;
            umma_commit(drain);
            mb_wait(drain, 0);
        }
    } else {
        // ---- warps 2-5: add the accumulator to the gradient; TMEM lane =
        // output channel, column = (kernel row, input channel)
        const int q = warp & 3;
        int t = 0;
        for (int it = blockIdx.x; it < w.items; it += gridDim.x, ++t) {
            int p0, p1, dx, cib, cob;
            item_of(it, p0, p1, dx, cib, cob);
            const int acc = t & 1;
            const int row = q * 32 + lane;
            const int co = cob * MB * CA + row;
            const bool mine = row < MB * CA && co < a.cout_real;
            // the warp has an output channel (uniform over its lanes)
            const bool busy = cob * MB * CA + q * 32 < a.cout_real && q * 32 < MB * CA;
            bool ready = true;
            if (lane == 0) ready = mb_wait_f(&tfull[acc], (uint32_t)((t >> 1) & 1), fail);
            ready = __shfl_sync(0xffffffffu, ready ? 1 : 0, 0) != 0;
            if (!ready) {
                if (lane == 0) *fail = 1;
                break;
            }
            tc_fence_after();
            // TMEM loads are warp-collective, so the lanes of a warp never part
            // in here: those without a channel add nothing
            if (busy) {
                const uint32_t base = tmem + (uint32_t)(acc * ACC) + ((uint32_t)(q * 32) << 16);
                float *g0 = a.g + a.off + (long long)(mine ? co : 0) * 9 * a.cin_real;
                const bool vec = ((a.off | a.cin_real) & 3) == 0;  // 16-byte aligned groups of four input channels
#pragma unroll
                for (int c = 0; c < N; c += 16) {
                    float v[16];
                    tmem_ld16(base + (uint32_t)c, v);
                    const int ci = cib * CB + c % CB;
                    float *g = g0 + ((c / CB) * 3 + dx) * a.cin_real + ci;
                    if (vec) {
#pragma unroll
                        for (int e = 0; e < 16; e += 4) red_add4_if(g + e, v + e, mine && ci + e < a.cin_real);
                    } else {
#pragma unroll
                        for (int e = 0; e < 16; ++e) red_add_if(g + e, v[e], mine && ci + e < a.cin_real);
                    }
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbarrier_arrive(&tempty[acc]);
        }
    }
    __syncthreads();
    if (s_fail) {
        if (tid == 0) {
            atomicCAS(err, 0, 1);
            for (int k = s_consumed; k < s_issued; ++k) mb_wait(&full[k % stages], (uint32_t)((k / stages) & 1));
        }
        __syncthreads();
    }
    tc_fence_after();
    if (warp == 1) tmem_dealloc(tmem, 2 * ACC);
}

// kp consecutive pixels: whole rows of whole images where a row is no longer
// than that, else a piece of one row.
bool wg_tile(int R, int kp, WgTile *t) {
    if (R < 8 || (R & (R - 1))) return false;
    t->kp = kp;
    t->Wx = R < kp ? R : kp;
    t->Hy = R < kp / t->Wx ? R : kp / t->Wx;
    t->Bn = kp / (t->Wx * t->Hy);
    return true;
}

template <int CA, int CB, int MB>
cudaError_t wg_launch(const WGradArgs &a, int num_sms, int *err, cudaStream_t st) {
    WgWork w;
    // the larger box has the fewer halo rows; it is taken where the ring holds
    // three of them (two boxes of 128 pixels always fit)
    for (int kp : {256, 128}) {
        if (!wg_tile(a.R, kp, &w.tile)) return cudaErrorInvalidValue;
        w.rows = w.tile.Bn * (w.tile.Hy + 2) * w.tile.Wx;
        w.stage = (MB * kp * CA * 2 + w.rows * CB * 2 + 1023) / 1024 * 1024;
        w.stages = WG_RING / w.stage < WG_MAX_STAGES ? WG_RING / w.stage : WG_MAX_STAGES;
        if (w.stages >= 3) break;
    }
    if (w.stages < 2) return cudaErrorInvalidValue;
    for (w.img_shift = 0; (1 << w.img_shift) < w.tile.Wx * w.tile.Hy;) ++w.img_shift;
    const WGradSplit split = wgrad_split(a, num_sms);
    w.nci = a.Cin / CB;
    w.nco = a.Cout / (MB * CA);
    const long long items = split.splits * 3 * w.nci * w.nco;
    if (items > (1ll << 30) || split.ktiles > (1ll << 25)) return cudaErrorInvalidValue;
    w.ktiles = (int)split.ktiles;
    w.chunk = (int)split.chunk;
    w.items = (int)items;
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
    auto k = wgrad_tc_kernel<CA, CB, MB>;
    static std::atomic<unsigned long long> configured{0};  // devices whose attribute is set
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const unsigned long long bit = 1ull << (dev & 63);
    if (!(configured.load() & bit)) {
        e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, WG_SMEM);
        if (e != cudaSuccess) return e;
        configured.fetch_or(bit);
    }
    const int grid = w.items < num_sms ? w.items : num_sms;
    k<<<(unsigned)grid, WG_THREADS, WG_SMEM, st>>>(zmap, xmap, a, w, err);
    return cudaGetLastError();
}

}  // namespace

bool conv_wgrad_tc_applies(const WGradArgs &a) {
    WgTile t;
    return wg_tile(a.R, 128, &t) && (a.Cin == 32 || a.Cin % 64 == 0) &&
           (a.Cout == 32 || a.Cout == 64 || a.Cout % 128 == 0);
}

// Boxes of 32 channels (64-byte pixel rows) where a layer has 32, of 64
// otherwise, two of dZ where it has 128 or more: a box never reaches past a
// tensor's channels.
cudaError_t conv_wgrad_tc(const WGradArgs &a, int num_sms, int *err, cudaStream_t st) {
    if (!conv_wgrad_tc_applies(a)) return cudaErrorInvalidValue;
    if (a.Cin == 32) {
        if (a.Cout == 32) return wg_launch<32, 32, 1>(a, num_sms, err, st);
        return a.Cout == 64 ? wg_launch<64, 32, 1>(a, num_sms, err, st) : wg_launch<64, 32, 2>(a, num_sms, err, st);
    }
    if (a.Cout == 32) return wg_launch<32, 64, 1>(a, num_sms, err, st);
    return a.Cout == 64 ? wg_launch<64, 64, 1>(a, num_sms, err, st) : wg_launch<64, 64, 2>(a, num_sms, err, st);
}

}  // namespace mdfnet
