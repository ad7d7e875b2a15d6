// 1x1 convolutions from codes to codes on the tensor cores (Algorithm 1 step 5
// on codes plus the fused steps 4, 1, 3): the expand, project and shortcut layers
// of the networks.
//
// These layers have few input channels per output element, so what bounds them
// is neither the tensor core nor memory but the instructions spent per element:
// expanding the input codes and, above all, turning accumulators into codes.
// The kernel is laid out around that:
//   * the whole weight matrix of the CTA's output channels is expanded once and
//     stays in shared memory (a CTA keeps its N tile and walks over M tiles);
//   * M tiles are MT x 128 pixels, MT = 1, 2 or 4, each 128 pixels an accumulator
//     of its own: a hand-off between the roles costs a few hundred clocks
//     whatever it carries, so a narrow layer hands over 512 pixels at a time;
//   * sixteen warps run the lean epilogue (dsq_epilogue.cuh), six expand, in two
//     groups each.  A lane's accumulators are eight consecutive channels of four
//     pixels, so the scales and biases sit in registers (reading them from shared
//     memory, one clock of that pipe per number and warp, took 33.6 us for
//     112x112 16->96 where the kernel without those loads took 22.9).
//   * the packed rows of a tile are contiguous in memory and come as one untiled
//     bulk copy (stride 2: im2col boxes with a traversal stride).
// Input channels are expanded and multiplied in planes of 128.
//
// MobileNetV2-shaped layers, batch 64, 4-bit, the im2col kernel that had them before and
// this one: 112x112 16->96 71.8 -> 28.5 us, 32->16 49.4 -> 14.3; 56x56 24->144 30.4 -> 14.4,
// 144->24 + residual 19.9 -> 12.2.
//
// Every wait on a barrier is bounded, as in the other tensor-core kernels.
#include "dsq_tc_common.cuh"
#include "dsq_tc_host.h"

namespace {

// Expansion and epilogue are two groups of warps each, working on alternate fills and
// alternate tiles: what a group waits for (a barrier, a fence, tensor memory) the
// other one's work covers.
constexpr int PW_WARP_TMA = 0, PW_WARP_MMA = 1, PW_WARP_A0 = 2, PW_A_GROUP = 3, PW_WARP_E0 = 8,
              PW_E_GROUP = 8, PW_WARPS = 24;
constexpr int PW_THREADS = PW_WARPS * 32;
constexpr int PW_EPQ = PW_E_GROUP / 4;        // warps of a group per tensor-memory lane quarter
constexpr int PW_A_SLOTS = 2;                 // expanded planes
constexpr int PW_MAX_STAGES = 4;              // packed planes in flight
constexpr int PW_BARS = 2 * PW_MAX_STAGES + 2 * PW_A_SLOTS + 4 + 1;

struct PwSmem {
    uint32_t a_slots, b_tiles, a_stage, epi, bars, tmem_slot, abort_flag, total;
};

struct PwParams {
    int M, K, Ncols, BN, n_tiles, mt;         // mt: 128-pixel subtiles of a tile
    int m_tiles, mstep;                       // tiles of mt * 128 pixels; tiles between two of a CTA
    int planes, P, PB;                        // planes of 128 channels; packed bytes of a pixel, of a plane
    int stages, tmem_cols;
    int early;                                // dsq_early_constants
    const uint8_t *act;
    int stride, Ho, Wo;                       // stride 2: output image (im2col boxes)
    int box_rows;                             // pixels of a TMA box
    int smem_bytes, shift, out_pitch;
    uint32_t orv;
    unsigned long long wait_ns;
    DsqEpi e;
    const uint8_t *w;
    PwSmem L;
    int *ws;
};

// row_bytes: packed bytes of a pixel in a stage
__host__ inline PwSmem pw_layout(int mt, int BN, int planes, int row_bytes, int stages)
{
    PwSmem L;
    uint32_t o = 0;
    L.a_slots = o; o += PW_A_SLOTS * mt * 128 * 128;
    L.b_tiles = o; o += planes * BN * 128;
    L.a_stage = o; o += stages * mt * 128 * row_bytes;
    L.epi = o;     o += 2 * BN * 4;
    o = (o + 127u) & ~127u;
    L.bars = o;    o += 8 * PW_BARS;
    L.tmem_slot = o; o += 8;
    L.abort_flag = o; o += 8;
    L.total = o;
    return L;
}

// instructions (32 bytes of K each) of a plane: the expanded bytes of its packed
// chunks (4-bit: 32 per chunk, 2-bit: 64), or of its codes (3-bit, natural order)
template <int BITS>
__device__ __forceinline__ int pw_groups(const PwParams &p, int pl)
{
    if (BITS == 3) return (min(128, p.K - 128 * pl) + 31) / 32;
    return min(p.PB, p.P - pl * p.PB) / 16 * (BITS == 2 ? 2 : 1);
}

// the packed bytes of a plane of one row -> int8 chunks of its 128-byte operand
// row at `dst` (swizzled by row & 7); `chunks` packed 16-byte chunks exist
template <int BITS, bool SIGNED>
__device__ __forceinline__ void pw_store_chunk(uint32_t dst, int sw, int ch, const uint4 v, uint32_t orv)
{
    constexpr int OUT = Chunks<BITS>::OUT;
#pragma unroll
    for (int c = 0; c < OUT; ++c)
        sts_128(dst + (uint32_t)(((ch * OUT + c) ^ sw) << 4), expand_word<BITS, SIGNED>(v.x, c, orv),
                expand_word<BITS, SIGNED>(v.y, c, orv), expand_word<BITS, SIGNED>(v.z, c, orv),
                expand_word<BITS, SIGNED>(v.w, c, orv));
}
template <bool SIGNED>
__device__ __forceinline__ void pw_store_row3(uint32_t dst, int sw, const uint4 (&v)[3], int groups,
                                              uint32_t orv)
{
    const uint32_t w[12] = {v[0].x, v[0].y, v[0].z, v[0].w, v[1].x, v[1].y,
                            v[1].z, v[1].w, v[2].x, v[2].y, v[2].z, v[2].w};
#pragma unroll
    for (int q = 0; q < 8; ++q)
        if (q < 2 * groups) {
            const uint4 c = expand3_chunk<SIGNED>(w, q, orv);
            sts_128(dst + (uint32_t)((q ^ sw) << 4), c.x, c.y, c.z, c.w);
        }
}

template <int BITS, bool RES, bool LO>
__global__ void __launch_bounds__(PW_THREADS, 1)
dsq_pw_kernel(const __grid_constant__ CUtensorMap tmap_a, const PwParams p)
{
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 1023u) & ~(uintptr_t)1023u);
    const PwSmem &L = p.L;
    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0);
    const int lane = threadIdx.x & 31;
    const int n_tile = p.n_tiles == 1 ? 0 : (int)blockIdx.x % p.n_tiles;
    const int m_first = p.n_tiles == 1 ? (int)blockIdx.x : (int)blockIdx.x / p.n_tiles;
    const int my_tiles = m_first < p.m_tiles ? (p.m_tiles - 1 - m_first) / p.mstep + 1 : 0;
    const int tile_px = p.mt * 128;
    const uint32_t a_slot_bytes = (uint32_t)tile_px * 128u;
    // a stage holds the tile's packed rows as they lie in memory (stride 1), or its
    // planes one behind the other
    const uint32_t px_bytes = p.stride == 1 ? (uint32_t)p.P : (uint32_t)p.PB;
    const uint32_t plane_at = p.stride == 1 ? (uint32_t)p.PB : (uint32_t)(tile_px * p.PB);
    const uint32_t stage_bytes = (uint32_t)tile_px * (p.stride == 1 ? p.P : p.planes * p.PB);
    const uint32_t n_fills = (uint32_t)my_tiles * p.planes;

    const uint32_t bars = smem_u32(smem + L.bars);
    auto bar_st_full = [&](int s) { return bars + 8u * s; };
    auto bar_st_empty = [&](int s) { return bars + 8u * (PW_MAX_STAGES + s); };
    constexpr int O_A = 2 * PW_MAX_STAGES;
    auto bar_a_full = [&](int s) { return bars + 8u * (O_A + s); };
    auto bar_a_empty = [&](int s) { return bars + 8u * (O_A + PW_A_SLOTS + s); };
    constexpr int O_ACC = O_A + 2 * PW_A_SLOTS;
    auto bar_acc_full = [&](int s) { return bars + 8u * (O_ACC + s); };
    auto bar_acc_empty = [&](int s) { return bars + 8u * (O_ACC + 2 + s); };
    const uint32_t bar_drain = bars + 8u * (O_ACC + 4);
    volatile uint32_t *tmem_slot = reinterpret_cast<volatile uint32_t *>(smem + L.tmem_slot);
    Ctl ctl{reinterpret_cast<volatile int *>(smem + L.abort_flag), p.ws, p.wait_ns};

    if (threadIdx.x == 0) {
        for (int s = 0; s < PW_MAX_STAGES; ++s) {
            mbar_init(bar_st_full(s), 1);             // TMA producer (+ bytes)
            mbar_init(bar_st_empty(s), PW_A_GROUP * p.planes);
        }
        for (int s = 0; s < PW_A_SLOTS; ++s) {
            mbar_init(bar_a_full(s), PW_A_GROUP);
            mbar_init(bar_a_empty(s), 1);             // tcgen05.commit
        }
        for (int s = 0; s < 2; ++s) {
            mbar_init(bar_acc_full(s), 1);            // tcgen05.commit
            mbar_init(bar_acc_empty(s), PW_E_GROUP);
        }
        mbar_init(bar_drain, 1);
        *ctl.abort_flag = 0;
        mbar_init_fence();
        if (p.stride != 1) tma_prefetch_desc(&tmap_a);
    }
    if (warp == PW_WARP_MMA) {
        tmem_alloc(smem_u32((const void *)tmem_slot), (uint32_t)p.tmem_cols);
        tmem_relinquish();
    }
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem_base = __shfl_sync(0xffffffffu, *tmem_slot, 0);
    float *sm_scale = reinterpret_cast<float *>(smem + L.epi);
    float *sm_bias = sm_scale + p.BN;
    if (warp != PW_WARP_TMA) {
        // ---------------- once: weights of this N tile, scales and biases ---------
        // (early: before the wait for the kernel ahead in the stream)
        if (!p.early) grid_dependency_wait();
        const int tid = threadIdx.x - 32;
        constexpr int NT = PW_THREADS - 32;
        const uint32_t bt = smem_u32(smem + L.b_tiles);
        const int cpr = p.P / 16;                                // packed chunks of a weight row
        const int rows = min(p.BN, p.Ncols - n_tile * p.BN);
        const uint8_t *w0 = p.w + (int64_t)n_tile * p.BN * p.P;
        if (BITS == 3) {
            for (int t = tid; t < rows * p.planes; t += NT) {
                const int row = t / p.planes, pl = t - row * p.planes;
                uint4 v[3];
#pragma unroll
                for (int l = 0; l < 3; ++l) {
                    const int at = 48 * pl + 16 * l;
                    v[l] = make_uint4(0u, 0u, 0u, 0u);
                    if (at < p.P) v[l] = __ldg(reinterpret_cast<const uint4 *>(w0 + (int64_t)row * p.P + at));
                }
                const int col = dsq_column_of(row);
                pw_store_row3<true>(bt + (uint32_t)((pl * p.BN + col) * 128), col & 7, v,
                                    pw_groups<3>(p, pl), p.orv);
            }
        } else {
            for (int t = tid; t < rows * cpr; t += NT) {
                const int row = t / cpr, c = t - row * cpr;
                const uint4 v = __ldg(reinterpret_cast<const uint4 *>(w0) + t);
                const int pl = c / BITS, ch = c - pl * BITS;     // BITS chunks per plane
                const int col = dsq_column_of(row);
                pw_store_chunk<BITS, true>(bt + (uint32_t)((pl * p.BN + col) * 128), col & 7, ch, v,
                                           p.orv);
            }
        }
        for (int c = tid; c < p.BN; c += NT) {
            float sc = 0.f, bi = -1e30f;                         // padding lanes: code 0
            if (n_tile * p.BN + c < p.Ncols)
                dsq_codes_affine(p.e.scale, p.e.bias, n_tile * p.BN + c, p.e.half_offset, -p.shift,
                                 sc, bi);
            sm_scale[c] = sc;
            sm_bias[c] = bi;
        }
        fence_proxy_async_smem();
        named_barrier_sync(1, NT);
    }
    // no activation is read and nothing is written before the kernels ahead of this
    // one have completed
    grid_dependency_wait();
    grid_launch_dependents();

    if (warp == PW_WARP_TMA) {
        // ---------------- producer: packed planes --------------------------------
        if (lane == 0) {
            uint32_t issued = 0, ph = 0;
            int s = 0, m0 = m_first * tile_px;
#pragma unroll 1
            for (int it = 0; it < my_tiles; ++it) {
                if (!wait_bar(bar_st_empty(s), ph ^ 1u, ctl, 31)) break;
                const uint32_t dst = smem_u32(smem + L.a_stage) + s * stage_bytes;
                const int px = min(tile_px, p.M - m0);
                if (p.stride == 1) {
                    mbar_arrive_expect_tx(bar_st_full(s), (uint32_t)(px * p.P));
                    bulk_load(dst, p.act + (int64_t)m0 * p.P, (uint32_t)(px * p.P), bar_st_full(s));
                } else {
                    // (boxes that start behind the last pixel are left out: an im2col
                    // load starts inside the tensor)
                    const int nb = (px + p.box_rows - 1) / p.box_rows;
                    mbar_arrive_expect_tx(bar_st_full(s), (uint32_t)(nb * p.box_rows * p.planes * p.PB));
                    for (int i = 0; i < nb; ++i) {
                        const int m = m0 + i * p.box_rows;
                        const int t = m / p.Wo, n = t / p.Ho;
                        for (int pl = 0; pl < p.planes; ++pl)
                            tma_load_im2col_4d(dst + pl * plane_at + (uint32_t)(i * p.box_rows * p.PB),
                                               &tmap_a, pl * p.PB, (m - t * p.Wo) * p.stride,
                                               (t - n * p.Ho) * p.stride, n, (uint16_t)0, (uint16_t)0,
                                               bar_st_full(s));
                    }
                }
                ++issued;
                m0 += p.mstep * tile_px;
                if (++s == p.stages) { s = 0; ph ^= 1u; }
            }
            const uint32_t S = (uint32_t)p.stages;
            for (uint32_t k = (issued > S ? issued - S : 0); k < issued; ++k)
                wait_bar_drain(bar_st_full(k % S), (k / S) & 1u);
        }
    } else if (warp == PW_WARP_MMA) {
        // ---------------- MMA issuer (whole warp, uniform; one lane issues) --------
        const uint32_t idesc = idesc_i8(p.BN, false, true, 128);
        const uint64_t d0 = smem_desc_sw128(0u);
        const uint32_t dhi = (uint32_t)(d0 >> 32), dlo = (uint32_t)d0;
        const uint32_t a_lo = dlo + (smem_u32(smem + L.a_slots) >> 4);
        const uint32_t b_lo = dlo + (smem_u32(smem + L.b_tiles) >> 4);
        int slot = 0;
        uint32_t pha = 0;
        bool ok = true;
#pragma unroll 1
        for (int it = 0; ok && it < my_tiles; ++it) {
            const int as = it & 1;
            if (!(ok = wait_bar_warp(bar_acc_empty(as), ((it >> 1) & 1) ^ 1u, ctl, 33))) break;
            tc_fence_after_sync();
#pragma unroll 1
            for (int pl = 0; pl < p.planes; ++pl) {
                if (!(ok = wait_bar_warp(bar_a_full(slot), pha, ctl, 34))) break;
                tc_fence_after_sync();
                const int groups = pw_groups<BITS>(p, pl);
                const uint32_t b = b_lo + (uint32_t)(pl * p.BN * 8);
#pragma unroll 1
                for (int mt = 0; mt < p.mt; ++mt) {
                    const uint32_t a = a_lo + slot * (a_slot_bytes >> 4) + mt * (128 * 128 / 16);
                    mma_i8_ss_x4_elect(tmem_base + (as * p.mt + mt) * p.BN, a,
                                       groups > 1 ? a + 2u : 0xFFFFFFFFu,
                                       groups > 2 ? a + 4u : 0xFFFFFFFFu,
                                       groups > 3 ? a + 6u : 0xFFFFFFFFu, dhi, b, dhi, idesc,
                                       (uint32_t)pl);
                }
                mma_commit_elect(bar_a_empty(slot));
                if (++slot == PW_A_SLOTS) { slot = 0; pha ^= 1u; }
            }
            if (ok) mma_commit_elect(bar_acc_full(as));
        }
        if (!ok) {
            // instructions already issued may still read the operands and write the
            // accumulators: let them finish before memory is given up
            mma_commit_elect(bar_drain);
            wait_bar_drain(bar_drain, 0u);
        }
    } else if (warp < PW_WARP_E0) {
        // ---------------- expand the packed planes ---------------------------------
        const int group = (warp - PW_WARP_A0) / PW_A_GROUP;
        const int tid = threadIdx.x - (PW_WARP_A0 + group * PW_A_GROUP) * 32;
        constexpr int NT = PW_A_GROUP * 32;
        // own fills: g = group, group + 2, ...; slot = group
        const int slot = group;
        int ss = 0, pl = group;
        while (pl >= p.planes) { pl -= p.planes; ++ss; }
        ss %= p.stages;
        uint32_t phs = (uint32_t)((group / p.planes) / p.stages) & 1u, pha = 0;
        // first task (pixel, packed chunk) of this thread and the step to its next, in
        // a full plane and in the last one
        const int ch_full = p.PB / 16, ch_last = (p.P - (p.planes - 1) * p.PB) / 16;
        const int row_f = tid / ch_full, row_l = tid / ch_last, dr_f = NT / ch_full, dr_l = NT / ch_last;
        bool ok = true;
#pragma unroll 1
        for (uint32_t g = group; ok && g < n_fills; g += 2) {
            if (!(ok = wait_bar_warp(bar_st_full(ss), phs, ctl, 32))) break;
            if (!(ok = wait_bar_warp(bar_a_empty(slot), pha ^ 1u, ctl, 35))) break;
            const uint32_t src = smem_u32(smem + L.a_stage) + ss * stage_bytes + pl * plane_at;
            const uint32_t dst = smem_u32(smem + L.a_slots) + slot * a_slot_bytes;
            if (BITS == 3) {
                const int chunks = pl == p.planes - 1 ? ch_last : ch_full;
                const int groups = pw_groups<BITS>(p, pl);
#pragma unroll 1
                for (int row = tid; row < tile_px; row += NT) {
                    uint4 v[3];
#pragma unroll
                    for (int l = 0; l < 3; ++l) {
                        v[l] = make_uint4(0u, 0u, 0u, 0u);
                        if (l < chunks) v[l] = lds_128(src + row * px_bytes + 16u * l);
                    }
                    pw_store_row3<false>(dst + (uint32_t)row * 128u, row & 7, v, groups, 0u);
                }
            } else {
                // task = (pixel, packed chunk); a thread's next task is NT further
                const bool last = pl == p.planes - 1;
                const int chunks = last ? ch_last : ch_full;
                int row = last ? row_l : row_f, ch = tid - row * chunks;
                const int d_row = last ? dr_l : dr_f, d_ch = NT - d_row * chunks;
#pragma unroll 2
                while (row < tile_px) {
                    const uint4 v = lds_128(src + row * px_bytes + 16u * ch);
                    pw_store_chunk<BITS, false>(dst + (uint32_t)row * 128u, row & 7, ch, v, 0u);
                    row += d_row;
                    ch += d_ch;
                    if (ch >= chunks) { ch -= chunks; ++row; }
                }
            }
            fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) {
                mbar_arrive(bar_a_full(slot));
                mbar_arrive(bar_st_empty(ss));
            }
            pha ^= 1u;
            pl += 2;
            while (pl >= p.planes) {
                pl -= p.planes;
                if (++ss == p.stages) { ss = 0; phs ^= 1u; }
            }
        }
    } else {
        // ---------------- epilogue -------------------------------------------------
        const int quarter = warp & 3;
        const int group = (warp - PW_WARP_E0) / PW_E_GROUP;
        const int k = ((warp - PW_WARP_E0) % PW_E_GROUP) >> 2;
        const DsqLean lean = dsq_make_lean(p.e);
        // columns with a place in the output row; unit = 32 columns of a subtile, the
        // subtiles of the same columns next to each other
        const int cols = min(p.BN, p.out_pitch * 8 / BITS - n_tile * p.BN);
        const int col_units = (cols + 31) / 32, units = col_units * p.mt;
        const int u0 = k * units / PW_EPQ, u1 = (k + 1) * units / PW_EPQ;
        const int j = lane & 3;                       // eight channels 8 j .. of the 32
        unsigned long long sc[4], bi[4];
        int cu_held = -1;
        // (only the last N tile's columns end near the pitch)
        const int spare_from = n_tile == p.n_tiles - 1
                                   ? (n_tile * p.BN + col_units * 32) * BITS / 8 + 4 * j : p.out_pitch;
        bool ok = true;
#pragma unroll 1
        for (int it = group; ok && it < my_tiles; it += 2) {
            const int as = group;                     // accumulator of the own tiles
            const int m0 = (m_first + it * p.mstep) * tile_px + quarter * 32 + (lane >> 2);
            if (!(ok = wait_bar_warp(bar_acc_full(as), (it >> 1) & 1u, ctl, 36))) break;
            tc_fence_after_sync();
            int cu = u0 / p.mt, mt = u0 - cu * p.mt;
#pragma unroll 1
            for (int u = u0; u < u1; ++u) {
                uint32_t r[2][16];
                const uint32_t taddr = tmem_base + ((uint32_t)(quarter * 32) << 16) +
                                       (as * p.mt + mt) * p.BN + cu * 32;
                __syncwarp();
                tmem_ld_16x256b_x4(taddr, r[0]);
                tmem_ld_16x256b_x4(taddr + (16u << 16), r[1]);
                // this lane's bytes of an output row: BITS bytes at byte0
                const int byte0 = (n_tile * p.BN + cu * 32) * BITS / 8 + j * BITS;
                const int mr = m0 + mt * 128;         // + 8 i: this lane's pixels
                uint32_t res[4];
                if (RES) {
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        res[i] = 0u;
                        const uint8_t *rp = p.e.residual + (int64_t)(mr + 8 * i) * p.out_pitch + byte0;
                        if (mr + 8 * i >= p.M || byte0 >= p.out_pitch) continue;
                        if (BITS == 4) res[i] = __ldg(reinterpret_cast<const uint32_t *>(rp));
                        else if (BITS == 2) res[i] = __ldg(reinterpret_cast<const uint16_t *>(rp));
                        else {
                            // three bytes; the row's last lane may reach past its pitch
#pragma unroll
                            for (int b = 0; b < 3; ++b)
                                if (byte0 + b < p.out_pitch) res[i] |= (uint32_t)__ldg(rp + b) << (8 * b);
                        }
                    }
                }
                if (cu != cu_held) {
                    cu_held = cu;
                    const ulonglong2 *s2 = reinterpret_cast<const ulonglong2 *>(sm_scale + cu * 32 + 8 * j);
                    const ulonglong2 *b2 = reinterpret_cast<const ulonglong2 *>(sm_bias + cu * 32 + 8 * j);
                    sc[0] = s2[0].x; sc[1] = s2[0].y; sc[2] = s2[1].x; sc[3] = s2[1].y;
                    bi[0] = b2[0].x; bi[1] = b2[0].y; bi[2] = b2[1].x; bi[3] = b2[1].y;
                }
                tmem_ld_wait();
                uint32_t cw[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const uint32_t (&q)[16] = r[i >> 1];
                    const int o = 2 * (i & 1);
                    const uint32_t v[8] = {q[o],     q[o + 1], q[o + 4],  q[o + 5],
                                           q[o + 8], q[o + 9], q[o + 12], q[o + 13]};
                    cw[i] = dsq_lean_codes8<BITS, RES, LO>(v, sc, bi, RES ? res[i] : 0u, lean);
                }
                if (BITS == 2) {
                    // a word is two lanes' half words: even lanes store pixels 0 and 2's, odd
                    // lanes pixels 1 and 3's
                    const int odd = j & 1;
#pragma unroll
                    for (int i = 0; i < 4; i += 2) {
                        const uint32_t got =
                            __shfl_xor_sync(0xffffffffu, odd ? cw[i] : cw[i + 1], 1);
                        const uint32_t word = odd ? got | (cw[i + 1] << 16) : cw[i] | (got << 16);
                        const int m = mr + 8 * (i + odd), at = byte0 - 2 * odd;
                        if (m < p.M && at < p.out_pitch)
                            *reinterpret_cast<uint32_t *>(p.e.y_codes + (int64_t)m * p.out_pitch + at) = word;
                    }
                } else {
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const int m = mr + 8 * i;
                        uint32_t word = cw[i];
                        int at = byte0;
                        bool live = m < p.M;
                        if (BITS == 3) {
                            // the four lanes' 3 x 4 bytes as three words
                            const uint32_t nx = __shfl_down_sync(0xffffffffu, cw[i], 1);
                            word = (cw[i] >> (8 * j)) | (nx << (24 - 8 * j));
                            at = byte0 + j;
                            live &= j < 3;
                        }
                        uint8_t *row = p.e.y_codes + (int64_t)m * p.out_pitch;
                        if (live && at < p.out_pitch) *reinterpret_cast<uint32_t *>(row + at) = word;
                    }
                }
                // the last unit may end before the row's pitch does (by at most 12 bytes): a
                // word per lane (one lane for all of them took 5 to 10 us of 48)
                if (BITS != 4 && cu == col_units - 1 && spare_from < p.out_pitch) {
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        if (mr + 8 * i < p.M)
                            *reinterpret_cast<uint32_t *>(p.e.y_codes + (int64_t)(mr + 8 * i) * p.out_pitch +
                                                          spare_from) = 0u;
                }
                if (++mt == p.mt) { mt = 0; ++cu; }
            }
            tc_fence_before_sync();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_acc_empty(as));
        }
    }

    // ---------------- teardown ------------------------------------------------------
    tc_fence_before_sync();
    __syncthreads();
    if (warp == PW_WARP_MMA) {
        __syncwarp();
        tc_fence_after_sync();
        tmem_dealloc(tmem_base, (uint32_t)p.tmem_cols);
    }
}

template <int BITS, bool RES, bool LO>
int pw_launch(const CUtensorMap &ta, const PwParams &p, cudaStream_t s, int pdl)
{
    static std::atomic<unsigned long long> configured{0ull};
    const int st = dsq_allow_smem((const void *)dsq_pw_kernel<BITS, RES, LO>, 227 * 1024, &configured);
    if (st) return st;
    return dsq_launch(dsq_pw_kernel<BITS, RES, LO>, dim3(p.mstep * p.n_tiles), dim3(PW_THREADS),
                      (size_t)p.smem_bytes, s, pdl, 0, ta, p);
}

template <int BITS>
int pw_dispatch(const CUtensorMap &ta, const PwParams &p, cudaStream_t s, int pdl)
{
    if (p.e.rq.lo != 0.0f)
        return p.e.residual ? pw_launch<BITS, true, true>(ta, p, s, pdl)
                            : pw_launch<BITS, false, true>(ta, p, s, pdl);
    return p.e.residual ? pw_launch<BITS, true, false>(ta, p, s, pdl)
                        : pw_launch<BITS, false, false>(ta, p, s, pdl);
}

}  // namespace

int dsq_pointwise(const void *act_codes, const dsq_nhwc_t *shape, int bits, const void *w_packed,
                  const dsq_conv_t *conv, const DsqEpi &e, void *workspace, cudaStream_t stream)
{
    if (conv->KH != 1 || conv->KW != 1 || conv->pad != 0) return DSQ_ERR_UNSUPPORTED;
    const DsqLaunchHooks hooks = dsq_launch_hooks();
    PwParams p = {};
    p.stride = conv->stride;
    p.Ho = (shape->H - 1) / conv->stride + 1;
    p.Wo = (shape->W - 1) / conv->stride + 1;
    p.M = shape->N * p.Ho * p.Wo;                      // (at most 2^30, checked by the caller)
    p.K = conv->Cin;
    p.Ncols = conv->Cout;
    p.P = (int)dsq_row_pitch(p.K, bits);
    p.planes = (p.K + 127) / 128;
    p.PB = p.P < 16 * bits ? p.P : 16 * bits;
    p.out_pitch = (int)dsq_row_pitch(p.Ncols, bits);
    const int sms = dsq_sm_count();
    if (sms <= 0) return DSQ_ERR_CUDA;

    // Tiling: the cheapest in a model of the launch in clocks - per tile the slowest
    // of epilogue (25 elements a clock), expansion and instructions (120 clocks
    // each, whatever their N), plus the hand-offs; once per CTA its weights and the
    // fill of the pipeline.  Constants fitted for the choice, not rates it reaches: 112x112
    // 16->96 makes 9 elements a clock and SM in all, 16 would fill the issue slots
    // (8 instructions an element, counted).
    const int subtiles = (p.M + 127) / 128;
    const int groups = bits == 3 ? (p.K + 31) / 32 : p.P / 16 * (bits == 2 ? 2 : 1);
    double best = 0;
    const int max_n = (p.Ncols + 31) / 32;
    for (int nt = (p.Ncols + 255) / 256; nt <= max_n && nt <= sms; ++nt) {
        const int bn = ((p.Ncols + nt - 1) / nt + 31) / 32 * 32;
        if ((p.Ncols + bn - 1) / bn != nt) continue;
        for (int mt = 1; mt <= 4; mt *= 2) {
            if (2 * mt * bn > 512) break;
            int stages = PW_MAX_STAGES;
            const int row_bytes = p.stride == 1 ? p.P : p.planes * p.PB;
            while (stages >= 2 &&
                   pw_layout(mt, bn, p.planes, row_bytes, stages).total + 1024 > 227u * 1024u)
                --stages;
            if (stages < 2) break;
            const int m_tiles = (subtiles + mt - 1) / mt;
            const int mstep = m_tiles < sms / nt ? m_tiles : sms / nt;
            const int per_cta = (m_tiles + mstep - 1) / mstep;
            const double epi = mt * 128.0 * bn / 25, expand = mt * 2.3 * p.P + 400.0 * p.planes,
                         mma = mt * groups * 120.0;
            double tile = epi > expand ? epi : expand;
            tile = (tile > mma ? tile : mma) + 300;
            const double cost = per_cta * tile + epi + expand + mma + 0.02 * bn * p.P;
            if (best == 0 || cost < best) {
                best = cost;
                p.n_tiles = nt; p.BN = bn; p.mt = mt; p.stages = stages;
                p.m_tiles = m_tiles; p.mstep = mstep;
            }
        }
    }
    if (best == 0) return DSQ_ERR_UNSUPPORTED;         // the weights do not fit beside the rings
    p.tmem_cols = 32;
    while (p.tmem_cols < 2 * p.mt * p.BN) p.tmem_cols *= 2;
    p.box_rows = p.mt * 128 < 256 ? p.mt * 128 : 256;
    p.L = pw_layout(p.mt, p.BN, p.planes, p.stride == 1 ? p.P : p.planes * p.PB, p.stages);
    p.act = (const uint8_t *)act_codes;
    p.early = dsq_early_constants();
    p.smem_bytes = (int)p.L.total + 1024;
    p.shift = e.half_offset ? 7 - bits : 8 - bits;
    p.orv = e.half_offset ? 0x01010101u << (7 - bits) : 0u;
    p.wait_ns = hooks.wait_ns;
    p.e = e;
    p.w = (const uint8_t *)w_packed;
    p.ws = (int *)workspace;

    CUtensorMap ta;
    std::memset(&ta, 0, sizeof(ta));
    if (p.stride != 1) {
        DsqEncodeIm2colFn enc = dsq_encode_im2col_fn();
        if (!enc) return DSQ_ERR_CUDA;
        const cuuint64_t P = (cuuint64_t)p.P;
        cuuint64_t dims[4] = {P, (cuuint64_t)shape->W, (cuuint64_t)shape->H, (cuuint64_t)shape->N};
        cuuint64_t strides[3] = {P, P * shape->W, P * shape->W * shape->H};
        int lower[2] = {0, 0}, upper[2] = {0, 0};
        cuuint32_t estr[4] = {1, (cuuint32_t)p.stride, (cuuint32_t)p.stride, 1};
        if (enc(&ta, CU_TENSOR_MAP_DATA_TYPE_UINT8, 4, const_cast<void *>(act_codes), dims, strides,
                lower, upper, (cuuint32_t)p.PB, (cuuint32_t)p.box_rows, estr,
                CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return DSQ_ERR_UNSUPPORTED;
    }
    switch (bits) {
    case 2: return pw_dispatch<2>(ta, p, stream, hooks.pdl);
    case 3: return pw_dispatch<3>(ta, p, stream, hooks.pdl);
    default: return pw_dispatch<4>(ta, p, stream, hooks.pdl);
    }
}
