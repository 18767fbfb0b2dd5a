// GEMM of few rows: the launch streams the weights once and does little arithmetic, so what counts is how many SMs take
// part, the bytes each has in flight and the latency of one pass, not the tensor rate.  Included by gemm_tcgen05.cu, once per
// code type and polarity count.
//
// The operands change places: 128 output channels are the 128 rows of the MMA (the weight tile is its A operand) and the
// tokens are its columns, both polarities of a dual layer side by side in ONE operand (pos rows, then neg rows), so a K-step
// is one MMA of 128 x (8 .. 256) instead of two of 128 padded token rows each.  An accumulator is 128 lanes x (tokens x
// polarities) columns; those of all K-segments of a CTA's K range stay in tensor memory.
// A cluster of 2, 4 or 8 CTAs may split the K range of a tile: each leaves its raw int32 accumulators in the shared memory of
// the CTA that finishes the token (token t: rank t mod split), which adds up the pieces of a segment -- exact -- before it
// scales them, so results do not depend on the split.  e4m3 sums are fp32 and would, so their K range is never split.
// With SRC != 0 the CTA quantizes its activations itself (its tokens x its K range, once, into the MMA's swizzled layout in
// shared memory, kept for all its tiles) while the first weights are on their way: one launch per layer and no code matrices.
//   warps 0..7  quantizer (SRC != 0), then epilogue: thread = output channel, two groups of four warps share the tokens
//   warp 8      TMA producer; warp 9 MMA issuer and owner of the tensor memory
// A CTA asks for at most 113 KiB of shared memory where it can, so that two share an SM and the set-up of one launch runs
// under the end of the one before.  Two resident CTAs must never ask for more than the 512 columns of tensor memory an SM
// has: one would wait for the other, and with clusters round in a circle.  Hence smem_for_columns: shared memory grows with
// the columns so that what fits in shared memory fits in tensor memory, too.
// Measured against the tile form, which takes one CTA per 64 or 128 output columns (us, tile form / here, device time in a graph
// over rotating buffers; GEMM alone): 1 x 10912 -> 2320 dual int8 23.0 / 9.2, 9 x 6720 -> 1336 three segments 15.5 / 8.2,
// 283 x 9248 -> 384 24.2 / 10, 1 x 4672 -> 288 dual e4m3 11.4 / 7.5; whole layers, where the quantizer's launch goes as well (a
// call): 8 x 3072 -> 18432 dual e4m3 18.1 / 12.2 (weights at copy bandwidth 8.8), 256 x 256 -> 768 7.7 / 5.3.  120 random layers of 1 .. 128
// rows: GEMM 0.79, layer 0.79 of its time.

constexpr int kRowsWarps = 8;                          // quantizer / epilogue
constexpr int kRowsThreads = (kRowsWarps + 2) * 32;
[[maybe_unused]] constexpr int kRowsStages = 16, kRowsGroups = 16;

struct RowsHeader {
    uint64_t full[kRowsStages], empty[kRowsStages];
    uint64_t acc_full[2], acc_empty[2];
    uint64_t x_full;
    uint64_t act_ready[kRowsGroups];     // quantized activations, in order of K
    uint32_t tmem_base, abort_flag;
};

enum : uint32_t { kWhereRowsProducer = 0x500, kWhereRowsFull = 0x600, kWhereRowsAct = 0x700, kWhereRowsAcc = 0x800, kWhereRowsEpilogue = 0x900, kWhereRowsInput = 0xA00 };

__device__ __forceinline__ void tc_ld8(uint32_t taddr, uint32_t (&r)[8])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr) : "memory");
}
__device__ __forceinline__ void st_cluster_u32(uint32_t addr, uint32_t v)
{
    asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }

template <typename Tin>
__device__ __forceinline__ float ld_shared_elem(uint32_t base, int j)
{
    if (sizeof(Tin) == 4) return ld_shared_f32(base + 4u * uint32_t(j));
    unsigned short v;
    asm volatile("ld.shared.u16 %0, [%1];" : "=h"(v) : "r"(base + 2u * uint32_t(j)));
    return __uint_as_float(uint32_t(v) << 16);
}
template <int KIND>
__device__ __forceinline__ float acc_to_float(uint32_t v) { return KIND == 0 ? __int2float_rn(int(v)) : __uint_as_float(v); }

// SRC: where the activations come from: 0 code matrices through TMA, 1 bf16 and 2 fp32 inputs quantized here.
template <int KIND, int NPOL, int SRC>
__global__ void __launch_bounds__(kRowsThreads, 2)
segquant_rows_kernel(const __grid_constant__ CUtensorMap tm_pos, const __grid_constant__ CUtensorMap tm_neg,
                     const __grid_constant__ CUtensorMap tm_w, const __grid_constant__ RowsParams prm)
{
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    const uint32_t w_bytes = uint32_t(prm.tile_rows) * BLOCK_K, act_block = uint32_t(prm.ncols) * BLOCK_K;
    const uint32_t block_bytes = w_bytes + (SRC == 0 ? act_block : 0u), stage_bytes = uint32_t(prm.stage_blocks) * block_bytes;
    const int stage_blocks = prm.stage_blocks;
    // [ring] [(SRC != 0) codes of the tokens' K range] [(SRC != 0) their inputs] [factors] [partial sums of the cluster] [header]
    const uint32_t ring0 = smem_u32(smem);
    const uint32_t act0 = ring0 + uint32_t(prm.stages) * stage_bytes;
    const uint32_t x0 = act0 + prm.act_bytes;
    float *sh_tab = reinterpret_cast<float *>(smem + size_t(prm.stages) * stage_bytes + prm.act_bytes + prm.x_bytes);
    uint8_t *sh_red = reinterpret_cast<uint8_t *>(sh_tab) + prm.tab_bytes;
    RowsHeader *hdr = reinterpret_cast<RowsHeader *>(sh_red + (prm.red_alias ? 0u : prm.red_bytes));
    if (prm.red_alias) sh_red = smem;                   // the ring's memory, free once every MMA of the cluster has retired

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int split = KIND == 0 ? prm.split : 1;        // e4m3: no exchange is compiled
    const uint32_t rank = split > 1 ? cluster_rank() : 0u;
    const int unit = int(blockIdx.x) / split, units = int(gridDim.x) / split;
    const int mt = unit % prm.num_m, m0 = mt * prm.tile_tokens;
    const int rows = min(prm.tile_tokens, prm.M - m0);              // tokens of this CTA
    const int kb0 = int(rank) * prm.kblocks / split, kb1 = (int(rank) + 1) * prm.kblocks / split;
    const int p_first = prm.rank_p0[rank], p_last = prm.rank_p1[rank];
    const int P = prm.sb.P, Q = prm.sb.Q;
    const uint32_t abort_flag = smem_u32(&hdr->abort_flag);
    const uint32_t full0 = smem_u32(&hdr->full[0]), empty0 = smem_u32(&hdr->empty[0]);
    const uint32_t acc_full0 = smem_u32(&hdr->acc_full[0]), acc_empty0 = smem_u32(&hdr->acc_empty[0]);

    // (SRC != 0) the quantizer's 16-element chunks, K-block by K-block, one per thread and pass; one barrier per group of passes
    using Tin = typename std::conditional<SRC == 2, float, __nv_bfloat16>::type;
    constexpr int kBatch = kRowsWarps * 32;
    const int kbeg = kb0 * BLOCK_K, per_block = rows * 8;
    const int act_chunks = (kb1 - kb0) * per_block;
    const int act_group = (act_chunks + kRowsGroups * kBatch - 1) / (kRowsGroups * kBatch) * kBatch;
    if (warp == kRowsWarps) {
        if (lane == 0) {
            asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tm_w)) : "memory");
            if (SRC == 0) asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tm_pos)) : "memory");
            if (SRC == 0 && NPOL == 2) asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tm_neg)) : "memory");
        }
        if (lane < prm.stages) {
            mbar_init(full0 + 8 * lane, 1);
            mbar_init(empty0 + 8 * lane, 1);
        }
        if (lane < 2) {
            mbar_init(acc_full0 + 8 * lane, 1);
            mbar_init(acc_empty0 + 8 * lane, kRowsWarps);
        }
        if (lane == 2) mbar_init(smem_u32(&hdr->x_full), 1);
        if (lane < kRowsGroups) mbar_init(smem_u32(&hdr->act_ready[lane]), kRowsWarps);
        if (lane == 0) hdr->abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == kRowsWarps + 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(smem_u32(&hdr->tmem_base)), "r"(uint32_t(prm.tmem_cols)) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    grid_launch_dependents();           // not before this CTA has its tensor memory: the next launch may take some on this SM
    const uint32_t tmem_base = hdr->tmem_base;
    const uint32_t set_cols = uint32_t(p_last - p_first + 1) * prm.ncols;
    // first of the cluster's two barriers: the others have started (or, where partial sums go into the ring's memory, are
    // done with it); every thread arrives and waits
    if (split > 1 && !prm.red_alias) cluster_arrive();

    bool ok = true;
    if (warp == kRowsWarps) {
        // ------------------------------------------------------------------ TMA producer
        // the first weights into L2 while the kernel in front finishes: L2 holds what memory holds, whoever wrote it last
        for (int kb = kb0 + lane; kb < min(kb1, kb0 + prm.ahead); kb += 32)
            asm volatile("cp.async.bulk.prefetch.tensor.2d.L2.global.tile [%0, {%1, %2}];"
                         ::"l"(reinterpret_cast<uint64_t>(&tm_w)), "r"(kb * BLOCK_K), "r"(unit / prm.num_m * prm.tile_rows) : "memory");
        grid_dependency_wait();
        if (SRC != 0) {                  // the inputs, ahead of the weights: behind them they would wait for all of those
            const uint32_t len = uint32_t(min(kb1 * BLOCK_K, prm.K) - kbeg) * uint32_t(sizeof(Tin)), bar = smem_u32(&hdr->x_full);
            if (lane == 0) mbar_expect_tx(bar, len * uint32_t(rows));
            __syncwarp();
            for (int r = lane; r < rows; r += 32)
                asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                             ::"r"(x0 + uint32_t(r) * prm.x_pitch), "l"(static_cast<const Tin *>(prm.X) + size_t(m0 + r) * prm.ldx + kbeg),
                             "r"(len), "r"(bar) : "memory");
            __syncwarp();
        }
        uint32_t s = 0, ph = 0, issued = 0;
        for (int nt = unit / prm.num_m; nt < prm.num_n && ok; nt += units / prm.num_m) {
            for (int kb = kb0; kb < kb1; kb += stage_blocks) {
                if (!mbar_wait_warp(empty0 + 8 * s, ph ^ 1, abort_flag, prm.status, kWhereRowsProducer)) {
                    ok = false;
                    break;
                }
                const uint32_t bar = full0 + 8 * s;
                const int blocks = min(stage_blocks, kb1 - kb);
                if (elect_one()) {
                    mbar_expect_tx(bar, uint32_t(blocks) * block_bytes);
                    for (int b = 0; b < blocks; b++) {
                        const uint32_t dst = ring0 + s * stage_bytes + uint32_t(b) * block_bytes;
                        const int k = (kb + b) * BLOCK_K;
                        tma_load_2d<1>(dst, &tm_w, bar, k, nt * prm.tile_rows);
                        if (SRC == 0) {
                            tma_load_2d<1>(dst + w_bytes, &tm_pos, bar, k, m0);
                            if (NPOL == 2) tma_load_2d<1>(dst + w_bytes + act_block / 2, &tm_neg, bar, k, m0);
                        }
                    }
                }
                __syncwarp();
                issued++;
                if (++s == uint32_t(prm.stages)) { s = 0; ph ^= 1; }
            }
        }
        if (SRC != 0 && !ok) {
            const long long t0 = clock64();
            while (!mbar_try_wait(smem_u32(&hdr->x_full), 0) && clock64() - t0 < 200000000ll) {}
        }
        if (!ok) {                       // let the copies this thread issued land before the CTA's shared memory goes away
            const uint32_t pending = min(issued, uint32_t(prm.stages));
            for (uint32_t j = 0; j < pending; j++) {
                if (s == 0) { s = prm.stages; ph ^= 1; }
                s--;
                const long long t0 = clock64();
                while (!mbar_try_wait(full0 + 8 * s, ph) && clock64() - t0 < 200000000ll) {}
            }
        }
        __syncwarp();
    } else if (warp == kRowsWarps + 1) {
        // ------------------------------------------------------------------ MMA issuer
        const uint32_t idesc = make_idesc(KIND, prm.ncols, TILE_M);
        const uint64_t w_desc0 = make_smem_desc(ring0), act_desc0 = make_smem_desc(SRC == 0 ? ring0 + w_bytes : act0);
        const uint32_t hi = uint32_t(w_desc0 >> 32);
        uint32_t s = 0, ph = 0, as = 0, aph = 0;
        int act_groups = 0, act_have = 0;                          // groups and chunks of activations known to be there
        for (int nt = unit / prm.num_m; nt < prm.num_n && ok; nt += units / prm.num_m) {
            if (!mbar_wait_warp(acc_empty0 + 8 * as, aph ^ 1, abort_flag, prm.status, kWhereRowsAcc)) {
                ok = false;
                break;
            }
            tc_fence_after();
            int p = p_first, k_end = prm.sb.kb[p + 1];
            uint32_t accumulate = 0, d = tmem_base + as * set_cols;
            for (int kb = kb0; kb < kb1; kb += stage_blocks) {
                if (!mbar_wait_warp(full0 + 8 * s, ph, abort_flag, prm.status, kWhereRowsFull)) {
                    ok = false;
                    break;
                }
                const int blocks = min(stage_blocks, kb1 - kb);
                if (SRC != 0) {
                    const int need = (kb + blocks - kb0) * per_block;
                    while (act_have < need && ok) {
                        ok = mbar_wait_warp(smem_u32(&hdr->act_ready[act_groups++]), 0, abort_flag, prm.status, kWhereRowsAct);
                        act_have += act_group;
                    }
                    if (!ok) break;
                }
                tc_fence_after();
                uint32_t a_lo = uint32_t(w_desc0) + s * (stage_bytes >> 4);
                uint32_t b_lo = uint32_t(act_desc0) + (SRC == 0 ? s * (stage_bytes >> 4) : uint32_t(kb - kb0) * (act_block >> 4));
                int k = kb * BLOCK_K;
                const uint32_t b_step = (SRC == 0 ? block_bytes : act_block) >> 4;
                if (k + blocks * BLOCK_K <= k_end) {               // whole blocks of one K-segment
                    if (elect_one()) {
#pragma unroll 1
                        for (int b = 0; b < blocks; b++, a_lo += block_bytes >> 4, b_lo += b_step) {
                            issue_full_kblock<KIND, 1>(d, a_lo, b_lo, hi, idesc, accumulate);
                            accumulate = 1;
                        }
                        tc_commit<1>(empty0 + 8 * s);
                    }
                    accumulate = 1;
                    k += blocks * BLOCK_K;
                } else {                                           // K-steps lie in one segment each (bounds are multiples of 32)
                    for (int b = 0; b < blocks; b++, a_lo += block_bytes >> 4, b_lo += b_step) {
                        const int stop = min(k + BLOCK_K, prm.K);
                        for (uint32_t off = 0; k < stop; k += MMA_K, off += MMA_K >> 4) {
                            if (k >= k_end) { k_end = prm.sb.kb[++p + 1]; d += prm.ncols; accumulate = 0; }
                            if (elect_one())
                                tc_mma<KIND, 1>(d, uint64_t(hi) << 32 | (a_lo + off), uint64_t(hi) << 32 | (b_lo + off), idesc, accumulate);
                            accumulate = 1;
                        }
                    }
                    if (elect_one()) tc_commit<1>(empty0 + 8 * s);
                }
                if (k >= k_end && p < p_last) { k_end = prm.sb.kb[++p + 1]; d += prm.ncols; accumulate = 0; }
                if (++s == uint32_t(prm.stages)) { s = 0; ph ^= 1; }
            }
            if (ok && elect_one()) tc_commit<1>(acc_full0 + 8 * as);
            if (++as == uint32_t(prm.acc_sets)) { as = 0; aph ^= 1; }
        }
        __syncwarp();
    } else {
        // Every warp that reads global memory waits for the kernel in front itself, also where its inputs come through the producer's
        // copies: the scales may be what that kernel computes (a calibration lets this launch start with its first instruction
        // and writes them with its last).
        grid_dependency_wait();
        if constexpr (SRC != 0) {
            // -------------------------------------------------------------- quantizer: this CTA's tokens x its K range
            // not unrolled, see the epilogue.  (Each CTA quantizes for itself, so an element by itself and a division each, as the
            // quantize kernel has for a bound of -127, would count many times: 8 x 976 -> 616 dual took 7.9 us, 6.5 in two kernels.)
            constexpr int MODE = NPOL == 2 ? kDual : kSingle;
            int cur_p = p_first;
            SegConst cp = seg_const(__ldg(prm.s_pos + cur_p)), cn = seg_const(NPOL == 2 ? __ldg(prm.s_neg + cur_p) : 1.0f);
            ok = mbar_wait_agreed(smem_u32(&hdr->x_full), 0, abort_flag, prm.status, kWhereRowsInput);
#pragma unroll 1
            for (int i0 = 0; i0 < act_chunks && ok; i0 += kBatch) {
                const int i = i0 + int(threadIdx.x);
                if (i < act_chunks) {
                    const int blk = i / per_block, rest = i - blk * per_block, row = rest >> 3, piece = rest & 7;
                    const int k = kbeg + blk * BLOCK_K + piece * kVec;
                    const uint32_t src = x0 + uint32_t(row) * prm.x_pitch + uint32_t(k - kbeg) * uint32_t(sizeof(Tin));
                    // 128-byte rows, 128-byte swizzle, one block of ncols rows per K-block
                    const uint32_t dst = act0 + uint32_t(blk) * act_block + uint32_t(row) * BLOCK_K + (uint32_t(piece ^ (row & 7)) << 4);
                    uint32_t wp[4] = {}, wn[4] = {};
                    bool stored = false;
                    if (k < prm.K) {                               // K is a multiple of 16: a chunk is inside or outside
                        if (k >= prm.sb.kb[cur_p + 1]) {           // the thread's chunks ascend in K
                            do cur_p++;
                            while (k >= prm.sb.kb[cur_p + 1]);
                            cp = seg_const(__ldg(prm.s_pos + cur_p));
                            cn = seg_const(NPOL == 2 ? __ldg(prm.s_neg + cur_p) : 1.0f);
                        }
                        const bool fast = cp.fast && cn.fast;
                        Raw16<Tin> raw;
#pragma unroll
                        for (int v = 0; v < int(sizeof(Tin)); v++) {
                            uint4 w;
                            asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(w.x), "=r"(w.y), "=r"(w.z), "=r"(w.w) : "r"(src + 16u * v) : "memory");
                            set_piece(raw, v, w);
                        }
                        if (KIND == 0 && NPOL == 2) bound16(raw);
#pragma unroll
                        for (int g4 = 0; g4 < 4; g4++) {
                            float x[4];
                            get4(raw, g4, x);
                            if (fast) quant4<KIND, MODE, kBounded<Tin>>(x, cp, cn, float(prm.q_hi), 0, wp[g4], wn[g4]);
                        }
                        if (KIND == 0 && NPOL == 2 && prm.q_lo != -128) {      // a negative bound of -127: -128 becomes -127
#pragma unroll
                            for (int g4 = 0; g4 < 4; g4++) wn[g4] = __vmaxs4(wn[g4], 0x81818181u);
                        }
                        if (!fast) {
#pragma unroll 1
                            for (int j = 0; j < kVec; j++) {       // the codes go straight to their place, a byte at a time
                                uint32_t a, b;
                                quant1<KIND, MODE>(ld_shared_elem<Tin>(src, j), cp.s, cn.s, 0, prm.q_lo, prm.q_hi, a, b);
                                asm volatile("st.shared.u8 [%0], %1;" ::"r"(dst + uint32_t(j)), "r"(a) : "memory");
                                if (NPOL == 2) asm volatile("st.shared.u8 [%0], %1;" ::"r"(dst + act_block / 2 + uint32_t(j)), "r"(b) : "memory");
                            }
                            stored = true;
                        }
                    }
                    if (!stored)
                        asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(dst), "r"(wp[0]), "r"(wp[1]), "r"(wp[2]), "r"(wp[3]) : "memory");
                    if (NPOL == 2 && !stored)
                        asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(dst + act_block / 2), "r"(wn[0]), "r"(wn[1]), "r"(wn[2]), "r"(wn[3]) : "memory");
                }
                if ((i0 + kBatch) % act_group == 0 || i0 + kBatch >= act_chunks) {
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    __syncwarp();
                    if (lane == 0) mbar_arrive(smem_u32(&hdr->act_ready[i0 / act_group]));
                }
            }
        }
        // ------------------------------------------------------------------ epilogue
        // y = bias, then y = fma(c[a], acc[a], y) over a = (K-segment, polarity) ascending, as in the other form of the kernel
        const int ch = (warp & 3) * 32 + lane, group = warp >> 2;
        const bool per_token = prm.col_scale != nullptr;
        float *sh_row = sh_tab + (per_token ? P * prm.tile_rows : 0);            // token scales [rows][P * NPOL]
        uint32_t as = 0, aph = 0;
        if (per_token) {
            for (int i = threadIdx.x; i < rows * P; i += kRowsWarps * 32) {
                const int r = i / P, p = i - r * P;
                sh_row[i * NPOL] = __ldg(prm.row_pos + size_t(m0 + r) * P + p);
                if (NPOL == 2) sh_row[i * NPOL + 1] = __ldg(prm.row_neg + size_t(m0 + r) * P + p);
            }
        } else {
            for (int i = threadIdx.x; i < P * NPOL * Q; i += kRowsWarps * 32) {
                const int a = i / Q, q = i - a * Q, p = a / NPOL;
                sh_tab[i] = __ldg((NPOL == 2 && (a & 1) ? prm.s_neg : prm.s_pos) + p) * __ldg(prm.s_w + p * Q + q);
            }
        }
        for (int nt = unit / prm.num_m; nt < prm.num_n; nt += units / prm.num_m) {
            const int n = nt * prm.tile_rows + ch;
            const bool mine = ch < prm.tile_rows && n < prm.N;
            float bias = 0.0f;
            int q = 0;
            if (mine) {
                if (prm.bias) bias = __ldg(prm.bias + n);
                if (!per_token) while (q + 1 < Q && n >= prm.sb.nb[q + 1]) q++;
            }
            asm volatile("bar.sync 1, %0;" ::"n"(kRowsWarps * 32) : "memory");      // the previous tile's factors are read
            if (per_token)
                for (int p = group; p < P; p += 2)
                    if (ch < prm.tile_rows) sh_tab[p * prm.tile_rows + ch] = mine ? __ldg(prm.col_scale + size_t(n) * P + p) : 0.0f;
            asm volatile("bar.sync 1, %0;" ::"n"(kRowsWarps * 32) : "memory");
            const uint32_t cur = as;
            if (ok) ok = mbar_wait_agreed(acc_full0 + 8 * cur, aph, abort_flag, prm.status, kWhereRowsEpilogue);
            if (++as == uint32_t(prm.acc_sets)) { as = 0; aph ^= 1; }
            tc_fence_after();
            const uint32_t t_row = tmem_base + (uint32_t((warp & 3) * 32) << 16) + cur * set_cols;
            const bool warp_rows = (warp & 3) * 32 < prm.tile_rows;     // this warp's lanes hold channels of the tile

            const int mpad = prm.ncols / NPOL, nacc = P * NPOL;          // accumulator a of token t: column a * mpad + t
            const int es = prm.y_is_f32 ? 4 : 2;
            const long long ystep = prm.ldy * es;
            char *ytile = static_cast<char *>(prm.Y) + (size_t(m0) * prm.ldy + n) * es;
            auto dump = [&](int a, int tok, uint32_t v) {
                static_cast<uint32_t *>(prm.acc_dump)[(size_t(a) * prm.M + m0 + tok) * size_t(prm.N) + n] = v;
            };
            // The loops are kept short: a launch runs each of them a few times, so unrolled code is fetched about as often as it runs.
            if (split == 1) {
#pragma unroll 1
                for (int t0 = group * 8; t0 < rows && ok && warp_rows; t0 += 16) {
                    float y[8];
#pragma unroll
                    for (int j = 0; j < 8; j++) y[j] = bias;
#pragma unroll 1
                    for (int a0 = 0; a0 < nacc; a0 += 2) {         // two accumulators' loads in flight
                        uint32_t r[2][8];
                        __syncwarp();
                        tc_ld8(t_row + uint32_t(a0 * mpad + t0), r[0]);
                        if (NPOL == 2 || a0 + 1 < nacc) tc_ld8(t_row + uint32_t((a0 + 1) * mpad + t0), r[1]);
                        tc_wait_ld();
#pragma unroll
                        for (int h = 0; h < 2; h++) {
                            const int a = a0 + h;
                            if (NPOL == 1 && a >= nacc) break;
                            if (per_token) {
                                const float cs = sh_tab[(a / NPOL) * prm.tile_rows + ch];
                                const float *rs = sh_row + t0 * nacc + a;            // (tokens beyond the last: nothing of them is stored)
#pragma unroll
                                for (int j = 0; j < 8; j++)
                                    y[j] = fmaf(t0 + j < rows ? rs[j * nacc] * cs : 0.0f, acc_to_float<KIND>(r[h][j]), y[j]);
                            } else {
                                const float c = sh_tab[a * Q + q];
#pragma unroll
                                for (int j = 0; j < 8; j++) y[j] = fmaf(c, acc_to_float<KIND>(r[h][j]), y[j]);
                            }
                            if (prm.acc_dump && mine) {
#pragma unroll
                                for (int j = 0; j < 8; j++)
                                    if (t0 + j < rows) dump(a, t0 + j, r[h][j]);
                            }
                        }
                    }
                    if (mine) {
                        char *yp = ytile + t0 * ystep;
                        const int left = rows - t0;
                        if (prm.y_is_f32) {
#pragma unroll
                            for (int j = 0; j < 8; j++, yp += ystep)
                                if (j < left) *reinterpret_cast<float *>(yp) = y[j];
                        } else {
#pragma unroll
                            for (int j = 0; j < 8; j++, yp += ystep)
                                if (j < left) *reinterpret_cast<__nv_bfloat16 *>(yp) = __float2bfloat16_rn(y[j]);
                        }
                    }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(acc_empty0 + 8 * cur);
            } else {
                // ---- one tile per cluster.  Piece c = (rank, local segment) of token t, polarity pol goes to rank t mod split,
                // to word [c * NPOL + pol][t / split][channel]
                if (prm.red_alias) cluster_arrive();
                cluster_wait();
                const int lg = 31 - __clz(split), slots = (prm.tile_tokens + split - 1) >> lg;
                const uint32_t slot_bytes = uint32_t(prm.tile_rows) * 4u;
                int c = 0;
                for (int r = 0; r < int(rank); r++) c += prm.rank_p1[r] - prm.rank_p0[r] + 1;
                uint32_t to[8];                                    // token j of an aligned group of eight
#pragma unroll
                for (int j = 0; j < 8; j++)
                    to[j] = map_to_cta(smem_u32(sh_red) + uint32_t(ch) * 4u, uint32_t(j & (split - 1))) + uint32_t((j >> lg) + c * NPOL * slots) * slot_bytes;
#pragma unroll 1
                for (int t0 = group * 8; t0 < rows && ok && warp_rows; t0 += 16) {
#pragma unroll 1
                    for (int a = 0; a < (p_last - p_first + 1) * NPOL; a++) {
                        uint32_t r[8];
                        __syncwarp();
                        tc_ld8(t_row + uint32_t(a * mpad + t0), r);
                        tc_wait_ld();
                        const uint32_t off = uint32_t(a * slots + (t0 >> lg)) * slot_bytes;
#pragma unroll
                        for (int j = 0; j < 8; j++)
                            if (t0 + j < rows) st_cluster_u32(to[j] + off, r[j]);
                    }
                }
                cluster_arrive();
                cluster_wait();
                constexpr int T = 4;                               // tokens of this rank in flight per thread
                const int tokens = (rows - int(rank) + split - 1) >> lg;
#pragma unroll 1
                for (int tl0 = group * T; tl0 < tokens && ok && mine; tl0 += 2 * T) {
                    const uint32_t *red = reinterpret_cast<const uint32_t *>(sh_red) + size_t(tl0) * prm.tile_rows + ch;
                    float y[T];
                    uint32_t acc[NPOL][T];
#pragma unroll
                    for (int j = 0; j < T; j++) y[j] = bias;
                    bool fresh = true;
                    int p = 0, r = 0;
#pragma unroll 1
                    while (true) {
                        const bool last_of_rank = p == prm.rank_p1[r];
                        const bool last = !last_of_rank || r + 1 == split || prm.rank_p0[r + 1] != p;     // piece of this segment
#pragma unroll
                        for (int pol = 0; pol < NPOL; pol++, red += size_t(slots) * prm.tile_rows) {
#pragma unroll
                            for (int j = 0; j < T; j++) {
                                const uint32_t v = tl0 + j < tokens ? red[j * prm.tile_rows] : 0u;
                                acc[pol][j] = fresh ? v : acc[pol][j] + v;
                            }
                            if (last) {
                                const int a = p * NPOL + pol;
                                const float cs = per_token ? sh_tab[p * prm.tile_rows + ch] : sh_tab[a * Q + q];
#pragma unroll
                                for (int j = 0; j < T; j++) {
                                    const int tok = ((tl0 + j) << lg) + int(rank);
                                    if (tl0 + j < tokens) {
                                        y[j] = fmaf(per_token ? sh_row[tok * nacc + a] * cs : cs, acc_to_float<KIND>(acc[pol][j]), y[j]);
                                        if (prm.acc_dump) dump(a, tok, acc[pol][j]);
                                    }
                                }
                            }
                        }
                        fresh = last;
                        if (!last_of_rank) p++;
                        else if (r + 1 == split) break;
                        else p = prm.rank_p0[++r];
                    }
#pragma unroll
                    for (int j = 0; j < T; j++) {
                        if (tl0 + j >= tokens) break;
                        char *yp = ytile + (((tl0 + j) << lg) + int(rank)) * ystep;
                        if (prm.y_is_f32) *reinterpret_cast<float *>(yp) = y[j];
                        else *reinterpret_cast<__nv_bfloat16 *>(yp) = __float2bfloat16_rn(y[j]);
                    }
                }
            }
        }
    }
    if (split > 1 && warp >= kRowsWarps) {              // the other roles' part in the cluster's barriers
        if (prm.red_alias) cluster_arrive();
        cluster_wait();
        cluster_arrive();
        cluster_wait();
    }
    tc_fence_before();
    __syncthreads();
    if (warp == kRowsWarps + 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(uint32_t(prm.tmem_cols)) : "memory");
    }
}

// ----------------------------------------------------------------------------- host side

[[maybe_unused]] constexpr double kRowsAheadBytes = 8e6;       // weights fetched into L2 ahead of the dependency wait

// Shapes one launch may take; all of them give the same results.
struct RowsShape { int tile_tokens, tile_rows, split; };

// Shared memory that a CTA with that many columns of tensor memory has to ask for at least (see the top of this file).
inline size_t smem_for_columns(int cols) { return size_t(228) * 1024 * cols / 512 - 1024; }

// Microseconds of the model below that no shape avoids: the start and end of a launch, and the weights from memory.
[[maybe_unused]] constexpr double kRowsStart = 2.64, kRowsByteTime = 0.183e-6;
inline double rows_floor(const GemmArgs &g) { return kRowsStart + kRowsByteTime * double(g.N) * double(g.K); }

// Works out a launch of the given shape; false where it does not fit.  *cost: estimated cycles, for rows_plan.
template <int KIND, int NPOL>
bool rows_layout(const GemmArgs &g, const RowsShape &sh, int sm_count, RowsParams *out, size_t *smem, unsigned *grid, double *cost)
{
    RowsParams &r = *out;
    const int split = sh.split, kblocks = int((g.K + BLOCK_K - 1) / BLOCK_K);
    const bool fused = g.X != nullptr, per_token = g.col_scale != nullptr;
    if (sh.tile_rows < 32 || sh.tile_rows > 128 || sh.tile_rows % 32 || split < 1 || split > 8 || (split & (split - 1))) return false;
    if (split > kblocks || (KIND != 0 && split > 1)) return false;
    r.tile_tokens = int(std::min<int64_t>(sh.tile_tokens, g.M));
    r.ncols = NPOL == 2 ? 2 * ((r.tile_tokens + 7) / 8 * 8) : (r.tile_tokens + 15) / 16 * 16;
    if (r.ncols > 256) return false;
    r.tile_rows = sh.tile_rows;
    r.split = split;
    r.kblocks = kblocks;
    r.num_m = int((g.M + r.tile_tokens - 1) / r.tile_tokens);
    r.num_n = int((g.N + r.tile_rows - 1) / r.tile_rows);
    int pieces = 0, most = 0, longest = 0;
    for (int i = 0; i < split; i++) {
        const int kb0 = i * kblocks / split, kb1 = (i + 1) * kblocks / split;
        const int64_t k0 = int64_t(kb0) * BLOCK_K, k1 = std::min<int64_t>(int64_t(kb1) * BLOCK_K, g.K);
        int p = 0;
        while (k0 >= g.sb.kb[p + 1]) p++;
        r.rank_p0[i] = p;
        while (k1 > g.sb.kb[p + 1]) p++;
        r.rank_p1[i] = p;
        pieces += r.rank_p1[i] - r.rank_p0[i] + 1;
        most = std::max(most, r.rank_p1[i] - r.rank_p0[i] + 1);
        longest = std::max(longest, kb1 - kb0);
    }
    if (most * r.ncols > kTmemCols) return false;
    r.tab_bytes = uint32_t(per_token ? g.sb.P * (r.tile_rows + r.tile_tokens * NPOL) : g.sb.P * NPOL * g.sb.Q) * 4u;
    r.tab_bytes = (r.tab_bytes + 15u) & ~15u;
    if (r.tab_bytes > 32 * 1024) return false;
    const uint32_t act_block = uint32_t(r.ncols) * BLOCK_K;
    r.act_bytes = fused ? uint32_t(longest) * act_block : 0u;
    const int es = g.x_dtype == SQ_F32 ? 4 : 2;
    r.x_pitch = fused ? uint32_t(longest) * BLOCK_K * es + 16u : 0u;       // rows 16 bytes apart in their banks
    r.x_bytes = (r.x_pitch * r.tile_tokens + 127u) & ~127u;
    r.red_bytes = split > 1 ? uint32_t(pieces * NPOL * ((r.tile_tokens + split - 1) / split) * r.tile_rows) * 4u : 0u;
    r.red_alias = r.red_bytes > 16 * 1024;
    const size_t block = size_t(r.tile_rows) * BLOCK_K + (fused ? 0u : act_block);
    // behind the ring: what follows, and at least what an MMA reads behind a tile of fewer than 128 rows
    const size_t fixed = 1024 + std::max<size_t>(r.act_bytes + r.x_bytes + r.tab_bytes + (r.red_alias ? 0u : r.red_bytes) + sizeof(RowsHeader),
                                                 size_t(TILE_M - r.tile_rows) * BLOCK_K);
    // K-blocks per ring stage: a wait, an election and a commit per stage cost the issuing loop some 75 ns (ns per block with 1, 2 and
    // 4 blocks a stage: 233, 146, 115); as many as the length of the K range and three stages allow.  Two CTAs per SM where three
    // stages fit half of its shared memory.
    auto ring = [&](size_t budget) {
        for (r.stage_blocks = longest >= 16 ? 4 : longest >= 4 ? 2 : 1; r.stage_blocks > 0; r.stage_blocks /= 2) {
            const int turns = (longest + r.stage_blocks - 1) / r.stage_blocks;
            const size_t stage = r.stage_blocks * block;
            r.stages = fixed + 2 * stage > budget ? 0 : int(std::min<size_t>((budget - fixed) / stage, kRowsStages));
            if (r.stages >= std::min(3, turns)) return turns;
        }
        return 0;
    };
    constexpr size_t kTwo = 113 * 1024, kOne = kSmemBudget;
    int per_sm = 2, turns = ring(kTwo);
    if (!turns) { turns = ring(kOne); per_sm = 1; }
    if (!turns) return false;
    const int64_t slots = int64_t(sm_count) * per_sm / split;
    if (slots < 1) return false;
    const int64_t per_m = split > 1 ? r.num_n : std::min<int64_t>(r.num_n, std::max<int64_t>(1, slots / r.num_m));
    *grid = unsigned(per_m * r.num_m * split);
    const int tiles_per_cta = int((r.num_n + per_m - 1) / per_m);
    if (per_sm == 2 && int(*grid) <= sm_count && turns * tiles_per_cta > r.stages) {
        // a CTA per SM and more blocks than that ring holds: a deeper one counts for more than the next launch's early start
        turns = ring(kOne);
        per_sm = 1;
    }
    const size_t stage = r.stage_blocks * block;
    if (tiles_per_cta == 1 && r.stages > turns) r.stages = std::max(2, turns);
    if (r.red_alias && r.red_bytes > r.stages * stage + r.act_bytes + r.x_bytes) return false;
    r.acc_sets = tiles_per_cta > 1 && 2 * most * r.ncols <= kTmemCols / per_sm ? 2 : 1;
    r.tmem_cols = 32;
    while (r.tmem_cols < r.acc_sets * most * r.ncols) r.tmem_cols *= 2;
    *smem = std::max(r.stages * stage + fixed, smem_for_columns(r.tmem_cols));
    if (*smem > kOne) return false;

    // microseconds, a model fitted to some 5000 timings of forced shapes (M 1 .. 300, K 256 .. 12288, N 256 .. 18432, up to 24
    // K-segments; half of them within 5 %, nine in ten within 18 %): weights from memory; the K loop, bound by the issuing loop,
    // the MMAs or the bytes that reach an SM; the quantizer's passes; accumulators per warp; the exchange of a split tile.
    static constexpr int kClusters[2][4] = {{148, 148, 132, 120}, {296, 296, 284, 264}};      // CTAs of 148 SMs, 1 and 2 per SM, by log2 split
    const int lg = split == 1 ? 0 : split == 2 ? 1 : split == 4 ? 2 : 3;
    const int capacity = std::max(split, kClusters[*smem > kTwo ? 0 : 1][lg] * sm_count / 148);
    const int resident = std::min(int(*grid), capacity), waves = (int(*grid) + capacity - 1) / capacity;
    const double per_sm_now = (resident + sm_count - 1) / sm_count, blocks = double(waves) * tiles_per_cta * longest;
    const double bytes = double(r.tile_rows + (fused ? 0 : r.ncols)) * BLOCK_K, g16 = (r.tile_tokens + 15) / 16;
    const double busy = per_sm_now > 1 ? 1.62 : 1.0, busy_half = per_sm_now > 1 ? 1.41 : 1.0;        // two CTAs on an SM
    const double quant = fused ? (KIND == 0 ? 0.31 : 0.49) + 0.4675 * ((r.tile_tokens * longest * 8 + 255) / 256) * busy : 0.0;
    const double per_block = std::max((r.stage_blocks == 4 ? 0.133 : r.stage_blocks == 2 ? 0.164 : 0.262) + 1.75e-4 * r.ncols * per_sm_now,
                                      6.8e-6 * bytes * per_sm_now);
    const double chain = blocks * per_block + waves * quant, memory = kRowsByteTime * double(g.N) * double(g.K) + (fused ? 0.27 : 0.0);
    const double stream = std::max(std::max(memory, chain), 0.04e-6 * resident * blocks * bytes + quant);
    const double epi = 0.148 * most * NPOL * g16 * busy_half + 0.157 * g16;
    const double comb = split > 1 ? 0.894 + 0.129 * pieces * NPOL * (((r.tile_tokens + split - 1) / split + 7) / 8) + 0.082 * most * NPOL * g16 : 0.0;
    *cost = kRowsStart + stream + waves * (tiles_per_cta * epi + comb) + (waves - 1) * 2.95;
    r.ahead = int(std::min<double>(longest, std::max(0.0, std::ceil(kRowsAheadBytes / (double(*grid) * r.tile_rows * BLOCK_K)))));
    return true;
}

// Where the model above falls short of the tile form's, in microseconds on top of it for a shape that has been picked.  900 layers of
// 1 .. 512 rows, GEMM alone, time here over time of the tile form; K-blocks are cut where a segment ends inside their ring
// stage, and are then issued MMA by MMA, which shows unless the weights take longer to arrive:
//   at least 12 cut blocks a CTA, one polarity: 0.86 .. 1.12, 1.00 in the median of 12 layers (8448 wide in 22 segments, 101 rows, 25.6 / 22.8);
//   at least 28, two polarities of e4m3, whose K range is not split: 1.06 .. 1.21 (4992 in 13 segments, 4 rows, 16.2 / 13.9);
//   with fewer, or of int8, 0.75 .. 0.93 (nine in ten);
//   one polarity, several token tiles, each of which reads the weights: 1.00 .. 1.20 for 20 MB of weights and more where the tile
//   form's 128-column tiles occupy 64 SMs (42 x 8016 -> 8936 19.7 / 16.4), 0.63 .. 0.95 where they do not (31 x 10192 -> 3392).
template <int KIND, int NPOL>
double rows_shortfall(const GemmArgs &g, const RowsParams &r, unsigned grid)
{
    if (NPOL == 1 && r.num_m > 1 && g.M <= TILE_M && g.N >= 64 * 128 && double(g.N) * double(g.K) >= 20e6) return 1e9;
    const int64_t stage = int64_t(r.stage_blocks) * BLOCK_K;
    int most = 0;
    for (int i = 0; i < r.split; i++) {
        const int kb0 = i * r.kblocks / r.split, kb1 = (i + 1) * r.kblocks / r.split;
        int64_t last = -1;
        int cut = 0;
        for (int p = r.rank_p0[i] + 1; p <= r.rank_p1[i]; p++) {
            const int64_t off = g.sb.kb[p] - int64_t(kb0) * BLOCK_K;
            if (off % stage == 0 || off / stage == last) continue;
            last = off / stage;
            cut += std::min(r.stage_blocks, kb1 - kb0 - int(last) * r.stage_blocks);
        }
        most = std::max(most, cut);
    }
    if (most < (NPOL == 1 ? 12 : 28) || (NPOL == 2 && KIND == 0)) return 0.0;
    const int per_m = int(grid) / r.num_m / r.split, tiles = (r.num_n + per_m - 1) / per_m;
    const double idle = kRowsByteTime * double(g.N) * double(g.K) - 0.133 * tiles * r.kblocks / r.split;        // the issuing loop's, uncut
    return std::max(0.0, (NPOL == 1 ? 0.16 : 0.12) * most * tiles - std::max(0.0, idle));
}

// The best shape for a layer and the time the models give it; false where none fits.  Working it out takes 1.2 (8 rows) to 6.2 us
// (250 rows) of a call that takes 5 to 10, so a thread keeps what it has decided, a function of sizes and segment bounds alone.
// An eager call asks two or three times (quantizing inside or not), so 256 decisions serve some eighty layers in rotation.
struct RowsKey {
    int64_t M, N, K;
    int P, Q, fused, x_f32, per_token, sm_count;
    uint16_t kb[SQ_MAX_P + 1];           // interior bounds are multiples of 32, K of 16 and at most 131072
    bool operator==(const RowsKey &o) const
    {
        return M == o.M && N == o.N && K == o.K && P == o.P && Q == o.Q && fused == o.fused && x_f32 == o.x_f32 &&
               per_token == o.per_token && sm_count == o.sm_count && std::equal(kb, kb + P + 1, o.kb);
    }
    uint32_t hash() const
    {
        int64_t w[8 + SQ_MAX_P] = {M, N, K, int64_t(P) << 32 | Q, fused << 2 | x_f32 << 1 | per_token, sm_count};
        size_t n = 6;
        for (int p = 1; p < P; p++) w[n++] = kb[p];
        return hash_words(w, n);
    }
};
struct RowsDecision {
    bool found;
    RowsShape shape;
    double cost;
};

template <int KIND, int NPOL>
RowsDecision rows_search(const GemmArgs &g, int sm_count, bool forced)
{
    RowsDecision best{};
    const int f_rows = forced ? g_tune_tile_n.load(std::memory_order_relaxed) : 0, f_tokens = forced ? g_tune_stages.load(std::memory_order_relaxed) : 0,
              f_split = forced ? g_tune_cta_group.load(std::memory_order_relaxed) : 0;
    RowsParams r{};
    size_t smem = 0;
    unsigned grid = 0;
    for (int tokens : {8, 16, 32, 64, 128, 256}) {
        if (tokens > 8 && tokens / 2 >= g.M && !forced) break;
        for (int rows : {128, 96, 64, 32})
            for (int split : {1, 2, 4, 8}) {
                if ((f_rows && rows != f_rows) || (f_tokens && tokens != f_tokens) || (f_split && split != f_split)) continue;
                double c = 0.0;
                if (!rows_layout<KIND, NPOL>(g, {tokens, rows, split}, sm_count, &r, &smem, &grid, &c)) continue;
                if (best.found && c >= best.cost) continue;
                best = {true, {tokens, rows, split}, c};
            }
    }
    if (best.found && !forced) {
        rows_layout<KIND, NPOL>(g, best.shape, sm_count, &r, &smem, &grid, &best.cost);
        best.cost += rows_shortfall<KIND, NPOL>(g, r, grid);
    }
    return best;
}

template <int KIND, int NPOL>
RowsDecision rows_plan(const GemmArgs &g, int sm_count)
{
    if (g_tune_seq.load(std::memory_order_relaxed) == kSegmentModeRows) return rows_search<KIND, NPOL>(g, sm_count, true);
    thread_local Recent<RowsKey, RowsDecision, 8, 32> kept;
    RowsKey key{};
    key.M = g.M; key.N = g.N; key.K = g.K;
    key.P = g.sb.P; key.Q = g.sb.Q;
    key.fused = g.X != nullptr;
    key.x_f32 = key.fused && g.x_dtype == SQ_F32;
    key.per_token = g.col_scale != nullptr;
    key.sm_count = sm_count;
    for (int p = 0; p <= g.sb.P; p++) key.kb[p] = uint16_t(g.sb.kb[p] / 16);
    const uint32_t hash = key.hash();
    if (const RowsDecision *d = kept.find(hash, key)) return *d;
    return kept.keep(hash, key, rows_search<KIND, NPOL>(g, sm_count, false));
}

template <int KIND, int NPOL>
sq_status prepare_rows_t(const GemmArgs &g, GemmLaunch &L, double limit, int device, int sm_count)
{
    RowsParams &r = L.rows;
    r = RowsParams{};
    const bool forced = g_tune_seq.load(std::memory_order_relaxed) == kSegmentModeRows;
    if (!forced && rows_floor(g) >= limit) return SQ_ERR_UNSUPPORTED;      // no shape can be the better one: nothing to search
    const RowsDecision d = rows_plan<KIND, NPOL>(g, sm_count);
    if (!d.found || d.cost >= limit) return SQ_ERR_UNSUPPORTED;
    if (g.X && !forced) {      // quantizing here also has to beat this form behind a quantizer of its own
        GemmArgs codes = g;
        codes.X = nullptr;
        const RowsDecision apart = rows_plan<KIND, NPOL>(codes, sm_count);
        if (apart.found && d.cost >= rows_gain(g.M, g.K, true) * (apart.cost + kQuantizeLaunch)) return SQ_ERR_UNSUPPORTED;
    }
    double cost = 0.0;
    rows_layout<KIND, NPOL>(g, d.shape, sm_count, &r, &L.smem, &L.grid, &cost);
    r.M = int(g.M); r.N = int(g.N); r.K = int(g.K);
    r.sb = g.sb;
    r.s_pos = g.s_pos; r.s_neg = g.s_neg; r.s_w = g.s_w; r.bias = g.bias;
    r.row_pos = g.row_pos; r.row_neg = g.row_neg; r.col_scale = g.col_scale;
    r.Y = g.Y; r.ldy = g.ldy; r.y_is_f32 = g.y_dtype == SQ_F32;
    r.acc_dump = g.acc_dump;
    r.status = g.status;
    r.X = g.X; r.ldx = g.ldx; r.q_lo = g.q_lo; r.q_hi = g.q_hi;
    if (!make_map(&L.tb, g.b, g.N, g.K, g.ldb, r.tile_rows)) return SQ_ERR_CUDA;
    const void *kern;
    if (g.X) {
        L.ta = L.tn = CUtensorMap{};
        kern = g.x_dtype == SQ_F32 ? reinterpret_cast<const void *>(segquant_rows_kernel<KIND, NPOL, 2>)
                                   : reinterpret_cast<const void *>(segquant_rows_kernel<KIND, NPOL, 1>);
    } else {
        if (!make_map(&L.ta, g.a_pos, g.M, g.K, g.lda, r.ncols / NPOL)) return SQ_ERR_CUDA;
        L.tn = L.ta;
        if (NPOL == 2 && !make_map(&L.tn, g.a_neg, g.M, g.K, g.lda, r.ncols / NPOL)) return SQ_ERR_CUDA;
        kern = reinterpret_cast<const void *>(segquant_rows_kernel<KIND, NPOL, 0>);
    }
    int clusters = 0;
    const sq_status fs = kernel_facts(device, kern, L.smem, 1, cudaLaunchConfig_t{}, &clusters);
    if (fs != SQ_OK) return fs;
    L.kernel = kern;
    L.cluster = unsigned(r.split);
    L.threads = kRowsThreads;
    L.few_rows = 1;
    L.device = device;
    return SQ_OK;
}
