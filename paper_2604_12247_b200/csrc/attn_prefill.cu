// Tiled causal attention of the wide prefill passes on the tensor cores (Section 4.3: prefill is the base model's; bf16
// models): tcgen05 MMAs with the scores, the probabilities and the outputs in tensor memory.
//
// A CTA takes a tile of 128 prompt rows of ONE query head (one row per thread of its four softmax warps = one row per
// tensor-memory lane) and walks the cached positions 0 .. (last row's position) in blocks of 128:
//
//   scores   S = Q K^T : Q is fp32; it enters as its high and low bf16 halves (two MMAs into the same sums), so the
//                        product is as accurate as an fp32 one; K is the cached bf16 row, exact.
//   softmax            : a thread owns a row: running maximum and sum in fp32 registers, no shuffles
//   out      P V       : P enters as high + low bf16 halves (two MMAs), straight from tensor memory, where it takes the
//                        place of the scores it came from; V is the cached bf16 row.  Every block's product goes to a
//                        tensor-memory buffer of its own and is added to the row's fp32 sums in registers (rounded, where
//                        accumulating on in the tensor core over the whole context would truncate; and the rescaling by
//                        the running maximum needs no pass over tensor memory).
// The low halves' products go into a sum first: the tensor core truncates as it accumulates, and behind the high halves every
// step of the low ones would be cut at the size of the whole sum.  Hidden state of a 7B layer after 100 prompt rows against
// 64 bits: 9.2e-6 high halves first, 8.9e-6 low halves first (8.9e-6 in two sums of their own).
//
// Warp 0 brings the K and V blocks (TMA boxes of a page's rows, 128-byte swizzle, two stages each), warp 1 issues the
// MMAs: S of the next block goes in front of P V of the current one, so the tensor pipe works while the softmax warps
// (2-5) do.  Bound: the tensor pipe, 2048 clocks per 128 x 128 block of a head at 128 channels (half of it for the low
// halves), beside about 1100 issue slots and 1024 clocks of exponentials per softmax warp; measured, a block takes about 5300
// clocks, the softmax warps' own latencies.  512 rows of the 7B shape: 22 us per layer, against 64 us with 16 rows per CTA
// and 39 us with 64 rows per CTA on mma.sync (13-16 clocks per m16n8k16: the legacy path was the bound).
//
// Output: the bf16 high/low operand rows of the output projection, in the block-major layout of the wide GEMMs.  Rows,
// their rotated queries (fp32) and the pass's K/V rows come from k_rope_append, launched before.
#include "attn_common.cuh"
#include "tc_ptx.cuh"

namespace sb {

constexpr int kPfRows = 128;         // prompt rows per CTA: the lanes of tensor memory
constexpr int kPfBlock = 128;        // cached positions per block
constexpr int kPfThreads = 6 * 32;   // producer, MMA issuer, four softmax warps
constexpr int kPfHalf = 128 * 128;   // bytes of a 128-row x 64-channel operand tile (128-byte swizzle)
constexpr int kPfBars = 15;
constexpr size_t kPfOneCta = 116 * 1024;   // dynamic shared memory that two CTAs of an SM cannot both have (228 KB)

struct alignas(64) PrefillAttnArgs {
    CUtensorMap tmK, tmV;      // the layer's page pool as [rows][Hkv * HD], boxes of box_rows x 64 channels
    const __nv_bfloat16* v;    // the same pool as plain rows
    const float* q;            // [M][H * hd] rotated queries, row i at position pos0 + i
    const int* page_table;
    __nv_bfloat16* act_out;    // [block of 8 rows][16][H * hd]: high halves in rows 0-7, low halves in rows 8-15
    int H, Hkv, page, page_shift, box_rows;
    int pos0, M;
    unsigned int* status;      // device status word: a wait that runs out raises a code here
};

// 2^x (results below 2^-126 flush to zero: they are no part of a sum that holds a 1)
__device__ __forceinline__ float exp2_flush(float x) {
    float r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
// x and y as one register of two bf16 (x in the low half): the high parts, and what is left of each as a second register
__device__ __forceinline__ void split_pair(float x, float y, uint32_t& hi, uint32_t& lo) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(x, y);
    hi = *reinterpret_cast<const uint32_t*>(&h);
    const __nv_bfloat162 l = __floats2bfloat162_rn(x - __uint_as_float(hi << 16), y - __uint_as_float(hi & 0xffff0000u));
    lo = *reinterpret_cast<const uint32_t*>(&l);
}

template <int HD>
__global__ void __launch_bounds__(kPfThreads, 1) k_attn_prefill(const __grid_constant__ PrefillAttnArgs a) {
    constexpr int NH = HD / 64;                          // 64-channel halves of a row
    constexpr int kOp = NH * kPfHalf;                    // one Q (high or low), K or V block
    extern __shared__ uint8_t smem_raw[];
    __shared__ uint32_t tmem_base_s;
    __shared__ volatile int abort_s;
    __shared__ __align__(8) unsigned long long bars_s[kPfBars];
    __shared__ uint32_t not_finite_s[2][4];              // positions whose V row is not finite, in the (at most two) masked blocks

    const uint32_t raw = smem_u32(smem_raw), tiles = (raw + 1023u) & ~1023u;   // swizzled tiles need 1024-byte alignment
    uint8_t* const q_p = smem_raw + (tiles - raw);                             // [high | low] operand tiles of Q
    uint8_t* const v_p = q_p + 4 * kOp;
    const uint32_t q_s = tiles, k_s = q_s + 2 * kOp, v_s = k_s + 2 * kOp;      // two K blocks, two V blocks
    const uint32_t bars = smem_u32(bars_s);
    auto kfull = [&](int b) { return bars + 8u * b; };
    auto kempty = [&](int b) { return bars + 8u * (2 + b); };
    auto vfull = [&](int b) { return bars + 8u * (4 + b); };
    auto vempty = [&](int b) { return bars + 8u * (6 + b); };
    auto sfull = [&](int b) { return bars + 8u * (8 + b); };        // a block's scores complete
    auto ofull = [&](int b) { return bars + 8u * (10 + b); };       // a block's P V complete
    auto pready = [&](int b) { return bars + 8u * (12 + b); };      // a block's P in place (128 threads)
    const uint32_t qready = bars + 8u * 14;                         // Q in place (128 threads)

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int h = blockIdx.x, tile = (int)gridDim.y - 1 - (int)blockIdx.y;   // the tiles with the most positions start first
    const int kvh = h / (a.H / a.Hkv), qd = a.H * HD;
    const int row0 = tile * kPfRows;
    const int n_rows = min(kPfRows, a.M - row0);
    const int last_pos = a.pos0 + row0 + n_rows - 1;     // the tile's last row attends over 0 .. last_pos
    const int n_blocks = last_pos / kPfBlock + 1;
    if (threadIdx.x == 0) {
        abort_s = 0;
        for (int b = 0; b < 8; ++b) not_finite_s[b >> 2][b & 3] = 0u;
        for (int b = 0; b < 12; ++b) mbar_init(bars + 8u * b, 1);
        for (int b = 12; b < kPfBars; ++b) mbar_init(bars + 8u * b, 128);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(&a.tmK) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(&a.tmV) : "memory");
    }
    // Tensor memory only after everything before this kernel has completed, and the next kernel only after that: a CTA of
    // this kernel takes all of an SM's tensor memory, and must neither keep it from a GEMM that it waits for nor find it
    // taken by one that waits for it.
    pdl_wait();
    if (warp == 1) {   // S of two blocks (128 columns each, P in their place), P V of two blocks
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_s)), "r"(512u));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::);
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    pdl_trigger();
    const uint32_t tmem = tmem_base_s;
    auto s_col = [&](int b) { return tmem + 128u * b; };
    auto o_col = [&](int b) { return tmem + 256u + 128u * b; };
    auto turn = [](int blk) { return (uint32_t)(blk >> 1) & 1u; };   // parity of the use of a two-slot resource by block blk

    if (warp == 0) {
        // ------------------------------ producer ------------------------------
        if (lane == 0) {
            auto bring = [&](int blk, const CUtensorMap* tm, uint32_t dst, uint32_t full) {
                const int first = blk * kPfBlock, n = min(last_pos - first + 1, kPfBlock);
                const int boxes = (n + a.box_rows - 1) / a.box_rows;
                mbar_expect_tx(full, (uint32_t)(boxes * a.box_rows * NH * 128));
                for (int b = 0; b < boxes; ++b) {
                    const int t = first + b * a.box_rows;
                    const int row = a.page_table[t >> a.page_shift] * a.page + (t & (a.page - 1));
#pragma unroll
                    for (int hf = 0; hf < NH; ++hf)
                        tma_load_2d(dst + hf * kPfHalf + b * a.box_rows * 128, tm, kvh * HD + hf * 64, row, full);
                }
            };
            for (int blk = 0; blk < n_blocks; ++blk) {
                const int b = blk & 1;
                if (!mbar_wait(kempty(b), turn(blk) ^ 1u, &abort_s, a.status, 6u)) break;
                bring(blk, &a.tmK, k_s + b * kOp, kfull(b));
                if (!mbar_wait(vempty(b), turn(blk) ^ 1u, &abort_s, a.status, 6u)) break;
                bring(blk, &a.tmV, v_s + b * kOp, vfull(b));
            }
        }
    } else if (warp == 1) {
        // ------------------------------ MMA issuer ------------------------------
        if (lane == 0) {
            bool ok = mbar_wait(qready, 0, &abort_s, a.status, 7u);
            for (int blk = 0; blk <= n_blocks && ok; ++blk) {
                if (blk < n_blocks) {   // S(blk): its buffer held P(blk - 2), whose MMAs were issued before these
                    const int b = blk & 1;
                    if (!(ok = mbar_wait(kfull(b), turn(blk), &abort_s, a.status, 7u))) break;
                    tc_fence_after();
#pragma unroll
                    for (int part = 1; part >= 0; --part)            // low halves, high halves (see the head of the file)
#pragma unroll
                        for (int ks = 0; ks < HD / 16; ++ks) {
                            const uint32_t off = (uint32_t)((ks >> 2) * kPfHalf + (ks & 3) * 32);
                            tc_mma(s_col(b), smem_desc(q_s + part * kOp + off), smem_desc(k_s + b * kOp + off), idesc_n(kPfBlock),
                                   (part < 1 || ks > 0) ? 1u : 0u);
                        }
                    tc_commit(kempty(b));
                    tc_commit(sfull(b));
                }
                if (blk > 0) {          // P V of the block before; whoever wrote that P has read P V of the block two before it
                    const int pb = blk - 1, b = pb & 1;
                    if (!(ok = mbar_wait(pready(b), turn(pb), &abort_s, a.status, 7u))) break;
                    if (!(ok = mbar_wait(vfull(b), turn(pb), &abort_s, a.status, 7u))) break;
                    tc_fence_after();
#pragma unroll
                    for (int part = 1; part >= 0; --part)
#pragma unroll
                        for (int ks = 0; ks < kPfBlock / 16; ++ks)   // P: of 32 positions, 16 columns of high halves, then 16 of low halves
                            tc_mma_ts(o_col(b), s_col(b) + (uint32_t)((ks >> 1) * 32 + part * 16 + (ks & 1) * 8),
                                      smem_desc_mn(v_s + b * kOp + ks * 2048, kPfHalf), idesc_n(HD) | (1u << 16),
                                      (part < 1 || ks > 0) ? 1u : 0u);
                    tc_commit(vempty(b));
                    tc_commit(ofull(b));
                }
            }
        }
    } else {
        // ------------------------------ softmax: one row per thread ------------------------------
        const int quad = warp & 3;                       // the quarter of the lanes this warp may touch
        const int r = quad * 32 + lane;                  // row in the tile
        const uint32_t lanes = (uint32_t)(quad * 32) << 16;
        {   // Q: the warp's 32 rows, whole rows at a time (coalesced), split into halves and put into the swizzled operand
            // tiles; rows past the pass repeat the last one (never stored)
            constexpr int LPR = HD / 4, RPI = 32 / LPR;  // lanes per row, rows per step
            const int c = (lane % LPR) * 4, sub = lane / LPR;
#pragma unroll 8
            for (int i = 0; i < 32; i += RPI) {
                const int rr = quad * 32 + i + sub;
                const float4 v = *reinterpret_cast<const float4*>(a.q + (size_t)min(row0 + rr, a.M - 1) * qd + (size_t)h * HD + c);
                uint2 hi, lo;
                split_pair(v.x, v.y, hi.x, lo.x);
                split_pair(v.z, v.w, hi.y, lo.y);
                uint8_t* dst = q_p + (c >> 6) * kPfHalf + rr * 128 + ((((c & 63) >> 3) ^ (rr & 7)) << 4) + (c & 4) * 2;
                *reinterpret_cast<uint2*>(dst) = hi;
                *reinterpret_cast<uint2*>(dst + kOp) = lo;
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // read by the tensor core
            mbar_arrive(qready);
        }
        // a wait of the whole warp: the tensor-memory accesses behind it are collective
        auto warp_wait = [&](uint32_t bar, uint32_t parity) {
            return __all_sync(0xffffffffu, mbar_wait(bar, parity, &abort_s, a.status, 8u)) != 0;
        };
        // probabilities as powers of two of (score - maximum) * scale * log2 e, the difference first: its rounding is the
        // difference's own size, where scaled scores and maxima far from zero would each bring one of theirs, and the
        // rescaling factor of the sums uses the same differences
        const float scale2 = attn_score_scale(HD) * 1.4426950408889634f;
        const int my_pos = a.pos0 + row0 + r;
        float m = -INFINITY, l = 0.f, f_prev = 0.f;
        float acc[HD];
#pragma unroll
        for (int e = 0; e < HD; ++e) acc[e] = 0.f;
        // adds P V of a block to the row's sums, which f brings to that block's running maximum
        auto take = [&](int blk, float f) {
            if (!warp_wait(ofull(blk & 1), turn(blk))) return false;
            tc_fence_after();
#pragma unroll
            for (int c = 0; c < HD; c += 32) {
                uint32_t v[32];
                tc_ld32_nowait(o_col(blk & 1) + lanes + (uint32_t)c, v);
                tc_wait_ld();
#pragma unroll
                for (int e = 0; e < 32; ++e) acc[c + e] = fmaf(acc[c + e], f, __uint_as_float(v[e]));
            }
            return true;
        };
        bool ok = true;
        for (int blk = 0; blk < n_blocks; ++blk) {
            const bool masked = blk * kPfBlock + kPfBlock - 1 > a.pos0 + row0;
            if (masked) {
                // V rows that some row of the tile does not see: its probability is 0, and 0 * V must stay 0.  Thread r looks
                // at row r of the block: past the last position it may hold anything and becomes 0; of the others, channels
                // that are not finite become 0 and the position is remembered for the rows that do see it.  (In front of the
                // wait for the block's scores: the tensor core is at them.)
                if (!(ok = warp_wait(vfull(blk & 1), turn(blk)))) break;
                const int t = blk * kPfBlock + r;
                auto piece_p = [&](int piece) {
                    return reinterpret_cast<uint4*>(v_p + (blk & 1) * kOp + (piece >> 3) * kPfHalf + r * 128 + (((piece & 7) ^ (r & 7)) << 4));
                };
                bool finite = true;
                if (t > last_pos) {
#pragma unroll
                    for (int piece = 0; piece < NH * 8; ++piece) *piece_p(piece) = make_uint4(0u, 0u, 0u, 0u);
                } else if (t > a.pos0 + row0) {
                    const __nv_bfloat162 zero = __floats2bfloat162_rn(0.f, 0.f);
                    __nv_bfloat162 z[4] = {zero, zero, zero, zero};   // 0 * v + z: stays 0 until a v is not finite
#pragma unroll
                    for (int piece = 0; piece < NH * 8; ++piece) {
                        const uint4 w = *piece_p(piece);
                        z[0] = __hfma2(*reinterpret_cast<const __nv_bfloat162*>(&w.x), zero, z[0]);
                        z[1] = __hfma2(*reinterpret_cast<const __nv_bfloat162*>(&w.y), zero, z[1]);
                        z[2] = __hfma2(*reinterpret_cast<const __nv_bfloat162*>(&w.z), zero, z[2]);
                        z[3] = __hfma2(*reinterpret_cast<const __nv_bfloat162*>(&w.w), zero, z[3]);
                    }
                    z[0] = __hadd2(__hadd2(z[0], z[1]), __hadd2(z[2], z[3]));
                    finite = !(__hisnan(z[0].x) || __hisnan(z[0].y));
                    if (!finite) {
                        auto clean = [](uint32_t w) {
                            return ((w & 0x7f80u) == 0x7f80u ? 0u : w & 0xffffu) | ((w & 0x7f800000u) == 0x7f800000u ? 0u : w & 0xffff0000u);
                        };
#pragma unroll 1
                        for (int piece = 0; piece < NH * 8; ++piece) {
                            uint4 w = *piece_p(piece);
                            w.x = clean(w.x); w.y = clean(w.y); w.z = clean(w.z); w.w = clean(w.w);
                            *piece_p(piece) = w;
                        }
                    }
                }
                const uint32_t found = __ballot_sync(0xffffffffu, !finite);
                if (lane == 0) not_finite_s[n_blocks - 1 - blk][quad] = found;
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            }
            if (!(ok = warp_wait(sfull(blk & 1), turn(blk)))) break;
            tc_fence_after();
            const uint32_t s0 = s_col(blk & 1) + lanes;
            const int seen = my_pos - blk * kPfBlock + 1;   // visible positions of the block (maybe more than it has, or none)
            float mx = -INFINITY;
#pragma unroll 1
            for (int c = 0; c < kPfBlock; c += 32) {
                uint32_t v[32];
                tc_ld32_nowait(s0 + (uint32_t)c, v);
                tc_wait_ld();
                if (masked) {
#pragma unroll
                    for (int e = 0; e < 32; ++e) mx = c + e < seen ? fmaxf(mx, __uint_as_float(v[e])) : mx;
                } else {
#pragma unroll
                    for (int e = 0; e < 32; ++e) mx = fmaxf(mx, __uint_as_float(v[e]));
                }
            }
            const float nm = fmaxf(m, mx);
            const float f = nm > -INFINITY ? exp2_flush((m - nm) * scale2) : 1.f, top = nm > -INFINITY ? nm : 0.f;
            float ls[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 1
            for (int c = 0; c < kPfBlock; c += 32) {
                uint32_t v[32], p[32];
                tc_ld32_nowait(s0 + (uint32_t)c, v);
                tc_wait_ld();
#pragma unroll
                for (int e = 0; e < 32; e += 2) {
                    float p0 = exp2_flush((__uint_as_float(v[e]) - top) * scale2), p1 = exp2_flush((__uint_as_float(v[e + 1]) - top) * scale2);
                    if (masked) {
                        p0 = c + e < seen ? p0 : 0.f;
                        p1 = c + e + 1 < seen ? p1 : 0.f;
                    }
                    ls[e & 2] += p0;
                    ls[(e & 2) + 1] += p1;
                    split_pair(p0, p1, p[e >> 1], p[16 + (e >> 1)]);
                }
                tc_st32(s0 + (uint32_t)c, p);            // 16 columns of high halves, 16 of low halves, over the scores they came from
            }
            l = l * f + ((ls[0] + ls[1]) + (ls[2] + ls[3]));
            m = nm;
            tc_wait_st();
            tc_fence_before();                           // (and behind the loads of P V in the previous step)
            mbar_arrive(pready(blk & 1));
            if (blk > 0 && !(ok = take(blk - 1, f_prev))) break;
            f_prev = f;
        }
        if (ok) ok = take(n_blocks - 1, f_prev);
        asm volatile("bar.sync 1, 128;" ::: "memory");   // not_finite_s of all four warps (reached by each of them, whatever it waited for)
#pragma unroll 1
        for (int b = 0; b < 8; ++b) {
#pragma unroll 1
            for (uint32_t left = not_finite_s[b >> 2][b & 3]; left; left &= left - 1) {
                const int t = (n_blocks - 1 - (b >> 2)) * kPfBlock + (b & 3) * 32 + __ffs(left) - 1;
                if (t > my_pos) continue;                // (a visible channel that is not finite decides the sum: its weight does not matter)
                const uint32_t* row = reinterpret_cast<const uint32_t*>(
                    a.v + ((size_t)a.page_table[t >> a.page_shift] * a.page + (t & (a.page - 1))) * (a.Hkv * HD) + kvh * HD);
#pragma unroll
                for (int e = 0; e < HD; e += 2) {
                    const uint32_t w = __ldcg(row + (e >> 1));
                    if ((w & 0x7f80u) == 0x7f80u) acc[e] += __uint_as_float(w << 16);
                    if ((w & 0x7f800000u) == 0x7f800000u) acc[e + 1] += __uint_as_float(w & 0xffff0000u);
                }
            }
        }
        if (ok && r < n_rows) {
            const int row = row0 + r, blk8 = row / kMaxW, i = row - blk8 * kMaxW;
            __nv_bfloat16* dst = a.act_out + ((size_t)blk8 * 16 + i) * qd + (size_t)h * HD;
            const float inv = 1.f / l;
#pragma unroll
            for (int e = 0; e < HD; e += 8) {
                uint4 hi, lo;
                split_pair(acc[e] * inv, acc[e + 1] * inv, hi.x, lo.x);
                split_pair(acc[e + 2] * inv, acc[e + 3] * inv, hi.y, lo.y);
                split_pair(acc[e + 4] * inv, acc[e + 5] * inv, hi.z, lo.z);
                split_pair(acc[e + 6] * inv, acc[e + 7] * inv, hi.w, lo.w);
                *reinterpret_cast<uint4*>(dst + e) = hi;
                *reinterpret_cast<uint4*>(dst + (size_t)8 * qd + e) = lo;
            }
        }
    }

    if (abort_s) {   // a wait expired: give copies and MMAs still in flight time to land before leaving
        unsigned long long t0 = clock64();
        while (clock64() - t0 < 4000000ull) {}
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u));
    }
}

template <int HD> static bool launch_hd(cudaStream_t st, const PrefillAttnArgs& a) {
    // More than half of an SM's shared memory, also where half would do (64 channels): a CTA takes all of the SM's tensor memory,
    // and a second one on the SM would sit in its allocation, a wait without a limit, and hold back the next launch.
    const size_t tiles = (size_t)6 * (HD / 64) * kPfHalf + 1024, smem = tiles > kPfOneCta ? tiles : kPfOneCta;
    static bool configured[kMaxDevices];             // function attributes are per device
    const int dev = current_device();
    if (dev < 0) return false;
    if (!configured[dev]) {
        if (cudaFuncSetAttribute(k_attn_prefill<HD>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) return false;
        configured[dev] = true;
    }
    return launch_kc(k_attn_prefill<HD>, dim3(a.H, (a.M + kPfRows - 1) / kPfRows), dim3(kPfThreads), smem, st, 1, a) == cudaSuccess;
}

// q: [M][H * hd] fp32 (launch_rope_append ran before and appended the pass's K/V rows); act_out: wide operand layout
bool launch_attention_prefill(cudaStream_t st, const float* q, const void* k_cache, const void* v_cache, const int* page_table,
                              void* act_out, int H, int Hkv, int hd, int page, int page_shift, int n_pages, int pos0, int M,
                              unsigned int* status) {
    if (hd != 64 && hd != 128) return false;
    PrefillAttnArgs a;
    a.v = static_cast<const __nv_bfloat16*>(v_cache);
    a.q = q; a.page_table = page_table; a.act_out = static_cast<__nv_bfloat16*>(act_out);
    a.H = H; a.Hkv = Hkv; a.page = page; a.page_shift = page_shift; a.pos0 = pos0; a.M = M; a.status = status;
    a.box_rows = page < kPfBlock ? page : kPfBlock;   // rows of one page, at most a block (pages are powers of two of 16 rows or more)
    if (!make_map(&a.tmK, k_cache, n_pages * page, Hkv * hd, a.box_rows) || !make_map(&a.tmV, v_cache, n_pages * page, Hkv * hd, a.box_rows)) return false;
    return hd == 128 ? launch_hd<128>(st, a) : launch_hd<64>(st, a);
}

}  // namespace sb
