// Block-quantized (INT8 / INT4) shard weights for decode: the host quantizer and packer, and the
// dequantizing matrix-vector kernel, sm_103a.
//
// What they compute (Voltron Section 3.2.2, precision heterogeneity: a device may hold its shard
// at a reduced precision; Section 4.2.2 allocates precisions per layer; Section 5.1 names k-quant
// formats without defining them).  Format: each weight row is cut into blocks of 32 consecutive
// weights along the input axis; a block keeps the fp16 scale d = fp16(amax / qmax) (qmax 127 for
// 8 bits, 7 for 4 bits) and every weight the code q = round-half-even(w / d) clamped to
// [-qmax, qmax] (0 when d = 0), both divisions in fp32.  A projection is y = sum_e (q_e d) x_e.
//
// The kernel keeps the codes as integers and multiplies them on the tensor cores (codes and
// an exact three-digit split of the input as whole numbers in fp16, whose products and sums in fp32
// are exact), so the work per code is a small fraction of an instruction (details at the kernel).
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>
#include <cmath>

#include "device.cuh"
#include "internal.h"

namespace vt {

// ================================================================== host: quantizer and packer

void quantize_rows_host(const __half* w, int64_t rows, int64_t k, int bits, int block, int8_t* q, __half* scales) {
    const int qmax = bits == 8 ? 127 : 7;
    const int64_t nb = (k + block - 1) / block;
    for (int64_t r = 0; r < rows; ++r)
        for (int64_t b = 0; b < nb; ++b) {
            const int64_t e0 = b * block, e1 = std::min(k, e0 + block);
            float amax = 0.0f;
            for (int64_t e = e0; e < e1; ++e) amax = std::max(amax, std::fabs(__half2float(w[r * k + e])));
            const __half d16 = __float2half_rn(amax / (float)qmax);  // fp32 division, one rounding to fp16
            const float d = __half2float(d16);
            scales[r * nb + b] = d16;
            for (int64_t e = e0; e < e1; ++e) {
                int c = 0;
                if (d != 0.0f) {
                    const float x = std::nearbyint(__half2float(w[r * k + e]) / d);  // fp32 division, ties to even
                    c = x > (float)qmax ? qmax : (x < (float)-qmax ? -qmax : (int)x);
                }
                q[r * k + e] = (int8_t)c;
            }
        }
}

static int64_t qmat_nb(int64_t k) { return (k + kQBlock - 1) / kQBlock; }

static int64_t qmat_rows(int64_t rows) { return (rows + kQTile - 1) / kQTile * kQTile; }  // whole row tiles

size_t qmat_code_bytes(int64_t rows, int64_t k, int bits) {
    return (size_t)qmat_rows(rows) * (size_t)qmat_nb(k) * (bits == 8 ? 32 : 16);
}

size_t qmat_scale_bytes(int64_t rows, int64_t k) { return (size_t)qmat_rows(rows) * (size_t)qmat_nb(k) * 2; }

// Byte offset of the codes of row r, block b, positions 8t .. 8t + 7, and index of the row's scale
// (the layout of QMatDev).
static __host__ __device__ __forceinline__ size_t qcode_at(int64_t r, int64_t b, int t, int64_t nb, int bits) {
    const int64_t tile = r / kQTile, g = r % 8, high = r / 8 % 2;
    return (size_t)(((tile * nb + b) * 32 + 4 * g + t) * 2 + high) * (bits == 8 ? 8 : 4);
}
static __host__ __device__ __forceinline__ size_t qscale_at(int64_t r, int64_t b, int64_t nb) {
    return (size_t)((r / kQTile * nb + b) * kQTile + r % 8 * 2 + r / 8 % 2);
}

void unpack_qmat(const uint8_t* codes, const __half* scales, int64_t rows, int64_t k, int bits, int8_t* q, __half* out) {
    const int64_t nb = qmat_nb(k);
    for (int64_t r = 0; r < rows; ++r) {
        for (int64_t b = 0; b < nb; ++b) out[r * nb + b] = scales[qscale_at(r, b, nb)];
        for (int64_t e = 0; e < k; ++e) {
            const uint8_t* at = codes + qcode_at(r, e / 32, (int)(e % 32 / 8), nb, bits);
            const int i = (int)(e % 8);
            q[r * k + e] = (int8_t)(bits == 8 ? at[i] - 128 : (i < 4 ? at[i] & 15 : at[i - 4] >> 4) - 8);
        }
    }
}

// ================================================================== device: dequantizing GEMV
//
// Tensor-core GEMV on exact integers.  Decode at batch 1 is bound by HBM only if the work per weight
// code stays far below one instruction; rebuilding weights as floats costs more than that.  So the
// codes go to `mma.sync m16n8k16` as fp16 integers, two MMAs per block of 32 weights of 16 rows:
//   - a biased code u (0 .. 255, or 0 .. 15) becomes the fp16 number 1024 + u by putting its bits
//     under the exponent of 1024: one byte permute, or a shift and an and-or, for two codes;
//   - the input x^ (fp32) of block b is split into three integer digits of at most 127 at scales s,
//     s / 254 and s / 254^2 (s = max|x^| / 127 over the block), which reproduce it to 2^-24 of the
//     block's largest value; the digits are the MMA's B columns 0, 1, 2, so one accumulation gives
//     all three dot products of each row with the block;
//   - every product and partial sum is an integer below 2^23, so the fp32 accumulation is exact; the
//     accumulator starts at -(1024 + bias) times the digit's sum, which takes the offsets out;
//   - a row's block term is s * D1 + s / 254 * D2 + s / 254^2 * D3, times the block's fp16 weight
//     scale, accumulated in fp32.
// Codes and scales are stored in the order in which a warp takes them: per row tile and block, lane
// (g, t) finds the positions 8t .. 8t + 7 of rows g and g + 8 side by side (one 16-byte load, or 8
// bytes at 4 bits), and rows g and g + 8's scales in one word, so a warp streams whole lines.  The
// k order within a block is the codes' order in the fragments, the same for the digits.
// What bounds it is the instructions around the MMAs and the start of a CTA (norm, digits), not the
// bytes: a warp takes 32 rows where there are enough (two row tiles share the input's fragments), a
// batch of two blocks runs without branches (past the end the last block again, with zero scales), and the input's
// divisions are done for four blocks at once, one lane each.  Llama-2-7B gate/up, four 8-bit shards
// in one launch (92 MB): 32.0 us, against 49 with rows stored one after another, 16 rows a warp and
// the integer MMA m16n8k32 (which takes the codes as they are, but is slow on this GPU).
// Work split: the blocks of a shard's rows are cut into `parts` (gemv_q_parts of the shard alone);
// a CTA takes 128 rows (64 in launches of few rows) and one or more consecutive parts, and computes
// the input digits of its parts only; a warp takes a quarter of the rows and
// one half of each part.  The CTAs of a row tile form a thread-block cluster: after a cluster barrier rank 0 adds the parts' row sums in part
// order (distributed shared memory) and runs the epilogue, and a second cluster barrier keeps the
// other ranks until it has read them.  No global scratch, no flags.
// How many parts a CTA takes depends on the launch (a single shard: one; a whole block's shards:
// enough for 2.5 CTAs an SM), the sums of a shard and their order do not, so a shard's results have
// the same bits alone and in a group.
// The first codes are loaded before griddepcontrol.wait: weights do not depend on the preceding
// kernel.
constexpr int kQWarps = 8;
constexpr int kQThreads = kQWarps * 32;
constexpr int kQUnroll = 2;  // blocks in flight per warp and buffer
constexpr int kQMaxParts = 8;

__device__ __forceinline__ void mma_f16f32(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                           uint32_t b1, float c0, float c1, float c2, float c3) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%11,%12,%13};"
        : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "f"(c0), "f"(c1), "f"(c2), "f"(c3));
}
// The eight codes of a row's position group as fp16 pairs 1024 + u: at 8 bits (two words) positions
// (0, 1), (2, 3), (4, 5), (6, 7); at 4 bits (one word) (0, 2), (1, 3), (4, 6), (5, 7).
template <int BITS>
__device__ __forceinline__ void codes_f16(uint32_t w0, uint32_t w1, uint32_t (&h)[4]) {
    if constexpr (BITS == 8) {
        h[0] = __byte_perm(w0, 0x64646464u, 0x4140);
        h[1] = __byte_perm(w0, 0x64646464u, 0x4342);
        h[2] = __byte_perm(w1, 0x64646464u, 0x4140);
        h[3] = __byte_perm(w1, 0x64646464u, 0x4342);
    } else {
        h[0] = (w0 & 0x000F000Fu) | 0x64006400u;
        h[1] = ((w0 >> 8) & 0x000F000Fu) | 0x64006400u;
        h[2] = ((w0 >> 4) & 0x000F000Fu) | 0x64006400u;
        h[3] = ((w0 >> 12) & 0x000F000Fu) | 0x64006400u;
    }
}

// First block of part `part` of `parts` over nb blocks (nb at most 512).
__host__ __device__ __forceinline__ int part_start(int nb, int part, int parts) { return part * nb / parts; }
// shared-memory bytes of a CTA whose parts have at most `pb` blocks: per block 3 x 32 fp16 digits, 16
// bytes of scales (s1, s2, s3) and 32 bytes of accumulator starts
static size_t gemv_q_smem(int pb) { return (size_t)pb * (192 + 16 + 32) + 16; }

// One CTA of 64 MT rows, four row groups of MT row tiles by two halves.  tile_row: the CTA's first row.
template <int EPI, int BITS, int MT>
__device__ __forceinline__ void gemv_q_cta(const QGemvArgs& a, int tile_row) {
    constexpr int kQRows = 64 * MT, kRowsW = 16 * MT;  // rows of the CTA, of a warp
    constexpr int OFFSET = 1024 + (BITS == 8 ? 128 : 8);  // of a code's fp16 number
    extern __shared__ __align__(16) uint8_t qsm[];
    __shared__ float red[kQWarps + 1];
    __shared__ float rsum[kQMaxParts][kQWarps][kRowsW];
    __shared__ float rows_sum[kQMaxParts][kQRows];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
    const QMatDev& W = a.w;
    const int nb = W.nb;
    // cluster (gridDim.x, 1, 1): this CTA has parts [p0, p1) of the shard, blocks [pb0, pb1)
    const int ranks = (int)gridDim.x, rank = (int)blockIdx.x, parts = a.parts;
    const int p0 = rank * parts / ranks, p1 = (rank + 1) * parts / ranks;
    const int pb0 = part_start(nb, p0, parts), npb = part_start(nb, p1, parts) - pb0;
    __half* xq = reinterpret_cast<__half*>(qsm);                       // [npb][3][32]
    float4* xsc = reinterpret_cast<float4*>(qsm + (size_t)npb * 192);  // [npb] (s1, s2, s3, -)
    float* xst = reinterpret_cast<float*>(xsc + npb);                  // [npb][8] accumulator start of each column
    const int tile = warp & 3, half = warp >> 2;
    __shared__ int2 span[kQMaxParts + 1][2];  // [part - p0][half]: its blocks
    if (tid < 2 * (p1 - p0)) {
        const int p = p0 + (tid >> 1), s0 = part_start(nb, p, parts), s1 = part_start(nb, p + 1, parts), mid = s0 + (s1 - s0) / 2;
        span[tid >> 1][tid & 1] = (tid & 1) == 0 ? make_int2(s0, mid) : make_int2(mid, s1);
    }
    __syncthreads();
    // Batches of kQUnroll of this warp's blocks: its half of the CTA's first part, then of the next, ...
    const int np = p1 - p0;
    struct Cursor {
        int p, b, end;
    };
    auto enter = [&](Cursor& c) {  // the first block of this warp's half of part c.p, skipping empty halves
        for (; c.p < np; ++c.p) {
            const int2 s = span[c.p][half];
            c.b = s.x;
            c.end = s.y;
            if (c.b < c.end) return;
        }
        c.b = pb0;  // past the last part: loads repeat the CTA's first blocks, nothing is consumed
        c.end = pb0 + 1;
    };
    auto next = [&](Cursor& c) {
        c.b += kQUnroll;
        if (c.b >= c.end) {
            ++c.p;
            enter(c);
        }
    };
    // this warp's row tiles (past the last one: that one again, its rows are not written)
    const int tiles = (W.rows + kQTile - 1) / kQTile, tile0 = tile_row / kQTile + MT * tile;
    constexpr uint32_t kCode = BITS == 8 ? 512 : 256;  // bytes of a row tile's block
    const uint8_t* const codes = W.codes + lane * (kCode / 32);
    const __half* const scales = W.scales + 2 * g;
    // block 0 of the row tile, in row tiles x blocks (rows * k / 512: at most 3 * 2^19 under the shape limits)
    uint32_t first[MT];
#pragma unroll
    for (int m = 0; m < MT; ++m) first[m] = (uint32_t)min(tile0 + m, tiles - 1) * (uint32_t)nb;
    struct Batch {
        uint4 q[kQUnroll][MT];     // codes of rows g, g + 8 of row tile m
        uint32_t d[kQUnroll][MT];  // their weight scales
    };
    auto load = [&](Batch& v, const Cursor& c) {
#pragma unroll
        for (int u = 0; u < kQUnroll; ++u)
#pragma unroll
            for (int m = 0; m < MT; ++m) {
                const uint32_t at = first[m] + (uint32_t)min(c.b + u, c.end - 1);
                if constexpr (BITS == 8) {
                    v.q[u][m] = ldg_stream(codes + (size_t)at * kCode);
                } else {
                    const uint2 w = ldg_stream_u2(codes + (size_t)at * kCode);
                    v.q[u][m].x = w.x;
                    v.q[u][m].z = w.y;
                }
                const uint32_t d = ldg_stream_u1(scales + (size_t)at * kQTile);
                v.d[u][m] = c.b + u < c.end ? d : 0u;
            }
    };
    Batch v0, v1;
    Cursor cl{0, 0, 0};  // the batch to load next
    enter(cl);
    Cursor cc = cl;      // the batch to consume next
    load(v0, cl);
    next(cl);
    load(v1, cl);
    next(cl);
    if (lane < kRowsW)
        for (int p = 0; p < kQMaxParts; ++p) rsum[p][warp][lane] = 0.f;  // (halves without blocks)
    pdl_wait();

    // ---------------------------------------------------------------- input digits of the part
    float rinv = 1.f;
    if (a.x != nullptr) {
        float ss = 0.f;
#pragma unroll 16
        for (int i = tid; i < W.k; i += kQThreads) {
            const float v = __half2float(a.x[i]);
            ss = fmaf(v, v, ss);
        }
        ss = warp_sum(ss);
        if (lane == 0) red[warp] = ss;
        __syncthreads();
        if (tid == 0) {
            float s = 0.f;
            for (int w = 0; w < kQWarps; ++w) s += red[w];
            red[kQWarps] = 1.0f / sqrtf(s / (float)W.k + a.eps);
        }
        __syncthreads();
        rinv = red[kQWarps];
    }
    for (int j0 = warp * 4; j0 < npb; j0 += kQWarps * 4) {  // four blocks at a time
        float v[4], am = 0.f;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int i = (pb0 + j0 + u) * kQBlock + lane;
            v[u] = 0.f;
            if (j0 + u < npb && i < W.k)
                v[u] = a.x != nullptr ? __half2float(a.x[i]) * rinv * __half2float(a.gain[i]) : __ldcg(a.vin + i);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            // the block's largest magnitude (non-negative floats order as their bit patterns)
            const float m = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(fabsf(v[u]))));
            if (lane == u) am = m;
        }
        // lane u: the scales of block u and the inverse of the first
        const float s1 = am / 127.0f, s2 = s1 / 254.0f, s3 = s2 / 254.0f;
        const float i1 = am > 0.f ? 127.0f / am : 0.f;
        if (lane < 4 && j0 + lane < npb) xsc[j0 + lane] = make_float4(s1, s2, s3, 0.f);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const float sc[2] = {__shfl_sync(0xffffffffu, s1, u), __shfl_sync(0xffffffffu, s2, u)};
            const float b1 = __shfl_sync(0xffffffffu, i1, u), b2 = b1 * 254.0f;
            const float iv[3] = {b1, b2, b2 * 254.0f};
            if (j0 + u >= npb) break;  // (the same for the whole warp)
            // three digits: each takes the remainder of the ones before, to within half its step, in
            // the order in which the codes unpack (codes_f16)
            const int at = BITS == 8 ? lane : (lane & ~3) | ((lane & 1) << 1) | ((lane >> 1) & 1);
            float r = v[u], start = 0.f;
#pragma unroll
            for (int e = 0; e < 3; ++e) {
                const int q = (int)fminf(fmaxf(rintf(r * iv[e]), -127.f), 127.f);
                if (e < 2) r = fmaf(-(float)q, sc[e], r);
                xq[(j0 + u) * 96 + e * 32 + at] = __int2half_rn(q);
                const int sum = __reduce_add_sync(0xffffffffu, q);
                if (lane == e) start = (float)(-OFFSET * sum);
            }
            if (lane < 8) xst[(j0 + u) * 8 + lane] = start;
        }
    }
    __syncthreads();
    pdl_launch_dependents();

    // ---------------------------------------------------------------- this warp's blocks
    float acc[2 * MT];  // rows g, g + 8 of each row tile
#pragma unroll
    for (int i = 0; i < 2 * MT; ++i) acc[i] = 0.f;
    auto consume = [&](const Batch& v) {
#pragma unroll
        for (int u = 0; u < kQUnroll; ++u) {
            const int j = min(cc.b + u, cc.end - 1) - pb0;  // (past the end: zero scales)
            uint4 bf = make_uint4(0u, 0u, 0u, 0u);
            if (g < 3) bf = *reinterpret_cast<const uint4*>(xq + j * 96 + g * 32 + 8 * t);
            const float2 st = *reinterpret_cast<const float2*>(xst + j * 8 + 2 * t);
            const float4 sc = xsc[j];
#pragma unroll
            for (int m = 0; m < MT; ++m) {
                uint32_t ha[4], hb[4];
                codes_f16<BITS>(v.q[u][m].x, v.q[u][m].y, ha);
                codes_f16<BITS>(v.q[u][m].z, v.q[u][m].w, hb);
                float c[4], d[4];
                mma_f16f32(c, ha[0], hb[0], ha[1], hb[1], bf.x, bf.y, st.x, st.y, st.x, st.y);
                mma_f16f32(d, ha[2], hb[2], ha[3], hb[3], bf.z, bf.w, c[0], c[1], c[2], c[3]);
                // lane t = 0 holds the digit-1 and digit-2 products of its rows, lane t = 1 digit 3 (the
                // other lanes' sums are not used)
                const float d3a = __shfl_down_sync(0xffffffffu, d[0], 1), d3b = __shfl_down_sync(0xffffffffu, d[2], 1);
                float va = sc.z * d3a, vb = sc.z * d3b;
                va = fmaf(sc.y, d[1], va);
                vb = fmaf(sc.y, d[3], vb);
                va = fmaf(sc.x, d[0], va);
                vb = fmaf(sc.x, d[2], vb);
                const float2 ds = h2_to_f2(v.d[u][m]);
                acc[2 * m] = fmaf(ds.x, va, acc[2 * m]);
                acc[2 * m + 1] = fmaf(ds.y, vb, acc[2 * m + 1]);
            }
        }
    };
    // after the last batch of a part: the part's sums of this warp's rows
    auto advance = [&]() {
        const int p = cc.p;
        next(cc);
        if (cc.p != p) {
#pragma unroll
            for (int i = 0; i < 2 * MT; ++i) {
                if (t == 0) rsum[p][warp][8 * i + g] = acc[i];
                acc[i] = 0.f;
            }
        }
    };
    __syncwarp();  // rsum is cleared
    while (cc.p < np) {
        consume(v0);
        load(v0, cl);
        next(cl);
        advance();
        if (cc.p < np) {
            consume(v1);
            load(v1, cl);
            next(cl);
            advance();
        }
    }
    __syncthreads();
    for (int i = tid; i < np * kQRows; i += kQThreads) {  // halves in order
        const int p = i / kQRows, r = i % kQRows;
        rows_sum[p][r] = rsum[p][r / kRowsW][r % kRowsW] + rsum[p][4 + r / kRowsW][r % kRowsW];
    }

    // ---------------------------------------------------------------- parts of the cluster
    if (ranks > 1) cluster_sync();  // every part's row sums are in its CTA's shared memory
    else __syncthreads();
    float tv = 0.f;
    const int r = tid, row = tile_row + r;
    if (rank == 0 && tid < kQRows) {
        for (int k = 0; k < ranks; ++k) {
            const int n = (k + 1) * parts / ranks - k * parts / ranks;
            for (int p = 0; p < n; ++p) tv += k == 0 ? rows_sum[p][r] : dsmem_ld(dsmem_addr(&rows_sum[p][r], (uint32_t)k));
        }
    }
    __syncthreads();
    if (rank == 0 && tid < kQRows) rows_sum[0][r] = tv;
    if (ranks > 1) cluster_sync();  // rank 0 has read the others' sums (they may leave), and its own are final
    else __syncthreads();
    if (rank != 0 || tid >= kQRows || row >= W.rows) return;

    // ---------------------------------------------------------------- epilogue (row pairs)
    if constexpr (EPI == kEpiPlain) {
        a.out[row] = tv;
    } else if ((r & 1) == 0 && row + 1 < W.rows) {
        const float t_odd = rows_sum[0][r + 1];
        if constexpr (EPI == kEpiSwiglu) {
            a.out[row >> 1] = silu(tv) * t_odd;
        } else {  // kEpiQkvRope: rows (row, row + 1) are the RoPE pair (i, i + dh / 2)
            const int p = *a.len;
            const bool ok = p >= 0 && p < a.cap;
            if (!ok && row == 0) set_status(a.status, VT_DEV_KV_OVERFLOW);
            const int hd = a.dh >> 1;
            const int blk = row / a.dh, i = (row - blk * a.dh) >> 1;
            if (blk < a.hq + a.hk) {
                const float2 cs2 = ok ? a.rope[(int64_t)p * hd + i] : make_float2(1.f, 0.f);
                const float re = tv * cs2.x - t_odd * cs2.y;
                const float ro = tv * cs2.y + t_odd * cs2.x;
                if (blk < a.hq) {
                    a.out[blk * a.dh + i] = re;
                    a.out[blk * a.dh + i + hd] = ro;
                } else if (ok) {
                    __half* kd = a.kcache + ((int64_t)(blk - a.hq) * a.cap + p) * a.dh;
                    kd[i] = __float2half_rn(re);
                    kd[i + hd] = __float2half_rn(ro);
                }
            } else if (ok) {
                __half* vd = a.vcache + ((int64_t)(blk - a.hq - a.hk) * a.cap + p) * a.dh;
                vd[i] = __float2half_rn(tv);
                vd[i + hd] = __float2half_rn(t_odd);
            }
        }
    }
}

template <int EPI, int NG, int MT>
__global__ void __launch_bounds__(kQThreads, 3) k_gemv_q(const __grid_constant__ DecodeGroup<QGemvArgs, NG> G) {
    int gi = 0, y = (int)blockIdx.y;  // the shard that owns this row tile
    if constexpr (NG > 1) {
        while (gi + 1 < G.n && y >= G.end[gi]) ++gi;
        if (gi > 0) y -= G.end[gi - 1];
    }
    const QGemvArgs& a = G.a[gi];
    if (a.w.bits == 8) gemv_q_cta<EPI, 8, MT>(a, y * 64 * MT);
    else gemv_q_cta<EPI, 4, MT>(a, y * 64 * MT);
}

// ================================================================== device: quantizer
//
// One thread per block of 32 weights of a row: the fp16 scale and the codes of the format
// above, packed into the kernel layout.  Every decision is the host quantizer's: IEEE fp32
// division (amax / qmax and w / d), one rounding of the scale to fp16, round-half-even of w / d,
// so the codes equal those of vt_quantize_rows bit for bit.
template <int BITS>
__global__ void k_quantize_rows(const __half* __restrict__ w, int64_t ld, int rows, int k, int nb,
                                uint8_t* __restrict__ codes, __half* __restrict__ scales) {
    constexpr int QMAX = BITS == 8 ? 127 : 7, BIAS = BITS == 8 ? 128 : 8;
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int r = (int)(t / nb), b = (int)(t - (int64_t)r * nb);
    if (r >= (rows + kQTile - 1) / kQTile * kQTile) return;
    const __half* src = w + (int64_t)r * ld + (int64_t)b * kQBlock;
    const int n = r < rows ? min(kQBlock, k - b * kQBlock) : 0;  // (rows past the end: zeros)
    float amax = 0.f;
    for (int e = 0; e < n; ++e) amax = fmaxf(amax, fabsf(__half2float(src[e])));
    const __half d16 = __float2half_rn(amax / (float)QMAX);
    const float d = __half2float(d16);
    scales[qscale_at(r, b, nb)] = d16;
    uint32_t u[kQBlock];
#pragma unroll
    for (int e = 0; e < kQBlock; ++e) {
        int c = 0;
        if (e < n && d != 0.f) {
            const float x = rintf(__half2float(src[e]) / d);
            c = x > (float)QMAX ? QMAX : (x < (float)-QMAX ? -QMAX : (int)x);
        }
        u[e] = (uint32_t)(c + BIAS);
    }
#pragma unroll
    for (int g = 0; g < 4; ++g) {  // positions 8g .. 8g + 7
        uint8_t* dst = codes + qcode_at(r, b, g, nb, BITS);
        if constexpr (BITS == 8) {
            uint32_t wd[2];
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const uint32_t* v = u + 8 * g + 4 * i;
                wd[i] = v[0] | (v[1] << 8) | (v[2] << 16) | (v[3] << 24);
            }
            *reinterpret_cast<uint2*>(dst) = make_uint2(wd[0], wd[1]);
        } else {
            uint32_t v = 0;
#pragma unroll
            for (int i = 0; i < 4; ++i) v |= (u[8 * g + i] | (u[8 * g + i + 4] << 4)) << (8 * i);
            *reinterpret_cast<uint32_t*>(dst) = v;
        }
    }
}

cudaError_t launch_quantize_rows(const __half* w, int64_t ld, const QMatDev& m, cudaStream_t st) {
    const int64_t n = qmat_rows(m.rows) * m.nb;
    if (n <= 0) return cudaSuccess;
    const int threads = 128;
    const unsigned blocks = (unsigned)((n + threads - 1) / threads);
    if (m.bits == 8)
        k_quantize_rows<8><<<blocks, threads, 0, st>>>(w, ld, m.rows, m.k, m.nb, m.codes, m.scales);
    else if (m.bits == 4)
        k_quantize_rows<4><<<blocks, threads, 0, st>>>(w, ld, m.rows, m.k, m.nb, m.codes, m.scales);
    else
        return cudaErrorInvalidValue;
    return cudaGetLastError();
}

// Parts of a shard's blocks: enough for about 2.5 pieces of 64 rows by one part per SM, each part at
// least 4 blocks, at most 8 (the portable cluster size).
static int gemv_q_parts(int tiles, int nb) {
    const int want = (int)std::lround(2.5 * (g_num_sms > 0 ? g_num_sms : 148) / std::max(tiles, 1));
    return std::max(1, std::min({kQMaxParts, want, std::max(1, nb / 4)}));
}

// The n shards of `a` in one launch of 64 MT-row tiles by cluster ranks.
template <int EPI, int NG, int MT>
static cudaError_t launch_q_group(const QGemvArgs* a, int n, cudaStream_t st) {
    DecodeGroup<QGemvArgs, NG> G{};
    int tiles = 0, min_parts = kQMaxParts, max_pb = 1;
    for (int s = 0; s < n; ++s) {
        tiles += (a[s].w.rows + 64 * MT - 1) / (64 * MT);
        G.a[s] = a[s];
        G.end[s] = tiles;
        G.a[s].parts = gemv_q_parts((a[s].w.rows + 63) / 64, a[s].w.nb);
        min_parts = std::min(min_parts, G.a[s].parts);
    }
    G.n = n;
    // CTAs per row tile: the parts of the shard, or, in a group, as many as the launch needs
    const int ranks = n == 1 ? min_parts : std::min(min_parts, gemv_q_parts(tiles, 4 * kQMaxParts));
    for (int s = 0; s < n; ++s)
        for (int k = 0; k < ranks; ++k)
            max_pb = std::max(max_pb, part_start(G.a[s].w.nb, (k + 1) * G.a[s].parts / ranks, G.a[s].parts) -
                                          part_start(G.a[s].w.nb, k * G.a[s].parts / ranks, G.a[s].parts));
    const size_t smem = gemv_q_smem(max_pb);
    if (smem > 200 * 1024) return cudaErrorInvalidValue;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)ranks, (unsigned)tiles);
    cfg.blockDim = dim3(kQThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    int na = 0;
    attr[na].id = cudaLaunchAttributeClusterDimension;
    attr[na].val.clusterDim.x = (unsigned)ranks;
    attr[na].val.clusterDim.y = 1;
    attr[na].val.clusterDim.z = 1;
    ++na;
    if (g_use_pdl) {
        attr[na].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[na].val.programmaticStreamSerializationAllowed = 1;
        ++na;
    }
    cfg.attrs = attr;
    cfg.numAttrs = (unsigned)na;
    return cudaLaunchKernelEx(&cfg, k_gemv_q<EPI, NG, MT>, G);
}

template <int EPI>
static cudaError_t launch_q_epi(const QGemvArgs* a, int n, cudaStream_t st) {
    QGemvArgs sel[VT_MAX_DEVICES];
    int m = 0, pieces = 0;
    for (int s = 0; s < n; ++s) {
        if (a[s].w.bits != 8 && a[s].w.bits != 4) return cudaErrorInvalidValue;
        if (a[s].w.rows > 0) {
            const int tiles = (a[s].w.rows + 63) / 64;
            sel[m++] = a[s];
            pieces += tiles * gemv_q_parts(tiles, a[s].w.nb);
        }
    }
    if (m == 0) return cudaSuccess;
    // Two row tiles a warp halve the instructions a row spends on the input, but also the CTAs: taken
    // where 1.75 CTAs an SM are left.  A token through four 8-bit Llama-2-7B shards (5 to 9 CTAs an SM)
    // 94 us a layer; through one such shard (at most 2.5 pieces an SM) 141 us a layer with one row tile a
    // warp against 205 with two.  A shard alone has 3.5 pieces from 34000 rows on, which only QKV can
    // have: an ATTN step of 96 heads and 4096 columns, 8 bits, 76 us with two row tiles and 92 with one.
    // (With two, the compiler spills 56 to 88 bytes a thread at the 80 registers that three CTAs leave.)
    const bool wide = 2 * pieces >= 7 * (g_num_sms > 0 ? g_num_sms : 148);
    if (m == 1) return wide ? launch_q_group<EPI, 1, 2>(sel, m, st) : launch_q_group<EPI, 1, 1>(sel, m, st);
    return wide ? launch_q_group<EPI, VT_MAX_DEVICES, 2>(sel, m, st) : launch_q_group<EPI, VT_MAX_DEVICES, 1>(sel, m, st);
}

cudaError_t launch_gemv_q(int epi, const QGemvArgs* a, int n, cudaStream_t st) {
    switch (epi) {
        case kEpiPlain: return launch_q_epi<kEpiPlain>(a, n, st);
        case kEpiSwiglu: return launch_q_epi<kEpiSwiglu>(a, n, st);
        case kEpiQkvRope: return launch_q_epi<kEpiQkvRope>(a, n, st);
        default: return cudaErrorInvalidValue;
    }
}

// ================================================================== quantized shard partials
//
// Communication scaling (Voltron Section 4.3.2): the activations sent between devices are lowered
// to 8 or 4 bits.  Under tensor parallelism those are the fp32 shard partials sent to the main
// device.  Format: blocks of 32 values, fp16 scale d = fp16(amax / qmax) and codes
// round-half-even(x / d) clamped to [-qmax, qmax], fp32 decisions (the oracle's vector format);
// stored as one int8 per value (8 bits) or two per byte (4 bits: value 2 i in the low nibble and
// 2 i + 1 in the high nibble, each as q + 8).

// The scale and this lane's code of a block of 32 values, one value per lane of the warp (0 past
// the end of the vector): every decision is the oracle's, in fp32.  A NaN takes no part in the
// maximum and has the code 0.
template <int QMAX>
__device__ __forceinline__ int block_code(float v, __half& d16, float& d) {
    const float amax = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(fmaxf(fabsf(v), 0.f))));
    d16 = __float2half_rn(amax / (float)QMAX);
    d = __half2float(d16);
    if (d == 0.f) return 0;
    const float r = rintf(v / d);
    return r > (float)QMAX ? QMAX : (r < (float)-QMAX ? -QMAX : (int)r);
}

// One warp per block of 32 values, one value per lane: the loads, the codes' stores and the 32
// divisions of a block run side by side.  It is latency bound (a few KB); a thread per block, with
// its 32 loads and divisions in a row on one CTA, took 10.5 us for a 4096-value partial.
template <int BITS>
__global__ void __launch_bounds__(256) k_quantize_vec(const float* __restrict__ x, int64_t n, uint8_t* __restrict__ codes,
                                                      __half* __restrict__ scales) {
    constexpr int QMAX = BITS == 8 ? 127 : 7;
    pdl_wait();
    const int lane = threadIdx.x & 31;
    const int64_t b = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), e = b * kQBlock + lane;
    if (b * kQBlock < n) {
        __half d16;
        float d;
        const int q = block_code<QMAX>(e < n ? x[e] : 0.f, d16, d);
        if (lane == 0) scales[b] = d16;
        if constexpr (BITS == 8) {
            if (e < n) codes[e] = (uint8_t)(int8_t)q;
        } else {
            const int hi = __shfl_down_sync(0xffffffffu, q, 1);  // (the code of 0 past the end)
            if ((lane & 1) == 0 && e < n) codes[e >> 1] = (uint8_t)((uint32_t)(q + 8) | ((uint32_t)(hi + 8) << 4));
        }
    }
    pdl_launch_dependents();
}

cudaError_t launch_quantize_vec(const float* x, int64_t n, int bits, uint8_t* codes, __half* scales, cudaStream_t st) {
    const int64_t nb = (n + kQBlock - 1) / kQBlock;
    if (nb <= 0) return cudaSuccess;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)((nb + 7) / 8));
    cfg.blockDim = dim3(256);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = g_use_pdl ? 1 : 0;
    if (bits == 8) return cudaLaunchKernelEx(&cfg, k_quantize_vec<8>, x, n, codes, scales);
    if (bits == 4) return cudaLaunchKernelEx(&cfg, k_quantize_vec<4>, x, n, codes, scales);
    return cudaErrorInvalidValue;
}

// out[e] = fp16(residual[e] + sum_s q_s[e] d_s[e / 32]), shards in order, fp32.
__global__ void k_combine_q(const __grid_constant__ CombineQArgs a) {
    pdl_wait();
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < a.count; e += (int64_t)gridDim.x * blockDim.x) {
        float acc = a.residual ? __half2float(a.residual[e]) : 0.f;
        for (int s = 0; s < a.n; ++s) {
            int q;
            if (a.bits == 8) {
                q = (int)(int8_t)a.codes[s][e];
            } else {
                const uint8_t byte = a.codes[s][e >> 1];
                q = (int)((e & 1) ? (byte >> 4) : (byte & 15)) - 8;
            }
            acc = fmaf((float)q, __half2float(a.scales[s][e / kQBlock]), acc);
        }
        a.out[e] = __float2half_rn(acc);
    }
    pdl_launch_dependents();
}

cudaError_t launch_combine_q(const CombineQArgs& a, cudaStream_t st) {
    if (a.count <= 0) return cudaSuccess;
    const int64_t blocks = std::min<int64_t>((a.count + 255) / 256, (int64_t)(g_num_sms > 0 ? g_num_sms : 148) * 8);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)blocks);
    cfg.blockDim = dim3(256);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = g_use_pdl ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, k_combine_q, a);
}

// The combine of one decode token whose partials travel at bits[s] (16: fp32): out = fp16(residual
// + sum_s p_s), shards in order, p_s the partial or, at 8 or 4 bits, its codes times their scale.
// One warp per block of 32 elements quantizes each shard's block as it leaves that shard and adds
// it at once (the same codes, scales and sums as k_quantize_vec followed by k_combine_q, which the
// tests compare with the oracle), so a block of the layer has one launch instead of one per shard
// and the codes need no memory.  Latency bound (n * 16 KB): the launches were what it cost.  Three
// layers of the 8B shapes on three devices, partials at 8 bits: 670 us a token with a quantizing
// launch per shard and a combine, 495 us with this.  The partials are cleared after reading (they
// are accumulated into zeroed buffers).
__global__ void __launch_bounds__(256) k_combine_token_q(const __grid_constant__ CombineTokenQArgs a) {
    pdl_wait();
    pdl_launch_dependents();
    const int lane = threadIdx.x & 31;
    const int e = (int)(blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) * kQBlock + lane;
    if (e - lane >= a.count) return;
    const bool on = e < a.count;
    float v[VT_MAX_DEVICES];
#pragma unroll
    for (int s = 0; s < VT_MAX_DEVICES; ++s) v[s] = on && s < a.n ? __ldcg(a.parts[s] + e) : 0.f;
    float acc = on ? __half2float(a.residual[e]) : 0.f;
#pragma unroll
    for (int s = 0; s < VT_MAX_DEVICES; ++s) {
        if (s >= a.n) break;
        if (a.bits[s] == 16) {
            acc += v[s];
        } else {
            __half d16;
            float d;
            const int q = a.bits[s] == 8 ? block_code<127>(v[s], d16, d) : block_code<7>(v[s], d16, d);
            acc = fmaf((float)q, d, acc);
        }
        if (on) a.parts[s][e] = 0.f;
    }
    if (on) a.out[e] = __float2half_rn(acc);
}

cudaError_t launch_combine_token_q(const CombineTokenQArgs& a, cudaStream_t st) {
    if (a.count <= 0) return cudaSuccess;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)((a.count + 255) / 256));
    cfg.blockDim = dim3(256);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = g_use_pdl ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, k_combine_token_q, a);
}

cudaError_t init_quant_kernels() {
    const int lim = 200 * 1024;
    cudaError_t e;
#define VT_Q_ATTR1(EPI, NG, MT)                                                                                  \
    if ((e = cudaFuncSetAttribute(k_gemv_q<EPI, NG, MT>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim)) != \
        cudaSuccess)                                                                                             \
        return e;
#define VT_Q_ATTR(EPI)                                                              \
    VT_Q_ATTR1(EPI, 1, 1) VT_Q_ATTR1(EPI, 1, 2) VT_Q_ATTR1(EPI, VT_MAX_DEVICES, 1) \
    VT_Q_ATTR1(EPI, VT_MAX_DEVICES, 2)
    VT_Q_ATTR(kEpiPlain)
    VT_Q_ATTR(kEpiSwiglu)
    VT_Q_ATTR(kEpiQkvRope)
#undef VT_Q_ATTR
#undef VT_Q_ATTR1
    return cudaSuccess;
}

}  // namespace vt
