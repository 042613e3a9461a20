// mc_gemm.cu -- prefill-path expert kernels (many pairs per expert): grouped
// dequant-GEMM on the 5th-generation tensor cores (Eq. 1's E_i on PMQ weights,
// Sec. 2.2, batched over the pairs routed to each expert).
//
// x_img_kernel: per token block (<= 128 pairs of one expert, from the block
//   list) and 128-column step, the fp16 activations of the block's pairs as the
//   K-major SW128 image the MMA reads (rows = pairs, zero rows past the block),
//   with the columns of every K = 16 slice ordered like the A operand below.
// gemm_kernel<W13>: persistent, one CTA per SM, warp-specialised:
//   weight producer    claims items (a token block x a 128-row block of W1|W3,
//                      or x a 256-row block pair of W2) from an atomic counter and
//                      streams the packed weights of both streams, one 128-column
//                      step per slot of the weight ring;
//   image producer     streams the activation images of the same items into a ring
//                      of its own (only the block's rows, rounded up to 16);
//   converter warps    16: four for each weight stream and step parity; each warp
//                      reads its two 16-row tiles of packed codes (the decode path's
//                      layout) into registers, gives the weight slot back, turns them
//                      into fp16 (q - z) s, waits until the MMAs have read its A
//                      buffer two steps ago and stores the tiles there with
//                      tcgen05.st 16x256b, whose thread -> (lane, column) order is the
//                      mma fragment order the packed tiles are stored in;
//   MMA warps (2)      one per weight stream: tcgen05.mma kind::f16, M = 128 rows,
//                      N = the block's pairs (rounded up to 16), K = 16, A from
//                      tensor memory, B from the image, fp32 accumulators in tensor
//                      memory;
//   epilogue warps     W13: h = silu(W1 x) * (W3 x) -> fp16 image of W2's input
//                      (the same image layout, one 128-column step per row block);
//                      W2: fp32 outputs per pair.
// What sets the pace.  The tensor pipe takes 1026 cycles for a step's 16 MMAs at
// N = 128 and 515 at N = 64, whatever copies, tensor-memory stores and shared-memory
// loads run beside it; the conversion alone takes ~51 cycles per 16x128 tile and SM
// (820 a step) with 8 warps as with 16: a probe's lop3, __hsub2 and __hfma2 each issue
// every other cycle.  What kept the MMAs from either pace was their issue: under
// `lane == 0` 8 MMAs take 541 cycles, and 859 beside 16 busy warps (elect_one).
// Mixtral-8x7b layer, W1,W3 / W2 launch: 256 tokens (N ~ 60) 157 / 99 -> 131 / 76 us,
// 4096 tokens 1424 / 755 -> 1316 / 657 us (1.46 PFLOP/s, 0.83 of the sustained cuBLAS
// rate; power-capped: 1298 / 646 in another run).
// Tensor memory (512 columns): accumulators of streams 0/1 at columns 0 / 128 (when
// every token block has <= 64 pairs, two accumulator sets of 64 columns each, so
// that an item's epilogue overlaps the next item's MMAs), each stream's two A
// buffers of 64 columns at 256 / 384.
#include "mc_host.h"
#include "mc_kernels.h"
#include "mc_profile.h"
#include "mc_umma.cuh"

namespace mc {

constexpr int kGN = 128;                  // pairs per token block (MMA N), at most
constexpr int kGNarrow = 64;              // a call whose blocks all have <= 64 pairs: narrow rings
constexpr int kImgBytes = kGN * kTileK * 2;  // one 128-column step image: 32 KB
constexpr int kGHdr = 2048;
constexpr size_t kGSmem = 232448;            // all of the CTA's shared memory
// warps 0-15: converters (warp w: tensor-memory lanes 32 (w % 4) .. +31, i.e. tiles
// 2 (w % 4) and 2 (w % 4) + 1, of stream (w / 4) % 2, in the steps of parity w / 8);
// 16-19 epilogue; 20 weight producer; 21 / 22 issue the MMAs of stream 0 / 1; 23
// image producer
constexpr int kGConv = 16, kGEpi0 = 16, kGProd = 20, kGMma = 21, kGMmaN = 2, kGImgProd = 23, kGConvGroup = 4;
constexpr int kGThreads = 24 * 32;
constexpr int kGMaxW = 8, kGMaxI = 6;        // ring slots, at most
// Items whose description may still be read while a new one is written: the weight
// producer is at most kGMaxW + 4 steps (so as many items, at one step per item)
// ahead of a completed MMA, the epilogue two items behind it, the end marker one
// more ahead.
constexpr int kGItemRing = 16;
static_assert(kGItemRing >= kGMaxW + 4 + 3, "item ring");

// Ring geometry of a call: the weight slots hold a 3-bit step of both streams, the
// image slots 128 or (narrow) 64 rows; what is left beside the h staging is split so
// that either ring covers a copy's latency (4 image and 5 weight slots, 4 of them at group
// 64; narrow 6 and 8).  One expert of more than 64 pairs makes the whole call wide, which
// costs 1 %: the Mixtral-8x7b layer narrow / forced wide at 200 tokens 211.5 / 213.7 us, at
// 256 with ODP 217.3 / 219.4.
struct GGeom {
    int atom;               // bytes between an image slot's two 64-column atoms
    int wslot, nw, ni;      // weight slot bytes, weight and image slots
    int img0, w0;           // offsets of the rings; the staging starts at kGHdr
};
__host__ __device__ __forceinline__ GGeom gemm_geom(int group, bool narrow)
{
    GGeom g;
    g.atom = (narrow ? kGNarrow : kGN) * 128;
    g.wslot = 2 * supertile_bytes(3, group);
    g.ni = narrow ? 6 : 4;
    g.img0 = kGHdr + 2 * g.atom;  // the staging: one h image
    g.w0 = g.img0 + g.ni * 2 * g.atom;
    const int nw = ((int)kGSmem - g.w0) / g.wslot;
    g.nw = nw < kGMaxW ? nw : kGMaxW;
    return g;
}

// Byte offset of (pair row n, column c of the 128-column step) in an image: two
// 64-column SW128 atoms; inside an atom the four 4-column groups of every
// 16-column run are transposed with the four K = 16 slices, so that K slice s of
// atom a holds, in order, columns 64a + 16t + 4s + {0..3} for t = 0..3 -- the
// columns the converter stores into tensor-memory columns 2t / 2t+1 of slice s.
__host__ __device__ __forceinline__ uint32_t img_off(int n, int c, int atom = kGN * 128)
{
    const int a = c >> 6, cc = c & 63;
    const int t = cc >> 4, s = (cc >> 2) & 3, e = cc & 3;
    return (uint32_t)(a * atom) + sw128_offset((uint32_t)n, (uint32_t)(16 * s + 4 * t + e));
}

// One step of the weight ring (item < 0: end of the CTA's work).
struct GWStage {
    int item, bits, nstream, info;  // info: the MMA warps' word (kInfo*)
};
constexpr int kInfoN = 0xff, kInfoFirst = 0x100, kInfoLast = 0x200, kInfoLone = 0x400,
              kInfoEnd = 0x800;

struct GItem {
    int k, u, nstream, n;  // token block (-1: end), unit, streams, MMA N
    int pair_base, nv;
};

// An expert's token blocks, in the order the items are taken (more bits first).
struct GRun {
    int e, bits, off, cnt, first, nb, base;  // expert, its pairs, first block, blocks, first item
};

struct GShared {
    uint64_t wfull[kGMaxW], wempty[kGMaxW];
    uint64_t ifull[kGMaxI], iempty[kGMaxI];
    uint64_t afull[2][2], aempty[2][2];  // [stream][buffer]
    uint64_t dfull[2], dempty[2], esync, drain;
    uint64_t itembar[kGItemRing];
    uint32_t tmem_base;
    volatile int abort;
    volatile int wissued, iissued;
    volatile int end_items;  // items this CTA's MMA warps completed, set once they saw the end marker
    int total, narrow;
    int ainfo[2][2];         // [stream][buffer]: the stored step's info word
    GRun run[kMaxE];
    GWStage wst[kGMaxW];
    GItem items[kGItemRing];
};
static_assert(sizeof(GShared) <= kGHdr, "gemm header");

__device__ __forceinline__ bool g_wait(uint64_t *bar, uint32_t parity, const ExpertParams &p, GShared *sh)
{
    if (mbar_try_wait(bar, parity)) return true;
    const uint64_t t0 = globaltimer_ns();
    while (true) {
        if (mbar_try_wait_sleep(bar, parity, kWaitHintNs)) return true;
        if (sh->abort) return false;
        if (globaltimer_ns() - t0 > p.timeout_ns) {
            set_status(p.status, MC_ERR_TIMEOUT);
            sh->abort = 1;
            return false;
        }
    }
}

// The same for a whole warp, with one answer for all of its lanes: what follows such a
// wait is executed by the warp together (tcgen05 st / ld, __syncwarp), and lanes that
// took different answers, when a phase completes just as a wait expires or the CTA
// aborts, would wait for one another for ever.  The vote is on the first test, so that a
// phase that is complete costs no divergent branch (256 tokens 221 -> 215 us, 512: 365 -> 351,
// against a vote on g_wait alone).
__device__ __forceinline__ bool warp_wait(uint64_t *bar, uint32_t parity, const ExpertParams &p, GShared *sh)
{
    if (__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) return true;
    return __all_sync(0xffffffffu, g_wait(bar, parity, p, sh));
}

// The packed buffer carries the header written for this shape and bit table
// (every expert's bit width and matrix offsets), so no copy reads outside it.
__device__ __forceinline__ bool g_header_ok(const ExpertParams &p)
{
    const PackHeader *hd = reinterpret_cast<const PackHeader *>(p.packed);
    bool ok = hd->magic == kMagic && hd->version == kFormatVersion && hd->E == p.E && hd->H == p.H &&
              hd->F == p.F && hd->group == p.group;
#pragma unroll
    for (int e = 0; e < kMaxE; ++e)
        if (e < p.E)
            ok &= hd->bits[e] == p.bits[e] && hd->mat_off[e][0] == p.mat_off[e][0] &&
                  hd->mat_off[e][1] == p.mat_off[e][1] && hd->mat_off[e][2] == p.mat_off[e][2];
    return ok;
}

__device__ __forceinline__ uint32_t h2_bits(__half2 v) { return *reinterpret_cast<const uint32_t *>(&v); }
__device__ __forceinline__ __half2 bits_h2(uint32_t v) { return *reinterpret_cast<const __half2 *>(&v); }

// ------------------------------------------------------------------ x image --
// A thread takes 32 consecutive columns of a pair (columns 64 a + 32 tp .. + 31), i.e.
// column quarters 2 tp and 2 tp + 1 of atom a, which are 16-byte chunk 2 s + tp of
// every slice s: four 16-byte loads, four 16-byte stores.  A warp stores whole
// 32-byte sectors of eight image rows (8-byte pieces scattered over the row, and the
// rows past the block's pairs written as zeros that no copy reads, took 85 us between
// events at 4096 tokens; this takes 25 us for 33 MB in, 67 MB out).
constexpr int kXRows = 32;  // pairs per CTA
__global__ void __launch_bounds__(kXRows * 4) x_img_kernel(ExpertParams p)
{
    const int k = blockIdx.x, kt = blockIdx.y, n = blockIdx.z * kXRows + (threadIdx.x >> 2), KT = p.H / kTileK;
    // CTA (0, 0, 0) checks the packed header for the two GEMM launches that follow
    // (they read only its verdict): the header's loads go out before the wait (the
    // packed buffer is complete before the layer starts), the verdict is written
    // after it, when the expert kernels of the call before have completed
    const bool hdr_thread = k == 0 && kt == 0 && blockIdx.z == 0 && threadIdx.x == 0;
    const bool hok = hdr_thread ? g_header_ok(p) : true;
    pdl_trigger();
    pdl_wait();
    if (hdr_thread) {
        *p.hdr_ok = hok ? 1 : 0;
        if (!hok) set_status(p.status, MC_ERR_BAD_PACK);
    }
    const int nblocks = *p.nchunks;
    const ChunkInfo ci = p.chunks[k];  // entry k < max_blocks exists even when unused
    if (k >= nblocks || n >= ((ci.nv + 15) & ~15)) return;  // the GEMM reads rows up to a multiple of 16
    const int a = (threadIdx.x >> 1) & 1, tp = threadIdx.x & 1;
    uint4 raw[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) raw[i] = make_uint4(0, 0, 0, 0);
    if (n < ci.nv) {
        const uint4 *src = reinterpret_cast<const uint4 *>(p.x + (size_t)(p.perm[ci.pair_base + n] >> 1) * p.H +
                                                           kt * kTileK + 64 * a + 32 * tp);
#pragma unroll
        for (int i = 0; i < 4; ++i) raw[i] = src[i];
    }
    // h[4 i + j]: columns 8 i + 2 j, + 1 of the 32
    uint32_t h[16];
    bool bad = false;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const __nv_bfloat162 *b2 = reinterpret_cast<const __nv_bfloat162 *>(&raw[i]);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float2 f = __bfloat1622float2(b2[j]);
            bad |= !(fabsf(f.x) <= 65504.f) || !(fabsf(f.y) <= 65504.f);
            h[4 * i + j] = h2_bits(__floats2half2_rn(f.x, f.y));
        }
    }
    // slice s: columns 4 s .. 4 s + 3 of the first quarter, then of the second
    uint8_t *row = p.ximg + ((size_t)k * KT + kt) * kImgBytes + (size_t)a * (kGN * 128) + n * 128;
#pragma unroll
    for (int s = 0; s < 4; ++s)
        *reinterpret_cast<uint4 *>(row + (((2 * s + tp) ^ (n & 7)) << 4)) =
            make_uint4(h[2 * s], h[2 * s + 1], h[8 + 2 * s], h[8 + 2 * s + 1]);
    if (bad) set_status(p.status, MC_ERR_RANGE);
}

// -------------------------------------------------------------- converters --

// Exponent-constant bits of pair j (the fp16 2^E the decoder adds, both halves).
template <int BITS>
__device__ __forceinline__ uint32_t pair_offset_bits(int j)
{
    const int f = BITS == 1 ? off1_pos(j) : BITS == 2 ? 2 * off2_pos(j) : off3_bit(j);
    return MC_C(25 - f);
}


// The code words and (scale, zero) pairs of one lane's part of a tile, as stored.
template <int GPT>
struct RawTile {
    uint32_t w[6];
    uint2 meta[GPT];
};

template <int GPT>
__device__ __forceinline__ void load_raw(const uint8_t *tile, int bits, int lane, RawTile<GPT> &t)
{
    if (bits >= 2) {
        const uint4 v = *reinterpret_cast<const uint4 *>(tile + 16 * lane);
        t.w[0] = v.x; t.w[1] = v.y; t.w[2] = v.z; t.w[3] = v.w;
    }
    if (bits != 2) {
        const uint2 v = *reinterpret_cast<const uint2 *>(tile + (bits == 3 ? 512 : 0) + 8 * lane);
        t.w[4] = v.x; t.w[5] = v.y;
    }
    const uint8_t *mt = tile + tile_code_bytes(bits);
#pragma unroll
    for (int g = 0; g < GPT; ++g) t.meta[g] = *reinterpret_cast<const uint2 *>(mt + 64 * g + (lane >> 2) * 8);
}

// One 16-row tile, one 128-column step: 32 fp16 pairs (q - z) s per lane, in the
// order tcgen05.st 16x256b.x8 takes them: per k-step s, the A-fragment registers
// a0, a2, a1, a3 (rows g8 / g8+8, k pairs t / t+4).
template <int BITS, int GPT>
__device__ __forceinline__ void convert_tile(const RawTile<GPT> &t, uint32_t (&out)[32])
{
    __half2 s2[GPT][2], nz2[GPT][2];  // [group][row half]: (s, s) and (-z s, -z s)
#pragma unroll
    for (int g = 0; g < GPT; ++g) {
        const __half2 a = bits_h2(t.meta[g].x), b = bits_h2(t.meta[g].y);  // (s0, z0), (s1, z1)
        const float sa = __low2float(a), za = __high2float(a), sb = __low2float(b), zb = __high2float(b);
        s2[g][0] = __floats2half2_rn(sa, sa);
        s2[g][1] = __floats2half2_rn(sb, sb);
        nz2[g][0] = __floats2half2_rn(-za * sa, -za * sa);
        nz2[g][1] = __floats2half2_rn(-zb * sb, -zb * sb);
    }
#pragma unroll
    for (int qd = 0; qd < 4; ++qd) {
        uint32_t r[8];
        if constexpr (BITS == 1) cvt1_half(t.w[4 + (qd >> 1)], 8 * (qd & 1), r);
        if constexpr (BITS == 2) cvt2(t.w[qd], r);
        if constexpr (BITS == 3) cvt3(t.w, qd, r);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int j = 8 * qd + i, s = j >> 2, rho = j & 3;
            const int gi = GPT == 2 ? (s >> 2) : 0;
            const __half2 q = __hsub2(bits_h2(r[i]), bits_h2(pair_offset_bits<BITS>(j)));  // exact
            const __half2 w = __hfma2(q, s2[gi][rho & 1], nz2[gi][rho & 1]);
            // st order per k-step: a0 (rho 0), a2 (rho 2), a1 (rho 1), a3 (rho 3)
            const int slot = rho == 0 ? 0 : rho == 2 ? 1 : rho == 1 ? 2 : 3;
            out[4 * s + slot] = h2_bits(w);
        }
    }
}

__device__ __forceinline__ void tmem_st_16x256_x8(uint32_t taddr, const uint32_t (&v)[32])
{
    asm volatile(
        "tcgen05.st.sync.aligned.16x256b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,"
        "%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32};" ::"r"(taddr),
        "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]), "r"(v[8]),
        "r"(v[9]), "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15]), "r"(v[16]),
        "r"(v[17]), "r"(v[18]), "r"(v[19]), "r"(v[20]), "r"(v[21]), "r"(v[22]), "r"(v[23]), "r"(v[24]),
        "r"(v[25]), "r"(v[26]), "r"(v[27]), "r"(v[28]), "r"(v[29]), "r"(v[30]), "r"(v[31])
        : "memory");
}

// A step's two tiles of one converter warp: converted and stored, the first store
// after the MMAs have read the buffer.  One code path per width from the packed words
// to the store (a store behind the widths' branches, shared by them: the ODP layer at
// 256 tokens 241 -> 245 us).  False once the CTA aborted.
template <int BITS, int GPT>
__device__ __forceinline__ bool convert_store(const RawTile<GPT> &ta, const RawTile<GPT> &tb, uint32_t abuf, bool wait,
                                              uint64_t *aempty, uint32_t parity, const ExpertParams &p, GShared *sh)
{
    uint32_t v[32];
    convert_tile<BITS, GPT>(ta, v);
    if (wait && !warp_wait(aempty, parity, p, sh)) return false;
    tc_fence_after();
    tmem_st_16x256_x8(abuf, v);
    convert_tile<BITS, GPT>(tb, v);
    tmem_st_16x256_x8(abuf + (16u << 16), v);
    tmem_st_wait();
    return true;
}

// ------------------------------------------------------------- epilogue --

__device__ __forceinline__ void tmem_ld_x16(uint32_t taddr, float (&v)[16])
{
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr)
        : "memory");
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

__device__ __forceinline__ void tmem_ld_x16_nowait(uint32_t taddr, uint32_t (&r)[16])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr)
        : "memory");
}

// Epilogue warps meet (bounded); false once the CTA aborted.
__device__ __forceinline__ bool epi_sync(const ExpertParams &p, GShared *sh, int lane, int &uses)
{
    __syncwarp();
    if (lane == 0) mbar_arrive(&sh->esync);
    return warp_wait(&sh->esync, (uses++) & 1, p, sh);
}

// ------------------------------------------------------------------ kernel --

template <bool W13, int GPT>
__global__ void __launch_bounds__(kGThreads, 1) gemm_kernel(ExpertParams p)
{
    extern __shared__ __align__(1024) uint8_t smem[];
    GShared *sh = reinterpret_cast<GShared *>(smem);
    uint8_t *staging = smem + kGHdr;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    constexpr int group = kTileK / GPT;
    const int nrb = W13 ? p.F / kBlockRows : p.H / kBlockRows;
    const int KTm = W13 ? p.H / kTileK : p.F / kTileK;  // column steps (K)
    const int U = W13 ? nrb : (nrb + 1) / 2;            // units of a token block: row block (pair)
    const uint8_t *img_base = W13 ? p.ximg : p.himg;

    if (threadIdx.x == 0) {
        for (int s = 0; s < kGMaxW; ++s) {
            mbar_init(&sh->wfull[s], 1);
            mbar_init(&sh->wempty[s], 2 * kGConvGroup);
        }
        for (int s = 0; s < kGMaxI; ++s) {
            mbar_init(&sh->ifull[s], 1);
            mbar_init(&sh->iempty[s], kGMmaN);
        }
        for (int b = 0; b < 2; ++b) {
            for (int c = 0; c < 2; ++c) {
                mbar_init(&sh->afull[c][b], kGConvGroup);
                mbar_init(&sh->aempty[c][b], 1);
            }
            mbar_init(&sh->dfull[b], kGMmaN);
            mbar_init(&sh->dempty[b], 4);
        }
        mbar_init(&sh->esync, 4);
        mbar_init(&sh->drain, kGMmaN);
        for (int i = 0; i < kGItemRing; ++i) mbar_init(&sh->itembar[i], 1);
        sh->abort = 0;
        sh->wissued = 0;
        sh->iissued = 0;
        sh->end_items = 0x7fffffff;
        fence_mbar_init();
    }
    if (warp == kGMma) tmem_alloc(&sh->tmem_base, 512);
    pdl_wait();
    if (warp == 0) {
        // the experts' runs of token blocks, from the routing's offsets, in the order
        // of the block list: more bits first, then by expert
        const int E = p.E;
        int off = 0, cnt = 0, bits = 0;
#pragma unroll
        for (int f = 0; f < kMaxE; ++f)
            if (f == lane) bits = p.bits[f];
        if (lane < E) {
            off = __ldcg(p.offsets + lane);
            cnt = __ldcg(p.offsets + lane + 1) - off;
        }
        const int nb = (cnt + kGN - 1) / kGN;
        int rank = 0, first = 0, blocks = 0;
        for (int f = 0; f < E; ++f) {
            const int bf = __shfl_sync(0xffffffffu, bits, f), nf = __shfl_sync(0xffffffffu, nb, f);
            blocks += nf;
            if (bf > bits || (bf == bits && f < lane)) {
                ++rank;
                first += nf;
            }
        }
        if (lane < E) sh->run[rank] = GRun{lane, bits, off, cnt, first, nb, first * U};
        const unsigned wide = __ballot_sync(0xffffffffu, cnt > kGNarrow);
        if (lane == 0) {
            sh->total = blocks * U;
            sh->narrow = wide == 0;
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tbase = sh->tmem_base;
    const int total = sh->total;
    const bool narrow = sh->narrow;
    const GGeom geo = gemm_geom(group, narrow);
    const int nbuf = narrow ? 2 : 1;  // accumulator sets

    if (warp == kGProd) {
        // ----------------------------------------------------- weight producer --
        if (lane == 0 && !(p.debug & kDebugNoProducer)) {
            const uint64_t pol = policy_evict_first();
            int *counter = &p.counters[W13 ? 2 : 3];
            // The packed header was checked once for the call by x_img_kernel, which
            // completed before this launch's wait returned: no copy unless its verdict
            // says the buffer matches
            const int verdict = __ldcg(p.hdr_ok);
            int item = atomicAdd(counter, 1);
            bool ok = verdict == 1;
            if (!ok) {
                set_status(p.status, MC_ERR_BAD_PACK);
                sh->abort = 1;
            }
            int it = 0, slot = 0, nitem = 0;
            uint32_t phase = 0;
            while (ok && item < total) {
                int r = 0;
                while (r + 1 < p.E && item >= sh->run[r + 1].base) ++r;
                const GRun run = sh->run[r];
                const int local = item - run.base;
                // W1,W3: the expert's token blocks vary fastest, so the CTAs that run
                // at the same time share a row block's weights (and the blocks' x
                // images stay in L2); W2: the 256-row block pairs vary fastest, so
                // they share one block's h image while the expert's W2 weights stay
                // in L2 from block to block
                const int u = W13 ? local / run.nb : local % U;
                const int blk = W13 ? local % run.nb : local / U;
                GItem gi;
                gi.k = run.first + blk;
                gi.u = u;
                gi.nstream = W13 ? 2 : w2_pair_width(u, nrb);
                gi.pair_base = run.off + blk * kGN;
                gi.nv = min(kGN, run.cnt - blk * kGN);
                gi.n = (gi.nv + 15) & ~15;
                sh->items[nitem % kGItemRing] = gi;
                mbar_arrive(&sh->itembar[nitem % kGItemRing]);
                ++nitem;
                const int STB = supertile_bytes(run.bits, group);
                const uint8_t *wsrc = p.packed + p.mat_off[run.e][W13 ? 0 : 2] +
                                      supertile_off(W13 ? 0 : 2, W13 ? u : 2 * u, 0, KTm, nrb, STB);
                const uint32_t wb = (uint32_t)(gi.nstream * STB);
                int next = total;
                for (int kt = 0; kt < KTm; ++kt, ++it) {
                    if (it >= geo.nw && !g_wait(&sh->wempty[slot], phase ^ 1u, p, sh)) {
                        ok = false;
                        break;
                    }
                    sh->wst[slot] = GWStage{item, run.bits, gi.nstream,
                                            gi.n | (kt == 0 ? kInfoFirst : 0) | (kt == KTm - 1 ? kInfoLast : 0) |
                                                (gi.nstream == 1 ? kInfoLone : 0)};
                    uint8_t *dst = smem + geo.w0 + slot * geo.wslot;
                    mbar_arrive_expect_tx(&sh->wfull[slot], wb);
                    // W1,W3 weights are read by the CTAs of one row block at about
                    // the same time: evict-first; a W2 row-block pair's weights come
                    // back for every token block of the expert: normal policy
                    if (W13) bulk_g2s_stream(dst, wsrc + (size_t)kt * wb, wb, &sh->wfull[slot], pol);
                    else bulk_g2s(dst, wsrc + (size_t)kt * wb, wb, &sh->wfull[slot]);
                    sh->wissued = it + 1;
                    // the next item's claim overlaps this item's last copies
                    if (kt == max(0, KTm - 2)) next = atomicAdd(counter, 1);
                    if (++slot == geo.nw) {
                        slot = 0;
                        phase ^= 1u;
                    }
                }
                item = next;
            }
            if (ok) {
                pdl_trigger();  // the CTA takes no further item: the next kernel may launch
                sh->items[nitem % kGItemRing].k = -1;
                mbar_arrive(&sh->itembar[nitem % kGItemRing]);
                // two end markers: each parity's converters take every other step
                for (int m = 0; m < 2; ++m, ++it) {
                    if (it >= geo.nw && !g_wait(&sh->wempty[slot], phase ^ 1u, p, sh)) break;
                    sh->wst[slot].item = -1;
                    mbar_arrive(&sh->wfull[slot]);
                    if (++slot == geo.nw) {
                        slot = 0;
                        phase ^= 1u;
                    }
                }
            }
        }
    } else if (warp == kGImgProd) {
        // ------------------------------------------------------ image producer --
        if (lane == 0) {
            int it = 0, slot = 0;
            uint32_t phase = 0;
            bool ok = true;
            for (int n = 0; ok; ++n) {
                if (!g_wait(&sh->itembar[n % kGItemRing], (n / kGItemRing) & 1, p, sh)) break;
                const GItem gi = sh->items[n % kGItemRing];
                if (gi.k < 0) break;
                const uint8_t *src = img_base + (size_t)gi.k * KTm * kImgBytes;
                const uint32_t ab = (uint32_t)gi.n * 128u;  // rows 0 .. n - 1 of an atom
                for (int kt = 0; kt < KTm; ++kt, ++it, src += kImgBytes) {
                    if (it >= geo.ni && !g_wait(&sh->iempty[slot], phase ^ 1u, p, sh)) {
                        ok = false;
                        break;
                    }
                    uint8_t *dst = smem + geo.img0 + slot * 2 * geo.atom;
                    mbar_arrive_expect_tx(&sh->ifull[slot], 2 * ab);
                    if (gi.n == kGN) {
                        bulk_g2s(dst, src, 2 * ab, &sh->ifull[slot]);
                    } else {
                        bulk_g2s(dst, src, ab, &sh->ifull[slot]);
                        bulk_g2s(dst + geo.atom, src + kImgBytes / 2, ab, &sh->ifull[slot]);
                    }
                    sh->iissued = it + 1;
                    if (++slot == geo.ni) {
                        slot = 0;
                        phase ^= 1u;
                    }
                }
            }
        }
    } else if (warp < kGConv) {
        // ---------------------------------------------------------- converters --
        // warp q of the group (stream cg, parity b) converts tiles 2q, 2q + 1 of the
        // stream (tensor-memory lanes 32q .. 32q + 31) in every other step, into the
        // stream's A buffer b
        const int q = warp & 3, cg = (warp >> 2) & 1, b = warp >> 3;
        const uint32_t abuf = tbase + 256u + 128u * (uint32_t)cg + 64u * (uint32_t)b + ((uint32_t)(32 * q) << 16);
        int slot = b;
        uint32_t phase = 0;
        for (int n = 0;; ++n) {
            if (!warp_wait(&sh->wfull[slot], phase, p, sh)) break;
            const GWStage st = sh->wst[slot];
            const bool active = st.item >= 0 && cg < st.nstream;
            RawTile<GPT> ta, tb;
            if (active) {
                const int TB = tile_bytes(st.bits, group);
                const uint8_t *w = smem + geo.w0 + slot * geo.wslot + cg * (kTilesPerBlock * TB) + 2 * q * TB;
                load_raw<GPT>(w, st.bits, lane, ta);
                load_raw<GPT>(w + TB, st.bits, lane, tb);
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&sh->wempty[slot]);  // the packed words are in registers
            slot += 2;
            if (slot >= geo.nw) {
                slot -= geo.nw;
                phase ^= 1u;
            }
            // the MMAs that read this buffer last are done (and afull's phase of that
            // step has been waited for)
            const bool wait = n > 0;
            const uint32_t par = (uint32_t)((n - 1) & 1);
            uint64_t *ae = &sh->aempty[cg][b];
            bool ok;
            if (!active) ok = !wait || warp_wait(ae, par, p, sh);
            else if (st.bits == 1) ok = convert_store<1, GPT>(ta, tb, abuf, wait, ae, par, p, sh);
            else if (st.bits == 2) ok = convert_store<2, GPT>(ta, tb, abuf, wait, ae, par, p, sh);
            else ok = convert_store<3, GPT>(ta, tb, abuf, wait, ae, par, p, sh);
            if (!ok) break;
            if (q == 0 && lane == 0) sh->ainfo[cg][b] = st.item < 0 ? kInfoEnd : st.info;
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&sh->afull[cg][b]);
            if (st.item < 0) break;
        }
    } else if (warp >= kGMma && warp < kGMma + kGMmaN) {
        // ----------------------------------------------------------------- MMA --
        // The whole warp runs the loop, one elected lane issues (elect_one).
        const int mx = warp - kGMma;  // the weight stream this warp multiplies
        int nitem = 0, slot = 0;
        uint32_t phase = 0;
        for (int it = 0;; ++it) {
            const int b = it & 1;
            if (!warp_wait(&sh->afull[mx][b], (it >> 1) & 1, p, sh)) break;
            const int info = sh->ainfo[mx][b];
            if (info & kInfoEnd) break;
            const int par = nitem % nbuf, use = nitem / nbuf;
            if ((info & kInfoFirst) && use > 0 && !warp_wait(&sh->dempty[par], (use - 1) & 1, p, sh)) break;
            if (!warp_wait(&sh->ifull[slot], phase, p, sh)) break;
            tc_fence_after();
            const uint32_t idesc = umma_idesc_f16(128, info & kInfoN);
            const uint64_t bd = umma_desc_sw128(smem + geo.img0 + slot * 2 * geo.atom);
            const uint64_t bd1 = bd + (uint64_t)(geo.atom >> 4);
            const uint32_t abuf = tbase + 256u + 128u * (uint32_t)mx + 64u * (uint32_t)b;
            const uint32_t d = tbase + 128u * (uint32_t)mx + (uint32_t)(kGNarrow * par);
            if (elect_one()) {
                // (a lone W2 block's second stream multiplies nothing: its converters
                // stored no tile and its accumulator is not read)
                if (mx == 0 || !(info & kInfoLone)) {
#pragma unroll
                    for (int s = 0; s < 8; ++s)
                        umma_f16_ts(d, abuf + 8u * (uint32_t)s, (s < 4 ? bd : bd1) + (uint64_t)(2 * (s & 3)), idesc,
                                    s > 0 || !(info & kInfoFirst));
                }
                umma_commit(&sh->aempty[mx][b]);
                umma_commit(&sh->iempty[slot]);
                if (info & kInfoLast) umma_commit(&sh->dfull[par]);
            }
            __syncwarp();
            if (info & kInfoLast) ++nitem;
            if (++slot == geo.ni) {
                slot = 0;
                phase ^= 1u;
            }
        }
        // every MMA of both warps has completed (and with it every commit to
        // dfull) before the epilogue is told that no item follows and before
        // TMEM is released
        __syncwarp();
        if (elect_one()) umma_commit(&sh->drain);
        __syncwarp();
        const uint64_t t0 = globaltimer_ns();
        while (!mbar_try_wait(&sh->drain, 0))
            if (globaltimer_ns() - t0 > p.timeout_ns) break;
        __syncwarp();
        // the epilogue has taken the last item of this accumulator set before its
        // dfull completes once more, so that it never sees two completions of one
        // barrier in one wait
        const int par = nitem % nbuf, use = nitem / nbuf;
        if ((use == 0 || warp_wait(&sh->dempty[par], (use - 1) & 1, p, sh)) && lane == 0) {
            if (mx == 0) sh->end_items = nitem;
            mbar_arrive(&sh->dfull[par]);
        }
    } else {
        // ------------------------------------------------------------ epilogue --
        const int ew = warp - kGEpi0;   // tensor-memory lanes 32 ew .. 32 ew + 31
        const int row = 32 * ew + lane;  // row of the 128-row block
        const int tid = threadIdx.x - 32 * kGEpi0;
        int uses = 0;
        for (int ic = 0;; ++ic) {
            const int par = ic % nbuf;
            if (!warp_wait(&sh->dfull[par], (ic / nbuf) & 1, p, sh)) break;
            if (ic >= sh->end_items) break;
            tc_fence_after();
            const GItem gi = sh->items[ic % kGItemRing];
            const uint32_t dbase = tbase + ((uint32_t)(32 * ew) << 16) + (uint32_t)(kGNarrow * par);
            if (W13) {
                // h of the thread's row, 64 pairs at a time packed in registers, so that D
                // is released before the last of the image is written (rows nv .. n - 1
                // of the block's x image are zero, so their h is)
                bool bad = false;
#pragma unroll 1
                for (int h0 = 0; h0 < gi.n; h0 += 64) {
                    uint32_t hp[32];
#pragma unroll
                    for (int n0 = 0; n0 < 64; n0 += 16) {
                        if (h0 + n0 >= gi.n) continue;
                        uint32_t g[16], v[16];
                        tmem_ld_x16_nowait(dbase + (uint32_t)(h0 + n0), g);
                        tmem_ld_x16_nowait(dbase + 128u + (uint32_t)(h0 + n0), v);
                        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
                        for (int i = 0; i < 16; i += 2) {
                            const float v0 = silu(__uint_as_float(g[i])) * __uint_as_float(v[i]);
                            const float v1 = silu(__uint_as_float(g[i + 1])) * __uint_as_float(v[i + 1]);
                            bad |= !(fabsf(v0) <= 65504.f) || !(fabsf(v1) <= 65504.f);
                            hp[(n0 + i) / 2] = h2_bits(__floats2half2_rn(v0, v1));
                        }
                    }
                    if (h0 + 64 >= gi.n) {
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(&sh->dempty[par]);
                    }
#pragma unroll
                    for (int n0 = 0; n0 < 64; n0 += 16) {
                        if (h0 + n0 >= gi.n) continue;
#pragma unroll
                        for (int i = 0; i < 16; i += 2) {
                            const __half2 h = bits_h2(hp[(n0 + i) / 2]);
                            *reinterpret_cast<__half *>(staging + img_off(h0 + n0 + i, row, geo.atom)) = __low2half(h);
                            *reinterpret_cast<__half *>(staging + img_off(h0 + n0 + i + 1, row, geo.atom)) = __high2half(h);
                        }
                    }
                }
                if (bad) set_status(p.status, MC_ERR_RANGE);
                // the image of W2's column step gi.u for token block gi.k
                if (!epi_sync(p, sh, lane, uses)) break;
                uint8_t *dst = p.himg + ((size_t)gi.k * (p.F / kTileK) + gi.u) * kImgBytes;
                for (int i = tid; i < gi.n * 8; i += 128) {
                    reinterpret_cast<uint4 *>(dst)[i] = reinterpret_cast<const uint4 *>(staging)[i];
                    reinterpret_cast<uint4 *>(dst + kImgBytes / 2)[i] =
                        reinterpret_cast<const uint4 *>(staging + geo.atom)[i];
                }
                if (!epi_sync(p, sh, lane, uses)) break;
            } else {
                float *out = p.opart;
                for (int x = 0; x < gi.nstream; ++x) {
                    const int blk = 2 * gi.u + x;
                    for (int n0 = 0; n0 < gi.nv; n0 += 16) {
                        float v[16];
                        tmem_ld_x16(dbase + 128u * (uint32_t)x + (uint32_t)n0, v);
#pragma unroll
                        for (int i = 0; i < 16; ++i)
                            if (n0 + i < gi.nv)
                                out[(size_t)(gi.pair_base + n0 + i) * p.H + blk * kBlockRows + row] = v[i];
                    }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&sh->dempty[par]);
            }
        }
    }

    tc_fence_before();
    __syncthreads();
    // On an abort, let copies that were issued but never consumed land before the
    // CTA's shared memory is released (bounded).
    if (threadIdx.x == 0 && sh->abort) {
        for (int it = max(0, sh->wissued - geo.nw); it < sh->wissued; ++it) {
            const uint64_t t0 = globaltimer_ns();
            while (!mbar_try_wait(&sh->wfull[it % geo.nw], (it / geo.nw) & 1))
                if (globaltimer_ns() - t0 > p.timeout_ns) break;
        }
        for (int it = max(0, sh->iissued - geo.ni); it < sh->iissued; ++it) {
            const uint64_t t0 = globaltimer_ns();
            while (!mbar_try_wait(&sh->ifull[it % geo.ni], (it / geo.ni) & 1))
                if (globaltimer_ns() - t0 > p.timeout_ns) break;
        }
    }
    if (warp == kGMma) {
        tc_fence_after();
        tmem_dealloc(tbase, 512);
    }
}

// --------------------------------------------------------------- launcher --

int launch_gemm(ExpertParams ep, cudaStream_t st)
{
    int dev = 0, maxsm = 0, nsm = 0;
    cudaError_t err = cudaGetDevice(&dev);
    if (err == cudaSuccess) err = cudaDeviceGetAttribute(&maxsm, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (err == cudaSuccess) err = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    if (err != cudaSuccess) return set_error(MC_ERR_CUDA, "device query: %s", cudaGetErrorString(err));
    if ((size_t)maxsm < kGSmem) return set_error(MC_ERR_UNSUPPORTED, "not enough shared memory for the GEMM ring");
    if (!ep.ximg || !ep.himg) return set_error(MC_ERR_INVALID_ARG, "prefill path without image buffers");
    auto k13 = ep.group == 64 ? gemm_kernel<true, 2> : gemm_kernel<true, 1>;
    auto k2 = ep.group == 64 ? gemm_kernel<false, 2> : gemm_kernel<false, 1>;
    err = cudaFuncSetAttribute(k13, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kGSmem);
    if (err == cudaSuccess) err = cudaFuncSetAttribute(k2, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kGSmem);
    if (err != cudaSuccess) return set_error(MC_ERR_CUDA, "cudaFuncSetAttribute: %s", cudaGetErrorString(err));

    profile_begin(kKXImg, st);
    err = launch_k(x_img_kernel, dim3(ep.max_blocks, ep.H / kTileK, kGN / kXRows), dim3(kXRows * 4), 0, st, ep);
    profile_end(kKXImg, st);
    if (err == cudaSuccess) {
        profile_begin(kKGemmW13, st);
        err = launch_k(k13, dim3(nsm), dim3(kGThreads), kGSmem, st, ep);
        profile_end(kKGemmW13, st);
    }
    if (err == cudaSuccess) {
        profile_begin(kKGemmW2, st);
        err = launch_k(k2, dim3(nsm), dim3(kGThreads), kGSmem, st, ep);
        profile_end(kKGemmW2, st);
    }
    if (err != cudaSuccess) return set_error(MC_ERR_CUDA, "GEMM launch: %s", cudaGetErrorString(err));
    return MC_OK;
}

size_t img_buffer_bytes(int max_blocks, int cols) { return (size_t)max_blocks * (cols / kTileK) * kImgBytes; }
int max_blocks_for(int T, int E) { return (2 * T + kGN - 1) / kGN + E; }

}  // namespace mc
