// Forward scan of the selective-scan layer core (MambaByte Section 2,
// "Implementation: parallel scans"; Eq. 2-3; Table 6 output and gating):
// prefill, and the training forward, which also keeps the state before every
// chunk. (Verify and the fused Delta projection: prefill.cu.)
//
// Work decomposition. Every (batch row, channel) is an independent recurrence
// over L with a 16-float state (A is diagonal). A CTA of four warps owns 32
// channels of one batch row for its span of L; a warp 8 channels, four lanes
// per channel, each with 4 states in registers. Stages of one to four chunks of
// 16 steps (kSub) come through a ring of TMA tiles (bounded waits); while a chunk
// is scanned the next one, of the same stage or the next, is converted.
//
// What bounds it: per (step, channel) 16 decays on the SFU and 64 multiply-adds,
// which leave the SM at about 0.6 instructions per scheduler and clock, because
// packed and scalar fp32 operations with three register operands take more
// than their pipe's cycles (a register-only loop of just these instructions
// runs at 0.57-0.61), and the shared-memory pipe, which every operand passes.
// The layout therefore spends as few instructions and shared-memory wavefronts
// as it can on everything else:
//  * Pairs of adjacent steps, not of states, fill the packed operations:
//    Delta_t, Delta_t+1 and (Delta x)_t, (Delta x)_t+1 of a channel lie in one
//    16-byte slot, B and C are widened to fp32 in pairs (t, t + 1), so decay
//    exponents, B Delta x and the sum C.h need no copies that duplicate a
//    scalar and no add across a pair; only the recurrence itself is scalar.
//    (Pairs of states: 35.3 instructions per lane and step; this: 29.6, 27.3 with 32-step stages, 27.0 with 64.)
//  * A 128-bit shared load takes 2 wavefronts instead of 4 if lanes that differ
//    in lane bit 0 (or in bit 1) read the same address. Lane bit 0 is a channel
//    bit and bit 1 a state bit (channel bits 0, 2, 3; state bits 1, 4), so that
//    both B, C (by state) and Delta (by channel) are read at that rate.
//  * The four lanes' shares of C.h are added through a warp's own tile instead
//    of shuffles and selects; the lane that adds them is the one that converts
//    those channels and steps, so that D x and silu(z) stay in its registers.
//  * Nothing is stored to shared memory between the loads of a chunk's scan:
//    the shares and the converted chunk i + 1 wait in registers, so that the
//    compiler may move every load ahead.
//  * Token tiles are swizzled by TMA: a warp reads 16-byte columns of them.
//
// Measured (B x L x D, bf16; before: pairs of states, shuffles): 8 x 8192 x 2048
// 850 -> 764 us, with 32-step stages 709, in even shares 650, of 64-step stages 623
// (0.47 of the SFU's rate); 4 x 8192 x 3584 708 -> 592 -> 553 -> 530 us; 1 x 8192 x
// 2048 (time split) 176 -> 122 us; fp32 3 x 1003 x 1544 (time split) 56 -> 39.8 us. At 764 / 592: two
// channels per lane (B and C loaded once for both: 17 % fewer wavefronts) 758 /
// 750 us on the first two: half the warps; two-warp CTAs (16 channels) 784 / 640.
#include <math.h>
#include <stddef.h>
#include <string.h>

#include <algorithm>

#include "common.cuh"
#include "pairs.cuh"
#include "tma.cuh"

namespace mbscan {
namespace {

constexpr int kT = 16;        // steps per chunk
constexpr int kSegUnit = 32;    // least steps of a segment of a time split
constexpr int kShareUnit = 64;  // shares are multiples of this many steps (whole stages)
constexpr int kTP = kT / 2;   // step pairs per chunk
constexpr int kWarps = 4;
constexpr int kThreads = 32 * kWarps;
constexpr int kWCh = 8;                     // channels per warp
constexpr int kCh = kWarps * kWCh;          // channels per CTA
constexpr int kPairs = kWCh / 2;            // channel pairs per warp
constexpr int kPartQ = kTP * kPairs + 4;    // float4s between the shares of two lanes q (the pad keeps them on other banks)

// Two forms, W: wide stages (64 steps for bf16, 32 for fp32) in a ring of 2 and at most 3 CTAs per SM, or stages of half
// that in a ring of 3 and 4 CTAs per SM. A stage is what lies between two CTA barriers. Microseconds per chunk of an
// SM's 1 to 4 CTAs, bf16: wide 0.56 0.78 1.07, narrow 0.61 0.82 1.10 1.40. Grids of at most 3 per SM take the wide form
// (8 x 8192 x 2048 in shares of 3 per SM: 650 -> 623 us), others the narrow one (608 tiles, 4 per SM: 179 us, wide 197).
template <bool W>
constexpr int kStages = W ? 2 : 3;
template <bool W>
constexpr int kCtas = W ? 3 : 4;   // CTAs per SM (shared memory and the register bound)
constexpr int kResident = kCtas<false>;
// Chunks per ring stage, one after the other between two CTA barriers
template <typename T, bool W>
constexpr int kSub = (sizeof(T) == 2 ? 2 : 1) * (W ? 2 : 1);
template <typename T, bool W>
constexpr int kRT = kT * kSub<T, W>;   // steps per stage

template <typename T, bool W>
struct Raw {   // TMA destinations; token tiles swizzled in their 64- (bf16) or 128-byte (fp32) rows
    T dt[kRT<T, W>][kCh];
    T x[kRT<T, W>][kCh];
    T z[kRT<T, W>][kCh];
    T B[kRT<T, W>][kDState];
    T C[kRT<T, W>][kDState];
};

template <typename T, bool W>
struct alignas(1024) Smem {
    Raw<T, W> raw[kStages<W>];
    T ys[2][kRT<T, W>][kCh];                          // output tiles (TMA stores), swizzled like the inputs
    float4 dg[2][kWarps][kTP][kWCh];   // (Delta_t, Delta_t+1, (Delta x)_t, (Delta x)_t+1), see dg_slot
    float4 bc[2][kSub<T, W>][2][2][kTP][4];           // [buffer][chunk][B, C][states 4q, 4q+1 or 4q+2, 4q+3][tp][q]
    float4 part[kWarps][4 * kPartQ];   // shares of C.h of lane q: [q][tp][channel pair]
    uint64_t full[kStages<W>];
    int ticket;
};

struct FwdArgs {
    CUtensorMap tm_dt, tm_x, tm_z, tm_B, tm_C, tm_y;
    ScanParams p;
    int has_gate;
    int seg0;        // first segment of L that the grid covers (blockIdx = (segment - seg0, batch row, channel tile))
    int len0, len;   // steps of the first segment and of the others (the last may be shorter)
};

// Slot of channel c of a warp at step pair tp in its dg tile. A lane stores channels 2 pp and 2 pp + 1 one after
// the other, eight lanes (four pp, two tp) at a time: the two halves change places on odd tp, so that these eight
// 16-byte stores fall on different banks. The scan's loads of all 8 channels at one tp cover 128 bytes either way.
__device__ __forceinline__ int dg_slot(int tp, int c) { return (((c ^ tp) & 1) << 2) | (c >> 1); }

template <typename T, bool kSummary, bool W>
__device__ __forceinline__ void issue_chunk(Smem<T, W> &s, const FwdArgs &a, int stage, int t, int d0, int b) {
    constexpr uint32_t tok = kRT<T, W> * kCh * sizeof(T), bc = kRT<T, W> * kDState * sizeof(T);
    const bool gate = !kSummary && a.has_gate;
    const uint32_t bytes = ((gate ? 3 : 2) * tok) + (kSummary ? 1 : 2) * bc;
    uint64_t *bar = &s.full[stage];
    mbar_arrive_expect_tx(bar, bytes);
    Raw<T, W> &r = s.raw[stage];
    tma_load_3d(&r.dt[0][0], &a.tm_dt, bar, d0, t, b);
    tma_load_3d(&r.x[0][0], &a.tm_x, bar, d0, t, b);
    if (gate) tma_load_3d(&r.z[0][0], &a.tm_z, bar, d0, t, b);
    tma_load_3d(&r.B[0][0], &a.tm_B, bar, 0, t, b);
    if (!kSummary) tma_load_3d(&r.C[0][0], &a.tm_C, bar, 0, t, b);
}

// kCkpt (training forward): also stores the state before every chunk.
// kSummary (first pass of a time-split span, every segment but the first and the
// last): scans the segment from a zero state and records its end state and the
// product of its decays, 2^(A log2 e * sum of Delta); no outputs. The first
// segment starts from h0, so that pass scans it for good and records only its
// end state. In the second pass segment s starts from what the first recorded,
// folded with the associative operator of Section 2: h <- P_s' * h + H_s'.
// kShares: the grid is p.shares CTAs; the channel tiles' spans, laid end to end,
// are cut into that many equal lengths, and a CTA scans the pieces in its own,
// the highest first. Its highest piece starts a tile (or it is all of a CTA's
// part of one) and depends on nothing; where it ends inside a tile, the CTA
// leaves the state for the next share. Only its lowest piece may start inside a
// tile: it comes last and waits (bounded) for the state that the share before
// has left as the first thing it did. Shares are numbered in the order in which
// their CTAs start (a ticket), so the one waited for is always running.
template <typename T, bool kCkpt, bool kSummary, bool kShares, bool W>
__device__ __forceinline__ void scan_spans(const FwdArgs &a) {
    using S = Smem<T, W>;
    using R = Raw<T, W>;
    constexpr int STAGES = kStages<W>, SUB = kSub<T, W>, RT = kRT<T, W>, kRowB = kCh * (int)sizeof(T);
    static_assert(sizeof(R) % (8 * kRowB) == 0 && offsetof(R, x) % (8 * kRowB) == 0 &&
                      offsetof(R, z) % (8 * kRowB) == 0 && offsetof(R, B) % 128 == 0 && offsetof(R, C) % 128 == 0 &&
                      offsetof(S, ys) % (8 * kRowB) == 0 && sizeof(T) * RT * kCh % (8 * kRowB) == 0,
                  "swizzled TMA tiles start on their pattern's boundary");
    extern __shared__ unsigned char smem_dyn[];
    S &s = *reinterpret_cast<S *>(smem_dyn + ((1024u - (smem_u32(smem_dyn) & 1023u)) & 1023u));
    const ScanParams &p = a.p;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int64_t D = p.d_inner;
    const int ntd = (int)((D + kCh - 1) / kCh);
    const int L = (int)p.seqlen;
    const int tiles = (int)p.batch * ntd;
    const int seg = kShares ? 0 : a.seg0 + (int)(blockIdx.x / tiles);
    const int nseg = p.nseg > 1 ? (int)p.nseg : 1;
    const int units = (L + kShareUnit - 1) / kShareUnit;   // kShares
    const bool gate = !kSummary && a.has_gate;

    if (tid == 0) {
        for (int st = 0; st < STAGES; ++st) mbar_init(&s.full[st], 1);
        fence_mbar_init();
    }
    __syncthreads();
    pdl_wait();   // everything below reads or writes global memory

    int st = 0;        // ring slot of the next stage
    uint32_t ph = 0;   // and its phase parity
    // this CTA's tile (batch row, 32 channels); with kShares the units of 64 steps lo .. hi - 1 of all tiles' spans
    // end to end, which it takes tile by tile from the highest
    int tile = (int)(blockIdx.x % tiles);
    int share = 0, lo = 0, hi = 0;
    if constexpr (kShares) {
        if (tid == 0) s.ticket = atomicAdd(p.share_sync(), 1);
        __syncthreads();
        share = s.ticket;
        const int total = tiles * units, len = (total + (int)p.shares - 1) / (int)p.shares;
        lo = min(share * len, total);
        hi = min(lo + len, total);
        if (lo == hi) return;
        tile = (hi - 1) / units;
    }
    for (;;) {   // pieces: one without kShares
        const int b = tile / ntd, d0 = (tile % ntd) * kCh;
        // its steps: tb .. te - 1
        const int tb = kShares ? max(lo - tile * units, 0) * kShareUnit : seg == 0 ? 0 : a.len0 + (seg - 1) * a.len;
        const int te = min(L, kShares ? (hi - tile * units) * kShareUnit : seg == 0 ? a.len0 : tb + a.len);
        const int nch = (te - tb + RT - 1) / RT;   // its stages
        if (tid == 0) {
            fence_proxy_async_smem();
            for (int j = 0, sl = st; j < STAGES && j < nch; ++j, sl = sl + 1 == STAGES ? 0 : sl + 1)
                issue_chunk<T, kSummary, W>(s, a, sl, tb + j * RT, d0, b);
        }

        // ---- conversion and output role: channels 8 warp + 2 pp + {0, 1} of the tile, steps 2 tp, 2 tp + 1
        const int pp = lane % kPairs, tp = lane / kPairs;
        const int off0 = tile_off<T, kCh>(2 * tp, kWCh * warp + 2 * pp), off1 = tile_off<T, kCh>(2 * tp + 1, kWCh * warp + 2 * pp);
        float2 bias = make_float2(0.f, 0.f), dsk = make_float2(0.f, 0.f);
        {
            const int64_t dc = (int64_t)d0 + kWCh * warp + 2 * pp;   // D % 8 == 0: both channels valid or neither
            if (dc < D) {
                if (p.dt_bias) bias = gld2(p.dt_bias + dc);
                if (p.D) dsk = gld2(p.D + dc);
            }
        }
        // widening role: two states of B or C at a step pair of every chunk (s.bc in the order of the threads)
        const int bc_off = ((2 * ((tid >> 2) & 7)) * kDState + 4 * (tid & 3) + 2 * ((tid >> 5) & 1)) * (int)sizeof(T);
        const bool bc_is_c = tid >= 64;

        // ---- scan role: channel c of the warp, states 4 q .. 4 q + 3 (the lane order of the file comment)
        const int c = (lane & 1) | ((lane >> 1) & 6), q = ((lane >> 1) & 1) | ((lane >> 4) << 1);
        const int64_t d = (int64_t)d0 + kWCh * warp + c;
        const bool chan_ok = d < D;
        float h[4], a2[4];
        float2 dsum = make_float2(0.f, 0.f);   // kSummary: sum of Delta over even and odd steps
        {
            float4 av = make_float4(0.f, 0.f, 0.f, 0.f), hv = av;
            if (chan_ok) {
                av = gld4(p.A + d * kDState + 4 * q);
                if (seg == 0 && tb == 0 && p.h0) hv = gld4(p.h0 + ((int64_t)b * D + d) * kDState + 4 * q);
                if constexpr (!kSummary) {
                    for (int sp = 0; sp < seg; ++sp) {
                        const int64_t o = (((int64_t)b * nseg + sp) * D + d) * kDState + 4 * q;
                        const float4 he = gld4(p.seg_h + o);
                        if (sp == 0) {
                            hv = he;
                        } else {
                            const float4 pe = gld4(p.seg_p + o);
                            hv = make_float4(fold(pe.x, hv.x, he.x), fold(pe.y, hv.y, he.y),
                                             fold(pe.z, hv.z, he.z), fold(pe.w, hv.w, he.w));
                        }
                    }
                }
            }
            a2[0] = av.x * kLog2e; a2[1] = av.y * kLog2e; a2[2] = av.z * kLog2e; a2[3] = av.w * kLog2e;
            h[0] = hv.x; h[1] = hv.y; h[2] = hv.z; h[3] = hv.w;
        }
        const int slot_e = dg_slot(0, c), slot_o = dg_slot(1, c);

        struct Conv {
            float4 c0, c1;
        };
        auto convert = [&](const R &r, int sub, int t0) {   // chunk `sub` of a stage, its first step t0
            constexpr int kSubB = kT * kRowB;
            const float2 x0 = ld2<T>(&r.x[0][0], off0 + sub * kSubB), x1 = ld2<T>(&r.x[0][0], off1 + sub * kSubB);
            float2 D0 = softplus2(add2(ld2<T>(&r.dt[0][0], off0 + sub * kSubB), bias));
            float2 D1 = softplus2(add2(ld2<T>(&r.dt[0][0], off1 + sub * kSubB), bias));
            const int rest = L - t0 - 2 * tp;   // steps left from this pair on
            const float m0 = rest < 1 ? 0.f : 1.f, m1 = rest < 2 ? 0.f : 1.f;
            D0 = mul2(D0, splat(m0));   // Delta = 0 past the end leaves h unchanged
            D1 = mul2(D1, splat(m1));
            const float2 g0 = mul2(D0, x0), g1 = mul2(D1, x1);
            return Conv{make_float4(D0.x, D1.x, g0.x, g1.x), make_float4(D0.y, D1.y, g0.y, g1.y)};
        };
        auto put = [&](int buf, const Conv &v) {
            s.dg[buf][warp][tp][dg_slot(tp, 2 * pp)] = v.c0;
            s.dg[buf][warp][tp][dg_slot(tp, 2 * pp + 1)] = v.c1;
        };
        struct Wide {
            float4 v[SUB];
        };
        auto widen = [&](const R &r) {
            Wide w;
            const T *src = !kSummary && bc_is_c ? &r.C[0][0] : &r.B[0][0];
#pragma unroll
            for (int u = 0; u < SUB; ++u) {
                const int o = bc_off + u * kT * kDState * (int)sizeof(T);
                const float2 v0 = ld2<T>(src, o), v1 = ld2<T>(src, o + kDState * (int)sizeof(T));
                w.v[u] = make_float4(v0.x, v1.x, v0.y, v1.y);
            }
            return w;
        };
        auto put_bc = [&](int buf, const Wide &w) {
#pragma unroll
            for (int u = 0; u < SUB; ++u) (&s.bc[buf][u][0][0][0][0])[tid] = w.v[u];
        };

        // ---- prologue: the first chunk, the first stage's B and C
        bool ok = mbar_wait(&s.full[st], ph);   // nch >= 1
        if (ok) {
            put(0, convert(s.raw[st], 0, tb));
            put_bc(0, widen(s.raw[st]));
        }
        if constexpr (kShares) {
            if (tid == 0) {
                bulk_wait_read_all();   // the piece before's last store no longer reads its output tile
                if (tb > 0) ok = flag_wait(p.share_sync() + share) && ok;   // share - 1's flag
            }
        }
        if (__syncthreads_or(ok ? 0 : 1)) {
            if (tid == 0) {
                report(p.status, 4 /* MB_ERR_TIMEOUT */, 0);
                for (int j = 0; j < STAGES && j < nch; ++j) {
                    mbar_wait(&s.full[st], ph);
                    st = st + 1 == STAGES ? 0 : st + 1;
                    ph ^= st == 0 ? 1u : 0u;
                }
                bulk_wait_all();
            }
            return;
        }
        if constexpr (kShares) {
            if (tb > 0 && chan_ok) {
                const float4 hv = __ldcg(reinterpret_cast<const float4 *>(
                    p.seg_h + ((int64_t)(share - 1) * kCh + kWCh * warp + c) * kDState + 4 * q));
                h[0] = hv.x; h[1] = hv.y; h[2] = hv.z; h[3] = hv.w;
            }
        }

        for (int i = 0; i < nch; ++i) {
            const int ts = tb + i * RT;   // its first step
            const R &r = s.raw[st];
            const int nst = st + 1 == STAGES ? 0 : st + 1;
            const uint32_t nph = st + 1 == STAGES ? ph ^ 1u : ph;
#pragma unroll
            for (int sub = 0; sub < SUB; ++sub) {
                const int t0 = ts + sub * kT;
                if (sub > 0 && t0 >= te) break;   // the span ends in an earlier chunk of this stage
                const int buf = SUB == 1 ? i & 1 : sub & 1;
                // (1) convert the next chunk, of this stage or (waiting for its tiles) the next one; past the last
                // chunk that is of no use, and not read. Stored after the scan below.
                const bool last = sub == SUB - 1;
                if (last) ok = i + 1 < nch ? mbar_wait(&s.full[nst], nph) : true;
                const Conv nv = last ? convert(s.raw[nst], 0, t0 + kT) : convert(r, sub + 1, t0 + kT);
                Wide nw;
                if (last) nw = widen(s.raw[nst]);
                // (2) D x and silu(z) of this lane's outputs
                const int o0 = off0 + sub * kT * kRowB, o1 = off1 + sub * kT * kRowB;
                float2 xd0, xd1, sz0 = splat(1.f), sz1 = sz0;
                if constexpr (!kSummary) {
                    xd0 = mul2(dsk, ld2<T>(&r.x[0][0], o0));
                    xd1 = mul2(dsk, ld2<T>(&r.x[0][0], o1));
                    if (gate) {
                        sz0 = silu2(ld2<T>(&r.z[0][0], o0));
                        sz1 = silu2(ld2<T>(&r.z[0][0], o1));
                    }
                }
                if constexpr (kCkpt) {   // state before the chunk, for the backward's recompute
                    static_assert(kT == kCkptSteps, "checkpoints are taken per chunk");
                    const int64_t nck = (L + kT - 1) / kT;
                    if (chan_ok)
                        *reinterpret_cast<float4 *>(p.h_ckpt + (((int64_t)b * nck + t0 / kT) * D + d) * kDState + 4 * q) =
                            make_float4(h[0], h[1], h[2], h[3]);
                }
                // (3) decays, recurrence, shares of C.h, a step pair at a time
                const float4(&dgw)[kTP][kWCh] = s.dg[buf][warp];
                const float4(&bcw)[2][2][kTP][4] = s.bc[i & 1][sub];
                float2 part[kTP], csum;
#pragma unroll
                for (int k = 0; k < kTP; ++k) {
                    const float4 v = dgw[k][(k & 1) ? slot_o : slot_e];
                    const float2 dd = make_float2(v.x, v.y), gg = make_float2(v.z, v.w);
                    const float4 b01 = bcw[0][0][k][q], b23 = bcw[0][1][k][q];
                    const float2 bp[4] = {make_float2(b01.x, b01.y), make_float2(b01.z, b01.w),
                                          make_float2(b23.x, b23.y), make_float2(b23.z, b23.w)};
                    float2 hp[4];
#pragma unroll
                    for (int n = 0; n < 4; ++n) {
                        const float2 e = mul2(dd, splat(a2[n]));
                        const float2 ab = make_float2(ex2(e.x), ex2(e.y));
                        const float2 bg = mul2(bp[n], gg);
                        hp[n].x = fmaf(ab.x, h[n], bg.x);
                        hp[n].y = fmaf(ab.y, hp[n].x, bg.y);
                        h[n] = hp[n].y;
                    }
                    if constexpr (kSummary) {
                        csum = k == 0 ? dd : add2(csum, dd);
                    } else {
                        const float4 c01 = bcw[1][0][k][q], c23 = bcw[1][1][k][q];
                        part[k] = mul2(make_float2(c01.x, c01.y), hp[0]);
                        part[k] = fma2(make_float2(c01.z, c01.w), hp[1], part[k]);
                        part[k] = fma2(make_float2(c23.x, c23.y), hp[2], part[k]);
                        part[k] = fma2(make_float2(c23.z, c23.w), hp[3], part[k]);
                    }
                }
                if constexpr (kSummary) dsum = add2(dsum, csum);
                // Not needed for order (other slots are read above): it keeps these stores behind the scan, 717 -> 711 us
                // on 8 x 8192 x 2048.
                if (!last) __syncwarp();
                put(buf ^ 1, nv);
                if (last) put_bc((i + 1) & 1, nw);
                // (4) add the four lanes' shares of each channel, skip term, gate
                if constexpr (!kSummary) {
                    float4 *pw = s.part[warp];
                    if (sub > 0) __syncwarp();   // the shares of the chunk before have been read
#pragma unroll
                    for (int k = 0; k < kTP; ++k) reinterpret_cast<float2 *>(pw + q * kPartQ + k * kPairs)[c] = part[k];
                    __syncwarp();
                    const float4 *src = pw + tp * kPairs + pp;   // (channel, step): (0, 0), (0, 1), (1, 0), (1, 1)
                    const float4 s0 = src[0], s1 = src[kPartQ], s2 = src[2 * kPartQ], s3 = src[3 * kPartQ];
                    const float2 ca = add2(add2(make_float2(s0.x, s0.y), make_float2(s1.x, s1.y)),
                                           add2(make_float2(s2.x, s2.y), make_float2(s3.x, s3.y)));
                    const float2 cb = add2(add2(make_float2(s0.z, s0.w), make_float2(s1.z, s1.w)),
                                           add2(make_float2(s2.z, s2.w), make_float2(s3.z, s3.w)));
                    st2<T>(&s.ys[i & 1][0][0], o0, mul2(add2(make_float2(ca.x, cb.x), xd0), sz0));
                    st2<T>(&s.ys[i & 1][0][0], o1, mul2(add2(make_float2(ca.y, cb.y), xd1), sz1));
                } else if (!last) {
                    __syncwarp();
                }
            }
            if constexpr (!kSummary) {
                fence_proxy_async_smem();   // y tile -> visible to the TMA store below
                if (tid == 0) bulk_wait_read_all();   // the store of stage i - 1 no longer reads its tile
            }
            if (__syncthreads_or(ok ? 0 : 1)) {
                if (tid == 0) {
                    report(p.status, 4 /* MB_ERR_TIMEOUT */, i + 1);
                    for (int j = i + 1; j < i + STAGES && j < nch; ++j) {
                        st = st + 1 == STAGES ? 0 : st + 1;
                        ph ^= st == 0 ? 1u : 0u;
                        mbar_wait(&s.full[st], ph);
                    }
                    bulk_wait_all();
                }
                return;
            }
            if (tid == 0) {
                if constexpr (!kSummary) {
#pragma unroll
                    for (int u = 0; u < SUB; ++u)   // the last stage may end in any chunk; what follows it is not this CTA's
                        if (ts + u * kT < te) tma_store_3d(&a.tm_y, &s.ys[i & 1][u * kT][0], d0, ts + u * kT, b);
                    bulk_commit();
                }
                if (i + STAGES < nch) {   // the slot is free: refill it with stage i + STAGES
                    fence_proxy_async_smem();
                    issue_chunk<T, kSummary, W>(s, a, st, tb + (i + STAGES) * RT, d0, b);
                }
            }
            st = nst;
            ph = nph;
        }
        if constexpr (kSummary) pdl_trigger();   // the second pass may set up while the last summaries are written
        if (!kShares && tid == 0) bulk_wait_all();

        if constexpr (kSummary) {
            if (chan_ok) {
                const int64_t o = (((int64_t)b * nseg + seg) * D + d) * kDState + 4 * q;
                const float sd = dsum.x + dsum.y;
                *reinterpret_cast<float4 *>(p.seg_h + o) = make_float4(h[0], h[1], h[2], h[3]);
                *reinterpret_cast<float4 *>(p.seg_p + o) =
                    make_float4(ex2(a2[0] * sd), ex2(a2[1] * sd), ex2(a2[2] * sd), ex2(a2[3] * sd));
            }
        } else if (te == L) {   // the span's last state
            if (p.h_out && chan_ok)
                *reinterpret_cast<float4 *>(p.h_out + ((int64_t)b * D + d) * kDState + 4 * q) =
                    make_float4(h[0], h[1], h[2], h[3]);
        } else if constexpr (!kShares) {
            if (seg == 0 && chan_ok)   // first pass: the first segment's end
                *reinterpret_cast<float4 *>(p.seg_h + ((int64_t)b * nseg * D + d) * kDState + 4 * q) =
                    make_float4(h[0], h[1], h[2], h[3]);
        } else {   // the share ends here: leave the state for the next one
            __stcg(reinterpret_cast<float4 *>(p.seg_h + ((int64_t)share * kCh + kWCh * warp + c) * kDState + 4 * q),
                   make_float4(h[0], h[1], h[2], h[3]));
            __threadfence();
            __syncthreads();
            if (tid == 0) flag_set(p.share_sync() + 1 + share);
        }
        if (!kShares || tile * units <= lo) break;
        --tile;
    }
    if (kShares && tid == 0) bulk_wait_all();
}

template <typename T, bool kCkpt, bool W>
__global__ void __launch_bounds__(kThreads, kCtas<W>) forward_kernel(const __grid_constant__ FwdArgs a) {
    scan_spans<T, kCkpt, false, false, W>(a);
}

template <typename T, bool kCkpt>
__global__ void __launch_bounds__(kThreads, kCtas<true>) forward_shares_kernel(const __grid_constant__ FwdArgs a) {
    scan_spans<T, kCkpt, false, true, true>(a);
}

template <typename T, bool kCkpt, bool W>
__global__ void __launch_bounds__(kThreads, kCtas<W>) first_pass_kernel(const __grid_constant__ FwdArgs a) {
    if (blockIdx.x < a.p.batch * ((a.p.d_inner + kCh - 1) / kCh))   // segment 0
        scan_spans<T, kCkpt, false, false, W>(a);
    else
        scan_spans<T, kCkpt, true, false, W>(a);
}

// ---------------------------------------------------------------------------
// Host side: tensor maps and the launch.

// [batch, L, inner] tensor with a (box_inner x rows x 1) box; rows (b, t) are
// `row` elements apart (row >= inner).
bool make_map(CUtensorMap *m, const void *base, int es, int64_t batch, int64_t L, int64_t inner, int box_inner,
              int64_t row, int swizzle, int rows) {
    const uint64_t dims[3] = {(uint64_t)inner, (uint64_t)L, (uint64_t)batch};
    const uint64_t strides[2] = {(uint64_t)(row * es), (uint64_t)(L * row * es)};
    const uint32_t box[3] = {(uint32_t)box_inner, (uint32_t)rows, 1};
    return encode_tmap(m, base, es, 3, dims, strides, box, swizzle);
}

// Split of a span into at most nseg segments, in whole chunks. The first
// is scanned for good while the others are summarised, which takes kFirst of its time per step, and is that much shorter
// (0.55 to 0.85 make no difference, bf16 1 x 8192 x 2048 and fp32 3 x 1003 x 1544).
constexpr double kFirst = 0.7;
struct Segments {
    int64_t n, len0, len;   // n <= nseg
};
Segments segments(int64_t L, int64_t nseg) {
    if (nseg < 2) return {1, L, L};
    const int64_t units = (L + kT - 1) / kT;
    int64_t others = (int64_t)((double)units / ((double)(nseg - 1) + kFirst));
    if (others < 1 || units - others * (nseg - 1) > others) ++others;   // the first is the shorter
    const int64_t m = std::min(nseg - 1, (units - 1) / others);
    return {m + 1, (units - m * others) * kT, others * kT};
}

template <typename T, bool kCkpt, bool W>
cudaError_t launch_form(const ScanParams &p, const Segments &g, int64_t grid, const DeviceLimits *lim, cudaStream_t s) {
    constexpr int es = sizeof(T), sw = kCh * es;   // one token row of a tile
    FwdArgs a;
    memset(&a, 0, sizeof(a));
    a.p = p;
    a.has_gate = p.z != nullptr;
    a.len0 = (int)g.len0;
    a.len = (int)g.len;
    const int64_t D = p.d_inner;
    auto tok = [&](CUtensorMap *m, const void *base, int rows = kRT<T, W>) {
        return make_map(m, base, es, p.batch, p.seqlen, D, kCh, D, sw, rows);
    };
    if (!tok(&a.tm_dt, p.dt) || !tok(&a.tm_x, p.x) || (p.z && !tok(&a.tm_z, p.z)) || !tok(&a.tm_y, p.y, kT) ||
        !make_map(&a.tm_B, p.B, es, p.batch, p.seqlen, kDState, kDState, p.bc_stride, 0, kRT<T, W>) ||
        !make_map(&a.tm_C, p.C, es, p.batch, p.seqlen, kDState, kDState, p.bc_stride, 0, kRT<T, W>))
        return cudaErrorInvalidValue;
    const size_t smem = sizeof(Smem<T, W>) + 1024;
    auto launch = [&](auto k, Placement at) {
        const cudaError_t e =
            cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)lim->smem_optin);
        if (e != cudaSuccess) return e;
        return launch_pdl(at.overlap, k, dim3((unsigned)grid), dim3(kThreads), at.smem, s, a);
    };
    cudaError_t e;
    if (g.n > 1) {   // first pass: segments 0 .. n-2
        if ((e = launch(first_pass_kernel<T, kCkpt, W>, {true, smem})) != cudaSuccess) return e;
        a.seg0 = 1;   // second pass: segments 1 .. n-1
        return launch(forward_kernel<T, kCkpt, W>, {true, smem});
    }
    if constexpr (W) {
        if (p.shares > 0) {
            if ((e = cudaMemsetAsync(p.share_sync(), 0, prefill_share_sync_bytes(p.shares), s)) != cudaSuccess) return e;
            return launch(forward_shares_kernel<T, kCkpt>, {true, spread_smem(smem, grid, kCtas<W>)});
        }
    }
    return launch(forward_kernel<T, kCkpt, W>, place_scan(p.seqlen, grid, kCtas<W>, smem));
}

template <typename T, bool kCkpt>
cudaError_t launch_typed(ScanParams p, cudaStream_t s) {
    const DeviceLimits *lim = device_limits();
    if (!lim) return cudaErrorInvalidDevice;
    if (p.nseg < 2 || !p.seg_h || !p.seg_p) p.nseg = 1;
    const Segments g = segments(p.seqlen, p.nseg);
    const int64_t ctas = ((p.d_inner + kCh - 1) / kCh) * p.batch;   // per segment of L
    const int64_t grid = g.n > 1 ? ctas * (g.n - 1) : p.shares > 0 ? p.shares : ctas;
    return p.shares > 0 || grid <= kCtas<true> * lim->sms ? launch_form<T, kCkpt, true>(p, g, grid, lim, s)
                                                          : launch_form<T, kCkpt, false>(p, g, grid, lim, s);
}

}  // namespace

// Time split: only when the batch rows and channel tiles give at most one CTA
// per SM (a CTA alone on an SM leaves most of its issue slots idle; the summary
// pass repeats most of a scan, so at 1.7 CTAs per SM, batch 4 x 2048 channels,
// the split measured slower) and the span is long enough to pay for the second
// launch: at 128 steps x 2048 channels unsplit 8.5 us, split 10.3; at 256 steps
// 14.4 and 12.3. Both passes run all segments but one, with at most 3 CTAs per SM
// (wide form) or 4: of the two numbers, the one with the less chunks x time per
// chunk of the SM that holds the most. (Microseconds with 3 and 4: bf16 1 x 4096 x
// 4608 130, 133; fp32 2 x 3000 x 1536 84, 77; 1 x 777 x 3584 25.2, 27.7; bf16 1 x
// 4096 x 4608 with 2: 139.) Every lane folds the summaries before its segment,
// about 0.07 us each, while a step costs about 0.1 us over both passes: their sum
// is least at sqrt(1.4 L) segments, which bounds spans of very few channels
// (8192 x 64: 86 segments 20 us, 256 segments 35 us, 16 segments 37 us; fp32
// 256 x 64: 8 segments 8.4 us, 2 segments 14.4 us).
// With the first segment summarised like the others, and scanned in the second
// pass: bf16 1 x 8192 x 2048 139 us (then 126, wide 122), fp32 3 x 1003 x 1544 42.7
// (then 40.7, wide 39.8).
constexpr int64_t kMinSplitSteps = 256;
constexpr double kFoldUs = 0.07;
// Microseconds per chunk of an SM's CTAs, 1 to 4 of them, as measured (fp32, bf16)
constexpr double kChunkUs[2][kResident] = {{0.79, 0.93, 1.20, 1.55}, {0.56, 0.78, 1.07, 1.40}};

int64_t prefill_segments(const ScanParams &p, bool bf16) {
    if (p.batch <= 0 || p.d_inner <= 0 || p.seqlen < kMinSplitSteps || p.dt_low) return 1;
    const int64_t sms = device_sms();
    const int64_t ctas = p.batch * ((p.d_inner + kCh - 1) / kCh);
    if (ctas > sms) return 1;
    const int64_t most = std::min((p.seqlen + kSegUnit - 1) / kSegUnit, (int64_t)sqrt(1.4 * (double)p.seqlen));
    int64_t best = 1;
    double least = 0;
    for (int64_t m = kCtas<true>; m <= kCtas<false>; ++m) {
        const int64_t nseg = std::min(m * sms / ctas + 1, most);
        if (nseg < 3) continue;   // two: one after the other
        const Segments g = segments(p.seqlen, nseg);
        const int64_t per_sm = (ctas * (g.n - 1) + sms - 1) / sms;
        const double us = (1 + kFirst) * kChunkUs[bf16][per_sm - 1] * (double)(g.len / kT) + kFoldUs * (double)g.n;
        if (best == 1 || us < 0.97 * least) {   // fewer segments at equal time: less summarised
            best = nseg;
            least = us;
        }
    }
    return best;
}

size_t prefill_split_bytes(const ScanParams &p, int64_t nseg) {
    return nseg > 1 ? (size_t)(2 * p.batch * nseg * p.d_inner * kDState) * sizeof(float) : 0;
}

// Even shares: CTAs of one tile each leave the GPU unevenly loaded when their
// number is little over a multiple of the SMs: the SMs that hold one more set
// the time (8 x 8192 x 2048: 512 tiles, 3.4 per SM). Then m = tiles / SMs
// (rounded down, at most 3: the wide form) CTAs per SM take equal shares of all
// tiles' steps. Microseconds per chunk of an SM's CTAs, 1 to 4 of them, as
// measured (kChunkUs, kShareUs; 4: the narrow form):
//                        bf16                  fp32
//   one CTA per tile     0.56 0.78 1.07 1.40   0.79 0.93 1.20 1.55
//   shares               0.63 0.83 1.10        0.87 1.02 1.22
// so m CTAs per SM finish tiles in tiles / (m SMs) times the second row, plus
// about 7 us for the clearing of the flags and the second prologue, against the
// first row's next number for one CTA per tile. More tiles than slots run in
// waves; the last one, of r per SM, takes about 0.85 of its number (its CTAs
// start as others end). Measured (bf16): 8 x 8192 x 2048 (3.4 tiles per SM)
// 709 -> 623 us, its training forward 740 -> 650 us; spans of 2048 steps at 2.1,
// 3.2, 3.4 and 4.3 tiles per SM 136 -> 118, 182 -> 156, 182 -> 164, 242 -> 209 us.
constexpr double kShareUs[2][kCtas<true>] = {{0.87, 1.02, 1.22}, {0.63, 0.83, 1.10}};

int64_t prefill_shares(const ScanParams &p, bool bf16) {
    if (p.batch <= 0 || p.d_inner <= 0 || p.seqlen < kMinSplitSteps || p.dt_low) return 0;
    const int64_t sms = device_sms(), tiles = p.batch * ((p.d_inner + kCh - 1) / kCh);
    if (sms <= 0 || tiles <= sms) return 0;
    const int64_t m = std::min<int64_t>(tiles / sms, kCtas<true>), rest = tiles % (kResident * sms);
    double plain = (double)(tiles / (kResident * sms)) * kChunkUs[bf16][kResident - 1];
    if (rest) plain += (tiles > rest ? 0.85 : 1.0) * kChunkUs[bf16][(rest - 1) / sms];
    const double even = (double)tiles / (double)(m * sms) * kShareUs[bf16][m - 1];
    const double chunks = (double)(p.seqlen / kT);
    return even * chunks + 7.0 < 0.97 * plain * chunks ? m * sms : 0;
}

size_t prefill_share_sync_bytes(int64_t shares) { return ((size_t)(shares + 1) * sizeof(int) + 255) / 256 * 256; }

size_t prefill_share_bytes(int64_t shares) {
    return shares > 0 ? prefill_share_sync_bytes(shares) + (size_t)shares * kCh * kDState * sizeof(float) : 0;
}

cudaError_t launch_forward(const ScanParams &p, bool bf16, cudaStream_t s) {
    if (p.h_ckpt)
        return bf16 ? launch_typed<__nv_bfloat16, true>(p, s) : launch_typed<float, true>(p, s);
    return bf16 ? launch_typed<__nv_bfloat16, false>(p, s) : launch_typed<float, false>(p, s);
}

}  // namespace mbscan
