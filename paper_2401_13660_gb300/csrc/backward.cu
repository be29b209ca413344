// Backward of the selective-scan layer core: the training path (MambaByte
// trains through this scan, Section 2 "parallel scans"; Section 4 setup).
// Given the forward inputs, the state checkpoints of the training forward
// (the state before every kCkptSteps-step chunk) and dJ/dout, dJ/dh_last, it
// returns every input gradient. For each (batch row, channel), from t = L-1
// down to 0, with g = dJ/dh_t:
//   dy = dout * silu(z);  dz = dout * y * silu'(z);  g += dy * C_t
//   dC_t += dy * h_t (summed over channels);  S1 = sum_n g B_t
//   dx = dy * D + Delta * S1;  dDelta = x * S1 + sum_n (g Abar h_{t-1}) A
//   dB_t += g * Delta * x (summed over channels);  dA += (g Abar h_{t-1}) Delta
//   g *= Abar;  ddt = dDelta * sigmoid(dt + bias);  dbias += ddt;  dD += dy x
// and dh0 = g at the end.
//
// Work decomposition. A CTA of two warps owns 32 channels of one batch row;
// four lanes share a channel pair, each with 4 states of both channels. Chunks
// of kCkptSteps steps are taken in reverse order through a ring of TMA tiles
// (dt, x, z, dout, B, C). Per chunk:
//  * conversion, once per (step, channel): Delta, Delta x, dy, sigmoid(dt +
//    bias) and the gate's factor of dz; B and C widened to fp32. Everything is
//    kept for pairs of adjacent steps, which fill the packed operations as in
//    forward.cu;
//  * the state before step 8, from the checkpoint; then for steps 8..15 and
//    then 0..7: their states and decays, forward, into registers (with each
//    lane's share of C.h), and the reverse sweep over them: the adjoint g and
//    dA in registers, each lane's shares of S1 and S2, and dB, dC;
//  * dB, dC of a step are sums over channels. A lane adds its own two; lanes
//    that differ in a channel bit exchange what they do not keep. Lanes hold
//    their four states in the order r -> r ^ perm with perm = their two low
//    channel bits (B and C lie in shared memory in both orders of a pair), so
//    that what is kept and sent is the same register on every lane: 7 shuffles
//    and 2 selects for 8 values. The warps' sums are added when the chunk is
//    done and sent to global memory with vector atomics;
//  * the shares of C.h, S1 and S2 are added through a warp's own tile; the lane
//    that adds them finishes dx, ddt, dz of those channels and steps (output
//    tiles written by TMA stores).
// dA, dD, dbias are accumulated in registers and added atomically at the end;
// dh0 is stored directly. Segments of a time-split span (backward_segments)
// start from the adjoints that a first pass (kSummary) leaves: each segment's
// adjoint from a zero one at its end, and its product of decays.
//
// What bounds it: issue at 2 warps per scheduler (registers hold half a chunk's
// states and decays: 254 of them), of which a loop of the core instructions
// alone reaches 0.52 per clock; it runs at 0.51. Two channels per lane halve
// the loads of B and C and the exchange of dB, dC per channel. Measured (8 x
// 8192 x 2048 bf16): 3.23 -> 2.43 ms, 2.08 -> 1.40 G warp instructions; before,
// the four warps added dB, dC with shared float atomics, a compare-and-swap loop
// that cost 5.5 clocks per instruction and kept the compiler from moving code
// across steps. Variants: quarters of a chunk in registers (193 registers, a
// longer first pass over the states) 2.63 ms, eighths 4.28 ms; both halves
// unrolled 3.38 ms (spills); states of the halves in registers instead of
// shared memory 2.74 ms.
#include <math.h>
#include <stddef.h>
#include <string.h>

#include "common.cuh"
#include "pairs.cuh"
#include "tma.cuh"

namespace mbscan {
namespace {

constexpr int kBT = kCkptSteps;            // steps per chunk
constexpr int kBTP = kBT / 2;              // step pairs per chunk
constexpr int kHTP = kBTP / 2;             // step pairs per half chunk
constexpr int kBWarps = 2;
constexpr int kBThreads = 32 * kBWarps;
constexpr int kBWCh = 16;                  // channels per warp, two per lane
constexpr int kBPairs = kBWCh / 2;
constexpr int kBCh = kBWarps * kBWCh;      // channels per CTA
constexpr int kBStages = 2;
// CTAs per SM: four by registers, fp32 three by shared memory (61 KB each)
template <typename T>
constexpr int kBResident = sizeof(T) == 2 ? 4 : 3;
constexpr int kShareQ = kHTP * kBPairs + 2;   // float4s between the shares of two lanes q (the pad moves them to other banks)

template <typename T>
struct BRaw {   // TMA destinations; token tiles swizzled in their 64- (bf16) or 128-byte (fp32) rows
    T dt[kBT][kBCh];
    T x[kBT][kBCh];
    T z[kBT][kBCh];
    T dout[kBT][kBCh];
    T B[kBT][kDState];
    T C[kBT][kDState];
};

template <typename T>
struct alignas(1024) BSmem {
    BRaw<T> raw[kBStages];
    T gx[kBT][kBCh], gdt[kBT][kBCh], gz[kBT][kBCh];   // output tiles (TMA stores), swizzled like the inputs
    float4 dg[kBWarps][kBTP][2][kBPairs];   // (Delta_t, Delta_t+1, (Delta x)_t, (Delta x)_t+1) of channel 2 j + k: [k][j]
    float4 dy[kBWarps][kBTP][kBPairs];      // dJ/dy: channel 2 j (t, t+1), channel 2 j + 1 (t, t+1)
    float4 bc[2][kBTP][4][4];               // B, C: [tp][q][2 h + s]: states 4q + 2h + s, 4q + 2h + 1 - s (t, t+1 each)
    float4 share[kBWarps][3][4 * kShareQ];  // shares of C.h, g.B, sum g Abar h A log2 e of lane q: [q][tp of the half][j]
    float4 fin[kBWarps][2][kBTP][kBPairs];  // sigmoid(dt + bias); dout d(gate)/dz: channels 2 j, 2 j + 1 at t, at t + 1
    float4 hq[kBWarps][2][2][32];           // states before each half of the chunk: [half][channel][lane]
    float2 sum[kBWarps][kBTP][32];          // the warp's dB, dC (t, t+1): [tp][8 q + 4 (dC) + state]
    uint64_t full[kBStages];
    int ticket;
};

struct BwdArgs {
    CUtensorMap tm_dt, tm_x, tm_z, tm_dout, tm_B, tm_C, tm_dx, tm_ddt, tm_dz;
    ScanParams p;
    GradParams g;
    int has_gate;
    int grid_segs, seg0;   // segments of L covered by the grid (blockIdx = (b, segment - seg0, channel tile))
};

template <typename T, bool kSummary>
__device__ __forceinline__ void issue_bchunk(BSmem<T> &s, const BwdArgs &a, int stage, int chunk, int d0, int b) {
    constexpr uint32_t tok = kBT * kBCh * sizeof(T), bc = kBT * kDState * sizeof(T);
    const uint32_t bytes = ((a.has_gate ? 3 : 2) + (kSummary ? 0 : 1)) * tok + (kSummary ? 1 : 2) * bc;
    uint64_t *bar = &s.full[stage];
    mbar_arrive_expect_tx(bar, bytes);
    const int t = chunk * kBT;
    BRaw<T> &r = s.raw[stage];
    tma_load_3d(&r.dt[0][0], &a.tm_dt, bar, d0, t, b);
    if (!kSummary) tma_load_3d(&r.x[0][0], &a.tm_x, bar, d0, t, b);
    if (a.has_gate) tma_load_3d(&r.z[0][0], &a.tm_z, bar, d0, t, b);
    tma_load_3d(&r.dout[0][0], &a.tm_dout, bar, d0, t, b);
    if (!kSummary) tma_load_3d(&r.B[0][0], &a.tm_B, bar, 0, t, b);
    tma_load_3d(&r.C[0][0], &a.tm_C, bar, 0, t, b);
}

// Delta = softplus(v) (as softplus2) and sigmoid(v) = u / (1 + u), u = e^v, 1 above v = 15 (1 - 3e-7 there)
__device__ __forceinline__ void softplus_sigmoid2(float2 v, float2 &delta, float2 &sig) {
    const float2 w = mul2(v, splat(kLog2e));
    const float2 u = make_float2(ex2(w.x), ex2(w.y));
    const float2 o = add2(u, splat(1.f));
    delta = softplus_of(v, u, o);
    sig = mul2(u, make_float2(rcp(o.x), rcp(o.y)));
    sig.x = v.x > 15.f ? 1.f : sig.x;
    sig.y = v.y > 15.f ? 1.f : sig.y;
}

// Four values of a lane's permuted state order (register r: state r ^ perm) from a row of four. kOnce: read this once
// and never again (checkpoints), past the L1 cache (8 x 8192 x 2048 with the forward: 3082 us, through it 3104); the
// few rows that every segment folds are better off in it (2 x 777 x 1544: 89.1 us, past it 89.9).
template <bool kOnce = false>
__device__ __forceinline__ void load_perm(float (&v)[4], const float *row, int perm) {
    const float *plo = row + (perm & 2), *phi = row + 2 - (perm & 2);
    const float2 lo = kOnce ? __ldcg(reinterpret_cast<const float2 *>(plo)) : gld2(plo);
    const float2 hi = kOnce ? __ldcg(reinterpret_cast<const float2 *>(phi)) : gld2(phi);
    const bool s = perm & 1;
    v[0] = s ? lo.y : lo.x;
    v[1] = s ? lo.x : lo.y;
    v[2] = s ? hi.y : hi.x;
    v[3] = s ? hi.x : hi.y;
}
__device__ __forceinline__ void store_perm(float *row, const float (&v)[4], int perm) {
    const bool s = perm & 1;
    *reinterpret_cast<float2 *>(row + (perm & 2)) = s ? make_float2(v[1], v[0]) : make_float2(v[0], v[1]);
    *reinterpret_cast<float2 *>(row + 2 - (perm & 2)) = s ? make_float2(v[3], v[2]) : make_float2(v[2], v[3]);
}

// dB, dC of one chunk: add the warps' sums to global memory (thread: step pair tid / 8, states 4q..4q+3 of dB or dC)
template <typename T>
__device__ __forceinline__ void flush_sums(const BSmem<T> &s, const GradParams &g, int64_t b, int t0, int64_t L) {
    static_assert(kBTP * 8 == kBThreads, "one thread per step pair and group of four");
    const int k = threadIdx.x >> 3, grp = threadIdx.x & 7;
    float4 lo = make_float4(0.f, 0.f, 0.f, 0.f), hi = lo;   // steps t, t + 1
#pragma unroll
    for (int w = 0; w < kBWarps; ++w) {
        const float4 *r = reinterpret_cast<const float4 *>(&s.sum[w][k][4 * grp]);
        const float4 u = r[0], v = r[1];
        lo = make_float4(lo.x + u.x, lo.y + u.z, lo.z + v.x, lo.w + v.z);
        hi = make_float4(hi.x + u.y, hi.y + u.w, hi.z + v.y, hi.w + v.w);
    }
    float *dst = ((grp & 1) ? g.dC : g.dB) + ((b * L + t0 + 2 * k) * kDState + 4 * (grp >> 1));
    if (t0 + 2 * k < L) atomicAdd(reinterpret_cast<float4 *>(dst), lo);
    if (t0 + 2 * k + 1 < L) atomicAdd(reinterpret_cast<float4 *>(dst + kDState), hi);
}

// kShares: as in forward.cu, the grid is p.shares CTAs of equal shares of all
// tiles' chunks (in the order the sweep takes them, the last chunk first); a
// share that ends inside a tile leaves the adjoint for the next one.
template <typename T, bool kSummary, bool kShares = false>
__global__ void __launch_bounds__(kBThreads, kBResident<T>) backward_kernel(const __grid_constant__ BwdArgs a) {
    constexpr int S = kBStages, kRowB = kBCh * (int)sizeof(T);
    using R = BRaw<T>;
    using SM = BSmem<T>;
    static_assert(sizeof(R) % (8 * kRowB) == 0 && offsetof(R, x) % (8 * kRowB) == 0 && offsetof(R, z) % (8 * kRowB) == 0 &&
                      offsetof(R, dout) % (8 * kRowB) == 0 && offsetof(R, B) % 128 == 0 && offsetof(R, C) % 128 == 0 &&
                      offsetof(SM, gx) % (8 * kRowB) == 0 && offsetof(SM, gdt) % (8 * kRowB) == 0 &&
                      offsetof(SM, gz) % (8 * kRowB) == 0,
                  "swizzled TMA tiles start on their pattern's boundary");
    extern __shared__ unsigned char smem_dyn[];
    const uint32_t sbase = (1024u - (smem_u32(smem_dyn) & 1023u)) & 1023u;
    SM &s = *reinterpret_cast<SM *>(smem_dyn + sbase);
    const ScanParams &p = a.p;
    const GradParams &gp = a.g;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int64_t D = p.d_inner;
    const int ntd = (int)((D + kBCh - 1) / kBCh);
    const int L = (int)p.seqlen;
    const int nchunks = (L + kBT - 1) / kBT;
    const int nseg = p.nseg > 1 ? (int)p.nseg : 1, cps = (nchunks + nseg - 1) / nseg;
    const int seg = kShares ? 0 : a.seg0 + (int)((blockIdx.x / ntd) % a.grid_segs);
    const bool gate = a.has_gate != 0;

    if (tid == 0) {
        for (int st = 0; st < S; ++st) mbar_init(&s.full[st], 1);
        fence_mbar_init();
    }
    __syncthreads();
    pdl_wait();   // everything below reads or writes global memory

    int tile = (int)(blockIdx.x / ntd / a.grid_segs) * ntd + (int)(blockIdx.x % ntd);   // batch row, 32 channels
    int share = 0, lo = 0, hi = 0;   // kShares: chunks lo .. hi - 1 of all tiles' sweeps end to end
    int n0 = 0;                      // ring stages consumed by the pieces before
    if constexpr (kShares) {
        if (tid == 0) s.ticket = atomicAdd(p.share_sync(), 1);
        __syncthreads();
        share = s.ticket;
        const int total = (int)p.batch * ntd * nchunks, len = (total + (int)p.shares - 1) / (int)p.shares;
        lo = min(share * len, total);
        hi = min(lo + len, total);
        if (lo == hi) return;
        tile = (hi - 1) / nchunks;
    }
    for (;;) {   // pieces: one without kShares
        const int b = tile / ntd, d0 = (tile % ntd) * kBCh;
        // chunks c0 + nch - 1 down to c0
        const int c0 = kShares ? max(nchunks - (hi - tile * nchunks), 0) : seg * cps;
        const int nch = (kShares ? nchunks - max(lo - tile * nchunks, 0) : min(nchunks, c0 + cps)) - c0;
        if (tid == 0) {
            fence_proxy_async_smem();
            for (int j = 0; j < S && j < nch; ++j) issue_bchunk<T, kSummary>(s, a, (n0 + j) % S, c0 + nch - 1 - j, d0, b);
        }

        // ---- conversion and finishing role: channels 16 warp + 2 pp + {0, 1} of the tile, step pairs ts and ts + 4
        const int wc0 = kBWCh * warp, pp = lane & 7, ts = lane >> 3;
        int off[2][2];
#pragma unroll
        for (int u = 0; u < 2; ++u)
#pragma unroll
            for (int e = 0; e < 2; ++e) off[u][e] = tile_off<T, kBCh>(2 * (ts + kHTP * u) + e, wc0 + 2 * pp);
        float2 bias = make_float2(0.f, 0.f), dsk = bias, dD_acc = bias, db_acc = bias;
        const int64_t dc = (int64_t)d0 + wc0 + 2 * pp;   // D % 8 == 0: both channels valid or neither
        if (dc < D) {
            if (p.dt_bias) bias = gld2(p.dt_bias + dc);
            if (p.D) dsk = gld2(p.D + dc);
        }

        // ---- scan role: channels 2 cl, 2 cl + 1 of the warp, states 4 q .. 4 q + 3 in the order r -> r ^ perm
        const int cl = ((lane >> 2) & 3) | ((lane & 1) << 2), q = ((lane >> 1) & 1) | ((lane >> 4) << 1);
        const int perm = cl & 3;
        const int ix0 = perm, ix1 = perm ^ 2;   // slots of s.bc that hold registers 0, 1 and 2, 3
        const int64_t d = (int64_t)d0 + wc0 + 2 * cl;
        const bool chan_ok = d < D;
        float a2[2][4], g[2][4];   // A log2 e; the adjoint Abar_{t+1} g_{t+1} on its way down
        float2 dA[2][4];           // even and odd steps
        float2 dsum[2];            // kSummary: sum of Delta
#pragma unroll
        for (int j = 0; j < 2; ++j) {
#pragma unroll
            for (int n = 0; n < 4; ++n) {
                a2[j][n] = g[j][n] = 0.f;
                dA[j][n] = make_float2(0.f, 0.f);
            }
            dsum[j] = make_float2(0.f, 0.f);
            if (chan_ok) {
                load_perm(a2[j], p.A + (d + j) * kDState + 4 * q, perm);
#pragma unroll
                for (int n = 0; n < 4; ++n) a2[j][n] *= kLog2e;
                if (kShares ? c0 + nch == nchunks : seg == nseg - 1) {
                    if (gp.dh_last) load_perm(g[j], gp.dh_last + ((int64_t)b * D + d + j) * kDState + 4 * q, perm);
                } else if (!kSummary && !kShares) {   // the last segment's summary starts from dh_last: fold down to this one
                    for (int sp = nseg - 1; sp > seg; --sp) {
                        const int64_t o = (((int64_t)b * nseg + sp) * D + d + j) * kDState + 4 * q;
                        float ge[4], pe[4];
                        load_perm(ge, p.seg_h + o, perm);
                        load_perm(pe, p.seg_p + o, perm);
#pragma unroll
                        for (int n = 0; n < 4; ++n) g[j][n] = sp == nseg - 1 ? ge[n] : fold(pe[n], g[j][n], ge[n]);
                    }
                }
            }
        }

        // Byte offsets (from smem_dyn) of what the scan's loops read and write, opaque to the compiler: it would compute
        // them again at every use rather than keep them.
        auto fixed = [&](size_t o) {
            uint32_t v = sbase + (uint32_t)o;
            asm volatile("" : "+r"(v));
            return v;
        };
        const uint32_t o_bc0 = fixed(offsetof(SM, bc) + (q * 4 + ix0) * 16), o_bc1 = o_bc0 + (ix1 - ix0) * 16;
        const uint32_t o_dg = fixed(offsetof(SM, dg) + (warp * kBTP * 2 * kBPairs + cl) * 16);
        const uint32_t o_dy = fixed(offsetof(SM, dy) + (warp * kBTP * kBPairs + cl) * 16);
        const uint32_t o_sh = fixed(offsetof(SM, share) + (warp * 3 * 4 * kShareQ + q * kShareQ + cl) * 16);
        auto at4 = [&](uint32_t o) -> float4 & { return *reinterpret_cast<float4 *>(smem_dyn + o); };
        constexpr uint32_t kC = kBTP * 4 * 4 * 16, kStepB = 4 * 4 * 16, kStepG = 2 * kBPairs * 16, kStepY = kBPairs * 16;
        constexpr uint32_t kShare = 4 * kShareQ * 16;

        if constexpr (kShares) {
            if (c0 + nch < nchunks) {   // the share before has left the adjoint
                bool set = true;
                if (tid == 0) set = flag_wait(p.share_sync() + share);
                if (__syncthreads_or(set ? 0 : 1)) {
                    if (tid == 0) {
                        report(p.status, 4 /* MB_ERR_TIMEOUT */, share);
                        for (int jj = 0; jj < S && jj < nch; ++jj)
                            mbar_wait(&s.full[(n0 + jj) % S], (uint32_t)(((n0 + jj) / S) & 1));
                        bulk_wait_all();
                    }
                    return;
                }
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    const float4 v = __ldcg(reinterpret_cast<const float4 *>(p.seg_h) +
                                            ((int64_t)(share - 1) * 2 + j) * kBThreads + tid);
                    g[j][0] = v.x; g[j][1] = v.y; g[j][2] = v.z; g[j][3] = v.w;
                }
            }
        }
        bool ok = true;
        for (int it = 0; it < nch; ++it) {
            const int sl = (n0 + it) % S;   // ring slot
            const int i = c0 + nch - 1 - it;   // chunk of this iteration
            const int t0 = i * kBT;
            const R &r = s.raw[sl];
            // the chunk's checkpoint, in flight during the conversion; the next one's on its way to L2
            float hm[2][4];
            if constexpr (!kSummary) {
                const float *ck = gp.h_ckpt + (((int64_t)b * nchunks + i) * D + d) * kDState + 4 * q;
#pragma unroll
                for (int j = 0; j < 2; ++j) {
#pragma unroll
                    for (int n = 0; n < 4; ++n) hm[j][n] = 0.f;
                    if (chan_ok) load_perm<true>(hm[j], ck + j * kDState, perm);
                }
                if (chan_ok && it + 1 < nch) asm volatile("prefetch.global.L2 [%0];" ::"l"(ck - D * kDState + (q & 1) * kDState));
            }
            // (1) convert chunk i; add dB, dC of chunk i + 1 to global memory
            ok = mbar_wait(&s.full[sl], (uint32_t)(((n0 + it) / S) & 1));
            if (ok) {
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    const int tp = ts + kHTP * u;
                    float2 de[2], dyv[2], gxv[2], sig[2], qz[2];
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        softplus_sigmoid2(add2(ld2<T>(&r.dt[0][0], off[u][e]), bias), de[e], sig[e]);
                        const float m = t0 + 2 * tp + e < L ? 1.f : 0.f;   // Delta = 0 past the end: h and g unchanged
                        de[e] = mul2(de[e], splat(m));
                        sig[e] = mul2(sig[e], splat(m));
                        dyv[e] = ld2<T>(&r.dout[0][0], off[u][e]);
                        if constexpr (!kSummary) gxv[e] = mul2(de[e], ld2<T>(&r.x[0][0], off[u][e]));
                        qz[e] = make_float2(0.f, 0.f);
                        if (gate) {
                            const float2 z = ld2<T>(&r.z[0][0], off[u][e]);
                            const float2 w = mul2(z, splat(-kLog2e));
                            const float2 o = add2(make_float2(ex2(w.x), ex2(w.y)), splat(1.f));
                            const float2 sz = make_float2(rcp(o.x), rcp(o.y));
                            qz[e] = mul2(mul2(dyv[e], sz), fma2(z, fma2(sz, splat(-1.f), splat(1.f)), splat(1.f)));
                            dyv[e] = mul2(dyv[e], mul2(z, sz));
                        }
                    }
                    if constexpr (kSummary) gxv[0] = gxv[1] = make_float2(0.f, 0.f);
                    s.dg[warp][tp][0][pp] = make_float4(de[0].x, de[1].x, gxv[0].x, gxv[1].x);
                    s.dg[warp][tp][1][pp] = make_float4(de[0].y, de[1].y, gxv[0].y, gxv[1].y);
                    s.dy[warp][tp][pp] = make_float4(dyv[0].x, dyv[1].x, dyv[0].y, dyv[1].y);
                    if constexpr (!kSummary) {
                        s.fin[warp][0][tp][pp] = make_float4(sig[0].x, sig[0].y, sig[1].x, sig[1].y);
                        s.fin[warp][1][tp][pp] = make_float4(qz[0].x, qz[0].y, qz[1].x, qz[1].y);
                    }
                }
                {   // two states of B and of C at a step pair, in both orders
                    const int wh = tid & 1, wq = (tid >> 1) & 3, wt = tid >> 3;
                    const bool swap = wq & 2;   // which order first: eight stores at a time on different banks
#pragma unroll
                    for (int u = kSummary ? 1 : 0; u < 2; ++u) {
                        const T *src = u ? &r.C[2 * wt][4 * wq + 2 * wh] : &r.B[2 * wt][4 * wq + 2 * wh];
                        const float2 v0 = ld2<T>(src, 0), v1 = ld2<T>(src, kDState * (int)sizeof(T));
                        float4 *dst = &s.bc[u][wt][wq][2 * wh];
                        const float4 f = make_float4(v0.x, v1.x, v0.y, v1.y), rv = make_float4(v0.y, v1.y, v0.x, v1.x);
                        dst[swap ? 1 : 0] = swap ? rv : f;
                        dst[swap ? 0 : 1] = swap ? f : rv;
                    }
                }
            }
            if constexpr (!kSummary) {
                if (it >= 1) flush_sums(s, gp, b, t0 + kBT, L);
                if (tid == 0) bulk_wait_read_all();   // the output tiles may be written again
            }
            if (__syncthreads_or(ok ? 0 : 1)) {
                if (tid == 0) {
                    report(p.status, 4 /* MB_ERR_TIMEOUT */, it);
                    for (int jj = it; jj <= it + S - 1 && jj < nch; ++jj)
                        mbar_wait(&s.full[(n0 + jj) % S], (uint32_t)(((n0 + jj) / S) & 1));
                    bulk_wait_all();
                }
                return;
            }

            const float4(&dgw)[kBTP][2][kBPairs] = s.dg[warp];
            const float4(&dyw)[kBTP][kBPairs] = s.dy[warp];
            if constexpr (kSummary) {
                float2 cs[2];
#pragma unroll
                for (int k = kBTP - 1; k >= 0; --k) {
                    const float4 c01 = s.bc[1][k][q][ix0], c23 = s.bc[1][k][q][ix1];
                    const float2 cp[4] = {make_float2(c01.x, c01.y), make_float2(c01.z, c01.w),
                                          make_float2(c23.x, c23.y), make_float2(c23.z, c23.w)};
                    const float4 yv = dyw[k][cl];
                    const float2 dyp[2] = {make_float2(yv.x, yv.y), make_float2(yv.z, yv.w)};
#pragma unroll
                    for (int j = 0; j < 2; ++j) {
                        const float2 dd = *reinterpret_cast<const float2 *>(&dgw[k][j][cl]);
                        cs[j] = k == kBTP - 1 ? dd : add2(cs[j], dd);
#pragma unroll
                        for (int n = 0; n < 4; ++n) {
                            const float2 e = mul2(dd, splat(a2[j][n]));
                            const float g1 = fmaf(dyp[j].y, cp[n].y, g[j][n]) * ex2(e.y);
                            g[j][n] = fmaf(dyp[j].x, cp[n].x, g1) * ex2(e.x);
                        }
                    }
                }
                dsum[0] = add2(dsum[0], cs[0]);
                dsum[1] = add2(dsum[1], cs[1]);
            } else {
                // (2) the state before step 8: steps 0 .. 7 from the checkpoint
                float4(&hq)[2][2][32] = s.hq[warp];
#pragma unroll
                for (int j = 0; j < 2; ++j) hq[0][j][lane] = make_float4(hm[j][0], hm[j][1], hm[j][2], hm[j][3]);
#pragma unroll
                for (int k = 0; k < kHTP; ++k) {
                    const float4 b01 = at4(o_bc0 + k * kStepB), b23 = at4(o_bc1 + k * kStepB);
                    const float2 bp[4] = {make_float2(b01.x, b01.y), make_float2(b01.z, b01.w), make_float2(b23.x, b23.y),
                                          make_float2(b23.z, b23.w)};
#pragma unroll
                    for (int j = 0; j < 2; ++j) {
                        const float4 v = at4(o_dg + k * kStepG + j * kBPairs * 16);
                        const float2 dd = make_float2(v.x, v.y), gg = make_float2(v.z, v.w);
#pragma unroll
                        for (int n = 0; n < 4; ++n) {
                            const float2 e = mul2(dd, splat(a2[j][n]));
                            const float2 bg = mul2(bp[n], gg);
                            hm[j][n] = fmaf(ex2(e.y), fmaf(ex2(e.x), hm[j][n], bg.x), bg.y);
                        }
                    }
                }
#pragma unroll
                for (int j = 0; j < 2; ++j) hq[1][j][lane] = make_float4(hm[j][0], hm[j][1], hm[j][2], hm[j][3]);
                float4(&sh)[3][4 * kShareQ] = s.share[warp];
                // (3) the two halves, the later one first (not unrolled: both at once spill registers)
#pragma unroll 1
                for (int u = 1; u >= 0; --u) {
                    const int k0 = kHTP * u;
                    const uint32_t ub0 = o_bc0 + u * kHTP * kStepB, ub1 = o_bc1 + u * kHTP * kStepB, ug = o_dg + u * kHTP * kStepG;
                    const float4 ha = hq[u][0][lane], hb = hq[u][1][lane];
                    const float hs[2][4] = {{ha.x, ha.y, ha.z, ha.w}, {hb.x, hb.y, hb.z, hb.w}};   // state before this half
                    // its decays and states, kept in registers, and the shares of C.h
                    float2 ab[kHTP][2][4], hp[kHTP][2][4];
                    float4 shy[kHTP];
#pragma unroll
                    for (int k = 0; k < kHTP; ++k) {
                        const float4 b01 = at4(ub0 + k * kStepB), b23 = at4(ub1 + k * kStepB);
                        const float4 c01 = at4(ub0 + kC + k * kStepB), c23 = at4(ub1 + kC + k * kStepB);
                        const float2 bp[4] = {make_float2(b01.x, b01.y), make_float2(b01.z, b01.w),
                                              make_float2(b23.x, b23.y), make_float2(b23.z, b23.w)};
                        const float2 cp[4] = {make_float2(c01.x, c01.y), make_float2(c01.z, c01.w),
                                              make_float2(c23.x, c23.y), make_float2(c23.z, c23.w)};
                        float2 acc[2];
#pragma unroll
                        for (int j = 0; j < 2; ++j) {
                            const float4 v = at4(ug + k * kStepG + j * kBPairs * 16);
                            const float2 dd = make_float2(v.x, v.y), gg = make_float2(v.z, v.w);
#pragma unroll
                            for (int n = 0; n < 4; ++n) {
                                const float2 e = mul2(dd, splat(a2[j][n]));
                                ab[k][j][n] = make_float2(ex2(e.x), ex2(e.y));
                                const float2 bg = mul2(bp[n], gg);
                                const float hl = k == 0 ? hs[j][n] : hp[k - 1][j][n].y;
                                hp[k][j][n].x = fmaf(ab[k][j][n].x, hl, bg.x);
                                hp[k][j][n].y = fmaf(ab[k][j][n].y, hp[k][j][n].x, bg.y);
                                acc[j] = n == 0 ? mul2(cp[0], hp[k][j][0]) : fma2(cp[n], hp[k][j][n], acc[j]);
                            }
                        }
                        shy[k] = make_float4(acc[0].x, acc[0].y, acc[1].x, acc[1].y);
                    }
#pragma unroll
                    for (int k = 0; k < kHTP; ++k) at4(o_sh + k * kBPairs * 16) = shy[k];
                    // reverse sweep
                    float4 sh1[kHTP], sh2[kHTP];
                    float2 sums[kHTP];
#pragma unroll
                    for (int k = kHTP - 1; k >= 0; --k) {
                        const float4 b01 = at4(ub0 + k * kStepB), b23 = at4(ub1 + k * kStepB);
                        const float4 c01 = at4(ub0 + kC + k * kStepB), c23 = at4(ub1 + kC + k * kStepB);
                        const float2 bp[4] = {make_float2(b01.x, b01.y), make_float2(b01.z, b01.w),
                                              make_float2(b23.x, b23.y), make_float2(b23.z, b23.w)};
                        const float2 cp[4] = {make_float2(c01.x, c01.y), make_float2(c01.z, c01.w),
                                              make_float2(c23.x, c23.y), make_float2(c23.z, c23.w)};
                        const float4 yv = at4(o_dy + u * kHTP * kStepY + k * kStepY);
                        const float2 dyp[2] = {make_float2(yv.x, yv.y), make_float2(yv.z, yv.w)};
                        float2 dBv[4], dCv[4], s1[2], s2[2];
#pragma unroll
                        for (int j = 0; j < 2; ++j) {
                            const float4 v = at4(ug + k * kStepG + j * kBPairs * 16);
                            const float2 dd = make_float2(v.x, v.y), gg = make_float2(v.z, v.w);
#pragma unroll
                            for (int n = 0; n < 4; ++n) {
                                const float2 A = ab[k][j][n], H = hp[k][j][n];
                                float2 gv, ga, w;
                                gv.y = fmaf(dyp[j].y, cp[n].y, g[j][n]);
                                ga.y = gv.y * A.y;
                                gv.x = fmaf(dyp[j].x, cp[n].x, ga.y);
                                ga.x = gv.x * A.x;
                                g[j][n] = ga.x;
                                w.x = ga.x * (k == 0 ? hs[j][n] : hp[k - 1][j][n].y);
                                w.y = ga.y * H.x;
                                dCv[n] = j == 0 ? mul2(dyp[0], H) : fma2(dyp[1], H, dCv[n]);
                                dBv[n] = j == 0 ? mul2(gg, gv) : fma2(gg, gv, dBv[n]);
                                s1[j] = n == 0 ? mul2(bp[0], gv) : fma2(bp[n], gv, s1[j]);
                                // scalar: a packed form would copy a2 into a pair at every use (2459 -> 2435 us)
                                s2[j].x = n == 0 ? a2[j][0] * w.x : fmaf(a2[j][n], w.x, s2[j].x);
                                s2[j].y = n == 0 ? a2[j][0] * w.y : fmaf(a2[j][n], w.y, s2[j].y);
                                dA[j][n] = fma2(dd, w, dA[j][n]);
                            }
                        }
                        sh1[k] = make_float4(s1[0].x, s1[0].y, s1[1].x, s1[1].y);
                        sh2[k] = make_float4(s2[0].x, s2[0].y, s2[1].x, s2[1].y);
                        // dB, dC over the warp's 16 channels: lanes that differ in channel bits exchange the states they do
                        // not keep; the state order r -> r ^ perm makes those registers 2, 3, then 1, on every lane
#pragma unroll
                        for (int n = 0; n < 2; ++n) {
                            dBv[n] = add2(dBv[n], shfl2(dBv[n + 2], 8));
                            dCv[n] = add2(dCv[n], shfl2(dCv[n + 2], 8));
                        }
                        dBv[0] = add2(dBv[0], shfl2(dBv[1], 4));
                        dCv[0] = add2(dCv[0], shfl2(dCv[1], 4));
                        const bool keepC = lane & 1;   // channel bit 2: this lane ends with dC of its state, or dB
                        const float2 keep = keepC ? dCv[0] : dBv[0], send = keepC ? dBv[0] : dCv[0];
                        sums[k] = add2(keep, shfl2(send, 1));
                    }
#pragma unroll
                    for (int k = 0; k < kHTP; ++k) {
                        at4(o_sh + kShare + k * kBPairs * 16) = sh1[k];
                        at4(o_sh + 2 * kShare + k * kBPairs * 16) = sh2[k];
                        s.sum[warp][k0 + k][8 * q + 4 * (lane & 1) + perm] = sums[k];
                    }
                    // finish this half's outputs
                    __syncwarp();
                    float2 tot[3][2];   // C.h, g.B, sum g Abar h A log2 e: [step] of (channel 2 pp, channel 2 pp + 1)
#pragma unroll
                    for (int v = 0; v < 3; ++v) {
                        const float4 *src = &sh[v][ts * kBPairs + pp];
                        const float4 x0 = src[0], x1 = src[kShareQ], x2 = src[2 * kShareQ], x3 = src[3 * kShareQ];
                        const float2 ca = add2(add2(make_float2(x0.x, x0.y), make_float2(x1.x, x1.y)),
                                               add2(make_float2(x2.x, x2.y), make_float2(x3.x, x3.y)));
                        const float2 cb = add2(add2(make_float2(x0.z, x0.w), make_float2(x1.z, x1.w)),
                                               add2(make_float2(x2.z, x2.w), make_float2(x3.z, x3.w)));
                        tot[v][0] = make_float2(ca.x, cb.x);
                        tot[v][1] = make_float2(ca.y, cb.y);
                    }
                    const float4 va = dgw[k0 + ts][0][pp], vb = dgw[k0 + ts][1][pp], yv = dyw[k0 + ts][pp];
                    const float4 fs = s.fin[warp][0][k0 + ts][pp], fq = s.fin[warp][1][k0 + ts][pp];
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        const int o = u ? off[1][e] : off[0][e];
                        const float2 sg = e ? make_float2(fs.z, fs.w) : make_float2(fs.x, fs.y);
                        const float2 qv = e ? make_float2(fq.z, fq.w) : make_float2(fq.x, fq.y);
                        const float2 de = e ? make_float2(va.y, vb.y) : make_float2(va.x, vb.x);
                        const float2 dyv = e ? make_float2(yv.y, yv.w) : make_float2(yv.x, yv.z);
                        const float2 xv = ld2<T>(&r.x[0][0], o);
                        const float2 ddt = mul2(fma2(xv, tot[1][e], mul2(tot[2][e], splat(kLn2))), sg);
                        st2<T>(&s.gx[0][0], o, fma2(de, tot[1][e], mul2(dyv, dsk)));
                        st2<T>(&s.gdt[0][0], o, ddt);
                        if (gate) st2<T>(&s.gz[0][0], o, mul2(fma2(dsk, xv, tot[0][e]), qv));
                        dD_acc = fma2(dyv, xv, dD_acc);
                        db_acc = add2(db_acc, ddt);
                    }
                    __syncwarp();   // the shares may be written again
                }
                fence_proxy_async_smem();   // output tiles -> visible to the TMA stores
            }
            __syncthreads();
            if (tid == 0) {
                if constexpr (!kSummary) {
                    tma_store_3d(&a.tm_dx, &s.gx[0][0], d0, t0, b);
                    tma_store_3d(&a.tm_ddt, &s.gdt[0][0], d0, t0, b);
                    if (gate) tma_store_3d(&a.tm_dz, &s.gz[0][0], d0, t0, b);
                    bulk_commit();
                }
                if (it + S < nch) {   // the stage is consumed: refill it
                    fence_proxy_async_smem();
                    issue_bchunk<T, kSummary>(s, a, sl, c0 + nch - 1 - (it + S), d0, b);
                }
            }
        }
        if constexpr (kSummary) pdl_trigger();   // the second pass may set up while the last summaries are written
        if constexpr (kSummary) {   // Abar g at the segment's start from a zero adjoint at its end; the product of its decays
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                if (!chan_ok) break;
                const int64_t o = (((int64_t)b * nseg + seg) * D + d + j) * kDState + 4 * q;
                const float sd = dsum[j].x + dsum[j].y;
                float pe[4];
#pragma unroll
                for (int n = 0; n < 4; ++n) pe[n] = ex2(a2[j][n] * sd);
                store_perm(p.seg_h + o, g[j], perm);
                store_perm(p.seg_p + o, pe, perm);
            }
        } else {
            flush_sums(s, gp, b, c0 * kBT, L);   // the last chunk's
#pragma unroll
            for (int o = 8; o <= 16; o += 8) {   // over the four lanes of a channel pair
                dD_acc = add2(dD_acc, shfl2(dD_acc, o));
                db_acc = add2(db_acc, shfl2(db_acc, o));
            }
            if (ts == 0 && dc < D) {
                if (gp.dD) atomicAdd(reinterpret_cast<float2 *>(gp.dD + dc), dD_acc);
                if (gp.ddt_bias) atomicAdd(reinterpret_cast<float2 *>(gp.ddt_bias + dc), db_acc);
            }
            if (chan_ok) {
#pragma unroll
                for (int j = 0; j < 2; ++j) {
#pragma unroll
                    for (int n = 0; n < 4; ++n)
                        atomicAdd(gp.dA + (d + j) * kDState + 4 * q + (n ^ perm), dA[j][n].x + dA[j][n].y);
                    if (gp.dh0 && c0 == 0)
                        store_perm(gp.dh0 + ((int64_t)b * D + d + j) * kDState + 4 * q, g[j], perm);
                }
            }
            if constexpr (kShares) {
                if (c0 > 0) {   // the share ends inside the tile: leave the adjoint for the next one
#pragma unroll
                    for (int j = 0; j < 2; ++j)
                        __stcg(reinterpret_cast<float4 *>(p.seg_h) + ((int64_t)share * 2 + j) * kBThreads + tid,
                               make_float4(g[j][0], g[j][1], g[j][2], g[j][3]));
                    __threadfence();
                    __syncthreads();
                    if (tid == 0) flag_set(p.share_sync() + 1 + share);
                }
            }
        }
        if (!kShares || tile * nchunks <= lo) break;
        n0 += nch;
        --tile;
    }
    if (!kSummary && tid == 0) bulk_wait_all();
}

// Zero the gradients that are accumulated atomically (16-byte aligned, sizes multiples of 16 bytes): one launch
// instead of five memsets, which with their gaps took a small span's backward from 70 to 89 us (2 x 777 x 1544).
struct ClearArgs {
    float4 *p[6];
    int64_t n[6];   // float4s
    int early;      // whether the next kernel may launch early
};
constexpr int kClearThreads = 256;
__global__ void __launch_bounds__(kClearThreads) clear_kernel(const __grid_constant__ ClearArgs a) {
    if (a.early) pdl_trigger();   // the next kernel may set up; it waits for this one before it adds anything
    pdl_wait();
    const int64_t step = (int64_t)gridDim.x * kClearThreads;
#pragma unroll
    for (int k = 0; k < 6; ++k)
        for (int64_t i = (int64_t)blockIdx.x * kClearThreads + threadIdx.x; i < a.n[k]; i += step)
            a.p[k][i] = make_float4(0.f, 0.f, 0.f, 0.f);
}

bool make_map3(CUtensorMap *m, const void *base, bool bf16, int64_t batch, int64_t L, int64_t inner,
               int box_inner, int64_t row, int swizzle) {
    const int64_t es = bf16 ? 2 : 4;
    const uint64_t dims[3] = {(uint64_t)inner, (uint64_t)L, (uint64_t)batch};
    const uint64_t strides[2] = {(uint64_t)(row * es), (uint64_t)(L * row * es)};
    const uint32_t box[3] = {(uint32_t)box_inner, (uint32_t)kBT, 1};
    return encode_tmap(m, base, (int)es, 3, dims, strides, box, swizzle);
}

template <typename T>
cudaError_t launch_backward_typed(const ScanParams &p, const GradParams &g, cudaStream_t s) {
    const bool bf16 = sizeof(T) == 2;
    BwdArgs a;
    memset(&a, 0, sizeof(a));
    a.p = p;
    a.g = g;
    a.has_gate = p.z != nullptr;
    const int64_t Bn = p.batch, L = p.seqlen, D = p.d_inner;
    if (p.nseg < 2 || !p.seg_h || !p.seg_p) a.p.nseg = 1;
    const int64_t nseg = a.p.nseg;
    auto tok = [&](CUtensorMap *m, const void *base) {
        return make_map3(m, base, bf16, Bn, L, D, kBCh, D, kBCh * (int)sizeof(T));
    };
    if (!tok(&a.tm_dt, p.dt) || !tok(&a.tm_x, p.x) || (p.z && !tok(&a.tm_z, p.z)) || !tok(&a.tm_dout, g.dout) ||
        !make_map3(&a.tm_B, p.B, bf16, Bn, L, kDState, kDState, p.bc_stride, 0) ||
        !make_map3(&a.tm_C, p.C, bf16, Bn, L, kDState, kDState, p.bc_stride, 0) || !tok(&a.tm_dx, g.dx) ||
        !tok(&a.tm_ddt, g.ddt) || (p.z && !tok(&a.tm_dz, g.dz)))
        return cudaErrorInvalidValue;
    constexpr size_t smem = sizeof(BSmem<T>) + 1024;
    static_assert(kBResident<T> * (smem + 1024) <= 228 * 1024, "an SM holds this many CTAs, 1 KB reserved for each");
    const DeviceLimits *lim = device_limits();
    if (!lim) return cudaErrorInvalidDevice;
    const int64_t ctas = ((D + kBCh - 1) / kBCh) * Bn;   // per segment of L
    cudaError_t e;
    if (nseg > 1) {   // first pass: summaries of segments 1 .. nseg - 1
        BwdArgs a1 = a;
        a1.seg0 = 1;
        a1.grid_segs = (int)(nseg - 1);
        auto k1 = backward_kernel<T, true>;
        if ((e = cudaFuncSetAttribute(k1, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)lim->smem_optin)) !=
            cudaSuccess)
            return e;
        const int64_t grid = ctas * (nseg - 1);
        if ((e = launch_pdl(true, k1, dim3((unsigned)grid), dim3(kBThreads), smem, s, a1)) != cudaSuccess) return e;
    }
    a.grid_segs = (int)nseg;
    if (nseg == 1 && p.shares > 0) {
        auto ks = backward_kernel<T, false, true>;
        if ((e = cudaFuncSetAttribute(ks, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)lim->smem_optin)) !=
            cudaSuccess)
            return e;
        return launch_pdl(true, ks, dim3((unsigned)p.shares), dim3(kBThreads), spread_smem(smem, p.shares, kBResident<T>),
                          s, a);
    }
    auto k = backward_kernel<T, false>;
    if ((e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)lim->smem_optin)) != cudaSuccess)
        return e;
    return launch_pdl(true, k, dim3((unsigned)(ctas * nseg)), dim3(kBThreads), smem, s, a);
}

}  // namespace

// Time split: when the batch rows and channel tiles fill at most half of the
// resident slots (kBResident per SM), into as many segments as fill them, each at
// least two chunks long. Only the adjoint is carried across a boundary (the
// states come from the checkpoints), so the first pass is short: decays and
// dy C, no sums over channels or states. Every lane folds the segments after
// its own; beyond sqrt(2 L) segments that costs more than shorter segments
// give. Measured: 2 x 777 x 1544 (98 CTAs) 156 us unsplit, 62 in 6 segments;
// 1 x 8192 x 64 1537 us unsplit, 53 in 128, 84 in 256; with the slots nearly
// filled (8 x 8192 x 2048: 512 CTAs) 2.63 ms unsplit, 2.90 ms in 6. fp32, spans
// of 2048 steps, tiles per SM 0.5, 1, 1.2, 1.6, 2: 141, 254, 353, 446, 448 us (cut
// for four slots per SM: 155, 270, 353, 500, 506). Three segments instead of two
// where they are at most one per SM beyond the slots (1.2 tiles per SM: 372 us in
// two): the CTAs of an SM do not end together, and a few more fill the gaps.
constexpr int64_t kMinBwdSplitSteps = 128;

int64_t backward_segments(const ScanParams &p, bool bf16) {
    if (p.batch <= 0 || p.d_inner <= 0 || p.seqlen < kMinBwdSplitSteps || p.dt_low) return 1;
    const int64_t slots = (int64_t)device_sms() * (bf16 ? kBResident<__nv_bfloat16> : kBResident<float>);
    const int64_t ctas = p.batch * ((p.d_inner + kBCh - 1) / kBCh);
    if (2 * ctas > slots) return 1;
    const int64_t nchunks = (p.seqlen + kBT - 1) / kBT;
    int64_t nseg = slots / ctas;
    const int64_t most = (int64_t)sqrt(2.0 * (double)p.seqlen);
    if (nseg > most) nseg = most;
    if (!bf16 && nseg == 2 && 3 * ctas <= slots + device_sms()) nseg = 3;
    if (nseg > nchunks / 2) nseg = nchunks / 2;
    if (nseg < 2) return 1;
    const int64_t cps = (nchunks + nseg - 1) / nseg;
    return (nchunks + cps - 1) / cps;   // no empty segment
}

// Even shares (as prefill_shares), where the tiles are little over two per SM
// or over a multiple of the slots. Microseconds per chunk of an SM's CTAs, one
// per tile, 1 to 4 (fp32: 3) of them, and of shares with two per SM and with
// all, as measured:
//   bf16   3.17 3.35 4.69 4.84   3.6  5.05
//   fp32   3.20 3.49 4.83        3.70 5.05
// (two CTAs of two warps fill the four schedulers once, so a third costs as much
// as two more). The last wave of fp32 takes about 0.9 of its number, of bf16 all.
// Measured, spans of 2048 steps: bf16 at 2.1, 4.2, 5.05 and 8.2 tiles per SM 600 ->
// 486, 1000 -> 681, 1003 -> 815, 1582 -> 1315 us; fp32 at 2.1, 3.1, 4.2 and 6.1 618 ->
// 501, 867 -> 670, 1007 -> 904, 1401 -> 1308 us, as it is at 2.9, 5.6 and 8.2.
int64_t backward_shares(const ScanParams &p, bool bf16) {
    if (p.batch <= 0 || p.d_inner <= 0 || p.seqlen < kMinBwdSplitSteps || p.dt_low) return 0;
    const int64_t sms = device_sms(), tiles = p.batch * ((p.d_inner + kBCh - 1) / kBCh);
    if (sms <= 0 || tiles <= 2 * sms) return 0;
    const int64_t resident = bf16 ? kBResident<__nv_bfloat16> : kBResident<float>, wave = resident * sms;
    constexpr double t[2][4] = {{3.20, 3.49, 4.83}, {3.17, 3.35, 4.69, 4.84}}, two[2] = {3.70, 3.6}, all = 5.05;
    const int64_t m = tiles < wave ? 2 : resident, rest = tiles % wave;
    double plain = (double)(tiles / wave) * t[bf16][resident - 1];
    if (rest) plain += (tiles > rest && !bf16 ? 0.9 : 1.0) * t[bf16][(rest - 1) / sms];
    const double even = (double)tiles / (double)(m * sms) * (m == 2 ? two[bf16] : all);
    const double chunks = (double)(p.seqlen / kBT);
    return even * chunks + 7.0 < 0.97 * plain * chunks ? m * sms : 0;
}

cudaError_t launch_backward(const ScanParams &p, const GradParams &g, bool bf16, cudaStream_t s) {
    const int64_t Bn = p.batch, L = p.seqlen, D = p.d_inner;
    // The sums are accumulated atomically: clear them first.
    cudaError_t e;
    ClearArgs c;
    const int64_t nbc = Bn * L * kDState / 4;
    void *const ptr[6] = {g.dB, g.dC, g.dA, g.dD, g.ddt_bias, p.share_sync()};
    const int64_t num[6] = {nbc, nbc, D * kDState / 4, g.dD ? D / 4 : 0, g.ddt_bias ? D / 4 : 0,
                            p.shares > 0 ? (int64_t)prefill_share_sync_bytes(p.shares) / 16 : 0};
    int64_t most = 0;
    for (int k = 0; k < 6; ++k) {
        c.p[k] = reinterpret_cast<float4 *>(ptr[k]);
        c.n[k] = num[k];
        if (num[k] > most) most = num[k];
    }
    // A grid that is not spread and leaves room on the SMs is placed unevenly where it launches early (2 x 2048 x 2048
    // 417 us, and 398).
    const int64_t tiles = Bn * ((D + kBCh - 1) / kBCh), per = bf16 ? kBResident<__nv_bfloat16> : kBResident<float>;
    c.early = p.shares > 0 || tiles * (p.nseg > 1 ? p.nseg - 1 : 1) > (per - 1) * (int64_t)device_sms();
    if (most > 0) {
        const int64_t want = (most + kClearThreads - 1) / kClearThreads, cap = 8 * (int64_t)device_sms();
        const int64_t grid = want < cap || cap == 0 ? want : cap;
        if ((e = launch_pdl(true, clear_kernel, dim3((unsigned)grid), dim3(kClearThreads), 0, s, c)) != cudaSuccess)
            return e;
    }
    if (Bn == 0 || D == 0) return cudaSuccess;
    if (L == 0) {   // nothing to scan: dJ/dh0 = dJ/dh_last
        if (!g.dh0) return cudaSuccess;
        const size_t bytes = (size_t)(Bn * D * kDState) * 4;
        if (g.dh_last) return cudaMemcpyAsync(g.dh0, g.dh_last, bytes, cudaMemcpyDeviceToDevice, s);
        return cudaMemsetAsync(g.dh0, 0, bytes, s);
    }
    return bf16 ? launch_backward_typed<__nv_bfloat16>(p, g, s) : launch_backward_typed<float>(p, g, s);
}

}  // namespace mbscan
