// The step kernel's plane pipeline in staged form (included by
// mmod_step_tma.cu, which documents the decomposition and the arithmetic).
//
// A CTA owns a TX x TY tile and marches down T planes from z0; each thread
// owns 2 (x) x 2 (y) points.  What differs from the ring form of
// mmod_step_tma.cu:
//   * One mbarrier per stage: stage t % 4 carries everything plane t needs that
//     is not on chip yet, i.e. the halo tile of u^n at z0 + t + 4, and u^{n-1}
//     and c at z0 + t.  A plane costs one wait instead of two, and with the
//     plane loop unrolled by 4 every shared-memory offset and the barrier are
//     constants; the eight halo slots alternate between two halves, so a group
//     of four planes reads its leading planes from one half and its centre
//     planes from the other.
//   * All the first planes are requested at once.  The planes z0-4 .. z0-1 are
//     only ever z neighbours of the thread's own points: they come as tile
//     boxes without x-y halo into a region of their own (TX x TY instead of
//     PITCH x (TY + 8) floats), so the eight halo slots hold z0 .. z0+7 from the
//     start and the leading planes of the first group do not wait for a slot
//     (one memory latency less per launch).
//   * A thread's own centre values come from its z queue, not from shared
//     memory again (4 of 24 loads per plane).
//   * Off the z layers e = e_x + e_y does not change along the march: each
//     thread keeps it and the damping factor 1 / (1 + e) of its four points in
//     registers (inside, e = 0 and the factor 1, where both operations are exact
//     identities), so that only z-layer planes form reciprocals (eight per
//     thread and plane, before on every plane of a tile that touches an x or y
//     layer: the CTAs that ended last).  240^3 38.6 -> 37.1 us per step,
//     batches of uneven shots 2-4 % faster, 1024 x 1024 x 512 1.3 %.
//   * Groups of four planes that touch a z layer run code of their own, so that
//     a plane has no branch between its two rows: with one there, the compiler
//     could not interleave the rows' loads and arithmetic.  240^3 37.1 -> 36.6 us
//     per step, 151 x 117 x 98 7.35 -> 7.1, batches 2-5 % faster; a third case
//     inside the plane (one reciprocal where a z-layer tile touches no x or y
//     layer) measured 2-6 % slower at every size.
// Bound by DRAM on large grids and by the pipeline's latencies on one-wave
// grids.  us per step, ring form -> staged: 64^3 4.47 -> 3.83, 128^3 8.68 ->
// 7.89, 200^3 34.98 -> 32.35, 240^3 41.96 -> 41.20, 512^3 337.0 -> 325.5 (6.60
// TB/s).  Then, with the tensor maps prefetched,
// u^n requested ahead of the block barrier, and the source and receiver
// look-ups taken off the critical path (they were dependent loads right after
// the wait and at the end): 64^3 3.83 -> 3.58, 151 x 117 x 98 7.8 -> 7.4, 240^3 39.4
// -> 38.8.  122 registers (123 with g^n, 106 to 108 in the imaging form, 128 in the
// claiming and persistent kernels), no spills.
// PITCH, the halo tile's row pitch, is chosen so that a half-warp whose lanes
// span two row pairs reads 16 different bank pairs: 2 PITCH = TX (mod 32).
#pragma once

namespace mmod {
namespace {

template <int TX_, int TY_, int PITCH_, int MINB_ = 2>
struct Staged {
    static constexpr bool kStaged = true;
    static constexpr int TX = TX_, TY = TY_, PITCH = PITCH_, HY = TY_ + 2 * kRadius;
    static constexpr int RY = 2, U = 4, NSU = 8;
    static constexpr int QD = 2 * kRadius + U;           // z queue: 8 planes and one group
    static constexpr int LX = TX / 2, NT = LX * (TY / RY);
    static constexpr int MINB = MINB_, MINB2 = MINB_ > 2 ? MINB_ : 2;
    static constexpr int CUR = PITCH * HY;               // floats of a halo slot
    static constexpr int OWN = TX * TY;                  // floats of a tile box
    static constexpr int OWN_S = (OWN + 31) / 32 * 32;   // its slot, 128-byte aligned
    static constexpr int CUR_S = (CUR + 31) / 32 * 32;
    static constexpr int RINGS = NSU * CUR_S + 4 * OWN_S + U * 2 * OWN_S;   // floats
    static constexpr int ABORT_OFF = RINGS * 4 + (U + 1) * 8;               // abort flag, then the claim words
    static constexpr int SMEM = ABORT_OFF + 16;
    static constexpr unsigned STAGE_BYTES = (CUR + 2 * OWN) * 4;
    static constexpr unsigned FIRST_BYTES = (4 * CUR + 4 * OWN) * 4;
    static_assert(TX % 4 == 0 && TY % RY == 0 && PITCH % 4 == 0 && PITCH >= TX + 2 * kRadius, "16-byte boxes");
    static_assert(NT <= 256 && SMEM <= 113 * 1024, "two CTAs per SM");
};

// What a launch computes.
enum StepMode {
    kStepOnly,
    kStepG,     // the step, and g^n = L u^n + s^n into StepArgs::gout
    kImage      // StepArgs::image: the accumulator's A += psi^{n+1} (L u^n + s^n).  A step without its own
                // field: where a reversed step needs g^n once, this one kernel takes the place of a
                // step that writes g^n and a pass that reads it (16 B per point instead of 36; the gradient
                // of 133 x 144 x 120 in the binomial schedule 15.3 -> 13.2 ms).
};

struct StagedCtx {
    float *col;          // the thread's column in halo slot 0 (row 2 py, column 2 px)
    float *pc;           // the thread's point in the first u^{n-1} tile
    uint64_t *full;      // U stage barriers
    int *abort_flag;
    int z0;
    bool full0, full1, part0, part1;   // row 0 / 1: both columns, or only the first, inside the grid
};

// One plane: step t of the range, J = t % 4, half = (t / 4) & 1.  out / gout:
// the thread's point of row 0 on this plane.
// Z: the group of planes touches a z layer.
template <class S, int J, int MODE, bool Z>
__device__ __forceinline__ void staged_plane(const StepArgs &a, const StagedCtx &c, int k, unsigned half,
                                             const float *ctr_half, const float *lead_half,
                                             float2 (&q)[S::QD][S::RY], const Wts &w,
                                             const float2 (&exy)[S::RY], const float2 (&rxy)[S::RY], float *out,
                                             float *gout) {
    const float ez = Z ? __ldg(a.ez + k) : 0.0f;
    if (!mbar_wait(&c.full[J], half, c.abort_flag, a.err)) return;
    // the leading plane k + 4 enters the queue
    const float *lead = lead_half + J * S::CUR_S + kRadius * S::PITCH + kRadius;
#pragma unroll
    for (int r = 0; r < S::RY; ++r) q[J + 2 * kRadius][r] = *reinterpret_cast<const float2 *>(lead + r * S::PITCH);
    // y neighbours: rows 2 py .. 2 py + 9 of the centre plane; the thread's own two rows are in the queue
    const float *ctr = ctr_half + J * S::CUR_S;
    float2 yc[S::RY + 2 * kRadius];
#pragma unroll
    for (int rr = 0; rr < S::RY + 2 * kRadius; ++rr)
        yc[rr] = rr >= kRadius && rr < kRadius + S::RY
                     ? q[J + kRadius][rr >= kRadius && rr < kRadius + S::RY ? rr - kRadius : 0]
                     : *reinterpret_cast<const float2 *>(ctr + rr * S::PITCH + kRadius);
    const float *upp = c.pc + J * 2 * S::OWN_S;
#pragma unroll
    for (int r = 0; r < S::RY; ++r) {
        const float *row = ctr + (kRadius + r) * S::PITCH;
        const float2 p = q[J + kRadius][r];
        const float2 x0 = *reinterpret_cast<const float2 *>(row), x1 = *reinterpret_cast<const float2 *>(row + 2);
        const float2 x3 = *reinterpret_cast<const float2 *>(row + 6), x4 = *reinterpret_cast<const float2 *>(row + 8);
        const float2 two_p = __fadd2_rn(p, p);
        const float2 ntp = neg2(two_p);
        // x: offsets 1 and 3 do not form aligned pairs, so they run scalar
        float2 lx;
        lx.x = pair_first(w.x1, p.y, x1.y, two_p.x);
        lx.y = pair_first(w.x1, x3.x, p.x, two_p.y);
        lx = pair_acc2(lx, w.x2, x3, x1, ntp);
        lx.x = pair_acc(lx.x, w.x3, x3.y, x0.y, two_p.x);
        lx.y = pair_acc(lx.y, w.x3, x4.x, x1.x, two_p.y);
        lx = pair_acc2(lx, w.x4, x4, x0, ntp);
        float2 ly = pair_first2(w.y[0], yc[kRadius + r + 1], yc[kRadius + r - 1], ntp);
        float2 lz = pair_first2(w.z[0], q[J + kRadius + 1][r], q[J + kRadius - 1][r], ntp);
#pragma unroll
        for (int m = 2; m <= kRadius; ++m) {
            ly = pair_acc2(ly, w.y[m - 1], yc[kRadius + r + m], yc[kRadius + r - m], ntp);
            lz = pair_acc2(lz, w.z[m - 1], q[J + kRadius + m][r], q[J + kRadius - m][r], ntp);
        }
        const float2 lap = __fadd2_rn(__fadd2_rn(lx, ly), lz);
        const float2 pp = *reinterpret_cast<const float2 *>(upp + r * S::TX);
        const float2 cc = *reinterpret_cast<const float2 *>(upp + S::OWN_S + r * S::TX);
        float2 num = __fadd2_rn(two_p, neg2(pp));
        if constexpr (MODE == kImage) {
            num = (a.fs && k == 0) ? pp : __ffma2_rn(cc, lap, pp);   // g = 0 on a free surface
        } else if constexpr (Z) {   // e = (e_x + e_y) + e_z
            const float2 e = __fadd2_rn(exy[r], bcast(ez));
            num = __ffma2_rn(cc, lap, __ffma2_rn(e, pp, num));
            num = __fmul2_rn(num, make_float2(damp_factor(e.x), damp_factor(e.y)));
        } else {
            num = __fmul2_rn(__ffma2_rn(cc, lap, __ffma2_rn(exy[r], pp, num)), rxy[r]);
        }
        if (MODE != kImage && a.fs && k == 0) num = make_float2(0.0f, 0.0f);   // p = 0 on a free surface
        float *dst = out + (r ? a.nxp : 0);
        if (r ? c.full1 : c.full0)
            *reinterpret_cast<float2 *>(dst) = num;
        else if (r ? c.part1 : c.part0)
            dst[0] = num.x;
        if constexpr (MODE == kStepG) {   // g^n = L u^n (sources added after the z range), 0 on a free surface
            const float2 gv = (a.fs && k == 0) ? make_float2(0.0f, 0.0f) : lap;
            float *gd = gout + (r ? a.nxp : 0);
            if (r ? c.full1 : c.full0)
                *reinterpret_cast<float2 *>(gd) = gv;
            else if (r ? c.part1 : c.part0)
                gd[0] = gv.x;
        }
    }
}

// The work of one CTA: block `bid` of the `nbid` blocks of one grid.
// halo_map: u^n, PITCH x HY box; own_map: u^n, prev_map: u^{n-1}, c_map: c, TX x TY boxes.
template <class S, class Dep, int MODE = kStepOnly>
__device__ __forceinline__ void step_staged_body(const StepArgs &a, const StepVar &v, const CUtensorMap *halo_map,
                                                 const CUtensorMap *own_map, const CUtensorMap *prev_map,
                                                 const CUtensorMap *c_map, const Geom &g, int bid, int nbid,
                                                 const Dep &dep) {
    extern __shared__ __align__(128) unsigned char smem[];
    float *const ring = reinterpret_cast<float *>(smem);
    float *const first = ring + S::NSU * S::CUR_S;       // planes z0-4 .. z0-1, tile boxes
    float *const pc = first + 4 * S::OWN_S;              // stage j: u^{n-1}, then c
    StagedCtx c;
    c.full = reinterpret_cast<uint64_t *>(pc + S::U * 2 * S::OWN_S);
    uint64_t *const init = c.full + S::U;
    c.abort_flag = reinterpret_cast<int *>(smem + S::ABORT_OFF);
    const int tid = threadIdx.x;
    int b = bid;
    const int tx = b % g.tiles_x;
    b /= g.tiles_x;
    const int ty = b % g.tiles_y;
    const int x0 = tx * S::TX, y0 = ty * S::TY, z0 = b / g.tiles_y * g.zlen;
    c.z0 = z0;
    const int T = min(a.nz - z0, g.zlen);

    auto load_pc = [&](int t) {   // u^{n-1} and c of plane t into its stage
        float *dst = pc + t % S::U * 2 * S::OWN_S;
        tma_load_3d(dst, prev_map, x0, y0, z0 + t, &c.full[t % S::U]);
        tma_load_3d(dst + S::OWN_S, c_map, x0, y0, z0 + t, &c.full[t % S::U]);
    };
    auto load_halo = [&](int p, uint64_t *bar) {   // u^n at z0 + p
        tma_load_3d(ring + p % S::NSU * S::CUR_S, halo_map, x0 - kRadius, y0 - kRadius, z0 + p, bar);
    };
    // The maps of u^n are first used on the critical path, right after the wait.
    if (tid == 32) {
        tma_prefetch_map(own_map);
        tma_prefetch_map(halo_map);
    }
    // This tile's run of the injection table, for the end of the kernel.
    int inj_lo = 0, inj_hi = 0;
    if (a.inj.npts > 0) {
        const long long bucket = ((long long)ty * a.inj.tiles_x + tx) * a.nz + z0;
        inj_lo = __ldg(a.inj.tile_start + bucket);
        inj_hi = __ldg(a.inj.tile_start + bucket + T);
    }
    // The first injection point of each thread past warp 0 (whose first thread
    // issues the copies), down to scale * w[n] and the damping factor: a chain
    // of four dependent loads, which at the end of the kernel made the whole grid
    // wait for the few CTAs that hold sources, and here runs while the previous
    // step drains or the first planes arrive.  What is left for the end is one
    // read-modify-write.  64^3 x 100 steps: 372 -> 325 us; gradient 200^3 41.0 ->
    // 40.0 ms.
    constexpr int kAhead = S::NT - 32;   // points looked up ahead
    SourcePoint src;
    if constexpr (MODE != kImage) {
        if (tid >= 32) {
            src = source_point(a, v.n, inj_lo + tid - 32, inj_hi);
            for (int p = inj_lo + kAhead + tid - 32; p < inj_hi; p += kAhead) prefetch_source_point(a, v.n, p);
        }
    }
    // Receivers of the previous step (u^n, read-only during this launch), one
    // per thread of the grid and more only where there are more: the offset is
    // loaded here, the value once u^n is there, and it is stored after the plane
    // loop, so the two dependent loads keep nobody waiting.
    const int r0 = bid * S::NT + tid;
    const bool rec0 = v.traces && r0 < a.nrec;
    const long long rec_off0 = rec0 ? __ldg(a.rec_off + r0) : 0;
    if (tid == 0) {
        if (dep.reinit()) {   // the previous unit consumed every copy it issued
            for (int s = 0; s <= S::U; ++s) mbar_inval(&c.full[s]);
        }
        for (int s = 0; s <= S::U; ++s) mbar_init(&c.full[s], 1);
        *c.abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if constexpr (Dep::kProxyFence) __syncthreads();   // the flag is 0 before any waiter may set it
    // c and u^{n-1} first where the dependency allows it (PdlDep), then wait, then u^n
    const bool early = dep.early();
    if (early && tid == 0) {
        if constexpr (Dep::kProxyFence) fence_proxy_async_global();
        for (int t = 0; t < S::U && t < T; ++t) {
            mbar_expect_tx(&c.full[t], S::STAGE_BYTES);
            load_pc(t);
        }
    }
    const int px = tid % S::LX, py = tid / S::LX;
    const int x = x0 + 2 * px, y = y0 + S::RY * py;
    // The layer profiles at the thread's points, loaded while the previous step
    // drains: after the wait their latency would delay the first plane (151 x
    // 117 x 98 2240 -> 2197 us, 160 x 120 x 100 forward and gradient 9.74 -> 9.43 ms).
    float ex[2], ey[S::RY];
    ex[0] = x < a.nx ? __ldg(a.ex + x) : 0.0f;
    ex[1] = x + 1 < a.nx ? __ldg(a.ex + x + 1) : 0.0f;
#pragma unroll
    for (int r = 0; r < S::RY; ++r) ey[r] = y + r < a.ny ? __ldg(a.ey + y + r) : 0.0f;
    dep.wait(tid, c.abort_flag, a.err);
    // a wait that cannot fail and that every thread makes itself: u^n may be
    // requested before the other warps are here
    if constexpr (Dep::kProxyFence) __syncthreads();
    const bool dep_ok = !Dep::kProxyFence || !*c.abort_flag;
    if (tid == 0 && dep_ok) {
        if constexpr (Dep::kProxyFence) fence_proxy_async_global();
        mbar_expect_tx(init, S::FIRST_BYTES);
        for (int p = 0; p < kRadius; ++p) {
            int z = z0 - kRadius + p;
            if (a.fs && z < 0) z = -z;   // plane -m is the odd image of plane m (negated when read)
            tma_load_3d(first + p * S::OWN_S, own_map, x0, y0, z, init);
        }
        for (int p = 0; p < kRadius; ++p) load_halo(p, init);
        for (int t = 0; t < S::U && t < T; ++t) {
            if (!early) {
                mbar_expect_tx(&c.full[t], S::STAGE_BYTES);
                load_pc(t);
            }
            load_halo(t + kRadius, &c.full[t]);
        }
    }
    int armed = dep_ok ? min(S::U, T) : 0;   // planes whose stage has been filled
    // kImage: the accumulator at this thread's source point (at most one: the
    // host keeps longer tables off this kernel), before anyone overwrites it
    long long img_off = 0;
    float img_acc = 0.0f;
    if constexpr (MODE == kImage) {
        if (inj_lo + tid < inj_hi) {
            img_off = __ldg(a.inj.pt_off + inj_lo + tid);
            img_acc = v.uout[img_off];
        }
    }
    if constexpr (!Dep::kProxyFence) __syncthreads();   // the barriers are set up
    const float rec_val0 = rec0 ? v.ucur[rec_off0] : 0.0f;
    if (v.traces) {
        for (int r = r0 + nbid * S::NT; r < a.nrec; r += nbid * S::NT) v.traces[r] = v.ucur[__ldg(a.rec_off + r)];
    }

    Wts w;
    w.x1 = a.w.x[0];
    w.x2 = bcast(a.w.x[1]);
    w.x3 = a.w.x[2];
    w.x4 = bcast(a.w.x[3]);
#pragma unroll
    for (int m = 0; m < kRadius; ++m) {
        w.y[m] = bcast(a.w.y[m]);
        w.z[m] = bcast(a.w.z[m]);
    }
    c.col = ring + S::RY * py * S::PITCH + 2 * px;
    c.pc = pc + S::RY * py * S::TX + 2 * px;
    // e_z = 0 on planes [z_top, z_bot): under a free surface there is no top
    // layer, but where the layers meet (nz = 2 nbl) plane nz - 1 - nbl keeps one
    const int z_top = a.fs ? 0 : a.nbl, z_bot = a.nz - a.nbl - (a.fs ? 1 : 0);
    float2 exy[S::RY], rxy[S::RY];   // e_x + e_y and its damping factor at the thread's points
#pragma unroll
    for (int r = 0; r < S::RY; ++r) {
        exy[r] = make_float2(__fadd_rn(ex[0], ey[r]), __fadd_rn(ex[1], ey[r]));
        rxy[r] = make_float2(1.0f, 1.0f);
        if (z0 + T > z_top && z0 < z_bot)   // not all planes in a z layer (64^3 2 % slower without the test)
            rxy[r] = make_float2(damp_factor(exy[r].x), damp_factor(exy[r].y));
    }
    c.full0 = y < a.ny && x + 1 < a.nx;
    c.full1 = y + 1 < a.ny && x + 1 < a.nx;
    c.part0 = y < a.ny && x + 1 == a.nx;
    c.part1 = y + 1 < a.ny && x + 1 == a.nx;
    const long long off = (long long)z0 * a.plane + (long long)y * a.nxp + x;
    float *out = v.uout + off;
    float *gout = MODE == kStepG ? a.gout + off : nullptr;

    float2 q[S::QD][S::RY];
    if (dep_ok && mbar_wait(init, 0, c.abort_flag, a.err)) {
        const float *own = first + S::RY * py * S::TX + 2 * px;
        const float *ctr = c.col + kRadius * S::PITCH + kRadius;
#pragma unroll
        for (int i = 0; i < kRadius; ++i) {
#pragma unroll
            for (int r = 0; r < S::RY; ++r) {
                q[i][r] = *reinterpret_cast<const float2 *>(own + i * S::OWN_S + r * S::TX);
                q[kRadius + i][r] = *reinterpret_cast<const float2 *>(ctr + i * S::CUR_S + r * S::PITCH);
            }
        }
        if (a.fs && z0 < kRadius) {   // queue planes above k = 0 hold the images: negate
#pragma unroll
            for (int i = 0; i < kRadius; ++i)
                if (i < kRadius - z0) {
#pragma unroll
                    for (int r = 0; r < S::RY; ++r) q[i][r] = neg2(q[i][r]);
                }
        }
    }
    // Plane t done by every thread: its centre slot and its u^{n-1} / c tiles
    // are free and take plane t + 4's data.
#define MMOD_STAGED(J, Z)                                                                                              \
    if (t + (J) < T) {                                                                                              \
        staged_plane<S, (J), MODE, Z>(a, c, z0 + t + (J), half, c.col + half * (4 * S::CUR_S),                            \
                                c.col + (half ^ 1) * (4 * S::CUR_S), q, w, exy, rxy, out, gout);                    \
        out += a.plane;                                                                                             \
        if constexpr (MODE == kStepG) gout += a.plane;                                                                           \
        __syncthreads();                                                                                            \
        if (tid == 0 && t + (J) + S::U < T && !*c.abort_flag) {                                                     \
            mbar_expect_tx(&c.full[J], S::STAGE_BYTES);                                                             \
            tma_load_3d(ring + (half * 4 + (J)) * S::CUR_S, halo_map, x0 - kRadius, y0 - kRadius,                   \
                        z0 + t + (J) + 2 * S::U, &c.full[J]);                                                       \
            tma_load_3d(pc + (J) * 2 * S::OWN_S, prev_map, x0, y0, z0 + t + (J) + S::U, &c.full[J]);                \
            tma_load_3d(pc + (J) * 2 * S::OWN_S + S::OWN_S, c_map, x0, y0, z0 + t + (J) + S::U, &c.full[J]);        \
            armed = t + (J) + S::U + 1;                                                                             \
        }                                                                                                           \
    }
    unsigned half = 0;
#pragma unroll 1
    for (int t = 0; t < T; t += S::U, half ^= 1) {
        if (*c.abort_flag) break;
        if (MODE != kImage && (z0 + t < z_top || z0 + t + S::U > z_bot)) {
            MMOD_STAGED(0, true)
            MMOD_STAGED(1, true)
            MMOD_STAGED(2, true)
            MMOD_STAGED(3, true)
        } else {
            MMOD_STAGED(0, false)
            MMOD_STAGED(1, false)
            MMOD_STAGED(2, false)
            MMOD_STAGED(3, false)
        }
#pragma unroll
        for (int i = 0; i < 2 * kRadius; ++i)
#pragma unroll
            for (int r = 0; r < S::RY; ++r) q[i][r] = q[i + S::U][r];
    }
#undef MMOD_STAGED
    if (rec0) v.traces[r0] = rec_val0;
    // Sources of this CTA's tile and planes: nothing in this launch reads the
    // u^{n+1} it writes, so they are added once the whole z range is stored
    // (the block barrier makes every thread's stores visible).  The points of
    // one tile over planes [z0, z0 + T) are one run of the table.
    __syncthreads();
    if constexpr (MODE == kImage) {
        // g^n at a source point is L u^n + w / cell per source, in that order,
        // before the product: the point's term is formed anew from the
        // accumulator as it was
        const int p = inj_lo + tid;
        if (!*c.abort_flag && p < inj_hi) {
            float gv = lap_point(a, v.ucur, v.ucur[img_off], __ldg(a.inj.pt_i + p), __ldg(a.inj.pt_j + p),
                                 __ldg(a.inj.pt_k + p));
            for (int s = __ldg(a.inj.pt_first + p); s < __ldg(a.inj.pt_first + p + 1); ++s)
                gv = __fmaf_rn(__ldg(a.wavelet + (long long)__ldg(a.inj.src_row + s) * a.wrs + (long long)v.n * a.wcs),
                               a.inv_cell, gv);
            v.uout[img_off] = __fmaf_rn(a.c[img_off], gv, img_acc);
        }
    } else if (!*c.abort_flag && inj_lo < inj_hi) {
        inject_source_point(a, v.uout, v.n, inj_lo + tid - 32, src);
        inject_points(a, v.uout, v.n, inj_lo + kAhead, inj_hi, tid, S::NT);
        if constexpr (MODE == kStepG) inject_g_points(a, v.n, inj_lo, inj_hi, tid, S::NT);
    }
    // After a give-up, wait (bounded) for the copies this CTA still has in
    // flight (the first planes and the latest phase of every stage) before its
    // shared memory is released.
    if (*c.abort_flag && tid == 0 && dep_ok) {
        mbar_drain(init, 0);
        for (int t = max(0, armed - S::U); t < armed; ++t) mbar_drain(&c.full[t % S::U], (t / S::U) & 1);
    }
}

}  // namespace
}  // namespace mmod
