// lk_stream_impl.cuh -- internal: the LK kernel of large levels, templated on
// the storage type of the pyramid planes. One pyramid level of dense
// Lucas-Kanade flow (Section III-C-1), all K steps fused, on column bands cut
// into segments of rows. Included once per storage type (lk_stream.cu: float,
// lk_stream_bf16.cu, lk_stream_f16.cu), each of which instantiates the entry
// points at the end of this file for its type only.
//
// Same arithmetic as lk_level_kernel (lk.cu): per step and pixel p
//   (G(p) + lambda I) v = sum_{q in W(p)} grad T(q) (grad T(q) . u(q) - It(q)) + lambda u(p),
//   It(q) = J(q + u(q)) - T(q), u(p) <- v,
// over the (2r+1)^2 box clipped to the image.
//
// Schedule. A segment of a band (RW columns, C * RH rows, halo included) is
// one cluster of C CTAs on top of each other; a thread owns two neighbouring
// columns of a run of R rows and keeps their flow, template and gradient in
// registers for all K steps. A step is
//   A  the residual products P = grad T (grad T . u - It) of the own pixels,
//      the r outer rows of the run first: they go to the neighbouring run's
//      halo, in this CTA or the one above or below (st.async, counted by a
//      barrier there);
//   B  the column sums over 2r+1 rows of the rows that need no outer halo,
//      from registers, to shared memory;
//   C  after a barrier of the warps that share the rows: their row sums, the
//      2x2 solve and the update;
// then B and C of the r outer rows, when the neighbours' rows have come. So
// the rows between the CTAs of a cluster are exchanged, not recomputed, and
// their way is hidden by the inner rows' work: only the band's sides and the
// cluster's top and bottom carry a halo of K r pixels, that the steps eat up
// from outside (108 x 204 of 128 x 224 pixels are left at K r = 10).
//
// What bounds it (level 0 of a 4000 x 1500 pair with smooth flows, both
// directions, 300 us in a CUDA graph of launches): the issue of instructions
// (half of the slots) and the shared-memory pipe (57%), at 128 registers a
// thread and 16 warps an SM. Before, 768 threads worked through 12-row chunks of
// a ring in shared memory, eleven CTA-wide barriers a chunk: 494 us, timed the
// same way. Registers instead of the ring, and two pixels per paired instruction:
// 353 to 197 M warp instructions (and 613 to 440 us, cold, under ncu on a pair
// with depth steps). Measured with the same arithmetic, on the whole smooth pair
// (603 us): one barrier.cluster a step, sent before and awaited after the inner
// rows' work, 3% slower (every thread's fence in it); counted halos without the
// inner rows in between 10%; the image's border masked behind a branch per row
// 2.5%; clusters of at most 4 CTAs 1 to 3%, of up to 12 4%, runs of 6 rows 2 to
// 6%, of 4 rows with 24 warps an SM 6%, 256-column regions 17%.
//
// The two halves of a warp own two runs on top of each other, the lower one
// upside down. "Outer" rows (towards another warp) and "inner" rows (towards
// the other half, exchanged by a shuffle) then have the same register names
// in both halves. The two halves' rows are an odd number apart, and so is the
// pitch of the staged target: the samples of the two halves, which cover every
// second column each, fall on different banks.
//
// The target J is staged as a box of the CTA's region, shifted by the integer
// part of the starting flow at its centre, with a margin of kMX columns and
// kMY rows and clamp-to-edge values; a sample whose four taps fall outside the
// box is read from global memory instead, one after the other in a thread: the
// margins are what two CTAs an SM leave of the shared memory. With 8 columns
// and 3 rows, 2.2% of the samples of a 4000 x 1500 pair with parallax steps and
// uncorrected gain (1.3% now) lay outside, half of them by rows: 826 us the
// flow of that pair against 681, and 592 against 578 where flows are smooth.
// 8 rows with 8 columns, 6 with 12 or 7 with 10 take the same time within 1%.
// Flows are kept relative to the cluster's reference flow (the starting flow at
// its centre) so that FP32 rounding does not grow with the size of the flow.
#pragma once

#include <type_traits>

#include "bounds.cuh"
#include "common.cuh"

namespace {
__device__ unsigned g_lost_halos;  // threads that gave up a wait, since the last read
}  // namespace

namespace pano {
namespace lks {

constexpr int kMX = 16;           // target box margin, columns
constexpr int kMY = 5;            // target box margin, rows

template <int RAD, int R, int WX, int WY>
struct StreamGeom {
    static constexpr int RW = 32 * WX;               // region columns
    static constexpr int NP = RW / 2;                // column pairs
    static constexpr int RH = 2 * R * WY;            // region rows of one CTA
    static constexpr int threads = 32 * WX * WY;
    static constexpr int JP = RW + 2 * kMX + 1;      // pitch of the target box (odd), RW + 2 kMX columns used
    static constexpr int JH = RH + 2 * kMY;
    static constexpr int VP = NP + 4;                // column sums: two zero pairs on either side
    static constexpr int TP = RW + 4, TH = RH + 2 * (RAD + 1);  // staged template
    static constexpr int NJ = JP * JH, NG = RH * NP, NV = RH * VP, NT = TP * TH, NO = 2 * WY * 2 * RAD * NP;
    static constexpr size_t kJ = 0;
    static constexpr size_t kGA = (kJ + sizeof(float) * NJ + 15) / 16 * 16;
    static constexpr size_t kGB = kGA + sizeof(float4) * NG;
    static constexpr size_t kO = kGB + sizeof(float2) * NG;
    static constexpr size_t kV = kO + sizeof(float4) * NO;
    static constexpr size_t kB = kV + sizeof(float4) * NV;  // barriers of the halos [parity][wy][half]
    static constexpr size_t bytes = kB + sizeof(unsigned long long) * 4 * WY;
    static constexpr size_t kT = kGA;                // the template is read before the normal matrices are written
    static_assert(sizeof(float) * NT <= sizeof(float4) * NG + sizeof(float2) * NG, "staged template too large");
    static_assert(R >= 2 * RAD, "a run must cover the rows it exchanges on both sides");
};

// Halo of K steps, rounded to even so that regions start on even pixels.
__host__ __device__ constexpr int stream_halo(int iters, int radius) { return (iters * radius + 1) & ~1; }

// Paired FP32 arithmetic: one instruction for the two pixels of a thread's
// column pair; each lane rounds exactly as the scalar operation would.
__device__ __forceinline__ float2 dup2(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.f, -1.f), a); }

__device__ __forceinline__ void copy_async4(void* dst_smem, const void* src) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst_smem);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void copy_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void copy_async_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory"); }

__device__ __forceinline__ unsigned cluster_rank() {
    unsigned r;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_arrive_relaxed() { asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
// address of this CTA's shared address `p` in the CTA of rank `r`
__device__ __forceinline__ unsigned cluster_map(unsigned p, unsigned r) {
    unsigned d;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(d) : "r"(p), "r"(r));
    return d;
}
// 16 bytes to a CTA of the cluster, counted by the barrier there
__device__ __forceinline__ void cluster_send(unsigned addr, unsigned bar, float2 a, float2 b) {
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.f32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(addr),
                 "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "r"(bar)
                 : "memory");
}
__device__ __forceinline__ void bar_init(unsigned bar) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar) : "memory");
}
// the barrier's current phase ends when `bytes` have arrived
__device__ __forceinline__ void bar_expect(unsigned bar, unsigned bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
// Waits until the phase of this parity has ended; false if it has not after
// kWaitTries tries, a quarter of a second (a try that fails takes 3.9 us). No
// launch that the host checks let through comes to that: a cluster is scheduled
// as a whole. (A limit by the clock instead, or no further waits for a thread
// that has given up once, cost 2 to 4% of the pairs and rigs: a flag carried
// from wait to wait, and spills.)
constexpr int kWaitTries = 1 << 16;
__device__ __forceinline__ bool bar_try(unsigned bar, unsigned parity) {
    unsigned done;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
        : "=r"(done)
        : "r"(bar), "r"(parity)
        : "memory");
    return done != 0;
}
__device__ __forceinline__ bool bar_retry(unsigned bar, unsigned parity) {
    for (int n = 0; n < kWaitTries; ++n)
        if (bar_try(bar, parity)) return true;
    return false;
}
__device__ __forceinline__ bool bar_wait(unsigned bar, unsigned parity) {
    return bar_try(bar, parity) || bar_retry(bar, parity);
}
// shared-memory load at a byte address plus a constant
template <int OFF>
__device__ __forceinline__ float ld_shared(unsigned addr) {
    float v;
    asm volatile("ld.shared.f32 %0, [%1+%2];" : "=f"(v) : "r"(addr), "n"(OFF));
    return v;
}
template <int N>
__device__ __forceinline__ void named_barrier(int id) { asm volatile("bar.sync %0, %1;" ::"r"(id), "n"(N) : "memory"); }

// Starting flow of pixel (x, y): zero, the given one, or twice the coarser
// level's flow at (x/2, y/2), bilinear.
__device__ __forceinline__ float2 start_flow_s(const LkArgs& a, const LkDir& D, int x, int y) {
    if (a.mode == 0 || D.uin == nullptr) return make_float2(0.f, 0.f);
    const float2* __restrict__ u = reinterpret_cast<const float2*>(D.uin);
    if (a.mode == 2) return u[(long long)y * D.uin_pitch + x];
    int x0 = x >> 1, y0 = y >> 1;
    float fx = (x & 1) ? 0.5f : 0.f, fy = (y & 1) ? 0.5f : 0.f;
    int xa = min(x0, a.in_w - 1), xb = min(x0 + 1, a.in_w - 1);
    int ya = min(y0, a.in_h - 1), yb = min(y0 + 1, a.in_h - 1);
    float2 u00 = u[(long long)ya * D.uin_pitch + xa], u10 = u[(long long)ya * D.uin_pitch + xb];
    float2 u01 = u[(long long)yb * D.uin_pitch + xa], u11 = u[(long long)yb * D.uin_pitch + xb];
    float tx = fmaf(fx, u10.x - u00.x, u00.x), bx = fmaf(fx, u11.x - u01.x, u01.x);
    float ty = fmaf(fx, u10.y - u00.y, u00.y), by = fmaf(fx, u11.y - u01.y, u01.y);
    return make_float2(2.f * fmaf(fy, bx - tx, tx), 2.f * fmaf(fy, by - ty, ty));
}

__device__ __forceinline__ float2 floor_clamped(float2 v, int w, int h) {
    return make_float2(floorf(fminf(fmaxf(v.x, -(float)(w + 2)), (float)(w + 2))),
                       floorf(fminf(fmaxf(v.y, -(float)(h + 2)), (float)(h + 2))));
}

// A sample outside the staged box (large or non-finite offsets): clamped taps
// of the global plane. Rare, and kept out of line.
template <class Ts>
__device__ __noinline__ float far_sample(const Ts* J, int pitch, int w, int h, int x, int y, float ox, float oy) {
    return sample_plane(J, pitch, w, h, x, y, ox, oy);
}

// Sums of 2 RAD + 1 consecutive elements of e: out[j] = e[j] + ... + e[j + 2 RAD].
template <int RAD, int N>
__device__ __forceinline__ void window_sums(const float2 (&e)[N + 2 * RAD], float2 (&out)[N]) {
    float2 s[N + 2 * RAD - 1];  // pairs
#pragma unroll
    for (int i = 0; i < N + 2 * RAD - 1; ++i) s[i] = add2(e[i], e[i + 1]);
#pragma unroll
    for (int j = 0; j < N; ++j) {
        if constexpr (RAD == 1) out[j] = add2(s[j], e[j + 2]);
        else if constexpr (RAD == 2) out[j] = add2(add2(s[j], s[j + 2]), e[j + 4]);
        else out[j] = add2(add2(add2(s[j], s[j + 2]), s[j + 4]), e[j + 6]);
    }
}

// Sums over the 2 RAD + 1 columns around each of a column pair c: l and r are
// the neighbouring pairs, ll and rr the columns beyond them (RAD 3).
template <int RAD>
__device__ __forceinline__ float2 row_sums(float ll, float2 l, float2 c, float2 r, float rr) {
    float m = c.x + c.y;
    if constexpr (RAD == 1) return make_float2(m + l.y, m + r.x);
    m += l.y + r.x;
    if constexpr (RAD == 2) return make_float2(m + l.x, m + r.y);
    m += l.x + r.y;
    return make_float2(m + ll, m + rr);
}

// One CTA's part of one segment: direction `dir`, region columns
// [ox, ox + RW), the cluster's region rows from oyc on; the pixels
// [x_lo, x_hi) x [y_lo, y_hi) of the result are written. ox and oyc are even
// and not negative. A float2 holds the same quantity of the thread's two
// columns. LATE: with a.early, what does not depend on the starting flow is done
// before the previous kernel (the coarser level) has ended.
template <int RAD, int R, int WX, int WY, bool LATE, class Ts>
__device__ __forceinline__ void lk_stream_item(const LkArgs& a, int dir, int ox, int oyc, int csize, int x_lo, int x_hi,
                                               int y_lo, int y_hi, unsigned char* smem) {
    using Geo = StreamGeom<RAD, R, WX, WY>;
    constexpr int RW = Geo::RW, RH = Geo::RH, NP = Geo::NP, JP = Geo::JP, JH = Geo::JH, VP = Geo::VP, TP = Geo::TP,
                  TH = Geo::TH;
    constexpr int NJ = Geo::NJ, NG = Geo::NG, NV = Geo::NV, NT = Geo::NT, NO = Geo::NO;
    (void)NG, (void)NV, (void)NT, (void)NO, (void)NJ;
    constexpr bool kAsync = std::is_same<Ts, float>::value;  // cp.async of 4-byte elements
    float* sJ = reinterpret_cast<float*>(smem + Geo::kJ);
    float4* sGA = reinterpret_cast<float4*>(smem + Geo::kGA);  // inverse normal matrices: (i11, i11', i12, i12')
    float2* sGB = reinterpret_cast<float2*>(smem + Geo::kGB);  // (i22, i22')
    float4* sO = reinterpret_cast<float4*>(smem + Geo::kO);    // outer halos [parity][wy][half][RAD][NP]: (Px, Px', Py, Py')
    float4* sV = reinterpret_cast<float4*>(smem + Geo::kV);    // column sums, rows in run order: (Vx, Vx', Vy, Vy')
    float* sT = reinterpret_cast<float*>(smem + Geo::kT);      // template, before the normal matrices

    const LkDir D = dir ? a.dir[1] : a.dir[0];
    const int w = a.w, h = a.h;
    const Ts* __restrict__ T = static_cast<const Ts*>(D.T);
    const Ts* __restrict__ J = static_cast<const Ts*>(D.J);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int wx = warp % WX, wy = warp / WX, half = lane >> 4;
    const int rank = (int)cluster_rank();
    const int oy = oyc + rank * RH;
    const int px = wx * 16 + (lane & 15), rx = 2 * px;    // the thread's column pair
    const int r0 = wy * 2 * R + (half ? 2 * R - 1 : 0);   // region row of row 0 of the run
    const int dr = half ? -1 : 1;                         // and the step from one of its rows to the next
    const int y0 = oy + r0, x0 = ox + rx;
    const int srow = (wy * 2 + half) * R;                 // the run's rows in the arrays that are in run order

    // ---- stage the template and the target box, with clamped borders
    auto stage = [&](const Ts* __restrict__ src, int pitch, int bx, int by, float* dst, int dp, int n, int rows, int site) {
        (void)site;
        constexpr int NC = (RW + 2 * kMX + 31) / 32;
        int xs[NC];
#pragma unroll
        for (int c = 0; c < NC; ++c) xs[c] = min(max(bx + lane + 32 * c, 0), w - 1);
        for (int r = warp; r < rows; r += WX * WY) {
            const Ts* row = src + (long long)min(max(by + r, 0), h - 1) * pitch;
            float* d = dst + r * dp + lane;
#pragma unroll
            for (int c = 0; c < NC; ++c)
                if (lane + 32 * c < n) {
                    if constexpr (kAsync) copy_async4(d + 32 * c, row + PANO_IDX(xs[c], w, site));
                    else d[32 * c] = ld_f32(row + PANO_IDX(xs[c], w, site));
                }
        }
        copy_async_commit();
    };
    if (!(LATE && a.early)) {
        grid_wait();
        // large levels: the successor's CTAs would only take slots (released
        // here, a 960 x 1000 pair takes 5% longer, a 4000 x 1500 one 1%)
        if (LATE) grid_release();
    }
    stage(T, D.pitchT, ox - 1, oy - (RAD + 1), sT + 1, TP, RW + 3, TH, 110);
    // reference flow of the cluster; the target box, shifted by the flow at the CTA's centre
    float2 ref, off;
    auto stage_target = [&]() {
        ref = start_flow_s(a, D, min(ox + RW / 2, w - 1), min(oyc + csize * RH / 2, h - 1));
        const float2 sh = floor_clamped(start_flow_s(a, D, min(ox + RW / 2, w - 1), min(oy + RH / 2, h - 1)), w, h);
        off = make_float2(ref.x - sh.x, ref.y - sh.y);
        stage(J, D.pitchJ, ox + (int)sh.x - kMX, oy + (int)sh.y - kMY, sJ, JP, RW + 2 * kMX, JH, 111);
    };
    const bool late = LATE && a.early;
    if (!late) stage_target();
    // the box's unused last column marks samples that fall outside the box
    if (tid < 4 * WY) bar_init((unsigned)__cvta_generic_to_shared(smem + Geo::kB) + 8 * tid);
    if (tid < JH) PANO_AT(sJ, tid * JP + JP - 1, NJ, 112) = __int_as_float(0x7fffffff);
    {
        const float4 z4 = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int i = tid; i < NO; i += Geo::threads) PANO_AT(sO, i, NO, 113) = z4;
        for (int i = tid; i < 4 * RH; i += Geo::threads)
            PANO_AT(sV, (i >> 2) * VP + ((i & 3) < 2 ? (i & 3) : NP + (i & 3)), NV, 114) = z4;
    }
    // pixels outside the image have no gradient, and count nowhere
    const bool edge = oy < RAD || oy + RH + RAD > h || ox + RW > w;
    const bool cin0 = x0 < w, cin1 = x0 + 1 < w;
    auto row_in = [&](int j) { return (unsigned)(y0 + dr * j) < (unsigned)h; };

    if (late) copy_async_wait<0>();
    else copy_async_wait<1>();
    __syncthreads();

    // ---- template, gradient and the normal matrices
    float2 t[R], gx[R], gy[R];
    {
        float2 q11[R + 2 * RAD], q12[R + 2 * RAD], q22[R + 2 * RAD];
        {
            const int to = (r0 + RAD + 1) * TP + 2 + rx, dt = dr * TP;  // row 0 of the run
            const float2 hs = dup2(half ? -0.5f : 0.5f);
            float2 pv = PANO_VEC(const float2, sT, to - (RAD + 1) * dt, 2, NT, 115);
            float2 cv = PANO_VEC(const float2, sT, to - RAD * dt, 2, NT, 116);
#pragma unroll
            for (int i = -RAD; i < R + RAD; ++i) {
                const float2 nv = PANO_VEC(const float2, sT, to + (i + 1) * dt, 2, NT, 117);
                const float lf = PANO_AT(sT, to + i * dt - 1, NT, 118), rt = PANO_AT(sT, to + i * dt + 2, NT, 119);
                float2 hx = make_float2(0.5f * (cv.y - lf), 0.5f * (rt - cv.x)), hy = mul2(hs, sub2(nv, pv));
                if (edge) {
                    const bool in = row_in(i);
                    if (!(in && cin0)) hx.x = hy.x = 0.f;
                    if (!(in && cin1)) hx.y = hy.y = 0.f;
                }
                if (i >= 0 && i < R) t[i] = cv, gx[i] = hx, gy[i] = hy;
                q11[i + RAD] = mul2(hx, hx);
                q12[i + RAD] = mul2(hx, hy);
                q22[i + RAD] = mul2(hy, hy);
                pv = cv;
                cv = nv;
            }
        }
        float2 c11[R], c12[R], c22[R];
        window_sums<RAD, R>(q11, c11);
        window_sums<RAD, R>(q12, c12);
        window_sums<RAD, R>(q22, c22);
        __syncthreads();  // the template is read
#pragma unroll
        for (int j = 0; j < R; ++j) {
            const int o = (srow + j) * NP + px;
            PANO_AT(sGA, o, NG, 120) = make_float4(c11[j].x, c11[j].y, c12[j].x, c12[j].y);
            PANO_AT(sGB, o, NG, 121) = c22[j];
        }
        named_barrier<32 * WX>(1 + wy);
        const bool hl = px > 0, hr = px + 1 < NP;                     // neighbouring pairs inside the region
        const bool hl2 = px > 1 && RAD == 3, hr2 = px + 2 < NP && RAD == 3;
#pragma unroll
        for (int j = 0; j < R; ++j) {
            const int o = (srow + j) * NP + px;
            const float4 z4 = make_float4(0.f, 0.f, 0.f, 0.f);
            const float2 z2 = make_float2(0.f, 0.f);
            const float4 l = hl ? PANO_AT(sGA, o - 1, NG, 122) : z4, r = hr ? PANO_AT(sGA, o + 1, NG, 123) : z4;
            const float2 lb = hl ? PANO_AT(sGB, o - 1, NG, 124) : z2, rb = hr ? PANO_AT(sGB, o + 1, NG, 125) : z2;
            float4 l2 = z4, r2 = z4;
            float2 lb2 = z2, rb2 = z2;
            if constexpr (RAD == 3) {
                if (hl2) l2 = PANO_AT(sGA, o - 2, NG, 126), lb2 = PANO_AT(sGB, o - 2, NG, 127);
                if (hr2) r2 = PANO_AT(sGA, o + 2, NG, 128), rb2 = PANO_AT(sGB, o + 2, NG, 129);
            }
            c11[j] = row_sums<RAD>(l2.y, make_float2(l.x, l.y), c11[j], make_float2(r.x, r.y), r2.x);
            c12[j] = row_sums<RAD>(l2.w, make_float2(l.z, l.w), c12[j], make_float2(r.z, r.w), r2.z);
            c22[j] = row_sums<RAD>(lb2.y, lb, c22[j], rb, rb2.x);
        }
        named_barrier<32 * WX>(1 + wy);
        const float2 lam2 = dup2(a.lambda);
#pragma unroll
        for (int j = 0; j < R; ++j) {
            const int o = (srow + j) * NP + px;
            const float2 p11 = add2(c11[j], lam2), p22 = add2(c22[j], lam2);
            const float2 det = fma2(p11, p22, mul2(c12[j], make_float2(-c12[j].x, -c12[j].y)));
            float2 iv = make_float2(1.0f / det.x, 1.0f / det.y);
            float2 i11 = mul2(p22, iv), i12 = mul2(c12[j], make_float2(-iv.x, -iv.y)), i22 = mul2(p11, iv);
            if (edge) {
                // pixels outside the image keep a zero (relative) flow
                const bool in = row_in(j);
                if (!(in && cin0)) i11.x = i12.x = i22.x = 0.f;
                if (!(in && cin1)) i11.y = i12.y = i22.y = 0.f;
            }
            PANO_AT(sGA, o, NG, 130) = make_float4(i11.x, i11.y, i12.x, i12.y);
            PANO_AT(sGB, o, NG, 131) = i22;
        }
    }

    if (late) {
        grid_begin();
        stage_target();
    }

    // ---- starting flow, relative to the reference
    float2 ux[R], uy[R];
    if (a.mode == 1 && D.uin != nullptr) {
        // x and y of the run's first pixel pair (in image order) are even: the
        // fine rows lie on or between NE coarse rows, e[i] in run order
        // (downwards in the upper half, upwards in the lower one)
        constexpr int NE = (R - 1) / 2 + 2;
        const float2* __restrict__ uc = reinterpret_cast<const float2*>(D.uin);
        const int xa = min(x0 >> 1, a.in_w - 1), xb = min((x0 >> 1) + 1, a.in_w - 1);
        const int cy = (oy + wy * 2 * R) / 2 + (half ? R : 0);
        const long long NUI = (long long)(a.in_h - 1) * D.uin_pitch + a.in_w;
        (void)NUI;
        float2 ex[NE], ey[NE];
#pragma unroll
        for (int i = 0; i < NE; ++i) {
            const long long ro = (long long)min(cy + dr * i, a.in_h - 1) * D.uin_pitch;
            const float2 ua = PANO_AT(uc, ro + xa, NUI, 132), ub = PANO_AT(uc, ro + xb, NUI, 133);
            ex[i] = fma2(make_float2(0.f, 0.5f), dup2(ub.x - ua.x), dup2(ua.x));
            ey[i] = fma2(make_float2(0.f, 0.5f), dup2(ub.y - ua.y), dup2(ua.y));
        }
        const float2 rx2 = dup2(-ref.x), ry2 = dup2(-ref.y);
#pragma unroll
        for (int j = 0; j < R; ++j) {
            const float2 fy = dup2(((j ^ half) & 1) ? 0.5f : 0.f);
            const float2 px_ = ex[j >> 1], qx = ex[(j >> 1) + 1], py_ = ey[j >> 1], qy = ey[(j >> 1) + 1];
            const float2 tx = half ? qx : px_, bx = half ? px_ : qx, ty = half ? qy : py_, by = half ? py_ : qy;
            ux[j] = fma2(dup2(2.f), fma2(fy, sub2(bx, tx), tx), rx2);
            uy[j] = fma2(dup2(2.f), fma2(fy, sub2(by, ty), ty), ry2);
        }
    } else {
#pragma unroll
        for (int j = 0; j < R; ++j) {
            const int y = min(y0 + dr * j, h - 1);
            const float2 s0 = start_flow_s(a, D, min(x0, w - 1), y), s1 = start_flow_s(a, D, min(x0 + 1, w - 1), y);
            ux[j] = make_float2(s0.x - ref.x, s1.x - ref.x);
            uy[j] = make_float2(s0.y - ref.y, s1.y - ref.y);
        }
    }
    if (edge) {
#pragma unroll
        for (int j = 0; j < R; ++j) {
            const bool in = row_in(j);
            if (!(in && cin0)) ux[j].x = uy[j].x = 0.f;
            if (!(in && cin1)) ux[j].y = uy[j].y = 0.f;
        }
    }

    // Where this run's outer rows go: the run above (upper half) or below
    // (lower half), in this CTA or its neighbour; none at the cluster's ends.
    // Every halo has a barrier that counts its bytes, one per parity of the
    // step: a run goes on as soon as its own two neighbours have sent. A halo
    // is overwritten two steps later, when the sender has received what its
    // reader sent after reading it.
    const int nwy = half ? wy + 1 : wy - 1;
    const int nrank = nwy < 0 ? rank - 1 : nwy >= WY ? rank + 1 : rank;
    const bool send = nrank >= 0 && nrank < csize;
    const int nslot = ((nwy + WY) % WY) * 2 + (half ^ 1);
    const unsigned so = (unsigned)__cvta_generic_to_shared(sO), sb = (unsigned)__cvta_generic_to_shared(smem + Geo::kB);
    const unsigned odst = cluster_map(so + (nslot * RAD * NP + px) * (unsigned)sizeof(float4), (unsigned)(send ? nrank : rank));
    const unsigned bdst = cluster_map(sb + nslot * 8, (unsigned)(send ? nrank : rank));
    const int oslot = ((wy * 2 + half) * RAD) * NP + px;  // this run's outer halo
    const bool from_above = wy > 0 || rank > 0, from_below = wy + 1 < WY || rank + 1 < csize;
    const unsigned bown = sb + wy * 16;  // this warp's barriers: above, below
    constexpr unsigned kHaloBytes = RAD * NP * sizeof(float4);
    bool lost = false;
    // Sample position: 1.5 * 2^23 + position, rounded down, holds the tap's
    // column / row of the box in its low mantissa bits (its bits are those of
    // 1.5 * 2^23 plus the integer, exact while |o| < 2^21).
    constexpr float kMagic = 12582912.0f;
    const float2 mgx = make_float2(kMagic + (float)(rx + kMX), kMagic + (float)(rx + 1 + kMX));
    const float mgy0 = kMagic + (float)(r0 + kMY), mgd = (float)dr;
    const unsigned sj = (unsigned)__cvta_generic_to_shared(sJ);
    const unsigned jbase = sj - 4u * (0x4B400000u * (unsigned)(JP + 1)), jnone = sj + 4u * (JP - 1);
    const float2 offx = dup2(off.x), offy = dup2(off.y), lam2 = dup2(a.lambda);
    const int vo = srow * VP + 2 + px, go = srow * NP + px;

    copy_async_wait<0>();
    if (wx == 0 && lane == 0) {
        // the barriers were initialised before the __syncthreads above
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            if (from_above) bar_expect(bown + q * (WY * 16), kHaloBytes);
            if (from_below) bar_expect(bown + q * (WY * 16) + 8, kHaloBytes);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncwarp();
    cluster_arrive();  // the staged target and the barriers are visible, the zeroed halos come before a neighbour's rows
    cluster_wait();

    // The steps, with and without the mask of the pixels outside the image (a
    // branch per row instead would keep the rows' loads from overlapping).
    auto steps = [&](auto masked) {
#pragma unroll 1
        for (int k = 0; k < a.iters; ++k) {
            float2 Px[R], Py[R];
            // ---- A: residual products of rows [JB, JE)
            auto products = [&](auto jb, auto je) {
                constexpr int JB = decltype(jb)::value, JE = decltype(je)::value;
                float2 acc = make_float2(0.f, 0.f);
#pragma unroll
                for (int j = JB; j < JE; ++j) {
                    // J at the pixel + ref + u
                    const float2 o_x = add2(offx, ux[j]), o_y = add2(offy, uy[j]);
                    const float my = fmaf((float)j, mgd, mgy0);
                    const float2 tx = make_float2(__fadd_rd(o_x.x, mgx.x), __fadd_rd(o_x.y, mgx.y));
                    const float2 ty = make_float2(__fadd_rd(o_y.x, my), __fadd_rd(o_y.y, my));
                    const float2 ax = sub2(o_x, sub2(tx, mgx)), ay = sub2(o_y, sub2(ty, dup2(my)));
                    unsigned p0 = (__float_as_uint(ty.x) * (unsigned)JP + __float_as_uint(tx.x)) * 4u + jbase;
                    unsigned p1 = (__float_as_uint(ty.y) * (unsigned)JP + __float_as_uint(tx.y)) * 4u + jbase;
                    // a sample outside the box reads the marker instead
                    p0 = fabsf(o_x.x) < (float)kMX && fabsf(o_y.x) < (float)kMY ? p0 : jnone;
                    p1 = fabsf(o_x.y) < (float)kMX && fabsf(o_y.y) < (float)kMY ? p1 : jnone;
                    PANO_FLAG(p0 - sj > 4u * (NJ - JP - 2) || p1 - sj > 4u * (NJ - JP - 2), 140);
                    const float2 i00 = make_float2(ld_shared<0>(p0), ld_shared<0>(p1));
                    const float2 i10 = make_float2(ld_shared<4>(p0), ld_shared<4>(p1));
                    const float2 i01 = make_float2(ld_shared<4 * JP>(p0), ld_shared<4 * JP>(p1));
                    const float2 i11 = make_float2(ld_shared<4 * JP + 4>(p0), ld_shared<4 * JP + 4>(p1));
                    const float2 top = fma2(ax, sub2(i10, i00), i00), bot = fma2(ax, sub2(i11, i01), i01);
                    const float2 jw = fma2(ay, sub2(bot, top), top);
                    float2 s = fma2(gx[j], ux[j], fma2(gy[j], uy[j], sub2(t[j], jw)));
                    if constexpr (decltype(masked)::value) {  // nothing from outside the image
                        const bool in = row_in(j);
                        if (!(in && cin0)) s.x = 0.f;
                        if (!(in && cin1)) s.y = 0.f;
                    }
                    acc = add2(acc, s);
                    Px[j] = mul2(gx[j], s);
                    Py[j] = mul2(gy[j], s);
                }
                if (__builtin_expect(!(acc.x + acc.y == acc.x + acc.y), 0)) {
                    // some samples (or their inputs) are not numbers: those outside
                    // the box are taken from the global plane
#pragma unroll
                    for (int j = JB; j < JE; ++j)
#pragma unroll
                        for (int c = 0; c < 2; ++c) {
                            const float vx = c ? ux[j].y : ux[j].x, vy = c ? uy[j].y : uy[j].x;
                            const float o_x = off.x + vx, o_y = off.y + vy;
                            if ((fabsf(o_x) < (float)kMX && fabsf(o_y) < (float)kMY) || !row_in(j) || !(c ? cin1 : cin0)) continue;
                            const float jw = far_sample(J, D.pitchJ, w, h, x0 + c, y0 + dr * j, ref.x + vx, ref.y + vy);
                            const float hx = c ? gx[j].y : gx[j].x, hy = c ? gy[j].y : gy[j].x;
                            const float s = fmaf(hx, vx, fmaf(hy, vy, (c ? t[j].y : t[j].x) - jw));
                            (c ? Px[j].y : Px[j].x) = hx * s;
                            (c ? Py[j].y : Py[j].x) = hy * s;
                        }
                }
            };
            // ---- C: row sums, solve, update of row j with column sums (vx, vy)
            auto update = [&](int j, float2 vx, float2 vy) {
                const float4 l = PANO_AT(sV, vo + j * VP - 1, NV, 146), r = PANO_AT(sV, vo + j * VP + 1, NV, 147);
                float4 l2 = make_float4(0.f, 0.f, 0.f, 0.f), r2 = l2;
                if constexpr (RAD == 3) {
                    l2 = PANO_AT(sV, vo + j * VP - 2, NV, 148);
                    r2 = PANO_AT(sV, vo + j * VP + 2, NV, 149);
                }
                const float2 mx = row_sums<RAD>(l2.y, make_float2(l.x, l.y), vx, make_float2(r.x, r.y), r2.x);
                const float2 my = row_sums<RAD>(l2.w, make_float2(l.z, l.w), vy, make_float2(r.z, r.w), r2.z);
                const float4 ga = PANO_AT(sGA, go + j * NP, NG, 152);
                const float2 gb = PANO_AT(sGB, go + j * NP, NG, 153), g11 = make_float2(ga.x, ga.y), g12 = make_float2(ga.z, ga.w);
                const float2 qx = fma2(lam2, ux[j], mx), qy = fma2(lam2, uy[j], my);
                ux[j] = fma2(g11, qx, mul2(g12, qy));
                uy[j] = fma2(g12, qx, mul2(gb, qy));
            };

            // the outer rows first: they are on their way while the others are formed
            products(std::integral_constant<int, 0>{}, std::integral_constant<int, RAD>{});
            if (send) {
#pragma unroll
                for (int j = 0; j < RAD; ++j)
                    cluster_send(odst + ((k & 1) * (NO / 2) + j * NP) * (unsigned)sizeof(float4), bdst + (k & 1) * (WY * 16), Px[j], Py[j]);
            }
            __syncwarp();
            // nobody sends any more: no CTA ends before its neighbours are here
            if (k + 1 == a.iters) cluster_arrive_relaxed();
            products(std::integral_constant<int, RAD>{}, std::integral_constant<int, R>{});
            __syncwarp();
            // ---- B: column sums of the rows that need no outer halo
            float2 hx[RAD], hy[RAD];  // sums of rows 0 .. i + RAD
            {
                float2 e[R + RAD], f[R + RAD];
#pragma unroll
                for (int j = 0; j < R; ++j) e[j] = Px[j], f[j] = Py[j];
#pragma unroll
                for (int i = 0; i < RAD; ++i) {
                    // the other half's inner rows
                    e[R + i].x = __shfl_xor_sync(0xffffffffu, Px[R - 1 - i].x, 16);
                    e[R + i].y = __shfl_xor_sync(0xffffffffu, Px[R - 1 - i].y, 16);
                    f[R + i].x = __shfl_xor_sync(0xffffffffu, Py[R - 1 - i].x, 16);
                    f[R + i].y = __shfl_xor_sync(0xffffffffu, Py[R - 1 - i].y, 16);
                }
                hx[0] = e[0], hy[0] = f[0];
#pragma unroll
                for (int i = 1; i <= RAD; ++i) hx[0] = add2(hx[0], e[i]), hy[0] = add2(hy[0], f[i]);
#pragma unroll
                for (int i = 1; i < RAD; ++i) hx[i] = add2(hx[i - 1], e[RAD + i]), hy[i] = add2(hy[i - 1], f[RAD + i]);
                float2 vx[R - RAD], vy[R - RAD];
                window_sums<RAD, R - RAD>(e, vx);
                window_sums<RAD, R - RAD>(f, vy);
#pragma unroll
                for (int j = RAD; j < R; ++j) {
                    Px[j] = vx[j - RAD], Py[j] = vy[j - RAD];
                    PANO_AT(sV, vo + j * VP, NV, 145) = make_float4(Px[j].x, Px[j].y, Py[j].x, Py[j].y);
                }
            }
            named_barrier<32 * WX>(1 + wy);
#pragma unroll
            for (int j = RAD; j < R; ++j) update(j, Px[j], Py[j]);
            // ---- and of the outer rows, when the neighbours' rows are here
            {
                const unsigned bar = bown + (k & 1) * (WY * 16);
                const unsigned ph = (unsigned)(k >> 1) & 1;
                if (from_above) lost |= !bar_wait(bar, ph);
                if (from_below) lost |= !bar_wait(bar + 8, ph);
                if (wx == 0 && lane == 0 && k + 2 < a.iters) {
                    if (from_above) bar_expect(bar, kHaloBytes);
                    if (from_below) bar_expect(bar + 8, kHaloBytes);
                }
                __syncwarp();
                float2 ex = make_float2(0.f, 0.f), ey = ex;
#pragma unroll
                for (int i = RAD - 1; i >= 0; --i) {
                    // row i lacks the halo's first RAD - i rows
                    const float4 o = PANO_AT(sO, (k & 1) * (NO / 2) + oslot + (RAD - 1 - i) * NP, NO, 144);
                    ex = i == RAD - 1 ? make_float2(o.x, o.y) : add2(ex, make_float2(o.x, o.y));
                    ey = i == RAD - 1 ? make_float2(o.z, o.w) : add2(ey, make_float2(o.z, o.w));
                    hx[i] = add2(hx[i], ex), hy[i] = add2(hy[i], ey);
                    PANO_AT(sV, vo + i * VP, NV, 145) = make_float4(hx[i].x, hx[i].y, hy[i].x, hy[i].y);
                }
            }
            named_barrier<32 * WX>(1 + wy);
#pragma unroll
            for (int i = 0; i < RAD; ++i) update(i, hx[i], hy[i]);
        }
    };
    if (edge) steps(std::true_type{});
    else steps(std::false_type{});

    cluster_wait();
    // ---- the result (not a number where a neighbour's rows never came)
    float2* uo = reinterpret_cast<float2*>(D.uout);
    const float2 end = lost ? dup2(__int_as_float(0x7fffffff)) : ref;
    const bool c0 = x0 >= x_lo && x0 < x_hi, c1 = x0 + 1 >= x_lo && x0 + 1 < x_hi;
    const long long NUO = (long long)(h - 1) * D.uout_pitch + w;
    (void)NUO;
#pragma unroll
    for (int j = 0; j < R; ++j) {
        const int y = y0 + dr * j;
        if (y < y_lo || y >= y_hi) continue;
        const long long o = (long long)y * D.uout_pitch + x0;
        if (c0) PANO_AT(uo, o, NUO, 154) = make_float2(ux[j].x + end.x, uy[j].x + end.y);
        if (c1) PANO_AT(uo, o + 1, NUO, 155) = make_float2(ux[j].y + end.x, uy[j].y + end.y);
    }
    if (__builtin_expect(lost, 0)) atomicAdd(&g_lost_halos, 1u);
}

// How a level is cut: nb bands, ns segments (clusters) per band of csize CTAs
// each; `small` selects the CTA shape.
struct StreamPlan {
    int nb, ns, csize, small;
};

// Rows per run and warps across and down of a CTA. Large levels: the largest
// run whose two CTAs per SM fit in registers (128 a thread) and shared memory
// (104 to 112 KB a CTA). Small levels: narrow, short regions, so that a level
// spreads over more SMs and each has fewer pixels to work through.
template <int RAD, bool SMALL>
struct StreamCfg { static constexpr int R = RAD == 3 ? 6 : 7, WX = 4, WY = 2; };
template <int RAD>
struct StreamCfg<RAD, true> { static constexpr int R = RAD == 3 ? 6 : 4, WX = 2, WY = 2; };

template <int RAD, bool SMALL>
struct CfgGeom : StreamGeom<RAD, StreamCfg<RAD, SMALL>::R, StreamCfg<RAD, SMALL>::WX, StreamCfg<RAD, SMALL>::WY> {
    static constexpr int min_ctas = 512 / StreamGeom<RAD, StreamCfg<RAD, SMALL>::R, StreamCfg<RAD, SMALL>::WX,
                                                     StreamCfg<RAD, SMALL>::WY>::threads;
};

// The region of band bx and segment sy, and the pixels it writes: neighbouring
// regions overlap by twice the halo, and the first and last ones reach the
// image's border, where no halo is needed.
template <int RAD, bool SMALL, class Ts>
__device__ __forceinline__ void lk_stream_cta(const LkArgs& a, int dir, int bx, int sy, int nb, int ns, int csize,
                                              unsigned char* smem) {
    using C = StreamCfg<RAD, SMALL>;
    using Geo = CfgGeom<RAD, SMALL>;
    const int halo = stream_halo(a.iters, RAD);
    const int ox = bx * (Geo::RW - 2 * halo), oy = sy * (csize * Geo::RH - 2 * halo);
    const int x_lo = bx ? ox + halo : 0, x_hi = bx + 1 < nb ? ox + Geo::RW - halo : a.w;
    const int y_lo = sy ? oy + halo : 0, y_hi = sy + 1 < ns ? oy + csize * Geo::RH - halo : a.h;
    lk_stream_item<RAD, C::R, C::WX, C::WY, SMALL, Ts>(a, dir, ox, oy, csize, x_lo, x_hi, y_lo, y_hi, smem);
}

template <int RAD, bool SMALL, class Ts>
__global__ void __launch_bounds__(CfgGeom<RAD, SMALL>::threads, CfgGeom<RAD, SMALL>::min_ctas)
    lk_stream_kernel(const __grid_constant__ LkArgs a, StreamPlan p) {
    extern __shared__ __align__(16) unsigned char smem[];
    const int item = blockIdx.x / p.csize;
    const int per_dir = p.nb * p.ns;
    const int dir = item / per_dir, rem = item - dir * per_dir;
    lk_stream_cta<RAD, SMALL, Ts>(a, dir, rem % p.nb, rem / p.nb, p.nb, p.ns, p.csize, smem);
}

// The same level of several strip pairs in one launch.
template <int RAD, bool SMALL, class Ts>
__global__ void __launch_bounds__(CfgGeom<RAD, SMALL>::threads, CfgGeom<RAD, SMALL>::min_ctas)
    lk_stream_batch_kernel(const __grid_constant__ LkBatch b, int csize) {
    extern __shared__ __align__(16) unsigned char smem[];
    const int item = blockIdx.x / csize;
    int p = 0;
    while (p + 1 < b.n && item >= b.start[p + 1]) ++p;
    const int local = item - b.start[p];
    const int per_dir = b.nb[p] * b.nseg[p];
    const int dir = local / per_dir, rem = local - dir * per_dir;
    lk_stream_cta<RAD, SMALL, Ts>(b.pair[p], dir, rem % b.nb[p], rem / b.nb[p], b.nb[p], b.nseg[p], csize, smem);
}

// Bands and segments of one level, from its size alone (a pair of a rig is cut
// as it is by itself). The number of CTAs on top of each other is made as
// small as possible (each row of a region is computed whether it is halo or
// not), then the clusters; seg_rows > 0 asks for segments of about that many
// rows instead.
template <int RAD>
StreamPlan stream_plan(int w, int h, int iters, int seg_rows) {
    const int halo = stream_halo(iters, RAD);
    StreamPlan p;
    p.small = (long long)w * h * halo < kStreamSmallWork && halo <= kStreamSmallHalo;
    const int RW = p.small ? CfgGeom<RAD, true>::RW : CfgGeom<RAD, false>::RW;
    const int RH = p.small ? CfgGeom<RAD, true>::RH : CfgGeom<RAD, false>::RH;
    auto parts = [halo](int n, int region) {
        return n <= region ? 1 : (n - 2 * halo + region - 2 * halo - 1) / (region - 2 * halo);
    };
    p.nb = parts(w, RW);
    const int c_min = 2 * halo / RH + 1;  // a region must be larger than its halo
    if (seg_rows > 0) {
        const long long c = ((long long)seg_rows + 2 * halo + RH - 1) / RH;
        p.csize = c < c_min ? c_min : c > kStreamMaxCluster ? kStreamMaxCluster : (int)c;
    } else {
        p.csize = c_min;
        long long best = -1;
        for (int c = c_min; c <= kStreamMaxCluster; ++c) {
            const long long n = (long long)parts(h, c * RH) * c;
            if (best < 0 || n < best) {
                best = n;
                p.csize = c;
            }
        }
    }
    p.ns = parts(h, p.csize * RH);
    return p;
}

// Rows of a segment that is a cluster of csize CTAs by itself, as seg_rows asks
// for it; 0 where the halo needs more CTAs, or fewer cover the level.
template <int RAD>
int stream_seg_rows(int w, int h, int iters, int csize) {
    const StreamPlan p = stream_plan<RAD>(w, h, iters, 0);
    const int RH = p.small ? CfgGeom<RAD, true>::RH : CfgGeom<RAD, false>::RH;
    const int rows = csize * RH - 2 * stream_halo(iters, RAD);
    return rows > 0 && (csize - 1) * RH < h ? rows : 0;
}

template <int RAD, class Ts>
cudaError_t launch_rad_stream(const LkArgs& a, int ndirs, cudaStream_t s) {
    const StreamPlan p = stream_plan<RAD>(a.w, a.h, a.iters, a.seg_rows);
    const int items = p.nb * p.ns * ndirs;
    if (p.small) {
        using Geo = CfgGeom<RAD, true>;
        return launch_dependent(lk_stream_kernel<RAD, true, Ts>, dim3(items * p.csize), dim3(Geo::threads), Geo::bytes, s, p.csize, a, p);
    }
    using Geo = CfgGeom<RAD, false>;
    return launch_dependent(lk_stream_kernel<RAD, false, Ts>, dim3(items * p.csize), dim3(Geo::threads), Geo::bytes, s, p.csize, a, p);
}

// One launch for the pairs that are cut with the same CTA shape and cluster
// size; adds the launches to *kernels.
template <int RAD, class Ts>
cudaError_t launch_rad_batch(const LkBatch& in, cudaStream_t s, int* kernels) {
    StreamPlan plan[kMaxBatch];
    for (int p = 0; p < in.n; ++p)
        plan[p] = stream_plan<RAD>(in.pair[p].w, in.pair[p].h, in.pair[p].iters, in.pair[p].seg_rows);
    bool done[kMaxBatch] = {};
    for (int first = 0; first < in.n; ++first) {
        if (done[first]) continue;
        LkBatch b;
        b.n = 0;
        b.start[0] = 0;
        for (int p = first; p < in.n; ++p) {
            if (done[p] || plan[p].small != plan[first].small || plan[p].csize != plan[first].csize) continue;
            done[p] = true;
            b.pair[b.n] = in.pair[p];
            b.nb[b.n] = plan[p].nb;
            b.nseg[b.n] = plan[p].ns;
            b.start[b.n + 1] = b.start[b.n] + 2 * plan[p].nb * plan[p].ns;
            ++b.n;
        }
        const int items = b.start[b.n], csize = plan[first].csize;
        cudaError_t e;
        if (plan[first].small) {
            using Geo = CfgGeom<RAD, true>;
            e = launch_dependent(lk_stream_batch_kernel<RAD, true, Ts>, dim3(items * csize), dim3(Geo::threads), Geo::bytes, s, csize, b, csize);
        } else {
            using Geo = CfgGeom<RAD, false>;
            e = launch_dependent(lk_stream_batch_kernel<RAD, false, Ts>, dim3(items * csize), dim3(Geo::threads), Geo::bytes, s, csize, b, csize);
        }
        if (e != cudaSuccess) return e;
        ++*kernels;
    }
    return cudaSuccess;
}

template <int RAD, bool SMALL, class Ts>
cudaError_t prepare_cfg(int max_smem) {
    using Geo = CfgGeom<RAD, SMALL>;
    if (Geo::bytes > (size_t)max_smem) return cudaErrorInvalidValue;
    cudaError_t e = cudaFuncSetAttribute(lk_stream_kernel<RAD, SMALL, Ts>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)Geo::bytes);
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(lk_stream_batch_kernel<RAD, SMALL, Ts>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)Geo::bytes);
}

template <int RAD, class Ts>
cudaError_t prepare_rad_stream(int max_smem) {
    const cudaError_t e = prepare_cfg<RAD, true, Ts>(max_smem);
    return e != cudaSuccess ? e : prepare_cfg<RAD, false, Ts>(max_smem);
}

// Entry points for one storage type (instantiated by exactly one .cu file).
template <class Ts>
cudaError_t stream_launch(const LkArgs& a, int ndirs, cudaStream_t s) {
    switch (a.radius) {
        case 1: return launch_rad_stream<1, Ts>(a, ndirs, s);
        case 2: return launch_rad_stream<2, Ts>(a, ndirs, s);
        case 3: return launch_rad_stream<3, Ts>(a, ndirs, s);
        default: return cudaErrorInvalidValue;
    }
}

template <class Ts>
cudaError_t stream_launch_batch(const LkBatch& b, cudaStream_t s, int* kernels) {
    switch (b.pair[0].radius) {
        case 1: return launch_rad_batch<1, Ts>(b, s, kernels);
        case 2: return launch_rad_batch<2, Ts>(b, s, kernels);
        case 3: return launch_rad_batch<3, Ts>(b, s, kernels);
        default: return cudaErrorInvalidValue;
    }
}

template <class Ts>
cudaError_t stream_prepare(int max_smem_bytes) {
    cudaError_t e;
    if ((e = prepare_rad_stream<1, Ts>(max_smem_bytes)) != cudaSuccess) return e;
    if ((e = prepare_rad_stream<2, Ts>(max_smem_bytes)) != cudaSuccess) return e;
    return prepare_rad_stream<3, Ts>(max_smem_bytes);
}

// host: add this unit's count of given-up waits to *n and clear it
#define PANO_LKS_LOST_READER(fn)                                                \
    cudaError_t fn(unsigned* n) {                                               \
        unsigned v = 0;                                                         \
        cudaError_t e = cudaMemcpyFromSymbol(&v, g_lost_halos, sizeof(v));      \
        if (e != cudaSuccess || v == 0) return e;                               \
        *n += v;                                                                \
        v = 0;                                                                  \
        return cudaMemcpyToSymbol(g_lost_halos, &v, sizeof(v));                 \
    }

#define PANO_LKS_INSTANTIATE(Ts)                                                      \
    template cudaError_t stream_launch<Ts>(const LkArgs&, int, cudaStream_t);        \
    template cudaError_t stream_launch_batch<Ts>(const LkBatch&, cudaStream_t, int*);    \
    template cudaError_t stream_prepare<Ts>(int);

#define PANO_LKS_EXTERN(Ts)                                                              \
    extern template cudaError_t stream_launch<Ts>(const LkArgs&, int, cudaStream_t);    \
    extern template cudaError_t stream_launch_batch<Ts>(const LkBatch&, cudaStream_t, int*);\
    extern template cudaError_t stream_prepare<Ts>(int);

}  // namespace lks
}  // namespace pano
