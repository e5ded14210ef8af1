// refine.cu -- energy and adjoint kernels for differentiable flow refinement.
//
// Not a step of the paper's method: a build extension that refines a flow by
// gradient steps on the energy
//   E(u) = sum_p (J(p + u(p)) - T(p))^2
//        + alpha sum_p sum_c [ (u_c(p + e_x) - u_c(p))^2 [x < w-1] + (u_c(p + e_y) - u_c(p))^2 [y < h-1] ]
// (data term of the LK step, smoothness term of the Horn-Schunck half of
// [20]). J is sampled with the bilinear clamp-to-edge sampler of the flow
// path. The kernels give E (as a double, used by finite-difference checks),
// dE/du, dE/dT and dE/dJ, and the transpose of the pyramid REDUCE so that
// gradients can be carried to full-resolution images without storing the
// pyramid.
#include <climits>

#include "bounds.cuh"
#include "common.cuh"

namespace pano {

namespace {

constexpr int kEgThreads = 256;
constexpr int kEgCtas = 152 * 8;  // CTAs of the energy alone: each adds one double to E

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
}

// a + b rounded, and the rounding error (Knuth's exact addition).
__device__ __forceinline__ float two_sum(float a, float b, float* err) {
    const float s = __fadd_rn(a, b), t = __fsub_rn(s, a);
    *err = __fadd_rn(__fsub_rn(a, __fsub_rn(s, t)), __fsub_rn(b, t));
    return s;
}

// A sum of squares in three floats: the rounding errors of the products and of
// the additions to `hi` go to `mid`, those of the additions to `mid` to `lo`.
// Over kSquares pixels (four squares each at most) that leaves less than the
// last bit of a double; then the sum goes into one. `big` is the largest
// magnitude added: the errors are exact, or below 2^-70 of the sum, for
// squares of 1e-12 .. 1e15.
constexpr int kSquares = 16;
struct SquareSum {
    float hi = 0.f, mid = 0.f, lo = 0.f, big = 0.f;
    __device__ __forceinline__ void add(float v) {
        const float p = __fmul_rn(v, v), e = __fmaf_rn(v, v, -p);
        float r, r1, r2;
        hi = two_sum(hi, p, &r);
        mid = two_sum(mid, r, &r1);
        mid = two_sum(mid, e, &r2);
        lo = __fadd_rn(lo, __fadd_rn(r1, r2));
        big = fmaxf(big, fabsf(v));
    }
    __device__ __forceinline__ bool exact() const { return big == 0.f || (big >= 1e-12f && big <= 1e15f); }
    __device__ __forceinline__ double value() const { return (double)hi + ((double)mid + (double)lo); }
};

// What a pixel's energy and gradients are made of.
struct EnergyPixel {
    float r;                  // J(p + u) - T
    float fx, fy;             // weights of the second column / row
    int xa, xb, ya, yb;       // taps
    float i00, i10, i01, i11;
    float2 u;
    float2 right, down;       // forward differences (zero at the border)
};

__device__ __forceinline__ EnergyPixel energy_pixel(const EnergyArgs& a, int x, int y) {
    EnergyPixel q;
    const int w = a.w, h = a.h;
    const long long p = (long long)y * w + x;
    const long long nf = (long long)h * w;                      // flow / gradient elements
    const long long nt = (long long)(h - 1) * a.pitch + w, nj = (long long)(h - 1) * a.pitchJ + w;  // elements of T and J
    (void)nf, (void)nt, (void)nj;
    const float2* U = reinterpret_cast<const float2*>(a.u);
    q.u = PANO_AT(U, p, nf, 601);
    // bilinear sample of J at p + u
    const float ox = fminf(fmaxf(q.u.x, -(float)(w + 2)), (float)(w + 2));
    const float oy = fminf(fmaxf(q.u.y, -(float)(h + 2)), (float)(h + 2));
    const float fxf = floorf(ox), fyf = floorf(oy);
    q.fx = ox - fxf, q.fy = oy - fyf;
    const int x0 = x + (int)fxf, y0 = y + (int)fyf;
    q.xa = min(max(x0, 0), w - 1), q.xb = min(max(x0 + 1, 0), w - 1);
    q.ya = min(max(y0, 0), h - 1), q.yb = min(max(y0 + 1, 0), h - 1);
    const long long ra = (long long)q.ya * a.pitchJ, rb = (long long)q.yb * a.pitchJ;
    q.i00 = PANO_AT(a.J, ra + q.xa, nj, 602), q.i10 = PANO_AT(a.J, ra + q.xb, nj, 602);
    q.i01 = PANO_AT(a.J, rb + q.xa, nj, 602), q.i11 = PANO_AT(a.J, rb + q.xb, nj, 602);
    const float top = fmaf(q.fx, q.i10 - q.i00, q.i00), bot = fmaf(q.fx, q.i11 - q.i01, q.i01);
    q.r = fmaf(q.fy, bot - top, top) - PANO_AT(a.T, (long long)y * a.pitch + x, nt, 603);
    q.right = q.down = make_float2(0.f, 0.f);
    if (x < w - 1) {
        const float2 n = PANO_AT(U, p + 1, nf, 604);
        q.right = make_float2(n.x - q.u.x, n.y - q.u.y);
    }
    if (y < h - 1) {
        const float2 n = PANO_AT(U, p + w, nf, 605);
        q.down = make_float2(n.x - q.u.x, n.y - q.u.y);
    }
    return q;
}

// Tiles of 32 x 8 pixels, from blockIdx.x on in steps of the grid.
template <class F>
__device__ __forceinline__ void energy_tiles(const EnergyArgs& a, F f) {
    const int tx = (a.w + 31) / 32, ty = (a.h + kEgThreads / 32 - 1) / (kEgThreads / 32);
    for (int t = blockIdx.x; t < tx * ty; t += gridDim.x) {
        const int by = t / tx, bx = t - by * tx;
        f(bx * 32 + (int)(threadIdx.x & 31), by * (kEgThreads / 32) + (int)(threadIdx.x >> 5));
    }
}

__device__ __noinline__ double energy_in_doubles(const EnergyArgs& a) {
    double d = 0.0, s = 0.0;
    energy_tiles(a, [&](int x, int y) {
        if (x >= a.w || y >= a.h) return;
        const EnergyPixel q = energy_pixel(a, x, y);
        d += (double)q.r * (double)q.r;
        s += (double)q.right.x * q.right.x + (double)q.right.y * q.right.y + (double)q.down.x * q.down.x +
             (double)q.down.y * q.down.y;
    });
    return d + (double)a.alpha * s;
}

// E alone. FP64 instructions run at 1/64 of the FP32 rate here: five squares a
// pixel in doubles, and a double atomic per 256 pixels, took 39 us on 1024^2
// pixels; sums of as many bits in three floats (22 us) and one atomic per CTA of a
// fixed grid take the place of both. A thread adds one double per kSquares
// pixels, so there are fewer roundings than with a double per pixel.
__global__ void __launch_bounds__(kEgThreads) energy_kernel(const __grid_constant__ EnergyArgs a) {
    __shared__ double s_part[kEgThreads / 32];
    grid_begin();
    SquareSum data, smooth;
    double e = 0.0;
    bool exact = true;
    int n = 0;
    auto flush = [&]() {
        exact = exact && data.exact() && smooth.exact();
        e += data.value() + (double)a.alpha * smooth.value();
        data = SquareSum();
        smooth = SquareSum();
        n = 0;
    };
    energy_tiles(a, [&](int x, int y) {
        if (x >= a.w || y >= a.h) return;
        const EnergyPixel q = energy_pixel(a, x, y);
        data.add(q.r);
        smooth.add(q.right.x);
        smooth.add(q.right.y);
        smooth.add(q.down.x);
        smooth.add(q.down.y);
        if (++n == kSquares) flush();
    });
    flush();
    if (!exact) e = energy_in_doubles(a);
    __syncwarp();
    e = warp_sum(e);
    if ((threadIdx.x & 31) == 0) s_part[threadIdx.x >> 5] = e;
    __syncthreads();
    if (threadIdx.x < 32) {
        double v = threadIdx.x < kEgThreads / 32 ? s_part[threadIdx.x] : 0.0;
        v = warp_sum(v);
        if (threadIdx.x == 0) atomicAdd(a.energy, v);
    }
}

// The gradients, times *scale if given. dE/dJ scatters to the four taps; where
// the neighbouring pixel's left taps are this pixel's right ones (a smooth
// flow), one addition serves both.
__global__ void __launch_bounds__(kEgThreads) energy_grad_kernel(const __grid_constant__ EnergyArgs a) {
    grid_begin();
    const int w = a.w, h = a.h;
    const float scale = a.scale ? (float)*a.scale : 1.f;
    energy_tiles(a, [&](int x, int y) {
        const bool in = x < w && y < h;
        const long long p = (long long)y * w + x;
        const long long nf = (long long)h * w;
        (void)nf;
        EnergyPixel q;
        q.xa = q.xb = q.ya = q.yb = -1;
        q.r = q.fx = q.fy = 0.f;
        if (in) {
            q = energy_pixel(a, x, y);
            if (a.grad_u) {
                const float2* U = reinterpret_cast<const float2*>(a.u);
                float2 lap = make_float2(-q.right.x - q.down.x, -q.right.y - q.down.y);
                if (x > 0) {
                    const float2 n = PANO_AT(U, p - 1, nf, 606);
                    lap.x += q.u.x - n.x;
                    lap.y += q.u.y - n.y;
                }
                if (y > 0) {
                    const float2 n = PANO_AT(U, p - w, nf, 607);
                    lap.x += q.u.x - n.x;
                    lap.y += q.u.y - n.y;
                }
                const float jdx = fmaf(q.fy, (q.i11 - q.i01) - (q.i10 - q.i00), q.i10 - q.i00);
                const float jdy = fmaf(q.fx, (q.i11 - q.i10) - (q.i01 - q.i00), q.i01 - q.i00);
                PANO_AT(reinterpret_cast<float2*>(a.grad_u), p, nf, 608) =
                    make_float2((2.f * q.r * jdx + 2.f * a.alpha * lap.x) * scale,
                                (2.f * q.r * jdy + 2.f * a.alpha * lap.y) * scale);
            }
            if (a.grad_T) PANO_AT(a.grad_T, p, nf, 609) = -2.f * q.r * scale;
        }
        if (a.grad_J) {
            const unsigned all = 0xffffffffu;
            const float g = 2.f * q.r * scale;
            float c00 = g * (1.f - q.fy) * (1.f - q.fx), c10 = g * (1.f - q.fy) * q.fx;
            float c01 = g * q.fy * (1.f - q.fx), c11 = g * q.fy * q.fx;
            const float l10 = __shfl_up_sync(all, c10, 1), l11 = __shfl_up_sync(all, c11, 1);
            const int lxb = __shfl_up_sync(all, q.xb, 1), lya = __shfl_up_sync(all, q.ya, 1), lyb = __shfl_up_sync(all, q.yb, 1);
            const bool take = in && (threadIdx.x & 31) > 0 && lxb == q.xa && lya == q.ya && lyb == q.yb;
            if (take) c00 += l10, c01 += l11;
            const bool taken = __shfl_down_sync(all, (int)take, 1) && (threadIdx.x & 31) < 31;
            if (in) {
                float* GJ = a.grad_J;
                atomicAdd(&PANO_AT(GJ, (long long)q.ya * w + q.xa, nf, 610), c00);
                atomicAdd(&PANO_AT(GJ, (long long)q.yb * w + q.xa, nf, 610), c01);
                if (!taken) {
                    atomicAdd(&PANO_AT(GJ, (long long)q.ya * w + q.xb, nf, 610), c10);
                    atomicAdd(&PANO_AT(GJ, (long long)q.yb * w + q.xb, nf, 610), c11);
                }
            }
        }
    });
}

// Rows (or columns) of the level below that a source row feeds, with their
// REDUCE weights: source index s receives weight k[t] from destination index
// d whenever clamp(2 d + t, 0, n - 1) == s, t in [-2, 2]. At most four
// destination indices qualify: d in [s/2 - 1, s/2 + 2] (border clamping adds
// weight, never indices); a weight of zero marks an unused candidate.
__device__ __forceinline__ void reduce_taps(int s, int n, int nd, int (&d)[4], float (&wt)[4]) {
    const float k[5] = {1.f / 16, 4.f / 16, 6.f / 16, 4.f / 16, 1.f / 16};
    const int base = (s >> 1) - 1;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int dd = base + i;
        float acc = 0.f;
#pragma unroll
        for (int t = -2; t <= 2; ++t)
            if (min(max(2 * dd + t, 0), n - 1) == s) acc += k[t + 2];
        const bool ok = dd >= 0 && dd < nd;
        d[i] = min(max(dd, 0), nd - 1);
        wt[i] = ok ? acc : 0.f;
    }
}

__device__ __noinline__ float adjoint_pixel(const float* gdst, int h, int w, int dst_pitch, int x, int y) {
    const int hd = (h + 1) / 2, wd = (w + 1) / 2;
    int dy[4], dx[4];
    float wy[4], wx[4];
    reduce_taps(y, h, hd, dy, wy);
    reduce_taps(x, w, wd, dx, wx);
    const long long nd = (long long)(hd - 1) * dst_pitch + wd;  // elements of the gradient of the output
    (void)nd;
    float acc = 0.f;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const long long ro = (long long)dy[i] * dst_pitch;
        float racc = 0.f;
#pragma unroll
        for (int j = 0; j < 4; ++j) racc = fmaf(wx[j], PANO_AT(gdst, ro + dx[j], nd, 611), racc);
        acc = fmaf(wy[i], racc, acc);
    }
    return acc;
}

// Transpose of REDUCE for up to two planes (blockIdx.z): a thread forms the
// 2 x 2 source pixels (2 yd, 2 xd) .. of one gradient pixel from the 3 x 3
// around it (even sources: 1 6 1, odd ones: 4 4, in sixteenths), with the
// order of operations of adjoint_pixel; pixels whose taps the border clamps
// use that. 40 us a plane of 1777 x 1210 with a thread and sixteen searched
// taps per source pixel.
__global__ void __launch_bounds__(256) pyr_down_adjoint_kernel(const __grid_constant__ AdjointArgs a) {
    grid_begin();
    const float* gdst = a.gdst[blockIdx.z];
    float* gsrc = a.gsrc[blockIdx.z];
    const int h = a.h, w = a.w, hd = (h + 1) / 2, wd = (w + 1) / 2;
    const int xd = blockIdx.x * blockDim.x + threadIdx.x, yd = blockIdx.y * blockDim.y + threadIdx.y;
    if (xd >= wd || yd >= hd) return;
    const long long nd = (long long)(hd - 1) * a.dst_pitch + wd, ns = (long long)(h - 1) * a.src_pitch + w;
    (void)nd, (void)ns;
    float v[2][2];
    if (xd > 0 && yd > 0 && xd + 2 < wd && yd + 2 < hd) {
        const float k1 = 1.f / 16, k4 = 4.f / 16, k6 = 6.f / 16;
        float e[3], o[3];  // even and odd column of the three rows
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            const long long ro = (long long)(yd - 1 + i) * a.dst_pitch + xd;
            const float l = PANO_AT(gdst, ro - 1, nd, 613), c = PANO_AT(gdst, ro, nd, 613), r = PANO_AT(gdst, ro + 1, nd, 613);
            e[i] = fmaf(k1, r, fmaf(k6, c, k1 * l));
            o[i] = fmaf(k4, r, k4 * c);
        }
        v[0][0] = fmaf(k1, e[2], fmaf(k6, e[1], k1 * e[0]));
        v[0][1] = fmaf(k1, o[2], fmaf(k6, o[1], k1 * o[0]));
        v[1][0] = fmaf(k4, e[2], k4 * e[1]);
        v[1][1] = fmaf(k4, o[2], k4 * o[1]);
    } else {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int x = 2 * xd + (i & 1), y = 2 * yd + (i >> 1);
            v[i >> 1][i & 1] = x < w && y < h ? adjoint_pixel(gdst, h, w, a.dst_pitch, x, y) : 0.f;
        }
    }
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const int y = 2 * yd + i;
        if (y >= h) break;
        float* o = &PANO_AT(gsrc, (long long)y * a.src_pitch + 2 * xd, ns, 612);
        if (2 * xd + 1 < w && (((uintptr_t)o) & 7) == 0) {
            *reinterpret_cast<float2*>(o) = make_float2(v[i][0], v[i][1]);
        } else {
            o[0] = v[i][0];
            if (2 * xd + 1 < w) o[1] = v[i][1];
        }
    }
}

}  // namespace

PANO_BOUNDS_READER(bounds_read_refine)

cudaError_t launch_energy_grad(const EnergyArgs& a, cudaStream_t s) {
    cudaError_t e;
    const long long tiles = (long long)((a.w + 31) / 32) * ((a.h + kEgThreads / 32 - 1) / (kEgThreads / 32));
    if (tiles > INT_MAX) return cudaErrorInvalidValue;
    if (a.energy) {
        if ((e = cudaMemsetAsync(a.energy, 0, sizeof(double), s)) != cudaSuccess) return e;
        const int ctas = tiles < kEgCtas ? (int)tiles : kEgCtas;
        if ((e = launch_dependent(energy_kernel, dim3(ctas), dim3(kEgThreads), 0, s, 0, a)) != cudaSuccess) return e;
    }
    if (!a.grad_u && !a.grad_T && !a.grad_J) return cudaSuccess;
    if (a.grad_J && (e = cudaMemsetAsync(a.grad_J, 0, sizeof(float) * (size_t)a.h * a.w, s)) != cudaSuccess) return e;
    return launch_dependent(energy_grad_kernel, dim3((unsigned)tiles), dim3(kEgThreads), 0, s, 0, a);
}

cudaError_t launch_pyr_down_adjoint(const AdjointArgs& a, cudaStream_t s) {
    dim3 block(32, 8);
    dim3 grid(((a.w + 1) / 2 + 31) / 32, ((a.h + 1) / 2 + 7) / 8, a.count);
    return launch_dependent(pyr_down_adjoint_kernel, grid, block, 0, s, 0, a);
}

}  // namespace pano
