// Curved-ray march (Sec. 3.3.2-3.3.3 of arXiv 2603.02048), one thread per
// pixel ray: pinhole ray generation, slab entry into the volume box, the
// march of Eq. 15 with the Eq. 16 update (or RK4) and the Eq. 18 adaptive
// step, the exit clip at the box face, and what the straight exit ray sees
// (textured scene planes, else the bilinear equirect environment map).
//
// Precision (everything FP32, no FP64 on the device):
//  - The direction is carried as w = w_ref + d, with w_ref the primary ray
//    direction (fixed per ray) and d the small accumulated deflection. The
//    Eq. 16 normalisation is done in that form, d' = d1 + r (w_ref + d1) with
//    1 + r = |w_ref + d1|^-1 (a Taylor polynomial in e = |w_ref + d1|^2 - 1,
//    see renormalize), so rounding never touches the O(1) part of w and the
//    deflection keeps full relative precision over thousands of steps.
//  - The position is a compensated pair (hi + lo): hi carries a power-of-two
//    bias B (hi = position + B, B above every coordinate and step), so every
//    increment is smaller than hi and Fast2Sum is error-free; its rounding
//    error goes to lo. The position proper is (hi - B) + lo, where hi - B is
//    exact (Sterbenz); the volume is sampled, and the exit tested, at the
//    lattice coordinate (hi - (B - 1/2)) + lo = position + 1/2, rounded once.
//  - Divisions and square roots whose operands are far from any cancellation
//    (ds / n, n theta / (|g_perp| + eps), the renormalisation term, |g_perp|)
//    use the approximate hardware forms (relative error ~1e-7, harmless next
//    to the 1e-6 rad tolerance: they perturb steps, not the path).
//
// Layout: a block of 128 threads covers a 16x8 pixel tile; each warp an 8x4
// sub-tile, so the rays of a warp stay close in the volume and their eight
// corner fetches per step share cache lines in L1. The volume is stored with
// its slices interleaved in pairs (ZPAIR) and a one-voxel halo of edge copies:
// the order spreads the distinct voxels of a warp's corner load over the L1
// bank groups at a cost of few address instructions, and the halo lets a
// sample in the box skip every index clamp.
// A sample whose eight corners are all zero (its first corner marked in the
// volume's free-corner mask, built with the volume) is read as zero from one
// bit of that mask instead of eight voxel loads, and the Eq. 16 step then
// takes n = 1, g_perp = 0 and their step length without the arithmetic (a
// warp whose lanes all sample zero skips it); every step is still taken with
// the values the general branch would compute, so the results do not depend
// on the skip, nor on when the mask is asked: only after a sample with dn = 0,
// as a ray that reads the plume mostly keeps to it for many steps.
//
// What bounds it: instruction issue and the L1 data pipe, of which a dense
// volume takes most (a load costs a cycle per distinct 16-byte unit in the
// fullest of eight banks). 1080p view of the 256^3 FP32 plume at h_max: 66 % of
// the issue slots, 65 % of the pipe; eight 720p views of it on FP16: 80 and 71 %;
// 32 views of a 512^3 FP16 volume: 86 % of the pipe. RK4 with few rays is bound
// by the four serial samples a step, ~340 cycles each. Against 2x2x2 bricks,
// scalar state and IEEE approximations the step took these launches from 360 to
// 277, 1227 to 1035 us and 10.1 to 8.84 ms.
#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <map>
#include <mutex>
#include <string>
#include <type_traits>
#include <vector>

#include "hh_internal.h"
#include "texels.h"

namespace hh {
namespace {

constexpr float kPi = 3.14159265358979323846f;

// Resident 128-thread blocks per SM the single-view march kernels are compiled
// for. Eq. 16: 8, i.e. at most 64 registers a thread, at which FP32 storage spills
// up to 28 bytes (9 or 10 blocks measured the same or slower). RK4: 6 (80
// registers) on FP16; 5 (96, of which up to 8 bytes still spill) on FP32 storage,
// whose four samples a step spill more at 6 (256^3 720p view 2514 against 2446 us,
// 64^3 128x128 164 against 140; FP16 1080p view 964 against 1014 with 5).
constexpr int march_blocks(int storage, int stepper) {
    return stepper != HH_STEP_RK4 ? 8 : storage == HH_STORE_FP32 ? 5 : 6;
}
// Resident 256-thread blocks per SM of the persistent batched kernel. More
// warps hide more of the L2 latency, until the step spills much of its state. Tile
// at a time, FP16: 5 blocks (48 registers, 4 to 28 bytes spilled) against 4, 8
// views of the 256^3 volume 1085 against 1088 us (views in turn: 1148 against
// 1195), 32 views of the 512^3 one 9.34 against 9.77 ms. FP32, whose eight corners
// take twice the registers: 4 blocks (64) against 3 and 5, 8 views 1171 against
// 1239 and 1367 us. RK4 and the refill state need more registers.
constexpr int batch_blocks(int storage, int stepper, bool refill) {
    if (stepper == HH_STEP_RK4 || refill) return 3;
    return storage == HH_STORE_FP32 ? 4 : 5;
}

// Volume-side arguments of a launch (shared by every view).
struct VolArgs {
    const void* vol;
    const float* scales;
    const unsigned* sparse;  // whether the volume's free-corner mask is worth testing
    int nx, ny, nz;
    ZPairStrides strides;
    unsigned long long mask_off;  // bytes from a volume's data to its free-corner mask
    float bias;         // power of two above every coordinate and step
    float bias_u;       // bias - 1/2: (hi - bias_u) + lo is the lattice coordinate
    float ux, uy, uz;   // n + 1/2: the far faces in lattice coordinates
    float h_fixed, h_min, h_max, theta, eps;
    int max_steps;
    const uint8_t* bg;
    int bgW, bgH;
    float bg_u, bg_v;   // texels per radian: bgW / 2 pi, bgH / pi
    int n_planes;
    hh_plane planes[HH_MAX_PLANES];
};

// View-side arguments: the camera, the caller's output buffers and the
// view's place in a batch's tile list.
struct alignas(16) ViewArgs {
    float3 eye;
    float3 f, r, u;    // camera basis: forward, right, up (computed on the host in FP64)
    float a0, b0, s;   // pixel (x, y) -> a = a0 + (x + 1/2) s, b = b0 - (y + 1/2) s
    int W, H;
    float* rgb;
    uint8_t* rgb8;
    float* exit_pos;
    float* exit_dir;
    int32_t* steps;
    uint32_t* flags;
    int tiles_x;     // 8x4-pixel tiles per row
    int tile_begin;  // index of the view's first tile in the batch
};

struct Sample {
    float dn, gx, gy, gz;
};

__device__ __forceinline__ float3 operator+(float3 a, float3 b) {
    return make_float3(a.x + b.x, a.y + b.y, a.z + b.z);
}
__device__ __forceinline__ float3 operator-(float3 a, float3 b) {
    return make_float3(a.x - b.x, a.y - b.y, a.z - b.z);
}
__device__ __forceinline__ float3 operator*(float s, float3 a) {
    return make_float3(s * a.x, s * a.y, s * a.z);
}
// Sums of products are written with explicit FMAs: a plain a * b + c * d lets
// the compiler fuse either product, and which one it fuses follows the
// surrounding code, so results would change with unrelated edits.
__device__ __forceinline__ float dot(float3 a, float3 b) {
    return fmaf(a.z, b.z, fmaf(a.y, b.y, a.x * b.x));
}
__device__ __forceinline__ float3 cross(float3 a, float3 b) {
    return make_float3(fmaf(a.y, b.z, -(a.z * b.y)), fmaf(a.z, b.x, -(a.x * b.z)),
                       fmaf(a.x, b.y, -(a.y * b.x)));
}
__device__ __forceinline__ float3 normalized(float3 v) {
    const float len = sqrtf(dot(v, v));
    return make_float3(v.x / len, v.y / len, v.z / len);
}
// a + s * b, component-wise with FMA
__device__ __forceinline__ float3 fma3(float s, float3 b, float3 a) {
    return make_float3(fmaf(s, b.x, a.x), fmaf(s, b.y, a.y), fmaf(s, b.z, a.z));
}
__device__ __forceinline__ float lerpf(float a, float b, float t) { return fmaf(t, b - a, a); }

// Error-free sum for |a| >= |b| (Dekker's Fast2Sum): s + e == a + b exactly.
__device__ __forceinline__ void fast_two_sum(float a, float b, float& s, float& e) {
    s = __fadd_rn(a, b);
    e = __fsub_rn(b, __fsub_rn(s, a));
}

// Packed FP32x2 (PTX fma.rn.f32x2 / sub.rn.f32x2): two FP32 lanes per
// instruction, each rounded like its scalar counterpart.
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
    float2 r;
    asm("{\n\t.reg .b64 pa, pb, pc, pd;\n\t"
        "mov.b64 pa, {%2, %3};\n\tmov.b64 pb, {%4, %5};\n\tmov.b64 pc, {%6, %7};\n\t"
        "fma.rn.f32x2 pd, pa, pb, pc;\n\tmov.b64 {%0, %1}, pd;\n\t}"
        : "=f"(r.x), "=f"(r.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
    return r;
}
__device__ __forceinline__ float2 sub2(float2 a, float2 b) {
    float2 r;
    asm("{\n\t.reg .b64 pa, pb, pd;\n\t"
        "mov.b64 pa, {%2, %3};\n\tmov.b64 pb, {%4, %5};\n\t"
        "sub.rn.f32x2 pd, pa, pb;\n\tmov.b64 {%0, %1}, pd;\n\t}"
        : "=f"(r.x), "=f"(r.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return r;
}
__device__ __forceinline__ float2 add2(float2 a, float2 b) {
    float2 r;
    asm("{\n\t.reg .b64 pa, pb, pd;\n\t"
        "mov.b64 pa, {%2, %3};\n\tmov.b64 pb, {%4, %5};\n\t"
        "add.rn.f32x2 pd, pa, pb;\n\tmov.b64 {%0, %1}, pd;\n\t}"
        : "=f"(r.x), "=f"(r.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return r;
}
__device__ __forceinline__ float2 mul2(float2 a, float2 b) {
    float2 r;
    asm("{\n\t.reg .b64 pa, pb, pd;\n\t"
        "mov.b64 pa, {%2, %3};\n\tmov.b64 pb, {%4, %5};\n\t"
        "mul.rn.f32x2 pd, pa, pb;\n\tmov.b64 {%0, %1}, pd;\n\t}"
        : "=f"(r.x), "=f"(r.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return r;
}
__device__ __forceinline__ float2 dup(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 xy(float3 a) { return make_float2(a.x, a.y); }
__device__ __forceinline__ float3 with_z(float2 a, float z) { return make_float3(a.x, a.y, z); }
// The march's vectors as a packed x, y pair and a scalar z, each component
// rounded as by the scalar operators above: two instructions for three, in a
// step that the issue rate bounds (march of the 256^3 1080p frame at h_max: 320
// against 308 us).
__device__ __forceinline__ float3 add_p(float3 a, float3 b) {
    return with_z(add2(xy(a), xy(b)), __fadd_rn(a.z, b.z));
}
__device__ __forceinline__ float3 mul_p(float s, float3 a) {
    return with_z(mul2(dup(s), xy(a)), __fmul_rn(s, a.z));
}
__device__ __forceinline__ float3 fma_p(float s, float3 b, float3 a) {
    return with_z(fma2(dup(s), xy(b), xy(a)), fmaf(s, b.z, a.z));
}
// a + t (b - a) on both halves of a float4 (t duplicated in tt).
__device__ __forceinline__ float4 lerp4x2(float4 a, float4 b, float2 tt) {
    const float2 lo = fma2(tt, sub2(make_float2(b.x, b.y), make_float2(a.x, a.y)),
                           make_float2(a.x, a.y));
    const float2 hi = fma2(tt, sub2(make_float2(b.z, b.w), make_float2(a.z, a.w)),
                           make_float2(a.z, a.w));
    return make_float4(lo.x, lo.y, hi.x, hi.y);
}

// The step length of a kernel: a fixed one, Eq. 18's with the approximations
// below that take subnormals for zero, or (LEN_SUBNORMAL, either of them) with
// ones that do not. step_len() picks for a launch.
enum { LEN_FIXED = 0, LEN_EQ18 = 1, LEN_SUBNORMAL = 2 };

// Hardware approximate square root and division (PTX *.approx[.ftz].f32, ~1 ulp):
// without .ftz each carries instructions for subnormal operands (march of the
// 1080p frame: 330 against 320 us).
template <int LEN>
__device__ __forceinline__ float sqrt_approx(float x) {
    float r;
    if (LEN == LEN_SUBNORMAL)
        asm("sqrt.approx.f32 %0, %1;" : "=f"(r) : "f"(x));
    else
        asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
template <int LEN>
__device__ __forceinline__ float div_approx(float a, float b) {
    float r;
    if (LEN == LEN_SUBNORMAL)
        asm("div.approx.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
    else
        asm("div.approx.ftz.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
    return r;
}

// What .ftz drops does not show where a subnormal |g_perp|^2, |g_perp| below
// 1.1e-19, is at most 2^-24 of eps, and the tolerance and the steps themselves are
// far from subnormal (n, near 1, takes them no further). Other parameters, which
// no scene in use has, march with LEN_SUBNORMAL.
int step_len(const hh_step_params& P) {
    const float least = 0x1p-100f;
    if (!P.adaptive) return P.h_fixed < least ? LEN_SUBNORMAL : LEN_FIXED;
    const bool tiny = P.eps < 0x1p-39f || P.h_min < least ||
                      (P.theta_max > 0.0f && P.theta_max < least);
    return tiny ? LEN_SUBNORMAL : LEN_EQ18;
}

// Lattice cell and weight along one axis from the lattice coordinate u =
// position + 1/2, the halo coordinate of the ZPAIR layout (the centre of
// grid voxel i at u = i + 1; the march carries u, not the position):
// i0 = floor(u), f = u - i0 (both from u itself: an index taken from the rounded
// value would wait for it; march of the 256^3 frame 309 against 305 us). A
// position in [0, n] has u in [0.5, n + 0.5], so both corners i0, i0 + 1 lie in
// the padded axis [0, n + 1], and the halo copies make this the sample with the
// lattice coordinate clamped to the voxel centres. The Euler march samples only
// accepted points, which lie in the box (a NaN gives i0 = 0); CLAMP first clamps u
// to [0.5, n + 0.5] (NaN to 0.5) for RK4 stage points, which may lie outside.
template <bool CLAMP>
__device__ __forceinline__ void axis_cell(float u, int n, int& i0, float& f) {
    if (CLAMP) u = fminf(fmaxf(u, 0.5f), static_cast<float>(n) + 0.5f);
    i0 = __float2int_rd(u);
    f = u - floorf(u);
}

// x-lerp of two FP16 corners read raw (four halves each), in FP32: the first
// corner converted, the second converted inside the subtraction
// (sub.rn.f32.f16: one rounding, as converting first and subtracting in FP32),
// then a + t (b - a) on both channel pairs.
__device__ __forceinline__ float4 xlerp_fp16(uint2 a, uint2 b, float2 tt) {
    const float2 a0 = __half22float2(*reinterpret_cast<const __half2*>(&a.x));
    const float2 a1 = __half22float2(*reinterpret_cast<const __half2*>(&a.y));
    float2 d0, d1;
    asm("{\n\t.reg .b16 l, h;\n\tmov.b32 {l, h}, %2;\n\t"
        "sub.rn.f32.f16 %0, l, %3;\n\tsub.rn.f32.f16 %1, h, %4;\n\t}"
        : "=f"(d0.x), "=f"(d0.y)
        : "r"(b.x), "f"(a0.x), "f"(a0.y));
    asm("{\n\t.reg .b16 l, h;\n\tmov.b32 {l, h}, %2;\n\t"
        "sub.rn.f32.f16 %0, l, %3;\n\tsub.rn.f32.f16 %1, h, %4;\n\t}"
        : "=f"(d1.x), "=f"(d1.y)
        : "r"(b.y), "f"(a1.x), "f"(a1.y));
    const float2 lo = fma2(tt, d0, a0), hi = fma2(tt, d1, a1);
    return make_float4(lo.x, lo.y, hi.x, hi.y);
}

// Trilinear sample of {dn, g} at lattice coordinate u = position + 1/2
// (Sec. 3.3.1: n and grad n sampled with trilinear interpolation); FP16
// volumes are interpolated as stored (code units, value / scale).
// With HH_DEBUG_BOUNDS the corner indices are checked against the padded
// axes (ix in [0, nx], so that ix + 1 <= nx + 1): a corner outside is counted
// in g_bounds_violations, flagged on the ray (HH_FLAG_CLAMP in `flags`) and
// clamped before the load. The release build has no check and no clamp.
#ifdef HH_DEBUG_BOUNDS
__device__ unsigned long long g_bounds_violations;
#endif

// The volume a kernel samples: with ADDR_BASE (zpair.h) the one at V.vol, else the
// one at the pointer passed.

// Returns false, leaving s unset, for a sample whose eight corners are all
// zero (the zero sample), read off the free-corner mask if `ask`. MASK = false
// (volumes not worth testing) never asks: the general arithmetic on eight zeros
// gives the zero sample's values.
template <int STORAGE, int ADDR, bool MASK, bool CLAMP>
__device__ __forceinline__ bool fetch_nonzero(const VolArgs& A, const void* __restrict__ vol,
                                              float3 u, bool ask, uint32_t& flags, Sample& s) {
    int ix, iy, iz;
    float fx, fy, fz;
    axis_cell<CLAMP>(u.x, A.nx, ix, fx);
    axis_cell<CLAMP>(u.y, A.ny, iy, fy);
    axis_cell<CLAMP>(u.z, A.nz, iz, fz);
#ifdef HH_DEBUG_BOUNDS
    if (ix < 0 || ix > A.nx || iy < 0 || iy > A.ny || iz < 0 || iz > A.nz) {
        atomicAdd(&g_bounds_violations, 1ull);
        flags |= HH_FLAG_CLAMP;
        ix = min(max(ix, 0), A.nx);
        iy = min(max(iy, 0), A.ny);
        iz = min(max(iz, 0), A.nz);
        fx = fminf(fmaxf(fx, 0.0f), 1.0f);
        fy = fminf(fmaxf(fy, 0.0f), 1.0f);
        fz = fminf(fmaxf(fz, 0.0f), 1.0f);
    }
#else
    (void)flags;
#endif
    const unsigned odd = static_cast<unsigned>(iz) & 1u;
    const unsigned b = zpair_element(A.strides, ix, iy, iz, odd);
    // the zero sample's bit: b & 31 of word b >> 5 (the funnel shift takes the
    // shift count mod 32)
    const char* base = static_cast<const char*>(ADDR == ADDR_BASE ? A.vol : vol);
    if (MASK && ask) {
        const unsigned w = __ldg(reinterpret_cast<const unsigned*>(base + A.mask_off) + (b >> 5));
        if (__funnelshift_r(w, w, b) & 1u) return false;
    }
    using V = typename std::conditional<STORAGE == HH_STORE_FP32, float4, uint2>::type;
    const V *c00, *c10, *c01, *c11;  // corners (ix, iy + 0 or 1, iz + 0 or 1)
    zpair_corners<ADDR>(A.strides, base, b, odd, c00, c10, c01, c11);
    float4 c;
    if constexpr (STORAGE == HH_STORE_FP16_SCALED) {
        // lerps along x (the second corner converted inside the subtraction),
        // then y, then z with packed FP32x2 arithmetic, two channels per
        // instruction (measured 8 % faster there; on FP32 storage the 8-weight
        // form below is faster)
        const uint2 r000 = __ldg(c00), r100 = __ldg(c00 + 2);
        const uint2 r010 = __ldg(c10), r110 = __ldg(c10 + 2);
        const uint2 r001 = __ldg(c01), r101 = __ldg(c01 + 2);
        const uint2 r011 = __ldg(c11), r111 = __ldg(c11 + 2);
        const float2 tx = dup(fx), ty = dup(fy), tz = dup(fz);
        c = lerp4x2(lerp4x2(xlerp_fp16(r000, r100, tx), xlerp_fp16(r010, r110, tx), ty),
                    lerp4x2(xlerp_fp16(r001, r101, tx), xlerp_fp16(r011, r111, tx), ty), tz);
    } else {
        // the standard 8-corner weights (formed two at a time; the sum over
        // corners packed two channels at a time was slower, 317 against 308 us)
        const float4 v000 = __ldg(c00), v100 = __ldg(c00 + 2);
        const float4 v010 = __ldg(c10), v110 = __ldg(c10 + 2);
        const float4 v001 = __ldg(c01), v101 = __ldg(c01 + 2);
        const float4 v011 = __ldg(c11), v111 = __ldg(c11 + 2);
        const float gx = 1.0f - fx, gy = 1.0f - fy, gz = 1.0f - fz;
        const float2 y0 = make_float2(gy, fy), yz0 = mul2(y0, dup(gz)), yz1 = mul2(y0, dup(fz));
        const float2 w00 = mul2(dup(gx), yz0), w10 = mul2(dup(fx), yz0);  // [x][z], over y
        const float2 w01 = mul2(dup(gx), yz1), w11 = mul2(dup(fx), yz1);
        c.x = w00.x * v000.x;
        c.y = w00.x * v000.y;
        c.z = w00.x * v000.z;
        c.w = w00.x * v000.w;
        auto add = [&c](float w, const float4& v) {
            c.x = fmaf(w, v.x, c.x);
            c.y = fmaf(w, v.y, c.y);
            c.z = fmaf(w, v.z, c.z);
            c.w = fmaf(w, v.w, c.w);
        };
        add(w10.x, v100);
        add(w00.y, v010);
        add(w10.y, v110);
        add(w01.x, v001);
        add(w11.x, v101);
        add(w01.y, v011);
        add(w11.y, v111);
    }
    // FP16 storage: the sample stays in code units (value / scale); the
    // power-of-two scales are applied downstream, where a product by them is
    // exact, so the result equals scaling here (see perp_of)
    s.dn = c.x;
    s.gx = c.y;
    s.gy = c.z;
    s.gz = c.w;
    return true;
}

template <int STORAGE, int ADDR, bool MASK, bool CLAMP>
__device__ __forceinline__ Sample fetch(const VolArgs& A, const void* __restrict__ vol, float3 u,
                                        uint32_t& flags) {
    Sample s;
    if (!fetch_nonzero<STORAGE, ADDR, MASK, CLAMP>(A, vol, u, true, flags, s))
        s.dn = s.gx = s.gy = s.gz = 0.0f;
    return s;
}

// Eq. 18 (second form) or the fixed step (LEN_SUBNORMAL's is Eq. 18's with h_min =
// h_max).
template <int LEN>
__device__ __forceinline__ float step_length(const VolArgs& A, float n, float gperp_norm) {
    if (LEN == LEN_FIXED) return A.h_fixed;
    return fminf(fmaxf(div_approx<LEN>(n * A.theta, gperp_norm + A.eps), A.h_min), A.h_max);
}

// Eq. 16's normalize, in deflection form: returns d' with w_ref + d' the unit
// vector along w1 = w_ref + d1: w_ref + d' = (1 + r) w1 with
// 1 + r = (1 + e)^(-1/2), e = |w1|^2 - 1, r by its Taylor polynomial
// -e/2 + 3e^2/8 - 5e^3/16 (error 35 e^4 / 128). e is the squared turn of one
// step plus the previous rounding (below 1e-5 when Eq. 18 bounds the turn by
// theta_max <= 3e-3; an e below FP32 resolution rounds to 0 and leaves w1 as
// it is, as FP32 normalisation would); r only scales w1, never turns it, and
// its error is undone at the next step. Only d is carried, so the rounding of
// the update never touches the O(1) part w_ref.
__device__ __forceinline__ float renorm_term(float3 w1) {
    const float e = fmaf(w1.x, w1.x, fmaf(w1.y, w1.y, fmaf(w1.z, w1.z, -1.0f)));
    return e * fmaf(e, fmaf(-0.3125f, e, 0.375f), -0.5f);
}
__device__ __forceinline__ float3 renormalize(float3 w1, float3 d1) {
    return fma3(renorm_term(w1), w1, d1);
}

struct LoadTexels {
    __device__ __forceinline__ uint32_t operator()(const uint8_t* p) const { return __ldg(p); }
    __device__ __forceinline__ uint32_t operator()(const uint16_t* p) const { return __ldg(p); }
};

// Channels of a pair of texels read as lo, hi.
__device__ __forceinline__ void texel_channels(uint32_t lo, uint32_t hi, float2& r, float2& g,
                                               float2& b) {
    r = make_float2(static_cast<float>(lo & 0xFFu), static_cast<float>(lo >> 24));
    g = make_float2(static_cast<float>((lo >> 8) & 0xFFu), static_cast<float>(hi & 0xFFu));
    b = make_float2(static_cast<float>((lo >> 16) & 0xFFu), static_cast<float>((hi >> 8) & 0xFFu));
}

// Bilinear colour between texels (i0, j0) and (i0 + 1, j0 + 1); value / 255.
__device__ __forceinline__ float3 texel_lerp(const uint8_t* __restrict__ tex, int W, int i0, int j0,
                                             float fs, float ft) {
    uint32_t lo0, hi0, lo1, hi1;
    texel_square(tex, W, i0, j0, LoadTexels(), lo0, hi0, lo1, hi1);
    float2 r0, g0, b0, r1, g1, b1;
    texel_channels(lo0, hi0, r0, g0, b0);
    texel_channels(lo1, hi1, r1, g1, b1);
    constexpr float k = 1.0f / 255.0f;
    return make_float3(lerpf(lerpf(r0.x, r0.y, fs), lerpf(r1.x, r1.y, fs), ft) * k,
                       lerpf(lerpf(g0.x, g0.y, fs), lerpf(g1.x, g1.y, fs), ft) * k,
                       lerpf(lerpf(b0.x, b0.y, fs), lerpf(b1.x, b1.y, fs), ft) * k);
}

// Colour of direction d in the equirect environment map (bilinear, u wraps,
// v clamps; value / 255).
__device__ __forceinline__ float3 environment(const VolArgs& A, float3 d) {
    const float phi = atan2f(d.y, d.x);
    const float theta = atan2f(sqrtf(fmaf(d.y, d.y, d.x * d.x)), d.z);
    const float W = static_cast<float>(A.bgW), H = static_cast<float>(A.bgH);
    const float u = fmaf(phi, A.bg_u, 0.5f * W - 0.5f);
    float v = fmaf(theta, A.bg_v, -0.5f);
    const float ufl = floorf(u);
    const float fu = u - ufl;
    // |phi| is at most pi (to a rounding): u lies within a texel of [0, W)
    int i0 = static_cast<int>(ufl);
    if (i0 < 0) i0 += A.bgW;
    if (i0 >= A.bgW) i0 -= A.bgW;
    v = fminf(fmaxf(v, 0.0f), H - 1.0f);
    const int j0 = min(static_cast<int>(floorf(v)), A.bgH - 2);
    const float fv = v - static_cast<float>(j0);
    if (i0 + 1 < A.bgW) return texel_lerp(A.bg, A.bgW, i0, j0, fu, fv);
    // the pair that wraps: the last texel of a row and its first
    const uint8_t* r0 = A.bg + static_cast<size_t>(j0) * A.bgW * 3;
    const uint8_t* r1 = r0 + static_cast<size_t>(A.bgW) * 3;
    float out[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const float t00 = __ldg(r0 + i0 * 3 + c), t01 = __ldg(r0 + c);
        const float t10 = __ldg(r1 + i0 * 3 + c), t11 = __ldg(r1 + c);
        out[c] = lerpf(lerpf(t00, t01, fu), lerpf(t10, t11, fu), fv) * (1.0f / 255.0f);
    }
    return make_float3(out[0], out[1], out[2]);
}

__device__ __forceinline__ float3 f3(const float v[3]) { return make_float3(v[0], v[1], v[2]); }

// Bilinear RGB8 texture lookup at texel coordinates (s, t), clamped to the
// texel centres; value / 255.
__device__ __forceinline__ float3 texel_bilinear(const uint8_t* tex, int W, int H, float s,
                                                 float t) {
    s = fminf(fmaxf(s, 0.0f), static_cast<float>(W - 1));
    t = fminf(fmaxf(t, 0.0f), static_cast<float>(H - 1));
    const int i0 = min(static_cast<int>(floorf(s)), W - 2);
    const int j0 = min(static_cast<int>(floorf(t)), H - 2);
    const float fs = s - static_cast<float>(i0), ft = t - static_cast<float>(j0);
    return texel_lerp(tex, W, i0, j0, fs, ft);
}

// What the straight ray P + t d (t > 0) sees: the nearest textured plane it
// hits, else the environment map.
// A call, not inlined: it runs once per ray, and keeping its registers out of
// the step loop's allocation is as fast as inlining it (measured).
__device__ __noinline__ float3 scene_color(const VolArgs& A, float3 P, float3 d) {
    float best_t = INFINITY, best_a = 0.0f, best_b = 0.0f;
    int best = -1;
#pragma unroll
    for (int k = 0; k < HH_MAX_PLANES; ++k) {
        if (k >= A.n_planes) break;
        const hh_plane& pl = A.planes[k];
        const float3 o = f3(pl.origin), u = f3(pl.u), v = f3(pl.v);
        const float3 nrm = cross(u, v);
        const float den = dot(d, nrm);
        if (den == 0.0f) continue;
        const float t = dot(o - P, nrm) / den;
        if (!(t > 0.0f) || !(t < best_t)) continue;
        const float3 r = fma3(t, d, P) - o;
        const float a = dot(r, u) / dot(u, u), b = dot(r, v) / dot(v, v);
        if (a >= 0.0f && a <= 1.0f && b >= 0.0f && b <= 1.0f) {
            best = k;
            best_t = t;
            best_a = a;
            best_b = b;
        }
    }
    if (best < 0) return environment(A, d);
    const uint8_t* tex = A.planes[0].rgb8_dev;
    int W = A.planes[0].width, H = A.planes[0].height;
#pragma unroll
    for (int k = 1; k < HH_MAX_PLANES; ++k)
        if (best == k) {
            tex = A.planes[k].rgb8_dev;
            W = A.planes[k].width;
            H = A.planes[k].height;
        }
    return texel_bilinear(tex, W, H, best_a * static_cast<float>(W) - 0.5f,
                          best_b * static_cast<float>(H) - 0.5f);
}

// Ray through the centre of pixel (px, py); row 0 at the top:
// normalize(f + a r + b u) with a = (2 (x + 1/2) / W - 1) t W / H and
// b = (1 - 2 (y + 1/2) / H) t, t = tan(vfov / 2), i.e. a = a0 + (x + 1/2) s,
// b = b0 - (y + 1/2) s with s = 2 t / H, a0 = -t W / H, b0 = t.
__device__ __forceinline__ float3 primary_ray(const ViewArgs& A, int px, int py) {
    const float a = fmaf(static_cast<float>(px) + 0.5f, A.s, A.a0);
    const float b = fmaf(static_cast<float>(py) + 0.5f, -A.s, A.b0);
    return normalized(fma3(b, A.u, fma3(a, A.r, A.f)));
}

// Slab test of o + t d against [0,nx]x[0,ny]x[0,nz]; hit iff
// t_out >= max(t_in, 0). An axis with d = 0 misses when o is outside it.
__device__ __forceinline__ bool slab(const VolArgs& A, float3 o, float3 d, float& t_in) {
    float tin = -INFINITY, tout = INFINITY;
    const float oo[3] = {o.x, o.y, o.z}, dd[3] = {d.x, d.y, d.z};
    const float bx[3] = {static_cast<float>(A.nx), static_cast<float>(A.ny),
                         static_cast<float>(A.nz)};
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        if (dd[a] == 0.0f) {
            if (oo[a] < 0.0f || oo[a] > bx[a]) return false;
            continue;
        }
        const float t1 = (0.0f - oo[a]) / dd[a];
        const float t2 = (bx[a] - oo[a]) / dd[a];
        tin = fmaxf(tin, fminf(t1, t2));
        tout = fminf(tout, fmaxf(t1, t2));
    }
    t_in = tin;
    return tout >= fmaxf(tin, 0.0f);
}

// Whether lattice coordinate u = position + 1/2 lies outside the box
// (position outside [0, n] on some axis).
__device__ __forceinline__ bool outside(const VolArgs& A, float3 u) {
    return u.x < 0.5f || u.y < 0.5f || u.z < 0.5f || u.x > A.ux || u.y > A.uy || u.z > A.uz;
}

// Fraction tau in [0, 1] of the increment `inc` from (hi + lo) at which the
// segment leaves the box (the slab exit along the segment).
__device__ __forceinline__ float exit_fraction(const VolArgs& A, float3 hi, float3 lo,
                                               float3 inc) {
    const float h3[3] = {hi.x, hi.y, hi.z}, l3[3] = {lo.x, lo.y, lo.z};
    const float i3[3] = {inc.x, inc.y, inc.z};
    const float bx[3] = {static_cast<float>(A.nx), static_cast<float>(A.ny),
                         static_cast<float>(A.nz)};
    float tau = 1.0f;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        if (i3[a] > 0.0f) tau = fminf(tau, ((bx[a] - h3[a]) - l3[a]) / i3[a]);
        else if (i3[a] < 0.0f) tau = fminf(tau, ((0.0f - h3[a]) - l3[a]) / i3[a]);
    }
    return fmaxf(tau, 0.0f);
}

// n and the transverse gradient g_perp = (I - w w^T) g at u (Eq. 15), with
// |g_perp|. With FP16 storage g_perp is returned in code units, g_perp / s_g:
// the caller multiplies the scalar that scales it by s_g (gsc in ray_step). s_n
// and s_g are powers of two, so every such product is exact and the results
// equal those of scaling the sample first: n = 1 + dn s_n is one rounding
// either way, and |g_perp| = s_g |g_perp / s_g| exactly.
template <int STORAGE, int LEN>
__device__ __forceinline__ float3 perp_of(const Sample& s, float3 w, float s_n, float s_g,
                                          float& n, float& gperp_norm) {
    n = STORAGE == HH_STORE_FP32 ? 1.0f + s.dn : fmaf(s.dn, s_n, 1.0f);
    const float3 g = make_float3(s.gx, s.gy, s.gz);
    const float3 gp = fma_p(-dot(w, g), w, g);
    gperp_norm = sqrt_approx<LEN>(dot(gp, gp));
    if (STORAGE != HH_STORE_FP32) gperp_norm *= s_g;
    return gp;
}
template <int STORAGE, int LEN, int ADDR, bool MASK, bool CLAMP>
__device__ __forceinline__ float3 perp_rate(const VolArgs& A, const void* __restrict__ vol,
                                            float3 u, float3 w, float s_n, float s_g, float& n,
                                            float& gperp_norm, uint32_t& flags) {
    return perp_of<STORAGE, LEN>(fetch<STORAGE, ADDR, MASK, CLAMP>(A, vol, u, flags), w, s_n, s_g,
                                 n, gperp_norm);
}

// Per-ray state of the march: primary direction w_ref, deflection d, biased
// compensated position (hi, lo) (position = (hi - B) + lo), its lattice
// coordinate rounded once, c = (hi - (B - 1/2)) + lo = position + 1/2 (where
// the volume is sampled and the exit is tested), steps taken and flags.
struct RayState {
    float3 wr, hi, lo, d, c;
    int k;
    uint32_t flags;
    float sn, sg;  // the volume's FP16 scales, read once per ray
    float ds0;     // the step length at a zero sample (n = 1, |g_perp| = 0)
    float last;    // Eq. 16: dn of the last sample
};

// Pixel (x, y) of slot p (0..31) of a tile_w x (32 / tile_w) warp tile. Each
// 8-lane quarter of the warp covers a 4x2 pixel block, not a row of 8: a
// 128-bit load is served a quarter-warp at a time, and the voxels of a 4x2
// block of neighbouring rays form a 2x2 patch across the view, which falls on
// four different L1 bank groups, where a row of 8 rays would walk a line of
// voxels that alternates between two.
__device__ __forceinline__ void tile_pixel(int p, int tile_w_log2, int& x, int& y) {
    const int q = p >> 3;
    const int qx_log2 = tile_w_log2 - 2;  // quarters per tile row: 1, 2 or 4
    x = ((q & ((1 << qx_log2) - 1)) << 2) | (p & 3);
    y = ((q >> qx_log2) << 1) | ((p >> 2) & 1);
}

// Ray generation and slab entry (flags = HIT when the ray enters the box).
template <int LEN>
__device__ __forceinline__ void ray_begin(const VolArgs& V, const float* __restrict__ scales,
                                          const ViewArgs& C, int px, int py, RayState& R) {
    R.wr = primary_ray(C, px, py);
    R.sn = __ldg(scales);
    R.sg = __ldg(scales + 1);
    R.ds0 = step_length<LEN>(V, 1.0f, 0.0f);
    R.last = 0.0f;
    R.k = 0;
    R.flags = 0;
    R.d = make_float3(0.0f, 0.0f, 0.0f);
    R.hi = R.lo = R.d;
    float t_in;
    if (slab(V, C.eye, R.wr, t_in)) {
        R.flags = HH_FLAG_HIT;
        // position = (hi - B) + lo with hi = position + B (see the header)
        // entry point, clamped into the box (rounding may put it just outside; the
        // march samples only positions in the box)
        float3 entry = fma3(fmaxf(t_in, 0.0f), R.wr, C.eye);
        entry.x = fminf(fmaxf(entry.x, 0.0f), static_cast<float>(V.nx));
        entry.y = fminf(fmaxf(entry.y, 0.0f), static_cast<float>(V.ny));
        entry.z = fminf(fmaxf(entry.z, 0.0f), static_cast<float>(V.nz));
        fast_two_sum(V.bias, entry.x, R.hi.x, R.lo.x);
        fast_two_sum(V.bias, entry.y, R.hi.y, R.lo.y);
        fast_two_sum(V.bias, entry.z, R.hi.z, R.lo.z);
    }
    R.c = make_float3((R.hi.x - V.bias_u) + R.lo.x, (R.hi.y - V.bias_u) + R.lo.y,
                      (R.hi.z - V.bias_u) + R.lo.z);
}

// One step of Eq. 16 (or RK4) with the Eq. 18 (or fixed) step length.
// Returns true when the step leaves the box: then R.hi and R.d, of no further
// use to the march, hold the exit point on the face and the new direction (six
// registers that the loop need not carry).
template <int STORAGE, int STEPPER, int LEN, int ADDR, bool MASK>
__device__ __forceinline__ bool ray_step(const VolArgs& V, const void* __restrict__ vol,
                                         RayState& R) {
    const float B = V.bias;
    const float3 wr = R.wr, d = R.d;
    const float3 C = R.c;
    float ds;
    float3 dnew, inc;
    const float gsc = STORAGE == HH_STORE_FP32 ? 1.0f : R.sg;  // see perp_rate
    if (STEPPER == HH_STEP_RK4) {
        float n1, gpn, n2, n3, n4, unused;
        const float3 w1 = wr + d;
        const float3 gp1 = perp_rate<STORAGE, LEN, ADDR, MASK, true>(V, vol, C, w1, R.sn, R.sg, n1,
                                                                     gpn, R.flags);
        ds = step_length<LEN>(V, n1, gpn);
        const float hds = 0.5f * ds;
        const float3 k1 = (div_approx<LEN>(1.0f, n1) * gsc) * gp1;
        const float3 d2 = fma3(hds, k1, d);
        const float3 w2 = wr + d2;
        const float3 gp2 = perp_rate<STORAGE, LEN, ADDR, MASK, true>(
            V, vol, fma3(hds, w1, C), w2, R.sn, R.sg, n2, unused, R.flags);
        const float3 k2 = (div_approx<LEN>(1.0f, n2) * gsc) * gp2;
        const float3 d3 = fma3(hds, k2, d);
        const float3 w3 = wr + d3;
        const float3 gp3 = perp_rate<STORAGE, LEN, ADDR, MASK, true>(
            V, vol, fma3(hds, w2, C), w3, R.sn, R.sg, n3, unused, R.flags);
        const float3 k3 = (div_approx<LEN>(1.0f, n3) * gsc) * gp3;
        const float3 d4 = fma3(ds, k3, d);
        const float3 w4 = wr + d4;
        const float3 gp4 = perp_rate<STORAGE, LEN, ADDR, MASK, true>(
            V, vol, fma3(ds, w3, C), w4, R.sn, R.sg, n4, unused, R.flags);
        const float3 k4 = (div_approx<LEN>(1.0f, n4) * gsc) * gp4;
        // k1 + 2 (k2 + k3) + k4 (every k is a product: the adds are kept
        // unfused, __fadd_rn, so no product is folded into them)
        const float3 ksum =
            make_float3(__fadd_rn(fmaf(2.0f, __fadd_rn(k2.x, k3.x), k1.x), k4.x),
                        __fadd_rn(fmaf(2.0f, __fadd_rn(k2.y, k3.y), k1.y), k4.y),
                        __fadd_rn(fmaf(2.0f, __fadd_rn(k2.z, k3.z), k1.z), k4.z));
        const float3 dsum = fma3(ds * (1.0f / 6.0f), ksum, d);
        dnew = renormalize(wr + dsum, dsum);
        const float3 dpos = (1.0f / 6.0f) * (d + 2.0f * (d2 + d3) + d4);
        inc = ds * (wr + dpos);
    } else {
        Sample smp;
        float3 d1;
        // The mask is asked after a sample with dn = 0 only, which spares the
        // nonzero steps its load and latency; a first zero sample behind nonzero
        // ones is read and computed like any other. 128^3 view of 320x240 43.0
        // against 38.8 us, 256^3 1080p 280.5 against 277.4, eight 720p views of it on
        // FP16 1032 against 1035 (at theta_max 3e-5 1183 against 1149, at 1e-5 2280
        // against 1962), 32 views of a 512^3 volume 9.12 against 8.84 ms. RK4, whose
        // stages step half as far, asks always (256^3 901 against 932 us with the
        // later stages asking after a zero first one).
        if (fetch_nonzero<STORAGE, ADDR, MASK, false>(V, vol, C, R.last == 0.0f, R.flags, smp)) {
            if (MASK) R.last = smp.dn;
            float n, gpn;
            const float3 gp = perp_of<STORAGE, LEN>(smp, add_p(wr, d), R.sn, R.sg, n, gpn);
            ds = step_length<LEN>(V, n, gpn);
            d1 = fma_p(div_approx<LEN>(ds, n) * gsc, gp, d);
        } else {
            // the zero sample: n = 1 and g_perp = 0 exactly, so the branch
            // above would give the step length ds0 (the same operations on
            // the same operands) and d1 = d + 0 = d (d is never -0: it starts
            // at +0 and a sum that rounds to zero is +0); a warp whose lanes
            // all sample zero skips the g_perp and Eq. 18 arithmetic
            ds = R.ds0;
            d1 = d;
        }
        // Eq. 16: w' = normalize(w1), C' = C + ds w'; with w' = (1 + r) w1
        // the increment is ds (1 + r) w1 (w' itself is formed only at the exit)
        const float3 w1 = add_p(wr, d1);
        const float rm1 = renorm_term(w1);
        dnew = fma_p(rm1, w1, d1);
        inc = mul_p(fmaf(ds, rm1, ds), w1);
    }
    // Fast2Sum of hi and the increment, x and y packed
    const float2 nhi2 = add2(xy(R.hi), xy(inc));
    const float2 err2 = sub2(xy(inc), sub2(nhi2, xy(R.hi)));
    float nhi_z, err_z;
    fast_two_sum(R.hi.z, inc.z, nhi_z, err_z);
    const float3 nhi = with_z(nhi2, nhi_z);
    const float3 nlo = add_p(R.lo, with_z(err2, err_z));
    const float Bu = V.bias_u;
    const float3 P = add_p(with_z(sub2(nhi2, dup(Bu)), __fsub_rn(nhi_z, Bu)), nlo);
    ++R.k;
    const float3 ohi = R.hi, olo = R.lo;
    R.hi = nhi;
    R.lo = nlo;
    R.c = P;
    R.d = dnew;
    if (outside(V, P)) {
        const float3 h0 = make_float3(ohi.x - B, ohi.y - B, ohi.z - B);  // exact
        const float tau = exit_fraction(V, h0, olo, inc);
        R.hi = h0 + fma3(tau, inc, olo);
        R.d = wr + dnew;
        R.flags |= HH_FLAG_EXITED;
        return true;
    }
    return false;
}

// Marches a ray that entered the box until it leaves it or runs out of steps.
// `sparse` (the same for every ray of the volume) picks the loop that tests the
// free-corner mask or the one that does not.
template <int STORAGE, int STEPPER, int LEN, int ADDR>
__device__ __forceinline__ void ray_march(const VolArgs& V, const void* __restrict__ vol,
                                          unsigned sparse, RayState& R) {
    if (sparse) {
        while (R.k < V.max_steps &&
               !ray_step<STORAGE, STEPPER, LEN, ADDR, true>(V, vol, R)) {
        }
    } else {
        while (R.k < V.max_steps &&
               !ray_step<STORAGE, STEPPER, LEN, ADDR, false>(V, vol, R)) {
        }
    }
}

// Display byte of a colour in [0, 1]: round-to-nearest-even of 255 v.
__device__ __forceinline__ uint8_t to_u8(float v) {
    return static_cast<uint8_t>(__float2uint_rn(__fmul_rn(fminf(fmaxf(v, 0.0f), 1.0f), 255.0f)));
}

// Final state, background lookup and the writes of one pixel. A ray that
// missed reports the eye and its primary direction; one that ran out of
// steps reports its current state (MAXSTEPS).
__device__ __forceinline__ void ray_end(const VolArgs& V, const ViewArgs& C, int px, int py,
                                        const RayState& R) {
    uint32_t flags = R.flags;
    float3 ep = R.hi, ed = R.d;  // of a ray that exited
    if (!(flags & HH_FLAG_HIT)) {
        ep = C.eye;
        ed = R.wr;
    } else if (!(flags & HH_FLAG_EXITED)) {
        flags |= HH_FLAG_MAXSTEPS;
        ep = make_float3((R.hi.x - V.bias) + R.lo.x, (R.hi.y - V.bias) + R.lo.y,
                         (R.hi.z - V.bias) + R.lo.z);
        ed = R.wr + R.d;
    }
    const float3 rgb = scene_color(V, ep, ed);
    const size_t pix = static_cast<size_t>(py) * C.W + px;
    if (C.rgb) {
        C.rgb[3 * pix + 0] = rgb.x;
        C.rgb[3 * pix + 1] = rgb.y;
        C.rgb[3 * pix + 2] = rgb.z;
    }
    if (C.rgb8) {
        C.rgb8[3 * pix + 0] = to_u8(rgb.x);
        C.rgb8[3 * pix + 1] = to_u8(rgb.y);
        C.rgb8[3 * pix + 2] = to_u8(rgb.z);
    }
    if (C.exit_pos) {
        C.exit_pos[3 * pix + 0] = ep.x;
        C.exit_pos[3 * pix + 1] = ep.y;
        C.exit_pos[3 * pix + 2] = ep.z;
    }
    if (C.exit_dir) {
        C.exit_dir[3 * pix + 0] = ed.x;
        C.exit_dir[3 * pix + 1] = ed.y;
        C.exit_dir[3 * pix + 2] = ed.z;
    }
    if (C.steps) C.steps[pix] = R.k;
    if (C.flags) C.flags[pix] = flags;
}

// Row of tiles taken i-th of n, from row mid outwards: mid, mid + 1, mid - 1, ...,
// then the rest of the longer side.
__device__ __forceinline__ int row_from(int i, int n, int mid) {
    if (i <= 2 * min(mid, n - 1 - mid)) return mid + ((i & 1) ? (i + 1) >> 1 : -(i >> 1));
    return mid < n - 1 - mid ? i : n - 1 - i;
}

// One view, one thread per pixel: a block of 128 threads covers 16x8 pixels,
// each warp an 8x4 tile. Blocks start with the row of tiles that sees the
// volume's centre and go outwards: the rays get shorter, so that the launch
// does not end on a few long ones (720p view of a 192x160x224 turbulence volume
// 180 us top to bottom, 166 so; 641x363 RK4 view 94 against 85; 1080p view of
// the 256^3 plume 295 against 285). Its blocks never release_next(): those of
// another view behind it would gather on the SMs that empty first (the RK4 view,
// launches back to back: 87.5 us, without 62.1, launched as ordinary ones 64.6).
template <int STORAGE, int STEPPER, int LEN, int ADDR>
__global__ void __launch_bounds__(128, march_blocks(STORAGE, STEPPER))
    march_kernel(const VolArgs V, const ViewArgs C, const int mid) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int tx, ty;
    tile_pixel(lane, 3, tx, ty);
    // (every load of the volume's depends on the pixel)
    asm volatile("griddepcontrol.wait;" : "+r"(tx), "+r"(ty) :: "memory");
    const int px = blockIdx.x * 16 + (warp & 1) * 8 + tx;
    const int py = row_from(blockIdx.y, gridDim.y, mid) * 8 + (warp >> 1) * 4 + ty;
    if (px >= C.W || py >= C.H) return;
    RayState R;
    ray_begin<LEN>(V, after_wait(V.scales), C, px, py, R);
    if (R.flags & HH_FLAG_HIT)
        ray_march<STORAGE, STEPPER, LEN, ADDR>(V, V.vol, __ldg(after_wait(V.sparse)), R);
    ray_end(V, C, px, py, R);
}

// View and place (column, row of tiles) of batch tile t: from the order table
// when there is one ({view, row << 16 | column}, the tiles of all views in the
// order the table gives; a view has at most 2^15 rows and 2^14 columns), else
// in the last view whose first tile is <= t (views one after the other).
__device__ __forceinline__ void tile_of(int t, int n_views, const int* s_begin,
                                        const ViewArgs* __restrict__ views,
                                        const uint2* __restrict__ order, int& view, int& tx,
                                        int& ty) {
    if (order) {
        const uint2 o = __ldg(order + t);
        view = static_cast<int>(o.x);
        tx = static_cast<int>(o.y & 0xFFFFu);
        ty = static_cast<int>(o.y >> 16);
        return;
    }
    int lo = 0, hi = n_views - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (s_begin[mid] <= t) lo = mid;
        else hi = mid - 1;
    }
    view = lo;
    const int local = t - s_begin[lo], tiles_x = __ldg(&views[lo].tiles_x);
    ty = local / tiles_x;
    tx = local - ty * tiles_x;
}

// Persistent batched march over many views of uneven size. Each warp pulls
// 32-pixel tiles (tile_w x 32/tile_w pixels) of any view from one atomic
// counter and marches them lane by lane. Warp-level compaction: when at
// least refill_min lanes are idle (their rays left the volume, missed it or
// ran out of steps), the idle lanes take the next pixels of the warp's
// current tile (and of the next tile when it runs out) while the other lanes
// keep marching; refill_min = 32 refills only when every lane is idle, i.e.
// plain tile-at-a-time scheduling, compiled separately (REFILL = false) as
// march_kernel's loop around a tile counter. In that mode `group` = 1 makes
// the block, not the warp, the unit of scheduling: one atomic fetches one
// tile per warp (consecutive tiles: neighbours in a view), the block's warps
// march them side by side on one SM, sharing its L1, and meet at a barrier
// before the next group, as march_kernel's blocks do when they retire. The
// per-ray arithmetic is march_kernel's.
template <int STORAGE, int STEPPER, int LEN, bool REFILL, int ADDR>
__global__ void __launch_bounds__(256, batch_blocks(STORAGE, STEPPER, REFILL))
    march_batch_kernel(const VolArgs V, const ViewArgs* __restrict__ views, int n_views,
                       int total_tiles, int tile_w, unsigned* __restrict__ counter,
                       int refill_min, const uint2* __restrict__ order, int group) {
    extern __shared__ int s_begin[];  // first tile of each view, then total_tiles
    for (int i = threadIdx.x; i <= n_views; i += blockDim.x)
        s_begin[i] = i < n_views ? views[i].tile_begin : total_tiles;
    __syncthreads();
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const unsigned lt_mask = (1u << lane) - 1u;
    const int tile_w_log2 = tile_w == 16 ? 4 : (tile_w == 8 ? 3 : 2);
    const unsigned sparse = __ldg(V.sparse);
    if (!REFILL) {
        __shared__ int s_group;  // first tile of the block's current group
        // the warps' current view records: one coalesced load where the view
        // changes, instead of a load per field and tile
        __shared__ ViewArgs s_view[8];
        constexpr int kWords = sizeof(ViewArgs) / sizeof(unsigned);
        const int warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
        ViewArgs& C = s_view[warp];
        int have_view = -1;
        int lx, ly;
        tile_pixel(lane, tile_w_log2, lx, ly);
        for (;;) {
            int t = 0;
            if (group) {  // block-uniform branch
                if (threadIdx.x == 0) s_group = static_cast<int>(atomicAdd(counter, 1u)) * warps;
                __syncthreads();
                const int g0 = s_group;
                __syncthreads();  // read by every warp before thread 0 writes it again
                if (g0 >= total_tiles) return;
                t = g0 + warp;
                if (t >= total_tiles) continue;
            } else {
                if (lane == 0) t = static_cast<int>(atomicAdd(counter, 1u));
                t = __shfl_sync(FULL, t, 0);
                if (t >= total_tiles) return;
            }
            int view, tx, ty;
            tile_of(t, n_views, s_begin, views, order, view, tx, ty);
            if (view != have_view) {  // warp-uniform
                __syncwarp();         // the last tile's reads are done
                const unsigned* src = reinterpret_cast<const unsigned*>(views + view);
                for (int w = lane; w < kWords; w += 32)
                    reinterpret_cast<unsigned*>(&C)[w] = __ldg(src + w);
                __syncwarp();
                have_view = view;
            }
            const int px = (tx << tile_w_log2) + lx, py = ty * (32 >> tile_w_log2) + ly;
            if (px < C.W && py < C.H) {
                RayState R;
                ray_begin<LEN>(V, V.scales, C, px, py, R);
                if (R.flags & HH_FLAG_HIT)
                    ray_march<STORAGE, STEPPER, LEN, ADDR>(V, V.vol, sparse, R);
                ray_end(V, C, px, py, R);
            }
        }
    }
    int tile_x = 0, tile_y = 0, tile_view = 0, pos = 32;  // the warp's pixel stream (warp-uniform)
    bool done = false, have = false;
    int vi = 0, px = 0, py = 0;
    RayState R;
    for (;;) {
        const unsigned free_mask = __ballot_sync(FULL, !have);
        if (!done && __popc(free_mask) >= refill_min) {
            unsigned todo = free_mask;
            while (todo && !done) {
                if (pos >= 32) {
                    int t = 0;
                    if (lane == 0) t = static_cast<int>(atomicAdd(counter, 1u));
                    t = __shfl_sync(FULL, t, 0);
                    if (t >= total_tiles) {
                        done = true;
                        break;
                    }
                    tile_of(t, n_views, s_begin, views, order, tile_view, tile_x, tile_y);
                    pos = 0;
                }
                const int avail = 32 - pos;
                const int rank = __popc(todo & lt_mask);
                const bool mine = ((todo >> lane) & 1u) && rank < avail;
                if (mine) {
                    const ViewArgs& C = views[tile_view];
                    const int p = pos + rank;
                    int lx, ly;
                    tile_pixel(p, tile_w_log2, lx, ly);
                    px = (tile_x << tile_w_log2) + lx;
                    py = tile_y * (32 >> tile_w_log2) + ly;
                    vi = tile_view;
                    if (px < C.W && py < C.H) {
                        ray_begin<LEN>(V, V.scales, C, px, py, R);
                        if ((R.flags & HH_FLAG_HIT) && V.max_steps > 0) have = true;
                        else ray_end(V, C, px, py, R);
                    }
                }
                pos += min(avail, __popc(todo));
                todo &= ~__ballot_sync(FULL, mine);
            }
        }
        if (__ballot_sync(FULL, have) == 0u) {
            if (done) break;
            continue;
        }
        if (have) {
            const bool left =
                sparse ? ray_step<STORAGE, STEPPER, LEN, ADDR, true>(V, V.vol, R)
                       : ray_step<STORAGE, STEPPER, LEN, ADDR, false>(V, V.vol, R);
            if (left || R.k >= V.max_steps) {
                ray_end(V, views[vi], px, py, R);
                have = false;
            }
        }
    }
}

// The render server's persistent worker (ray-level continuous batching):
// jobs (requests) are published by the host into a device queue while the
// kernel runs. A warp keeps a cursor j on the job table: it waits for job j
// to be published (n_jobs > j) and written (its entry's seq == j), takes
// tiles of it from the job's counter until they run out, then moves on. The
// warp that finishes a job's last tile raises the job's flag in host-mapped
// memory. Every wait is bounded in time (the global nanosecond timer): a warp
// whose queue has stayed empty for idle_ns counts itself idle, and once every
// warp of the launch is idle they all leave together (a warp that finds work
// again uncounts itself; the host launches the worker again when new work
// arrives, so the whole grid, not a remnant of it, serves the next burst); a
// warp told to stop leaves when idle; and a job whose entry does not appear
// within entry_ns of its publication being seen is failed (flag
// HH_JOB_FAILED) instead of waited for. Idle polls back off
// from 1 to 32 us, so thousands of idle warps do not crowd the queue's cache
// line. The per-ray arithmetic is march_kernel's (ray_begin / ray_step /
// ray_end) on the volume of the tile's job.
__device__ __forceinline__ int ld_acquire_int(const int* p) {
    int v;
    asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ unsigned atom_add_acq_rel(unsigned* p, unsigned v) {
    unsigned old;
    asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], %2;"
                 : "=r"(old)
                 : "l"(p), "r"(v)
                 : "memory");
    return old;
}
__device__ __forceinline__ unsigned long long global_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// What a warp of the serving worker keeps between tiles, in shared memory: the
// view record of its current tile and its job. In registers they made the
// march's loop spill more (six requests of three views on a 384^3 FP16 volume, four
// blocks: 12.2 against 11.4 ms).
struct alignas(16) WorkerWarp {
    ViewArgs view;
    unsigned long long vol, scales;  // addresses of the job's volume and its FP16 scales
    unsigned sparse;
    int view_begin, n_views, n_tiles;
    int view_first, view_end;  // job-relative tiles of the view held
    unsigned long long idle_since;
    unsigned backoff;          // ns
    int counted_idle;
};

// Resident 256-thread blocks per SM of the serving worker: as the batched
// kernel's (FP16: 5 against 4, six requests of three views on a 384^3 volume in
// 10.65 against 11.4 ms, although 60 to 68 bytes spill at 5).
constexpr int worker_blocks(int storage, int stepper) {
    return batch_blocks(storage, stepper, false);
}

template <int STORAGE, int STEPPER, int LEN, int ADDR>
__global__ void __launch_bounds__(256, worker_blocks(STORAGE, STEPPER))
    serve_worker_kernel(const VolArgs V, const ServeWorkerArgs W) {
    extern __shared__ __align__(16) unsigned char s_raw[];  // a WorkerWarp per warp
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    WorkerWarp& S = reinterpret_cast<WorkerWarp*>(s_raw)[warp];
    ViewArgs& C = S.view;
    const int tile_w_log2 = W.tile_w == 16 ? 4 : (W.tile_w == 8 ? 3 : 2);
    const int tile_h = 32 >> tile_w_log2;
    const char* views = static_cast<const char*>(W.views);
    constexpr int kWords = sizeof(ViewArgs) / sizeof(unsigned);
    int j = ld_acquire_int(W.first_open);
    int have_job = -1;
    unsigned t = 0;  // this warp's claimed tile of job j (valid while have_job == j)
    bool claimed_next = false;
    // lane 0's alone: since when the warp has been idle, whether it counts so
    if (lane == 0) {
        S.idle_since = 0;
        S.backoff = 1000;
        S.counted_idle = 0;
        atomicAdd(W.started_warps, 1);
    }
    __syncwarp();
    for (;;) {
        if (j != have_job) {
            // wait for job j: published, then written (both bounded in time)
            int ok = 0;
            if (lane == 0) {
                if (j < ld_acquire_int(W.n_jobs)) {
                    ok = 1;
                    if (*reinterpret_cast<const volatile unsigned*>(W.claimed + j) >=
                        HH_JOB_CLAIM_FAILED) {
                        ok = 2;  // failed by another warp: skip it
                    } else if (ld_acquire_int(&W.jobs[j].seq) != j) {
                        const unsigned long long t0 = global_ns();
                        while (ld_acquire_int(&W.jobs[j].seq) != j) {
                            if (global_ns() - t0 > W.entry_ns) {
                                ok = 2;
                                if (atomicOr(W.claimed + j, HH_JOB_CLAIM_FAILED) <
                                    HH_JOB_CLAIM_FAILED) {
                                    __threadfence_system();
                                    W.host_done[j] = HH_JOB_FAILED;
                                }
                                break;
                            }
                            __nanosleep(1000);
                        }
                    }
                } else if (ld_acquire_int(W.stop) != 0) {
                    ok = -1;  // stop requested
                }
            }
            ok = __shfl_sync(FULL, ok, 0);
            if (ok == -1) {
                if (lane == 0) W.host_ctl[1] = HH_WORKER_STOPPED;
                break;
            }
            if (ok == 0) {  // nothing published beyond j: idle (bounded)
                int leave = 0;
                if (lane == 0) {
                    const unsigned long long now = global_ns();
                    if (S.idle_since == 0) S.idle_since = now;
                    if (!S.counted_idle && now - S.idle_since > W.idle_ns) {
                        S.counted_idle = 1;
                        // all warps that have started are idle: the launch leaves
                        // (a block that starts later sees the flag and leaves too)
                        if (atomicAdd(W.idle_warps, 1) + 1 == ld_acquire_int(W.started_warps))
                            atomicExch(W.leave, 1);
                    }
                    leave = ld_acquire_int(W.leave);
                }
                if (__shfl_sync(FULL, leave, 0)) break;
                __nanosleep(S.backoff);
                __syncwarp();
                if (lane == 0) S.backoff = min(S.backoff * 2u, 32000u);
                __syncwarp();
                j = max(j, ld_acquire_int(W.first_open));
                continue;
            }
            if (ok == 2) {
                ++j;
                continue;
            }
            __syncwarp();
            if (lane == 0) {
                S.idle_since = 0;
                S.backoff = 1000;
                if (S.counted_idle) atomicSub(W.idle_warps, 1);
                S.counted_idle = 0;
                const ServeJob* e = W.jobs + j;
                S.vol = __ldcg(reinterpret_cast<const unsigned long long*>(&e->vol));
                S.scales = __ldcg(reinterpret_cast<const unsigned long long*>(&e->scales));
                S.sparse = __ldcg(reinterpret_cast<const unsigned*>(
                    __ldcg(reinterpret_cast<const unsigned long long*>(&e->sparse))));
                S.view_begin = __ldcg(&e->view_begin);
                S.n_views = __ldcg(&e->n_views);
                S.n_tiles = __ldcg(&e->n_tiles);
                S.view_first = S.view_end = 0;
            }
            __syncwarp();
            have_job = j;
            claimed_next = false;
        }
        if (!claimed_next) {
            if (lane == 0) t = atomicAdd(W.claimed + j, 1u);
            t = __shfl_sync(FULL, t, 0);
        }
        claimed_next = false;
        if (t >= static_cast<unsigned>(S.n_tiles)) {  // exhausted (or failed): next job
            ++j;
            if (lane == 0) atomicMax(W.first_open, j);
            continue;
        }
        const int ti = static_cast<int>(t);
        if (ti < S.view_first || ti >= S.view_end) {
            // the tile's view: the last view of the job whose first tile is <= t
            int lo = 0, hi = S.n_views - 1;
            while (lo < hi) {
                const int mid = (lo + hi + 1) >> 1;
                const ViewArgs* vm = reinterpret_cast<const ViewArgs*>(
                    views + static_cast<size_t>(S.view_begin + mid) * sizeof(ViewArgs));
                if (__ldcg(&vm->tile_begin) <= ti) lo = mid;
                else hi = mid - 1;
            }
            __syncwarp();
            const unsigned* src = reinterpret_cast<const unsigned*>(
                views + static_cast<size_t>(S.view_begin + lo) * sizeof(ViewArgs));
            for (int w = lane; w < kWords; w += 32)
                reinterpret_cast<unsigned*>(&C)[w] = __ldcg(src + w);
            __syncwarp();
            if (lane == 0) {
                S.view_first = C.tile_begin;
                S.view_end = C.tile_begin + C.tiles_x * ((C.H + tile_h - 1) / tile_h);
            }
            __syncwarp();
        }
        const int local = ti - S.view_first;
        const int ty = local / C.tiles_x, tx = local - ty * C.tiles_x;
        int lx, ly;
        tile_pixel(lane, tile_w_log2, lx, ly);
        const int px = (tx << tile_w_log2) + lx, py = ty * tile_h + ly;
        if (px < C.W && py < C.H) {
            RayState R;
            ray_begin<LEN>(V, reinterpret_cast<const float*>(S.scales), C, px, py, R);
            if (R.flags & HH_FLAG_HIT)
                ray_march<STORAGE, STEPPER, LEN, ADDR>(
                    V, reinterpret_cast<const void*>(S.vol), S.sparse, R);
            ray_end(V, C, px, py, R);
        }
        // count the tile (release: its outputs are ordered before the count,
        // so the warp that sees the count reach n_tiles sees every tile) and
        // claim the next one in the same breath, unless the launch is leaving
        // (then the next launch takes the job's remaining tiles)
        __syncwarp();
        unsigned next = 0;
        int leave = 0;
        if (lane == 0) {
            const unsigned before = atom_add_acq_rel(W.done + j, 1u);
            leave = ld_acquire_int(W.leave);
            if (!leave) next = atomicAdd(W.claimed + j, 1u);
            if (before + 1u == static_cast<unsigned>(S.n_tiles)) {
                __threadfence_system();
                W.host_done[j] = HH_JOB_DONE;
            }
        }
        if (__shfl_sync(FULL, leave, 0)) break;
        t = __shfl_sync(FULL, next, 0);
        claimed_next = true;
    }
}

// Whether the volume needs ADDR_ANY: its byte offsets do not fit 32 bits (mask_off
// is the end of its data).
bool addr_any(unsigned long long mask_off) { return mask_off >= (1ull << 32); }
// The form of a kernel for volumes that do not: `addr`, or ADDR_ANY, compiled
// anyway, where speed does not matter.
constexpr int narrow(int len, int addr) { return len == LEN_SUBNORMAL ? ADDR_ANY : addr; }

template <int STORAGE, int STEPPER, int LEN>
void launch_one(const VolArgs& V, const ViewArgs& C, cudaStream_t s) {
    const dim3 block(128);
    const dim3 grid((C.W + 15) / 16, (C.H + 7) / 8);
    // row of blocks that sees the volume's centre (the middle one if it is behind
    // the camera)
    const float o[3] = {0.5f * V.nx - C.eye.x, 0.5f * V.ny - C.eye.y, 0.5f * V.nz - C.eye.z};
    const float ahead = C.f.x * o[0] + C.f.y * o[1] + C.f.z * o[2];
    const float up = C.u.x * o[0] + C.u.y * o[1] + C.u.z * o[2];
    float row = 0.5f * C.H;
    if (ahead > 0.0f) row = (C.b0 - up / ahead) / C.s;
    const int mid = static_cast<int>(fminf(fmaxf(row, 0.0f), C.H - 1.0f)) / 8;
    if (addr_any(V.mask_off))
        launch_next(march_kernel<STORAGE, STEPPER, LEN, ADDR_ANY>, grid, block, s, V, C, mid);
    else
        launch_next(march_kernel<STORAGE, STEPPER, LEN, narrow(LEN, ADDR_BASE)>, grid, block,
                    s, V, C, mid);
}

// Calls F<STORAGE, STEPPER, LEN>::run(args...) for the runtime choice.
template <template <int, int, int> class F, int STORAGE, int STEPPER, typename... Args>
void dispatch_len(int len, Args&&... args) {
    if (len == LEN_FIXED) F<STORAGE, STEPPER, LEN_FIXED>::run(args...);
    else if (len == LEN_EQ18) F<STORAGE, STEPPER, LEN_EQ18>::run(args...);
    else F<STORAGE, STEPPER, LEN_SUBNORMAL>::run(args...);
}
template <template <int, int, int> class F, typename... Args>
void dispatch(int storage, const hh_step_params& P, Args&&... args) {
    const bool fp16 = storage == HH_STORE_FP16_SCALED, rk4 = P.stepper == HH_STEP_RK4;
    const int len = step_len(P);
    if (!fp16 && !rk4) dispatch_len<F, HH_STORE_FP32, HH_STEP_EULER_PAPER>(len, args...);
    else if (!fp16) dispatch_len<F, HH_STORE_FP32, HH_STEP_RK4>(len, args...);
    else if (!rk4) dispatch_len<F, HH_STORE_FP16_SCALED, HH_STEP_EULER_PAPER>(len, args...);
    else dispatch_len<F, HH_STORE_FP16_SCALED, HH_STEP_RK4>(len, args...);
}

template <int ST, int SP, int LEN>
struct SingleLaunch {
    static void run(const VolArgs& V, const ViewArgs& C, cudaStream_t s) {
        launch_one<ST, SP, LEN>(V, C, s);
    }
};

// The batch kernel of a launch: refill_min >= 32 runs the tile-at-a-time
// instantiation (REFILL = false).
template <int ST, int SP, int LEN>
auto batch_kernel(bool any, int refill_min) {
    if (refill_min >= 32)
        return any ? march_batch_kernel<ST, SP, LEN, false, ADDR_ANY>
                   : march_batch_kernel<ST, SP, LEN, false, narrow(LEN, ADDR_BASE)>;
    return any ? march_batch_kernel<ST, SP, LEN, true, ADDR_ANY>
               : march_batch_kernel<ST, SP, LEN, true, narrow(LEN, ADDR_BASE)>;
}

template <int ST, int SP, int LEN>
struct BatchLaunch {
    static void run(const VolArgs& V, const ViewArgs* views, int n_views, int total_tiles,
                    int tile_w, unsigned* counter, int refill_min, const uint2* order, int group,
                    int blocks, int threads, cudaStream_t s) {
        const size_t smem = (n_views + 1) * sizeof(int);
        batch_kernel<ST, SP, LEN>(addr_any(V.mask_off), refill_min)<<<blocks, threads, smem, s>>>(
            V, views, n_views, total_tiles, tile_w, counter, refill_min, order,
            refill_min >= 32 ? group : 0);
    }
};

// The worker on volumes of one grid and storage: all below 4 GiB, or none.
template <int ST, int SP, int LEN>
auto worker_kernel(bool any) {
    return any ? serve_worker_kernel<ST, SP, LEN, ADDR_ANY>
               : serve_worker_kernel<ST, SP, LEN, narrow(LEN, ADDR_PTR)>;
}

template <int ST, int SP, int LEN>
struct WorkerLaunch {
    static void run(const VolArgs& V, const ServeWorkerArgs& W, int blocks, int threads,
                    cudaStream_t s) {
        const size_t smem = (threads / 32) * sizeof(WorkerWarp);
        worker_kernel<ST, SP, LEN>(addr_any(V.mask_off))<<<blocks, threads, smem, s>>>(V, W);
    }
};

template <int ST, int SP, int LEN>
struct WorkerOccupancy {
    static void run(bool any, int threads, int* blocks_per_sm) {
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(
            blocks_per_sm, worker_kernel<ST, SP, LEN>(any), threads,
            (threads / 32) * sizeof(WorkerWarp));
    }
};

template <int ST, int SP, int LEN>
struct BatchOccupancy {
    static void run(int threads, size_t smem, bool any, int refill_min, int* blocks_per_sm) {
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(
            blocks_per_sm, batch_kernel<ST, SP, LEN>(any, refill_min), threads, smem);
    }
};

VolArgs make_vol_args(const hh_volume_s* vol, const hh_step_params& P, const hh_background& bg) {
    VolArgs A;
    A.vol = vol->data;
    A.scales = vol->scales_dev;
    A.nx = vol->nx;
    A.ny = vol->ny;
    A.nz = vol->nz;
    A.sparse = vol->sparse_dev;
    A.strides = zpair_strides(vol->row, vol->pair, vol->storage == HH_STORE_FP32 ? 16u : 8u);
    A.mask_off = vol->mask_off;
    // bias: a power of two B with B >= 2 * step and B >= extent + step + 1, so
    // positions in [-step, extent + step] keep hi in [B/2, 2B - 1] and both
    // hi - B and hi - (B - 1/2) are exact (Sterbenz)
    const float step = P.adaptive ? P.h_max : P.h_fixed;
    const float need =
        fmaxf(static_cast<float>(max(vol->nx, max(vol->ny, vol->nz))) + step + 1.0f, 2.0f * step);
    float B = 8.0f;
    while (B < need) B *= 2.0f;
    A.bias = B;
    A.bias_u = B - 0.5f;
    A.ux = static_cast<float>(vol->nx) + 0.5f;
    A.uy = static_cast<float>(vol->ny) + 0.5f;
    A.uz = static_cast<float>(vol->nz) + 0.5f;
    A.h_fixed = P.h_fixed;
    A.h_min = P.adaptive ? P.h_min : P.h_fixed;
    A.h_max = P.adaptive ? P.h_max : P.h_fixed;
    A.theta = P.adaptive ? P.theta_max : 0.0f;
    A.eps = P.adaptive ? P.eps : 1.0f;
    A.max_steps = P.max_steps;
    A.bg = bg.rgb8_dev;
    A.bgW = bg.width;
    A.bgH = bg.height;
    A.bg_u = static_cast<float>(bg.width) / (2.0f * kPi);
    A.bg_v = static_cast<float>(bg.height) / kPi;
    A.n_planes = bg.n_planes;
    for (int k = 0; k < HH_MAX_PLANES; ++k) A.planes[k] = bg.planes[k];
    return A;
}

ViewArgs make_view_args(const hh_camera& cam, const hh_view_out& out, int tile_w) {
    ViewArgs C;
    C.eye = make_float3(cam.eye[0], cam.eye[1], cam.eye[2]);
    // camera basis and pixel mapping, once per view in FP64 (see primary_ray)
    double f[3], r[3], u[3], fn = 0.0, rn = 0.0;
    for (int a = 0; a < 3; ++a) {
        f[a] = static_cast<double>(cam.look_at[a]) - cam.eye[a];
        fn += f[a] * f[a];
    }
    for (int a = 0; a < 3; ++a) f[a] /= std::sqrt(fn);
    const double up[3] = {cam.up[0], cam.up[1], cam.up[2]};
    r[0] = f[1] * up[2] - f[2] * up[1];
    r[1] = f[2] * up[0] - f[0] * up[2];
    r[2] = f[0] * up[1] - f[1] * up[0];
    for (int a = 0; a < 3; ++a) rn += r[a] * r[a];
    for (int a = 0; a < 3; ++a) r[a] /= std::sqrt(rn);
    u[0] = r[1] * f[2] - r[2] * f[1];
    u[1] = r[2] * f[0] - r[0] * f[2];
    u[2] = r[0] * f[1] - r[1] * f[0];
    C.f = make_float3(static_cast<float>(f[0]), static_cast<float>(f[1]), static_cast<float>(f[2]));
    C.r = make_float3(static_cast<float>(r[0]), static_cast<float>(r[1]), static_cast<float>(r[2]));
    C.u = make_float3(static_cast<float>(u[0]), static_cast<float>(u[1]), static_cast<float>(u[2]));
    const double t = std::tan(0.5 * static_cast<double>(cam.vfov_deg) * (M_PI / 180.0));
    C.a0 = static_cast<float>(-t * cam.width / cam.height);
    C.b0 = static_cast<float>(t);
    C.s = static_cast<float>(2.0 * t / cam.height);
    C.W = cam.width;
    C.H = cam.height;
    C.rgb = out.rgb;
    C.rgb8 = out.rgb8;
    C.exit_pos = out.exit_pos;
    C.exit_dir = out.exit_dir;
    C.steps = out.steps;
    C.flags = out.flags;
    C.tiles_x = (cam.width + tile_w - 1) / tile_w;
    C.tile_begin = 0;
    return C;
}
}  // namespace

cudaError_t launch_trace(const hh_volume_s* vol, const hh_camera& cam, const hh_step_params& P,
                         const hh_background& bg, const hh_view_out& out, cudaStream_t s) {
    if (vol->layout != HH_LAYOUT_ZPAIR) return cudaErrorInvalidValue;
    const VolArgs V = make_vol_args(vol, P, bg);
    const ViewArgs C = make_view_args(cam, out, 8);
    dispatch<SingleLaunch>(vol->storage, P, V, C, s);
    count_launch();
    return cudaGetLastError();
}

}  // namespace hh

namespace hh {

size_t view_record_bytes() { return sizeof(ViewArgs); }

int build_view_table(const hh_camera* cams, const hh_view_out* outs, int n, int tile_w,
                     void* host_records) {
    ViewArgs* v = static_cast<ViewArgs*>(host_records);
    const int tile_h = 32 / tile_w;
    int64_t tiles = 0;
    for (int i = 0; i < n; ++i) {
        v[i] = make_view_args(cams[i], outs[i], tile_w);
        v[i].tile_begin = static_cast<int>(tiles);
        tiles += static_cast<int64_t>(v[i].tiles_x) * ((cams[i].height + tile_h - 1) / tile_h);
        if (tiles > (int64_t(1) << 30)) return -1;
    }
    return static_cast<int>(tiles);
}

int serve_worker_blocks_per_sm(const hh_volume_s* like, const hh_step_params& P, int threads) {
    int bps = 0;
    dispatch<WorkerOccupancy>(like->storage, P, addr_any(like->mask_off), threads, &bps);
    return max(bps, 1);
}

cudaError_t launch_serve_worker(const hh_volume_s* like, const hh_step_params& P,
                                const hh_background& bg, const ServeWorkerArgs& W, int blocks,
                                int threads, cudaStream_t s) {
    if (like->layout != HH_LAYOUT_ZPAIR) return cudaErrorInvalidValue;
    const VolArgs V = make_vol_args(like, P, bg);
    dispatch<WorkerLaunch>(like->storage, P, V, W, blocks, threads, s);
    count_launch();
    return cudaGetLastError();
}

}  // namespace hh

// ------------------------------------------------------------------------
// Batched multi-view launches (hh_batch_*)
// ------------------------------------------------------------------------
struct hh_batch_s {
    hh_volume vol = nullptr;
    hh_step_params params{};
    hh_background bg{};
    std::vector<hh_camera> cams;
    std::vector<hh_view_out> outs;
    hh_batch_config cfg{};
    int total_tiles = 0;
    hh::ViewArgs* views_dev = nullptr;
    unsigned* counter_dev = nullptr;
    uint2* order_dev = nullptr;  // tile order table (NULL: views one after the other)
    int sm_count = 0;
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
    cudaStream_t graph_stream = nullptr;
};

namespace {

using hh::fail;
using hh::cuda_fail;

void drop_graph(hh_batch b) {
    if (b->exec) cudaGraphExecDestroy(b->exec);
    if (b->graph) cudaGraphDestroy(b->graph);
    b->exec = nullptr;
    b->graph = nullptr;
    b->graph_stream = nullptr;
}

// The interleaved tile order (tile_order 1): the tiles of all views sorted by
// their relative row in their view (then by view, then by column), so that
// every view sweeps the volume top to bottom at the same time. The top quarter,
// whose rays are short, is not taken first but beside the bottom quarter, in
// mirrored order, so that the launch ends on its shortest rays (8 views of a
// 256^3 FP16 volume 1054 -> 1033 us, 12 uneven ones of 384^3 2293 -> 2275; from
// the middle outwards 1034, but 2309: two sweeps share fewer lines in L2; 32
// views of 512^3 the same 9.14 ms).
std::vector<uint2> interleaved_order(const std::vector<hh::ViewArgs>& v, int tile_w) {
    struct Key {
        double k;
        uint32_t view, place;  // place: row << 16 | column
    };
    std::vector<Key> keys;
    const int tile_h = 32 / tile_w;
    for (size_t i = 0; i < v.size(); ++i) {
        const int tiles_y = (v[i].H + tile_h - 1) / tile_h;
        for (int ty = 0; ty < tiles_y; ++ty)
            for (int tx = 0; tx < v[i].tiles_x; ++tx)
                keys.push_back({ty + 0.5 < 0.25 * tiles_y ? 1.0 - (ty + 0.5) / tiles_y
                                                          : (ty + 0.5) / tiles_y,
                                static_cast<uint32_t>(i),
                                static_cast<uint32_t>(ty) << 16 | static_cast<uint32_t>(tx)});
    }
    std::stable_sort(keys.begin(), keys.end(), [](const Key& x, const Key& y) { return x.k < y.k; });
    std::vector<uint2> ord(keys.size());
    for (size_t j = 0; j < keys.size(); ++j) ord[j] = make_uint2(keys[j].view, keys[j].place);
    return ord;
}

// Uploads the view table for the current tile width (synchronous).
hh_status upload_views(hh_batch b) {
    std::vector<hh::ViewArgs> v(b->cams.size());
    int tiles = 0;
    const int tile_w = b->cfg.tile_w, tile_h = 32 / tile_w;
    for (size_t i = 0; i < v.size(); ++i) {
        v[i] = hh::make_view_args(b->cams[i], b->outs[i], tile_w);
        v[i].tile_begin = tiles;
        const int64_t t = static_cast<int64_t>(v[i].tiles_x) * ((b->cams[i].height + tile_h - 1) / tile_h);
        if (tiles + t > (int64_t(1) << 30)) return fail(HH_ERR_INVALID_ARG, "batch has too many pixels");
        tiles += static_cast<int>(t);
    }
    b->total_tiles = tiles;
    cudaError_t e = cudaMemcpy(b->views_dev, v.data(), v.size() * sizeof(hh::ViewArgs),
                               cudaMemcpyHostToDevice);
    if (e != cudaSuccess) return cuda_fail(e, "uploading the view table");
    hh::dev_free(b->order_dev);
    b->order_dev = nullptr;
    if (b->cfg.tile_order == 1) {
        std::vector<uint2> ord = interleaved_order(v, tile_w);
        e = hh::dev_alloc(reinterpret_cast<void**>(&b->order_dev), ord.size() * sizeof(uint2));
        if (e == cudaSuccess)
            e = cudaMemcpy(b->order_dev, ord.data(), ord.size() * sizeof(uint2),
                           cudaMemcpyHostToDevice);
        if (e != cudaSuccess) return cuda_fail(e, "uploading the tile order");
    }
    return HH_OK;
}

hh_status check_config(const hh_batch_config* c) {
    if (!c) return fail(HH_ERR_INVALID_ARG, "config is NULL");
    if (c->block_threads < 32 || c->block_threads > 256 || c->block_threads % 32)
        return fail(HH_ERR_INVALID_ARG, "block_threads must be a multiple of 32 in [32, 256]");
    if (c->blocks_per_sm < 0 || c->blocks_per_sm > 64)
        return fail(HH_ERR_INVALID_ARG, "blocks_per_sm must be in [0, 64]");
    if (c->refill_min < 1 || c->refill_min > 32)
        return fail(HH_ERR_INVALID_ARG, "refill_min must be in [1, 32]");
    if (c->tile_w != 4 && c->tile_w != 8 && c->tile_w != 16)
        return fail(HH_ERR_INVALID_ARG, "tile_w must be 4, 8 or 16");
    if (c->tile_order != 0 && c->tile_order != 1)
        return fail(HH_ERR_INVALID_ARG, "tile_order must be 0 or 1");
    if (c->tile_group != 0 && c->tile_group != 1)
        return fail(HH_ERR_INVALID_ARG, "tile_group must be 0 or 1");
    if (c->tile_group == 1 && c->refill_min != 32)
        return fail(HH_ERR_INVALID_ARG, "tile_group 1 needs tile-at-a-time scheduling (refill_min 32)");
    return HH_OK;
}

int resident_blocks(hh_batch b, int threads, int refill_min) {
    int bps = 0;
    const size_t smem = (b->cams.size() + 1) * sizeof(int);
    hh::dispatch<hh::BatchOccupancy>(b->vol->storage, b->params, threads, smem,
                                     hh::addr_any(b->vol->mask_off), refill_min, &bps);
    return std::max(bps, 1);
}

int grid_blocks(hh_batch b) {
    const int bps = b->cfg.blocks_per_sm > 0
                        ? b->cfg.blocks_per_sm
                        : resident_blocks(b, b->cfg.block_threads, b->cfg.refill_min);
    return b->sm_count * bps;
}

// Counter reset + one persistent launch of `blocks` blocks (no host queries,
// so it can run inside a stream capture).
cudaError_t enqueue(hh_batch b, int blocks, cudaStream_t s) {
    cudaError_t e = cudaMemsetAsync(b->counter_dev, 0, sizeof(unsigned), s);
    if (e != cudaSuccess) return e;
    const int threads = b->cfg.block_threads;
    const hh::VolArgs V = hh::make_vol_args(b->vol, b->params, b->bg);
    hh::dispatch<hh::BatchLaunch>(b->vol->storage, b->params, V, b->views_dev,
                                  static_cast<int>(b->cams.size()), b->total_tiles,
                                  b->cfg.tile_w, b->counter_dev, b->cfg.refill_min,
                                  static_cast<const uint2*>(b->order_dev), b->cfg.tile_group,
                                  blocks, threads, s);
    hh::count_launch();
    return cudaGetLastError();
}

// Autotuner results by workload signature (grid, storage, schedule, views).
std::mutex g_tune_mutex;
std::map<std::string, hh_batch_config> g_tune_cache;

std::string signature(hh_batch b) {
    std::string k = std::to_string(b->vol->nx) + "x" + std::to_string(b->vol->ny) + "x" +
                    std::to_string(b->vol->nz) + "/" + std::to_string(b->vol->storage) + "/" +
                    std::to_string(b->params.stepper) + std::to_string(b->params.adaptive);
    for (const auto& c : b->cams) k += "/" + std::to_string(c.width) + "x" + std::to_string(c.height);
    return k;
}

}  // namespace

extern "C" {

hh_status hh_batch_create(hh_volume vol, const hh_camera* cams, int n_cams,
                          const hh_step_params* params, const hh_background* bg,
                          const hh_view_out* outs, hh_batch* out) {
    if (!out) return fail(HH_ERR_INVALID_ARG, "out is NULL");
    *out = nullptr;
    if (!vol) return fail(HH_ERR_INVALID_ARG, "volume is NULL");
    if (n_cams < 1 || n_cams > 4096 || !cams || !outs)
        return fail(HH_ERR_INVALID_ARG, "a batch needs 1 to 4096 cameras and outputs");
    hh_status st = hh::check_params(params);
    if (st != HH_OK) return st;
    if ((st = hh::check_background(bg)) != HH_OK) return st;
    for (int i = 0; i < n_cams; ++i) {
        if ((st = hh::check_camera(cams[i], i)) != HH_OK) return st;
        if (!outs[i].rgb && !outs[i].rgb8)
            return fail(HH_ERR_INVALID_ARG, "view %d: rgb and rgb8 outputs are both NULL", i);
    }
    hh_batch b = new (std::nothrow) hh_batch_s();
    if (!b) return fail(HH_ERR_OOM, "host allocation failed");
    b->vol = vol;
    b->params = *params;
    b->bg = *bg;
    b->cams.assign(cams, cams + n_cams);
    b->outs.assign(outs, outs + n_cams);
    b->cfg = hh_batch_config{128, 0, 32, 8, 0, 0};
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&b->sm_count, cudaDevAttrMultiProcessorCount, dev);
    cudaError_t e = hh::dev_alloc(reinterpret_cast<void**>(&b->views_dev), n_cams * sizeof(hh::ViewArgs));
    if (e == cudaSuccess) e = hh::dev_alloc(reinterpret_cast<void**>(&b->counter_dev), sizeof(unsigned));
    if (e != cudaSuccess) {
        hh::dev_free(b->views_dev);
        delete b;
        return cuda_fail(e, "batch allocation");
    }
    if ((st = upload_views(b)) != HH_OK) {
        hh_batch_free(b);
        return st;
    }
    *out = b;
    return hh::ok();
}

hh_status hh_batch_set_config(hh_batch b, const hh_batch_config* cfg) {
    if (!b) return fail(HH_ERR_INVALID_ARG, "batch is NULL");
    hh_status st = check_config(cfg);
    if (st != HH_OK) return st;
    const bool retile = cfg->tile_w != b->cfg.tile_w || cfg->tile_order != b->cfg.tile_order;
    b->cfg = *cfg;
    drop_graph(b);
    if (retile && (st = upload_views(b)) != HH_OK) return st;
    return hh::ok();
}

hh_status hh_batch_get_config(hh_batch b, hh_batch_config* cfg) {
    if (!b || !cfg) return fail(HH_ERR_INVALID_ARG, "batch or config is NULL");
    *cfg = b->cfg;
    if (cfg->blocks_per_sm == 0)
        cfg->blocks_per_sm = resident_blocks(b, b->cfg.block_threads, b->cfg.refill_min);
    return hh::ok();
}

hh_status hh_batch_launch(hh_batch b, void* stream) {
    if (!b) return fail(HH_ERR_INVALID_ARG, "batch is NULL");
    cudaError_t e = enqueue(b, grid_blocks(b), static_cast<cudaStream_t>(stream));
    if (e != cudaSuccess) return cuda_fail(e, "batch launch");
    return hh::ok();
}

hh_status hh_batch_launch_graph(hh_batch b, void* stream) {
    if (!b) return fail(HH_ERR_INVALID_ARG, "batch is NULL");
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (!s) return fail(HH_ERR_INVALID_ARG, "graph launches need a created (non-default) stream");
    if (b->exec && b->graph_stream != s) drop_graph(b);
    if (!b->exec) {
        const int blocks = grid_blocks(b);
        cudaError_t e = cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal);
        if (e != cudaSuccess) return cuda_fail(e, "begin capture");
        cudaError_t le = enqueue(b, blocks, s);
        e = cudaStreamEndCapture(s, &b->graph);
        if (le != cudaSuccess) {
            drop_graph(b);
            return cuda_fail(le, "batch launch during capture");
        }
        if (e == cudaSuccess) e = cudaGraphInstantiate(&b->exec, b->graph, 0);
        if (e != cudaSuccess) {
            drop_graph(b);
            return cuda_fail(e, "graph capture");
        }
        b->graph_stream = s;
    }
    cudaError_t e = cudaGraphLaunch(b->exec, s);
    if (e != cudaSuccess) return cuda_fail(e, "graph launch");
    hh::count_launch();
    return hh::ok();
}

hh_status hh_batch_autotune(hh_batch b, int reps, void* stream, hh_batch_config* best) {
    if (!b) return fail(HH_ERR_INVALID_ARG, "batch is NULL");
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const std::string key = signature(b);
    if (reps > 0) {
        std::lock_guard<std::mutex> lock(g_tune_mutex);
        auto it = g_tune_cache.find(key);
        if (it != g_tune_cache.end()) {
            hh_status st = hh_batch_set_config(b, &it->second);
            if (st == HH_OK && best) *best = it->second;
            return st;
        }
    }
    if (reps == 0) return fail(HH_ERR_INVALID_ARG, "reps must be non-zero");
    const int n = reps < 0 ? -reps : reps;
    std::vector<hh_batch_config> cand;
    for (int to : {0, 1})
        for (int tw : {8, 4, 16})
            for (int th : {128, 256, 64})
                for (int rm : {32, 16, 8})
                    for (int bps : {0, -2})
                        for (int tg : {0, 1})
                            if (tg == 0 || rm == 32)
                                cand.push_back(hh_batch_config{th, bps, rm, tw, to, tg});
    cudaEvent_t e0, e1;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    float best_ms = 1e30f;
    hh_batch_config best_cfg = b->cfg;
    hh_status st = HH_OK;
    for (auto c : cand) {
        if (c.blocks_per_sm < 0)
            c.blocks_per_sm = std::max(1, resident_blocks(b, c.block_threads, c.refill_min) / 2);
        if ((st = hh_batch_set_config(b, &c)) != HH_OK) break;
        std::vector<float> t;
        const int blocks = grid_blocks(b);
        cudaError_t e = enqueue(b, blocks, s);  // warm-up
        for (int r = 0; r < n && e == cudaSuccess; ++r) {
            cudaEventRecord(e0, s);
            e = enqueue(b, blocks, s);
            cudaEventRecord(e1, s);
            if (e == cudaSuccess) e = cudaEventSynchronize(e1);
            float ms = 0.0f;
            cudaEventElapsedTime(&ms, e0, e1);
            t.push_back(ms);
        }
        if (e != cudaSuccess) {
            st = cuda_fail(e, "autotune trial");
            break;
        }
        std::sort(t.begin(), t.end());
        const float med = t[t.size() / 2];
        if (med < best_ms) {
            best_ms = med;
            best_cfg = c;
        }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    if (st != HH_OK) return st;
    if ((st = hh_batch_set_config(b, &best_cfg)) != HH_OK) return st;
    {
        std::lock_guard<std::mutex> lock(g_tune_mutex);
        g_tune_cache[key] = best_cfg;
    }
    if (best) *best = best_cfg;
    return hh::ok();
}

hh_status hh_debug_bounds_violations(uint64_t* count, int reset) {
    if (!count) return fail(HH_ERR_INVALID_ARG, "count is NULL");
#ifdef HH_DEBUG_BOUNDS
    unsigned long long c = 0;
    cudaError_t e = cudaDeviceSynchronize();
    if (e == cudaSuccess) e = cudaMemcpyFromSymbol(&c, hh::g_bounds_violations, sizeof c);
    if (e == cudaSuccess && reset) {
        const unsigned long long zero = 0;
        e = cudaMemcpyToSymbol(hh::g_bounds_violations, &zero, sizeof zero);
    }
    if (e != cudaSuccess) return cuda_fail(e, "reading the bounds counter");
    *count = c;
    return hh::ok();
#else
    (void)reset;
    *count = 0;
    return fail(HH_ERR_NOT_FOUND, "this library was built without HH_DEBUG_BOUNDS");
#endif
}

hh_status hh_batch_free(hh_batch b) {
    if (!b) return hh::ok();
    drop_graph(b);
    hh::dev_free(b->views_dev);
    hh::dev_free(b->counter_dev);
    hh::dev_free(b->order_dev);
    delete b;
    return hh::ok();
}

}  // extern "C"
