// kernels.cu -- sm_103a kernels of the plateau-reduced gradient estimator.
//
//   k_instantiate   one CTA per render: Philox draws -> perturbation tau and weight
//                   w (Sec. 3.2, Eq. 11, Algorithm 1), theta +- tau bound into the
//                   scene (Eq. 10's P(theta - tau_i)), derived constants precomputed;
//                   the scene is built in shared memory and written out in one copy.
//   k_trace         persistent render kernel. Each warp pulls (render, pixel block)
//                   work items from a queue, stages the render's scene in its own
//                   shared-memory slot, and traces the block's pixels x samples as a
//                   pool of path tasks: a lane whose path ends takes the next task
//                   at once (ballot + popc), so live paths stay packed in the warp.
//                   Radiance is accumulated per pixel in 2^-32 fixed point (integer
//                   adds are order-independent, so results do not depend on which
//                   lane traced which path). Each pixel's error against the target is
//                   formed exactly in integers, squared in FP32, and summed per block
//                   in FP64 -- the perturbed image never reaches HBM. Variants: path
//                   sharing (a block of all renders traced once in the scene without
//                   the perturbed primitives, recording the paths that may differ) and
//                   the pathwise estimator (Eq. 9, forward-mode tangents).
//   k_trace_affected  path sharing, per-render pass: each render traces again the
//                   recorded paths that may meet its own primitives, resuming where
//                   the renders part, and adds its radiance minus the shared one.
//   k_shared_epilogue path sharing: the blocks with recorded paths, all renders.
//   k_trace_group   render groups: the renders of a path sample traced side by side.
//   k_trace_replay  replay: each path traced once for all renders of a job, recording the
//                   events that can differ; each render replays them with its own
//                   primitives, albedos and (Eq. 9) tangents.
//   k_trace_prefix  paths shared up to the first ray that could meet a moving object that is not
//                   black; from there the renders go on side by side.
//   k_finalize      one CTA per render: L_r from the block partials (fixed order); the
//                   CTA completing a job's last render forms the gradient of Eq. 10
//                   (or the mean of Eq. 9's pathwise gradients) and applies Adam.
//   k_hd_norms, k_hd_perturb, k_hd_grad  high-dimensional parameters (texture scenes):
//                   D-dimensional draws and the gradient W^T dL with Adam.
//   k_adam          standalone Adam update.
//   k_philox        raw Philox words (for bit-exact checks of the random streams).
//   k_ffma_probe    FMA-chain throughput probe (the FP32 peak of the roofline).
//
// FP32 throughout the path tracer; every floating-point reduction is in a fixed order
// and every per-pixel sum is an integer sum, so results are deterministic and
// independent of the launch shape and of other jobs sharing the launch.
#include <cstddef>
#include <cstdint>

#include "internal.h"

namespace prdpt {

constexpr unsigned kFull = 0xffffffffu;  // all lanes of a warp

// Programmatic dependent launch: the kernels of a step are launched so that the next one
// may be scheduled while the previous one drains. Each kernel reads only host-written data
// (job descriptors, the base scene) before pdl_enter, which waits until every kernel
// before it in the stream has completed and its writes are visible (a no-op for a launch
// without the attribute), then lets the next kernel be scheduled.
__device__ __forceinline__ void pdl_enter() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// ---------------------------------------------------------------------------
// small vector helpers
// ---------------------------------------------------------------------------
__device__ __forceinline__ float3 f3(float x, float y, float z) { return make_float3(x, y, z); }
__device__ __forceinline__ float3 xyz(float4 a) { return make_float3(a.x, a.y, a.z); }
__device__ __forceinline__ float3 operator+(float3 a, float3 b) { return f3(a.x + b.x, a.y + b.y, a.z + b.z); }
__device__ __forceinline__ float3 operator-(float3 a, float3 b) { return f3(a.x - b.x, a.y - b.y, a.z - b.z); }
__device__ __forceinline__ float3 operator*(float3 a, float s) { return f3(a.x * s, a.y * s, a.z * s); }
__device__ __forceinline__ float3 operator*(float3 a, float3 b) { return f3(a.x * b.x, a.y * b.y, a.z * b.z); }
// Rounded in this order wherever it is inlined (the order that the compiler chose for the plain
// sum of products), so that kernels that trace the same path agree bit for bit.
__device__ __forceinline__ float dot3(float3 a, float3 b) {
    return __fmaf_rn(a.z, b.z, __fmaf_rn(a.x, b.x, __fmul_rn(a.y, b.y)));
}
__device__ __forceinline__ float3 cross3(float3 a, float3 b) {
    return f3(a.y * b.z - a.z * b.y, a.z * b.x - a.x * b.z, a.x * b.y - a.y * b.x);
}
// The approximate reciprocal, quotient and reciprocal root of the path tracer, without the code
// that the plain intrinsics carry for subnormal operands: their operands in the tracer are never
// subnormal (directions, cosines, roulette probabilities, distances; a subnormal under the root of
// the sphere test gives a miss), and for the others the results are the same. A quad's u x v can
// have a subnormal square: k_instantiate takes the plain root for its normal.
__device__ __forceinline__ float rcp_fast(float a) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(a));
    return r;
}
__device__ __forceinline__ float div_fast(float a, float b) {
    float r;
    asm("div.approx.ftz.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ float rsqrt_fast(float a) {
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(a));
    return r;
}
__device__ __forceinline__ float3 normalized(float3 a) { return a * rsqrt_fast(dot3(a, a)); }
__device__ __forceinline__ float maxc(float3 a) { return fmaxf(a.x, fmaxf(a.y, a.z)); }
// Approximate reciprocal (MUFU.RCP, 1 ulp); +-0 gives +-inf as the slab test needs.
__device__ __forceinline__ float3 rcp3(float3 d) {
    return f3(rcp_fast(d.x), rcp_fast(d.y), rcp_fast(d.z));
}
__device__ __forceinline__ int as_int(float f) { return __float_as_int(f); }

// ---------------------------------------------------------------------------
// Philox4x32-10 (Salmon et al., SC'11) and the open-interval uniform
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint4 philox(uint4 c, unsigned k0, unsigned k1) {
#pragma unroll
    for (int i = 0; i < 10; ++i) {
        if (i) {
            k0 += 0x9E3779B9u;
            k1 += 0xBB67AE85u;
        }
        const unsigned lo0 = 0xD2511F53u * c.x, hi0 = __umulhi(0xD2511F53u, c.x);
        const unsigned lo1 = 0xCD9E8D57u * c.z, hi1 = __umulhi(0xCD9E8D57u, c.z);
        c = make_uint4(hi1 ^ c.y ^ k0, lo1, hi0 ^ c.w ^ k1, lo0);
    }
    return c;
}

// The same generator kept out of line: one copy of its code instead of one per call site,
// for the kernels whose code outgrows the instruction cache (replay, render groups; measured on
// an earlier kernel for caustic: 7.16 -> 6.72 ms a step; the per-render kernel is 4 % faster inline).
__device__ __noinline__ uint4 philox_ool(uint4 c, unsigned k0, unsigned k1) { return philox(c, k0, k1); }

// ((x >> 9) * 2 + 1) / 2^24: exact in FP32, never 0, 1 or 1/2.
__device__ __forceinline__ float u01(unsigned x) { return __uint2float_rn((x >> 9) * 2u + 1u) * 0x1p-24f; }

// ---------------------------------------------------------------------------
// Perturbation sampler (Sec. 3.2; Eq. 11 positivized; supplemental inverse CDF)
// ---------------------------------------------------------------------------
__device__ __forceinline__ int sampler_uniforms(int mode, int D) {
    if (mode == kRadial) {
        if (D == 1) return 2;
        const int n_exp = (D + 1) / 2, extra = (D % 2 == 0);
        return n_exp + 2 * ((D + extra + 1) / 2);
    }
    if (mode == kPerDim) return D;
    return 2 * ((D + 1) / 2);
}

// Box-Muller normal number j of the pairs starting at uniform index `base`.
__device__ __forceinline__ float bm_normal(const float* u, int base, int j) {
    const float a = u[base + 2 * (j / 2)], b = u[base + 2 * (j / 2) + 1];
    const float rad = sqrtf(-2.0f * logf(a));
    float s, c;
    sincospif(2.0f * b, &s, &c);
    return rad * ((j & 1) ? s : c);
}

// Bandwidth at step t: constant, or the warm-started linear decay (Sec. 3.3).
__device__ __forceinline__ float sigma_sched(const float* sigma, int anneal, int total_steps, float sigma_min, int d,
                                             int t) {
    const float s0 = sigma[d];
    if (!anneal) return s0;
    const int w = total_steps / 2;
    if (t < w || total_steps - w <= 0) return s0;
    float frac = float(t - w) / float(total_steps - w);
    frac = fminf(frac, 1.0f);
    return s0 - frac * (s0 - sigma_min);
}
__device__ __forceinline__ float sigma_at(const InstJob& J, int d, int t) {
    return sigma_sched(J.sigma, J.anneal, J.total_steps, J.sigma_min, d, t);
}

// Axis-aligned bounds of a primitive record, inflated by 1e-3 scene units plus 1e-5
// relative, so that a slab test against them is conservative for the exact FP32
// intersection tests of the primitive (path sharing).
template <class Rec>
__device__ __forceinline__ void prim_bounds(const Rec& P, int type, float3& lo, float3& hi) {
    if (type == kSphere) {
        const float4 c = P[0];
        const float rad = fabsf(c.w);
        lo = f3(c.x - rad, c.y - rad, c.z - rad);
        hi = f3(c.x + rad, c.y + rad, c.z + rad);
    } else if (type == kQuad) {
        const float3 c = xyz(P[0]), u = xyz(P[2]), v = xyz(P[3]);
        const float3 e = f3(0.5f * (fabsf(u.x) + fabsf(v.x)), 0.5f * (fabsf(u.y) + fabsf(v.y)),
                            0.5f * (fabsf(u.z) + fabsf(v.z)));
        lo = c - e;
        hi = c + e;
    } else {
        lo = xyz(P[0]);
        hi = xyz(P[1]);
    }
    const float3 m = f3(1e-3f + 1e-5f * fmaxf(fabsf(lo.x), fabsf(hi.x)), 1e-3f + 1e-5f * fmaxf(fabsf(lo.y), fabsf(hi.y)),
                        1e-3f + 1e-5f * fmaxf(fabsf(lo.z), fabsf(hi.z)));
    lo = lo - m;
    hi = hi + m;
}

// Largest float x with (x e) w <= 1/2 in FP32 (e, w > 0), or 0 when it is not found near 0.5 / (e w).
// (x e) w does not decrease with x, so |x| <= the result is that test, exactly.
__device__ __forceinline__ float half_extent(float e, float w) {
    float x = 0.5f / (e * w);
    for (int i = 0; i < 32; ++i) {
        const float up = __int_as_float(__float_as_int(x) + 1);
        if (__fmul_rn(__fmul_rn(x, e), w) > 0.5f) x = __int_as_float(__float_as_int(x) - 1);
        else if (__fmul_rn(__fmul_rn(up, e), w) <= 0.5f) x = up;
        else return x;
    }
    return 0.0f;
}

// An axis-aligned quad (unit normal along one axis, edges along the other two): returns 1 + the
// normal's axis and replaces uw, vw by the half extents along the lower and the higher edge axis, for
// quad_any_t's short test; 0 for any other quad, and for one whose plane the camera's eye is `near`.
template <class Near>
__device__ __forceinline__ int axis_quad(float3 n, float3 u, float3 v, float& uw, float& vw, const Near& near) {
    const float nn[3] = {n.x, n.y, n.z}, uu[3] = {u.x, u.y, u.z}, vv[3] = {v.x, v.y, v.z};
    int a = -1, b = -1, c = -1;
    float eu = 0.0f, ev = 0.0f;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        if ((nn[k] == 0.0f) + (uu[k] == 0.0f) + (vv[k] == 0.0f) != 2) continue;
        if (fabsf(nn[k]) == 1.0f) a = k;
        if (uu[k] != 0.0f) { b = k; eu = fabsf(uu[k]); }
        if (vv[k] != 0.0f) { c = k; ev = fabsf(vv[k]); }
    }
    if (a < 0 || b < 0 || c < 0) return 0;
    const float hu = half_extent(eu, uw), hv = half_extent(ev, vw);
    if (!(hu > 1e-30f && hu < 1e30f && hv > 1e-30f && hv < 1e30f) || near(a)) return 0;
    uw = b < c ? hu : hv;
    vw = b < c ? hv : hu;
    return 1 + a;
}

// ---------------------------------------------------------------------------
// k_instantiate: one CTA (kInstBlock threads) per render
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(kInstBlock) k_instantiate(const InstLaunch L) {
    __shared__ float s_u[4 * 32];
    __shared__ float s_red[kInstBlock];
    __shared__ float s_theta[kMaxD];
    __shared__ float s_scalar[2], s_tex[2];
    __shared__ int s_job;
    __shared__ __align__(16) BaseScene s_base;  // the job's base scene, staged once (int4 stores)
    __shared__ InstScene s_inst;  // render r's scene, built here and written out in one copy

    const int tid = threadIdx.x;
    // Before waiting on the previous kernel: only data the host wrote (job descriptors, the
    // base scene). Parameters, step counters and work counters come after the wait.
    if (tid == 0) {
        int j = 0;
        if (L.jobs) {
            int lo = 0, hi = L.njobs - 1;  // last job with block_begin <= blockIdx.x
            while (lo < hi) {
                const int mid = (lo + hi + 1) / 2;
                if (L.jobs[mid].block_begin <= (int)blockIdx.x) lo = mid; else hi = mid - 1;
            }
            j = lo;
        }
        s_job = j;
    }
    __syncthreads();
    const InstJob& J = L.jobs ? L.jobs[s_job] : L.job0;
    const int r = blockIdx.x - J.block_begin;
    const int D = J.D;
    {  // stage the base scene: all loads in flight at once, then the shared-memory stores
        constexpr int n16 = int(sizeof(BaseScene) / 16), n4 = int(sizeof(BaseScene) / 4);
        constexpr int kPer = (n16 + kInstBlock - 1) / kInstBlock;
        if (J.base && (reinterpret_cast<size_t>(J.base) & 15) == 0) {
            const int4* src = reinterpret_cast<const int4*>(J.base);
            int4* dst = reinterpret_cast<int4*>(&s_base);
            int4 v[kPer];
#pragma unroll
            for (int q = 0; q < kPer; ++q)
                if (tid + q * kInstBlock < n16) v[q] = __ldg(src + tid + q * kInstBlock);
#pragma unroll
            for (int q = 0; q < kPer; ++q)
                if (tid + q * kInstBlock < n16) dst[tid + q * kInstBlock] = v[q];
            for (int i = 4 * n16 + tid; i < n4; i += kInstBlock)
                reinterpret_cast<int*>(&s_base)[i] = __ldg(reinterpret_cast<const int*>(J.base) + i);
        } else if (J.base) {
            for (int i = tid; i < n4; i += kInstBlock)
                reinterpret_cast<int*>(&s_base)[i] = __ldg(reinterpret_cast<const int*>(J.base) + i);
        }
    }
    pdl_enter();
    if (blockIdx.x == 0 && tid == 0) {
        if (L.queue_reset) *L.queue_reset = 0u;
        if (L.queue_reset2) *L.queue_reset2 = 0u;
        if (L.queue_reset3) *L.queue_reset3 = 0u;
        if (L.queue_reset4) *L.queue_reset4 = 0u;
    }
    if (r == 0 && tid == 0 && J.queue_reset) *J.queue_reset = 0u;
    if (r == 0 && tid == 0 && J.share_reset)
        for (int i = 0; i < 4; ++i) J.share_reset[i] = 0u;
    if (tid == 0 && J.aff_cursor) J.aff_cursor[r] = 0u;
    if (J.aff_flags)  // this render's corrected-block bits, read by the last step's epilogue
        for (int i = tid; i < J.flag_words; i += kInstBlock) J.aff_flags[size_t(r) * J.flag_words + i] = 0u;
    const unsigned step = J.step + (J.step_dev ? (unsigned)*J.step_dev : 0u);
    const float theta_d = (tid < D && J.theta) ? J.theta[(J.render_mode ? r * D : 0) + tid] : 0.0f;
    __syncthreads();

    // ---- a1: perturbation and weight of render r --------------------------------
    // (texture scenes: the draws are made by the high-dimensional kernels, k_hd_*)
    const bool texscene = J.base && s_base.tex_mat >= 0;
    if (texscene) {
    } else if (J.render_mode) {
        if (tid < D) s_theta[tid] = theta_d;
    } else {
        const bool anti = J.antithetic && (r & 1);
        const unsigned index = (J.antithetic ? unsigned(r >> 1) : unsigned(r)) +
                               unsigned(J.antithetic ? J.pair_begin : 2 * J.pair_begin);
        const int nu = sampler_uniforms(J.sampler, D);
        const int nblk = (nu + 3) / 4;
        if (tid < nblk) {
            const uint4 w = philox(make_uint4(index, tid, step, kTagPerturb << 28), unsigned(J.seed),
                                   unsigned(J.seed >> 32));
            s_u[4 * tid + 0] = u01(w.x);
            s_u[4 * tid + 1] = u01(w.y);
            s_u[4 * tid + 2] = u01(w.z);
            s_u[4 * tid + 3] = u01(w.w);
        }
        __syncthreads();
        float tt = 0.0f, wt = 0.0f;  // unit-bandwidth tau~_d and w~_d of this thread's d
        if (J.sampler == kRadial && D == 1) {
            if (tid == 0) {
                const float rho = sqrtf(-2.0f * logf(s_u[0]));
                const float sg = (s_u[1] < 0.5f) ? -1.0f : 1.0f;
                tt = sg * rho;
                wt = sg * J.c_radial;
            }
        } else if (J.sampler == kRadial) {
            const int n_exp = (D + 1) / 2, extra = (D % 2 == 0);
            const float z = (tid < D) ? bm_normal(s_u, n_exp, tid) : 0.0f;
            // squared direction norm and chi^2_{D+1} radius, summed in a fixed order
            s_red[tid] = z * z;
            __syncthreads();
            if (tid == 0) {
                float zn = 0.0f;
                for (int d = 0; d < D; ++d) zn += s_red[d];
                float r2 = 0.0f;
                for (int j = 0; j < n_exp; ++j) r2 += -2.0f * logf(s_u[j]);
                if (extra) {  // one more degree of freedom when D + 1 is odd: normal number D
                    const float ze = bm_normal(s_u, n_exp, D);
                    r2 += ze * ze;
                }
                s_scalar[0] = sqrtf(zn);
                s_scalar[1] = r2;
            }
            __syncthreads();
            if (tid < D) {
                const float dir = z / s_scalar[0];
                tt = sqrtf(s_scalar[1]) * dir;
                wt = J.c_radial * dir;
            }
        } else if (J.sampler == kPerDim) {
            if (tid < D) {
                const float xi = s_u[tid];
                const float c1 = 0.7978845608028654f;  // sqrt(2/pi)
                if (xi < 0.5f) {
                    tt = -sqrtf(-2.0f * logf(2.0f * xi));
                    wt = -c1;
                } else {
                    tt = sqrtf(-2.0f * logf(2.0f * (1.0f - xi)));
                    wt = c1;
                }
            }
        } else {
            if (tid < D) {
                tt = bm_normal(s_u, 0, tid);
                wt = tt;
            }
        }
        if (tid < D) {
            const float sg = sigma_at(J, tid, (int)step);
            float tau = sg * tt;
            float w = wt / sg;
            if (anti) {
                tau = -tau;
                w = -w;
            }
            s_theta[tid] = theta_d + tau;  // FP32 sum: the parameters this render gets
            if (J.tau_out) J.tau_out[r * D + tid] = tau;
            if (J.w_out) J.w_out[r * D + tid] = w;
        }
    }
    __syncthreads();
    if (!J.scenes) return;  // draws only

    // ---- a2: bind theta_r into the scene -----------------------------------------
    const BaseScene& B = s_base;
    InstScene& S = s_inst;
    if (tid < kMaxDiff) {  // pathwise estimator: derivative of each parameter's clamp
        float dc = 0.0f;
        if (J.diff && !texscene && tid < D) {
            const float t = s_theta[tid];
            dc = B.bind_kind[tid] == kBindAlbedo ? ((t >= 0.0f && t <= 1.0f) ? 1.0f : 0.0f) : (t >= 0.0f ? 1.0f : 0.0f);
        }
        S.dclamp[tid] = dc;
    }
    if (tid < B.n_prims) {
        const int i = tid;
        const int type = B.prim_type[i], mat = B.prim_mat[i], slot = B.prim_slot[i];
        float g[9];
#pragma unroll
        for (int q = 0; q < 9; ++q) g[q] = B.prim_geom[i][q];
        for (int d = 0; d < (texscene ? 0 : D); ++d) {
            if (B.bind_index[d] != i) continue;
            if (B.bind_kind[d] == kBindPos) g[B.bind_comp[d]] = s_theta[d];
            if (B.bind_kind[d] == kBindRadius && type == kSphere) g[3] = fabsf(s_theta[d]);
        }
        float4* P = S.prim[slot];
        const float3 c = f3(g[0], g[1], g[2]);
        if (type == kSphere) {
            P[0] = make_float4(c.x, c.y, c.z, g[3]);
            P[1] = make_float4(g[3] * g[3], 1.0f / g[3], __int_as_float(mat), __int_as_float(i));
        } else if (type == kQuad) {
            const float3 u = f3(g[3], g[4], g[5]), v = f3(g[6], g[7], g[8]);
            const float3 uv = cross3(u, v);
            const float3 n = uv * rsqrtf(dot3(uv, uv));  // subnormal for |u x v| < 1.1e-19: not rsqrt_fast
            float uw = 1.0f / dot3(u, u), vw = 1.0f / dot3(v, v);
            bool plain = true;  // textured quads: the first keeps 1/(u.u), 1/(v.v) in the scene's header
            for (int k = 0; k < i && mat == B.tex_mat; ++k)
                plain = plain && !(B.prim_mat[k] == mat && B.prim_type[k] == kQuad);
            if (mat == B.tex_mat && plain) {
                s_tex[0] = uw;
                s_tex[1] = vw;
            }
            // The eye within 1e-6 of the quad's plane (see quad_any_t). Renders share the rows of a moving
            // quad that no binding changes, so one that moves along its normal is judged in forward
            // renders only.
            auto near = [&](int a) {
                if (!(fabsf(g[a] - B.eye[a]) < 1e-6f)) return false;
                for (int d = 0; d < B.D && !J.render_mode && B.tex_mat < 0; ++d)
                    if (B.bind_kind[d] == kBindPos && B.bind_index[d] == i && B.bind_comp[d] == a) return false;
                return true;
            };
            const int axis = plain ? axis_quad(n, u, v, uw, vw, near) : 0;
            P[0] = make_float4(c.x, c.y, c.z, __int_as_float(mat | (axis << 8)));
            P[1] = make_float4(n.x, n.y, n.z, __int_as_float(i));
            P[2] = make_float4(u.x, u.y, u.z, uw);
            P[3] = make_float4(v.x, v.y, v.z, vw);
        } else {
            P[0] = make_float4(g[0] - g[3], g[1] - g[4], g[2] - g[5], __int_as_float(mat));
            P[1] = make_float4(g[0] + g[3], g[1] + g[4], g[2] + g[5], __int_as_float(i));
        }
    }
    if (tid < B.n_mats) {
        const int i = tid;
        float p[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) p[q] = B.mat_param[i][q];
        for (int d = 0; d < (texscene ? 0 : D); ++d) {
            if (B.bind_index[d] != i) continue;
            if (B.bind_kind[d] == kBindAlbedo) p[B.bind_comp[d]] = s_theta[d];
            if (B.bind_kind[d] == kBindEmission) p[3 + B.bind_comp[d]] = s_theta[d];
        }
        for (int q = 0; q < 3; ++q) p[q] = fminf(fmaxf(p[q], 0.0f), 1.0f);
        for (int q = 3; q < 6; ++q) p[q] = fmaxf(p[q], 0.0f);
        S.mat[i][0] = make_float4(p[0], p[1], p[2], __int_as_float(B.mat_type[i]));
        S.mat[i][1] = make_float4(p[3], p[4], p[5], p[6]);
    }
    __syncthreads();
    if (J.var_box && tid < J.n_var) {  // path sharing: this render's bounds of a perturbed primitive
        const int i = J.var_prim[tid];
        float3 lo, hi;
        prim_bounds(static_cast<const float4*>(S.prim[B.prim_slot[i]]), B.prim_type[i], lo, hi);
        J.var_box[(size_t(r) * kMaxVariant + tid) * 2 + 0] = make_float4(lo.x, lo.y, lo.z, 0.0f);
        J.var_box[(size_t(r) * kMaxVariant + tid) * 2 + 1] = make_float4(hi.x, hi.y, hi.z, 0.0f);
    }
    if (tid == 32) {
        S.tex = texscene ? J.tex_all + size_t(r) * size_t(J.tex_D) : nullptr;
        S.tex_mat = texscene ? B.tex_mat : -1;
        S.tex_res = texscene ? B.tex_res : 0;
        S.n_sph = B.n_sph;
        S.n_quad = B.n_quad;
        S.n_box = B.n_box;
        const unsigned field =
            J.render_mode ? (J.crn ? 0u : unsigned(r)) : (J.crn ? 0u : unsigned(r + 1 + 2 * J.pair_begin));
        S.seed_lo = unsigned(J.seed);
        S.seed_hi = unsigned(J.seed >> 32);
        S.step = step;
        S.c3 = (J.tag << 28) | (field & 0x0fffffffu);
        S.eye = make_float4(B.eye[0], B.eye[1], B.eye[2], B.tan_half);
        S.fwd = make_float4(B.fwd[0], B.fwd[1], B.fwd[2], float(J.W) / float(J.H));
        S.right = make_float4(B.right[0], B.right[1], B.right[2], texscene ? s_tex[0] : 0.0f);
        S.up = make_float4(B.up[0], B.up[1], B.up[2], texscene ? s_tex[1] : 0.0f);
        S.bg = make_float4(B.bg[0], B.bg[1], B.bg[2], 0.0f);
    }
    if (tid < 32) {  // emitters, in primitive order: lane = primitive
        bool emits = false;
        int mat = 0;
        if (tid < B.n_prims) {
            mat = B.prim_mat[tid];
            const float4 e = S.mat[mat][1];
            emits = (e.x > 0.0f || e.y > 0.0f || e.z > 0.0f) && B.prim_type[tid] != kBox;
        }
        const unsigned m = __ballot_sync(kFull, emits);
        const int nl = __popc(m & ((1u << tid) - 1u));
        if (emits && nl < kMaxLights) {
            const int slot = B.prim_slot[tid];
            float area;
            if (B.prim_type[tid] == kQuad) {
                const float3 u = xyz(S.prim[slot][2]), v = xyz(S.prim[slot][3]);
                const float3 cr = cross3(u, v);
                area = sqrtf(dot3(cr, cr));
            } else {
                const float rad = S.prim[slot][0].w;
                area = 4.0f * 3.14159265358979f * rad * rad;
            }
            S.light[nl] = make_int4(B.prim_type[tid], slot, tid, mat);
            S.light_area[nl] = area;
        }
        if (tid == 0) S.n_lights = min(__popc(m), kMaxLights);
    }
    __syncthreads();
    {  // write out what the render kernels stage: header, used materials, used primitives
        const float4* src = reinterpret_cast<const float4*>(&s_inst);
        float4* dst = reinterpret_cast<float4*>(J.scenes + r);
        constexpr int kHead = int(offsetof(InstScene, mat) / 16);
        constexpr int kPrim = int(offsetof(InstScene, prim) / 16);
        const int nm = 2 * B.n_mats, np = 4 * B.n_prims;
        for (int i = tid; i < kHead + nm + np; i += kInstBlock) {
            const int o = (i < kHead + nm) ? i : kPrim + (i - kHead - nm);
            dst[o] = src[o];
        }
    }
}

// ---------------------------------------------------------------------------
// Ray casting against the shared-memory scene (brute force over <= 32 primitives)
// ---------------------------------------------------------------------------
// Work counters (only counted when the launch asks for them): primitive tests by
// type, camera paths, surface vertices, shadow rays, closest-hit rays.
constexpr int kNumCounters = 8;
struct Counters {
    unsigned sph, quad, box, paths, vertices, shadow, rays, pad;
};

// The intersection tests read a primitive record through P[j]: a pointer to its four float4,
// or a strided view of a per-render table (SRec).
template <class Rec>
__device__ __forceinline__ float sphere_t(const Rec& P, float3 o, float3 d) {
    const float4 a = P[0];
    const float r2 = P[1].x;
    const float3 oc = o - xyz(a);
    const float b = dot3(oc, d);
    const float3 l = oc - d * b;  // centre offset from the ray line: better conditioned than b^2 - c
    const float disc = r2 - dot3(l, l);
    if (!(disc > 0.0f)) return INFINITY;  // tangent rays (disc == 0) count as misses
    const float sq = disc * rsqrt_fast(disc);
    float t = -b - sq;
    if (t <= kEps) t = -b + sq;
    return (t > kEps) ? t : INFINITY;
}

template <class Rec>
__device__ __forceinline__ float quad_t(const Rec& P, float3 o, float3 d) {
    const float4 a = P[0], nb = P[1], uu = P[2], vv = P[3];
    const float3 n = xyz(nb);
    const float den = dot3(n, d);
    if (fabsf(den) < 1e-12f) return INFINITY;
    const float3 co = xyz(a) - o;
    const float t = div_fast(dot3(n, co), den);
    if (!(t > kEps)) return INFINITY;
    const float3 q = d * t - co;  // hit point relative to the centre
    const float pa = dot3(q, xyz(uu)) * uu.w, pb = dot3(q, xyz(vv)) * vv.w;
    return (fabsf(pa) <= 0.5f && fabsf(pb) <= 0.5f) ? t : INFINITY;
}

// A quad of either kind. An axis-aligned one (walls, floors, ceiling lights) needs no dot products:
// with n = +-e_a the plane distance is (c_a - o_a) / d_a, which is (c_a - o_a) rcp(d_a) in the
// approximate quotient's own terms, and each in-plane test compares one coordinate with the half
// extent; every rounding is that of quad_t, so the result is the same bit for bit. About 12
// instructions and one reciprocal per axis and ray instead of 38 and one per quad: four 512 x 512
// renders of the GI box at 32 spp 6.35 -> 6.06 ms, occlusion with independent samples 478 -> 468 us
// (together with div_fast and its kin).
// quad_t's bound on the cosine (1e-12) is left out: with a smaller one that is not zero, t > kEps
// needs a ray that starts within 1e-12 t of the plane but not in it. Points on surfaces lie kEps off
// parallel planes and anywhere beside the others; the camera's eye can lie so near, and then the
// quad takes the general test (k_instantiate). Testing the bound here costs 1 to 5 % (per quad: GI box
// 512 x 512, 32 renders 14.58 -> 15.03 ms, Eq. 9 on 256 x 256 walls 2.02 -> 2.10; per ray, with the
// reciprocal cleared: 14.91 and 2.10).
template <class Rec>
__device__ __forceinline__ float quad_any_t(const Rec& P, float3 o, float3 d, float3 inv) {
    const float4 a = P[0];
    const int axis = as_int(a.w) >> 8;
    if (axis) {
        const float3 co = xyz(a) - o;
        const bool ax = axis == 1, az = axis == 3;
        const float t = ax ? co.x * inv.x : (az ? co.z * inv.z : co.y * inv.y);
        const float qb = ax ? fmaf(d.y, t, -co.y) : fmaf(d.x, t, -co.x);
        const float qc = az ? fmaf(d.y, t, -co.y) : fmaf(d.z, t, -co.z);
        return (t > kEps && fabsf(qb) <= P[2].w && fabsf(qc) <= P[3].w) ? t : INFINITY;
    }
    return quad_t(P, o, d);
}

// Slab test; returns the nearest t > eps (entering, or leaving from inside).
template <class Rec>
__device__ __forceinline__ float box_t(const Rec& P, float3 o, float3 inv) {
    const float3 lo = xyz(P[0]), hi = xyz(P[1]);
    const float tx0 = (lo.x - o.x) * inv.x, tx1 = (hi.x - o.x) * inv.x;
    const float ty0 = (lo.y - o.y) * inv.y, ty1 = (hi.y - o.y) * inv.y;
    const float tz0 = (lo.z - o.z) * inv.z, tz1 = (hi.z - o.z) * inv.z;
    const float tn = fmaxf(fmaxf(fminf(tx0, tx1), fminf(ty0, ty1)), fminf(tz0, tz1));
    const float tf = fminf(fminf(fmaxf(tx0, tx1), fmaxf(ty0, ty1)), fmaxf(tz0, tz1));
    if (tn > tf) return INFINITY;
    if (tn > kEps) return tn;
    return (tf > kEps) ? tf : INFINITY;
}

// Outward normal of box record P at the hit found by box_t.
template <class Rec>
__device__ __forceinline__ float3 box_normal(const Rec& P, float3 o, float3 d, float3 inv) {
    const float3 lo = xyz(P[0]), hi = xyz(P[1]);
    float tn[3], tf[3];
    const float oo[3] = {o.x, o.y, o.z}, dd[3] = {d.x, d.y, d.z}, ii[3] = {inv.x, inv.y, inv.z};
    const float l3[3] = {lo.x, lo.y, lo.z}, h3[3] = {hi.x, hi.y, hi.z};
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const float t0 = (l3[a] - oo[a]) * ii[a], t1 = (h3[a] - oo[a]) * ii[a];
        tn[a] = fminf(t0, t1);
        tf[a] = fmaxf(t0, t1);
    }
    int an = 0, af = 0;
    float bn = tn[0], bf = tf[0];
#pragma unroll
    for (int a = 1; a < 3; ++a) {
        if (tn[a] > bn) { bn = tn[a]; an = a; }
        if (tf[a] < bf) { bf = tf[a]; af = a; }
    }
    const bool entering = bn > kEps;
    const int axis = entering ? an : af;
    const float s = (dd[axis] > 0.0f ? 1.0f : -1.0f) * (entering ? -1.0f : 1.0f);
    return f3(axis == 0 ? s : 0.0f, axis == 1 ? s : 0.0f, axis == 2 ? s : 0.0f);
}

struct Hit {
    float t;
    int slot;   // record slot, -1 = miss
    int type;
};

// Closest hit over all primitives, grouped by type. With kSkip, primitives whose
// record slot is set in `skip` are left out (the perturbed ones, in shared mode).
template <bool kCount, bool kSkip, class Scn>
__device__ __forceinline__ Hit closest_hit(const Scn& S, float3 o, float3 d, Counters& cnt, unsigned skip) {
    Hit h{INFINITY, -1, 0};
    const float3 inv = rcp3(d);
    const int ns = S.n_sph, nq = S.n_quad, nb = S.n_box;
    if (kCount) {
        const unsigned sk = kSkip ? skip : 0u;
        cnt.sph += ns - __popc(sk & ((1u << ns) - 1u));
        cnt.quad += nq - __popc((sk >> ns) & ((1u << nq) - 1u));
        cnt.box += nb - __popc((sk >> (ns + nq)) & ((1u << nb) - 1u));
        ++cnt.rays;
    }
#pragma unroll 1
    for (int i = 0; i < ns; ++i) {
        if (kSkip && ((skip >> i) & 1u)) continue;
        const float t = sphere_t(S.prim[i], o, d);
        if (t < h.t) { h.t = t; h.slot = i; h.type = kSphere; }
    }
#pragma unroll 1
    for (int i = ns; i < ns + nq; ++i) {
        if (kSkip && ((skip >> i) & 1u)) continue;
        const float t = quad_any_t(S.prim[i], o, d, inv);
        if (t < h.t) { h.t = t; h.slot = i; h.type = kQuad; }
    }
    if (nb) {
#pragma unroll 1
        for (int i = ns + nq; i < ns + nq + nb; ++i) {
            if (kSkip && ((skip >> i) & 1u)) continue;
            const float t = box_t(S.prim[i], o, inv);
            if (t < h.t) { h.t = t; h.slot = i; h.type = kBox; }
        }
    }
    return h;
}

// Is anything but primitive slot `light` (and, with kSkip, the slots in `skip`) hit
// closer than dist?
template <bool kCount, bool kSkip, class Scn>
__device__ __forceinline__ bool occluded(const Scn& S, float3 o, float3 d, float dist, int light,
                                         Counters& cnt, unsigned skip) {
    const float3 inv = rcp3(d);
    const int ns = S.n_sph, nq = S.n_quad, nb = S.n_box;
    if (kCount) ++cnt.shadow;
#pragma unroll 1
    for (int i = 0; i < ns; ++i) {
        if (i == light || (kSkip && ((skip >> i) & 1u))) continue;
        if (kCount) ++cnt.sph;
        if (sphere_t(S.prim[i], o, d) < dist) return true;
    }
#pragma unroll 1
    for (int i = ns; i < ns + nq; ++i) {
        if (i == light || (kSkip && ((skip >> i) & 1u))) continue;
        if (kCount) ++cnt.quad;
        if (quad_any_t(S.prim[i], o, d, inv) < dist) return true;
    }
    if (nb) {
#pragma unroll 1
        for (int i = ns + nq; i < ns + nq + nb; ++i) {
            if (i == light || (kSkip && ((skip >> i) & 1u))) continue;
            if (kCount) ++cnt.box;
            if (box_t(S.prim[i], o, inv) < dist) return true;
        }
    }
    return false;
}

// Render-group mode: the lanes of a warp trace the same path samples for up to 32
// renders of a job at once (with common random numbers the renders' paths agree until a
// perturbed primitive intervenes, so the lanes stay coherent). The invariant part of the
// scene is the warp's staged InstScene; each lane reads what differs between renders from
// its row of a per-warp table:
//   [0 .. n - 1]  the rows of the perturbed primitives' records that a position or radius
//                 binding changes (a quad's centre row; a sphere's and a box's two rows), in
//                 record-slot order; the other rows are the staged scene's
//   [n + j]       albedo row (albedo, type) of the j-th bound material (only albedos are bound
//                 in this mode; the emission row is the staged scene's)
//   [n + m .. + 1]  the render's emitter areas (8 floats), only when a radius binding can
//                 change an emitter's area (m = bound materials)
// A record in a per-render table kept field-major (field j of every render contiguous), so
// that lanes reading their own renders' fields load consecutive float4 without bank
// conflicts: row j at p[j * s] for the first n rows, in the staged scene's record for the others.
struct SRec {
    const float4* p;
    int s, n;
    const float4* base;
    __device__ __forceinline__ float4 operator[](int j) const { return *(j < n ? p + j * s : base + j); }
};

struct GroupLane {
    const float4* rec;  // this lane's row: field q at rec[q * rs]
    unsigned prims;     // record-slot mask of the perturbed primitives
    unsigned mats;      // mask of the bound materials
    unsigned offs;      // first field of the k-th perturbed primitive's own rows: bits 8 k .. 8 k + 7
    int var_rows;       // fields of all of them
    int areas;          // 1: the row holds the emitter areas
    const uint4* rng;   // the sample group's Philox blocks: [0] jitter, [1 + 2 b + k] vertex b, slot k
    int bpre;           // vertices b < bpre have their blocks in `rng`
    int rs;             // float4 between consecutive fields of a row (the table's render count)
};

// Record of primitive slot `slot`: the lane's own for a perturbed primitive, else the
// staged scene's.
template <bool kGroup, class Scn>
__device__ __forceinline__ auto prim_rec(const Scn& S, int slot, const GroupLane* g) {
    if constexpr (kGroup) {
        const bool quad = slot >= S.n_sph && slot < S.n_sph + S.n_quad;
        const int k = __popc(g->prims & ((1u << slot) - 1u));
        const bool own = (g->prims >> slot) & 1u;
        return SRec{g->rec + ((g->offs >> (8 * k)) & 255u) * g->rs, g->rs, own ? (quad ? 1 : 2) : 0, S.prim[slot]};
    } else {
        return static_cast<const float4*>(S.prim[slot]);
    }
}

// Albedo row (albedo, type) of material m: the lane's own for a bound material.
template <bool kGroup, class Scn>
__device__ __forceinline__ float4 mat_albedo(const Scn& S, int m, const GroupLane* g) {
    if constexpr (kGroup) {
        if ((g->mats >> m) & 1u) return g->rec[(g->var_rows + __popc(g->mats & ((1u << m) - 1u))) * g->rs];
    }
    return S.mat[m][0];
}

template <bool kGroup, class Scn>
__device__ __forceinline__ float light_area(const Scn& S, int li, const GroupLane* g) {
    if constexpr (kGroup) {
        if (g->areas)
            return reinterpret_cast<const float*>(g->rec + (g->var_rows + __popc(g->mats) + (li >> 2)) * g->rs)[li & 3];
    }
    return S.light_area[li];
}

// The lane's perturbed primitives against a ray: closer hits replace h (the staged scene's
// closest hit over the other primitives).
template <bool kCount, class Scn>
__device__ __forceinline__ void group_hit(const Scn& S, const GroupLane& g, float3 o, float3 d, Hit& h,
                                          Counters& cnt) {
    const float3 inv = rcp3(d);
    unsigned m = g.prims;
#pragma unroll 1
    for (unsigned offs = g.offs; m; offs >>= 8) {
        const int slot = __ffs(m) - 1;
        m &= m - 1u;
        const float4* own = g.rec + (offs & 255u) * g.rs;
        float t;
        int type;
        if (slot < S.n_sph) {
            t = sphere_t(SRec{own, g.rs, 2, S.prim[slot]}, o, d);
            type = kSphere;
            if (kCount) ++cnt.sph;
        } else if (slot < S.n_sph + S.n_quad) {
            t = quad_any_t(SRec{own, g.rs, 1, S.prim[slot]}, o, d, inv);
            type = kQuad;
            if (kCount) ++cnt.quad;
        } else {
            t = box_t(SRec{own, g.rs, 2, S.prim[slot]}, o, inv);
            type = kBox;
            if (kCount) ++cnt.box;
        }
        if (t < h.t) { h.t = t; h.slot = slot; h.type = type; }
    }
}

// Is one of the lane's perturbed primitives other than slot `light` hit closer than dist?
template <bool kCount, class Scn>
__device__ __forceinline__ bool group_occluded(const Scn& S, const GroupLane& g, float3 o, float3 d, float dist,
                                               int light, Counters& cnt) {
    const float3 inv = rcp3(d);
    unsigned m = g.prims;
#pragma unroll 1
    for (unsigned offs = g.offs; m; offs >>= 8) {
        const int slot = __ffs(m) - 1;
        m &= m - 1u;
        const float4* own = g.rec + (offs & 255u) * g.rs;
        if (slot == light) continue;
        float t;
        if (slot < S.n_sph) {
            t = sphere_t(SRec{own, g.rs, 2, S.prim[slot]}, o, d);
            if (kCount) ++cnt.sph;
        } else if (slot < S.n_sph + S.n_quad) {
            t = quad_any_t(SRec{own, g.rs, 1, S.prim[slot]}, o, d, inv);
            if (kCount) ++cnt.quad;
        } else {
            t = box_t(SRec{own, g.rs, 2, S.prim[slot]}, o, inv);
            if (kCount) ++cnt.box;
        }
        if (t < dist) return true;
    }
    return false;
}

// Union over the job's R renders of the perturbed primitives' bounds (shared mode; each
// render's bounds are inflated so that a slab test is conservative against the exact
// intersection tests), and the pool that keeps the segments touching them.
// One live path sample (Eq. 1's integrand along one path; Eq. 3 averages them).
struct Path {
    float3 o, d, beta, L;
    unsigned pixel;  // y * W + x
    int s, b;        // sample index, vertex index
    int slot;        // pixel slot inside the warp's block (per-render pass: the path's record)
    bool specular;   // emission counts: camera rays and rays after specular bounces
    unsigned seg;    // shared pass: touching-segment word (see note_touch)
};

struct VarBoxes {
    float4 lo[kMaxVariant], hi[kMaxVariant];  // union over renders
    float4* seg_pool;                         // touching segments, kSeg slots per path
    float4* seg_state;                        // 4 per path group: where the path's renders part
    unsigned* seg_ctr;                        // slots claimed
    unsigned seg_cap;                         // slots available
    int n;
    unsigned skip, mats;
};

// Does the segment o + t inv^-1, 0 <= t <= tm, touch the box [lo, hi]?
__device__ __forceinline__ bool slab_touch(float3 lo, float3 hi, float3 o, float3 inv, float tm) {
    const float tx0 = (lo.x - o.x) * inv.x, tx1 = (hi.x - o.x) * inv.x;
    const float ty0 = (lo.y - o.y) * inv.y, ty1 = (hi.y - o.y) * inv.y;
    const float tz0 = (lo.z - o.z) * inv.z, tz1 = (hi.z - o.z) * inv.z;
    const float tn = fmaxf(fmaxf(fminf(tx0, tx1), fminf(ty0, ty1)), fmaxf(fminf(tz0, tz1), 0.0f));
    const float tf = fminf(fminf(fmaxf(tx0, tx1), fmaxf(ty0, ty1)), fminf(fmaxf(tz0, tz1), tm));
    return tn <= tf;
}

// Touching segments of a shared-pass path. A path that touches a union box of the
// perturbed primitives claims a group g of kSeg segment slots and keeps, besides the
// segments, its state at the start of the vertex of the first touch: up to there none of
// its rays can meet a render's own primitive, so every render's path agrees with the
// shared one and the per-render pass resumes from that state instead of the camera.
// A path's segment word p.seg is
//   0                          no ray touched a union box;
//   (g + 1) << 3 | count       count <= kSeg touching segments (o, tmax), (d, 0) in slots
//                              kSeg g ..; a render traces the path again only if one of them
//                              touches that render's own bounds;
//   kSegAll | (g + 1) << 3     every render traces the path again from state g (a bound
//                              material was hit, or more than kSeg segments touched);
//   kSegFull                   every render traces the path again from the camera (the pool
//                              ran out before the first touch).
// State g: (o, d.x), (d.y, d.z, beta.x, beta.y), (beta.z, L), (vertex b, emission flag).
// A first touch by a shadow ray is kept as the vertex's state after its emission was
// added (o and d from the stash below), with the emission flag cleared so that the
// resumed vertex does not add it again.
constexpr unsigned kSegAll = 0x80000000u, kSegFull = 0xffffffffu;

// Ray (o, d) of each shared-pass thread's current vertex, kept while its path has not
// touched (a shadow ray's first touch records the vertex's state).
__shared__ float s_stash[6][kBlock];

template <bool kNee>
__device__ __forceinline__ unsigned open_group(const VarBoxes& V, const Path& p) {
    const unsigned base = atomicAdd(V.seg_ctr, unsigned(kSeg));
    if (base + unsigned(kSeg) > V.seg_cap) return kSegFull;
    const unsigned g = base / unsigned(kSeg);
    float3 o = p.o, d = p.d;
    if (kNee) {
        const int t = threadIdx.x;
        o = f3(s_stash[0][t], s_stash[1][t], s_stash[2][t]);
        d = f3(s_stash[3][t], s_stash[4][t], s_stash[5][t]);
    }
    float4* st = V.seg_state + 4 * size_t(g);
    st[0] = make_float4(o.x, o.y, o.z, d.x);
    st[1] = make_float4(d.y, d.z, p.beta.x, p.beta.y);
    st[2] = make_float4(p.beta.z, p.L.x, p.L.y, p.L.z);
    st[3] = make_float4(__int_as_float(p.b), __int_as_float((!kNee && p.specular) ? 1 : 0), 0.0f, 0.0f);
    return (g + 1u) << 3;
}

// Test the segment o + t d, 0 <= t <= tmax, of path p against the union boxes and keep it
// if it touches (kNee: a shadow ray). The caller returns kAffected once kSegAll is set.
template <bool kCount, bool kNee>
__device__ __forceinline__ void note_touch(const VarBoxes& V, float3 o, float3 d, float tmax, Path& p,
                                           Counters& cnt) {
    const float3 inv = rcp3(d);
    const float tm = tmax * 1.0001f + 1e-3f;
    bool hit = false;
    for (int k = 0; k < V.n; ++k) hit = hit || slab_touch(xyz(V.lo[k]), xyz(V.hi[k]), o, inv, tm);
    if (kCount) cnt.box += V.n;
    if (!hit) return;
    unsigned seg = p.seg;
    if (seg == 0u) {
        seg = open_group<kNee>(V, p);
        if (seg == kSegFull) {
            p.seg = kSegFull;
            return;
        }
    } else if ((seg & 7u) == unsigned(kSeg)) {
        p.seg = seg | kSegAll;
        return;
    }
    const size_t slot = size_t((seg >> 3) - 1u) * kSeg + (seg & 7u);
    V.seg_pool[2 * slot + 0] = make_float4(o.x, o.y, o.z, tmax);
    V.seg_pool[2 * slot + 1] = make_float4(d.x, d.y, d.z, 0.0f);
    p.seg = seg + 1u;
}

template <bool kOol = false, class Scn>
__device__ __forceinline__ uint4 path_words(const Scn& S, unsigned pixel, int s, int b, int slot) {
    const unsigned c1 = unsigned(s) | (unsigned(b) << 16) | (unsigned(slot) << 24);
    if constexpr (kOol) return philox_ool(make_uint4(pixel, c1, S.step, S.c3), S.seed_lo, S.seed_hi);
    return philox(make_uint4(pixel, c1, S.step, S.c3), S.seed_lo, S.seed_hi);
}

// Block `slot` of the path's current vertex: from the render group's table while the
// vertex is within it (the same words, drawn ahead by the group's lanes), else drawn here.
template <bool kGroup, bool kOol = false, class Scn>
__device__ __forceinline__ uint4 vertex_words(const Scn& S, const Path& p, int slot, const GroupLane* gl) {
    if constexpr (kGroup) {
        if (p.b < gl->bpre) return gl->rng[1 + 2 * p.b + slot];
    }
    return path_words<kOol>(S, p.pixel, p.s, p.b, slot);
}

// Orthonormal basis around unit n (Duff et al. 2017).
__device__ __forceinline__ void onb(float3 n, float3& t1, float3& t2) {
    const float sg = n.z >= 0.0f ? 1.0f : -1.0f;
    const float a = div_fast(-1.0f, sg + n.z);
    const float b = n.x * n.y * a;
    t1 = f3(1.0f + sg * n.x * n.x * a, sg * b, -sg * n.x);
    t2 = f3(b, sg + n.y * n.y * a, -n.y);
}

// Albedo of a textured quad at hit point pt: texel (floor(s T), floor(t T)) with
// s = (pt - c).u / |u|^2 + 1/2, t = (pt - c).v / |v|^2 + 1/2 (each clamped to [0, T-1]) of
// the render's texture [T][T][3]; channels clamped to [0, 1].
template <class Scn, class Rec>
__device__ __forceinline__ float3 tex_albedo(const Scn& S, const Rec& P, float3 pt) {
    const float4 c = P[0], u = P[2], v = P[3];
    const float3 l = pt - xyz(c);
    const bool axis = (as_int(c.w) >> 8) != 0;  // the record holds half extents, the header these
    const float uw = axis ? S.right.w : u.w, vw = axis ? S.up.w : v.w;
    const float s = fmaf(dot3(l, xyz(u)), uw, 0.5f), t = fmaf(dot3(l, xyz(v)), vw, 0.5f);
    const int T = S.tex_res;
    const int tx = min(max(int(floorf(s * float(T))), 0), T - 1);
    const int ty = min(max(int(floorf(t * float(T))), 0), T - 1);
    const float* q = S.tex + (size_t(ty) * T + tx) * 3;
    return f3(fminf(fmaxf(__ldg(q), 0.0f), 1.0f), fminf(fmaxf(__ldg(q + 1), 0.0f), 1.0f),
              fminf(fmaxf(__ldg(q + 2), 0.0f), 1.0f));
}

// Camera ray of sample s through pixel (x, y): pinhole, box-filtered jitter (slot 2). The
// jitter block is drawn here unless the caller passes it (`pre`).
template <bool kOol = false, class Scn>
__device__ __forceinline__ void start_path(const Scn& S, int W, int H, int x, int y, int s, int slot,
                                           Path& p, const uint4* pre = nullptr) {
    p.pixel = unsigned(y * W + x);
    const uint4 jw = pre ? *pre : path_words<kOol>(S, p.pixel, s, 0, 2);
    const float th = S.eye.w, aspect = S.fwd.w;
    const float sx = (float(2 * x - W) + 2.0f * u01(jw.x)) * div_fast(aspect * th, float(W));
    const float sy = (float(H - 2 * y) - 2.0f * u01(jw.y)) * div_fast(th, float(H));
    p.o = xyz(S.eye);
    p.d = normalized(xyz(S.fwd) + xyz(S.right) * sx + xyz(S.up) * sy);
    p.L = f3(0.f, 0.f, 0.f);
    p.beta = f3(1.f, 1.f, 1.f);
    p.s = s;
    p.b = 0;
    p.slot = slot;
    p.specular = true;
}

// One surface interaction of a path: unidirectional path tracing with next-event
// estimation on diffuse vertices. Returns kEnded when the path has ended.
// Random slots of vertex b: slot 0 = (light point u, v, BSDF u1, u2); slot 1 =
// (light choice, Russian roulette, dielectric choice), drawn only when needed.
//
// With kShared (path sharing across renders), the scene is the invariant part only. A
// render whose perturbed primitives no ray segment of the path can meet traces exactly
// this path, because all renders share its random numbers. Segments that touch a union
// box are kept (note_touch) for the per-render pass, which traces the path again in the
// renders whose own bounds a kept segment touches. A path that hits a material whose
// parameters are bound, or that every render must trace again, returns kAffected.
constexpr int kLive = 0, kEnded = 1, kAffected = 2;

// Forward-mode tangents of one path for the pathwise estimator (Eq. 9): dL[k] is the
// derivative of radiance channel c_k with respect to parameter k (an albedo or emission of
// material m_k), dB[k] that of the throughput's channel c_k. The path's discrete choices
// are held fixed and the Russian-roulette probability is a constant of the derivative,
// which keeps the derivative estimate unbiased as it keeps the radiance unbiased.
template <int kND>
struct Tangents {
    float dB[kND > 0 ? kND : 1], dL[kND > 0 ? kND : 1];
};

__device__ __forceinline__ float comp3(float3 v, int c) { return c == 0 ? v.x : (c == 1 ? v.y : v.z); }

template <int kND>
__device__ __forceinline__ void tan_reset(Tangents<kND>& t) {
#pragma unroll
    for (int k = 0; k < kND; ++k) t.dB[k] = t.dL[k] = 0.0f;
}

// L += beta * E (background or emitter seen on a camera or specular ray); E may be bound.
template <int kND, class Clamp>
__device__ __forceinline__ void tan_emit(Tangents<kND>& t, const TraceJob& J, const Clamp& dclamp, float3 beta,
                                         float3 E, int mat) {
#pragma unroll
    for (int k = 0; k < kND; ++k) {
        if (k >= J.diff_n) break;
        const int c = J.diff_comp[k];
        float d = t.dB[k] * comp3(E, c);
        if (J.diff_kind[k] == kBindEmission && J.diff_mat[k] == mat) d = fmaf(comp3(beta, c), dclamp[k], d);
        t.dL[k] += d;
    }
}

// L += beta * albedo * Le * g (next-event estimation at a vertex of material mat).
template <int kND, class Clamp>
__device__ __forceinline__ void tan_nee(Tangents<kND>& t, const TraceJob& J, const Clamp& dclamp, float3 beta,
                                        float3 albedo, int mat, float3 Le, int lmat, float g) {
#pragma unroll
    for (int k = 0; k < kND; ++k) {
        if (k >= J.diff_n) break;
        const int c = J.diff_comp[k];
        const float bc = comp3(beta, c), rc = comp3(albedo, c), ec = comp3(Le, c);
        float d = t.dB[k] * rc * ec;
        if (J.diff_kind[k] == kBindAlbedo && J.diff_mat[k] == mat) d = fmaf(bc * dclamp[k], ec, d);
        if (J.diff_kind[k] == kBindEmission && J.diff_mat[k] == lmat) d = fmaf(bc * rc, dclamp[k], d);
        t.dL[k] = fmaf(d, g, t.dL[k]);
    }
}

// beta <- beta * albedo (scattering at a vertex of material mat); beta is the old value.
template <int kND, class Clamp>
__device__ __forceinline__ void tan_scatter(Tangents<kND>& t, const TraceJob& J, const Clamp& dclamp, float3 beta,
                                            float3 albedo, int mat) {
#pragma unroll
    for (int k = 0; k < kND; ++k) {
        if (k >= J.diff_n) break;
        const int c = J.diff_comp[k];
        float d = t.dB[k] * comp3(albedo, c);
        if (J.diff_kind[k] == kBindAlbedo && J.diff_mat[k] == mat) d = fmaf(comp3(beta, c), dclamp[k], d);
        t.dB[k] = d;
    }
}

template <int kND>
__device__ __forceinline__ void tan_rr(Tangents<kND>& t, float inv_q) {
#pragma unroll
    for (int k = 0; k < kND; ++k) t.dB[k] *= inv_q;
}

// Next-event estimation at a diffuse vertex po with shading normal ns: emitter li chosen by
// slot 1's first word wl, a uniform point on it from slot 0's first two words (wx, wy).
// True, with the geometry term g (cosines over squared distance, times the emitter's area
// and count over pi) and the emitter's material, when the point is visible from po.
// Emitter of a next-event estimate: floor(u n) of slot 1's first word, exactly.
template <class Scn>
__device__ __forceinline__ int nee_light(const Scn& S, unsigned wl) {
    const int li = int((((wl >> 9) * 2u + 1u) * unsigned(S.n_lights)) >> 24);
    return min(li, S.n_lights - 1);
}

// Is one of the primitives whose record slots are set in `cand` hit closer than dist?
template <bool kCount, class Scn>
__device__ __forceinline__ bool occluded_set(const Scn& S, float3 o, float3 d, float dist, unsigned cand,
                                             Counters& cnt) {
    if (kCount) ++cnt.shadow;
    const int ns = S.n_sph, nsq = S.n_sph + S.n_quad;
    const float3 inv = rcp3(d);
#pragma unroll 1
    while (cand) {
        const int i = __ffs(cand) - 1;
        cand &= cand - 1u;
        float t;
        if (i < ns) {
            if (kCount) ++cnt.sph;
            t = sphere_t(S.prim[i], o, d);
        } else if (i < nsq) {
            if (kCount) ++cnt.quad;
            t = quad_any_t(S.prim[i], o, d, inv);
        } else {
            if (kCount) ++cnt.box;
            t = box_t(S.prim[i], o, inv);
        }
        if (t < dist) return true;
    }
    return false;
}

// The estimate toward emitter li at the point (lu, lv) of its parameterisation (see
// nee_visible).
template <bool kCount, bool kShared, bool kGroup, class Scn>
__device__ __forceinline__ bool nee_to(const Scn& S, float3 po, float3 ns, float lu, float lv, int li, Counters& cnt,
                                       unsigned skip, const GroupLane* gl, float3& wi, float& dist, float& g,
                                       int& lmat) {
    const int4 lt = S.light[li];
    const auto LP = prim_rec<kGroup>(S, lt.y, gl);
    float3 yl, ny;
    if (lt.x == kQuad) {
        const float3 uu = xyz(LP[2]), vv = xyz(LP[3]);
        yl = xyz(LP[0]) + uu * (lu - 0.5f) + vv * (lv - 0.5f);
        ny = xyz(LP[1]);
    } else {
        const float z = 1.0f - 2.0f * lu;
        const float rr2 = fmaxf(0.0f, 1.0f - z * z);
        const float rr_ = rr2 * rsqrt_fast(fmaxf(rr2, 1e-30f));
        float sp, cp;
        sincospif(2.0f * lv, &sp, &cp);
        ny = f3(rr_ * cp, rr_ * sp, z);
        yl = xyz(LP[0]) + ny * LP[0].w;
    }
    const float3 dv = yl - po;
    const float dist2 = dot3(dv, dv);
    const float inv_dist = rsqrt_fast(dist2);
    wi = dv * inv_dist;
    const float cx = dot3(ns, wi), cl = -dot3(ny, wi);
    if (!(cx > 0.0f && cl > 0.0f)) return false;
    dist = dist2 * inv_dist;
    bool blocked;
    if constexpr (kGroup) {  // skip: invariant primitives known not to meet the shadow ray
        const int np = S.n_sph + S.n_quad + S.n_box;
        const unsigned all = np >= 32 ? 0xffffffffu : (1u << np) - 1u;
        blocked = occluded_set<kCount>(S, po, wi, dist, all & ~(gl->prims | skip | (1u << lt.y)), cnt) ||
                  ((gl->prims & ~(1u << lt.y)) != 0u && group_occluded<kCount>(S, *gl, po, wi, dist, lt.y, cnt));
    } else {
        blocked = occluded<kCount, kShared>(S, po, wi, dist, lt.y, cnt, skip);
    }
    if (blocked) return false;
    g = cx * cl * (inv_dist * inv_dist) * light_area<kGroup>(S, li, gl) * float(S.n_lights) * 0.3183098861837907f;
    lmat = lt.w;
    return true;
}

template <bool kCount, bool kShared, bool kGroup, class Scn>
__device__ __forceinline__ bool nee_visible(const Scn& S, float3 po, float3 ns, unsigned wx, unsigned wy, unsigned wl,
                                            Counters& cnt, unsigned skip, const GroupLane* gl, float3& wi,
                                            float& dist, float& g, int& lmat) {
    return nee_to<kCount, kShared, kGroup>(S, po, ns, u01(wx), u01(wy), nee_light(S, wl), cnt, skip, gl, wi, dist, g,
                                          lmat);
}

// The radiance terms of a path: L + ba Le g (next-event estimation, ba = beta * albedo) and
// L + beta bg (a ray that leaves the scene).
__device__ __forceinline__ float3 nee_add(float3 L, float3 ba, float3 Le, float g) { return L + ba * Le * g; }
__device__ __forceinline__ float3 bg_add(float3 L, float3 beta, float3 bg) { return L + beta * bg; }

// Normal and material of the hit at pt (surfaces' own orientation).
template <class Rec>
__device__ __forceinline__ float3 surface_normal(const Rec& P, int type, float3 pt, float3 o, float3 d, int& mat) {
    float3 ng;
    if (type == kSphere) {
        const float4 a = P[0];
        ng = (pt - xyz(a)) * P[1].y;
        mat = as_int(P[1].z);
    } else if (type == kQuad) {
        ng = xyz(P[1]);
        mat = as_int(P[0].w) & 255;
    } else {
        ng = box_normal(P, o, d, rcp3(d));
        mat = as_int(P[0].w) & 255;
    }
    return ng;
}

// Cosine-distributed direction around ns (not normalised to the last bit).
__device__ __forceinline__ float3 diffuse_dir(float3 ns, float u1, float u2) {
    const float rad = u1 * rsqrt_fast(u1);
    float sp, cp;
    sincospif(2.0f * u2, &sp, &cp);
    float3 t1, t2;
    onb(ns, t1, t2);
    const float cz2 = fmaxf(0.0f, 1.0f - u1);
    return t1 * (rad * cp) + t2 * (rad * sp) + ns * (cz2 * rsqrt_fast(fmaxf(cz2, 1e-30f)));
}

// Smooth dielectric (exact unpolarised Fresnel): reflect or refract the path's ray at pt.
__device__ __forceinline__ void dielectric(Path& p, float3 pt, float3 ng, float ior, float u) {
    float ci = -dot3(p.d, ng);
    float eta;
    float3 n;
    if (ci > 0.0f) {
        eta = rcp_fast(ior);
        n = ng;
    } else {
        eta = ior;
        n = ng * -1.0f;
        ci = -ci;
    }
    const float s2t = eta * eta * (1.0f - ci * ci);
    float F, ct = 0.0f;
    if (s2t >= 1.0f) {
        F = 1.0f;
    } else {
        ct = sqrtf(1.0f - s2t);
        const float rs = div_fast(eta * ci - ct, eta * ci + ct);
        const float rp = div_fast(ci - eta * ct, ci + eta * ct);
        F = 0.5f * (rs * rs + rp * rp);
    }
    if (u < F) {
        p.d = normalized(p.d + n * (2.0f * ci));
        p.o = pt + n * kEps;
    } else {
        p.d = normalized(p.d * eta + n * (eta * ci - ct));
        p.o = pt - n * kEps;
    }
}

template <bool kCount, bool kShared, int kND = 0, bool kGroup = false, class Scn>
__device__ __forceinline__ int advance(const Scn& S, int depth, int rr_start, Path& p, Counters& cnt,
                                       const VarBoxes* V = nullptr, Tangents<kND>* tn = nullptr,
                                       const TraceJob* Jd = nullptr, const GroupLane* gl = nullptr) {
    if (kShared && p.seg == 0u) {
        const int t = threadIdx.x;
        s_stash[0][t] = p.o.x;
        s_stash[1][t] = p.o.y;
        s_stash[2][t] = p.o.z;
        s_stash[3][t] = p.d.x;
        s_stash[4][t] = p.d.y;
        s_stash[5][t] = p.d.z;
    }
    Hit h;
    if constexpr (kGroup) {  // the staged scene without the perturbed primitives, then the lane's own
        h = closest_hit<kCount, true>(S, p.o, p.d, cnt, gl->prims);
        group_hit<kCount>(S, *gl, p.o, p.d, h, cnt);
    } else {
        h = closest_hit<kCount, kShared>(S, p.o, p.d, cnt, kShared ? V->skip : 0u);
    }
    if (kShared) {
        note_touch<kCount, false>(*V, p.o, p.d, h.slot < 0 ? 3.0e38f : h.t, p, cnt);
        if (p.seg & kSegAll) return kAffected;
    }
    if (h.slot < 0) {
        if (kND > 0) tan_emit(*tn, *Jd, S.dclamp, p.beta, xyz(S.bg), -1);
        p.L = bg_add(p.L, p.beta, xyz(S.bg));
        return kEnded;
    }
    if (kCount) ++cnt.vertices;
    const float3 pt = p.o + p.d * h.t;
    const auto P = prim_rec<kGroup>(S, h.slot, gl);
    int mat;
    const float3 ng = surface_normal(P, h.type, pt, p.o, p.d, mat);
    if (kShared && ((V->mats >> mat) & 1u)) {  // every render from here (state: this vertex)
        p.seg = (p.seg == 0u ? open_group<false>(*V, p) : p.seg) | kSegAll;
        return kAffected;
    }
    const float4 m0 = mat_albedo<kGroup>(S, mat, gl), m1 = S.mat[mat][1];
    const int mtype = as_int(m0.w);
    const float3 emission = xyz(m1);
    float3 albedo = xyz(m0);
    if (mat == S.tex_mat && h.type == kQuad) albedo = tex_albedo(S, P, pt);
    if (p.specular && (emission.x > 0.f || emission.y > 0.f || emission.z > 0.f) && dot3(p.d, ng) < 0.0f) {
        if (kND > 0) tan_emit(*tn, *Jd, S.dclamp, p.beta, emission, mat);
        p.L = p.L + p.beta * emission;
    }
    const bool last = (p.b + 1 >= depth);
    const bool rr = !last && rr_start >= 0 && p.b >= rr_start;
    uint4 w1 = make_uint4(0u, 0u, 0u, 0u);
    if (mtype == kDiffuse) {
        const float3 ns = dot3(ng, p.d) < 0.0f ? ng : ng * -1.0f;
        const float3 po = pt + ns * kEps;
        const uint4 w0 = vertex_words<kGroup, kGroup>(S, p, 0, gl);
        if (S.n_lights > 1 || rr) w1 = vertex_words<kGroup, kGroup>(S, p, 1, gl);
        if (S.n_lights > 0) {  // next-event estimation: one emitter, uniform area sample
            float3 wi;
            float dist, g;
            int lmat;
            if (nee_visible<kCount, kShared, kGroup>(S, po, ns, w0.x, w0.y, w1.x, cnt, kShared ? V->skip : 0u, gl,
                                                     wi, dist, g, lmat)) {
                if (kShared) {
                    note_touch<kCount, true>(*V, po, wi, dist, p, cnt);
                    if (p.seg & kSegAll) return kAffected;
                }
                const float3 Le = xyz(S.mat[lmat][1]);
                if (kND > 0) tan_nee(*tn, *Jd, S.dclamp, p.beta, albedo, mat, Le, lmat, g);
                p.L = nee_add(p.L, p.beta * albedo, Le, g);
            }
        }
        if (last) return kEnded;
        const float3 wo = diffuse_dir(ns, u01(w0.z), u01(w0.w));
        if (kND > 0) tan_scatter(*tn, *Jd, S.dclamp, p.beta, albedo, mat);
        p.beta = p.beta * albedo;
        p.o = po;
        p.d = normalized(wo);
        p.specular = false;
    } else if (mtype == kMirror) {
        if (last) return kEnded;
        if (rr) w1 = vertex_words<kGroup, kGroup>(S, p, 1, gl);
        const float3 ns = dot3(ng, p.d) < 0.0f ? ng : ng * -1.0f;
        p.d = normalized(p.d - ns * (2.0f * dot3(p.d, ns)));
        p.o = pt + ns * kEps;
        if (kND > 0) tan_scatter(*tn, *Jd, S.dclamp, p.beta, albedo, mat);
        p.beta = p.beta * albedo;
        p.specular = true;
    } else {  // smooth dielectric: exact unpolarised Fresnel, reflect or refract
        if (last) return kEnded;
        w1 = vertex_words<kGroup, kGroup>(S, p, 1, gl);
        dielectric(p, pt, ng, m1.w, u01(w1.z));
        if (kND > 0) tan_scatter(*tn, *Jd, S.dclamp, p.beta, albedo, mat);
        p.beta = p.beta * albedo;
        p.specular = true;
    }
    if (maxc(p.beta) <= 0.0f) return kEnded;
    if (rr) {  // Russian roulette on slot 1's second uniform
        const float q = fminf(0.95f, maxc(p.beta));
        if (u01(w1.y) >= q) return kEnded;
        const float inv_q = rcp_fast(q);
        if (kND > 0) tan_rr(*tn, inv_q);
        p.beta = p.beta * inv_q;
    }
    ++p.b;
    return kLive;
}

// ---------------------------------------------------------------------------
// k_trace: persistent render + fused loss/gradient/Adam epilogue
// ---------------------------------------------------------------------------
constexpr int kWarps = kBlock / 32;
#ifndef PRDPT_TRACE_MIN_BLOCKS
#define PRDPT_TRACE_MIN_BLOCKS 3  // <= 85 registers: 24 resident warps per SM
#endif
constexpr int kTraceMinBlocks = PRDPT_TRACE_MIN_BLOCKS;
constexpr int kDiffMinBlocks = 5;  // pathwise-estimator CTAs of kDiffBlock threads: <= 102 registers
constexpr float kFix = 4294967296.0f;  // 2^32: fixed-point scale of the radiance accumulators

__device__ __forceinline__ double warp_sum_d(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
    return v;
}
__device__ __forceinline__ unsigned warp_sum_u(unsigned v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
    return v;
}

// n / d for d >= 1 given m = ceil(2^32 / d) (m wraps to 0 for d = 1).
__device__ __forceinline__ int div_magic(int n, int d, unsigned m) {
    return d == 1 ? n : int(__umulhi(unsigned(n), m));
}

// Radiance to fixed point (2^-32 units): integer sums are exact and independent of
// the order in which the warp's lanes finish their paths. The conversion is done
// on the significand bits (a float -> int64 conversion would run on the FP64 pipe):
// v * 2^32 = m * 2^(e + 9) for v = m * 2^(e - 23); values below 2^-9 are truncated.
__device__ __forceinline__ unsigned long long to_fixed(float v) {
    v = fminf(fmaxf(v, 0.0f), 2.0e9f);  // NaN -> 0
    const unsigned bits = __float_as_uint(v);
    const int e = int(bits >> 23) - 127;
    if (e < -32) return 0ull;
    const unsigned long long m = (bits & 0x7fffffu) | 0x800000u;
    const int sh = e + 9;
    return sh >= 0 ? (m << sh) : (m >> (-sh));
}

// Signed value to 2^-32 fixed point as a two's-complement 64-bit word (tangent sums).
__device__ __forceinline__ unsigned long long to_fixed_signed(float v) {
    return v >= 0.0f ? to_fixed(v) : 0ull - to_fixed(-v);
}

// Two's-complement 64-bit integer to float (magnitude split into 32-bit halves, so no
// 64-bit conversion instruction is needed); relative rounding error below 2^-23.
__device__ __forceinline__ float signed_word_to_float(long long D) {
    const unsigned long long m = D < 0 ? (unsigned long long)(-D) : (unsigned long long)D;
    const float f = fmaf(float(unsigned(m >> 32)), 4294967296.0f, float(unsigned(m)));
    return D < 0 ? -f : f;
}

// Squared error of one pixel against the target, summed over RGB (a4). The pixel's sums
// are 2^-32 fixed point over spp samples; acc - T * spp * 2^32 is formed exactly in 64-bit
// integers (T truncated to 2^-32), so the difference suffers no cancellation, and is then
// scaled to the mean and squared in FP32. Only the sums over pixels are FP64.
__device__ __forceinline__ float fixed_diff(unsigned long long a, float t, unsigned spp, float inv) {
    return signed_word_to_float((long long)(a - to_fixed(t) * (unsigned long long)spp)) * inv;
}

__device__ __forceinline__ double pixel_sq_error(unsigned long long ax, unsigned long long ay, unsigned long long az,
                                                 float4 T, unsigned spp, float inv) {
    const float dx = fixed_diff(ax, T.x, spp, inv), dy = fixed_diff(ay, T.y, spp, inv),
                dz = fixed_diff(az, T.z, spp, inv);
    return double(fmaf(dx, dx, fmaf(dy, dy, dz * dz)));
}

// 1 / (spp * 2^32): scale of a pixel's fixed-point sum to its mean.
__device__ __forceinline__ float mean_scale(int spp) { return 1.0f / (float(spp) * 4294967296.0f); }

// Per-warp shared-memory workspace of the render kernel.
struct WarpSmem {
    InstScene scene;                  // the render being traced (render 0 in shared phase A)
    TraceJob job;
    unsigned long long acc[3][32];    // radiance of the block's pixels, 2^-32 fixed point
    unsigned recorded;                // shared mode: the block has recorded paths
    VarBoxes vb;                      // shared mode: bounds of the perturbed primitives

};

// Copy render r's scene (header, used materials, used primitives) into a warp's slot.
__device__ __forceinline__ void stage_scene(InstScene& S, const TraceJob& J, int r, int lane) {
    const float4* src = reinterpret_cast<const float4*>(J.scenes + r);
    float4* dst = reinterpret_cast<float4*>(&S);
    constexpr int kHead = int(offsetof(InstScene, mat) / 16);
    constexpr int kPrim = int(offsetof(InstScene, prim) / 16);
    const int nm = 2 * J.n_mats, np = 4 * J.n_prims;
    for (int i = lane; i < kHead + nm + np; i += 32) {
        const int o = (i < kHead + nm) ? i : kPrim + (i - kHead - nm);
        dst[o] = __ldg(src + o);
    }
    __syncwarp();
}

// Union over the job's R renders of each perturbed primitive's bounds (shared mode).
__device__ void build_var_boxes(WarpSmem& W, const TraceJob& J, int lane) {
    for (int k = 0; k < J.n_var; ++k) {
        float3 lo = f3(INFINITY, INFINITY, INFINITY), hi = f3(-INFINITY, -INFINITY, -INFINITY);
        for (int r = lane; r < J.R; r += 32) {
            const float4* b = J.var_box + (size_t(r) * kMaxVariant + k) * 2;
            const float3 a = xyz(__ldg(b)), c = xyz(__ldg(b + 1));
            lo = f3(fminf(lo.x, a.x), fminf(lo.y, a.y), fminf(lo.z, a.z));
            hi = f3(fmaxf(hi.x, c.x), fmaxf(hi.y, c.y), fmaxf(hi.z, c.z));
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            lo.x = fminf(lo.x, __shfl_xor_sync(kFull, lo.x, o));
            lo.y = fminf(lo.y, __shfl_xor_sync(kFull, lo.y, o));
            lo.z = fminf(lo.z, __shfl_xor_sync(kFull, lo.z, o));
            hi.x = fmaxf(hi.x, __shfl_xor_sync(kFull, hi.x, o));
            hi.y = fmaxf(hi.y, __shfl_xor_sync(kFull, hi.y, o));
            hi.z = fmaxf(hi.z, __shfl_xor_sync(kFull, hi.z, o));
        }
        if (lane == 0) {
            W.vb.lo[k] = make_float4(lo.x, lo.y, lo.z, 0.f);
            W.vb.hi[k] = make_float4(hi.x, hi.y, hi.z, 0.f);
        }
    }
    if (lane == 0) {
        W.vb.seg_pool = J.seg_pool;
        W.vb.seg_state = J.seg_state;
        W.vb.seg_ctr = J.share_ctl + 2;
        W.vb.seg_cap = J.seg_cap;
        W.vb.n = J.n_var;
        W.vb.skip = J.var_prims;
        W.vb.mats = J.var_mats;
    }
    __syncwarp();
}

// a += v modulo 2^64 on a shared-memory word, as two native 32-bit atomics: the low
// word's carry (seen from the value it held before the add) goes into the high word.
// Concurrent adds give the exact sum whatever their order; the word is read only after
// every add has completed.
__device__ __forceinline__ void smem_add_u64(unsigned long long* a, unsigned long long v) {
    unsigned* w = reinterpret_cast<unsigned*>(a);  // little-endian: w[0] low, w[1] high
    const unsigned lo = unsigned(v), old = atomicAdd(w, lo);
    atomicAdd(w + 1, unsigned(v >> 32) + (old + lo < old ? 1u : 0u));
}

// k-th (0-based) set bit of m.
__device__ __forceinline__ int nth_set_bit(unsigned long long m, int k) {
    int pos = 0;
    unsigned x = unsigned(m);
    const int c = __popc(x);
    if (k >= c) {
        k -= c;
        x = unsigned(m >> 32);
        pos = 32;
    }
#pragma unroll
    for (int w = 16; w > 0; w >>= 1) {
        const int cw = __popc(x & ((1u << w) - 1u));
        if (k >= cw) {
            k -= cw;
            x >>= w;
            pos += w;
        }
    }
    return pos;
}

// Trace `ntasks` path tasks with the warp as a pool: each lane holds one live path and,
// when it ends, takes the next task (ballot + popc). decode(task, slot, sample) maps a
// task to its pixel slot and sample; every lane calls it (it may use warp shuffles).
// Ended paths add their radiance to acc[.][slot]. In shared mode a path that touched a
// perturbed primitive's union box is also recorded -- its code, segment word and
// shared-pass radiance -- in the job's list, and *recorded is set.
template <bool kCount, bool kShared, class Decode, int kND = 0, class Scn>
__device__ __forceinline__ void run_pool(const Scn& S, const TraceJob& J, int ntasks, int x0, int y0, int vw,
                                         unsigned magic_w, Decode decode, unsigned long long (&acc)[3][32],
                                         unsigned* recorded, const VarBoxes* V, Counters& cnt, int lane,
                                         unsigned long long (*dacc)[32] = nullptr) {
    const unsigned lt_mask = (1u << lane) - 1u;
    Path p;
    Tangents<kND> tn;
    bool alive = false, ended = true;  // every lane takes its first task at the first refill
    int next = 0, slot, smp;
    for (;;) {
        // lanes whose path ended take the next tasks, in lane order (one code site for the
        // first tasks and the later ones)
        const unsigned need = __ballot_sync(kFull, ended);
        const int mine = next + __popc(need & lt_mask);
        decode((ended && mine < ntasks) ? mine : 0, slot, smp);
        if (ended) {
            alive = mine < ntasks;
            if (alive) {
                const int row = div_magic(slot, vw, magic_w);
                start_path(S, J.W, J.H, x0 + slot - row * vw, y0 + row, smp, slot, p);
                if (kShared) p.seg = 0u;
                if (kND > 0) tan_reset(tn);
                if (kCount) ++cnt.paths;
            }
        }
        next += __popc(need);
        if (!__any_sync(kFull, alive)) break;
        int st = kLive;
        if (alive) st = advance<kCount, kShared, kND>(S, J.depth, J.rr_start, p, cnt, V, &tn, &J);
        ended = alive && st != kLive;
        // every ended path counts in the shared radiance; the per-render pass later adds,
        // for each render in a recorded path's mask, its own radiance minus this value
        if (ended) {
            smem_add_u64(&acc[0][p.slot], to_fixed(p.L.x));
            smem_add_u64(&acc[1][p.slot], to_fixed(p.L.y));
            smem_add_u64(&acc[2][p.slot], to_fixed(p.L.z));
#pragma unroll
            for (int k = 0; k < kND; ++k)  // tangents: signed fixed point, exact and order-free
                if (k < J.diff_n) smem_add_u64(&dacc[k][p.slot], to_fixed_signed(tn.dL[k]));
        }
        if (kShared) {  // record the paths some render must trace itself
            const bool rec = ended && p.seg != 0u;
            const unsigned am = __ballot_sync(kFull, rec);
            if (am) {
                unsigned base = 0;
                if (lane == __ffs(am) - 1) base = atomicAdd(J.share_ctl + 1, unsigned(__popc(am)));
                base = __shfl_sync(kFull, base, __ffs(am) - 1);
                if (rec) {
                    const unsigned e = base + __popc(am & lt_mask);
                    J.aff_codes[e] = (p.pixel << 6) | unsigned(p.s);
                    J.aff_segw[e] = p.seg;
                    J.aff_lsh[3 * size_t(e) + 0] = p.L.x;
                    J.aff_lsh[3 * size_t(e) + 1] = p.L.y;
                    J.aff_lsh[3 * size_t(e) + 2] = p.L.z;
                }
                if (lane == 0) *recorded = 1u;
            }
        }
    }
    __syncwarp();
}

// Pixel means of render r's block, then either the image (render mode) or the squared
// error and the block partial.
template <bool kRender>
__device__ __forceinline__ void block_epilogue(const TraceJob& J, int r, int t, const WarpSmem& W, int x0, int y0,
                                               int vw, int npx, int lane) {
    double e = 0.0;
    const int px = x0 + lane % vw, py = y0 + lane / vw;
    if (lane < npx && px < J.W && py < J.H) {
        const unsigned long long ax = W.acc[0][lane], ay = W.acc[1][lane], az = W.acc[2][lane];
        if (kRender) {
            const double inv = 1.0 / (double(J.spp) * double(kFix));
            J.images[(size_t(r) * J.H + py) * J.W + px] =
                make_float4(float(double(ax) * inv), float(double(ay) * inv), float(double(az) * inv), 0.0f);
        } else {
            e = pixel_sq_error(ax, ay, az, __ldg(J.target + size_t(py) * J.W + px), unsigned(J.spp),
                               mean_scale(J.spp));
        }
    }
    if (!kRender) {
        e = warp_sum_d(e);
        if (lane == 0) J.partials[size_t(r) * J.tiles + t] = e;  // a5: one partial per block
    }
    __syncwarp();
}

// The same squared error for all R renders of a block whose paths are all shared.
__device__ __forceinline__ void shared_block_epilogue(const TraceJob& J, int t, const WarpSmem& W, int x0, int y0,
                                                      int vw, int npx, int lane) {
    double e = 0.0;
    const int px = x0 + lane % vw, py = y0 + lane / vw;
    if (lane < npx && px < J.W && py < J.H) {
        e = pixel_sq_error(W.acc[0][lane], W.acc[1][lane], W.acc[2][lane], __ldg(J.target + size_t(py) * J.W + px),
                           unsigned(J.spp), mean_scale(J.spp));
    }
    e = warp_sum_d(e);
    for (int r = lane; r < J.R; r += 32) J.partials[size_t(r) * J.tiles + t] = e;
    __syncwarp();
}

// Pathwise estimator (Eq. 9): the block's loss partial as in block_epilogue, and for each
// parameter k the partial sum over its pixels of (I - T)_c dI_c/dtheta_k (c = c_k), where
// dI is the tangent sum divided by spp; the 2 / (3HW) factor is applied in k_finalize.
template <int kND>
__device__ __forceinline__ void diff_epilogue(const TraceJob& J, int r, int t, const unsigned long long (&acc)[3][32],
                                              const unsigned long long (*dacc)[32], int x0, int y0, int vw, int npx,
                                              int lane) {
    const int px = x0 + lane % vw, py = y0 + lane / vw;
    const bool ok = lane < npx && px < J.W && py < J.H;
    const float inv = mean_scale(J.spp);
    float3 res = f3(0.f, 0.f, 0.f);
    double e = 0.0;
    if (ok) {
        const float4 T = __ldg(J.target + size_t(py) * J.W + px);
        res = f3(fixed_diff(acc[0][lane], T.x, unsigned(J.spp), inv), fixed_diff(acc[1][lane], T.y, unsigned(J.spp), inv),
                 fixed_diff(acc[2][lane], T.z, unsigned(J.spp), inv));
        e = double(fmaf(res.x, res.x, fmaf(res.y, res.y, res.z * res.z)));
    }
    e = warp_sum_d(e);
    if (lane == 0) J.partials[size_t(r) * J.tiles + t] = e;
#pragma unroll
    for (int k = 0; k < kND; ++k) {
        if (k >= J.diff_n) break;
        double g = 0.0;
        if (ok) g = double(comp3(res, J.diff_comp[k]) * (signed_word_to_float((long long)dacc[k][lane]) * inv));
        g = warp_sum_d(g);
        if (lane == 0) J.gpartials[(size_t(r) * J.tiles + t) * J.diff_n + k] = g;
    }
    __syncwarp();
}

// kShare: every item is a pixel block of all renders of a path-sharing job (single-job
// launches only); otherwise every item is one render's block and job.share is ignored.
// kND > 0: the pathwise estimator (Eq. 9) with tangents of up to kND parameters, in CTAs
// of kDiffBlock threads (room for the per-pixel tangent sums in shared memory).
template <bool kRender, bool kCount, bool kShare, int kND>
__global__ void __launch_bounds__(kND > 0 ? kDiffBlock : kBlock, kND > 0 ? kDiffMinBlocks : kTraceMinBlocks)
    k_trace(const __grid_constant__ TraceLaunch L) {
    constexpr int kW = (kND > 0 ? kDiffBlock : kBlock) / 32;
    __shared__ WarpSmem s_warp[kW];
    __shared__ unsigned long long s_dacc[kND > 0 ? kW : 1][kND > 0 ? kND : 1][32];

    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    WarpSmem& W = s_warp[warp];
    const TraceJob& J = W.job;
    int cur_job = -1, cur_r = -1;
    Counters cnt{0u, 0u, 0u, 0u, 0u, 0u, 0u, 0u};
    if (!L.jobs) {  // a single job's descriptor is host data: copied before the wait
        const unsigned* src = reinterpret_cast<const unsigned*>(&L.job0);
        unsigned* dst = reinterpret_cast<unsigned*>(&W.job);
        for (int i = lane; i < int(sizeof(TraceJob) / 4); i += 32) dst[i] = src[i];
        __syncwarp();
    }
    pdl_enter();
    if (!L.jobs) {
        if (kShare) build_var_boxes(W, J, lane);  // the renders' bounds: written by k_instantiate
        cur_job = 0;
    }

    for (;;) {
        // ---- pop one work item for this warp --------------------------------------
        unsigned item = 0;
        int j = 0;
        if (lane == 0) {
            item = atomicAdd(L.queue, 1u);
            if (item < unsigned(L.total_items) && L.jobs) {
                int lo = 0, hi = L.njobs - 1;
                while (lo < hi) {
                    const int mid = (lo + hi + 1) / 2;
                    if (L.jobs[mid].item_begin <= int(item)) lo = mid; else hi = mid - 1;
                }
                j = lo;
            }
        }
        item = __shfl_sync(kFull, item, 0);
        if (item >= unsigned(L.total_items)) break;
        j = __shfl_sync(kFull, j, 0);
        if (j != cur_job) {
            const unsigned* src = reinterpret_cast<const unsigned*>(L.jobs ? L.jobs + j : &L.job0);
            unsigned* dst = reinterpret_cast<unsigned*>(&W.job);
            for (int i = lane; i < int(sizeof(TraceJob) / 4); i += 32) dst[i] = src[i];
            __syncwarp();
            if (kShare) build_var_boxes(W, J, lane);
            cur_job = j;
            cur_r = -1;
        }
        const int li = int(item) - J.item_begin;
        const int r = kShare ? 0 : li % J.R;  // render-interleaved: neighbouring items share pixels
        const int t = kShare ? li : li / J.R;
        if (r >= J.R || t >= J.tiles) {
            if (lane == 0) atomicOr(L.status, kStatusBadItem);
            break;
        }
        if (r != cur_r) {  // a2 -> shared memory
            stage_scene(W.scene, J, r, lane);
            cur_r = r;
        }

        // ---- block geometry and task decoding ------------------------------------------
        const int x0 = (t % J.tiles_x) * J.bw, y0 = (t / J.tiles_x) * J.bh;
        const int vw = min(J.bw, J.W - x0), vh = min(J.bh, J.H - y0);
        const int npx = vw * vh, ntasks = npx * J.spp;
        // task -> (pixel slot, sample) by multiply-high with m = ceil(2^32 / d): exact for
        // n < 2^32 / d (here n < 2^21, d <= 32); d = 1 has no 32-bit m and is special-cased
        const unsigned magic = 0xffffffffu / unsigned(npx) + 1u, magic_w = 0xffffffffu / unsigned(vw) + 1u;
        auto dense = [&](int task, int& slot, int& smp) {
            smp = div_magic(task, npx, magic);
            slot = task - smp * npx;
        };
        W.acc[0][lane] = 0ull;
        W.acc[1][lane] = 0ull;
        W.acc[2][lane] = 0ull;
        __syncwarp();

        if (!kShare && kND > 0) {
            // ---- pathwise estimator: radiance and tangents of every pixel x sample ----------
#pragma unroll
            for (int k = 0; k < (kND > 0 ? kND : 1); ++k) s_dacc[warp][k][lane] = 0ull;
            __syncwarp();
            run_pool<kCount, false, decltype(dense), kND>(W.scene, J, ntasks, x0, y0, vw, magic_w, dense, W.acc,
                                                          nullptr, nullptr, cnt, lane, s_dacc[warp]);
            diff_epilogue<kND>(J, r, t, W.acc, s_dacc[warp], x0, y0, vw, npx, lane);
            continue;
        }
        if (!kShare) {
            // ---- a3: every pixel x sample of this render ----------------------------------
            run_pool<kCount, false>(W.scene, J, ntasks, x0, y0, vw, magic_w, dense, W.acc, nullptr, nullptr, cnt,
                                    lane);
            block_epilogue<kRender>(J, r, t, W, x0, y0, vw, npx, lane);  // a4/a5
            continue;
        }

        // ---- shared pass: every path once in the invariant scene ---------------------------
        if (lane == 0) W.recorded = 0u;
        __syncwarp();
        run_pool<kCount, true>(W.scene, J, ntasks, x0, y0, vw, magic_w, dense, W.acc, &W.recorded, &W.vb, cnt, lane);
        if (W.recorded == 0u) {  // every path is shared by all renders
            shared_block_epilogue(J, t, W, x0, y0, vw, npx, lane);
            continue;
        }
        // some paths differ between renders: keep the shared radiance for the epilogue pass
        // and list the block; its affected paths are already in the job's list
        unsigned long long* dst = J.share_acc + size_t(t) * 96;
        dst[lane] = W.acc[0][lane];
        dst[32 + lane] = W.acc[1][lane];
        dst[64 + lane] = W.acc[2][lane];
        if (lane == 0) J.aff_tiles[atomicAdd(J.share_ctl + 0, 1u)] = t;
        __syncwarp();
    }
    if (kCount) {
        const unsigned v[kNumCounters] = {warp_sum_u(cnt.sph), warp_sum_u(cnt.quad), warp_sum_u(cnt.box),
                                          warp_sum_u(cnt.paths), warp_sum_u(cnt.vertices), warp_sum_u(cnt.shadow),
                                          warp_sum_u(cnt.rays), 0u};
        if (lane == 0)
            for (int i = 0; i < kNumCounters; ++i) atomicAdd(L.counters + i, (unsigned long long)v[i]);
    }
}

// ---------------------------------------------------------------------------
// k_trace_group: render-group variant of the per-render kernel (a3-a5)
// ---------------------------------------------------------------------------
// A work item is (pixel block t, render group g): G = J.gsize consecutive renders of a
// job (G divides R; 32 / G lanes per render). Lane l traces render g G + (l mod G), and
// the 32 / G lanes of one render take the samples s = l / G, l / G + 32 / G, ... of the
// current pixel: all lanes follow one pixel, so with common random numbers the renders'
// paths agree until a perturbed primitive intervenes and the warp stays coherent. The
// block's pixels are taken in bit-reversed slot order and their squared errors summed
// pairwise in that order, which is the shuffle tree of the per-render kernel's epilogue:
// with the same block shape, the same integer pixel sums and the same FP32 path
// arithmetic, every partial is bit-identical to the per-render kernel's.
constexpr int kGroupTab = kGroupTabRows;  // float4 per warp for the group's per-render records
static_assert(offsetof(InstScene, light_area) % 16 == 0, "emitter areas are copied as two float4");

// The render-group kernel's staged scene: the fields of InstScene with arrays for at most
// kGroupPrims primitives and kGroupMats materials (the per-warp copy is then 1.9 KB instead
// of 3.4 KB, so more warps fit an SM). Its header is laid out as InstScene's.
struct __align__(16) GroupScene {
    int n_sph, n_quad, n_box, n_lights;
    unsigned seed_lo, seed_hi, step, c3;
    float4 eye, fwd, right, up, bg;
    int4 light[kMaxLights];
    float light_area[kMaxLights];
    float dclamp[kMaxDiff];
    const float* tex;
    int tex_mat, tex_res;
    float4 mat[kGroupMats][2];
    float4 prim[kGroupPrims][4];
};
static_assert(offsetof(GroupScene, light) == offsetof(InstScene, light) &&
                  offsetof(GroupScene, light_area) == offsetof(InstScene, light_area) &&
                  offsetof(GroupScene, tex) == offsetof(InstScene, tex) &&
                  offsetof(GroupScene, mat) == offsetof(InstScene, mat),
              "GroupScene's header must be laid out as InstScene's");

// Copy render r's scene (header, used materials, used primitives) into a warp's GroupScene
// (the job has at most kGroupPrims primitives and kGroupMats materials).
__device__ __forceinline__ void stage_group_scene(GroupScene& S, const TraceJob& J, int r, int lane) {
    const float4* src = reinterpret_cast<const float4*>(J.scenes + r);
    float4* dst = reinterpret_cast<float4*>(&S);
    constexpr int kHead = int(offsetof(InstScene, mat) / 16);
    constexpr int kPrimSrc = int(offsetof(InstScene, prim) / 16);
    constexpr int kPrimDst = int(offsetof(GroupScene, prim) / 16);
    const int nm = 2 * J.n_mats, np = 4 * J.n_prims;
    for (int i = lane; i < kHead + nm + np; i += 32) {
        const bool is_prim = i >= kHead + nm;
        const int o = is_prim ? i - kHead - nm : i;
        dst[is_prim ? kPrimDst + o : o] = __ldg(src + (is_prim ? kPrimSrc + o : o));
    }
    __syncwarp();
}

struct GroupSmem {
    GroupScene scene;  // the invariant part (render g G's records of the other primitives)
    TraceJob job;
    float4 tab[kGroupTab];
    double pair[5][32];  // each lane's pairwise-sum stack (touched once per pixel)
    unsigned long long acc[3][32];  // each lane's radiance sums of the current pixel, 2^-32 fixed point
    uint4 rng[32];  // each sample group's Philox blocks of its current path (G per group)
};

#ifndef PRDPT_GROUP_MIN_BLOCKS
#define PRDPT_GROUP_MIN_BLOCKS 6  // 128-thread CTAs, <= 85 registers: 24 resident warps per SM
#endif
constexpr int kGroupMinBlocks = PRDPT_GROUP_MIN_BLOCKS;

__device__ __forceinline__ int brev5(int q) { return int(__brev(unsigned(q)) >> 27); }

// Pairwise sum over 32 values pushed in order: level l of the stack (s[l][lane]) holds a
// completed subtree of 2^l values; value q merges with levels 0, 1, ... while bit l of q is
// set. After the 32nd push the result is the total, summed as ((v0 + v1) + (v2 + v3)) + ...
__device__ __forceinline__ double pairwise_push(int q, double v, double (*s)[32], int lane) {
    int l = 0;
    for (; (q >> l) & 1; ++l) v = s[l][lane] + v;
    if (l < 5) s[l][lane] = v;
    return v;
}

template <bool kCount>
__global__ void __launch_bounds__(kGroupBlock, kGroupMinBlocks) k_trace_group(const __grid_constant__ TraceLaunch L) {
    __shared__ GroupSmem s_grp[kGroupBlock / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    GroupSmem& W = s_grp[warp];
    const TraceJob& J = W.job;
    int cur_job = -1, cur_item_g = -1;
    Counters cnt{0u, 0u, 0u, 0u, 0u, 0u, 0u, 0u};
    if (!L.jobs) {  // a single job's descriptor is host data: copied before the wait
        const unsigned* src = reinterpret_cast<const unsigned*>(&L.job0);
        unsigned* dst = reinterpret_cast<unsigned*>(&W.job);
        for (int i = lane; i < int(sizeof(TraceJob) / 4); i += 32) dst[i] = src[i];
        __syncwarp();
        cur_job = 0;
    }
    pdl_enter();
    for (;;) {
        unsigned item = 0;
        int j = 0;
        if (lane == 0) {
            item = atomicAdd(L.queue, 1u);
            if (item < unsigned(L.total_items) && L.jobs) {
                int lo = 0, hi = L.njobs - 1;
                while (lo < hi) {
                    const int mid = (lo + hi + 1) / 2;
                    if (L.jobs[mid].item_begin <= int(item)) lo = mid; else hi = mid - 1;
                }
                j = lo;
            }
        }
        item = __shfl_sync(kFull, item, 0);
        if (item >= unsigned(L.total_items)) break;
        j = __shfl_sync(kFull, j, 0);
        if (j != cur_job) {
            const unsigned* src = reinterpret_cast<const unsigned*>(L.jobs ? L.jobs + j : &L.job0);
            unsigned* dst = reinterpret_cast<unsigned*>(&W.job);
            for (int i = lane; i < int(sizeof(TraceJob) / 4); i += 32) dst[i] = src[i];
            __syncwarp();
            cur_job = j;
            cur_item_g = -1;
        }
        const int G = J.gsize, ngr = J.R / G, stride = J.gstride;
        const int li = int(item) - J.item_begin;
        const int g = li % ngr, t = li / ngr;  // group-interleaved: neighbouring items share pixels
        if (G < 1 || G > 32 || (32 % G) != 0 || t >= J.tiles || G * stride > kGroupTab || J.n_prims > kGroupPrims ||
            J.n_mats > kGroupMats) {
            if (lane == 0) atomicOr(L.status, kStatusBadItem);
            break;
        }
        if (g != cur_item_g) {  // stage render g G's scene and the group's per-render records
            stage_group_scene(W.scene, J, g * G, lane);
            const int n = J.var_rows, nm = __popc(J.var_mats);
            for (int i = lane; i < G * stride; i += 32) {
                const int gi = i / stride, q = i - gi * stride;
                const InstScene& R = J.scenes[g * G + gi];
                float4 v;
                if (q < n) {  // own row of a perturbed primitive
                    v = __ldg(&R.prim[J.row_src[q] >> 1][J.row_src[q] & 1]);
                } else if (q < n + nm) {  // albedo row of a bound material
                    v = __ldg(&R.mat[nth_set_bit(J.var_mats, q - n)][0]);
                } else {  // emitter areas
                    v = __ldg(reinterpret_cast<const float4*>(R.light_area) + (q - n - nm));
                }
                W.tab[q * G + gi] = v;  // field-major: the lanes' loads of one field are contiguous
            }
            __syncwarp();
            cur_item_g = g;
        }
        const int gi = lane % G, ks = lane / G, nsg = 32 / G;  // render in group, sample group, groups
        // Under common random numbers the G renders of a path sample draw the same Philox
        // blocks, so the group's lanes draw them ahead, one block each: the jitter and
        // slots 0 and 1 of vertices b < bpre.
        const int bpre = (G - 1) >> 1;
        const GroupLane gl{W.tab + gi, J.var_prims, J.var_mats, J.var_offs, J.var_rows,
                           stride > J.var_rows + __popc(J.var_mats) ? 1 : 0, W.rng + ks * G, bpre, G};
        const unsigned gmask = G == 32 ? kFull : ((1u << G) - 1u) << (ks * G);
        const int x0 = (t % J.tiles_x) * J.bw, y0 = (t / J.tiles_x) * J.bh;
        const int vw = min(J.bw, J.W - x0), vh = min(J.bh, J.H - y0);
        const int npx = vw * vh;
        const unsigned magic_w = 0xffffffffu / unsigned(vw) + 1u;
        const float inv = mean_scale(J.spp);
        double part = 0.0;
        for (int q = 0; q < 32; ++q) {
            const int slot = brev5(q);  // pixels in bit-reversed slot order (see above)
            double e = 0.0;
            if (slot < npx) {
                const int row = div_magic(slot, vw, magic_w);
                const int px = x0 + slot - row * vw, py = y0 + row;
                W.acc[0][lane] = 0ull;
                W.acc[1][lane] = 0ull;
                W.acc[2][lane] = 0ull;
                for (int smp = ks; smp < J.spp; smp += nsg) {
                    __syncwarp(gmask);  // the group's lanes are done with the previous path's blocks
                    if (gi == 0 || gi <= 2 * bpre)
                        W.rng[lane] = path_words(W.scene, unsigned(py * J.W + px), smp, gi == 0 ? 0 : (gi - 1) >> 1,
                                                 gi == 0 ? 2 : (gi - 1) & 1);
                    __syncwarp(gmask);
                    Path p;
                    start_path(W.scene, J.W, J.H, px, py, smp, slot, p, gl.rng);
                    if (kCount) ++cnt.paths;
                    while (advance<kCount, false, 0, true>(W.scene, J.depth, J.rr_start, p, cnt, nullptr, nullptr,
                                                          nullptr, &gl) == kLive) {
                    }
                    W.acc[0][lane] += to_fixed(p.L.x);
                    W.acc[1][lane] += to_fixed(p.L.y);
                    W.acc[2][lane] += to_fixed(p.L.z);
                }
                unsigned long long a0 = W.acc[0][lane], a1 = W.acc[1][lane], a2 = W.acc[2][lane];
                for (int o = G; o < 32; o <<= 1) {  // the render's other sample groups
                    a0 += __shfl_xor_sync(kFull, a0, o);
                    a1 += __shfl_xor_sync(kFull, a1, o);
                    a2 += __shfl_xor_sync(kFull, a2, o);
                }
                e = pixel_sq_error(a0, a1, a2, __ldg(J.target + size_t(py) * J.W + px), unsigned(J.spp), inv);
            }
            part = pairwise_push(q, e, W.pair, lane);
        }
        if (ks == 0) J.partials[size_t(g * G + gi) * J.tiles + t] = part;  // a5: one partial per block
        __syncwarp();
    }
    if (kCount) {
        const unsigned v[kNumCounters] = {warp_sum_u(cnt.sph), warp_sum_u(cnt.quad), warp_sum_u(cnt.box),
                                          warp_sum_u(cnt.paths), warp_sum_u(cnt.vertices), warp_sum_u(cnt.shadow),
                                          warp_sum_u(cnt.rays), 0u};
        if (lane == 0)
            for (int i = 0; i < kNumCounters; ++i) atomicAdd(L.counters + i, (unsigned long long)v[i]);
    }
}

// Replay mode (k_trace_replay): a path is traced once in the invariant scene for all renders.
// What is the same in every render -- the path up to its first event that can differ -- is its
// lane's own radiance; from there on the path is recorded as a chain of groups of entries (one
// group per vertex) in a per-warp pool of float4 granules, which every render replays with its
// own primitives and albedos. The first granule's w is the entry's info word:
//   bits 0-1 kind, 16: last entry of its group
//   kVert      a vertex: bits 2-3 the next-event estimate, 4 Russian roulette, 5-7 light, 8-11
//              material, 12-15 surface slot, 17 flipped normal, 18 normal kept in full, 19-31 the
//              estimate's cull mask. With bound materials (throughput replayed per render):
//                0 none                (-, u_rr, -, info)
//                1 perturbed emitter   (po, info) (light u, v, u_rr, -) [(ns, -)]: each render's
//                                      own point on it, occlusion and geometry term
//                2 fixed emitter       (g, u_rr, -, info): seen by every render
//                3 fixed emitter       (po, info) (wi, distance) (g, u_rr, -, -): the render's own
//                                      primitives may hide it
//              without: 1 (po, info) (ba, light u) (ns, light v), 2 (-, info) - (ba, g),
//              3 (po, info) (wi, distance) (ba, g), with ba = beta * albedo
//   kSegment   a ray that could meet a perturbed primitive: (o, info) (d, t) [(beta, -) without
//              bound materials], t the invariant scene's closest hit; bit 4 emission counts, 8-14
//              vertex index. A render whose own primitive is closer parts from the path here
//   kEmission  emission seen on a camera or specular ray: (beta, info), bits 8-11 material, 5 the
//              background
//   kPrefix    radiance (and throughput) before the first entry: (L, info) [(beta, -)]
enum : unsigned { kVert = 0u, kSegment = 1u, kEmission = 2u, kPrefix = 3u };
constexpr unsigned kLastEntry = 1u << 16;
constexpr int kNoEntry = 0xffff;  // end of a chain
constexpr int kCullBits = 13;

struct ReplayLane {
    const float4* ulo;   // union over the renders of each perturbed primitive's bounds
    const float4* uhi;
    const float4* amax;  // per bound material: the largest albedo over the renders
    const float4* ball;  // per record slot: an enclosing ball, inflated
    int n_var;
    unsigned skip;       // record slots of the perturbed primitives
    unsigned mats;       // bound materials
    float4* ent;         // the warp's pool
    unsigned short* nxt; // per group (its first granule): the chain's next group
    unsigned* ctr;       // granules claimed
    int cap;
    int first, last;     // this lane's chain
    bool rec;            // recording (the renders may differ from here on)
    bool varied;         // a bound material was met: p.beta is an upper bound over the renders
    bool full;           // the pool ran out: the path is traced again in a later batch
    bool cull;           // look for primitives that no render's shadow ray can meet (kMove 1, no bound materials)
};

// Enclosing ball of a primitive record, inflated beyond the FP32 rounding of its test.
__device__ __forceinline__ float4 prim_ball(const float4* P, int type) {
    float3 c;
    float rad;
    if (type == kSphere) {
        c = xyz(P[0]);
        rad = fabsf(P[0].w);
    } else if (type == kQuad) {
        const float3 u = xyz(P[2]), w = xyz(P[3]);
        c = xyz(P[0]);
        rad = 0.5f * (sqrtf(dot3(u, u)) + sqrtf(dot3(w, w)));
    } else {
        const float3 a = xyz(P[0]), b = xyz(P[1]), e = (b - a) * 0.5f;
        c = (a + b) * 0.5f;
        rad = sqrtf(dot3(e, e));
    }
    return make_float4(c.x, c.y, c.z, rad * 1.00001f + 1e-3f + 1e-5f * (fabsf(c.x) + fabsf(c.y) + fabsf(c.z)));
}

// Invariant primitives that no render's shadow ray from po to its emitter in record slot `slot`
// can meet, as a mask of the first kCullBits record slots: every such ray lies in the cone from
// po over the emitter's union bounds (centre b, half-diagonal rb: the ray to a point y deviates
// from the axis po -> b by at most t rb at parameter t). A primitive is left out when its
// enclosing ball keeps clear of that cone, or when a quad's plane has po and the whole union
// box strictly on one side. The margins exceed the FP32 rounding of the intersection tests and
// of the approximate roots and quotients here, so leaving these primitives out never changes a
// shadow ray's outcome.
template <class Lane>
__device__ __forceinline__ unsigned shadow_cull(const GroupScene& S, const Lane& E, float3 po, int slot) {
    const int k = __popc(E.skip & ((1u << slot) - 1u));
    const float3 lo = xyz(E.ulo[k]), hi = xyz(E.uhi[k]);
    const float3 bc = (lo + hi) * 0.5f, bh = (hi - lo) * 0.5f;
    const float bb = dot3(bh, bh), rb = bb * rsqrt_fast(bb) * 1.0001f;  // the bounds are inflated: bb > 0
    const float3 v = bc - po;
    const float vv = dot3(v, v);
    if (!(vv > 1e-12f)) return 0u;
    const float ilv = rsqrt_fast(vv) * 1.0001f, ivv = rcp_fast(vv);
    unsigned m = 0u;
    const int ns = S.n_sph, nq = S.n_quad, np = min(ns + nq + S.n_box, kCullBits);
#pragma unroll 1
    for (int i = 0; i < np; ++i) {
        if ((E.skip >> i) & 1u) continue;
        const float4 ball = E.ball[i];
        const float3 w = xyz(ball) - po;
        const float t0 = dot3(w, v) * ivv;
        const float3 q = w - v * fminf(fmaxf(t0, 0.0f), 1.0f);
        const float lim = ball.w + fmaxf(fminf(1.0f, t0 + (ball.w + rb) * ilv), 0.0f) * rb;
        bool clear = dot3(q, q) > lim * lim * 1.0001f;
        if (!clear && i >= ns && i < ns + nq) {
            const float4* P = S.prim[i];
            const float3 c = xyz(P[0]), n = xyz(P[1]), pc = po - c;
            const float pp = dot3(pc, pc), mg = 1.1e-5f + 2.1e-6f * pp * rsqrt_fast(fmaxf(pp, 1e-30f));
            const float sp = dot3(pc, n), sb = dot3(bc - c, n);
            const float eb = fabsf(n.x) * bh.x + fabsf(n.y) * bh.y + fabsf(n.z) * bh.z;
            clear = (sp > mg && sb - eb > mg) || (sp < -mg && sb + eb < -mg);
        }
        if (clear) m |= 1u << i;
    }
    return m;
}

// Does the segment o + t d, 0 <= t <= tmax, touch a union box of the perturbed primitives?
template <bool kCount, class Lane>
__device__ __forceinline__ bool replay_touch(const Lane& E, float3 o, float3 d, float tmax, Counters& cnt) {
    const float3 inv = rcp3(d);
    const float tm = tmax * 1.0001f + 1e-3f;
    bool hit = false;
#pragma unroll 1
    for (int k = 0; k < E.n_var; ++k) hit = hit || slab_touch(xyz(E.ulo[k]), xyz(E.uhi[k]), o, inv, tm);
    if (kCount) cnt.box += E.n_var;
    return hit;
}

// One vertex of a path of a replay job (as advance), recording what can differ between the
// renders. kMat: the job binds albedos; kMove: it perturbs primitives (1: every emitter is one).
template <bool kCount, bool kMat, int kMove>
__device__ __forceinline__ int replay_vertex(const GroupScene& S, int depth, int rr_start, Path& p, ReplayLane& E,
                                             Counters& cnt) {
    const Hit h = closest_hit<kCount, (kMove != 0)>(S, p.o, p.d, cnt, kMove ? E.skip : 0u);
    const bool miss = h.slot < 0;
    const bool touch = kMove && replay_touch<kCount>(E, p.o, p.d, miss ? 3.0e38f : h.t, cnt);
    bool rec = E.rec || touch, bound = false, last = true, rr = false;
    unsigned emis = 0u, vert = 0u;  // info words of the entries to record (emission: 0 none)
    int nvert = 0;                  // granules of the vertex entry
    float4 v0 = make_float4(0.f, 0.f, 0.f, 0.f), v1 = v0, v2 = v0;
    float3 pt = p.o, ng = p.d, ns = p.d, po = p.o, albedo = p.d;
    int mtype = kDiffuse;
    float ior = 1.0f;
    uint4 w0 = make_uint4(0u, 0u, 0u, 0u), w1 = w0;
    if (miss) {
        if (!rec) p.L = bg_add(p.L, p.beta, xyz(S.bg));
        else if (S.bg.x != 0.0f || S.bg.y != 0.0f || S.bg.z != 0.0f) emis = kEmission | 32u;
    } else {
        if (kCount) ++cnt.vertices;
        pt = p.o + p.d * h.t;
        int mat = 0;
        ng = surface_normal(static_cast<const float4*>(S.prim[h.slot]), h.type, pt, p.o, p.d, mat);
        const float4 m0 = S.mat[mat][0], m1 = S.mat[mat][1];
        mtype = as_int(m0.w);
        ior = m1.w;
        const float3 emission = xyz(m1);
        albedo = xyz(m0);
        if (p.specular && (emission.x > 0.f || emission.y > 0.f || emission.z > 0.f) && dot3(p.d, ng) < 0.0f) {
            if (rec) emis = kEmission | (unsigned(mat) << 8);
            else p.L = p.L + p.beta * emission;
        }
        if (kMat && ((E.mats >> mat) & 1u)) {
            bound = rec = true;
            albedo = xyz(E.amax[mat]);
        }
        last = p.b + 1 >= depth;
        rr = !last && rr_start >= 0 && p.b >= rr_start;
        const bool flip = !(dot3(ng, p.d) < 0.0f);
        ns = flip ? ng * -1.0f : ng;
        po = pt + ns * kEps;
        const bool diffuse = mtype == kDiffuse;
        if (diffuse) w0 = path_words<true>(S, p.pixel, p.s, p.b, 0);
        if (diffuse ? (S.n_lights > 1 || rr) : (!last && (rr || mtype == kDielectric)))
            w1 = path_words<true>(S, p.pixel, p.s, p.b, 1);
        const float urr = u01(w1.y);
        unsigned est = 0u;
        int li = 0;
        if (diffuse && S.n_lights > 0) {  // next-event estimation: one emitter, uniform area sample
            const float3 ba = p.beta * albedo;
            if (maxc(ba) > 0.0f || bound) {  // (a black vertex adds nothing, nor has it derivatives unless bound)
                li = nee_light(S, w1.x);
                const int lslot = S.light[li].y;
                const float lu = u01(w0.x), lv = u01(w0.y);
                if (kMove == 1 || (kMove && ((E.skip >> lslot) & 1u))) {  // each render's own estimate
                    est = 1u;
                    rec = true;
                    if (kMat || kMove != 1 || E.cull) vert = shadow_cull(S, E, po, lslot) << (32 - kCullBits);
                    v0 = make_float4(po.x, po.y, po.z, 0.f);
                    if (kMat) {
                        v1 = make_float4(lu, lv, urr, 0.f);
                        v2 = make_float4(ns.x, ns.y, ns.z, 0.f);
                        vert |= (flip ? 1u << 17 : 0u) | (h.type != kQuad ? 1u << 18 : 0u) | (unsigned(h.slot) << 12);
                        nvert = h.type != kQuad ? 3 : 2;
                    } else {
                        v1 = make_float4(ba.x, ba.y, ba.z, lu);
                        v2 = make_float4(ns.x, ns.y, ns.z, lv);
                        nvert = 3;
                    }
                } else {
                    float3 wi;
                    float dist, g;
                    int lmat;
                    if (nee_to<kCount, (kMove != 0), false>(S, po, ns, lu, lv, li, cnt, kMove ? E.skip : 0u, nullptr, wi, dist,
                                                     g, lmat)) {
                        const bool own = kMove && replay_touch<kCount>(E, po, wi, dist, cnt);
                        rec = rec || own;
                        if (!rec) {
                            p.L = nee_add(p.L, ba, xyz(S.mat[lmat][1]), g);
                        } else if (own) {
                            est = 3u;
                            v0 = make_float4(po.x, po.y, po.z, 0.f);
                            v1 = make_float4(wi.x, wi.y, wi.z, dist);
                            v2 = kMat ? make_float4(g, urr, 0.f, 0.f) : make_float4(ba.x, ba.y, ba.z, g);
                            nvert = 3;
                        } else {
                            est = 2u;
                            v0 = make_float4(g, urr, 0.f, 0.f);
                            v2 = make_float4(ba.x, ba.y, ba.z, g);
                            nvert = kMat ? 1 : 3;
                        }
                    }
                }
            }
        }
        if (kMat && rec && est == 0u) {
            v0 = make_float4(0.f, urr, 0.f, 0.f);
            nvert = 1;
        }
        vert |= kVert | (est << 2) | (rr ? 16u : 0u) | (unsigned(li) << 5) | (unsigned(mat) << 8);
    }
    // ---- record the vertex's group: prefix, segment, emission, vertex ------------------------
    const bool pre = rec && !E.rec &&
                     (p.L.x != 0.0f || p.L.y != 0.0f || p.L.z != 0.0f ||
                      (kMat && (p.beta.x != 1.0f || p.beta.y != 1.0f || p.beta.z != 1.0f)));
    const int npre = pre ? (kMat ? 2 : 1) : 0, nseg = touch ? (kMat ? 2 : 3) : 0;
    const int total = npre + nseg + (emis ? 1 : 0) + nvert;
    E.rec = rec;
    if (total) {
        int i = int(atomicAdd(E.ctr, unsigned(total)));
        if (unsigned(i) >= unsigned(E.cap) || i + total > E.cap) {
            E.full = true;
            return kEnded;
        }
        E.nxt[i] = (unsigned short)(kNoEntry);
        if (E.first == kNoEntry) E.first = i;
        else E.nxt[E.last] = (unsigned short)(i);
        E.last = i;
        const int end = i + total;
        if (pre) {
            E.ent[i] = make_float4(p.L.x, p.L.y, p.L.z, __uint_as_float(kPrefix | (i + npre == end ? kLastEntry : 0u)));
            if (kMat) E.ent[i + 1] = make_float4(p.beta.x, p.beta.y, p.beta.z, 0.f);
            i += npre;
        }
        if (kMove && touch) {
            const unsigned info = kSegment | (p.specular ? 16u : 0u) | (unsigned(p.b) << 8) |
                                  (i + nseg == end ? kLastEntry : 0u);
            E.ent[i] = make_float4(p.o.x, p.o.y, p.o.z, __uint_as_float(info));
            E.ent[i + 1] = make_float4(p.d.x, p.d.y, p.d.z, miss ? INFINITY : h.t);
            if (!kMat) E.ent[i + 2] = make_float4(p.beta.x, p.beta.y, p.beta.z, 0.f);
            i += nseg;
        }
        if (emis) {
            E.ent[i] = make_float4(p.beta.x, p.beta.y, p.beta.z, __uint_as_float(emis | (i + 1 == end ? kLastEntry : 0u)));
            ++i;
        }
        if (nvert) {
            v0.w = __uint_as_float(vert | kLastEntry);
            E.ent[i] = v0;
            if (kMove && nvert > 1) E.ent[i + 1] = v1;
            if (kMove && nvert > 2) E.ent[i + 2] = v2;
        }
    }
    if (miss || last) return kEnded;
    // ---- the next ray ---------------------------------------------------------------------------
    if (mtype == kDiffuse) {
        p.d = normalized(diffuse_dir(ns, u01(w0.z), u01(w0.w)));
        p.o = po;
        p.specular = false;
    } else {
        if (mtype == kMirror) {
            p.d = normalized(p.d - ns * (2.0f * dot3(p.d, ns)));
            p.o = po;
        } else {
            dielectric(p, pt, ng, ior, u01(w1.z));
        }
        p.specular = true;
    }
    p.beta = p.beta * albedo;
    if (kMat) E.varied = E.varied || bound;
    if (maxc(p.beta) <= 0.0f) return kEnded;
    if (rr) {  // Russian roulette on slot 1's second uniform
        if (kMat && E.varied) {
            // A render survives when u < q_r = min(0.95, max beta_r), and q_r <= q here; its
            // largest throughput is then max(1, max beta_r / 0.95) up to rounding.
            const float bm = maxc(p.beta);
            if (u01(w1.y) >= fminf(0.95f, bm * 1.000001f)) return kEnded;
            const float nb = fmaxf(1.0f, bm * 1.0527f) * 1.00001f;
            p.beta = f3(nb, nb, nb);
        } else {
            const float q = fminf(0.95f, maxc(p.beta));
            if (u01(w1.y) >= q) return kEnded;
            p.beta = p.beta * rcp_fast(q);
        }
    }
    ++p.b;
    return kLive;
}

// ---------------------------------------------------------------------------
// k_trace_replay: every path traced once, replayed by each render (a3-a5)
// ---------------------------------------------------------------------------
// Under common random numbers the renders of a job differ only where a perturbed primitive
// meets a ray, where an emitter that moved is sampled, and in the albedos that are bound. A
// work item is one of a pixel block's J.parts parts (1/parts of the positions of the bit-reversed
// slot order) for all R <= 64 renders (more: 64 of them), taken by one warp, which takes the part's (pixel, sample)
// tasks in batches of 32, pixels in that order:
//   phase A  lane = task: the path is traced once in the invariant scene (replay_vertex). What
//            is the same in every render goes into the pixel's common sum, the rest into a
//            chain of entries in the warp's pool. A batch whose pool runs out keeps the paths
//            before the first one that did not fit, and the next batch starts there (with that
//            path alone if it was the batch's first: the pool holds any one path);
//   phase B  lane = render (lane and lane + 32; with R < 32 the lanes hold floor(32 / R)
//            samples side by side): each render replays the chains with its own primitives,
//            albedos and tangents (replay_sample). A render that parts from the path (its own
//            primitive is hit first) traces the rest as k_trace_group does, unless that
//            primitive is black (most emitters), where the path ends.
// Each render's radiance is the same sum, term by term and in the same order, as tracing the
// path in that render alone, and the pairwise pixel sum is the shuffle tree of the per-render
// epilogue (see k_trace_group): with the same block shape every partial is bit-identical to
// the per-render kernel's; a part's sum is a subtree, and the warp that finishes a block's last
// part adds them. The warps of a CTA share the staged scene and the per-render table
// and meet only when the launch goes on to another job.
//
// Tracing a path once instead of once per render leaves per render only its estimates (light
// sample, occlusion by the few primitives the cull leaves, geometry term) and products of
// albedos. Before, the GI box's renders retraced every path side by side (k_trace_group) and Eq. 9
// traced each render alone (k_trace; Eq. 10 with albedos only shared paths, but nearly every path meets a
// bound wall): GI box 512 x 512, 32 renders at 32 spp 40.9 -> 16.2 ms, its
// walls by Eq. 9 87.6 -> 7.5 ms, by Eq. 10 at 256 x 256 11.3 -> 1.26 ms, caustic 512 x 512, 64 renders at
// 64 spp 7.8 -> 7.3 ms. Leaving fixed emitters out of the variant for jobs whose emitters all move
// (80 -> 74 KB of code: instruction fetch is among the largest stalls) took the GI box to 15.1 ms and
// caustic to 7.0 ms. Bound by instruction issue (60 % of cycles, 20 warps per SM): fixed-latency
// dependencies and instruction fetch are the largest stalls, phase A takes about a quarter of the
// GI box's time and half of Eq. 9's. Groups of entries are 16-byte granules because the pool's
// shared memory sets how many paths fit a batch.
constexpr int kReplayWarps = kGroupBlock / 32;

// Shared memory of a CTA: this head, the per-render table, and per warp (replay_warp_bytes)
//   double pair[halves][levels][32]   pairwise-sum stacks of the lane's renders
//   u64 acc[halves][3][32]            radiance of the current pixel, 2^-32 fixed point
//   u64 dacc[halves][nd][32]          Eq. 9: its tangent sums
//   double gsum[halves][nd][32]       Eq. 9: the block's gradient partials
//   u64 common[replay_common][3]      radiance common to all renders, per pixel of the block
//   float4 ent[pool], u16 nxt[pool], u16 first[32], unsigned ctr
struct ReplayHead {
    GroupScene scene;  // the invariant part (render 0's records of the other primitives)
    TraceJob job;
    float4 ulo[kMaxVariant], uhi[kMaxVariant];
    float4 amax[kGroupMats];   // largest albedo of each bound material over the renders
    float4 ball[kGroupPrims];  // enclosing balls of the invariant primitives
    unsigned left, pad[3];     // has the job items left?
};
static_assert(sizeof(ReplayHead) % 16 == 0, "float4 arrays follow");

__host__ __device__ constexpr int replay_levels(int pixels) {
    return pixels <= 1 ? 0 : (pixels <= 2 ? 1 : (pixels <= 4 ? 2 : (pixels <= 8 ? 3 : (pixels <= 16 ? 4 : 5))));
}
// Entries of `common`: the pixels, rounded up to an even number so that the pool after it is aligned.
__host__ __device__ constexpr int replay_common(int pixels) { return pixels + (pixels & 1); }
__host__ __device__ constexpr size_t replay_warp_bytes(int pool, int halves, int pixels, int nd) {
    return size_t(halves) * (replay_levels(pixels) + 3 + 2 * nd) * 256 + size_t(replay_common(pixels)) * 24 + size_t(pool) * 18 + 80;
}
// (pool in multiples of 8: 16-byte alignment throughout)
static_assert(replay_warp_bytes(8, 1, 1, 0) % 16 == 0 && replay_warp_bytes(8, 1, 2, 3) % 16 == 0 &&
                  replay_warp_bytes(24, 2, 4, 6) % 16 == 0 && replay_warp_bytes(512, 2, 32, 12) % 16 == 0,
              "the next warp's sums are aligned");
size_t replay_smem(const TraceLaunch& L) {
    return sizeof(ReplayHead) + size_t(L.tab_rows) * 16 +
           kReplayWarps * replay_warp_bytes(L.pool, L.halves, L.pixels, L.diff_nd);
}

// Resident CTAs per SM that a variant is compiled for: 6 (<= 80 registers, 24 warps), or 5 (<= 102)
// with perturbed primitives, where the pool needs the shared memory (the GI box with only its
// light moving, 32 renders at 16 spp: 8.4 ms with 5, 15.6 ms with 6; the GI box's walls, 256 x 256:
// 1.33 ms with 5, 1.25 ms with 6).
constexpr int replay_min_blocks(bool move) { return move ? 5 : 6; }

// The pool takes the shared memory that replay_min_blocks CTAs per SM (the registers' limit) leave,
// up to kReplayPoolMax granules, or that fewer CTAs leave where it would be too small to hold a
// batch of common paths: a pool that runs out costs part of a batch's phase A (GI box at 32
// renders, 224 granules of 3 float4 instead of 128: 73 -> 27 ms), a CTA less per SM a tenth or so
// (Eq. 9 on the box's walls with 44 renders, whose sums fill 6 CTAs' shared memory: 232 x 274 at 50 spp
// 29.9 ms with 24 granules, 5.2 ms with what 3 CTAs leave; 64 renders, 256 x 256 at 16 spp, 10.9 and 1.9).
constexpr int kReplayPoolMax = 512, kReplayPoolMove = 256, kReplayPoolFixed = 128;
static int replay_pool(const TraceLaunch& L) {
    const size_t head = sizeof(ReplayHead) + size_t(L.tab_rows) * 16;
    const size_t rest = replay_warp_bytes(0, L.halves, L.pixels, L.diff_nd);
    const int need = (L.granules + 7) & ~7, want = L.replay_move ? kReplayPoolMove : kReplayPoolFixed;
    int fits = 0;
    for (int ctas = replay_min_blocks(L.replay_move != 0); ctas >= 2 && fits < want; --ctas) {
        const size_t cta = 227 * 1024 / ctas - 1024;  // 1 KB of a CTA's is the system's
        if (cta > head + kReplayWarps * rest) fits = int((cta - head - kReplayWarps * rest) / (18 * kReplayWarps));
    }
    fits = fits < kReplayPoolMax ? fits : kReplayPoolMax;
    return fits > need ? fits & ~7 : need;
}

// The pool is fitted anew to the tables, sums and pixels of all jobs so far: taken as the least pool
// for the next job, the first one's would keep the launch to fewer CTAs than its jobs need (8
// renders on one pixel, then 32 on 4: 4 CTAs per SM instead of the reverse order's 5).
void replay_cover(TraceLaunch& L, const TraceJob& J) {
    auto most = [](int& a, int b) { a = a > b ? a : b; };
    L.replay_mat |= J.var_mats ? 1 : 0;
    most(L.replay_move, J.n_var > 0 ? (J.black ? 1 : 2) : 0);
    most(L.halves, J.R > 32 ? 2 : 1);
    most(L.tab_rows, J.R * J.gstride);
    most(L.pixels, J.bw * J.bh / J.parts);
    L.replay_chunked |= J.chunks > 1 ? 1 : 0;
    most(L.granules, replay_path_granules(J.depth, J.n_var > 0));
    if (J.diff) L.diff_nd = J.nd;
    L.pool = replay_pool(L);
}

// A render's clamp derivatives (Eq. 9) in its row of the table.
struct ClampRow {
    const float4* p;
    int s;
    __device__ __forceinline__ float operator[](int k) const {
        return reinterpret_cast<const float*>(p + (k >> 2) * s)[k & 3];
    }
};

// Sum of non-negative floats below 2^14 in 2^-32 fixed point, as to_fixed adds them, without
// 64-bit arithmetic: hi counts units of 2^-9 (the bits that an addition of 2^14 rounded toward
// zero keeps), lo the rest in units of 2^-32. The sum is (hi << 23) + lo; 32 terms fit.
__device__ __forceinline__ void fix_add(unsigned& hi, unsigned& lo, float v) {
    const float s = __fadd_rz(v, 16384.0f);
    hi += __float_as_uint(s) - 0x46800000u;
    const float r = v - (s - 16384.0f);  // exact, in [0, 2^-9)
    lo += __float_as_uint(__fadd_rz(r, 0x1p-9f)) - 0x3b000000u;
}
__device__ __forceinline__ unsigned long long fix_sum(unsigned hi, unsigned lo) {
    return ((unsigned long long)hi << 23) + lo;
}
// The same for |v| < 2^13 (tangents): rounded down to 2^-32, hi signed.
__device__ __forceinline__ void fix_add_signed(unsigned& hi, unsigned& lo, float v) {
    const float s = __fadd_rz(v, 24576.0f);
    hi += __float_as_uint(s) - 0x46c00000u;
    const float r = v - (s - 24576.0f);
    lo += __float_as_uint(__fadd_rz(r, 0x1p-9f)) - 0x3b000000u;
}
__device__ __forceinline__ unsigned long long fix_sum_signed(unsigned hi, unsigned lo) {
    return (unsigned long long)((long long)int(hi) << 23) + lo;
}

// The rest of a path in one render's scene (as k_trace_group traces it).
template <bool kCount>
__device__ __forceinline__ float3 replay_alone(const GroupScene& S, int depth, int rr_start, const GroupLane& gl,
                                               Path p, Counters& cnt) {
    while (advance<kCount, false, 0, true>(S, depth, rr_start, p, cnt, nullptr, nullptr, nullptr, &gl) == kLive) {
    }
    return p.L;
}

// One render's radiance from a path's chain (without the common part). kMove: 0 no perturbed
// primitive, 1 only black ones (a render that meets its own primitive ends there) with every emitter
// among them, 2 any. Tangent slot k is a parameter of channel k mod 3 (kND: 0 or a multiple of 3);
// J.mat_slots[m] holds the slots of material m's parameters.
template <bool kCount, bool kMat, int kMove, int kND>
__device__ __forceinline__ float3 replay_sample(const GroupScene& S, const TraceJob& J, const GroupLane& gl,
                                                const float4* ent, const unsigned short* nxt, int i, unsigned pixel,
                                                int s, int slot, Counters& cnt, Tangents<kND>& tn) {
    float3 Lr = f3(0.f, 0.f, 0.f), beta = f3(1.f, 1.f, 1.f);
    const ClampRow dclamp{gl.rec + (gl.var_rows + __popc(gl.mats)) * gl.rs, gl.rs};
    bool on = true, parted = false;  // on the shared path; left it to go on alone
    Path p;
    int next = nxt[i];
#pragma unroll 1
    while (i != kNoEntry) {
        const float4 a = ent[i];
        const unsigned info = __float_as_uint(a.w), kind = info & 3u;
        const int mat = int(info >> 8) & 15;
        int size = 1;
        if (kind == kVert) {
            const unsigned est = (info >> 2) & 3u;
            size = !kMove ? 1 : (!kMat || est == 3u || (info & (1u << 18)) ? 3 : (est == 1u ? 2 : 1));
            if ((!kMat && !kMove) || on) {
                float3 ba, albedo = f3(0.f, 0.f, 0.f);
                float urr = 0.0f;
                if (kMat) {
                    albedo = xyz(mat_albedo<true>(S, mat, &gl));
                    ba = beta * albedo;
                    urr = a.y;
                    if (kND > 0) {  // tangents of beta * albedo
                        const unsigned ms = J.mat_slots[mat];
#pragma unroll
                        for (int k = 0; k < kND; ++k) {
                            tn.dB[k] *= comp3(albedo, k % 3);
                            if ((ms >> k) & 1u) tn.dB[k] = fmaf(comp3(beta, k % 3), dclamp[k], tn.dB[k]);
                        }
                    }
                }
                if (est) {
                    const int li = int(info >> 5) & 7;
                    bool seen = true;
                    float g;
                    int lmat;
                    if (kMove == 1 || (kMove && est == 1u)) {
                        const float4 b = ent[i + 1];
                        float3 ns;
                        float lu, lv;
                        if (kMat) {
                            urr = b.z;
                            lu = b.x;
                            lv = b.y;
                            if (info & (1u << 18)) {
                                ns = xyz(ent[i + 2]);
                            } else {  // a quad's normal, from its record
                                ns = xyz(S.prim[(info >> 12) & 15u][1]);
                                if (info & (1u << 17)) ns = ns * -1.0f;
                            }
                        } else {
                            const float4 c = ent[i + 2];
                            ba = xyz(b);
                            ns = xyz(c);
                            lu = b.w;
                            lv = c.w;
                        }
                        float3 wi;
                        float dist;
                        seen = nee_to<kCount, false, true>(S, xyz(a), ns, lu, lv, li, cnt, info >> (32 - kCullBits), &gl,
                                                           wi, dist, g, lmat);
                    } else {
                        const int4 lt = S.light[li];
                        lmat = lt.w;
                        g = a.x;
                        if (kMove && (est == 3u || !kMat)) {
                            const float4 c = ent[i + 2];
                            g = kMat ? c.x : c.w;
                            if (kMat) urr = c.y;
                            else ba = xyz(c);
                            if (est == 3u) {
                                const float4 b = ent[i + 1];
                                seen = !group_occluded<kCount>(S, gl, xyz(a), xyz(b), b.w, lt.y, cnt);
                            }
                        }
                    }
                    if (seen) {
                        const float3 Le = xyz(S.mat[lmat][1]);
                        if (kND > 0) {
                            const float3 leg = Le * g;
#pragma unroll
                            for (int k = 0; k < kND; ++k) tn.dL[k] = fmaf(tn.dB[k], comp3(leg, k % 3), tn.dL[k]);
                        }
                        Lr = nee_add(Lr, ba, Le, g);
                    }
                }
                if (kMat) {
                    const float mb = maxc(ba);
                    on = mb > 0.0f;
                    beta = ba;
                    if (info & 16u) {  // Russian roulette
                        const float q = fminf(0.95f, mb);
                        on = on && urr < q;
                        const float inv_q = rcp_fast(q);
                        beta = beta * inv_q;
#pragma unroll
                        for (int k = 0; k < kND; ++k) tn.dB[k] *= inv_q;
                    }
                }
            }
        } else if (kMove && kind == kSegment) {
            size = kMat ? 2 : 3;
            if (on) {
                const float4 b = ent[i + 1];
                Hit h{b.w, -1, 0};
                group_hit<kCount>(S, gl, xyz(a), xyz(b), h, cnt);
                if (h.slot >= 0) {  // this render's own primitive comes first
                    on = false;
                    const float3 bt = kMat ? beta : xyz(ent[i + 2]);
                    const auto P = prim_rec<true>(S, h.slot, &gl);
                    const int hm = as_int(h.type == kSphere ? P[1].z : P[0].w) & 255;
                    const float4 al = mat_albedo<true>(S, hm, &gl);
                    if (kMove == 1 || (as_int(al.w) == kDiffuse && al.x == 0.0f && al.y == 0.0f && al.z == 0.0f)) {
                        // a black surface: its emission, and the path ends
                        const float3 em = xyz(S.mat[hm][1]);
                        if ((info & 16u) && (em.x > 0.f || em.y > 0.f || em.z > 0.f)) {
                            const float3 d = xyz(b), pt = xyz(a) + d * h.t;
                            const float3 ng = h.type == kSphere ? (pt - xyz(P[0])) * P[1].y : xyz(P[1]);
                            if (dot3(d, ng) < 0.0f) Lr = Lr + bt * em;
                        }
                    } else {
                        parted = true;
                        p.o = xyz(a);
                        p.d = xyz(b);
                        p.beta = bt;
                        p.specular = (info & 16u) != 0u;
                        p.b = int(info >> 8) & 127;
                    }
                }
            }
        } else if (kind == kEmission) {
            if ((!kMat && !kMove) || on) {
                const float3 E = (info & 32u) ? xyz(S.bg) : xyz(S.mat[mat][1]);
#pragma unroll
                for (int k = 0; k < kND; ++k) tn.dL[k] = fmaf(tn.dB[k], comp3(E, k % 3), tn.dL[k]);
                Lr = Lr + (kMat ? beta : xyz(a)) * E;
            }
        } else if (kind == kPrefix) {
            Lr = xyz(a);
            if (kMat) {
                beta = xyz(ent[i + 1]);
                size = 2;
            }
        }
        if (info & kLastEntry) {
            i = next;
            if (i != kNoEntry) next = nxt[i];
        } else {
            i += size;
        }
    }
    if (kMove == 2 && parted) {
        p.L = Lr;
        p.pixel = pixel;
        p.s = s;
        p.slot = slot;
        p.seg = 0u;
        Lr = replay_alone<kCount>(S, J.depth, J.rr_start, gl, p, cnt);
    }
    return Lr;
}

// Sum number k (0 the squared error, 1 + slot a tangent slot's) of work item `item` in render r. Out
// of line, like replay_combine: both run once per item, and inlined they cost the loops registers.
template <int kND>
__device__ __noinline__ void replay_store(const TraceJob& J, unsigned item, int r, int k, double v) {
    if (J.parts > 1) {
        J.part_sums[(size_t(item) * J.R + r) * (1 + kND) + k] = v;
    } else if (k == 0) {
        J.partials[size_t(r) * J.tiles + item] = v;
    } else if (J.slot_param[k - 1] >= 0) {
        J.gpartials[(size_t(r) * J.tiles + item) * J.diff_n + J.slot_param[k - 1]] = v;
    }
}

// The warp that finishes a block's last part adds the parts' subtrees in the pairwise sum's order.
template <int kND>
__device__ __noinline__ void replay_combine(const TraceJob& J, unsigned item, int lane) {
    const int parts = J.parts, t = int(item) / parts;
    unsigned done = 0;
    __threadfence();  // the part's sums before its count
    __syncwarp();
    if (lane == 0) {
        done = atomicAdd(J.part_done + t, 1u);
        __threadfence();
    }
    done = __shfl_sync(kFull, done, 0);
    if (done != unsigned(parts - 1)) return;
    const int n = J.R * (1 + kND);
    for (int i = lane; i < n; i += 32) {
        const int r = i / (1 + kND), k = i - r * (1 + kND);
        const int param = k > 0 ? J.slot_param[k - 1] : 0;
        if (param < 0) continue;
        double s[5], v = 0.0;
        for (int p = 0; p < parts; ++p) {
            v = __ldcg(J.part_sums + (size_t(t) * parts + p) * n + i);
            int l = 0;
            for (; (p >> l) & 1; ++l) v = s[l] + v;
            if (p + 1 < parts) s[l] = v;
        }
        if (k == 0) J.partials[size_t(r) * J.tiles + t] = v;
        else J.gpartials[(size_t(r) * J.tiles + t) * J.diff_n + param] = v;
    }
    if (lane == 0) J.part_done[t] = 0u;  // ready for the next launch
}

// kChunked: jobs of more than 64 renders (a variant of its own: the chunk costs the others 1 %).
template <bool kCount, bool kMat, int kMove, int kND, bool kChunked>
__global__ void __launch_bounds__(kGroupBlock, replay_min_blocks(kMove != 0)) k_trace_replay(const __grid_constant__ TraceLaunch L) {
    extern __shared__ __align__(16) unsigned char s_replay[];
    ReplayHead& E = *reinterpret_cast<ReplayHead*>(s_replay);
    float4* tab = reinterpret_cast<float4*>(s_replay + sizeof(ReplayHead));
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int levels = replay_levels(L.pixels), halves = L.halves;
    unsigned char* wbase = s_replay + sizeof(ReplayHead) + size_t(L.tab_rows) * 16 +
                           size_t(warp) * replay_warp_bytes(L.pool, halves, L.pixels, kND);
    double (*pair)[32] = reinterpret_cast<double (*)[32]>(wbase);
    unsigned long long (*acc)[32] = reinterpret_cast<unsigned long long (*)[32]>(pair + halves * levels);
    unsigned long long (*dacc)[32] = acc + halves * 3;
    double (*gsum)[32] = reinterpret_cast<double (*)[32]>(dacc + halves * kND);
    unsigned long long (*common)[3] = reinterpret_cast<unsigned long long (*)[3]>(gsum + halves * kND);
    float4* ent = reinterpret_cast<float4*>(common + replay_common(L.pixels));
    unsigned short* nxt = reinterpret_cast<unsigned short*>(ent + L.pool);
    unsigned short* firsts = nxt + L.pool;
    unsigned* ctr = reinterpret_cast<unsigned*>(firsts + 32);
    const TraceJob& J = E.job;
    Counters cnt{0u, 0u, 0u, 0u, 0u, 0u, 0u, 0u};
    const int njobs = L.jobs ? L.njobs : 1;
    for (int jb = 0; jb < njobs; ++jb) {  // a packed launch's jobs one after another, each CTA from another one
    {  // job descriptors are host data: the first is copied before the wait on the previous kernel
        const unsigned* src =
            reinterpret_cast<const unsigned*>(L.jobs ? L.jobs + (int(blockIdx.x) + jb) % njobs : &L.job0);
        unsigned* dst = reinterpret_cast<unsigned*>(&E.job);
        __syncthreads();  // every warp is done with the previous job
        for (int i = threadIdx.x; i < int(sizeof(TraceJob) / 4); i += kGroupBlock) dst[i] = src[i];
        if (jb == 0) pdl_enter();
        __syncthreads();
    }
    if (threadIdx.x == 0) E.left = __ldcg(J.queue) < unsigned(J.tiles * J.parts * J.chunks) ? 1u : 0u;
    __syncthreads();
    if (!E.left) continue;
    const int n = J.n_var, nr = J.var_rows, nm = __popc(J.var_mats), stride = J.gstride, ncl = (kND + 3) / 4;
    if (J.R < 1 || J.R > 64 * J.chunks || (!kChunked && J.chunks > 1) || (J.R > 32 && halves < 2) || (J.chunks > 1 && J.parts > 1) || J.R * stride > L.tab_rows || stride < nr + nm + ncl || n < 0 ||
        n > kMaxVariant || J.n_prims > kGroupPrims || J.n_mats > kGroupMats || (!kMat && nm) || (!kMove && n) ||
        (kMove == 1 && !J.black && n) || J.parts < 1 || J.parts > J.bw * J.bh ||
        J.bw * J.bh > L.pixels * J.parts || (J.parts & (J.parts - 1)) != 0 || replay_path_granules(J.depth, kMove != 0) > L.pool) {
        if (threadIdx.x == 0) atomicOr(L.status, kStatusBadItem);
        continue;
    }
    // ---- stage the job: invariant scene, per-render rows, union bounds --------------------------
    if (warp == 0) stage_group_scene(E.scene, J, 0, lane);
    for (int i = threadIdx.x; i < J.R * stride; i += kGroupBlock) {
        const int r = i / stride, q = i - r * stride;
        const InstScene& R = J.scenes[r];
        float4 v;
        if (q < nr) {
            v = __ldg(&R.prim[J.row_src[q] >> 1][J.row_src[q] & 1]);
        } else if (q < nr + nm) {
            v = __ldg(&R.mat[nth_set_bit(J.var_mats, q - nr)][0]);
        } else if (kND > 0) {  // clamp derivatives by tangent slot
            const int k = 4 * (q - nr - nm);
            auto dc = [&](int slot) { return slot < kND && J.slot_param[slot] >= 0 ? __ldg(R.dclamp + J.slot_param[slot]) : 0.0f; };
            v = make_float4(dc(k), dc(k + 1), dc(k + 2), dc(k + 3));
        } else {
            v = __ldg(reinterpret_cast<const float4*>(R.light_area) + (q - nr - nm));
        }
        tab[q * J.R + r] = v;  // field-major, as k_trace_group's table
    }
    __syncthreads();
    if (kMat && int(threadIdx.x) < nm) {
        float4 m = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int r = 0; r < J.R; ++r) {
            const float4 v = tab[(nr + int(threadIdx.x)) * J.R + r];
            m = make_float4(fmaxf(m.x, v.x), fmaxf(m.y, v.y), fmaxf(m.z, v.z), 0.f);
        }
        E.amax[nth_set_bit(J.var_mats, int(threadIdx.x))] = m;
    }
    if (kMove && warp == 1 && lane < J.n_prims && lane < kCullBits)
        E.ball[lane] = prim_ball(E.scene.prim[lane], lane < E.scene.n_sph ? kSphere
                                                     : (lane < E.scene.n_sph + E.scene.n_quad ? kQuad : kBox));
    if (kMove && warp == 0) {
        for (int k = 0; k < n; ++k) {
            const int slot = nth_set_bit(J.var_prims, k);
            const int type = slot < E.scene.n_sph ? kSphere : (slot < E.scene.n_sph + E.scene.n_quad ? kQuad : kBox);
            float3 lo = f3(INFINITY, INFINITY, INFINITY), hi = f3(-INFINITY, -INFINITY, -INFINITY);
            for (int r = lane; r < J.R; r += 32) {
                float3 a, c;
                const SRec own{tab + ((J.var_offs >> (8 * k)) & 255u) * J.R + r, J.R, type == kQuad ? 1 : 2, E.scene.prim[slot]};
                prim_bounds(own, type, a, c);
                lo = f3(fminf(lo.x, a.x), fminf(lo.y, a.y), fminf(lo.z, a.z));
                hi = f3(fmaxf(hi.x, c.x), fmaxf(hi.y, c.y), fmaxf(hi.z, c.z));
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                lo.x = fminf(lo.x, __shfl_xor_sync(kFull, lo.x, o));
                lo.y = fminf(lo.y, __shfl_xor_sync(kFull, lo.y, o));
                lo.z = fminf(lo.z, __shfl_xor_sync(kFull, lo.z, o));
                hi.x = fmaxf(hi.x, __shfl_xor_sync(kFull, hi.x, o));
                hi.y = fmaxf(hi.y, __shfl_xor_sync(kFull, hi.y, o));
                hi.z = fmaxf(hi.z, __shfl_xor_sync(kFull, hi.z, o));
            }
            if (lane == 0) {
                E.ulo[k] = make_float4(lo.x, lo.y, lo.z, 0.f);
                E.uhi[k] = make_float4(hi.x, hi.y, hi.z, 0.f);
            }
        }
    }
    __syncthreads();
    // Positions of the bit-reversed order that can hold a pixel of a block of 2^k pixels are
    // multiples of 2^(5 - k): the other levels of the pairwise sum would add zeros.
    const int qshift = 5 - replay_levels(J.bw * J.bh), qend = (32 / J.parts) >> qshift;
    for (;;) {  // ---- the warp's work items ------------------------------------------------------
        unsigned item = 0;
        if (lane == 0) item = atomicAdd(J.queue, 1u);
        item = __shfl_sync(kFull, item, 0);
        // jobs of more than 64 renders: every block once per chunk of 64
        const unsigned units = unsigned(J.tiles * J.parts), chunk = kChunked ? item / units : 0u;
        if (kChunked ? int(chunk) >= J.chunks : item >= units) break;
        if (kChunked) item -= chunk * units;
        const int r0 = int(chunk) * 64;
        const int t = int(item) / J.parts, q0 = (int(item) - t * J.parts) * (qend << qshift);
        const int R = kChunked ? min(J.R - r0, 64) : J.R, nh = R > 32 ? 2 : 1, spp = J.spp;
        // phase B lanes: render gi of sample group ks; with R < 32, nsg = floor(32 / R) samples
        // side by side (lanes beyond nsg R repeat the last group's; they are not counted)
        const int G = R < 32 ? R : 32, nsg = 32 / G, gi = lane % G, ks = lane / G;
        const int areas = !kND && J.gstride > J.var_rows + __popc(J.var_mats) ? 1 : 0;
        const int x0 = (t % J.tiles_x) * J.bw, y0 = (t / J.tiles_x) * J.bh;
        const int vw = min(J.bw, J.W - x0), vh = min(J.bh, J.H - y0);
        const int npx = vw * vh;
        const unsigned magic_w = 0xffffffffu / unsigned(vw) + 1u;
        const float inv = mean_scale(spp);
        // the part's positions that hold a pixel (bit q: position q0 + q)
        const unsigned vm = __ballot_sync(kFull, lane < (qend << qshift) && brev5(q0 + lane) < npx);
        const int npix = __popc(vm);
        auto pixel_of = [&](int k, int& slot) {  // k-th pixel of the block
            slot = brev5(q0 + nth_set_bit(vm, k));
            const int row = div_magic(slot, vw, magic_w);
            return unsigned((y0 + row) * J.W + x0 + slot - row * vw);
        };
        if (lane < npix)
            for (int i = 0; i < 3; ++i) common[lane][i] = 0ull;
#pragma unroll 1
        for (int i = 0; i < 3 * nh; ++i) acc[i][lane] = 0ull;
#pragma unroll 1
        for (int i = 0; i < kND * nh; ++i) {
            dacc[i][lane] = 0ull;
            gsum[i][lane] = 0.0;
        }
        auto push_pair = [&](int h, int q, double v) {  // position q << qshift of the pairwise sum
            double (*s)[32] = pair + h * levels;
            int l = 0;
#pragma unroll 1
            for (; (q >> l) & 1; ++l) v = s[l][lane] + v;
            if (q + 1 < qend) s[l][lane] = v;
            else if (ks == 0 && gi + 32 * h < R) replay_store<kND>(J, item, r0 + gi + 32 * h, 0, v);  // a5
        };
        int k0 = 0, s0 = 0;    // the next task: pixel k0 of the block, sample s0
        int nextq = 0;         // positions below are summed
        bool alone = false;    // the next batch holds one path only
        // The loops below stay rolled: unrolled copies of the tracer overflow the instruction
        // cache (measured on the caustic step: 13.1 ms unrolled, 11.0 ms rolled).
#pragma unroll 1
        while (k0 < npix) {
            // ---- phase A: one path per lane, traced once for all renders ----------------------
            __syncwarp();  // phase B of the previous batch is done with the pool
            if (lane == 0) *ctr = 0u;
            __syncwarp();
            int kp = k0, sp = s0 + lane;  // this lane's task
            while (sp >= spp && kp < npix) {
                sp -= spp;
                ++kp;
            }
            const bool have = kp < npix && (!alone || lane == 0);
            // (culling costs more than two renders' tests: GI box with only its light moving, 96 x 96 at 64 spp,
            // 560 -> 436 us)
            ReplayLane el{E.ulo,    E.uhi,    E.amax, E.ball, J.n_var, J.var_prims, J.var_mats, ent, nxt, ctr,
                          L.pool, kNoEntry, kNoEntry, false,  false,   false, R > 2};
            Path p;
            p.L = f3(0.f, 0.f, 0.f);
            if (have) {
                int slot;
                const unsigned pixel = pixel_of(kp, slot);
                const int py = int(pixel) / J.W, px = int(pixel) - py * J.W;
                start_path<true>(E.scene, J.W, J.H, px, py, sp, slot, p);
            }
            bool live = have;
            const Counters before = cnt;
#pragma unroll 1
            while (__any_sync(kFull, live)) {
                if (live) live = replay_vertex<kCount, kMat, kMove>(E.scene, J.depth, J.rr_start, p, el, cnt) == kLive;
            }
            const unsigned fm = __ballot_sync(kFull, el.full), hm = __ballot_sync(kFull, have);
            const int nb = fm ? __ffs(fm) - 1 : __popc(hm);  // the batch: tasks of lanes 0 .. nb - 1
            if (kCount && lane >= nb) cnt = before;  // traced again in the next batch
            if (nb == 0) {
                if (alone) {  // cannot happen: the host sizes the pool for any one path
                    if (lane == 0) atomicOr(L.status, kStatusBadItem);
                    break;
                }
                alone = true;
                continue;
            }
            alone = false;
            if (lane < nb) {
                if (kCount) ++cnt.paths;
                firsts[lane] = (unsigned short)(el.first);
                if (!el.rec && (p.L.x != 0.0f || p.L.y != 0.0f || p.L.z != 0.0f)) {
                    smem_add_u64(&common[kp][0], to_fixed(p.L.x));
                    smem_add_u64(&common[kp][1], to_fixed(p.L.y));
                    smem_add_u64(&common[kp][2], to_fixed(p.L.z));
                }
            }
            const unsigned work = __ballot_sync(kFull, lane < nb && el.first != kNoEntry);
            __syncwarp();
            // ---- phase B: each render's terms, pixel by pixel ---------------------------------
            int i0 = 0;  // first task of the current pixel in the batch
#pragma unroll 1
            while (i0 < nb) {
                const int i1 = min(nb, i0 + spp - s0);
                const unsigned in = (i1 >= 32 ? kFull : (1u << i1) - 1u) & ~((1u << i0) - 1u);
                int slot;
                const unsigned pixel = pixel_of(k0, slot);
                const bool ends = s0 + (i1 - i0) == spp;  // the pixel's last samples
#pragma unroll 1
                for (int h = 0; h < nh; ++h) {
                    const int r = gi + 32 * h;
                    const GroupLane gl{tab + r0 + (r < R ? r : 0), J.var_prims, J.var_mats, J.var_offs, J.var_rows, areas,
                                       nullptr, 0, kChunked ? J.R : R};
                    unsigned hi0 = 0u, hi1 = 0u, hi2 = 0u, lo0 = 0u, lo1 = 0u, lo2 = 0u;
                    unsigned dhi[kND > 0 ? kND : 1], dlo[kND > 0 ? kND : 1];
#pragma unroll
                    for (int k = 0; k < kND; ++k) dhi[k] = dlo[k] = 0u;
                    unsigned todo = work & in;
#pragma unroll 1
                    while (todo) {
                        int jj = __ffs(todo) - 1;
                        todo &= todo - 1u;
#pragma unroll 1
                        for (int i = 1; i < nsg; ++i) {  // sample group ks takes the ks-th of the next nsg tasks
                            if (i <= ks) jj = __ffs(todo) - 1;
                            todo &= todo - 1u;
                        }
                        if (jj < 0 || r >= R || (kCount && ks >= nsg)) continue;
                        Tangents<kND> tn;
                        if (kND > 0) tan_reset(tn);
                        const float3 v = replay_sample<kCount, kMat, kMove, kND>(
                            E.scene, J, gl, ent, nxt, firsts[jj], pixel, s0 + jj - i0, slot, cnt, tn);
                        if (v.x + v.y + v.z < 16384.0f && fminf(v.x, fminf(v.y, v.z)) >= 0.0f) {
                            fix_add(hi0, lo0, v.x);
                            fix_add(hi1, lo1, v.y);
                            fix_add(hi2, lo2, v.z);
                        } else {
#pragma unroll 1
                            for (int c = 0; c < 3; ++c) acc[3 * h + c][lane] += to_fixed(comp3(v, c));
                        }
#pragma unroll
                        for (int k = 0; k < kND; ++k) {
                            if (fabsf(tn.dL[k]) < 8192.0f) fix_add_signed(dhi[k], dlo[k], tn.dL[k]);
                            else dacc[h * kND + k][lane] += to_fixed_signed(tn.dL[k]);
                        }
                    }
                    unsigned long long a0 = acc[3 * h][lane] + fix_sum(hi0, lo0),
                                       a1 = acc[3 * h + 1][lane] + fix_sum(hi1, lo1),
                                       a2 = acc[3 * h + 2][lane] + fix_sum(hi2, lo2);
                    acc[3 * h][lane] = ends ? 0ull : a0;
                    acc[3 * h + 1][lane] = ends ? 0ull : a1;
                    acc[3 * h + 2][lane] = ends ? 0ull : a2;
                    if (!ends) {
#pragma unroll
                        for (int k = 0; k < kND; ++k) dacc[h * kND + k][lane] += fix_sum_signed(dhi[k], dlo[k]);
                        continue;
                    }
                    // the pixel is complete: add its sample groups and the common part, form the error
                    auto groups = [&](unsigned long long v) {
                        unsigned long long sum = v;
                        if (kMat || kMove != 1) {
                            _Pragma("unroll 1") for (int q = 1; q < nsg; ++q) sum += __shfl_sync(kFull, v, (lane + q * G) & 31);
                        } else {  // by halves (caustic 400 x 400 at 32 spp, 2 renders: 16 groups, 679 -> 612 us)
                            _Pragma("unroll 1") for (int q = 1; q < nsg; q *= 2) {
                                const unsigned long long o = __shfl_sync(kFull, sum, (lane + q * G) & 31);
                                if (ks + q < nsg) sum += o;
                            }
                        }
                        return sum;
                    };
                    if (nsg > 1) {  // valid in the lanes of sample group 0
                        a0 = groups(a0);
                        a1 = groups(a1);
                        a2 = groups(a2);
                    }
                    a0 += common[k0][0];
                    a1 += common[k0][1];
                    a2 += common[k0][2];
                    const float4 T = __ldg(J.target + pixel);
                    const int q = nth_set_bit(vm, k0) >> qshift;
                    _Pragma("unroll 1") for (int z = nextq; z < q; ++z) push_pair(h, z, 0.0);
                    if (kND > 0) {
                        const float3 res = f3(fixed_diff(a0, T.x, unsigned(spp), inv), fixed_diff(a1, T.y, unsigned(spp), inv),
                                              fixed_diff(a2, T.z, unsigned(spp), inv));
                        push_pair(h, q, double(fmaf(res.x, res.x, fmaf(res.y, res.y, res.z * res.z))));
#pragma unroll
                        for (int k = 0; k < kND; ++k) {
                            unsigned long long d = dacc[h * kND + k][lane] + fix_sum_signed(dhi[k], dlo[k]);
                            dacc[h * kND + k][lane] = 0ull;
                            if (nsg > 1) d = groups(d);
                            gsum[h * kND + k][lane] += double(comp3(res, k % 3) * (signed_word_to_float((long long)d) * inv));
                        }
                    } else {
                        push_pair(h, q, pixel_sq_error(a0, a1, a2, T, unsigned(spp), inv));
                    }
                }
                if (ends) {
                    nextq = (nth_set_bit(vm, k0) >> qshift) + 1;
                    ++k0;
                    s0 = 0;
                } else {
                    s0 += i1 - i0;
                }
                i0 = i1;
            }
        }
        for (int h = 0; h < nh; ++h) {
            _Pragma("unroll 1") for (int z = nextq; z < qend; ++z) push_pair(h, z, 0.0);
            if (kND > 0 && ks == 0 && gi + 32 * h < R) {
#pragma unroll
                for (int k = 0; k < kND; ++k) replay_store<kND>(J, item, r0 + gi + 32 * h, 1 + k, gsum[h * kND + k][lane]);
            }
        }
        __syncwarp();
        if (J.parts > 1) replay_combine<kND>(J, item, lane);
    }
    }
    if (kCount) {
        const unsigned v[kNumCounters] = {warp_sum_u(cnt.sph), warp_sum_u(cnt.quad), warp_sum_u(cnt.box),
                                          warp_sum_u(cnt.paths), warp_sum_u(cnt.vertices), warp_sum_u(cnt.shadow),
                                          warp_sum_u(cnt.rays), 0u};
        if (lane == 0)
            for (int i = 0; i < kNumCounters; ++i) atomicAdd(L.counters + i, (unsigned long long)v[i]);
    }
}

// ---------------------------------------------------------------------------
// k_trace_prefix: path vertices shared up to the first ray that could meet a moving object (a3-a5)
// ---------------------------------------------------------------------------
// For a job of R <= 64 renders whose perturbed primitives include every emitter and at least one
// that is not black, and whose materials are not bound (e.g. a moving ball and light): the renders'
// paths agree until one of their rays could meet a perturbed primitive, and differ before that only
// in the next-event estimates. A work item is one pixel block of all renders, taken by a
// CTA of kPrefixWarps warps; warp w takes the pixel slots of positions q = 8w .. 8w + 7 of
// the bit-reversed order. For each pixel, 32 samples at a time:
//   phase A  lane = sample: the path is traced once in the invariant scene, keeping its
//            diffuse vertices (PrefixLane) and its end: left the scene (the background term),
//            ended, or stopped where a ray could meet a perturbed primitive;
//   phase B  lane = render (lane and lane + 32; with R <= 16, render lane mod G of sample
//            group lane / G, G the power of two >= R): for each sample that adds anything,
//            the render's own next-event estimates at the kept vertices (occlusion tested
//            against the primitives the vertex's cull mask leaves), then the background term
//            or, for a stopped path, the rest of the path traced in the render's scene (as in
//            k_trace_group).
// Each render's radiance is the same sum, term by term and in the same order, as tracing
// the path in that render alone, so with the same block shape every partial is
// bit-identical to the per-render kernel's; the warps' subtrees of the pairwise pixel sum
// are combined as that sum's top two levels.
// Replay shares such a path further, but where some renders part from it and others do not, a warp
// waits for both; here all renders of a stopped path go on side by side (237 x 141, 16 renders at 16 spp,
// replayed and here: a glass ball moving beside the light 540 and 337 us, a grey box beside the GI box's
// light 4.06 and 1.77 ms). Bound by instruction issue like the other render kernels.
constexpr int kPrefixCap = 2;      // diffuse vertices kept per path
constexpr int kPrefixFields = 13;  // po, ns, beta * albedo, the emitter point (lu, lv), emitter li, cull mask
constexpr int kPrefixWarps = kGroupBlock / 32;
constexpr int kPrefixSlots = 32 / kPrefixWarps;
static_assert(kPrefixSlots == 8, "the warps' subtrees are the pairwise sum's levels 0-2");
constexpr int kPrefixMinBlocks = 5;  // <= 102 registers: 20 resident warps per SM

struct PrefixLane {
    const float4* ulo;   // as ReplayLane's
    const float4* uhi;
    const float4* ball;
    int n_var;
    unsigned skip;
    float* ent;          // the warp's kept vertices: ent[(k * kPrefixFields + field) * 32 + lane]
    int lane;
    int n;               // vertices kept by this lane's path
    bool miss;           // the path ended by leaving the scene
};
struct PrefixWarp {
    float ent[kPrefixCap * kPrefixFields * 32];  // kept vertices of the warp's 32 paths
    float st[10][32];                            // end state: o, d, beta, vertex b (bits)
    int n[32];                                   // vertices kept
    int kind[32];                                // 0 ended, 1 left the scene, 2 stopped (specular flag: 4)
    double pair[2][3][32];                       // pairwise-sum stacks of the lane's two renders
};
struct PrefixSmem {
    GroupScene scene;  // the invariant part (render 0's records of the other primitives)
    TraceJob job;
    float4 tab[kPrefixTabRows];  // per-render rows (as k_trace_group's), R x gstride
    float4 ulo[kMaxVariant], uhi[kMaxVariant];
    float4 ball[kGroupPrims];
    double sub[kPrefixWarps][64];
    PrefixWarp w[kPrefixWarps];
    unsigned item;
    int job_index;
};

// One vertex of a path in the invariant scene (as advance; no invariant primitive emits): kAffected
// where the renders trace on themselves, from the path's present ray.
template <bool kCount>
__device__ __forceinline__ int prefix_vertex(const GroupScene& S, int depth, int rr_start, Path& p, PrefixLane& E,
                                             Counters& cnt) {
    const Hit h = closest_hit<kCount, true>(S, p.o, p.d, cnt, E.skip);
    if (replay_touch<kCount>(E, p.o, p.d, h.slot < 0 ? 3.0e38f : h.t, cnt)) return kAffected;
    if (h.slot < 0) {
        E.miss = true;  // the background term is added per render, after its vertex terms
        return kEnded;
    }
    if (kCount) ++cnt.vertices;
    const float3 pt = p.o + p.d * h.t;
    int mat;
    const float3 ng = surface_normal(static_cast<const float4*>(S.prim[h.slot]), h.type, pt, p.o, p.d, mat);
    const float4 m0 = S.mat[mat][0];
    const int mtype = as_int(m0.w);
    const float3 albedo = xyz(m0);
    const bool last = p.b + 1 >= depth, rr = !last && rr_start >= 0 && p.b >= rr_start;
    uint4 w1 = make_uint4(0u, 0u, 0u, 0u);
    if (mtype == kDiffuse) {
        const float3 ns = dot3(ng, p.d) < 0.0f ? ng : ng * -1.0f;
        const float3 po = pt + ns * kEps;
        const uint4 w0 = path_words<true>(S, p.pixel, p.s, p.b, 0);
        if (S.n_lights > 1 || rr) w1 = path_words<true>(S, p.pixel, p.s, p.b, 1);
        if (S.n_lights > 0) {  // kept for the renders' own estimates (the renders' emitters differ)
            if (E.n == kPrefixCap) return kAffected;
            float* e = E.ent + E.n * kPrefixFields * 32 + E.lane;
            const float3 ba = p.beta * albedo;
            const int li = nee_light(S, w1.x);
            e[0] = po.x; e[32] = po.y; e[64] = po.z;
            e[96] = ns.x; e[128] = ns.y; e[160] = ns.z;
            e[192] = ba.x; e[224] = ba.y; e[256] = ba.z;
            e[288] = u01(w0.x); e[320] = u01(w0.y); e[352] = __int_as_float(li);
            e[384] = __uint_as_float(shadow_cull(S, E, po, S.light[li].y));
            ++E.n;
        }
        if (last) return kEnded;
        p.d = normalized(diffuse_dir(ns, u01(w0.z), u01(w0.w)));
        p.o = po;
        p.specular = false;
    } else {
        if (last) return kEnded;
        if (rr || mtype == kDielectric) w1 = path_words<true>(S, p.pixel, p.s, p.b, 1);
        if (mtype == kMirror) {
            const float3 ns = dot3(ng, p.d) < 0.0f ? ng : ng * -1.0f;
            p.d = normalized(p.d - ns * (2.0f * dot3(p.d, ns)));
            p.o = pt + ns * kEps;
        } else {
            dielectric(p, pt, ng, S.mat[mat][1].w, u01(w1.z));
        }
        p.specular = true;
    }
    p.beta = p.beta * albedo;
    if (maxc(p.beta) <= 0.0f) return kEnded;
    if (rr) {  // Russian roulette on slot 1's second uniform
        const float q = fminf(0.95f, maxc(p.beta));
        if (u01(w1.y) >= q) return kEnded;
        p.beta = p.beta * rcp_fast(q);
    }
    ++p.b;
    return kLive;
}

template <bool kCount>
__global__ void __launch_bounds__(kGroupBlock, kPrefixMinBlocks) k_trace_prefix(const __grid_constant__ TraceLaunch L) {
    __shared__ PrefixSmem E;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    PrefixWarp& Wp = E.w[warp];
    const TraceJob& J = E.job;
    int cur_job = -1;
    Counters cnt{0u, 0u, 0u, 0u, 0u, 0u, 0u, 0u};
    if (!L.jobs) {  // a single job's descriptor is host data: copied before the wait
        const unsigned* src = reinterpret_cast<const unsigned*>(&L.job0);
        unsigned* dst = reinterpret_cast<unsigned*>(&E.job);
        for (int i = threadIdx.x; i < int(sizeof(TraceJob) / 4); i += kGroupBlock) dst[i] = src[i];
    }
    __syncthreads();
    pdl_enter();
    for (;;) {
        if (threadIdx.x == 0) {
            const unsigned item = atomicAdd(L.queue, 1u);
            int j = 0;
            if (item < unsigned(L.total_items) && L.jobs) {
                int lo = 0, hi = L.njobs - 1;
                while (lo < hi) {
                    const int mid = (lo + hi + 1) / 2;
                    if (L.jobs[mid].item_begin <= int(item)) lo = mid; else hi = mid - 1;
                }
                j = lo;
            }
            E.item = item;
            E.job_index = j;
        }
        __syncthreads();
        const unsigned item = E.item;
        const int j = E.job_index;
        if (item >= unsigned(L.total_items)) break;
        if (j != cur_job) {  // stage the job, its invariant scene, per-render rows and union bounds
            if (L.jobs) {
                const unsigned* src = reinterpret_cast<const unsigned*>(L.jobs + j);
                unsigned* dst = reinterpret_cast<unsigned*>(&E.job);
                for (int i = threadIdx.x; i < int(sizeof(TraceJob) / 4); i += kGroupBlock) dst[i] = src[i];
                __syncthreads();
            }
            if (J.R < 1 || J.R > 64 || J.R * J.gstride > kPrefixTabRows || J.gstride < J.var_rows || J.n_var < 1 ||
                J.n_var > kMaxVariant || J.n_prims > kGroupPrims || J.n_mats > kGroupMats) {
                if (threadIdx.x == 0) atomicOr(L.status, kStatusBadItem);
                break;
            }
            if (warp == 0) stage_group_scene(E.scene, J, 0, lane);
            const int stride = J.gstride, n = J.n_var, nr = J.var_rows;
            for (int i = threadIdx.x; i < J.R * stride; i += kGroupBlock) {
                const int r = i / stride, q = i - r * stride;
                const InstScene& R = J.scenes[r];
                float4 v;
                if (q < nr) v = __ldg(&R.prim[J.row_src[q] >> 1][J.row_src[q] & 1]);
                else v = __ldg(reinterpret_cast<const float4*>(R.light_area) + (q - nr));  // emitter areas
                E.tab[q * J.R + r] = v;  // field-major, as k_trace_group's table
            }
            __syncthreads();
            if (warp == 1 && lane < J.n_prims && lane < kCullBits)
                E.ball[lane] = prim_ball(E.scene.prim[lane], lane < E.scene.n_sph ? kSphere
                                                             : (lane < E.scene.n_sph + E.scene.n_quad ? kQuad : kBox));
            if (warp == 0) {
                for (int k = 0; k < n; ++k) {
                    const int slot = nth_set_bit(J.var_prims, k);
                    const int type = slot < E.scene.n_sph ? kSphere : (slot < E.scene.n_sph + E.scene.n_quad ? kQuad : kBox);
                    float3 lo = f3(INFINITY, INFINITY, INFINITY), hi = f3(-INFINITY, -INFINITY, -INFINITY);
                    for (int r = lane; r < J.R; r += 32) {
                        float3 a, c;
                        const SRec own{E.tab + ((J.var_offs >> (8 * k)) & 255u) * J.R + r, J.R, type == kQuad ? 1 : 2, E.scene.prim[slot]};
                        prim_bounds(own, type, a, c);
                        lo = f3(fminf(lo.x, a.x), fminf(lo.y, a.y), fminf(lo.z, a.z));
                        hi = f3(fmaxf(hi.x, c.x), fmaxf(hi.y, c.y), fmaxf(hi.z, c.z));
                    }
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) {
                        lo.x = fminf(lo.x, __shfl_xor_sync(kFull, lo.x, o));
                        lo.y = fminf(lo.y, __shfl_xor_sync(kFull, lo.y, o));
                        lo.z = fminf(lo.z, __shfl_xor_sync(kFull, lo.z, o));
                        hi.x = fmaxf(hi.x, __shfl_xor_sync(kFull, hi.x, o));
                        hi.y = fmaxf(hi.y, __shfl_xor_sync(kFull, hi.y, o));
                        hi.z = fmaxf(hi.z, __shfl_xor_sync(kFull, hi.z, o));
                    }
                    if (lane == 0) {
                        E.ulo[k] = make_float4(lo.x, lo.y, lo.z, 0.f);
                        E.uhi[k] = make_float4(hi.x, hi.y, hi.z, 0.f);
                    }
                }
            }
            __syncthreads();
            cur_job = j;
        }
        const int t = int(item) - J.item_begin;
        if (t < 0 || t >= J.tiles) {
            if (threadIdx.x == 0) atomicOr(L.status, kStatusBadItem);
            break;
        }
        const int R = J.R, nh = R > 32 ? 2 : 1, stride = J.gstride;
        // phase B lanes: render gi = lane mod G of sample group ks = lane / G (G the power of
        // two >= R, at most 32): with few renders a warp takes 32 / G samples at a time
        const int G = R >= 32 ? 32 : (R <= 1 ? 1 : 1 << (32 - __clz(R - 1)));
        const int nsg = 32 / G, gi = lane % G, ks = lane / G;
        const int areas = stride > J.var_rows ? 1 : 0;
        const int x0 = (t % J.tiles_x) * J.bw, y0 = (t / J.tiles_x) * J.bh;
        const int vw = min(J.bw, J.W - x0), vh = min(J.bh, J.H - y0);
        const int npx = vw * vh;
        const unsigned magic_w = 0xffffffffu / unsigned(vw) + 1u;
        const float inv = mean_scale(J.spp);
        PrefixLane el{E.ulo, E.uhi, E.ball, J.n_var, J.var_prims, Wp.ent, lane, 0, false};
        const bool bg_nonzero = E.scene.bg.x != 0.0f || E.scene.bg.y != 0.0f || E.scene.bg.z != 0.0f;
        double sub[2] = {0.0, 0.0};
        // The loops below stay rolled: unrolled copies of the tracer overflow the instruction
        // cache (measured on the caustic step: 13.1 ms unrolled, 11.0 ms rolled).
#pragma unroll 1
        for (int qq = 0; qq < kPrefixSlots; ++qq) {
            const int slot = brev5(warp * kPrefixSlots + qq);  // pixels in bit-reversed slot order
            double e[2] = {0.0, 0.0};
            if (slot < npx) {
                const int row = div_magic(slot, vw, magic_w);
                const int px = x0 + slot - row * vw, py = y0 + row;
                unsigned long long acc[2][3] = {{0ull, 0ull, 0ull}, {0ull, 0ull, 0ull}};
                for (int s0 = 0; s0 < J.spp; s0 += 32) {
                    // ---- phase A: one path per lane, traced once for all renders ----------
                    __syncwarp();  // phase B of the previous samples is done with the table
                    bool work = false;  // does the sample add anything to a render?
                    if (s0 + lane < J.spp) {
                        Path p;
                        start_path<true>(E.scene, J.W, J.H, px, py, s0 + lane, slot, p);
                        if (kCount) ++cnt.paths;
                        el.n = 0;
                        el.miss = false;
                        int res;
                        while ((res = prefix_vertex<kCount>(E.scene, J.depth, J.rr_start, p, el, cnt)) == kLive) {
                        }
                        Wp.n[lane] = el.n;
                        Wp.kind[lane] = (res == kAffected ? 2 : (el.miss ? 1 : 0)) | (p.specular ? 4 : 0);
                        Wp.st[0][lane] = p.o.x;
                        Wp.st[1][lane] = p.o.y;
                        Wp.st[2][lane] = p.o.z;
                        Wp.st[3][lane] = p.d.x;
                        Wp.st[4][lane] = p.d.y;
                        Wp.st[5][lane] = p.d.z;
                        Wp.st[6][lane] = p.beta.x;
                        Wp.st[7][lane] = p.beta.y;
                        Wp.st[8][lane] = p.beta.z;
                        Wp.st[9][lane] = __int_as_float(p.b);
                        work = el.n > 0 || res == kAffected || (el.miss && bg_nonzero);
                    }
                    // ---- phase B: each render's terms of each sample, in sample order -----
                    // (samples that add nothing to any render -- no kept vertex, not stopped,
                    // no background term -- are passed over: their sums would add zero)
                    __syncwarp();
                    unsigned todo = __ballot_sync(kFull, work);
#pragma unroll 1
                    while (todo) {
                        int jj = -1;  // sample group ks takes the ks-th of the next nsg samples
                        for (int i = 0; i < nsg && todo; ++i) {
                            if (i == ks) jj = __ffs(todo) - 1;
                            todo &= todo - 1u;
                        }
                        if (jj < 0) continue;
                        const int nk = Wp.n[jj], kind = Wp.kind[jj];
#pragma unroll 1
                        for (int h = 0; h < nh; ++h) {
                            const int r = gi + 32 * h;
                            if (r >= R) continue;
                            const GroupLane gl{E.tab + r, J.var_prims, 0u, J.var_offs, J.var_rows, areas, nullptr, 0, R};
                            float3 Lr = f3(0.f, 0.f, 0.f);
#pragma unroll 1
                            for (int k = 0; k < nk; ++k) {
                                const float* en = Wp.ent + k * kPrefixFields * 32 + jj;
                                const float3 po = f3(en[0], en[32], en[64]), nsv = f3(en[96], en[128], en[160]);
                                float3 wi;
                                float dist, g;
                                int lmat;
                                if (nee_to<kCount, false, true>(E.scene, po, nsv, en[288], en[320],
                                                                __float_as_int(en[352]), cnt, __float_as_uint(en[384]),
                                                                &gl, wi, dist, g, lmat))
                                    Lr = nee_add(Lr, f3(en[192], en[224], en[256]), xyz(E.scene.mat[lmat][1]), g);
                            }
                            const float3 beta = f3(Wp.st[6][jj], Wp.st[7][jj], Wp.st[8][jj]);
                            if ((kind & 3) == 1) {
                                Lr = bg_add(Lr, beta, xyz(E.scene.bg));
                            } else if ((kind & 3) == 2) {  // the rest of the path in render r's scene
                                Path p;
                                p.o = f3(Wp.st[0][jj], Wp.st[1][jj], Wp.st[2][jj]);
                                p.d = f3(Wp.st[3][jj], Wp.st[4][jj], Wp.st[5][jj]);
                                p.beta = beta;
                                p.L = Lr;
                                p.pixel = unsigned(py * J.W + px);
                                p.s = s0 + jj;
                                p.b = __float_as_int(Wp.st[9][jj]);
                                p.slot = slot;
                                p.specular = (kind & 4) != 0;
                                p.seg = 0u;
                                Lr = replay_alone<kCount>(E.scene, J.depth, J.rr_start, gl, p, cnt);
                            }
                            if (Lr.x != 0.0f || Lr.y != 0.0f || Lr.z != 0.0f) {
                                acc[h][0] += to_fixed(Lr.x);
                                acc[h][1] += to_fixed(Lr.y);
                                acc[h][2] += to_fixed(Lr.z);
                            }
                        }
                    }
                }
                for (int o = G; o < 32; o <<= 1) {  // the render's other sample groups
                    acc[0][0] += __shfl_xor_sync(kFull, acc[0][0], o);
                    acc[0][1] += __shfl_xor_sync(kFull, acc[0][1], o);
                    acc[0][2] += __shfl_xor_sync(kFull, acc[0][2], o);
                }
                const float4 T = __ldg(J.target + size_t(py) * J.W + px);
                for (int h = 0; h < nh; ++h)
                    e[h] = pixel_sq_error(acc[h][0], acc[h][1], acc[h][2], T, unsigned(J.spp), inv);
            }
            for (int h = 0; h < 2; ++h) {  // levels 0-2 of the pairwise sum over this warp's slots
                double v = e[h];
                int l = 0;
                for (; (qq >> l) & 1; ++l) v = Wp.pair[h][l][lane] + v;
                if (l < 3) Wp.pair[h][l][lane] = v;
                else sub[h] = v;
            }
        }
        for (int h = 0; h < nh; ++h)
            if (ks == 0 && gi + 32 * h < R) E.sub[warp][gi + 32 * h] = sub[h];
        __syncthreads();
        for (int r = threadIdx.x; r < R; r += kGroupBlock)  // a5: levels 3 and 4
            J.partials[size_t(r) * J.tiles + t] = (E.sub[0][r] + E.sub[1][r]) + (E.sub[2][r] + E.sub[3][r]);
        __syncthreads();
    }
    if (kCount) {
        const unsigned v[kNumCounters] = {warp_sum_u(cnt.sph), warp_sum_u(cnt.quad), warp_sum_u(cnt.box),
                                          warp_sum_u(cnt.paths), warp_sum_u(cnt.vertices), warp_sum_u(cnt.shadow),
                                          warp_sum_u(cnt.rays), 0u};
        if (lane == 0)
            for (int i = 0; i < kNumCounters; ++i) atomicAdd(L.counters + i, (unsigned long long)v[i]);
    }
}

// Per-render pass of a path-sharing job: render r traces again each recorded path one of
// whose kept segments touches render r's bounds of a perturbed primitive, and adds its radiance minus the shared-pass radiance (2^-32 fixed point,
// modulo 2^64) to the render's image-sized buffer with global atomic adds -- integer
// sums, so the order does not matter and the block sums equal those of tracing every
// path in every render.
// Work distribution: warp g starts on render g mod R and streams that render's paths.
// Batches of 32 list entries are claimed from the render's cursor, the entries that
// render r must trace are compacted into a per-warp ring, and a lane whose path ends takes the
// next ring entry at once, so the warp's pool only drains when the render's list is
// used up; the warp then moves on to the next render with entries left.
constexpr int kAffRing = 64;  // ring entries per warp (the ring never holds more than 63)

template <bool kCount>
__global__ void __launch_bounds__(kBlock, kTraceMinBlocks) k_trace_affected(const __grid_constant__ TraceLaunch L) {
    __shared__ InstScene s_scene[kWarps];
    __shared__ TraceJob s_job[kWarps];
    __shared__ unsigned s_ring[kWarps][kAffRing];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned lt_mask = (1u << lane) - 1u;
    InstScene& S = s_scene[warp];
    TraceJob& J = s_job[warp];
    unsigned* ring = s_ring[warp];
    const int gwarp = int(blockIdx.x) * kWarps + warp;
    Counters cnt{0u, 0u, 0u, 0u, 0u, 0u, 0u, 0u};
    const int njobs = L.jobs ? L.njobs : 1;
    for (int jb = 0; jb < njobs; ++jb) {  // the jobs of a packed launch one after another
    {  // job descriptors are host data: the first is copied before the wait on the previous kernel
        const unsigned* src = reinterpret_cast<const unsigned*>(L.jobs ? L.jobs + jb : &L.job0);
        unsigned* dst = reinterpret_cast<unsigned*>(&J);
        for (int i = lane; i < int(sizeof(TraceJob) / 4); i += 32) dst[i] = src[i];
        __syncwarp();
        if (jb == 0) pdl_enter();
    }
    const bool job_shares = J.share != 0;
    __syncwarp();  // every lane has read the descriptor before the next copy may overwrite it
    if (!job_shares) continue;
    const unsigned n_codes = __ldcg(J.share_ctl + 1);
    const unsigned magic_W = 0xffffffffu / unsigned(J.W) + 1u;
    for (int k = 0; k < J.R; ++k) {
        {  // the next render, in the order gwarp + k, ..., with entries left: 32 cursors at a time
            const bool left = k + lane < J.R && __ldcg(J.aff_cursor + (gwarp + k + lane) % J.R) < n_codes;
            const unsigned m = __ballot_sync(kFull, left);
            if (!m) {
                k += 31;
                continue;
            }
            k += __ffs(m) - 1;
        }
        const int r = (gwarp + k) % J.R;
        unsigned* cursor = J.aff_cursor + r;
        {  // stage render r's scene
            const float4* src = reinterpret_cast<const float4*>(J.scenes + r);
            float4* dst = reinterpret_cast<float4*>(&S);
            constexpr int kHead = int(offsetof(InstScene, mat) / 16);
            constexpr int kPrim = int(offsetof(InstScene, prim) / 16);
            const int nm = 2 * J.n_mats, np = 4 * J.n_prims;
            for (int i = lane; i < kHead + nm + np; i += 32) {
                const int o = (i < kHead + nm) ? i : kPrim + (i - kHead - nm);
                dst[o] = __ldg(src + o);
            }
            __syncwarp();
        }
        unsigned long long* acc = J.acc_aff + size_t(r) * J.W * J.H * 3;
        unsigned head = 0, tail = 0;  // ring positions, the same in every lane
        bool src_done = false, alive = false;
        Path p;
        for (;;) {
            while (!src_done && tail - head < 32u) {  // claim 32 entries, keep render r's
                unsigned base = 0;
                if (lane == 0) base = atomicAdd(cursor, 32u);
                base = __shfl_sync(kFull, base, 0);
                if (base >= n_codes) {
                    src_done = true;
                    break;
                }
                const unsigned e = base + unsigned(lane);
                bool need = false;
                if (e < n_codes) {  // does a kept segment of the path touch render r's bounds?
                    const unsigned sw = __ldcg(J.aff_segw + e);
                    need = (sw & kSegAll) != 0u;
                    const unsigned s0 = ((sw >> 3) - 1u) * unsigned(kSeg), ns = need ? 0u : (sw & 7u);
                    for (unsigned q = 0; q < ns && !need; ++q) {
                        const float4 A = __ldcg(J.seg_pool + 2 * size_t(s0 + q));
                        const float4 B = __ldcg(J.seg_pool + 2 * size_t(s0 + q) + 1);
                        const float3 o = xyz(A), inv = rcp3(xyz(B));
                        const float tm = A.w * 1.0001f + 1e-3f;
                        for (int k = 0; k < J.n_var && !need; ++k) {
                            const float4* bx = J.var_box + (size_t(r) * kMaxVariant + k) * 2;
                            need = slab_touch(xyz(__ldg(bx)), xyz(__ldg(bx + 1)), o, inv, tm);
                        }
                    }
                }
                const unsigned nb = __ballot_sync(kFull, need);
                if (need) ring[(tail + __popc(nb & lt_mask)) % kAffRing] = e;
                tail += unsigned(__popc(nb));
            }
            __syncwarp();
            const unsigned fr = __ballot_sync(kFull, !alive);  // lanes free for a new path
            const unsigned avail = tail - head, rank = unsigned(__popc(fr & lt_mask));
            if (!alive && rank < avail) {
                const unsigned e = ring[(head + rank) % kAffRing];
                const unsigned code = __ldcg(J.aff_codes + e), sw = __ldcg(J.aff_segw + e);
                const int pixel = int(code >> 6), smp = int(code & 63u);
                if (sw == kSegFull) {
                    const int y = div_magic(pixel, J.W, magic_W);
                    start_path(S, J.W, J.H, pixel - y * J.W, y, smp, int(e), p);
                } else {  // resume where the path's renders part
                    const float4* st = J.seg_state + 4 * size_t(((sw & ~kSegAll) >> 3) - 1u);
                    const float4 a = __ldcg(st), b = __ldcg(st + 1), c = __ldcg(st + 2), q = __ldcg(st + 3);
                    p.o = f3(a.x, a.y, a.z);
                    p.d = f3(a.w, b.x, b.y);
                    p.beta = f3(b.z, b.w, c.x);
                    p.L = f3(c.y, c.z, c.w);
                    p.b = __float_as_int(q.x);
                    p.specular = __float_as_int(q.y) != 0;
                    p.pixel = unsigned(pixel);
                    p.s = smp;
                    p.slot = int(e);
                }
                if (kCount) ++cnt.paths;
                alive = true;
            }
            head += min(avail, unsigned(__popc(fr)));
            __syncwarp();
            if (!__any_sync(kFull, alive)) break;  // ring empty and the render's list used up
            int st = kLive;
            if (alive) st = advance<kCount, false>(S, J.depth, J.rr_start, p, cnt);
            if (alive && st != kLive) {
                unsigned long long* a = acc + size_t(p.pixel) * 3;
                const float* ls = J.aff_lsh + 3 * size_t(p.slot);
                const unsigned long long dx = to_fixed(p.L.x) - to_fixed(__ldcg(ls + 0));
                const unsigned long long dy = to_fixed(p.L.y) - to_fixed(__ldcg(ls + 1));
                const unsigned long long dz = to_fixed(p.L.z) - to_fixed(__ldcg(ls + 2));
                if (dx) atomicAdd(a + 0, dx);
                if (dy) atomicAdd(a + 1, dy);
                if (dz) atomicAdd(a + 2, dz);
                if (dx | dy | dz) {  // mark the pixel as corrected in render r
                    unsigned* fw = J.aff_flags + size_t(r) * J.flag_words + (p.pixel >> 5);
                    const unsigned bit = 1u << (p.pixel & 31u);
                    if (!(__ldcg(fw) & bit)) atomicOr(fw, bit);
                }
                alive = false;
            }
        }
        __syncwarp();
    }
    }
    if (kCount) {
        const unsigned v[kNumCounters] = {warp_sum_u(cnt.sph), warp_sum_u(cnt.quad), warp_sum_u(cnt.box),
                                          warp_sum_u(cnt.paths), warp_sum_u(cnt.vertices), warp_sum_u(cnt.shadow),
                                          warp_sum_u(cnt.rays), 0u};
        if (lane == 0)
            for (int i = 0; i < kNumCounters; ++i) atomicAdd(L.counters + i, (unsigned long long)v[i]);
    }
}

// Epilogue pass of a path-sharing job: one item per listed block, all renders. Lanes form
// segments of `pw` lanes (one render each, one pixel per lane); a segment's error sum uses
// the same shuffle tree as a full warp whose other lanes hold zeros, so the partial is
// bit-identical to the per-render path. Clears the affected radiance it read, so the
// buffers are zero for the next step.
__global__ void __launch_bounds__(kBlock) k_shared_epilogue(const __grid_constant__ TraceLaunch L) {
    __shared__ TraceJob s_job[kWarps];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    TraceJob& J = s_job[warp];
    const int njobs = L.jobs ? L.njobs : 1;
    for (int jb = 0; jb < njobs; ++jb) {  // the jobs of a packed launch one after another
    {  // job descriptors are host data: the first is copied before the wait on the previous kernel
        const unsigned* src = reinterpret_cast<const unsigned*>(L.jobs ? L.jobs + jb : &L.job0);
        unsigned* dst = reinterpret_cast<unsigned*>(&J);
        for (int i = lane; i < int(sizeof(TraceJob) / 4); i += 32) dst[i] = src[i];
        __syncwarp();
        if (jb == 0) pdl_enter();
    }
    const bool job_shares = J.share != 0;
    __syncwarp();  // every lane has read the descriptor before the next copy may overwrite it
    if (!job_shares) continue;
    const unsigned n_items = __ldcg(J.share_ctl + 0);
    const float inv = mean_scale(J.spp);
    const unsigned gw = blockIdx.x * kWarps + unsigned(warp), nw = gridDim.x * kWarps;
    for (unsigned item = gw; item < n_items; item += nw) {  // listed blocks cost alike: a static split
        const int t = __ldcg(J.aff_tiles + item);
        if (t < 0 || t >= J.tiles) {
            if (lane == 0) atomicOr(L.status, kStatusBadItem);
            break;
        }
        const int x0 = (t % J.tiles_x) * J.bw, y0 = (t / J.tiles_x) * J.bh;
        const int vw = min(J.bw, J.W - x0), vh = min(J.bh, J.H - y0);
        const int npx = vw * vh;
        const int pw = npx <= 8 ? 8 : (npx <= 16 ? 16 : 32);  // lanes per render segment
        const int G = 32 / pw, sub = lane / pw, pl = lane % pw;
        const int px = x0 + pl % vw, py = y0 + pl / vw;
        const bool pix_ok = pl < npx && px < J.W && py < J.H;
        const unsigned long long* sh = J.share_acc + size_t(t) * 96;
        const unsigned long long s0 = pix_ok ? __ldcg(sh + pl) : 0ull, s1 = pix_ok ? __ldcg(sh + 32 + pl) : 0ull,
                                 s2 = pix_ok ? __ldcg(sh + 64 + pl) : 0ull;
        const float4 T = pix_ok ? __ldg(J.target + size_t(py) * J.W + px) : make_float4(0.f, 0.f, 0.f, 0.f);
        const size_t plane = size_t(J.W) * J.H * 3, pix3 = (size_t(py) * J.W + px) * 3;
        const unsigned pixel = pix_ok ? unsigned(py * J.W + px) : 0u, pbit = 1u << (pixel & 31u);
        constexpr int kBatch = 4;  // rounds whose loads are issued before any store
        for (int rb = 0; rb < J.R; rb += kBatch * G) {
            unsigned long long a[kBatch][3];
            bool corr[kBatch];  // render r corrected this pixel: read (and clear) its correction
#pragma unroll
            for (int q = 0; q < kBatch; ++q) {
                const int r = rb + q * G + sub;
                corr[q] = pix_ok && r < J.R &&
                          (__ldcg(J.aff_flags + size_t(r) * J.flag_words + (pixel >> 5)) & pbit) != 0u;
                const bool ok = corr[q];
                const unsigned long long* af = J.acc_aff + size_t(ok ? r : 0) * plane + (ok ? pix3 : 0);
                a[q][0] = ok ? __ldcg(af + 0) : 0ull;
                a[q][1] = ok ? __ldcg(af + 1) : 0ull;
                a[q][2] = ok ? __ldcg(af + 2) : 0ull;
            }
#pragma unroll
            for (int q = 0; q < kBatch; ++q) {
                const int r = rb + q * G + sub;
                double e = 0.0;
                if (pix_ok && r < J.R) {
                    if (corr[q]) {
                        unsigned long long* af = J.acc_aff + size_t(r) * plane + pix3;
                        af[0] = 0ull;
                        af[1] = 0ull;
                        af[2] = 0ull;
                    }
                    e = pixel_sq_error(s0 + a[q][0], s1 + a[q][1], s2 + a[q][2], T, unsigned(J.spp), inv);
                }
                for (int o = pw / 2; o > 0; o >>= 1) e += __shfl_xor_sync(kFull, e, o);
                if (pl == 0 && r < J.R) J.partials[size_t(r) * J.tiles + t] = e;
            }
        }
        __syncwarp();
    }
    }
}

// One Adam update (Sec. 3.4: Adam with PyTorch's default betas and eps) of one parameter
// in FP32, as PyTorch's FP32 Adam. The bias corrections 1 - beta^t are formed as
// -expm1(t log1p(beta - 1)), which keeps their relative accuracy while beta^t is near 1.
__device__ __forceinline__ void adam_update(float& th, float& m, float& v, float g, int t, float lr, float b1,
                                            float b2, float eps) {
    m = fmaf(b1, m, (1.0f - b1) * g);
    v = fmaf(b2, v, (1.0f - b2) * g * g);
    const float bc1 = -expm1f(float(t) * log1pf(b1 - 1.0f));
    const float bc2 = -expm1f(float(t) * log1pf(b2 - 1.0f));
    th -= lr * (m / bc1) / (sqrtf(v / bc2) + eps);
}

// ---------------------------------------------------------------------------
// k_finalize: a5 (per-render loss), a6 (gradient, Eq. 10), a7 (Adam)
// ---------------------------------------------------------------------------
// One 256-thread CTA per render of every job in the launch: L_r = (1/3HW) sum of the
// render's block partials in a fixed order (strided per thread into eight accumulators, a
// warp shuffle tree, then the eight warp sums in order). The CTA that completes a job's
// last render forms the gradient in FP64 (one warp per parameter) and applies Adam.
__global__ void __launch_bounds__(kBlock) k_finalize(const __grid_constant__ TraceLaunch L) {
    __shared__ double s_red[kBlock / 32];
    __shared__ int s_job, s_last;
    const int tid = threadIdx.x;
    if (tid == 0) {
        int j = 0;
        if (L.jobs) {
            int lo = 0, hi = L.njobs - 1;  // last job with fin_begin <= blockIdx.x
            while (lo < hi) {
                const int mid = (lo + hi + 1) / 2;
                if (L.jobs[mid].fin_begin <= int(blockIdx.x)) lo = mid; else hi = mid - 1;
            }
            j = lo;
        }
        s_job = j;
    }
    __syncthreads();
    pdl_enter();  // the job lookup above reads host data only
    const TraceJob& J = L.jobs ? L.jobs[s_job] : L.job0;
    const int r = int(blockIdx.x) - J.fin_begin;
    // fixed-order sum of src[i * stride], i < n: strided per thread into eight
    // accumulators, a warp shuffle tree, then the eight warp sums in order (thread 0)
    auto reduce = [&](const double* src, int n, int stride) -> double {
        double a[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) a[q] = 0.0;
        int i = tid;
        for (; i + 31 * kBlock < n; i += 32 * kBlock) {  // 32 loads in flight, then the same adds
            double v[32];
#pragma unroll
            for (int q = 0; q < 32; ++q) v[q] = __ldcg(src + size_t(i + q * kBlock) * stride);
#pragma unroll
            for (int q = 0; q < 32; ++q) a[q & 7] += v[q];
        }
        for (; i + 7 * kBlock < n; i += 8 * kBlock) {
#pragma unroll
            for (int q = 0; q < 8; ++q) a[q] += __ldcg(src + size_t(i + q * kBlock) * stride);
        }
        for (; i < n; i += kBlock) a[0] += __ldcg(src + size_t(i) * stride);
        double v = ((a[0] + a[1]) + (a[2] + a[3])) + ((a[4] + a[5]) + (a[6] + a[7]));
        v = warp_sum_d(v);
        if ((tid & 31) == 0) s_red[tid >> 5] = v;
        __syncthreads();
        double sum = 0.0;
        if (tid == 0)
            for (int w = 0; w < kBlock / 32; ++w) sum += s_red[w];
        __syncthreads();
        return sum;
    };
    const double lsum = reduce(J.partials + size_t(r) * J.tiles, J.tiles, 1);
    if (tid == 0) {
        const double Lr = lsum / (3.0 * double(J.W) * double(J.H));
        J.losses[r] = Lr;
        if (J.loss_out) J.loss_out[r] = float(Lr);
    }
    if (J.diff)  // pathwise estimator: render r's loss gradient (without the 2 / 3HW factor)
        for (int k = 0; k < J.diff_n; ++k) {
            const double gsum = reduce(J.gpartials + size_t(r) * J.tiles * J.diff_n + k, J.tiles, J.diff_n);
            if (tid == 0) J.rgrads[size_t(r) * kMaxDiff + k] = gsum;
        }
    if (tid == 0) {
        __threadfence();
        s_last = (atomicAdd(J.done, 1u) == unsigned(J.R - 1));
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    // a6: one warp per parameter, lanes over pairs (fixed order), FP64; a7: Adam in FP32
    const int t = J.step_dev ? __ldcg(J.step_dev) : 0;
    const int warp = tid >> 5, lane = tid & 31;
    for (int d = warp; d < (J.hd ? 0 : J.D); d += kBlock / 32) {  // hd: k_hd_grad
        double g = 0.0;
        if (J.diff) {  // Eq. 9: mean over renders of the pathwise loss gradients
            for (int q = lane; q < J.R; q += 32) g += __ldcg(J.rgrads + size_t(q) * kMaxDiff + d);
            g = warp_sum_d(g) * (2.0 / (3.0 * double(J.W) * double(J.H))) / double(J.R);
        } else if (J.antithetic) {
            const int P = J.R / 2;
            for (int p = lane; p < P; p += 32)
                g += double(J.w[size_t(2 * p) * J.D + d]) * (__ldcg(J.losses + 2 * p) - __ldcg(J.losses + 2 * p + 1));
            g = warp_sum_d(g) / double(2 * P);
        } else {
            for (int q = lane; q < J.R; q += 32) g += double(J.w[size_t(q) * J.D + d]) * __ldcg(J.losses + q);
            g = warp_sum_d(g) / double(J.R);
        }
        if (lane == 0) {
            const float gf = float(g);
            if (J.grad_out) J.grad_out[d] = gf;
            if (J.theta) adam_update(J.theta[d], J.m[d], J.v[d], gf, t + 1, J.lr, J.b1, J.b2, J.eps);
        }
    }
    __syncthreads();
    if (tid == 0) {
        if (J.step_dev) *J.step_dev = t + 1;
        *J.done = 0u;  // ready for the next launch
    }
}

// ---------------------------------------------------------------------------
// standalone Adam and raw Philox
// ---------------------------------------------------------------------------
__global__ void k_adam(int D, float* theta, float* m, float* v, const float* g, int t, float lr, float b1, float b2,
                       float eps) {
    const int d = blockIdx.x * blockDim.x + threadIdx.x;
    if (d >= D) return;
    adam_update(theta[d], m[d], v[d], g[d], t, lr, b1, b2, eps);
}

__global__ void k_philox(unsigned long long seed, unsigned c0, unsigned c1, unsigned c2, unsigned c3, int n,
                         uint4* out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    out[i] = philox(make_uint4(c0 + unsigned(i), c1, c2, c3), unsigned(seed), unsigned(seed >> 32));
}

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------
// Launch with the programmatic-stream-serialisation attribute (see pdl_enter).
template <typename... Args>
static cudaError_t launch_pdl_smem(void (*kernel)(Args...), int grid, int block, size_t smem, cudaStream_t stream,
                                   const Args&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(unsigned(grid));
    cfg.blockDim = dim3(unsigned(block));
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}
template <typename... Args>
static cudaError_t launch_pdl(void (*kernel)(Args...), int grid, int block, cudaStream_t stream, const Args&... args) {
    return launch_pdl_smem(kernel, grid, block, 0, stream, args...);
}

cudaError_t launch_instantiate(const InstLaunch& L, cudaStream_t stream) {
    if (L.total_blocks <= 0) return cudaSuccess;
    return launch_pdl(k_instantiate, L.total_blocks, kInstBlock, stream, L);
}

int trace_diff_blocks_per_sm() {
    int n = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_trace<false, false, false, 8>, kDiffBlock, 0);
    return n > 0 ? n : 1;
}

int trace_blocks_per_sm(bool render_mode) {
    int n = 0;
    if (render_mode)
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_trace<true, false, false, 0>, kBlock, 0);
    else
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_trace<false, false, false, 0>, kBlock, 0);
    return n > 0 ? n : 1;
}

int trace_group_blocks_per_sm() {
    int n = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_trace_group<false>, kGroupBlock, 0);
    return n > 0 ? n : 1;
}

// Kernel variant of a replay launch: bound materials, perturbed primitives, tangent slots. A
// packed launch runs the variant that covers all of its jobs.
constexpr size_t kReplaySmemMax = 160 * 1024;
static_assert(sizeof(ReplayHead) + kReplayTabRows * 16 +
                      kReplayWarps * replay_warp_bytes(replay_path_granules(64, true), 2, 32, 12) <= kReplaySmemMax,
              "the largest table, pool (depth 64) and tangent sums fit");
using ReplayKernel = void (*)(const TraceLaunch);
template <bool kCount>
static ReplayKernel replay_kernel_of(const TraceLaunch& L) {
    if (L.replay_chunked)
        return L.replay_move == 2 ? k_trace_replay<kCount, true, 2, 0, true>
                                  : (L.replay_move ? k_trace_replay<kCount, true, 1, 0, true>
                                                   : k_trace_replay<kCount, true, 0, 0, true>);
    if (L.diff_nd == 3) return k_trace_replay<kCount, true, 0, 3, false>;
    if (L.diff_nd == 6) return k_trace_replay<kCount, true, 0, 6, false>;
    if (L.diff_nd == 12) return k_trace_replay<kCount, true, 0, 12, false>;
    if (!L.replay_mat)
        return L.replay_move == 2 ? k_trace_replay<kCount, false, 2, 0, false> : k_trace_replay<kCount, false, 1, 0, false>;
    return L.replay_move == 2 ? k_trace_replay<kCount, true, 2, 0, false>
                              : (L.replay_move ? k_trace_replay<kCount, true, 1, 0, false>
                                               : k_trace_replay<kCount, true, 0, 0, false>);
}
static ReplayKernel replay_kernel(const TraceLaunch& L) {
    return L.counters ? replay_kernel_of<true>(L) : replay_kernel_of<false>(L);
}

int trace_replay_blocks_per_sm(const TraceLaunch& L) {
    const ReplayKernel k = replay_kernel(L);
    const size_t smem = replay_smem(L);
    int n = 0;
    // the same bound for every launch of the kernel: a later one may need more than this one
    if (smem > kReplaySmemMax ||
        cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, int(kReplaySmemMax)) != cudaSuccess)
        return 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k, kGroupBlock, smem) != cudaSuccess) return 0;
    return n;
}

int trace_prefix_blocks_per_sm() {
    int n = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_trace_prefix<false>, kGroupBlock, 0);
    return n > 0 ? n : 1;
}

cudaError_t launch_trace(const TraceLaunch& L, bool render_mode, int grid, cudaStream_t stream) {
    if (L.total_items <= 0) return cudaSuccess;
    const bool count = L.counters != nullptr;
    if (L.group == 3 && !render_mode)
        return launch_pdl(count ? k_trace_prefix<true> : k_trace_prefix<false>, grid, kGroupBlock, stream, L);
    if (L.group == 2 && !render_mode)
        return launch_pdl_smem(replay_kernel(L), grid, kGroupBlock, replay_smem(L), stream, L);
    if (L.group && !render_mode)
        return launch_pdl(count ? k_trace_group<true> : k_trace_group<false>, grid, kGroupBlock, stream, L);
    const bool share = !render_mode && L.share;
    if (render_mode) return launch_pdl(count ? k_trace<true, true, false, 0> : k_trace<true, false, false, 0>, grid, kBlock,
                                       stream, L);
    if (share) return launch_pdl(count ? k_trace<false, true, true, 0> : k_trace<false, false, true, 0>, grid, kBlock,
                                 stream, L);
    if (L.diff_nd == 4)
        return launch_pdl(count ? k_trace<false, true, false, 4> : k_trace<false, false, false, 4>, grid, kDiffBlock,
                          stream, L);
    if (L.diff_nd == 6)
        return launch_pdl(count ? k_trace<false, true, false, 6> : k_trace<false, false, false, 6>, grid, kDiffBlock,
                          stream, L);
    if (L.diff_nd == 8)
        return launch_pdl(count ? k_trace<false, true, false, 8> : k_trace<false, false, false, 8>, grid, kDiffBlock,
                          stream, L);
    return launch_pdl(count ? k_trace<false, true, false, 0> : k_trace<false, false, false, 0>, grid, kBlock, stream, L);
}

cudaError_t launch_trace_affected(const TraceLaunch& L, int grid, cudaStream_t stream) {
    return launch_pdl(L.counters ? k_trace_affected<true> : k_trace_affected<false>, grid, kBlock, stream, L);
}

cudaError_t launch_shared_epilogue(const TraceLaunch& L, int grid, cudaStream_t stream) {
    return launch_pdl(k_shared_epilogue, grid, kBlock, stream, L);
}

cudaError_t launch_finalize(const TraceLaunch& L, int n_renders, cudaStream_t stream) {
    if (n_renders <= 0) return cudaSuccess;
    return launch_pdl(k_finalize, n_renders, kBlock, stream, L);
}

cudaError_t launch_adam(int D, float* theta, float* m, float* v, const float* g, int t, float lr, float b1,
                        float b2, float eps, cudaStream_t stream) {
    k_adam<<<(D + 63) / 64, 64, 0, stream>>>(D, theta, m, v, g, t, lr, b1, b2, eps);
    return cudaGetLastError();
}

cudaError_t launch_philox(unsigned long long seed, unsigned c0, unsigned c1, unsigned c2, unsigned c3, int n,
                          uint32_t* out, cudaStream_t stream) {
    if (n <= 0) return cudaSuccess;
    k_philox<<<(n + 255) / 256, 256, 0, stream>>>(seed, c0, c1, c2, c3, n, reinterpret_cast<uint4*>(out));
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// High-dimensional parameters (texture scenes): a1 and a6/a7 over D > kMaxD
// ---------------------------------------------------------------------------
// Uniform number k of draw `index` (stream PERTURB): word k mod 4 of Philox block k / 4,
// the same counter layout as the small-D sampler of k_instantiate.
__device__ __forceinline__ float perturb_uniform(const HdDraws& H, unsigned index, unsigned step, int k) {
    const uint4 w = philox(make_uint4(index, unsigned(k >> 2), step, kTagPerturb << 28), unsigned(H.seed),
                           unsigned(H.seed >> 32));
    const unsigned x = (k & 3) == 0 ? w.x : ((k & 3) == 1 ? w.y : ((k & 3) == 2 ? w.z : w.w));
    return u01(x);
}

// Uniforms k and k + 1 of a draw (one Philox block unless k is a block's last word).
__device__ __forceinline__ float2 perturb_uniform_pair(const HdDraws& H, unsigned index, unsigned step, int k) {
    const uint4 w = philox(make_uint4(index, unsigned(k >> 2), step, kTagPerturb << 28), unsigned(H.seed),
                           unsigned(H.seed >> 32));
    const int q = k & 3;
    const unsigned xa = q == 0 ? w.x : (q == 1 ? w.y : (q == 2 ? w.z : w.w));
    unsigned xb;
    if (q < 3) {
        xb = q == 0 ? w.y : (q == 1 ? w.z : w.w);
    } else {
        xb = philox(make_uint4(index, unsigned(k >> 2) + 1u, step, kTagPerturb << 28), unsigned(H.seed),
                    unsigned(H.seed >> 32)).x;
    }
    return make_float2(u01(xa), u01(xb));
}

// Box-Muller normals 2m and 2m + 1 of a draw whose pairs start at uniform `base` (as
// bm_normal): (cos, sin) parts.
__device__ __forceinline__ float2 hd_normal_pair(const HdDraws& H, unsigned index, unsigned step, int base, int m) {
    const float2 ab = perturb_uniform_pair(H, index, step, base + 2 * m);
    const float rad = sqrtf(-2.0f * logf(ab.x));
    float sn, cs;
    sincospif(2.0f * ab.y, &sn, &cs);
    return make_float2(rad * cs, rad * sn);
}

__device__ __forceinline__ unsigned hd_step(const HdDraws& H) {
    return H.step + (H.step_dev ? unsigned(*H.step_dev) : 0u);
}

// Radial sampler (Sec. 3.2, reading R1) in D dimensions: the norm of the D Box-Muller
// normals and the chi_{D+1} radius (sum of (D+1)/2 exponentials, plus one more squared
// normal when D is even). Each draw's terms are split into norm_split contiguous parts,
// one CTA each, summed in FP64 in a fixed order; the CTA that finishes a draw's last part
// adds the parts in order.
__global__ void __launch_bounds__(kBlock) k_hd_norms(const HdDraws H) {
    __shared__ double s_z[kBlock / 32], s_r[kBlock / 32];
    __shared__ int s_last;
    const int split = H.norm_split, part = int(blockIdx.x) % split;
    const unsigned local = blockIdx.x / unsigned(split);
    pdl_enter();
    const unsigned index = local + unsigned(H.draw_begin), step = hd_step(H);
    const int D = H.D, n_exp = (D + 1) / 2, nz = D + (D % 2 == 0 ? 1 : 0), npair = (nz + 1) / 2;
    const int m0 = int((long long)npair * part / split), m1 = int((long long)npair * (part + 1) / split);
    const int e0 = int((long long)n_exp * part / split), e1 = int((long long)n_exp * (part + 1) / split);
    double zs = 0.0, rs = 0.0;
    for (int m = m0 + int(threadIdx.x); m < m1; m += kBlock) {  // normals 2m and 2m + 1
        const float2 z = hd_normal_pair(H, index, step, n_exp, m);
        const float q0 = z.x * z.x, q1 = z.y * z.y;
        if (2 * m < D) zs += double(q0); else rs += double(q0);
        if (2 * m + 1 < D) zs += double(q1); else if (2 * m + 1 < nz) rs += double(q1);
    }
    for (int j = e0 + int(threadIdx.x); j < e1; j += kBlock)
        rs += double(-2.0f * logf(perturb_uniform(H, index, step, j)));
    zs = warp_sum_d(zs);
    rs = warp_sum_d(rs);
    if ((threadIdx.x & 31) == 0) {
        s_z[threadIdx.x >> 5] = zs;
        s_r[threadIdx.x >> 5] = rs;
    }
    __syncthreads();
    HdNorm& N = H.norms[local];
    if (threadIdx.x == 0) {
        double z = 0.0, r = 0.0;
        for (int w = 0; w < kBlock / 32; ++w) {
            z += s_z[w];
            r += s_r[w];
        }
        N.part[part] = make_double2(z, r);
        __threadfence();
        s_last = atomicAdd(&N.ctr, 1u) == unsigned(split - 1);
    }
    __syncthreads();
    if (!s_last) return;
    // the parts loaded side by side, then added in order by one thread (one thread loading each
    // part as it adds it waited a round trip to L2 per part: 36 at D = 49,152)
    __threadfence();
    __shared__ double2 s_part[kNormSplitMax];
    if (int(threadIdx.x) < split) s_part[threadIdx.x] = __ldcg(&N.part[threadIdx.x]);
    __syncthreads();
    if (threadIdx.x == 0) {
        double z = 0.0, r = 0.0;
        for (int q = 0; q < split; ++q) {
            z += s_part[q].x;
            r += s_part[q].y;
        }
        N.v = make_float2(float(sqrt(z)), float(sqrt(r)));
        N.ctr = 0u;  // ready for the next launch
    }
}

// One thread per (render, pair of parameters 2m, 2m + 1): tau, w and theta + tau of every
// sampler (as the small-D sampler, per dimension), antithetic renders negated. A pair of
// Box-Muller normals comes from one pair of uniforms, so a thread forms both.
__global__ void __launch_bounds__(kBlock) k_hd_perturb(const HdDraws H) {
    pdl_enter();
    const size_t half = (size_t(H.D) + 1) / 2;
    const size_t i = size_t(blockIdx.x) * kBlock + threadIdx.x;
    if (i >= size_t(H.R) * half) return;
    const int r = int(i / half), m = int(i - size_t(r) * half);
    const bool anti = H.antithetic && (r & 1);
    const unsigned local = H.antithetic ? unsigned(r >> 1) : unsigned(r), step = hd_step(H);
    const unsigned index = local + unsigned(H.draw_begin);
    float tt[2], wt[2];
    if (H.sampler == kRadial) {
        const float2 z = hd_normal_pair(H, index, step, (H.D + 1) / 2, m);
        const float2 nr = H.norms[local].v;
        const float dir0 = z.x / nr.x, dir1 = z.y / nr.x;
        tt[0] = nr.y * dir0;
        wt[0] = H.c_radial * dir0;
        tt[1] = nr.y * dir1;
        wt[1] = H.c_radial * dir1;
    } else if (H.sampler == kPerDim) {
        const float2 xi2 = perturb_uniform_pair(H, index, step, 2 * m);
        const float c1 = 0.7978845608028654f;  // sqrt(2/pi)
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const float xi = k == 0 ? xi2.x : xi2.y;
            if (xi < 0.5f) {
                tt[k] = -sqrtf(-2.0f * logf(2.0f * xi));
                wt[k] = -c1;
            } else {
                tt[k] = sqrtf(-2.0f * logf(2.0f * (1.0f - xi)));
                wt[k] = c1;
            }
        }
    } else {
        const float2 z = hd_normal_pair(H, index, step, 0, m);
        tt[0] = wt[0] = z.x;
        tt[1] = wt[1] = z.y;
    }
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const int d = 2 * m + k;
        if (d >= H.D) break;
        const float sg = sigma_sched(H.sigma, H.anneal, H.total_steps, H.sigma_min, d, int(step));
        float tau = sg * tt[k], w = wt[k] / sg;
        if (anti) {
            tau = -tau;
            w = -w;
        }
        const size_t o = size_t(r) * size_t(H.D) + size_t(d);
        if (H.theta_out) H.theta_out[o] = H.theta[d] + tau;  // FP32 sum: the parameters this render gets
        if (H.tau_out) H.tau_out[o] = tau;
        if (H.w_out) H.w_out[o] = w;
    }
}

// a6 + a7 over D parameters: g_d = (1/2P) sum_p w_{2p,d} (L_2p - L_2p+1) (a skinny GEMV,
// W^T dL, fixed order over p in FP64), then Adam with t = the already advanced step. Bound by the
// latency of its loads (3 MB of weights at D = 49,152, 16 renders): the losses are read once per
// CTA, the weights eight at a time, and CTAs of 128 threads spread over every SM.
constexpr int kGradBlock = 128;
__global__ void __launch_bounds__(kGradBlock) k_hd_grad(const HdGrad G) {
    __shared__ double s_dl[kMaxRenders];  // pair differences (antithetic) or losses
    pdl_enter();
    const int n = G.antithetic ? G.R / 2 : G.R, stride = G.antithetic ? 2 : 1;
    for (int p = threadIdx.x; p < n; p += kGradBlock)
        s_dl[p] = G.antithetic ? __ldcg(G.losses + 2 * p) - __ldcg(G.losses + 2 * p + 1) : __ldcg(G.losses + p);
    __syncthreads();
    const int d = int(blockIdx.x) * kGradBlock + int(threadIdx.x);
    if (d >= G.D) return;
    const float* w = G.w + d;
    const size_t step = size_t(stride) * G.D;
    double g = 0.0;
    int p = 0;
    for (; p + 8 <= n; p += 8) {  // eight weights in flight, then the same sums
        float v[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) v[q] = w[size_t(p + q) * step];
#pragma unroll
        for (int q = 0; q < 8; ++q) g += double(v[q]) * s_dl[p + q];
    }
    for (; p < n; ++p) g += double(w[size_t(p) * step]) * s_dl[p];
    g /= double(G.antithetic ? 2 * n : n);
    const float gf = float(g);
    if (G.grad_out) G.grad_out[d] = gf;
    if (G.theta) adam_update(G.theta[d], G.m[d], G.v[d], gf, __ldcg(G.step_dev), G.lr, G.b1, G.b2, G.eps);
}

cudaError_t launch_hd_draws(const HdDraws& H, cudaStream_t stream) {
    if (H.D <= 0 || H.R <= 0) return cudaSuccess;
    if (H.sampler == kRadial) {
        if (H.norm_split < 1 || H.norm_split > kNormSplitMax) return cudaErrorInvalidValue;
        const cudaError_t e = launch_pdl(k_hd_norms, (H.antithetic ? H.R / 2 : H.R) * H.norm_split, kBlock, stream, H);
        if (e != cudaSuccess) return e;
    }
    const size_t n = size_t(H.R) * ((size_t(H.D) + 1) / 2);  // one thread per (render, parameter pair)
    return launch_pdl(k_hd_perturb, int((n + kBlock - 1) / kBlock), kBlock, stream, H);
}

cudaError_t launch_hd_grad(const HdGrad& G, cudaStream_t stream) {
    if (G.D <= 0) return cudaSuccess;
    return launch_pdl(k_hd_grad, (G.D + kGradBlock - 1) / kGradBlock, kGradBlock, stream, G);
}

// ---------------------------------------------------------------------------
// FP32 issue-rate probe: the denominator of the render kernels' roofline
// ---------------------------------------------------------------------------
// Every thread runs kFfmaChains independent fused multiply-add chains, so each warp
// always has an FMA ready; a full-occupancy grid then issues FFMA on every FP32 lane
// of every SM each cycle, up to the loop's few integer instructions.
constexpr int kFfmaChains = 8;

__global__ void __launch_bounds__(kBlock) k_ffma_probe(float* out, int iters, float b, float c) {
    float a[kFfmaChains];
#pragma unroll
    for (int i = 0; i < kFfmaChains; ++i) a[i] = float(threadIdx.x) * 1e-7f + float(i);
    for (int k = 0; k < iters; ++k) {
#pragma unroll 16
        for (int i = 0; i < kFfmaChains; ++i) a[i] = fmaf(a[i], b, c);
    }
    float s = 0.f;
#pragma unroll
    for (int i = 0; i < kFfmaChains; ++i) s += a[i];
    out[size_t(blockIdx.x) * blockDim.x + threadIdx.x] = s;
}

int ffma_probe_flops_per_thread_iter() { return 2 * kFfmaChains; }

cudaError_t launch_ffma_probe(float* out, int blocks, int iters, cudaStream_t stream) {
    if (blocks <= 0 || iters <= 0) return cudaErrorInvalidValue;
    k_ffma_probe<<<blocks, kBlock, 0, stream>>>(out, iters, 0.9999999f, 1e-7f);
    return cudaGetLastError();
}

}  // namespace prdpt
