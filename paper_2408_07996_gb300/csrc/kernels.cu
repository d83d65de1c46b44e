// kernels.cu -- wavefront path tracer and statistical event detector.
//
// One chunk of paths goes through
//   camera rays + extend -> [shade(+NEE) -> shadow + extend] x max_depth -> shade -> stats
// Every path keeps one slot of the wavefront for its ray and state; extend,
// shade and shadow walk device-side queues of slots (sizes in device
// counters, no host round trip) that shade fills tile by tile in direction
// order.  `stats` fuses, per queued pixel, the log-luminance batch statistics
// (Sec. 3.1, Eq. 3-4), the Chan merge into the running statistics, the t-test
// of Eq. 7 (Sec. 3.2), a bit for the re-queue of undecided pixels in order
// (Sec. 3.3) and the event rule with the reference update (Alg. 1, Eq. 1).
#include <cuda_runtime.h>
#include <stdint.h>

#include <mutex>

#include "../../include/mcev.h"
#include "device.cuh"
#include "kernels.h"
#include "tdist.h"

namespace mcev {

// Resident blocks of 128 threads per SM of the traversal kernel, which fix its
// registers: 10 blocks (48) for the two-wide layout; traversal waits on node
// fetches, so more warps pay (terrain frame at 9 / 10 / 12 blocks: 778 / 766 /
// 767 ms, the last spilling at 40 registers; eight batched jobs at 8 / 9 / 10
// blocks 140.9 / 136.9 / 135.4 ms).  The TLAS loop carries more state (frames of
// 12 moving spheres at 8 / 9 / 10 blocks 15.9 / 15.7 / 16.6 ms).  The wide-node
// traversal keeps a whole node (five 16-byte words) and its eight child tests in
// flight.
__host__ __device__ constexpr int trav_blocks(bool wide, bool tlas) {
    return wide ? 8 : (tlas ? 9 : 10);
}

static constexpr uint32_t NO_FLAGS = 0xFFFFFFFFu;

// Direction cell of a ray for the queues' order: its octant (which plane of a
// box is near on each axis) and its dominant axis (the shear of the
// watertight test), so rays of one cell take the same side of every
// sign-dependent choice of the traversal.
static constexpr uint32_t KEY_NONE = 0xFFu;
static constexpr int KEY_CELLS = 32;    // 24 used
__device__ __forceinline__ uint32_t dir_cell(f3 d) {
    const float ax = fabsf(d.x), ay = fabsf(d.y), az = fabsf(d.z);
    const uint32_t kz = (ay > ax && ay >= az) ? 1u : ((az > ax && az > ay) ? 2u : 0u);
    const uint32_t oct = (d.x < 0.0f ? 1u : 0u) | (d.z < 0.0f ? 2u : 0u) | (d.y < 0.0f ? 4u : 0u);
    return 3u * oct + kz;
}

// shadow-ray count of the bounce whose ray queue is `cur` (double-buffered so
// a launch can trace one bounce's shadow rays while the next bounce's shade
// appends to the other slot)
__device__ __forceinline__ int sh_slot(int cur) { return cur ? 19 : 2; }
static constexpr uint32_t FNV_BASIS = 2166136261u;

// ------------------------------------------------------------------ camera rays
// Starts path p of a chunk: sample k_base + p % spp_r of queue entry j0 + p / spp_r.
// kBatch: queue entries are (job << 24 | pixel) and every path reads its
// job's frame and settings from the job table; otherwise entries are pixels
// of the single context whose frame and settings are kernel arguments.
template <bool kBatch>
__device__ __forceinline__ void start_path(const DevFrame& fr, const DevParams& P, const Wave& w, const Chunk& ch,
                                           int p, const Job* __restrict__ jobs) {
    const int j = p / ch.spp_r;
    const int32_t s = p - j * ch.spp_r;
    const int32_t entry = __ldg(ch.queue + ch.j0 + j);
    const int job = kBatch ? (int)((uint32_t)entry >> 24) : 0;
    const int32_t pix = kBatch ? (entry & 0xFFFFFF) : entry;
    const DevFrame& F = kBatch ? jobs[job].fr : fr;
    const DevParams& Q = kBatch ? jobs[job].P : P;
    const uint32_t k = (uint32_t)(ch.k_base + s);
    const uint4 x = philox4x32_10(make_uint4((uint32_t)pix, k, 0u, 0u), F.key0, F.key1);
    const int px = pix % Q.width, py = pix / Q.width;
    const float fx = 2.0f * ((float)px + u01(x.x)) / (float)Q.width - 1.0f;
    const float fy = 1.0f - 2.0f * ((float)py + u01(x.y)) / (float)Q.height;
    const f3 d = norm3(mk3(F.fwd[0] + fx * F.right[0] + fy * F.up[0],
                           F.fwd[1] + fx * F.right[1] + fy * F.up[1],
                           F.fwd[2] + fx * F.right[2] + fy * F.up[2]));
    w.ray_o[p] = make_float4(F.eye[0], F.eye[1], F.eye[2], 1.0f);
    w.ray_d[p] = make_float4(d.x, d.y, d.z, 0.0f);
    w.L[p] = 0.0f;
    w.pix_k[p] = make_int2(entry, (int)k);
    if (Q.adjoint && Q.grad_mean) {
        // d loss / d L of this path: d loss / d mean * d mean / d ln(L + eps) * d ln(L + eps) / dL
        const float Lt = w.Ltot[p];
        w.delta[p] = isfinite(Lt) ? __ldg(Q.grad_mean + pix) / ((float)Q.spp * (Lt + Q.eps)) : 0.0f;
    }
    if (Q.want_sig) {
        w.sig[p] = FNV_BASIS;
        w.pflags[p] = NO_FLAGS;
    }
}

// ------------------------------------------------------------------ gradient sums
// Millions of contributions land on a few lights and, within a warp, on a few
// texels; atomics on one word serialise (FP64 ones on four lights' words took
// 140 us of a 200-us traversal launch and 140 us of a 250-us shading launch of
// the 256x256 gradient step).  They are added up first: per warp, and for the
// first EMIT_SLOTS materials per block.
constexpr int EMIT_SLOTS = 32;

// acc[m] (or grad_emit[m]) += v for the lanes with m >= 0; the whole warp calls
__device__ __forceinline__ void warp_add_emit(double* acc, double* grad_emit, int m, double v) {
    const unsigned full = 0xffffffffu;
    unsigned todo = __ballot_sync(full, m >= 0);
    while (todo) {
        const int lead = __ffs(todo) - 1;
        const int mm = __shfl_sync(full, m, lead);
        double x = m == mm ? v : 0.0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(full, x, o);
        if ((int)(threadIdx.x & 31) == lead) atomicAdd((mm < EMIT_SLOTS ? acc : grad_emit) + mm, x);
        todo &= ~__ballot_sync(full, m == mm);
    }
}

// d loss / d texel += g * (luminance weights) for the lanes with texel >= 0; the
// whole warp calls.  Texels that several lanes share are added up first.
__device__ __forceinline__ void warp_add_tex(float* grad_tex, int texel, float g) {
    const unsigned full = 0xffffffffu;
    unsigned todo = __ballot_sync(full, texel >= 0);
    while (todo) {
        const int lead = __ffs(todo) - 1;
        const int tt = __shfl_sync(full, texel, lead);
        const unsigned same = __ballot_sync(full, texel == tt);
        if (__popc(same) < 4) break;       // scattered: the loop would cost more than it saves
        float x = texel == tt ? g : 0.0f;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(full, x, o);
        if (texel == tt) {
            g = x;
            if ((int)(threadIdx.x & 31) != lead) texel = -1;
        }
        if ((int)(threadIdx.x & 31) == lead) {
            float* gt = grad_tex + 3 * (int64_t)tt;
            atomicAdd(gt, x * MCEV_Y_R);
            atomicAdd(gt + 1, x * MCEV_Y_G);
            atomicAdd(gt + 2, x * MCEV_Y_B);
            texel = -1;
        }
        todo &= ~same;
    }
    if (texel >= 0) {
        float* gt = grad_tex + 3 * (int64_t)texel;
        atomicAdd(gt, g * MCEV_Y_R);
        atomicAdd(gt + 1, g * MCEV_Y_G);
        atomicAdd(gt + 2, g * MCEV_Y_B);
    }
}

// what a shaded vertex adds to the gradients (material / texel -1: nothing)
struct VertexGrad {
    int mat, texel;
    float emit, tex;
};

// Per-block accumulation of the traversal work counters: work_begin at the
// top of the kernel, add_work at its end.  Each warp adds its sums in shared
// memory; the last warp of the block to finish adds the block's totals to
// the global counters, so no warp waits for another.  v: nodes, triangles
// and box tests of closest-hit rays, then of shadow rays.
struct WorkAcc {
    unsigned long long v[6];
    double emit[EMIT_SLOTS];      // adjoint: the block's emission gradients
    unsigned int done;
};

__device__ __forceinline__ WorkAcc& work_acc() {
    __shared__ WorkAcc acc;
    return acc;
}

__device__ __forceinline__ void work_begin() {
    WorkAcc& a = work_acc();
    if (threadIdx.x < 6) a.v[threadIdx.x] = 0ull;
    if (threadIdx.x < EMIT_SLOTS) a.emit[threadIdx.x] = 0.0;
    if (threadIdx.x == 0) a.done = 0u;
    __syncthreads();
}

__device__ __forceinline__ void warp_work(WorkAcc& a, int at, int3 work) {
    const unsigned m = 0xffffffffu;
    const int nodes = __reduce_add_sync(m, work.x);
    const int tris = __reduce_add_sync(m, work.y);
    const int boxes = __reduce_add_sync(m, work.z);
    if ((threadIdx.x & 31) == 0 && (nodes | tris)) {
        atomicAdd(&a.v[at], (unsigned long long)nodes);
        atomicAdd(&a.v[at + 1], (unsigned long long)tris);
        atomicAdd(&a.v[at + 2], (unsigned long long)boxes);
    }
}

// the whole warp, converged after its ray loops
__device__ __forceinline__ void add_work(const Wave& w, int3 closest, int3 shadow, double* grad_emit) {
    WorkAcc& a = work_acc();
    warp_work(a, 0, closest);
    warp_work(a, 3, shadow);
    __syncwarp();      // orders the other lanes' additions to a.emit before lane 0's fence
    if ((threadIdx.x & 31) == 0) {
        __threadfence_block();
        if (atomicAdd(&a.done, 1u) == (blockDim.x >> 5) - 1u) {
            __threadfence_block();
            // 64-bit words after the int32 counters (layout.h)
            unsigned long long* c = reinterpret_cast<unsigned long long*>(w.counters + 32);
            const int word[6] = {0, 1, 7, 2, 3, 8};
            for (int i = 0; i < 6; ++i) {
                const unsigned long long v = atomicAdd(&a.v[i], 0ull);
                if (v) atomicAdd(c + word[i], v);
            }
            if (grad_emit)
                for (int m = 0; m < EMIT_SLOTS; ++m) {
                    const double v = atomicAdd(&a.emit[m], 0.0);
                    if (v != 0.0) atomicAdd(grad_emit + m, v);
                }
        }
    }
}

// ------------------------------------------------------------------ shade + NEE + BSDF sampling
// Shades a bounce's hits and queues the rays it leaves.  A block takes tiles of
// up to Q_TILE consecutive entries of the bounce's queue: it shades them, one
// path per thread and step, and then appends the paths that go on and the ones
// with a shadow ray to their queues, grouped by direction cell (a counting
// sort in shared memory) with one atomic per tile and queue.  Consecutive
// entries stay paths of neighbouring pixels (the samples of a pixel are
// consecutive path slots, a tile is 8 pixels at 512 samples), so a traversal
// warp holds rays that start at nearly the same point and leave it in nearly
// the same direction.
//
// What bounds it: the latency of the per-path gathers (64 registers, 1024
// threads per SM; 15 % faster than an unconstrained 80-register build).
// Against appending rays in the order shade's warps finish, which mixes the
// pixels of a whole wave of blocks, the 1280x720 terrain frame with the converged
// traversal loop takes: 687 ms of traversal with one cell per tile (pixel
// order kept, no sort), 609 ms with the 24 cells, 624 and 614 ms with an octahedral
// grid of 4 x 4 and 8 x 8 cells, 640 ms with the octants alone; shading and
// queues 139, 139, 143, 148 and 136 ms (more cells scatter shade's reads).
// Tiles of 2048 and 8192 entries within 1 % of 4096.  Queues filled by a kernel of
// their own cost 9 ms more (139 -> 130 ms, 4 bytes per path and a launch per
// bounce); blocks of 128 / 256 / 512 threads 138 / 130 / 370 ms.
static constexpr int Q_BLOCK = 256, Q_TILE = 4096, Q_ITEMS = Q_TILE / Q_BLOCK;
static constexpr int Q_RESIDENT = 1024 / Q_BLOCK;   // blocks per SM

// kAdjoint: the replay pass of mcev_backward (never batched)
template <bool kBatch, bool kAdjoint>
__device__ __forceinline__ uint32_t shade_path(const DevScene& sc, const DevFrame& fr, const DevParams& P,
                                               const Wave& w, int p, int depth, const Job* __restrict__ jobs,
                                               VertexGrad& vg) {
    const float4 ro = w.ray_o[p];
    const float4 rd = w.ray_d[p];
    const int2 rs = w.pix_k[p];
    const int job = kBatch ? (int)((uint32_t)rs.x >> 24) : 0;
    const DevScene& S = kBatch ? jobs[job].sc : sc;
    const DevFrame& F = kBatch ? jobs[job].fr : fr;
    const DevParams& Q = kBatch ? jobs[job].P : P;
    const float2 hv = w.hit[p];
    const int tri = __float_as_int(hv.y);
    float beta = ro.w;
    // radiance this vertex adds to the path (emission on a hit, the
    // environment on a miss); the path's total is updated only when
    // something is added
    float Ladd = 0.0f;
    const float pdf_prev = rd.w;
    float pdf_next = 0.0f;
    uint32_t sig = 0, pflags = NO_FLAGS;
    if (Q.want_sig) {
        sig = w.sig[p];
        const uint32_t pf = w.pflags[p];
        if (pf != NO_FLAGS) sig = fnv(sig, pf);
    }
    const f3 d = xyz(rd);
    bool cont = false, shadow = false;
    f3 P0 = mk3(0, 0, 0), wi_next = mk3(0, 0, 0), sh_dir = mk3(0, 0, 0);
    float sh_tmax = 0.0f, sh_c = 0.0f, sh_g = 0.0f;
    int sh_m = -1;
    if (tri < 0) {
        // miss: environment radiance (Sec. 3.1 samples the light reaching the pixel)
        if (Q.want_sig) sig = fnv(sig, 0xFFFFFFFFu);
        if (S.has_env) {
            int row, col;
            float st;
            env_texel(S, d, row, col, st);
            if (Q.want_sig) sig = fnv(sig, (uint32_t)(row * S.env_w + col));
            const float Le = __ldg(S.env + (int64_t)row * S.env_w + col);
            float wgt = 1.0f;
            if (depth > 0 && Q.nee) wgt = Q.mis ? power_heuristic(pdf_prev, F.p_env * texel_pdf(S, row, col, st)) : 0.0f;
            Ladd = beta * wgt * Le;
        } else if (Q.want_sig) {
            sig = fnv(sig, 0xFFFFFFFEu);
        }
    } else {
        const int rec = F.n_inst > 1 ? w.hit_rec[p] : 0;
        // the shading record (edge cross product, material) serves most
        // hits; the vertices are read only for textured albedo, emitter
        // MIS weights and the decision signature
        const float4 tsh = __ldg(S.tshade + tri);
        const float4* tp = S.tris + 3 * tri;
        const float4* ip = F.inst + 7 * rec;
        const float4 i0 = __ldg(ip + 3), i1 = __ldg(ip + 4), i2 = __ldg(ip + 5);
        const int ovr = __float_as_int(__ldg(ip + 6).y);
        if (Q.want_sig) {
            sig = fnv(sig, (uint32_t)hit_inst(F, rec, __ldg(tp + 2).w));
            sig = fnv(sig, (uint32_t)__float_as_int(__ldg(tp).w));
        }
        const float t = hv.x;
        P0 = xyz(ro) + d * t;
        const f3 ng = norm3(xf_normal(i0, i1, i2, xyz(tsh)));
        const f3 wo = d * -1.0f;
        const int mat = ovr >= 0 ? ovr : __float_as_int(tsh.w);
        const float4 mv = __ldg(S.mats + mat);
        const int tword = __float_as_int(mv.x);
        const int type = tword & 0xFF;
        float alb = mv.y;
        const float rough = mv.z;
        // the override applies to the scene's emitters only (NEE samples that fixed set)
        const float emit = (S.emit && mv.w > 0.0f) ? __ldg(S.emit + mat) : mv.w;
        int texel = -1;
        if ((tword & MAT_TEXTURED) && S.tex && S.tri_uv) {
            // albedo = luminance of the nearest texel at the hit's texture coordinates
            const float4 q0 = __ldg(tp), q1 = __ldg(tp + 1), q2 = __ldg(tp + 2);
            float b1, b2;
            barycentric(xf_point(i0, i1, i2, P0), xyz(q0), xyz(q1), xyz(q2), b1, b2);
            const float b0 = 1.0f - b1 - b2;
            const float2 t0 = __ldg(S.tri_uv + 3 * tri), t1 = __ldg(S.tri_uv + 3 * tri + 1),
                         t2 = __ldg(S.tri_uv + 3 * tri + 2);
            texel = texel_of(S, b0 * t0.x + b1 * t1.x + b2 * t2.x, b0 * t0.y + b1 * t1.y + b2 * t2.y);
            const float* rgb = S.tex + 3 * (int64_t)texel;
            alb = MCEV_Y_R * __ldg(rgb) + MCEV_Y_G * __ldg(rgb + 1) + MCEV_Y_B * __ldg(rgb + 2);
            if (Q.want_sig) sig = fnv(sig, (uint32_t)texel);
        }
        const float dlt = kAdjoint ? w.delta[p] : 0.0f;
        uint32_t flags = 0;
        const float cos_o = dot3(ng, wo);
        if (emit > 0.0f && cos_o > 0.0f) {
            flags |= 1u;
            float wgt = 1.0f;
            if (depth > 0 && Q.nee) {
                if (!Q.mis) {
                    wgt = 0.0f;
                } else {
                    const float4 q0 = __ldg(tp), q1 = __ldg(tp + 1), q2 = __ldg(tp + 2);
                    const float4 m0 = __ldg(ip), m1 = __ldg(ip + 1), m2 = __ldg(ip + 2);
                    const f3 e1 = xyz(q1) - xyz(q0), e2 = xyz(q2) - xyz(q0);
                    const f3 we1 = xf_vec(m0, m1, m2, e1), we2 = xf_vec(m0, m1, m2, e2);
                    const f3 wc = cross3(we1, we2);
                    const float area = 0.5f * sqrtf(dot3(wc, wc));
                    const float pl = F.p_area / ((float)F.n_lights * area) * t * t / cos_o;
                    wgt = power_heuristic(pdf_prev, pl);
                }
            }
            Ladd = beta * wgt * emit;
            if (kAdjoint && Q.grad_emit) {
                vg.mat = mat;
                vg.emit = dlt * beta * wgt;
            }
        }
        if (depth < Q.max_depth && alb > 0.0f) {
            // adjoint: every contribution after this vertex carries one factor of its albedo
            if (kAdjoint && texel >= 0 && Q.grad_tex && dlt != 0.0f) {
                vg.texel = texel;
                vg.tex = dlt * (w.Ltot[p] - (w.L[p] + Ladd)) / alb;
            }
            const f3 nn = cos_o < 0.0f ? ng * -1.0f : ng;
            f3 tb, bt;
            onb(nn, tb, bt);
            const f3 wol = mk3(dot3(wo, tb), dot3(wo, bt), dot3(wo, nn));
            const uint32_t ent = (uint32_t)rs.x;
            const uint2 pk = make_uint2(kBatch ? (ent & 0xFFFFFFu) : ent, (uint32_t)rs.y);
            // next-event estimation
            if (Q.nee && (S.env_ok || F.n_lights > 0)) {
                const uint4 x = philox4x32_10(make_uint4(pk.x, pk.y, (uint32_t)(depth + 1), 0u), F.key0, F.key1);
                const bool use_env = S.env_ok && (F.n_lights == 0 || u01(x.x) < 0.5f);
                f3 wi = mk3(0, 0, 0);
                float pl = 0.0f, Le = 0.0f, tmax = __int_as_float(0x7f800000);
                int lmat = -1;
                if (use_env) {
                    float pdf;
                    wi = env_sample(S, u01(x.z), u01(x.w), pdf, Le);
                    pl = F.p_env * pdf;
                } else {
                    const uint64_t mm = (uint64_t)(x.y >> 8);
                    const int li = (int)((mm * (uint64_t)F.n_lights) >> 24);
                    const float4* lp = F.lights + 4 * li;
                    const float4 a0 = __ldg(lp), a1 = __ldg(lp + 1), a2 = __ldg(lp + 2), an = __ldg(lp + 3);
                    const float su = sqrtf(u01(x.z));
                    const float b0 = 1.0f - su, b1 = u01(x.w) * su, b2 = 1.0f - b0 - b1;
                    const f3 Ql = xyz(a0) * b0 + xyz(a1) * b1 + xyz(a2) * b2;
                    const f3 dv = Ql - P0;
                    const float dist = sqrtf(dot3(dv, dv));
                    wi = dv * (1.0f / dist);
                    const float cl = -dot3(xyz(an), wi);
                    if (cl > 0.0f) {
                        pl = F.p_area / ((float)F.n_lights * a1.w) * dist * dist / cl;
                        lmat = __float_as_int(a2.w);
                        Le = S.emit ? __ldg(S.emit + lmat) : a0.w;
                    }
                    tmax = dist - Q.t_min;
                }
                if (pl > 0.0f && Le > 0.0f) {
                    const f3 wil = mk3(dot3(wi, tb), dot3(wi, bt), dot3(wi, nn));
                    float pb;
                    const float f = bsdf_eval(type, alb, rough, wol, wil, &pb);
                    if (f > 0.0f && wil.z > 0.0f) {
                        flags |= 2u;
                        const float wgt = Q.mis ? power_heuristic(pl, pb) : 1.0f;
                        sh_c = beta * f * wil.z * Le * wgt / pl;
                        sh_g = beta * f * wil.z * wgt / pl;
                        sh_m = lmat;
                        sh_dir = wi;
                        sh_tmax = tmax;
                        shadow = true;
                    }
                }
            }
            // BSDF sampling of the continuation
            const uint4 y = philox4x32_10(make_uint4(pk.x, pk.y, (uint32_t)(depth + 1), 1u), F.key0, F.key1);
            const f3 wil = bsdf_sample(type, rough, wol, u01(y.x), u01(y.y));
            float pb;
            const float f = bsdf_eval(type, alb, rough, wol, wil, &pb);
            if (f > 0.0f && pb > 0.0f && wil.z > 0.0f) {
                flags |= 8u;
                beta *= f * wil.z / pb;
                pdf_next = pb;
                wi_next = norm3(tb * wil.x + bt * wil.y + nn * wil.z);
                cont = true;
            }
        }
        pflags = flags;
    }
    if (Ladd != 0.0f) w.L[p] += Ladd;
    if (Q.want_sig) {
        w.sig[p] = sig;
        w.pflags[p] = pflags;
    }
    if (shadow || cont) w.ray_o[p] = make_float4(P0.x, P0.y, P0.z, beta);
    if (shadow) {
        w.sh_d[p] = make_float4(sh_dir.x, sh_dir.y, sh_dir.z, sh_tmax);
        w.sh_c[p] = sh_c;
        if (kAdjoint) {
            w.sh_g[p] = sh_g;
            w.sh_m[p] = sh_m;
        }
    }
    if (cont) w.ray_d[p] = make_float4(wi_next.x, wi_next.y, wi_next.z, pdf_next);
    return (cont ? dir_cell(wi_next) : KEY_NONE) | (shadow ? dir_cell(sh_dir) : KEY_NONE) << 8;
}

template <bool kBatch, bool kAdjoint>
__global__ void __launch_bounds__(Q_BLOCK, Q_RESIDENT)
    k_shade(DevScene sc, DevFrame fr, DevParams P, Wave w, int cur, int depth, int last, int resident,
            const Job* __restrict__ jobs) {
    __shared__ uint16_t keys[Q_TILE];
    __shared__ uint16_t order[Q_TILE];  // the tile's entries, misses first
    __shared__ int n_miss, n_hit;
    __shared__ double emit[EMIT_SLOTS];
    __shared__ int cnt[2][KEY_CELLS];   // next rays, shadow rays
    const int32_t n = *(volatile int32_t*)(w.counters + cur);
    const int32_t* list = depth > 0 ? w.list[cur] : nullptr;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    if (blockIdx.x == 0 && tid == 0) w.counters[20] = 0;   // the next traversal's cursor
    // a small queue is cut into smaller tiles, so that every resident block has one
    if (kAdjoint && tid < EMIT_SLOTS) emit[tid] = 0.0;     // (synchronised by the first tile)
    const int step = resident * Q_BLOCK;
    const int items = max(1, min(Q_ITEMS, (n + step - 1) / step));
    for (int64_t t0 = (int64_t)blockIdx.x * items * Q_BLOCK; t0 < n; t0 += (int64_t)gridDim.x * items * Q_BLOCK) {
        if (tid < 2 * KEY_CELLS) (&cnt[0][0])[tid] = 0;
        if (tid == 0) n_miss = n_hit = 0;
        __syncthreads();
        const int size = (int)min((int64_t)items * Q_BLOCK, n - t0);
        // After the camera rays (whose pixels mostly see one thing), rays that hit and
        // rays that leave the scene are shaded apart: mixed, 15 of 32 lanes were active.
        const bool split = list != nullptr;
        if (split) {
            for (int k = 0; k < items; ++k) {
                const int e = k * Q_BLOCK + tid;
                const bool in = e < size;
                const bool miss = in && __float_as_int(w.hit[__ldg(list + t0 + e)].y) < 0;
                const unsigned bm = __ballot_sync(0xffffffffu, miss), bh = __ballot_sync(0xffffffffu, in && !miss);
                int am = 0, ah = 0;
                if (lane == 0) {
                    if (bm) am = atomicAdd(&n_miss, __popc(bm));
                    if (bh) ah = atomicAdd(&n_hit, __popc(bh));
                }
                am = __shfl_sync(0xffffffffu, am, 0) + __popc(bm & ((1u << lane) - 1u));
                ah = size - 1 - __shfl_sync(0xffffffffu, ah, 0) - __popc(bh & ((1u << lane) - 1u));
                if (in) order[miss ? am : ah] = (uint16_t)e;
            }
            __syncthreads();
        }
        for (int k = 0; k < items; ++k) {
            int e = k * Q_BLOCK + tid;
            uint32_t key = KEY_NONE | (KEY_NONE << 8);
            VertexGrad vg{-1, -1, 0.0f, 0.0f};
            if (e < size) {
                if (split) e = order[e];
                const int p = list ? __ldg(list + t0 + e) : (int)(t0 + e);
                key = shade_path<kBatch, kAdjoint>(sc, fr, P, w, p, depth, jobs, vg);
            }
            if (kAdjoint) {
                __syncwarp();
                if (P.grad_emit) warp_add_emit(emit, P.grad_emit, vg.mat, (double)vg.emit);
                if (P.grad_tex) warp_add_tex(P.grad_tex, vg.texel, vg.tex);
            }
            keys[e] = (uint16_t)key;
            if ((key & 0xFFu) != KEY_NONE) atomicAdd(&cnt[0][key & 0xFFu], 1);
            if ((key >> 8) != KEY_NONE) atomicAdd(&cnt[1][key >> 8], 1);
        }
        if (last) continue;   // no ray goes on from the last bounce
        __syncthreads();
        // first queue position of each cell, one warp per queue
        if (wid < 2) {
            const int c = cnt[wid][lane];
            int v = c;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, v, o);
                if (lane >= o) v += y;
            }
            int base = 0;
            if (lane == 31 && v) base = atomicAdd(w.counters + (wid ? sh_slot(cur) : 1 - cur), v);
            cnt[wid][lane] = __shfl_sync(0xffffffffu, base, 31) + v - c;
        }
        __syncthreads();
        for (int k = 0; k < items; ++k) {
            const uint32_t kn = keys[k * Q_BLOCK + tid] & 0xFFu, ks = keys[k * Q_BLOCK + tid] >> 8;
            if (kn == KEY_NONE && ks == KEY_NONE) continue;
            const int64_t i = t0 + k * Q_BLOCK + tid;
            const int p = list ? __ldg(list + i) : (int)i;
            if (kn != KEY_NONE) w.list[1 - cur][atomicAdd(&cnt[0][kn], 1)] = p;
            if (ks != KEY_NONE) w.sh_list[atomicAdd(&cnt[1][ks], 1)] = p;
        }
        __syncthreads();
    }
    if (kAdjoint && P.grad_emit && (int64_t)blockIdx.x * items * Q_BLOCK < n) {
        __syncthreads();
        if (tid < EMIT_SLOTS && emit[tid] != 0.0) atomicAdd(P.grad_emit + tid, emit[tid]);
    }
}

// ------------------------------------------------------------------ traversal
// The groups of 32 consecutive queue entries that a warp of the traversal
// kernel takes: first its own number, then the next of a device cursor, fetched
// while the current group is traced.  Per-ray cost is heavy-tailed: a fixed
// share of the queues per block left SMs idle at the end of a launch (terrain
// frame traversal 650 ms -> 624 ms, sphere field 183 -> 178 ms; groups of 128
// rays 635 and 181 ms).
struct Groups {
    int g, n_warps, total;   // current group, warps of the grid, groups of both queues
    int32_t* cursor;
    int ahead;               // lane 0: the group after g
    __device__ __forceinline__ void prefetch() {
        ahead = total;
        if (n_warps < total && (threadIdx.x & 31) == 0) ahead = n_warps + atomicAdd(cursor, 1);
    }
    __device__ __forceinline__ void advance() { g = __shfl_sync(0xffffffffu, ahead, 0); }
};

// Traces the warp's groups below `g_end` of a queue whose first group is
// `g0`, one ray per lane: closest hits (kAny = false) of `list` (null: slots
// 0 .. n-1) into w.hit, or occlusion of the shadow rays.  (Refilling a warp's
// idle lanes with further rays while others are still traced was slower on
// the sphere field, 178 -> 200 ms and more at every threshold: the lanes' state
// machine costs more than it fills.)
template <bool kAny, bool kBatch, bool kWide, bool kTlas>
__device__ __forceinline__ int3 trace_queue(const DevScene& sc, const DevFrame& fr, const DevParams& P, const Wave& w,
                                            const int32_t* __restrict__ list, const Chunk* ch, int32_t n, Groups& gr,
                                            int g0, int g_end, int* stack, int32_t* err,
                                            const Job* __restrict__ jobs) {
    const int lane = threadIdx.x & 31;
    const float4* dirs = kAny ? w.sh_d : w.ray_d;
    int2 work = make_int2(0, 0);
    int3 wwork = make_int3(0, 0, 0);
    while (gr.g < g_end) {
        gr.prefetch();
        const int g = (gr.g - g0) * 32;
        const bool live = g + lane < n;
        const int i = live ? g + lane : n - 1;
        const int p = list ? __ldg(list + i) : i;
        if (!kAny && ch) {
            if (live) start_path<kBatch>(fr, P, w, *ch, p, jobs);
            __syncwarp();
        }
        const int job = kBatch ? (int)((uint32_t)w.pix_k[p].x >> 24) : 0;
        const DevScene& S = kBatch ? jobs[job].sc : sc;
        const DevFrame& F = kBatch ? jobs[job].fr : fr;
        const DevParams& Q = kBatch ? jobs[job].P : P;
        const float4* op = w.ray_o + p;
        const float4* dp = dirs + p;
        const float tmin = Q.t_min;
        THit h{kAny ? dp->w : __int_as_float(0x7f800000), -1, 0};
        if (kWide) {
            Hit wh;
            int e = 0;
            const bool occ = trace_wide<kAny>(S, F, op, dp, live, tmin, h.t, wh, stack, &e, wwork);
            if (e) atomicOr(err, 1);
            h = THit{wh.t, kAny ? (occ ? 0 : -1) : wh.tri, wh.rec};
        } else {
            // the merged never-moving geometry, then the one moving instance
            // (variants without the TLAS are launched for frames with at most one)
#pragma unroll 1
            for (int step = 0; step < (kTlas ? 1 : 2); ++step) {
                const int rec = step == 0 ? F.static_rec : (F.n_tlas > 0 ? 0 : -1);
                if (!kBatch && rec < 0) continue;   // the same for the whole warp
                const bool on = live && rec >= 0 && !(kAny && h.tri >= 0);
                int root = 0;
                TRay r;
                if (on) r = object_tray(F, rec, op, dp, root);
                two_wide<kAny>(S, F, root, rec, r, on, tmin, h, stack, err, work);
            }
            if (kTlas && (kBatch || F.n_tlas > 0))
                two_level<kAny>(S, F, op, dp, live && F.n_tlas > 0 && !(kAny && h.tri >= 0), tmin, h, stack, err, work);
        }
        if (!kAny) {
            if (live) {
                __stcs(w.hit + p, make_float2(h.t, __int_as_float(h.tri)));
                if (F.n_inst > 1) w.hit_rec[p] = h.rec;
            }
        } else {
            // the light sample reaches the path's vertex: add its contribution
            const bool lit = live && h.tri < 0;
            if (lit) {
                w.L[p] += w.sh_c[p];
                if (Q.want_sig) w.pflags[p] |= 4u;
            }
            if (!kBatch && P.adjoint && P.grad_emit) {
                const int m = lit ? w.sh_m[p] : -1;
                warp_add_emit(work_acc().emit, P.grad_emit, m, m >= 0 ? (double)(w.delta[p] * w.sh_g[p]) : 0.0);
            }
        }
        gr.advance();
    }
    return kWide ? wwork : make_int3(work.x, work.y, 2 * work.x);
}

// One launch traces the closest hits of bounce `depth` (ray queue `ecur`) and,
// with scur >= 0, then the shadow rays of the bounce before (appended with queue
// scur).
// At depth 0 the rays are the chunk's camera rays (rc: the device-resident round
// loop's current chunk), started here: a kernel of their own wrote and this one
// read 32 bytes more per path (7.8 ms of a terrain 720p frame).
// The grid is the resident warps only; queue sizes are read on the device.
// The first thread also clears the counters the next queues append to.
template <bool kBatch, bool kWide, bool kTlas>
__global__ void __launch_bounds__(MCEV_TRAV_BLOCK, trav_blocks(kWide, kTlas))
    k_trace(DevScene sc, DevFrame fr, DevParams P, Wave w, int ecur, int scur, int depth, Chunk ch, int32_t* err,
            const Job* __restrict__ jobs, const RoundCtl* __restrict__ rc) {
    int stack[MCEV_STACK];
    work_begin();
    if (rc) ch = Chunk{rc->queue[rc->qi], rc->j0, rc->n_done, (int32_t)(rc->nj * rc->spp_r), rc->spp_r};
    const int32_t n = depth == 0 ? ch.n_paths : *(volatile int32_t*)(w.counters + ecur);
    const int32_t ns = scur >= 0 ? *(volatile int32_t*)(w.counters + sh_slot(scur)) : 0;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        if (depth == 0) w.counters[ecur] = n;
        w.counters[1 - ecur] = 0;
        w.counters[sh_slot(ecur)] = 0;
        unsigned long long* c = reinterpret_cast<unsigned long long*>(w.counters + 32);
        atomicAdd(c + 4, (unsigned long long)n);
        if (ns) atomicAdd(c + 5, (unsigned long long)ns);
    }
    const int ge = (n + 31) >> 5;
    Groups gr{(int)(blockIdx.x * (MCEV_TRAV_BLOCK / 32) + (threadIdx.x >> 5)), (int)gridDim.x * (MCEV_TRAV_BLOCK / 32),
              ge + ((ns + 31) >> 5), w.counters + 20, 0};
    const int3 wc = trace_queue<false, kBatch, kWide, kTlas>(sc, fr, P, w, depth > 0 ? w.list[ecur] : nullptr,
                                                             depth > 0 ? nullptr : &ch, n, gr, 0, ge, stack, err, jobs);
    int3 ws = make_int3(0, 0, 0);
    if (scur >= 0)
        ws = trace_queue<true, kBatch, kWide, kTlas>(sc, fr, P, w, w.sh_list, nullptr, ns, gr, ge, gr.total, stack, err,
                                                       jobs);
    add_work(w, wc, ws, !kBatch && P.adjoint ? P.grad_emit : nullptr);
}

// ------------------------------------------------------------------ per-pixel statistics + test + requeue + events
struct Moments {
    float n, mean, m2;
};
__device__ __forceinline__ Moments chan(Moments a, Moments b) {
    const float n = a.n + b.n;
    if (n == 0.0f) return a;
    const float dl = b.mean - a.mean;
    Moments r;
    r.n = n;
    r.mean = a.mean + dl * (b.n / n);
    r.m2 = a.m2 + b.m2 + dl * dl * (a.n * b.n / n);
    return r;
}

// kChecked: caller-supplied pixel ids and counts are range-checked (the
// allocation-free entry point); the renderer's own queues use <false>.
// log of a path value: the fast hardware logarithm by default (its error,
// ~1e-7 absolute near 1, is far below the statistics' own noise)
#ifndef MCEV_FAST_LOG
#define MCEV_FAST_LOG 1
#endif
#if MCEV_FAST_LOG
#define MCEV_LOG(x) __logf(x)
#else
#define MCEV_LOG(x) logf(x)
#endif

// Lanes per pixel of the statistics kernel: a warp, or four lanes (eight pixels per
// warp).  A round traced spp_r samples of a pixel: one batch, or a window of
// several batches of `sub`.  Each batch is merged and tested in order exactly as
// Alg. 1 would; once the pixel is decided, the rest of the window is left unused.
//
// What bounds it: with short batches the instructions of the merge and the test (six
// divisions and a square root), which every lane of a pixel repeats: 90k pixels x
// 15 batches of 16 431 us with a warp per pixel, 137 us with four lanes; eight jobs
// 131 -> 124 ms, terrain 720p 751 -> 742 ms.  With long batches and few pixels the
// latency of a pixel's own chain of loads and additions, which a warp shortens eightfold.
// Whole detector steps, four lanes / a warp: 5000 pixels x 17 samples 19 / 27 us, 80000 x
// 16 27 / 53, 20000 x 64 27 / 27, 20000 x 512 39 / 39, 9728 x 512 39 / 27, 1 x 64 27 / 19, 40000 x
// 2048 138 / 103, 9728 x 2048 100 / 39, 1 x 8192 286 / 39 (a mean of 2^20 samples of one pixel
// 38 / 3.9 ms).  So long batches (64 and more) have a warp per pixel up to 32 pixels per
// sample.  Batches of 32 and more have one also where a warp for every pixel is resident at
// once (152 SMs x 40), and the shortest below 1024 pixels: mean-only steps on 3072 pixels
// with batches of 32 and 64 104 / 91 us, of 16 97 / 103; on 64 pixels of 16 96 / 92.
//
// The order of the additions is fixed: sample s of a batch belongs to leaf s % 32,
// leaves add up pairwise 16, 8, 4, 2 and 1 apart (a warp's butterfly).  A lane holds
// every LANES-th leaf, so the last steps are shuffles (a + b on one lane, b + a on its
// partner: the same bits), and every lane of a pixel ends with identical
// statistics and takes the same decisions.
__host__ __device__ __forceinline__ bool stats_by_warp(int64_t n_pix, int64_t sub) {
    const int64_t resident = 152 * 40;
    const int64_t most = sub >= 64 && 32 * sub > resident ? 32 * sub : (sub >= 32 ? resident : 1024);
    return n_pix <= most;
}

constexpr int STATS_STEPS = 8;
template <bool kChecked, bool kBatch, int LANES>
__device__ __forceinline__ void stats_tiles(const Wave& w, const StatsArgs& A0, const int32_t* __restrict__ queue,
                                            int64_t j0, int64_t n_pix, int32_t* __restrict__ next_queue,
                                            const Job* __restrict__ jobs, uint32_t* again_bits, int& again_at) {
    constexpr unsigned full = 0xffffffffu;
    constexpr int PIX = 32 / LANES, LEAVES = 32 / LANES;
    constexpr bool kOwnList = kChecked && LANES == 32;     // few pixels: listed one by one, in any order
    constexpr int AHEAD = 8;       // samples that a lane of a warp's pixel loads at a time
    const int lane = threadIdx.x & 31, q = lane & (LANES - 1);
    const int test0 = A0.mode == MODE_DETECT ? (int)((A0.k_base - A0.spp_min) / A0.spp_batch) : 0;
    // a block's tile: up to 8 steps of 64 (8) pixels, fewer when there are few pixels
    constexpr int STEP = 256 / LANES, STEPS = STATS_STEPS;
    const int64_t per_step = (int64_t)gridDim.x * STEP;
    const int steps = (int)max((int64_t)1, min((int64_t)STEPS, n_pix / per_step));
    for (int64_t t0 = (int64_t)blockIdx.x * steps * STEP; t0 < n_pix; t0 += per_step * steps) {
        if (!kOwnList) {
            if (threadIdx.x < STEP * STEPS / 32) again_bits[threadIdx.x] = 0;
            __syncthreads();
        }
        for (int it = 0; it < steps; ++it) {
            const int in_tile = it * STEP + (threadIdx.x >> 5) * PIX + lane / LANES;
            const int64_t j = t0 + in_tile;
            bool on = j < n_pix;
            const int32_t entry = on ? __ldg(queue + j0 + j) : 0;
            const int32_t pix = kBatch ? (entry & 0xFFFFFF) : entry;
            // per-pixel state and outputs of the pixel's job
            StatsArgs A = A0;
            if (kBatch && on) {
                const Job& J = jobs[(uint32_t)entry >> 24];
                A.cur = J.cur;
                A.ref = J.ref;
                A.events = J.events;
                A.spp_out = J.spp_out;
                A.mean_out = J.mean_out;
                A.eps = J.P.eps;
            }
            if (kChecked && on && (pix < 0 || (int64_t)pix >= A.n_total)) {
                if (q == 0) atomicOr(w.counters + 8, 1);
                on = false;
            }
            Moments c{0.0f, 0.0f, 0.0f};
            if (on && A.k_base > 0) c = Moments{(float)A.cur.n[pix], A.cur.mean[pix], A.cur.m2[pix]};
            const bool detect = A.mode == MODE_DETECT;
            const float ma = detect && on ? A.ref.mean[pix] : 0.0f;
            const int32_t na = detect && on ? A.ref.n[pix] : 0;
            const float va = (detect && na > 1) ? A.ref.m2[pix] / (float)(na - 1) : 0.0f;
            int bad = 0;
            bool open = on;        // neither decided nor off
            int32_t n = (int32_t)c.n;
            // number of the last test: spp_min + test * spp_batch samples
            int test = A.k_base == 0 ? -1 : test0;
            const float* Lp = w.L + (on ? j : 0) * A.spp_r;
            for (int s0 = 0; s0 < A.spp_r && __any_sync(full, open); s0 += A.sub) {
                const int s1 = min(s0 + A.sub, A.spp_r);
                // moments of this batch from sums shifted by one value (the running
                // mean, or the batch's first sample for a pixel's first batch), so
                // lanes merge by plain addition
                float sh = c.mean;
                if (open && !(c.n > 0.0f)) {
                    const float L0 = Lp[s0];
                    sh = MCEV_LOG((isfinite(L0) ? L0 : 0.0f) + A.eps);
                }
                float a1[LEAVES], a2[LEAVES];
#pragma unroll
                for (int m = 0; m < LEAVES; ++m) a1[m] = a2[m] = 0.0f;
                if (open) {
                    auto add = [&](int m, float x) {
                        if (!isfinite(x)) {
                            x = 0.0f;
                            ++bad;
                        }
                        const float d = MCEV_LOG(x + A.eps) - sh;
                        a1[m] += d;
                        a2[m] = fmaf(d, d, a2[m]);
                    };
                    if constexpr (LANES == 32) {
                        for (int b = s0 + q; b < s1; b += 32 * AHEAD) {
                            float x[AHEAD];
#pragma unroll
                            for (int u = 0; u < AHEAD; ++u) x[u] = b + 32 * u < s1 ? Lp[b + 32 * u] : 0.0f;
#pragma unroll
                            for (int u = 0; u < AHEAD; ++u)
                                if (b + 32 * u < s1) add(0, x[u]);
                        }
                    } else {
                        for (int b = s0; b < s1; b += 32) {
#pragma unroll
                            for (int m = 0; m < LEAVES; ++m) {
                                if (b + LANES * m >= s1) break;     // the same for the whole warp
                                const int s = b + LANES * m + q;
                                if (s < s1) add(m, Lp[s]);
                            }
                        }
                    }
                }
#pragma unroll
                for (int h = LEAVES / 2; h > 0; h >>= 1) {
#pragma unroll
                    for (int m = 0; m < h; ++m) {
                        a1[m] += a1[m + h];
                        a2[m] += a2[m + h];
                    }
                }
                float s1d = a1[0], s2d = a2[0];
#pragma unroll
                for (int off = LANES / 2; off > 0; off >>= 1) {
                    s1d += __shfl_xor_sync(full, s1d, off);
                    s2d += __shfl_xor_sync(full, s2d, off);
                }
                if (!open) continue;
                const float fn = (float)(s1 - s0);
                const float md = s1d / fn;
                const Moments m{fn, sh + md, fmaxf(s2d - s1d * md, 0.0f)};
                c = (A.k_base == 0 && s0 == 0) ? m : chan(c, m);
                n = (int32_t)c.n;
                if (!detect) continue;
                ++test;
                bool decided = n >= A.spp_max;
                if (!decided && A.variant != VAR_UNIFORM) {
                    const float gap = fabsf(c.mean - ma);
                    if (A.variant == VAR_MEAN_ONLY) {
                        decided = gap < A.C;
                    } else {
                        const float vb = c.m2 / (float)(n - 1);
                        const float se2 = A.se_mode == SE_WELCH ? va / (float)na + vb / (float)n : (va + vb) / (float)n;
                        if (se2 == 0.0f) {
                            decided = gap < A.C;
                        } else if (kChecked && n < A.spp_min) {
                            decided = false;
                        } else {
                            const float t = (gap - A.C) / sqrtf(se2);
                            int r = test;
                            if (kChecked)      // by the caller's own counts
                                r = min((n - A.spp_min) / A.spp_batch,
                                        (A.spp_max - A.spp_min + A.spp_batch - 1) / A.spp_batch - 1);
                            const float tc = __ldg(A.tcrit + r);
                            decided = A.variant == VAR_TWO_TAILED ? (t < tc || t > -tc) : (t < tc);
                        }
                    }
                }
                open = !decided;
            }
#pragma unroll
            for (int off = LANES / 2; off > 0; off >>= 1) bad += __shfl_xor_sync(full, bad, off);
            // the pixel's first lane writes it back
            const bool own = on && q == 0;
            const bool again = own && (detect ? open : n < A.spp_max);
            if (kOwnList && again) next_queue[atomicAdd(w.counters + 3, 1)] = entry;
            if (!kOwnList && again) atomicOr(&again_bits[in_tile >> 5], 1u << (in_tile & 31));
            // Nothing is queued in the round that reaches spp_max; a pixel it leaves open (its
            // FP32 count cannot reach every spp_max above 2^24) is counted, which ends the call
            // with an error.
            if (!kChecked && again && A.k_base + A.spp_r >= A.spp_max) atomicAdd(w.counters + 3, 1);
            if (!own) continue;
            if (bad) atomicAdd(w.counters + 4, bad);
            A.cur.n[pix] = n;
            A.cur.mean[pix] = c.mean;
            A.cur.m2[pix] = c.m2;
            if (again) continue;
            if (!detect) {
                if (A.mode == MODE_MEAN) {
                    A.mean_out[pix] = c.mean;
                    if (A.spp_out) A.spp_out[pix] = n;
                } else {
                    A.ref.n[pix] = n;
                    A.ref.mean[pix] = c.mean;
                    A.ref.m2[pix] = c.m2;
                }
                continue;
            }
            const float delta = c.mean - ma;
            int8_t ev = 0;
            if (fabsf(delta) > A.C) {
                ev = delta > 0.0f ? 1 : -1;
                A.ref.n[pix] = n;
                A.ref.mean[pix] = c.mean;
                A.ref.m2[pix] = c.m2;
                atomicAdd(w.counters + (ev > 0 ? 5 : 6), 1);
            }
            if (n >= A.spp_max) atomicAdd(w.counters + 7, 1);
            atomicAdd(reinterpret_cast<unsigned long long*>(w.counters + 32) + 6, (unsigned long long)n);
            A.events[pix] = ev;
            if (A.spp_out) A.spp_out[pix] = n;
            if (A.mean_out) A.mean_out[pix] = c.mean;
        }
        if (kOwnList) continue;
        __syncthreads();
        if (!kChecked) {
            // requeue() queues them
            const int64_t at = (t0 >> 3) + threadIdx.x;
            if (threadIdx.x < steps * STEP / 8 && at < (n_pix + 7) >> 3)
                reinterpret_cast<uint8_t*>(w.again)[at] = reinterpret_cast<const uint8_t*>(again_bits)[threadIdx.x];
            __syncthreads();
            continue;
        }
        // the allocation-free step lists its tile's undecided pixels itself (any order of tiles)
        if (threadIdx.x < 32) {
            const uint32_t bits = lane < STEP * STEPS / 32 ? again_bits[lane] : 0u;
            const int total = __reduce_add_sync(full, __popc(bits));
            if (lane == 0 && total) again_at = atomicAdd(w.counters + 3, total);
        }
        __syncthreads();
        for (int i = threadIdx.x; i < steps * STEP; i += blockDim.x) {
            const uint32_t bits = again_bits[i >> 5];
            if (!(bits >> (i & 31) & 1u)) continue;
            int at = again_at + __popc(bits & ((1u << (i & 31)) - 1u));
            for (int k = 0; k < i >> 5; ++k) at += __popc(again_bits[k]);
            next_queue[at] = __ldg(queue + j0 + t0 + i);
        }
        __syncthreads();
    }
}

template <bool kChecked, bool kBatch>
__global__ void __launch_bounds__(256) k_stats(Wave w, StatsArgs A, const int32_t* __restrict__ queue, int64_t j0,
                                               int64_t n_pix, int32_t* __restrict__ next_queue,
                                               const Job* __restrict__ jobs, const RoundCtl* __restrict__ rc) {
    __shared__ uint32_t again_bits[64 * STATS_STEPS / 32];
    __shared__ int again_at;
    if (rc) {
        // sizes of the current chunk of the device-resident round loop
        queue = rc->queue[rc->qi];
        next_queue = rc->queue[rc->qi ^ 1];
        j0 = rc->j0;
        n_pix = rc->nj;
        A.spp_r = rc->spp_r;
        A.sub = rc->sub;
        A.k_base = rc->n_done;
    }
    if (stats_by_warp(n_pix, A.sub))
        stats_tiles<kChecked, kBatch, 32>(w, A, queue, j0, n_pix, next_queue, jobs, again_bits, again_at);
    else
        stats_tiles<kChecked, kBatch, 4>(w, A, queue, j0, n_pix, next_queue, jobs, again_bits, again_at);
}

// Appends a chunk's undecided pixels (w.again, one bit per entry) to the next
// round's queue in their order, by one block.  Neighbours in the image stay
// neighbours in the queue from round to round, so that their paths keep meeting
// in the same traversal warps.  Appended warp by warp (eight pixels at a time) as
// warps finished, a terrain 720p frame took 727 ms, a sphere-field frame 190 ms and
// eight jobs 121.7 ms; by tiles of 64 to 512 pixels 713, 187.0 and 110.9 ms; with
// the first queue in image tiles (tiled_pixel) 709, 186.7 and 109.4 ms; in full order
// 695, 183.2 and 108.7 ms.
constexpr int REQUEUE_BLOCK = 1024;
__device__ __forceinline__ void requeue(const Wave& w, const int32_t* __restrict__ queue, int64_t j0, int64_t n_pix,
                                        int32_t* __restrict__ next_queue) {
    __shared__ int sums[REQUEUE_BLOCK / 32];
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int64_t words = (n_pix + 31) >> 5;
    int at = *(volatile int32_t*)(w.counters + 3);
    for (int64_t t0 = 0; t0 < words; t0 += REQUEUE_BLOCK) {
        const int64_t k = t0 + threadIdx.x;
        uint32_t bits = k < words ? w.again[k] : 0u;
        if (32 * k + 32 > n_pix && k < words) bits &= (1u << (n_pix & 31)) - 1u;    // (written up to a whole byte)
        const int c = __popc(bits);
        int v = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(full, v, o);
            if (lane >= o) v += y;
        }
        if (lane == 31) sums[wid] = v;
        __syncthreads();
        const int s = sums[lane];
        const int before = __reduce_add_sync(full, lane < wid ? s : 0), total = __reduce_add_sync(full, s);
        int to = at + before + v - c;
        for (; bits; bits &= bits - 1) next_queue[to++] = __ldg(queue + j0 + 32 * k + __ffs(bits) - 1);
        at += total;
        __syncthreads();
    }
    if (threadIdx.x == 0) *(volatile int32_t*)(w.counters + 3) = at;
}

__global__ void __launch_bounds__(REQUEUE_BLOCK) k_requeue(Wave w, const int32_t* queue, int64_t j0, int64_t n_pix,
                                                           int32_t* next_queue) {
    requeue(w, queue, j0, n_pix, next_queue);
}

// ------------------------------------------------------------------ tracePaths output
__global__ void k_write_samples(Wave w, int64_t out0, int64_t n_paths, float* __restrict__ L_out,
                                uint32_t* __restrict__ sig_out) {
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < n_paths; p += (int64_t)gridDim.x * blockDim.x) {
        L_out[out0 + p] = w.L[p];
        if (sig_out) {
            uint32_t s = w.sig[p];
            const uint32_t pf = w.pflags[p];
            if (pf != NO_FLAGS) s = fnv(s, pf);
            sig_out[out0 + p] = s;
        }
    }
}

// Pixel at place i of the order that a frame's queue starts in: tiles of 16 x 16
// pixels, row by row within each.
constexpr int PIXEL_TILE = 16;
__device__ __forceinline__ int32_t tiled_pixel(int64_t i, int W, int H) {
    const int64_t band_size = (int64_t)PIXEL_TILE * W;
    const int band = (int)(i / band_size);
    const int bh = min(PIXEL_TILE, H - band * PIXEL_TILE);       // rows of the band
    const int in_band = (int)(i - band * band_size);
    const int tile = in_band / (PIXEL_TILE * bh);
    const int x0 = tile * PIXEL_TILE, tw = min(PIXEL_TILE, W - x0);
    const int in_tile = in_band - tile * (PIXEL_TILE * bh);
    const int y = in_tile / tw;
    return (band * PIXEL_TILE + y) * W + x0 + (in_tile - y * tw);
}

__global__ void k_pixel_queue(int32_t* q, int W, int H) {
    const int64_t n = (int64_t)W * H;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        q[i] = tiled_pixel(i, W, H);
}

// ------------------------------------------------------------------ launchers
static int grid_for(int64_t work, int block, int sms, int per_sm) {
    int64_t g = (work + block - 1) / block;
    const int64_t cap = (int64_t)sms * per_sm;
    if (g > cap) g = cap;
    if (g < 1) g = 1;
    return (int)g;
}

// traversal kernels by (batched jobs, BLAS layout, moving instances under a TLAS)
cudaError_t launch_trace(const DevScene& sc, const DevFrame& fr, const DevParams& P, const Wave& w, int ecur, int scur,
                         int depth, const Chunk& ch, int64_t max_n, int32_t* err, int sms, cudaStream_t st,
                         const Job* jobs, int trav, const RoundCtl* rc) {
    // both queues of at most max_n rays
    const int64_t work = scur >= 0 ? 2 * max_n : max_n;
#define MCEV_TRACE(kb, kw, kt)                                                                                      \
    k_trace<kb, kw, kt><<<grid_for(work, MCEV_TRAV_BLOCK, sms, trav_blocks(kw, kt)), MCEV_TRAV_BLOCK, 0, st>>>( \
        sc, fr, P, w, ecur, scur, depth, ch, err, jobs, depth == 0 ? rc : nullptr)
    switch ((jobs ? 4 : 0) | ((trav & TRAV_WIDE) ? 2 : 0) | ((trav & TRAV_TLAS) ? 1 : 0)) {
    case 0: MCEV_TRACE(false, false, false); break;
    case 1: MCEV_TRACE(false, false, true); break;
    case 2:
    case 3: MCEV_TRACE(false, true, true); break;
    case 4: MCEV_TRACE(true, false, false); break;
    case 5: MCEV_TRACE(true, false, true); break;
    default: MCEV_TRACE(true, true, true); break;
    }
#undef MCEV_TRACE
    return cudaGetLastError();
}

cudaError_t launch_shade(const DevScene& sc, const DevFrame& fr, const DevParams& P, const Wave& w, int cur,
                         int depth, bool last, int64_t max_n, int sms, cudaStream_t st, const Job* jobs) {
    const int resident = sms * Q_RESIDENT;
    const int grid = grid_for(max_n, Q_BLOCK, sms, 4 * Q_RESIDENT);
    if (jobs)
        k_shade<true, false><<<grid, Q_BLOCK, 0, st>>>(sc, fr, P, w, cur, depth, last ? 1 : 0, resident, jobs);
    else if (P.adjoint)
        k_shade<false, true><<<grid, Q_BLOCK, 0, st>>>(sc, fr, P, w, cur, depth, last ? 1 : 0, resident, nullptr);
    else
        k_shade<false, false><<<grid, Q_BLOCK, 0, st>>>(sc, fr, P, w, cur, depth, last ? 1 : 0, resident, nullptr);
    return cudaGetLastError();
}

cudaError_t launch_stats(const Wave& w, const StatsArgs& A, const int32_t* queue, int64_t j0, int64_t n_pix,
                         int32_t* next_queue, int sms, cudaStream_t st, const Job* jobs, const RoundCtl* rc) {
    // with rc, n_pix is an upper bound of the chunk's pixels (the size is on the device)
    const int64_t lanes = n_pix * (rc || stats_by_warp(n_pix, A.sub) ? 32 : 4);
    if (jobs)
        k_stats<false, true><<<grid_for(lanes, 256, sms, 8), 256, 0, st>>>(w, A, queue, j0, n_pix, next_queue,
                                                                                 jobs, rc);
    else
        k_stats<false, false><<<grid_for(lanes, 256, sms, 8), 256, 0, st>>>(w, A, queue, j0, n_pix, next_queue,
                                                                                  nullptr, rc);
    return cudaGetLastError();
}

cudaError_t launch_requeue(const Wave& w, const int32_t* queue, int64_t j0, int64_t n_pix, int32_t* next_queue,
                           cudaStream_t st) {
    k_requeue<<<1, REQUEUE_BLOCK, 0, st>>>(w, queue, j0, n_pix, next_queue);
    return cudaGetLastError();
}

static cudaError_t launch_stats_checked(const Wave& w, const StatsArgs& A, const int32_t* queue, int64_t n_pix,
                                        int32_t* next_queue, int sms, cudaStream_t st) {
    const int64_t lanes = n_pix * (stats_by_warp(n_pix, A.sub) ? 32 : 4);
    k_stats<true, false><<<grid_for(lanes, 256, sms, 8), 256, 0, st>>>(w, A, queue, 0, n_pix, next_queue, nullptr,
                                                                         nullptr);
    return cudaGetLastError();
}

// ------------------------------------------------------------------ device-resident round loop
// The rounds of Alg. 1's sampling schedule (Sec. 3.3) without the host: a
// CUDA graph runs k_round_init, then a conditional WHILE node whose body is
// one wavefront chunk (bounces, statistics) followed by
// k_round_next, which moves to the next chunk of the round or, at the end
// of a round, reads the number of re-queued pixels and sizes the next round
// (first round spp_min samples, then windows of spp_batch batches:
// round_window), and clears the condition when no pixel is left.  The loop
// is bounded: after plan.max_iters chunks, or plan.timeout_ns of wall clock
// (%globaltimer), it stops with RC_TIMEOUT, which the host reports as
// MCEV_ERR_TIMEOUT.
__device__ __forceinline__ unsigned long long global_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ void round_first_chunk(RoundCtl* rc, const RoundPlan& plan) {
    rc->per_chunk = max((int64_t)1, plan.cap / rc->spp_r);
    rc->j0 = 0;
    rc->nj = min(rc->per_chunk, rc->Q);
}

__global__ void k_round_init(RoundCtl* rc, Wave w, RoundPlan plan, int32_t* q0, int32_t* q1, int W, int H) {
    if (W > 0)
        for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < plan.Q0; i += (int64_t)gridDim.x * blockDim.x)
            q0[i] = tiled_pixel(i, W, H);
    if (blockIdx.x != 0 || threadIdx.x != 0) return;
    rc->queue[0] = q0;
    rc->queue[1] = q1;
    rc->Q = plan.Q0;
    rc->n_done = 0;
    rc->paths = 0;
    rc->stats_pix = 0;
    rc->qi = 0;
    rc->rounds = 0;
    rc->iters = 0;
    rc->status = RC_OK;
    rc->spp_r = rc->sub = min(plan.spp_min, plan.spp_max);
    round_first_chunk(rc, plan);
    w.counters[3] = 0;
    rc->t_start = global_ns();
}

__global__ void __launch_bounds__(REQUEUE_BLOCK) k_round_next(RoundCtl* rc, Wave w, RoundPlan plan,
                                                              cudaGraphConditionalHandle h) {
    // (no pixel goes on from the round that reaches spp_max; k_stats counts those it leaves open)
    if (rc->n_done + rc->spp_r < plan.spp_max)
        requeue(w, rc->queue[rc->qi], rc->j0, rc->nj, rc->queue[rc->qi ^ 1]);
    if (threadIdx.x != 0) return;
    rc->iters += 1;
    rc->stats_pix += rc->nj;
    unsigned int go = 1;
    if (rc->iters >= plan.max_iters || global_ns() - rc->t_start > plan.timeout_ns) {
        rc->status = RC_TIMEOUT;
        go = 0;
    } else if (rc->j0 + rc->per_chunk < rc->Q) {
        rc->j0 += rc->per_chunk;
        rc->nj = min(rc->per_chunk, rc->Q - rc->j0);
    } else {
        // the round is done: its undecided pixels form the next round
        rc->paths += rc->Q * (int64_t)rc->spp_r;
        rc->n_done += rc->spp_r;
        rc->rounds += 1;
        const int32_t q = *(volatile int32_t*)(w.counters + 3);
        w.counters[3] = 0;
        rc->qi ^= 1;
        rc->Q = q;
        if (q == 0) {
            go = 0;
        } else if (rc->n_done >= plan.spp_max) {
            rc->status = RC_CAP;
            go = 0;
        } else {
            const int64_t sub = plan.spp_batch;
            const int64_t m = round_window(plan.cap, q, sub, rc->n_done, plan.spp_max, plan.window_max,
                                           plan.uniform != 0);
            rc->sub = (int32_t)sub;
            rc->spp_r = (int32_t)min(m * sub, (int64_t)plan.spp_max - rc->n_done);
            round_first_chunk(rc, plan);
        }
    }
    cudaGraphSetConditional(h, go);
}

cudaError_t launch_round_init(RoundCtl* rc, const Wave& w, const RoundPlan& plan, int32_t* q0, int32_t* q1,
                              int W, int H, int sms, cudaStream_t st) {
    k_round_init<<<W > 0 ? grid_for(plan.Q0, 256, sms, 8) : 1, 256, 0, st>>>(rc, w, plan, q0, q1, W, H);
    return cudaGetLastError();
}

cudaError_t launch_round_next(RoundCtl* rc, const Wave& w, const RoundPlan& plan, cudaGraphConditionalHandle h,
                              cudaStream_t st) {
    k_round_next<<<1, REQUEUE_BLOCK, 0, st>>>(rc, w, plan, h);
    return cudaGetLastError();
}

// out[i] += (float)acc[i]
__global__ void k_add_f64(float* __restrict__ out, const double* __restrict__ acc, int n) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
        out[i] += (float)acc[i];
}

cudaError_t launch_add_f64(float* out, const double* acc, int n, cudaStream_t st) {
    k_add_f64<<<(n + 255) / 256, 256, 0, st>>>(out, acc, n);
    return cudaGetLastError();
}

// queue entries (job << 24 | pixel) of one job
__global__ void k_fill_entries(int32_t* q, int W, int H, int job) {
    const int64_t n = (int64_t)W * H;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        q[i] = (int32_t)(((uint32_t)job << 24) | (uint32_t)tiled_pixel(i, W, H));
}

cudaError_t launch_fill_entries(int32_t* q, int W, int H, int job, int sms, cudaStream_t st) {
    k_fill_entries<<<grid_for((int64_t)W * H, 256, sms, 8), 256, 0, st>>>(q, W, H, job);
    return cudaGetLastError();
}

cudaError_t launch_write_samples(const Wave& w, int64_t out0, int64_t n_paths, float* L_out, uint32_t* sig_out,
                                 int sms, cudaStream_t st) {
    k_write_samples<<<grid_for(n_paths, 256, sms, 8), 256, 0, st>>>(w, out0, n_paths, L_out, sig_out);
    return cudaGetLastError();
}

cudaError_t launch_pixel_queue(int32_t* q, int W, int H, int sms, cudaStream_t st) {
    k_pixel_queue<<<grid_for((int64_t)W * H, 256, sms, 8), 256, 0, st>>>(q, W, H);
    return cudaGetLastError();
}

}  // namespace mcev

// ------------------------------------------------------------------ allocation-free detector step
// Scratch of mcev_detect_batch_static: int32 counters [0, 256) in the layout
// of Wave::counters (layout.h lists every slot; k_stats uses [3]-[8] and the
// uint64 word [32 + 6]) followed by the critical-t table.  It lives in the
// library image so the call never allocates; host code reaches it only
// through the address cudaGetSymbolAddress returns for the current device.
static __device__ __align__(256) unsigned char g_detect_scratch[MCEV_DETECT_STATIC_SCRATCH_BYTES];

namespace {

struct StaticDevice {
    void* scratch = nullptr;
    int sms = 0;
    bool ready = false;
};
constexpr int kMaxDevices = 64;
StaticDevice g_static_dev[kMaxDevices];
std::mutex g_static_mu;

mcev_status static_fail(const mcev_detect_args* a, mcev_status s, const char* msg) {
    if (a && a->err_msg && a->err_len > 0) {
        size_t i = 0;
        for (; msg[i] && i + 1 < a->err_len; ++i) a->err_msg[i] = msg[i];
        a->err_msg[i] = 0;
    }
    return s;
}

}  // namespace

extern "C" mcev_status mcev_detect_batch_static(const mcev_detect_args* a, int64_t* n_undecided) {
    using namespace mcev;
    if (!a || !n_undecided) return MCEV_ERR_ARG;
    if (!a->L || !a->pixels || !a->cur_n || !a->cur_mean || !a->cur_m2 || !a->ref_n || !a->ref_mean ||
        !a->ref_m2 || !a->events || !a->undecided)
        return static_fail(a, MCEV_ERR_ARG, "mcev_detect_batch_static: a required pointer is NULL");
    if (a->n_pix < 0 || a->n_total < 1 || a->spp_r < 1 || a->k_base < 0 || a->reserved0 != 0 || a->spp_min < 2 ||
        a->spp_batch < 1 || a->spp_max < a->spp_min || a->k_base + a->spp_r > a->spp_max ||
        (a->k_base == 0 && a->spp_r != a->spp_min) || !(a->eps > 0.0f) || !(a->C >= 0.0f) ||
        !(a->alpha > 0.0f && a->alpha < 1.0f) || a->variant < 0 || a->variant > 3 || a->se_mode < 0 ||
        a->se_mode > 1 || (int64_t)a->n_pix * a->spp_r > ((int64_t)1 << 40))
        return static_fail(a, MCEV_ERR_ARG, "mcev_detect_batch_static: inconsistent sizes or settings");
    // Later calls must start on the test schedule spp_min + r * spp_batch and
    // cover whole batches (only the last batch of the frame may be shorter, as
    // it ends at spp_max), so that the kernel tests at every schedule point the
    // window crosses and each test reads the critical value of its own count.
    if (a->k_base > 0 && (a->k_base < a->spp_min || (a->k_base - a->spp_min) % a->spp_batch != 0 ||
                          (a->spp_r % a->spp_batch != 0 && a->k_base + a->spp_r != a->spp_max)))
        return static_fail(a, MCEV_ERR_ARG,
                           "mcev_detect_batch_static: call off the test schedule: k_base must be spp_min + r * "
                           "spp_batch and spp_r a multiple of spp_batch (or end at spp_max)");
    const int64_t n_tests = (a->spp_max - a->spp_min + a->spp_batch - 1) / a->spp_batch;
    if (n_tests > MCEV_DETECT_STATIC_MAX_TESTS)
        return static_fail(a, MCEV_ERR_ARG,
                           "mcev_detect_batch_static: the schedule needs more than 4096 t-tests; the fixed "
                           "scratch holds 4096 critical values (raise spp_batch or lower spp_max)");
    *n_undecided = 0;
    if (a->n_pix == 0) return MCEV_OK;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) {
        cudaGetLastError();
        return static_fail(a, MCEV_ERR_CUDA, "mcev_detect_batch_static: no usable current CUDA device");
    }
    StaticDevice sd;
    {
        std::lock_guard<std::mutex> lock(g_static_mu);
        StaticDevice& s = g_static_dev[dev];
        if (!s.ready) {
            void* p = nullptr;
            if (cudaGetSymbolAddress(&p, g_detect_scratch) != cudaSuccess || !p) {
                cudaGetLastError();
                return static_fail(a, MCEV_ERR_CUDA, "mcev_detect_batch_static: cudaGetSymbolAddress failed");
            }
            int sms = 0;
            if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
                cudaGetLastError();
                return static_fail(a, MCEV_ERR_CUDA, "mcev_detect_batch_static: device query failed");
            }
            s.scratch = p;
            s.sms = sms;
            s.ready = true;
        }
        sd = s;
    }
    cudaStream_t st = (cudaStream_t)a->stream;
    int32_t* counters = (int32_t*)sd.scratch;
    float* tcrit = (float*)((unsigned char*)sd.scratch + 256);
    float tab[MCEV_DETECT_STATIC_MAX_TESTS];
    int nt = 0;
    if (a->variant == VAR_ONE_TAILED || a->variant == VAR_TWO_TAILED) {
        const double p = a->variant == VAR_TWO_TAILED ? 0.5 * (double)a->alpha : (double)a->alpha;
        for (int n = a->spp_min; n < a->spp_max; n += a->spp_batch) tab[nt++] = (float)t_quantile_int(p, n - 1);
    }
    if (cudaMemsetAsync(counters, 0, 256, st) != cudaSuccess ||
        (nt > 0 && cudaMemcpyAsync(tcrit, tab, sizeof(float) * nt, cudaMemcpyHostToDevice, st) != cudaSuccess)) {
        cudaGetLastError();
        return static_fail(a, MCEV_ERR_CUDA, "mcev_detect_batch_static: scratch initialisation failed");
    }
    Wave w{};
    w.L = const_cast<float*>(a->L);
    w.counters = counters;
    StatsArgs A{};
    A.cur = PixStats{a->cur_n, a->cur_mean, a->cur_m2};
    A.ref = PixStats{a->ref_n, a->ref_mean, a->ref_m2};
    A.tcrit = tcrit;
    A.events = a->events;
    A.spp_out = a->spp_out;
    A.mean_out = a->mean_out;
    A.eps = a->eps;
    A.C = a->C;
    A.spp_r = a->spp_r;
    // the first call is the first batch (spp_min samples, one test at its
    // end); a later call's samples are merged and tested one spp_batch at a time
    A.sub = a->k_base == 0 ? a->spp_r : a->spp_batch;
    A.k_base = a->k_base;
    A.spp_min = a->spp_min;
    A.spp_batch = a->spp_batch;
    A.spp_max = a->spp_max;
    A.mode = MODE_DETECT;
    A.variant = a->variant;
    A.se_mode = a->se_mode;
    A.n_total = a->n_total;
    if (launch_stats_checked(w, A, a->pixels, a->n_pix, a->undecided, sd.sms, st) != cudaSuccess)
        return static_fail(a, MCEV_ERR_CUDA, "mcev_detect_batch_static: kernel launch failed");
    int32_t c[16];
    if (cudaMemcpyAsync(c, counters, sizeof c, cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess) {
        cudaGetLastError();
        return static_fail(a, MCEV_ERR_CUDA, "mcev_detect_batch_static: kernel or copy failed");
    }
    *n_undecided = c[3];
    if (c[8])
        return static_fail(a, MCEV_ERR_ARG,
                           "mcev_detect_batch_static: a pixel id was outside [0, n_total); those pixels were skipped");
    return MCEV_OK;
}
