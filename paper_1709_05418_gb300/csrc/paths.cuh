// paths.cuh -- warp-wide tracing of many independent L_i paths (Sec. 4.4, Sec. 5.1), for the
// path-traced render mode and the training labels.
//
// A path alternates phase sampling, delta tracking to the next collision, survival with
// probability albedo and next-event estimation there, and its length varies by orders of
// magnitude (HG 0.85, albedo 0.99).  With a path per lane in nested loops a warp ran 4 of its
// 32 lanes per instruction: every loop ends with its longest lane.  Here each lane is a state
// machine and the warp runs one step of all lanes at a time: a step is one tentative
// collision, of a free flight (global majorant) or of a shadow ray (brick majorants), whose
// random block, logarithm and density lookup both kinds share; a shadow ray crosses at most
// kWalkSteps bricks a step.  What happens once per bounce (the end of a shadow ray, survival
// and the next shadow ray's set-up, a new direction, the next path for a lane that ended one)
// waits, each of the two kinds by itself, until kEventLanes lanes need it or as many as run.
// The arithmetic whose contraction the compiler would otherwise choose by the code around it
// (positions, the optical depth spent, the phase cosine) is written out with one rounding
// sequence.  Every path does the arithmetic and the draws of its own stream in the order direction block,
// tracking blocks, survival block, shadow blocks, per bounce, so its estimate does not depend
// on the lane, the warp or the other paths.  The vertex the path starts from is its first
// bounce (full phase function); everything after it uses the medium behind the first bounce
// (v.lmc, v.dscale, v.albedo_c).
#pragma once
#include "common.cuh"
#include "rules.h"

namespace rpnn {

constexpr int kEventLanes = 11;               // 5 to 18 lanes, 3 to 6 bricks: within 5 % of one another
constexpr int kWalkSteps = 4;

// Source of paths and sink of estimates for trace_paths:
//   int fetch(bool want, x, d, rng)  warp-collective; 1: the lane got a path, 0: none yet, -1: none
//   void finish(L, capped)           the lane's path ended (capped: a device loop reached its cap)
//   bool stopped()                   warp-uniform: drop everything in flight
//   bool keep()                      warp-uniform: stay although no lane has work left
//   void beat()                      a bounce of this warp's lanes: what other warps' waits see as progress
//   bool idle(bound)                 warp-uniform: one more poll for other warps; false: the bound is reached
template <class Src>
__device__ __forceinline__ void trace_paths(const VolumeView& v, const float3 wl, const float E, Src& src) {
    enum { kHit, kFetch, kEnd, kExit, kTurn, kFly, kShadow, kWait, kDone };
    int state = kFetch, b = 0;
    float3 x = f3(0.f, 0.f, 0.f), d = f3(0.f, 0.f, 1.f);
    float t = 0.0f, t1 = 0.0f, L = 0.0f, T = 1.0f, te = 0.0f, mu_b = 0.0f;
    float tau = -1.0f;                  // shadow ray: optical depth left to spend, < 0: draw first
    uint32_t ctr = 0, n = 0;
    Rng rng = make_rng(0, 0, 0, 0);
    BrickWalk w{};
    bool capped = false;
    const float maj_s = v.majorant * v.dscale;
    // the point at t along e from x
    auto at = [&](const float3 e) { return f3(__fmaf_rn(t, e.x, x.x), __fmaf_rn(t, e.y, x.y), __fmaf_rn(t, e.z, x.z)); };
    auto brick = [&]() { te = walk_exit(w, t1); mu_b = walk_majorant(v, w); };
    // the shadow ray into its next brick; false once it has left the grid or reached its cap
    auto advance = [&]() {
        if (te >= t1) return false;
        t = te;
        if (!walk_step(v, w)) return false;
        if (++n >= v.track_cap) { capped = true; return false; }
        brick();
        return true;
    };
    for (;;) {
        const int run = __popc(__ballot_sync(0xffffffffu, state == kFly || state == kShadow));
        const int hits = __popc(__ballot_sync(0xffffffffu, state == kHit));
        const int turns = __popc(__ballot_sync(0xffffffffu, state > kHit && state <= kTurn));
        if (run + hits + turns == 0 && !__any_sync(0xffffffffu, state == kWait) && !src.keep()) break;
        if (src.stopped()) break;
        const bool do_hits = hits >= min(kEventLanes, run), do_turns = turns >= min(kEventLanes, run);
        if (do_hits && hits) {
            src.beat();
            if (state == kHit) {
                const float4 xi = rng.draw(ctr++);
                float t0;
                if (!(xi.x < v.albedo_c)) {
                    state = kEnd;
                } else {
                    T = 1.0f;
                    if (v.majorant <= 0.0f || !box_clip(v.ext, x, wl, t0, t1)) {
                        state = kExit;
                    } else {
                        walk_init(v, x, wl, t0, w);
                        t = t0;
                        n = 0;
                        brick();
                        bool in = true;
                        while (in && !(mu_b > 0.0f)) in = advance();    // empty bricks spend nothing
                        state = in ? kShadow : kExit;
                        tau = -1.0f;
                    }
                }
            }
            continue;
        }
        if (do_turns && (turns || run == 0)) {
            if (turns) src.beat();
            if (state == kExit) {
                // next-event estimate of the vertex x from the shadow ray's transmittance; next bounce
                const float ct = __fmaf_rn(d.z, wl.z, __fmaf_rn(d.x, wl.x, __fmul_rn(d.y, wl.y)));
                L = __fmaf_rn(__fmul_rn(E, phase_eval(v, v.lmc, ct)), T, L);
                ++b;
                state = kTurn;
            }
            if (state == kEnd) {
                src.finish(L, capped);
                state = kFetch;
            }
            const int got = src.fetch(state == kFetch || state == kWait, x, d, rng);
            if (state == kFetch || state == kWait) {
                if (got > 0) { state = kTurn; b = 0; ctr = 0; L = 0.0f; capped = false; }
                else state = got < 0 ? kDone : kWait;
            }
            if (state == kTurn) {
                if (b >= kBounceCap) {
                    capped = true;
                    state = kEnd;
                } else {
                    const float4 xi = rng.draw(ctr++);
                    d = phase_sample(v, b == 0 ? v.lm : v.lmc, d, xi.x, xi.y);
                    float t0;
                    const bool in = v.majorant > 0.0f && box_clip(v.ext, x, d, t0, t1);
                    state = in ? kFly : kEnd;
                    if (in) { t = t0; n = 0; }
                }
            }
            if (run == 0 && turns == 0 && !__any_sync(0xffffffffu, state < kWait)) {
                // only waiting for other warps of the block
                if (!src.idle(path_poll_bound(v.track_cap))) break;
                __nanosleep(200);
            }
            continue;
        }
        const bool fly = state == kFly;
        bool look = false;
        float xy = 0.0f;
        if (fly || (state == kShadow && tau < 0.0f)) {
            const float4 xi = rng.draw(ctr++);
            const float lg = logf(1.0f - xi.x);
            xy = xi.y;
            tau = -lg;
            if (fly) {
                t -= lg / maj_s;
                look = t < t1;
                if (!look) state = kEnd;
            }
        }
        if (state == kShadow) {
            for (int k = 0; k < kWalkSteps; ++k) {
                if (mu_b > 0.0f) {
                    const float mu_s = mu_b * v.dscale;
                    const float seg = __fmul_rn(mu_s, __fsub_rn(te, t));
                    if (tau < seg) {
                        t += tau / mu_s;
                        look = true;
                        break;
                    }
                    tau = __fsub_rn(tau, seg);
                }
                if (!advance()) { state = kExit; break; }
            }
        }
        if (look) {
            const float3 p = at(fly ? d : wl);
            const float mu = raw_density(v, p);
            if (fly) {
                if (xy * v.majorant < mu) { x = p; state = kHit; }
                else if (++n >= v.track_cap) { capped = true; state = kEnd; }
            } else {
                T *= 1.0f - mu / mu_b;
                tau = -1.0f;
                if (++n >= v.track_cap) { capped = true; state = kExit; }
            }
        }
    }
}

// One path by itself, in nested loops: the same draws and the same rounding sequence as trace_paths,
// so the same estimate.  For a lane of the primary pass, where paths are so short that listing
// them for a second launch costs more than its shared steps save (path_in_primary).
__device__ __forceinline__ float trace_path(const VolumeView& v, float3 x, float3 d, const float3 wl, const float E,
                                            const Rng& rng, bool& capped) {
    const float maj_s = v.majorant * v.dscale;
    uint32_t ctr = 0;
    float L = 0.0f;
    for (int b = 0; b < kBounceCap; ++b) {
        float4 xi = rng.draw(ctr++);
        d = phase_sample(v, b == 0 ? v.lm : v.lmc, d, xi.x, xi.y);
        float t, t1;
        if (!(v.majorant > 0.0f) || !box_clip(v.ext, x, d, t, t1)) return L;
        for (uint32_t n = 0;;) {
            xi = rng.draw(ctr++);
            t -= logf(1.0f - xi.x) / maj_s;
            if (!(t < t1)) return L;
            const float3 p = f3(__fmaf_rn(t, d.x, x.x), __fmaf_rn(t, d.y, x.y), __fmaf_rn(t, d.z, x.z));
            if (xi.y * v.majorant < raw_density(v, p)) { x = p; break; }
            if (++n >= v.track_cap) { capped = true; return L; }
        }
        xi = rng.draw(ctr++);
        if (!(xi.x < v.albedo_c)) return L;
        // next-event estimate: ratio tracking towards the light
        float T = 1.0f;
        if (box_clip(v.ext, x, wl, t, t1)) {
            BrickWalk w;
            walk_init(v, x, wl, t, w);
            float tau = -1.0f;
            for (uint32_t n = 0;;) {
                const float te = walk_exit(w, t1), mu_b = walk_majorant(v, w);
                if (mu_b > 0.0f) {
                    if (tau < 0.0f) tau = -logf(1.0f - rng.draw(ctr++).x);
                    const float mu_s = mu_b * v.dscale;
                    const float seg = __fmul_rn(mu_s, __fsub_rn(te, t));
                    if (tau < seg) {
                        t += tau / mu_s;
                        const float3 p = f3(__fmaf_rn(t, wl.x, x.x), __fmaf_rn(t, wl.y, x.y), __fmaf_rn(t, wl.z, x.z));
                        T *= 1.0f - raw_density(v, p) / mu_b;
                        tau = -1.0f;
                        if (++n >= v.track_cap) { capped = true; break; }
                        continue;
                    }
                    tau = __fsub_rn(tau, seg);
                }
                if (te >= t1) break;
                t = te;
                if (!walk_step(v, w)) break;
                if (++n >= v.track_cap) { capped = true; break; }
            }
        }
        const float ct = __fmaf_rn(d.z, wl.z, __fmaf_rn(d.x, wl.x, __fmul_rn(d.y, wl.y)));
        L = __fmaf_rn(__fmul_rn(E, phase_eval(v, v.lmc, ct)), T, L);
    }
    capped = true;
    return L;
}

}  // namespace rpnn
