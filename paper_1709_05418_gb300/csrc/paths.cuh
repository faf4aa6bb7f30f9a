// paths.cuh -- warp-wide tracing of many independent L_i paths (Sec. 4.4, Sec. 5.1), for the
// path-traced render mode and the training labels.
//
// A path alternates phase sampling, delta tracking to the next collision, survival with
// probability albedo and next-event estimation there, and its length varies by orders of
// magnitude (HG 0.85, albedo 0.99).  With a path per lane in nested loops a warp ran 4 of its
// 32 lanes per instruction: every loop ends with its longest lane.  Here each lane is a state
// machine and the warp runs one step of all lanes at a time: a step is one tentative
// collision, of a free flight (global majorant) or of a shadow ray (brick majorants), whose
// random block, logarithm and density lookup both kinds share.  What happens once per bounce
// (a new direction, survival and the shadow ray's set-up, the next path for a lane that ended
// one) waits until several lanes need it (kEventLanes) or as many lanes wait as run.
// The arithmetic whose contraction the compiler would otherwise choose by the code around it
// (positions, the optical depth spent, the phase cosine) is written out with one rounding
// sequence.  Every path does the arithmetic and the draws of its own stream in the order direction block,
// tracking blocks, survival block, shadow blocks, per bounce, so its estimate does not depend
// on the lane, the warp or the other paths.  The vertex the path starts from is its first
// bounce (full phase function); everything after it uses the medium behind the first bounce
// (v.lmc, v.dscale, v.albedo_c).
#pragma once
#include "common.cuh"

namespace rpnn {

constexpr int kEventLanes = 8;
constexpr uint32_t kPathPolls = 1u << 24;     // bound on a warp's polls for other warps' results

// Source of paths and sink of estimates for trace_paths:
//   int fetch(bool want, x, d, rng)  warp-collective; 1: the lane got a path, 0: none yet, -1: none
//   void finish(L, capped)           the lane's path ended (capped: a device loop reached its cap)
//   bool stopped()                   warp-uniform: drop everything in flight
//   bool keep()                      warp-uniform: stay although no lane has work left
//   void gave_up()                   the bound on polls was reached
template <class Src>
__device__ __forceinline__ void trace_paths(const VolumeView& v, const float3 wl, const float E, Src& src) {
    enum { kFetch, kTurn, kHit, kFly, kShadow, kWait, kDone };
    int state = kFetch, b = 0;
    float3 x = f3(0.f, 0.f, 0.f), d = f3(0.f, 0.f, 1.f);
    float t = 0.0f, t1 = 0.0f, L = 0.0f, T = 1.0f, te = 0.0f, mu_b = 0.0f;
    uint32_t ctr = 0, n = 0, polls = 0;
    Rng rng = make_rng(0, 0, 0, 0);
    BrickWalk w{};
    bool capped = false;
    const float maj_s = v.majorant * v.dscale;
    // the point at t along e from x
    auto at = [&](const float3 e) { return f3(__fmaf_rn(t, e.x, x.x), __fmaf_rn(t, e.y, x.y), __fmaf_rn(t, e.z, x.z)); };
    auto end = [&]() { src.finish(L, capped); state = kFetch; };
    // next-event estimate of the vertex x from the shadow ray's transmittance; next bounce
    auto nee_done = [&]() {
        const float ct = __fmaf_rn(d.z, wl.z, __fmaf_rn(d.x, wl.x, __fmul_rn(d.y, wl.y)));
        L = __fmaf_rn(__fmul_rn(E, phase_eval(v, v.lmc, ct)), T, L);
        ++b;
        state = kTurn;
    };
    // the shadow ray's brick at t; false once it has left the grid or reached its cap
    auto brick = [&]() { te = walk_exit(w, t1); mu_b = walk_majorant(v, w); };
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
        const int ev = __popc(__ballot_sync(0xffffffffu, state <= kHit));
        if (run == 0 && ev == 0 && !__any_sync(0xffffffffu, state == kWait) && !src.keep()) break;
        if (src.stopped()) break;
        if (run == 0 || ev >= kEventLanes || ev >= run) {
            if (state == kHit) {
                const float4 xi = rng.draw(ctr++);
                float t0;
                if (!(xi.x < v.albedo_c)) {
                    end();
                } else {
                    T = 1.0f;
                    if (v.majorant <= 0.0f || !box_clip(v.ext, x, wl, t0, t1)) {
                        nee_done();
                    } else {
                        walk_init(v, x, wl, t0, w);
                        t = t0;
                        n = 0;
                        brick();
                        bool in = true;
                        while (in && !(mu_b > 0.0f)) in = advance();    // empty bricks spend nothing
                        if (in) state = kShadow;
                        else nee_done();
                    }
                }
            }
            const int got = src.fetch(state == kFetch || state == kWait, x, d, rng);
            if (state == kFetch || state == kWait) {
                if (got > 0) { state = kTurn; b = 0; ctr = 0; L = 0.0f; capped = false; }
                else state = got < 0 ? kDone : kWait;
            }
            if (state == kTurn) {
                if (b >= kBounceCap) {
                    capped = true;
                    end();
                } else {
                    const float4 xi = rng.draw(ctr++);
                    d = phase_sample(v, b == 0 ? v.lm : v.lmc, d, xi.x, xi.y);
                    float t0;
                    if (v.majorant <= 0.0f || !box_clip(v.ext, x, d, t0, t1)) end();
                    else { t = t0; n = 0; state = kFly; }
                }
            }
            if (run == 0 && !__any_sync(0xffffffffu, state < kWait)) {
                // only waiting for other warps of the block
                if (++polls >= kPathPolls) { src.gave_up(); break; }
                __nanosleep(200);
            }
            continue;
        }
        const bool fly = state == kFly, shadow = state == kShadow;
        bool look = false;
        float3 p = x;
        float xy = 0.0f;
        if (fly || shadow) {
            const float4 xi = rng.draw(ctr++);
            const float lg = logf(1.0f - xi.x);
            xy = xi.y;
            if (fly) {
                t -= lg / maj_s;
                if (t >= t1) end();
                else { p = at(d); look = true; }
            } else {
                float tau = -lg;
                bool in = true;
                while (in) {
                    if (mu_b > 0.0f) {
                        const float mu_s = mu_b * v.dscale;
                        const float seg = __fmul_rn(mu_s, __fsub_rn(te, t));
                        if (tau < seg) {
                            t += tau / mu_s;
                            break;
                        }
                        tau = __fsub_rn(tau, seg);
                    }
                    in = advance();
                }
                if (in) { p = at(wl); look = true; }
                else nee_done();
            }
        }
        if (look) {
            const float mu = raw_density(v, p);
            if (fly) {
                if (xy * v.majorant < mu) { x = p; state = kHit; }
                else if (++n >= v.track_cap) { capped = true; end(); }
            } else {
                T *= 1.0f - mu / mu_b;
                if (++n >= v.track_cap) { capped = true; nee_done(); }
            }
        }
    }
}

}  // namespace rpnn
