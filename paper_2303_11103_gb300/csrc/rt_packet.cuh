// rt_packet.cuh -- traversal by whole warps: the rays of a warp that lie close
// together go through the scene as one beam.
//
// Besides the binary hierarchy the scene has an implicit tree of 32 children a
// node: groups of 32 leaves (along a Hilbert curve in flat scenes, else in
// Morton order), sets of 32 groups; the
// large triangles stand apart, 32 a round. A lane tests one child's box
// against the beam (the interval of the rays' origins moving with the interval
// of their directions), so one round answers for 32 boxes and all rays of the
// beam, where the per-ray traversal spends a visit per node and lane. Children
// are taken nearest first while they begin before the farthest current hit;
// triangles that the beam reaches are tested by every ray, with the per-ray
// traversal's test and ties, so both find the same hits: a hit is the smallest
// distance over all triangles, equal ones to the lowest id, and the boxes are
// widened beyond what rounding can shift: by 4e-6 of the scene's extent or of
// its largest coordinate, where a plane at p seen from o is off by at most
// 3.6e-7 (|p| + |o|) (rounded products and a reciprocal within two units).
//
// Boxes at s.pk, 32-byte records: first (groups, sets, large triangles rounded
// up to 32, records of a copy), then 8 copies, one for each octant of
// directions, of: 32 leaves a group; 32 groups a set; the sets and the large
// triangles, padded to multiples of 32 by boxes no beam meets. A record holds
// the entry and exit planes of its octant in pairs (lo and hi where the
// direction is positive, hi and lo where it is negative) and, for a triangle,
// its index in s.tris. With the planes in this order a box test is three packed
// FMAs and four min / max; with one copy of lo and hi, chosen between and
// subtracted in the test, it took three times the instructions (64-transmitter
// map 99.4 ms, 92.7 with the copies).
#pragma once
#include "rt_common.cuh"

// Rays of a beam differ by at most PK_DIR in each direction component, and by
// at most the scene's pk_rho (half the spacing of its groups) in each origin
// coordinate. A warp whose rays fall into more than PK_BEAMS beams, or into more
// than one with fewer than PK_FEW rays in all, traces those of PK_MIN rays or
// more as beams and the others ray by ray, all at once: a beam costs about half
// of such a traversal. (0.05 to 0.3, 0.125 to 0.8 and 2 to 10 beams: within 5 %
// where the rays are dense; a limit on a beam's triangle tests, 16 to 64, cost
// 2 to 10 %.)
constexpr float PK_DIR = 0.2f;
constexpr int PK_MIN = 12, PK_FEW = 16, PK_BEAMS = 4;

__device__ __forceinline__ float warp_min(float x) {
    float r;
    asm volatile("redux.sync.min.f32 %0, %1, 0xffffffff;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ float warp_max(float x) {
    float r;
    asm volatile("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(r) : "f"(x));
    return r;
}

// At t the beam covers [olo + dlo t, ohi + dhi t] on an axis; it overlaps
// [lo, hi] where lo <= ohi + dhi t and hi >= olo + dlo t, each a bound on t
// from below or above by the sign of the slope. Where both slopes are upward
// or both downward, one plane bounds the entry (n) and the other the exit (f),
// as for a ray; where they part, both bound the entry (open), and where they
// close in, both the exit (shut).
struct BeamAxis {
    float2 r, c;            // reciprocal slopes and -origin * slope, for the entry and the exit plane
    bool neg, open, shut;   // neg: the entry plane is hi
};
struct Beam {
    BeamAxis x, y, z;
    bool odd;               // some axis open or shut
};

__device__ __forceinline__ BeamAxis beam_axis(float olo, float ohi, float dlo, float dhi) {
    const float rlo = __fdividef(1.0f, dlo >= 0.0f ? fmaxf(dlo, 1e-30f) : fminf(dlo, -1e-30f));
    BeamAxis a;
    a.neg = dlo < 0.0f && dhi <= 0.0f;
    a.open = dlo < 0.0f && dhi > 0.0f;
    a.shut = dlo > 0.0f && dhi < 0.0f;
    const float rhi = __fdividef(1.0f, dhi > 0.0f || (dlo >= 0.0f && !a.shut) ? fmaxf(dhi, 1e-30f) : fminf(dhi, -1e-30f));
    a.r = a.neg ? make_float2(rlo, rhi) : make_float2(rhi, rlo);
    a.c = a.neg ? make_float2(-olo * rlo, -ohi * rhi) : make_float2(-ohi * rhi, -olo * rlo);
    return a;
}
// rays: origin and direction
__device__ __forceinline__ BeamAxis ray_axis(bool mine, float o, float d) {
    const float inf = __int_as_float(0x7f800000);
    return beam_axis(warp_min(mine ? o : inf), warp_max(mine ? o : -inf), warp_min(mine ? d : inf),
                     warp_max(mine ? d : -inf));
}
// segments: start (t = 0) and end (t = 1); the chords between the extremes
// bound the segments in between
__device__ __forceinline__ BeamAxis seg_axis(bool mine, float o, float e) {
    const float inf = __int_as_float(0x7f800000);
    const float olo = warp_min(mine ? o : inf), ohi = warp_max(mine ? o : -inf);
    return beam_axis(olo, ohi, warp_min(mine ? e : inf) - olo, warp_max(mine ? e : -inf) - ohi);
}

// Where the beam enters a record's box (bits of the distance, or of +inf when
// it misses the box before tmax). ref: the record's triangle.
__device__ __forceinline__ unsigned beam_box(const Beam& b, const float4* box, float tmin, float tmax, int& ref) {
    const float inf = __int_as_float(0x7f800000);
    float4 p, q;
    ldg8(box, p, q);
    ref = __float_as_int(q.z);
    const float2 x = fma2(p.x, p.y, b.x.r, b.x.c), y = fma2(p.z, p.w, b.y.r, b.y.c), z = fma2(q.x, q.y, b.z.r, b.z.c);
    const float nx = x.x, fx = x.y, ny = y.x, fy = y.y, nz = z.x, fz = z.y;
    float tn = fmax3(nx, ny, fmaxf(nz, tmin)), tf;
    if (!b.odd) {
        tf = fmin3(fx, fy, fminf(fz, tmax));
    } else {
        tn = fmax3(b.x.shut ? -inf : nx, b.y.shut ? -inf : ny, fmaxf(b.z.shut ? -inf : nz, tmin));
        tn = fmax3(fmaxf(tn, b.x.open ? fx : -inf), b.y.open ? fy : -inf, b.z.open ? fz : -inf);
        tf = fmin3(b.x.open ? inf : fx, b.y.open ? inf : fy, fminf(b.z.open ? inf : fz, tmax));
        tf = fmin3(fminf(tf, b.x.shut ? nx : inf), b.y.shut ? ny : inf, b.z.shut ? nz : inf);
    }
    return tn <= tf ? __float_as_uint(tn) : 0x7f800000u;
}

// The nearest remaining child of a level: its lane, or -1 when none begins by
// `far`. The child is taken off.
__device__ __forceinline__ int take_nearest(unsigned& key, unsigned far) {
    const unsigned k = __reduce_min_sync(0xffffffffu, key);
    if (k > far || k == 0x7f800000u) return -1;
    const int src = __ffs(__ballot_sync(0xffffffffu, key == k)) - 1;
    if ((int)(threadIdx.x & 31) == src) key = 0x7f800000u;
    return src;
}

// One beam. SEG false, for the rays of `mine`: the closest hit before t (t,
// id), or for rays of `any` whether something is hit before t (id >= 0 then, t
// is left). SEG: for the segments of `mine`, o + [0, t] d from the beam's 0 to
// 1, whether something is hit before t (id: the triangle's index in s.tris).
// Triangles ex0 and ex1 are skipped. Called by all 32 lanes. One loop serves
// all levels (one copy of the box and triangle tests: the kernels around it
// are large enough to miss the instruction cache).
template <bool SEG>
__device__ __forceinline__ void beam_walk(const DevScene& s, const Beam& b, bool mine, bool any, f3 o, f3 d, int ex0,
                                          int ex1, float& t, int& id) {
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const float tmin = s.tmin;
    // distance up to which some ray still looks for a hit
    auto far_of = [&]() {
        return __reduce_max_sync(full, mine && !(any && id >= 0) ? __float_as_uint(SEG ? 1.0f : t) : 0u);
    };
    unsigned far = far_of();
    const int4 n = __ldg(reinterpret_cast<const int4*>(s.pk));   // groups, sets, large triangles, records
    const int oct = (b.x.neg ? 1 : 0) | (b.y.neg ? 2 : 0) | (b.z.neg ? 4 : 0);
    const float4* boxes = s.pk + 2 * (1 + (size_t)oct * n.w + lane);
    const int r1 = 32 * n.x, r2 = r1 + 32 * n.y, rb = r2 + (n.y + 31) / 32 * 32;   // first records of the levels
    unsigned key1 = 0x7f800000u, key2 = 0x7f800000u;
    int level = 2, rec = r2, next2 = r2, next1 = 0;   // the round's level and first record; those of key2, key1
    int k2 = r2, kb = rb;                             // sets and large triangles not yet looked at
    while (true) {
        if (level == 2) {
            if (k2 < r2 + n.y) {
                rec = next2 = k2;
                k2 += 32;
            } else if (kb < rb + n.z) {
                rec = kb;
                kb += 32;
                level = 0;
            } else {
                break;
            }
        }
        int ref;
        unsigned key = beam_box(b, boxes + 2 * (size_t)rec, SEG ? 0.0f : tmin, __uint_as_float(far), ref);
        if (level == 2) {
            key2 = key;
        } else if (level == 1) {
            key1 = key;
            next1 = rec;
        } else {
            int src;
            while ((src = take_nearest(key, far)) >= 0) {
                const int at = __shfl_sync(full, ref, src);
                const float4* tp = s.tris + 3 * (size_t)at;
                const float4 q0 = ldg4(tp), q1 = ldg4(tp + 1), q2 = ldg4(tp + 2);
                const int k = __float_as_int(q0.w);
                if (mine && k != ex0 && (!SEG || k != ex1)) {
                    const float th = tri_hit(q0, q1, q2, o, d);
                    if (th > tmin && (th < t || (!any && th == t && k < id))) {
                        id = SEG ? at : k;
                        if (!any) t = th;
                    }
                }
                far = far_of();
            }
        }
        // segments: all are blocked (far is 0, where boxes around their starts begin too;
        // the same test in the other traces cost dense maps 1 to 2 %)
        if (SEG && far == 0u) break;
        // the nearest group, else the nearest set, else the next sets
        int src = take_nearest(key1, far);
        level = 0;
        rec = 32 * (next1 - r1 + src);
        if (src < 0) {
            key1 = 0x7f800000u;
            src = take_nearest(key2, far);
            level = src < 0 ? 2 : 1;
            rec = r1 + 32 * (next2 - r2 + src);
        }
    }
}

__device__ __forceinline__ void beam_trace(const DevScene& s, bool mine, bool any, f3 o, f3 d, int ex, float& t, int& id) {
    Beam b;
    b.x = ray_axis(mine, o.x, d.x);
    b.y = ray_axis(mine, o.y, d.y);
    b.z = ray_axis(mine, o.z, d.z);
    b.odd = b.x.open || b.y.open || b.z.open;
    beam_walk<false>(s, b, mine, any, o, d, ex, ex, t, id);
}

// Any occluder (any_hit) of the segments from o to e, d = (e - o) / |e - o|, for
// the lanes of `need`, called by all 32: those that start and end near the
// first one's ends as a beam, the others one by one. found: the occluder
// (index in s.tris), or RT_NO_REF. Without boxes for beams all one by one; layout
// 8: no occluder named either.
template <int LY>
__device__ __forceinline__ bool warp_segments(const DevScene& s, bool need, f3 o, f3 e, f3 d, float tmax, int ex0, int ex1,
                                              int& found) {
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    found = RT_NO_REF;
    TravCount cnt;
    if (LY == 8) return need && any_hit<false, 8>(s, nullptr, 0, o, d, tmax, ex0, ex1, cnt);
    unsigned todo = __ballot_sync(full, need);
    if (s.n_tris == 0 || !todo) return false;
    const float rho = s.pk_rho;
    const int lead = __ffs(todo) - 1;
    const float ox = o.x - __shfl_sync(full, o.x, lead), oy = o.y - __shfl_sync(full, o.y, lead),
                oz = o.z - __shfl_sync(full, o.z, lead);
    const float ex = e.x - __shfl_sync(full, e.x, lead), ey = e.y - __shfl_sync(full, e.y, lead),
                ez = e.z - __shfl_sync(full, e.z, lead);
    const bool in = need && (lane == lead || (fmax3(fabsf(ox), fabsf(oy), fabsf(oz)) <= rho &&
                                              fmax3(fabsf(ex), fabsf(ey), fabsf(ez)) <= rho));
    const unsigned m = __ballot_sync(full, in);
    const bool beam = s.pk && __popc(m) >= PK_MIN;
    if (beam) {
        Beam b;
        b.x = seg_axis(in, o.x, e.x);
        b.y = seg_axis(in, o.y, e.y);
        b.z = seg_axis(in, o.z, e.z);
        b.odd = b.x.open || b.y.open || b.z.open || b.x.shut || b.y.shut || b.z.shut;
        beam_walk<true>(s, b, in, true, o, d, ex0, ex1, tmax, found);
    }
    bool hit = in && beam && found >= 0;
    if (need && !(in && beam)) hit = any_hit_b<false, true, true>(s, nullptr, 0, o, d, tmax, ex0, ex1, cnt, &found);
    __syncwarp();
    return hit;
}

// A single ray through the binary hierarchy: closest_hit_b's tests and ties, for
// hits before t, or with `any` whether there is one (t is left). The next node is
// selected and not branched to: with a branch for each case (both children, one,
// none) the lanes went on apart until the last one's end in kernels of many
// registers, whatever they had in common (orientation gradient at 120 rays a
// triangle and depth 5, geometric mean over 21 cities: 1.5 times the time).
__device__ __forceinline__ int single_ray(const DevScene& s, bool any, f3 o, f3 d, int ex, float& t) {
    const f3 inv = safe_inv(d);
    const f3 oi = {o.x * inv.x, o.y * inv.y, o.z * inv.z};
    int stack[RT_STACK];
    int sp = 0, node = 0, best = -1;
    float tb = t;
    const float tmin = s.tmin;
    auto test = [&](const float4* tp) {
        const float4 r0 = ldg4(tp), r1 = ldg4(tp + 1), r2 = ldg4(tp + 2);
        const int id = __float_as_int(r0.w);
        if (id != ex) {
            const float th = tri_hit(r0, r1, r2, o, d);
            if (th > tmin && (th < tb || (th == tb && id < best))) {
                tb = th;
                best = id;
            }
        }
    };
#pragma unroll 1
    for (int k = 0; k < s.n_big; k++) test(s.big + 3 * k);
    const float4* onodes = octant_nodes(s, inv);
    const PairRay pr = pair_ray(inv, oi);
    const int no_top = 0x7fffffff;   // top: the child deferred last, the others in the stack
    int top = no_top;
    bool live = s.n_nodes > 0 && !(any && best >= 0);
    while (live) {
        float4 a, b, c, e;
        load_node<true>(onodes + 4 * (size_t)node, a, b, c, e);
        float tn0, tf0, tn1, tf1;
        box_pair(a, b, c, pr, tmin, tb, tn0, tf0, tn1, tf1);
        const int c0 = __float_as_int(e.x), c1 = __float_as_int(e.y);
        bool h0 = tn0 <= tf0, h1 = tn1 <= tf1;
        if (h0 && c0 < 0) {
            test(s.tris + 3 * (size_t)~c0);
            h0 = false;
        }
        if (h1 && c1 < 0) {
            test(s.tris + 3 * (size_t)~c1);
            h1 = false;
        }
        const bool first = tn0 <= tn1, both = h0 && h1, none = !h0 && !h1, empty = top == no_top;
        if (both && !empty) stack[sp++] = top;
        int below = no_top;
        if (none && empty && sp > 0) below = stack[--sp];
        node = both ? (first ? c0 : c1) : h0 ? c0 : h1 ? c1 : empty ? below : top;
        top = both ? (first ? c1 : c0) : none ? no_top : top;
        live = node != no_top && !(any && best >= 0);
    }
    if (!any) t = tb;
    return best;
}

// For the lanes of `need`, called by all 32: rays near one another are traced
// as beams, the others one by one. Closest hit before t, or any (see
// beam_trace); id -1 without one.
__device__ __forceinline__ void warp_trace(const DevScene& s, bool need, bool any, f3 o, f3 d, int ex, float& t,
                                           int& id) {
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    id = -1;
    const unsigned want = __ballot_sync(full, need);
    unsigned todo = want, rest = 0;
    if (s.n_tris == 0) return;
    // each ray's beam: the first ray of those not yet in one and what lies near it
    int mine = -1, beams = 0;
    while (todo && beams < PK_BEAMS) {
        const int lead = __ffs(todo) - 1;
        const float dx = d.x - __shfl_sync(full, d.x, lead), dy = d.y - __shfl_sync(full, d.y, lead),
                    dz = d.z - __shfl_sync(full, d.z, lead);
        const float ox = o.x - __shfl_sync(full, o.x, lead), oy = o.y - __shfl_sync(full, o.y, lead),
                    oz = o.z - __shfl_sync(full, o.z, lead);
        const bool in = ((todo >> lane) & 1u) && (lane == lead || (fmax3(fabsf(dx), fabsf(dy), fabsf(dz)) <= PK_DIR &&
                                                                   fmax3(fabsf(ox), fabsf(oy), fabsf(oz)) <= s.pk_rho));
        if (in) mine = beams;
        todo &= ~__ballot_sync(full, in);
        beams++;
    }
    const int least = todo || (beams > 1 && __popc(want) < PK_FEW) ? PK_MIN : 1;
    for (int n = 0; n < beams; n++) {
        const unsigned m = __ballot_sync(full, mine == n);
        if (__popc(m) < least) rest |= m;
        else beam_trace(s, mine == n, any, o, d, ex, t, id);
    }
    rest |= todo;
    if (rest) {   // for the warp: its set-up is not computed where all went as beams
        if ((rest >> lane) & 1u) id = single_ray(s, any, o, d, ex, t);
        __syncwarp();
    }
}
