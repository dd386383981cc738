// rt_scatter.cu -- first-order diffuse scattering (Sec. II-B lists diffuse
// reflections, i.e. scattering, among the features and leaves the model to
// the documentation). Reading used here: the effective-roughness model with
// a Lambertian pattern, the scattered wave depolarised.
//
// Each of the N Fibonacci-lattice rays of a transmitter carries the fraction
// |F_tx,q(d)|^2 / N of the transmitted power. Where it first hits a surface
// of scattering coefficient S, the fraction S^2 is re-radiated with the
// intensity pattern cos(theta_s)/pi on the side the ray came from; a
// receiver there, with the segment to it unoccluded, collects with the
// effective aperture lambda^2/(4 pi) |F_rx,p|^2, half of the depolarised
// wave per port:
//   g[pair][p][q] += S^2 (|F_tx,q(d)|^2/N) (cos theta_s/pi) (lambda^2/(4 pi r^2)) |F_rx,p(-k_s)|^2 / 2.
// The result is the incoherent scattered gain of every pair and port pair.
// A material with a directive pattern (exponent alpha >= 0) replaces
// cos(theta_s)/pi by ((1 + k_r . k_s)/2)^alpha / F_alpha, k_r the specular
// direction and F_alpha the lobe's integral over the hemisphere.
//
// The gain is quadratic in S, so its vector-Jacobian product with respect to
// the coefficients (Sec. II: gradients with respect to the parameters of the
// scattering functions) is, for material m,
//   dL/dS_m = 2 S_m sum over rays hitting m, receivers and ports of dL/dg * g / S_m^2,
// accumulated by the same kernel in its VJP mode.
#include "rt_field.cuh"
#include "rt_internal.h"

namespace {

struct ScatParams {
    DevScene s;
    const float* tx_pos;
    const float* tx_ypr;
    const float* rx_pos;
    const float* rx_ypr;
    const int32_t* rx_off;   // [n_tx+1] or null
    const float* scat;       // [n_mat] scattering coefficients
    const float4* dirs;      // [N] directions in the direction-coherent ray order, or null
    const int32_t* alpha;    // [n_mat] pattern exponent, -1 Lambertian; null: all Lambertian
    const float* up;         // VJP: upstream dL/dgain [n_pairs][nrp][ntp]
    float* grad;             // VJP: dL/dS [n_mat]
    int n_mat;
    bool grad_smem;          // VJP: per-block partial sums in shared memory
    int n_tx, n_rx;
    int rays, n_chunks;      // rays of a work unit, chunks of each transmitter's receivers
    long long N;
    DevAntenna txa, rxa;
    float w0;                // lambda^2 / (4 pi) / (2 pi N)
    float* gain;             // [n_pairs][nrp][ntp]
};

// F_alpha: the integral of ((1 + k_r . k_s)/2)^alpha over the hemisphere
// k_s . n > 0, with cos(theta_i) = k_r . n = ci. Binomial expansion in
// x = k_r . k_s; the hemisphere integral of x^j is 2 pi/(j+1) for even j
// (half the sphere's) and, for odd j = 2w+1,
//   2 pi/(j+1) ci sum_{u=0..w} C(2u, u) (sin^2(theta_i)/4)^u.
__device__ float directive_norm(int alpha, float ci) {
    const float q = 0.25f * fmaxf(0.0f, 1.0f - ci * ci);
    float tot = 0.0f, binom = 1.0f, part = 0.0f, term = 1.0f;
    int u = 0;
    for (int j = 0; j <= alpha; j++) {
        float I;
        if ((j & 1) == 0) {
            I = 2.0f * RT_PI_F / (float)(j + 1);
        } else {
            part += term;                                   // adds C(2u, u) q^u
            term *= q * 2.0f * (float)(2 * u + 1) / (float)(u + 1);
            u++;
            I = 2.0f * RT_PI_F / (float)(j + 1) * ci * part;
        }
        tot += binom * I;
        binom *= (float)(alpha - j) / (float)(j + 1);
    }
    return ldexpf(tot, -alpha);
}

// Rays of a work unit at most, warps of its block, entries of a warp's queue.
constexpr int SC_RAYS = 256, SC_WARPS = 4, SC_Q = 64;

// A unit's scattering hits, in shared memory.
struct ScatHits {
    float4 pt[SC_RAYS];    // hit point, hit triangle
    float4 nm[SC_RAYS];    // normal on the side the ray came from, material
    float4 tx[SC_RAYS];    // transmit power of both ports, coefficient S, pattern exponent
    float4 dir[SC_RAYS];   // specular direction, F_alpha / pi (directive patterns only)
};

// Any occluder between a queued (hit, receiver) pair, then its contribution:
// lane < take handles entry n + lane. Called by all 32 lanes; the occluder
// found last goes to ref0, the one before it to ref1.
template <bool VJP, int LY>
__device__ __forceinline__ void scatter_batch(const ScatParams& p, const ScatHits& h, const int* qr,
                                              const uint16_t* qh, int n, int take, int t, float* sgrad, int& ref0,
                                              int& ref1, TravCount& cnt) {
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    int r = -1, found = RT_NO_REF, m = 0;
    float w = 0.0f, sc = 0.0f, ptx[2] = {0.0f, 0.0f}, prx[2] = {0.0f, 0.0f};
    if (lane < take) {
        r = qr[n + lane];
        const int k = qh[n + lane];
        const float4 hp = h.pt[k], hn = h.nm[k], ht = h.tx[k];
        const f3 rx = mk(p.rx_pos[3 * r], p.rx_pos[3 * r + 1], p.rx_pos[3 * r + 2]);
        const f3 P = xyz(hp), v = rx - P;
        const float dist = sqrtf(dot(v, v));
        const f3 ks = v * (1.0f / dist);
        if (!any_hit_ref<LY>(p.s, P, ks, dist - p.s.tmin, __float_as_int(hp.w), -1, cnt, found)) {
            const float cs = dot(v, xyz(hn)) / dist;
            const int am = __float_as_int(ht.w);
            float pat = cs;
            if (am >= 0) {
                const float4 hd = h.dir[k];
                pat = powf(0.5f * (1.0f + dot(xyz(hd), ks)), (float)am) / hd.w;
            }
            m = __float_as_int(hn.w);
            sc = ht.z;
            w = (VJP ? 1.0f : sc * sc) * pat * p.w0 / (dist * dist);
            ptx[0] = ht.x;
            ptx[1] = ht.y;
            const Rot<float> Rr = rot_ypr(p.rx_ypr[3 * r], p.rx_ypr[3 * r + 1], p.rx_ypr[3 * r + 2]);
            for (int pp = 0; pp < p.rxa.n_ports; pp++) {
                const V3<float> f = antenna_vec<float>(p.rxa.kind, p.rxa.slant[pp], Rr, V3<float>{-ks.x, -ks.y, -ks.z});
                prx[pp] = f.x * f.x + f.y * f.y + f.z * f.z;
            }
        }
    }
    const unsigned fm = __ballot_sync(full, found != RT_NO_REF);
    const int last = fm ? __shfl_sync(full, found, 31 - __clz(fm)) : ref0;
    if (last != ref0) {
        ref1 = ref0;
        ref0 = last;
    }
    unsigned open = __ballot_sync(full, w != 0.0f);
    const long long pair = p.rx_off ? (long long)r : (long long)t * p.n_rx + r;
    float acc = 0.0f;
    if (VJP) {   // w is g / S^2 here
        if (w != 0.0f) {
            for (int pp = 0; pp < p.rxa.n_ports; pp++)
                for (int q = 0; q < p.txa.n_ports; q++)
                    acc += __ldg(p.up + (pair * p.rxa.n_ports + pp) * p.txa.n_ports + q) * w * prx[pp] * ptx[q];
            acc *= 2.0f * sc;
        }
    }
    // the entries are in receiver order, so the batch has few receivers (or,
    // for the VJP, materials): one sum over the warp and one atomic for each
    while (open) {
        const int g = __shfl_sync(full, VJP ? m : r, __ffs(open) - 1);
        const bool mine = w != 0.0f && (VJP ? m : r) == g;
        open &= ~__ballot_sync(full, mine);
        if (VJP) {
            float c = mine ? acc : 0.0f;
            for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(full, c, o);
            if (lane == 0 && c != 0.0f) atomicAdd((p.grad_smem ? sgrad : p.grad) + g, c);
            continue;
        }
        const long long gp = p.rx_off ? (long long)g : (long long)t * p.n_rx + g;
        for (int pp = 0; pp < p.rxa.n_ports; pp++)
            for (int q = 0; q < p.txa.n_ports; q++) {
                float c = mine ? w * prx[pp] * ptx[q] : 0.0f;
                for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(full, c, o);
                if (lane == 0 && c != 0.0f) atomicAdd(p.gain + (gp * p.rxa.n_ports + pp) * p.txa.n_ports + q, c);
            }
    }
    __syncwarp();
}

// Every (ray's first hit, receiver): a block takes up to SC_RAYS rays of one
// transmitter and a chunk of its receivers. The rays are traced first (in the
// direction-coherent order of the tracing kernels, so the hits of a block lie
// near each other) and the hits that scatter are packed in shared memory; then
// each warp takes one receiver at a time against all of them, a lane per hit.
// The last two occluders of pairs of this warp are tried first (ref_hit: a
// triangle instead of a traversal), and what they do not block is queued,
// across receivers, so that traversals run with full warps. VJP:
// the sum of dL/dg * g / S^2, times 2 S, goes to the hit's material (per block
// in shared memory first).
// Bound by the pairs no kept occluder answers and by the pairs' own
// arithmetic. 1e5 rays x 1000 receivers in the city, mean of six sites: 1.32
// ms, where a thread per (ray, chunk of receivers) with a traversal per pair
// took 3.83 ms. (One occluder kept instead of two: 7 % slower; the queued
// segments as beams: 4 % slower, they fan out over the receivers.)
template <bool VJP, int LY>
__global__ void __launch_bounds__(32 * SC_WARPS, 7) k_scatter(ScatParams p) {
    constexpr int W = SC_WARPS;
    extern __shared__ float sgrad[];
    __shared__ ScatHits h;
    __shared__ int q_rx[W][SC_Q];
    __shared__ uint16_t q_hit[W][SC_Q];
    __shared__ int n_hit;
    const unsigned full = 0xffffffffu, lt = lanemask_lt();
    const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
    if (VJP && p.grad_smem)
        for (int i = threadIdx.x; i < p.n_mat; i += blockDim.x) sgrad[i] = 0.0f;
    const long long batches = (p.N + p.rays - 1) / p.rays;
    const long long units = (long long)p.n_tx * batches * p.n_chunks;
    TravCount cnt;
    int ref0 = RT_NO_REF, ref1 = RT_NO_REF;   // the last two occluders of recent pairs
    for (long long u = blockIdx.x; u < units; u += gridDim.x) {
        const long long tb = div_ll(u, p.n_chunks);
        const int chunk = (int)(u - tb * p.n_chunks);
        const int t = (int)div_ll(tb, batches);
        const long long i0 = (tb - (long long)t * batches) * p.rays;
        // this chunk of the transmitter's receivers
        const int rb0 = p.rx_off ? p.rx_off[t] : 0, re0 = p.rx_off ? p.rx_off[t + 1] : p.n_rx;
        const int len = (re0 - rb0 + p.n_chunks - 1) / p.n_chunks;
        const int rb = min(re0, rb0 + chunk * len), re = min(re0, rb + len);
        if (rb >= re) continue;   // the same for the whole block
        __syncthreads();          // the last unit's hits are no longer read
        if (threadIdx.x == 0) n_hit = 0;
        __syncthreads();
        for (int k0 = 0; k0 < p.rays; k0 += 32 * W) {
            const long long i = i0 + k0 + threadIdx.x;
            const bool in = k0 + (int)threadIdx.x < p.rays && i < p.N;
            float sc = 0.0f, th = 0.0f;
            int hit = -1, m = 0;
            f3 d = mk(0, 0, 1);
            if (in) {
                const f3 o = mk(p.tx_pos[3 * t], p.tx_pos[3 * t + 1], p.tx_pos[3 * t + 2]);
                d = p.dirs ? xyz(__ldg(p.dirs + i)) : fib_dir(p.N, i);
                hit = closest_hit<false, LY>(p.s, nullptr, 0, o, d, -1, th, cnt);
                if (hit >= 0) {
                    m = __ldg(p.s.mat + hit);
                    sc = __ldg(p.scat + m);
                }
            }
            const bool keep = sc > 0.0f;   // S <= 0: no scattering
            const unsigned km = __ballot_sync(full, keep);
            int at = 0;
            if (lane == 0 && km) at = atomicAdd(&n_hit, __popc(km));
            at = __shfl_sync(full, at, 0) + __popc(km & lt);
            if (keep) {
                const f3 o = mk(p.tx_pos[3 * t], p.tx_pos[3 * t + 1], p.tx_pos[3 * t + 2]);
                f3 n = xyz(__ldg(p.s.planes + hit));
                if (dot(d, n) > 0.0f) n = n * -1.0f;   // the side the ray came from
                const f3 P = o + d * th;
                const int am = p.alpha ? __ldg(p.alpha + m) : -1;
                if (am >= 0) {
                    const float dn = dot(d, n);                 // < 0: n faces the incoming ray
                    const f3 kr = d - n * (2.0f * dn);
                    // pi / F_alpha replaces 1/pi in w0
                    h.dir[at] = make_float4(kr.x, kr.y, kr.z, directive_norm(am, -dn) / RT_PI_F);
                }
                const Rot<float> Rt = rot_ypr(p.tx_ypr[3 * t], p.tx_ypr[3 * t + 1], p.tx_ypr[3 * t + 2]);
                float ptx[2] = {0.0f, 0.0f};
                for (int q = 0; q < p.txa.n_ports; q++) {
                    const V3<float> f = antenna_vec<float>(p.txa.kind, p.txa.slant[q], Rt, V3<float>{d.x, d.y, d.z});
                    ptx[q] = f.x * f.x + f.y * f.y + f.z * f.z;
                }
                h.pt[at] = make_float4(P.x, P.y, P.z, __int_as_float(hit));
                h.nm[at] = make_float4(n.x, n.y, n.z, __int_as_float(m));
                h.tx[at] = make_float4(ptx[0], ptx[1], sc, __int_as_float(am));
            }
        }
        __syncthreads();
        const int nh = n_hit;
        int nq = 0;   // queued pairs (warp-uniform)
        // (receiver, 32 hits) in receiver order, an equal run of them for each warp
        const int nt = (nh + 31) / 32;
        const long long steps = (long long)(re - rb) * nt;
        const long long step0 = steps * wp / W, step1 = steps * (wp + 1) / W;
        const int r0 = nt ? (int)div_ll(step0, nt) : 0;
        int r = rb + r0, tile = (int)(step0 - (long long)r0 * nt);
        f3 rx = mk(0, 0, 0);
        for (long long step = step0; step < step1; step++) {
            if (step == step0 || tile == 0) rx = mk(p.rx_pos[3 * r], p.rx_pos[3 * r + 1], p.rx_pos[3 * r + 2]);
            const int k = 32 * tile + lane;
            bool open = false;
            if (k < nh) {
                const float4 hp = h.pt[k];
                const f3 P = xyz(hp), v = rx - P;
                const float dist = sqrtf(dot(v, v));
                const f3 ks = v * (1.0f / dist);
                const int hit = __float_as_int(hp.w);
                if (dot(v, xyz(h.nm[k])) / dist > 0.0f)
                    open = !ref_hit(p.s, ref0, P, ks, dist - p.s.tmin, hit, -1) &&
                           !ref_hit(p.s, ref1, P, ks, dist - p.s.tmin, hit, -1);
            }
            const unsigned om = __ballot_sync(full, open);
            if (open) {
                q_rx[wp][nq + __popc(om & lt)] = r;
                q_hit[wp][nq + __popc(om & lt)] = (uint16_t)k;
            }
            nq += __popc(om);
            __syncwarp();
            // 32 of them, or what is left at the end (one call: a second copy of the
            // traversal costs a cold instruction cache 2 to 4 us)
            while (nq >= 32 || (step + 1 == step1 && nq > 0)) {
                const int take = min(nq, 32);
                nq -= take;
                scatter_batch<VJP, LY>(p, h, q_rx[wp], q_hit[wp], nq, take, t, sgrad, ref0, ref1, cnt);
            }
            if (++tile == nt) {
                tile = 0;
                r++;
            }
        }
    }
    if (VJP && p.grad_smem) {
        __syncthreads();
        for (int i = threadIdx.x; i < p.n_mat; i += blockDim.x)
            if (sgrad[i] != 0.0f) atomicAdd(p.grad + i, sgrad[i]);
    }
}


// The same for few receivers, where the first hits weigh more than the pairs:
// a thread a ray, which keeps its hit in registers and takes every receiver of
// its transmitter in turn; the warp's lanes visit the same receiver together and
// add up their contributions with one atomic when they share the transmitter.
// Nothing is packed or queued, so one chain of first hit, segment and sum bounds
// it: 1e5 rays x 1 receiver 60 us, k_scatter 63. VJP: each ray's sum of
// dL/dg * g / S^2 goes, times 2 S, to its material.
template <bool VJP, int LY>
__global__ void __launch_bounds__(128) k_scatter_few(ScatParams p) {
    extern __shared__ float sgrad[];
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    if (VJP && p.grad_smem) {
        for (int i = threadIdx.x; i < p.n_mat; i += blockDim.x) sgrad[i] = 0.0f;
        __syncthreads();
    }
    const long long total = (long long)p.n_tx * p.N, step = (long long)gridDim.x * blockDim.x;
    TravCount cnt;
    for (long long b = (long long)blockIdx.x * blockDim.x + threadIdx.x - lane; b < total; b += step) {
        const bool in = b + lane < total;
        const long long slot = in ? b + lane : total - 1;
        const int t = (int)div_ll(slot, p.N);
        const long long i = slot - (long long)t * p.N;
        const bool uniform = __all_sync(full, t == __shfl_sync(full, t, 0));
        float sc = 0.0f, acc = 0.0f, fa = 1.0f, ptx[2] = {0.0f, 0.0f};
        f3 P = mk(0, 0, 0), n = mk(0, 0, 1), kr = mk(0, 0, 1);
        int hit = -1, m = 0, am = -1;
        if (in) {
            const f3 o = mk(p.tx_pos[3 * t], p.tx_pos[3 * t + 1], p.tx_pos[3 * t + 2]);
            const f3 d = p.dirs ? xyz(__ldg(p.dirs + i)) : fib_dir(p.N, i);
            float th;
            hit = closest_hit<false, LY>(p.s, nullptr, 0, o, d, -1, th, cnt);
            if (hit >= 0) {
                m = __ldg(p.s.mat + hit);
                sc = fmaxf(__ldg(p.scat + m), 0.0f);   // S <= 0: no scattering
                n = xyz(__ldg(p.s.planes + hit));
                if (dot(d, n) > 0.0f) n = n * -1.0f;   // the side the ray came from
                P = o + d * th;
                am = p.alpha ? __ldg(p.alpha + m) : -1;
                if (am >= 0) {
                    const float dn = dot(d, n);                 // < 0: n faces the incoming ray
                    kr = d - n * (2.0f * dn);
                    fa = directive_norm(am, -dn) / RT_PI_F;     // pi / F_alpha replaces 1/pi in w0
                }
                const Rot<float> Rt = rot_ypr(p.tx_ypr[3 * t], p.tx_ypr[3 * t + 1], p.tx_ypr[3 * t + 2]);
                for (int q = 0; q < p.txa.n_ports; q++) {
                    const V3<float> f = antenna_vec<float>(p.txa.kind, p.txa.slant[q], Rt, V3<float>{d.x, d.y, d.z});
                    ptx[q] = f.x * f.x + f.y * f.y + f.z * f.z;
                }
            }
        }
        if (!__any_sync(full, sc > 0.0f)) continue;
        const int rb = p.rx_off ? p.rx_off[t] : 0, nr = (p.rx_off ? p.rx_off[t + 1] : p.n_rx) - rb;
        const int nr_max = __reduce_max_sync(full, (unsigned)nr);
        for (int k = 0; k < nr_max; k++) {
            float w = 0.0f, prx[2] = {0.0f, 0.0f};
            const int r = rb + k;
            if (sc > 0.0f && k < nr) {
                const f3 rx = mk(p.rx_pos[3 * r], p.rx_pos[3 * r + 1], p.rx_pos[3 * r + 2]);
                const f3 v = rx - P;
                const float dist = sqrtf(dot(v, v));
                const float cs = dot(v, n) / dist;
                const f3 ks = v * (1.0f / dist);
                if (cs > 0.0f && !any_hit<false, LY>(p.s, nullptr, 0, P, ks, dist - p.s.tmin, hit, -1, cnt)) {
                    const float pat = am < 0 ? cs : powf(0.5f * (1.0f + dot(kr, ks)), (float)am) / fa;
                    w = (VJP ? 1.0f : sc * sc) * pat * p.w0 / (dist * dist);
                    const Rot<float> Rr = rot_ypr(p.rx_ypr[3 * r], p.rx_ypr[3 * r + 1], p.rx_ypr[3 * r + 2]);
                    for (int pp = 0; pp < p.rxa.n_ports; pp++) {
                        const V3<float> f = antenna_vec<float>(p.rxa.kind, p.rxa.slant[pp], Rr, V3<float>{-ks.x, -ks.y, -ks.z});
                        prx[pp] = f.x * f.x + f.y * f.y + f.z * f.z;
                    }
                }
            }
            const long long pair = p.rx_off ? (long long)r : (long long)t * p.n_rx + r;
            if (VJP) {   // w is g / S^2 here
                if (w != 0.0f)
                    for (int pp = 0; pp < p.rxa.n_ports; pp++)
                        for (int q = 0; q < p.txa.n_ports; q++)
                            acc += __ldg(p.up + (pair * p.rxa.n_ports + pp) * p.txa.n_ports + q) * w * prx[pp] * ptx[q];
                continue;
            }
            for (int pp = 0; pp < p.rxa.n_ports; pp++)
                for (int q = 0; q < p.txa.n_ports; q++) {
                    float c = w * prx[pp] * ptx[q];
                    if (uniform)
                        for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(full, c, o);
                    if (c != 0.0f && (!uniform || lane == 0))
                        atomicAdd(p.gain + (pair * p.rxa.n_ports + pp) * p.txa.n_ports + q, c);
                }
        }
        if (VJP && acc != 0.0f) atomicAdd((p.grad_smem ? sgrad : p.grad) + m, 2.0f * sc * acc);
    }
    if (VJP && p.grad_smem) {
        __syncthreads();
        for (int i = threadIdx.x; i < p.n_mat; i += blockDim.x)
            if (sgrad[i] != 0.0f) atomicAdd(p.grad + i, sgrad[i]);
    }
}

}  // namespace

// gain != null: forward; else up / grad: the VJP with respect to S.
int scattering_impl(rt_ctx* ctx, int64_t N, float* gain, const float* up, float* grad) {
    const int64_t n_pairs = ctx->rx_sets ? (int64_t)ctx->rx_off[ctx->n_tx] : (int64_t)ctx->n_tx * ctx->n_rx;
    const int np = ctx->tx_ant.n_ports * ctx->rx_ant.n_ports;
    const bool vjp = gain == nullptr;
    if (vjp) RT_TRY(cudaMemsetAsync(grad, 0, sizeof(float) * (size_t)ctx->n_mat, ctx->stream));
    else RT_TRY(cudaMemsetAsync(gain, 0, sizeof(float) * (size_t)n_pairs * np, ctx->stream));
    if (N == 0 || ctx->n_tris == 0 || !ctx->scat_set) return RT_OK;
    ScatParams p;
    p.s = dev_scene(ctx);
    p.tx_pos = bp<float>(ctx->tx_pos);
    p.tx_ypr = bp<float>(ctx->tx_ypr);
    p.rx_pos = bp<float>(ctx->rx_pos);
    p.rx_ypr = bp<float>(ctx->rx_ypr);
    p.rx_off = ctx->rx_sets ? bp<int32_t>(ctx->rx_off_d) : nullptr;
    p.scat = bp<float>(ctx->scat);
    {
        int e = ensure_perm(ctx, N);
        if (e) return e;
    }
    p.dirs = ctx->dirs_ok ? bp<float4>(ctx->dirs) : nullptr;
    p.alpha = ctx->scat_alpha_set ? bp<int32_t>(ctx->scat_alpha) : nullptr;
    p.up = up;
    p.grad = grad;
    p.n_mat = ctx->n_mat;
    p.grad_smem = vjp && ctx->n_mat <= 4096;
    p.n_tx = ctx->n_tx;
    p.n_rx = ctx->n_rx;
    p.N = N;
    p.txa = ctx->tx_ant;
    p.rxa = ctx->rx_ant;
    const double lam = RT_C0_D / ctx->fc;
    p.w0 = (float)(lam * lam / (4.0 * RT_PI_D) / (2.0 * RT_PI_D * (double)N));
    p.gain = gain;
    // work units: up to SC_RAYS rays against a chunk of the receivers. The rays
    // of a unit share its occluders and its chunk's receivers amortise their
    // first hits, so both shrink only while the units would not fill the chip:
    // to 128 rays and 32 receivers for 24 units per SM (city, 1000 receivers, mean
    // of six sites: 16 units 1.41 ms, 24 1.32, 32 1.35, 48 1.44: first hits against
    // the last wave's gap), to 32 rays and 4 receivers for one wave (2 x 1464 rays
    // x 127 receivers: 0.10 ms; one thread per ray and 64 receivers took 1.22 ms).
    int nr_max = ctx->n_rx;
    if (ctx->rx_sets) {
        nr_max = 0;
        for (int t = 0; t < ctx->n_tx; t++) nr_max = std::max(nr_max, ctx->rx_off[t + 1] - ctx->rx_off[t]);
    }
    const long long sms = ctx->num_sms, wave = 7 * sms;
    auto n_units = [&](int rays, long long chunks) { return (long long)ctx->n_tx * ((N + rays - 1) / rays) * chunks; };
    auto chunks_for = [&](int rays, long long units, int receivers) {
        return std::max<long long>(1, std::min<long long>(nr_max / receivers, (units + n_units(rays, 1) - 1) / n_units(rays, 1)));
    };
    // a thread a ray (k_scatter_few): for one receiver, and up to eight while units
    // of 128 rays would make one to four waves, whose last one is partly empty
    // (3e5 rays x 2 receivers: 82 us, k_scatter 93; x 8: 143 both; but 1e5 x 2: 72
    // and 68, 1e6 x 2: 153 and 152, and 1e5 x 8: 107 and 87)
    const long long coarse = n_units(128, 1);
    const bool few = nr_max == 1 || (nr_max <= 8 && coarse > wave && coarse < 4 * wave);
    p.rays = SC_RAYS;
    if (n_units(p.rays, std::max(1, nr_max / 32)) < 24 * sms) p.rays = 128;
    p.n_chunks = (int)chunks_for(p.rays, 24 * sms, 32);
    if (n_units(p.rays, p.n_chunks) < wave) p.n_chunks = (int)chunks_for(p.rays, wave, 4);
    while (p.rays > 32 && n_units(p.rays, p.n_chunks) < wave) p.rays /= 2;
    const long long units = few ? std::min<long long>(((long long)ctx->n_tx * N + 127) / 128, 16 * sms)
                                : std::min<long long>(n_units(p.rays, p.n_chunks), 1ll << 30);
    const size_t smem = p.grad_smem ? sizeof(float) * ctx->n_mat : 0;
    const bool wide = wide_layout(ctx);
    auto kern = few ? (vjp ? (wide ? k_scatter_few<true, 8> : k_scatter_few<true, 2>)
                           : (wide ? k_scatter_few<false, 8> : k_scatter_few<false, 2>))
                    : (vjp ? (wide ? k_scatter<true, 8> : k_scatter<true, 2>)
                           : (wide ? k_scatter<false, 8> : k_scatter<false, 2>));
    prof_begin(ctx, vjp ? "k_scatter_vjp" : "k_scatter");
    kern<<<(unsigned)units, 32 * SC_WARPS, smem, ctx->stream>>>(p);
    prof_end(ctx);
    RT_TRY(cudaGetLastError());
    return RT_OK;
}
