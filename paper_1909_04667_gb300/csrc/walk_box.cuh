// Short-range walk of a periodic TreePM box (paper Sec. 3.1, 3.4).
//
// A warp serves 32 key-consecutive targets, one per lane.  The cutoff sphere
// (2.8 mean spacings on the 128^3 box) is about as wide as the group, so a
// lock-step walk visits the union of 32 spheres: 626 nodes and 1000 leaf
// particles, of which most lanes need few.  Candidate nodes therefore come
// from a stack 32 at a time, one per LANE, and are first held against the
// group's bounding box: nodes beyond the cutoff for all targets are dropped,
// for the others the bounds say whether every target opens them, or every
// target that is not beyond the cutoff, or neither.  Only what is left is
// looked at target by target (the node's record handed round the warp): the
// distance to the cube, or the whole decision, in the lane walk's FP32
// operations, so that the decisions are the same bits.  An opened leaf's
// particles are held against the box in the same way, a particle per lane, and
// those in reach taken two at a time through the two-wide instructions.
// Bound by instruction issue (57 thousand warp instructions for 32 targets, the
// lane walk 71 thousand): 128^3 box, relative criterion, 4.68 -> 3.7 ms; 40^3
// box, theta = 0.5, 0.59 -> 0.53 ms; a Zel'dovich box of 128^3 with 98
// interactions a particle, cold caches, 5.18 -> 4.67 ms (65 thousand
// instructions).  Images looked up per node instead of per target where one
// serves the whole group: 6.15 -> 5.4 ms a step.
//
// Small boxes leave the chip idle behind 32-target warps (40^3: 2000 of them,
// four to six thousand fit).  Then `split` warps of a block share a chunk: all
// descend to the cells of side split_side (the largest not above the cutoff),
// each goes on into its share of those, dealt by node index, and the first
// alone takes what lies above (40^3 box with the spectral gradient, a step:
// 0.95 -> 0.76 ms).
//
// Leaves of a particle or two (more nodes than half the particles) leave little
// to hold against the box: a lane of the candidates, and a turn of the warp,
// for each.  Calls that fill the chip then keep the lane walk (box_rule): steps
// of its walk and of this one with leaf bucket 4, relative criterion, 56^3 (0.91
// nodes a particle) 903 / 981 us, 72^3 (0.82) 2247 / 2416, 120^3 (1.03) 7124 /
// 8188; theta = 0.5 64^3 (1.06) 1478 / 1343, 90^3 (0.63) 3271 / 3176, 110^3
// (0.86) 3970 / 4135, 120^3 5948 / 6261.  With four warps a group this walk is
// ahead all the same (40^3, bucket 4, relative 838 / 578).
constexpr int kBoxWarps = 4;

inline int box_split(int64_t groups, int num_sms) {
    // warps per chunk: four while they fit the chip about once, two up to twice
    // (steps with 1 / 2 / 4: 40^3 0.98 / 0.82 / 0.78 ms, 52^3 0.84 / 0.82 / 0.85,
    // 64^3 2.16 / 2.07 / 2.04, 80^3 2.61 / 2.66 / 2.82)
    return groups <= 24 * (int64_t)num_sms ? 4 : groups <= 64 * (int64_t)num_sms ? 2 : 1;
}

inline bool box_rule(const System *s, int64_t n_act, bool relative, int num_sms) {
    const int64_t groups = (n_act + 31) / 32;
    return 2 * s->nnodes <= s->n || groups <= (relative ? 24 : 200) * (int64_t)num_sms;
}

constexpr int kBoxStack = 384;  // child ranges, as in the walk with two targets per warp
constexpr int kBoxSafe = kBoxStack - 64;

struct BoxShared {
    uint2 stack[kBoxStack];    // (first child, targets that need the children)
    uint8_t count[kBoxStack];  // children
    // the step's nodes: centre offset from the frame and side; box offset to
    // the nearest image and the targets that need (later: open) the node;
    // centre of mass and mass
    float4 d[32], c[32], o[32];
};

template <bool RELATIVE>
__global__ void __launch_bounds__(kBoxWarps * 32, 7)
    k_walk_box(TreeView T, const uint32_t *__restrict__ sidx, const uint32_t *__restrict__ slot,
               const float *__restrict__ a_old, int64_t n_act, int split, float split_side, WalkConsts k,
               float *__restrict__ acc, float *__restrict__ pot, uint32_t *__restrict__ nint, int *__restrict__ err) {
    __shared__ BoxShared shared[kBoxWarps];
    const int warp = threadIdx.x >> 5;
    BoxShared &sh = shared[warp];
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const uint32_t part = (uint32_t)(warp % split);  // which of the chunk's warps
    const unsigned lt_mask = (1u << lane) - 1u;
    const int64_t g0 = ((int64_t)blockIdx.x * kBoxWarps + warp) / split * 32;
    if (g0 >= n_act)
        return;  // whole warp
    const int64_t gi = g0 + lane;
    const bool valid = gi < n_act;
    const uint32_t s = sidx ? sidx[valid ? gi : g0] : (uint32_t)(valid ? gi : g0);
    const uint32_t j = T.perm[s];
    const uint32_t out = slot ? slot[valid ? gi : g0] : j;

    // group frame: the smallest key cell holding the group's first and last particle
    const uint64_t kk = T.key[s];
    const uint64_t kf = __shfl_sync(FULL, kk, 0), kx = kf ^ __shfl_sync(FULL, kk, (int)min((int64_t)31, n_act - 1 - g0));
    const int glevel = kx ? min((__clzll(kx) - 1) / 3, kMaxLevel) : kMaxLevel;
    const uint64_t gpre = kf >> (3 * (kMaxLevel - glevel));
    const double ghalf = ldexp(T.L0, -(glevel + 1));
    const double gcx_d = (double)(2 * (uint64_t)compact3w(gpre) + 1) * ghalf;
    const double gcy_d = (double)(2 * (uint64_t)compact3w(gpre >> 1) + 1) * ghalf;
    const double gcz_d = (double)(2 * (uint64_t)compact3w(gpre >> 2) + 1) * ghalf;
    const float gcx = (float)gcx_d, gcy = (float)gcy_d, gcz = (float)gcz_d;
    const float x = (float)(T.pos[3 * (size_t)j] - (T.x0 + gcx_d)), y = (float)(T.pos[3 * (size_t)j + 1] - (T.y0 + gcy_d)),
                z = (float)(T.pos[3 * (size_t)j + 2] - (T.z0 + gcz_d));
    float thr = k.thr_const;
    if (RELATIVE)
        thr = valid ? k.alpha_over_G * fabsf(a_old[out]) : 0.0f;

    // bounding box (middle and half size) and largest threshold
    const float inf = __int_as_float(0x7f800000);
    float lox = valid ? x : inf, loy = valid ? y : inf, loz = valid ? z : inf;
    float hix = valid ? x : -inf, hiy = valid ? y : -inf, hiz = valid ? z : -inf, tmax = thr;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        lox = fminf(lox, __shfl_xor_sync(FULL, lox, o));
        loy = fminf(loy, __shfl_xor_sync(FULL, loy, o));
        loz = fminf(loz, __shfl_xor_sync(FULL, loz, o));
        hix = fmaxf(hix, __shfl_xor_sync(FULL, hix, o));
        hiy = fmaxf(hiy, __shfl_xor_sync(FULL, hiy, o));
        hiz = fmaxf(hiz, __shfl_xor_sync(FULL, hiz, o));
        if (RELATIVE)
            tmax = fmaxf(tmax, __shfl_xor_sync(FULL, tmax, o));
    }
    const float bcx = 0.5f * (lox + hix), bcy = 0.5f * (loy + hiy), bcz = 0.5f * (loz + hiz);
    // half sizes with a margin for the rounding of the middle
    const float pad = 2e-6f * k.box;
    const float bhx = 0.5f * (hix - lox) + pad, bhy = 0.5f * (hiy - loy) + pad, bhz = 0.5f * (hiz - loz) + pad;
    const float ext = fmaxf(fmaxf(fmaxf(-lox, hix), fmaxf(-loy, hiy)), fmaxf(-loz, hiz));
    // a group wider than an eighth of the box may see several images of a node:
    // no bounds, every target looks for itself
    const bool wide = ext > 0.125f * k.box;
    const float rcut = sqrtf(k.rcut2), reach2 = (rcut * 1.0001f + pad) * (rcut * 1.0001f + pad);

    PairSums ps;
    ps.x = ps.y = ps.z = ps.p = make_float2(0.f, 0.f);
    float ax = 0.f, ay = 0.f, az = 0.f, ph = 0.f;
    uint32_t cnt = 0;
    const unsigned valid_mask = __ballot_sync(FULL, valid);
    if (lane == 0) {
        sh.stack[0] = make_uint2(0u, valid_mask);  // the root, breadth-first index 0
        sh.count[0] = 1;
    }
    __syncwarp();
    int sn = 1;
    while (sn > 0) {
        // ---- up to 32 nodes from the top child ranges
        const int cap = sn > kBoxSafe ? 1 : 32;
        const int idx = sn - 1 - lane;
        const uint2 R = idx >= 0 ? sh.stack[idx] : make_uint2(0u, 0u);
        const int c = idx >= 0 ? (int)sh.count[idx] : 0;
        int total;
        const int excl = warp_exclusive(c, total);
        const bool some = c > 0 && excl < cap;
        const bool whole = some && excl + c <= cap;
        const unsigned starts = __reduce_or_sync(FULL, some ? 1u << excl : 0u);
        const int r = __popc(starts & (0xffffffffu >> (31 - lane))) - 1;
        const uint32_t node = __shfl_sync(FULL, R.x, r) + (uint32_t)(lane - __shfl_sync(FULL, excl, r));
        const unsigned need = __shfl_sync(FULL, R.y, r);
        sn -= __popc(__ballot_sync(FULL, whole));
        if (some && !whole) {  // the partly taken range stays on top
            sh.stack[idx].x = R.x + (uint32_t)(cap - excl);
            sh.count[idx] = (uint8_t)(c - (cap - excl));
        }
        __syncwarp();
        // ---- the lane's node against the group's bounding box
        enum { kDrop, kOpenAll, kOpenNear, kLook };
        int cls = kDrop;
        float4 C = make_float4(0.f, 0.f, 0.f, 0.f), O = C;
        int4 Lk = make_int4(0, 0, 0, 0);
        float dx = 0.f, dy = 0.f, dz = 0.f, cx = 0.f, cy = 0.f, cz = 0.f;
        bool general = false;  // images differ between targets, or between a target and the node's parts
        if (lane < min(total, cap)) {
            C = __ldg(&T.bcen[node]);
            O = __ldg(&T.bcom[node]);
            Lk = __ldg(&T.blink[node]);
            dx = C.x - gcx, dy = C.y - gcy, dz = C.z - gcz;  // exact
            // the box offset that brings every target of the group to its
            // nearest image of the node (0 or one box side)
            cx = k.box * rintf(dx * k.boxinv), cy = k.box * rintf(dy * k.boxinv), cz = k.box * rintf(dz * k.boxinv);
            const float wx = dx - cx, wy = dy - cy, wz = dz - cz;
            const float L = C.w;
            general = wide || L > k.bigL || fmaxf(fabsf(wx), fmaxf(fabsf(wy), fabsf(wz))) + ext > 0.4999f * k.box;
            cls = kLook;
            const float up = 1.0f + 1e-5f, dn = 1.0f - 1e-5f;
            // nearest and farthest |target - node centre| per axis
            const float ux = fabsf(bcx - wx), uy = fabsf(bcy - wy), uz = fabsf(bcz - wz);
            const float nx = fmaxf(ux - bhx, 0.0f), ny = fmaxf(uy - bhy, 0.0f), nz = fmaxf(uz - bhz, 0.0f);
            const float fx = ux + bhx, fy = uy + bhy, fz = uz + bhz;
            const float hl = 0.5f * L;
            const float ex = fmaxf(nx - hl, 0.0f), ey = fmaxf(ny - hl, 0.0f), ez = fmaxf(nz - hl, 0.0f);
            if (!(wide || L > k.bigL) && fmaf(ex, ex, fmaf(ey, ey, ez * ez)) > reach2) {
                cls = kDrop;
            } else if (L == split_side && node % (uint32_t)split != part) {
                cls = kDrop;  // another warp's
            } else if (!general) {
                const float hx = fmaxf(fx - hl, 0.0f), hy = fmaxf(fy - hl, 0.0f), hz = fmaxf(fz - hl, 0.0f);
                const bool none_far = fmaf(hx, hx, fmaf(hy, hy, hz * hz)) <= k.rcut2 * dn;
                const bool guard_all = k.box_guard && fmaxf(fx, fmaxf(fy, fz)) <= 0.6f * L * dn;
                // farthest target from the centre of mass: inside the box, and
                // -- of those that are not beyond the cutoff -- inside the
                // cutoff and the cube's diagonal
                const float mx = fabsf(bcx - (wx + O.x)) + bhx, my = fabsf(bcy - (wy + O.y)) + bhy,
                            mz = fabsf(bcz - (wz + O.z)) + bhz;
                const float far2 = fmaf(mx, mx, fmaf(my, my, mz * mz));
                const float lim = rcut * 1.0001f + pad + 1.7321f * L;
                const float d2 = fminf(far2, lim * lim);
                const float q = RELATIVE ? O.w * L * L : L * L;
                const bool open_near = q > (RELATIVE ? tmax * d2 * d2 : k.thr_const * d2) * up;
                if (guard_all || open_near)
                    cls = none_far ? kOpenAll : kOpenNear;
            }
        }
        unsigned om = cls == kOpenAll ? need : 0u;  // targets that open the lane's node
        sh.d[lane] = make_float4(dx, dy, dz, C.w);
        sh.c[lane] = make_float4(cx, cy, cz, __uint_as_float(need));
        sh.o[lane] = O;
        const unsigned gen = __ballot_sync(FULL, general);
        const unsigned look = __ballot_sync(FULL, cls == kLook);
        __syncwarp();
        // ---- target by target: the lane's target against node `from`; GEN: the
        // node's image is the target's own matter
        auto offset = [&](auto general_image, float4 D, float4 S, float &px, float &py, float &pz) {
            px = x - D.x, py = y - D.y, pz = z - D.z;
            if constexpr (decltype(general_image)::value) {
                px = wrap_min_image(px, k);
                py = wrap_min_image(py, k);
                pz = wrap_min_image(pz, k);
            } else {
                px += S.x;
                py += S.y;
                pz += S.z;
            }
        };
        auto targets = [&](auto general_image, unsigned nodes) {
            for (unsigned todo = nodes; todo; todo &= todo - 1u) {
                const int from = __ffs(todo) - 1;
                const float4 D = sh.d[from], S = sh.c[from];
                const float L = D.w;
                float px, py, pz;
                offset(general_image, D, S, px, py, pz);
                const float ex = fmaxf(fabsf(px) - 0.5f * L, 0.0f), ey = fmaxf(fabsf(py) - 0.5f * L, 0.0f),
                            ez = fmaxf(fabsf(pz) - 0.5f * L, 0.0f);
                const bool in = ((__float_as_uint(S.w) >> lane) & 1u) &&
                                !(fmaf(ex, ex, fmaf(ey, ey, ez * ez)) > k.rcut2);
                bool open = in;
                if ((look >> from) & 1u) {
                    const float4 Q = sh.o[from];
                    float rx = Q.x - px, ry = Q.y - py, rz = Q.z - pz;  // target -> centre of mass
                    if constexpr (decltype(general_image)::value) {
                        if (L > k.bigL) {
                            rx = wrap_min_image(rx, k);
                            ry = wrap_min_image(ry, k);
                            rz = wrap_min_image(rz, k);
                        }
                    }
                    const float r2 = fmaf(rx, rx, fmaf(ry, ry, rz * rz));
                    const float gl = k.box_guard ? 0.6f * L : -1.0f;
                    const bool guard = fmaxf(fabsf(px), fmaxf(fabsf(py), fabsf(pz))) <= gl;
                    const bool crit = RELATIVE ? Q.w * L * L > thr * r2 * r2 : L * L > thr * r2;
                    open = in && (guard || crit);
                    const bool accept = in && !open && (part == 0u || L <= split_side);
                    if (__any_sync(FULL, accept)) {
                        cnt += accept ? 1u : 0u;
                        if (__any_sync(FULL, accept && r2 < k.h2)) {
                            if (accept)
                                pair_term<true>(rx, ry, rz, r2, Q.w, k, ax, ay, az, ph);
                        } else {
                            const float ri = rsqrtf(fmaxf(r2, k.h2));
                            float gs, gp;
                            short_range_factors(r2 * ri, k.inv2rs, gs, gp);
                            const float mr = (accept ? Q.w : 0.0f) * ri, f = mr * ri * ri * gs;
                            ax = fmaf(f, rx, ax);
                            ay = fmaf(f, ry, ay);
                            az = fmaf(f, rz, az);
                            ph = fmaf(-mr, gp, ph);
                        }
                    }
                }
                const unsigned b = __ballot_sync(FULL, open);
                if (lane == from)
                    om = b;
            }
        };
        const unsigned left = __ballot_sync(FULL, cls >= kOpenNear);
        targets(std::true_type{}, left & gen);
        targets(std::false_type{}, left & ~gen);
        // ---- children of opened nodes to the stack
        const bool push = om != 0u && Lk.y != 0;
        const unsigned bp = __ballot_sync(FULL, push);
        if (push) {
            const int at = sn + __popc(bp & lt_mask);
            if (at < kBoxStack) {
                sh.stack[at] = make_uint2((uint32_t)Lk.x, om);
                sh.count[at] = (uint8_t)Lk.y;
            } else {
                atomicOr(err, 2);
            }
        }
        sn = min(sn + __popc(bp), kBoxStack);
        // ---- opened leaves: their particles against the box, a particle per
        // lane, then those in reach two at a time, a target per lane
        auto leaves = [&](auto general_image, unsigned nodes) {
            constexpr bool GEN = decltype(general_image)::value;
            for (unsigned todo = nodes; todo; todo &= todo - 1u) {
                const int from = __ffs(todo) - 1;
                const float4 D = sh.d[from], S = sh.c[from];
                const bool mine = (__shfl_sync(FULL, om, from) >> lane) & 1u;
                const int j0 = __shfl_sync(FULL, Lk.z, from), j1 = j0 + __shfl_sync(FULL, Lk.w, from);
                float px, py, pz;
                offset(general_image, D, S, px, py, pz);
                const float ux = D.x - S.x - bcx, uy = D.y - S.y - bcy, uz = D.z - S.z - bcz;
                for (int jb = j0; jb < j1; jb += 32) {
                    bool near = jb + lane < j1;
                    if (near && !GEN) {
                        const float4 P = __ldg(&T.spart[jb + lane]);
                        const float ex = fmaxf(fabsf(ux + P.x) - bhx, 0.0f), ey = fmaxf(fabsf(uy + P.y) - bhy, 0.0f),
                                    ez = fmaxf(fabsf(uz + P.z) - bhz, 0.0f);
                        near = fmaf(ex, ex, fmaf(ey, ey, ez * ez)) <= reach2;
                    }
                    for (unsigned rest = __ballot_sync(FULL, near); rest;) {
                        const int ja = jb + __ffs(rest) - 1;
                        rest &= rest - 1u;
                        const bool two = rest != 0u;
                        const int jc = two ? jb + __ffs(rest) - 1 : ja;
                        rest &= rest - 1u;
                        const float4 A = __ldg(&T.spart[ja]), B = __ldg(&T.spart[jc]);
                        float2 qx = __fadd2_rn(make_float2(px, px), make_float2(-A.x, -B.x)),
                               qy = __fadd2_rn(make_float2(py, py), make_float2(-A.y, -B.y)),
                               qz = __fadd2_rn(make_float2(pz, pz), make_float2(-A.z, -B.z));
                        if (GEN && D.w > k.bigL) {
                            qx = make_float2(wrap_min_image(qx.x, k), wrap_min_image(qx.y, k));
                            qy = make_float2(wrap_min_image(qy.x, k), wrap_min_image(qy.y, k));
                            qz = make_float2(wrap_min_image(qz.x, k), wrap_min_image(qz.y, k));
                        }
                        const float2 q2 = __ffma2_rn(qx, qx, __ffma2_rn(qy, qy, __fmul2_rn(qz, qz)));
                        const bool a = mine && (uint32_t)ja != s && q2.x <= k.rcut2;
                        const bool b = mine && two && (uint32_t)jc != s && q2.y <= k.rcut2;
                        if (!__any_sync(FULL, a || b))
                            continue;
                        cnt += (a ? 1u : 0u) + (b ? 1u : 0u);
                        far_pair<true>(qx, qy, qz, make_float2(fmaxf(q2.x, k.h2), fmaxf(q2.y, k.h2)),
                                       make_float2(a ? A.w : 0.0f, b ? B.w : 0.0f), k, ps);
                        const bool ca = a && q2.x < k.h2, cb = b && q2.y < k.h2;
                        if (__any_sync(FULL, ca || cb)) {
                            if (ca)
                                soft_correction<true>(qx.x, qy.x, qz.x, q2.x, A.w, k.h2, k.hinv, k.hinv3, k, ps.x.x,
                                                      ps.y.x, ps.z.x, ps.p.x);
                            if (cb)
                                soft_correction<true>(qx.y, qy.y, qz.y, q2.y, B.w, k.h2, k.hinv, k.hinv3, k, ps.x.y,
                                                      ps.y.y, ps.z.y, ps.p.y);
                        }
                    }
                }
            }
        };
        const unsigned opened = __ballot_sync(FULL, om != 0u && Lk.y == 0 && (part == 0u || C.w <= split_side));
        leaves(std::true_type{}, opened & gen);
        leaves(std::false_type{}, opened & ~gen);
        __syncwarp();
    }
    ax -= ps.x.x + ps.x.y;
    ay -= ps.y.x + ps.y.y;
    az -= ps.z.x + ps.z.y;
    ph -= ps.p.x + ps.p.y;
    if (split > 1) {  // the parts of the chunk's warps, in order
        sh.o[lane] = make_float4(ax, ay, az, ph);
        sh.d[lane].x = __uint_as_float(cnt);
        __syncthreads();
        if (part != 0u)
            return;
        for (int v = 1; v < split; v++) {
            const float4 q = shared[warp + v].o[lane];
            ax += q.x;
            ay += q.y;
            az += q.z;
            ph += q.w;
            cnt += __float_as_uint(shared[warp + v].d[lane].x);
        }
    }
    if (!valid)
        return;
    // added to the mesh force, which is there already
    const float G = k.G;
    acc[3 * (size_t)out] += G * ax;
    acc[3 * (size_t)out + 1] += G * ay;
    acc[3 * (size_t)out + 2] += G * az;
    if (pot)
        pot[out] += G * ph;
    if (nint)
        nint[out] = cnt;
}
