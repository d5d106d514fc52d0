// Walk with two targets per warp (open boundaries).
//
// The group walk gives a warp 32 targets and is bound by instruction issue
// once there are some four thousand such warps.  Fewer targets leave the chip
// idle, and a warp's serial chain is the time of the call: 46 thousand
// instructions for 32 neighbours of a 2^20 Hernquist halo, four times that for
// targets scattered over the tree, where hardly any node gets one answer from
// all of them.  Here the lanes hold SOURCES (32 candidate nodes, or 32 leaf
// particles, at a time) and a warp serves two consecutive active particles.
// Every candidate is decided for both by the per-particle rule (the lane
// walk's FP32 operations, in the frame of the chunk's run), a target that
// accepts it takes its monopole from the same registers, and what some target
// opens goes back to the warp's stack (children) or to its leaf list.  Sums
// stay in registers, one set per lane and target, and are added up over the
// lanes at the end.  The work per target is about twice the group walk's, the
// chain a tenth of it, and 16 times as many warps share the work.
//
// Measured, one force call on the relative criterion (Hernquist, leaf bucket
// 16), group walk / this walk: 1000 random particles of 2^20 1.24 / 0.07 ms,
// 16384 of 2^20 0.86 / 0.15 ms, 65536 of 2^20 0.72 / 0.34 ms, 32768 of 2^17
// 0.43 / 0.19 ms; tree build and forces on a whole small system: 4096 0.32 /
// 0.20 ms, 32768 0.52 / 0.42 ms; all of 2^20 1.58 / 3.8 ms.  One target a warp
// or four took 63 and 95 us for the 1000, 547 and 346 us for the 65536.

// A run's targets as one warp's registers: lane l holds target l.
struct RunTargets {
    uint32_t s, out;          // sorted position, output slot
    float x, y, z, thr, sup;  // offset from the frame centre, threshold, support
    float gcx, gcy, gcz;      // frame centre relative to the root corner
};

// The targets of a run of gcount <= 32 active particles at [g0, g0 + gcount)
// of the sorted active list, in the frame that the group walk gives them: the
// smallest key cell holding the first and last target, moved to the middle of
// their bounding box on the grid of the node centres (2^-22 L0, so that
// node-to-frame offsets stay exact in FP32).  Offsets are FP64 differences
// rounded once.  The plain FP32 form takes absolute coordinates.
template <bool RELATIVE, bool VARH>
__device__ __forceinline__ RunTargets run_targets(const TreeView &T, const WalkConsts &k,
                                                  const uint32_t *__restrict__ sidx,
                                                  const uint32_t *__restrict__ slot, int64_t g0, int gcount,
                                                  const float *__restrict__ a_old) {
    const unsigned FULL = 0xffffffffu;
    RunTargets t;
    const int lane = threadIdx.x & 31;
    const double L0 = T.L0;
    const bool valid = lane < gcount;
    const int64_t gi = valid ? g0 + lane : g0;
    t.s = sidx ? sidx[gi] : (uint32_t)gi;
    const uint32_t j = T.perm[t.s];
    t.out = slot ? slot[gi] : j;
    const uint64_t kk = T.key[t.s];
    const uint64_t kf = __shfl_sync(FULL, kk, 0), kl = __shfl_sync(FULL, kk, gcount - 1);
    const uint64_t kx = kf ^ kl;
    const int glevel = kx ? min((__clzll(kx) - 1) / 3, kMaxLevel) : kMaxLevel;
    const uint64_t gpre = kf >> (3 * (kMaxLevel - glevel));
    const double ghalf = ldexp(L0, -(glevel + 1));
    double gcx = (double)(2 * (uint64_t)compact3w(gpre) + 1) * ghalf;
    double gcy = (double)(2 * (uint64_t)compact3w(gpre >> 1) + 1) * ghalf;
    double gcz = (double)(2 * (uint64_t)compact3w(gpre >> 2) + 1) * ghalf;
    if (k.plain) {
        gcx = -T.x0;
        gcy = -T.y0;
        gcz = -T.z0;
    }
    const double dx = T.pos[3 * (size_t)j] - (T.x0 + gcx), dy = T.pos[3 * (size_t)j + 1] - (T.y0 + gcy),
                 dz = T.pos[3 * (size_t)j + 2] - (T.z0 + gcz);
    t.x = (float)dx, t.y = (float)dy, t.z = (float)dz;
    if (!k.plain) {
        const float inf = __int_as_float(0x7f800000);
        float lox = valid ? t.x : inf, loy = valid ? t.y : inf, loz = valid ? t.z : inf;
        float hix = valid ? t.x : -inf, hiy = valid ? t.y : -inf, hiz = valid ? t.z : -inf;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            lox = fminf(lox, __shfl_xor_sync(FULL, lox, o));
            loy = fminf(loy, __shfl_xor_sync(FULL, loy, o));
            loz = fminf(loz, __shfl_xor_sync(FULL, loz, o));
            hix = fmaxf(hix, __shfl_xor_sync(FULL, hix, o));
            hiy = fmaxf(hiy, __shfl_xor_sync(FULL, hiy, o));
            hiz = fmaxf(hiz, __shfl_xor_sync(FULL, hiz, o));
        }
        const float q = (float)ldexp(L0, -22), iq = (float)ldexp(1.0 / L0, 22);  // powers of two
        const float sx = q * rintf(0.5f * (lox + hix) * iq), sy = q * rintf(0.5f * (loy + hiy) * iq),
                    sz = q * rintf(0.5f * (loz + hiz) * iq);
        gcx += (double)sx;
        gcy += (double)sy;
        gcz += (double)sz;
        t.x = (float)(dx - (double)sx);
        t.y = (float)(dy - (double)sy);
        t.z = (float)(dz - (double)sz);
    }
    t.gcx = (float)gcx, t.gcy = (float)gcy, t.gcz = (float)gcz;
    t.thr = k.thr_const;
    if (RELATIVE)
        t.thr = valid ? k.alpha_over_G * fabsf(a_old[t.out]) : 0.0f;
    t.sup = VARH ? __ldg(&T.psoft[t.s]) : 0.0f;
    return t;
}

// Exclusive prefix sum over the warp, and the total.
__device__ __forceinline__ int warp_exclusive(int v, int &total) {
    const int lane = threadIdx.x & 31;
    int incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o)
            incl += u;
    }
    total = __shfl_sync(0xffffffffu, incl, 31);
    return incl - v;
}

constexpr int kFewWarps = 4;
// Stack of child ranges.  A step takes 32 nodes (at least four ranges) and
// pushes at most 32 ranges; above kFewSafe ranges it takes one node at a time,
// and the descent of a single node adds at most one range a level.
constexpr int kFewStack = 384;
constexpr int kFewSafe = kFewStack - 64;
constexpr int kFewLeaves = 64;

struct FewShared {
    uint2 stack[kFewStack];   // (first child, children << 8 | targets that need them)
    float4 lsrc[kFewLeaves];  // opened leaf: centre (group frame), first particle
    uint2 lmeta[kFewLeaves];  // targets, particle count
};

// A warp's two targets (the second repeats the first where there is but one)
// and their sums.
template <bool TREEPM, bool VARH>
struct FewTargets {
    float2 x, y, z, thr, sup;
    PairSums s;
    uint32_t self0, self1;  // sorted positions
    uint32_t cnt0, cnt1;

    __device__ __forceinline__ void init(const RunTargets &t, int a, int b) {
        const unsigned FULL = 0xffffffffu;
        x = make_float2(__shfl_sync(FULL, t.x, a), __shfl_sync(FULL, t.x, b));
        y = make_float2(__shfl_sync(FULL, t.y, a), __shfl_sync(FULL, t.y, b));
        z = make_float2(__shfl_sync(FULL, t.z, a), __shfl_sync(FULL, t.z, b));
        thr = make_float2(__shfl_sync(FULL, t.thr, a), __shfl_sync(FULL, t.thr, b));
        if (VARH)
            sup = make_float2(__shfl_sync(FULL, t.sup, a), __shfl_sync(FULL, t.sup, b));
        self0 = __shfl_sync(FULL, t.s, a);
        self1 = __shfl_sync(FULL, t.s, b);
        s.x = s.y = s.z = s.p = make_float2(0.f, 0.f);
        cnt0 = cnt1 = 0u;
    }

    // Pair terms of one source per lane at (target - source) offset r, for the
    // targets that take it (a the first, b the second).
    __device__ __forceinline__ void term(float2 rx, float2 ry, float2 rz, float2 r2, bool a, bool b, float m, float hs,
                                         const WalkConsts &k) {
        cnt0 += a ? 1u : 0u;
        cnt1 += b ? 1u : 0u;
        float2 he = make_float2(0.f, 0.f), h2 = make_float2(k.h2, k.h2);
        if (VARH) {  // the larger support of the two
            he = make_float2(fmaxf(sup.x, hs), fmaxf(sup.y, hs));
            h2 = __fmul2_rn(he, he);
        }
        const bool ca = a && r2.x < h2.x, cb = b && r2.y < h2.y;
        far_pair<TREEPM>(rx, ry, rz, make_float2(fmaxf(r2.x, h2.x), fmaxf(r2.y, h2.y)),
                         make_float2(a ? m : 0.0f, b ? m : 0.0f), k, s);
        if (ca) {  // inside the softening length: the spline's difference
            const float hi = VARH ? 1.0f / he.x : k.hinv, hi3 = VARH ? hi * hi * hi : k.hinv3;
            soft_correction<TREEPM>(rx.x, ry.x, rz.x, r2.x, m, h2.x, hi, hi3, k, s.x.x, s.y.x, s.z.x, s.p.x);
        }
        if (cb) {
            const float hi = VARH ? 1.0f / he.y : k.hinv, hi3 = VARH ? hi * hi * hi : k.hinv3;
            soft_correction<TREEPM>(rx.y, ry.y, rz.y, r2.y, m, h2.y, hi, hi3, k, s.x.y, s.y.y, s.z.y, s.p.y);
        }
    }

    // All listed leaves, their particles 32 to a tile.  The small
    // particle-to-leaf-centre vector is subtracted first so that close pairs
    // keep their precision.
    __device__ __forceinline__ void leaves(const FewShared &sh, int nl, const TreeView &T, const WalkConsts &k) {
        const unsigned FULL = 0xffffffffu;
        const int lane = threadIdx.x & 31;
        for (int e0 = 0; e0 < nl; e0 += 32) {
            const int c = e0 + lane < nl ? (int)sh.lmeta[e0 + lane].y : 0;
            int total;
            const int start = warp_exclusive(c, total);
            int before = 0;  // leaves that start before the tile
            for (int b = 0; b < total; b += 32) {
                // the leaves that start inside the tile, a bit at their first lane
                const bool in = c > 0 && start >= b && start < b + 32;
                const unsigned starts = __reduce_or_sync(FULL, in ? 1u << (start - b) : 0u);
                const int e = before + __popc(starts & (0xffffffffu >> (31 - lane))) - 1;
                before += __popc(starts);
                const int off = b + lane - __shfl_sync(FULL, start, e & 31);
                float4 P = make_float4(0.f, 0.f, 0.f, 0.f), E = P;
                unsigned mask = 0u;
                uint32_t jj = 0u;
                float hs = 0.0f;
                if (b + lane < total) {
                    E = sh.lsrc[e0 + e];
                    mask = sh.lmeta[e0 + e].x;
                    jj = (uint32_t)(__float_as_int(E.w) + off);
                    P = __ldg(&T.spart[jj]);
                    if (VARH)
                        hs = __ldg(&T.psoft[jj]);
                }
                const float2 px = __fadd2_rn(x, make_float2(-E.x, -E.x)), py = __fadd2_rn(y, make_float2(-E.y, -E.y)),
                             pz = __fadd2_rn(z, make_float2(-E.z, -E.z));
                const float2 rx = __fadd2_rn(px, make_float2(-P.x, -P.x)), ry = __fadd2_rn(py, make_float2(-P.y, -P.y)),
                             rz = __fadd2_rn(pz, make_float2(-P.z, -P.z));
                const float2 r2 = __ffma2_rn(rx, rx, __ffma2_rn(ry, ry, __fmul2_rn(rz, rz)));
                // no target takes a term from itself, or from beyond the short-range cutoff
                const bool a = (mask & 1u) && jj != self0 && !(TREEPM && r2.x > k.rcut2);
                const bool bb = (mask & 2u) && jj != self1 && !(TREEPM && r2.y > k.rcut2);
                term(rx, ry, rz, r2, a, bb, P.w, hs, k);
            }
        }
    }

    // The walk for nt targets (1 or 2).
    template <bool RELATIVE>
    __device__ __forceinline__ void walk(const TreeView &T, const WalkConsts &k, FewShared &sh, float gcx, float gcy,
                                         float gcz, int nt, int *__restrict__ err) {
        const unsigned FULL = 0xffffffffu;
        const int lane = threadIdx.x & 31;
        const unsigned lt_mask = (1u << lane) - 1u;
        if (lane == 0)
            sh.stack[0] = make_uint2(0u, 256u | (nt > 1 ? 3u : 1u));  // the root, breadth-first index 0
        __syncwarp();
        int sn = 1, nl = 0;
        while (sn > 0) {
            // ---- up to 32 nodes from the top child ranges, of which lane l
            // holds the l-th; a node's range is the last that starts at or
            // before its lane
            const int cap = sn > kFewSafe ? 1 : 32;
            const int idx = sn - 1 - lane;
            const uint2 R = idx >= 0 ? sh.stack[idx] : make_uint2(0u, 0u);
            const int c = (int)(R.y >> 8);
            int total;
            const int excl = warp_exclusive(c, total);
            const bool some = c > 0 && excl < cap;
            const bool whole = some && excl + c <= cap;
            const unsigned starts = __reduce_or_sync(FULL, some ? 1u << excl : 0u);
            const int r = __popc(starts & (0xffffffffu >> (31 - lane))) - 1;
            const uint32_t node = __shfl_sync(FULL, R.x, r) + (uint32_t)(lane - __shfl_sync(FULL, excl, r));
            unsigned need = __shfl_sync(FULL, R.y, r);
            sn -= __popc(__ballot_sync(FULL, whole));
            if (some && !whole)  // the partly taken range stays on top
                sh.stack[idx] = make_uint2(R.x + (uint32_t)(cap - excl),
                                           ((uint32_t)(c - (cap - excl)) << 8) | (R.y & 0xffu));
            __syncwarp();
            float4 C = make_float4(0.f, 0.f, 0.f, 0.f), O = C;
            int4 Lk = make_int4(0, 0, 0, 0);
            float hsig = 0.0f;
            if (lane < min(total, cap)) {
                C = __ldg(&T.bcen[node]);
                O = __ldg(&T.bcom[node]);
                Lk = __ldg(&T.blink[node]);
                if (VARH)
                    hsig = __ldg(&T.bsoft[node]);
            } else {
                need = 0u;
            }
            // ---- the decision of each target for the lane's node
            const float dx = C.x - gcx, dy = C.y - gcy, dz = C.z - gcz;  // exact
            const float L = C.w;
            const float q = RELATIVE ? O.w * L * L : L * L;
            const float gl = k.box_guard ? 0.6f * L : -1.0f;
            const float2 px = __fadd2_rn(x, make_float2(-dx, -dx)), py = __fadd2_rn(y, make_float2(-dy, -dy)),
                         pz = __fadd2_rn(z, make_float2(-dz, -dz));
            const float2 rx = __fadd2_rn(px, make_float2(-O.x, -O.x)), ry = __fadd2_rn(py, make_float2(-O.y, -O.y)),
                         rz = __fadd2_rn(pz, make_float2(-O.z, -O.z));
            const float2 r2 = __ffma2_rn(rx, rx, __ffma2_rn(ry, ry, __fmul2_rn(rz, rz)));
            float2 th = __fmul2_rn(thr, r2);
            if (RELATIVE)
                th = __fmul2_rn(th, r2);
            bool oa = fmaxf(fabsf(px.x), fmaxf(fabsf(py.x), fabsf(pz.x))) <= gl || q > th.x;
            bool ob = fmaxf(fabsf(px.y), fmaxf(fabsf(py.y), fabsf(pz.y))) <= gl || q > th.y;
            if (VARH) {  // Sec. 3.2: a node of mixed softenings is opened inside its largest one
                oa = oa || (hsig < 0.0f && sup.x < -hsig && r2.x < hsig * hsig);
                ob = ob || (hsig < 0.0f && sup.y < -hsig && r2.y < hsig * hsig);
            }
            bool na = need & 1u, nb = need & 2u;
            if (TREEPM) {  // beyond the short-range cutoff for a target: neither opened nor accepted
                const float hl = 0.5f * L;
                float ex = fmaxf(fabsf(px.x) - hl, 0.0f), ey = fmaxf(fabsf(py.x) - hl, 0.0f),
                      ez = fmaxf(fabsf(pz.x) - hl, 0.0f);
                na = na && !(fmaf(ex, ex, fmaf(ey, ey, ez * ez)) > k.rcut2);
                ex = fmaxf(fabsf(px.y) - hl, 0.0f), ey = fmaxf(fabsf(py.y) - hl, 0.0f),
                ez = fmaxf(fabsf(pz.y) - hl, 0.0f);
                nb = nb && !(fmaf(ex, ex, fmaf(ey, ey, ez * ez)) > k.rcut2);
            }
            const unsigned om = (na && oa ? 1u : 0u) | (nb && ob ? 2u : 0u);
            // ---- what the targets open, and the monopoles they accept
            const bool push = om != 0u && Lk.y != 0, leaf = om != 0u && Lk.y == 0;
            const unsigned bp = __ballot_sync(FULL, push), bl = __ballot_sync(FULL, leaf);
            if (push) {
                const int at = sn + __popc(bp & lt_mask);
                if (at < kFewStack)
                    sh.stack[at] = make_uint2((uint32_t)Lk.x, ((uint32_t)Lk.y << 8) | om);
                else
                    atomicOr(err, 2);
            }
            sn = min(sn + __popc(bp), kFewStack);
            if (leaf) {
                const int l = nl + __popc(bl & lt_mask);
                sh.lsrc[l] = make_float4(dx, dy, dz, __int_as_float(Lk.z));
                sh.lmeta[l] = make_uint2(om, (uint32_t)Lk.w);
            }
            nl += __popc(bl);
            __syncwarp();
            term(rx, ry, rz, r2, na && !oa, nb && !ob, O.w, fabsf(hsig), k);
            __syncwarp();
            if (nl >= 32 || sn == 0) {
                leaves(sh, nl, T, k);
                nl = 0;
                __syncwarp();
            }
        }
    }

    // Adds up the lanes' parts and writes one target's results.
    __device__ __forceinline__ void write(float sx, float sy, float sz, float sp, uint32_t cnt, uint32_t out,
                                          const WalkConsts &k, float *__restrict__ acc, float *__restrict__ pot,
                                          uint32_t *__restrict__ nint, int accumulate) const {
        const unsigned FULL = 0xffffffffu;
        const int lane = threadIdx.x & 31;
        float v[4] = {sx, sy, sz, sp};
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
#pragma unroll
            for (int c = 0; c < 4; c++)
                v[c] += __shfl_xor_sync(FULL, v[c], o);
        const float r = -k.G * (lane == 0 ? v[0] : lane == 1 ? v[1] : lane == 2 ? v[2] : v[3]);
        const uint32_t n = __reduce_add_sync(FULL, cnt);
        if (lane < 3) {
            float *p = acc + 3 * (size_t)out + lane;
            *p = accumulate ? *p + r : r;
        } else if (lane == 3 && pot) {
            pot[out] = accumulate ? pot[out] + r : r;
        } else if (lane == 4 && nint) {
            nint[out] = n;
        }
    }
};

// Targets [lo, hi) (two at most) of the chunk of gcount <= 32 consecutive
// active particles at g0, each in the frame of its run (chunk_cuts).
template <bool RELATIVE, bool TREEPM, bool VARH>
__device__ __forceinline__ void few_walk_chunk(const TreeView &T, const WalkConsts &k, FewShared &sh,
                                               const uint32_t *__restrict__ sidx, const uint32_t *__restrict__ slot,
                                               int64_t g0, int gcount, int lo, int hi, const float *__restrict__ a_old,
                                               float *__restrict__ acc, float *__restrict__ pot,
                                               uint32_t *__restrict__ nint, int accumulate, int *__restrict__ err) {
    unsigned cut = k.plain ? 0u : chunk_cuts(T.key, sidx, g0, gcount);  // the plain FP32 form has one frame
    int start = 0;
    for (;;) {
        const int end = cut ? __ffs(cut) : gcount;
        const int a = max(lo, start) - start, nt = min(hi, end) - start - a;
        if (nt > 0) {
            const RunTargets t = run_targets<RELATIVE, VARH>(T, k, sidx, slot, g0 + start, end - start, a_old);
            FewTargets<TREEPM, VARH> f;
            f.init(t, a, a + nt - 1);
            f.template walk<RELATIVE>(T, k, sh, t.gcx, t.gcy, t.gcz, nt, err);
            const uint32_t o0 = __shfl_sync(0xffffffffu, t.out, a), o1 = __shfl_sync(0xffffffffu, t.out, a + nt - 1);
            f.write(f.s.x.x, f.s.y.x, f.s.z.x, f.s.p.x, f.cnt0, o0, k, acc, pot, nint, accumulate);
            if (nt > 1)
                f.write(f.s.x.y, f.s.y.y, f.s.z.y, f.s.p.y, f.cnt1, o1, k, acc, pot, nint, accumulate);
            __syncwarp();
        }
        if (!cut)
            break;
        cut &= cut - 1u;
        start = end;
    }
}

// ----------------------------------------------------------------------
// Which chunks of a call's sorted active list get two targets a warp.  A group
// walk is one warp's chain, as long for 20 groups as for 2000; this walk
// spreads it over 16 warps for twice the instructions.  It is the faster one
// until the targets in flight fill the chip, whatever their tree's size, so
// the rule goes by the number of targets in the call:
//   kFewAll   every chunk, for requests of at most kFewBH, kFewRelative or
//             kFewOther ids, by themselves or in a batch of at most kFewBatch
//             (whose one walk serves all requests).  Group walk / this walk in
//             us, Hernquist and Plummer spheres, leaf bucket 16:
//                                        theta 0.7   theta 0.5    alpha 0.0025
//               batch of 12 x 4096       437 / 344   626 / 427    605 / 363
//               batch of 3 x 16384       406 / 369   765 / 526    649 / 372
//               batch of 6 x 16384       487 / 576   792 / 856    827 / 575
//               all of 32768             212 / 187   444 / 319    282 / 153
//               all of 49152             221 / 262   452 / 472    292 / 215
//               all of 65536             244 / 336   479 / 617    310 / 275
//               32768 densest of 2^17    298 / 290   550 / 510    374 / 281
//               49152 densest of 2^17    327 / 380   592 / 686    365 / 349
//               65536 densest of 2^17    373 / 463   695 / 851    382 / 413
//             two softenings (the mesh is kinder to this walk):
//               32768 densest of 2^19    392 / 370   755 / 703    608 / 382
//               65536 densest of 2^19    439 / 629   851 / 1257   650 / 580
//             The relative criterion has longer and more uneven chains: batches
//             with it keep this walk to kFewSmall ids where the systems have at
//             most kFewSystem particles (5 x 16384 772 / 507, 10 x 8192 776 / 504).
//   span > 0  larger requests of at most 2^16 ids: the chunks whose neighbours
//             are on average at least that many particles apart in key order;
//             closer ones keep the group walk.  From 4 in a plain call (65536
//             random ids of 2^19, 2^20 at theta = 0.5 834 / 808, 967 / 845 us, at
//             alpha = 0.0025 563 / 361, 645 / 375), and in a batch, whose other
//             requests may fill the chip, from 20 (theta) or 10 (16 requests for
//             random ids of 2^19: span 16 4544 / 5675 us at theta = 0.5, 2265 /
//             2333 at alpha = 0.0025; span 32 3162 / 3001, 1724 / 1285).
//   kFewNone  larger requests.
// At 32 particles a group a request has the same bits in a plain call and in
// every batch of at most kFewBatch ids, and in every batch larger than kFewSmall;
// the two differ by FP32 rounding.  Groups of 64 particles never come here.
// ----------------------------------------------------------------------
constexpr int64_t kFewBH = 1 << 15;
constexpr int64_t kFewRelative = 3 << 14;  // uniform softening, no mesh
constexpr int64_t kFewOther = 1 << 16;     // relative criterion with the mesh or per-particle softening
constexpr int64_t kFewBatch = 3 << 14;
constexpr int64_t kFewSmall = 9 << 13, kFewSystem = 1 << 15;
constexpr int64_t kFewRequest = 1 << 16;

inline int few_rule(bool relative, bool uniform, int64_t n_act) {
    const int64_t line = !relative ? kFewBH : uniform ? kFewRelative : kFewOther;
    return n_act <= line ? (int)kFewAll : n_act <= kFewRequest ? 4 : (int)kFewNone;
}

inline int few_rule_in_batch(const System *s, bool relative, int64_t n_ids, int64_t batch_ids) {
    if (batch_ids <= kFewBatch || (relative && s->n <= kFewSystem && batch_ids <= kFewSmall))
        return few_rule(relative, true, n_ids);
    return n_ids > kFewRequest ? (int)kFewNone : relative ? 10 : 20;
}

// A call with chunks for both walks launches the group walk first and this one
// right behind it in the same stream, allowed to start as soon as all blocks of
// the group walk run (they say so with cudaTriggerProgrammaticLaunchCompletion):
// its warps then fill what the group walk leaves idle.  Beside it on a second
// stream this walk took the places that the group walk's blocks spread over, and
// its long chains met on few SMs.  Batches of requests for 2048 random ids of
// 2^16 at theta = 0.5, chunks of spread 32 and more to this walk (us, groups
// only / second stream / one after the other / this way): 64 requests 1810 / 2320
// / 2310 / 1760, 16 requests 1650 / 1850 / 1450 / 1180.
// Block 0 of this walk waits for the group walk before it ends, so that what
// follows in the stream follows both.
inline cudaLaunchConfig_t beside_config(unsigned blocks, int threads, cudaLaunchAttribute *attr, cudaStream_t st) {
    attr->id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr->val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t c{};
    c.gridDim = dim3(blocks);
    c.blockDim = dim3((unsigned)threads);
    c.stream = st;
    c.attrs = attr;
    c.numAttrs = 1;
    return c;
}

__device__ __forceinline__ void end_after_group_walk() {
    if (blockIdx.x == 0)
        cudaGridDependencySynchronize();  // no wait in a launch that stands alone
}

// A warp per two active particles of a chunk, for the chunks that the rule
// gives to this walk (the others' warps do nothing).
template <bool RELATIVE, bool TREEPM, bool VARH>
__global__ void __launch_bounds__(kFewWarps * 32)
    k_walk_few(TreeView T, const uint32_t *__restrict__ sidx, const uint32_t *__restrict__ slot,
               const float *__restrict__ a_old, int64_t n_act, int rule, WalkConsts k, float *__restrict__ acc,
               float *__restrict__ pot, uint32_t *__restrict__ nint, int accumulate, int *__restrict__ err) {
    __shared__ FewShared shared[kFewWarps];
    const int64_t first = ((int64_t)blockIdx.x * kFewWarps + (threadIdx.x >> 5)) * 2;
    const int64_t g0 = first & ~int64_t(31);
    const int gcount = (int)min((int64_t)32, n_act - g0);
    if (first < n_act && few_chunk(rule, sidx, g0, gcount)) {
        const int lo = (int)(first - g0);
        few_walk_chunk<RELATIVE, TREEPM, VARH>(T, k, shared[threadIdx.x >> 5], sidx, slot, g0, gcount, lo,
                                               min(lo + 2, gcount), a_old, acc, pot, nint, accumulate, err);
    }
    end_after_group_walk();
}
