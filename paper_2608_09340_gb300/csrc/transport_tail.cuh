// The end of a launch: the last packets of a CTA, a few lanes' worth, each
// walked by a group of lanes (FP32 walk). Included by transport_impl.cuh.
//
// What bounds it. Scattering counts are heavy-tailed, so a launch ends with
// packets that have up to 1e6 events left and nothing else to run: its time
// is the latency of one packet's event, 1420 cycles when a lane walks its
// packet alone (two Philox blocks, the draws, the profile, the test, then the
// sampler, one after the other). Most of that work does not depend on the
// packet's frequency. A group of G lanes therefore takes the next G
// scatterings of its packet, one per lane: each lane makes its scattering's
// draws, the angle to the previous scattering's direction, and the sampler's
// inversion at its ln(xi) in the kUWin rows around the packet's |x|. What
// remains serial is the chain of frequencies, x -> row -> u_par -> x' (136
// cycles a step with 128 registers, 173 with 64), walked for up to G
// scatterings on the assumption that all happen in this cell. Then each lane evaluates the profile and the distance
// of its own segment, the positions follow as a chain of fused multiply-adds,
// and the first lane whose point lies outside the cell (or that ends the
// packet) marks how many of the scatterings stand; the rest are walked again
// from the next cell, with the same draws. A packet alone then takes 150 to
// 200 ns per event (690 to 1000 before): 1e5 packets in the outflowing sphere
// 938 -> 389 ms, 1e4 in the slab 143 -> 35.5 ms (183 -> 44 with the packets
// of another seed), together with the other steps.
//
// Every value is formed by the functions and in the order of advance(), so a
// packet continues bit for bit as it would have in a lane of its own.
#pragma once

// Warps of a CTA that walk packets this way (their buffers take the stash's
// place in shared memory). A CTA starts with up to kTailWide packets per warp
// in groups of 8 lanes, or with nearly twice as many in groups of 4: these
// use three times the issue slots per event of a lane's walk and gain less,
// and a CTA with few packets above kTailWide rather waits for some to end.
// Measured with both / with groups of 8 only, means of three seeds: outflow of
// 1e5 packets 368 / 369 ms, static sphere 492 / 500, dusty slab 107 / 109,
// 64 models 162 / 167, 1e4-packet slab 35.8 / 35.1 (all but the models'
// within the scatter of these calls); with groups of 4 from 2 kTailWide down
// the slab (33 packets per CTA) took 52 for 44 with a fourth seed's packets.
//
// Runs with an emissivity tally (TransportArgs::tail_warps) use kTailWarpsL1:
// a segment that the walk deposits itself reads the R_IIA table through L1,
// and with 8 warps' buffers two CTAs need the SM's largest shared-memory
// split, which leaves L1 28 of 256 KB; with 6 they leave it 60. Medians of 8
// runs, without groups (17 KB for the stash) / 8 warps / 6: 128^3 envelope, 3
// cameras x 64 channels, 1e6 packets deposited in the walk 20.3 / 27.0 / 22.0
// ms, 4e6 with the default buffer 46.9 / 52.3 / 46.1, a box of tau0 = 100 with
// 1e5 packets 32.5 / 41.1 / 31.8. Without that tally 8 are better (box of
// tau0 = 1000 with mean intensity, 1e5 packets: 27.0 / 12.5 / 13.4). The 32
// packets of one warp's draw of ids, a CTA's all in a run of few, are among
// those that 6 warps start with in groups of 4.
//
// With the tables in the constant bank (mode 4) the lanes of a group read
// different addresses, which that bank serves one after the other, so that
// many groups stand in one another's way: kTailWarpsConst, unless a CTA's
// packets all go to groups at once. Slab of 128 cells, tau = 32000, without
// groups / 8 warps / 4: 2e3 packets 610 / 151 / 183 ms, 2e4 788 / 707 / 567,
// 2e5 2496 / 2608 / 2421; dusty slab, 1e5 packets 104 / 113 / 100.
constexpr int kTailWarps = 8, kTailWarpsL1 = 6, kTailWarpsConst = 4;
constexpr int kTailWide = 4;
constexpr bool tail_starts(int total, int warps)
{
    return total <= warps * kTailWide || (total <= warps * 2 * kTailWide && 3 * total >= warps * 4 * kTailWide);
}

// Rows inverted ahead (odd: no bank conflicts between slots). In the line's
// core the frequency spreads by 0.7 and rows 0 to 6 (|x| < 2.67) hold nearly
// all scatterings; a chain that leaves the window ends there and the window
// moves.
constexpr int kUWin = 7;

// A warp's buffers. Slots are lanes; the arrays of the two serial loops are in
// chain order (index: first lane of the group + place in the chain), so that
// the loops read at constant offsets. They run in fours and may read past
// their group's part, whose values are then not used.
struct TailBuf {
    float4 a[32];               // {z1, sin(gamma), g - 1, byte offset of the slot's row 0 in u}
    float2 b[32];               // {first row of u, z2}
    float u[32 * kUWin + kUsNx]; // u of kUWin rows per slot (any row at any slot reads inside the buffer)
    union {
        struct {
            float4 ac[64];      // a in chain order
            float vc[64];       // n_out.V/b
            float xs[68];       // [2 x first lane + k]: lab-frame frequency in front of scattering k
        };
        struct {
            float4 d[32];       // rich: {absorbed fraction, mean-weight factor, H, 0}
            float2 c[3][32];    // {ds, n_in's component}
            float o[3][32];     // position in front of the segment, by component
        };
    };
};
static_assert(sizeof(TailBuf) % 16 == 0, "warps' buffers stay aligned");
static_assert(kUsNx * sizeof(float) <= sizeof(float4) * 32, "rows below a slot's window fall into a and b");

constexpr size_t tail_bytes(int block, int warps)
{
    const int w = block / 32 < warps ? block / 32 : warps;
    return (size_t)w * sizeof(TailBuf);
}

// u at L in N rows from i0: us_sample's inversion of each row, side by side
// so that the rows' reads overlap. The node is bisected between the entries
// of this guide bin and the next one: where a row is flat (between the
// Gaussian core and the Lorentz spike) one bin spans up to 27 nodes, and with
// 32 lanes and several rows some walk would almost always be that long.
template <int N>
__device__ __forceinline__ void us_invert_rows(float L, int m, int i0, const Tabs& T, float* u)
{
    int j[N], h[N];
    const float* c = T.sc + i0 * kUsNu;
    const int m1 = m < kGuideN - 1 ? m + 1 : m;
#pragma unroll
    for (int r = 0; r < N; ++r) {
        j[r] = T.sg[(i0 + r) * kGuideN + m];
        h[r] = (m1 > m ? T.sg[(i0 + r) * kGuideN + m1] : kUsNu - 2) + 1;
    }
    for (;;) {
        bool more = false;
#pragma unroll
        for (int r = 0; r < N; ++r) {
            const int mid = (j[r] + h[r]) >> 1;         // (j itself once h = j + 1)
            const bool le = c[r * kUsNu + mid] <= L;
            j[r] = le ? mid : j[r];
            h[r] = le ? h[r] : mid;
            more = more || h[r] - j[r] > 1;
        }
        if (!more) break;
    }
    float c0[N], c1[N];
    bool off = false;
#pragma unroll
    for (int r = 0; r < N; ++r) {
        c0[r] = c[r * kUsNu + j[r]];
        c1[r] = c[r * kUsNu + j[r] + 1];
        off = off || c0[r] > L || c1[r] <= L;
    }
    if (off) {          // the bin of a rounded logit can be a neighbour's: walk on
#pragma unroll
        for (int r = 0; r < N; ++r) {
            while (c0[r] > L) { --j[r]; c1[r] = c0[r]; c0[r] = c[r * kUsNu + j[r]]; }
            while (c1[r] <= L) { ++j[r]; c0[r] = c1[r]; c1[r] = c[r * kUsNu + j[r] + 1]; }
        }
    }
#pragma unroll
    for (int r = 0; r < N; ++r) {
        const float fr = __fmul_rn(L - c0[r], Ops<float>::rcp(c1[r] - c0[r]));
        u[r] = fmaf((float)kUsDu, fr, fmaf((float)kUsDu, (float)j[r], (float)kUsU0));
    }
}

// A segment's part of the visit sums and the weight, as advance() adds them.
template <unsigned F>
__device__ __forceinline__ void visit(const TransportArgs& A, bool absorbs, float ab, float fct, float ds, float H,
                                      float& w, float& ve, float& va)
{
    float wseg = w;
    if (absorbs) wseg = w * fct;
    if (A.rich & KRL_TALLY_EXC) ve = fmaf(wseg * ds, H, ve);
    if (absorbs) {
        va = fmaf(w, ab, va);
        w = w * (1.0f - ab);
    }
}

// Takes over the packet of lane src (state that a later event reads).
template <unsigned F>
__device__ __forceinline__ void shfl_packet(Pkt<float>& p, int src)
{
    p.c = __shfl_sync(kFull, p.c, src);
    p.cx = __shfl_sync(kFull, p.cx, src);
    p.cy = __shfl_sync(kFull, p.cy, src);
    p.cz = __shfl_sync(kFull, p.cz, src);
    p.px = __shfl_sync(kFull, p.px, src);
    p.py = __shfl_sync(kFull, p.py, src);
    p.pz = __shfl_sync(kFull, p.pz, src);
    p.nx = __shfl_sync(kFull, p.nx, src);
    p.ny = __shfl_sync(kFull, p.ny, src);
    p.nz = __shfl_sync(kFull, p.nz, src);
    p.x = __shfl_sync(kFull, p.x, src);
    p.tau = __shfl_sync(kFull, p.tau, src);
    p.rec.x = __shfl_sync(kFull, p.rec.x, src);
    p.rec.y = __shfl_sync(kFull, p.rec.y, src);
    p.rec.z = __shfl_sync(kFull, p.rec.z, src);
    p.rec.w = __shfl_sync(kFull, p.rec.w, src);
    p.nscat = __shfl_sync(kFull, p.nscat, src);
    p.ncross = __shfl_sync(kFull, p.ncross, src);
    p.id = __shfl_sync(kFull, p.id, src);
    p.vis_scat = __shfl_sync(kFull, p.vis_scat, src);
    if (F & F_RICH) {
        p.vis_exc = __shfl_sync(kFull, p.vis_exc, src);
        p.vis_abs = __shfl_sync(kFull, p.vis_abs, src);
        p.wgt = __shfl_sync(kFull, p.wgt, src);
    }
}

// Walks the warp's packets to their ends. On entry the lanes of group
// lane / G hold the same packet p (alive: the group has one).
template <unsigned F, int PH>
__device__ __forceinline__ void walk_tail(const TransportArgs& A, const RoundKeys& K, Pkt<float>& p, bool alive, int G, TailBuf* tb,
                          const Tabs& T, float a, float H0, LaneStats& st)
{
    using O = Ops<float>;
    constexpr bool VEL = (F & F_VEL) != 0, RICH = (F & F_RICH) != 0, SEG = (F & F_SEG) != 0;
    const int lane = (int)(threadIdx.x & 31u);
    const bool absorbs = RICH && A.tau_abs;
    int sub = lane & (G - 1), base = lane - sub;
    uint32_t ev = 0;            // the scattering whose draws this lane holds (0: none)
    int have = 0;               // draws held of the group's packet, from its next scattering on
    int known = 0;              // of these, with frequencies
    float xe = 0.0f;            // the frequency after the last known one
    float myc = 0.0f, myo = 0.0f, H = 0.0f;     // this lane's scattering: gas-frame frequency, lab frame after it, profile
    bool out = false, far = false;              // its row lies outside its window; |x| > 300
    float mx = 0.0f, my = 0.0f, mz = 0.0f, tn = 0.0f, ueps = 1.0f;
    tb->a[lane] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);   // (offset 0: every slot's window lies in u from here on)
    tb->b[lane] = make_float2(0.0f, 0.0f);
    int len = 16;               // about the run of scatterings between two crossings
    for (;;) {
        // ---- packets that ended leave room: the remaining ones take wider groups
        const unsigned heads = __ballot_sync(kFull, alive && sub == 0);
        if (!heads) break;
        const int ng = __popc(heads);
        if (2 * G * ng <= 32) {
            do G *= 2;
            while (2 * G * ng <= 32);
            sub = lane & (G - 1);
            base = lane - sub;
            const int j = lane / G;
            unsigned t = heads;
            for (int q = 0; q < j && (t & (t - 1u)); ++q) t &= t - 1u;
            shfl_packet<F>(p, __ffs(t) - 1);
            alive = j < ng;
            ev = 0;
            have = known = 0;
        }
        // ---- the event budget
        const uint32_t cnt = p.nscat + p.ncross;
        if (alive && cnt >= A.max_iters32) {
            flush_visit<float, F>(A, p, sub == 0);
            if (sub == 0) end_packet(A, p, 3, st.stuck, st);
            alive = false;
        }
        const uint32_t room = A.max_iters32 - cnt;      // events that may still run (wraps once ended: unused)
        const uint32_t e0 = p.nscat + 1u;
        const int s0 = (int)(e0 & (uint32_t)(G - 1));   // slot of scattering e0: slots hold e mod G
        const int pos = (sub - s0) & (G - 1);           // this lane's place in the chain

        // A scattering's frequency does not depend on the cell, unless the gas
        // moves: then a crossing ends what is known, and chains are kept
        // short. Otherwise they run over all G scatterings.
        if (__any_sync(kFull, alive && known == 0)) {
        // ---- draws of the next G scatterings, once the held ones run short
        if (__any_sync(kFull, alive && have < (VEL ? (len < 8 ? len : 8) : G))) {
            have = G;
            const uint32_t e = e0 + (uint32_t)pos;
            const bool fresh = e != ev;
            float L = 0.0f, z1 = 0.0f, z2 = 0.0f;
            int gm = 0;
            if (fresh) {
                const uint32_t lo = (uint32_t)p.id, hi = (uint32_t)(p.id >> 32);
                const Words w0 = philox(lo, hi, e, 0u, K), w1 = philox(lo, hi, e, 1u, K);
                const DrawsF D = draws_f32(w0, w1);
                const float2 z = __fmul2_rn(make_float2(D.rad, D.rad), make_float2(D.bc, D.bs));
                z1 = z.x;
                z2 = z.y;
                L = D.L;
                gm = D.gm;
                mx = D.mx;
                my = D.my;
                mz = D.mz;
                tn = D.tau;
                if (RICH) ueps = O::uni(w1.w[2]);
                ev = e;
            }
            __syncwarp();
            const int prev = base + ((sub - 1) & (G - 1));
            float ix = __shfl_sync(kFull, mx, prev), iy = __shfl_sync(kFull, my, prev), iz = __shfl_sync(kFull, mz, prev);
            if (fresh) {
                if (pos == 0) {
                    ix = p.nx;
                    iy = p.ny;
                    iz = p.nz;
                }
                float gm1, sg;
                scatter_angle<float>(ix, iy, iz, mx, my, mz, gm1, sg);
                // rows around the packet's |x|: in the core from row 0 up
                float xc = p.x;
                if (VEL) xc = p.x - vdot<float>(p.nx, p.ny, p.nz, p.rec);
                int r0 = us_row(fabsf(xc), T) - kUWin / 2;
                r0 = r0 < 0 ? 0 : (r0 > kUsNx - kUWin ? kUsNx - kUWin : r0);
                tb->a[lane] = make_float4(z1, sg, gm1, __int_as_float((lane * kUWin - r0) * 4));
                tb->b[lane] = make_float2(__int_as_float(r0), z2);
                us_invert_rows<4>(L, gm, r0, T, tb->u + lane * kUWin);
                us_invert_rows<kUWin - 4>(L, gm, r0 + 4, T, tb->u + lane * kUWin + 4);
            }
        }
        // ---- the chain of frequencies: scattering e0 + k at gas-frame frequency xc
        if (VEL) known = 0;
        const int goal = VEL && len < have ? len : have;
        const int steps = (int)__reduce_max_sync(kFull, (unsigned)(alive ? goal - known : 0));
        // (+ 0 turns a negative zero into a positive one: the sign of x_in
        // then is its sign bit)
        float x = (known ? xe : p.x) + 0.0f;
        const float xb = x, vb = VEL ? vdot<float>(p.nx, p.ny, p.nz, p.rec) : 0.0f;
        float vd = vb;
        // (both halves of ac: a group with known scatterings reads past its part
        // into the next one's or the upper half, and every offset there has to
        // be a slot's)
        tb->ac[base + pos] = tb->a[lane];
        tb->ac[32 + lane] = tb->a[lane];
        if (VEL) tb->vc[base + pos] = vdot<float>(mx, my, mz, p.rec);
        __syncwarp();
        const float4* pa = tb->ac + (base + known);
        const float* pv = tb->vc + (base + known);
        float* px = tb->xs + (2 * base + known + 1);
#pragma unroll 1
        for (int k0 = 0; k0 < steps; k0 += 4, pa += 4, pv += 4, px += 4) {
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const float4 qa = pa[q];
                const float vo = VEL ? pv[q] : 0.0f;
                const float xc = VEL ? x - vd : x;
                const float ax = fabsf(xc);
                const float4* rb = T.rb + 2 * row_bin_in(ax);
                const float4 g = rb[0];
                const float2 g2 = *reinterpret_cast<const float2*>(rb + 1);
                const float* u = reinterpret_cast<const float*>(
                    reinterpret_cast<const char*>(tb->u) + (4 * __float_as_int(g.y) + __float_as_int(qa.w)));
                const float u0 = u[0], u1 = u[1], u2 = u[2];
                const bool up = g.x <= ax;
                const float t = __fmul_rn(ax - (up ? g2.x : g.z), up ? g2.y : g.w);
                // the sign of x_in, which u_par takes, on g - 1
                const float gs = __uint_as_float(__float_as_uint(qa.z) ^ (__float_as_uint(xc) & 0x80000000u));
                x = scatter_x<float>(xc, us_lerp<float>(t, up ? u1 : u0, up ? u2 : u1), gs, qa.x, qa.y);
                if (VEL) {
                    x = x + vo;
                    vd = vo;
                }
                px[q] = x;
            }
        }
        __syncwarp();
        // each lane picks its own scattering up. Beyond |x| = 300 u_par is the
        // second Gaussian; the chain goes wrong there and is taken up after it
        if (pos >= known && pos < goal) {
            const float xl = pos == known ? xb : tb->xs[2 * base + pos];
            myo = tb->xs[2 * base + pos + 1];
            myc = VEL ? xl - (pos == 0 ? vb : tb->vc[base + pos - 1]) : xl;
            const float ax = fabsf(myc);
            const float2 q = tb->b[lane];
            far = ax > 300.0f;
            out = !far && (unsigned)(us_row(ax, T) - __float_as_int(q.x)) >= (unsigned)(kUWin - 1);
            if (far) {
                const float4 qa = tb->a[lane];
                myo = scatter_x<float>(myc, q.y, qa.z, qa.x, qa.y);
                if (VEL) myo = myo + tb->vc[base + pos];
            }
        }
        known = goal;
        xe = __shfl_sync(kFull, myo, base + ((s0 + goal - 1) & (G - 1)));
        H = profile<float, PH>(A, myc, T.sv, a, H0);
        __syncwarp();
        }

        // ---- each lane: the distance of its own segment
        const int now = known < len ? known : len;      // segments looked at
        const int now4 = (int)(__reduce_max_sync(kFull, (unsigned)(alive ? now : 0)) + 3u) & ~3;
        const int prev = base + ((sub - 1) & (G - 1));
        float ix = __shfl_sync(kFull, mx, prev), iy = __shfl_sync(kFull, my, prev), iz = __shfl_sync(kFull, mz, prev);
        float ti = __shfl_sync(kFull, tn, prev);
        if (pos == 0) {
            ix = p.nx;
            iy = p.ny;
            iz = p.nz;
            ti = p.tau;
        }
        const float alpha = __fmul_rn(p.rec.x, H);
        const float ds = O::dv(ti, alpha);
        tb->c[0][base + pos] = make_float2(ds, ix);
        tb->c[1][base + pos] = make_float2(ds, iy);
        tb->c[2][base + pos] = make_float2(ds, iz);
        float ab = 0.0f, fct = 1.0f;
        if (RICH) {
            if (absorbs) fct = seg_factor<float>(__ldg(A.tau_abs + p.c) * ds, ab);
            tb->d[base + pos] = make_float4(ab, fct, H, 0.0f);
        }
        __syncwarp();

        // ---- positions (and, rich, weights and visit sums) in front of each
        // segment: a lane follows one component, which leaves a step one read,
        // one write and one fused multiply-add
        const int comp = (sub & 3) < 3 ? sub & 3 : 2;
        float qc = comp == 0 ? p.px : (comp == 1 ? p.py : p.pz);
        float w = p.wgt, ve = p.vis_exc, va = p.vis_abs, ow = w, oe = ve, oa = va;
        const float2* pc = &tb->c[comp][base];
        float* po = &tb->o[comp][base];
        const float4* pd = tb->d + base;
#pragma unroll 1
        for (int k0 = 0; k0 < now4; k0 += 4, pc += 4, po += 4, pd += 4) {
            float2 v[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) v[q] = pc[q];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                po[q] = qc;
                qc = fmaf(v[q].x, v[q].y, qc);
                if (RICH) {
                    const bool mine = k0 + q == pos;
                    const float4 d = pd[q];
                    ow = mine ? w : ow;
                    oe = mine ? ve : oe;
                    oa = mine ? va : oa;
                    visit<F>(A, absorbs, d.x, d.y, v[q].x, d.z, w, ve, va);
                }
            }
        }
        __syncwarp();
        const float2 oxy = make_float2(tb->o[0][base + pos], tb->o[1][base + pos]);
        const float oz = tb->o[2][base + pos];
        // ---- how many of the scatterings stand: up to the first segment that
        // leaves the cell or ends the packet, or whose row was not at hand,
        // and within the event budget
        const float2 exy = __ffma2_rn(make_float2(ds, ds), make_float2(ix, iy), oxy);
        const float ez = fmaf(ds, iz, oz);
        const bool scat = in_cell(exy, ez);
        bool gone = false, dead = false;                // absorbed; destroyed
        float aw = ow, ae = oe, aa = oa;                // after this lane's segment
        if (RICH) {
            visit<F>(A, absorbs, ab, fct, ds, H, aw, ae, aa);
            gone = scat && absorbs && aw < (float)kWeightCut;
            dead = scat && !gone && (A.rich & kRichEps) && ueps < __ldg(A.eps + p.c);
        }
        // bit k: the chain's k-th segment
        unsigned stop = __ballot_sync(kFull, pos < now && (!scat || gone || dead)) >> base;
        const unsigned group = G < 32 ? (1u << G) - 1u : kFull;
        auto order = [&](unsigned bits) {
            bits &= group;
            return ((bits >> s0) | (s0 ? bits << (G - s0) : 0u)) & group;
        };
        stop = order(stop);
        // A scattering without its row has its own profile and place: a
        // crossing, absorption or destruction there stands, its outcome does
        // not. The place after one beyond |x| = 300 was evaluated with another
        // frequency than the packet has: whether it stops there is not known.
        unsigned lost = 0u;
        if (__any_sync(kFull, pos < now && (out || far))) {     // rare
            lost = order(__ballot_sync(kFull, pos < now && out) >> base);
            const unsigned wrong = order(__ballot_sync(kFull, pos < now && far) >> base) << 1;
            stop &= ~wrong;
            lost |= wrong;
        }
        int lim = room < (uint32_t)now ? (int)room : now;
        const int fo = lost ? __ffs(lost) - 1 : 64;
        int f = stop ? __ffs(stop) - 1 : now;
        const bool ends = f < lim && f <= fo;           // segment f runs, and is not a plain scattering
        if (fo < lim) lim = fo;
        f = alive ? (f < lim ? f : lim) : 0;            // (a group without a packet keeps known >= 0)
        have -= f;
        known -= f;
        if (!ends && f == fo) {                         // draw again, the window around x
            have = known = 0;
            ev = 0;
        }
        if (VEL && ends) known = 0;
        // rich: the tallies of the segments that scattered, each by its lane
        if (SEG && alive && (A.rich & (KRL_TALLY_J | KRL_TALLY_EMISS)) && pos < now &&
            (pos < f || (pos == f && ends && scat))) {
            float wseg = ow;
            if (absorbs) wseg = ow * fct;
            rich_segment<float, F>(A, T, p.c, p.rec, ix, iy, iz, ds, myc, H, wseg);
        }
        // ---- the state in front of segment f, or after the whole chain
        const bool whole = f == now;
        const int src = base + ((s0 + (whole ? now - 1 : f)) & (G - 1));
        const int kind = gone ? 2 : (dead ? 3 : 1);
        p.nx = __shfl_sync(kFull, whole ? mx : ix, src);
        p.ny = __shfl_sync(kFull, whole ? my : iy, src);
        p.nz = __shfl_sync(kFull, whole ? mz : iz, src);
        p.tau = __shfl_sync(kFull, whole ? tn : ti, src);
        p.px = __shfl_sync(kFull, whole ? exy.x : oxy.x, src);
        p.py = __shfl_sync(kFull, whole ? exy.y : oxy.y, src);
        p.pz = __shfl_sync(kFull, whole ? ez : oz, src);
        const float xf = __shfl_sync(kFull, myo, base + ((s0 + f - 1) & (G - 1)));
        p.x = f > 0 ? xf : p.x;
        const float fH = __shfl_sync(kFull, H, src);
        p.nscat += (uint32_t)f;
        p.vis_scat += (uint32_t)f;
        float fds = 0.0f, fc = 0.0f;
        int fk = 1;
        if (RICH) {
            fds = __shfl_sync(kFull, ds, src);
            fc = __shfl_sync(kFull, myc, src);
            fk = __shfl_sync(kFull, kind, src);
            p.wgt = __shfl_sync(kFull, whole ? aw : ow, src);
            p.vis_exc = __shfl_sync(kFull, whole ? ae : oe, src);
            p.vis_abs = __shfl_sync(kFull, whole ? aa : oa, src);
        }
        // look as far ahead as the runs of scatterings between crossings go
        const bool any_end = __any_sync(kFull, alive && ends);
        len = any_end ? (len > 7 ? len - 4 : 4) : (len + 4 < 32 ? len + 4 : 32);
        if (alive && ends) {
            const bool lead = sub == 0;
            const float falpha = __fmul_rn(p.rec.x, fH);
            int axis = 0;
            float nd = 0.0f, s = fds;
            const float4 rec = p.rec;
            if (!RICH || fk == 1) s = to_face(p, axis, nd);
            bool over = false;
            if (RICH) {
                // segment f: to the face, or the scattering that ended the packet
                float wseg = p.wgt, fab = 0.0f;
                if (absorbs) wseg = p.wgt * seg_factor<float>(__ldg(A.tau_abs + p.c) * s, fab);
                if (A.rich & KRL_TALLY_EXC) p.vis_exc = fmaf(wseg * s, fH, p.vis_exc);
                if (SEG && fk == 1 && lead && (A.rich & (KRL_TALLY_J | KRL_TALLY_EMISS)))
                    rich_segment<float, F>(A, T, p.c, rec, p.nx, p.ny, p.nz, s, fc, fH, wseg);
                if (absorbs) {
                    p.vis_abs = fmaf(p.wgt, fab, p.vis_abs);
                    p.wgt = p.wgt * (1.0f - fab);
                    if (p.wgt < (float)kWeightCut) {
                        flush_visit<float, F>(A, p, lead);
                        if (lead) end_packet(A, p, 4, st.absorbed, st);
                        over = true;
                    }
                }
                if (!over && fk == 3) {
                    ++p.nscat;
                    ++p.vis_scat;
                    flush_visit<float, F>(A, p, lead);
                    if (lead) end_packet(A, p, 2, st.des, st);
                    over = true;
                }
            }
            if (!over) over = !cross_face<float, F>(A, p, falpha, s, axis, nd, st, lead);
            if (over) alive = false;
        }
        __syncwarp();
    }
}
