// Groups of time steps in one pass over memory.
//
// Between two steps the carriers of a stack depend on one another only
// through the slots and ids of new carriers: a carrier's random words are
// keyed by its slot and the step, so a slot that exists can be advanced
// through several steps without knowing what the others do.  A group runs m
// steps as
//   k_group   every slot present at the group's start, through all m steps: a
//             warp holds a sub-tile of slots in shared memory, steps them
//             together and runs the general step for the eventful ones; the
//             secondaries go, in slot order, to a list per sub-tile and step
//   k_tail    the carriers created in the group, step by step: the source's,
//             the secondaries' slots and ids (the counts of the lists give
//             them), and the steps that the new carriers themselves take in
//             the rest of the group
// The slot order, the ids, the random words and the order of capacity drops
// are those of single steps, so the results are the same bit for bit.
//
// A group is closed when no carrier can be created in it (every buffer full, or
// secondaries switched off, and no source): it then runs to the end of its
// range (the next density or compaction step) in one pass, and k_tail only keeps
// the books.  An open group has at most GROUP_OPEN steps, for which the record
// lists have room whatever happens (one record per slot and step).  Which of
// the two a group is, only the device knows: every launch compares the device
// step counter with its own first step and leaves at once if an earlier
// group has run past it.
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <type_traits>
#include <vector>

#include "pic_step.cuh"

namespace pic {

namespace {

// Most warps of a k_group block (20 and 24, at the fewer registers that leaves,
// were not faster) and quads per turn of the sweep (2: 39.9 ms for 50 steps of
// 4e8 carriers, 4: 39.5).
constexpr int GW_MAX = 16;
constexpr int UNROLL = 4;

template <bool DET>
__device__ __forceinline__ float fly(float z, float w, float t)
{
    return DET ? __fadd_rn(z, __fmul_rn(w, t)) : __fmaf_rn(w, t, z);
}

__device__ __forceinline__ int cell_at(float z, float inv_dz, int nc)
{
    const int c = __float_as_int(__fmaf_rd(z, inv_dz, 8388608.0f)) - 0x4B000000;
    return c < nc - 1 ? c : nc - 1;
}

// Shared-memory addition at a 32-bit address.  Unconditional: a lane with
// nothing to add adds 0 (a predicate became branches around every addition).
__device__ __forceinline__ void red_shared(uint32_t addr, uint32_t v)
{
    asm volatile("red.shared::cta.add.u32 [%0], %1;" ::"r"(addr), "r"(v));
}

// Philox4x32-10 of the scattering tests of one step, x the quad's index: the
// other three counter words are the same for every quad, so the first two
// rounds need one product each and the constants below.
struct TestKey {
    uint32_t u0, u1, u2, u3, u4, u5;
};

__device__ __forceinline__ TestKey test_key(const Args &a, uint32_t ctr_hi, uint32_t step)
{
    TestKey t;
    const unsigned long long p1 = 0xCD9E8D57ull * step;
    t.u0 = (uint32_t)(p1 >> 32) ^ ctr_hi ^ a.rk0[0];        // word 0 after round 0
    t.u1 = SUB_TEST ^ a.rk1[0];                             // word 2: hi(p0) ^ u1
    const unsigned long long q0 = 0xD2511F53ull * t.u0;     // round 1
    t.u2 = (uint32_t)p1 ^ a.rk0[1];                         // word 0: hi(q1) ^ u2
    t.u3 = (uint32_t)(q0 >> 32) ^ a.rk1[1];                 // word 2: lo(p0) ^ u3
    t.u4 = (uint32_t)q0;                                    // word 3 after round 1
    t.u5 = t.u4 ^ a.rk1[2];
    return t;
}

__device__ __forceinline__ uint4 philox_test(uint32_t x, const TestKey &t, const Args &a)
{
    const unsigned long long p0 = 0xD2511F53ull * x;
    const uint32_t c2 = (uint32_t)(p0 >> 32) ^ t.u1, c3 = (uint32_t)p0;
    const unsigned long long q1 = 0xCD9E8D57ull * c2;
    const uint32_t d0 = (uint32_t)(q1 >> 32) ^ t.u2, d1 = (uint32_t)q1, d2 = c3 ^ t.u3;
    const unsigned long long r0 = 0xD2511F53ull * d0, r1 = 0xCD9E8D57ull * d2;
    uint4 c = make_uint4((uint32_t)(r1 >> 32) ^ d1 ^ a.rk0[2], (uint32_t)r1,
                         (uint32_t)(r0 >> 32) ^ t.u5, (uint32_t)r0);
#pragma unroll
    for (int r = 3; r < 10; ++r) {
        const unsigned long long s0 = 0xD2511F53ull * c.x, s1 = 0xCD9E8D57ull * c.z;
        c = make_uint4((uint32_t)(s1 >> 32) ^ c.y ^ a.rk0[r], (uint32_t)s1,
                       (uint32_t)(s0 >> 32) ^ c.w ^ a.rk1[r], (uint32_t)s0);
    }
    return c;
}

// First step and length of the group, or length 0 where an earlier group has
// run past its first step.  Uniform over the grid: nothing it reads changes
// before every block of the launch has passed here (k_tail's counters are
// written by the last block to finish).
struct Span {
    uint32_t s0;
    int len;
    bool closed;
};

template <bool DEP>
__device__ __forceinline__ Span group_span(const Args &a, uint32_t s0, int span, int m, bool no_src)
{
    Span sp{};
    sp.s0 = s0;
    if (__ldcg(&a.ctl->step) != s0) return sp;
    bool open = !no_src;
    if (!(a.flags & PIC_F_NO_SECONDARIES))
        for (int s = threadIdx.x; s < a.n_stacks; s += TPB) {
            const long long n = (long long)__ldcg(&a.cnt[s].n_slots);
            if (n > 0 && n < a.stacks[s].cap) open = true;
        }
    sp.closed = !cta_sync_or(open);
    // densities inside the group: as many steps as windows are held
    sp.len = sp.closed && !DEP ? span : (m < span ? m : span);
    return sp;
}

__device__ __forceinline__ uint2 *list_of(const GroupArgs &g, int j)
{
    uint2 *p = j < 4 ? (j < 2 ? g.list[0] : g.list[1]) : (j < 6 ? g.list[2] : g.list[3]);
    return p + (j & 1) * g.list_n;
}

// A slot's test word: the upper half of its threshold plus one, and the edge
// ahead as a half-precision number rounded down (its sign kept, that of zero
// too).  A random word below the threshold is below the test word.
__device__ __forceinline__ uint32_t test_word(uint32_t P, float edge)
{
    return (P ? (P & 0xFFFF0000u) + 0x10000u : 0u) | (uint32_t)__half_as_ushort(__float2half_rd(edge));
}

__device__ __forceinline__ float edge_of(uint32_t t)
{
    return __half2float(__ushort_as_half((unsigned short)(t & 0xFFFFu)));
}

struct GroupSmem {               // byte offsets in dynamic shared memory
    size_t ent, mv, q, t, j, n, gs, v, tiles, warps, total, per_warp;
};

// Shared memory of a warp: per slot the depth, the speed, the test word (upper
// half of the threshold, edge ahead) and, with densities, the bin word; rows of
// one lane's 4 Q slots padded by one vector, so that the vector accesses of
// consecutive lanes fall into different banks; 32 queue entries.
__host__ __device__ constexpr size_t warp_bytes(bool dep, int quads)
{
    return (size_t)32 * (quads + 1) * 16 * (dep ? 4 : 3) + 64;
}

__host__ __device__ inline GroupSmem group_smem(const Args &a, bool dep, int quads, int warps, int nd,
                                                int nj)
{
    GroupSmem o{};
    auto up = [](size_t x) { return (x + 15) & ~(size_t)15; };
    size_t p = 0;
    o.ent = p; p = up(p + (size_t)a.ftab_max * sizeof(FastEnt));
    o.mv = p; p = up(p + (size_t)a.ftab_max * 16);
    o.q = p; p = up(p + (size_t)a.tab_max * 4);
    o.t = p; p = up(p + (size_t)a.T_max * 4);
    o.j = p; p = up(p + (size_t)nj * a.jbin_max * 4);
    o.n = p; if (dep) p = up(p + (size_t)nd * (a.nbin_max + a.gbin_max) * 4);
    o.gs = p; if (dep) p = up(p + (size_t)nd * a.gbin_max * 4);
    o.v = p; if (dep && (a.flags & PIC_F_VELOCITY_MOMENTS)) p = up(p + (size_t)nd * a.gbin_max * 16);
    o.tiles = p; p = up(p + (size_t)(2 * a.n_stacks + 1) * 8);
    o.warps = p;
    o.per_warp = warp_bytes(dep, quads);
    o.total = p + (size_t)warps * o.per_warp;
    return o;
}

// Adds a block's nb bins (an even number) to those in memory, two at a time: the
// sums stay below 2^32, so a pair of bins is one 64-bit number without a carry
// between them, and the additions at the L2 are what this takes.  Every block
// starts at bins of its own.
__device__ __forceinline__ void flush_bins(uint32_t *dst, const uint32_t *src, int nb)
{
    const int np = nb / 2, rot = (int)((long long)blockIdx.x * np / (int)gridDim.x) & ~15;
    unsigned long long *d = reinterpret_cast<unsigned long long *>(dst);
    for (int i = threadIdx.x; i < np; i += (int)blockDim.x) {
        const int b = i + rot < np ? i + rot : i + rot - np;
        const uint32_t lo = src[2 * b], hi = src[2 * b + 1];
        if (lo | hi) atomicAdd(&d[b], (unsigned long long)lo | ((unsigned long long)hi << 32));
    }
}

// ---------------------------------------------------------------------------
// k_group.  A lane owns 4 Q consecutive slots of its warp's sub-tile of 128 Q
// slots.  The depth is kept in the direction of flight: z' = z for a carrier
// flying up and -z for one flying down, with |v mu| and the one layer edge
// ahead of it (hi or -lo), so that a step is two additions and one compare
// (rounding to nearest is symmetric: the bits are those of the signed
// flight).  A slot's test word holds the upper half of its threshold and the
// edge ahead rounded down to 16 bits: a superset of the events passes the
// sweep (exact for edges up to 2048 cells of 1 nm; 2^-16 too many tests), and the
// general step finds out.  Tables looked up per carrier and step instead cost
// six shared-memory wavefronts per warp where the own word costs one.  The
// edge's sign is the direction; a removed slot has speed 0, edge +inf and
// threshold 0.
// ---------------------------------------------------------------------------
template <bool DET, bool DEP, int Q>
__device__ __forceinline__ void phase_group(const Args &a, const GroupArgs &g, const Span sp)
{
    constexpr int S = 128 * Q;               // slots of a sub-tile
    constexpr int RQ = Q + 1;                // padded row of a lane, vectors
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ DevStack s_st;
    __shared__ uint32_t s_abs[GROUP_MAX];
    __shared__ unsigned long long s_led[9];
    __shared__ unsigned int s_next;

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, NT = (int)blockDim.x;
    const GroupSmem o = group_smem(a, DEP, Q, 0, g.nd, g.nj);
    FastEnt *s_ent = reinterpret_cast<FastEnt *>(smem + o.ent);
    uint4 *s_mv = reinterpret_cast<uint4 *>(smem + o.mv);    // speed, test words up and down, bin row
    uint32_t *s_Q = reinterpret_cast<uint32_t *>(smem + o.q);
    uint32_t *s_T = reinterpret_cast<uint32_t *>(smem + o.t);
    int32_t *s_J = reinterpret_cast<int32_t *>(smem + o.j);
    uint32_t *s_n = reinterpret_cast<uint32_t *>(smem + o.n);
    uint32_t *s_gs = reinterpret_cast<uint32_t *>(smem + o.gs);
    unsigned long long *s_v = reinterpret_cast<unsigned long long *>(smem + o.v);
    long long *s_tpref = reinterpret_cast<long long *>(smem + o.tiles);
    long long *s_nsl = s_tpref + a.n_stacks + 1;
    unsigned char *wmem = smem + o.warps + (size_t)warp * warp_bytes(DEP, Q);
    float4 *wz = reinterpret_cast<float4 *>(wmem), *ww = wz + 32 * RQ;
    uint4 *wt = reinterpret_cast<uint4 *>(ww + 32 * RQ), *wb = wt + 32 * RQ;      // wb: DEP only
    uint16_t *wq = reinterpret_cast<uint16_t *>(wt + (DEP ? 2 : 1) * 32 * RQ);

    const int cur = (int)__ldcg(&a.ctl->cur);
    const int ne = a.n_e;
    const float half = a.half_dt;
    const bool vmom = DEP && (a.flags & PIC_F_VELOCITY_MOMENTS);
    const uint32_t me = (uint32_t)a.moment_every;
    const int tj0 = (int)(sp.s0 / me);                       // the running window

    for (int s = tid; s < a.n_stacks; s += NT) s_nsl[s] = (long long)__ldcg(&a.cnt[s].n_slots);
    __syncthreads();
    if (tid == 0) {
        long long acc = 0;
        for (int s = 0; s < a.n_stacks; ++s) {
            s_tpref[s] = acc;
            acc += (s_nsl[s] + S - 1) / S;
        }
        s_tpref[a.n_stacks] = acc;
    }
    __syncthreads();
    const long long T = s_tpref[a.n_stacks];
    const long long t0 = chunk_lo(T, blockIdx.x, gridDim.x), t1 = chunk_lo(T, blockIdx.x + 1, gridDim.x);
    if (t0 >= t1) return;
    const int s_first = stack_of(s_tpref, a.n_stacks, t0);
    const int s_last = stack_of(s_tpref, a.n_stacks, t1 - 1);

    for (int s = s_first; s <= s_last; ++s) {
        const long long ta = t0 > s_tpref[s] ? t0 : s_tpref[s];
        const long long tb = t1 < s_tpref[s + 1] ? t1 : s_tpref[s + 1];
        if (ta >= tb) continue;
        // the stack's tables and the counts of this block's part of it
        __syncthreads();
        if (tid == 0) {
            s_st = a.stacks[s];
            s_next = 0u;
        }
        if (tid < 9) s_led[tid] = 0ull;
        for (int i = tid; i < GROUP_MAX; i += NT) s_abs[i] = 0u;
        __syncthreads();
        const DevStack &st = s_st;
        const int nc = st.n_cells, nf = nc + 1, nb = 2 * ne * nc, hb = nb + nc;
        for (int i = tid; i < st.ftab_n; i += NT) {
            const FastEnt e = a.fent[st.fent_off + i];
            s_ent[i] = e;
            // byte offset of the (spin, k) row of bins; removed slots have a row
            // of their own after the last
            const int k = i & ((1 << a.kb) - 1), sg = (i >> a.kb) & 1;
            s_mv[i] = make_uint4(__float_as_uint(e.v), test_word(e.P, e.hi), test_word(e.P, -e.lo),
                                 (uint32_t)(4 * (k >= 1 && k <= ne ? (sg * ne + k - 1) * nc : nb)));
        }
        for (int i = tid; i < st.tab_n; i += NT) s_Q[i] = a.ent[st.ent_off + i].Q;
        for (int i = tid; i < st.T_n; i += NT) s_T[i] = a.T_thr[st.T_off + i];
        for (int i = tid; i < g.nj * 2 * nf; i += NT) s_J[i] = 0;
        if (DEP) {
            for (int i = tid; i < g.nd * hb; i += NT) s_n[i] = 0u;
            for (int i = tid; i < g.nd * nc; i += NT) s_gs[i] = 0u;
            if (vmom)
                for (int i = tid; i < g.nd * 2 * nc; i += NT) s_v[i] = 0ull;
        }
        __syncthreads();
        const uint32_t ctr_hi = (uint32_t)(a.stack_base + s) << 16;
        const int nsl = (int)s_nsl[s];
        const bool full = s_nsl[s] >= st.cap;
        float *Z = a.z[cur] + st.base;
        float *MU = a.mu[cur] + 2 * st.base;
        const unsigned int n_sub = (unsigned int)(tb - ta);

        for (;;) {
            unsigned int u = 0;
            if (lane == 0) u = atomicAdd(&s_next, 1u);
            u = __shfl_sync(0xffffffffu, u, 0);
            if (u >= n_sub) break;
            const int sub = (int)(ta - s_tpref[s]) + (int)u;     // sub-tile of the stack
            const int slot0 = sub * S;
            const int nvalid = nsl - slot0;                      // at least 1
            const bool ragged = nvalid < S;
            // ---- load: quads of consecutive lanes are consecutive in memory
#pragma unroll
            for (int q = 0; q < Q; ++q) {
                const int i4 = (q * 32 + lane) * 4;
                const float4 z4 = *reinterpret_cast<const float4 *>(Z + slot0 + i4);
                const uint4 *mp = reinterpret_cast<const uint4 *>(MU + 2 * (long long)(slot0 + i4));
                const uint4 m0 = mp[0], m1 = mp[1];
                const float zi[4] = {z4.x, z4.y, z4.z, z4.w};
                const uint32_t mi[4] = {m0.x, m0.z, m1.x, m1.z};
                const uint32_t pi[4] = {m0.y, m0.w, m1.y, m1.w};
                float zo[4], wo[4];
                uint32_t to[4], bo[4];
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    const uint32_t pk = ragged && i4 + c >= nvalid ? 0u : pi[c];
                    const uint4 e = s_mv[fast_index(a, pk)];
                    const float w = __fmul_rn(__uint_as_float(e.x), __uint_as_float(mi[c]));
                    const bool dn = w < 0.f;
                    zo[c] = dn ? -zi[c] : zi[c];
                    wo[c] = dn ? -w : w;
                    to[c] = dn ? e.z : e.y;
                    if (DEP) bo[c] = e.w | ((pk & 0xFFu) ? (pk << 11) & 0xFF000000u : 0u);
                }
                const int i = q * 32 + lane, v = (i / Q) * RQ + i % Q;
                wz[v] = make_float4(zo[0], zo[1], zo[2], zo[3]);
                ww[v] = make_float4(wo[0], wo[1], wo[2], wo[3]);
                wt[v] = make_uint4(to[0], to[1], to[2], to[3]);
                if (DEP) wb[v] = make_uint4(bo[0], bo[1], bo[2], bo[3]);
            }
            __syncwarp();
            const uint32_t quad0 = (uint32_t)(slot0 >> 2) + (uint32_t)(lane * Q);
            float4 *rz = wz + lane * RQ;
            const float4 *rw = ww + lane * RQ;
            const uint4 *rt = wt + lane * RQ, *rb = wb + lane * RQ;
            // the lane's counts for this sub-tile: at most 64 x 32 items
            uint32_t c_hit = 0, c_chg = 0, c_abs = 0, c_bath = 0, c_qdrop = 0, n_event = 0;

#pragma unroll 1
            for (int j = 0; j < sp.len; ++j) {
                const uint32_t step = sp.s0 + (uint32_t)j;
                const TestKey tk = test_key(a, ctr_hi, step);
                const bool dep = DEP && (step + 1) % me == 0;
                const int hd = (int)(step / me) - tj0;       // window held at hd
                uint32_t *h_n = s_n + hd * hb, *h_gs = s_gs + hd * nc;
                unsigned long long *h_v = s_v + hd * 2 * nc;
                const uint32_t a_n = smem_addr(h_n) - 4u * 0x4B000000u, a_gs = smem_addr(h_gs) - 4u * 0x4B000000u;
                const uint32_t cl_max = 0x4B000000u + (uint32_t)(nc - 1);
                // ---- the step of every slot that meets no boundary and does
                // not scatter; the others keep their start and are marked
                uint32_t mask = 0;
                auto sweep = [&](auto depc, auto velc) {
                    constexpr bool D = decltype(depc)::value, V = decltype(velc)::value;
#pragma unroll (Q < UNROLL ? Q : UNROLL)
                    for (int q = 0; q < Q; ++q) {
                        const uint4 x4 = philox_test(quad0 + (uint32_t)q, tk, a);
                        const float4 z4 = rz[q], w4 = rw[q];
                        const uint4 t4 = rt[q];
                        const float zi[4] = {z4.x, z4.y, z4.z, z4.w}, wi[4] = {w4.x, w4.y, w4.z, w4.w};
                        const uint32_t ti[4] = {t4.x, t4.y, t4.z, t4.w}, xi[4] = {x4.x, x4.y, x4.z, x4.w};
                        uint4 b4 = make_uint4(0u, 0u, 0u, 0u);
                        if (D) b4 = rb[q];
                        const uint32_t bi[4] = {b4.x, b4.y, b4.z, b4.w};
                        float zo[4];
                        uint32_t nib = 0;
#pragma unroll
                        for (int c = 0; c < 4; ++c) {
                            const float z2 = fly<DET>(fly<DET>(zi[c], wi[c], half), wi[c], half);
                            const bool slow = (z2 > edge_of(ti[c])) | (xi[c] < ti[c]);
                            zo[c] = slow ? zi[c] : z2;
                            if (slow) nib |= 1u << c;
                            if (D) {
                                // the cell's index plus the exponent bits of
                                // 2^23, which a_n and a_gs have taken off
                                const uint32_t cl = min((uint32_t)__float_as_int(
                                                            __fmaf_rd(fabsf(z2), a.inv_dz, 8388608.0f)), cl_max);
                                red_shared(a_n + (bi[c] & 0xFFFFFFu) + 4u * cl, slow ? 0u : 1u);
                                red_shared(a_gs + 4u * cl, slow ? 0u : bi[c] >> 24);
                                if (V && !slow && (bi[c] & 0xFFFFFFu) < (uint32_t)(4 * nb)) {
                                    const long long v = vel_q(wi[c]);
                                    add_u64_split(&h_v[((bi[c] & 0xFFFFFFu) >= (uint32_t)(4 * ne * nc) ? nc : 0) +
                                                       (int)(cl - 0x4B000000u)],
                                                  (unsigned long long)((ti[c] & 0x8000u) ? -v : v));
                                }
                            }
                        }
                        mask |= nib << (4 * q);
                        rz[q] = make_float4(zo[0], zo[1], zo[2], zo[3]);
                    }
                };
                if (!DEP || !dep) sweep(std::false_type{}, std::false_type{});
                else if (!vmom) sweep(std::true_type{}, std::false_type{});
                else sweep(std::true_type{}, std::true_type{});
                // ---- the general step of the marked slots, 32 at a time in slot order
                const uint32_t cnt = (uint32_t)__popc(mask);
                uint32_t incl = cnt;
#pragma unroll
                for (int d = 1; d < 32; d <<= 1) {
                    const uint32_t y = __shfl_up_sync(0xffffffffu, incl, d);
                    if (lane >= d) incl += y;
                }
                const uint32_t total = __shfl_sync(0xffffffffu, incl, 31);
                uint32_t n_spawn = 0;
#pragma unroll 1
                for (uint32_t b0 = 0; b0 < total; b0 += 32u) {
                    {
                        uint32_t idx = incl - cnt - b0, mm = mask;   // below 0 wraps past 32
                        while (mm) {
                            const int bit = __ffs(mm) - 1;
                            mm &= mm - 1u;
                            if (idx < 32u) wq[idx] = (uint16_t)(lane * (4 * Q) + bit);
                            ++idx;
                        }
                    }
                    __syncwarp();
                    bool act = b0 + (uint32_t)lane < total;
                    const int p = act ? (int)wq[lane] : 0;           // slot within the sub-tile
                    act = act && p < nvalid;        // (memory past the stack's slots holds old records)
                    const int pv = ((p >> 2) / Q * RQ + (p >> 2) % Q) * 4 + (p & 3);
                    const int slot = slot0 + p;
                    uint2 *mps = reinterpret_cast<uint2 *>(MU + 2 * (long long)slot);
                    float z = 0.f, mu = 1.f;
                    uint32_t pk = 1u;
                    if (act) {
                        const uint2 mp = *mps;
                        mu = __uint_as_float(mp.x);
                        pk = mp.y;
                        z = reinterpret_cast<const float *>(wz)[pv];
                    }
                    const float mu_in = mu;
                    const uint32_t pk_in = pk;
                    int k = (int)(pk & 0xFFu), layer = (int)((pk >> 9) & 0xFu);
                    const int sg = (int)((pk >> 8) & 1u);
                    FastEnt e = s_ent[(((layer * 2 + sg) << a.kb) + k)];
                    // What the sweep suspected, settled: the first boundary of
                    // the step, if any, and the test.  The word that comes next
                    // is known but for a carrier that scatters before it meets
                    // its boundary (it draws again), so both Philox calls run
                    // side by side.
                    bool dead = false, second, pend = false;
                    float tau = half, zb;
                    int hit = 0;
                    uint32_t xs, sub_;
                    uint4 r;
                    bool up, ev;
                    {
                        const float w = __fmul_rn(e.v, mu);
                        z = w < 0.f ? -z : z;
                        const float z1 = fly<DET>(z, w, half), z2 = fly<DET>(z1, w, half);
                        up = mu > 0.f;
                        zb = up ? e.hi : e.lo;
                        const bool bnd = act && (up ? z2 > zb : z2 < zb);
                        second = !(bnd && (up ? z1 > zb : z1 < zb));     // first event in the second half
                        sub_ = !bnd ? SUB_EVT : SUB_IF + (second ? 16u : 0u);
                        const uint4 x = philox_test((uint32_t)slot >> 2, tk, a);
                        r = philox_rk(make_uint4((uint32_t)slot, ctr_hi, step, sub_), a);
                        xs = (slot & 2) ? ((slot & 1) ? x.w : x.z) : ((slot & 1) ? x.y : x.x);
                        const bool scat = xs < e.P;
                        ev = bnd || (act && scat);
                        if (!ev) {
                            z = z2;
                            sub_ = 0u;
                        } else {
                            if (second) z = z1;
                            if (bnd && second && scat) {
                                pend = true;
                                sub_ = 0u;
                            } else if (bnd) {
                                tau = __fsub_rn(half, __fdiv_rn(__fsub_rn(zb, z), w));
                                if (!(tau > 0.f)) tau = 0.f;
                                z = zb;
                            }
                        }
                    }
                    n_event += (uint32_t)__popc(__ballot_sync(0xffffffffu, ev));
                    bool done = !ev;
                    uint2 srec = make_uint2(0u, 0u);
                    // apply the word, fly until the next one is needed or the
                    // step is done; one Philox call serves every lane
#pragma unroll 1
                    for (;;) {
                        if (sub_ == SUB_EVT) {
                            const bool inel = r.y < s_Q[(layer * 2 + sg) * ne + (k - 1)];
                            if (k == 1 && (inel || (a.flags & PIC_F_LOWEST_BIN_ANY))) {
                                dead = done = true;
                                c_abs += 1u;
                                c_bath += 1u;
                            } else {
                                mu = mu_of(r.z);
                                if (inel) {
                                    const int kp = 1 + (int)__umulhi(r.w, (uint32_t)(k - 1));
                                    const int ks = k - kp;
                                    k = kp;
                                    e = s_ent[(((layer * 2 + sg) << a.kb) + k)];
                                    if (a.flags & PIC_F_NO_SECONDARIES) {
                                        c_bath += (uint32_t)ks;
                                    } else if (full) {
                                        c_chg += 1u << 16;                   // dropped
                                        c_qdrop += (uint32_t)ks;
                                        if (a.flags & PIC_F_STRICT_CAPACITY)
                                            atomicCAS(&a.ctl->status, 0u, (unsigned int)PIC_ERR_CAPACITY);
                                    } else {
                                        srec = make_uint2(__float_as_uint(z),
                                                          (uint32_t)ks | ((uint32_t)layer << 8) |
                                                              (((pk >> 13) & 0xFFu) << 12) | ((uint32_t)p << 20));
                                    }
                                }
                            }
                        } else if (sub_ != 0u) {
                            // at the boundary zb
                            ++hit;
                            if (up ? layer == st.n_layers - 1 : layer == 0) {        // vacuum
                                mu = -mu;
                            } else {
                                const int iface = up ? layer : layer - 1, dir = up ? 0 : 1;
                                c_hit += 1u;
                                if ((a.flags & PIC_F_TRANSPARENT) ||
                                    r.x < s_T[((iface * 2 + dir) * 2 + sg) * ne + (k - 1)]) {
                                    layer += up ? 1 : -1;
                                    c_hit += 1u << 16;                       // transmitted
                                    e = s_ent[(((layer * 2 + sg) << a.kb) + k)];
                                } else {
                                    mu = -mu;
                                }
                            }
                        }
                        sub_ = 0u;
                        if (!done) {
                            if (pend) {
                                pend = false;
                                sub_ = SUB_EVT;
                            } else {
#pragma unroll 1
                                for (;;) {
                                    const float w = __fmul_rn(e.v, mu);
                                    const float z1 = fly<DET>(z, w, tau);
                                    up = mu > 0.f;
                                    zb = up ? e.hi : e.lo;
                                    const bool cross = up ? z1 > zb : z1 < zb;
                                    if (!cross || hit == PIC_MAX_HITS) {
                                        if (cross) c_abs += 1u << 16;        // truncated
                                        z = cross ? zb : z1;
                                        if (second) { done = true; break; }
                                        // the test at mid-step
                                        second = true;
                                        tau = half;
                                        hit = 0;
                                        if (xs < e.P) { sub_ = SUB_EVT; break; }
                                        continue;
                                    }
                                    tau = __fsub_rn(tau, __fdiv_rn(__fsub_rn(zb, z), w));
                                    if (!(tau > 0.f)) tau = 0.f;
                                    z = zb;
                                    sub_ = SUB_IF + (second ? 16u : 0u) + (uint32_t)hit;
                                    break;
                                }
                            }
                        }
                        if (!__any_sync(0xffffffffu, sub_ != 0u)) break;
                        r = philox_rk(make_uint4((uint32_t)slot, ctr_hi, step, sub_), a);
                    }
                    // ---- results
                    if (act) {
                        pk = (pk & ~0x1FFFu) | ((uint32_t)sg << 8) | ((uint32_t)layer << 9);
                        if (dead) {
                            const int ce = cell_at(z, a.inv_dz, nc);
                            e.v = 0.f;
                            atomicAdd(&s_J[hd * 2 * nf + sg * nf + ce], -1);
                            atomicAdd(&s_abs[j], 1u);
                            if (a.w[0])
                                atomicAdd(reinterpret_cast<unsigned long long *>(a.bdw) + st.J_off +
                                              ((long long)(tj0 + hd) * 2 + sg) * nf + ce,
                                          0ull - (unsigned long long)a.w[cur][st.base + slot]);
                        } else {
                            pk |= (uint32_t)k;
                        }
                        const float w = __fmul_rn(e.v, mu);
                        const bool dn = w < 0.f;
                        const uint4 en = s_mv[fast_index(a, pk)];
                        reinterpret_cast<float *>(wz)[pv] = dn ? -z : z;
                        reinterpret_cast<float *>(ww)[pv] = dn ? -w : w;
                        reinterpret_cast<uint32_t *>(wt)[pv] = dn ? en.z : en.y;
                        if (DEP) {
                            reinterpret_cast<uint32_t *>(wb)[pv] =
                                en.w | ((pk & 0xFFu) ? (pk << 11) & 0xFF000000u : 0u);
                            if (dep && (pk & 0xFFu)) {
                                const int ce = cell_at(z, a.inv_dz, nc);
                                atomicAdd(&h_n[(sg * ne + k - 1) * nc + ce], 1u);
                                atomicAdd(&h_gs[ce], (pk >> 13) & 0xFFu);
                                if (vmom) add_u64_split(&h_v[sg * nc + ce], (unsigned long long)vel_q(w));
                            }
                        }
                        if (__float_as_uint(mu) != __float_as_uint(mu_in) || pk != pk_in) {
                            c_chg += 1u;
                            *mps = make_uint2(__float_as_uint(mu), pk);
                        }
                    }
                    if (!sp.closed) {
                        const unsigned int sb = __ballot_sync(0xffffffffu, srec.y != 0u);
                        if (srec.y != 0u)
                            list_of(g, j)[st.base + slot0 + (int)n_spawn + __popc(sb & ((1u << lane) - 1u))] = srec;
                        n_spawn += (uint32_t)__popc(sb);
                    }
                    __syncwarp();
                }
                if (!sp.closed && lane == 0)
                    g.cnt[(long long)j * g.cnt_n + (st.base / S + sub)] = (uint16_t)n_spawn;
            }
            // ---- store the depths
#pragma unroll
            for (int q = 0; q < Q; ++q) {
                const int i4 = (q * 32 + lane) * 4;
                const int i = q * 32 + lane, v = (i / Q) * RQ + i % Q;
                const float4 z4 = wz[v];
                const uint4 t4 = wt[v];
                const float4 zo = make_float4(
                    __uint_as_float(__float_as_uint(z4.x) ^ ((t4.x & 0x8000u) << 16)),
                    __uint_as_float(__float_as_uint(z4.y) ^ ((t4.y & 0x8000u) << 16)),
                    __uint_as_float(__float_as_uint(z4.z) ^ ((t4.z & 0x8000u) << 16)),
                    __uint_as_float(__float_as_uint(z4.w) ^ ((t4.w & 0x8000u) << 16)));
                float *zp = Z + slot0 + i4;
                if (i4 + 4 <= nvalid) {
                    *reinterpret_cast<float4 *>(zp) = zo;
                } else {
                    if (i4 < nvalid) zp[0] = zo.x;
                    if (i4 + 1 < nvalid) zp[1] = zo.y;
                    if (i4 + 2 < nvalid) zp[2] = zo.z;
                }
            }
            // ---- the sub-tile's counts
            const uint32_t vals[8] = {c_abs & 0xFFFFu, c_bath, c_hit & 0xFFFFu, c_hit >> 16, c_abs >> 16,
                                      c_chg >> 16, c_qdrop, c_chg & 0xFFFFu};
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const uint32_t v = __reduce_add_sync(0xffffffffu, vals[q]);
                if (lane == 0 && v) atomicAdd(&s_led[q], (unsigned long long)v);
            }
            if (lane == 0) atomicAdd(&s_led[8], (unsigned long long)n_event);
            __syncwarp();
        }

        // ---- the block's counts of this stack
        __syncthreads();
        if (tid < 9 && s_led[tid]) {
            const int idx[9] = {L_ABSORBED, L_Q_BATH, L_IFACE_HITS, L_IFACE_TRANSMIT, L_TRUNCATED,
                                L_SPAWN_DROPPED, L_Q_DROPPED, L_CHANGED, L_EVENTFUL};
            atomicAdd(&a.cnt[s].led[idx[tid]], s_led[tid]);
        }
        for (int i = tid; i < sp.len; i += NT)
            if (s_abs[i]) atomicAdd(&g.abs[s * GROUP_MAX + i], s_abs[i]);
        int32_t *gB = a.bd_hist + st.J_off + (long long)tj0 * 2 * nf;
        for (int i = tid; i < g.nj * 2 * nf; i += NT) {
            const int v = s_J[i];
            if (v) atomicAdd(&gB[i], v);
        }
        if (DEP) {
            const int ndep = (int)((sp.s0 + (uint32_t)sp.len) / me) - tj0;   // windows ended
            uint32_t *gN = a.n_hist + st.n_off + (long long)tj0 * nb;
            unsigned long long *gG = a.g_hist + st.n_off / (2 * ne) + (long long)tj0 * nc;
            unsigned long long *gV = reinterpret_cast<unsigned long long *>(a.v_hist) + st.n_off / ne +
                                     (long long)tj0 * 2 * nc;
            for (int h = 0; h < ndep; ++h) {
                flush_bins(gN + (long long)h * nb, s_n + h * hb, nb);
                for (int i = tid; i < nc; i += NT) {
                    const uint32_t v = s_gs[h * nc + i];
                    if (v) atomicAdd(&gG[(long long)h * nc + i], (unsigned long long)v);
                }
                if (vmom)
                    for (int i = tid; i < 2 * nc; i += NT) {
                        const unsigned long long v = s_v[h * 2 * nc + i];
                        if (v) atomicAdd(&gV[(long long)h * 2 * nc + i], v);
                    }
            }
        }
    }
}

// The span is decided by the block's first TPB threads (the width of k_tail's
// blocks, which decide the same) and handed to the others.
template <bool DEP>
__device__ __forceinline__ Span block_span(const Args &a, uint32_t s0, int span, int m, bool no_src)
{
    __shared__ Span s_sp;
    if (threadIdx.x < TPB) {
        const Span sp = group_span<DEP>(a, s0, span, m, no_src);
        if (threadIdx.x == 0) s_sp = sp;
    }
    __syncthreads();
    return s_sp;
}

template <bool DET, bool DEP, int Q>
__global__ void __launch_bounds__(32 * GW_MAX, 1) k_group(const Args a, const GroupArgs g)
{
    const uint32_t s0 = (g.base ? __ldcg(g.base) : 0u) + (uint32_t)g.off;
    const Span sp = block_span<DEP>(a, s0, g.end - g.off, g.m, g.no_src != 0);
    if (sp.len != 0) phase_group<DET, DEP, Q>(a, g, sp);
}

// ---------------------------------------------------------------------------
// k_tail: the carriers created in the steps of an open group.  Every stack has
// blocks of its own (in proportion to its capacity) with a barrier among them;
// they know the counts of the lists, hence for each step the slot and id of
// every new carrier: the source's first half, the secondaries of the slots of
// the group's start (list order), those of the new carriers (slot order), the
// source's second half.  A new carrier takes the remaining steps of the group
// here.  Few carriers: direct, warp-aggregated sums in memory.
// ---------------------------------------------------------------------------
constexpr int TAIL_PIECE = 1024;     // sub-tiles whose counts are held at a time

// add 1 (or v) to *p, the calling lanes with the same address together
__device__ __forceinline__ void agg_add(uint32_t *p, int v)
{
    const unsigned int m = __match_any_sync(__activemask(), (unsigned long long)p);
    if ((int)(threadIdx.x & 31) == __ffs(m) - 1) atomicAdd(p, (uint32_t)(v * __popc(m)));
}

__device__ __forceinline__ void agg_sum(unsigned long long *p, uint32_t v)
{
    const unsigned int m = __match_any_sync(__activemask(), (unsigned long long)p);
    const uint32_t t = __reduce_add_sync(m, v);
    if ((int)(threadIdx.x & 31) == __ffs(m) - 1) atomicAdd(p, (unsigned long long)t);
}

// Barrier of the stack's nb blocks (all resident: a cooperative launch) in two
// halves, between which a block works on what needs no other block: one
// counter that only grows, `target` the arrivals that end this barrier.  One
// trip to memory to arrive, then polls; bounded in polls.  The second half is
// false, for the whole block, where the wait was given up: the lists and counts
// that it waited for cannot be read.
__device__ __forceinline__ void stack_arrive(unsigned int *bar)
{
    cta_sync();
    if (threadIdx.x == 0) asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(bar) : "memory");
}

__device__ __forceinline__ bool stack_wait(const Args &a, unsigned int *bar, unsigned int target)
{
    bool given_up = false;
    if (threadIdx.x == 0) {
        unsigned int it = 0, v;
        for (;;) {
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(bar) : "memory");
            if ((int)(v - target) >= 0) break;
            if (++it > a.spin_limit) {
                atomicMax(&a.ctl->status, (unsigned int)PIC_ERR_TIMEOUT);
                a.ctl->timeout_where = 7u;
                given_up = true;
                break;
            }
            if ((it & 63u) == 0 && timed_out(a)) {
                given_up = true;
                break;
            }
            if (it > 1024) __nanosleep(128);
        }
    }
    return !cta_sync_or(given_up);
}

struct TailChild {                   // a secondary before its slot is known
    float z, mu, zb, v;              // depth and direction after its half flight; where it was born; speed
    uint32_t pk, pslot;              // packed word without the id; the parent's slot
    uint32_t hits, trans, trunc;
};

struct TailStack {                   // what a tail block keeps of its stack
    const DevStack *st;
    int s, nc, nf, ne;
    uint32_t ctr_hi;
    float *Z, *MU;
    uint32_t *ID, *W;
    bool vmom;
    // SUMS: births minus removals, generation and velocity sums of the group's
    // windows (from tj0) in shared memory; else added in memory
    int tj0;
    int32_t *J;
    uint32_t *G;
    unsigned long long *V;
};

// Their shared memory.  In memory the sums fall on a few lines (115 cells: 7 lines
// of generation sums and 8 of births), whose additions one after another were
// most of what many new carriers cost: k_tail's part of 20 steps of 2e7 carriers
// that start at 1.5 eV, 1.7e7 secondaries, took 9.0 ms with densities every step
// (single steps' event and placement passes 5.1) and 4.5 ms without, now 1.9 and 1.4.
__host__ __device__ inline size_t tail_sums(const Args &a, int nd, int nj)
{
    const bool vmom = nd > 0 && (a.flags & PIC_F_VELOCITY_MOMENTS);
    return (size_t)nj * a.jbin_max * 4 + (size_t)nd * a.gbin_max * (vmom ? 20 : 4) + 8;
}

// the density, generation and velocity sums of one carrier at the end of window t
template <bool SUMS>
__device__ __forceinline__ void tail_deposit(const Args &a, const TailStack &x, int t, int sg, int k,
                                             uint32_t gen, float z, float w)
{
    const int c = cell_at(z, a.inv_dz, x.nc);
    agg_add(&a.n_hist[x.st->n_off + ((long long)t * 2 + sg) * x.ne * x.nc + (long long)(k - 1) * x.nc + c], 1);
    if (SUMS) atomicAdd(&x.G[(t - x.tj0) * x.nc + c], gen);
    else agg_sum(&a.g_hist[x.st->n_off / (2 * x.ne) + (long long)t * x.nc + c], gen);
    if (SUMS && x.vmom)
        add_u64_split(&x.V[((t - x.tj0) * 2 + sg) * x.nc + c], (unsigned long long)vel_q(w));
    else if (x.vmom)
        atomicAdd(reinterpret_cast<unsigned long long *>(a.v_hist) + x.st->n_off / x.ne +
                      ((long long)t * 2 + sg) * x.nc + c,
                  (unsigned long long)vel_q(w));
}

// a birth (+1) or removal (-1) in window t, with its weight
template <bool SUMS>
__device__ __forceinline__ void tail_change(const Args &a, const TailStack &x, int t, int sg, float z, int by, uint32_t w)
{
    const int c = cell_at(z, a.inv_dz, x.nc);
    const long long i = x.st->J_off + ((long long)t * 2 + sg) * x.nf + c;
    if (SUMS) atomicAdd(&x.J[((t - x.tj0) * 2 + sg) * x.nf + c], by);
    else agg_add(reinterpret_cast<uint32_t *>(&a.bd_hist[i]), by);
    if (a.w[0])
        atomicAdd(reinterpret_cast<unsigned long long *>(a.bdw) + i,
                  by > 0 ? (unsigned long long)w : 0ull - (unsigned long long)w);
}

// Source(dt/2): the carrier with id `id` in slot `slot`
template <bool SUMS>
__device__ __forceinline__ void tail_source(const Args &a, const TailStack &x, uint32_t step, int t,
                                            unsigned long long id, long long slot, bool deposit,
                                            unsigned long long &q, unsigned long long &wsum)
{
    const DevStack &st = *x.st;
    const uint32_t cy = (uint32_t)(id >> 32) | x.ctr_hi;
    const uint4 r0 = philox_rk(make_uint4((uint32_t)id, cy, step, SUB_INJ + 0), a);
    const uint4 r1 = philox_rk(make_uint4((uint32_t)id, cy, step, SUB_INJ + 1), a);
    // first entry whose threshold lies above the word (the last one otherwise)
    const uint32_t *thr = a.cdf_thr + st.cdf_off;
    int lo = 0, hi = st.n_cdf - 1;
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (r0.x < thr[mid]) hi = mid; else lo = mid + 1;
    }
    const int i = lo;
    const float z = __fmul_rn(__fadd_rn((float)a.cdf_cell[st.cdf_off + i], unit_of(r0.y)), a.dz);
    const uint32_t sg = r0.z < st.up_thr ? 0u : 1u;
    uint32_t k;
    if (st.e_mode == 1) {
        k = (uint32_t)(sg ? st.k_mono1 : st.k_mono0);
    } else if (st.has_ebias) {
        const uint32_t *kt = a.kthr + (long long)x.s * x.ne;
        k = 1u;
        while ((int)k < x.ne && !(r0.w < kt[k - 1])) ++k;
    } else {
        k = 1u + __umulhi(r0.w, (uint32_t)x.ne);
    }
    const uint32_t layer = (uint32_t)a.cdf_layer[st.cdf_off + i];
    const float mu = mu_of(r1.x);
    x.Z[slot] = z;
    *reinterpret_cast<uint2 *>(x.MU + 2 * slot) = make_uint2(
        __float_as_uint(mu), k | (sg << 8) | (layer << 9) | (1u << 13) | ((uint32_t)(id >> 32) << 21));
    x.ID[slot] = (uint32_t)id;
    q += k;
    uint32_t wq = 1u << 20;
    if (a.w[0]) {
        // weight p/q of the birth cell and bin (Eq. PIC), 2^-20 units
        const double wr = __dmul_rn(__dmul_rn(a.wcell[st.cdf_off + i], a.wbin[(long long)x.s * x.ne + k - 1]),
                                    1048576.0);
        wq = wr < 1.0 ? 1u : (wr > 4294967295.0 ? 0xFFFFFFFFu : __double2uint_rn(wr));
        x.W[slot] = wq;
        wsum += wq;
    }
    tail_change<SUMS>(a, x, t, (int)sg, z, 1, wq);
    if (deposit) {
        const float v = x.vmom ? a.ent[st.ent_off + (layer * 2 + sg) * x.ne + (k - 1)].v : 0.f;
        tail_deposit<SUMS>(a, x, t, (int)sg, (int)k, 1u, z, __fmul_rn(v, mu));
    }
}

// The static shared memory of phase_tail, one for both of its forms in k_run (with
// two of them it had room for fewer warps: 100 steps of 4e5 slots 0.83 -> 0.98 ms).
struct TailShared {
    DevStack st;
    float edge[PIC_MAX_LAYERS + 1];
    uint32_t p0[PIC_MAX_LAYERS];
    uint32_t pre[TAIL_PIECE + 1];
    uint32_t tot[GROUP_OPEN], mine[GROUP_OPEN];
    uint32_t tt[2];
    int w[TPB / 32], flag;
    unsigned long long r8[(TPB / 32) * 10];
};

__device__ __forceinline__ TailShared &tail_shared()
{
    __shared__ TailShared sh;
    return sh;
}

template <bool DET, bool SUMS>
__device__ __forceinline__ void phase_tail(const Args &a, const GroupArgs &g, const Span sp, bool no_src)
{
    extern __shared__ __align__(128) unsigned char smem[];
    TabEnt *s_ent = reinterpret_cast<TabEnt *>(smem);
    uint32_t *s_T = reinterpret_cast<uint32_t *>(s_ent + a.tab_max);
    TailShared &sh = tail_shared();
    DevStack &s_st = sh.st;
    auto &s_edge = sh.edge;
    auto &s_p0 = sh.p0;
    auto &s_pre = sh.pre;
    auto &s_tot = sh.tot;
    auto &s_mine = sh.mine;
    auto &s_tt = sh.tt;
    auto &s_w = sh.w;
    int &s_flag = sh.flag;
    auto &s_r8 = sh.r8;

    const int tid = threadIdx.x, lane = tid & 31;
    const int4 bl = g.blk[blockIdx.x];
    const int s = bl.x, ib = bl.y, nbk = bl.z, b0 = bl.w;
    unsigned int *bar = g.bar + 32 * s, bar_t = 0;       // the last block of the launch resets it
    unsigned long long psum = 0, adds = 0;       // advanced carriers and created ones, without removals
    const unsigned long long live0 = __ldcg(&a.cnt[s].live);
    const long long n0 = (long long)__ldcg(&a.cnt[s].n_slots);
    unsigned long long nid = __ldcg(&a.cnt[s].next_id);
    long long nsl = n0;

    if (sp.closed) {
        psum = (unsigned long long)sp.len * live0;
    } else {
        Stk S{};
        load_stack(a, s, S, &s_st, s_ent, s_T, s_edge, s_p0);
        const DevStack &st = s_st;
        const int cur = (int)__ldcg(&a.ctl->cur);
        const uint32_t me = (uint32_t)a.moment_every;
        TailStack x;
        x.st = &s_st; x.s = s; x.nc = st.n_cells; x.nf = st.n_cells + 1; x.ne = a.n_e;
        x.ctr_hi = S.ctr_hi;
        x.Z = a.z[cur] + st.base;
        x.MU = a.mu[cur] + 2 * st.base;
        x.ID = a.id[cur] + st.base;
        x.W = a.w[0] ? a.w[cur] + st.base : nullptr;
        x.vmom = (a.flags & PIC_F_VELOCITY_MOMENTS) != 0;
        x.tj0 = (int)(sp.s0 / me);
        // the windows that the group's steps lie in, and of these the ones that may end
        const int wj = (int)((sp.s0 + (uint32_t)sp.len - 1u) / me) - x.tj0 + 1, wd = wj < g.nd ? wj : g.nd;
        const int nv = x.vmom ? wd * 2 * x.nc : 0, nj = wj * 2 * x.nf, ng = wd * x.nc;
        if (SUMS) {
            x.V = reinterpret_cast<unsigned long long *>((reinterpret_cast<uintptr_t>(s_T + a.T_max) + 7) & ~uintptr_t(7));
            x.J = reinterpret_cast<int32_t *>(x.V + nv);
            x.G = reinterpret_cast<uint32_t *>(x.J + nj);
            for (int i = tid; i < nv; i += TPB) x.V[i] = 0ull;
            for (int i = tid; i < nj + ng; i += TPB) x.J[i] = 0;
        }
        const float half = a.half_dt;
        const bool dep_in = g.nd > 0;            // densities deposited inside the group
        const long long U = (n0 + g.sub - 1) / g.sub;      // sub-tiles of the group's start
        const long long u0 = U * ib / nbk, u1 = U * (ib + 1) / nbk;
        const uint16_t *cnt = g.cnt + st.base / g.sub;
        Tally ty{};
        uint32_t kept_here = 0;
        unsigned long long q_src = 0, w_src = 0, n_event = 0;

        // the lists' counts: this block's, those before it, all
        if (tid < GROUP_OPEN) s_tot[tid] = s_mine[tid] = 0u;
        cta_sync();
#pragma unroll 1
        for (int j = 0; j < sp.len; ++j) {
            uint32_t c = 0;
            for (long long u = u0 + tid; u < u1; u += TPB) c += cnt[j * g.cnt_n + u];
            c = __reduce_add_sync(0xffffffffu, c);
            if (lane == 0 && c) atomicAdd(&s_tot[j], c);
        }
        cta_sync();
        if (tid < sp.len) g.bsum[(long long)(b0 + ib) * GROUP_OPEN + tid] = s_tot[tid];
        stack_arrive(bar);

        // A secondary from its record; it depends on nothing but the record.
        auto make = [&](uint32_t step, const uint2 rec, long long pslot) -> TailChild {
            const int ks = (int)(rec.y & 0xFFu);
            int layer = (int)((rec.y >> 8) & 0xFu);
            const uint32_t g0 = (rec.y >> 12) & 0xFFu, gen = g0 < 255u ? g0 + 1u : 255u;
            const uint4 y = philox_rk(make_uint4((uint32_t)pslot, x.ctr_hi, step, SUB_SEC), a);
            const int sg = y.x < s_p0[layer] ? 0 : 1;
            TailChild c;
            c.zb = __uint_as_float(rec.x);
            c.z = c.zb;
            c.mu = mu_of(y.y);
            float lo = s_edge[layer], hi = s_edge[layer + 1];
            TabEnt e = s_ent[(layer * 2 + sg) * x.ne + (ks - 1)];
            Tally tq{};
            flight<DET>(a, S, c.z, c.mu, layer, e, lo, hi, sg, ks, half, (uint32_t)pslot, x.ctr_hi, step,
                        SUB_SIF, tq);
            c.v = e.v;
            c.pk = (uint32_t)ks | ((uint32_t)sg << 8) | ((uint32_t)layer << 9) | (gen << 13);
            c.pslot = (uint32_t)pslot;
            c.hits = tq.hits;
            c.trans = tq.trans;
            c.trunc = tq.trunc;
            return c;
        };
        // The records of step j in sub-tiles [p0, p0 + np) of this block: a prefix
        // of their counts in s_pre; the number of records.
        auto prefix = [&](int j, long long p0, int np) -> int {
            int c[TAIL_PIECE / TPB], sum = 0;
#pragma unroll
            for (int q = 0; q < TAIL_PIECE / TPB; ++q) {
                const int i = tid * (TAIL_PIECE / TPB) + q;
                c[q] = i < np ? (int)cnt[j * g.cnt_n + p0 + i] : 0;
                sum += c[q];
            }
            int excl;
            const int tot = block_scan(sum, excl, s_w);
            if (tot == 0) return 0;
#pragma unroll
            for (int q = 0; q < TAIL_PIECE / TPB; ++q) {
                s_pre[tid * (TAIL_PIECE / TPB) + q] = (uint32_t)excl;
                excl += c[q];
            }
            cta_sync();
            return tot;
        };
        auto record = [&](int j, long long p0, int r) -> TailChild {
            int lo = 0, hi = TAIL_PIECE - 1;         // last sub-tile with prefix <= r
            while (lo < hi) {
                const int mid = (lo + hi + 1) >> 1;
                if (s_pre[mid] <= (uint32_t)r) lo = mid; else hi = mid - 1;
            }
            const long long sl0 = (p0 + lo) * g.sub;
            const uint2 rec = __ldcg(&(list_of(g, j) + st.base)[sl0 + (r - (int)s_pre[lo])]);
            return make(sp.s0 + (uint32_t)j, rec, sl0 + (rec.y >> 20));
        };
        // The first TPB secondaries of the next step (most often all) are made
        // while the block waits for the others at the barrier before it.
        const int np0 = (int)(u1 - u0 < TAIL_PIECE ? u1 - u0 : TAIL_PIECE);
        TailChild ch{};
        int tot0 = 0;
        auto prepare = [&](int j) {
            tot0 = prefix(j, u0, np0);
            if (tid < tot0) ch = record(j, u0, tid);
        };
        prepare(0);
        if (!stack_wait(a, bar, bar_t += (unsigned int)nbk)) return;
        if (tid < GROUP_OPEN) s_tot[tid] = 0u;
        cta_sync();
        for (int i = tid; i < nbk * sp.len; i += TPB) {
            const int b = i / sp.len, j = i % sp.len;
            const uint32_t v = __ldcg(&g.bsum[(long long)(b0 + b) * GROUP_OPEN + j]);
            if (v) {
                atomicAdd(&s_tot[j], v);
                if (b < ib) atomicAdd(&s_mine[j], v);
            }
        }
        cta_sync();

#pragma unroll 1
        for (int j = 0; j < sp.len; ++j) {
            const uint32_t step = sp.s0 + (uint32_t)j;
            const int t = (int)(step / me);
            const bool dep = dep_in && (step + 1) % me == 0;
            uint2 *list = list_of(g, j) + st.base;
            // ---- the source's first half: slots [nsl, nsl + i0)
            const long long in0 = no_src ? 0 : a.inj[st.inj_off + 2 * (long long)step];
            const long long r0 = st.cap - nsl;
            const long long i0 = in0 < r0 ? in0 : (r0 > 0 ? r0 : 0);
            psum += live0 + adds + (unsigned long long)i0;
            // ---- the step of the new carriers, in slot order: block ib's share
            const long long L = nsl + i0 - n0;
            const long long x0 = L * ib / nbk, x1 = L * (ib + 1) / nbk;
            uint32_t mine = 0;
            float z_next = 0.f;              // the next carrier's record, asked for one round ahead
            uint2 mp_next = make_uint2(0u, 0u);
            auto ask = [&](long long xi) {
                if (xi < x1 && n0 + xi < nsl) {
                    z_next = __ldcg(x.Z + n0 + xi);
                    mp_next = __ldcg(reinterpret_cast<const uint2 *>(x.MU + 2 * (n0 + xi)));
                }
            };
            ask(x0 + tid);
#pragma unroll 1
            for (long long xi = x0 + tid; xi < x1; xi += TPB) {
                const long long slot = n0 + xi;
                float z = z_next;
                uint2 mp = mp_next;
                ask(xi + TPB);
                if (slot >= nsl) {
                    tail_source<SUMS>(a, x, step, t, nid + (unsigned long long)(slot - nsl), slot, false, q_src, w_src);
                    z = __ldcg(x.Z + slot);
                    mp = __ldcg(reinterpret_cast<const uint2 *>(x.MU + 2 * slot));
                }
                float mu = __uint_as_float(mp.x);
                uint32_t pk = mp.y;
                uint2 rec = make_uint2(0u, 0u);
                int k = (int)(pk & 0xFFu);
                if (k != 0) {
                    const int sg = (int)((pk >> 8) & 1u);
                    int layer = (int)((pk >> 9) & 0xFu);
                    TabEnt e = s_ent[(layer * 2 + sg) * x.ne + (k - 1)];
                    float lo = s_edge[layer], hi = s_edge[layer + 1];
                    const uint4 xg = philox_rk(make_uint4((uint32_t)(slot >> 2), x.ctr_hi, step, SUB_TEST), a);
                    const uint32_t xs = (slot & 2) ? ((slot & 1) ? xg.w : xg.z) : ((slot & 1) ? xg.y : xg.x);
                    const float w = __fmul_rn(e.v, mu);
                    const float z2 = fly<DET>(fly<DET>(z, w, half), w, half);
                    bool dead = false;
                    float w_end = w;
                    if (!((z2 > hi) | (z2 < lo) | (xs < e.P))) {
                        z = z2;
                    } else {
                        ++n_event;
                        flight<DET>(a, S, z, mu, layer, e, lo, hi, sg, k, half, (uint32_t)slot, x.ctr_hi,
                                    step, SUB_IF, ty);
                        if (xs < e.P) {
                            const uint4 r = philox_rk(make_uint4((uint32_t)slot, x.ctr_hi, step, SUB_EVT), a);
                            const bool inel = r.y < e.Q;
                            if (k == 1 && (inel || (a.flags & PIC_F_LOWEST_BIN_ANY))) {
                                dead = true;
                                ++ty.absorbed;
                                ++ty.bath;
                            } else {
                                mu = mu_of(r.z);
                                if (inel) {
                                    const int kp = 1 + (int)__umulhi(r.w, (uint32_t)(k - 1));
                                    const int ks = k - kp;
                                    k = kp;
                                    e = s_ent[(layer * 2 + sg) * x.ne + (k - 1)];
                                    if (a.flags & PIC_F_NO_SECONDARIES) {
                                        ty.bath += (uint32_t)ks;
                                    } else {
                                        // (a full buffer drops it at its placement)
                                        rec = make_uint2(__float_as_uint(z),
                                                         (uint32_t)ks | ((uint32_t)layer << 8) |
                                                             (((pk >> 13) & 0xFFu) << 12));
                                        ++mine;
                                    }
                                }
                            }
                        }
                        if (dead) {
                            pk = (pk & ~0x1FFFu) | ((uint32_t)sg << 8) | ((uint32_t)layer << 9);
                            tail_change<SUMS>(a, x, t, sg, z, -1, a.w[0] ? x.W[slot] : 0u);
                            atomicAdd(&g.abs[s * GROUP_MAX + j], 1u);
                        } else {
                            flight<DET>(a, S, z, mu, layer, e, lo, hi, sg, k, half, (uint32_t)slot, x.ctr_hi,
                                        step, SUB_IF + 16, ty);
                            pk = (pk & ~0x1FFFu) | (uint32_t)k | ((uint32_t)sg << 8) | ((uint32_t)layer << 9);
                            w_end = __fmul_rn(e.v, mu);
                        }
                        if (__float_as_uint(mu) != mp.x || pk != mp.y) {
                            ++ty.changed;
                            *reinterpret_cast<uint2 *>(x.MU + 2 * slot) = make_uint2(__float_as_uint(mu), pk);
                        }
                    }
                    x.Z[slot] = z;
                    if (dep && !dead) tail_deposit<SUMS>(a, x, t, sg, k, (pk >> 13) & 0xFFu, z, w_end);
                }
                list[slot] = rec;
            }
            // ---- secondaries of the new carriers per block
            uint32_t tail_tot = 0, tail_pre = 0;
            if (L > 0) {
                if (tid < 2) s_tt[tid] = 0u;
                cta_sync();
                mine = __reduce_add_sync(0xffffffffu, mine);
                if (lane == 0 && mine) atomicAdd(&s_tt[0], mine);
                cta_sync();
                if (tid == 0) g.tsum[(long long)(b0 + ib) * GROUP_OPEN + j] = s_tt[0];
                stack_arrive(bar);
                if (!stack_wait(a, bar, bar_t += (unsigned int)nbk)) return;
                if (tid == 0) s_tt[0] = 0u;
                cta_sync();
                for (int b = tid; b < nbk; b += TPB) {
                    const uint32_t v = __ldcg(&g.tsum[(long long)(b0 + b) * GROUP_OPEN + j]);
                    if (v) {
                        atomicAdd(&s_tt[0], v);
                        if (b < ib) atomicAdd(&s_tt[1], v);
                    }
                }
                cta_sync();
                tail_tot = s_tt[0];
                tail_pre = s_tt[1];
                cta_sync();
            }
            nid += (unsigned long long)i0;
            nsl += i0;
            if (ib == 0 && tid == 0 && in0 > 0) {
                unsigned long long *led = a.cnt[s].led;
                if (i0) atomicAdd(&led[L_INJECTED], (unsigned long long)i0);
                if (in0 > i0) atomicAdd(&led[L_INJECT_DROPPED], (unsigned long long)(in0 - i0));
            }
            // ---- the slots and ids of the step's secondaries
            const long long room = st.cap - nsl;
            const long long total = (long long)s_tot[j] + tail_tot;
            const long long kept = total < room ? total : (room > 0 ? room : 0);
            auto place = [&](const TailChild &c, long long rank) {
                const int ks = (int)(c.pk & 0xFFu), sg = (int)((c.pk >> 8) & 1u);
                if (rank >= room) {
                    ++ty.spawn_drop;
                    ty.q_drop += (uint32_t)ks;
                    return;
                }
                ty.hits += c.hits;
                ty.trans += c.trans;
                ty.trunc += c.trunc;
                const unsigned long long id = nid + (unsigned long long)rank;
                const long long d = nsl + rank;
                x.Z[d] = c.z;
                *reinterpret_cast<uint2 *>(x.MU + 2 * d) =
                    make_uint2(__float_as_uint(c.mu), c.pk | ((uint32_t)(id >> 32) << 21));
                x.ID[d] = (uint32_t)id;
                ++kept_here;
                uint32_t wp = 0;
                if (a.w[0]) {
                    wp = __ldcg(&x.W[c.pslot]);
                    x.W[d] = wp;
                }
                tail_change<SUMS>(a, x, t, sg, c.zb, 1, wp);
                if (dep) tail_deposit<SUMS>(a, x, t, sg, ks, (c.pk >> 13) & 0xFFu, c.z, __fmul_rn(c.v, c.mu));
            };
            if (s_tot[j] > 0) {
                // a thread per record, in pieces of the block's sub-tiles
                long long run = s_mine[j];
                if (tid < tot0) place(ch, run + tid);
#pragma unroll 1
                for (int r = tid + TPB; r < tot0; r += TPB) place(record(j, u0, r), run + r);
                run += tot0;
                for (long long p0 = u0 + TAIL_PIECE; p0 < u1; p0 += TAIL_PIECE) {
                    cta_sync();
                    const int tot = prefix(j, p0, (int)(u1 - p0 < TAIL_PIECE ? u1 - p0 : TAIL_PIECE));
#pragma unroll 1
                    for (int r = tid; r < tot; r += TPB) place(record(j, p0, r), run + r);
                    run += tot;
                }
            }
            if (tail_tot > 0) {
                long long run = (long long)s_tot[j] + tail_pre;
                for (long long p0 = x0; p0 < x1; p0 += TPB) {
                    const long long slot = n0 + p0 + tid;
                    const uint2 rec = p0 + tid < x1 ? list[slot] : make_uint2(0u, 0u);
                    int excl;
                    const int tot = block_scan((rec.y & 0xFFu) != 0u ? 1 : 0, excl, s_w);
                    if ((rec.y & 0xFFu) != 0u) place(make(step, rec, slot), run + excl);
                    run += tot;
                }
            }
            if (ib == 0 && tid == 0 && total > room && (a.flags & PIC_F_STRICT_CAPACITY))
                atomicCAS(&a.ctl->status, 0u, (unsigned int)PIC_ERR_CAPACITY);
            nsl += kept;
            nid += (unsigned long long)kept;
            // ---- the source's second half: slots [nsl, nsl + i1), not moved
            const long long in1 = no_src ? 0 : a.inj[st.inj_off + 2 * (long long)step + 1];
            const long long r1 = st.cap - nsl;
            const long long i1 = in1 < r1 ? in1 : (r1 > 0 ? r1 : 0);
            for (long long xi = (long long)ib * TPB + tid; xi < i1; xi += (long long)nbk * TPB)
                tail_source<SUMS>(a, x, step, t, nid + (unsigned long long)xi, nsl + xi, dep, q_src, w_src);
            if (ib == 0 && tid == 0) {
                unsigned long long *led = a.cnt[s].led;
                if (i1) atomicAdd(&led[L_INJECTED], (unsigned long long)i1);
                if (in1 > i1) atomicAdd(&led[L_INJECT_DROPPED], (unsigned long long)(in1 - i1));
                if ((in0 > i0 || in1 > i1) && (a.flags & PIC_F_STRICT_CAPACITY))
                    atomicCAS(&a.ctl->status, 0u, (unsigned int)PIC_ERR_CAPACITY);
            }
            nsl += i1;
            nid += (unsigned long long)i1;
            adds += (unsigned long long)(i0 + kept + i1);
            // the carriers written here are read by other blocks in the next step
            if (j + 1 < sp.len) {
                if (nsl > n0) stack_arrive(bar); else cta_sync();
                prepare(j + 1);
                if (nsl > n0 && !stack_wait(a, bar, bar_t += (unsigned int)nbk)) return;
            }
        }
        // ---- the block's sums and counts
        if (SUMS) {
            cta_sync();
            int32_t *gJ = a.bd_hist + st.J_off + (long long)x.tj0 * 2 * x.nf;
            unsigned long long *gG = a.g_hist + st.n_off / (2 * x.ne) + (long long)x.tj0 * x.nc;
            unsigned long long *gV = reinterpret_cast<unsigned long long *>(a.v_hist) + st.n_off / x.ne +
                                     (long long)x.tj0 * 2 * x.nc;
            for (int i = tid; i < nj; i += TPB)
                if (x.J[i]) atomicAdd(&gJ[i], x.J[i]);
            for (int i = tid; i < ng; i += TPB)
                if (x.G[i]) atomicAdd(&gG[i], (unsigned long long)x.G[i]);
            for (int i = tid; i < nv; i += TPB)
                if (x.V[i]) atomicAdd(&gV[i], x.V[i]);
        }
        const uint32_t vals[10] = {ty.absorbed, ty.bath, ty.hits, ty.trans, ty.trunc, ty.spawn_drop,
                                   ty.q_drop, ty.changed, kept_here, (uint32_t)n_event};
        const unsigned long long v = block_sums<10>(vals, s_r8);
        if (tid < 10 && v) {
            const int idx[10] = {L_ABSORBED, L_Q_BATH, L_IFACE_HITS, L_IFACE_TRANSMIT, L_TRUNCATED,
                                 L_SPAWN_DROPPED, L_Q_DROPPED, L_CHANGED, L_SPAWNED, L_EVENTFUL};
            atomicAdd(&a.cnt[s].led[idx[tid]], v);
        }
        const unsigned long long qs = block_sum_u64(q_src, s_r8), wsm = block_sum_u64(w_src, s_r8);
        if (tid == 0) {
            if (qs) atomicAdd(&a.cnt[s].led[L_Q_INJECTED], qs);
            if (wsm) atomicAdd(&a.cnt[s].w_injected, wsm);
        }
    }
    if (ib == 0 && tid == 0)
        g.res[s] = GroupRes{(unsigned long long)nsl, nid, psum, live0 + adds};

    // ---- the last block of the launch moves the counters on
    if (last_block(a, &s_flag)) {
        for (int q = tid; q < a.n_stacks; q += TPB) {
            const GroupRes r = {__ldcg(&g.res[q].n_slots), __ldcg(&g.res[q].next_id),
                                __ldcg(&g.res[q].steps0), __ldcg(&g.res[q].live0)};
            unsigned long long gone = 0, gone_steps = 0;
            for (int j = 0; j < sp.len; ++j) {
                const unsigned long long c = __ldcg(&g.abs[q * GROUP_MAX + j]);
                if (!c) continue;
                g.abs[q * GROUP_MAX + j] = 0u;
                gone += c;
                gone_steps += c * (unsigned long long)(sp.len - 1 - j);
            }
            g.bar[32 * q] = 0u;
            DevCounters &c = a.cnt[q];
            c.n_slots = r.n_slots;
            c.next_id = r.next_id;
            c.live = r.live0 - gone;
            c.led[L_PARTICLE_STEPS] += r.steps0 - gone_steps;
        }
        if (tid == 0) {
            a.ctl->done = 0u;
            a.ctl->step = sp.s0 + (uint32_t)sp.len;
        }
    }
}

template <bool DET, bool SUMS>
__global__ void __launch_bounds__(TPB, 2) k_tail(const Args a, const GroupArgs g)
{
    const uint32_t s0 = (g.base ? __ldcg(g.base) : 0u) + (uint32_t)g.off;
    const Span sp = g.nd > 0 ? group_span<true>(a, s0, g.end - g.off, g.m, g.no_src != 0)
                             : group_span<false>(a, s0, g.end - g.off, g.m, g.no_src != 0);
    if (sp.len != 0) phase_tail<DET, SUMS>(a, g, sp, g.no_src != 0);
}

// ---------------------------------------------------------------------------
// k_dens: the densities, generation and velocity sums of the window that the
// step before ended, from the state: 12 bytes read per slot and two or three
// shared-memory additions per carrier.
// ---------------------------------------------------------------------------
constexpr int DENS_T = 1024;     // (with 512 threads and branches around the additions 1.06 ms
                                 // for 4e8 slots, now 0.72: the bandwidth of a copy)

__device__ __forceinline__ void phase_dens(const Args &a)
{
    const int NT = (int)blockDim.x;
    extern __shared__ __align__(128) unsigned char smem[];
    uint32_t *s_n = reinterpret_cast<uint32_t *>(smem);
    uint32_t *s_gs = s_n + a.nbin_max;
    unsigned long long *s_v = reinterpret_cast<unsigned long long *>(
        (reinterpret_cast<uintptr_t>(s_gs + a.gbin_max) + 7) & ~uintptr_t(7));
    const bool vmom = (a.flags & PIC_F_VELOCITY_MOMENTS) != 0;
    long long *s_tpref = reinterpret_cast<long long *>(s_v + (vmom ? 2 * a.gbin_max : 0));
    FastEnt *s_ent = reinterpret_cast<FastEnt *>(
        (reinterpret_cast<uintptr_t>(s_tpref + 2 * a.n_stacks + 1) + 15) & ~uintptr_t(15));
    long long *s_nsl = s_tpref + a.n_stacks + 1;
    const int tid = threadIdx.x, ne = a.n_e;
    const int cur = (int)__ldcg(&a.ctl->cur);
    const int t = (int)(__ldcg(&a.ctl->step) / (uint32_t)a.moment_every) - 1;
    const RangeEnd end(a);
    for (int s = tid; s < a.n_stacks; s += NT) s_nsl[s] = (long long)a.cnt[s].n_slots;
    __syncthreads();
    if (tid == 0) {
        long long acc = 0;
        for (int s = 0; s < a.n_stacks; ++s) {
            s_tpref[s] = acc;
            acc += (s_nsl[s] + TILE - 1) / TILE;
        }
        s_tpref[a.n_stacks] = acc;
    }
    __syncthreads();
    const long long T = s_tpref[a.n_stacks];
    const long long t0 = chunk_lo(T, blockIdx.x, gridDim.x), t1 = chunk_lo(T, blockIdx.x + 1, gridDim.x);
    if (t0 >= t1 || !end.reached(a)) return;
    const int s_first = stack_of(s_tpref, a.n_stacks, t0), s_last = stack_of(s_tpref, a.n_stacks, t1 - 1);
    for (int s = s_first; s <= s_last; ++s) {
        const long long ta = t0 > s_tpref[s] ? t0 : s_tpref[s];
        const long long tb = t1 < s_tpref[s + 1] ? t1 : s_tpref[s + 1];
        if (ta >= tb) continue;
        const DevStack &st = a.stacks[s];
        const int nc = st.n_cells, nb = 2 * ne * nc;
        __syncthreads();
        for (int i = tid; i < nb; i += NT) s_n[i] = 0u;
        for (int i = tid; i < nc; i += NT) s_gs[i] = 0u;
        if (vmom) {
            for (int i = tid; i < 2 * nc; i += NT) s_v[i] = 0ull;
            for (int i = tid; i < st.ftab_n; i += NT) s_ent[i] = a.fent[st.fent_off + i];
        }
        __syncthreads();
        const uint32_t a_n = smem_addr(s_n), a_gs = smem_addr(s_gs);
        const float *Z = a.z[cur] + st.base;
        const float *MU = a.mu[cur] + 2 * st.base;
        const long long i0 = (ta - s_tpref[s]) * TILE;
        long long i1 = (tb - s_tpref[s]) * TILE;
        if (i1 > s_nsl[s]) i1 = s_nsl[s];
#pragma unroll 2
        for (long long i = i0 + 4 * tid; i < i1; i += 4 * NT) {
            const float4 z4 = *reinterpret_cast<const float4 *>(Z + i);
            const uint4 *mp = reinterpret_cast<const uint4 *>(MU + 2 * i);
            const uint4 m0 = mp[0], m1 = mp[1];
            const float zi[4] = {z4.x, z4.y, z4.z, z4.w};
            const uint32_t pi[4] = {m0.y, m0.w, m1.y, m1.w}, mi[4] = {m0.x, m0.z, m1.x, m1.z};
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                // a removed slot adds 0 to the first row (z of a slot past the last
                // one may be anything: its cell is held inside)
                const uint32_t pk = i + c < i1 ? pi[c] : 0u;
                const int k = (int)(pk & 0xFFu), sg = (int)((pk >> 8) & 1u);
                const uint32_t on = k != 0 ? 1u : 0u;
                const int cl = max(cell_at(zi[c], a.inv_dz, nc), 0);
                red_shared(a_n + 4u * (uint32_t)((on ? sg * ne + k - 1 : 0) * nc + cl), on);
                red_shared(a_gs + 4u * (uint32_t)cl, on ? (pk >> 13) & 0xFFu : 0u);
                if (vmom && on)
                    add_u64_split(&s_v[sg * nc + cl],
                                  (unsigned long long)vel_q(__fmul_rn(s_ent[fast_index(a, pk)].v,
                                                                      __uint_as_float(mi[c]))));
            }
        }
        __syncthreads();
        uint32_t *gN = a.n_hist + st.n_off + (long long)t * nb;
        unsigned long long *gG = a.g_hist + st.n_off / (2 * ne) + (long long)t * nc;
        flush_bins(gN, s_n, nb);
        for (int i = tid; i < nc; i += NT)
            if (s_gs[i]) atomicAdd(&gG[i], (unsigned long long)s_gs[i]);
        if (vmom) {
            unsigned long long *gV = reinterpret_cast<unsigned long long *>(a.v_hist) + st.n_off / ne +
                                     (long long)t * 2 * nc;
            for (int i = tid; i < 2 * nc; i += NT)
                if (s_v[i]) atomicAdd(&gV[i], s_v[i]);
        }
    }
}

__global__ void __launch_bounds__(DENS_T) k_dens(const Args a)
{
    phase_dens(a);
}

// ---------------------------------------------------------------------------
// k_run: n_steps whole steps of every stack in one cooperative launch, the
// phases of each group separated by grid barriers.  All threads of a block work
// on k_group's and k_dens's phases, the first TPB on the others.  `src_end`:
// the first step after which no source carrier comes.
// ---------------------------------------------------------------------------
template <bool DET, bool DEP, int Q>
__global__ void __launch_bounds__(32 * GW_MAX, 1) k_run(const Args a, const GroupArgs g, int n_steps, int src_end)
{
    uint32_t s = __ldcg(&a.ctl->step);
    const uint32_t end = s + (uint32_t)n_steps, me = (uint32_t)a.moment_every, ce = (uint32_t)a.compact_every;
    const bool low = threadIdx.x < TPB;
    // (decisions of the whole block; a status other than a given-up wait's changes
    // nothing here, as in single launches)
    if (__syncthreads_or(threadIdx.x == 0 && timed_out(a))) return;
    while (s < end) {
        uint32_t e = (s / ce + 1) * ce;
        if (e > s + GROUP_MAX) e = s + GROUP_MAX;
        if (!DEP && e > (s / me + 1) * me) e = (s / me + 1) * me;
        if (e > end) e = end;
        while (s < e) {
            const bool no_src = s >= (uint32_t)src_end;
            const Span sp = block_span<DEP>(a, s, (int)(e - s), group_part((int)(e - s), g.m), no_src);
            if (sp.len == 0) return;         // (only after a wait was given up in k_tail's part)
            phase_group<DET, DEP, Q>(a, g, sp);
            if (!grid_sync(a)) return;
            if (low && g.tail_sums) phase_tail<DET, true>(a, g, sp, no_src);
            else if (low) phase_tail<DET, false>(a, g, sp, no_src);
            if (!grid_sync(a)) return;
            s += (uint32_t)sp.len;
        }
        if (!DEP && e % me == 0) {
            phase_dens(a);
            if ((e < end || e % ce == 0) && !grid_sync(a)) return;
        }
        if (e % ce == 0) {
            if (low) phase_compact<0>(a);
            if (e < end && !grid_sync(a)) return;
        }
    }
}

// (after a wait was given up no group of the graph finds its first step)
__global__ void k_mark_base(DevCtl *ctl)
{
    ctl->base = ctl->status == (unsigned int)PIC_ERR_TIMEOUT ? 0x80000000u : ctl->step;
}

size_t dens_smem(const Args &a)
{
    const bool vmom = (a.flags & PIC_F_VELOCITY_MOMENTS) != 0;
    return (size_t)(a.nbin_max + a.gbin_max) * 4 + 8 + (vmom ? (size_t)a.gbin_max * 16 : 0) +
           (size_t)(2 * a.n_stacks + 1) * 8 + 16 + (vmom ? (size_t)a.ftab_max * sizeof(FastEnt) : 0);
}

template <bool DEP, int Q>
cudaError_t group_fits(size_t smem, int threads, bool *ok)
{
    int o1 = 0, o2 = 0;
    cudaError_t e = occupancy(k_group<false, DEP, Q>, smem, &o1, threads);
    if (e == cudaSuccess) e = occupancy(k_group<true, DEP, Q>, smem, &o2, threads);
    *ok = e == cudaSuccess && o1 >= 1 && o2 >= 1;
    return e;
}

// The shapes that k_group may take, the preferred one first; none: the steps are
// not grouped.  Every one has TPB threads or more: a block decides the group's
// span at a barrier of its first TPB threads (group_span).
struct GroupShape {
    int m, quads, warps, nd, nj;
    size_t smem;
};

// densities deposited inside the groups
bool group_dep(const Args &a) { return a.moment_every < GROUP_DEP_EVERY && !(a.flags & PIC_F_WEIGHTS); }

std::vector<GroupShape> group_shapes(const Args &a, long long slots, int sms, size_t cap)
{
    const int me = a.moment_every;
    const bool dep = group_dep(a);
    std::vector<GroupShape> r;
    // Slots per sub-tile: 1024, so that the 2 % of eventful carriers fill most of
    // a warp (41.5 ms for 50 steps of 4e8 carriers; 52.9 with 512); 512 beside
    // the density histograms, which leave room for too few warps otherwise
    // (batched stacks 171 ms for 50 steps against 251); 256 or 512 where larger
    // ones would leave warps without any.
    int quads = dep ? 4 : 8;
    if (slots < (long long)sms * 12 * 1024) quads = 4;
    if (slots < (long long)sms * 12 * 512) quads = 2;
    for (int m = slots <= GROUP_LIST_SLOTS ? GROUP_OPEN : GROUP_OPEN_LARGE; m >= 1; --m) {
        const int nd = dep ? (me - 1 + m) / me : 0;
        const int nj = dep ? (me + m - 2) / me + 1 : 1;
        // groups of one step (50 steps of 245 cells x 60 bins: 1.2e6 slots 1.57 ms, single
        // steps 2.02; 1.2e7 slots 6.43 and 5.44; densities every third step, 275
        // cells: 1.69 and 1.63)
        if (m == 1 && (me > 1 || slots > LONE_SLOTS)) break;
        // too few warps beside the histograms: fewer windows
        const int least = m == 1 || quads == 8 ? TPB / 32 : quads == 4 ? (m > GROUP_OPEN_LARGE ? 14 : TPB / 32) : 12;
        for (int w = GW_MAX; w >= least; --w) {
            const GroupSmem o = group_smem(a, dep, quads, w, nd, nj);
            if (o.total <= cap) r.push_back({m, quads, w, nd, nj, o.total});
        }
    }
    return r;
}

}  // namespace

static cudaError_t configure_run(const Args &a, GroupCfg *c);

cudaError_t configure_group(const Args &a, long long slots, GroupCfg *gc)
{
    *gc = GroupCfg{};
    int dev = 0, sms = 0, optin = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e != cudaSuccess) return e;
    const size_t cap = (size_t)optin - 2048;         // less the kernels' static shared memory
    // the edges have to do as half-precision numbers
    if (a.dz * (float)a.gbin_max > 32768.f || a.dz < 1.f / 1024.f) return cudaSuccess;
    GroupCfg c;
    c.dep = group_dep(a);
    for (const GroupShape &x : group_shapes(a, slots, sms, cap)) {
        bool ok = false;
        if (c.dep) {
            if (x.quads == 4) e = group_fits<true, 4>(x.smem, 32 * x.warps, &ok);
            else e = group_fits<true, 2>(x.smem, 32 * x.warps, &ok);
        } else {
            if (x.quads == 8) e = group_fits<false, 8>(x.smem, 32 * x.warps, &ok);
            else if (x.quads == 4) e = group_fits<false, 4>(x.smem, 32 * x.warps, &ok);
            else e = group_fits<false, 2>(x.smem, 32 * x.warps, &ok);
        }
        if (e != cudaSuccess) return e;
        if (!ok) continue;
        c.m = x.m; c.quads = x.quads; c.warps = x.warps; c.nd = x.nd; c.nj = x.nj; c.smem = x.smem;
        c.grid = sms;
        c.ok = true;
        break;
    }
    if (!c.ok) return cudaSuccess;
    // Blocks: every one resident (they wait on one another), few for few carriers.
    // Two per SM keep their sums over cells beside the tables.  Births and removals
    // alone are too few in small contexts to pay for clearing and flushing (300
    // steps from 1e5 carriers 4.56 ms without, 4.67 with), and 32 bits hold the
    // generation sums of the carriers that a block moves and of those that it
    // places, each at most its stack's share (pic_init) of 2^23 slots, 255 each.
    auto tail = [&](bool sums) -> cudaError_t {
        c.tail_sums = sums;
        c.smem_tail = (size_t)a.tab_max * sizeof(TabEnt) + (size_t)a.T_max * 4 + 16 + (sums ? tail_sums(a, c.nd, c.nj) : 0);
        int o[4] = {2, 2, 2, 2};                 // (a step by itself takes the form without sums)
        cudaError_t r = occupancy(k_tail<false, false>, c.smem_tail, &o[0]);
        if (r == cudaSuccess) r = occupancy(k_tail<true, false>, c.smem_tail, &o[1]);
        if (sums && r == cudaSuccess) r = occupancy(k_tail<false, true>, c.smem_tail, &o[2]);
        if (sums && r == cudaSuccess) r = occupancy(k_tail<true, true>, c.smem_tail, &o[3]);
        const long long most = (long long)sms * std::min({o[0], o[1], o[2], o[3], 2});
        c.grid_tail = (int)std::max<long long>(std::min<long long>(std::max<long long>(slots / 4096, 8), most), a.n_stacks);
        if (most < a.n_stacks) c.grid_tail = 0;
        return r;
    };
    e = tail((c.dep || slots > (1ll << 20)) && tail_sums(a, c.nd, c.nj) <= 48 * 1024);
    if (e == cudaSuccess && c.tail_sums &&
        slots / std::max(std::min(c.grid_tail, c.grid) - a.n_stacks, 1) > (1ll << 23))
        e = tail(false);
    if (e != cudaSuccess) return e;
    if (c.grid_tail == 0) return cudaSuccess;
    if (!c.dep) {
        c.smem_dens = dens_smem(a);
        int od = 0;
        e = occupancy(k_dens, c.smem_dens, &od, DENS_T);
        if (e != cudaSuccess) return e;
        if (od < 1) return cudaSuccess;
        c.grid_dens = sms * std::min(od, 2);
    }
    e = configure_run(a, &c);
    *gc = c;
    return e;
}

// The persistent form's blocks: one per SM, which also have to be enough for a
// block per stack; shared memory for the largest of its phases.
template <bool DEP, int Q>
static cudaError_t run_fits(size_t smem, int threads, bool *ok)
{
    int o1 = 0, o2 = 0;
    cudaError_t e = occupancy(k_run<false, DEP, Q>, smem, &o1, threads);
    if (e == cudaSuccess) e = occupancy(k_run<true, DEP, Q>, smem, &o2, threads);
    *ok = e == cudaSuccess && o1 >= 1 && o2 >= 1;
    return e;
}

static cudaError_t configure_run(const Args &a, GroupCfg *c)
{
    c->run = false;
    if ((a.flags & PIC_F_WEIGHTS) || c->grid < a.n_stacks) return cudaSuccess;
    cudaError_t e = cudaSuccess;
    // (its static shared memory is larger: a warp or two less)
    for (int w = c->warps; w >= TPB / 32 && !c->run && e == cudaSuccess; --w) {
        c->smem_run = std::max({group_smem(a, c->dep, c->quads, w, c->nd, c->nj).total, c->smem_tail, c->smem_dens});
        c->warps_run = w;
        if (c->dep) {
            if (c->quads == 4) e = run_fits<true, 4>(c->smem_run, 32 * w, &c->run);
            else e = run_fits<true, 2>(c->smem_run, 32 * w, &c->run);
        } else {
            if (c->quads == 8) e = run_fits<false, 8>(c->smem_run, 32 * w, &c->run);
            else if (c->quads == 4) e = run_fits<false, 4>(c->smem_run, 32 * w, &c->run);
            else e = run_fits<false, 2>(c->smem_run, 32 * w, &c->run);
        }
    }
    return e;
}

cudaError_t launch_run(const Args &a, const GroupArgs &g, const GroupCfg &c, bool det, int n_steps, int src_end,
                       cudaStream_t s)
{
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)c.grid);
    cfg.blockDim = dim3((unsigned)(32 * c.warps_run));
    cfg.dynamicSmemBytes = c.smem_run;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
#define PIC_RUN_LAUNCH(DEP, Q)                                                                     \
    return det ? cudaLaunchKernelEx(&cfg, k_run<true, DEP, Q>, a, g, n_steps, src_end)             \
               : cudaLaunchKernelEx(&cfg, k_run<false, DEP, Q>, a, g, n_steps, src_end)
    if (c.dep) {
        if (c.quads == 4) PIC_RUN_LAUNCH(true, 4);
        PIC_RUN_LAUNCH(true, 2);
    }
    if (c.quads == 8) PIC_RUN_LAUNCH(false, 8);
    if (c.quads == 4) PIC_RUN_LAUNCH(false, 4);
    PIC_RUN_LAUNCH(false, 2);
#undef PIC_RUN_LAUNCH
}

cudaError_t launch_group(const Args &a, const GroupArgs &g, const GroupCfg &c, bool det, cudaStream_t s)
{
    const int nt = 32 * c.warps;
    if (nt < TPB) return cudaErrorInvalidConfiguration;
#define PIC_GROUP_LAUNCH(DEP, Q)                                                                   \
    do {                                                                                           \
        if (det) k_group<true, DEP, Q><<<c.grid, nt, c.smem, s>>>(a, g);                           \
        else k_group<false, DEP, Q><<<c.grid, nt, c.smem, s>>>(a, g);                              \
    } while (0)
    if (c.dep) {
        if (c.quads == 4) PIC_GROUP_LAUNCH(true, 4);
        else PIC_GROUP_LAUNCH(true, 2);
    } else {
        if (c.quads == 8) PIC_GROUP_LAUNCH(false, 8);
        else if (c.quads == 4) PIC_GROUP_LAUNCH(false, 4);
        else PIC_GROUP_LAUNCH(false, 2);
    }
#undef PIC_GROUP_LAUNCH
    return cudaGetLastError();
}

cudaError_t launch_tail(const Args &a, const GroupArgs &g, const GroupCfg &c, bool det, cudaStream_t s)
{
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)c.grid_tail);
    cfg.blockDim = dim3((unsigned)TPB);
    cfg.dynamicSmemBytes = c.smem_tail;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    // a step by itself has little to add up: clearing and flushing took 1 us of the
    // 66 of a call of one step and its window
    if (g.tail_sums && g.end - g.off > 1)
        return det ? cudaLaunchKernelEx(&cfg, k_tail<true, true>, a, g) : cudaLaunchKernelEx(&cfg, k_tail<false, true>, a, g);
    return det ? cudaLaunchKernelEx(&cfg, k_tail<true, false>, a, g) : cudaLaunchKernelEx(&cfg, k_tail<false, false>, a, g);
}

cudaError_t launch_dens(const Args &a, const GroupCfg &c, cudaStream_t s)
{
    k_dens<<<c.grid_dens, DENS_T, c.smem_dens, s>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_mark_base(DevCtl *ctl, cudaStream_t s)
{
    k_mark_base<<<1, 1, 0, s>>>(ctl);
    return cudaGetLastError();
}

}  // namespace pic

// The shapes of a context of n_stacks stacks with `slots` slots in all and at
// most `layers` layers and `cells` cells each, from the preferred one: up to
// `most` of (m, quads, warps) into out; their number.  For checks without a
// device.
extern "C" int pic_group_shapes(int n_stacks, int n_e, int layers, int cells, int moment_every, unsigned int flags,
                                long long slots, int sms, long long smem, int *out, int most)
{
    using namespace pic;
    Args a{};
    int kb = 0;
    while ((1 << kb) < n_e + 1) ++kb;
    a.n_stacks = n_stacks; a.n_e = n_e; a.moment_every = moment_every; a.flags = flags;
    a.ftab_max = layers * 2 << kb;
    a.tab_max = layers * 2 * n_e;
    a.T_max = std::max((layers - 1) * 4 * n_e, 1);
    a.nbin_max = 2 * n_e * cells;
    a.gbin_max = cells;
    a.jbin_max = 2 * (cells + 1);
    const std::vector<GroupShape> v = group_shapes(a, slots, sms, (size_t)smem);
    for (int i = 0; i < (int)v.size() && i < most; ++i) {
        out[3 * i] = v[i].m;
        out[3 * i + 1] = v[i].quads;
        out[3 * i + 2] = v[i].warps;
    }
    return (int)v.size();
}
