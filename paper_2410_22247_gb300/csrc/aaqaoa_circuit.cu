// Whole MaxCut circuits in one launch (k_circuit): the phase tables, p layers,
// the energy and, for a gradient, the adjoint sweep, for states that fit the
// shared memory of one CTA or of a team of CTAs.
//
// A state is the flip-symmetric half of k_pass (m = n - 1 stored bits, vertex
// n - 1 on side 0, twisted frame i^|y| psi(y)). A team of 2^c CTAs holds one
// point's vectors, 2^Tl amplitudes per CTA (m = Tl + c), in one of two layouts
// of the stored index y:
//   low:  y = rank | i                      (i: the CTA's local index, Tl bits)
//   high: i = P | hi | lo, the CTA's tile of fixed middle bits f = 0 | rank and
//         its mirrored tile ~f: y = hi | (P ? ~f : f) | lo
// The low layout mixes qubits 0..Tl-1, the high layout the c top stored bits
// (in hi) and vertex n - 1, whose partner of y is ~y, i.e. local index ~i. A
// layer is one part, an exchange of the tiles through global memory (L2
// resident), the other part; the next layer starts in the layout that this one
// ended in, so a layer costs one exchange and one barrier of the team. A team
// of up to 16 CTAs is a cluster and exchanges through distributed shared
// memory. With c = 0 there is one layout and no exchange.
//
// What bounds it: latency (a few thousand amplitudes per CTA, one barrier per
// register stage), so the aim is few launches, few barriers and little code.
// The register stages take up to four bits and share one loop for every bit
// position; shared memory is swizzled (amplitude index low bits XOR the next
// four), which keeps the strided accesses of all stages free of bank conflicts.
// Measured (device, p = 2, one point; before: the tables' launch and a kernel
// with one barrier per qubit, above n = 13 the passes): complex64 gradient
// n = 10 54 -> 21 us, n = 14 140 -> 28, n = 16 137 -> 40, n = 20 151 -> 75;
// 256 complex128 energies at n = 12 157 -> 84 us.
#include <atomic>

#include "aaqaoa_pass.cuh"

namespace aaq {

namespace {

constexpr int CIRC_MAXP = 64;
constexpr int CIRC_MAXN = CIRCUIT_MASKS;  // row length of the neighbour masks

__device__ __forceinline__ uint32_t cswz(uint32_t i) { return i ^ ((i >> 4) & 15u); }

// A thread's sum of terms in the amplitude type. complex64: a float and the
// rounding errors of its additions (TwoSum), 48 bits, so that a term costs six
// FP32 operations and no FP64 one: the FP64 unit takes 16 cycles per warp, and
// three such additions per register stage were 1.2 us of a 33 us gradient at
// n = 10. Sums over threads are FP64.
template <typename R> struct CircSum {
    double v = 0.0;
    __device__ __forceinline__ void add(double x) { v += x; }
    __device__ __forceinline__ double value() const { return v; }
};
template <> struct CircSum<float> {
    float hi = 0.f, lo = 0.f;
    __device__ __forceinline__ void add(float x)
    {
        const float t = __fadd_rn(hi, x), z = __fsub_rn(t, hi);
        lo = __fadd_rn(lo, __fadd_rn(__fsub_rn(hi, __fsub_rn(t, z)), __fsub_rn(x, z)));
        hi = t;
    }
    __device__ __forceinline__ double value() const { return (double)hi + (double)lo; }
};

struct CircLayer {  // one layer's mixer: rotation t, dropped factor f, f^n; of the inverse: -t, fi, fi^n
    double f, fi, fn, fin;
    double t;
};

// register-stage bits of a launch: up to KMAX (16 amplitudes of each vector in
// registers; 8 for two complex128 vectors)
template <typename R, int NV>
constexpr int circ_kmax = (NV == 2 && !std::is_same<R, float>::value) ? 3 : 4;

// thread/CTA view of one point; its vectors start the dynamic shared memory
// (phi, lambda; for a cluster twice, the exchange alternates the two)
extern __shared__ __align__(16) unsigned char circ_smem[];

struct CircCtx {
    int m, Tl, c, rank, a;  // a: low bits of the high layout
    int km;                 // bits of a full register stage
    int pair;               // as StageCtx::pair
    uint32_t off;           // first amplitude of the current phi
};

// stored index of local index i
__device__ __forceinline__ uint32_t circ_index(const CircCtx &X, int high, uint32_t i)
{
    if (!high)
        return ((uint32_t)X.rank << X.Tl) | i;
    const uint32_t lo = i & ((1u << X.a) - 1u), hi = (i >> X.a) & ((1u << (X.Tl - 1 - X.a)) - 1u);
    const uint32_t fm = (1u << (X.c + 1)) - 1u, f = (i >> (X.Tl - 1)) ? ~(uint32_t)X.rank & fm : (uint32_t)X.rank;
    return (hi << (X.a + X.c + 1)) | (f << X.a) | lo;
}

// One register stage: the butterflies of local bits q0..q0+K-1 and, for MIR,
// then those of vertex n - 1 (local index ~i), on the vectors at `off`. run:
// f^j before the stage; acc: the thread's sum of dE/dbeta terms. sg0: the sign
// of vertex n - 1's rotation at local index 0 (the stored index of a local
// index has its bit count plus the rank's in either layout). A function of its
// own with its arguments in registers, so that every bit position and layer
// runs the same code (a launch meets it cold).
template <typename R> struct CircMix {
    R run;
    CircSum<R> acc;
};
template <typename R, int NV, int K, bool MIR>
__device__ __noinline__ CircMix<R> circ_stage(uint32_t off, int Tl, int q0, int pair, R sg0, R t, R f, R run,
                                              CircSum<R> acc)
{
    using C = typename CT<R>::T;
    C *phi = reinterpret_cast<C *>(circ_smem) + off, *lam = phi + ((size_t)1 << Tl);
    constexpr int RB = K + (MIR ? 1 : 0), NR = 1 << RB, H = 1 << K;
    const uint32_t items = 1u << (Tl - RB), full = (1u << Tl) - 1u, gm = (uint32_t)(H - 1) << q0;
    R sc = run;
    for (uint32_t it = threadIdx.x; it < items; it += blockDim.x) {
        const uint32_t i = ((it >> q0) << (q0 + K)) | (it & ((1u << q0) - 1u));
        const uint32_t s0 = cswz(i), s1 = MIR ? cswz(i ^ full ^ gm) : 0u;
        C a[NR], l[NR];
#pragma unroll
        for (int r = 0; r < NR; r++) {
            const uint32_t x = (MIR && r >= H ? s1 : s0) ^ cswz((uint32_t)(r & (H - 1)) << q0);
            a[r] = phi[x];
            if constexpr (NV == 2)
                l[r] = lam[x];
        }
        sc = run;
#pragma unroll
        for (int k = 0; k < K; k++) {
            C ipp[2], ipn[2];
            ipp[0] = ipp[1] = ipn[0] = ipn[1] = mkc<C>((R)0, (R)0);
#pragma unroll
            for (int r = 0; r < NR; r++) {
                if (r & (1 << k))
                    continue;
                const int r1 = r | (1 << k);
                if constexpr (NV == 2) {
                    const int h = (r >> (k == 0 ? 1 : 0)) & 1;
                    dot_acc(ipp[h], l[r1], a[r]);
                    dot_acc(ipn[h], l[r], a[r1]);
                    rot(l[r], l[r1], t);
                }
                rot(a[r], a[r1], t);
            }
            if constexpr (NV == 2) {
                const R q = ((ipp[0].x + ipp[0].y) + (ipp[1].x + ipp[1].y)) -
                            ((ipn[0].x + ipn[0].y) + (ipn[1].x + ipn[1].y));
                acc.add(q * (sc * sc));
            }
            sc *= f;
        }
        if constexpr (MIR) {
            const R sg = (__popc(i) & 1) ? -sg0 : sg0;
            const R q = sg * mix_mirror<R, NV, RB, NV == 1>(pair, sg * t, a, l);
            if constexpr (NV == 2)
                acc.add(q * (sc * sc));
            sc *= f;
        }
#pragma unroll
        for (int r = 0; r < NR; r++) {
            const uint32_t x = (MIR && r >= H ? s1 : s0) ^ cswz((uint32_t)(r & (H - 1)) << q0);
            phi[x] = a[r];
            if constexpr (NV == 2)
                lam[x] = l[r];
        }
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < RB; k++)  // (threads without an item too)
        run *= f;
    return CircMix<R>{run, acc};
}

// The mixer's part in one layout: local bits q0..q1-1, and vertex n - 1 if
// mir, as stages of km bits (the last one with vertex n - 1 takes one fewer).
template <typename R, int NV>
__device__ __forceinline__ CircMix<R> circ_mix(const CircCtx &X, int q0, int q1, bool mir, R t, R f, CircMix<R> M)
{
    constexpr int KMAX = circ_kmax<R, NV>;
    const R sg0 = ((__popc(X.rank) + (X.m >> 1)) & 1) ? (R)-1 : (R)1;
    while (q0 < q1 || mir) {
        const int k = q1 - q0 < X.km ? q1 - q0 : X.km;
        if (mir && k < X.km) {  // the last stage
            if (k == 0)
                M = circ_stage<R, NV, 0, true>(X.off, X.Tl, q0, X.pair, sg0, t, f, M.run, M.acc);
            else if (k == 1)
                M = circ_stage<R, NV, 1, true>(X.off, X.Tl, q0, X.pair, sg0, t, f, M.run, M.acc);
            else if (k == 2)
                M = circ_stage<R, NV, 2, true>(X.off, X.Tl, q0, X.pair, sg0, t, f, M.run, M.acc);
            else if constexpr (KMAX > 3)
                M = circ_stage<R, NV, 3, true>(X.off, X.Tl, q0, X.pair, sg0, t, f, M.run, M.acc);
            break;
        }
        if (k == 1)
            M = circ_stage<R, NV, 1, false>(X.off, X.Tl, q0, X.pair, sg0, t, f, M.run, M.acc);
        else if (k == 2)
            M = circ_stage<R, NV, 2, false>(X.off, X.Tl, q0, X.pair, sg0, t, f, M.run, M.acc);
        else if (k == 3)
            M = circ_stage<R, NV, 3, false>(X.off, X.Tl, q0, X.pair, sg0, t, f, M.run, M.acc);
        else if constexpr (KMAX > 3)
            M = circ_stage<R, NV, 4, false>(X.off, X.Tl, q0, X.pair, sg0, t, f, M.run, M.acc);
        q0 += k;
    }
    return M;
}

// cut values of the 4 states with stored indices y | 0..3
__device__ __noinline__ int4 circ_cuts(const uint32_t *nbr, const int *w, int K, int m, uint32_t y)
{
    int base = 0, d0 = 0, d1 = 0, w01 = 0;
    for (int c = 0; c < K; c++) {
        const uint32_t *nb = nbr + c * CIRC_MAXN;
        const int wc = w[c];
        int bc = 0;
#pragma unroll 4
        for (int u = 2; u < m; u++)
            bc += ((y >> u) & 1u) ? __popc(nb[u] & ~y) : 0;
        base += wc * bc;
        d0 += wc * (__popc(nb[0]) - 2 * __popc(nb[0] & y));
        d1 += wc * (__popc(nb[1]) - 2 * __popc(nb[1] & y));
        w01 += wc * (int)((nb[1]) & 1u);
    }
    return make_int4(base, base + d0, base + d1, base + d0 + d1 - 2 * w01);
}

// cluster (distributed shared memory) helpers
__device__ __forceinline__ void circ_cluster_sync()
{
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}
__device__ __forceinline__ uint32_t circ_map(uint32_t addr, uint32_t rank)
{
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
__device__ __forceinline__ void circ_st(uint32_t addr, float2 v)
{
    asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(addr), "f"(v.x), "f"(v.y) : "memory");
}
__device__ __forceinline__ void circ_st(uint32_t addr, double2 v)
{
    asm volatile("st.shared::cluster.v2.f64 [%0], {%1, %2};" ::"r"(addr), "d"(v.x), "d"(v.y) : "memory");
}
__device__ __forceinline__ void circ_st(uint32_t addr, double v)
{
    asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(addr), "d"(v) : "memory");
}

// i^e z
template <typename C>
__device__ __forceinline__ C circ_turn(C z, int e)
{
    const bool sw = e & 1;
    C v;
    v.x = sw ? z.y : z.x;
    v.y = sw ? z.x : z.y;
    if (((e + 1) & 2))
        v.x = -v.x;
    if (e & 2)
        v.y = -v.y;
    return v;
}

}  // namespace

// CL: the team is a cluster (exchange through distributed shared memory)
template <typename R, bool GRAD, bool CL>
__global__ void __launch_bounds__(512) k_circuit(const __grid_constant__ CircuitArgs A)
{
    using C = typename CT<R>::T;
    constexpr int NV = GRAD ? 2 : 1;
    __shared__ uint32_t s_cost[MAXK * CIRC_MAXN], s_obs[MAXK * CIRC_MAXN];
    __shared__ int s_cw[MAXK], s_ow[MAXK];
    __shared__ CircLayer lay[CIRC_MAXP];
    __shared__ int s_stop;
    __shared__ unsigned s_last;

    const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, warp = tid >> 5, nw = nt >> 5;
    const int n = A.n, p = A.p, c = A.c, Tl = A.Tl, m = n - 1, tab_len = A.tab_len;
    const uint32_t NL = 1u << Tl;
    CircCtx X;
    C *const vec = reinterpret_cast<C *>(circ_smem);
    C *tabs = vec + (size_t)(CL ? 2 : 1) * NV * NL;
    const int tslots = A.resident ? p : 1, rows = GRAD ? 1 + 2 * p : 1;
    double *red = reinterpret_cast<double *>(tabs + (size_t)2 * tslots * tab_len);  // [rows][nw]
    double *xred = red + (size_t)rows * nw;                                         // CL: [rows][2^c], rank 0's
    uint16_t *cval = reinterpret_cast<uint16_t *>(xred + (CL ? (size_t)rows << c : 0));  // [layouts][2^Tl]
    X.m = m;
    X.Tl = Tl;
    X.c = c;
    X.rank = (int)(blockIdx.x & ((1u << c) - 1u));
    X.a = A.a;
    X.km = A.km;
    X.pair = (m & 1) ? 1 : 2;
    X.off = 0;
    const unsigned b = blockIdx.x >> c;  // the team's point

    // The error flag of earlier launches that was not fetched yet. A team stops (its
    // counters are not at zero); a host call that reads no other word back gets it.
    const bool stops = !CL && c;
    int pending = 0;
    if (tid == 0) {
        if (stops || (A.err_out && X.rank == 0))
            pending = *reinterpret_cast<volatile int *>(A.err);
        s_stop = stops && pending ? 1 : 0;
    }
    if (CL)
        circ_cluster_sync();  // every CTA of the cluster runs before its memory is written
    else
        __syncthreads();
    // A team that gives up leaves NaN in its point's row, not what an earlier call put
    // there (each CTA that gives up writes it; no other result follows, since the
    // last CTA to finish writes that and needs all of them).
    auto give_up = [&] {
        for (int r = tid; r < rows; r += nt)
            A.out[(size_t)b * A.out_stride + r] = __longlong_as_double(0x7ff8000000000000ll);
    };
    if (!CL && s_stop) {
        give_up();
        return;
    }

    // cut functions. A graph per point reads all classes, so that no load waits
    // for their number; one graph's are launch constants, only those in use (a
    // constant read by lane-dependent index costs one access per lane).
    const GraphFns *const pt = A.fns ? A.fns + b : nullptr;
    const int Kc = pt ? pt->cost.K : A.fn[0].K, Ko = pt ? pt->obs[A.obs].K : A.fn[1].K;
    if (pt) {
        const CutFn &cost = pt->cost, &obs = pt->obs[A.obs];
        for (int i = tid; i < MAXK * CIRC_MAXN; i += nt) {
            const int k = i / CIRC_MAXN, u = i % CIRC_MAXN;
            s_cost[i] = u < n ? (uint32_t)cost.nbr[k][u] : 0u;
            s_obs[i] = u < n ? (uint32_t)obs.nbr[k][u] : 0u;
        }
        if (tid < MAXK) {
            s_cw[tid] = cost.w[tid];
            s_ow[tid] = obs.w[tid];
        }
    } else {
        for (int i = tid; i < (Kc + Ko) * CIRC_MAXN; i += nt) {
            const int e = i >= Kc * CIRC_MAXN, j = e ? i - Kc * CIRC_MAXN : i;
            (e ? s_obs : s_cost)[j] = A.fn[e].nbr[j / CIRC_MAXN][j % CIRC_MAXN];
        }
        for (int k = tid; k < 2 * MAXK; k += nt)
            (k < MAXK ? s_cw : s_ow)[k % MAXK] = A.fn[k / MAXK].w[k % MAXK];
    }
    __syncthreads();
    const double *gam = A.gamma ? A.gamma + (size_t)b * p : A.ang, *bet = A.gamma ? A.beta + (size_t)b * p : A.ang + p;
    // ------------------------------------------------ angles, tables
    // Warps take layers, lanes table entries; the first entry of a lane is
    // computed beside the mixer's angles (the last warps), its scale
    // follows once those are known.
    double2 z0 = make_double2(1.0, 0.0);
    if (A.resident && warp < p && lane < tab_len)
        z0 = phase_sincos(gam[warp] * (double)lane);
    for (int l = nt - 1 - tid; l < p; l += nt) {
        const double2 z = phase_sincos(bet[l]);
        const bool sh = fabs(z.y) > fabs(z.x);  // rotate by beta - pi/2 (see rot)
        double t;
        MixFactor m;
        mix_ratio<R>(sh ? -z.x : z.y, sh ? z.y : z.x, t, m);
        const double fn = mix_power<R>(m, n);
        lay[l] = CircLayer{m.f, sh ? -m.f : m.f, fn, (sh && (n & 1)) ? -fn : fn, t};
    }
    // cut values of the tile's states in both layouts
    for (int h = 0; h < (c > 0 ? 2 : 1); h++)
        for (uint32_t i = 4u * tid; i < NL; i += 4u * nt) {
            const int4 v = circ_cuts(s_cost, s_cw, Kc, m, circ_index(X, h, i));
            *reinterpret_cast<uint2 *>(cval + (size_t)h * NL + i) =
                make_uint2((uint32_t)v.x | ((uint32_t)v.y << 16), (uint32_t)v.z | ((uint32_t)v.w << 16));
        }
    __syncthreads();
    auto entry = [&](int l, int c0, double2 z, C *dst) {  // [0] forward, [1] inverse
        const double fs = l > 0 ? lay[l - 1].fn : 1.0, fb = lay[l].fin;
        dst[c0] = mkc<C>((R)(z.x * fs), (R)(-z.y * fs));
        dst[tab_len + c0] = mkc<C>((R)(z.x * fb), (R)(z.y * fb));
    };
    if (A.resident) {
        for (int l = warp; l < p; l += nw)
            for (int i = lane; i < tab_len; i += 32) {
                const double2 z = l == warp && i == lane ? z0 : phase_sincos(gam[l] * (double)i);
                entry(l, i, z, tabs + (size_t)2 * l * tab_len);
            }
        __syncthreads();
    }
    auto layer_table = [&](int l) -> const C * {
        if (A.resident)
            return tabs + (size_t)2 * l * tab_len;
        __syncthreads();
        for (int i = tid; i < tab_len; i += nt)
            entry(l, i, phase_sincos(gam[l] * (double)i), tabs);
        __syncthreads();
        return tabs;
    };

    // exchange of the tiles between the layouts (all CTAs of the team)
    C *xphi = c && !CL ? reinterpret_cast<C *>(A.phi) + ((size_t)b << n) : nullptr;
    C *xlam = c && !CL && GRAD ? reinterpret_cast<C *>(A.lam) + ((size_t)b << n) : nullptr;
    unsigned arrivals = 0;
    int parity = 0;
    auto exchange = [&](int from, bool both) -> bool {
        C *phi = vec + X.off, *lam = phi + NL;
        if constexpr (CL) {  // every amplitude straight to its place in the other layout
            X.off ^= (uint32_t)NV * NL;
            const uint32_t dst = smem_u32(vec + X.off), amask = (1u << X.a) - 1u, fm = (2u << c) - 1u;
#pragma unroll 4
            for (uint32_t i = tid; i < NL; i += nt) {
                const uint32_t y = circ_index(X, from, i), x = cswz(i);
                uint32_t r, j;
                if (from) {
                    r = y >> Tl;
                    j = y & (NL - 1u);
                } else {
                    const uint32_t f = (y >> X.a) & fm, P = f >> c;
                    r = P ? ~f & (fm >> 1) : f;
                    j = (P << (Tl - 1)) | ((y >> (X.a + c + 1)) << X.a) | (y & amask);
                }
                const uint32_t at = circ_map(dst + cswz(j) * (uint32_t)sizeof(C), r);
                circ_st(at, phi[x]);
                if (GRAD && both)
                    circ_st(at + NL * (uint32_t)sizeof(C), lam[x]);
            }
            circ_cluster_sync();
            return true;
        }
        C *bp = xphi + ((size_t)parity << m), *bl = xlam + ((size_t)parity << m);
        parity ^= 1;
#pragma unroll 4
        for (uint32_t i = tid; i < NL; i += nt) {
            const uint32_t y = circ_index(X, from, i), x = cswz(i);
            __stcg(bp + y, phi[x]);
            if (GRAD && both)
                __stcg(bl + y, lam[x]);
        }
        arrivals += 1u << c;
        __syncthreads();
        if (tid == 0) {
            __threadfence();
            if (!(A.drop_arrival && X.rank == 0))
                atomicAdd(A.bar + b, 1u);
            const long long t0 = clock64();
            while (*reinterpret_cast<volatile unsigned *>(A.bar + b) < arrivals)
                if (clock64() - t0 > WAIT_BUDGET_CYCLES) {
                    atomicExch(A.err, 1);
                    s_stop = 1;
                    break;
                }
            __threadfence();
        }
        __syncthreads();
        if (s_stop) {
            give_up();
            return false;
        }
#pragma unroll 4
        for (uint32_t i = tid; i < NL; i += nt) {
            const uint32_t y = circ_index(X, from ^ 1, i), x = cswz(i);
            phi[x] = __ldcg(bp + y);
            if (GRAD && both)
                lam[x] = __ldcg(bl + y);
        }
        __syncthreads();
        return true;
    };
    const int hq0 = Tl - 1 - c, hq1 = Tl - 1;  // the high layout's bits

    // ------------------------------------------------ forward sweep
    int high = 0;
    {
        C *phi = vec + X.off;
        const C *T = layer_table(0);
        const R amp0 = (R)A.amp0;
        for (uint32_t i = tid; i < NL; i += nt) {  // 2^(-n/2) i^|y| times the first cost phase
            const C z = T[cval[i]];
            phi[cswz(i)] = circ_turn(mkc<C>(amp0 * z.x, amp0 * z.y), __popc(circ_index(X, 0, i)));
        }
    }
    __syncthreads();
    for (int l = 0; l < p; l++) {
        if (l > 0) {
            C *phi = vec + X.off;
            const C *T = layer_table(l);
            for (uint32_t i = tid; i < NL; i += nt) {
                const uint32_t x = cswz(i);
                phi[x] = cmul(phi[x], T[cval[(size_t)high * NL + i]]);
            }
            __syncthreads();
        }
        const R t = (R)lay[l].t, f = (R)lay[l].f;
        for (int part = 0; part < (c ? 2 : 1); part++) {
            if (part) {
                if (!exchange(high, false))
                    return;
                high ^= 1;
            }
            circ_mix<R, 1>(X, high ? hq0 : 0, high ? hq1 : Tl, high || c == 0, t, f, CircMix<R>{(R)1, {}});
        }
    }

    // ------------------------------ energy, lambda = O phi, the state
    {
        C *phi = vec + X.off, *lam = phi + NL;
        const R fn = (R)lay[p - 1].fn;
        CircSum<R> es;
        for (uint32_t i0 = 4u * tid; i0 < NL; i0 += 4u * nt) {
            const int4 o4 = circ_cuts(s_obs, s_ow, Ko, m, circ_index(X, high, i0));
            const int ov[4] = {o4.x, o4.y, o4.z, o4.w};
#pragma unroll
            for (int j = 0; j < 4; j++) {
                const uint32_t x = cswz(i0 + j);
                C v = phi[x];
                v.x *= fn;
                v.y *= fn;
                const R o = (R)ov[j];
                es.add((v.x * v.x + v.y * v.y) * o);
                if (GRAD || A.state)
                    phi[x] = v;
                if (GRAD)
                    lam[x] = mkc<C>(v.x * o, v.y * o);
            }
        }
        double e = es.value();
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
            e += __shfl_xor_sync(0xffffffffu, e, o);
        if (lane == 0)
            red[warp] = e;
    }
    __syncthreads();
    if (A.state) {  // psi(x) = (-i)^(nK) i^(-|x|) psi~(x) and psi(~x) = psi(x)
        int K = 0;
        for (int l = 0; l < p; l++)
            K += lay[l].fi == lay[l].f ? 0 : 1;
        const C *phi = vec + X.off;
        C *dst = reinterpret_cast<C *>(A.state) + ((size_t)b << n);
        for (uint32_t i = tid; i < NL; i += nt) {
            const uint32_t y = circ_index(X, high, i);
            const C v = circ_turn(phi[cswz(i)], 4 * CIRC_MAXN - ((n * K) & 3) - __popc(y));
            dst[y] = v;
            dst[(2u << m) - 1u - y] = v;
        }
    }

    // ------------------------------------------------- adjoint sweep
    if constexpr (GRAD) {
        for (int l = p - 1; l >= 0; l--) {
            const R t = (R)-lay[l].t, f = (R)lay[l].fi;
            CircMix<R> M{(R)1, {}};
            for (int part = 0; part < (c ? 2 : 1); part++) {
                if (part) {
                    if (!exchange(high, true))
                        return;
                    high ^= 1;
                }
                M = circ_mix<R, NV>(X, high ? hq0 : 0, high ? hq1 : Tl, high || c == 0, t, f, M);
            }
            // dE/dgamma (both vectors carry 1/f^n) and the inverse cost phase
            C *phi = vec + X.off, *lam = phi + NL;
            const C *T = l > 0 ? layer_table(l) + tab_len : nullptr;
            CircSum<R> g;
            for (uint32_t i = tid; i < NL; i += nt) {
                const uint32_t x = cswz(i);
                const int cv = cval[(size_t)high * NL + i];
                const C u = phi[x], v = lam[x];
                g.add((R)cv * im_conj_mul(v, u));
                if (l > 0) {
                    const C z = T[cv];
                    phi[x] = cmul(u, z);
                    lam[x] = cmul(v, z);
                }
            }
            double gb = M.acc.value(), gg = g.value() * (lay[l].fn * lay[l].fn);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                gg += __shfl_xor_sync(0xffffffffu, gg, o);
                gb += __shfl_xor_sync(0xffffffffu, gb, o);
            }
            if (lane == 0) {
                red[(1 + l) * nw + warp] = gg;
                red[(1 + p + l) * nw + warp] = gb;
            }
            __syncthreads();
        }
    }

    // -------------------------------------------------- the results
    if (A.err_out && tid == 0 && X.rank == 0)
        *A.err_out = pending;
    // sums over the stored half count twice; dE/dgamma and dE/dbeta are
    // 2 Im of theirs. A team's CTAs are added in rank order.
    double *part = CL ? nullptr : A.partials + (((size_t)b * rows) << c);
    for (int r = tid; r < rows; r += nt) {
        double s = 0.0;
        for (int w = 0; w < nw; w++)
            s += red[r * nw + w];
        if (c == 0)
            A.out[(size_t)b * A.out_stride + r] = (r ? 4.0 : 2.0) * s;
        else if (CL)
            circ_st(circ_map(smem_u32(xred + ((size_t)r << c) + X.rank), 0), s);
        else
            __stcg(part + ((size_t)r << c) + X.rank, s);
    }
    if (c) {
        bool mine = X.rank == 0;
        if constexpr (CL) {
            circ_cluster_sync();
        } else {
            __syncthreads();
            if (tid == 0) {
                __threadfence();
                s_last = atomicAdd(A.bar + b, 1u) == arrivals + (1u << c) - 1u;
                __threadfence();
            }
            __syncthreads();
            mine = s_last;
        }
        if (mine) {
            for (int r = tid; r < rows; r += nt) {
                double s = 0.0;
                for (int k = 0; k < (1 << c); k++)
                    s += CL ? xred[((size_t)r << c) + k] : __ldcg(part + ((size_t)r << c) + k);
                A.out[(size_t)b * A.out_stride + r] = (r ? 4.0 : 2.0) * s;
            }
            if (!CL && tid == 0)
                A.bar[b] = 0u;  // every CTA is past its waits
        }
    }
}

// shared memory of one CTA with 2^Tl amplitudes per vector
static size_t circuit_smem(bool c128, bool grad, const CircuitPlan &q, int p, int tab_len)
{
    const size_t amp = c128 ? 16 : 8, rows = grad ? 1 + 2 * (size_t)p : 1;
    return ((size_t)(grad ? 2 : 1) * (q.cluster ? 2 : 1) << q.Tl) * amp +
           (size_t)2 * (q.resident ? p : 1) * tab_len * amp + rows * (q.nt / 32) * 8 +
           (q.cluster ? (rows << q.c) * 8 : 0) + ((size_t)(q.c ? 2 : 1) << q.Tl) * 2;
}

constexpr size_t CIRC_SMEM = 210 * 1024;  // dynamic; the static part is 6 KB
constexpr int CIRC_MAX_TL = 12;

// the shape with 2^c CTAs per point, or false if it does not fit
static bool circuit_shape(bool c128, bool grad, int n, int p, int tab_len, int B, int c, CircuitPlan *q)
{
    q->c = c;
    q->Tl = n - 1 - c;
    q->cluster = c >= 1 && c <= 4;
    q->a = c ? (q->Tl - 1 - c < 8 ? q->Tl - 1 - c : 8) : 0;
    if (q->Tl < 4 || q->Tl > CIRC_MAX_TL || (c && q->a < 3))
        return false;
    // Bits per register stage. A launch that leaves SMs idle is bound by the
    // latency of a stage: few amplitudes per thread (complex64 n = 10 gradient
    // 2 / 3 / 4 bits: 22.0 / 22.5 / 22.7 us, n = 11 28.0 / 24.7 us; complex128
    // n = 12, 8 CTAs, 2 / 3 bits: 63 / 79 us). A fuller one by shared memory
    // and issue: many (256 energies at n = 13 in complex64 38 -> 28 us).
    const bool fullchip = (long long)B << c > device_sms();
    q->km = fullchip ? 4 : (c128 || q->Tl < 9) ? 2 : 3;
    if (c128 && grad && q->km > 3)
        q->km = 3;
    q->nt = q->Tl > q->km ? 1 << (q->Tl - q->km) : 1;
    q->nt = q->nt < 128 ? 128 : q->nt > 512 ? 512 : q->nt;
    for (q->resident = 1; q->resident >= 0; q->resident--) {
        q->smem = circuit_smem(c128, grad, *q, p, tab_len);
        if (q->smem <= CIRC_SMEM)
            break;
    }
    if (q->resident < 0)
        return false;
    if (c && !q->cluster) {  // the CTAs of a team wait for one another: all are resident
        if (B > (device_sms() >> c) || B > CIRCUIT_MAX_POINTS)
            return false;
    }
    return true;
}

// Which calls run as one launch, and with how many CTAs per point; the passes
// take the others (measured p = 2, one point unless said, us, circuit / passes).
// * One point: complex64 up to n = 20 (n = 14 gradient 28 / 140, n = 16 40 / 137,
//   n = 20 75 / 151; energies 19 / 67, 24 / 67, 38 / 71), complex128 likewise
//   (n = 14 81 / 304, n = 16 143 / 330, n = 20 499 / 567). Few amplitudes per
//   CTA (latency, FP64 rate) against more partners to exchange with: 2^9 and up
//   to 16 CTAs (a cluster) in complex64, 2^8 in complex128; beyond that teams
//   that exchange through L2.
// * Batches: as few CTAs per point as keep the chip busy. Up to n = 14 the
//   circuit wins at every size (256 points, n = 14: energy 83 / 143, gradient
//   158 / 500; complex128 392 / 486, 1554 / 1815); above, while its CTAs are
//   few: n = 15, 64 points 48 / 84, 92 / 226; n = 16, 64 points 112 / 98 and
//   217 / 260, 256 points 396 / 198 and 801 / 764; complex128 n = 15, 16 points
//   97 / 147, 343 / 345, n = 16, 16 points 206 / 152.
bool circuit_plan(bool c128, bool grad, int n, int p, int tab_len, int B, CircuitPlan *q)
{
    if (n < CIRCUIT_MIN_QUBITS || n > CIRCUIT_MAX_QUBITS || p > CIRC_MAXP)
        return false;
    const int m = n - 1;
    int c = c128 ? (m <= 8 ? 0 : m <= 12 ? m - 8 : m <= 14 ? 4 : m <= 15 ? 5 : m <= 17 ? 6 : 7)
                 : (m <= 10 ? 0 : m <= 13 ? m - 9 : m <= 15 ? 4 : m <= 18 ? m - 11 : 7);
    const long long few = c128 ? 256 : 76;
    CircuitPlan s;
    while (c > 0 && ((long long)B << c) > few && circuit_shape(c128, grad, n, p, tab_len, B, c - 1, &s))
        c--;
    while (c <= 7 && !circuit_shape(c128, grad, n, p, tab_len, B, c, q))
        c++;
    if (c > 7)
        return false;
    if (n <= 14 || !q->cluster)
        return true;
    return c128 ? ((long long)B << m) <= (1 << 18) : ((long long)B << c) <= (grad ? 512 : 256);
}

template <typename R, bool GRAD, bool CL>
static int launch_circuit_t(const CircuitArgs &a, const CircuitPlan &q, cudaStream_t st)
{
    static std::atomic<unsigned long long> ready{0};  // devices whose kernel attributes are set
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess)
        return (int)e;
    const unsigned long long bit = 1ull << (dev & 63);
    if (dev > 63 || !(ready.load() & bit)) {
        e = cudaFuncSetAttribute(k_circuit<R, GRAD, CL>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)CIRC_SMEM);
        if (e == cudaSuccess && CL)
            e = cudaFuncSetAttribute(k_circuit<R, GRAD, CL>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        if (e != cudaSuccess)
            return (int)e;
        ready.fetch_or(bit);
    }
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    if (CL) {
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = 1u << q.c;
        at[0].val.clusterDim.y = 1;
        at[0].val.clusterDim.z = 1;
    } else {
        at[0].id = cudaLaunchAttributeCooperative;
        at[0].val.cooperative = 1;
    }
    cfg.gridDim = dim3((unsigned)a.B << q.c);
    cfg.blockDim = dim3(q.nt);
    cfg.dynamicSmemBytes = q.smem;
    cfg.stream = st;
    cfg.attrs = at;
    cfg.numAttrs = q.c ? 1 : 0;
    e = cudaLaunchKernelEx(&cfg, k_circuit<R, GRAD, CL>, a);
    return (int)(e != cudaSuccess ? e : cudaGetLastError());
}

template <typename R>
static int launch_circuit_r(bool grad, const CircuitArgs &a, const CircuitPlan &q, cudaStream_t st)
{
    if (q.cluster)
        return grad ? launch_circuit_t<R, true, true>(a, q, st) : launch_circuit_t<R, false, true>(a, q, st);
    return grad ? launch_circuit_t<R, true, false>(a, q, st) : launch_circuit_t<R, false, false>(a, q, st);
}

int launch_circuit(bool c128, bool grad, const CircuitArgs &a, const CircuitPlan &q, cudaStream_t st)
{
    return c128 ? launch_circuit_r<double>(grad, a, q, st) : launch_circuit_r<float>(grad, a, q, st);
}

}  // namespace aaq
