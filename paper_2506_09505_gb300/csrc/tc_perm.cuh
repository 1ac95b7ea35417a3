// Poseidon-12 permutation with its dense contractions on the tensor cores
// (tcgen05, sm_103a), 128 states per group of 128 threads.
//
// Alg. 1's full rounds are x <- M S(x + c_r); the 12x12 products M y of a
// whole group are one tensor-core contraction of byte limbs (the digit scheme
// of TcTables and TcDev in pg12_internal.h):
//
//   thread t: y_j = S(x_j) R^-6 (Montgomery products, field.cuh), its 8 bytes
//             -> row t of A (fp16 subnormals, bits = byte), in shared memory
//   leader  : D[128 x 96] = A[128 x 96] * B^T + bias   (7 tcgen05.mma, K = 16
//             each, fp32 accumulators in tensor memory), commit -> mbarrier
//   thread t: reads row t of D (tcgen05.ld), y_i = sum_b 2^(8b) bits(D[t][8i+b])
//             folded mod p: M is stored times R^6 and the bias holds the next
//             round's constants, so this is the next S-box input
//
// The 22 partial rounds (Alg. 1, MDSPartial) run in their unrolled form
// (ChainParams): the dot products U_q with the partial rounds' input and the
// deferred cell updates W s are contractions of round 3's S-box bytes and of
// the 22 partial S-box outputs; only the chain c_q -> s_q = S(c_q + k_q) ->
// c_(q+1) = U_q + sum_(r<=q) beta[q][r] s_r runs on the integer pipes, one
// thread per state, in two halves: the first half's terms in the second
// half's chain values are one more contraction, and the values are scaled so
// that beta[q][q] = 1 (KernelParams), so each thread forms 90 of the 231
// products beta[q][r] s_r.
//
// Every fp32 sum is an exact integer below 2^24 (times 2^-24), so each result
// is the exact residue: the same function as the integer-pipe form, bit for
// bit after canonicalisation.  A group's threads meet at one named barrier
// per contraction (operands written, the previous accumulators read) and
// wait on the group's mbarrier for the tensor cores; every wait is bounded.
#pragma once
#include <cstddef>

#include "poseidon.cuh"
#include "tcgen05.cuh"

namespace pg12 {
namespace dev {

constexpr int kTcGroup = 128;                   // states per group
constexpr int kTcAChunk = 128;                  // bytes of one 8 x 8 fp16 core matrix
constexpr int kTcAChunks = kTcK / 8;            // core-matrix columns of A (12 input words)
constexpr int kTcABytes = kTcGroup * kTcK * 2;  // A operand of a group: 24 KiB
constexpr int kTcRegion = 128;                  // tensor-memory columns of one group
constexpr int kTcUStore = kTcN;                 // columns 96..119 of a region hold chain values as words
// tensor-memory columns one CTA of `groups` groups allocates (a power of two)
constexpr int tc_tmem_alloc(int groups) { return groups <= 1 ? 128 : groups <= 2 ? 256 : 512; }

// byte offsets of the tables inside TcDev (and inside its shared-memory copy)
constexpr uint32_t kTabM = offsetof(TcDev, m), kTabPre = offsetof(TcDev, pre);
constexpr uint32_t kTabBBias = offsetof(TcDev, b_bias), kTabABias = offsetof(TcDev, a_bias);
constexpr uint32_t kTabZcap = offsetof(TcDev, a_zcap);
constexpr uint32_t kTabVpa = offsetof(TcDev, vpa), kTabVpb = offsetof(TcDev, vpb), kTabBs = offsetof(TcDev, bs);
constexpr uint32_t kTabW1 = offsetof(TcDev, w1), kTabW2 = offsetof(TcDev, w2);
static_assert(kTabVpa % 128 == 0 && kTabVpb % 128 == 0 && kTabBs % 128 == 0 && kTabW1 % 128 == 0 &&
                  kTabW2 % 128 == 0 && kTabBBias % 128 == 0 && kTabABias % 128 == 0 && kTabZcap % 128 == 0,
              "tables are 128-byte aligned");

__device__ __align__(16) TcDev g_tc;        // uploaded with the other constant tables
__constant__ uint64_t c_beta[kRP][kRP];     // the chain's coefficients beta~ times R

// One group's share of the CTA's shared memory and tensor memory.  A state is
// held by TPS threads: 1 where many groups are in flight (the fewest
// instructions), 4 where a launch leaves SMs with one group or two and the
// latency of a permutation counts (each thread then does a quarter of the
// S-boxes and combinations of a round; the chain stays in one thread per state).
template <int TPS>
struct TcGroup {
    static constexpr int kThreads = kTcGroup * TPS;
    static constexpr int kWords = kT / TPS;  // words of a state held by one thread
    uint8_t *a;           // A operand, kTcABytes
    uint64_t *mbar;       // tensor-core completion barrier
    uint32_t tmem;        // the group's kTcRegion columns, lanes 0..127
    uint32_t phase;       // parity of the mbarrier's next completion
    int bar;              // named barrier of the group's threads
    int t;                // thread index within the group
    uint32_t failed;      // this thread saw a tensor-core wait run out
    volatile uint32_t *bcast;  // one word through which thread 0 hands the group a value
    uint32_t a_addr, tab;      // shared addresses of A and of the tables

    __device__ __forceinline__ int row() const { return TPS == 1 ? t : t % kTcGroup; }   // its state
    __device__ __forceinline__ int part() const { return TPS == 1 ? 0 : t / kTcGroup; }  // which of the TPS threads
    // word i of the thread is word TPS i + part of the state: every part holds the
    // same number of rate, capacity and digest words
    __device__ __forceinline__ int word(int i) const { return TPS * i + part(); }
    // its warp's lanes of the group's tensor memory
    __device__ __forceinline__ uint32_t lane_base() const { return tmem + ((uint32_t)(row() & ~31) << 16); }
};

// The row's chunk j of A (K columns 8j..8j+7) <- the 8 bytes of y as fp16 subnormals.
template <int TPS>
__device__ __forceinline__ void tc_put(const TcGroup<TPS> &G, int j, uint64_t y) {
    const int r = G.row();
    *reinterpret_cast<uint4 *>(G.a + ((r >> 3) * kTcAChunks + j) * kTcAChunk + (r & 7) * 16) = tc_bytes(y);
}

// One contraction into the group's D (columns 0 .. n-1): the group meets
// (its A stores visible to the tensor cores, its earlier tensor-memory
// accesses done), a lane of warp 0 issues the bias block of kind `bias` (D starts at
// the bias; bias < 0: D accumulates) and the six K = 16 blocks of A (cells
// 8..11 from the zero-capacity block when z) against the table at byte offset
// b_off, and commits; every thread waits.  Returns false, in every thread of
// the group, once a wait of the group has run out.
template <int TPS>
__device__ __forceinline__ bool tc_contract(TcGroup<TPS> &G, uint32_t b_off, int n, int bias, bool z) {
    fence_async_smem();   // this thread's A stores -> the tensor cores' proxy
    tc_fence_before();    // its tensor-memory accesses are complete
    if (group_sync_or(G.bar, G.failed, TcGroup<TPS>::kThreads)) return false;
    if (G.t < 32) {
        tc_fence_after();
        const uint32_t idesc = tc_idesc(n);
        const uint32_t sbo = kTcAChunks * kTcAChunk;
        // warp-uniform operands and an elected lane: the descriptors stay in
        // uniform registers, which the instruction reads
        const uint32_t d = __shfl_sync(0xFFFFFFFFu, G.tmem, 0);
        const uint64_t a0 = tc_desc(__shfl_sync(0xFFFFFFFFu, G.a_addr, 0), kTcAChunk, sbo);
        const uint64_t b0 = tc_desc(G.tab + b_off, kTcAChunk, sbo);
        if (tc_elect()) {
            if (bias >= 0) {
                // K chunks (H_k, Z) for kind k < 8, (Z, H_(k-8)) above: see TcDev::a_bias
                const uint32_t first = bias < 8 ? 1u + bias : 0u, lbo = bias < 8 ? 8u - bias : bias - 7u;
                tc_mma(d, tc_desc(G.tab + kTabABias + first * kTcAChunk, lbo * kTcAChunk, 0),
                       tc_desc(G.tab + kTabBBias, kTcAChunk, 2 * kTcAChunk), idesc, 0);
            }
#pragma unroll
            for (int kb = 0; kb < kTcK / 16; ++kb) {
                uint64_t a = a0 + (kb * 2 * kTcAChunk >> 4);
                if (z && kb >= 4) a = tc_desc(G.tab + kTabZcap + (kb - 4) * 2 * kTcAChunk, kTcAChunk, 0);
                tc_mma(d, a, b0 + (kb * 2 * kTcAChunk >> 4), idesc, 1);
            }
            tc_commit(G.mbar);
        }
        __syncwarp();
    }
    const bool ok = mbar_wait(G.mbar, G.phase);
    G.phase ^= 1u;
    if (!ok) G.failed = 1;
    tc_fence_after();
    return true;
}

// f(i, w) for the rows G.word(i) < ROWS of D, i = 0 .. n-1, w their eight column
// words; the next load is in flight during f.  One thread per state loads pairs
// of rows.  Row counts that are no multiple of TPS leave the last row to some
// parts (whole warps).
template <int TPS, int ROWS, class F>
__device__ __forceinline__ void tc_rows(const TcGroup<TPS> &G, F &&f) {
    constexpr int kStep = TPS == 1 ? 2 : 1, kN = (ROWS + TPS - 1) / TPS;
    const uint32_t base = G.lane_base();
    auto has = [&](int i) { return ROWS % TPS == 0 || i < ROWS / TPS || G.word(i) < ROWS; };
    auto load = [&](int i, uint32_t(&w)[16]) {
        if (TPS == 1) tmem_ld16_start(base + 8 * i, w);
        else tmem_ld8_start(base + 8 * G.word(i), w);
    };
    uint32_t w[2][16];
    load(0, w[0]);
#pragma unroll
    for (int i = 0; i < kN; i += kStep) {
        const int k = (i / kStep) & 1;
        tmem_ld_wait();
        if (i + kStep < kN && has(i + kStep)) load(i + kStep, w[k ^ 1]);
        if (has(i)) {
            f(i, w[k]);
            if (kStep == 2) f(i + 1, w[k] + 8);
        }
    }
}

// Dense layer of round r (table at m_off) on the S-box outputs in A, plus the
// next constants (the bias of kind r); with `digest` only words 0..3 of the
// result are formed.  z: round 0 of states whose capacity entered as zero (A
// holds cells 0..7; cells 8..11 come from the constant zcap block).
template <int TPS>
__device__ __forceinline__ bool tc_dense(TcGroup<TPS> &G, uint32_t m_off, int r, bool z, bool digest,
                                         uint64_t (&x)[kT / TPS]) {
    if (!tc_contract(G, m_off, kTcN, kBiasDense + r, z)) return false;
    auto out = [&](int i, const uint32_t *w) { x[i] = tc_combine(w); };
    if (digest) tc_rows<TPS, kDigest>(G, out);
    else tc_rows<TPS, kT>(G, out);
    return true;
}

// One half of the chain on the scaled values of KernelParams: s_q = f(z_q) for
// q = q0 .. q0 + 10, each into A's chunk q - q0, from c = z_q0; between them
// z_(q+1) = U_q + sum_(r = q0 .. q-1) beta~[q][r] s_r + s_q, U_q (its bias
// includes the round constant) the word in tensor-memory column kTcUStore +
// 2 (q - u0).  The sum does not wait for s_q's S-box.  Unrolled, so the s_r stay
// in registers (reading them back from A's bytes in a loop: a 2^22 x 8 tree
// 5.69 ms against 5.57).
static_assert(kRP == 2 * kTcSplit, "the halves have the same length");
// u: the words U_(q0) .. as pairs, u[2 k] and u[2 k + 1] from column kTcUStore + 2 k.
template <int TPS>
__device__ __forceinline__ void chain_half(const TcGroup<TPS> &G, uint64_t c, int q0, const uint32_t *u) {
    uint64_t s[kTcSplit];
#pragma unroll
    for (int q = 0;; ++q) {
        uint64_t t = 0;
        if (q < kTcSplit - 1) {
            t = ((uint64_t)u[2 * q + 1] << 32) | u[2 * q];
            if (q > 0) {
                MAcc A;
                macc_init(A, t);
#pragma unroll
                for (int r = 0; r < q; ++r) macc(A, s[r], c_beta[q + q0][r + q0]);
                t = macc_reduce(A);
            }
        }
        s[q] = msbox(c);
        tc_put(G, q, s[q]);
        if (q == kTcSplit - 1) break;
        c = add_fold(t, s[q]);
    }
}
// The stored words 0 .. 11 of the thread's state as 24 columns.
__device__ __forceinline__ void tc_load_words(uint32_t base, uint32_t (&u)[32]) {
    uint32_t a[16], b[16];
    tmem_ld16_start(base, a);
    tmem_ld8_start(base + 16, b);
    tmem_ld_wait();
#pragma unroll
    for (int i = 0; i < 16; ++i) u[i] = a[i];
#pragma unroll
    for (int i = 0; i < 8; ++i) u[16 + i] = b[i];
}

// Rows 0 .. ROWS-1 of D combined into words, stored at tensor-memory columns
// kTcUStore + 2 i.
template <int ROWS, int TPS>
__device__ __forceinline__ void tc_store_rows(const TcGroup<TPS> &G) {
    const uint32_t base = G.lane_base() + kTcUStore;
    uint64_t even = 0;
    tc_rows<TPS, ROWS>(G, [&](int i, const uint32_t *w) {
        const uint64_t v = tc_combine(w);
        if (TPS > 1) tmem_st_word(base + 2 * G.word(i), v);
        else if (i & 1) tmem_st_words(base + 2 * (i - 1), even, v);
        else even = v;
    });
    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}

// The 22 partial rounds in their unrolled form, after round 3's dense layer
// (A still holds round 3's S-box bytes y3, x holds x^(0) = P y3, cell 0 as z_0);
// x leaves with round 4's constants added.  The chain runs in the threads that
// hold cell 0; the others wait at the next contraction.
template <int TPS>
__device__ __forceinline__ bool tc_partial(TcGroup<TPS> &G, uint64_t (&x)[kT / TPS]) {
    const uint32_t lane_base = G.lane_base();
    // U_0 .. U_9 as words
    if (!tc_contract(G, kTabVpa, kTcUa * 8, kBiasUa, false)) return false;
    tc_store_rows<kTcUa>(G);
    // U_10 .. U_21 as column sums in D (A still holds y3)
    if (!tc_contract(G, kTabVpb, kTcN, kBiasUb, false)) return false;
    // first half: s_0 .. s_10 into A's chunks 0..10
    if (G.part() == 0) {
        uint32_t u[32];
        tc_load_words(lane_base + kTcUStore, u);
        chain_half(G, x[0], 0, u);
    }
    // D += their terms in z_11 .. z_21: the second half's U'_q (q = 10 .. 20) and U_21, as words
    if (!tc_contract(G, kTabBs, kTcN, -1, false)) return false;
    tc_store_rows<kT>(G);
    // the deferred updates W s, from s_0 .. s_10 now, s_11 .. s_21 after the second half
    if (!tc_contract(G, kTabW1, kTcN, kBiasW, false)) return false;
    if (G.part() == 0) {
        uint32_t u[32];
        tc_load_words(lane_base + kTcUStore, u);
        chain_half(G, ((uint64_t)u[1] << 32) | u[0], kTcSplit, u + 2);
    }
    if (!tc_contract(G, kTabW2, kTcN, -1, false)) return false;
    // cell 0 = c_22 = U_21 + (W s)_0, cell i = x_i^(0) + (W s)_i
    const uint64_t u21 = tmem_ld_word(lane_base + kTcUStore + 2 * (kRP - 1 - kTcUa));
    if (G.part() == 0) x[0] = u21;
    tc_rows<TPS, kT>(G, [&](int i, const uint32_t *w) { x[i] = tc_combine(w, x[i]); });
    return true;
}

// The permutation on x, the thread's words of a state in registers (weak words
// in, weak words out).  zcap: cells 8..11 enter as zero (their round 0 S-box
// outputs are constants, read from a_zcap); digest: only cells 0..3 of the
// result are read and formed.  Each round's S-boxes and output rows are
// unrolled (the state never leaves registers).  Round 0's constants are added
// here, all later ones by the contractions' biases.
template <int TPS>
__device__ __forceinline__ bool tc_permute(TcGroup<TPS> &G, uint64_t (&x)[kT / TPS], bool zcap, bool digest) {
#pragma unroll
    for (int i = 0; i < kT / TPS; ++i) x[i] = add_canon(x[i], c_dev.full_rc[0][G.word(i)]);
#pragma unroll 1
    for (int r = 0; r < kRF; ++r) {
        const bool z = zcap && r == 0;
#pragma unroll
        for (int i = 0; i < kRate / TPS; ++i) tc_put(G, G.word(i), msbox(x[i]));
        if (!z) {
#pragma unroll
            for (int i = kRate / TPS; i < kT / TPS; ++i) tc_put(G, G.word(i), msbox(x[i]));
        }
        const bool mid = r == kRF / 2 - 1;
        if (!tc_dense(G, mid ? kTabPre : kTabM, r, z, digest && r == kRF - 1, x)) return false;
        if (mid && !tc_partial(G, x)) return false;
    }
    return true;
}

// Shared-memory layout of a CTA of GROUPS groups: the tables, then each
// group's A operand, then the barriers.
template <int GROUPS>
struct TcLayout {
    static_assert(GROUPS * kTcRegion <= 512, "the groups' tensor memory exceeds the SM's");
    static constexpr int kTmemCols = tc_tmem_alloc(GROUPS);
    static constexpr size_t kTables = 0;
    static constexpr size_t kA = (sizeof(TcDev) + 127) & ~(size_t)127;
    static constexpr size_t kBar = kA + (size_t)GROUPS * kTcABytes;
    static constexpr size_t kTabBar = kBar + 8 * GROUPS;
    static constexpr size_t kTmemSlot = kTabBar + 8;
    static constexpr size_t kBcast = kTmemSlot + 8;
    static constexpr size_t kBytes = kBcast + 4 * GROUPS;
    static_assert(kBytes <= 232448, "a block has at most 227 KB of shared memory");
};

__device__ int g_tc_fault;  // set when a tensor-core wait ran out (read by pg_device_faults)

// Prologue of a tensor-core kernel: the copy of the tables into shared memory
// started (one bulk copy; with 131 KB of 16-byte loads through registers a launch
// of one unit took 28.7 us instead of 21.6), the groups' barriers, one
// tensor-memory allocation for all groups.  tc_tables_ready follows.
template <int TPS, int GROUPS>
__device__ __forceinline__ TcGroup<TPS> tc_setup(uint8_t *sm) {
    using L = TcLayout<GROUPS>;
    uint64_t *bars = reinterpret_cast<uint64_t *>(sm + L::kBar);
    uint64_t *tab_bar = reinterpret_cast<uint64_t *>(sm + L::kTabBar);
    uint32_t *tslot = reinterpret_cast<uint32_t *>(sm + L::kTmemSlot);
    if (threadIdx.x == 0) {
        for (int g = 0; g <= GROUPS; ++g)  // the groups' barriers, then the tables'
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(bars + g)));
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        fence_async_smem();
        bulk_copy(sm + L::kTables, &g_tc, sizeof(TcDev), tab_bar);
    }
    if (threadIdx.x < 32) {
        __syncwarp();
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(tslot)),
                     "r"(L::kTmemCols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    fence_async_smem();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const int g = threadIdx.x / TcGroup<TPS>::kThreads;
    TcGroup<TPS> G;
    G.t = threadIdx.x % TcGroup<TPS>::kThreads;
    G.failed = 0;
    G.a = sm + L::kA + (size_t)g * kTcABytes;
    G.mbar = bars + g;
    G.tmem = *tslot + (uint32_t)(g * kTcRegion);
    G.phase = 0;
    G.bar = 1 + g;
    G.bcast = reinterpret_cast<volatile uint32_t *>(sm + L::kBcast) + g;
    G.a_addr = smem_addr(G.a);
    G.tab = smem_addr(sm + L::kTables);
    return G;
}

// The warps that issue the contractions wait for the tables (bounded); every
// kernel calls this once, after whatever else it has to wait for.
template <int TPS, int GROUPS>
__device__ __forceinline__ void tc_tables_ready(uint8_t *sm, TcGroup<TPS> &G) {
    if (G.t < 32 && !mbar_wait(reinterpret_cast<uint64_t *>(sm + TcLayout<GROUPS>::kTabBar), 0)) G.failed = 1;
}

// Thread 0 adds one to *counter; every thread of the group gets the old
// value.  The first barrier orders the group's earlier stores (each thread
// fences its own first) before the atomic and keeps thread 0 from
// overwriting a value others have not read yet.
template <int TPS>
__device__ __forceinline__ uint32_t group_fetch_add(TcGroup<TPS> &G, uint32_t *counter) {
    group_sync(G.bar, TcGroup<TPS>::kThreads);
    if (G.t == 0) *G.bcast = atomicAdd(counter, 1u);
    group_sync(G.bar, TcGroup<TPS>::kThreads);
    return *G.bcast;
}

// Epilogue: every group is done with tensor memory; the allocating warp
// frees it.  A group whose wait ran out records the fault and gives the table
// copy and its last contraction one more bounded wait each before the memory is
// freed: neither may land in shared or tensor memory that is no longer ours.
template <int TPS, int GROUPS>
__device__ __forceinline__ void tc_teardown(uint8_t *sm, TcGroup<TPS> &G) {
    using L = TcLayout<GROUPS>;
    if (G.failed) {
        atomicExch(&g_tc_fault, 1);
        if (G.t == 0) {
            mbar_wait(reinterpret_cast<uint64_t *>(sm + L::kTabBar), 0);
            mbar_wait(G.mbar, G.phase ^ 1u);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (threadIdx.x < 32) {
        tc_fence_after();
        const uint32_t base = *reinterpret_cast<uint32_t *>(sm + L::kTmemSlot);
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(base), "r"(L::kTmemCols));
    }
}

}  // namespace dev
}  // namespace pg12
