// cluster.cu -- step (ii) of the EMCS (Sec. 3): the all-cluster Houdayer
// update (ACU) and the original single-cluster Houdayer move.
//
// One replica pair at one temperature belongs to a group of LN lanes of a
// warp (LN = 4, 8, 16 or 32 lanes, the smallest that holds L): lane = y, and
// the rows z = 0..L-1 of that y sit in the lane's registers as L-bit masks
// (bit x).  The site overlaps q_i = s^a_i s^b_i (Eq. (2)) are one XOR per
// row.  The clusters -- connected components of {i ~ j : neighbours,
// q_i = q_j} -- are flooded as bit masks:
//  1. sites with no equal neighbour are clusters of their own; they drop out
//     in one pass of bit operations over all rows;
//  2. the first unlabelled site in site order is the next cluster's canonical
//     label (its smallest site).  Its cluster grows from that site: a row
//     takes in what its y and z neighbours hold, and a carry through the row's
//     mask (m + s, and the same on the reversed row) fills whole runs along x,
//     until a pass changes nothing.  For L <= 16 one cluster of each sign of q
//     floods at a time, in the two halves of a word.
// A thermalised pair (L = 12 to 16) has one large cluster of each sign, which
// take about ten passes, and one to three others of more than one site.  A
// pair that needs more than MAX_FLOODS turns (an overlap of hundreds of small
// domains) is relabelled by the whole block with a union-find over its sites,
// whose cost does not depend on the number of clusters.
// One sign per cluster is drawn from Philox keyed by the label; the flips are
// XORed into both clones' words and the energies are updated (on the coupling
// grid from the bonds that the flips cut or spare, whichever are fewer, H_b
// following from the conserved H_a + H_b).  Every loop is bounded; hitting a
// bound sets STATUS_NOCONVERGE and leaves the pair as it was.
//
// What bounds it: instruction issue and latency of the floods' serial chains
// (40% issue active, DRAM 12% at L = 12); it reads each clone once and the rows
// that flip twice.
// Whole launch, thermalised, against the block-per-pair union-find over sites
// that it replaces: L = 12, 28672 pairs 203 us (611 us); L = 16, 18432 pairs
// 247 us (887 us); L = 8, 5120 pairs 36 us (44 us); at a random start, where
// clusters are many, 269 us (705 us) and 356 us (1000 us).  Launches of few
// pairs have a block each (pair_kernel); between the two, a launch lasts as
// long as one warp's chain: L = 14, 840 pairs 45 us (49 us).
#include "kernels.cuh"
#include "bitrows.cuh"

namespace pthr {

namespace {

constexpr int MAX_FLOODS = 64;   // turns of flooding per pair before the union-find takes over

template <int L>
struct ClusterGeom {
    static constexpr int LN = L <= 4 ? 4 : (L <= 8 ? 8 : (L <= 16 ? 16 : 32));   // lanes per pair
    static constexpr int PPW = 32 / LN;                                          // pairs per warp
};
template <bool WIDE> struct RowType { typedef uint16_t T; };
template <> struct RowType<true> { typedef uint32_t T; };

// A list of bonds of one pair: site, direction (2 bits), sign (1 bit).
template <int L>
struct BondList {
    static constexpr int SITE_BITS = L <= 16 ? 12 : 14;
    typedef typename RowType<(L > 16)>::T Entry;         // 15 or 17 bits
    static constexpr int N = 3 * L * L + L * L / 2;      // entries
};

// Shared memory: three row arrays and a bond list per pair of the block, then
// the union-find's parents [V] and sizes [V], 16 bits each (V <= 24^3), and
// the pairs' records.
template <int L>
constexpr size_t cluster_smem(int threads) {
    typedef typename RowType<(L > 16)>::T Row;
    const size_t slots = (size_t)(threads / 32) * ClusterGeom<L>::PPW;
    const size_t rows = slots * (3 * L * L + BondList<L>::N) * sizeof(Row);
    return ((rows + 15) & ~(size_t)15) + 2 * (((size_t)L * L * L * 2 + 15) & ~(size_t)15) + slots * 7 * sizeof(int);
}

// ------------------------------------------------------------ union-find
// Parent: 16 bits, or int where the memory allows it.
template <typename Parent>
__device__ __forceinline__ int find_root(volatile Parent *parent, int x, int cap, bool &ok,
                                         uint32_t *status, int V) {
    for (int it = 0; it < cap; ++it) {
        const int p = parent[x];
        if (p == x) return x;
#ifdef PTHR_DEBUG
        if (!PTHR_DCHECK(status, p >= 0 && p < V && (int)parent[p] < V)) { ok = false; return x; }
#endif
        const int gp = parent[p];
        if (gp != p) parent[x] = (Parent)gp;   // path halving: gp is an ancestor of x
        x = gp;
    }
    ok = false;
    return x;
}

// The root of x without writing anything.  For flattening after every join
// is done: the forest no longer changes, but other threads are writing the
// final roots, and a path-halving store could replace a final root with an
// intermediate ancestor after its owner wrote it.
template <typename Parent>
__device__ __forceinline__ int find_root_readonly(volatile Parent *parent, int x, int cap, bool &ok,
                                                  uint32_t *status, int V) {
    for (int it = 0; it < cap; ++it) {
        const int p = parent[x];
        if (p == x) return x;
#ifdef PTHR_DEBUG
        if (!PTHR_DCHECK(status, p >= 0 && p < V)) { ok = false; return x; }
#endif
        x = p;
    }
    ok = false;
    return x;
}

__device__ __forceinline__ uint16_t swap_root(volatile uint16_t *p, uint16_t a, uint16_t b) {
    return atomicCAS(const_cast<unsigned short *>((volatile unsigned short *)p), a, b);
}
__device__ __forceinline__ int swap_root(volatile int *p, int a, int b) {
    return atomicCAS(const_cast<int *>(p), a, b);
}

template <typename Parent>
__device__ __forceinline__ void unite(volatile Parent *parent, int a, int b, int cap, bool &ok,
                                      uint32_t *status, int V) {
    for (int it = 0; it < cap; ++it) {
        a = find_root(parent, a, cap, ok, status, V);
        b = find_root(parent, b, cap, ok, status, V);
        if (!ok || a == b) return;
        if (a < b) { const int t = a; a = b; b = t; }   // hook the larger root a under b
        if (swap_root(&parent[a], (Parent)a, (Parent)b) == (Parent)a) return;
    }
    ok = false;
}

struct PairStats { int nclus, top1, top2; };

__device__ __forceinline__ void add_size(PairStats &s, int c) {
    ++s.nclus;
    if (c > s.top1) { s.top2 = s.top1; s.top1 = c; } else if (c > s.top2) { s.top2 = c; }
}

// ------------------------------------------------------------ rows
// Rows whose words are loaded together (a divisor of L)
__host__ __device__ constexpr int rows_in_flight(int L) {
    const int most = L > 16 ? 4 : 8;
    for (int n = most; n > 1; --n)
        if (L % n == 0) return n;
    return 1;
}

// flip mask of packed word j (bit 7 of byte k: site 4j + k of the colour
// row) from the natural row's flip bits shifted to the colour's parity
__device__ __forceinline__ uint32_t word_flips(uint32_t v, int j) {
    return (((v >> (8 * j)) & 0x55u) * 0x02082080u) & 0x80808080u;
}

// 2^18 J (negated: -2^18 J) as an integer (adding 1.5 2^23 rounds to one); bad
// is set where the integer does not give J back.  By value: a zero of either
// sign is on the grid.
__device__ __forceinline__ int bond_int(float j, bool negated, uint32_t &bad) {
    const int v = __float_as_int(fmaf(j, 262144.f, 12582912.f)) - 0x4B400000;
    bad |= (float)v * 3.814697265625e-06f != j;
    return negated ? -v : v;
}

// Adds the sums of J s_i s_j over the forward bonds of row r after the flips to
// Ea (clone a) and Eb (clone b): FP32 pairs over half a row's bonds (at most 36
// terms), added up in FP64.  (The low part of one pair over a lane's 3 L^2
// bonds would itself round: L = 24 2e-14 of the energy, 2e-16 so.)  U: sites
// whose couplings are loaded together.
template <int L, int U, typename Row>
__device__ __forceinline__ void row_energies(const float *J, const Row *qs, const Row *as, const Row *Fs, int r,
                                             double &Ea, double &Eb) {
    constexpr int V = L * L * L;
    const int y = r % L, z = r / L;
    const int ry = (y + 1 == L ? 0 : y + 1) + L * z, rz = y + L * (z + 1 == L ? 0 : z + 1);
    const uint32_t ar = as[r] ^ Fs[r], ay = as[ry] ^ Fs[ry], az = as[rz] ^ Fs[rz];
    const uint32_t br = ar ^ qs[r], by = ay ^ qs[ry], bz = az ^ qs[rz];
    const uint32_t na[3] = {ar ^ rot_next<L>(ar), ar ^ ay, ar ^ az};
    const uint32_t nb[3] = {br ^ rot_next<L>(br), br ^ by, br ^ bz};
#pragma unroll 1
    for (int x0 = 0; x0 < L; x0 += L / 2) {
        float h = 0.f, l = 0.f, h2 = 0.f, l2 = 0.f;
#pragma unroll U
        for (int x = x0; x < x0 + L / 2; ++x) {
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                const float j = __ldg(J + d * V + L * r + x);
                two_sum_acc(h, l, ((na[d] >> x) & 1u) ? -j : j);
                two_sum_acc(h2, l2, ((nb[d] >> x) & 1u) ? -j : j);
            }
        }
        Ea += (double)h + (double)l;
        Eb += (double)h2 + (double)l2;
    }
}

// The same over the rows z of one y; a call of its own, so that its registers are
// not the flooding kernel's (L = 12, 256 samples, three batches, on the grid 50.4
// us per launch inline, 48.3 so; 48.7 before the energies summed half rows).
template <int L, typename Row>
__device__ __noinline__ double2 column_energies(const float *J, const Row *qs, const Row *as, const Row *Fs, int y) {
    double Ea = 0.0, Eb = 0.0;
    for (int z = 0; z < L; ++z) row_energies<L, L / 2>(J, qs, as, Fs, y + L * z, Ea, Eb);
    return make_double2(Ea, Eb);
}

// flip bits of bit word i of a lattice in the bit layout, from its flip rows
template <int L, typename Row>
__device__ __forceinline__ uint32_t flip_bits(const Row *Fs, int i) {
    constexpr int ROWS = Geom<L>::ROWS, W = Geom<L>::W;
    uint32_t m = 0;
#pragma unroll
    for (int t = 0; t < 8; ++t) {
        const int w = 8 * i + t;
        const int c = w / (ROWS * W), g = w - c * ROWS * W;
        const int r = g / W, j = g - r * W;
        m |= (compact_bits((uint32_t)Fs[r] >> ((c + r % L + r / L) & 1)) >> (4 * j) & 0xFu) << (4 * t);
    }
    return m;
}

// ------------------------------------------------------------ items
struct PairItem {
    bool live;
    int s, P, k, la, lb;
    uint32_t emcs, pair_id;
    unsigned long long seed;
};

__device__ __forceinline__ PairItem pair_item(const ClusterArgs &a, int item) {
    const Batch &b = a.b;
    PairItem p{};
    if (item >= a.sample_count * b.NPAIR * b.n_acu) return p;
    int t = item;
    p.k = t % b.n_acu; t /= b.n_acu;
    p.P = t % b.NPAIR; t /= b.NPAIR;
    p.s = a.sample_first + t;
    if (!PTHR_DCHECK(b.status, p.s >= 0 && p.s < b.S && p.k < b.NT && p.P < b.NPAIR)) return PairItem{};
    if (!b.active[p.s]) return p;
    p.emcs = b.emcs[p.s];
    if (!a.label_only && (p.emcs % (uint32_t)b.acu_interval) != 0u) return p;
    p.seed = b.seeds[p.s];
    const int ga = 2 * p.P, gb = 2 * p.P + 1;
    p.la = ga * b.NSLOT + b.perm[((size_t)p.s * b.NR + ga) * b.NSLOT + p.k];
    p.lb = gb * b.NSLOT + b.perm[((size_t)p.s * b.NR + gb) * b.NSLOT + p.k];
    if (!PTHR_DCHECK(b.status, p.la >= ga * b.NSLOT && p.la < (ga + 1) * b.NSLOT &&
                                p.lb >= gb * b.NSLOT && p.lb < (gb + 1) * b.NSLOT && gb < b.NR)) return PairItem{};
    p.pair_id = (uint32_t)(p.P * b.NT + p.k);
    p.live = true;
    return p;
}

// eta = -1 iff the top bit of word 0 of (label, pair_id, emcs, TAG_ACU)
__device__ __forceinline__ bool cluster_sign(const PairItem &p, int label) {
    return (philox_word0(p.seed, (uint32_t)label, p.pair_id, p.emcs, TAG_ACU) >> 31) != 0u;
}

// Labels, flips and sizes of one pair of the block by union-find over its
// sites (all threads of the block).  Fs receives the flip rows.
//  1. runs of equal q along each x row (with the periodic wrap) become stars
//     rooted at their smallest site;
//  2. a lock-free union-find in shared memory joins runs across y and z
//     edges, always hooking the larger root under the smaller one, so every
//     root is the smallest site index of its cluster (the canonical label).
//     An edge whose left neighbours in both rows are in the same two runs is
//     implied by that neighbouring edge and skipped; x = 0 never skips.
template <int L, typename Row, typename Parent>
__device__ __forceinline__ bool union_find(const ClusterArgs &a, const PairItem &p, int target, const Row *qs,
                                           Row *Fs, Parent *parent, uint16_t *cnt, int cap, PairStats &st) {
    constexpr int V = L * L * L;
    constexpr uint32_t M = (1u << L) - 1u;
    __shared__ int s_ok, s_nclus, s_top[2][32];
    const Batch &b = a.b;
    const int tid = threadIdx.x, T = blockDim.x;
    if (tid == 0) { s_ok = 1; s_nclus = 0; }
    for (int i = tid; i < (V + 1) / 2; i += T) reinterpret_cast<uint32_t *>(cnt)[i] = 0u;
    for (int r = tid; r < L * L; r += T) {
        const int i0 = L * r;
        const uint32_t q = qs[r];
        const uint32_t st_ = (q ^ (q << 1)) & M & ~1u;         // bit x >= 1: q[x] != q[x-1]
        const bool wrap = ((q ^ (q >> (L - 1))) & 1u) == 0u;   // q[0] == q[L-1]
        const int last = st_ ? 31 - __clz(st_) : L;            // start of the last run
        int root = i0;
        for (int x = 0; x < L; ++x) {
            if ((st_ >> x) & 1u) root = i0 + x;
            parent[i0 + x] = (Parent)((wrap && x >= last) ? i0 : root);
        }
    }
    __syncthreads();
    bool ok = true;
    volatile Parent *vp = parent;
    for (int tsk = tid; tsk < 2 * L * L; tsk += T) {
        const int r = tsk >> 1;
        const int y = r % L, z = r / L;
        const int r2 = (tsk & 1) ? y + L * ((z + 1) % L) : ((y + 1) % L) + L * z;
        const uint32_t q1 = qs[r], q2 = qs[r2];
        uint32_t C = ~(q1 ^ q2) & M & ((q1 ^ (q1 << 1)) | (q2 ^ (q2 << 1)) | 1u);
        while (C) {
            const int x = __ffs(C) - 1;
            C &= C - 1u;
            unite(vp, L * r + x, L * r2 + x, cap, ok, b.status, V);
        }
    }
    __syncthreads();
    // every site points straight at its root; only final roots are written
    // here (no path halving), so after the barrier parent[i] is the root
    for (int i = tid; i < V; i += T) parent[i] = (Parent)find_root_readonly(vp, i, cap, ok, b.status, V);
    if (!ok) s_ok = 0;
    __syncthreads();
    if (!s_ok) return false;
    if (a.label_only) {
        int32_t *out = a.labels_out + ((size_t)(p.s * b.NPAIR + p.P) * b.NT + p.k) * V;
        for (int i = tid; i < V; i += T) out[i] = parent[i];
        __syncthreads();
        return true;
    }
    // cluster sizes (statistics): one atomic per distinct root per warp
    for (int i0 = 0; i0 < V; i0 += T) {
        const int i = i0 + tid;
        const int root = i < V ? parent[i] : -1;
        const unsigned peers = __match_any_sync(0xffffffffu, root);
        if (i < V && (tid & 31) == __ffs(peers) - 1)
            atomicAdd(reinterpret_cast<uint32_t *>(cnt) + (root >> 1), (uint32_t)__popc(peers) << (16 * (root & 1)));
    }
    __syncthreads();
    PairStats my{0, 0, 0};
    for (int i = tid; i < V; i += T)
        if (parent[i] == i) add_size(my, cnt[i]);
    atomicAdd(&s_nclus, my.nclus);
    int t1 = my.top1, t2 = my.top2;
    for (int o = 16; o > 0; o >>= 1) {
        const int u1 = __shfl_xor_sync(0xffffffffu, t1, o), u2 = __shfl_xor_sync(0xffffffffu, t2, o);
        int n1, n2;
        if (u1 > t1) { n1 = u1; n2 = max(t1, u2); } else { n1 = t1; n2 = max(t2, u1); }
        t1 = n1; t2 = n2;
    }
    if ((tid & 31) == 0) { s_top[0][tid >> 5] = t1; s_top[1][tid >> 5] = t2; }
    __syncthreads();
    // the sizes are read: a root's entry now holds its flip bit
    const int root_t = target >= 0 ? parent[target] : -1;
    for (int i = tid; i < V; i += T)
        if (parent[i] == i)
            cnt[i] = (uint16_t)(b.cluster_mode == PTHR_CLUSTER_ACU ? cluster_sign(p, i) : i == root_t);
    int a1 = 0, a2 = 0;
    for (int w = 0; w < T / 32; ++w) {
        const int u1 = s_top[0][w], u2 = s_top[1][w];
        if (u1 > a1) { a2 = max(a1, u2); a1 = u1; } else { a2 = max(a2, u1); }
    }
    st = PairStats{s_nclus, a1, a2};
    __syncthreads();
    for (int r = tid; r < L * L; r += T) {
        uint32_t f = 0u;
        for (int x = 0; x < L; ++x) f |= (uint32_t)cnt[parent[L * r + x]] << x;
        Fs[r] = (Row)f;
    }
    __syncthreads();
    return true;
}

// The same as a call of its own, so that its registers are not the floods'.
template <int L, typename Row>
__device__ __noinline__ bool union_find_pair(const ClusterArgs &a, const PairItem &p, int target, const Row *qs,
                                             Row *Fs, uint16_t *parent, uint16_t *cnt, int cap, PairStats &st) {
    return union_find<L, Row, uint16_t>(a, p, target, qs, Fs, parent, cnt, cap, st);
}

// A lane's rows hold the unlabelled sites of both signs of q: for L <= 16 the
// q = +1 sites in the low and the q = -1 sites in the high half of one word,
// so that one cluster of each sign floods at a time; for larger L two words.
template <int L>
struct FloodWords {
    static constexpr bool PACKED = L <= 16;
    static constexpr uint32_t M = (1u << L) - 1u;
    // bits of the row's first and last site, in both halves
    static constexpr uint32_t FIRST = PACKED ? 0x00010001u : 1u;
    static constexpr uint32_t LAST = FIRST << (L - 1);
};

// a + b, by halves where the row fills a half (otherwise a carry out of the
// low row ends in the gap above it, which no mask holds)
template <int L>
__device__ __forceinline__ uint32_t add_rows(uint32_t a, uint32_t b) {
    if (L != 16) return a + b;
    uint32_t d;
    asm("add.u16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
    return d;
}

// One row of a flood: row z takes in what its neighbour rows hold and fills
// whole runs of its mask m (mr: reversed).  The carries of m + s run from a
// seed to its run's top, on the reversed row to its bottom.  Returns the new
// bits.
template <int L>
__device__ __forceinline__ uint32_t flood_row(uint32_t (&f)[L], const uint32_t (&m)[L], const uint32_t (&mr)[L],
                                              int z, int lp, int lm) {
    using Fw = FloodWords<L>;
    const uint32_t f0 = f[z];
    const uint32_t fy = __shfl_sync(0xffffffffu, f0, lp) | __shfl_sync(0xffffffffu, f0, lm);
    uint32_t s = f0 | f[(z + 1) % L] | f[(z + L - 1) % L];
    s = s | fy | ((f0 >> (L - 1)) & Fw::FIRST);
    s = (s | ((f0 << (L - 1)) & Fw::LAST)) & m[z];
    const uint32_t sr = __brev(s);
    const uint32_t up = (m[z] & ~add_rows<L>(m[z], s)) | s;
    const uint32_t dn = (mr[z] & ~add_rows<L>(mr[z], sr)) | sr;
    f[z] = up | __brev(dn);
    return f[z] ^ f0;
}

// Energies, flips and statistics of the pairs of a warp, from their flip rows.
template <int L, typename Row>
__device__ __forceinline__ void finish_pair(const ClusterArgs &a, const PairItem &p, const Row *qs, const Row *as,
                                         const Row *Fs, typename BondList<L>::Entry *list, int *count, int sub, int yl, bool ok,
                                            bool rest, const PairStats &st) {
    using Gm = Geom<L>;
    constexpr int V = Gm::V, LW = Gm::LAT_WORDS, W = Gm::W, ROWS = Gm::ROWS;
    constexpr int LN = ClusterGeom<L>::LN, SITE_BITS = BondList<L>::SITE_BITS;
    constexpr unsigned FULLW = 0xffffffffu;
    typedef typename BondList<L>::Entry Entry;
    const Batch &b = a.b;
    const int y = yl < L ? yl : L - 1, yp = (y + 1) % L;
    uint32_t *A = b.spins + ((size_t)p.s * b.NLAT + p.la) * b.lat_words;
    uint32_t *B = b.spins + ((size_t)p.s * b.NLAT + p.lb) * b.lat_words;
    if (p.live && !ok && yl == 0) set_status(b.status, STATUS_NOCONVERGE);
    __syncwarp();
    if (a.label_only) {
        if (p.live && !ok) {                             // no label rather than those of some clusters
            int32_t *out = a.labels_out + ((size_t)(p.s * b.NPAIR + p.P) * b.NT + p.k) * V;
            for (int i = yl; i < V; i += LN) out[i] = -1;
        }
        return;
    }
    const bool go = p.live && ok;                        // the same for all lanes of the pair

    // ---- energies (Eq. (1)).  Only bonds with exactly one flipped end change:
    // for them s'_i s'_j = -s_i s_j, so Delta H_a = sum of 2 J s_i s_j (old
    // spins of clone a).  Such a bond joins sites of opposite q, where the two
    // clones' terms cancel, so H_a + H_b is conserved and Delta H_b =
    // -Delta H_a.  Over all bonds between opposite q the same sum is
    // H_b - H_a, so with R the sum over those that are NOT cut, the new
    // energies are H_b - R and H_a + R.  `rest` picks the shorter sum: when
    // the two large clusters (one of each sign) flip differently, nearly
    // every bond between them is cut and R runs over the bonds at small
    // clusters only, and when they flip alike the cut bonds do (a thermalised
    // pair has 30% of its bonds between opposite q and cuts none or nearly
    // all of them; either sum then has a few dozen terms).
    // On the coupling grid (J a multiple of 2^-18) the sum is exact in
    // integers and both energies are updated exactly in FP64; the energies
    // before are those of the resident spins (every entry point that changes
    // spins recomputes them).  Off the grid both energies are recomputed.
    const float *J = b.J + (size_t)p.s * 3 * V;
    long long dE = 0;
    int nflip = 0;
    uint32_t bad = 0;                                    // a coupling off the grid
    // The bonds go through a list in shared memory (site, direction and the
    // sign of s_i s_j in one entry): the lanes' rows hold very different
    // numbers of them, and from the list every lane sums an equal share with
    // its couplings' loads (600 to 800 cycles each) in flight together.
    if (yl == 0) *count = 0;
    __syncwarp();
    int listed = 0;                                      // entries, the same for all lanes of the pair
    for (int z = 0; z < L; ++z) {
        const int r = y + L * z, ry = yp + L * z, rz = y + L * (z + 1 == L ? 0 : z + 1);
        uint32_t w[3] = {0u, 0u, 0u}, n[3];
        if (go && yl < L) {
            const uint32_t f = Fs[r], av = as[r];
            nflip += __popc(f);
            w[0] = f ^ rot_next<L>(f);
            w[1] = f ^ Fs[ry];
            w[2] = f ^ Fs[rz];
            if (rest) {
                const uint32_t q = qs[r];
                w[0] ^= q ^ rot_next<L>(q);
                w[1] ^= q ^ qs[ry];
                w[2] ^= q ^ qs[rz];
            }
            n[0] = av ^ rot_next<L>(av);
            n[1] = av ^ as[ry];
            n[2] = av ^ as[rz];
            const int mine = __popc(w[0]) + __popc(w[1]) + __popc(w[2]);
            if (mine) {
                int at = atomicAdd(count, mine);
#pragma unroll
                for (int d = 0; d < 3; ++d) {
                    while (w[d]) {
                        const int sh = __clz(w[d]), x = 31 - sh;
                        w[d] ^= 1u << x;
                        list[at++] = (Entry)((L * r + x) | (d << SITE_BITS) | (((n[d] >> x) & 1u) << (SITE_BITS + 2)));
                    }
                }
            }
        }
        __syncwarp();
        listed = *count;
        // a plane holds at most 3 L^2 bonds: sum the list up when the next plane
        // may not fit (or at the end)
        if (__any_sync(FULLW, listed > BondList<L>::N - 3 * L * L) || z == L - 1) {
            int sum = 0;
#pragma unroll 4
            for (int i = yl; i < listed; i += LN) {
                const uint32_t e = list[i];
                const uint32_t site = e & ((1u << SITE_BITS) - 1u), d = (e >> SITE_BITS) & 3u;
                // (at most N / LN terms below 2^23)
                sum += bond_int(__ldg(J + d * V + site), (e >> (SITE_BITS + 2)) != 0u, bad);
            }
            dE += sum;
            __syncwarp();
            if (yl == 0) *count = 0;
            __syncwarp();
        }
    }
    const unsigned off = __ballot_sync(FULLW, bad != 0u);
    const bool exact_E = ((off >> (sub * LN)) & (unsigned)((1ull << LN) - 1ull)) == 0u;
    double Ea = 0.0, Eb = 0.0;
    if (go && !exact_E && yl < L) {
        const double2 e = column_energies<L>(J, qs, as, Fs, y);
        Ea = e.x;
        Eb = e.y;
    }
    for (int o = LN / 2; o > 0; o >>= 1) {
        dE += __shfl_xor_sync(FULLW, dE, o);
        nflip += __shfl_xor_sync(FULLW, nflip, o);
    }
    if (off) {                                           // warp-uniform
        for (int o = LN / 2; o > 0; o >>= 1) {
            Ea += __shfl_xor_sync(FULLW, Ea, o);
            Eb += __shfl_xor_sync(FULLW, Eb, o);
        }
    }
    if (!go) return;
    // ---- flip both clones
    if (b.bits) {
        for (int i = yl; i < LW / 8; i += LN) {
            const uint32_t m = flip_bits<L>(Fs, i);
            if (m) { A[i] ^= m; B[i] ^= m; }
        }
    } else if (yl < L) {
        // four rows at a time, so that their loads are in flight together
        constexpr int ZB = L % 4 == 0 ? 4 : 2;
        for (int z0 = 0; z0 < L; z0 += ZB) {
            uint32_t f[ZB], wa[ZB][2][W], wb[ZB][2][W];
#pragma unroll
            for (int i = 0; i < ZB; ++i) {
                const int r = y + L * (z0 + i);
                f[i] = Fs[r];
                if (f[i]) {
#pragma unroll
                    for (int c = 0; c < 2; ++c) {
                        load_words<W>(A + (c * ROWS + r) * W, wa[i][c]);
                        load_words<W>(B + (c * ROWS + r) * W, wb[i][c]);
                    }
                }
            }
#pragma unroll
            for (int i = 0; i < ZB; ++i) {
                const int r = y + L * (z0 + i);
                if (!f[i]) continue;
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    const uint32_t v = f[i] >> ((c + y + z0 + i) & 1);
#pragma unroll
                    for (int j = 0; j < W; ++j) {
                        const uint32_t mj = word_flips(v, j);
                        wa[i][c][j] ^= mj;
                        wb[i][c][j] ^= mj;
                    }
                    store_words<W>(A + (c * ROWS + r) * W, wa[i][c]);
                    store_words<W>(B + (c * ROWS + r) * W, wb[i][c]);
                }
            }
        }
    }
    if (yl == 0) {
        double *E = b.E + (size_t)p.s * b.NLAT;
        if (exact_E) {
            const double dH = (double)(2 * dE) * (1.0 / 262144.0);
            const double Ha = E[p.la], Hb = E[p.lb];
            E[p.la] = rest ? Hb - dH : Ha + dH;
            E[p.lb] = rest ? Ha + dH : Hb - dH;
        } else {
            E[p.la] = -Ea;
            E[p.lb] = -Eb;
        }
        long long *cs = b.cstat + (((size_t)p.s * b.NPAIR + p.P) * b.NT + p.k) * 4;
        cs[0] = st.nclus;
        cs[1] = st.top1;
        cs[2] = st.top2;
        cs[3] = nflip;
    }
}


// ------------------------------------------------------------ the block
template <int L>
__device__ __forceinline__ void cluster_block(const ClusterArgs &a, int bid, unsigned char *smem) {
    using Gm = Geom<L>;
    constexpr int V = Gm::V, ROWS = Gm::ROWS, W = Gm::W;
    constexpr int LN = ClusterGeom<L>::LN, PPW = ClusterGeom<L>::PPW;
    constexpr uint32_t M = (1u << L) - 1u;
    constexpr unsigned FULLW = 0xffffffffu;
    typedef typename RowType<(L > 16)>::T Row;
    const Batch &b = a.b;
    const int tid = threadIdx.x, T = blockDim.x;
    const int lane = tid & 31, sub = lane / LN, yl = lane % LN;
    const int slots = (T / 32) * PPW, slot = (tid >> 5) * PPW + sub;
    Row *rows = reinterpret_cast<Row *>(smem);
    Row *qs = rows + (size_t)slot * 3 * ROWS, *as = qs + ROWS, *Fs = as + ROWS;
    Row *list = rows + (size_t)slots * 3 * ROWS + (size_t)slot * BondList<L>::N;
    uint16_t *parent = reinterpret_cast<uint16_t *>(
        smem + (((size_t)slots * (3 * ROWS + BondList<L>::N) * sizeof(Row) + 15) & ~(size_t)15));
    uint16_t *cnt = parent + (((size_t)V * 2 + 15) & ~(size_t)15) / 2;
    __shared__ int s_nslow;
    int *s_list = reinterpret_cast<int *>(cnt + (((size_t)V * 2 + 15) & ~(size_t)15) / 2);   // [slots] slow pairs
    int *s_target = s_list + slots, *s_count = s_target + slots;                          // [slots] each
    int *s_res = s_count + slots;                                                         // [slots][4]
    if (tid == 0) s_nslow = 0;
    __syncthreads();

    const PairItem p = pair_item(a, bid * slots + slot);
    const bool acu = b.cluster_mode == PTHR_CLUSTER_ACU;
    const int cap = a.iter_cap > 0 ? a.iter_cap : 4 * V + 64;
    const bool mine = p.live && yl < L;              // this lane holds rows
    const int y = yl < L ? yl : L - 1;
    const int yp = (y + 1) % L, ym = (y + L - 1) % L;
    const int lp = sub * LN + yp, lm = sub * LN + ym;   // lanes of the y neighbours
    uint32_t *A = b.spins + ((size_t)p.s * b.NLAT + p.la) * b.lat_words;
    uint32_t *B = b.spins + ((size_t)p.s * b.NLAT + p.lb) * b.lat_words;

    // ---- rows of q and of clone a's signs
    uint32_t u[L];                                   // unlabelled sites
    if (b.bits) {
#pragma unroll
        for (int z = 0; z < L; ++z) {
            const int r = y + L * z, p0 = (y + z) & 1;
            const uint32_t av = mine ? row_of_bits<L>(A, r, p0) : 0u, bv = mine ? row_of_bits<L>(B, r, p0) : 0u;
            u[z] = av ^ bv;
            if (yl < L) as[r] = (Row)av;
        }
    } else {
        constexpr int ZB = rows_in_flight(L);
#pragma unroll
        for (int z0 = 0; z0 < L; z0 += ZB) {
            uint32_t wa[ZB][2][W], wb[ZB][2][W];
#pragma unroll
            for (int i = 0; i < ZB; ++i)
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    load_words<W>(A + (c * ROWS + y + L * (z0 + i)) * W, wa[i][c]);
                    load_words<W>(B + (c * ROWS + y + L * (z0 + i)) * W, wb[i][c]);
                }
#pragma unroll
            for (int i = 0; i < ZB; ++i) {
                const int r = y + L * (z0 + i), p0 = (y + z0 + i) & 1;
                const uint32_t av = row_of_words<L>(wa[i], p0), bv = row_of_words<L>(wb[i], p0);
                u[z0 + i] = mine ? av ^ bv : 0u;
                if (yl < L) as[r] = (Row)av;
            }
        }
    }
#pragma unroll
    for (int z = 0; z < L; ++z) {
        const int r = y + L * z;
        if (yl < L) {
            qs[r] = (Row)u[z];
            Fs[r] = 0;
        }
    }
    // ---- single-cluster move: the floor(u*n)-th q = -1 site in site order
    int target = -1;
    if (!acu && !a.label_only) {
        int n = 0;
#pragma unroll
        for (int z = 0; z < L; ++z) n += __popc(u[z]);
        for (int o = LN / 2; o > 0; o >>= 1) n += __shfl_xor_sync(FULLW, n, o);
        int want = -1;
        if (n > 0) {
            const uint32_t w = philox_word0(p.seed, 0u, p.pair_id, p.emcs, TAG_SINGLE);
            want = (int)(((unsigned long long)(w >> 8) * (unsigned long long)n) >> 24);
        }
        int seen = 0;                                // sites of the planes below z
#pragma unroll
        for (int z = 0; z < L; ++z) {
            const int c = __popc(u[z]);
            int incl = c;
            for (int o = 1; o < LN; o <<= 1) {
                const int t = __shfl_up_sync(FULLW, incl, o, LN);
                if (yl >= o) incl += t;
            }
            const int first = seen + incl - c;
            if (want >= first && want < first + c) {
                uint32_t v = u[z];
                for (int m = want - first; m > 0; --m) v &= v - 1u;
                target = L * (y + L * z) + __ffs(v) - 1;
            }
            seen += __shfl_sync(FULLW, incl, LN - 1, LN);
        }
        for (int o = LN / 2; o > 0; o >>= 1) target = max(target, __shfl_xor_sync(FULLW, target, o));
    }
    __syncwarp();
    // ---- sites with no equal neighbour
    int32_t *labels = nullptr;
    if (a.label_only && p.live) labels = a.labels_out + ((size_t)(p.s * b.NPAIR + p.P) * b.NT + p.k) * V;
    PairStats st{0, 0, 0};
    {
        int niso = 0;
#pragma unroll
        for (int z = 0; z < L; ++z) {
            const uint32_t q = u[z];
            const uint32_t ex = ~(q ^ rot_next<L>(q)) & M;             // x and x + 1 equal
            const uint32_t ey = ~(q ^ qs[yp + L * z]) | ~(q ^ qs[ym + L * z]);
            const uint32_t ez = ~(q ^ u[(z + 1) % L]) | ~(q ^ u[(z + L - 1) % L]);
            const uint32_t eq = ex | (ex << 1) | (ex >> (L - 1)) | ey | ez;
            const uint32_t iso = M & ~eq;
            if (mine) Fs[y + L * z] = (Row)iso;          // for now
            niso += mine ? __popc(iso) : 0;
        }
#pragma unroll
        for (int z = 0; z < L; ++z) u[z] = mine ? M & ~(uint32_t)Fs[y + L * z] : 0u;
        // one site per lane and turn, so that the lanes draw their signs
        // together (turns = the most such sites of one lane)
        int z = -1;
        uint32_t v = 0, f = 0;
        while (mine) {
            while (v == 0u && z < L) {
                if (z >= 0) Fs[y + L * z] = (Row)f;
                f = 0u;
                if (++z < L) v = Fs[y + L * z];
            }
            if (z >= L) break;
            const int x = 31 - __clz(v), i = L * (y + L * z) + x;
            v ^= 1u << x;
            if (a.label_only) labels[i] = i;
            else if (acu ? cluster_sign(p, i) : i == target) f |= 1u << x;
        }
        __syncwarp();
        for (int o = LN / 2; o > 0; o >>= 1) niso += __shfl_xor_sync(FULLW, niso, o);
        st = PairStats{niso, niso > 0 ? 1 : 0, niso > 1 ? 1 : 0};
    }
    // ---- the other clusters, by their smallest site: in each turn the first
    // unlabelled q = +1 site's cluster and the first q = -1 site's
    using Fw = FloodWords<L>;
    bool ok = true, slow = false;
    int big0 = 0, big1 = 0;                              // largest cluster of each sign so far
    bool flip0 = false, flip1 = false;                   // and whether it flips
    if (Fw::PACKED) {
#pragma unroll
        for (int z = 0; z < L; ++z) {
            const uint32_t q = qs[y + L * z];
            u[z] = (u[z] & ~q) | ((u[z] & q) << 16);
        }
    }
    uint32_t ur[L];
#pragma unroll
    for (int z = 0; z < L; ++z) ur[z] = __brev(u[z]);
    for (int nf = 0; nf <= MAX_FLOODS; ++nf) {
        // first sites; 0xFFFF: none (V < 2^16)
        uint32_t key = 0xFFFFFFFFu;
        {
            int z0 = -1, z1 = -1;
            uint32_t w0 = 0, w1 = 0;
#pragma unroll
            for (int z = L - 1; z >= 0; --z) {
                if (Fw::PACKED) {
                    if (u[z] & 0xFFFFu) { z0 = z; w0 = u[z]; }
                    if (u[z] > 0xFFFFu) { z1 = z; w1 = u[z]; }
                } else if (u[z]) {
                    z0 = z;
                    w0 = u[z];
                }
            }
            if (z0 >= 0) key = (uint32_t)(L * (y + L * z0) + __ffs(w0) - 1);
            if (Fw::PACKED) {
                key &= 0xFFFFu;
                key |= z1 >= 0 ? (uint32_t)(L * (y + L * z1) + __ffs(w1 >> 16) - 1) << 16 : 0xFFFF0000u;
            }
        }
        for (int o = LN / 2; o > 0; o >>= 1) {
            const uint32_t other = __shfl_xor_sync(FULLW, key, o);
            key = Fw::PACKED ? __vminu2(key, other) : min(key, other);
        }
        const bool act = key != 0xFFFFFFFFu;
        if (!__any_sync(FULLW, act)) break;
        if (nf == MAX_FLOODS) { slow = act; break; }
        const int lab[2] = {(int)(Fw::PACKED ? key & 0xFFFFu : key), (int)(Fw::PACKED ? key >> 16 : 0xFFFFu)};
        uint32_t m[L], f[L];
        int sign1 = 0;                                   // unpacked: the cluster's sign is -1
        if (Fw::PACKED) {
            // (a label 0xFFFF lies in no plane: V <= 16^3)
            const int r0 = lab[0] / L, r1 = lab[1] / L, z0 = r0 / L, z1 = r1 / L;
            const uint32_t b0 = yl == r0 - L * z0 ? 1u << (lab[0] - L * r0) : 0u;
            const uint32_t b1 = yl == r1 - L * z1 ? 0x10000u << (lab[1] - L * r1) : 0u;
#pragma unroll
            for (int z = 0; z < L; ++z) {
                m[z] = u[z];
                f[z] = (z == z0 ? b0 : 0u) | (z == z1 ? b1 : 0u);
            }
        } else {
            // one cluster at a time, of the sign of its first site
            const int rs = act ? lab[0] / L : 0, xs = act ? lab[0] - rs * L : 0;
            sign1 = (int)((qs[rs] >> xs) & 1u);
            const uint32_t inv = sign1 ? 0u : FULLW;
#pragma unroll
            for (int z = 0; z < L; ++z) {
                const int r = y + L * z;
                m[z] = act ? u[z] & (qs[r] ^ inv) : 0u;
                ur[z] = __brev(m[z]);
                f[z] = act && yl < L && r == rs ? 1u << xs : 0u;
            }
        }
        // passes over the rows, upwards and downwards in turn, until one
        // changes nothing; four chains of L/4 rows advance side by side, since
        // one row's shuffles, reversals and carries are a serial chain of about
        // 90 cycles (on thermalised pairs four chains need 5% more row visits
        // than one, and a quarter of the serial steps)
        constexpr int CH = (L + 3) / 4;
        unsigned more = FULLW;                           // lanes with changes in the last pass
        for (int it = 0; more && it < 2 * cap; ++it) {
            uint32_t ch = 0;
            if ((it & 1) == 0) {
#pragma unroll
                for (int v = 0; v < CH; ++v)
#pragma unroll
                    for (int z = v; z < L; z += CH) ch |= flood_row<L>(f, m, ur, z, lp, lm);
            } else {
#pragma unroll
                for (int v = CH - 1; v >= 0; --v)
#pragma unroll
                    for (int z = v; z < L; z += CH) ch |= flood_row<L>(f, m, ur, z, lp, lm);
            }
            more = __ballot_sync(FULLW, ch != 0u);
        }
        // (of this pair: its neighbours in the warp may have converged)
        if ((more >> (sub * LN)) & (unsigned)((1ull << LN) - 1ull)) ok = false;
        int size = 0;                                    // both clusters' sites, 16 bits each
#pragma unroll
        for (int z = 0; z < L; ++z)
            size += Fw::PACKED ? __popc(f[z] & 0xFFFFu) + (__popc(f[z] >> 16) << 16) : __popc(f[z]);
        for (int o = LN / 2; o > 0; o >>= 1) size += __shfl_xor_sync(FULLW, size, o);
        bool flip[2] = {false, false};                   // of the two clusters
        bool holds[2] = {false, false};                  // the single move's target site
        if (!acu) {
#pragma unroll
            for (int z = 0; z < L; ++z) {
                const int x = target - L * (y + L * z);
                if (yl < L && x >= 0 && x < L) {
                    holds[0] = (f[z] >> x) & 1u;
                    holds[1] = Fw::PACKED && ((f[z] >> (16 + x)) & 1u);
                }
            }
        }
        // even lanes draw the sign of one cluster, odd lanes of the other
        const unsigned drawn = __ballot_sync(FULLW, acu && cluster_sign(p, lab[Fw::PACKED ? yl & 1 : 0]));
#pragma unroll
        for (int h = 0; h < (Fw::PACKED ? 2 : 1); ++h) {
            const int sz = Fw::PACKED ? (h ? (int)((uint32_t)size >> 16) : size & 0xFFFF) : size;
            if (sz > 0) add_size(st, sz);
            if (acu) {
                flip[h] = sz > 0 && ((drawn >> (sub * LN + h)) & 1u);
            } else {
                const unsigned any = __ballot_sync(FULLW, holds[h]);
                flip[h] = ((any >> (sub * LN)) & (unsigned)((1ull << LN) - 1ull)) != 0u;
            }
            const int sign = Fw::PACKED ? h : sign1;
            if (sz > (sign ? big1 : big0)) {
                if (sign) { big1 = sz; flip1 = flip[h]; } else { big0 = sz; flip0 = flip[h]; }
            }
        }
        if (a.label_only) {
            if (mine) {
#pragma unroll
                for (int z = 0; z < L; ++z) as[y + L * z] = (Row)(f[z] & Fw::M);
                if (Fw::PACKED) {
#pragma unroll
                    for (int z = 0; z < L; ++z) Fs[y + L * z] = (Row)(f[z] >> 16);
                }
                for (int z = 0; z < L; ++z) {
#pragma unroll
                    for (int h = 0; h < (Fw::PACKED ? 2 : 1); ++h) {
                        uint32_t v = h ? Fs[y + L * z] : as[y + L * z];
                        while (v) {
                            const int x = 31 - __clz(v);
                            v ^= 1u << x;
                            labels[L * (y + L * z) + x] = lab[h];
                        }
                    }
                }
            }
        } else if (flip[0] || flip[1]) {
            const uint32_t k0 = flip[0] ? Fw::M : 0u, k1 = flip[1] ? Fw::M : 0u;
#pragma unroll
            for (int z = 0; z < L; ++z) {
                const uint32_t v = Fw::PACKED ? (f[z] & k0) | ((f[z] >> 16) & k1) : f[z];
                if (v) Fs[y + L * z] |= (Row)v;
            }
        }
#pragma unroll
        for (int z = 0; z < L; ++z) {
            u[z] &= ~f[z];
            if (Fw::PACKED) ur[z] = __brev(u[z]);
        }
    }
    // ---- flips, energies and statistics; then, if the block has any, the pairs
    // of many clusters (the whole block, one pair after another) and theirs
#pragma unroll 1
    for (int turn = 0; turn < 2; ++turn) {
        if (turn == 1) {
            if (slow && yl == 0) {
                const int i = atomicAdd(&s_nslow, 1);
                s_list[i] = slot;
                s_target[i] = target;
            }
            __syncthreads();
            const int nslow = s_nslow;
            if (nslow == 0) return;
            for (int i = 0; i < nslow; ++i) {
                const int sl = s_list[i];
                const PairItem ps = pair_item(a, bid * slots + sl);
                PairStats r{0, 0, 0};
                const bool good = union_find_pair<L, Row>(a, ps, s_target[i], rows + (size_t)sl * 3 * ROWS,
                                                          rows + (size_t)sl * 3 * ROWS + 2 * ROWS, parent, cnt,
                                                          cap, r);
                if (tid == 0) {
                    s_res[4 * sl] = good;
                    s_res[4 * sl + 1] = r.nclus;
                    s_res[4 * sl + 2] = r.top1;
                    s_res[4 * sl + 3] = r.top2;
                }
                __syncthreads();
            }
            if (slow) {
                ok = s_res[4 * slot] != 0;
                st = PairStats{s_res[4 * slot + 1], s_res[4 * slot + 2], s_res[4 * slot + 3]};
            }
        }
        if (__any_sync(FULLW, slow) == (turn == 1))
            finish_pair<L, Row>(a, p, qs, as, Fs, list, s_count + slot, sub, yl, ok, !slow && flip0 != flip1, st);
    }
}

// ------------------------------------------------------------ one block per pair
// Launches of few pairs: a warp's flood is one serial chain, which such a
// launch lasts as long as, while most of the GPU idles.  Here a whole block
// labels its pair by the union-find over sites and shares out rows, bonds and
// words among its threads; the pair's rows, int parents and sizes are all its
// shared memory.  One sample, 28 pairs, thermalised (warps): L = 8 17 us (21
// us), L = 16 26 us (46 us), L = 20 37 us (90 us), L = 24 58 us (142 us).
// Registers for three blocks of 512 threads per SM to L = 18 (above it the
// memory takes two): 64 registers cost 40% at L = 14, 336 pairs, 32 registers 8%.
template <int L>
constexpr size_t pair_smem() {
    typedef typename RowType<(L > 16)>::T Row;
    return (size_t)L * L * L * 4 + (((size_t)L * L * L * 2 + 15) & ~(size_t)15) + 3 * L * L * sizeof(Row) + 16;
}

template <int L>
__device__ __forceinline__ void pair_block(const ClusterArgs &a, int bid, unsigned char *smem) {
    using Gm = Geom<L>;
    constexpr int V = Gm::V, ROWS = Gm::ROWS, W = Gm::W, LW = Gm::LAT_WORDS;
    constexpr int CAP = 4 * V + 64;
    typedef typename RowType<(L > 16)>::T Row;
    int *parent = reinterpret_cast<int *>(smem);
    uint16_t *cnt = reinterpret_cast<uint16_t *>(parent + V);
    Row *qs = reinterpret_cast<Row *>(smem + (size_t)V * 4 + (((size_t)V * 2 + 15) & ~(size_t)15));
    Row *as = qs + ROWS, *Fs = as + ROWS;
    __shared__ int s_n, s_target, s_part[16][2];
    __shared__ double s_E[16][2];
    __shared__ long long s_dE[16];
    const Batch &b = a.b;
    const int tid = threadIdx.x, T = blockDim.x, lane = tid & 31, wid = tid >> 5, nw = T >> 5;
    const PairItem p = pair_item(a, bid);
    if (!p.live) return;                                 // the same for the block
    uint32_t *A = b.spins + ((size_t)p.s * b.NLAT + p.la) * b.lat_words;
    uint32_t *B = b.spins + ((size_t)p.s * b.NLAT + p.lb) * b.lat_words;
    if (tid == 0) { s_n = 0; s_target = -1; }
    for (int r = tid; r < ROWS; r += T) {
        const int p0 = (r % L + r / L) & 1;
        uint32_t av, bv;
        if (b.bits) {
            av = row_of_bits<L>(A, r, p0);
            bv = row_of_bits<L>(B, r, p0);
        } else {
            uint32_t wa[2][W], wb[2][W];
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                load_words<W>(A + (c * ROWS + r) * W, wa[c]);
                load_words<W>(B + (c * ROWS + r) * W, wb[c]);
            }
            av = row_of_words<L>(wa, p0);
            bv = row_of_words<L>(wb, p0);
        }
        as[r] = (Row)av;
        qs[r] = (Row)(av ^ bv);
    }
    __syncthreads();
    // ---- single-cluster move: the floor(u*n)-th q = -1 site in site order
    if (b.cluster_mode != PTHR_CLUSTER_ACU && !a.label_only) {
        const int chunk = (ROWS + T - 1) / T;
        const int lo = min(ROWS, tid * chunk), hi = min(ROWS, lo + chunk);
        int my = 0;
        for (int r = lo; r < hi; ++r) my += __popc((uint32_t)qs[r]);
        int incl = my;
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += t;
        }
        if (lane == 31) s_part[wid][0] = incl;
        __syncthreads();
        int before = incl - my, n = 0;
        for (int w = 0; w < nw; ++w) {
            if (w < wid) before += s_part[w][0];
            n += s_part[w][0];
        }
        if (n > 0) {
            const uint32_t w = philox_word0(p.seed, 0u, p.pair_id, p.emcs, TAG_SINGLE);
            const int want = (int)(((unsigned long long)(w >> 8) * (unsigned long long)n) >> 24);
            if (want >= before && want < before + my) {
                for (int r = lo; r < hi; ++r) {
                    uint32_t v = qs[r];
                    const int c = __popc(v);
                    if (want < before + c) {
                        for (int m = want - before; m > 0; --m) v &= v - 1u;
                        s_target = L * r + __ffs(v) - 1;
                        break;
                    }
                    before += c;
                }
            }
        }
        __syncthreads();
    }
    PairStats st{0, 0, 0};
    if (!union_find<L, Row, int>(a, p, s_target, qs, Fs, parent, cnt, CAP, st)) {
        if (tid == 0) set_status(b.status, STATUS_NOCONVERGE);
        return;
    }
    if (a.label_only) return;
    // ---- energies from the cut bonds (see finish_pair)
    const float *J = b.J + (size_t)p.s * 3 * V;
    int sum = 0, nflip = 0;                              // at most 2 rows of 3 L terms below 2^23
    uint32_t bad = 0;
    for (int r = tid; r < ROWS; r += T) {
        const int y = r % L, z = r / L;
        const int ry = (y + 1 == L ? 0 : y + 1) + L * z, rz = y + L * (z + 1 == L ? 0 : z + 1);
        const uint32_t f = Fs[r], av = as[r];
        const uint32_t cut[3] = {f ^ rot_next<L>(f), f ^ Fs[ry], f ^ Fs[rz]};
        const uint32_t neg[3] = {av ^ rot_next<L>(av), av ^ as[ry], av ^ as[rz]};
        nflip += __popc(f);
#pragma unroll
        for (int d = 0; d < 3; ++d)
            for (uint32_t cb = cut[d]; cb; cb &= cb - 1u) {
                const int x = __ffs(cb) - 1;
                sum += bond_int(__ldg(J + d * V + L * r + x), (neg[d] >> x) & 1u, bad);
            }
    }
    const bool exact_E = __syncthreads_or(bad != 0u) == 0;
    double ea = 0.0, eb = 0.0;
    if (!exact_E)
#pragma unroll 1
        for (int r = tid; r < ROWS; r += T) row_energies<L, 1>(J, qs, as, Fs, r, ea, eb);
    // (a warp's sums of both, below 2^31 where cut into 16-bit halves)
    int hi = __reduce_add_sync(0xffffffffu, sum >> 12);
    const unsigned lo = __reduce_add_sync(0xffffffffu, (unsigned)(sum & 0xFFF));
    nflip = __reduce_add_sync(0xffffffffu, nflip);
    if (!exact_E)
        for (int o = 16; o > 0; o >>= 1) {
            ea += __shfl_xor_sync(0xffffffffu, ea, o);
            eb += __shfl_xor_sync(0xffffffffu, eb, o);
        }
    if (lane == 0) {
        s_dE[wid] = (long long)hi * 4096 + (long long)lo;
        s_part[wid][0] = nflip;
        s_E[wid][0] = ea;
        s_E[wid][1] = eb;
    }
    // ---- flip both clones
    if (b.bits) {
        for (int i = tid; i < LW / 8; i += T) {
            const uint32_t m = flip_bits<L>(Fs, i);
            if (m) { A[i] ^= m; B[i] ^= m; }
        }
    } else {
        for (int r = tid; r < ROWS; r += T) {
            const uint32_t f = Fs[r];
            if (!f) continue;
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                uint32_t wa[W], wb[W];
                load_words<W>(A + (c * ROWS + r) * W, wa);
                load_words<W>(B + (c * ROWS + r) * W, wb);
                const uint32_t v = f >> ((c + r % L + r / L) & 1);
#pragma unroll
                for (int j = 0; j < W; ++j) {
                    wa[j] ^= word_flips(v, j);
                    wb[j] ^= word_flips(v, j);
                }
                store_words<W>(A + (c * ROWS + r) * W, wa);
                store_words<W>(B + (c * ROWS + r) * W, wb);
            }
        }
    }
    __syncthreads();
    if (tid == 0) {
        long long dE = 0;
        int flips = 0;
        double Ea = 0.0, Eb = 0.0;
        for (int w = 0; w < nw; ++w) {
            dE += s_dE[w];
            flips += s_part[w][0];
            Ea += s_E[w][0];
            Eb += s_E[w][1];
        }
        double *E = b.E + (size_t)p.s * b.NLAT;
        if (exact_E) {
            const double dH = (double)(2 * dE) * (1.0 / 262144.0);
            E[p.la] += dH;
            E[p.lb] -= dH;
        } else {
            E[p.la] = -Ea;
            E[p.lb] = -Eb;
        }
        long long *cs = b.cstat + (((size_t)p.s * b.NPAIR + p.P) * b.NT + p.k) * 4;
        cs[0] = st.nclus;
        cs[1] = st.top1;
        cs[2] = st.top2;
        cs[3] = flips;
    }
}

template <int L>
__global__ void __launch_bounds__(512, L <= 18 ? 3 : 2) pair_kernel(ClusterArgs a) {
    extern __shared__ __align__(16) unsigned char smem[];
    pair_block<L>(a, blockIdx.x, smem);
}

template <int L>
cudaError_t launch_pairs_L(const ClusterArgs &a, int threads, cudaStream_t st) {
    static bool configured = false;
    if (!configured) {
        cudaError_t e = allow_max_dynamic_smem(pair_kernel<L>);
        if (e != cudaSuccess) return e;
        configured = true;
    }
    const int blocks = a.sample_count * a.b.NPAIR * a.b.n_acu;
    if (blocks <= 0) return cudaSuccess;
    pair_kernel<L><<<blocks, threads, pair_smem<L>(), st>>>(a);
    return cudaGetLastError();
}

template <int L>
__global__ void __launch_bounds__(CLUSTER_MAX_THREADS, L <= 8 || L > 16 ? 4 : 5) cluster_kernel(ClusterArgs a) {
    extern __shared__ __align__(16) unsigned char smem[];
    cluster_block<L>(a, blockIdx.x, smem);
}

template <int L>
cudaError_t launch_cluster_L(const ClusterArgs &a, int threads, cudaStream_t st) {
    static bool configured = false;
    if (!configured) {
        cudaError_t e = allow_max_dynamic_smem(cluster_kernel<L>);
        if (e != cudaSuccess) return e;
        configured = true;
    }
    const int blocks = cluster_blocks_for(L, a.sample_count * a.b.NPAIR * a.b.n_acu, threads);
    if (blocks <= 0) return cudaSuccess;
    cluster_kernel<L><<<blocks, threads, cluster_smem<L>(threads), st>>>(a);
    return cudaGetLastError();
}

// The cluster step of a mixed-L group (see kernels.cuh): the blocks of every
// batch's cluster launch, dispatching on its lattice size; one block size and
// one form for the group.
template <bool PAIRS>
__global__ void __launch_bounds__(PAIRS ? 512 : CLUSTER_MAX_THREADS, PAIRS ? 2 : 5)
group_cluster_kernel(GroupClusterArgs g) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ ClusterArgs ca;
    const int i = group_member(g.off, g.n, (int)blockIdx.x);
    if (threadIdx.x == 0) {
        switch (i) {
#define PICK(J) case J: ca = g.a[J]; break;
            PICK(0) PICK(1) PICK(2) PICK(3) PICK(4) PICK(5) PICK(6) PICK(7)
#undef PICK
        }
    }
    __syncthreads();
    const int bid = (int)blockIdx.x - g.off[i];
    switch (ca.b.L) {
#define X(LL) case LL: PAIRS ? pair_block<LL>(ca, bid, smem) : cluster_block<LL>(ca, bid, smem); break;
        X(4) X(6) X(8) X(10) X(12) X(14) X(16)
#undef X
    }
}

}  // namespace

int cluster_blocks_for(int L, int pairs, int threads) {
    const int lanes = L <= 4 ? 4 : (L <= 8 ? 8 : (L <= 16 ? 16 : 32));
    const int slots = (threads / 32) * (32 / lanes);
    return (pairs + slots - 1) / slots;
}

template <bool PAIRS>
static cudaError_t launch_group_cluster_form(const GroupClusterArgs &g, int blocks, int threads, size_t smem,
                                             cudaStream_t st) {
    static bool configured = false;
    if (!configured) {
        cudaError_t e = allow_max_dynamic_smem(group_cluster_kernel<PAIRS>);
        if (e != cudaSuccess) return e;
        configured = true;
    }
    group_cluster_kernel<PAIRS><<<blocks, threads, smem, st>>>(g);
    return cudaGetLastError();
}

cudaError_t launch_group_cluster(const GroupClusterArgs &g, int pairs, int blocks, int threads, size_t smem,
                                 cudaStream_t st) {
    if (blocks <= 0) return cudaSuccess;
    return pairs ? launch_group_cluster_form<true>(g, blocks, threads, smem, st)
                 : launch_group_cluster_form<false>(g, blocks, threads, smem, st);
}

size_t cluster_pair_smem_bytes_for(int L) {
#define X(LL) if (L == LL) return pair_smem<LL>();
    PTHR_FOR_EACH_L(X)
#undef X
    return 0;
}

cudaError_t launch_cluster_pairs(const ClusterArgs &a, int threads, cudaStream_t st) {
#define X(LL) if (a.b.L == LL) return launch_pairs_L<LL>(a, threads, st);
    PTHR_FOR_EACH_L(X)
#undef X
    return cudaErrorInvalidValue;
}

size_t cluster_smem_bytes_for(int L, int threads) {
#define X(LL) if (L == LL) return cluster_smem<LL>(threads);
    PTHR_FOR_EACH_L(X)
#undef X
    return 0;
}

cudaError_t launch_cluster(const ClusterArgs &a, int threads, cudaStream_t st) {
#define X(LL) if (a.b.L == LL) return launch_cluster_L<LL>(a, threads, st);
    PTHR_FOR_EACH_L(X)
#undef X
    return cudaErrorInvalidValue;
}

}  // namespace pthr
