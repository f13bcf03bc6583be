// resident.cu -- many time steps in one cooperative launch, the populations
// held in shared memory, for lattices that fit the chip's shared memory.
//
// A step of such a lattice as a launch of its own is bound by latency: the
// launch, the drain of its stores and three dependent trips to L2 cost 6 to
// 10 us whatever the size. Here the lattice is cut into rectangular patches,
// one CTA (one SM) each; a CTA keeps its patch and a halo of three nodes in
// shared memory for all the steps, and after each step the CTAs exchange what
// their neighbours' pulls reach.
//
// Measured (us per step in runs of 1000, one launch per step -> resident; the
// launches in brackets overlap their heads and tails, launch_after):
// FP32 100 x 50 6.16 (5.1) -> 1.85, 256 x 128 6.17 (5.8) -> 2.29, 400 x 200 with
// a 30 degree slope 8.21 (6.6) -> 2.62, 512 x 512 with a disc 10.3 (9.7) -> 5.8
// (BF16 10.7 (9.9) -> 4.8); FP64 100 x 50 18.4 -> 6.1, 400 x 200 41.0 -> 18.2. What a step of 256 x 128
// takes (cycles, a patch at the wall): bounce-back copies, pulls and phi
// 1,100, ghost values 800, collision 1,000, publishing 400, the wait 1,650. With
// larger patches the pulls (shared-memory bandwidth) and the collision (FP32
// pipe) grow to 2,500 and 4,400; in FP64 the FP64 pipe is the bound (19 cycles
// per warp instruction and SM).
//
// The exchange goes through global memory (L2) in 128-bit words, {three 32-bit
// payloads, 32-bit step tag}, written and read with relaxed 128-bit accesses; a
// reader polls the word itself until it has the tag of the step. There is no
// flag and no fence: the payload is there when its tag is. (A ring of 152 CTAs
// exchanging 256 such words each takes 1,600 cycles a step, at 512 words 2,000;
// a release fence, a flag and an acquire fence take 9,000.) Words are
// double-buffered by the parity of the step. A CTA overwrites a word of step s
// at step s + 2; by then it has had the heartbeat of step s + 1 of every patch
// that its halo reaches, which that patch sent after it had read its words of
// step s. A poll has an iteration limit; a CTA that gives up sets bit 2 of the
// status word and returns, and so do its neighbours in turn.
//
// Which values cross is worked out once per launch, by both sides, from the
// node words. A patch pulls f and g on its own nodes, and g for phi on the ring
// of one around it and, next to ghost nodes, of two (the ghost average reaches
// one node further): each source that lies in another patch is wanted from it.
// The owner publishes the same set, seen from its side. A word's place follows
// from its owner, type and node, so neither asks the other.
//
// Bounce-back: where a node's source keeps no population, what the node takes
// instead is copied, once per step, to the solid cell where the plain pull looks
// for it (each such cell and direction serves one node). So every pull has
// the same constant offsets.
//
// Updates are in place: all pulls of a step (own nodes into registers, the
// ring's into phi) are over at the barrier before the collision.
//
// The per-node arithmetic is node_core (step_core.cuh): two x-adjacent nodes
// per thread in packed FP32x2 lanes, or one node in FP64, so the fields
// equal those of the other step kernels bit for bit.
#include "step_core.cuh"

#include <cmath>
#include <cstring>
#include <type_traits>

namespace pfk {
namespace {

// Polls of one word before a wait gives up: a poll is a round trip to L2 (0.4
// us and more), so some seconds; in a healthy run a word is there within a step.
constexpr int kSpinLimit = 1 << 22;
constexpr int kHaloX = 4, kHaloY = 3;   // three nodes are read; four in x keeps pairs aligned
// patches that a halo of three reaches, at most: one of three nodes or more at
// each side, three of one row above and below
constexpr int kMostHeartbeats = 3 * 7 - 1;
constexpr int kMaxResident = 152;       // CTAs of a one-lattice launch at most (one per SM)

// A word of the exchange: three 32-bit payloads and the step tag, one 128-bit
// access of memory.
struct Word { unsigned long long lo, hi; };
__device__ __forceinline__ Word ld_word(const Word* p)
{
    Word w;
    asm volatile("{\n\t.reg .b128 t;\n\tld.relaxed.gpu.global.b128 t, [%2];\n\tmov.b128 {%0, %1}, t;\n\t}"
                 : "=l"(w.lo), "=l"(w.hi)
                 : "l"(p)
                 : "memory");
    return w;
}
__device__ __forceinline__ void st_word(Word* p, unsigned a, unsigned b, unsigned c, unsigned tag)
{
    const unsigned long long lo = (unsigned long long)b << 32 | a, hi = (unsigned long long)tag << 32 | c;
    asm volatile("{\n\t.reg .b128 t;\n\tmov.b128 t, {%1, %2};\n\tst.relaxed.gpu.global.b128 [%0], t;\n\t}" ::"l"(p),
                 "l"(lo), "l"(hi)
                 : "memory");
}
__device__ __forceinline__ unsigned word_tag(const Word& w) { return (unsigned)(w.hi >> 32); }
__device__ __forceinline__ unsigned word_at(const Word& w, int k)
{
    return k == 0 ? (unsigned)w.lo : k == 1 ? (unsigned)(w.lo >> 32) : (unsigned)w.hi;
}

// The three populations of a word. Across a horizontal border (and a corner)
// directions are grouped by c_y: types 0, 1, 2 hold c_y = +1, 0, -1; across a
// vertical one by c_x: types 3, 4, 5. f takes types 0..5, g types 6..11.
constexpr int kTypes = 12;
__device__ __forceinline__ int type_of(int i, bool horizontal)
{
    const int x = (i == 1 || i == 5 || i == 8) ? 1 : ((i == 3 || i == 6 || i == 7) ? -1 : 0);
    const int y = (i == 2 || i == 5 || i == 6) ? 1 : ((i == 4 || i == 7 || i == 8) ? -1 : 0);
    return horizontal ? 1 - y : 4 - x;
}
// direction k (0..2) of type t (0..5)
__device__ __forceinline__ int type_dir(int t, int k)
{
    const unsigned d = t == 0 ? 0x652u : t == 1 ? 0x310u : t == 2 ? 0x874u : t == 3 ? 0x851u : t == 4 ? 0x420u : 0x763u;
    return (int)(d >> (4 * k)) & 0xf;
}

// Patches of a lattice: columns in units of UNIT nodes (2 in packed lanes)
// and the rows 1..ny-2, each cut into nearly equal parts (ResidentCut).
struct Rect { int x0, y0, w, h; };   // w without columns past nx

template <int UNIT>
__host__ __device__ __forceinline__ Rect patch_rect(const ResidentCut& c, int id, int nx)
{
    const int i = id % c.px, j = id / c.px;
    Rect r;
    r.x0 = UNIT * (int)((long long)i * c.units / c.px);
    r.y0 = 1 + (int)((long long)j * c.rows / c.py);
    const int x1 = UNIT * (int)((long long)(i + 1) * c.units / c.px);
    r.w = (x1 < nx ? x1 : nx) - r.x0;
    r.h = 1 + (int)((long long)(j + 1) * c.rows / c.py) - r.y0;
    return r;
}

// Place of the word of type t of a border node among its patch's words. A type
// that crosses horizontal borders takes rows of nodes, one that crosses
// vertical ones columns: of f the outermost at each side (what a pull reaches),
// of g the three outermost (a pull on the ring of one, or of two next to a
// ghost), so 24 (w + h) words in all. The words of a row lie side by side, those of
// the columns at both sides too: a warp publishes them together (400 steps of 256 x
// 128 FP32: the two sides apart 956 us, together 922; column after column 512 x 512
// FP32 took 3.5 % more).
// ROOMY (batches, whose words are one buffer however many the members): the place
// among the type's, each of which takes all 6 (w + h) border nodes, rows first.
// With the compact places a step of 256 uneven lattices in BF16 took 179 us
// instead of 175.
template <bool ROOMY>
__device__ __forceinline__ int slot_of(const ResidentCut& c, const Rect& r, int t, int lx, int ly)
{
    const int row = ly < 3 ? ly : ly - r.h + 6, col = lx < 3 ? lx : lx - r.w + 6;
    if (ROOMY) return ly < 3 || ly >= r.h - 3 ? row * r.w + lx : 6 * r.w + ly * 6 + col;
    const int tt = t % 6, g = 6 * (c.w + c.h);
    if (tt < 3) return t < 6 ? (2 * tt + (ly != 0)) * c.w + lx : g + (6 * tt + row) * c.w + lx;
    if (t < 6) return 6 * c.w + 2 * (tt - 3) * c.h + 2 * ly + (lx != 0);
    return g + 18 * c.w + 6 * (tt - 3) * c.h + 6 * ly + col;
}

// Words of a patch in one buffer: its types' places, then the heartbeat in a line
// of its own. Only active patches have words, in their order.
constexpr int kHeartbeat = 8;
template <bool ROOMY> __host__ __device__ __forceinline__ int patch_words(int w, int h) { return (ROOMY ? 72 : 24) * (w + h) + kHeartbeat; }
// (places of a ROOMY patch count from the type's first word)
template <bool ROOMY> __device__ __forceinline__ int type_words(const ResidentCut& c) { return ROOMY ? 6 * (c.w + c.h) : 0; }
// An entry of the publish list: type, place, cell. (Two orders of the bits: the
// other order costs 0.5 to 1.5 % of a step in each case.)
template <bool ROOMY> __device__ __forceinline__ uint32_t pub_entry(int t, int slot, int c)
{
    return ROOMY ? (uint32_t)t << 28 | (uint32_t)slot << 13 | (uint32_t)c : (uint32_t)slot << 17 | (uint32_t)t << 13 | (uint32_t)c;
}
template <bool ROOMY> __device__ __forceinline__ unsigned pub_type(uint32_t u) { return ROOMY ? u >> 28 : (u >> 13) & 0xfu; }
template <bool ROOMY> __device__ __forceinline__ unsigned pub_slot(uint32_t u) { return ROOMY ? (u >> 13) & 0x7fffu : u >> 17; }
template <bool ROOMY> __device__ __forceinline__ int first_word(const ResidentCut& c, int id)
{
    return (c.before[id >> 5] + __popc(c.active[id >> 5] & ((1u << (id & 31)) - 1u))) * patch_words<ROOMY>(c.w, c.h);
}

// Shared memory of a patch of at most WM x HM nodes: byte offsets of the
// arrays. Row and plane strides are constants, so a pull's offset is an
// immediate of its load.
constexpr int kMaxList(int w, int h) { return 8 * 2 * (w + h) + 512; }   // entries of an exchange list at most
constexpr int align16(int b) { return (b + 15) & ~15; }
template <int PREC, int WM, int HM>
struct Lay {
    static constexpr int E = PREC == PFLBM_FP64 ? 8 : PREC == PFLBM_FP32 ? 4 : 2, C = PREC == PFLBM_FP64 ? 8 : 4;
    // (one cell to spare at the end: the payload of heartbeats goes there)
    static constexpr int RS = WM + 2 * kHaloX, ROWS = HM + 2 * kHaloY, CELLS = (RS * ROWS + 8) & ~7, OWN = WM * HM;
    // exchange lists: 4 words per border node on each side are usual (f, g one
    // node deep, g two deep), 8 possible next to ghost nodes, more at corners:
    // what the lists do not hold waits in global memory
    static constexpr int CAP = 5 * 2 * (WM + HM) + 128, MAXLIST = kMaxList(WM, HM);
    static constexpr int kS = 0;
    static constexpr int kG0 = kS + align16(17 * CELLS * E);
    static constexpr int kPhi = kG0 + align16(CELLS * C);
    static constexpr int kSprev = kPhi + align16(CELLS * C);
    static constexpr int kWet = kSprev + align16(OWN * C);
    static constexpr int kWord = kWet + align16(OWN * C);
    static constexpr int kRing = kWord + align16(CELLS * 2);
    static constexpr int kGhost = kRing + align16((4 * (WM + HM) + 32) * 2);
    // bounce-back copies: up to 3 unknown links per node of a wall are usual;
    // more than the list holds wait in global memory
    static constexpr int COPIES = 6 * (WM + HM) + 64, MAXCOPY = 8 * (WM + 4) * (HM + 4);
    // whole lists, which no mask can exceed
    static constexpr ResidentSpill kMost{MAXLIST, MAXCOPY};
    static constexpr int kCopy = kGhost + align16((WM + 2) * (HM + 2) * 4);
    static constexpr int kPoll = kCopy + align16(COPIES * 4);
    static constexpr int kPollC = kPoll + align16(CAP * 4);
    static constexpr int kPub = kPollC + align16(CAP * 2);
    static constexpr int kBytes = kPub + align16(CAP * 4);
    static_assert(9 * CELLS <= 32768 && CELLS <= 8192, "packed offsets of the lists");
    static_assert(kBytes <= 227 * 1024 - 1024, "shared memory of one CTA");
};

// One lattice: its descriptor and cut are launch parameters. A batch: CTA b
// runs patch item[b].y (its place among the active ones in the upper half) of
// member item[b].x, whose words start at item[b].zw.
template <int PREC, bool BATCH> struct ResArgs;
struct ResCommon {
    Word* ll;                        // two buffers of ll_half words
    unsigned long long ll_half;
    uint32_t* spill;                 // list entries past what shared memory holds
    unsigned tag;                    // words of step s carry tag + s
    int steps;
};
template <int PREC> struct ResArgs<PREC, false> : ResCommon {
    StepArgs<PREC> a;
    ResidentCut cut;
    ResidentSpill room;              // of each CTA in spill (batches: Lay::kMost)
    int* need;                       // COUNT: the largest overflow of a list and of the copies
    uint16_t item[kMaxResident];     // patch of each CTA
};
template <int PREC> struct ResArgs<PREC, true> : ResCommon {
    const StepArgs<PREC>* a;
    const ResidentCut* cut;
    const uint4* item;
};

// Pulled populations of a lane: raw 16-bit pairs, F2, or double.
struct Hold1 {
    double w[9];
    __device__ __forceinline__ double operator[](int i) const { return w[i]; }
};
template <int PREC> struct LaneKind { using Hold = Hold2<PREC>; using C = F2; static constexpr int N = 2; };
template <> struct LaneKind<PFLBM_FP64> { using Hold = Hold1; using C = double; static constexpr int N = 1; };

// One pull for all nodes of the lane at cell c: plane PL (of f, or 8 + i of g)
// at the cell c_I back. (Where that cell keeps no population the bounce-back
// copies have put there what the node takes instead.)
template <int I, int PL, int PREC, int rs, int cells>
__device__ __forceinline__ void pull_lane(typename LaneKind<PREC>::Hold& v, const typename Store<PREC>::S* s, int c)
{
    constexpr int X = cx(I), Y = cy(I);
    const int at = c + (PL * cells - (Y * rs + X));
    if constexpr (PREC == PFLBM_FP64) {
        v.w[I] = PFLBM_LD(s, at, 17 * cells);
    } else if constexpr (PREC == PFLBM_FP32) {
        if constexpr (X == 0) v.w[I] = v2f(PFLBM_LD(reinterpret_cast<const float2*>(s), at >> 1, 17 * cells / 2));
        else v.w[I] = F2(PFLBM_LD(s, at, 17 * cells), PFLBM_LD(s, at + 1, 17 * cells));
    } else {
        const uint16_t* b = reinterpret_cast<const uint16_t*>(s);
        if constexpr (X == 0)
            v.w[I] = PFLBM_LD(reinterpret_cast<const uint32_t*>(s), at >> 1, 17 * cells / 2);
        else
            v.w[I] = (uint32_t)PFLBM_LD(b, at, 17 * cells) | ((uint32_t)PFLBM_LD(b, at + 1, 17 * cells) << 16);
    }
}
// Directions 1..8 of f (G = 0) or g (G = 8).
template <int G, int PREC, int rs, int cells>
__device__ __forceinline__ void pull_moving(typename LaneKind<PREC>::Hold& v, const typename Store<PREC>::S* s, int c)
{
    pull_lane<1, G + 1, PREC, rs, cells>(v, s, c);
    pull_lane<2, G + 2, PREC, rs, cells>(v, s, c);
    pull_lane<3, G + 3, PREC, rs, cells>(v, s, c);
    pull_lane<4, G + 4, PREC, rs, cells>(v, s, c);
    pull_lane<5, G + 5, PREC, rs, cells>(v, s, c);
    pull_lane<6, G + 6, PREC, rs, cells>(v, s, c);
    pull_lane<7, G + 7, PREC, rs, cells>(v, s, c);
    pull_lane<8, G + 8, PREC, rs, cells>(v, s, c);
}
// g_i of one node (the ring), in work units.
template <int I, int PREC, int rs, int cells>
__device__ __forceinline__ typename Store<PREC>::C pull_node(const typename Store<PREC>::S* s, int c)
{
    return Store<PREC>::template ldp<I>(PFLBM_LD(s, c + ((8 + I) * cells - (cy(I) * rs + cx(I))), 17 * cells));
}

// phi = sum_i g_i of the lane's nodes, in the order of the scalar code.
template <int PREC>
__device__ __forceinline__ typename LaneKind<PREC>::C lane_phi(const typename LaneKind<PREC>::Hold& v,
                                                               const typename Store<PREC>::G0T raw[])
{
    using T = Store<PREC>;
    using C = typename LaneKind<PREC>::C;
    C s;
    if constexpr (T::kNorm)
        s = fmadd(C(T::template unit<1>()), (v[1] + v[2]) + (v[3] + v[4]),
                  C(T::template unit<5>()) * ((v[5] + v[6]) + (v[7] + v[8])));
    else
        s = ((v[1] + v[2]) + (v[3] + v[4])) + ((v[5] + v[6]) + (v[7] + v[8]));
    if constexpr (LaneKind<PREC>::N == 2) return F2(T::g0(raw[0]), T::g0(raw[1])) + s;
    else return raw[0] + s;
}

// The lane's stores go to its own cells in shared memory. `pair`: both
// columns exist (the last column of an odd-width lattice is alone; the cell
// beside it is halo).
template <int PREC, int cells, int PARTS>
struct LaneS {
    using T = Store<PREC>;
    using S = typename T::S;
    using C = typename LaneKind<PREC>::C;
    using FArr = typename LaneKind<PREC>::Hold;
    using R = typename T::C;
    static constexpr int N = LaneKind<PREC>::N, kParts = PARTS;
    S* s;                       // plane 0 of f at the lane's cell; g_i is plane 8 + i
    typename T::G0T* g0;
    R* sp;
    const R* wt;
    int k;
    bool valid[2], pair;
    typename T::G0T g0raw[2];
    __device__ __forceinline__ C wet(const StepArgs<PREC>&) const
    {
        if constexpr (N == 2) return v2f(*reinterpret_cast<const float2*>(wt));
        else return *wt;
    }
    __device__ __forceinline__ void check_u(const StepArgs<PREC>& a, C uu) const
    {
        if constexpr (N == 2) {
            if ((valid[0] && !(uu.x < 0.09f)) || (valid[1] && !(uu.y < 0.09f))) atomicOr(a.status, 1);
        } else {
            if (!(uu < 0.09)) atomicOr(a.status, 1);
        }
    }
    __device__ __forceinline__ void put(int plane, C v) const
    {
        if constexpr (PREC == PFLBM_FP64) {
            s[plane * cells] = v;
        } else if constexpr (PREC == PFLBM_FP32) {
            if (pair) *reinterpret_cast<float2*>(s + plane * cells) = f2v(v);
            else s[plane * cells] = v.x;
        }
    }
    __device__ __forceinline__ void put_raw(int plane, uint32_t u) const
    {
        if (pair) *reinterpret_cast<uint32_t*>(s + plane * cells) = u;
        else *reinterpret_cast<uint16_t*>(s + plane * cells) = (uint16_t)u;
    }
    template <int I>
    __device__ __forceinline__ void store_f(const StepArgs<PREC>&, C v) const
    {
        if constexpr (T::kNorm) put_raw(I, Hold2<PREC>::pack_raw(v));
        else put(I, v);
    }
    template <int I>
    __device__ __forceinline__ C store_g(const StepArgs<PREC>&, C v) const
    {
        if constexpr (T::kNorm) {
            const uint32_t u = Hold2<PREC>::pack_raw(v);
            put_raw(8 + I, u);
            return v - Hold2<PREC>::unpack_raw(u);
        } else {
            put(8 + I, v);
            return C(0);
        }
    }
    __device__ __forceinline__ int32_t g0_lane(int32_t raw, float d, bool ok, const StepArgs<PREC>& a) const
    {
        long long q = (long long)raw + __float2ll_rn(d * 1073741824.0f);
        if (q > INT_MAX || q < -INT_MAX) {
            if (ok) atomicOr(a.status, 2);
            q = q > 0 ? INT_MAX : -INT_MAX;
        }
        return (int32_t)q;
    }
    __device__ __forceinline__ void store_g0(const StepArgs<PREC>& a, C d) const
    {
        if constexpr (N == 2) {
            const int2 v = make_int2(g0_lane(g0raw[0], d.x, valid[0], a), g0_lane(g0raw[1], d.y, valid[1], a));
            if (pair) *reinterpret_cast<int2*>(g0) = v;
            else *g0 = v.x;
        } else {
            *g0 = T::g0_add(g0raw[0], d, a.status);
        }
    }
    __device__ __forceinline__ void store_sprev(const StepArgs<PREC>&, C v) const
    {
        if constexpr (N == 2) *reinterpret_cast<float2*>(sp) = f2v(v);
        else *sp = v;
    }
};

// COUNT: only the lengths of the lists, into need.
template <int PREC, int VV, int WM, int HM, int P, int NTMAX, bool BATCH, bool COUNT>
__global__ void __launch_bounds__(NTMAX, 1) k_resident(const __grid_constant__ ResArgs<PREC, BATCH> q)
{
    using T = Store<PREC>;
    using S = typename T::S;
    using G0T = typename T::G0T;
    using R = typename T::C;                      // scalar arithmetic type
    using C = typename LaneKind<PREC>::C;         // lane arithmetic type
    using Hold = typename LaneKind<PREC>::Hold;
    constexpr int N = LaneKind<PREC>::N;
    extern __shared__ __align__(16) unsigned char sm[];
    __shared__ int4 s_off[kTypes];                // element offsets of a word type's populations
    __shared__ int s_n[6];                        // poll, publish, ring, ghost, copy entries; give-up

    __shared__ uint32_t s_seen[kMaxPatches / 32];
    __shared__ __align__(16) unsigned char s_arg[BATCH ? sizeof(StepArgs<PREC>) + sizeof(ResidentCut) : 16];
    const StepArgs<PREC>* ap;
    const ResidentCut* cp;
    Word* ll = q.ll;
    int id, rank = 0;                             // patch; its place among the member's active ones
    if constexpr (BATCH) {
        // the member's descriptor and cut, read field by field where used
        const uint4 it = q.item[blockIdx.x];
        constexpr int NA = sizeof(StepArgs<PREC>) / 4, NC = sizeof(ResidentCut) / 4;
        static_assert(sizeof(StepArgs<PREC>) % 8 == 0 && sizeof(ResidentCut) % 4 == 0, "copied in words");
        const int* sa = reinterpret_cast<const int*>(q.a + it.x);
        const int* sc = reinterpret_cast<const int*>(q.cut + it.x);
        for (int i = threadIdx.x; i < NA + NC; i += blockDim.x)
            reinterpret_cast<int*>(s_arg)[i] = i < NA ? sa[i] : sc[i - NA];
        ap = reinterpret_cast<const StepArgs<PREC>*>(s_arg);
        cp = reinterpret_cast<const ResidentCut*>(s_arg + sizeof(StepArgs<PREC>));
        id = (int)(it.y & 0xffffu);
        rank = (int)(it.y >> 16);
        ll += (unsigned long long)it.w << 32 | it.z;
        __syncthreads();
    } else {
        ap = &q.a;
        cp = &q.cut;
        id = q.item[blockIdx.x];
    }
    const StepArgs<PREC>& a = *ap;
    const ResidentCut& cut = *cp;
    const Rect r = patch_rect<N>(cut, id, a.nx);
    const int tid = threadIdx.x, NT = blockDim.x;
    const int nx = a.nx, ny = a.ny, pitch = a.pitch, plane = a.plane;
    const int w2 = (r.w + N - 1) / N * N;
    using L = Lay<PREC, WM, HM>;
    constexpr int rs = L::RS, cells = L::CELLS;
    const int area = rs * (r.h + 2 * kHaloY);     // cells in use
    S* sS = reinterpret_cast<S*>(sm + L::kS);
    G0T* sG0 = reinterpret_cast<G0T*>(sm + L::kG0);
    R* sPhi = reinterpret_cast<R*>(sm + L::kPhi);
    R* sSp = reinterpret_cast<R*>(sm + L::kSprev);
    R* sWet = reinterpret_cast<R*>(sm + L::kWet);
    uint16_t* sW = reinterpret_cast<uint16_t*>(sm + L::kWord);
    uint16_t* sRing = reinterpret_cast<uint16_t*>(sm + L::kRing);
    uint32_t* sGhost = reinterpret_cast<uint32_t*>(sm + L::kGhost);
    uint32_t* sCopy = reinterpret_cast<uint32_t*>(sm + L::kCopy);
    uint32_t* sPoll = reinterpret_cast<uint32_t*>(sm + L::kPoll);
    uint16_t* sPollC = reinterpret_cast<uint16_t*>(sm + L::kPollC);
    uint32_t* sPub = reinterpret_cast<uint32_t*>(sm + L::kPub);

    // entry `at` of the lists (0: poll, 1: its cell, 2: publish) and of the copies
    // past shared memory, in the CTA's part of the overflow. A batch's has room
    // for whole lists, list by list.
    int room_list = L::MAXLIST, room_copy = L::MAXCOPY;
    uint32_t* gList = q.spill + (size_t)blockIdx.x * L::kMost.words();
    uint32_t* gCopy = gList + 3 * L::MAXLIST;
    if constexpr (!BATCH) {
        room_list = L::CAP + q.room.list;
        room_copy = L::COPIES + q.room.copies;
        gList = q.spill + (size_t)blockIdx.x * q.room.words() - 3 * L::CAP;
        gCopy = gList + 3 * room_list - L::COPIES;
    }
    auto over = [&](int list, int at) { return gList + (BATCH ? list * L::MAXLIST + at : 3 * at + list); };

    // ---- set-up: the state, the node words, the lists ----
    if (tid < 6) s_n[tid] = 0;
    for (int i = tid; i < kMaxPatches / 32; i += NT) s_seen[i] = 0;
    if (tid < kTypes) {
        // g_0, the first of its types (7 and 10), has an array of its own
        // (32-bit elements in the 16-bit formats)
        const int t = tid % 6, g = tid < 6 ? 0 : 8 * cells;
        const bool g0 = tid == 7 || tid == 10;
        s_off[tid] = make_int4(g0 ? (L::kG0 - L::kS) / (T::kNorm ? 4 : (int)sizeof(S)) : g + type_dir(t, 0) * cells,
                               g + type_dir(t, 1) * cells, g + type_dir(t, 2) * cells, g0 ? 1 : 0);
    }
    uint32_t* mask = reinterpret_cast<uint32_t*>(sPhi);   // wanted / published word types per cell, until the lists exist
    for (int c = tid; c < area; c += NT) {
        const int ly = c / rs - kHaloY, lx = c % rs - kHaloX;
        const int gy = r.y0 + ly;
        const bool in = gy >= 0 && gy < ny;
        const int k = in ? gy * pitch + wrapn(r.x0 + lx, nx) : 0;
        sW[c] = in ? PFLBM_LD(a.cls, k, plane) : (uint8_t)CLS_OUT;
        mask[c] = 0;
        if constexpr (COUNT) continue;
        sG0[c] = in ? PFLBM_LD(a.in.g0, k, plane) : G0T(0);
#pragma unroll
        for (int p = 0; p < 17; ++p) {
            S v;
            if (p < 9) v = PFLBM_LD(a.in.f, p * plane + (in ? k : 0), 9LL * plane);
            else v = PFLBM_LD(a.in.g, (p - 8) * plane + (in ? k : 0), 9LL * plane);
            sS[p * cells + c] = v;
        }
        if (lx >= 0 && lx < w2 && ly >= 0 && ly < r.h) {
            const int o = ly * WM + lx;
            const bool own = lx < r.w;
            sSp[o] = own ? PFLBM_LD(a.sprev, k, plane) : R(0);
            sWet[o] = own && (sW[c] & F_WET) ? PFLBM_LD(a.wet, k, plane) : R(0);
        }
    }
    __syncthreads();
    for (int c = tid; c < area; c += NT) {
        const int ly = c / rs - kHaloY, lx = c % rs - kHaloX;
        if (lx < -2 || lx > r.w + 1 || ly < -2 || ly > r.h + 1) continue;
        unsigned w = sW[c] & 0xffu;
#pragma unroll
        for (int j = 1; j < 9; ++j)
            if (zeta_of((uint8_t)sW[c + cy(j) * rs + cx(j)])) w |= 256u << (j - 1);
        sW[c] = (uint16_t)w;
    }
    __syncthreads();
    for (int c = tid; c < area; c += NT) {
        const int ly = c / rs - kHaloY, lx = c % rs - kHaloX;
        if (lx < -2 || lx > r.w + 1 || ly < -2 || ly > r.h + 1) continue;
        const unsigned w = sW[c];
        const bool near1 = lx >= -1 && lx <= r.w && ly >= -1 && ly <= r.h;
        if (near1 && (uint8_t)w != CLS_OUT && (w & CLS_MASK) == CLS_GHOST)
            sGhost[atomicAdd(&s_n[3], 1)] = w << 16 | (uint32_t)c;
        if (!zeta_of((uint8_t)w)) continue;
        auto mine = [&](int x, int y) { return x >= 0 && x < r.w && y >= 0 && y < r.h; };
        const bool own = mine(lx, ly), ng = (w & F_NEARGHOST) != 0;
        const bool want = own || near1 || ng;   // this patch needs phi here
        // another patch needs phi here: it has a node within one (two next to a
        // ghost), across a horizontal border or a corner, or a vertical one
        const int d = ng ? 2 : 1;
        const bool give_h = ly < d || ly >= r.h - d, give_v = lx < d || lx >= r.w - d;
        auto mark = [&](int i, int o) {
            const unsigned zm = w >> 8;
            int p = o, dx = 0, dy = 0;
            if (zm & (1u << (i - 1))) { dx = cx(i); dy = cy(i); }
            if (zm & (1u << (o - 1))) { p = i; dx = -cx(i); dy = -cy(i); }
            const bool src = mine(lx + dx, ly + dy), src_h = ly + dy < 0 || ly + dy >= r.h;
            uint32_t m = 0;
            if (src) {
                if (give_h) m |= 64u << type_of(p, true);
                if (give_v) m |= 64u << type_of(p, false);
                if (!own) m |= 1u << type_of(p, ly < 0 || ly >= r.h);
            } else {
                if (want) m |= 64u << type_of(p, src_h);
                if (own) m |= 1u << type_of(p, src_h);
            }
            if (m) atomicOr(&mask[c + dy * rs + dx], m);
            // an unknown population: copied to where the plain pull looks for it
            if (p == o && (own || want)) {
                const uint32_t dst = (uint32_t)(i * cells + c - (cy(i) * rs + cx(i)));
                const uint32_t from = (uint32_t)(o * cells + c + dy * rs + dx);
                const int at = atomicAdd(&s_n[4], 1);
                if (at < room_copy)
                    (at < L::COPIES ? sCopy + at : gCopy + at)[0] = (own ? 1u << 31 : 0u) | dst << 16 | from;
            }
        };
#pragma unroll
        for (int i = 1; i < 9; ++i) mark(i, opp(i));
        uint32_t m0 = 0;
        if (own) m0 = (give_h ? 64u << type_of(0, true) : 0u) | (give_v ? 64u << type_of(0, false) : 0u);
        else if (want) m0 = 64u << type_of(0, ly < 0 || ly >= r.h);
        if (m0) atomicOr(&mask[c], m0);
        if (!own && want) sRing[atomicAdd(&s_n[2], 1)] = (uint16_t)c;
    }
    __syncthreads();
    if constexpr (COUNT) {
        for (int c = tid; c < area; c += NT) {
            const int ly = c / rs - kHaloY, lx = c % rs - kHaloX, n = __popc(mask[c]);
            if (n) atomicAdd(&s_n[lx >= 0 && lx < r.w && ly >= 0 && ly < r.h], n);
        }
        __syncthreads();
        if (tid == 0) {
            const int poll = s_n[0] + kMostHeartbeats;
            atomicMax(&q.need[0], (poll > s_n[1] ? poll : s_n[1]) - L::CAP);
            atomicMax(&q.need[1], s_n[4] - L::COPIES);
        }
        return;
    }
    for (int p = 0; p < kTypes; ++p) {
        for (int c0 = tid & ~31; c0 < area; c0 += NT) {
            const int c = c0 + (tid & 31), ly = c / rs - kHaloY, lx = c % rs - kHaloX;
            const bool set = c < area && ((mask[c] >> p) & 1u);
            const bool own = lx >= 0 && lx < r.w && ly >= 0 && ly < r.h;
#pragma unroll
            for (int side = 0; side < 2; ++side) {
                const bool on = set && own == (side == 1);
                const unsigned m = __ballot_sync(0xffffffffu, on);
                if (!m) continue;
                int at = 0;
                if ((tid & 31) == 0) at = atomicAdd(&s_n[side], __popc(m));
                at = __shfl_sync(0xffffffffu, at, 0) + __popc(m & ((1u << (tid & 31)) - 1u));
                if (!on || at >= room_list) continue;
                if (side == 1) {
                    (at < L::CAP ? sPub + at : over(2, at))[0] =
                        pub_entry<BATCH>(p, slot_of<BATCH>(cut, r, p, lx, ly), c);
                } else {
                    const int gx = wrapn(r.x0 + lx, nx), gy = r.y0 + ly;
                    const int i = ((gx / N + 1) * cut.px - 1) / cut.units, j = (gy * cut.py - 1) / cut.rows;
                    const int from = j * cut.px + i;
                    const Rect o = patch_rect<N>(cut, from, nx);
                    const uint32_t u = (uint32_t)p << 28 | (uint32_t)(first_word<BATCH>(cut, from) + p * type_words<BATCH>(cut) +
                                                                      slot_of<BATCH>(cut, o, p, gx - o.x0, gy - o.y0));
                    atomicOr(&s_seen[from >> 5], 1u << (from & 31));
                    if (at < L::CAP) {
                        sPoll[at] = u;
                        sPollC[at] = (uint16_t)c;
                    } else {
                        *over(0, at) = u;
                        *over(1, at) = (uint32_t)c;
                    }
                }
            }
        }
    }
    __syncthreads();
    // heartbeats: one word of every patch that this one's halo reaches and that
    // it wants nothing else from, so that neither runs ahead of the other
    for (int c = tid; c < area; c += NT) {
        const int ly = c / rs - kHaloY, lx = c % rs - kHaloX, gy = r.y0 + ly;
        if (lx < -3 || lx > r.w + 2 || gy < 1 || gy > ny - 2) continue;
        const int gx = wrapn(r.x0 + lx, nx);
        const int of = ((gy * cut.py - 1) / cut.rows) * cut.px + ((gx / N + 1) * cut.px - 1) / cut.units;
        if (of == id || !(cut.active[of >> 5] >> (of & 31) & 1u)) continue;
        if (s_seen[of >> 5] >> (of & 31) & 1u) continue;
        if (atomicOr(&s_seen[of >> 5], 1u << (of & 31)) >> (of & 31) & 1u) continue;
        const int at = atomicAdd(&s_n[0], 1);
        const uint32_t u = (uint32_t)(first_word<BATCH>(cut, of) + patch_words<BATCH>(cut.w, cut.h) - kHeartbeat);
        if (at < L::CAP) {
            sPoll[at] = u;
            sPollC[at] = (uint16_t)(cells - 1);
        } else if (at < room_list) {
            *over(0, at) = u;
            *over(1, at) = (uint32_t)(cells - 1);
        }
    }
    __syncthreads();
    for (int c = tid; c < area; c += NT) sPhi[c] = R(0);
    const int n_poll = s_n[0], n_pub = s_n[1], n_ring = s_n[2], n_ghost = s_n[3], n_copy = s_n[4];
    if (n_poll > room_list || n_pub > room_list || n_copy > room_copy) {   // cannot happen (the room was worked out); nothing was written past the lists
        if (tid == 0) atomicOr(a.status, 4);
        return;
    }

    // ---- the thread's lanes: cell, node words, place among the own nodes.
    // FP64, patches of at most 32 nodes per four warps: a node's collision is
    // shared by three warps of different schedulers, each of which evaluates the
    // moments (half of the work). One scheduler takes 64 cycles for a warp's FP64
    // instruction, the SM 19, so a patch of one warp leaves two thirds of the
    // pipe idle: 100 x 50 in 150 patches 7.9 -> 6.1 us a step. ----
    const int wl = w2 / N, nl = wl * r.h;
    const bool team = PREC == PFLBM_FP64 && nl <= NT / 128 * 32;
    const int part = team ? (tid >> 5) & 3 : 0;        // 3: no lane
    const int t_first = !team ? tid : part == 3 ? nl : (tid >> 7) * 32 + (tid & 31);
    int cell[P], own[P];
    unsigned word[P][2];
#pragma unroll
    for (int j = 0; j < P; ++j) {
        const int t = t_first + j * NT;
        const int ly = t / wl, lx = N * (t - ly * wl);
        cell[j] = t < nl ? (ly + kHaloY) * rs + lx + kHaloX : kHaloY * rs + kHaloX;
        own[j] = t < nl ? ly * WM + lx : 0;
        word[j][0] = t < nl ? sW[cell[j]] : (unsigned)CLS_OUT;
        word[j][1] = t < nl && N == 2 && lx + 1 < r.w ? sW[cell[j] + 1] : (unsigned)CLS_OUT;
    }
    __syncthreads();

    for (int s = 1; s <= q.steps; ++s) {
        // ---- bounce-back (Sec. 2.2.2): copies for the links of the wall nodes ----
        if (n_copy > 0) {
            for (int t = tid; t < n_copy; t += NT) {
                const uint32_t e = t < L::COPIES ? sCopy[t] : gCopy[t];
                const int dst = (int)(e >> 16) & 0x7fff, from = (int)e & 0xffff;
                PFLBM_ST(sS, 8 * cells + dst, 17 * cells, PFLBM_LD(sS, 8 * cells + from, 17 * cells));
                if (e >> 31) PFLBM_ST(sS, dst, 17 * cells, PFLBM_LD(sS, from, 17 * cells));
            }
            __syncthreads();
        }
        // ---- pulls and phi: the own nodes, the ring ----
        Hold g[P], f[P];
        G0T raw[P][2];
#pragma unroll
        for (int j = 0; j < P; ++j) {
            const bool z0 = zeta_of((uint8_t)word[j][0]), z1 = zeta_of((uint8_t)word[j][1]);
            if (!z0 && !z1) continue;
            const int c = cell[j];
            if constexpr (N == 2) {
                const int2 v = PFLBM_LD(reinterpret_cast<const int2*>(sG0), c >> 1, cells / 2);
                raw[j][0] = v.x;
                raw[j][1] = v.y;
            } else {
                raw[j][0] = PFLBM_LD(sG0, c, cells);
            }
            if constexpr (PREC == PFLBM_FP64) f[j].w[0] = sS[c];
            else if constexpr (PREC == PFLBM_FP32) f[j].w[0] = v2f(*reinterpret_cast<const float2*>(sS + c));
            else f[j].w[0] = *reinterpret_cast<const uint32_t*>(sS + c);
            pull_moving<8, PREC, rs, cells>(g[j], sS, c);
            pull_moving<0, PREC, rs, cells>(f[j], sS, c);
            const C ph = lane_phi<PREC>(g[j], raw[j]);
            if constexpr (N == 2) {
                if (z0) sPhi[c] = ph.x;
                if (z1) sPhi[c + 1] = ph.y;
            } else if (part == 0) {
                sPhi[c] = ph;
            }
        }
        for (int t = NT - 1 - tid; t < n_ring; t += NT) {
            const int c = sRing[t];
            R v[9];
            v[0] = T::g0(PFLBM_LD(sG0, c, cells));
            v[1] = pull_node<1, PREC, rs, cells>(sS, c);
            v[2] = pull_node<2, PREC, rs, cells>(sS, c);
            v[3] = pull_node<3, PREC, rs, cells>(sS, c);
            v[4] = pull_node<4, PREC, rs, cells>(sS, c);
            v[5] = pull_node<5, PREC, rs, cells>(sS, c);
            v[6] = pull_node<6, PREC, rs, cells>(sS, c);
            v[7] = pull_node<7, PREC, rs, cells>(sS, c);
            v[8] = pull_node<8, PREC, rs, cells>(sS, c);
            PFLBM_ST(sPhi, c, cells, phi_of<PREC>(v));
        }
        __syncthreads();

        // ---- ghost values (Sec. 2.2.2; Robin on flat walls in Appendix A cases 1 and 3) ----
        if (n_ghost > 0) {
            for (int t = tid; t < n_ghost; t += NT) {
                const uint32_t e = sGhost[t], w = e >> 16;
                const int c = (int)(e & 0xffffu);
                if (w & (F_GHOST_UP | F_GHOST_DOWN)) {
                    const int ly = c / rs - kHaloY, lx = c % rs - kHaloX;
                    const R coef = PFLBM_LD(a.wet, (r.y0 + ly) * pitch + wrapn(r.x0 + lx, nx), plane);
                    sPhi[c] = robin_ghost<R>(sPhi[(w & F_GHOST_UP) ? c + rs : c - rs], coef);
                } else {
                    R num = R(0), den = R(0);
#pragma unroll
                    for (int j = 1; j < 9; ++j)
                        if (w & (256u << (j - 1))) {
                            num += sPhi[c + cy(j) * rs + cx(j)];
                            den += R(1);
                        }
                    sPhi[c] = num / den;
                }
            }
            __syncthreads();
        }

        // ---- collision, in place ----
        auto collide = [&](const int j, auto parts) {
            LaneS<PREC, cells, decltype(parts)::value> lane;
            lane.valid[0] = zeta_of((uint8_t)word[j][0]);
            lane.valid[1] = zeta_of((uint8_t)word[j][1]);
            if (!lane.valid[0] && !lane.valid[1]) return;
            const int c = cell[j];
            lane.pair = N == 1 || (uint8_t)word[j][1] != CLS_OUT;
            lane.s = sS + c;
            lane.g0 = sG0 + c;
            lane.sp = sSp + own[j];
            lane.wt = sWet + own[j];
            lane.k = 0;
            lane.g0raw[0] = raw[j][0];
            lane.g0raw[1] = raw[j][1];
            C gpx, gpy, lap, ph;
            if constexpr (N == 2) {
                F2 Wr[3], Cr[3], Er[3];
#pragma unroll
                for (int y = 0; y < 3; ++y) {
                    const float2* row = reinterpret_cast<const float2*>(sPhi + c + (y - 1) * rs);
                    const float2 l = row[-1], m = row[0], e = row[1];
                    Wr[y] = F2(l.y, m.x);
                    Cr[y] = F2(m.x, m.y);
                    Er[y] = F2(m.y, e.x);
                }
                ph = Cr[1];
                stencil9<F2>(Cr[1], Er[1], Wr[1], Cr[2], Cr[0], Er[2], Wr[2], Wr[0], Er[0], gpx, gpy, lap);
            } else {
                const R* b = sPhi + c;
                ph = b[0];
                stencil9<double>(b[0], b[1], b[-1], b[rs], b[-rs], b[rs + 1], b[rs - 1], b[-rs - 1], b[-rs + 1], gpx, gpy,
                                 lap);
            }
            node_core<PREC, true, VV>(
                a, lane, ph, gpx, gpy, lap, g[j], [&](Hold& fv) { fv = f[j]; },
                [&](int) {
                    if constexpr (N == 2) return v2f(*reinterpret_cast<const float2*>(lane.sp));
                    else return *lane.sp;
                },
                [](C, C, C, C) {});
        };
        if constexpr (PREC == PFLBM_FP64) {
            if (!team) collide(0, std::integral_constant<int, kPartAll>());
            else if (part == 0) collide(0, std::integral_constant<int, kPartAxes>());
            else if (part == 1) collide(0, std::integral_constant<int, kPartDiagonals>());
            else if (part == 2) collide(0, std::integral_constant<int, kPartG>());
        } else {
#pragma unroll
            for (int j = 0; j < P; ++j) collide(j, std::integral_constant<int, kPartAll>());
        }
        if (s == q.steps) break;
        __syncthreads();

        // ---- exchange: publish the border, then wait for the halo ----
        const unsigned tag = q.tag + (unsigned)s;
        constexpr int WPT = PREC == PFLBM_FP64 ? 2 : 1;   // words per triple
        constexpr int NS = (L::kPhi - L::kS) / (int)sizeof(S), NW = (L::kPhi - L::kS) / 4;   // elements of sS and sG0
        Word* buf = ll + (s & 1) * q.ll_half;
        {
            const int words = patch_words<BATCH>(cut.w, cut.h);
            Word* to = buf + (unsigned long long)((BATCH ? rank : (int)blockIdx.x) * words) * WPT;
            if (tid < WPT) st_word(to + (words - kHeartbeat) * WPT + tid, 0u, 0u, 0u, tag);
            for (int e = tid; e < n_pub; e += NT) {
                const uint32_t u = e < L::CAP ? sPub[e] : *over(2, e);
                const int c = (int)(u & 0x1fffu);
                Word* d = to + (pub_type<BATCH>(u) * type_words<BATCH>(cut) + pub_slot<BATCH>(u)) * WPT;
                const int4 off = s_off[pub_type<BATCH>(u)];
                if constexpr (PREC == PFLBM_FP64) {
                    const double v0 = PFLBM_LD(sS, c + off.x, NS), v1 = PFLBM_LD(sS, c + off.y, NS),
                                 v2 = PFLBM_LD(sS, c + off.z, NS);
                    st_word(d, (unsigned)__double2loint(v0), (unsigned)__double2hiint(v0), (unsigned)__double2loint(v1), tag);
                    st_word(d + 1, (unsigned)__double2hiint(v1), (unsigned)__double2loint(v2), (unsigned)__double2hiint(v2),
                            tag);
                } else if constexpr (PREC == PFLBM_FP32) {
                    const uint32_t* b = reinterpret_cast<const uint32_t*>(sS);
                    st_word(d, PFLBM_LD(b, c + off.x, NS), PFLBM_LD(b, c + off.y, NS), PFLBM_LD(b, c + off.z, NS), tag);
                } else {
                    const uint16_t* b = reinterpret_cast<const uint16_t*>(sS);
                    const unsigned v0 = off.w ? PFLBM_LD(reinterpret_cast<const uint32_t*>(sS), c + off.x, NW)
                                              : (unsigned)PFLBM_LD(b, c + off.x, NS);
                    st_word(d, v0, PFLBM_LD(b, c + off.y, NS), PFLBM_LD(b, c + off.z, NS), tag);
                }
            }
        }
        constexpr int U = 2;   // words a thread waits for together
        bool late = false;
        for (int e0 = tid; e0 < n_poll; e0 += U * NT) {
            Word v[U][WPT];
            bool have[U];
            const Word* src[U];
            int4 off[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int e = e0 + u * NT;
                have[u] = e >= n_poll;
                const uint32_t ent = have[u] ? 0u : e < L::CAP ? sPoll[e] : *over(0, e);
                const int c = have[u] ? 0 : e < L::CAP ? (int)sPollC[e] : (int)*over(1, e);
                src[u] = buf + (ent & 0xfffffffu) * WPT;
                off[u] = s_off[ent >> 28];
                off[u].x += c;
                off[u].y += c;
                off[u].z += c;
            }
            for (int tries = 0;; ++tries) {
                bool all = true;
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    if (have[u]) continue;
                    bool ok = true;
#pragma unroll
                    for (int x = 0; x < WPT; ++x) {
                        v[u][x] = ld_word(src[u] + x);
                        ok = ok && word_tag(v[u][x]) == tag;
                    }
                    have[u] = ok;
                    all = all && ok;
                }
                if (all) break;
                if (tries >= kSpinLimit) { late = true; break; }
            }
            if (late) break;
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int e = e0 + u * NT;
                if (e >= n_poll) continue;
                const Word& w = v[u][0];
                if constexpr (PREC == PFLBM_FP64) {
                    const Word& y = v[u][1];
                    PFLBM_ST(sS, off[u].x, NS, __hiloint2double((int)word_at(w, 1), (int)word_at(w, 0)));
                    PFLBM_ST(sS, off[u].y, NS, __hiloint2double((int)word_at(y, 0), (int)word_at(w, 2)));
                    PFLBM_ST(sS, off[u].z, NS, __hiloint2double((int)word_at(y, 2), (int)word_at(y, 1)));
                } else if constexpr (PREC == PFLBM_FP32) {
                    uint32_t* b = reinterpret_cast<uint32_t*>(sS);
                    PFLBM_ST(b, off[u].x, NS, word_at(w, 0));
                    PFLBM_ST(b, off[u].y, NS, word_at(w, 1));
                    PFLBM_ST(b, off[u].z, NS, word_at(w, 2));
                } else {
                    uint16_t* b = reinterpret_cast<uint16_t*>(sS);
                    if (off[u].w) PFLBM_ST(reinterpret_cast<uint32_t*>(sS), off[u].x, NW, word_at(w, 0));
                    else PFLBM_ST(b, off[u].x, NS, (uint16_t)word_at(w, 0));
                    PFLBM_ST(b, off[u].y, NS, (uint16_t)word_at(w, 1));
                    PFLBM_ST(b, off[u].z, NS, (uint16_t)word_at(w, 2));
                }
            }
        }
        if (late) s_n[5] = 1;
        __syncthreads();
        if (s_n[5]) {
            if (tid == 0) atomicOr(a.status, 4);
            return;
        }
    }

    // ---- the state back to global memory: the copy that as many single steps
    // would end in. For an even count that is the copy the launch began with;
    // by now every patch that reads this one's nodes from it has done so (it
    // has sent the heartbeat of a step). ----
    __syncthreads();
    const Planes<PREC> to = q.steps & 1 ? a.out : a.in;
    for (int o = tid; o < w2 * r.h; o += NT) {
        const int ly = o / w2, lx = o - ly * w2, c = (ly + kHaloY) * rs + lx + kHaloX;
        if (lx >= r.w || !zeta_of((uint8_t)sW[c])) continue;
        const int k = (r.y0 + ly) * pitch + r.x0 + lx;
        PFLBM_ST(to.g0, k, plane, sG0[c]);
#pragma unroll
        for (int p = 0; p < 17; ++p) {
            if (p < 9) PFLBM_ST(to.f, p * plane + k, 9LL * plane, sS[p * cells + c]);
            else PFLBM_ST(to.g, (p - 8) * plane + k, 9LL * plane, sS[p * cells + c]);
        }
        if (!a.dgdt) PFLBM_ST(a.sprev, k, plane, sSp[ly * WM + lx]);
    }
}

// Patch classes: the largest patch, lanes per thread and threads per CTA. A
// lane needs 115 to 140 registers unconstrained, and 512 threads may have 128.
struct Class { int wm, hm, p, nt; };
constexpr int kClassCount = 3;
constexpr Class class_of(int precision, int k)
{
    if (precision == PFLBM_FP64) return k == 0 ? Class{16, 16, 1, 256} : Class{32, 16, 1, 512};
    if (k == 0) return Class{16, 16, 1, 256};
    if (k == 1) return Class{32, 32, 1, 512};
    return precision == PFLBM_FP32 ? Class{52, 34, 2, 448} : Class{64, 32, 2, 512};
}
constexpr int classes(int precision) { return precision == PFLBM_FP64 ? 2 : kClassCount; }

template <int PREC, int K> constexpr ResidentSpill spill_k() { return Lay<PREC, class_of(PREC, K).wm, class_of(PREC, K).hm>::kMost; }

template <int PREC, int VV, int K, bool BATCH>
cudaError_t launch_k(const ResArgs<PREC, BATCH>& q, int n_items, int nt, cudaStream_t stream)
{
    constexpr Class c = class_of(PREC, K);
    auto* k = k_resident<PREC, VV, c.wm, c.hm, c.p, c.nt, BATCH, false>;
    if constexpr (!BATCH)
        if (q.steps == 0) k = k_resident<PREC, 0, c.wm, c.hm, c.p, c.nt, false, true>;
    constexpr int smem = Lay<PREC, c.wm, c.hm>::kBytes;
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    void* args[] = {(void*)&q};
    if (q.steps == 0) return cudaLaunchKernel((const void*)k, dim3(n_items), dim3(nt), args, smem, stream);   // no exchange
    return cudaLaunchCooperativeKernel((const void*)k, dim3(n_items), dim3(nt), args, smem, stream);
}

template <int PREC>
cudaError_t launch_prec(pflbm_t* h, const ResidentPlan& pl, int steps, int* need)
{
    ResArgs<PREC, false> q;
    write_step_args(h, 0, &q.a);
    q.cut = pl.cut;
    q.ll = (Word*)h->res_words;
    q.ll_half = pl.words / 2;
    q.spill = (uint32_t*)h->res_spill;
    q.room = pl.room;
    q.need = need;
    q.tag = h->res_tag;
    q.steps = steps;
    int n = 0;
    for (int i = 0; i < pl.cut.px * pl.cut.py; ++i)
        if (pl.cut.active[i >> 5] >> (i & 31) & 1u) q.item[n++] = (uint16_t)i;
    const bool vv = q.a.varvisc != 0;
    if (pl.cls == 0)
        return vv ? launch_k<PREC, 1, 0, false>(q, n, pl.nt, h->stream) : launch_k<PREC, 0, 0, false>(q, n, pl.nt, h->stream);
    if (pl.cls == 1)
        return vv ? launch_k<PREC, 1, 1, false>(q, n, pl.nt, h->stream) : launch_k<PREC, 0, 1, false>(q, n, pl.nt, h->stream);
    if constexpr (PREC != PFLBM_FP64)
        return vv ? launch_k<PREC, 1, 2, false>(q, n, pl.nt, h->stream) : launch_k<PREC, 0, 2, false>(q, n, pl.nt, h->stream);
    return cudaErrorInvalidValue;
}

template <int PREC>
cudaError_t launch_batch_prec(const ResidentWave& w, int cls, int nt, cudaStream_t stream)
{
    ResArgs<PREC, true> q;
    q.a = (const StepArgs<PREC>*)w.args;
    q.cut = w.cuts;
    q.item = w.items;
    q.ll = (Word*)w.words;
    q.ll_half = w.half;
    q.spill = w.spill;
    q.tag = w.tag;
    q.steps = w.steps;
    if constexpr (PREC != PFLBM_FP64)
        if (cls == 2) return launch_k<PREC, 2, 2, true>(q, w.n_items, nt, stream);
    return cudaErrorInvalidValue;
}

// Which patches of a cut hold a zeta = 1 node: a fluid node in them or next to them
// (from the 8 x 8 blocks with fluid, so it may say yes too often, never no).
// The block columns of the patches' columns (and where those reach over the
// periodic seam) and the block rows of their rows are worked out once per px and py:
// a plan looks at tens of thousands of patches.
struct PatchTest {
    struct Span { int lo, hi, seam; };     // blocks lo..hi-1; and block column `seam` (or -1)
    const SolidMap& m;
    int nx, unit, px = 0, py = 0;
    std::vector<Span> cols, rows;
    PatchTest(const SolidMap& map, int nx_, int unit_) : m(map), nx(nx_), unit(unit_) {}
    Rect rect(const ResidentCut& c, int i) const { return unit == 1 ? patch_rect<1>(c, i, nx) : patch_rect<2>(c, i, nx); }
    void columns(const ResidentCut& c)
    {
        px = c.px;
        cols.resize(px);
        for (int i = 0; i < px; ++i) {
            const Rect r = rect(c, i);
            const int x0 = r.x0 - 1, x1 = r.x0 + r.w;
            cols[i] = {(x0 < 0 ? 0 : x0) / 8, (x1 >= nx ? nx - 1 : x1) / 8 + 1, x0 < 0 ? (nx - 1) / 8 : x1 >= nx ? 0 : -1};
            // a single column of patches reaches over the seam at both sides, and
            // holds both columns itself
        }
    }
    void lines(const ResidentCut& c)
    {
        py = c.py;
        rows.resize(py);
        for (int j = 0; j < py; ++j) {
            const Rect r = rect(c, j * c.px);
            rows[j] = {(r.y0 - 1) / 8, (r.y0 + r.h) / 8 + 1, -1};   // rows 0 and ny - 1 exist beside every patch
        }
    }
    bool active(int i, int j) const
    {
        const Span &x = cols[i], &y = rows[j];
        const int* lo = m.sum.data() + (size_t)y.lo * (m.bw + 1);
        const int* hi = m.sum.data() + (size_t)y.hi * (m.bw + 1);
        if (hi[x.hi] - lo[x.hi] - hi[x.lo] + lo[x.lo] > 0) return true;
        return x.seam >= 0 && hi[x.seam + 1] - lo[x.seam + 1] - hi[x.seam] + lo[x.seam] > 0;
    }
    // active patches, counted row by row of patches until they are more than cap
    int count(int cap, int* tests) const
    {
        if (m.sum.back() == m.bw * m.bh) return px * py;
        int n = 0;
        for (int j = 0; j < py && n <= cap; ++j, *tests += px)
            for (int i = 0; i < px; ++i) n += active(i, j);
        return n;
    }
    // the set of active patches, how many lie below each of its words; their number
    int fill(ResidentCut* c) const
    {
        int n = 0;
        for (int i = 0; i < px * py; ++i) {
            if (i % 32 == 0) c->before[i >> 5] = (uint16_t)n;
            if (!active(i % px, i / px)) continue;
            c->active[i >> 5] |= 1u << (i & 31);
            ++n;
        }
        return n;
    }
};

}  // namespace

void SolidMap::build(const uint8_t* solid, int nx, int ny)
{
    bw = (nx + 7) / 8;
    bh = (ny + 7) / 8;
    sum.assign((size_t)(bw + 1) * (bh + 1), 0);
    for (int y = 0; y < ny; ++y) {
        const uint8_t* row = solid + (size_t)y * nx;
        int* out = sum.data() + (size_t)(y / 8 + 1) * (bw + 1) + 1;
        for (int b = 0; b < nx / 8; ++b) {       // a zero byte among eight
            uint64_t v;
            memcpy(&v, row + 8 * b, 8);
            out[b] |= ((v - 0x0101010101010101ull) & ~v & 0x8080808080808080ull) != 0;
        }
        for (int x = nx / 8 * 8; x < nx; ++x) out[x / 8] |= row[x] == 0;
    }
    // kinds of 64 x 8 tiles; solid nodes of each row within two columns of a tile first
    const int tx = (nx + 63) / 64, ty = (ny + 7) / 8;
    std::vector<uint8_t> near((size_t)ny * tx, 0);
    for (int y = 0; y < ny; ++y)
        for (int i = 0; i < tx; ++i) {
            const uint8_t* row = solid + (size_t)y * nx;
            const int x0 = 64 * i, x1 = x0 + 64 < nx ? x0 + 64 : nx;
            uint64_t v = 0;
            int x = x0;
            for (uint64_t w; x + 8 <= x1; x += 8, v |= w) memcpy(&w, row + x, 8);
            for (; x < x1; ++x) v |= row[x];
            for (int d = 1; d <= 2; ++d) v |= row[(x0 - d + nx) % nx] | row[(x1 + d - 1) % nx];
            near[(size_t)y * tx + i] = v != 0;
        }
    for (int j = 0; j < ty; ++j)
        for (int i = 0; i < tx; ++i) {
            const int* f = sum.data() + (size_t)(j + 1) * (bw + 1) + 1;   // blocks, not summed yet
            bool fluid = false, clear = j > 0 && 8 * j + 10 <= ny;
            for (int b = 8 * i; b < 8 * i + 8 && b < bw; ++b) fluid = fluid || f[b];
            for (int y = 8 * j - 2; clear && y < 8 * j + 10; ++y) clear = !near[(size_t)y * tx + i];
            ++tiles[!fluid ? kTileSolid : clear ? kTilePlain : kTileMixed];
        }
    for (int y = 1; y <= bh; ++y)
        for (int x = 1; x <= bw; ++x)
            sum[(size_t)y * (bw + 1) + x] += sum[(size_t)(y - 1) * (bw + 1) + x] + sum[(size_t)y * (bw + 1) + x - 1] -
                                             sum[(size_t)(y - 1) * (bw + 1) + x - 1];
}

constexpr int kPlanTests = 45000;

// Cycles of a step that depend on the largest patch: its collision and pulls, and
// its border. Those per node and per border node are measured (FP32 and 16-bit:
// about 2.4 and 4.3; FP64: the FP64 pipe takes 19 cycles a warp instruction).
// Rows of 16 or 32 lanes are 6 to 12 % faster than others (a warp then reads
// whole rows: fewer bank conflicts).
double step_cycles(int precision, int w, int h)
{
    const int unit = precision == PFLBM_FP64 ? 1 : 2, lw = w / unit, lanes = lw * h;
    return ((precision == PFLBM_FP64 ? 100.0 : 2.4) * ((lanes + 31) / 32 * 32 * unit) + 4.3 * 2 * (w + h)) *
           (lw == 16 ? 0.88 : lw == 32 ? 0.94 : 1.0);
}

// The cut with the smallest estimated step.
bool plan_resident(int nx, int ny, int precision, const SolidMap& map, int max_ctas, int only_class, ResidentPlan* out)
{
    const int unit = precision == PFLBM_FP64 ? 1 : 2, units = (nx + unit - 1) / unit, rows = ny - 2;
    const int cap = max_ctas < kMaxResident ? max_ctas : kMaxResident;
    if (map.sum.empty() || map.sum.back() == 0) return false;
    const double fluid = map.sum.back() / ((double)map.bw * map.bh);
    double best = 1e300;
    bool found = false;
    // columns of patches from the one that makes them square outwards, so that
    // most of the others are dropped by their cost alone
    const int ideal = (int)(sqrt((double)cap / fluid * nx / ny) + 0.5), most = units < kMaxPatches ? units : kMaxPatches;
    int tests = 0;   // patches looked at; the search ends after about a tenth of a millisecond of it
    PatchTest test(map, nx, unit);
    const long long least = 64LL * map.sum.back() - 8LL * (nx + 8) - 8LL * (ny + 8) - 2LL * nx;   // nodes in blocks with fluid, at least
    for (int turn = 0; turn <= 2 * (ideal + most) && tests < kPlanTests; ++turn) {
        const int px = ideal + (turn & 1 ? -(turn + 1) / 2 : turn / 2);
        if (px < 1 || px > most) continue;
        const int w2 = (units + px - 1) / px * unit, lw = w2 / unit;
        if (px > 1 && lw < 4) continue;
        ResidentCut cut{};
        cut.px = px;
        cut.py = 1;
        cut.units = units;
        cut.rows = rows;
        cut.w = w2;
        bool columns = false;
        for (int k = 0; k < classes(precision); ++k) {
            if (only_class >= 0 && k != only_class) continue;
            const Class c = class_of(precision, k);
            if (w2 > c.wm) continue;
            // rows of patches, from more than can be active down
            int py = (int)(cap / (px * fluid)) + 2;
            if (py > rows) py = rows;
            if (py > kMaxPatches / px) py = kMaxPatches / px;
            for (; py >= 1; --py) {
                const int h = (rows + py - 1) / py, lanes = lw * h;
                if (h > c.hm || lanes > c.p * c.nt) break;
                const double cost = step_cycles(precision, w2, h);
                if (cost >= best) break;      // fewer rows of patches only cost more
                // every node of a block with fluid lies in an active patch
                if (least > (long long)cap * w2 * h) continue;
                cut.py = py;
                cut.h = h;
                if (!columns) test.columns(cut);
                columns = true;
                test.lines(cut);
                int n = test.count(cap, &tests);
                if (n > cap) continue;
                if (n == 0) break;
                ResidentCut full = cut;
                n = test.fill(&full);
                best = cost;
                found = true;
                out->cut = full;
                out->cls = k;
                out->n_active = n;
                const int per = ((lanes + c.p - 1) / c.p + 31) / 32 * 32;
                // the exchange and the ring want threads too
                out->nt = per < 256 ? 256 : per;
                out->words = 2ull * n * patch_words<false>(w2, h) * (precision == PFLBM_FP64 ? 2 : 1);
                out->room = {0, 0};
                out->bytes = out->words * sizeof(Word);
                break;
            }
        }
    }
    return found;
}

size_t resident_word_bytes() { return sizeof(Word); }
int resident_batch_class(int precision) { return precision == PFLBM_FP64 ? -1 : 2; }
bool cut_resident(int nx, int ny, int precision, const SolidMap& map, int cls, double split, ResidentCut* cut, int* n_active,
                  unsigned long long* half_words)
{
    if (map.sum.empty() || precision == PFLBM_FP64) return false;
    const Class c = class_of(precision, cls);
    const int units = (nx + 1) / 2, rows = ny - 2;
    *cut = ResidentCut{};
    cut->px = (units + c.wm / 2 - 1) / (c.wm / 2);
    const int least = (rows + c.hm - 1) / c.hm, most = rows / 8 > least ? rows / 8 : least;
    cut->py = (int)(least * split) < most ? (int)(least * split) : most;
    if (cut->py < least) cut->py = least;
    if ((long long)cut->px * cut->py > kMaxPatches) return false;
    cut->units = units;
    cut->rows = rows;
    cut->w = (units + cut->px - 1) / cut->px * 2;
    cut->h = (rows + cut->py - 1) / cut->py;
    PatchTest test(map, nx, 2);
    test.columns(*cut);
    test.lines(*cut);
    const int n = test.fill(cut);
    *n_active = n;
    *half_words = (unsigned long long)n * patch_words<true>(cut->w, cut->h);
    return true;
}
// (the layouts of the two 16-bit formats are the same)
ResidentSpill resident_spill(int precision, int cls)
{
    if (precision == PFLBM_FP64) return cls == 0 ? spill_k<PFLBM_FP64, 0>() : spill_k<PFLBM_FP64, 1>();
    if (precision == PFLBM_FP32)
        return cls == 0 ? spill_k<PFLBM_FP32, 0>() : cls == 1 ? spill_k<PFLBM_FP32, 1>() : spill_k<PFLBM_FP32, 2>();
    return cls == 0 ? spill_k<PFLBM_BF16, 0>() : cls == 1 ? spill_k<PFLBM_BF16, 1>() : spill_k<PFLBM_BF16, 2>();
}

// The overflow that a handle's footprint allows for: 32-bit words per patch, a third
// of its exchange words' memory. Dense obstacles need it: 5 x 5 solid blocks every 8
// nodes take about 900 of a 64 x 32 patch's 5760, single fluid nodes every 4 nodes,
// which have the most links a mask can have, about 4600 of a 52 x 34 patch's 5160.
static int spill_allowed(int w, int h) { return 60 * (w + h); }

bool add_spill(ResidentPlan* pl, const int need[2])
{
    pl->room = {need[0] > 0 ? need[0] : 0, need[1] > 0 ? need[1] : 0};
    if (pl->room.words() > spill_allowed(pl->cut.w, pl->cut.h)) return false;
    pl->spill_bytes = (size_t)pl->n_active * pl->room.words() * 4;
    return true;
}

// The largest over all cuts that plan_resident may come to, whatever the mask.
size_t resident_bytes_at_most(int nx, int ny, int precision)
{
    const int unit = precision == PFLBM_FP64 ? 1 : 2, units = (nx + unit - 1) / unit, rows = ny - 2;
    const Class big = class_of(precision, classes(precision) - 1);
    size_t most = 0;
    for (int px = 1; px <= units && px <= kMaxPatches; ++px) {
        const int w2 = (units + px - 1) / px * unit;
        if (w2 > big.wm || (px > 1 && w2 / unit < 4)) continue;
        for (int py = 1; py <= rows && py <= kMaxPatches / px; ++py) {
            const int h = (rows + py - 1) / py, n = px * py < kMaxResident ? px * py : kMaxResident;
            if (h > big.hm) continue;
            const size_t bytes = n * (2 * patch_words<false>(w2, h) * (precision == PFLBM_FP64 ? 2 : 1) * sizeof(Word) +
                                      spill_allowed(w2, h) * sizeof(uint32_t));
            if (bytes > most) most = bytes;
        }
    }
    return most;
}

cudaError_t launch_resident(pflbm_t* h, const ResidentPlan& pl, int steps, int* need)
{
    cudaError_t e;
    switch (h->precision) {
        case PFLBM_FP64: e = launch_prec<PFLBM_FP64>(h, pl, steps, need); break;
        case PFLBM_FP32: e = launch_prec<PFLBM_FP32>(h, pl, steps, need); break;
        case PFLBM_BF16: e = launch_prec<PFLBM_BF16>(h, pl, steps, need); break;
        default: e = launch_prec<PFLBM_FP16>(h, pl, steps, need); break;
    }
    if (e == cudaSuccess) {
        h->cur ^= steps & 1;
        h->res_tag += (unsigned)steps;
    }
    return e;
}

cudaError_t launch_resident_wave(int precision, const ResidentWave& w, int cls, cudaStream_t stream)
{
    const int nt = class_of(precision, cls).nt;
    switch (precision) {
        case PFLBM_FP32: return launch_batch_prec<PFLBM_FP32>(w, cls, nt, stream);
        case PFLBM_BF16: return launch_batch_prec<PFLBM_BF16>(w, cls, nt, stream);
        case PFLBM_FP16: return launch_batch_prec<PFLBM_FP16>(w, cls, nt, stream);
        default: return cudaErrorInvalidValue;
    }
}

#ifdef PFLBM_BOUNDS
unsigned bounds_violations_resident()
{
    unsigned v = 0;
    cudaMemcpyFromSymbol(&v, g_bounds_viol, sizeof(v));
    return v;
}
#else
unsigned bounds_violations_resident() { return 0; }
#endif

}  // namespace pfk
