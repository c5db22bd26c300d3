// balls.cu -- per-graph tables of bounded distances, built once when a graph
// (or its commit region) is set up and read by every decode.
//
// Ball table: for every detector v the detectors within a radius of v with
// their exact distances, in one list per detector: higher detectors within
// b_1, lower ones within b_1 (Algorithm 1's level-1 neighbourhood), then those
// beyond b_1 up to the table radius.  A decode finds the events near an event
// by testing a list against the syndrome row instead of searching the graph.
//
// Six largest weights of radius hold 279 entries per detector on average at
// d = 21 (11 MB), four, at d = 51, 119 (64 MB).  A list starts on its own
// 128-byte line with the entries level 1 reads (12 on average, one line).
// Building takes one bounded search per detector, a warp each, in shared memory;
// it runs twice, once for the sizes (a d = 5 graph is created in 0.22 instead of
// 0.15 ms, d = 25 in 2.9 instead of 2.4, d = 51 in 19.2 instead of 20.6, its
// distance runs being faster).
//
// Seam distances: for every detector a lower bound on its distance to the
// nearest detector on the other side of the commit region's border (sliding
// windows): a path shorter than that stays on one side.

#include <climits>

#include "qec_internal.h"

namespace qec {

namespace {

constexpr unsigned FULL = 0xffffffffu;
constexpr int CAP = 1024;    // entries of one ball; a larger one is stored to b_1 only, or not at all
constexpr int HS = 2048;     // hash slots per warp, at most half full (plus one entry per lane)
constexpr int WPB = 4;       // warps per block, one ball at a time each
constexpr int ALIGN = 16;    // lists start on 128-byte lines

struct Ball {
    int key[HS], dist[HS];               // vertex (-1: empty), distance so far
    unsigned queued[HS / 32];            // slot waits in the next round's work list
    unsigned short list[CAP], wl[2][CAP];
    int count, nwl[2];
};

// Ball of radius R around v by label-correcting relaxation in shared memory
// (one warp).  Returns the number of entries (v itself included), -1 if more
// than CAP.  Rounds are bounded by the ball's size, since every round with
// work lowers a distance that a path with one more edge explains.
__device__ int grow(const DGraph &g, Ball &B, int v, int R, int lane) {
    for (int i = lane; i < HS; i += 32) { B.key[i] = -1; B.dist[i] = INT_MAX; }
    for (int i = lane; i < HS / 32; i += 32) B.queued[i] = 0;
    __syncwarp();
    auto home = [](int x) { return ((unsigned)x * 2654435761u) >> 21; };   // HS = 2^11
    static_assert(HS == 2048, "home slot");
    if (lane == 0) {
        const unsigned h = home(v);
        B.key[h] = v;
        B.dist[h] = 0;
        B.list[0] = (unsigned short)h;
        B.wl[0][0] = (unsigned short)h;
        B.count = 1;
        B.nwl[0] = 1;
    }
    __syncwarp();
    for (int it = 0; it <= CAP; it++) {
        const int cur = it & 1, n = B.nwl[cur];
        __syncwarp();
        if (lane == 0) B.nwl[cur ^ 1] = 0;
        __syncwarp();
        for (int i = lane; i < n; i += 32) {
            const unsigned h = B.wl[cur][i];
            atomicAnd(&B.queued[h >> 5], ~(1u << (h & 31)));
            const int x = B.key[h], dx = *(volatile int *)&B.dist[h];
            const int r1 = g.row[x + 1];
            for (int j = g.row[x]; j < r1; j++) {
                const Slot sl = g.slot[j];
                const int nd = dx + sl.w;
                if (sl.code < 0 || nd > R) continue;
                unsigned p = home(sl.code);
                for (int probe = 0; probe < HS; probe++, p = (p + 1) & (HS - 1)) {
                    int k = *(volatile int *)&B.key[p];
                    if (k == -1) {
                        if (*(volatile int *)&B.count >= CAP) { atomicAdd(&B.count, 1); break; }
                        k = atomicCAS(&B.key[p], -1, sl.code);
                        if (k == -1) {
                            const int c = atomicAdd(&B.count, 1);
                            if (c < CAP) B.list[c] = (unsigned short)p;
                            k = sl.code;
                        }
                    }
                    if (k != sl.code) continue;
                    if (nd < atomicMin(&B.dist[p], nd)) {
                        const unsigned bit = 1u << (p & 31);
                        if (!(atomicOr(&B.queued[p >> 5], bit) & bit)) {
                            const int w = atomicAdd(&B.nwl[cur ^ 1], 1);
                            if (w < CAP) B.wl[cur ^ 1][w] = (unsigned short)p;
                        }
                    }
                    break;
                }
            }
        }
        __syncwarp();
        const int c = B.count, nn = B.nwl[cur ^ 1];
        __syncwarp();
        if (c > CAP || nn > CAP) return -1;
        if (nn == 0) return c;
    }
    return -1;
}

// One warp per detector.  out == NULL: add every list's room to *cursor, or with
// `whole`, once some ball of radius R is too large, only mark cursor[1]; else
// write the lists and their headers, each list where *cursor stands.
__global__ void __launch_bounds__(32 * WPB) ball_kernel(DGraph g, int R, bool whole, unsigned long long *cursor, int4 *hdr,
                                                        int2 *out) {
    extern __shared__ __align__(16) char dyn[];
    Ball *const ball = reinterpret_cast<Ball *>(dyn);
    const int lane = threadIdx.x & 31;
    Ball &B = ball[threadIdx.x >> 5];
    const int nw = gridDim.x * WPB;
    unsigned long long room = 0;
    for (int v = blockIdx.x * WPB + (threadIdx.x >> 5); v < g.n; v += nw) {
        bool far = true;
        int n = R > g.b1 ? grow(g, B, v, R, lane) : -1;
        if (n < 0 && whole && R > g.b1) {
            if (lane == 0) *(volatile unsigned long long *)(cursor + 1) = 1;
            return;
        }
        if (whole && *(volatile unsigned long long *)(cursor + 1)) return;
        if (n < 0) {   // too many entries: b_1 only
            far = R <= g.b1;
            __syncwarp();
            n = grow(g, B, v, g.b1, lane);
        }
        if (!out) {
            if (n > 0) room += (unsigned long long)((n - 1 + ALIGN - 1) / ALIGN * ALIGN);
            __syncwarp();
            continue;
        }
        int4 h = make_int4(0, 0, -1, -1);
        if (n > 0) {
            unsigned long long beg = 0;
            if (lane == 0) beg = atomicAdd(cursor, (unsigned long long)((n - 1 + ALIGN - 1) / ALIGN * ALIGN));
            beg = __shfl_sync(FULL, beg, 0);
            // three sweeps, one per section of the list
            int at = 0, up = 0, near = 0;
            for (int part = 0; part < 3; part++) {
                for (int b = 0; b < n; b += 32) {
                    const int i = b + lane;
                    int u = v, d = 0;
                    if (i < n) { u = B.key[B.list[i]]; d = B.dist[B.list[i]]; }
                    const int mine = u == v ? -1 : (d > g.b1 ? 2 : (u > v ? 0 : 1));
                    const unsigned m = __ballot_sync(FULL, mine == part);
                    if (mine == part) out[beg + at + __popc(m & ((1u << lane) - 1u))] = make_int2(u, d);
                    at += __popc(m);
                }
                if (part == 0) up = at;
                if (part == 1) near = at;
            }
            h = make_int4((int)(unsigned)beg, up, near, far ? at - near : -1);
        }
        if (lane == 0) hdr[v] = h;
        __syncwarp();
    }
    if (!out && lane == 0 && room) atomicAdd(cursor, room);
}

__global__ void seam_kernel(DGraph g, const unsigned *commit, int *seam) {
    const int lane = threadIdx.x & 31;
    const int nw = gridDim.x * (blockDim.x >> 5);
    for (int v = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); v < g.n; v += nw) {
        const int4 h = g.bhdr[v];
        const unsigned side = (commit[v >> 5] >> (v & 31)) & 1u;
        // nothing on the other side within the list: beyond the list's radius
        int best = h.w >= 0 ? g.brad + 1 : (h.z >= 0 ? g.b1 + 1 : 0);
        const int n = h.z + max(h.w, 0);
        for (int k = lane; k < n; k += 32) {
            const int2 e = g.ball[(unsigned)h.x + k];
            if (((commit[e.x >> 5] >> (e.x & 31)) & 1u) != side) best = min(best, e.y);
        }
        best = __reduce_min_sync(FULL, best);
        if (lane == 0) seam[v] = best;
    }
}

int grid_for(int n, int wpb) { return (int)std::min<long long>(((long long)n + wpb - 1) / wpb, 8192); }

}  // namespace

cudaError_t build_ball_table(DGraph &g, bool wide, int4 **hdr, int2 **ball) {
    *hdr = nullptr;
    *ball = nullptr;
    unsigned long long *cursor = nullptr, total[2] = {0, 0};
    cudaError_t e = cudaMalloc(hdr, sizeof(int4) * (size_t)g.n);
    if (e == cudaSuccess) e = cudaMalloc(&cursor, sizeof(total));
    const int smem = (int)sizeof(Ball) * WPB;
    if (e == cudaSuccess) e = cudaFuncSetAttribute(ball_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    // Radius: six largest weights (a region of up to four edges' radius and
    // smaller ones stay within it of each other), for windows of a sliding decode
    // eight (an event at an open end has no boundary near), where every ball fits
    // and the table stays below 128 MB; else four below 512 MB, with single balls
    // that are too large stored to b_1 only; else b_1, at whatever size that takes
    // (128 bytes to 8 KB per detector, at most 16 GB).  Six instead of four: 3,000
    // d = 31 windows 0.52 -> 0.37 ms, 1,024 circuit-level d = 13 shots 0.19 -> 0.12 ms.
    constexpr unsigned long long WIDE_LIMIT = 1ull << 24, FAR_LIMIT = 1ull << 26, LIMIT = (1ull << 31) - 1;   // entries
    const int grid = grid_for(g.n, WPB);
    int R = g.b1;
    for (int k : {8, 6, 4, 0}) {
        if (k == 8 && !wide) continue;
        if (k > 4 && (unsigned long long)g.n * 256 > WIDE_LIMIT) continue;
        R = (int)std::min<long long>(std::max<long long>(g.b1, (long long)k * g.wmax + 4), INT_MAX / 4);
        if (e == cudaSuccess) e = cudaMemset(cursor, 0, sizeof(total));
        if (e != cudaSuccess) break;
        ball_kernel<<<grid, 32 * WPB, smem>>>(g, R, k > 4, cursor, *hdr, nullptr);
        e = cudaMemcpy(total, cursor, sizeof(total), cudaMemcpyDeviceToHost);
        if (e != cudaSuccess || (!total[1] && total[0] <= (k > 4 ? WIDE_LIMIT : FAR_LIMIT))) break;
    }
    if (e == cudaSuccess && total[0] <= LIMIT) {
        e = cudaMalloc(ball, sizeof(int2) * (size_t)(total[0] + 1));
        if (e != cudaSuccess) { (void)cudaGetLastError(); *ball = nullptr; e = cudaSuccess; }
    }
    if (e == cudaSuccess && *ball) {
        e = cudaMemset(cursor, 0, sizeof(total));
        if (e == cudaSuccess) ball_kernel<<<grid, 32 * WPB, smem>>>(g, R, false, cursor, *hdr, *ball);
    } else if (e == cudaSuccess) {
        e = cudaMemset(*hdr, 0xff, sizeof(int4) * (size_t)g.n);   // no room: no list is complete
    }
    if (e == cudaSuccess) e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaStreamSynchronize(nullptr);
    if (cursor) cudaFree(cursor);
    g.bhdr = *hdr;
    g.ball = *ball;
    g.brad = R;
    return e;
}

cudaError_t build_seam(const DGraph &g, const unsigned *commit, int *seam) {
    seam_kernel<<<grid_for(g.n, 8), 256>>>(g, commit, seam);
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? cudaStreamSynchronize(nullptr) : e;
}

}  // namespace qec
