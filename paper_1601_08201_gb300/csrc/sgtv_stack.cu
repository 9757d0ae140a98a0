// sgtv_stack.cu -- set-up of the stacked row form (FP32 vectors; read by
// k_rows_stack in sgtv_kernels.cuh).
//
// A tile is tr consecutive rows, and one warp's work. Its distinct columns
// (at most 32 * kStkMaxWords) are dealt to the warp: column k of the tile's
// ascending list belongs to word k / 32 and, inside the word, to one lane, so
// a lane owns one column per word for the whole tile and keeps that column's
// f and its sum of a_ij * ratio_i in registers. What is stored per row is a
// bit per (lane, word). The values stand in 32 stacks, a [levels][32] array:
// for each pair of rows every lane is given one stack, and its values of the
// first row, then of the second, word after word, lie on consecutive levels of
// it. Reading them takes a pointer per lane that steps one level per set bit:
// no index, and never a bank conflict, since no two lanes share a stack.
//
// A tile is as long as its tallest stack, and the levels that a pair of rows
// touches have to be in shared memory together, so the stacks are kept level:
// the columns of a word are handed to its lanes heaviest column to the lane
// with the fewest values so far, and in each pair the lane with the most
// values gets the lowest stack. (Which columns a word holds is left alone: 32
// neighbours of the list, so that the gathers of f and the adds into e stay
// in runs.)
//
// The kernel streams the stacks through a ring of shared memory, one copy per
// pair of rows: the levels above the last pair's highest, up to this pair's.
// The copies run kStkAhead pairs ahead, so the ring is as high as the largest
// step from the lowest stack after a pair to the highest one kStkAhead pairs
// on.
//
// One record per lane and pair: the first row's bits, the second row's bits,
// the first value's place in the ring (level * 32 + stack); 32 bits of
// 10 + 10 + 12 for up to 10 words, else 64 of 24 + 24 + 16.
#include <limits.h>

#include "sgtv_internal.h"

namespace sgtv {

namespace {

constexpr int kT = 256;
constexpr int kMaxCols = 32 * kStkMaxWords;
constexpr int kMaxBitWords = 44 * 1024;  // 176 KB bitmap; a wider index range is swept in chunks

struct Span {
    int64_t p0, p1;
    int32_t mn, mx;
};

// The tile's nonzeros and index range (rows are ascending inside).
__device__ Span tile_span(const int64_t *__restrict__ ptr, const int32_t *__restrict__ idx, int64_t I, int tr,
                          int64_t t)
{
    __shared__ int32_t smn, smx;
    const int64_t r0 = t * tr, r1 = r0 + tr < I ? r0 + tr : I;
    __syncthreads();
    if (threadIdx.x == 0) {
        smn = INT_MAX;
        smx = -1;
    }
    __syncthreads();
    for (int64_t r = r0 + threadIdx.x; r < r1; r += blockDim.x) {
        const int64_t a = ptr[r], b = ptr[r + 1];
        if (b > a) {
            atomicMin(&smn, idx[a]);
            atomicMax(&smx, idx[b - 1]);
        }
    }
    __syncthreads();
    return Span{ptr[r0], ptr[r1], smn, smx};
}

__device__ __forceinline__ int chunk_words(int64_t lo, int32_t mx, int max_words)
{
    if (lo > mx) return 0;
    const int64_t w = (int64_t(mx) - lo) / 32 + 1;
    return int(w < max_words ? w : max_words);
}

__device__ void chunk_bitmap(const int32_t *__restrict__ idx, const Span &s, int64_t lo, int words, uint32_t *bits)
{
    for (int w = threadIdx.x; w < words; w += blockDim.x) bits[w] = 0u;
    __syncthreads();
    const int64_t hi = lo + int64_t(words) * 32;
    for (int64_t p = s.p0 + threadIdx.x; p < s.p1; p += blockDim.x) {
        const int64_t v = int64_t(idx[p]);
        if (v >= lo && v < hi) atomicOr(&bits[(v - lo) >> 5], 1u << ((v - lo) & 31));
    }
    __syncthreads();
}

// out[0] = largest number of distinct columns of a tile.
__global__ void __launch_bounds__(kT)
k_stk_count(int64_t I, int tr, const int64_t *__restrict__ ptr, const int32_t *__restrict__ idx, int max_words,
            int *__restrict__ out)
{
    extern __shared__ uint32_t bits[];
    __shared__ int total;
    const Span s = tile_span(ptr, idx, I, tr, blockIdx.x);
    if (threadIdx.x == 0) total = 0;
    __syncthreads();
    for (int64_t lo = s.mn; s.mx >= 0; lo += int64_t(max_words) * 32) {
        const int words = chunk_words(lo, s.mx, max_words);
        if (words == 0) break;
        chunk_bitmap(idx, s, lo, words, bits);
        int c = 0;
        for (int w = threadIdx.x; w < words; w += blockDim.x) c += __popc(bits[w]);
        atomicAdd(&total, c);
        __syncthreads();
    }
    if (threadIdx.x == 0) atomicMax(out, total);
}

// One lane's record of a pair of rows.
template <typename M> struct Rec;
template <> struct Rec<uint32_t> {
    __device__ static uint32_t make(uint32_t a, uint32_t b, uint32_t at) { return a | (b << 10) | (at << 20); }
    __device__ static uint32_t first(uint32_t v) { return v & 0x3FFu; }
    __device__ static uint32_t second(uint32_t v) { return (v >> 10) & 0x3FFu; }
    __device__ static uint32_t place(uint32_t v) { return v >> 20; }
};
template <> struct Rec<uint64_t> {
    __device__ static uint64_t make(uint32_t a, uint32_t b, uint32_t at)
    {
        return uint64_t(a) | (uint64_t(b) << 24) | (uint64_t(at) << 48);
    }
    __device__ static uint32_t first(uint64_t v) { return uint32_t(v) & 0xFFFFFFu; }
    __device__ static uint32_t second(uint64_t v) { return uint32_t(v >> 24) & 0xFFFFFFu; }
    __device__ static uint32_t place(uint64_t v) { return uint32_t(v >> 48); }
};

// Per tile: the column list, the lanes, the records without their places
// (absolute, in `start`: level * 32 + stack), each pair's levels (first | count
// << 16) and the stack height; rank[p] = the nonzero's place in the column
// list. stats[0] = levels the ring needs.
template <typename M>
__global__ void __launch_bounds__(kT)
k_stk_build(int64_t I, int tr, int words_per_tile, const int64_t *__restrict__ ptr, const int32_t *__restrict__ idx,
            int max_words, int32_t *__restrict__ uidx, uint8_t *__restrict__ lanes, uint16_t *__restrict__ rank,
            M *__restrict__ rec, uint16_t *__restrict__ start, uint32_t *__restrict__ ctl,
            int32_t *__restrict__ height, int *__restrict__ stats)
{
    extern __shared__ uint32_t bits[];  // bitmap, then one prefix per 32 bitmap words
    int32_t *pre = reinterpret_cast<int32_t *>(bits + max_words);
    __shared__ int32_t ucol[kMaxCols], cnt[kMaxCols];
    __shared__ uint8_t lane_of[kMaxCols];
    __shared__ uint32_t ms[kStkMaxRows][32];
    __shared__ int32_t load[32], inv[32], top[kStkMaxRows / 2], low[kStkMaxRows / 2];
    __shared__ int base, run;
    const int64_t t = blockIdx.x;
    const int64_t r0 = t * tr;
    const int nr = int(I - r0 < tr ? I - r0 : tr);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const Span s = tile_span(ptr, idx, I, tr, t);
    for (int k = threadIdx.x; k < kMaxCols; k += blockDim.x) {
        ucol[k] = -1;
        cnt[k] = 0;
    }
    for (int k = threadIdx.x; k < kStkMaxRows * 32; k += blockDim.x) ms[k >> 5][k & 31] = 0u;
    if (threadIdx.x == 0) base = 0;
    __syncthreads();
    for (int64_t lo = s.mn; s.mx >= 0; lo += int64_t(max_words) * 32) {
        const int words = chunk_words(lo, s.mx, max_words);
        if (words == 0) break;
        chunk_bitmap(idx, s, lo, words, bits);
        const int ng = (words + 31) / 32;
        for (int g = threadIdx.x; g < ng; g += blockDim.x) {
            int c = 0;
            for (int w = g * 32; w < words && w < g * 32 + 32; w++) c += __popc(bits[w]);
            pre[g] = c;
        }
        __syncthreads();
        if (warp == 0) {  // exclusive scan of the groups, 32 at a time
            int r = base;
            for (int g0 = 0; g0 < ng; g0 += 32) {
                const int c = g0 + lane < ng ? pre[g0 + lane] : 0;
                int x = c;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int y = __shfl_up_sync(0xffffffffu, x, o);
                    if (lane >= o) x += y;
                }
                if (g0 + lane < ng) pre[g0 + lane] = r + x - c;
                r += __shfl_sync(0xffffffffu, x, 31);
            }
            if (lane == 0) run = r;
        }
        __syncthreads();
        const int64_t hi = lo + int64_t(words) * 32;
        for (int64_t p = s.p0 + threadIdx.x; p < s.p1; p += blockDim.x) {
            const int64_t v = int64_t(idx[p]);
            if (v < lo || v >= hi) continue;
            const int b = int(v - lo), w = b >> 5;
            int k = pre[w >> 5];
            for (int w2 = w & ~31; w2 < w; w2++) k += __popc(bits[w2]);
            k += __popc(bits[w] & ((1u << (b & 31)) - 1u));
            rank[p] = uint16_t(k);
            ucol[k] = int32_t(v);
            atomicAdd(&cnt[k], 1);
        }
        __syncthreads();
        if (threadIdx.x == 0) base = run;
        __syncthreads();
    }
    if (warp == 0) {
        // word by word: the heaviest column to the lane with the lowest stack
        int mine = 0;
        for (int w = 0; w < words_per_tile; w++) {
            const int c = cnt[32 * w + lane];
            int rc = 0, rl = 0;
            for (int j = 0; j < 32; j++) {
                const int cj = __shfl_sync(0xffffffffu, c, j), lj = __shfl_sync(0xffffffffu, mine, j);
                rc += (cj > c || (cj == c && j < lane)) ? 1 : 0;
                rl += (lj < mine || (lj == mine && j < lane)) ? 1 : 0;
            }
            inv[rl] = lane;
            __syncwarp();
            const int to = inv[rc];
            lane_of[32 * w + lane] = uint8_t(to);
            load[to] = c;
            __syncwarp();
            mine += load[lane];
            __syncwarp();
        }
    }
    __syncthreads();
    for (int k = threadIdx.x; k < 32 * words_per_tile; k += blockDim.x) {
        uidx[t * 32 * words_per_tile + (k & ~31) + lane_of[k]] = ucol[k];
        lanes[t * 32 * words_per_tile + k] = lane_of[k];
    }
    for (int r = warp; r < nr; r += kT / 32)
        for (int64_t p = ptr[r0 + r] + lane; p < ptr[r0 + r + 1]; p += 32) {
            const int k = rank[p];
            atomicOr(&ms[r][lane_of[k]], 1u << (k >> 5));
        }
    __syncthreads();
    if (warp == 0) {
        int mine = 0, last = 0;  // height of stack `lane`, of the highest one
        for (int r = 0; r < nr; r += 2) {
            const uint32_t ma = ms[r][lane], mb = r + 1 < nr ? ms[r + 1][lane] : 0u;
            const int c = __popc(ma) + __popc(mb);
            int rc = 0, rl = 0;
            for (int j = 0; j < 32; j++) {
                const int cj = __shfl_sync(0xffffffffu, c, j), lj = __shfl_sync(0xffffffffu, mine, j);
                rc += (cj > c || (cj == c && j < lane)) ? 1 : 0;
                rl += (lj < mine || (lj == mine && j < lane)) ? 1 : 0;
            }
            inv[rl] = lane;
            load[lane] = mine;
            __syncwarp();
            const int to = inv[rc], at = load[to];
            __syncwarp();
            load[to] = at + c;
            const int64_t k = ((r0 + r) >> 1) * 32 + lane;
            rec[k] = Rec<M>::make(ma, mb, 0u);
            start[k] = uint16_t(at * 32 + to);
            __syncwarp();
            mine = load[lane];
            __syncwarp();
            int hi = mine, lo = mine;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                hi = max(hi, __shfl_xor_sync(0xffffffffu, hi, o));
                lo = min(lo, __shfl_xor_sync(0xffffffffu, lo, o));
            }
            if (lane == 0) {
                ctl[(r0 + r) >> 1] = uint32_t(last) | (uint32_t(hi - last) << 16);
                top[r >> 1] = hi;
                low[r >> 1] = lo;
            }
            last = hi;
        }
        __syncwarp();
        if (lane == 0) {
            const int np = (nr + 1) / 2;
            int ring = top[(kStkAhead < np ? kStkAhead : np) - 1];
            for (int p = 0; p + kStkAhead < np; p++) ring = max(ring, top[p + kStkAhead] - low[p]);
            height[t] = last;
            atomicMax(stats, ring);
        }
    }
}

// The copy of a pair's `n` levels from level `first` on into a ring of `ring`
// levels: to place a = first mod ring, on past the end as far as the repeated
// levels reach, and what is missing then to a second place -- the levels past
// the end to the ring's start, or those among the first kStkMirror again
// behind the end (never both: the ring is higher than n + kStkMirror). Bits: a
// 7, n 6, levels of the first copy 7, of the second 6, 1 if the second goes to
// the ring's start.
__device__ __forceinline__ uint32_t copy_code(int first, int n, int ring)
{
    const int a = first % ring;
    const int n1 = n < ring + kStkMirror - a ? n : ring + kStkMirror - a;
    const bool over = a + n > ring;
    const int n2 = over ? a + n - ring : (a < kStkMirror ? (n < kStkMirror - a ? n : kStkMirror - a) : 0);
    return uint32_t(a) | (uint32_t(n) << 7) | (uint32_t(n1) << 13) | (uint32_t(n2) << 20) | (over ? 1u << 26 : 0u);
}

// The values at their places in the stacks (the array zeroed beforehand), and
// the records and copies of a ring of `ring` levels.
template <typename M, typename VB>
__global__ void __launch_bounds__(kT)
k_stk_fill(int64_t I, int tr, int words_per_tile, int ring, const int64_t *__restrict__ ptr,
           const VB *__restrict__ val, const uint8_t *__restrict__ lanes, const uint16_t *__restrict__ rank,
           const uint16_t *__restrict__ start, M *__restrict__ rec, uint32_t *__restrict__ ctl,
           const int64_t *__restrict__ lvl, VB *__restrict__ out)
{
    __shared__ uint8_t lane_of[kMaxCols];
    const int64_t t = blockIdx.x;
    const int64_t r0 = t * tr;
    const int nr = int(I - r0 < tr ? I - r0 : tr);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int k = threadIdx.x; k < 32 * words_per_tile; k += blockDim.x)
        lane_of[k] = lanes[t * 32 * words_per_tile + k];
    __syncthreads();
    for (int r = warp; r < nr; r += kT / 32) {
        const int64_t pair = ((r0 + r) >> 1) * 32;
        for (int64_t p = ptr[r0 + r] + lane; p < ptr[r0 + r + 1]; p += 32) {
            const int k = rank[p];
            const int l = lane_of[k];
            const M v = rec[pair + l];
            const uint32_t a = Rec<M>::first(v), below = (1u << (k >> 5)) - 1u;
            const int up = (r & 1) ? __popc(a) + __popc(Rec<M>::second(v) & below) : __popc(a & below);
            const int at = start[pair + l];
            out[(lvl[t] + (at >> 5) + up) * 32 + (at & 31)] = val[p];
        }
    }
    __syncthreads();
    for (int64_t k = (r0 >> 1) * 32 + threadIdx.x; k < ((r0 + nr + 1) >> 1) * 32; k += blockDim.x) {
        const M v = rec[k];
        const int at = start[k];
        rec[k] = Rec<M>::make(Rec<M>::first(v), Rec<M>::second(v),
                              uint32_t(((at >> 5) % ring) * 32 + (at & 31)));
    }
    for (int64_t k = (r0 >> 1) + threadIdx.x; k < ((r0 + nr + 1) >> 1); k += blockDim.x)
        ctl[k] = copy_code(int(ctl[k] & 0xFFFFu), int(ctl[k] >> 16), ring);
}

// Reads the stacks as the kernel does and compares each row with the CSR
// form: count, sums of the columns, of the values' bits and of their products
// (integers, modulo 2^64). Also bounds: every level inside the tile and among
// those in the ring, no copy over a level still to be read, every column
// inside the image, no two lanes on one stack. Sets flag bit 64.
template <typename M, typename VB>
__global__ void __launch_bounds__(kT)
k_stk_check(int64_t I, int64_t J, int tr, int words_per_tile, int ring, int64_t ntiles,
            const int64_t *__restrict__ ptr, const int32_t *__restrict__ idx, const VB *__restrict__ val,
            const int32_t *__restrict__ uidx, const M *__restrict__ rec, const uint32_t *__restrict__ ctl,
            const int64_t *__restrict__ lvl, const VB *__restrict__ sval, int *__restrict__ flag)
{
    const int lane = threadIdx.x & 31;
    const int64_t nwarps = (int64_t(gridDim.x) * blockDim.x) >> 5;
    bool bad = ring > kStkMaxRing || ring < 2 * words_per_tile + kStkMirror;
    for (int64_t t = (int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5; t < ntiles; t += nwarps) {
        const int64_t r0 = t * tr;
        const int nr = int(I - r0 < tr ? I - r0 : tr);
        const int h = int(lvl[t + 1] - lvl[t]);
        int level = 0, stack = 0, top = 0, low = 0;  // levels below top have been copied, those below low used up
        for (int r = 0; r < nr; r++) {
            const M v = rec[((r0 + r) >> 1) * 32 + lane];
            if ((r & 1) == 0) {
                const uint32_t k = ctl[(r0 + r) >> 1];
                const int cnt = int((k >> 7) & 63u);
                bad |= k != copy_code(top, cnt, ring);
                top += cnt;
                // before this pair, the copies of kStkAhead - 1 further ones have been issued
                int ahead = top;
                for (int q = 1; q < kStkAhead && r + 2 * q < nr; q++)
                    ahead += int((ctl[((r0 + r) >> 1) + q] >> 7) & 63u);
                bad |= ahead - low > ring || top > h;
                const int at = int(Rec<M>::place(v));
                stack = at & 31;
                level = top - ring + (((at >> 5) - (top - ring)) % ring + ring) % ring;
                const uint32_t same = __match_any_sync(0xffffffffu, stack);  // by every lane, also one out of the ring
                bad |= (at >> 5) >= ring || __popc(same) != 1;
                // a lane without values in the pair may stand at the top of the highest stack
                if ((Rec<M>::first(v) | Rec<M>::second(v)) == 0u && level < low) level = top;
                bad |= level < low;
            }
            unsigned long long n = 0, c = 0, b = 0, x = 0;
            const int64_t a = ptr[r0 + r], e = ptr[r0 + r + 1];
            for (int64_t p = a + lane; p < e; p += 32) {
                n += 1;
                c += (unsigned long long)idx[p];
                b += (unsigned long long)val[p];
                x += (unsigned long long)idx[p] * (unsigned long long)val[p];
            }
            const uint32_t m = (r & 1) ? Rec<M>::second(v) : Rec<M>::first(v);
#pragma unroll 4
            for (int w = 0; w < words_per_tile; w++) {  // several words' loads in flight
                const int at = level + __popc(m & ((1u << w) - 1u));
                const bool in = ((m >> w) & 1u) && at >= 0 && at < top && at < h;
                const int32_t col = uidx[(t * words_per_tile + w) * 32 + lane];
                const unsigned long long y = in ? (unsigned long long)sval[(lvl[t] + at) * 32 + stack] : 0ull;
                if (!((m >> w) & 1u)) continue;
                bad |= !in || col < 0 || col >= J;
                n -= 1;
                c -= (unsigned long long)col;
                b -= y;
                x -= (unsigned long long)col * y;
            }
            level += __popc(m);
            bad |= (m >> words_per_tile) != 0u;
            __syncwarp();
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                n += __shfl_xor_sync(0xffffffffu, n, o);
                c += __shfl_xor_sync(0xffffffffu, c, o);
                b += __shfl_xor_sync(0xffffffffu, b, o);
                x += __shfl_xor_sync(0xffffffffu, x, o);
            }
            bad |= n != 0 || c != 0 || b != 0 || x != 0;
            if ((r & 1) || r + 1 == nr) {
                low = level;
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) low = min(low, __shfl_xor_sync(0xffffffffu, low, o));
            }
        }
    }
    if (__any_sync(0xffffffffu, bad) && lane == 0) atomicOr(flag, 64);
}

// Partial sums by column (two-pass form): how many tiles hold each column,
// where each (tile, word, lane) writes, in ascending tile order per column.
__global__ void k_stk_colcount(int64_t n, const int32_t *__restrict__ uidx, int32_t *__restrict__ cnt)
{
    for (int64_t k = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; k < n; k += int64_t(gridDim.x) * blockDim.x)
        if (uidx[k] >= 0) atomicAdd(cnt + uidx[k], 1);
}

__global__ void k_stk_place(int64_t n, const int32_t *__restrict__ uidx, const int32_t *__restrict__ poff,
                            int32_t *__restrict__ cnt, int32_t *__restrict__ ent)
{
    for (int64_t k = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; k < n; k += int64_t(gridDim.x) * blockDim.x)
        if (uidx[k] >= 0) ent[poff[uidx[k]] + atomicSub(cnt + uidx[k], 1) - 1] = int32_t(k);
}

__global__ void k_stk_order(int64_t J, const int32_t *__restrict__ poff, int32_t *__restrict__ ent,
                            int32_t *__restrict__ ppos)
{
    for (int64_t j = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; j < J; j += int64_t(gridDim.x) * blockDim.x) {
        const int a = poff[j], b = poff[j + 1];
        for (int i = a + 1; i < b; i++) {  // the set-up bounds b - a
            const int v = ent[i];
            int k = i;
            for (; k > a && ent[k - 1] > v; k--) ent[k] = ent[k - 1];
            ent[k] = v;
        }
        for (int i = a; i < b; i++) ppos[ent[i]] = i;
    }
}

int grid_of(int64_t n)
{
    const int64_t b = (n + kT - 1) / kT;
    return int(b < 1 ? 1 : (b < 8192 ? b : 8192));
}

template <typename K>
cudaError_t opt_in(K kernel, size_t smem)
{
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
}

int bitmap_words(int64_t J)
{
    const int64_t w = (J + 31) / 32;
    return int(w < kMaxBitWords ? w : kMaxBitWords);
}

}  // namespace

cudaError_t stk_count(int64_t I, int64_t J, int tr, const int64_t *ptr, const int32_t *idx, int *out, cudaStream_t st)
{
    const int words = bitmap_words(J);
    const size_t smem = size_t(words) * 4;
    cudaError_t e = opt_in(k_stk_count, smem);
    if (e != cudaSuccess) return e;
    k_stk_count<<<unsigned((I + tr - 1) / tr), kT, smem, st>>>(I, tr, ptr, idx, words, out);
    return cudaGetLastError();
}

namespace {

template <typename M>
cudaError_t build_typed(int64_t I, int64_t J, const StackMat &m, const int64_t *ptr, const int32_t *idx,
                        uint8_t *lanes, uint16_t *rank, uint16_t *start, int32_t *height, int *stats, cudaStream_t st)
{
    const int words = bitmap_words(J);
    const size_t smem = size_t(words) * 4 + size_t(words / 32 + 1) * 4;
    cudaError_t e = opt_in(k_stk_build<M>, smem);
    if (e != cudaSuccess) return e;
    k_stk_build<M><<<unsigned(m.ntiles), kT, smem, st>>>(I, m.tr, m.words, ptr, idx, words, m.uidx, lanes, rank,
                                                         static_cast<M *>(m.rec), start, m.ctl, height, stats);
    return cudaGetLastError();
}

template <typename M, typename VB>
void fill_typed(int64_t I, int64_t J, const StackMat &m, const int64_t *ptr, const int32_t *idx, const void *val,
                const uint8_t *lanes, const uint16_t *rank, const uint16_t *start, int *flag, int sm_count,
                cudaStream_t st)
{
    M *rec = static_cast<M *>(m.rec);
    const VB *v = static_cast<const VB *>(val);
    VB *sv = static_cast<VB *>(m.val);
    k_stk_fill<M, VB><<<unsigned(m.ntiles), kT, 0, st>>>(I, m.tr, m.words, m.ring, ptr, v, lanes, rank, start, rec,
                                                         m.ctl, m.lvl, sv);
    const int64_t blocks = (m.ntiles + kT / 32 - 1) / (kT / 32), cap = int64_t(sm_count) * 8;
    k_stk_check<M, VB><<<unsigned(blocks < cap ? blocks : cap), kT, 0, st>>>(
        I, J, m.tr, m.words, m.ring, m.ntiles, ptr, idx, v, m.uidx, rec, m.ctl, m.lvl, sv, flag);
}

}  // namespace

cudaError_t stk_build(int64_t I, int64_t J, const StackMat &m, const int64_t *ptr, const int32_t *idx, uint8_t *lanes,
                      uint16_t *rank, uint16_t *start, int32_t *height, int *stats, cudaStream_t st)
{
    return stk_rec_bytes(m.words) == 4
               ? build_typed<uint32_t>(I, J, m, ptr, idx, lanes, rank, start, height, stats, st)
               : build_typed<uint64_t>(I, J, m, ptr, idx, lanes, rank, start, height, stats, st);
}

cudaError_t stk_fill(int64_t I, int64_t J, const StackMat &m, const int64_t *ptr, const int32_t *idx, const void *val,
                     int val_bytes, const uint8_t *lanes, const uint16_t *rank, const uint16_t *start, int *flag,
                     int sm_count, cudaStream_t st)
{
    const bool small = stk_rec_bytes(m.words) == 4;
    if (val_bytes == 2) {
        if (small)
            fill_typed<uint32_t, uint16_t>(I, J, m, ptr, idx, val, lanes, rank, start, flag, sm_count, st);
        else
            fill_typed<uint64_t, uint16_t>(I, J, m, ptr, idx, val, lanes, rank, start, flag, sm_count, st);
    } else {
        if (small)
            fill_typed<uint32_t, uint32_t>(I, J, m, ptr, idx, val, lanes, rank, start, flag, sm_count, st);
        else
            fill_typed<uint64_t, uint32_t>(I, J, m, ptr, idx, val, lanes, rank, start, flag, sm_count, st);
    }
    return cudaGetLastError();
}

void stk_colcount(const StackMat &m, int32_t *cnt, cudaStream_t st)
{
    const int64_t n = m.ntiles * 32 * m.words;
    k_stk_colcount<<<grid_of(n), kT, 0, st>>>(n, m.uidx, cnt);
}

void stk_place(int64_t J, const StackMat &m, int32_t *cnt, int32_t *ent, cudaStream_t st)
{
    const int64_t n = m.ntiles * 32 * m.words;
    k_stk_place<<<grid_of(n), kT, 0, st>>>(n, m.uidx, m.poff, cnt, ent);
    k_stk_order<<<grid_of(J), kT, 0, st>>>(J, m.poff, ent, m.ppos);
}

}  // namespace sgtv
