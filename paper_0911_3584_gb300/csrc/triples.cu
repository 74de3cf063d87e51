// Symbolic phase of the listed-triple product kernel.
//
// For C = mask_C(op(A) op(B)) every block C_ij is a sum over the k with both
// op(A)_ik and op(B)_kj stored.  This pass lists, once per plan, those pairs
// of storage positions for every block of C, k ascending, so the numeric
// kernel neither searches B's rows nor multiplies blocks that are absent.
// The blocks of C are ordered by groups of four consecutive rows, and inside
// a group by the length of their lists, longest first (ties: by column, then
// row).  The numeric kernel runs eight blocks per warp and a warp lasts as
// long as its longest list, so lists of like length keep its lanes busy: on
// the products whose lists vary with the distance |r_i - r_j| (T = SX, U = SY
// and X = LS, Y = LH), column order left a third of the lanes idle.  Every
// block still sums its own list in k order, so the order changes no result.
#include <algorithm>
#include <cstdint>
#include <vector>

#include "lnv_impl.cuh"

namespace lnv {
namespace {

constexpr int kTripleGroup = 4;

__device__ __forceinline__ int64_t lower_bound_i32(const int32_t *__restrict__ a, int64_t lo, int64_t hi,
                                                   int32_t key)
{
    while (lo < hi) {
        const int64_t mid = lo + ((hi - lo) >> 1);
        if (a[mid] < key) lo = mid + 1;
        else hi = mid;
    }
    return lo;
}

// Count (tri == nullptr; items are C's blocks as stored where item_cb is null) or list the
// triples of each item.  op(A) and op(B) have the patterns of A and B (a transposed operand has
// a symmetric pattern); a transposed operand's block is read at the transpose position.
__global__ void k_triples(int64_t n_items, const int32_t *__restrict__ item_cb,
                          const int32_t *__restrict__ c_row, const int32_t *__restrict__ c_col,
                          const int64_t *__restrict__ a_rp, const int32_t *__restrict__ a_col,
                          const int64_t *__restrict__ a_tr, const int64_t *__restrict__ b_rp,
                          const int32_t *__restrict__ b_col, const int64_t *__restrict__ b_tr, int ta,
                          int tb, int64_t *cnt, const int64_t *__restrict__ t_off, int2 *tri)
{
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (t >= n_items) return;
    const int32_t cb = item_cb ? item_cb[t] : (int32_t)t;
    const int32_t i = c_row[cb], j = c_col[cb];
    int64_t c = 0, w = tri ? t_off[t] : 0;
    for (int64_t q = a_rp[i]; q < a_rp[i + 1]; ++q) {
        const int32_t k = a_col[q];
        const int64_t be = b_rp[k + 1];
        const int64_t p = lower_bound_i32(b_col, b_rp[k], be, j);
        if (p < be && b_col[p] == j) {
            if (tri) tri[w + c] = make_int2((int32_t)(ta ? a_tr[q] : q), (int32_t)(tb ? b_tr[p] : p));
            ++c;
        }
    }
    if (!tri) cnt[t] = c;
}

// The items of one group of C's rows, one CTA per group: the blocks by column, then row
// (at), and, in groups that fit shared memory, by length of their lists, longest first
// (a bitonic sort of length and first order; cap: a power of two, 0: the first order stays).
// 2010 atoms, X = LS (11 million triples, 1.3 million items): 0.11 ms, and the lists 2.2 ms
// in all; with both orders made on the host 6.9.
__global__ void __launch_bounds__(512)
k_order(int64_t n, const int64_t *__restrict__ rp, const int32_t *__restrict__ col, const int64_t *__restrict__ cnt,
        int cap, int32_t *__restrict__ item_cb, int64_t *__restrict__ cnt_out)
{
    extern __shared__ uint32_t key[];  // [cap], then uint16 at[cap]
    uint16_t *at = reinterpret_cast<uint16_t *>(key + cap);
    const int64_t r0 = (int64_t)blockIdx.x * kTripleGroup, r1 = min(n, r0 + kTripleGroup);
    const int64_t q0 = rp[r0], q1 = rp[r1];
    const int nq = (int)(q1 - q0);
    for (int64_t r = r0; r < r1; ++r)
        for (int64_t q = rp[r] + threadIdx.x; q < rp[r + 1]; q += blockDim.x) {
            const int32_t c = col[q];
            int64_t w = q - rp[r];
            for (int64_t o = r0; o < r1; ++o)  // ties go to the lower row
                if (o != r) w += lower_bound_i32(col, rp[o], rp[o + 1], o < r ? c + 1 : c) - rp[o];
            if (cap) {
                key[w] = (uint32_t)(0xFFFF - cnt[q]) << 16 | (uint32_t)w;
                at[w] = (uint16_t)(q - q0);
            } else {
                item_cb[q0 + w] = (int32_t)q;
                cnt_out[q0 + w] = cnt[q];
            }
        }
    if (!cap) return;
    int m = 1;
    while (m < nq) m <<= 1;
    for (int i = nq + threadIdx.x; i < m; i += blockDim.x) key[i] = 0xFFFFFFFFu;
    __syncthreads();
    for (int k = 2; k <= m; k <<= 1)
        for (int d = k >> 1; d > 0; d >>= 1) {
            for (int i = threadIdx.x; i < m / 2; i += blockDim.x) {
                const int a = 2 * i - (i & (d - 1)), b = a + d;
                const uint32_t x = key[a], y = key[b];
                if ((x > y) == ((a & k) == 0)) {
                    key[a] = y;
                    key[b] = x;
                }
            }
            __syncthreads();
        }
    for (int i = threadIdx.x; i < nq; i += blockDim.x) {
        item_cb[q0 + i] = (int32_t)(q0 + at[key[i] & 0xFFFF]);
        cnt_out[q0 + i] = 0xFFFF - (int64_t)(key[i] >> 16);
    }
}

}  // namespace

void triple_plan_free(TriplePlan *tp)
{
    cudaFree(tp->item_cb);
    cudaFree(tp->t_off);
    cudaFree(tp->tri);
    cudaFree(tp->up);
    *tp = TriplePlan();
}

lnv_status triple_plan_build(lnv_ctx *ctx, lnv_plan *pl, size_t budget_bytes)
{
    TriplePlan &tp = pl->tri;
    if (tp.tri || (tp.t_off && pl->triples == 0)) return LNV_OK;
    const lnv_pattern *A = pl->A, *B = pl->B, *C = pl->C;
    if (A->nnzb >= ((int64_t)1 << 31) || B->nnzb >= ((int64_t)1 << 31) || C->nnzb >= ((int64_t)1 << 31)) {
        set_error("triple-list plan: 2^31 or more blocks in an operand");
        return LNV_ERR_UNSUPPORTED;
    }
    const size_t need = sizeof(int2) * (size_t)pl->triples + (sizeof(int64_t) * 2 + sizeof(int32_t)) * (size_t)(C->nnzb + 1);
    if (need > budget_bytes) {
        set_error("triple-list plan needs %zu bytes, over the %zu budget", need, budget_bytes);
        return LNV_ERR_UNSUPPORTED;
    }
    const int64_t n = C->n, ng = (n + kTripleGroup - 1) / kTripleGroup;
    const size_t nc = (size_t)std::max<int64_t>(C->nnzb, 1);
    size_t bytes = sizeof(int32_t) * nc + sizeof(int64_t) * (size_t)(C->nnzb + 1);
    int64_t *by_block = nullptr, *cnt = nullptr;  // list lengths by block, by item
    cudaError_t e = dev_alloc(&tp.item_cb, sizeof(int32_t) * nc);
    if (e == cudaSuccess) e = dev_alloc(&tp.t_off, sizeof(int64_t) * (size_t)(C->nnzb + 1));
    if (e == cudaSuccess) e = dev_alloc(&by_block, sizeof(int64_t) * nc);
    if (e == cudaSuccess) e = dev_alloc(&cnt, sizeof(int64_t) * nc);
    if (e != cudaSuccess) {
        cudaFree(by_block);
        triple_plan_free(&tp);
        set_error("triple-list plan: allocation failed (%s)", cudaGetErrorString(e));
        return LNV_ERR_OOM;
    }
    tp.n_items = C->nnzb;
    const unsigned nb = (unsigned)((C->nnzb + 255) / 256);
    lnv_status s = LNV_OK;
    if (C->nnzb > 0) {
        k_triples<<<nb, 256, 0, ctx->stream>>>(C->nnzb, nullptr, C->row, C->col, A->row_ptr, A->col, A->tr,
                                               B->row_ptr, B->col, B->tr, pl->trans_a, pl->trans_b, by_block,
                                               nullptr, nullptr);
        if (cudaGetLastError() != cudaSuccess) s = LNV_ERR_CUDA;
        count_launch();
        // shared memory for the longest group (6 bytes an item); a list is no longer than a row of A
        int64_t longest = (int64_t)kTripleGroup * C->max_row, cap = 1;
        while (cap < longest) cap <<= 1;
        if (6 * cap > (int64_t)ctx->smem_optin || cap > 65536 || A->max_row > 0xFFFF) cap = 0;
        if (s == LNV_OK && ensure_smem((const void *)k_order, 6 * (size_t)cap) != cudaSuccess) s = LNV_ERR_CUDA;
        if (s == LNV_OK) {
            k_order<<<(unsigned)ng, 512, 6 * (size_t)cap, ctx->stream>>>(n, C->row_ptr, C->col, by_block, (int)cap,
                                                                         tp.item_cb, cnt);
            if (cudaGetLastError() != cudaSuccess) s = LNV_ERR_CUDA;
            count_launch();
        }
    }
    if (s == LNV_OK) s = scan_exclusive(ctx->stream, cnt, C->nnzb, tp.t_off);
    int64_t total = 0;
    if (s == LNV_OK && cudaMemcpyAsync(&total, tp.t_off + C->nnzb, sizeof(int64_t), cudaMemcpyDeviceToHost,
                                       ctx->stream) != cudaSuccess)
        s = LNV_ERR_CUDA;
    if (s == LNV_OK && cudaStreamSynchronize(ctx->stream) != cudaSuccess) s = LNV_ERR_CUDA;
    if (s == LNV_OK && total != pl->triples) {
        set_error("triple-list plan: %lld triples listed, %lld counted", (long long)total, (long long)pl->triples);
        s = LNV_ERR_PATTERN;
    }
    if (s == LNV_OK && total > 0) {
        if (dev_alloc(&tp.tri, sizeof(int2) * (size_t)total) != cudaSuccess) {
            set_error("triple-list plan: allocation of %lld triples failed", (long long)total);
            s = LNV_ERR_OOM;
        } else {
            bytes += sizeof(int2) * (size_t)total;
            k_triples<<<nb, 256, 0, ctx->stream>>>(C->nnzb, tp.item_cb, C->row, C->col, A->row_ptr, A->col,
                                                   A->tr, B->row_ptr, B->col, B->tr, pl->trans_a, pl->trans_b,
                                                   nullptr, tp.t_off, tp.tri);
            if (cudaGetLastError() != cudaSuccess) s = LNV_ERR_CUDA;
            count_launch();
            if (s == LNV_OK && cudaStreamSynchronize(ctx->stream) != cudaSuccess) s = LNV_ERR_CUDA;
        }
    }
    cudaFree(cnt);
    cudaFree(by_block);
    if (s == LNV_OK && pl->sym1) {
        // the items of C's upper triangle (col >= row), in item order
        s = pattern_host_cols(ctx, C);
        std::vector<int32_t> items((size_t)C->nnzb), row_of((size_t)C->nnzb), up;
        if (s == LNV_OK && cudaMemcpy(items.data(), tp.item_cb, sizeof(int32_t) * items.size(),
                                      cudaMemcpyDeviceToHost) != cudaSuccess)
            s = LNV_ERR_CUDA;
        if (s == LNV_OK) {
            for (int64_t r = 0; r < n; ++r)
                for (int64_t q = C->h_row_ptr[r]; q < C->h_row_ptr[r + 1]; ++q) row_of[(size_t)q] = (int32_t)r;
            up.reserve(items.size() / 2 + 1);
            for (size_t t = 0; t < items.size(); ++t)
                if (C->h_col[(size_t)items[t]] >= row_of[(size_t)items[t]]) up.push_back((int32_t)t);
        }
        tp.n_up = (int64_t)up.size();
        if (s == LNV_OK && !up.empty()) {
            if (dev_alloc(&tp.up, sizeof(int32_t) * up.size()) != cudaSuccess ||
                cudaMemcpy(tp.up, up.data(), sizeof(int32_t) * up.size(), cudaMemcpyHostToDevice) != cudaSuccess) {
                set_error("triple-list plan: allocation of the upper-triangle items failed");
                s = LNV_ERR_OOM;
            }
            bytes += sizeof(int32_t) * up.size();
        }
    }
    if (s != LNV_OK) {
        if (s == LNV_ERR_CUDA) set_error("triple-list plan: kernel failed");
        triple_plan_free(&tp);
        return s;
    }
    tp.bytes = bytes;
    return LNV_OK;
}

}  // namespace lnv
