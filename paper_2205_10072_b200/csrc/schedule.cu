// The calls that build schedules of one p (arXiv 2205.10072, Algorithms 1-5 and the lookup of Algorithm 9): they check
// their arguments and launch the kernels of rows.cu.  Many p at once: batch.cuh.
#include "bcs_common.cuh"

namespace bcs {

bcs_status make_table(uint32_t p, PTable *tab)
{
    if (p == 0) return BCS_ERR_RANGE;
    if (p > 0x7fffffffu) return BCS_ERR_UNSUPPORTED;
    const int q = ceil_log2_u32(p);
    for (int k = 0; k < kRow; ++k) tab->s[k] = 0;
    uint32_t v = p;
    for (int k = q; k >= 0; --k) {   // Algorithm 1: successive ceil-halving
        tab->s[k] = v;
        v = (v + 1u) / 2u;
    }
    tab->p = p;
    tab->q = q;
    return BCS_OK;
}

}  // namespace bcs

using namespace bcs;

extern "C" {

size_t bcs_build_workspace_bytes(uint32_t p, uint64_t r_begin, uint64_t r_end)
{
    if (check_range(p, r_begin, r_end) != BCS_OK) return 0;
    const int q = ceil_log2_u32(p);
    const uint64_t count = r_end - r_begin;
    if (q == 0 || count == 0) return 0;
    return (size_t)(align_up(4ull * p, 256) + (uint64_t)q * align_up(count, 16));
}

bcs_status bcs_build(uint32_t p, uint64_t r_begin, uint64_t r_end, int8_t *recv_out,
                     int8_t *send_out, void *workspace, size_t workspace_bytes,
                     void *cuda_stream)
{
    bcs_status st = check_range(p, r_begin, r_end);
    if (st != BCS_OK) return st;
    if (r_begin == r_end || p == 1) return BCS_OK;
    if (recv_out == nullptr && send_out == nullptr) return BCS_ERR_ARG;
    if (!aligned16(recv_out) || !aligned16(send_out) || !aligned16(workspace)) return BCS_ERR_ALIGN;
    (void)workspace_bytes;                   // the rows need no scratch memory, see rows.cuh
    return launch_rows(p, r_begin, r_end - r_begin, recv_out, send_out, static_cast<cudaStream_t>(cuda_stream));
}

size_t bcs_prepare_workspace_bytes(uint32_t p)
{
    if (p == 0 || p > 0x7fffffffu) return 0;
    const int q = ceil_log2_u32(p);
    if (q == 0) return 0;
    return (size_t)(align_up(4ull * p, 256) + (uint64_t)q * align_up(p, 16));
}

// A prepared p.  The call that writes a row computes it (rows.cuh), in no more time than the transposition of a
// prepared copy took, so preparing is no more than the checks, and the workspace is not touched.
static bcs_status prepare_check(uint32_t p, const void *workspace, size_t workspace_bytes)
{
    if (p == 0) return BCS_ERR_RANGE;
    if (p > 0x7fffffffu) return BCS_ERR_UNSUPPORTED;
    if (p == 1) return BCS_OK;
    if (workspace == nullptr || workspace_bytes < bcs_prepare_workspace_bytes(p)) return BCS_ERR_ARG;
    if (!aligned16(workspace)) return BCS_ERR_ALIGN;
    return BCS_OK;
}

bcs_status bcs_prepare_codes(uint32_t p, void *workspace, size_t workspace_bytes, void *)
{
    return prepare_check(p, workspace, workspace_bytes);
}

bcs_status bcs_prepare_rows(uint32_t p, uint64_t r_begin, uint64_t r_end, int8_t *recv_out,
                            void *workspace, size_t workspace_bytes, void *cuda_stream)
{
    bcs_status st = check_range(p, r_begin, r_end);
    if (st != BCS_OK) return st;
    st = prepare_check(p, workspace, workspace_bytes);
    if (st != BCS_OK || p == 1 || r_begin == r_end) return st;
    if ((r_begin & 15u) != 0 || !aligned16(recv_out)) return BCS_ERR_ALIGN;
    if (recv_out == nullptr) return BCS_OK;
    return launch_rows(p, r_begin, r_end - r_begin, recv_out, nullptr, static_cast<cudaStream_t>(cuda_stream));
}

bcs_status bcs_prepare(uint32_t p, void *workspace, size_t workspace_bytes, void *)
{
    return prepare_check(p, workspace, workspace_bytes);
}

bcs_status bcs_build_prepared(uint32_t p, uint64_t r_begin, uint64_t r_end, int8_t *recv_out,
                              int8_t *send_out, const void *workspace, size_t workspace_bytes,
                              void *cuda_stream)
{
    bcs_status st = check_range(p, r_begin, r_end);
    if (st != BCS_OK) return st;
    if (r_begin == r_end || p == 1) return BCS_OK;
    if (recv_out == nullptr && send_out == nullptr) return BCS_ERR_ARG;
    if (workspace == nullptr || workspace_bytes < bcs_prepare_workspace_bytes(p)) return BCS_ERR_ARG;
    if (!aligned16(recv_out) || !aligned16(send_out) || !aligned16(workspace)) return BCS_ERR_ALIGN;
    return launch_rows(p, r_begin, r_end - r_begin, recv_out, send_out, static_cast<cudaStream_t>(cuda_stream));
}

// The runs of virtual ranks (r - root) mod p of the range [r_begin, r_end): [v0, v0 + len_a) and,
// when the range passes virtual rank p - 1, [0, len_b).
struct RootedRuns {
    uint64_t v0, len_a, len_b;
};

static RootedRuns rooted_runs(uint32_t p, uint32_t root, uint64_t r_begin, uint64_t r_end)
{
    RootedRuns rr;
    const uint64_t count = r_end - r_begin;
    rr.v0 = count ? (r_begin + p - root) % p : 0;
    rr.len_a = count < p - rr.v0 ? count : p - rr.v0;
    rr.len_b = count - rr.len_a;
    return rr;
}

size_t bcs_build_rooted_workspace_bytes(uint32_t p, uint32_t root, uint64_t r_begin, uint64_t r_end)
{
    if (check_range(p, r_begin, r_end) != BCS_OK || root >= p) return 0;
    const int q = ceil_log2_u32(p);
    const RootedRuns rr = rooted_runs(p, root, r_begin, r_end);
    const size_t a = bcs_build_workspace_bytes(p, rr.v0, rr.v0 + rr.len_a);
    const size_t b = bcs_build_workspace_bytes(p, 0, rr.len_b);
    // two staging tables for the second run (used only where it lands off a 16-byte boundary)
    return (size_t)align_up(a > b ? a : b, 256) + 2 * (size_t)align_up(rr.len_b * (uint64_t)q, 256);
}

bcs_status bcs_build_rooted(uint32_t p, uint32_t root, uint64_t r_begin, uint64_t r_end,
                            int8_t *recv_out, int8_t *send_out, void *workspace,
                            size_t workspace_bytes, void *cuda_stream)
{
    bcs_status st = check_range(p, r_begin, r_end);
    if (st != BCS_OK) return st;
    if (root >= p) return BCS_ERR_RANGE;
    const int q = ceil_log2_u32(p);
    if (r_begin == r_end || q == 0) return BCS_OK;
    if (recv_out == nullptr && send_out == nullptr) return BCS_ERR_ARG;
    if (!aligned16(recv_out) || !aligned16(send_out) || !aligned16(workspace)) return BCS_ERR_ALIGN;
    const RootedRuns rr = rooted_runs(p, root, r_begin, r_end);
    const bool fast = workspace != nullptr &&
                      workspace_bytes >= bcs_build_rooted_workspace_bytes(p, root, r_begin, r_end);
    // (the kernel would not mind, but without a workspace such a range was always refused)
    if (rr.len_b != 0 && ((rr.len_a * (uint64_t)q) & 15u) != 0 && !fast) return BCS_ERR_ARG;
    return launch_rows(p, rr.v0, r_end - r_begin, recv_out, send_out, static_cast<cudaStream_t>(cuda_stream));
}

bcs_status bcs_build_to_host(uint32_t p, uint64_t r_begin, uint64_t r_end, int8_t *recv_host,
                             int8_t *send_host, void *stage_dev, size_t stage_bytes,
                             void *cuda_stream)
{
    bcs_status st = check_range(p, r_begin, r_end);
    if (st != BCS_OK) return st;
    const int q = ceil_log2_u32(p);
    const uint64_t bytes = (r_end - r_begin) * (uint64_t)q;
    if (bytes == 0) return BCS_OK;
    if (recv_host == nullptr && send_host == nullptr) return BCS_ERR_ARG;
    if (stage_dev == nullptr) return BCS_ERR_ARG;
    if (!aligned16(stage_dev)) return BCS_ERR_ALIGN;
    const uint64_t half = align_up(bytes, 256);
    if ((uint64_t)stage_bytes < 2 * half) return BCS_ERR_ARG;
    int8_t *recv_dev = static_cast<int8_t *>(stage_dev);
    int8_t *send_dev = recv_dev + half;
    st = launch_rows(p, r_begin, r_end - r_begin, recv_host ? recv_dev : nullptr, send_host ? send_dev : nullptr,
                     static_cast<cudaStream_t>(cuda_stream));
    if (st != BCS_OK) return st;
    cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
    if (recv_host &&
        cudaMemcpyAsync(recv_host, recv_dev, bytes, cudaMemcpyDeviceToHost, stream) != cudaSuccess)
        return BCS_ERR_CUDA;
    if (send_host &&
        cudaMemcpyAsync(send_host, send_dev, bytes, cudaMemcpyDeviceToHost, stream) != cudaSuccess)
        return BCS_ERR_CUDA;
    return BCS_OK;
}

bcs_status bcs_wait_expired(uint64_t *count_host)
{
    if (count_host == nullptr) return BCS_ERR_ARG;
    if (cudaDeviceSynchronize() != cudaSuccess) return BCS_ERR_CUDA;
    unsigned long long count = 0;            // (the kernel that hands out turns waits for its answers with a limit)
    if (!expired_wait_count(&count)) return BCS_ERR_CUDA;
    *count_host = count;
    return BCS_OK;
}

bcs_status bcs_build_static(uint32_t p, uint64_t r_begin, uint64_t r_end, int8_t *recv_out,
                            int8_t *send_out, void *cuda_stream)
{
    bcs_status st = check_range(p, r_begin, r_end);
    if (st != BCS_OK) return st;
    if (bcs_build_workspace_bytes(p, r_begin, r_end) > (size_t)BCS_STATIC_WORKSPACE_BYTES)
        return BCS_ERR_UNSUPPORTED;          // the stated limit of this entry point
    return bcs_build(p, r_begin, r_end, recv_out, send_out, nullptr, 0, cuda_stream);
}

}  // extern "C"
