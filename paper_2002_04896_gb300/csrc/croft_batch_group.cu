// croft_batch_group.cu - the grouped schedule of batched plans (CROFT_BATCH_GROUPED):
// for each pass, one launch per distinct axis length over all grids that have it
// (croft_group_kernel.cuh), the launches of a pass concurrent in the plan's CUDA
// graph, the passes ordered by graph edges.
//
// Paper mapping: "option 4" of Sec. 5.1 - one 1D plan (here: one specialised
// kernel) reused for every pencil of that length, across grids as well.
#include <cuda_runtime.h>

#include <limits.h>
#include <string.h>

#include <algorithm>
#include <map>
#include <new>
#include <vector>

#include "../../include/croft.h"
#include "croft_group_kernel.cuh"
#include "croft_sizes.h"

namespace croft {

typedef void (*group_fn)(const GroupArgs);

template <int LAYOUT, int N>
static group_fn group_kernel_of() {
    if constexpr (group_two<LAYOUT, N>().r1 != 0) return croft_group_two_kernel<LAYOUT, N>;
    else return croft_group_kernel<LAYOUT, N>;
}

static group_fn group_kernel_for(int layout, int n) {
    switch (n) {
#define CROFT_G_CASE(N) \
    case N: return layout == LAYOUT_ROW ? group_kernel_of<LAYOUT_ROW, N>() : group_kernel_of<LAYOUT_COL, N>();
        CROFT_BATCH_SIZES(CROFT_G_CASE)
#undef CROFT_G_CASE
        default: return nullptr;
    }
}

int host_build_twiddles(int n, float* out);  // croft_plan.cu
void host_build_two_twiddles(int n, int r1, float* out);

struct GroupLaunch {
    int pass, layout, n;
    int nseg, ctas;
    int grid_of[kGroupSegs];     // batch index of each segment
    int reads_in[kGroupSegs];    // 1: the segment's pass is its grid's first pass (reads `in`)
    GroupArgs args;              // (pointers and isign filled per exec)
    cudaGraphNode_t node[2];     // its node in the graph of each direction
    int W, block, smem;
    int tw_off;           // float2 offset of N's twiddles in the pool
};

struct GroupState {
    std::vector<GroupLaunch> launches;
    float2* d_tw = nullptr;
};

void group_state_destroy(GroupState* s) {
    if (!s) return;
    dev_free(s->d_tw);
    delete s;
}

// Builds the launches of the grids `pgrid` (axes all in the batched size list).
croft_status group_state_build(const std::vector<int>& dims, const std::vector<int>& pgrid, GroupState** out) {
    *out = nullptr;
    GroupState* s = new (std::nothrow) GroupState();
    if (!s) return CROFT_ERR_OOM;
    static const int kAxis[3] = {2, 1, 0};
    std::vector<float> pool;
    std::map<std::pair<int, int>, int> tw_off;  // (length, first radix of a two-stage pass or 0) -> offset
    // first pass of each grid (lowest pass index whose axis is longer than 1)
    std::vector<int> first(pgrid.size(), -1);
    for (size_t i = 0; i < pgrid.size(); ++i)
        for (int p = 0; p < 3 && first[i] < 0; ++p)
            if (dims[3 * pgrid[i] + kAxis[p]] > 1) first[i] = p;
    for (int p = 0; p < 3; ++p) {
        std::map<std::pair<int, int>, std::vector<int>> by_len;  // (layout, n) -> grids
        for (size_t i = 0; i < pgrid.size(); ++i) {
            const int g = pgrid[i];
            const int n = dims[3 * g + kAxis[p]];
            if (n <= 1) continue;
            const int nz = dims[3 * g + 2], ny = dims[3 * g + 1];
            const long long M = kAxis[p] == 2 ? 1 : (kAxis[p] == 1 ? (long long)nz : (long long)ny * nz);
            by_len[{M == 1 ? LAYOUT_ROW : LAYOUT_COL, n}].push_back((int)i);
        }
        for (auto& kv : by_len) {
            const int layout = kv.first.first, n = kv.first.second;
            group_fn f = group_kernel_for(layout, n);
            if (!f) {
                group_state_destroy(s);
                return CROFT_ERR_UNSUPPORTED_SIZE;
            }
            const bool row = layout == LAYOUT_ROW;
            const CroftTwo K = croft_two_batch(n, row);
            const std::pair<int, int> key{n, K.r1};
            if (!tw_off.count(key)) {
                tw_off[key] = (int)(pool.size() / 2);
                std::vector<float> t(2 * (size_t)n + 2, 0.f);
                if (K.r1) {
                    host_build_two_twiddles(n, K.r1, t.data());
                } else if (n > 1 && host_build_twiddles(n, t.data()) != n - 1) {
                    group_state_destroy(s);
                    return CROFT_ERR_UNSUPPORTED_SIZE;
                }
                pool.insert(pool.end(), t.begin(), t.begin() + 2 * n);
            }
            GroupLaunch L;
            L.pass = p;
            L.layout = layout;
            L.n = n;
            if (K.r1) {
                L.W = K.w;
                L.block = K.w * K.t;
                L.smem = croft_two_smem(K, n, row);
            } else {
                const int T = croft_threads_per_pencil(n);
                const int tw_pad = ((n + 1) / 2) * 2;
                L.W = row ? 256 / T : croft_col_width(n, 8);
                L.block = L.W * T;
                const long long tile_elems = row ? (long long)L.W * croft_row_ld_staged(n) : (long long)n * L.W;
                L.smem = (int)((tw_pad + tile_elems) * sizeof(float2));
            }
            L.tw_off = tw_off[key];
            L.nseg = L.ctas = 0;
            memset(&L.args, 0, sizeof(L.args));
            for (int& t : L.args.first_tile) t = INT_MAX;
            if (allow_smem((const void*)f, L.smem) != cudaSuccess) {
                cudaGetLastError();
                group_state_destroy(s);
                return CROFT_ERR_CUDA;
            }
            for (int i : kv.second) {
                const int g = pgrid[i];
                const long long N = (long long)dims[3 * g] * dims[3 * g + 1] * dims[3 * g + 2];
                const int nz = dims[3 * g + 2], ny = dims[3 * g + 1];
                if (L.nseg == kGroupSegs) {  // full: the rest in another launch
                    s->launches.push_back(L);
                    L.nseg = L.ctas = 0;
                    for (int& t : L.args.first_tile) t = INT_MAX;
                }
                GroupSeg& S = L.args.seg[L.nseg];
                S.M = kAxis[p] == 2 ? 1 : (kAxis[p] == 1 ? (long long)nz : (long long)ny * nz);
                S.ncols = N / n;
                S.cdiv = croft_coldiv_make(S.M, S.ncols + L.W);
                const long long tiles = (S.ncols + L.W - 1) / L.W;
                if (L.ctas + tiles > 0x7ffffffeLL) {
                    group_state_destroy(s);
                    return CROFT_ERR_UNSUPPORTED_SIZE;
                }
                L.args.first_tile[L.nseg] = L.ctas;
                L.grid_of[L.nseg] = g;
                L.reads_in[L.nseg] = first[i] == p ? 1 : 0;
                L.ctas += (int)tiles;
                ++L.nseg;
            }
            s->launches.push_back(L);
        }
    }
    if (s->launches.empty()) {
        *out = s;
        return CROFT_OK;
    }
    if (dev_alloc((void**)&s->d_tw, sizeof(float) * std::max<size_t>(2, pool.size())) != cudaSuccess) {
        cudaGetLastError();
        group_state_destroy(s);
        return CROFT_ERR_OOM;
    }
    if (!pool.empty() && cudaMemcpy(s->d_tw, pool.data(), sizeof(float) * pool.size(), cudaMemcpyHostToDevice) != cudaSuccess) {
        cudaGetLastError();
        group_state_destroy(s);
        return CROFT_ERR_CUDA;
    }
    for (GroupLaunch& L : s->launches) {
        L.args.tw = s->d_tw + L.tw_off;
        L.args.W = L.W;
    }
    *out = s;
    return CROFT_OK;
}

static cudaKernelNodeParams group_node_params(const GroupLaunch& L, void** params) {
    cudaKernelNodeParams kp;
    memset(&kp, 0, sizeof(kp));
    kp.func = (void*)group_kernel_for(L.layout, L.n);
    kp.gridDim = dim3((unsigned)L.ctas, 1, 1);
    kp.blockDim = dim3((unsigned)L.block, 1, 1);
    kp.sharedMemBytes = (unsigned)L.smem;
    kp.kernelParams = params;
    return kp;
}

// The grids' pointers for the next launch of direction dir's graph: every kernel's parameters (a change
// reaches later launches only, so an exec in flight keeps its own).
croft_status group_graph_fill(GroupState* s, cudaGraphExec_t ge, int dir, void* const* in, void* const* out) {
    for (GroupLaunch& L : s->launches) {
        for (int k = 0; k < L.nseg; ++k) {
            const int g = L.grid_of[k];
            L.args.seg[k].in = (const float2*)(L.reads_in[k] ? in[g] : out[g]);
            L.args.seg[k].out = (float2*)out[g];
        }
        L.args.isign = dir == 0 ? 1.f : -1.f;
        void* params[1] = {&L.args};
        const cudaKernelNodeParams kp = group_node_params(L, params);
        if (cudaGraphExecKernelNodeSetParams(ge, L.node[dir], &kp) != cudaSuccess) {
            cudaGetLastError();
            return CROFT_ERR_CUDA;
        }
    }
    return CROFT_OK;
}

// Adds pass 0 launches -> pass 1 launches -> pass 2 launches to direction dir's graph.
// With pdl, the edges from one pass's launches to the next pass's are programmatic:
// the next pass's CTAs may become resident (and load their twiddles) while the
// previous pass drains, and wait in the kernel (griddepcontrol.wait) for every
// upstream launch to complete before they read the grid.
croft_status group_graph_add(GroupState* s, cudaGraph_t g, int dir, bool pdl) {
    std::vector<cudaGraphNode_t> prev;
    for (int p = 0; p < 3; ++p) {
        std::vector<cudaGraphNode_t> cur;
        for (GroupLaunch& L : s->launches) {
            if (L.pass != p) continue;
            void* params[1] = {&L.args};
            const cudaKernelNodeParams kp = group_node_params(L, params);
            cudaGraphNode_t kn;
            if (prev.empty() || !pdl) {
                if (cudaGraphAddKernelNode(&kn, g, prev.data(), prev.size(), &kp) != cudaSuccess) return CROFT_ERR_CUDA;
            } else {
                if (cudaGraphAddKernelNode(&kn, g, nullptr, 0, &kp) != cudaSuccess) return CROFT_ERR_CUDA;
                std::vector<cudaGraphNode_t> to(prev.size(), kn);
                std::vector<cudaGraphEdgeData> ed(prev.size());
                for (cudaGraphEdgeData& e : ed) {
                    memset(&e, 0, sizeof(e));
                    e.from_port = cudaGraphKernelNodePortProgrammatic;
                    e.type = cudaGraphDependencyTypeProgrammatic;
                }
                if (cudaGraphAddDependencies(g, prev.data(), to.data(), ed.data(), prev.size()) != cudaSuccess) {
                    cudaGetLastError();  // programmatic edges refused: plain edges (the kernel's wait returns at once)
                    if (cudaGraphAddDependencies(g, prev.data(), to.data(), nullptr, prev.size()) != cudaSuccess)
                        return CROFT_ERR_CUDA;
                }
            }
            L.node[dir] = kn;
            cur.push_back(kn);
        }
        if (!cur.empty()) prev = cur;
    }
    return CROFT_OK;
}

int group_state_launches(const GroupState* s) { return s ? (int)s->launches.size() : 0; }

}  // namespace croft
