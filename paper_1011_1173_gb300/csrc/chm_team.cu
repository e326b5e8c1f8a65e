// Host side of the team kernel (chm_team.cuh): the scratch of one or many
// problems and the launch.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdlib>
#include <cstring>

#include "chm.h"
#include "chm_internal.h"
#include "chm_team.cuh"

namespace chm {

ScratchNeed team_need(const ProbShape *shapes, int count)
{
    ScratchNeed r;
    for (int i = 0; i < count; ++i) {
        const int nb = (int)((shapes[i].n + kW - 1) / kW), k = shapes[i].k;
        r.iflags += team::prob_flags(nb, k);
        r.progress += team::prob_tags(nb, k);
        r.data += team::prob_data(nb, k);
    }
    return r;
}

ScratchNeed team_need_cap(const ProbShape &sh)
{
    ScratchNeed r;
    const int nb = (int)((sh.n + kW - 1) / kW);
    r.iflags = team::prob_flags(nb, sh.k);
    r.progress = team::prob_tags(nb, sh.k);
    r.data = team::prob_data_cap(nb, sh.k);
    return r;
}

void team_carve(const ProbShape *shapes, int count, int dtype, const Scratch &sc, Prob *problems)
{
    size_t fi = 0, fp = 0, fd = 0;
    for (int i = 0; i < count; ++i) {
        const int nb = (int)((shapes[i].n + kW - 1) / kW), k = shapes[i].k;
        Prob &p = problems[i];
        p.nb = nb;
        p.k = k;
        p.ntasks = team::prob_tasks(nb, k, dtype == CHM_F64);
        p.iflags = sc.iflags + fi;
        p.progress = sc.progress + fp;
        p.data = sc.data + fd;
        fi += team::prob_flags(nb, k);
        fp += team::prob_tags(nb, k);
        fd += team::prob_data(nb, k);
    }
}

// Three blocks per SM in double, four in float.
static_assert(3 * (sizeof(team::TaskSmem<double>) + 1536) <= 228 * 1024, "shared memory of three blocks");
static_assert(4 * (sizeof(team::TaskSmem<float>) + 1536) <= 228 * 1024, "shared memory of four blocks");

namespace {

// One-time per-(device, type) set-up: the shared-memory attribute and the
// occupancy limit; allocates nothing.
template <typename T>
int occupancy(int dev, int *bps_out)
{
    static int occ[64] = {0};
    if (dev < 0 || dev >= 64) return CHM_ERR_ARG;
    if (!occ[dev]) {
        const int smem = (int)sizeof(team::TaskSmem<T>);
        if (cudaFuncSetAttribute(team::team_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess)
            return CHM_ERR_CUDA;
        int b = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, team::team_kernel<T>, team::kThreads, smem) != cudaSuccess ||
            b < 1)
            return CHM_ERR_CUDA;
        const char *e = getenv("CHM_MAX_CTAS_PER_SM");
        const int cap = e ? atoi(e) : 0;
        if (cap > 0 && cap < b) b = cap;
        occ[dev] = b;
    }
    *bps_out = occ[dev];
    return CHM_OK;
}

// Teams: one for a single problem; for many, about fourteen blocks each, so
// that the largest problems, which start first, end with the rest (512
// factors of order 64 to 4096 in double, two executions: 54.0 ms with 14
// blocks a team against 54.3 with 28 and 55.0 with four; 96 float factors
// up to order 2048, 608 blocks: 4.1 ms with 14, 3.9 with 38 and 4.5 with four).
int default_teams(int nprobs, int grid)
{
    const char *e = getenv("CHM_GROUPS");
    int g = e ? atoi(e) : 0;
    if (g <= 0) g = std::max(1, grid / 14);
    return std::max(1, std::min(std::min(g, nprobs), kMaxTeams));
}

template <typename T>
int launch_t(const Prob *single, const Prob *d_probs, int nprobs, long long tasks, const Scratch &sc,
             const LaunchCfg &cfg, long long *trace, cudaStream_t stream)
{
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return CHM_ERR_CUDA;
    int bps = 0;
    const int rc = occupancy<T>(dev, &bps);
    if (rc != CHM_OK) return rc;
    if (cfg.ctas_per_sm > 0) bps = std::min(bps, cfg.ctas_per_sm);
    long long grid = (long long)sm_count(dev) * bps;
    if (cfg.grid > 0) grid = std::min<long long>(grid, cfg.grid);
    grid = std::max<long long>(1, std::min(grid, tasks));
    team::Launch<T> P;
    memset(&P, 0, sizeof(P));
    P.probs = d_probs;
    if (single) P.prob0 = *single;
    P.nprobs = nprobs;
    P.nteams = cfg.groups > 0 ? std::max(1, std::min(std::min(cfg.groups, nprobs), kMaxTeams))
                              : default_teams(nprobs, (int)grid);
    P.nteams = (int)std::min<long long>(P.nteams, grid);
    P.ctl = sc.ctl;
    P.status = sc.status;
    P.trace = trace;
    P.timeout_ns = timeout_ns();
    P.skip_publish = cfg.skip_publish;
    P.ws_data = sc.data;
    P.ws_data_bytes = sc.data_bytes;
    P.ws_iflags = sc.iflags;
    P.ws_iflags_n = sc.iflags_cap;
    P.ws_progress = sc.progress;
    P.ws_progress_n = sc.progress_cap;
    P.chk_cut = check_cut();
    team::team_kernel<T><<<(int)grid, team::kThreads, sizeof(team::TaskSmem<T>), stream>>>(P);
    return cudaGetLastError() == cudaSuccess ? CHM_OK : CHM_ERR_CUDA;
}

}  // namespace

int team_occupancy(int dtype, int dev, int *ctas_per_sm)
{
    return dtype == CHM_F64 ? occupancy<double>(dev, ctas_per_sm) : occupancy<float>(dev, ctas_per_sm);
}

int launch_team(int dtype, const Prob *single, const Prob *d_probs, int nprobs, long long tasks, const Scratch &sc,
                const LaunchCfg &cfg, long long *trace, cudaStream_t stream)
{
    return dtype == CHM_F64 ? launch_t<double>(single, d_probs, nprobs, tasks, sc, cfg, trace, stream)
                            : launch_t<float>(single, d_probs, nprobs, tasks, sc, cfg, trace, stream);
}

}  // namespace chm
