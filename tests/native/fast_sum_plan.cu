// Host side of the fast image sum without a GPU: the allocations and copies that
// fmm_plan and fmm_fit make land in host memory (linked with --wrap for the
// calls below), and the n-th allocation can be made to fail.
//
// Input: doubled n_coll n_cells, then per cell e1 e2 C n_bodies and per body n a b x y;
// then commands, each printing one line per precision and cell:
//   plan F    fmm_plan, allocation F (1, 2, ...) failing (0: none)
//   set ...   per cell e2, per body x y; then fmm_fit
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <iostream>
#include <string>

#include "../../paper_1912_04501_gb300/csrc/bie_internal.cuh"

static int g_calls = 0, g_fail = 0, g_live = 0;
static cudaError_t g_last = cudaSuccess;

extern "C" {
cudaError_t __wrap_cudaMalloc(void** p, size_t n) {
    if (++g_calls == g_fail) {
        *p = nullptr;
        return g_last = cudaErrorMemoryAllocation;
    }
    *p = std::calloc(1, n);
    ++g_live;
    return cudaSuccess;
}
cudaError_t __wrap_cudaFree(void* p) {
    if (p) --g_live;
    std::free(p);
    return cudaSuccess;
}
cudaError_t __wrap_cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) {
    std::memcpy(d, s, n);
    return cudaSuccess;
}
cudaError_t __wrap_cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t) {
    std::memset(d, v, n);
    return cudaSuccess;
}
cudaError_t __wrap_cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t __wrap_cudaGetLastError() {
    const cudaError_t e = g_last;
    g_last = cudaSuccess;
    return e;
}
}

int main() {
    using namespace bie;
    bie_ctx c;
    int doubled;
    std::cin >> doubled >> c.m >> c.ncell;
    c.sms = 152;
    c.utilde = doubled != 0;
    c.srcmul = doubled ? 4 : 1;
    for (int k = 0; k < c.ncell; ++k) {
        Cell cl{};
        double e1[2], e2[2];
        std::cin >> e1[0] >> e1[1] >> e2[0] >> e2[1] >> cl.C[0] >> cl.C[1] >> cl.n_bodies;
        cell_set_lattice(cl, e1, e2);
        cl.body_off = c.nb;
        cl.node_off = c.N;
        for (int j = 0; j < cl.n_bodies; ++j, ++c.nb) {
            double n, a, b, x, y;
            std::cin >> n >> a >> b >> x >> y;
            c.n_nodes.push_back((int)n);
            c.offsets.push_back(c.N);
            for (double v : {a, b, x, y, 0.0, n, (double)c.N, 0.0}) c.body_host.push_back(v);
            for (double v : {0.0, a, b, 0.0}) c.bshape_host.push_back(v);
            c.N += (int)n;
        }
        cl.n_nodes = c.N - cl.node_off;
        c.cells_h.push_back(cl);
    }
    c.offsets.push_back(c.N);
    std::string cmd;
    while (std::cin >> cmd) {
        int rc = 0;
        if (cmd == "plan") {
            std::cin >> g_fail;
            g_calls = 0;
            rc = fmm_plan(&c);
        } else {
            for (Cell& cl : c.cells_h) {
                double e2[2];
                const double e1[2] = {cl.e1[0], cl.e1[1]};
                std::cin >> e2[0] >> e2[1];
                cell_set_lattice(cl, e1, e2);
                for (int b = cl.body_off; b < cl.body_off + cl.n_bodies; ++b)
                    std::cin >> c.body_host[8 * b + 2] >> c.body_host[8 * b + 3];
            }
            rc = fmm_fit(&c);
        }
        const bool work = c.ws.fsq && c.ws.fmp && c.ws.floc && c.ws.ftick;
        std::printf("%s rc %d calls %d live %d work %d error %d\n", cmd.c_str(), rc, g_calls, g_live, (int)work, (int)g_last);
        for (int prec = 0; prec < 3; ++prec) {
            const Fmm& f = c.fmm[prec];
            std::printf("prec %d on %d walls %d held %d\n", prec, (int)f.on, (int)f.walls, (int)(f.arena != nullptr));
            if (!f.on || !f.arena) continue;
            for (int k = 0; k < c.ncell; ++k) {
                const FmmCell& q = f.cells[k];
                std::printf("cell %.17g %.17g %.17g %d %d %d %d %.17g %.17g\n", q.ox, q.oy, q.h, q.gx[0], q.gy[0], q.nlev,
                            q.wall, (double)f.t.centre[q.off[0]].x, (double)f.t.centre[q.off[0]].z);
            }
        }
    }
    free_fmm(&c);
    std::printf("freed live %d\n", g_live);
    return 0;
}
