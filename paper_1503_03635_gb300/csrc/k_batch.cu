// k_batch.cu -- many facility-location instances solved in one pass.
//
// A batch is one graph U whose connected parts are the instances, so every
// phase (sketch hops, radii, keys, MIS sweeps, BFS) runs once over all of
// them, with the launch and synchronisation costs of one instance:
//   * a union batch: independent graphs placed side by side (graph i holds
//     vertices [off_i, off_{i+1}) of U); U's sketches are built per solve;
//   * a replica batch: R instances (own costs and client sets) on one
//     resident graph G whose sketches are built once.  U is R copies of G's
//     CSR; the instances share G's ADS: radii of all R instances are read
//     off it in one kernel, and only keys, MIS and BFS run on U.
// Ranks and priorities use part-local ids (fl_graph::vbase), so each part
// is solved exactly as it would be alone (Sections 3.1 and 4.1: the instances share no
// client, facility or edge).
#include <algorithm>
#include <cstdio>
#include <vector>

#include "fl_internal.cuh"

namespace fl {

namespace {

int grid_for(int64_t items, int per_block) {
    int64_t b = (items + per_block - 1) / per_block;
    if (b < 1) b = 1;
    if (b > 152 * 32) b = 152 * 32;
    return (int)b;
}

// Part i's CSR, already copied into U (its first n_i row offsets at voff,
// its columns at eoff), shifted to U's numbering.
__global__ void k_place_part(int part, int64_t n_i, int64_t nnz_i, int64_t voff, int64_t eoff,
                             int64_t* __restrict__ rowp, int32_t* __restrict__ cols, int32_t* __restrict__ vbase,
                             int32_t* __restrict__ vpart, int32_t* __restrict__ rid) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < n_i || t < nnz_i; t += stride) {
        if (t < n_i) {
            rowp[voff + t] += eoff;
            vbase[voff + t] = (int32_t)voff;
            vpart[voff + t] = part;
            rid[voff + t] = (int32_t)t;
        }
        if (t < nnz_i) cols[eoff + t] += (int32_t)voff;
    }
}

// Every CSR entry stays inside its vertex's part.
__global__ void k_check_parts(const int64_t* __restrict__ rowp, const int32_t* __restrict__ cols, int64_t n,
                              const int32_t* __restrict__ vbase, Counters* ctr) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += stride) {
        const int32_t b = vbase[v];
        for (int64_t e = rowp[v]; e < rowp[v + 1]; ++e)
            if (vbase[cols[e]] != b) {
                atomicOr(&ctr->error, 1ULL);
                break;
            }
    }
}

// U = R copies of G: vertex i*n + v, entries i*nnz + e.
__global__ void k_replicate_csr(const int64_t* __restrict__ rowp, const int32_t* __restrict__ cols, int64_t n,
                                int64_t nnz, int64_t R, int64_t* __restrict__ Urowp, int32_t* __restrict__ Ucols,
                                int32_t* __restrict__ vbase, int32_t* __restrict__ vpart,
                                const int32_t* __restrict__ base_rid, int32_t* __restrict__ rid) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const int64_t total_e = R * nnz, total_v = R * n;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < total_e || t <= total_v; t += stride) {
        if (t < total_e) {
            const int64_t i = t / nnz, e = t - i * nnz;
            Ucols[t] = (int32_t)(i * n + cols[e]);
        }
        if (t < total_v) {
            const int64_t i = t / n, v = t - i * n;
            Urowp[t] = i * nnz + rowp[v];
            vbase[t] = (int32_t)(i * n);
            vpart[t] = (int32_t)i;
            rid[t] = base_rid ? base_rid[v] : (int32_t)v;
        } else if (t == total_v) {
            Urowp[t] = total_e;
        }
    }
}

__global__ void k_replicate_i32(const int32_t* __restrict__ a, int64_t n, int64_t R, int32_t* __restrict__ out) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < n * R; t += stride) out[t] = a[t % n];
}

// Per instance: opening cost of its open facilities, open count, distance sum
// and unserved clients.  kObjParts blocks share an instance (one block each
// read 16 instances of 262 k vertices in 1.24 ms, now 0.04); block (i, c) sums its part
// in a fixed tree order, and k_batch_totals adds the parts up in order.
constexpr int kObjParts = 64;

struct ObjPart {
    double cost;
    long long n_open, dist_sum, unserved;
};

__global__ void __launch_bounds__(256) k_batch_objective(const int64_t* __restrict__ off, int n_inst, int parts,
                                                         const uint8_t* __restrict__ open,
                                                         const double* __restrict__ cost,
                                                         const uint8_t* __restrict__ client,
                                                         const int32_t* __restrict__ dist,
                                                         ObjPart* __restrict__ out) {
    __shared__ ObjPart red[256];
    for (int64_t b = blockIdx.x; b < (int64_t)n_inst * parts; b += gridDim.x) {
        const int i = (int)(b / parts), c = (int)(b % parts);
        const int64_t v0 = off[i], len = off[i + 1] - v0;
        const int64_t end = v0 + len * (c + 1) / parts;
        ObjPart p = {0.0, 0, 0, 0};
        for (int64_t v = v0 + len * c / parts + threadIdx.x; v < end; v += blockDim.x) {
            if (open[v]) {
                p.cost += cost[v];
                ++p.n_open;
            }
            if (client[v]) {
                const int32_t d = dist[v];
                if (d < 0) ++p.unserved;
                else p.dist_sum += d;
            }
        }
        red[threadIdx.x] = p;
        __syncthreads();
        for (int s = 128; s > 0; s >>= 1) {
            if ((int)threadIdx.x < s) {
                ObjPart& a = red[threadIdx.x];
                const ObjPart& o = red[threadIdx.x + s];
                a.cost += o.cost;
                a.n_open += o.n_open;
                a.dist_sum += o.dist_sum;
                a.unserved += o.unserved;
            }
            __syncthreads();
        }
        if (threadIdx.x == 0) out[b] = red[0];
        __syncthreads();
    }
}

__global__ void k_batch_totals(const ObjPart* __restrict__ part, int n_inst, int parts, double* __restrict__ obj,
                               long long* __restrict__ n_open, long long* __restrict__ dist_sum,
                               long long* __restrict__ unserved) {
    const int stride = gridDim.x * blockDim.x;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n_inst; i += stride) {
        ObjPart t = {0.0, 0, 0, 0};
        for (int c = 0; c < parts; ++c) {
            const ObjPart& p = part[(int64_t)i * parts + c];
            t.cost += p.cost;
            t.n_open += p.n_open;
            t.dist_sum += p.dist_sum;
            t.unserved += p.unserved;
        }
        obj[i] = t.cost + (double)t.dist_sum;
        n_open[i] = t.n_open;
        dist_sum[i] = t.dist_sum;
        unserved[i] = t.unserved;
    }
}

}  // namespace


int batch_place_parts(fl_graph* U, const std::vector<int64_t>& voff, const std::vector<int64_t>& eoff) {
    cudaStream_t st = U->stream;
    const int n_parts = (int)voff.size() - 1;
    for (int i = 0; i < n_parts; ++i) {
        const int64_t n_i = voff[i + 1] - voff[i], nnz_i = eoff[i + 1] - eoff[i];
        FL_LAUNCH(kProfOther, k_place_part<<<grid_for(std::max(n_i, nnz_i), 256), 256, 0, st>>>(
                                  i, n_i, nnz_i, voff[i], eoff[i], U->rowp.as<int64_t>(), U->cols.as<int32_t>(),
                                  U->vbase.as<int32_t>(), U->vpart.as<int32_t>(), U->rid.as<int32_t>()));
    }
    FL_CUDA(cudaGetLastError());
    return FL_OK;
}

int batch_check_parts(fl_graph* U) {
    cudaStream_t st = U->stream;
    FL_CUDA(cudaMemsetAsync(U->ctr.p, 0, sizeof(Counters), st));
    FL_LAUNCH(kProfOther, k_check_parts<<<grid_for(U->n, 256), 256, 0, st>>>(
                              U->rowp.as<int64_t>(), U->cols.as<int32_t>(), U->n, U->vbase.as<int32_t>(),
                              U->ctr.as<Counters>()));
    FL_CUDA(cudaGetLastError());
    FL_TRY(read_counters(U));
    if (U->h_ctr->error) FL_FAIL(FL_EINVAL, "a CSR entry leaves its graph (column outside [0, n_i))");
    return FL_OK;
}

int batch_replicate(const fl_graph* G, int64_t R, fl_graph* U) {
    cudaStream_t st = U->stream;
    FL_LAUNCH(kProfOther, k_replicate_csr<<<grid_for(std::max(R * G->nnz, R * G->n + 1), 256), 256, 0, st>>>(
                              G->rowp.as<int64_t>(), G->cols.as<int32_t>(), G->n, G->nnz, R, U->rowp.as<int64_t>(),
                              U->cols.as<int32_t>(), U->vbase.as<int32_t>(), U->vpart.as<int32_t>(),
                              G->rid.p ? G->rid.as<int32_t>() : nullptr, U->rid.as<int32_t>()));
    FL_CUDA(cudaGetLastError());
    return FL_OK;
}

int batch_replicate_ecc(const fl_graph* G, int64_t R, fl_graph* U) {
    FL_TRY(dalloc(U->ecc_ub, (size_t)U->n * 4));
    FL_LAUNCH(kProfOther, k_replicate_i32<<<grid_for(U->n, 256), 256, 0, U->stream>>>(
                              G->ecc_ub.as<int32_t>(), G->n, R, U->ecc_ub.as<int32_t>()));
    FL_CUDA(cudaGetLastError());
    return FL_OK;
}

int batch_objective(fl_solve* s, const int64_t* off_d, int n_inst, double* obj, long long* n_open,
                    long long* dist_sum, long long* unserved) {
    fl_graph* g = s->g;
    // about 1000 vertices per block at least
    const int64_t mean = g->n / n_inst;
    const int parts = (int)std::max<int64_t>(1, std::min<int64_t>(kObjParts, mean / 1024));
    FL_TRY(dalloc(s->obj_tmp, (size_t)n_inst * parts * sizeof(ObjPart)));
    ObjPart* part = s->obj_tmp.as<ObjPart>();
    const int64_t blocks = std::min<int64_t>((int64_t)n_inst * parts, 152 * 16);
    FL_LAUNCH(kProfOther, k_batch_objective<<<(unsigned)blocks, 256, 0, g->stream>>>(
                              off_d, n_inst, parts, s->open.as<uint8_t>(), s->cost.as<double>(),
                              s->client.as<uint8_t>(), s->dist.as<int32_t>(), part));
    FL_LAUNCH(kProfOther, k_batch_totals<<<(unsigned)std::min((n_inst + 127) / 128, 152), 128, 0, g->stream>>>(
                              part, n_inst, parts, obj, n_open, dist_sum, unserved));
    FL_CUDA(cudaGetLastError());
    return FL_OK;
}


}  // namespace fl
