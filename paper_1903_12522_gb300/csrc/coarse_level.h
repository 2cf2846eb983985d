// A level of the V-cycle's coarse end as the cluster kernel sees it (riesz.cu).
#pragma once

namespace cmcg {

struct CoarseLevel {
    int np, lo, cnt;  // nodes, and the CTA's run of them
    int halo;         // entries of the neighbours' runs that x and r hold copies of, on either side
    int chunk, sx, sy, sxy, nx, ny, nz, dim;
    int fused;                 // see lap_rn
    float cK, cB, inv2d;       // MGConst
    unsigned x, r, b;          // offsets in shared memory: iterate, residual / second buffer, right-hand side
    unsigned node;             // a byte per node
    unsigned long long m_chunk, m_sx, m_sy;  // factors of the divisions by chunk, sx, sy
};

}  // namespace cmcg
