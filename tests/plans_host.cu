// Prints the plans the library makes, on the host: each input line
//     precision problem flow streaming n  nx ny  nx ny ...
// describes a batch of n lattices (streaming: -1 as lbm_batch_create leaves it);
// the output line holds the batch's plan and the first lattice's own:
//     batch tile w h t  band threads rows | solo tile w h t  band threads rows
//     | solo tiles, dynamic shared memory of one | default prefetch of the first lattice
//     with 16-bit storage, and of the batch
//     | rows per block of the batch's sweeps | whether the lattice, and the batch, take several steps
//     per launch after lbm_(batch_)set_streaming to one buffer, and after -1
#include "lbm_api.cu"

#include <iostream>

int main() {
    int precision, problem, flow, streaming, n;
    while (std::cin >> precision >> problem >> flow >> streaming >> n) {
        std::vector<lbm_s> lats(n);
        lbm_batch_s b;
        b.precision = precision;
        b.problem = problem;
        b.flow = flow;
        b.streaming = streaming;
        for (lbm_s &h : lats) {
            std::cin >> h.nx >> h.ny;
            h.precision = precision;
            h.esize = precision == LBM_FP64 ? 8 : (precision == LBM_FP32 ? 4 : 2);
            h.ntx = (h.nx + kTW - 1) / kTW;
            h.num_sms = 152;
            h.p.problem = problem;
            h.p.flow_on = flow;
            set_grid(&h);
            plan_steps(&h);
            b.members.push_back(&h);
        }
        int prefetch = 0;
        if (precision == LBM_FP64) {
            batch_build<double>(&b);
        } else {
            batch_build<float>(&b);
            prefetch = reinterpret_cast<BatchEntry<float> *>(b.host_entries.data())->a[0].prefetch;
        }
        lbm_s &h = lats[0];
        TileArgs tl{};
        if (h.tile.t) tl = tile_args(&h, h.tile, h.tile.t, tile_cells(&h, h.tile.w, h.tile.h, h.tile.t, 1));
        std::printf("%d %d %d %d %d %d %d %d %d %d %d %u %d %d %d", b.tile.w, b.tile.h, b.tile.t, b.band.threads, b.band.rows,
                    h.tile.w, h.tile.h, h.tile.t, h.band.threads, h.band.rows, tl.tiles_x * tl.tiles_y, tl.smem,
                    default_prefetch16(&h), prefetch, batch_shape(&b).rows);
        for (int mode : {1, -1}) {
            const int rc = lbm_set_streaming(&h, mode) | lbm_batch_set_streaming(&b, mode);
            std::printf(" %d %d", rc == 0 && (use_tiles(&h) || use_bands(&h)),
                        rc == 0 && !batch_sweeps_chosen(&b) && (b.tile.t > 0 || b.band.threads > 0));
        }
        std::printf("\n");
    }
    return 0;
}
