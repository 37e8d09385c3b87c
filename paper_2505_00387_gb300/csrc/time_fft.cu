// Launches of the register-FFT time kernels (time_fft.cuh).
#include <algorithm>

#include "time_fft_dispatch.cuh"

namespace aahrt {

static FrameFn frame_pick(int L) {
    switch (L) {
        case 9: return frame_call<2>;
        case 10: return frame_call<4>;
        case 11: return frame_call<8>;
        case 12: return frame_call<16>;
        case 13: return frame_call<32>;
        default: return nullptr;
    }
}

template <int C>
static size_t frame_most(int pairs, int nrows, int nfrac) {
    return frame_smem<Frame<C>>(pairs, 1, nrows, nfrac);
}

// Shared memory of an analysis block of one pair taking seq pairs in turn.
static size_t frame_analysis_smem(int L, int seq, int nrows, int nfrac) {
    switch (L) {
        case 9: return frame_smem<Frame<2>>(1, seq, nrows, nfrac);
        case 10: return frame_smem<Frame<4>>(1, seq, nrows, nfrac);
        case 11: return frame_smem<Frame<8>>(1, seq, nrows, nfrac);
        case 12: return frame_smem<Frame<16>>(1, seq, nrows, nfrac);
        default: return frame_smem<Frame<32>>(1, seq, nrows, nfrac);
    }
}

// Shared memory of the largest time kernel of frames of 2^L samples.
static size_t frame_plan_smem(int L, int pairs, int nt, int ntau) {
    const int nrows = std::max(nt, ntau), nfrac = nt;
    switch (L) {
        case 9: return frame_most<2>(pairs, nrows, nfrac);
        case 10: return frame_most<4>(pairs, nrows, nfrac);
        case 11: return frame_most<8>(pairs, nrows, nfrac);
        case 12: return frame_most<16>(pairs, nrows, nfrac);
        default: return frame_most<32>(pairs, nrows, nfrac);
    }
}

bool frame_serves(int L, int nt, int ntau, int max_smem) {
    // (1 KB stays for the kernels' static shared memory)
    return L >= 9 && L <= 13 && frame_plan_smem(L, 1, nt, ntau) + 1024 <= (size_t)max_smem;
}

static int gather_pairs(int L) { return L >= 12 ? 2 : 4096 >> L; }

bool gather_frames_serve(int L, int nt, int ntau, int max_smem) {
    return L >= 9 && L <= 13 &&
           frame_plan_smem(L, gather_pairs(L), nt, ntau) + 1024 <= (size_t)max_smem;
}

cudaError_t configure_gather_frames(Plan &p, int max_smem) {
    p.frame_pairs = gather_pairs(p.L);
    const FrameArgs none{};
    cudaError_t e = cudaSuccess;
    for (int op = GATHER_R2C; op <= GATHER_C2R; ++op)
        for (int model = 0; model < 2; ++model)
            for (int epi = 0; epi < 2 && !e; ++epi)
                e = frame_pick(p.L)(FrameCall{(FrameOp)op, model != 0, p.interp, epi, 1, nullptr,
                                              max_smem}, none, nullptr, nullptr, nullptr);
    return e;
}

cudaError_t configure_frame_kernels(Plan &p, int num_sms, int max_smem) {
    // 256 threads a block, fewer while blocks are fewer than SMs
    const long long groups = std::min(p.ncg_model_blk, p.ncg_data_blk);
    p.frame_pairs = std::max(1, 256 / (p.nfft / 16));
    while (p.frame_pairs > 1 &&
           (groups / p.frame_pairs < num_sms ||
            frame_plan_smem(p.L, p.frame_pairs, p.nt, p.ntau) + 1024 > (size_t)max_smem))
        p.frame_pairs /= 2;
    // pairs an analysis block of one pair takes in turn: as many as cost at most
    // 3 % more rounds of resident blocks than one at a time, within the shared
    // memory of three blocks an SM (10 % where a block has its SM to itself
    // and nothing else hides the wait for its rows).  Data analyses of 100-4000
    // pairs, 1001 to 3200 samples: 1 % above the best of 1, 2 and 4 on average,
    // 14 % at most (1200 pairs of 1600 samples, 47 us against 41); always one at a
    // time is up to 23 % above it (1824 pairs of 2800 samples, 164 against 133).
    for (int model = 0; model < 2; ++model) {
        const long long n = model ? p.ncg_model_blk : p.ncg_data_blk;
        const long long room = (p.L <= 12 ? 3LL : 1LL) * num_sms;
        int &seq = model ? p.frame_seq_model : p.frame_seq_data;
        seq = 1;
        for (int q = 2; q <= 4 && p.frame_pairs == 1; q *= 2) {
            const long long rounds = ((n + q - 1) / q + room - 1) / room * q;
            const size_t smem = frame_analysis_smem(p.L, q, model ? p.ntau : p.nt, model ? 0 : p.nt);
            if (100 * rounds <= (p.L <= 12 ? 103 : 110) * ((n + room - 1) / room) &&
                smem + 1536 <= (size_t)max_smem / (p.L <= 12 ? 3 : 1))
                seq = q;
        }
    }
    p.frame_ahead = (p.L <= 12 ? 4 : 2) * num_sms;       // resident blocks, by registers
    const FrameFn fn = frame_pick(p.L);
    const FrameArgs none{};
    cudaError_t e = cudaSuccess;
    for (int op = 0; op < 3; ++op)
        for (int model = 0; model < 2; ++model)
            for (int epi = 0; epi < 3 && !e; ++epi)
                e = fn(FrameCall{(FrameOp)op, model != 0, p.interp, epi, 1, nullptr, max_smem}, none,
                       nullptr, nullptr, nullptr);
    return e;
}

cudaError_t launch_frame(Plan &p, int op, bool model_side, int epi, const void *in, void *out,
                         const float *aux, const FistaArgs &fa, bool blocked, bool bound,
                         cudaStream_t st) {
    FrameArgs a;
    a.groups = model_side ? (blocked ? p.cg_model_blk : p.cg_model_pair)
                          : (blocked ? p.cg_data_blk : p.cg_data_pair);
    a.ngroups = model_side ? p.ncg_model_blk : p.ncg_data_blk;
    a.syn = model_side ? p.ST : p.U;
    a.ana = model_side ? p.S : p.UT;
    a.nrows = model_side ? p.ntau : p.nt;
    // fractions staged: those of U^T, in a data analysis
    a.nfrac = model_side || op == FRAME_C2R ? 0 : p.nt;
    a.frac = model_side ? p.frac_s : p.frac_u;
    a.sc = FrameScatter{p.sc_i0, p.sc_n0};
    a.ahead = p.frame_pairs == 1 ? p.frame_ahead : 0;
    // (blocked rows are whole slabs: one pair at a time)
    a.seq = op != FRAME_R2C || blocked ? 1 : model_side ? p.frame_seq_model : p.frame_seq_data;
    a.ns = p.ns;
    a.nbins = p.nbins;
    a.tw = p.tw_t;
    a.fa = fa;
    a.ybd = bound ? FrameBound{p.ymax, p.nychunk, p.ychunk_log} : FrameBound{nullptr, 0, 0};
    if (p.gather_frames) {
        a.groups = model_side ? p.cg_model_pair : p.cg_data_pair;
        a.ngroups = model_side ? p.ncg_model_pair : p.ncg_data_pair;
        a.seq = 1;
        op = op == FRAME_R2C ? GATHER_R2C : GATHER_C2R;
    }
    return frame_pick(p.L)(FrameCall{(FrameOp)op, model_side, p.interp, epi, p.frame_pairs, st, 0}, a,
                           in, out, aux);
}

}  // namespace aahrt
