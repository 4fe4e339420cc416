// walk_steps.cu -- one thread per query, the walk kernels' step code in two forms: fast_step where it
// applies (walker_advance's way) and walker_step alone, so that every ordinary crossing is half_step's.
// Built by test_gpu_walk_steps.py; not part of the library.
#include "../paper_2603_15780_gb300/csrc/walk.cuh"

struct Out {
    int32_t *face, *ncross;
    uint32_t *st;
    uint64_t *hash;
    float *state;  // [nq][4] end point and direction in the end face's frame
};

template <bool MIX, bool FAST>
__global__ void k_steps(int64_t nq, WalkParams P, QueryIn in, Out o) {
    const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= nq) return;
    Walker w;
    Carry<0> cw;
    if (walker_init<0>(P, in, q, w, cw)) {
        if (MIX) walker_start_mix(P, in, q, w);
        NoHook h;
        for (;;) {
            const int r = FAST ? fast_step<MIX, true>(w, P, h) : SG_FAST_SLOW;
            if (r == SG_FAST_CROSSED) continue;
            if (r == SG_FAST_END) break;
            if (walker_step<true, false, MIX>(w, P)) break;
        }
        walker_settle<MIX>(w, P);
    }
    o.face[q] = w.f; o.ncross[q] = w.ncross; o.st[q] = w.st; o.hash[q] = w.hash;
    o.state[4 * q] = w.px; o.state[4 * q + 1] = w.py; o.state[4 * q + 2] = w.dx; o.state[4 * q + 3] = w.dy;
}

extern "C" int walk_steps(const sg_mesh *m, int mix, int fast, int64_t nq, const int32_t *face, const float *bary,
                          const float *v, int max_steps, float tau_near, int32_t *out_face, int32_t *out_ncross,
                          uint32_t *out_st, uint64_t *out_hash, float *out_state) {
    WalkParams P{};
    P.rec = m->d_rec; P.fv = m->d_fv; P.frm = m->d_frm; P.half = m->d_half; P.V = m->d_V; P.face_off = m->d_face_off;
    P.lref = m->d_lref; P.half48 = m->d_half48; P.frm64 = m->d_frm64;
    P.max_steps = max_steps; P.tau_near = tau_near; P.tau_snap = 1e-6f; P.want_hash = 1;
    QueryIn in{};
    in.n_mesh = m->n_mesh; in.face = face; in.bary = bary; in.v = v;
    const Out o{out_face, out_ncross, out_st, out_hash, out_state};
    const unsigned grid = (unsigned)((nq + 127) / 128);
    if (mix) {
        if (fast) k_steps<true, true><<<grid, 128>>>(nq, P, in, o);
        else k_steps<true, false><<<grid, 128>>>(nq, P, in, o);
    } else {
        if (fast) k_steps<false, true><<<grid, 128>>>(nq, P, in, o);
        else k_steps<false, false><<<grid, 128>>>(nq, P, in, o);
    }
    return (int)cudaGetLastError();
}
