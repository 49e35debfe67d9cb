// The host side of the multi-step kernel (march.cu) without a GPU: its launches are recorded instead of
// made, or answered with an error, and its order of tiles is walked on the host.
#include <cuda_runtime.h>

namespace {
cudaError_t fake_memset(void*, int, size_t, cudaStream_t) { return cudaSuccess; }
}  // namespace
#define cudaMemsetAsync fake_memset
#include "../paper_2608_23786_gb300/csrc/march.cu"

namespace mclbm {

namespace {
struct Launch {
    int64_t steps, src, dst, parity, lanes;
};
std::vector<Launch> g_launches;
cudaError_t g_answer;
constexpr int64_t kBase = int64_t(1) << 40;  // never dereferenced

template <class E>
cudaError_t record(MarchArgs<E>& a)
{
    if (g_answer != cudaSuccess) return g_answer;
    g_launches.push_back({a.steps, (int64_t)a.lev.src, (int64_t)a.lev.dst, a.lev.parity, a.lanes});
    return cudaSuccess;
}

// 0 if the order holds every tile of every step once, each after the tiles it waits for.
template <class E>
int walk(const mclbm_ctx* c, int vec, int64_t steps)
{
    MarchArgs<E> a;
    memset(&a, 0, sizeof(a));
    if (!march_order(a, c, vec, steps)) return 1;
    const unsigned units = 1u << a.logU, um = units - 1, tpu = 1u << a.logT;
    std::vector<unsigned> done((size_t)c->M * units, 0);  // tiles of a unit, all steps, as cnt
    std::vector<char> seen((size_t)c->M * units * tpu * steps, 0);
    MarchWalk w = march_begin(a, 0, 1);
    for (MarchTile t = march_next(a, w); t.valid; t = march_next(a, w)) {
        const size_t id = ((size_t)t.step * c->M * units + t.ctr) * tpu + t.tile;
        if (id >= seen.size() || seen[id]) return 2;
        seen[id] = 1;
        for (unsigned d : {um, 0u, 1u})
            if (done[(t.ctr & ~um) | ((t.ctr + d) & um)] < (t.step << a.logT)) return 3;
        ++done[t.ctr];
    }
    for (unsigned d : done)
        if (d != tpu * steps) return 4;
    return 0;
}
}  // namespace

cudaError_t launch_march_f32(MarchArgs<float>& a, int, int, int, int64_t, cudaStream_t) { return record(a); }
cudaError_t launch_march_f16(MarchArgs<__half>& a, int, int, int, int64_t, cudaStream_t) { return record(a); }
cudaError_t launch_march_f64(MarchArgs<double>& a, int, int, int, int64_t, cudaStream_t) { return record(a); }
void* lattice_ptr(const mclbm_ctx* c, int which) { return (char*)kBase + which * (int64_t)c->pop_bytes; }

}  // namespace mclbm

using namespace mclbm;

static mclbm_ctx context(int N, int M, int precision, int pattern)
{
    mclbm_ctx c{};
    c.cfg.N = N;
    c.cfg.M = M;
    c.cfg.precision = precision;
    c.cfg.pattern = pattern;
    c.N = N;
    c.M = M;
    c.logN = ilog2(N);
    c.n = (int64_t)N * N * N;
    c.elem_bytes = precision == MCLBM_FP64 ? 8 : (precision == MCLBM_FP32 ? 4 : 2);
    c.pop_bytes = c.elem_bytes * Q * c.n * M;
    c.units.omega = 1.0;
    c.num_sms = 152;
    return c;
}

extern "C" {

// Steps taken by the multi-step kernel of a call for nsteps (negative: the CUDA error of the call).
int64_t take(int N, int M, int precision, int pattern, int64_t nsteps, int answer, int64_t limit, int trajectory)
{
    g_launches.clear();
    g_answer = (cudaError_t)answer;
    mclbm_ctx c = context(N, M, precision, pattern);
    c.step_limit = limit;
    int64_t taken = -1;
    const cudaError_t e = trajectory ? launch_march_trajectory(&c, (void*)(kBase / 2), (void*)kBase, c.pop_bytes, nsteps, &taken)
                                     : launch_march(&c, nsteps, &taken);
    if (e != cudaSuccess) return -(int64_t)e;
    const bool counted = c.multi_launches == (int64_t)g_launches.size() && c.multi_steps == taken;
    return counted && c.steps == (trajectory ? 0 : taken) ? taken : -100000;
}

int velocities() { return Q; }

int launches(int64_t* out, int most)  // [][5]: steps, source, destination, parity of the first step, lanes
{
    for (int k = 0; k < most && k < (int)g_launches.size(); ++k) memcpy(out + 5 * k, &g_launches[k], sizeof(Launch));
    return (int)g_launches.size();
}

int order(int N, int M, int precision, int64_t steps)
{
    const mclbm_ctx c = context(N, M, precision, MCLBM_AA);
    const int vec = march_vec(precision, N, (int64_t)M * c.n);
    switch (precision) {
        case MCLBM_FP64: return walk<double>(&c, vec, steps);
        case MCLBM_FP32: return walk<float>(&c, vec, steps);
        default: return walk<__half>(&c, vec, steps);
    }
}
}
