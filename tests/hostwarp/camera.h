// The surroundings of the camera-side warp kernel for a run on the host. Its march stands in the kernel: every
// uniform the model draws moves it by one, and a march of L steps ends beyond L.
enum { FLR_C_PATHS, FLR_C_CONNECT_BUDGET };
constexpr int MAX_CONNECT_STEPS = 1 << 16;
constexpr float RT_RR_THRESHOLD = 0.0f;
struct SceneDev { int B = 1; bool homogeneous = false; };
struct RunDev { uint64_t n_paths, path_offset; unsigned long long *work_counter; void *tallies; };
struct Smem { const float *maj, *inv_maj; };
struct SmemLayout { int unused; };
struct RegCnt { uint32_t steps, nulls, events, scatters, connections, connect_steps, cell_walks; };
struct MarchRng { uint32_t s0, s1, s2, s3; };
static const float g_ones[256] = {1.0f};
constexpr int FLR_FORM_PLAIN = 0;
inline SmemLayout smem_layout(int, int, int) { return {0}; }
inline int camera_queue_offset(int, int) { return 0; }
inline Smem block_prologue(const SceneDev &, unsigned char *, const SmemLayout &, void *, bool) { return {g_ones, g_ones}; }
inline void block_epilogue(const SceneDev &, const RunDev &, const Smem &, const RegCnt &) {}
inline void counters_carry(const Smem &) {}
inline void cnt_add(const Smem &, int) {}
inline float3 inv_dir(float3 w) { return w; }
template <bool> struct MedS_ { const SceneDev &S; const Smem &sm; };
struct CamPath { float3 x, w, iw; int pix, bin; float pb, beta; uint32_t step; int n_events; uint64_t pid; bool alive; };
struct CamStart { float3 x, w; int pix, bin; float pb; };
struct LightGeom { float3 start, dir; float len, geom; int bx; bool ok; };
struct CamRec { LightGeom g; float wt; bool valid; };
inline bool camera_start(const SceneDev &, const RunDev &, const Smem &, uint64_t, CamStart &cs) { cs = CamStart{}; return true; }
inline CamRec camera_step(const SceneDev &, const RunDev &, const Smem &, CamPath &cp, RegCnt &)
{
    const uint32_t step = cp.step++;
    cp.alive = cp.step < path_steps(cp.pid);
    cp.pix = (int)(cp.pid * MAX_STEPS + step);   // the film value of this connection
    CamRec r{};
    r.g.len = (float)march_steps(cp.pid, step) + 0.5f;
    r.wt = 1.0f;
    r.valid = asks(cp.pid, step);
    return r;
}
inline MarchRng march_rng(const RunDev &, uint64_t, uint32_t, uint32_t) { return {}; }
inline float march_next(MarchRng &) { return 0.63212056f; }   // -log(1 - u) = 1
template <class M> float sigma_t_at(const M &, float3, int) { return 0.0f; }
inline void film_add(const SceneDev &, const RunDev &, size_t idx, float) { made(idx / MAX_STEPS, (uint32_t)(idx % MAX_STEPS)); }
