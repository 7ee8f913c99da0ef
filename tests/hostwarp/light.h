// The surroundings of the light tracer's warp kernels for a run on the host: what a step and a march do is the model
// of warp.h; queues, stacks, stocks of path ids and rounds are the kernels' own source.
constexpr int FLR_FORM_WAVEFRONT_WARP = 2;
struct SceneDev { int B = 1; };
struct RunDev { uint64_t n_paths, path_offset; unsigned long long *work_counter; int regroup, hero; void *tallies; };
struct Smem { const float *inv_maj; };
struct AdjDev { int K; const float *ak, *ovf; float *grad_sigma_s; };
struct SmemLayout { int queue_off_bytes; };
static const float g_table[256] = {};
inline SmemLayout smem_layout(int, int, int) { return {0}; }
inline Smem block_prologue(const SceneDev &, unsigned char *, const SmemLayout &, void *, bool) { return {g_table}; }
inline void counters_carry(const Smem &) {}
inline void budget_flag(const RunDev &, const Smem &) {}
inline float3 inv_dir(float3 w) { return w; }
template <bool, bool, bool, bool = false> struct MedS_ { const SceneDev &S; const Smem &sm; };
