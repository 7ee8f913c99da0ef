template <int MODE, bool MC>
bool march_begin(const SceneDev &, const RunDev &, const Smem &, const AdjDev &, float3, int, float, int, int, uint64_t pid,
                 uint32_t step, March &mc, RegCnt &, float &)
{
    model_march(mc, pid, step);
    return true;
}
template <int MODE, bool LZ>
bool march_advance(const SceneDev &, const RunDev &, const Smem &, const AdjDev &, March &mc, RegCnt &) { return model_march_step(mc); }
template <int MODE, bool LZ>
bool march_matter(const SceneDev &, const RunDev &, const Smem &, const AdjDev &, March &, RegCnt &, float &) { return true; }
template <bool MC> float adjoint_weight(const SceneDev &, const RunDev &, const Smem &, const AdjDev &, const Conn &, RegCnt &) { return 0.0f; }
