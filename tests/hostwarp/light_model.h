inline void block_epilogue(const SceneDev &, const RunDev &, const Smem &, const RegCnt &) {}
struct AdjObs { const SceneDev &S; const Smem &sm; const AdjDev &A; float left; float *g; };

// The connection that step `p.step - 1` of the path asks for, if any; ends the path at its last step.
inline Conn model_step(Path &p)
{
    const uint32_t step = p.step++;
    p.alive = p.step < path_steps(p.pid);
    return Conn{p.x, 1.0f, 0, -1, p.pid, step, asks(p.pid, step)};
}

inline Conn model_spawn(uint64_t pid, Path &p)
{
    p = Path{};
    p.pid = pid;
    p.alive = true;
    Conn c{};
    return c;   // valid = false
}

template <class M, class Obs = int>
Conn spawn_or_track(const M &, const RunDev &, const Smem &, Path &p, RegCnt &, const Obs & = Obs())
{
    return p.step == STEP_SPAWN ? model_spawn(p.pid, p) : model_step(p);
}

inline void model_march(March &mc, uint64_t pid, uint32_t step)
{
    mc = March{};
    mc.it = march_steps(pid, step);
    mc.g = MarchRng{(uint32_t)pid, step, 0u, 0u};
}

inline bool model_march_step(March &mc)   // false once the march has ended, which makes the connection
{
    if (mc.it-- > 0) return true;
    made(mc.g.s0, mc.g.s1);
    return false;
}
