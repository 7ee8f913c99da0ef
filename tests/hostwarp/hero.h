struct HeroSet { int n, hero, bin[4]; float q[4]; };
struct HMarch { March mc; };
inline SmemLayout hero_warp_layout(int, int) { return {0}; }
template <class M> Conn spawn_rolled(const M &, const RunDev &, const Smem &, uint64_t pid, Path &p, int *) { return model_spawn(pid, p); }
template <class M> void hero_lines(const M &, const SceneDev &, int, int, HeroSet &h) { h = HeroSet{}; }
template <class M> Conn track_step_hero(const M &, const RunDev &, const Smem &, Path &p, HeroSet &, RegCnt &) { return model_step(p); }
