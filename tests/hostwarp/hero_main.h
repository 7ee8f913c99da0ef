bool hero_march_begin(const SceneDev &, const RunDev &, const Smem &, const HQueue &q, int k, HMarch &hm, RegCnt &)
{
    model_march(hm.mc, ((uint64_t)q.pid_hi[k] << 32) | q.pid_lo[k], q.step[k]);
    return true;
}
bool hero_march_step(const SceneDev &, const RunDev &, const Smem &, HMarch &hm, RegCnt &) { return model_march_step(hm.mc); }
