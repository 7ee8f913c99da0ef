"""Memory ordering of the warp-regrouped kernels' shared queues and stacks. The lanes of a warp pass records to one
another through shared memory; a vote (ballot, any) orders their execution but not their memory, only __syncwarp does
both. Here the kernels' own source runs on the host, 32 threads for the lanes, under a race detector that
knows the difference (tests/hostwarp/warp.h); it also checks that every connection is made exactly once and that no
queue or stack index leaves its bounds."""
import os
import re
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
SRC = os.path.join(os.path.dirname(HERE), "paper_1706_03024_gb300", "csrc", "fluoro_kernels.cu")


def _definition(text, head):
    """The definition that starts with `head` (with a template line before it), up to its closing brace."""
    m = re.search(r"^(template <[^\n]*>\n)?" + head, text, re.M)
    assert m, head
    i = text.index("{", m.end())
    depth, j = 0, i
    while True:
        depth += {"{": 1, "}": -1}.get(text[j], 0)
        j += 1
        if depth == 0:
            return text[m.start():j] + ";\n"


def _source(heads, constants):
    text = open(SRC).read()
    out = [re.search(rf"^constexpr (?:int|uint32_t) {c} = [^;]*;", text, re.M).group(0) + "\n" for c in constants]
    return out, {h: _definition(text, h) for h in heads}


def _f(name, kind="__device__ __forceinline__"):
    return rf"{kind} [^\n]*\b{name}\("


LIGHT = [r"struct RegCnt\b", r"struct MarchRng\b", r"struct Path\b", r"struct Conn\b", r"struct Queue\b", r"struct March\b"]
MAIN = """
int main()
{
    for (const unsigned long long n : {1ull, 33ull, 150ull}) {
        unsigned long long work = 0;
        RunDev R{};
        R.n_paths = n;
        R.work_counter = &work;
        RUN
        if (run_warp(n, [=] { CALL; })) return 1;
    }
    return 0;
}
"""


def _program(kernel):
    def inc(f):
        return f'#include "{f}"\n'

    if kernel == "camera":
        const, d = _source([_f("queue_length"), _f("k_trace_camera_warp", "__global__ void")],
                           ["SPAWN_MIN", "CARRY_ROUNDS", "CQ_CAP", "CQ_DRAIN", "CQ_WORDS"])
        body = [inc("camera.h"), *const, *d.values()]
        return body, MAIN.replace("RUN", "").replace("CALL", "k_trace_camera_warp(SceneDev{}, R)")
    const = ["WARP_BLOCK", "SPAWN_MIN", "CARRY_ROUNDS"]
    if kernel == "hero":
        const, d = _source(LIGHT + [_f("queue_length"), r"struct HQueue\b", _f("hq_push"),
                                    _f("k_trace_hero_warp", "__global__ void")],
                           const + ["HERO_MAX", "HQ_CAP", "HQ_DRAIN", "HQ_WORDS"])
        d = list(d.values())
        n = len(LIGHT)
        body = [inc("light.h"), "constexpr uint32_t STEP_SPAWN = 0xFFFFFFFFu;\n", *const, *d[:n], inc("light_model.h"),
                inc("hero.h"), *d[n:n + 3], inc("hero_main.h"), *d[n + 3:]]
        return body, MAIN.replace("RUN", "R.hero = 4;").replace("CALL", "k_trace_hero_warp(SceneDev{}, R)")
    const, d = _source(LIGHT + [r"struct PathIds\b", _f("wq_push"), _f("ids_left"), _f("queue_length"), _f("claim_path"),
                                _f("path_claimed"), _f("stack_store"), _f("stack_load"), _f("wq_drain"),
                                _f("k_trace_wavefront_warp", "__global__ void")],
                       const + ["WARP_BLOCKS", "WQ_CAP", "WQ_DRAIN", "MS_CAP", "MS_WORDS", "DRAIN_KEEP", "CLAIM_MIN",
                                "WARP_WORDS", "MAX_REGROUP", "WM_RENDER", "WM_ADJ_WEIGHTS", "WM_ADJ_GRAD", "WQ_ORD_MAX"])
    d = list(d.values())
    n = len(LIGHT)
    body = [inc("light.h"), "constexpr uint32_t STEP_SPAWN = 0xFFFFFFFFu;\n", *const, *d[:n], inc("light_model.h"),
            inc("warp_main.h"), *d[n:]]
    regroup = kernel.split("/")[1]
    return body, MAIN.replace("RUN", f"R.regroup = {regroup};").replace(
        "CALL", "k_trace_wavefront_warp<WM_RENDER, false, false, true>(SceneDev{}, R, AdjDev{})")


@pytest.mark.parametrize("kernel", ["light/1", "light/3", "hero", "camera"])
def test_lanes_exchange_records_only_across_a_syncwarp(tmp_path, kernel):
    body, main = _program(kernel)
    src, exe = tmp_path / "warp.cpp", tmp_path / "warp"
    src.write_text('#include "warp.h"\n' + "".join(body) + main)
    subprocess.run(["g++", "-std=c++17", "-O1", "-g", "-fsanitize=thread", "-pthread", "-w", "-I",
                    os.path.join(HERE, "hostwarp"), str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=600)
    if "unexpected memory mapping" in r.stderr:
        pytest.skip("the race detector cannot run under this kernel's address layout")
    assert "data race" not in r.stderr, r.stderr[:6000]
    assert r.returncode == 0, r.stderr[:6000]
