"""Kernels that may be set up while the one before on the stream ends (launch_next.cuh): an earlier grid's
writes are promised to be visible only behind the wait, so it is the first statement of each of them."""
import os
import re

import pytest

from paper_2310_07182_gb300 import build

SRC = {f: open(os.path.join(build.CSRC, f)).read() for f in os.listdir(build.CSRC) if f.endswith((".cu", ".cuh", ".cpp"))}


def _kernels():
    """(file, name, body) of every kernel."""
    for f, s in SRC.items():
        s = re.sub(r"#else\n__global__.*\n|#.*\n", "", s)  # a kernel's other heading; directives
        for m in re.finditer(r"__global__\s+void\s+(?:__\w+__\((?:[^()]|\([^()]*\))*\)\s*)?(k_\w+)\s*\(", s):
            i = s.index("{", m.end())
            depth, j = 1, i + 1
            while depth:
                depth += {"{": 1, "}": -1}.get(s[j], 0)
                j += 1
            yield f, m.group(1), s[i + 1:j - 1]


CHAINED = [k for k in _kernels() if "start_of_step" in k[2]]


def test_kernels_are_found():
    names = {k[1] for k in CHAINED}
    assert {"k_raygen", "k_trace_bvh2", "k_trace_shadow", "k_trace_bvh8", "k_finish_accumulate"} <= names


@pytest.mark.parametrize("f,name,body", CHAINED, ids=[k[1] for k in CHAINED])
def test_nothing_comes_before_the_wait(f, name, body):
    assert re.match(r"\s*(if \(kOne\) )?start_of_step\(\);", body)
    assert body.count("start_of_step") == 1


def test_no_kernel_lets_the_next_one_in_early():
    for s in SRC.values():
        assert "cudaTriggerProgrammaticLaunchCompletion" not in s and "griddepcontrol" not in s


def test_stage_events_and_chained_launches_exclude_each_other():
    """A launch behind a recorded event is not behind a kernel: no launch of a timed plan is chained."""
    s = SRC["cr_api.cpp"]
    plan = s[s.index("cr_status enqueue_plan("):]
    plan = plan[:plan.index("\n}\n")]
    decide = re.search(r"const bool chained = ([^;]*);", plan).group(1)
    assert decide.startswith("!times && ")
    assert all("chained" in v for v in re.findall(r"\.chained = ([^;]*);", plan))


def test_shared_memory_beyond_48_kb_is_allowed_before_occupancy_is_asked():
    """Otherwise the answer is 0 blocks, and such launches (32 stack entries, 352 threads or more) get the plain
    variant."""
    s = SRC["trace_common.cuh"]
    body = s[s.index("static uint32_t resident_blocks("):]
    body = body[:body.index("\n}\n")]
    assert 0 < body.find("allow_smem<kKernel>(smem)") < body.index("cudaOccupancyMaxActiveBlocksPerMultiprocessor")


def test_uploads_from_pageable_memory_are_waited_for():
    """cudaMemcpy from pageable memory may return before the data has arrived, and the render streams do not
    wait for the legacy stream that it runs on: a wait follows the scene's uploads and the server's table."""
    s = SRC["cr_api.cpp"]
    create = s[s.index("cr_status cr_scene_create("):s.index("static void free_workspace(")]
    assert create.rindex("cudaStreamSynchronize(cudaStreamLegacy)") > create.rindex("cudaMemcpyHostToDevice")
    t = SRC["server.cpp"]
    for i in [m.end() for m in re.finditer(r"cudaMemcpy\(", t)]:
        assert "cudaStreamSynchronize(cudaStreamLegacy)" in t[i:i + 250]


def test_the_server_clears_its_path_state():
    """A queue position that was reserved but not written must not hold uninitialised memory: it is used as
    an index.  The lanes' state, job tables and the scene table are cleared before the first iteration."""
    s = SRC["server.cpp"]
    body = s[s.index("cr_status cr_server_create("):s.index("r->loop()")]
    wait = body.index("cudaStreamSynchronize(cudaStreamLegacy)")
    for clear in ("cudaMemset(ws.base, 0, ws.bytes)", "cudaMemset(r->lanes[l].d_table[q], 0,", "cudaMemset(r->d_scenes, 0,"):
        assert 0 < body.index(clear) < wait
