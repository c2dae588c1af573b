"""The host code of the arena and the server on a stand-in for the CUDA runtime
(tests/engine_host.cu; no GPU): what happens when copies run as late as the
runtime allows, when launches fail, and when memory is full."""
import os
import subprocess

import pytest

from conftest import ROOT


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    from paper_2208_14870_gb300 import build
    exe = str(tmp_path_factory.mktemp("engine") / "engine_host")
    csrc = os.path.join(ROOT, "paper_2208_14870_gb300", "csrc")
    r = subprocess.run([build.nvcc(), *build.ARCH, "-O1", "-std=c++17", "-cudart", "none", "-I", csrc,
                        os.path.join(ROOT, "tests", "engine_host.cu"), "-o", exe, "-lpthread"],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return exe


@pytest.mark.parametrize("scenario", ["server_force", "server_force_failing", "server_device_ms", "server_recovery_fails",
                                      "staging_f32", "staging_f16s", "full_arena_f32", "full_arena_f16s", "pinned_parts_f32",
                                      "pinned_parts_f16s", "narrow_launches_f32", "narrow_launches_f16s",
                                      "small_forces_f32", "small_forces_f16s", "small_fields_f32", "small_fields_f16s"])
def test_scenario(program, scenario, tmp_path):
    env = dict(os.environ, LBM_AUTOTUNE_CACHE=str(tmp_path / "autotune.txt"))
    r = subprocess.run([program, scenario], capture_output=True, text=True, timeout=120, env=env)
    assert r.stdout == "ok\n", (r.returncode, r.stdout, r.stderr)
