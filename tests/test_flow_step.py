"""Step completion of the decoupled kernel, every interleaving on the CPU.

The walkers report a step's batches and blocks of put-aside streams and the
appliers wait for them through the code of csrc/tmcs_flow_step.h. The model in
flow_step_model.cpp runs that code with two walkers, one applier and a slot
that two steps use in turn, in every order of their accesses: no walker may
take a later step's count for its own, no step may be applied before its
streams have ended, and none may wait forever.
"""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_every_interleaving(tmp_path):
    exe = str(tmp_path / "flow_step_model")
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", os.path.join(ROOT, "paper_2504_05611_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "flow_step_model.cpp"), "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stdout
