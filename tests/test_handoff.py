"""CPU model of the kernels' hand-offs (tests/handoff_model.cpp over the kernels'
own csrc/handoff.h): under random schedules, with waits that time out anywhere,
every role ends.  Nothing here, and nothing in the GPU tests, makes a GPU wait
without limit; the mistakes are planted in the model."""
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2609_36757_gb300", "csrc")


@pytest.fixture(scope="module")
def model(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("handoff") / "handoff_model")
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", CSRC, "-o", exe,
                    os.path.join(HERE, "handoff_model.cpp")], check=True)

    def run(kernel, protocol, seeds):
        out = subprocess.run([exe, kernel, protocol, str(seeds)], check=True,
                             capture_output=True, text=True, timeout=600).stdout
        return tuple(int(x) for x in out.split())
    return run


@pytest.mark.parametrize("kernel", ["fwd64", "fwd128", "dkdv", "dq"])
def test_every_role_ends_whatever_wait_fails(model, kernel):
    runs, failed, stuck = model(kernel, "shipped", 2000)
    assert failed > runs // 4  # the failures are there
    assert stuck == 0


@pytest.mark.parametrize("kernel,mistake", [
    ("fwd64", "burst"), ("fwd128", "burst"), ("dkdv", "burst"),
    ("dq", "burst"), ("fwd64", "blocking"), ("dkdv", "blocking"),
    ("dq", "one-ds")])
def test_the_model_sees_arrivals_that_stand_in_for_others(model, kernel,
                                                          mistake):
    assert model(kernel, mistake, 2000)[2] > 0
