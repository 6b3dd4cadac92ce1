"""A job whose wait gave up on the device (status 2 of its record) is an
error to its caller, from svm_train_batch and from the server alike, and never
a solve; the mapping that both use, built for the host, on every status."""
import os
import re
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1406_5161_gb300", "csrc")


def test_a_wait_that_gave_up_is_an_error(tmp_path):
    exe = str(tmp_path / "batch_status_check")
    subprocess.run(["g++", "-O1", "-std=c++17", "-I", CSRC, "-I", os.path.join(ROOT, "include"),
                    os.path.join(ROOT, "tests", "batch_status_check.cpp"), "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout


def test_both_callers_use_it():
    src = open(os.path.join(CSRC, "svm_api.cu")).read()
    for fn in ("srv_finish", "train_batch_impl"):
        body = src[re.search(rf"^\w+ {fn}\(", src, re.M).start():]
        body = body[:body.index("\n}\n")]
        assert "job_result(" in body and not re.search(r"\.status == [012]", body), fn
