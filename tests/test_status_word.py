"""Every launch with bounded waits reports to the status word that
ns_problem_status reads.  The waits cannot be made to expire from outside, so the
wiring is read from the sources."""

import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2509_13307_gb300", "csrc")


def _source(name):
    with open(os.path.join(CSRC, name)) as f:
        return f.read()


def test_status_call_reads_the_workspace_word():
    body = _source("problem.cu").split("int ns_problem_status(")[1].split("\n}")[0]
    assert set(re.findall(r"[\w>.-]*d_err", body)) == {"p->ws.d_err"}


def test_gradient_launches_report_to_it():
    src = re.sub(r"//[^\n]*", "", _source("adjoint.cu"))
    assert set(re.findall(r"[\w>.-]*d_err", src)) == {"p->ws.d_err"}
    for call in ("launch_layer_f64(", "launch_gemm_planes(", "launch_projection_adj<double>(",
                 "launch_projection_adj<float>("):
        parts = src.split(call)[1:]
        assert parts
        for part in parts:
            assert "p->ws.d_err" in part[:part.index(";")], (call, part[:200])
