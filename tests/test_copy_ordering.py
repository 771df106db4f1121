"""Host-to-device copies against the kernels that read them.  A handle's stream may be non-blocking (torch's are):
nothing then orders it after the legacy stream, where a plain cudaMemcpy runs; from pageable memory, and between
device arrays, such a copy may still be under way when the call returns.  So what a set-up kernel reads is
copied on the handle's stream, or the copy is waited for before the launch."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_16863_gb300", "csrc")


def _source(name):
    return re.sub(r"//.*", "", open(os.path.join(CSRC, name)).read())


def test_preconditioner_copies_run_on_its_stream():
    text = _source("precond.cuh")
    assert not re.search(r"\bcudaMemcpy(?:2D)?\s*\(", text) and not re.search(r"\bcudaMemset\s*\(", text)
    # the cluster program: copied before the images' kernel, its host array read until the stream is waited for
    body = text[text.index("aao_status store_cluster_plan"):]
    body = body[:body.index("aao_status build_cluster")]
    copy, image = body.index("cudaMemcpyAsync(dprog"), body.index("k_cluster_image")
    assert copy < image < body.rindex("cudaStreamSynchronize(st())")


def test_kappa_has_arrived_before_the_faces_are_formed():
    text = _source("solver.cu")
    copy, faces = text.index("cudaMemcpy(kap, grid->kappa"), text.index("launch(k_faces")
    assert copy < text.index("cudaStreamSynchronize(cudaStreamLegacy)", copy) < faces
