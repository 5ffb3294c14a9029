"""Kernels that reach into the shared memory of their cluster's other CTAs: CUDA requires every CTA of the
cluster to have started before its distributed shared memory is accessed, so a cluster barrier has to
stand before the first such access in the order of execution, and one behind the last, before a CTA
may leave. Checked on the source (a run cannot be expected to show it)."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2606_19224_gb300", "csrc")


def _kernels():
    """(file, kernel name, body) of every __global__ function that uses map_shared_rank."""
    out = []
    for f in sorted(os.listdir(CSRC)):
        if not f.endswith((".cu", ".cuh")):
            continue
        src = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, f)).read())
        for m in re.finditer(r"__global__[^;{]*?(\w+)\s*\((?=[^;{]*\)\s*\{)", src):
            at = src.index("{", m.end())
            depth, end = 1, at + 1
            while depth:
                depth += {"{": 1, "}": -1}.get(src[end], 0)
                end += 1
            body = src[at:end]
            if "map_shared_rank" in body:
                name = [n for n in re.findall(r"(\w+)\s*\(", src[m.start():at]) if n not in ("__launch_bounds__", "__cluster_dims__")]
                out.append((f, name[0], body))
    return out


def _without_lambdas(body):
    """The body without its named lambdas, and their texts by name."""
    lambdas = {}
    while True:
        m = re.search(r"auto (\w+) = \[&?\]\s*\([^)]*\)[^{;]*\{", body)
        if not m:
            return body, lambdas
        depth, end = 1, m.end()
        while depth:
            depth += {"{": 1, "}": -1}.get(body[end], 0)
            end += 1
        lambdas[m.group(1)] = body[m.end():end]
        body = body[:m.start()] + body[end + 1:]


KERNELS = _kernels()


def test_the_kernels_are_found():
    assert {k for _, k, _ in KERNELS} >= {"small_cg_f64_kernel", "small_cg_f32_kernel", "mlp_gemm_kernel", "mse_kernel"}


@pytest.mark.parametrize("file,kernel,body", KERNELS, ids=[k for _, k, _ in KERNELS])
def test_a_cluster_barrier_stands_before_the_first_and_behind_the_last_remote_access(file, kernel, body):
    main, lambdas = _without_lambdas(body)
    remote = {"map_shared_rank"}
    for _ in lambdas:   # lambdas that reach a remote access through others
        remote |= {n for n, text in lambdas.items() if any(re.search(rf"\b{r}\b", text) for r in remote)}
    access = [m.start() for r in remote for m in re.finditer(rf"\b{r}\(", main)]
    barrier = [m.start() for m in re.finditer(r"\bcluster\.sync\(\)", main)]
    assert access and barrier, (file, kernel)
    assert min(barrier) < min(access), f"{kernel}: remote access before the first cluster barrier"
    assert max(barrier) > max(access), f"{kernel}: no cluster barrier behind the last remote access"
