"""Shared helpers of the GPU parity tests: move one seeded draw to both sides, compare masks."""
from __future__ import annotations

import numpy as np
import torch

from paper_2502_19078_b200 import workloads as wl


def gpu_layer(weights, binding, dev="cuda", activation=0):
    """binding.Layer (neuron-major, on the GPU) from a workloads.layer_weights() draw, norms included.
    The non-gated form (activation 2) leaves the drawn w_up out."""
    wg = weights["w_gate"].to(dev).contiguous()
    wu = None if activation == 2 else weights["w_up"].to(dev).contiguous()
    wdt = weights["w_down"].to(dev).t().contiguous()      # row j = column j of W_out
    layer = binding.Layer(wg, wu, wdt, activation=activation)
    norms = torch.empty(layer.d_ff, dtype=torch.float32, device=dev)
    binding.clada_down_norms(layer, norms)
    layer.set_down_norm(norms)
    return layer


def oracle_weights(weights, activation=0):
    """(W_in, V_in, W_out) numpy arrays in the paper's layout for the oracle (V_in None when non-gated)."""
    return (wl.to_numpy_bits(weights["w_gate"]),
            None if activation == 2 else wl.to_numpy_bits(weights["w_up"]),
            wl.to_numpy_bits(weights["w_down"]))


def compare_masks(mask_gpu: np.ndarray, scores_oracle: np.ndarray, tau: float, rel=1e-6):
    """Masks must agree bit for bit except where the oracle's score lies within `rel` of tau.
    Returns (n_excused, n_mismatched)."""
    mask_or = scores_oracle >= tau
    diff = np.nonzero(mask_or != mask_gpu.astype(bool))[0]
    if diff.size == 0:
        return 0, 0
    near = np.abs(scores_oracle[diff] - tau) <= rel * abs(tau)
    return int(near.sum()), int((~near).sum())


def rel_inf(a: np.ndarray, ref: np.ndarray) -> float:
    denom = float(np.max(np.abs(ref)))
    if denom == 0.0:
        return float(np.max(np.abs(a)))
    return float(np.max(np.abs(a.astype(np.float64) - ref)) / denom)


def launches(fn):
    """[(kernel name, grid)] of the library's kernels that `fn` launches, in order: the kernel nodes of a CUDA graph that
    captures the call."""
    import subprocess

    from cuda.bindings import driver

    def get(result):
        assert int(result[0]) == 0, result[0]
        return result[1]

    fn()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(graph):
        fn()
    raw = graph.raw_cuda_graph()
    n = driver.cuGraphGetNodes(raw, 0)
    assert int(n[0]) == 0, n[0]
    ran = []
    for node in get(driver.cuGraphGetNodes(raw, n[2]))[:n[2]]:
        if get(driver.cuGraphNodeGetType(node)) != driver.CUgraphNodeType.CU_GRAPH_NODE_TYPE_KERNEL:
            continue
        k = get(driver.cuGraphKernelNodeGetParams(node))
        name = get(driver.cuFuncGetName(k.func) if int(k.func) else driver.cuKernelGetName(k.kern)).decode()
        ran.append((name, (k.gridDimX, k.gridDimY, k.gridDimZ)))
    names = subprocess.run(["c++filt"], input="\n".join(n for n, _ in ran), capture_output=True, text=True, check=True)
    return [(n, grid) for n, (_, grid) in zip(names.stdout.splitlines(), ran) if "clada::" in n]
