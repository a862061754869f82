"""Early-launched step kernels (griddepcontrol.wait): resident while the kernel
before them writes their inputs, they may not read through the read-only path,
whose data has to stay unwritten for the whole kernel.  And runs of them repeat
bit for bit, directly and from a captured graph."""
import os
import re

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2402_05240_gb300", "csrc")


def _functions(text):
    """name -> signature and body of every function template in the file."""
    out = {}
    text = re.sub(r"__launch_bounds__\([^)]*\)", "", text)
    for m in re.finditer(r"(?:__global__|__device__)[^;{}()]*?(\w+)\s*\(", text):
        i = text.find("{", m.end())
        depth, j = 1, i + 1
        while depth:
            depth += {"{": 1, "}": -1}.get(text[j], 0)
            j += 1
        out.setdefault(m.group(1), "")
        out[m.group(1)] += text[m.start():j]
    return out


def test_no_read_only_loads_in_early_launched_kernels():
    text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, "mhd_kernels.cuh")).read())
    fns = _functions(text)
    early = set(re.findall(r"launch_step\((k_\w+)", text)) | {"k_finish_dt"}
    assert {"k_flux_pcm", "k_recon3", "k_flux_hlld_r", "k_emf_r", "k_update_half", "k_update_full"} <= early
    todo, seen = set(early), set()
    while todo:
        name = todo.pop()
        seen.add(name)
        body = fns[name]
        assert not re.search(r"__ldg|ld\.global\.nc|\bldg\b", body), name
        if name == "load_dir":  # (two overloads: the kernels' one takes the table of pointers)
            body = body[body.index("Fields<const T, 8>"):]
        assert not re.search(r"\bconst\s+\w+\s*\*\s*__restrict__", body), name
        todo |= {f for f in re.findall(r"\b(\w+)\s*(?:<[^;(){}]*>)?\s*\(", body) if f in fns} - seen
    assert {"load_dir", "edge_field_r", "hydro_update", "face_update", "flux_hlld_cell"} <= seen


@pytest.mark.gpu
@pytest.mark.parametrize("precision", ["fp64", "fp64_df", "fp32_bulk"])
@pytest.mark.parametrize("n", [(33, 20, 17), (4, 5, 16500)])
def test_replay_and_repeat(precision, n):
    import torch

    from paper_2402_05240_gb300 import inputs as I
    from paper_2402_05240_gb300 import mhd
    U0 = torch.from_numpy(np.ascontiguousarray(I.turbulent_box(I.Box(*n), seed_v=3, seed_b=4, kmax=4))).cuda()
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s):
        sim = mhd.Sim(*n, cfl=0.3, recon="ppmc", precision=precision, stream=s.cuda_stream)
        A, B, C = U0.clone(), U0.clone(), U0.clone()
        sim.run(A, 4)
        sim.run(B, 4)
        s.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=s):
            sim.run(C, 4)
        graph.replay()
        s.synchronize()
    assert bool(torch.isfinite(A).all())
    assert torch.equal(A, B) and torch.equal(A, C)


@pytest.mark.gpu
@pytest.mark.parametrize("precision", ["fp64", "fp64_df", "fp32_bulk"])
def test_two_contexts_side_by_side(precision):
    """Two contexts on two streams, their runs enqueued in turn, give the bits
    of runs by themselves."""
    import torch

    from paper_2402_05240_gb300 import inputs as I
    from paper_2402_05240_gb300 import mhd
    shapes = [(33, 20, 17), (48, 9, 21)]
    U0 = [torch.from_numpy(np.ascontiguousarray(I.turbulent_box(I.Box(*n), seed_v=3 + i, seed_b=4, kmax=4))).cuda()
          for i, n in enumerate(shapes)]
    alone = []
    for n, u in zip(shapes, U0):
        sim, A = mhd.Sim(*n, cfl=0.3, recon="ppmc", precision=precision), u.clone()
        for _ in range(10):
            sim.run(A, 3)
        torch.cuda.synchronize()
        alone.append(A)
    streams = [torch.cuda.Stream() for _ in shapes]
    sims = [mhd.Sim(*n, cfl=0.3, recon="ppmc", precision=precision, stream=s.cuda_stream)
            for n, s in zip(shapes, streams)]
    got = [u.clone() for u in U0]
    torch.cuda.synchronize()
    for _ in range(10):
        for sim, A in zip(sims, got):
            sim.run(A, 3)
    torch.cuda.synchronize()
    assert all(torch.equal(a, b) for a, b in zip(alone, got))
