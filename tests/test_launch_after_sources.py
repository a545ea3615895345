"""Kernels launched before their stream's previous kernel has ended (launch_after):
they wait for it in their first statement, and of what they read only tables made
before the render's first kernel are declared unchanging (__restrict__)."""
import glob
import os
import re

from paper_2510_12901_gb300 import _build

# sensor tables, scene planes and the caller's poses: written before the projection,
# which is launched without overlap
TABLES = {"const float4 pix", "const float4 pix2", "const double tile_dir",
          "const float tile_basis", "const LidarItem items", "const uint32_t item_rays",
          "const float4 ray_e", "const float2 ray_tau", "const double item_u",
          "const double item_ref", "const uint2 tile_items", "const LidarItemRays tab",
          "const float planes", "const float poses"}


def _kernels():
    """(name, parameters, body) of every __global__ function."""
    for path in sorted(glob.glob(os.path.join(_build.CSRC, "*.cu*"))):
        src = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"__global__\s+void\s+(?:__launch_bounds__\([^;{]*?\)\s*)?(k_\w+)\(", src):
            end = src.index("{", m.end())
            yield m.group(1), src[m.end():end], src[end + 1:src.index("\n}", end)]


def test_kernels_launched_after_wait_first():
    launched = set()
    for path in glob.glob(os.path.join(_build.CSRC, "*.cu")):
        for args in re.findall(r"launch_after\(([^;]*?)\bst,", open(path).read()):
            launched |= set(re.findall(r"\bk_\w+", args))
    # launched through a variable
    launched -= {"k_off"}
    launched |= {"k_pair_offsets", "k_render_camera", "k_param_grads"}
    waits = {}
    for name, params, body in _kernels():
        waits[name] = body.strip().startswith("after_previous();")
        assert waits[name] or "after_previous" not in body, name
        if not waits[name]:
            continue
        for p in params.split(","):
            m = re.match(r"\s*(const\s+\w+)\s*\*\s*__restrict__\s*(\w+)", p)
            assert m is None or f"{m.group(1)} {m.group(2)}" in TABLES, (name, p.strip())
    assert len(launched) >= 15 and all(waits[k] for k in launched), launched
    assert {k for k, w in waits.items() if w} == launched
