"""Sizes the host plan chooses, from host_plan.cpp alone (no GPU)."""
import ctypes
import os
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))


def _call(name, geom, cluster_size, transforms, folder, count):
    from paper_1302_3734_gb300 import build, geometry_struct
    lib = os.path.join(str(folder), "libhostplan.so")
    if not os.path.exists(lib):
        subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", f"-I{build.INCLUDE}", f"-I{build.CSRC}",
                        f"-I{os.path.join(build._cuda_home(), 'include')}", os.path.join(HERE, "host_plan_probe.cpp"),
                        os.path.join(build.CSRC, "host_plan.cpp"), "-o", lib], check=True)
    g, keep = geometry_struct(geom)
    out = (ctypes.c_longlong * count)()
    st = getattr(ctypes.CDLL(lib), name)(ctypes.byref(g), cluster_size, transforms, out)
    assert st == 0, st
    return list(out)


def gather_sizes(geom, cluster_size, transforms, folder):
    """(bands, shared memory, terms of the largest band) of the separate gather."""
    return _call("host_plan_gather", geom, cluster_size, transforms, folder, 3)


def coarse_sides(geom, cluster_size, transforms, folder):
    """Per layer, the side of the block that one CTA of its cluster finishes."""
    return _call("host_plan_coarse", geom, cluster_size, transforms, folder, len(geom["layers"]))


def forward_ctas(geom, cluster_size, transforms, folder):
    """(CTAs of one forward launch, CTAs up to which a launch takes the small form)."""
    n = _call("host_plan_forward", geom, cluster_size, transforms, folder, 1)[0]
    return n, ctypes.CDLL(os.path.join(str(folder), "libhostplan.so")).host_plan_forward_small()
