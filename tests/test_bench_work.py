"""The work that bench.py charges to a pipe, per active (bin, detector). No GPU."""
import os
import re

import bench

CSRC = os.path.join(bench.ROOT, "paper_2601_02336_gb300", "csrc")


def test_fp64_path_is_charged_what_its_kernel_does():
    """The FP64 path's carrier, data product and moments are integer work: its FP64 share is the phase (7.3 FLOP with
    three detectors) and the per-particle phases, and the pipe that binds is the integer one, which has no measured
    peak, so no fraction of another pipe's is reported for it."""
    assert bench.work("fp64")["flop"] < 8.0
    for kernel, workload in (("nuts", "bbh11"), ("loglike", "bbh11"), ("loglike", "bns")):
        f64, f32, _ = bench.counted(kernel, "fp64", workload)
        assert f64 < 20.0 and f32 < 1.0
    assert bench.binding_pipe("fp64", 7.5, 0.0, 1.05, 76.6) == ("imad", 93.0, None)
    assert bench.binding_pipe("mixed", 2.96, 113.0, 1.05, 76.6)[0] == "fp64"
    assert bench.binding_pipe("split", 0.27, 132.7, 1.05, 76.6)[0] == "fp32"


def test_counts_are_keyed_to_every_device_source():
    """Each header that a counted kernel's unit includes, directly or not, is in the hash (the host-side context and
    the public header aside)."""
    for kernel, unit in (("nuts", "nuts_kernel.cuh"), ("loglike", "loglike_kernel.cuh")):
        seen, todo = set(), [unit]
        while todo:
            f = todo.pop()
            if f in seen or f == "context.cuh" or "/" in f:
                continue
            seen.add(f)
            todo += re.findall(r'#include "([^"]+)"', open(os.path.join(CSRC, f)).read())
        assert seen == set(bench.COUNTED_SOURCES[kernel])
