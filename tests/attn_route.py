"""The attention kernel that a launch runs, from the library's own rule (attn_choice.h, compiled for the host): tests that are about one kernel
say so."""
import ctypes
import functools
import os
import subprocess
import tempfile

from paper_2505_13254_b200 import build

SOURCE = r"""
#include "attn_choice.h"
extern "C" int route(int blocks, int mblocks, int sm_count, int tiles) {
    int cap[ATT_MAX_SPLIT + 1];
    for (int s = 1; s <= ATT_MAX_SPLIT; ++s) cap[s] = sm_count / s * s;
    const AttnChoice c = attn_choice(blocks, mblocks, sm_count, tiles, cap);
    return c.duo ? c.splits : c.follow ? -1 : 0;
}
extern "C" int operand(int blocks, int mblocks, int sm_count, int tiles, int tree_tiles) {
    int cap[ATT_MAX_SPLIT + 1];
    for (int s = 1; s <= ATT_MAX_SPLIT; ++s) cap[s] = sm_count / s * s;
    const AttnChoice c = attn_choice(blocks, mblocks, sm_count, tiles, cap);
    return q_from_tensor_memory(blocks, mblocks, sm_count, tiles, tree_tiles, c) ? c.splits : 0;
}
"""


@functools.lru_cache(None)
def _library():
    where = tempfile.mkdtemp()
    src, so = os.path.join(where, "route.cpp"), os.path.join(where, "route.so")
    with open(src, "w") as f:
        f.write(SOURCE)
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", build.CSRC, src, "-o", so])
    return ctypes.CDLL(so)


def _shape(batch, nodes, hq, hkv, longest, sm_count):
    if sm_count is None:
        import torch
        sm_count = torch.cuda.get_device_properties(0).multi_processor_count
    mblocks = (hq // hkv * nodes + 127) // 128
    return batch * hkv * mblocks, mblocks, sm_count, (longest + 63) // 64


def route(batch, nodes, hq, hkv, longest, sm_count=None):
    """1 or 2: tree_attn_duo_kernel with so many splits; -1: tree_attn_umma_kernel<true>; 0: tree_attn_umma_kernel<false>."""
    return _library().route(*_shape(batch, nodes, hq, hkv, longest, sm_count))


def splits_with_q_in_tensor_memory(batch, nodes, hq, hkv, longest, sm_count=None):
    """0: every CTA takes the query rows from shared memory; else those of many tiles from tensor memory, and the launch has so many splits (as many
    clusters as SMs allow; the device may run fewer of the largest at once)."""
    return _library().operand(*_shape(batch, nodes, hq, hkv, longest, sm_count), (nodes + 63) // 64)
