"""The library's host path on devices that do not exist: host/fake_cudart.c stands in for the CUDA runtime (preloaded in
a child process), so that what a call launches, on which device and under which limits, can be checked without a GPU and
for more devices than one."""
import json
import os
import shutil
import subprocess
import sys

import pytest

from paper_2507_18181_b200 import build

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)

PRELUDE = """
import ctypes as C, json, os, sys
sys.path.insert(0, %r)
from paper_2507_18181_b200 import binding as B
fake = C.CDLL(os.environ["LD_PRELOAD"])
fake.fake_launch.restype = C.c_char_p

def launches(since=0):
    out = []
    for i in range(since, fake.fake_launches()):
        dev, x, y, z, name = fake.fake_launch(i).decode().split(" ", 4)
        out.append((int(dev), (int(x), int(y), int(z)), name))
    return out

keep = []
def buf(n):
    b = (C.c_char * (n + 256))()
    keep.append(b)
    return (C.addressof(b) + 255) // 256 * 256

def model(head_dim=128, heads=8, kv_heads=2, d=512, ffn=1408, layers=2, vocab=1000, page=16, positions=4096):
    wp = B.WeightPtrs(embed=16, lm_head=16, g_final=16)
    arr = (C.c_void_p * layers)(*[16] * layers)
    keep.append(arr)
    for f in ("wqkv", "wo", "wgu", "wd", "g_attn", "g_ffn"):
        setattr(wp, f, C.cast(arr, C.POINTER(C.c_void_p)))
    return B.specasr_model_create(B.ModelConfig(n_layers=layers, d_model=d, n_heads=heads, n_kv_heads=kv_heads, head_dim=head_dim,
                                                ffn=ffn, vocab=vocab, page_size=page, max_positions=positions, rms_eps=1e-6,
                                                rope_base=1e4, gemm_path=0), wp)

def cache(m, pages=64, nodes=256):
    return B.specasr_kv_create(m, buf(16), buf(16), pages, buf(4 * pages), pages, buf(B.specasr_workspace_bytes(m, nodes)), nodes)

def verify(m, kv, n):
    B.specasr_verify_tree(m, kv, 16, 16, n, 16, 16, 16, 0)
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    """run(code): the JSON that `code`, run behind PRELUDE in front of the stand-in runtime, prints."""
    build.build()
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    so = str(tmp_path_factory.mktemp("host") / "fake_cudart.so")
    subprocess.run([shutil.which("gcc") or "cc", "-O1", "-shared", "-fPIC", "-I", os.path.join(cuda, "include"),
                    os.path.join(HERE, "host", "fake_cudart.c"), "-o", so], check=True)

    def call(code):
        res = subprocess.run([sys.executable, "-c", PRELUDE % ROOT + code], capture_output=True, text=True, timeout=120,
                             env=dict(os.environ, LD_PRELOAD=so, CUDA_VISIBLE_DEVICES=""))
        assert res.returncode == 0, res.stdout + res.stderr
        return json.loads(res.stdout)
    return call


@pytest.mark.parametrize("head_dim,heads,kv_heads,d", [(128, 8, 2, 512), (64, 4, 4, 256), (128, 32, 8, 4096)])
def test_models_on_two_devices_of_one_process(run, head_dim, heads, kv_heads, d):
    """A kernel's shared-memory limit belongs to one device: calls of all sizes run on the second device too."""
    got = run(f"""
for dev in (0, 1):
    fake.fake_set_device(dev)
    m = model(head_dim={head_dim}, heads={heads}, kv_heads={kv_heads}, d={d})
    kv = cache(m)
    B.specasr_prefill_embeds(m, kv, 16, 300, 0)
    for n in (1, 9, 33, 64, 65, 128, 129, 256):
        verify(m, kv, n)
print(json.dumps([[l[2] for l in launches() if l[0] == dev] for dev in (0, 1)]))
""")
    assert got[0] == got[1] and any("k_stack" in k for k in got[0]) and any("k_proj" in k for k in got[0])


def test_a_device_that_refuses_the_shared_memory_refuses_the_model(run):
    got = run("""
fake.fake_refuse_limit(1, 1)
out = []
for dev in (0, 1):
    fake.fake_set_device(dev)
    try:
        out.append(bool(model()))
    except B.SpecasrError as e:
        out.append(e.status)
print(json.dumps(out))
""")
    assert got == [True, 7]          # SPECASR_ERR_CUDA


def test_accept_slices_follow_the_device(run):
    """Slices of the vocabulary per row: about four blocks per SM of the device at hand, at most 64 and at most one per 1024
    tokens, from the smallest to the widest vocabulary."""
    cases = [(1, 32000), (64, 32000), (256, 32000), (5, 70000), (3, 1), (1, 2**31 - 1)]
    got = run(f"""
out = []
for dev, sms in ((0, 148), (1, 18)):
    fake.fake_set_device(dev)
    fake.fake_set_sm_count(dev, sms)
    for n, vocab in {cases}:
        at = fake.fake_launches()
        B.specasr_accept_logits_static(16, vocab, 16, 16, n, 16, 16, 16, 0)
        out.append(launches(at)[0][1])
print(json.dumps(out))
""")
    want = [[min(-(-4 * sms // n), 64, (vocab - 1) // 1024 + 1), n, 1] for sms in (148, 18) for n, vocab in cases]
    assert got == want


@pytest.mark.parametrize("shape", ["", "head_dim=64, heads=14, kv_heads=2, d=896, ffn=4864, vocab=32000, layers=24",
                                   "heads=32, kv_heads=8, d=4096, ffn=14336, vocab=32000, layers=32"])
def test_a_workspace_grows_with_the_nodes_of_a_tree(run, shape):
    """Twice the nodes, twice the bytes at most: large context-fill chunks live in what a tree has."""
    got = run(f"""
m = model({shape})
print(json.dumps([B.specasr_workspace_bytes(m, n) for n in (16, 32, 64, 128, 256)]))
""")
    assert all(a < b <= 2 * a for a, b in zip(got, got[1:])), got


def test_large_fill_chunks_are_planned_on_devices_of_any_size(run):
    got = run("""
out = []
for dev, sms in ((0, 16), (1, 148), (2, 300)):
    fake.fake_set_device(dev)
    fake.fake_set_sm_count(dev, sms)
    m = model(head_dim=64, heads=14, kv_heads=2, d=896, ffn=4864)
    kv = cache(m)
    at = fake.fake_launches()
    B.specasr_prefill_embeds(m, kv, 16, 750, 0)
    out.append([grid for _, grid, name in launches(at) if "k_tree_attention" in name])
print(json.dumps(out))
""")
    assert all(len(g) == 1 and 0 < g[0][0] <= sms for g, sms in zip(got, (16, 148, 300))), got
