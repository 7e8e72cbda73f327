"""Which kernels a step is made of, without a device: the library runs over a CUDA runtime that does nothing but note the launches
(tests/host/fake_cudart.c).  The row counts that steps leave for the host are written by the test, as the kernels would.  Each test is a
process of its own, as the library takes the runtime that it finds first."""
import os
import subprocess
import sys
import textwrap

import pytest

from paper_2509_23094_b200 import build

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)

PRELUDE = """
import ctypes as C, sys, types
from dataclasses import replace
sys.modules["torch"] = types.ModuleType("torch")          # (only names of it are in annotations)
sys.path.insert(0, sys.argv[1])
from paper_2509_23094_b200 import binding, inputs
lib, fake = binding.load(), C.CDLL("libcudart.so.12")
fake.fake_log.restype = C.c_char_p
fake.fake_host_words.restype = C.POINTER(C.c_int32)
fake.fake_refuse.argtypes = [C.c_char_p, C.c_int]


class Ctx:
    def __init__(self, shape, batch, seq, flags=0):
        cfg = binding.make_config(shape, batch, seq, flags=flags)
        self.batch, self.seq, self.n = batch, seq, 0
        w, at = binding.Weights(), (C.c_void_p * shape.n_layers)(*[1 << 20] * shape.n_layers)
        for name in ("wqkv", "bqkv", "wo", "w_gate", "w_up", "w_down", "g_attn", "g_ffn"):
            setattr(w, name, C.cast(at, C.POINTER(C.c_void_p)))
        w.g_final = w.w_lm = 1 << 20
        self.handle = C.c_void_p()
        need = lib.d2c_workspace_bytes(C.byref(cfg))
        binding._check(lib.d2c_create(C.byref(cfg), C.byref(w), 1 << 30, need, None, C.byref(self.handle)))
        self.words = fake.fake_host_words()

    def step(self, k, p, rows, block=(0, 0)):
        # the kernels of a step that then finds `rows` rows
        fake.fake_clear()
        a = binding.StepArgs(self.batch, self.seq, 1 << 21, 1 << 22, None, None, k, p, None, None, *block)
        rc = lib.d2c_step(self.handle, C.byref(a), None)
        slot = 2 * (self.n & 1)
        self.words[slot], self.words[slot + 1] = rows, self.n
        self.n += 1
        if rc:
            return rc
        names = fake.fake_log().decode().split()
        assert names
        one = [n for n in names if "small_step_kernel" in n]
        assert not one or len(names) == 1
        return "one" if one else "separate"
"""


@pytest.fixture(scope="module")
def runtime(tmp_path_factory):
    build.build()
    d = tmp_path_factory.mktemp("fake_cuda")
    (d / "v.map").write_text("libcudart.so.12 { *; };\n")
    subprocess.run(["gcc", "-shared", "-fPIC", "-O1", "-Wall", "-Werror", "-o", str(d / "libcudart.so.12"), os.path.join(HERE, "host", "fake_cudart.c"),
                    "-Wl,-soname,libcudart.so.12", f"-Wl,--version-script={d / 'v.map'}"], check=True)
    return str(d)


def _run(runtime, body):
    r = subprocess.run([sys.executable, "-c", PRELUDE + textwrap.dedent(body), ROOT], env=dict(os.environ, LD_LIBRARY_PATH=runtime),
                       stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True, timeout=120)
    assert r.returncode == 0, r.stdout


def test_small_steps_go_by_the_count_of_a_step_that_asked_for_no_less(runtime):
    """Few rows behind few of the same call: one launch.  A call that asks for more rows of stage 1 or for more of the mass than the step
    before did, as the select-all step of the next request does, takes the separate kernels, whatever that one found."""
    _run(runtime, """
    c = Ctx(inputs.TOY, 1, 2048)
    few = (16, 0.1, 40)
    assert c.step(2048, 1.0, 2048) == "separate"
    assert c.step(*few) == "separate"                                    # behind many
    assert c.step(*few) == "one" and c.step(*few) == "one"
    for more in ((2048, 1.0), (16, 0.9), (17, 0.1), (10 ** 6, 0.1)):
        assert c.step(*more, 2048) == "separate", more
        assert c.step(*few) == "separate"                                # behind many
        assert c.step(*few) == "one"
    assert c.step(8, 0.05, 20) == "one" and c.step(16, 0.05, 30) == "separate" and c.step(16, 0.05, 30) == "one"
    assert c.step(16, 0.0, 2000) == "one" and c.step(16, 0.0, 16) == "separate" and c.step(16, 0.0, 16) == "one"      # (found many: the next goes by it)
    assert c.step(2048, 0.0, 32, block=(100, 132)) == "separate"          # of a block 32 at most, more than 16
    assert c.step(2048, 0.0, 32, block=(132, 164)) == "one" and c.step(2048, 0.0, 32, block=(0, 32)) == "one"
    assert c.step(2048, 0.0, 32, block=(2040, 4096)) == "one"             # eight positions of it are there
    assert c.step(2048, 0.0, 32, block=(164, 196)) == "separate"
    assert c.step(2048, 0.0, 500) == "separate"
    c = Ctx(inputs.TOY, 1, 128)                                            # room for few rows only
    assert c.step(128, 1.0, 128) == "one" and c.step(8, 0.5, 60) == "one" and c.step(128, 1.0, 128) == "one"
    c = Ctx(inputs.TOY, 1, 2048, flags=16)                                 # a flag that asks for the separate kernels
    assert all(c.step(*few) == "separate" for _ in range(4))
    """)


def test_a_step_asks_once_for_the_count_of_the_one_before(runtime):
    """Whether the stream is captured, and the event behind the selection of the step before: each a call of 0.5 us in front of the step's
    first launch, made once whichever way the step then goes."""
    _run(runtime, """
    for shape in (inputs.TOY, inputs.TOY_HD128):
        c = Ctx(shape, 1, 2048)
        for i in range(4):
            assert c.step(2048, 1.0, 2048) == "separate"
            assert fake.fake_asked() == 2, (shape.name, i)
    c = Ctx(inputs.TOY, 1, 2048)
    assert [c.step(16, 0.1, 40) for _ in range(3)] == ["separate", "one", "one"]
    fake.fake_asked()
    assert c.step(16, 0.1, 40) == "one" and fake.fake_asked() == 1           # (the count of a step in one launch is behind no event)
    """)


def test_a_context_counts_clusters_for_itself(runtime):
    """What the first context of a process found while its kernel's attributes could not be set, or were not set yet by the thread that had
    begun to, is not what the others find."""
    _run(runtime, """
    fake.fake_unset(1)
    a = Ctx(inputs.TOY, 1, 128)
    fake.fake_unset(0)
    b = Ctx(inputs.TOY, 1, 128)
    assert a.step(128, 1.0, 128) == "separate" and b.step(128, 1.0, 128) == "one"
    """)


# cudaErrorInvalidValue, cudaErrorLaunchOutOfResources, cudaErrorIllegalAddress, cudaErrorCooperativeLaunchTooLarge, cudaErrorInvalidClusterSize
@pytest.mark.parametrize("code,goes_on", [(1, False), (701, True), (700, False), (720, True), (912, True)])
def test_a_refused_one_launch_step_takes_the_separate_kernels(runtime, code, goes_on):
    """A GPU that has fewer SMs than were counted (a part of one) refuses a launch that needs all its CTAs at once: the step is done by the
    separate kernels, and so are those behind it.  Any other error is the call's answer, and nothing else is enqueued."""
    _run(runtime, f"""
    c = Ctx(inputs.TOY, 1, 128)
    assert c.step(128, 1.0, 128) == "one"
    fake.fake_refuse(b"small_step_kernel", {code})
    if {goes_on}:
        assert c.step(8, 0.5, 60) == "separate" and fake.cudaGetLastError() == 0
        fake.fake_refuse(b"", 0)
        assert c.step(8, 0.5, 60) == "separate"
    else:
        assert c.step(8, 0.5, 60) == binding.D2C_ECUDA and fake.fake_log() == b""
        c.n -= 1                                                           # (a step that was not enqueued)
        fake.fake_refuse(b"", 0)
        assert c.step(8, 0.5, 60) == "one"
    """)


def test_attention_of_more_query_heads_than_a_tile_has_rows(runtime):
    """129 query heads and more of a K/V head do not share a tile of 128 rows; each then has tiles of its own, on the tensor cores like any."""
    _run(runtime, """
    for heads in (128, 129, 160, 512):
        c = Ctx(replace(inputs.TOY_HD128, name="many", n_layers=1, n_q_heads=heads, n_kv_heads=1), 1, 300)
        for rows in (300, 20, 20):
            assert c.step(16, 0.1, rows) == "separate"
            assert "attn_fwd_tc" in fake.fake_log().decode(), (heads, rows)
    """)


def test_attention_of_few_rows_of_many_long_sequences(runtime):
    """Tiles of a few rows, room for thousands of them in each of many sequences: no dimension of a grid has room for all of them."""
    _run(runtime, """
    for heads, batch in ((32, 64), (32, 66), (128, 16), (64, 32)):
        c = Ctx(replace(inputs.TOY_HD128, name="long", n_layers=1, n_q_heads=heads, n_kv_heads=1), batch, 8192)
        for rows in (8192 * batch, batch, batch, 2 * batch, 4 * batch, 40 * batch):
            assert c.step(1, 0.1, rows) == "separate", (heads, batch, rows, lib.d2c_last_error(c.handle))
    """)


def test_probabilities_of_few_rows_are_numbered_in_turn(runtime):
    """The form of the probabilities kernel that the GPU test of it means to reach, with the rows that it has (p of the known ones)."""
    from test_gpu_branches import IN_TURN
    _run(runtime, f"""
    for layers, batch, seq, heads, kv, p in {IN_TURN}:
        c = Ctx(replace(inputs.TOY_HD128, name="turn", n_layers=layers, n_q_heads=heads, n_kv_heads=kv), batch, seq)
        rows = batch * int(p * (seq - 100))
        forms = []
        for n in (batch * seq, rows, rows, rows):
            c.step(0, p, n)
            forms.append({{name.split("AbarFormE")[1][0] for name in fake.fake_log().decode().split() if "AbarForm" in name}})
        assert forms == [{{"0"}}, {{"0"}}, {{"1"}}, {{"1"}}], (heads, seq, forms)
    """)


def test_places_of_the_forward(runtime):
    """Which form of the forward a step takes: with shared keys places for half of the tiles where those for all would be far more CTAs than
    SMs, for all else; without, by place where one of two places is expected to be taken."""
    from test_gpu_branches import PLACES
    _run(runtime, f"""
    def form(heads, kv, batch, seq, rows):
        c = Ctx(replace(inputs.TOY_HD128, name="places", n_layers=1, n_q_heads=heads, n_kv_heads=kv), batch, seq)
        for n in (batch * seq, rows, rows):
            c.step(20, 0.0, n)
        names = [n for n in fake.fake_log().decode().split() if "attn_fwd_tc" in n]
        return names[0].split("attn_fwd_tc")[1][:13]
    for want, heads, kv, seq in {PLACES}:
        assert form(heads, kv, 1, seq, 20) == want, want
    assert form(4, 2, 1, 570, 194) == "ILb1ELb0ELb1E"
    assert form(32, 32, 5, 215, 100) == "ILb0ELb0ELb1E" and form(32, 32, 5, 700, 100) == "ILb0ELb0ELb0E"
    """)
