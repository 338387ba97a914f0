"""Rules of the CUDA sources whose breach a run need not show, checked in the text."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2506_08889_b200", "csrc")


def _sources():
    """File name -> its text without comments."""
    found = {}
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        with open(path) as f:
            found[os.path.basename(path)] = re.sub(r"//[^\n]*|/\*.*?\*/", "", f.read(), flags=re.S)
    return found


def test_aligned_cluster_barriers_bring_the_warp_together_first():
    # barrier.cluster.*.aligned behind a branch of some lanes (a rotary pair that two lanes finish, predicated copies)
    # is undefined unless the lanes have met again
    wrapped = 0
    for name, text in _sources().items():
        assert "cluster.sync()" not in text, name
        for m in re.finditer(r"barrier\.cluster\.", text):
            assert re.search(r"__syncwarp\(\);\s*asm volatile\(\"$", text[:m.start()]), (name, text[m.start():m.start() + 40])
            wrapped += 1
    assert wrapped == 2


def _kernel(name):
    """The text of a kernel, from its name to the next kernel's."""
    for text in _sources().values():
        m = re.search(r"\n%s\(|__global__[^;{]*\b%s\(" % (name, name), text)
        if m:
            end = text.find("__global__", m.end())
            return text[m.end():end if end > 0 else len(text)]
    raise AssertionError(name)


def test_weights_are_read_after_the_wait_for_the_kernel_before():
    # that kernel may be the one that writes them
    for name, load in (("kcomp_stream_kernel", r"\bload_w\("), ("step_cluster_kernel", r"\bload_w\("), ("gate_cluster_kernel", r"__ldg\(")):
        text = _kernel(name)
        calls = [m.start() for m in re.finditer(load, text)]
        assert calls and min(calls) > text.index("pdl_wait()"), name


def test_the_one_launch_step_reads_no_compressed_key_through_the_read_only_path():
    # it appends one in the same launch, and the next step starts under its end
    assert not re.search(r"__ldg\(\s*kc\b", _kernel("step_cluster_kernel"))


def test_nothing_is_read_behind_a_wait_that_ran_out():
    # what it stood for need not be there: numbers made of it are no indices.  (Tensor memory is given back all the same.)
    for name, text in _sources().items():
        for m in re.finditer(r"[;{})]\s*mbar_wait\(&sm\.([\w.]+)", text):
            assert m.group(1).endswith("tmem_done"), (name, m.group(0))
    # (the deal of uneven lists: behind a barrier of the hardware, whose warps all come)
    text = _sources()["seer_lists.cu"]
    shares = [m.start() for m in re.finditer(r"\btake_share\(\);", text)]
    assert len(shares) == 2 and all(re.search(r"await_deal\(\w+\);\s*$", text[:at]) for at in shares)
