"""Rules on the CUDA sources that no run can show to be kept."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2112_02644_b200", "csrc")


def sources():
    return {os.path.basename(f): re.sub(r"//[^\n]*", "", open(f).read()) for f in glob.glob(os.path.join(CSRC, "*.cu*"))}


def test_what_the_kernel_before_writes_is_read_by_ordinary_loads():
    # kernels become resident while the kernel before them in the stream is still writing: loads that ask for data
    # nothing writes meanwhile (ld.global.nc) are not for them, but for the stash the update reads
    src = sources()
    assert {f for f, text in src.items() if re.search(r"__ldg|\.nc\b", text)} <= {"memory.cu"}
    assert set(re.findall(r"__ldg\(([^+(]*)", src["memory.cu"])) <= {"rp ", "reinterpret_cast<const float4*>"}
    for f, text in src.items():
        for params in re.findall(r"__global__[^{;]*?\bk_\w+\(([^)]*)\)", text):
            assert not re.search(r"const[^,]*__restrict__", params), (f, params)


def test_a_peer_is_known_to_have_started_before_its_shared_memory_is_written():
    # the CTAs of a cluster need not begin together: a barrier all of them have arrived on comes before the first store
    stores, checked = r"peer_store|peer_arrive|send_column\(|score_slots\(|slice_norm\(|deliver\(", set()
    for f, text in sources().items():
        for body in re.split(r"\n__(?:global|device)__|\ntemplate", text):
            store = re.search(stores, body)
            name = re.search(r"\b(k_\w+|tables_of_lone_stream)\(", body)
            if not (store and name and name.start() < body.index("{")):
                continue
            wait = re.search(r"cluster_wait\(\)|cluster_sync_all\(\)", body)
            assert wait and wait.start() < store.start(), (f, name.group(1))
            checked.add(name.group(1))
    assert checked >= {"k_lookup_nchw", "k_lookup_sparse", "k_lookup_frame", "k_lookup_frame_nhwc", "k_encode_nhwc", "k_score_shared",
                       "tables_of_lone_stream"}


def test_a_wait_that_gives_up_is_heeded():
    # no vector and no decision is made of what has not arrived, and a CTA that peers store into (counted on its barrier) stays
    # for a second wait
    for f, text in sources().items():
        if f != "lookup.cu":   # (its self-test of the waits has nothing to make of the result)
            # ((void), and the ring's copies that are left to land: the CTA only stays)
            assert not re.findall(r"(?<!\(void)[;{})]\s*mbar_wait_[\w<>]+\(&(?!full\[s\])\w+[^;]*", text), f
    encode = sources()["encode.cu"]
    for bar in ("delivered", "summed"):
        assert set(re.findall(r"([\w<>]+)\(&%s, 0, [\w.]*status\)" % bar, encode)) == {"mbar_wait_arrivals<true>"}
