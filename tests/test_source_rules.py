"""Properties of the CUDA sources that no run on one GPU can show (read from the text of csrc/, no GPU)."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2605_29707_gb300", "csrc")


def _code(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def test_packed_states_are_published_in_the_size_they_are_read():
    """The GRU's packed states cross CTAs without a barrier: the memory model orders a strong read with a
    strong write of the same 32-bit word, and says nothing of a weak 16-bit write to half of it."""
    code = _code("gru.cu")
    assert "ld.relaxed.gpu.global.v4.u32" in code
    assert re.search(r"hxp\s*\[|__st\w+\(\s*hxp", code) is None
    stores = re.findall(r"(\w+)\(reinterpret_cast<(\w+)\*>\(hxp", code)
    assert stores == [("st_relaxed", "uint32_t")], stores
    assert re.search(r"st_relaxed\(uint32_t\*[^}]*st\.relaxed\.gpu\.global\.u32", code)


def test_kernel_attributes_are_set_per_device():
    """A kernel's attributes belong to a device: only ensure_smem_attr, which keeps what it set by (device,
    kernel) under a lock, sets them, and no launch keeps a flag for the whole process."""
    for name in sorted(os.listdir(CSRC)):
        code = _code(name)
        assert code.count("cudaFuncSetAttribute(") == (2 if name == "api.cu" else 0), name
        assert re.search(r"static\s+bool\s+\w+\s*=", code) is None, name


def test_sizes_of_the_chip_come_from_the_device():
    """No launch rule names the SM count of one chip: it is read from the device (api.cu's 152 is what
    domino_launches_per_step answers for where none is visible)."""
    for name in sorted(os.listdir(CSRC)):
        found = re.findall(r"\b152\b", _code(name))
        assert len(found) == (1 if name == "api.cu" else 0), (name, found)
