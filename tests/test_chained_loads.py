"""Kernels that may start while their predecessor still writes (they call wait_previous) read what
earlier kernels write by plain loads: no const __restrict__ parameter but the constant tables, which
the compiler may turn into non-coherent loads, and no explicit __ldg of anything but those."""
import pathlib
import re

CSRC = pathlib.Path(__file__).resolve().parent.parent / "paper_2404_02783_gb300" / "csrc"
TABLES = {"kf_arr", "scale_arr"}  # written when a context or batch is made


def _kernels():
    for path in sorted([*CSRC.glob("*.cu"), *CSRC.glob("*.cuh")]):
        text = path.read_text()
        for part in re.split(r"(?=__global__ void)", text)[1:]:
            m = re.search(r"(k_\w+)\(", part)
            head, body = part[m.end():].split("{", 1)
            yield path.name, m.group(1), head, body


def _chained():
    return [k for k in _kernels() if "wait_previous()" in k[3]]


def test_there_are_chained_kernels():
    assert len(_chained()) >= 9


def test_inputs_of_chained_kernels_are_plain_loads():
    for file, name, head, _ in _chained():
        for param in re.findall(r"const[^,()]*__restrict__\s+(\w+)", head):
            assert param in TABLES, (file, name, param)
    # read and never written, a restrict pointer counts as constant too
    x_cols = next(head for _, name, head, _ in _chained() if name == "k_x_cols")
    assert re.search(r"cplx<T>\*\s+data,", x_cols)


def test_no_explicit_non_coherent_load():
    for file, name, _, body in _chained():
        if file != "fft_impl.cuh":  # there the tables alone, through TwGlobal and SpecOp::amp
            assert "__ldg" not in body.split("\n}\n")[0], (file, name)
    assert "__ldg" not in (CSRC / "update_dev.cuh").read_text()  # the update's particle step
