"""Kernels launched as programmatic dependents are resident before the kernel
before them has ended, so __ldg (ld.global.nc, defined for memory that nothing
writes during the kernel's whole lifetime) may name setup tables only: never a
field, a spectrum, its scales, a partial projection or mode columns."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1111_4971_gb300", "csrc")

# the setup tables that each source of such a kernel reads with __ldg
TABLES = {
    "modes.cu": set(),
    "modes_z.cu": {"zp"},                       # z recurrences
    "modes_sums.cu": {"sy", "p", "a.sx"},       # sine tables (p: a row of the y table)
    "modes_split.cu": {"tb", "a.scale.rows"},        # digit fragments, row scales
    "zfft_impl.cuh": {"w2", "a.w2_z"},          # phases
    "tdst_impl.cuh": {"tw", "grow"},            # twiddles, Green spectrum
    "fft_common.cuh": {"tw"},
}


def source(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def ldg_operands(text):
    for m in re.finditer(r"__ldg\(", text):
        depth, at = 1, m.end()
        while depth:
            depth += {"(": 1, ")": -1}.get(text[at], 0)
            at += 1
        arg = re.sub(r"reinterpret_cast<[^>]*>", "", text[m.end():at - 1]).lstrip("&( ")
        yield re.match(r"[\w.]+", arg).group(0)


def test_dependent_kernels_read_only_tables_through_ldg():
    for name, tables in TABLES.items():
        assert set(ldg_operands(source(name))) <= tables, name


def test_every_dependent_kernel_is_listed_and_waits():
    for name in sorted(os.listdir(CSRC)):
        text = source(name)
        if "launch_stage(" in text and name != "fft_common.cuh":
            assert "wait_stage()" in text, name
            # zfft.cu and transverse_sym.cu launch the routines of their headers
            assert name in TABLES or name in ("zfft.cu", "transverse_sym.cu"), name
