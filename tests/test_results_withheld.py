"""A step or a batch run whose kernels reported an error writes nothing into the caller's arrays: the kernels that
write results, compiled for the host, with the pass over the cells replaced by a counter."""
import pytest

from device_code import compile_host, definition, source

STUBS = """
struct dim { int x; };
static dim threadIdx{0}, blockIdx{0}, blockDim{1}, gridDim{1};
struct DevStats { unsigned err = 0, bad_input = 0; };
struct FieldCheck {};
struct FieldJob { double* gamma_out = nullptr; double* heat = nullptr; const FieldCheck* valid = nullptr; const unsigned long long* more = nullptr; DevStats* st = nullptr; unsigned block0 = 0; };
struct FieldOut { double* gamma = nullptr; double* heat = nullptr; };
static int written = 0;
static void finalize_cells(const FieldJob&, int64_t, int64_t) { ++written; }
static int job_of_block(const FieldJob*, int) { return 0; }
static void atomicOr(unsigned* p, unsigned v) { *p |= v; }
"""
MAIN = """
extern "C" int step(unsigned bad, unsigned err, unsigned left) {
    DevStats st; st.err = err; st.bad_input = bad;
    unsigned long long more = left;
    FieldCheck chk; FieldJob j; j.valid = &chk; j.st = &st; j.more = &more;
    written = 0; finalize_kernel(j); return written;
}
extern "C" int batch(unsigned run_err, unsigned solve_err) {
    DevStats st[3]; st[2].err = solve_err;
    FieldJob jobs[4]; FieldOut outs[3]; unsigned err = run_err;
    fold_errors_kernel(st, 3, &err);
    written = 0; finalize_many_kernel(jobs, outs, &err, 3); return written;
}
"""


@pytest.fixture(scope="module")
def dev(tmp_path_factory):
    f, b = source("fields.cu"), source("batch.cu")
    body = "".join(definition(f, "__global__ void __launch_bounds__(kBlock) " + k) for k in ("finalize_kernel(", "finalize_many_kernel("))
    return compile_host(tmp_path_factory.mktemp("withheld"), STUBS + body + definition(b, "__global__ void fold_errors_kernel(") + MAIN)


@pytest.mark.parametrize("left", [0, 7])
@pytest.mark.parametrize("bad,err", [(0, 0), (1, 0), (0, 1), (0, 2), (3, 4)])
def test_step(dev, bad, err, left):
    assert dev.step(bad, err, left) == int(bad == 0 and err == 0 and left == 0)


@pytest.mark.parametrize("run_err,solve_err", [(0, 0), (4, 0), (0, 1), (2, 1)])
def test_batch(dev, run_err, solve_err):
    assert dev.batch(run_err, solve_err) == int(run_err == 0 and solve_err == 0)
