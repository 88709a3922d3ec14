"""The key of the benchmark's traffic record: the code of a kernel's sources."""
import bench


def test_key_follows_code_and_not_comments():
    a = "int f(int x) {  // doubles x\n  return 2 * x; /* exact */\n}\n"
    b = "/* doubles */ int f(int x) {\n  return 2 * x;\n}"
    c = "int f(int x) { return 3 * x; }"
    assert bench._code_only(a) == bench._code_only(b)
    assert bench._code_only(a) != bench._code_only(c)
    for tag in ("fp32", "fp64"):
        assert len(bench._kernel_hash(tag)) == 16
