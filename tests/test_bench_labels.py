"""The kernel names of the bench's apply objects: in FP64 schedule code 4 runs the fixed-point
kernel and code 5 the staged one, in FP32 both run the staged one."""
import bench


def test_labels_name_what_runs():
    assert bench.kernel_name(4, 3, 8) == "k_apply_fix<4,double>"
    assert bench.kernel_name(5, 4, 8) == "k_apply_stage<5,double,double,4,1,0>"
    assert bench.kernel_name(4, 3, 4) == "k_apply_stage<4,float,float,2,1,0>"
    # the fixed-point kernel takes no other kernel's traffic
    assert bench.captured_traffic(bench.kernel_name(4, 3, 8)) is None
