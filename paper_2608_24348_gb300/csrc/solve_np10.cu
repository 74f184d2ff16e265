// solve_np10.cu -- persistent solver kernels for order N = 9 (up to 8 problems).
#include "solver.cuh"

int sem_solve_launch_np10(const SolveParams<8> &p, int mode, int sms, cudaStream_t s)
{
    switch (mode) {
        case MODE_F64: return launch_solve<8, MODE_F64, 10>(p, sms, s);
        case MODE_F64N: return launch_solve<8, MODE_F64N, 10>(p, sms, s);
        case MODE_F32: return launch_solve<8, MODE_F32, 10>(p, sms, s);
        case MODE_TC: return launch_solve<8, MODE_TC, 10>(p, sms, s);
        default: return SEM_ERR_ARG;
    }
}

int sem_solve_tables_np10(const double *D) { return solver_upload_tables(10, D); }
