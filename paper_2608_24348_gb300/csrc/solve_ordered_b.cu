// solve_ordered_b.cu -- the ordered solver of Taylor-Green steps, N + 1 in {2, 5, 8}.
#include "solver_ordered.cuh"

int sem_solve_ordered_b(const SolveParams<8> &p, int n, int sms, cudaStream_t s)
{
    switch (n) {
        case 2: return ordered::launch<2>(p, sms, s);
        case 5: return ordered::launch<5>(p, sms, s);
        case 8: return ordered::launch<8>(p, sms, s);
        default: return SEM_ERR_ARG;
    }
}

int sem_solve_ordered_tables_b(int n, const double *D) { return solver_upload_tables(n, D); }
